// dvc_mlp.cuh -- the value network's inference for small batches in one launch:
// features, three dense layers, the output layer and the softmax of 128 rows by
// a cluster of four CTAs.
//
// A batch of a few hundred leaves (a chain of a value-mode search, a server's
// lane, a caller's handful) fills a handful of GEMM tiles, and features, three
// layers and the softmax, one launch after another, each cost their latency: 4-12
// us on 2-6 CTAs.  Here every CTA of a cluster builds the features of the same 128
// rows, then computes 128 of each layer's 512 columns: it streams only its quarter
// of the weights (TMA into a ring, issued ahead of the layers that use them),
// and writes its quarter of the activations into the shared memory of all four
// (distributed shared memory), where the next layer reads them as its A operand.
// Nothing but the states and the probabilities crosses the SMs' edge.
// Accumulation order, epilogues and the order in which partial logits are added
// are those of the layer-by-layer path (dvc_gemm.cuh), so the results are the
// same bits.  What bounds it is latency: of about 52,000 cycles the features take
// 7,400, the three layers' MMAs 14,000 (about 540 a slice of 64 columns, with the
// weights' copies ahead of them), their epilogues 6,800 and the exchanges of
// activations (96 KB out of every SM, fences, waits for the slowest neighbour)
// 14,000.  333 rows: 29 us a call against 50 by layers.
//
// Roles: warps 0-15 features and epilogue, warp 16 copies, warp 17 MMA.  Shared
// memory: H (128 x 512 BF16 in the K-blocked layout: 128 KB) and five 16 KB ring
// slots; the features (128 x 640) take H and the last two slots at first.
//   xready the features stand in shared memory;
//   hfull  all four CTAs' quarters of H are here (per layer);
//   hfree  all four CTAs' MMAs have read what H held, so that it may be overwritten;
//   pfull  the partial logits of this CTA's 32 output rows are here.
// Every wait is bounded; a CTA whose wait gives up latches DVC_E_TIMEOUT and
// still takes part in the cluster's last barrier, which no CTA leaves before its
// neighbours have finished writing into it.
#pragma once
#include "dvc_features.cuh"
#include "dvc_gemm.cuh"

namespace dvc {

constexpr int kMlpCluster = 4;
constexpr int kMlpCols = 128;  // columns of a layer per CTA
constexpr int kMlpSlots = 5;
constexpr uint32_t kMlpSlot = 16384u, kMlpH = 131072u;
constexpr uint32_t kMlpSmem = kMlpH + kMlpSlots * kMlpSlot + 1024u;
constexpr int kMlpThreads = 32 * 18;

struct MlpArgs {
    const float* bias[3];
    const __nv_bfloat16* W4;  // 4 x 512
    const float* b4;
    const dvc_state* states;
    int n;
    float* out;  // n x 4 win probabilities per absolute seat
    int32_t* flags;
    uint64_t wait_ns;
};

__device__ __forceinline__ uint32_t map_cta(uint32_t saddr, uint32_t cta) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(cta));
    return r;
}
__device__ __forceinline__ void st_shared_v4(uint32_t addr, uint4 v) {
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w)
                 : "memory");
}
__device__ __forceinline__ void st_cluster_v4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d)
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t addr) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(addr) : "memory");
}
// ... where no data goes with it.
__device__ __forceinline__ void mbar_arrive_cluster_relaxed(uint32_t addr) {
    asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(addr) : "memory");
}
// mbar_wait with acquire at cluster scope.
__device__ __forceinline__ bool mbar_wait_cluster(uint64_t* bar, uint32_t phase, uint64_t limit_ns) {
    uint64_t t0 = 0;
    for (uint32_t i = 0; i < kWaitLimit; ++i) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(smem_u32(bar)), "r"(phase)
            : "memory");
        if (ok) return true;
        if ((i & 63u) != 63u) continue;
        const uint64_t t = global_ns();
        if (i == 63u) t0 = t;
        else if (t - t0 > limit_ns) return false;
    }
    return false;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Softmax over relative seats 0..P-1 of logits z, written per absolute seat.
__device__ __forceinline__ void softmax_seats(const dvc_state& s, float4 z, float* o) {
    const int P = (s.nplayers >= 2 && s.nplayers <= 4) ? s.nplayers : 2;
    const int cur = s.cur < P ? s.cur : 0;
    const float zz[4] = {z.x, z.y, z.z, z.w};
    float mx = zz[0];
    for (int r = 1; r < P; ++r) mx = fmaxf(mx, zz[r]);
    float e[4], sum = 0.0f;
    for (int r = 0; r < P; ++r) {
        e[r] = expf(zz[r] - mx);
        sum += e[r];
    }
    o[0] = o[1] = o[2] = o[3] = 0.0f;
    for (int r = 0; r < P; ++r) o[(cur + r) % P] = e[r] / sum;
}

// Ring order of the weight slices (10 of layer 1, 8 each of layers 2 and 3):
// layer 1 goes round slots 0-2, since features stand in 3 and 4, the others
// round all five from slot 1 on (slice 9 is in slot 0).  mlp_fill: copies into the
// slot before slice `it`; mlp_use: contents before it, features included.
__host__ __device__ constexpr int mlp_slot(int it) { return it < 10 ? it % 3 : (it - 9) % 5; }
__host__ __device__ constexpr int mlp_fill(int it) {
    if (it < 10) return it / 3;
    const int j = it - 9, s = j % 5;
    return j / 5 + (s == 0 ? 3 : s < 3 ? 3 : 0);
}
__host__ __device__ constexpr int mlp_use(int it) { return mlp_fill(it) + (mlp_slot(it) >= 3 ? 1 : 0); }
constexpr bool mlp_ring_counts() {
    int n[kMlpSlots] = {0, 0, 0, 0, 0};
    for (int it = 0; it < 26; ++it)
        if (n[mlp_slot(it)]++ != mlp_fill(it)) return false;
    return true;
}
static_assert(mlp_ring_counts(), "mlp_fill counts the copies into each slot");

__global__ void __cluster_dims__(kMlpCluster, 1, 1) __launch_bounds__(kMlpThreads, 1)
    mlp_kernel(const __grid_constant__ CUtensorMap w1, const __grid_constant__ CUtensorMap w2,
               const __grid_constant__ CUtensorMap w3, const __grid_constant__ MlpArgs a) {
    extern __shared__ __align__(1024) unsigned char gsm[];
    __shared__ uint64_t s_full[kMlpSlots], s_empty[kMlpSlots], s_acc, s_xready, s_hfull, s_hfree, s_pfull, s_done;
    __shared__ uint32_t s_tmem;
    __shared__ int s_fail, s_issued, s_consumed;
    __shared__ float4 s_head[kMlpCols];                      // output weights of this CTA's columns
    __shared__ __align__(16) float4 s_parts[32][kHeadParts];  // partial logits of its 32 rows
    __shared__ uint32_t s_rows[128 * kFeatPitch];             // feature bits
    volatile int* fail = &s_fail;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t rank = blockIdx.x & (kMlpCluster - 1);
    const int m0 = (int)(blockIdx.x / kMlpCluster) * 128;
    const uint32_t base = (smem_u32(gsm) + 1023u) & ~1023u;  // the same offset in every CTA
    const uint32_t ring = base + kMlpH;
    if (tid == 0) {
        for (int s = 0; s < kMlpSlots; ++s) {
            mbar_init(&s_full[s], 1);
            mbar_init(&s_empty[s], 1);
        }
        mbar_init(&s_acc, 1);
        mbar_init(&s_xready, 16);
        mbar_init(&s_hfull, 16 * kMlpCluster);  // every epilogue warp of the cluster
        mbar_init(&s_hfree, kMlpCluster);
        mbar_init(&s_pfull, 2 * kMlpCluster);
        mbar_init(&s_done, 1);
        s_fail = s_issued = s_consumed = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int c = tid; c < kMlpCols; c += kMlpThreads) {
        const __nv_bfloat16* w = a.W4 + kMlpCols * rank + c;
        s_head[c] = make_float4(__bfloat162float(w[0]), __bfloat162float(w[512]), __bfloat162float(w[1024]),
                                __bfloat162float(w[1536]));
    }
    for (int e = tid; e < 128 * kFeatPitch; e += kMlpThreads) s_rows[e] = 0u;
    if (warp == 0) tc_alloc(&s_tmem, 128u);
    tc_fence_before();
    __syncthreads();
    cluster_sync();  // barriers stand before a neighbour arrives on them
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    chain_next();
    if (warp != 16) chain_wait();  // the first weights are copied while the leaves are made
    if (warp == 16) {
        int it = 0;
        bool waited = false;
        bool stop = false;
        for (int L = 0; L < 3 && !stop; ++L) {
            const CUtensorMap* w = L == 0 ? &w1 : L == 1 ? &w2 : &w3;
            for (int kc = 0; kc < (L == 0 ? 10 : 8); ++kc, ++it) {
                const int s = mlp_slot(it);
                const int use = mlp_use(it);  // earlier contents of the slot, features included
                if (use > 0 && !waited) {
                    chain_wait();
                    waited = true;
                }
                if (__any_sync(0xFFFFFFFFu, (use > 0 && !mbar_wait(&s_empty[s], (uint32_t)(use - 1) & 1u, a.wait_ns)) ||
                                                *fail)) {
                    *fail = 1;
                    stop = true;
                    break;
                }
                mbar_expect_tx(&s_full[s], kMlpSlot);
                tma_load_2d(ring + (uint32_t)s * kMlpSlot, w, kc * 64, kMlpCols * (int)rank, &s_full[s]);
            }
        }
        if (lane == 0) s_issued = it;
    } else if (warp == 17) {
        const uint32_t idesc = idesc_bf16_f32(128, kMlpCols);
        int it = 0;
        bool stop = false;
        for (int L = 0; L < 3 && !stop; ++L) {
            if (__any_sync(0xFFFFFFFFu, !(L == 0 ? mbar_wait(&s_xready, 0u, a.wait_ns)
                                                 : mbar_wait_cluster(&s_hfull, (uint32_t)(L - 1) & 1u, a.wait_ns)))) {
                *fail = 1;
                break;
            }
            tc_fence_after();
            for (int kc = 0; kc < (L == 0 ? 10 : 8); ++kc, ++it) {
                const int s = mlp_slot(it);
                if (__any_sync(0xFFFFFFFFu, !mbar_wait(&s_full[s], (uint32_t)mlp_fill(it) & 1u, a.wait_ns) || *fail)) {
                    *fail = 1;
                    stop = true;
                    break;
                }
                tc_fence_after();
                // 64 columns of H, or of the features: H's place and then slots 3 and 4
                const uint32_t sa = kc < 8 ? base + (uint32_t)kc * kMlpSlot : ring + (uint32_t)(kc - 5) * kMlpSlot;
                const uint32_t sb = ring + (uint32_t)s * kMlpSlot;
#pragma unroll
                for (int kk = 0; kk < 4; ++kk)
                    tc_mma(tmem, smem_desc_noswz(sa + (uint32_t)kk * 4096u, 2048u, 128u),
                           smem_desc_sw128(sb + (uint32_t)kk * 32u), idesc, (kc > 0 || kk > 0) ? 1u : 0u);
                tc_commit(&s_empty[s]);
                if (kc >= 8) tc_commit(&s_empty[kc - 5]);  // the features' slot
            }
            if (!stop) tc_commit(&s_acc);
        }
        if (lane == 0) s_consumed = it;
        tc_commit(&s_done);  // arrives when every MMA issued above has completed
    } else {
        const int quarter = warp & 3, group = warp >> 2;
        const int row = quarter * 32 + lane;
        const uint32_t acc = tmem + ((uint32_t)(quarter * 32) << 16);
        bool go = true;
        {
            // features: warp (quarter, group) sets part `group` of 32 rows, then
            // writes every fourth 8-feature column of them
            uint32_t* mine = s_rows + row * kFeatPitch;
            if (m0 + row < a.n) feature_bits(load_state(a.states[m0 + row]), group, mine);
            asm volatile("bar.sync 1, 512;" ::: "memory");
#pragma unroll 4
            for (int b = group; b < kFeatures / 8; b += 4) {
                const uint4 x = feature_bf16((mine[b >> 2] >> (8 * (b & 3))) & 0xFFu);
                const uint32_t at = b < 64 ? base + (uint32_t)(b >> 1) * 4096u
                                           : ring + 3u * kMlpSlot + (uint32_t)((b - 64) >> 1) * 4096u;
                st_shared_v4(at + (uint32_t)(b & 1) * 2048u + (uint32_t)row * 16u, x);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // read by the MMAs
            __syncwarp();
            if (lane == 0) mbar_arrive(&s_xready);
        }
        for (int L = 0; L < 2 && go; ++L) {
            go = __all_sync(0xFFFFFFFFu, mbar_wait(&s_acc, (uint32_t)L & 1u, a.wait_ns)) && !*fail;
            if (!go) break;
            tc_fence_after();
            // this CTA's MMAs have read what H held (the features, H1)
            if (warp == 0 && lane < kMlpCluster)
                mbar_arrive_cluster_relaxed(map_cta(smem_u32(&s_hfree), (uint32_t)lane));
            uint32_t w[2][8];
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                float v[16];
                const int col = group * 32 + c * 16;
                const float4* b4 = reinterpret_cast<const float4*>(a.bias[L] + kMlpCols * rank + col);
                float4 b[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) b[j] = __ldg(b4 + j);
                tc_ld16(acc + (uint32_t)col, v);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    v[4 * j] += b[j].x;
                    v[4 * j + 1] += b[j].y;
                    v[4 * j + 2] += b[j].z;
                    v[4 * j + 3] += b[j].w;
                }
#pragma unroll
                for (int i = 0; i < 16; ++i) v[i] = gelu(v[i]);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    __nv_bfloat162 p = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
                    w[c][i] = *reinterpret_cast<uint32_t*>(&p);
                }
            }
            // every CTA's MMAs have: this layer's activations may take its place
            go = __all_sync(0xFFFFFFFFu, mbar_wait_cluster(&s_hfree, (uint32_t)L & 1u, a.wait_ns));
            if (!go) break;
#pragma unroll
            for (uint32_t q = 0; q < kMlpCluster; ++q) {
                // block of 16 columns: two halves of 8 columns x 128 rows x 16 bytes
                const uint32_t dst = map_cta(base + (uint32_t)(kMlpCols / 16 * rank + 2u * group) * 4096u, q) +
                                     (uint32_t)row * 16u;
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    st_cluster_v4(dst + (uint32_t)c * 4096u, w[c][0], w[c][1], w[c][2], w[c][3]);
                    st_cluster_v4(dst + (uint32_t)c * 4096u + 2048u, w[c][4], w[c][5], w[c][6], w[c][7]);
                }
            }
            asm volatile("fence.proxy.async;" ::: "memory");  // read by the neighbours' MMAs
            tc_fence_before();
            __syncwarp();
            if (lane < kMlpCluster) mbar_arrive_cluster(map_cta(smem_u32(&s_hfull), (uint32_t)lane));
        }
        if (go && group < 2) {
            // layer 3 and the output layer's products: 64 columns per warp, in column order
            go = __all_sync(0xFFFFFFFFu, mbar_wait(&s_acc, 0u, a.wait_ns)) && !*fail;
            if (go) {
                tc_fence_after();
                float4 head = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll 1
                for (int c = 0; c < 4; ++c) {
                    float v[16];
                    const int col = group * 64 + c * 16;
                    const float4* b4 = reinterpret_cast<const float4*>(a.bias[2] + kMlpCols * rank + col);
                    float4 b[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) b[j] = __ldg(b4 + j);
                    tc_ld16(acc + (uint32_t)col, v);
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        v[4 * j] += b[j].x;
                        v[4 * j + 1] += b[j].y;
                        v[4 * j + 2] += b[j].z;
                        v[4 * j + 3] += b[j].w;
                    }
#pragma unroll
                    for (int i = 0; i < 16; ++i) v[i] = gelu(v[i]);
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        const float4 hw = s_head[col + i];
                        head.x += v[i] * hw.x;
                        head.y += v[i] * hw.y;
                        head.z += v[i] * hw.z;
                        head.w += v[i] * hw.w;
                    }
                }
                // rows 32 q .. of the tile are finished by CTA q
                const uint32_t dst = map_cta(smem_u32(&s_parts[lane][2 * rank + group]), (uint32_t)quarter);
                st_cluster_v4(dst, __float_as_uint(head.x), __float_as_uint(head.y), __float_as_uint(head.z),
                              __float_as_uint(head.w));
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(map_cta(smem_u32(&s_pfull), (uint32_t)quarter));
            }
        } else if (go && warp == 8) {
            go = __all_sync(0xFFFFFFFFu, mbar_wait_cluster(&s_pfull, 0u, a.wait_ns));
            const int r = m0 + 32 * (int)rank + lane;
            if (go && r < a.n) {
                float4 z = make_float4(a.b4[0], a.b4[1], a.b4[2], a.b4[3]);
#pragma unroll
                for (int p = 0; p < kHeadParts; ++p) {
                    const float4 x = s_parts[lane][p];
                    z.x += x.x;
                    z.y += x.y;
                    z.z += x.z;
                    z.w += x.w;
                }
                softmax_seats(a.states[r], z, a.out + (size_t)r * 4);
            }
        }
        if (!go && lane == 0) *fail = 1;
    }
    __syncthreads();
    // every MMA has completed before tensor memory is freed; on failure the
    // copies still in flight land first
    const bool ok = __syncthreads_and(mbar_wait(&s_done, 0, a.wait_ns) && !*fail) != 0;
    if (!ok && tid == 0) {
        for (int it = s_consumed; it < s_issued; ++it)
            mbar_wait(&s_full[mlp_slot(it)], (uint32_t)mlp_fill(it) & 1u, a.wait_ns);
        if (a.flags) atomicCAS(a.flags, 0, -4);  // DVC_E_TIMEOUT
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();  // no neighbour writes into this CTA any more
    if (warp == 0) {
        tc_fence_after();
        tc_dealloc(tmem, 128u);
    }
}

}  // namespace dvc
