// dvc_value.cu -- the value network: a learned leaf evaluator that can stand in
// for random playouts (the workload's extension of the method; the paper's
// own leaf evaluation is the playout of Sec. II-B).
//
// Features (640): per tile, owner seat relative to the mover, face-down/up
// and drawn-this-turn; per opponent slot, the values it may hold given the
// face-up numbered neighbours and the tiles the mover cannot see.  Network
// 640 -> 512 -> 512 -> 512 (GELU) -> 4 logits over relative seats, softmax
// over the seats in play.  BF16 weights and activations, FP32 accumulation in
// tensor memory (tcgen05), FP32 master weights and AdamW moments.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cstdio>
#include <cstring>
#include <vector>

#include "dvc_device.cuh"
#include "dvc_features.cuh"
#include "dvc_gemm.cuh"
#include "dvc_internal.h"
#include "dvc_mlp.cuh"

using namespace dvc;
using namespace dvc_host;

namespace {

constexpr int VF = 640, VH = 512, VO = 16;
// floats per row of the logit buffers: VO logits (training) or kHeadParts x 4
// partial logits (inference with the output layer folded into layer 3)
constexpr int kLogitFloats = kHeadParts * 4 > VO ? kHeadParts * 4 : VO;
constexpr size_t OFF_W1 = 0, OFF_B1 = OFF_W1 + (size_t)VH * VF, OFF_W2 = OFF_B1 + VH, OFF_B2 = OFF_W2 + (size_t)VH * VH,
                 OFF_W3 = OFF_B2 + VH, OFF_B3 = OFF_W3 + (size_t)VH * VH, OFF_W4 = OFF_B3 + VH,
                 OFF_B4 = OFF_W4 + 4 * VH, NPARAM = OFF_B4 + 4;

}  // namespace

struct dvc_value_net {
    float *master, *m, *v, *grad;
    __nv_bfloat16 *W1, *W2, *W3, *W4;  // W4: 64 x 512, rows 4.. zero
    float* b4p;                        // 16
    int clusters;                      // clusters of the small-batch kernel that run at once
    int cap;                           // workspace rows (multiple of 128)
    __nv_bfloat16 *X, *H1, *H2, *H3, *dZ[3], *dZ4;  // dZ of layers 1..3; of the output layer, 64 columns
    float *Z1, *Z2, *Z3, *L;
    float* colsum;                     // bias gradients of layers 1..3 by 32 rows: 3 x (rows / 32) x 512
    float* rowpart;                    // per CTA of the loss kernel: four output-bias gradients, padding (8); kLossSum
    long long step;
};

namespace {

// ------------------------------------------------------------------ kernels

// Feature bits of 32 states per CTA, four warps: warp 0 sets the tiles' bits,
// warp k the slots of opponent k, lane r works on row r.  The bits meet in
// shared memory, from where all threads write the rows: a byte of feature bits
// becomes 8 BF16 values through a 256-entry table (4 FP32 values per nibble for
// Xf).  Rows n .. npad-1 are written as zeros.  What bounds it is the chain of one
// row's slots; with a thread per row 8,192 rows took 11.9 us, now 6.4.
constexpr int kFeatThreads = 128, kFeatRows = 32;

__global__ void __launch_bounds__(kFeatThreads)
    features_kernel(const dvc_state* states, int n, int npad, __nv_bfloat16* X, float* Xf, int blocked) {
    chain_next();
    __shared__ uint32_t s_rows[kFeatRows * kFeatPitch];
    __shared__ uint4 s_lut[256];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int row0 = blockIdx.x * kFeatRows, row = row0 + lane;
    dvc_state st = {};
    if (row < n) st = states[row];
    for (int b = tid; b < 256; b += kFeatThreads) s_lut[b] = feature_bf16((uint32_t)b);
    for (int e = tid; e < kFeatRows * kFeatPitch; e += kFeatThreads) s_rows[e] = 0u;
    __syncthreads();
    uint32_t* mine = s_rows + lane * kFeatPitch;
    if (row < n) feature_bits(load_state(st), warp, mine);
    __syncthreads();
    if (blocked) {
        // K-blocked X (npad a multiple of 128): 16 bytes per 8 features; a warp's
        // 32 rows are contiguous in a block
        if (X && row < npad) {
            __nv_bfloat16* xr = X + kblocked_index(row, 0, VF);
            for (int b = warp; b < VF / 8; b += kFeatThreads / 32)
                *reinterpret_cast<uint4*>(xr + (size_t)(b >> 1) * 2048 + (size_t)(b & 1) * 1024) =
                    s_lut[(mine[b >> 2] >> (8 * (b & 3))) & 0xFFu];
        }
        return;
    }
    const int nrows = min(kFeatRows, npad - row0);
    if (X && nrows > 0) {
        uint4* dst = reinterpret_cast<uint4*>(X + (size_t)row0 * VF);
        for (int c = tid; c < nrows * (VF / 8); c += kFeatThreads) {
            const int r = c / (VF / 8), k = c - r * (VF / 8);
            dst[c] = s_lut[(s_rows[r * kFeatPitch + (k >> 2)] >> (8 * (k & 3))) & 0xFFu];
        }
    }
    if (Xf && nrows > 0) {
        float4* dst = reinterpret_cast<float4*>(Xf + (size_t)row0 * VF);
        for (int c = tid; c < nrows * (VF / 4); c += kFeatThreads) {
            const int r = c / (VF / 4), k = c - r * (VF / 4);
            const uint32_t nib = (s_rows[r * kFeatPitch + (k >> 3)] >> (4 * (k & 7))) & 0xFu;
            dst[c] = make_float4((float)(nib & 1u), (float)((nib >> 1) & 1u), (float)((nib >> 2) & 1u),
                                 (float)((nib >> 3) & 1u));
        }
    }
}

// Softmax over relative seats 0..P-1, written per absolute seat, of logits
// given as 8 partial sums per row (the output layer folded into layer 3):
// z[r] = b4[r] + parts[0][r] + ... + parts[7][r].
__global__ void softmax_head_kernel(const float* parts, const float* b4, const dvc_state* states, int n, float* out) {
    chain_wait();
    const int row = blockIdx.x * blockDim.x + threadIdx.x;
    if (row >= n) return;
    const float4* pp = reinterpret_cast<const float4*>(parts) + (size_t)row * kHeadParts;
    float4 z = make_float4(b4[0], b4[1], b4[2], b4[3]);
#pragma unroll
    for (int p = 0; p < kHeadParts; ++p) {
        const float4 q = pp[p];
        z.x += q.x;
        z.y += q.y;
        z.z += q.z;
        z.w += q.w;
    }
    softmax_seats(states[row], z, out + (size_t)row * 4);
}

// Cross-entropy against soft labels (absolute seats) and dL/dlogits / n.
// Rows >= n get zero gradient.  dZ4 (npad x 64, BF16, K-padded); the rows' losses
// in rowloss, and per CTA the sums of the FP32 logit gradients in rowpart[cta][0..3].
constexpr int kLossThreads = 128;
constexpr int kLossSum = 7;  // in the first CTA's padding of rowpart: the sum of the losses
static_assert(kLogitFloats > VO, "the rows' losses stand behind the logits");
__global__ void __launch_bounds__(kLossThreads)
    loss_grad_kernel(const float* L, const dvc_state* states, const float* labels, int n, int npad,
                     __nv_bfloat16* dZ4, float* rowloss, float* rowpart) {
    chain_next();
    chain_wait();
    __shared__ float s_sum[kLossThreads / 32][4];
    const int row = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float d[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    float loss = 0.0f;
    if (row < n) {
        const dvc_state& s = states[row];
        const int P = (s.nplayers >= 2 && s.nplayers <= 4) ? s.nplayers : 2;
        const int cur = s.cur < P ? s.cur : 0;
        const float4 zv = *reinterpret_cast<const float4*>(L + (size_t)row * VO);
        const float z[4] = {zv.x, zv.y, zv.z, zv.w};
        float mx = z[0];
#pragma unroll
        for (int r = 1; r < 4; ++r)
            if (r < P) mx = fmaxf(mx, z[r]);
        float sum = 0.0f;
#pragma unroll
        for (int r = 0; r < 4; ++r)
            if (r < P) sum += expf(z[r] - mx);
        const float lse = mx + logf(sum);
#pragma unroll
        for (int r = 0; r < 4; ++r)
            if (r < P) {
                const float y = labels[(size_t)row * 4 + (cur + r) % P];
                const float p = expf(z[r] - lse);
                if (y > 0.0f) loss -= y * (z[r] - lse);
                d[r] = (p - y) / (float)n;
            }
    }
    if (row < npad) {
        rowloss[row] = loss;
        uint4* out = reinterpret_cast<uint4*>(dZ4 + (size_t)row * 64);
        const __nv_bfloat162 lo = __floats2bfloat162_rn(d[0], d[1]), hi = __floats2bfloat162_rn(d[2], d[3]);
        out[0] = make_uint4(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi), 0u, 0u);
#pragma unroll
        for (int j = 1; j < 8; ++j) out[j] = make_uint4(0u, 0u, 0u, 0u);
    }
    float v[4] = {d[0], d[1], d[2], d[3]};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_xor_sync(0xFFFFFFFFu, v[k], o);
        if (lane == 0) s_sum[warp][k] = v[k];
    }
    __syncthreads();
    if (threadIdx.x < 4) {
        float acc = 0.0f;
        for (int w = 0; w < kLossThreads / 32; ++w) acc += s_sum[w][threadIdx.x];
        rowpart[(size_t)blockIdx.x * 8 + threadIdx.x] = acc;
    }
}

// AdamW on one FP32 master parameter (weight decay on weight matrices only).
struct AdamCoef {
    float lr, b1, b2, eps, wd, c1, c2;
};
__device__ __forceinline__ float adamw_one(float w, float& m, float& v, float gi, bool is_bias, const AdamCoef& a) {
    const float mi = a.b1 * m + (1.0f - a.b1) * gi;
    const float vi = a.b2 * v + (1.0f - a.b2) * gi * gi;
    m = mi;
    v = vi;
    float upd = (mi / a.c1) / (sqrtf(vi / a.c2) + a.eps);
    if (!is_bias) upd += a.wd * w;
    return w - a.lr * upd;
}

__device__ __forceinline__ bool is_bias_index(size_t i) {
    return (i >= OFF_B1 && i < OFF_W2) || (i >= OFF_B2 && i < OFF_W3) || (i >= OFF_B3 && i < OFF_W4) || i >= OFF_B4;
}

// The BF16 working copy of master weights i .. i + 3 (no biases).
__device__ __forceinline__ void store_bf16_weights(const dvc_value_net& v, size_t i, float4 w) {
    __nv_bfloat16* dst = i < OFF_B1 ? v.W1 + i : i < OFF_B2 ? v.W2 + (i - OFF_W2) : i < OFF_B3 ? v.W3 + (i - OFF_W3)
                                                                                            : v.W4 + (i - OFF_W4);
    const __nv_bfloat162 lo = __floats2bfloat162_rn(w.x, w.y), hi = __floats2bfloat162_rn(w.z, w.w);
    *reinterpret_cast<uint2*>(dst) =
        make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
}

// End of a training step in one launch: sum the partial gradients (biases over the
// 32-row column sums, output biases over the loss kernel's CTAs, in a fixed
// order), AdamW, BF16 copies.  CTAs 0 .. kAdamMain-1 take four weights per
// thread; then 16 CTAs per hidden layer take 32 biases each, and the last one the
// output biases and the loss.  What bounds it is memory: gradients, master,
// moments and their updates.
constexpr int kAdamThreads = 256;
constexpr int kAdamMain = (int)((NPARAM / 4 + kAdamThreads - 1) / kAdamThreads);
constexpr int kAdamGrid = kAdamMain + 3 * (VH / 32) + 1;
__global__ void __launch_bounds__(kAdamThreads)
    adamw_kernel(dvc_value_net v, int row_blocks, int loss_ctas, int n, AdamCoef a, float* loss_out) {
    chain_wait();
    const int tid = threadIdx.x;
    if ((int)blockIdx.x < kAdamMain) {
        const size_t i = ((size_t)blockIdx.x * kAdamThreads + tid) * 4;
        if (i >= NPARAM || is_bias_index(i)) return;  // tensors begin at multiples of four
        const float4 g = *reinterpret_cast<const float4*>(v.grad + i);
        float4 w = *reinterpret_cast<const float4*>(v.master + i), m = *reinterpret_cast<const float4*>(v.m + i);
        float4 u = *reinterpret_cast<const float4*>(v.v + i);
        w.x = adamw_one(w.x, m.x, u.x, g.x, false, a);
        w.y = adamw_one(w.y, m.y, u.y, g.y, false, a);
        w.z = adamw_one(w.z, m.z, u.z, g.z, false, a);
        w.w = adamw_one(w.w, m.w, u.w, g.w, false, a);
        *reinterpret_cast<float4*>(v.master + i) = w;
        *reinterpret_cast<float4*>(v.m + i) = m;
        *reinterpret_cast<float4*>(v.v + i) = u;
        store_bf16_weights(v, i, w);
        return;
    }
    __shared__ float s_part[kAdamThreads];
    const int e = (int)blockIdx.x - kAdamMain;
    size_t i = 0;
    float acc = 0.0f;
    bool mine = false;
    if (e < 3 * (VH / 32)) {
        const int layer = e / (VH / 32), col = e % (VH / 32) * 32 + (tid & 31);
        const float* p = v.colsum + (size_t)layer * row_blocks * VH + col;
        for (int r = tid >> 5; r < row_blocks; r += kAdamThreads / 32) acc += p[(size_t)r * VH];
        s_part[tid] = acc;
        __syncthreads();
        acc = 0.0f;
        for (int w = 0; w < kAdamThreads / 32; ++w) acc += s_part[w * 32 + (tid & 31)];
        i = (layer == 0 ? OFF_B1 : layer == 1 ? OFF_B2 : OFF_B3) + (size_t)col;
        mine = tid < 32;
    } else {
        const int k = tid & 7;  // 0..3: output biases
        if (k < 4)
            for (int r = tid >> 3; r < loss_ctas; r += kAdamThreads / 8) acc += v.rowpart[(size_t)r * 8 + k];
        s_part[tid] = acc;
        __syncthreads();
        acc = 0.0f;
        for (int w = 0; w < kAdamThreads / 8; ++w) acc += s_part[w * 8 + k];
        if (tid == 0 && loss_out) *loss_out = v.rowpart[kLossSum] / (float)n;
        i = OFF_B4 + (size_t)k;
        mine = tid < 4;
    }
    if (!mine) return;
    float m = v.m[i], u = v.v[i];
    const float w = adamw_one(v.master[i], m, u, acc, true, a);
    v.grad[i] = acc;
    v.master[i] = w;
    v.m[i] = m;
    v.v[i] = u;
    if (i >= OFF_B4) v.b4p[i - OFF_B4] = w;
}

// BF16 working copies of the master weights, zero padding included.
__global__ void refresh_kernel(dvc_value_net v) {
    const size_t nthr = (size_t)gridDim.x * blockDim.x, t0 = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (size_t q = t0; q < NPARAM / 4; q += nthr)
        if (!is_bias_index(4 * q))
            store_bf16_weights(v, 4 * q, *reinterpret_cast<const float4*>(v.master + 4 * q));
    for (size_t j = 4 * VH + t0; j < 64 * (size_t)VH; j += nthr) v.W4[j] = __float2bfloat16_rn(0.0f);
    if (t0 < VO) v.b4p[t0] = t0 < 4 ? v.master[OFF_B4 + t0] : 0.0f;
}

// Glorot-uniform weights from Philox (key = seed, counter = index), zero biases.
__global__ void init_params_kernel(float* w, uint64_t seed) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < NPARAM; i += (size_t)gridDim.x * blockDim.x) {
        float fan_in = 0.0f, fan_out = 0.0f;
        bool bias = true;
        if (i < OFF_B1) { fan_in = VF; fan_out = VH; bias = false; }
        else if (i >= OFF_W2 && i < OFF_B2) { fan_in = VH; fan_out = VH; bias = false; }
        else if (i >= OFF_W3 && i < OFF_B3) { fan_in = VH; fan_out = VH; bias = false; }
        else if (i >= OFF_W4 && i < OFF_B4) { fan_in = VH; fan_out = 4; bias = false; }
        if (bias) {
            w[i] = 0.0f;
            continue;
        }
        uint32_t a = (uint32_t)i, b = (uint32_t)(i >> 32), c = 7u, d = 0u;
        philox10(a, b, c, d, (uint32_t)seed, (uint32_t)(seed >> 32));
        const float u = ((float)(a >> 8) + 0.5f) * (1.0f / 16777216.0f);  // (0, 1)
        const float lim = sqrtf(6.0f / (fan_in + fan_out));
        w[i] = (2.0f * u - 1.0f) * lim;
    }
}

// ------------------------------------------------------------------ host helpers

// The network's own tile widths have a chained build.
template <int BN>
constexpr bool kChainedGemm = BN == 256 || BN == 16;

template <int BN, bool BMN = false, bool BACK = false>
cudaError_t gemm_attributes() {
    cudaError_t e = cudaFuncSetAttribute(gemm_bf16_tc_kernel<BN, BMN, BACK, false>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)GemmCfg<BN>::kSmem);
    if constexpr (kChainedGemm<BN>)
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(gemm_bf16_tc_kernel<BN, BMN, BACK, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)GemmCfg<BN>::kSmem);
    return e;
}

// cuTensorMapEncodeTiled through the runtime's driver entry point, so the
// library needs no link against the driver library.
PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
    static const PFN_cuTensorMapEncodeTiled_v12000 fn = [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) !=
                cudaSuccess ||
            q != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            p = nullptr;
        }
        return (PFN_cuTensorMapEncodeTiled_v12000)p;
    }();
    return fn;
}

// A row-major rows x K BF16 matrix as the 2-D tensor (K, rows) read in boxes
// of 64 x box_rows with the 128-byte swizzle; rows past the end read as zero.
// (For an operand read MN-major, "K" is its M or N and the rows are K.)
bool encode_kmajor(CUtensorMap* m, const __nv_bfloat16* p, int rows, int K, int box_rows) {
    const PFN_cuTensorMapEncodeTiled_v12000 enc = tensor_map_encoder();
    if (!enc) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)K * 2u};
    const cuuint32_t box[2] = {(cuuint32_t)kGemmBK, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1u, 1u};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<__nv_bfloat16*>(p), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int BN, bool BMN = false, bool BACK = false>
cudaError_t launch_gemm(const GemmArgs& a, cudaStream_t st, bool chained) {
    // inside a stream capture the attributes were set beforehand (dvc_value_prepare)
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    cudaError_t e = cudaStreamIsCapturing(st, &cs);
    if (e == cudaSuccess && cs == cudaStreamCaptureStatusNone) e = gemm_attributes<BN, BMN, BACK>();
    if (e != cudaSuccess) return e;
    CUtensorMap tA, tB;
    if (!encode_kmajor(&tA, a.A, a.M, a.K, kGemmBM) ||
        !(BMN ? encode_kmajor(&tB, a.B, a.K, a.N, 64) : encode_kmajor(&tB, a.B, a.N, a.K, BN)))
        return cudaErrorInvalidValue;
    const long long tiles = (long long)((a.M + kGemmBM - 1) / kGemmBM) * (a.N / BN);
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const unsigned grid = (unsigned)std::min<long long>(tiles, std::max(sms, 1));
    // chained while every tile has an SM of its own, where the launch and the prologue
    // are a good part of the time (a training step of 8,192 rows 179 -> 158 us); a
    // persistent grid gains nothing and its build without is faster (65,536 rows: the
    // whole evaluation 148 us against 151 chained)
    if constexpr (kChainedGemm<BN>)
        if (chained && tiles <= sms)
            return launch_chained(gemm_bf16_tc_kernel<BN, BMN, BACK, true>, grid, kGemmThreads, GemmCfg<BN>::kSmem, st,
                                  tA, tB, a);
    gemm_bf16_tc_kernel<BN, BMN, BACK, false><<<grid, kGemmThreads, GemmCfg<BN>::kSmem, st>>>(tA, tB, a);
    return cudaGetLastError();
}

constexpr uint64_t kGemmWaitNs = 2000000000ull;  // 2 s: far beyond any wait of a working GEMM

// a_blocked / c_blocked: A read / C written in the K-blocked layout (M a
// multiple of 128; the inference path's activations).
cudaError_t gemm(const __nv_bfloat16* A, const __nv_bfloat16* B, const float* bias, __nv_bfloat16* C, float* Cf, int M,
                 int N, int K, int act, int32_t* flags, cudaStream_t st, bool a_blocked = false,
                 bool c_blocked = false) {
    const int wide = ((uintptr_t)C % 32 == 0 && (uintptr_t)Cf % 32 == 0) ? 1 : 0;  // null counts as aligned
    GemmArgs a{A, B, bias, C, Cf, M, N, K, act, flags, kGemmWaitNs, 0, nullptr, nullptr, wide,
               bias && (uintptr_t)bias % 16 == 0, a_blocked ? 1 : 0, c_blocked ? 1 : 0};
    if (N % 256 == 0) return launch_gemm<256>(a, st, true);
    if (N % 128 == 0) return launch_gemm<128>(a, st, true);
    if (N % 64 == 0) return launch_gemm<64>(a, st, true);
    if (N % 32 == 0) return launch_gemm<32>(a, st, true);
    return launch_gemm<16>(a, st, true);
}

// Layer 3 with the 512 -> 4 output layer folded into its epilogue: no H3
// written; 8 partial logit vectors per row into `parts` (rows x 8 x 4).
cudaError_t gemm_head(const __nv_bfloat16* A, const __nv_bfloat16* B, const float* bias, float* Cf, int M,
                      const __nv_bfloat16* W4, float* parts, int32_t* flags, cudaStream_t st, bool a_blocked) {
    GemmArgs a{A,     B,  bias, nullptr, Cf, M, VH, VH, kActGelu, flags, kGemmWaitNs, 0, W4, parts,
               (uintptr_t)Cf % 32 == 0, bias && (uintptr_t)bias % 16 == 0, a_blocked ? 1 : 0, 0};
    return launch_gemm<256>(a, st, true);  // N = 512: two 256-column tiles x four column groups = kHeadParts
}

// dZ = (dZn Wn) * gelu'(Z): the gradient at the layer below, Wn (512 outputs of
// the layer above, K rows) x 512 read MN-major, with the bias gradient's sums.
cudaError_t gemm_back(const __nv_bfloat16* dZn, int K, const __nv_bfloat16* Wn, const float* Z, __nv_bfloat16* dZ,
                      float* colsum, int M, int32_t* flags, cudaStream_t st) {
    GemmArgs a{};
    a.A = dZn;
    a.B = Wn;
    a.C = dZ;
    a.M = M;
    a.N = VH;
    a.K = K;
    a.act = kActNone;
    a.flags = flags;
    a.wait_ns = kGemmWaitNs;
    a.Z = Z;
    a.colsum = colsum;
    return launch_gemm<256, true, true>(a, st, true);
}

// Weight gradients of all four layers into v->grad.
cudaError_t gemm_dw(dvc_value_net* v, int n, int npad, int32_t* flags, cudaStream_t st) {
    DwArgs a{};
    const __nv_bfloat16* A[4] = {v->dZ[0], v->dZ[1], v->dZ[2], v->H3};
    const __nv_bfloat16* B[4] = {v->X, v->H1, v->H2, v->dZ4};
    const int wb[4] = {VF, VH, VH, 64};
    const size_t off[4] = {OFF_W1, OFF_W2, OFF_W3, OFF_W4};
    int first = 0;
    for (int q = 0; q < 4; ++q) {
        if (!encode_kmajor(&a.a[q], A[q], npad, VH, 64) || !encode_kmajor(&a.b[q], B[q], npad, wb[q], 64))
            return cudaErrorInvalidValue;
        a.p[q] = DwProblem{first, wb[q] / 64, wb[q], q == 3 ? 1 : 0, off[q]};
        first += VH / 128 * (wb[q] / 64);
    }
    a.tiles = first;
    a.losses = v->L + (size_t)npad * VO;
    a.n = n;
    a.loss_sum = v->rowpart + kLossSum;
    a.nk = npad / 64;
    a.grad = v->grad;
    a.flags = flags;
    a.wait_ns = kGemmWaitNs;
    return launch_chained(gemm_dw_kernel, (unsigned)first + 1u, kDwThreads, kDwSmem, st, a);
}

cudaError_t mlp_attributes() {
    return cudaFuncSetAttribute(mlp_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMlpSmem);
}

// Clusters of mlp_kernel that the device holds at once.
cudaError_t mlp_clusters(int* out) {
    cudaError_t e = mlp_attributes();
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kMlpCluster);
    cfg.blockDim = dim3(kMlpThreads);
    cfg.dynamicSmemBytes = kMlpSmem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kMlpCluster;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaOccupancyMaxActiveClusters(out, mlp_kernel, &cfg);
}

int net_alloc(dvc_ctx* c) {
    if (c->vnet) return DVC_OK;
    dvc_value_net* v = new dvc_value_net();
    std::memset(v, 0, sizeof(*v));
    bool ok = cudaMalloc(&v->master, NPARAM * 4) == cudaSuccess && cudaMalloc(&v->m, NPARAM * 4) == cudaSuccess &&
              cudaMalloc(&v->v, NPARAM * 4) == cudaSuccess && cudaMalloc(&v->grad, NPARAM * 4) == cudaSuccess &&
              cudaMalloc(&v->W1, (size_t)VH * VF * 2) == cudaSuccess &&
              cudaMalloc(&v->W2, (size_t)VH * VH * 2) == cudaSuccess &&
              cudaMalloc(&v->W3, (size_t)VH * VH * 2) == cudaSuccess &&
              cudaMalloc(&v->W4, (size_t)64 * VH * 2) == cudaSuccess && cudaMalloc(&v->b4p, VO * 4) == cudaSuccess;
    if (!ok || cudaMemset(v->m, 0, NPARAM * 4) != cudaSuccess || cudaMemset(v->v, 0, NPARAM * 4) != cudaSuccess ||
        cudaMemset(v->grad, 0, NPARAM * 4) != cudaSuccess) {
        cudaGetLastError();
        c->vnet = v;
        return fail(c, DVC_E_OOM, "value network: parameter allocation");
    }
    const cudaError_t e = mlp_clusters(&v->clusters);
    if (e != cudaSuccess) v->clusters = 0;  // the layer-by-layer path serves every size
    cudaGetLastError();
    c->vnet = v;
    return DVC_OK;
}

void free_work(dvc_value_net* v) {
    void* ptrs[] = {v->X, v->H1, v->H2, v->H3, v->dZ[0], v->dZ[1], v->dZ[2], v->dZ4,
                    v->Z1, v->Z2, v->Z3, v->L, v->colsum, v->rowpart};
    for (void* p : ptrs)
        if (p) cudaFree(p);
    v->X = v->H1 = v->H2 = v->H3 = v->dZ[0] = v->dZ[1] = v->dZ[2] = v->dZ4 = nullptr;
    v->Z1 = v->Z2 = v->Z3 = v->L = v->colsum = v->rowpart = nullptr;
    v->cap = 0;
}

int ensure_work(dvc_ctx* c, int npad) {
    dvc_value_net* v = c->vnet;
    if (npad <= v->cap) return DVC_OK;
    free_work(v);
    const size_t r = (size_t)npad;
    auto al = [&](void** p, size_t bytes) { return cudaMalloc(p, bytes) == cudaSuccess; };
    const bool ok = al((void**)&v->X, r * VF * 2) && al((void**)&v->H1, r * VH * 2) && al((void**)&v->H2, r * VH * 2) &&
                    al((void**)&v->H3, r * VH * 2) && al((void**)&v->dZ[0], r * VH * 2) &&
                    al((void**)&v->dZ[1], r * VH * 2) && al((void**)&v->dZ[2], r * VH * 2) &&
                    al((void**)&v->dZ4, r * 64 * 2) && al((void**)&v->Z1, r * VH * 4) && al((void**)&v->Z2, r * VH * 4) &&
                    al((void**)&v->Z3, r * VH * 4) && al((void**)&v->L, r * kLogitFloats * 4) &&
                    al((void**)&v->colsum, 3 * (r / 32) * VH * 4) && al((void**)&v->rowpart, r / kLossThreads * 8 * 4);
    if (!ok) {
        cudaGetLastError();
        free_work(v);
        return fail(c, DVC_E_OOM, "value network: workspace of " + std::to_string(npad) + " rows");
    }
    // Attributes of a training step's kernels, set here so that a step of as many rows may
    // be captured after any call: evaluations of up to a wave of clusters launch none of
    // its forward GEMMs.
    cudaError_t e = gemm_attributes<256>();
    if (e == cudaSuccess) e = gemm_attributes<16>();
    if (e == cudaSuccess) e = gemm_attributes<256, true, true>();
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(gemm_dw_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDwSmem);
    if (e != cudaSuccess) return cuda_fail(c, e, "value network attributes");
    v->cap = npad;
    return DVC_OK;
}

int refresh(dvc_ctx* c, cudaStream_t st) {
    dvc_value_net* v = c->vnet;
    refresh_kernel<<<256, 256, 0, st>>>(*v);
    return check_launch(c, "refresh_kernel");
}

int need_net(dvc_ctx* c) {
    if (!c->vnet || !c->vnet->master) return fail(c, DVC_E_INVALID, "value network not initialised (dvc_value_init)");
    return DVC_OK;
}

// Features and the four layers of npad rows (n live) into the given
// activation buffers; Z1..Z3 (pre-activation FP32, training) may be null.
// With head = true (inference) the output layer is folded into layer 3's
// epilogue: L receives 8 partial logit vectors per row (softmax_head_kernel
// sums them) and H3 is not written; with head = false (training) layer 4 is
// a GEMM of its own and L holds the logits (16 columns per row).
int forward_into(dvc_ctx* c, const dvc_state* states, int n, int npad, __nv_bfloat16* X, __nv_bfloat16* H1,
                 __nv_bfloat16* H2, __nv_bfloat16* H3, float* L, float* Z1, float* Z2, float* Z3, bool head,
                 cudaStream_t st) {
    dvc_value_net* v = c->vnet;
    int32_t* fl = c->d_flags;
    // inference (head folded in): X, H1 and H2 in the K-blocked layout; training keeps them row-major
    const bool kb = head;
    features_kernel<<<(npad + kFeatRows - 1) / kFeatRows, kFeatThreads, 0, st>>>(states, n, npad, X, nullptr, kb ? 1 : 0);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = gemm(X, v->W1, v->master + OFF_B1, H1, Z1, npad, VH, VF, kActGelu, fl, st, kb, kb);
    if (e == cudaSuccess) e = gemm(H1, v->W2, v->master + OFF_B2, H2, Z2, npad, VH, VH, kActGelu, fl, st, kb, kb);
    if (head) {
        if (e == cudaSuccess) e = gemm_head(H2, v->W3, v->master + OFF_B3, Z3, npad, v->W4, L, fl, st, kb);
    } else {
        if (e == cudaSuccess) e = gemm(H2, v->W3, v->master + OFF_B3, H3, Z3, npad, VH, VH, kActGelu, fl, st);
        if (e == cudaSuccess) e = gemm(H3, v->W4, v->b4p, nullptr, L, npad, VO, VH, kActNone, fl, st);
    }
    if (e != cudaSuccess) return cuda_fail(c, e, "value forward");
    return DVC_OK;
}

// Win probabilities of n leaves, activations in the given buffers (npad rows).
// One launch of clusters (dvc_mlp.cuh) while its 128-row tiles run at once: 28.9
// us for 128 rows, 30.8 for 3,000, against 45 us layer by layer up to 7,000 rows;
// a second wave would take 57 us (4,864 rows), and the layers use a full chip
// better (65,536 rows: 148 us against 418).
int infer(dvc_ctx* c, const dvc_state* states, int n, int npad, __nv_bfloat16* X, __nv_bfloat16* H1, __nv_bfloat16* H2,
          float* L, float* probs, cudaStream_t st, bool chained) {
    dvc_value_net* v = c->vnet;
    if (npad / 128 <= v->clusters) {
        cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
        cudaError_t e = cudaStreamIsCapturing(st, &cs);
        if (e == cudaSuccess && cs == cudaStreamCaptureStatusNone) e = mlp_attributes();
        CUtensorMap w1, w2, w3;
        if (e == cudaSuccess && (!encode_kmajor(&w1, v->W1, VH, VF, kMlpCols) || !encode_kmajor(&w2, v->W2, VH, VH, kMlpCols) ||
                                 !encode_kmajor(&w3, v->W3, VH, VH, kMlpCols)))
            e = cudaErrorInvalidValue;
        if (e != cudaSuccess) return cuda_fail(c, e, "value network");
        const MlpArgs a{{v->master + OFF_B1, v->master + OFF_B2, v->master + OFF_B3}, v->W4, v->b4p, states, n,
                        probs, c->d_flags, kGemmWaitNs};
        if (chained) e = launch_chained(mlp_kernel, (unsigned)(npad / 128 * kMlpCluster), kMlpThreads, kMlpSmem, st, w1, w2, w3, a);
        else {
            mlp_kernel<<<npad / 128 * kMlpCluster, kMlpThreads, kMlpSmem, st>>>(w1, w2, w3, a);
            e = cudaGetLastError();
        }
        return e == cudaSuccess ? DVC_OK : cuda_fail(c, e, "mlp_kernel");
    }
    if (int rc = forward_into(c, states, n, npad, X, H1, H2, nullptr, L, nullptr, nullptr, nullptr, true, st)) return rc;
    const cudaError_t e = launch_chained(softmax_head_kernel, (unsigned)(n + 127) / 128, 128, 0, st, L, v->b4p, states, n, probs);
    return e == cudaSuccess ? DVC_OK : cuda_fail(c, e, "softmax_head_kernel");
}

int check_states_args(dvc_ctx* c, const void* d_states, int n) {
    if (n < 0) return fail(c, DVC_E_INVALID, "value network: n < 0");
    if (n > (1 << 24)) return fail(c, DVC_E_UNSUPPORTED, "value network: more than 2^24 rows");
    if (n > 0 && !is_device_ptr(d_states, c->device)) return fail(c, DVC_E_INVALID, "value network: states must be device memory");
    return DVC_OK;
}

}  // namespace

extern "C" {

int dvc_value_init(dvc_ctx* c, uint64_t seed, void* stream) {
    if (!c) return DVC_E_INVALID;
    if (int rc = set_device(c)) return rc;
    if (int rc = net_alloc(c)) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    dvc_value_net* v = c->vnet;
    init_params_kernel<<<512, 256, 0, st>>>(v->master, seed);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemsetAsync(v->m, 0, NPARAM * 4, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(v->v, 0, NPARAM * 4, st);
    if (e != cudaSuccess) return cuda_fail(c, e, "dvc_value_init");
    v->step = 0;
    return refresh(c, st);
}

int dvc_value_params(dvc_ctx* c, float* d_params, int direction, void* stream) {
    if (!c) return DVC_E_INVALID;
    if (!is_device_ptr(d_params, c->device) || (direction != 0 && direction != 1))
        return fail(c, DVC_E_INVALID, "dvc_value_params: device pointer and direction 0 (out) or 1 (in)");
    if (int rc = set_device(c)) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    if (direction == 1 && !c->vnet) {
        if (int rc = net_alloc(c)) return rc;
    }
    if (int rc = need_net(c)) return rc;
    dvc_value_net* v = c->vnet;
    const cudaError_t e = direction == 0 ? cudaMemcpyAsync(d_params, v->master, NPARAM * 4, cudaMemcpyDeviceToDevice, st)
                                         : cudaMemcpyAsync(v->master, d_params, NPARAM * 4, cudaMemcpyDeviceToDevice, st);
    if (e != cudaSuccess) return cuda_fail(c, e, "dvc_value_params");
    return direction == 1 ? refresh(c, st) : DVC_OK;
}

int dvc_value_features(dvc_ctx* c, const dvc_state* d_states, int n, float* d_out, void* stream) {
    if (!c) return DVC_E_INVALID;
    if (int rc = check_states_args(c, d_states, n)) return rc;
    if (n == 0) return DVC_OK;
    if (!is_device_ptr(d_out, c->device)) return fail(c, DVC_E_INVALID, "dvc_value_features: d_out must be device memory");
    if (int rc = set_device(c)) return rc;
    features_kernel<<<(n + kFeatRows - 1) / kFeatRows, kFeatThreads, 0, (cudaStream_t)stream>>>(d_states, n, n, nullptr, d_out, 0);
    return check_launch(c, "features_kernel");
}

int dvc_value_eval(dvc_ctx* c, const dvc_state* d_leaves, int n, float* d_winprob, void* stream) {
    if (!c) return DVC_E_INVALID;
    if (int rc = check_states_args(c, d_leaves, n)) return rc;
    if (n == 0) return DVC_OK;
    if (!is_device_ptr(d_winprob, c->device)) return fail(c, DVC_E_INVALID, "dvc_value_eval: d_winprob must be device memory");
    if (int rc = set_device(c)) return rc;
    if (int rc = need_net(c)) return rc;
    const int npad = (n + 127) / 128 * 128;
    if (int rc = ensure_work(c, npad)) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    dvc_value_net* v = c->vnet;
    return infer(c, d_leaves, n, npad, v->X, v->H1, v->H2, v->L, d_winprob, st, false);
}

int dvc_value_train_step(dvc_ctx* c, const dvc_state* d_states, const float* d_labels, int n, float lr, float* d_loss,
                         void* stream) {
    if (!c) return DVC_E_INVALID;
    if (int rc = check_states_args(c, d_states, n)) return rc;
    if (n == 0) return DVC_OK;
    if (!is_device_ptr(d_labels, c->device) || (d_loss && !is_device_ptr(d_loss, c->device)) || !(lr >= 0.0f))
        return fail(c, DVC_E_INVALID, "dvc_value_train_step: device labels/loss, lr >= 0");
    if (int rc = set_device(c)) return rc;
    if (int rc = need_net(c)) return rc;
    const int npad = (n + 127) / 128 * 128;
    if (int rc = ensure_work(c, npad)) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    dvc_value_net* v = c->vnet;
    int32_t* fl = c->d_flags;
    if (int rc = forward_into(c, d_states, n, npad, v->X, v->H1, v->H2, v->H3, v->L, v->Z1, v->Z2, v->Z3, false, st))
        return rc;
    cudaError_t e = launch_chained(loss_grad_kernel, (unsigned)(npad / kLossThreads), kLossThreads, 0, st, v->L, d_states,
                                   d_labels, n, npad, v->dZ4, v->L + (size_t)npad * VO, v->rowpart);
    // the gradient at each hidden layer, from the top
    const size_t blocks = (size_t)npad / 32 * VH;
    if (e == cudaSuccess) e = gemm_back(v->dZ4, 64, v->W4, v->Z3, v->dZ[2], v->colsum + 2 * blocks, npad, fl, st);
    if (e == cudaSuccess)
        e = gemm_back(v->dZ[2], VH, v->W3, v->Z2, v->dZ[1], v->colsum + blocks, npad, fl, st);
    if (e == cudaSuccess) e = gemm_back(v->dZ[1], VH, v->W2, v->Z1, v->dZ[0], v->colsum, npad, fl, st);
    if (e == cudaSuccess) e = gemm_dw(v, n, npad, fl, st);
    if (e != cudaSuccess) return cuda_fail(c, e, "value backward");
    v->step += 1;
    AdamCoef a{lr, 0.9f, 0.999f, 1e-8f, 1e-4f, 0.0f, 0.0f};
    a.c1 = 1.0f - powf(a.b1, (float)v->step);
    a.c2 = 1.0f - powf(a.b2, (float)v->step);
    e = launch_chained(adamw_kernel, kAdamGrid, kAdamThreads, 0, st, *v, npad / 32, npad / kLossThreads, n, a, d_loss);
    return e == cudaSuccess ? DVC_OK : cuda_fail(c, e, "adamw_kernel");
}

int dvc_value_grads(dvc_ctx* c, float* d_out, void* stream) {
    if (!c) return DVC_E_INVALID;
    if (!is_device_ptr(d_out, c->device)) return fail(c, DVC_E_INVALID, "dvc_value_grads: d_out must be device memory");
    if (int rc = need_net(c)) return rc;
    if (int rc = set_device(c)) return rc;
    const cudaError_t e =
        cudaMemcpyAsync(d_out, c->vnet->grad, NPARAM * 4, cudaMemcpyDeviceToDevice, (cudaStream_t)stream);
    return e == cudaSuccess ? DVC_OK : cuda_fail(c, e, "dvc_value_grads");
}

// File: "DVCV" magic, u32 version 1, u64 parameter count, i64 Adam step,
// then master weights, first and second moments (FP32 each).
int dvc_value_save(dvc_ctx* c, const char* path) {
    if (!c || !path) return DVC_E_INVALID;
    if (int rc = need_net(c)) return rc;
    if (int rc = set_device(c)) return rc;
    if (cudaDeviceSynchronize() != cudaSuccess) return fail(c, DVC_E_CUDA, "dvc_value_save: sync");
    dvc_value_net* v = c->vnet;
    std::vector<float> buf(3 * NPARAM);
    if (cudaMemcpy(buf.data(), v->master, NPARAM * 4, cudaMemcpyDeviceToHost) != cudaSuccess ||
        cudaMemcpy(buf.data() + NPARAM, v->m, NPARAM * 4, cudaMemcpyDeviceToHost) != cudaSuccess ||
        cudaMemcpy(buf.data() + 2 * NPARAM, v->v, NPARAM * 4, cudaMemcpyDeviceToHost) != cudaSuccess)
        return fail(c, DVC_E_CUDA, "dvc_value_save: copy");
    FILE* f = std::fopen(path, "wb");
    if (!f) return fail(c, DVC_E_INVALID, std::string("dvc_value_save: cannot open ") + path);
    const char magic[4] = {'D', 'V', 'C', 'V'};
    const uint32_t ver = 1;
    const uint64_t np = NPARAM;
    const int64_t step = v->step;
    bool ok = std::fwrite(magic, 1, 4, f) == 4 && std::fwrite(&ver, 4, 1, f) == 1 && std::fwrite(&np, 8, 1, f) == 1 &&
              std::fwrite(&step, 8, 1, f) == 1 && std::fwrite(buf.data(), 4, buf.size(), f) == buf.size();
    ok = (std::fclose(f) == 0) && ok;
    return ok ? DVC_OK : fail(c, DVC_E_INVALID, "dvc_value_save: write failed");
}

int dvc_value_load(dvc_ctx* c, const char* path) {
    if (!c || !path) return DVC_E_INVALID;
    if (int rc = set_device(c)) return rc;
    if (int rc = net_alloc(c)) return rc;
    FILE* f = std::fopen(path, "rb");
    if (!f) return fail(c, DVC_E_INVALID, std::string("dvc_value_load: cannot open ") + path);
    char magic[4];
    uint32_t ver = 0;
    uint64_t np = 0;
    int64_t step = 0;
    std::vector<float> buf(3 * NPARAM);
    bool ok = std::fread(magic, 1, 4, f) == 4 && std::memcmp(magic, "DVCV", 4) == 0 && std::fread(&ver, 4, 1, f) == 1 &&
              ver == 1 && std::fread(&np, 8, 1, f) == 1 && np == NPARAM && std::fread(&step, 8, 1, f) == 1 &&
              std::fread(buf.data(), 4, buf.size(), f) == buf.size();
    std::fclose(f);
    if (!ok) return fail(c, DVC_E_INVALID, "dvc_value_load: not a version-1 value-network file");
    dvc_value_net* v = c->vnet;
    if (cudaMemcpy(v->master, buf.data(), NPARAM * 4, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(v->m, buf.data() + NPARAM, NPARAM * 4, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(v->v, buf.data() + 2 * NPARAM, NPARAM * 4, cudaMemcpyHostToDevice) != cudaSuccess)
        return fail(c, DVC_E_CUDA, "dvc_value_load: copy");
    v->step = step;
    if (int rc = refresh(c, nullptr)) return rc;
    return cudaDeviceSynchronize() == cudaSuccess ? DVC_OK : fail(c, DVC_E_CUDA, "dvc_value_load: sync");
}

int dvc_gemm_timeout_probe(dvc_ctx* c, const void* d_A, const void* d_B, float* d_Cf, int M, int N, int K,
                           int wait_ms, void* stream) {
    if (!c) return DVC_E_INVALID;
    if (M < 1 || N < 16 || N % 16 || K < 64 || K % 64 || wait_ms < 1 || wait_ms > 1000)
        return fail(c, DVC_E_INVALID, "dvc_gemm_timeout_probe: M >= 1, N % 16 == 0, K % 64 == 0, wait 1..1000 ms");
    if (!is_device_ptr(d_A, c->device) || !is_device_ptr(d_B, c->device) || !is_device_ptr(d_Cf, c->device))
        return fail(c, DVC_E_INVALID, "dvc_gemm_timeout_probe: device pointers");
    if (int rc = set_device(c)) return rc;
    GemmArgs a{(const __nv_bfloat16*)d_A, (const __nv_bfloat16*)d_B, nullptr, nullptr, d_Cf, M, N, K, kActNone,
               c->d_flags, (uint64_t)wait_ms * 1000000ull, 1, nullptr, nullptr, 0};
    cudaError_t e;
    if (N % 256 == 0) e = launch_gemm<256>(a, (cudaStream_t)stream, false);
    else if (N % 128 == 0) e = launch_gemm<128>(a, (cudaStream_t)stream, false);
    else if (N % 64 == 0) e = launch_gemm<64>(a, (cudaStream_t)stream, false);
    else if (N % 32 == 0) e = launch_gemm<32>(a, (cudaStream_t)stream, false);
    else e = launch_gemm<16>(a, (cudaStream_t)stream, false);
    return e == cudaSuccess ? DVC_OK : cuda_fail(c, e, "dvc_gemm_timeout_probe");
}

int dvc_gemm_bf16(dvc_ctx* c, const void* d_A, const void* d_B, const float* d_bias, void* d_C, float* d_Cf, int M,
                  int N, int K, int act, void* stream) {
    if (!c) return DVC_E_INVALID;
    if (M < 1 || N < 16 || N % 16 || K < 64 || K % 64 || (act != kActNone && act != kActGelu))
        return fail(c, DVC_E_INVALID, "dvc_gemm_bf16: M >= 1, N % 16 == 0, K % 64 == 0, act 0 or 1");
    if (!is_device_ptr(d_A, c->device) || !is_device_ptr(d_B, c->device) || (d_bias && !is_device_ptr(d_bias, c->device)) ||
        (d_C && !is_device_ptr(d_C, c->device)) || (d_Cf && !is_device_ptr(d_Cf, c->device)) || (!d_C && !d_Cf))
        return fail(c, DVC_E_INVALID, "dvc_gemm_bf16: device pointers, at least one output");
    if ((uintptr_t)d_C % 16 || (uintptr_t)d_Cf % 16 || (uintptr_t)d_A % 16 || (uintptr_t)d_B % 16)
        return fail(c, DVC_E_INVALID, "dvc_gemm_bf16: A, B, C and Cf must be 16-byte aligned");
    if (int rc = set_device(c)) return rc;
    const cudaError_t e = gemm((const __nv_bfloat16*)d_A, (const __nv_bfloat16*)d_B, d_bias, (__nv_bfloat16*)d_C, d_Cf,
                               M, N, K, act, c->d_flags, (cudaStream_t)stream);
    return e == cudaSuccess ? DVC_OK : cuda_fail(c, e, "dvc_gemm_bf16");
}

}  // extern "C"

int dvc_value_rows_alloc(dvc_ctx* c, dvc_value_rows* r, int rows) {
    dvc_value_rows_free(r);
    const size_t n = (size_t)rows;
    const bool ok = cudaMalloc(&r->X, n * VF * 2) == cudaSuccess && cudaMalloc(&r->H1, n * VH * 2) == cudaSuccess &&
                    cudaMalloc(&r->H2, n * VH * 2) == cudaSuccess &&
                    cudaMalloc(&r->L, n * kLogitFloats * 4) == cudaSuccess;
    if (!ok) {
        cudaGetLastError();
        dvc_value_rows_free(r);
        return fail(c, DVC_E_OOM, "value network: activation rows");
    }
    r->rows = rows;
    return DVC_OK;
}

void dvc_value_rows_free(dvc_value_rows* r) {
    void* ptrs[] = {r->X, r->H1, r->H2, r->L};
    for (void* p : ptrs)
        if (p) cudaFree(p);
    *r = dvc_value_rows{};
}

int dvc_value_prepare(dvc_ctx* c) {
    if (int rc = need_net(c)) return rc;
    cudaError_t e = gemm_attributes<256>();
    if (e == cudaSuccess) e = gemm_attributes<128>();
    if (e == cudaSuccess) e = gemm_attributes<64>();
    if (e == cudaSuccess) e = gemm_attributes<32>();
    if (e == cudaSuccess) e = gemm_attributes<16>();
    if (e == cudaSuccess) e = mlp_attributes();
    return e == cudaSuccess ? DVC_OK : cuda_fail(c, e, "value network attributes");
}

int dvc_value_forward_rows(dvc_ctx* c, const dvc_state* d_leaves, int n, dvc_value_rows* r, int row0, float* d_probs,
                           cudaStream_t st, bool chained) {
    if (n <= 0) return DVC_OK;
    const int npad = (n + 127) / 128 * 128;
    if (row0 < 0 || row0 + npad > r->rows) return fail(c, DVC_E_INVALID, "value network: activation rows");
    const size_t o = (size_t)row0;
    return infer(c, d_leaves, n, npad, (__nv_bfloat16*)r->X + o * VF, (__nv_bfloat16*)r->H1 + o * VH,
                 (__nv_bfloat16*)r->H2 + o * VH, r->L + o * kLogitFloats, d_probs, st, chained);
}

void dvc_value_free(dvc_ctx* c) {
    if (!c || !c->vnet) return;
    dvc_value_net* v = c->vnet;
    free_work(v);
    void* ptrs[] = {v->master, v->m, v->v, v->grad, v->W1, v->W2, v->W3, v->W4, v->b4p};
    for (void* p : ptrs)
        if (p) cudaFree(p);
    delete v;
    c->vnet = nullptr;
}
