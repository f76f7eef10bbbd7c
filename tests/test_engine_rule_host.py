"""The default engine of a forest (host logic, no GPU): the library's own rule,
compiled for the host, follows the fullest CTA of the fused engine, not the
chip's average, and under the ordering-aware policy a forest of few trees never
leaves the fused engine, whose CTAs of one and two trees its pipeline loses to."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r'''
#include <cstdio>
#include "dvc_shape.cuh"
int main() {
    char what;
    int a, b, c, d, e;
    while (std::scanf(" %c %d %d %d %d %d", &what, &a, &b, &c, &d, &e) == 6)
        std::printf("%d\n", what == 'e'   ? dvc::default_engine(a, b, c, d != 0)
                            : what == 'p' ? (int)dvc::play_alone(a, b, c, d, e)
                            : what == 'l' ? dvc::fused_launch_iterations(a, b, c)
                                          : dvc::default_value_chains(a, b));
    return 0;
}
'''


@pytest.fixture(scope="module")
def engine(tmp_path_factory):
    if shutil.which("nvcc") is None:
        pytest.skip("nvcc not found")
    d = tmp_path_factory.mktemp("rule")
    src, exe = d / "r.cu", d / "r"
    src.write_text(SRC)
    subprocess.run(["nvcc", "-std=c++17", "-I" + os.path.join(ROOT, "paper_2403_10720_gb300", "csrc"), str(src), "-o",
                    str(exe)], check=True, capture_output=True)

    def ask(rows, what="e"):
        text = "\n".join(" ".join(map(str, (what, *r, *[0] * (5 - len(r))))) for r in rows)
        out = subprocess.run([str(exe)], input=text, check=True, capture_output=True, text=True).stdout
        return [int(x) for x in out.split()]
    return ask


TREES = [1, 2, 3, 40, 75, 151, 152, 153, 304, 305, 457, 608, 609, 1217, 2281, 2432, 2433, 4864, 4865, 1 << 20]
PLAYOUTS = [1, 15, 16, 17, 32, 33, 57, 128, 129, 170, 171, 256, 257, 512, 513, 1024, 65536, 1 << 20]


@pytest.mark.parametrize("sms", [152, 76, 1])
def test_uniform_playouts_follow_the_fullest_cta(engine, sms):
    rows = [(n, sms, P, 0) for n in TREES for P in PLAYOUTS]
    for (n, _, P, _), e in zip(rows, engine(rows)):
        trees = -(-n // sms)
        assert e == (1 if trees <= 32 and trees * P <= 512 else 2), (n, P)


def test_ordering_aware(engine):
    rows = [(n, 152, P, 1) for n in TREES for P in PLAYOUTS]
    for (n, _, P, _), e in zip(rows, engine(rows)):
        if n <= 304:
            assert e == 1, (n, P)
        elif n > 608:
            assert e == 2, (n, P)
        elif -(-n // 152) * P <= 512:
            assert e == 1, (n, P)
    assert engine([(400, 152, 200, 1), (400, 152, 256, 1), (400, 152, 400, 1), (608, 152, 129, 1)]) == [2, 2, 1, 2]


def test_form_of_two_player_playouts(engine):
    # CTAs, SMs, trees and warps of a CTA, playouts
    rows = {(1, 152, 1, 1, 1): 1, (1, 152, 1, 12, 384): 1, (1, 152, 1, 13, 385): 0, (1, 152, 1, 16, 1 << 20): 0,
            (152, 152, 7, 7, 32): 1, (143, 152, 14, 14, 32): 0, (152, 152, 32, 16, 8): 1, (152, 152, 32, 16, 16): 0,
            (456, 152, 4, 4, 32): 1, (457, 152, 4, 4, 32): 0, (457, 152, 4, 4, 1): 0, (1 << 18, 152, 4, 5, 1): 1}
    assert engine(list(rows), "p") == list(rows.values())


def test_value_chains(engine):
    # 152 SMs: eight chains of up to five tiles of 128 leaves
    rows = {(1, 152): 1, (2432, 152): 1, (2433, 152): 8, (5120, 152): 8, (5121, 152): 1, (1 << 20, 152): 1,
            (1216, 76): 1, (1217, 76): 8, (2048, 76): 8, (2049, 76): 1, (100, 4): 1}
    assert engine(list(rows), "v") == list(rows.values())


def test_launches_end_before_their_counts_wrap(engine):
    # trees and warps of a CTA, playouts; a game has at most 128 steps of four words
    rows = [(T, W, P) for T in (1, 2, 14, 32, 64) for W in (1, 3, 16, 32) for P in (1, 32, 256, 4096, 1 << 20)]
    for (T, W, P), n in zip(rows, engine(rows, "l")):
        games = -(-T * P // (32 * W))
        assert n >= 1 and n * games * 512 < 1 << 32
        assert (n + 1) * games * 512 > 0.99 * (1 << 32) or n > 1000
