"""Host checks of the FP32 phase 1's shared memory (no GPU), with the numbers the
kernel is compiled with: two CTAs of every shape fit an SM, the two 32-bit words
that a thread decodes its two samples from lie inside a row's copied bytes for
every alignment of the first sample (the last row's may reach into the ring's 16
bytes of slack), and they give back the samples."""
import json
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2303_09886_gb300 import synth

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_2303_09886_gb300", "csrc")
SHAPES = [(8, 64), (16, 32), (32, 16), (64, 8), (8, 32), (8, 16), (8, 8), (8, 4)]
SMEM_PER_SM, RESERVED_PER_CTA, SMEM_PER_CTA = 228 * 1024, 1024, 227 * 1024

PROGRAM = """
#include "k_phase1.cuh"
#include <cstdio>
template <int T, int N1, int W> void row(const char *end) {
    using S = fe::P1Shape<T, N1, W>;
    std::printf("{\\"T\\": %d, \\"N1\\": %d, \\"W\\": %d, \\"smem\\": %d, \\"seg\\": %d, \\"ns\\": %d, \\"rowb\\": %d, "
                "\\"ring\\": %d, \\"align\\": %d, \\"nw\\": %d, \\"stage\\": %d}%s\\n", T, N1, W, (int)S::SMEM, S::SEG, S::NS,
                S::ROWB, S::RING, (int)S::ALIGN, S::NW, S::STAGE_BYTES, end);
}
template <int T> void rows(const char *end) {
    row<T, 8, 64>(","); row<T, 16, 32>(","); row<T, 32, 16>(","); row<T, 64, 8>(",");
    row<T, 8, 32>(","); row<T, 8, 16>(","); row<T, 8, 8>(","); row<T, 8, 4>(end);
}
int main() {
    std::printf("["); rows<1>(","); rows<2>(","); rows<4>(","); rows<8>(","); rows<16>(","); rows<32>("]");
}
"""


@pytest.fixture(scope="module")
def shapes(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc is needed")
    d = tmp_path_factory.mktemp("layout")
    (d / "l.cu").write_text(PROGRAM)
    subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I" + CSRC, str(d / "l.cu"), "-o",
                    str(d / "l")], check=True)
    return json.loads(subprocess.run([str(d / "l")], check=True, capture_output=True, text=True).stdout)


def test_two_ctas_fit(shapes):
    assert {(s["N1"], s["W"]) for s in shapes} == set(SHAPES) and len(shapes) == 6 * len(SHAPES)
    for s in shapes:
        per_cta = s["smem"] + 32 * 4 + RESERVED_PER_CTA      # and a block's coarse delays
        assert 2 * per_cta <= SMEM_PER_SM and s["smem"] <= SMEM_PER_CTA, s


def _byte(s):
    return 10 * s // 8


def test_both_words_lie_in_the_copied_row_and_give_the_samples(shapes):
    rng = np.random.default_rng(20230317)
    for sh in [s for s in shapes if s["T"] == 16]:
        W, seg, align = sh["W"], sh["seg"], sh["align"]
        x = rng.integers(-512, 512, 512 + 4 * W + 64).astype(np.int16)
        x = x[:x.size // 4 * 4]
        b = synth.pack10(x)
        for s0 in range(0, 512):
            first = _byte(s0) // align * align                # the segment's copy starts here
            copied = np.zeros(seg + 16, np.uint8)             # (the next segment's bytes or the slack)
            n = min(seg, b.size - first)
            copied[:n] = b[first:first + n]
            for c in range(0, W, 2):
                o = _byte(s0 + c) - first
                lo = o & ~3
                # the second sample's second byte is copied; the two words end in the slack at most
                assert _byte(s0 + c + 1) + 1 - first < seg and lo + 8 <= seg + 16, (sh, s0, c)
                v = int.from_bytes(copied[o:o + 4].tobytes(), "big") >> (12 - 2 * ((s0 + c) & 3))
                got = [(v >> 10) & 0x3FF, v & 0x3FF]
                assert [g - ((g & 0x200) << 1) for g in got] == [int(x[s0 + c]), int(x[s0 + c + 1])], (sh, s0, c)
        assert sh["rowb"] == sh["ns"] * seg and sh["stage"] == sh["nw"] * sh["ring"] * sh["rowb"] + 16
