"""Host checks of the sine-Gordon FP32 sine (no GPU needed): the polynomial that
threads with small values run alone gives, bit for bit, what the general sine
gives there, and a build with PSS_SG_LIBM_SIN never takes it.  Compiled from the
kernel header with nvcc, its FP32 intrinsics standing for the host's own
correctly rounded operations."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1206_3215_gb300", "csrc")

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <cuda_runtime.h>
// the header's device functions as host functions
#undef __device__
#undef __forceinline__
#define __device__
#define __forceinline__ inline
static inline float host_fma(float a, float b, float c) { return fmaf(a, b, c); }
#define __fmaf_rn host_fma
#include "sg_sin.cuh"
int main()
{
    long n = 0, bad = 0;
    for (unsigned i = 1; i < 0x3f800000u; i += 97) {  // positive floats below 1
        float x;
        memcpy(&x, &i, 4);
        for (float s : {x, -x}) {
            float2 v[2] = {{s, 0.0f}, {0.0f, s}};
            if (pss::sg_all_small(v, true) != (fabsf(s) <= pss::sg_sin_small && !PSS_SG_LIBM_SIN)) ++bad;
            if (fabsf(s) > pss::sg_sin_small) continue;
            const float a = pss::sg_sin_poly(s), b = pss::sg_sin(s);
            if (!PSS_SG_LIBM_SIN && memcmp(&a, &b, 4)) ++bad;
            ++n;
        }
    }
    const float nan = NAN;
    float2 w[1] = {{nan, nan}};
    if (!pss::sg_all_small(w, true) && !PSS_SG_LIBM_SIN) ++bad;  // (the polynomial carries NaN through)
    if (!std::isnan(pss::sg_sin_poly(nan)) || !std::isnan(pss::sg_sin_poly(-nan))) ++bad;
    std::printf("%ld %ld\n", n, bad);
    return 0;
}
"""


def _nvcc():
    for cand in (shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    return None


@pytest.mark.parametrize("libm", [0, 1])
def test_small_value_path_equals_the_general_sine(tmp_path, libm):
    nvcc = _nvcc()
    if nvcc is None:
        pytest.skip("nvcc not available")
    src, exe = tmp_path / "sine.cpp", tmp_path / "sine"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, "-x", "c++", "-std=c++17", "-O1", "-Xcompiler", "-ffp-contract=off",
                    f"-DPSS_SG_LIBM_SIN={libm}", "-I", CSRC, "-I", os.path.join(os.path.dirname(nvcc), "..", "include"),
                    str(src), "-o", str(exe)], check=True, capture_output=True)
    n, bad = (int(x) for x in subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split())
    assert n > 10_000_000
    assert bad == 0
