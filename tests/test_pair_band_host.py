"""The binary32 band around the cutoff (csrc/band.cuh), compiled for the host."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2204_03756_gb300 import build

SRC = """
#include "band.cuh"
extern "C" void band(double psi2, double eta, float* out) {
    const mtpt::PairBand b = mtpt::pair_band(psi2, eta);
    out[0] = b.lo;
    out[1] = b.hi;
    out[2] = b.reach2;
}
"""


@pytest.fixture(scope="module")
def band(tmp_path_factory):
    d = tmp_path_factory.mktemp("band")
    src, out = d / "band.cpp", d / "band.so"
    src.write_text(SRC)
    subprocess.run(["g++", "-O2", "-std=gnu++17", "-shared", "-fPIC", "-I", build.SRC_DIR,
                    "-o", str(out), str(src)], check=True)
    so = ctypes.CDLL(os.fspath(out))
    so.band.argtypes = [ctypes.c_double, ctypes.c_double, ctypes.c_void_p]

    def call(psi2, eta):
        r = np.empty(3, np.float32)
        so.band(psi2, eta, r.ctypes.data)
        return r
    return call


# (0 and infinity: what psi^2 and w / psi become beyond binary64's range)
@pytest.mark.parametrize("eta", [1e-14, 1e-6, 0.5, 1.0 - 1e-9, 1.0, 1.0 + 1e-9, 1.013, 10.6, 4e6,
                                 1e30, np.inf])
@pytest.mark.parametrize("psi2", [0.0, 1e-300, 1e-42, 1.8e-8, 1.0, 1.5625, 4e3, 1e37, 1e200, np.inf])
def test_the_searches_may_compare_the_band_by_its_bits(band, psi2, eta):
    """The search takes the sign of bits(d2) - bits(lo) for d2 < lo, and
    bits(d2) - bits(lo) <= bits(hi) - bits(lo), unsigned, for d2 inside the band:
    right for every d2 >= 0 as long as neither bound has a sign bit or is a NaN."""
    lo, hi, reach2 = band(psi2, eta)
    assert not np.signbit(lo) and lo <= hi <= reach2
    # around psi2 as far as binary32 and eta reach
    assert float(lo) <= psi2 * max(1.0 - eta, 0.0) if psi2 * eta < np.inf else True
    assert float(hi) >= min(psi2, 3.4e38)
    rng = np.random.default_rng(1)
    d2 = np.concatenate([np.float32([0.0, 1e-45, 1.0, np.inf, lo, hi]),
                         np.exp(rng.uniform(-103.0, 88.0, 4000)).astype(np.float32),
                         rng.uniform(0.0, 3.0, 2000).astype(np.float32) * np.float32(min(psi2, 1e38))])
    t = d2.view(np.uint32) - lo.view(np.uint32)
    assert np.array_equal(t.view(np.int32) < 0, d2 < lo)
    assert np.array_equal((d2 >= lo) & (t <= hi.view(np.uint32) - lo.view(np.uint32)),
                          (d2 >= lo) & (d2 <= hi))
