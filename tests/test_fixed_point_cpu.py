"""CPU checks of the fixed-point weights of the FP64 form: the very functions the kernels call
(csrc/pic_fixed.cuh, csrc/pic_ttable.cu), compiled for the host."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import paper_1909_09613_gb300 as pic
from paper_1909_09613_gb300 import _build

SOURCE = r"""
#include "pic_ttable.cu"
#include "pic_fixed.cuh"
using namespace pic;

template <int L, int KT>
static int eval(const TTable &t, const uint64_t *f, int n, int *base, uint64_t *w)
{
    for (int i = 0; i < n; ++i) base[i] = ttable_weights62<L, KT>(t, f[i], w + (size_t)i * KT);
    return KT;
}

// integer-node weights at n offsets f (units of 2^-64): base[n], w[n * K] in units of 2^-62;
// returns the number of nodes K, 0 where no table is built
extern "C" int weights62(int l, int scheme, double dtt, const uint64_t *f, int n, int *base,
                         uint64_t *w)
{
    TTable t;
    if (!build_ttable(l, scheme, dtt, &t, true)) return 0;
    const bool wide = t.K > l + 1;
    switch (l) {
    case 1: return wide ? eval<1, 3>(t, f, n, base, w) : eval<1, 2>(t, f, n, base, w);
    case 2: return wide ? eval<2, 4>(t, f, n, base, w) : eval<2, 3>(t, f, n, base, w);
    case 3: return wide ? eval<3, 5>(t, f, n, base, w) : eval<3, 4>(t, f, n, base, w);
    default: return wide ? eval<4, 6>(t, f, n, base, w) : eval<4, 5>(t, f, n, base, w);
    }
}
"""


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    _build.build()
    pic.load_library()
    d = tmp_path_factory.mktemp("fixed")
    src, so = str(d / "fixed.cu"), str(d / "fixed.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run([_build._nvcc(), "-O2", "-std=c++17", "--expt-relaxed-constexpr", "-Xcompiler",
                    "-fPIC", "-shared", "-I", _build.CSRC, "-I", _build.INCLUDE, src, "-o", so],
                   check=True, capture_output=True)
    lib = ctypes.CDLL(so)
    lib.weights62.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_double, ctypes.c_void_p,
                              ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p]
    return lib


def _weights62(host, l, scheme, dtt, deltas):
    f = np.array([int(d * 2.0 ** 64) for d in deltas], dtype=np.uint64)  # exact: 53 bits each
    base = np.zeros(len(f), dtype=np.int32)
    w = np.zeros(6 * len(f), dtype=np.uint64)
    k = host.weights62(l, scheme, dtt, f.ctypes.data, len(f), base.ctypes.data, w.ctypes.data)
    return k, base, w[: k * len(f)].reshape(len(f), k).astype(np.float64) * 2.0 ** -62


def _near(x):
    lo = np.nextafter(x, 0.0)
    hi = np.nextafter(x, 2.0)
    return [np.nextafter(lo, 0.0), lo, x, hi, np.nextafter(hi, 2.0)]


STEPS = _near(0.5) + [0.7 * 0.1 / 0.14, 0.25, 0.1, 0.7, 1 / 3] + _near(1.0)[:2]


@pytest.mark.parametrize("l", [1, 2, 3, 4])
@pytest.mark.parametrize("scheme", [pic.PIC_SCHEME_WT, pic.PIC_SCHEME_MC])
@pytest.mark.parametrize("dtt", STEPS)
def test_fixed_point_weights_equal_the_fp64_ones(host, l, scheme, dtt):
    """As functions of the node (a node one side leaves out counts as zero there): both sides
    round a few times at 2^-53 of a weight of at most 1.  A support less than half an FP32 ulp
    below an integer number of cells has no table in either form."""
    rng = np.random.default_rng(l)
    deltas = np.concatenate([rng.random(60), [0.0, 2.0 ** -53, 0.25, 0.5, 1.0 - 2.0 ** -53]])
    try:
        pic.pic_axis_weights(l, scheme, dtt, 0.5)
    except pic.PicError:
        below = -(l / 2 + dtt) % 1.0
        assert 0.0 < below < 2.0 ** -25
        assert host.weights62(l, scheme, dtt, None, 0, None, None) == 0
        return
    k, base, w = _weights62(host, l, scheme, dtt, deltas)
    assert k in (l + 1, l + 2)
    for i, d in enumerate(deltas):
        b0, w0 = pic.pic_axis_weights(l, scheme, dtt, float(d))
        a, b = np.zeros(24), np.zeros(24)
        a[12 + base[i]: 12 + base[i] + k] = w[i]
        b[12 + b0: 12 + b0 + len(w0)] = w0
        assert np.max(np.abs(a - b)) <= 4e-15, (d, dtt, base[i], b0)


@pytest.mark.parametrize("l", [1, 2, 3, 4])
@pytest.mark.parametrize("dtt", [0.25, 0.6, 1e-3, 1e-6, 1e-9])
def test_fixed_point_weights_sum_to_one(host, l, dtt):
    """In units of 2^-62, but where the others leave nothing for the middle weight, which is not
    negative (a few units of 2^-59 each; the table's own rounding of 2^-64 / dtt in the others)."""
    f = np.random.default_rng(l).integers(0, 2 ** 64, 2000, dtype=np.uint64)
    base, w = np.zeros(len(f), dtype=np.int32), np.zeros(6 * len(f), dtype=np.uint64)
    k = host.weights62(l, pic.PIC_SCHEME_WT, dtt, f.ctypes.data, len(f), base.ctypes.data, w.ctypes.data)
    w = w[: k * len(f)].reshape(len(f), k)
    left = w.sum(axis=1).astype(np.int64) - 2 ** 62
    assert np.all((left == 0) | ((w[:, k // 2] == 0) & (left > 0) & (left < 8 * 30 + 2 / dtt)))
    assert l == 1 or np.all(left == 0)
