"""Every length of the two-pass transforms (FP32) at the edges of its range, against the FP64 oracle.

A length P serves lattices of n <= P/2 sites along an axis; the largest n, the smallest one that is padded to
P, and odd ones between take different numbers of zero inputs and dropped outputs.  Layer counts 1 to 8 each
have their own y/z kernel.  Tolerance as in the other field tests: 1e-5 of max |h|, the FP32 field bound.
"""
import numpy as np
import pytest

import oracle
from paper_1804_07135_gb300 import binding
from paper_1804_07135_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# (P, smallest n padded to P, largest n)
LENGTHS = [(32, 13, 16), (48, 17, 24), (64, 25, 32), (80, 33, 40), (96, 41, 48), (112, 49, 54), (128, 55, 64),
           (144, 65, 72), (160, 73, 80), (192, 81, 96), (224, 97, 108), (256, 109, 128), (288, 129, 144),
           (320, 145, 160), (384, 161, 192), (448, 193, 216), (512, 217, 256)]


def _check(case, seed):
    nx, ny, nz, J, D, K, w, n = case
    path = W.random_spins((n, nx * ny * nz, 3), seed=seed).astype(np.float32)
    with binding.StringMethod([case]) as sm:
        sm.set_path(0, path)
        start = sm.get_path(0)
        got = sm.field(0, dtype=np.float32)
        cfg = sm.launch_config(0)
    m = oracle.model(nx, ny, nz, J, D, K, w)
    for k in range(n):
        s = start[k] / np.linalg.norm(start[k], axis=-1, keepdims=True)
        ref = oracle.field(m, s)
        assert np.abs(got[k] - ref).max() <= 1e-5 * np.abs(ref).max(), (case, k)
    return cfg


@pytest.mark.parametrize("i", range(len(LENGTHS)))
def test_x_and_yz_kernels_at_the_edges_of_each_length(i):
    P, lo, hi = LENGTHS[i]
    nz = 1 + i % 8
    for n in (lo, (lo + hi) // 2 | 1, hi):
        if n > hi:
            continue
        other = 14 if P < 200 else 5
        assert _check((n, other, nz, 1.0, 0.3, 0.1, 0.03, 3), seed=i)["Px"] == P
        assert _check((other + 1, n, nz, 1.0, -0.3, 0.1, 0.03, 2), seed=50 + i)["Py"] == P


@pytest.mark.parametrize("nz", range(1, 10))
def test_every_layer_count(nz):
    # 9 layers leave the two-pass y/z kernel for the runtime plan
    cfg = _check((22, 29, nz, 1.0, 0.3, 0.1, 0.03, 3), seed=nz)
    assert cfg["Px"] == 48 and cfg["Py"] == 64
    cfg = _check((13, 37, nz, 1.0, 0.3, 0.1, 0.03, 2), seed=90 + nz)
    assert cfg["Px"] == 32 and cfg["Py"] == (80 if nz <= 8 else 81)


@pytest.mark.parametrize("case", [(13, 30, 1), (24, 40, 2), (50, 17, 3), (33, 20, 4), (75, 6, 5), (4, 100, 6),
                                  (45, 8, 7), (5, 129, 8), (150, 4, 8)])
def test_fp64_kernels(case):
    # the same kernels in FP64: the FP64 field bound of the other parity tests, 1e-12 of max |h|
    nx, ny, nz = case
    desc = (nx, ny, nz, 1.0, 0.3, 0.1, 0.03, 3)
    path = W.random_spins((3, nx * ny * nz, 3), seed=nx)
    with binding.StringMethod([desc], precision=binding.SS_PREC_FP64) as sm:
        sm.set_path(0, path)
        got, e = sm.field(0), sm.energies(0)
    m = oracle.model(*desc[:7])
    want = oracle.energies(m, path)
    assert np.abs(e - want).max() <= 1e-11 * np.abs(want).max()
    for k in range(3):
        ref = oracle.field(m, path[k])
        assert np.abs(got[k] - ref).max() <= 1e-12 * np.abs(ref).max(), k
