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


# Energies alone stop at the spectrum (two columns of it in shared memory): every layer count, even and odd image
# counts, x lengths with and without a middle column, the largest y length that fits and the first that does not
@pytest.mark.parametrize("case", [(20, 33, 1, 3), (40, 30, 2, 2), (17, 24, 3, 4), (30, 64, 4, 5), (5, 30, 5, 2),
                                  (21, 50, 6, 3), (7, 16, 7, 2), (33, 20, 8, 3), (5, 128, 8, 3), (4, 129, 8, 2),
                                  (6, 256, 1, 3), (3, 14, 2, 2), (150, 9, 5, 3), (4, 222, 4, 2), (2, 130, 5, 2)])
def test_energies_without_the_field(case):
    # bounds of the other energy tests: FP64 context 1e-11 of the largest energy's terms, an FP32 context's FP64
    # energies the same against the oracle at its own stored (FP32) spins
    nx, ny, nz, n = case
    desc = (nx, ny, nz, 1.0, 0.3, 0.1, 0.4, n)
    m = oracle.model(*desc[:7])
    path = W.random_spins((n, nx * ny * nz, 3), seed=nx)
    for prec in (binding.SS_PREC_FP64, binding.SS_PREC_FP32):
        with binding.StringMethod([desc], precision=prec) as sm:
            sm.set_path(0, path)
            s = sm.get_path(0)
            s = s / np.linalg.norm(s, axis=-1, keepdims=True)
            want = oracle.energies(m, s)
            e = sm.energies(0)
        scale = np.abs(want).max() + nx * ny * nz
        assert np.abs(e - want).max() <= 1e-11 * scale


def test_fp32_input_spins_normalised_to_the_last_bit():
    # FP32 spins of any norm, in and beyond the range the FP32-pair arithmetic takes (squared norms 1e-6 to 1e6),
    # with components that vanish or underflow.  Tolerance: one rounding to FP32 (0.5 units in the last place), and
    # 1e-6 for what the arithmetic before it may leave.
    rng = np.random.default_rng(5)
    nx, ny, K = 23, 13, 5
    v = W.random_spins((K, nx * ny, 3), seed=3)
    scale = 10.0 ** rng.choice([0, 0, -1, 1, -2.9, 2.9, -3.1, 3.1, -15, 15], (K, nx * ny, 1))
    v = (v * scale).astype(np.float32)
    v[0, ::3, 0] = 0.0
    v[1, ::4, 1:] = 0.0
    v[2, ::5, 2] *= np.float32(1e-20)
    v[3, :, 0] = np.float32(2.0 ** -63)
    with binding.StringMethod([(nx, ny, 1, 1.0, 0.3, 0.1, 0.0, K)]) as sm:
        sm.set_path(0, v)
        got = sm.get_path(0)
        w = v.astype(np.longdouble)
        ref = w / np.sqrt((w * w).sum(-1, keepdims=True))
        ulp = np.maximum(np.spacing(np.abs(ref).astype(np.float32)), np.float32(1e-45)).astype(np.longdouble)
        assert (np.abs(got.astype(np.float32) - ref) / ulp).max() <= 0.5 + 1e-6
        for bad in ([0, 0, 0], [np.inf, 0, 1], [np.nan, 1, 0]):
            w = v.copy()
            w[4, -1] = bad
            with pytest.raises(binding.SsError):
                sm.set_path(0, w)
                sm.get_path(0)
            sm.set_path(0, v)


# FP64 lengths at the lines of their rule: few y/z CTAs (short lengths), a two-pass x length too much longer (short x
# beside a two-pass y), about as long, and one whose short x the y/z kernel does not take
@pytest.mark.parametrize("case,Px,Py", [((13, 17, 2, 11), 27, 36), ((13, 17, 2, 13), 32, 48), ((25, 32, 8, 8), 54, 64),
                                        ((19, 14, 5, 10), 48, 32), ((14, 20, 4, 14), 32, 48), ((5, 14, 3, 6), 9, 27)])
def test_fp64_padded_lengths(case, Px, Py):
    nx, ny, nz, n = case
    desc = (nx, ny, nz, 1.0, 0.3, 0.1, 0.03, n)
    path = W.random_spins((n, nx * ny * nz, 3), seed=ny)
    with binding.StringMethod([desc], precision=binding.SS_PREC_FP64) as sm:
        cfg = sm.launch_config(0)
        sm.set_path(0, path)
        got = sm.field(0)
    assert (cfg["Px"], cfg["Py"]) == (Px, Py)
    m = oracle.model(*desc[:7])
    for k in (0, n - 1):  # the FP64 field bound
        ref = oracle.field(m, path[k])
        assert np.abs(got[k] - ref).max() <= 1e-12 * np.abs(ref).max(), k
