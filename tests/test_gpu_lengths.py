"""Fields and energies where the x length keeps the two-pass y/z kernel away: narrow strips and wide films whose Px its
columns per CTA do not divide, with a ny whose two-pass length has a factor 5 or 7, in both precisions, against the
FP64 oracle.  Bounds of the other parity tests: FP32 field 1e-5 of max |h|, FP64 field 1e-12, energies 1e-11 of the
largest energy's terms.
"""
import numpy as np
import pytest

import oracle
from paper_1804_07135_gb300 import binding
from paper_1804_07135_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# (nx, ny, nz, images); the last three have the image pairs that take FP64 past its rule for small grids
CASES = [(9, 35, 1, 2), (9, 100, 1, 3), (6, 50, 1, 2), (5, 76, 3, 3), (2, 100, 4, 2), (3, 150, 2, 2), (350, 35, 1, 2), (5, 81, 1, 3),
         (326, 33, 2, 2), (9, 33, 1, 240), (2, 40, 4, 140), (9, 50, 1, 240)]


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("case", CASES)
def test_field_and_energies(case, precision):
    nx, ny, nz, n = case
    desc = (nx, ny, nz, 1.0, 0.3, 0.1, 0.4, n)
    path = W.random_spins((n, nx * ny * nz, 3), seed=nx + ny)
    prec = binding.SS_PREC_FP64 if precision == "fp64" else binding.SS_PREC_FP32
    with binding.StringMethod([desc], precision=prec) as sm:
        sm.set_path(0, path)
        s = sm.get_path(0)
        field, energies = sm.field(0), sm.energies(0)
    s = s / np.linalg.norm(s, axis=-1, keepdims=True)
    m = oracle.model(*desc[:7])
    some = sorted({0, 1, n - 1})
    want = oracle.energies(m, s[some])
    assert np.abs(energies[some] - want).max() <= 1e-11 * (np.abs(want).max() + nx * ny * nz)
    for k in some:
        ref = oracle.field(m, s[k])
        assert np.abs(field[k] - ref).max() <= (1e-12 if precision == "fp64" else 1e-5) * np.abs(ref).max(), k


# FP64 at Px = 32: the two-pass x kernels (two rows per CTA, 128 threads) up to 700 CTAs, the runtime-plan ones beyond
@pytest.mark.parametrize("case", [(16, 40, 2, 34), (16, 40, 2, 36), (14, 33, 1, 82), (13, 35, 3, 27)])
def test_fp64_x_kernels_at_32_points(case):
    nx, ny, nz, n = case
    desc = (nx, ny, nz, 1.0, 0.3, 0.1, 0.03, n)
    path = W.random_spins((n, nx * ny * nz, 3), seed=ny)
    with binding.StringMethod([desc], precision=binding.SS_PREC_FP64) as sm:
        cfg = sm.launch_config(0)
        sm.set_path(0, path)
        field, energies = sm.field(0), sm.energies(0)
    assert cfg["Px"] == 32
    two_pass = (ny + 1) // 2 * nz * ((n + 1) // 2) <= 700
    assert ((cfg["rows_xfwd"], cfg["threads_xfwd"]) == (2, 128)) == two_pass
    m = oracle.model(*desc[:7])
    want = oracle.energies(m, path)
    assert np.abs(energies - want).max() <= 1e-11 * (np.abs(want).max() + nx * ny * nz)
    for k in (0, n // 2, n - 1):
        ref = oracle.field(m, path[k])
        assert np.abs(field[k] - ref).max() <= 1e-12 * np.abs(ref).max(), k


# FP64 with 13 or 14 sites along y: short lengths up to the line of each layer count, two-pass lengths beyond it
@pytest.mark.parametrize("case,Px,Py", [((14, 14, 2, 22), 27, 27), ((14, 14, 2, 24), 32, 32), ((10, 14, 3, 20), 24, 27),
                                        ((10, 13, 3, 22), 24, 32), ((15, 13, 4, 14), 32, 27), ((15, 13, 4, 16), 32, 32),
                                        ((15, 15, 3, 16), 32, 32), ((10, 14, 5, 18), 24, 32)])
def test_fp64_lengths_at_13_and_14_sites(case, Px, Py):
    nx, ny, nz, n = case
    desc = (nx, ny, nz, 1.0, 0.3, 0.1, 0.03, n)
    path = W.random_spins((n, nx * ny * nz, 3), seed=n)
    with binding.StringMethod([desc], precision=binding.SS_PREC_FP64) as sm:
        cfg = sm.launch_config(0)
        sm.set_path(0, path)
        field, energies = sm.field(0), sm.energies(0)
    assert (cfg["Px"], cfg["Py"]) == (Px, Py)
    m = oracle.model(*desc[:7])
    want = oracle.energies(m, path)
    assert np.abs(energies - want).max() <= 1e-11 * (np.abs(want).max() + nx * ny * nz)
    for k in (0, n - 1):
        ref = oracle.field(m, path[k])
        assert np.abs(field[k] - ref).max() <= 1e-12 * np.abs(ref).max(), k


# FP32 over the runtime-plan y/z kernel.  17 or 18 sites along x: 48 points until that kernel needs more rounds for them
@pytest.mark.parametrize("case,Px", [((18, 12, 2, 40), 48), ((18, 12, 2, 64), 36), ((17, 5, 1, 130), 36), ((17, 9, 9, 6), 48),
                                     ((18, 9, 9, 16), 36), ((17, 20, 12, 17), 48), ((17, 20, 12, 16), 36), ((18, 40, 10, 17), 36),
                                     ((18, 13, 8, 64), 48),
                                     # strips: 324 (162) points instead of 384 (192) where the x kernels save too little
                                     ((162, 3, 1, 40), 324), ((162, 3, 1, 16), 384), ((162, 12, 4, 40), 384), ((81, 2, 1, 60), 162),
                                     ((81, 2, 1, 30), 192)])
def test_fp32_x_length_over_the_runtime_plan_kernel(case, Px):
    nx, ny, nz, n = case
    desc = (nx, ny, nz, 1.0, 0.3, 0.1, 0.03, n)
    path = W.random_spins((n, nx * ny * nz, 3), seed=n).astype(np.float32)
    with binding.StringMethod([desc]) as sm:
        cfg = sm.launch_config(0)
        sm.set_path(0, path)
        s = sm.get_path(0)
        field, energies = sm.field(0, dtype=np.float32), sm.energies(0)
    assert cfg["Px"] == Px
    s = s / np.linalg.norm(s, axis=-1, keepdims=True)
    m = oracle.model(*desc[:7])
    want = oracle.energies(m, s)
    assert np.abs(energies - want).max() <= 1e-11 * (np.abs(want).max() + nx * ny * nz)
    for k in (0, n - 1):
        ref = oracle.field(m, s[k])
        assert np.abs(field[k] - ref).max() <= 1e-5 * np.abs(ref).max(), k


# FP64 on small grids at lengths both y/z kernels have: 64 to 256 threads of the two-pass one, 384 of the runtime plan's.
# Energies come from the spectrum with either, whose tensor carries the two-pass kernel's factor or not.
@pytest.mark.parametrize("case,two_pass", [((15, 15, 2, 16), False), ((15, 15, 2, 18), True), ((8, 29, 2, 3), False),
                                           ((24, 16, 3, 8), False), ((24, 16, 3, 10), True), ((4, 46, 3, 7), False),
                                           ((16, 15, 4, 12), False), ((16, 15, 4, 14), True), ((16, 24, 4, 4), True),
                                           ((12, 16, 5, 16), False), ((12, 16, 5, 18), True), ((12, 24, 1, 4), True),
                                           ((12, 16, 6, 4), True), ((8, 16, 8, 3), True)])
def test_fp64_yz_kernel_of_small_grids(case, two_pass):
    nx, ny, nz, n = case
    desc = (nx, ny, nz, 1.0, 0.3, 0.1, 0.3, n)
    path = W.random_spins((n, nx * ny * nz, 3), seed=ny + nz)
    with binding.StringMethod([desc], precision=binding.SS_PREC_FP64) as sm:
        cfg = sm.launch_config(0)
        sm.set_path(0, path)
        field, energies, terms = sm.field(0), sm.energies(0), sm.energy_terms(0)
    assert (cfg["threads_yz"] != 384) == two_pass
    m = oracle.model(*desc[:7])
    want = oracle.energies(m, path)
    scale = np.abs(want).max() + nx * ny * nz
    assert np.abs(energies - want).max() <= 1e-11 * scale
    assert np.abs(terms @ np.array(desc[3:7]) - want).max() <= 1e-11 * scale
    for k in (0, n - 1):
        ref = oracle.field(m, path[k])
        assert np.abs(field[k] - ref).max() <= 1e-12 * np.abs(ref).max(), k


# An FP32 context's FP64 energies over the runtime-plan y/z kernel take an x length of their own
@pytest.mark.parametrize("case", [(26, 30, 9, 3), (14, 5, 1, 4), (41, 12, 3, 2), (17, 4, 10, 5), (26, 14, 2, 3)])
def test_energies_and_barrier_of_an_fp32_context(case):
    nx, ny, nz, n = case
    desc = (nx, ny, nz, 1.0, 0.3, 0.1, 0.3, n)
    path = W.random_spins((n, nx * ny * nz, 3), seed=nx + nz).astype(np.float32)
    with binding.StringMethod([desc]) as sm:
        sm.set_path(0, path)
        s = sm.get_path(0)
        energies, terms, (barrier, k) = sm.energies(0), sm.energy_terms(0), sm.barrier(0)
    s = s / np.linalg.norm(s, axis=-1, keepdims=True)
    want = oracle.energies(oracle.model(*desc[:7]), s)
    scale = np.abs(want).max() + nx * ny * nz
    assert np.abs(energies - want).max() <= 1e-11 * scale
    assert np.abs(terms @ np.array(desc[3:7]) - want).max() <= 1e-11 * scale
    assert k == int(np.argmax(want)) and abs(barrier - (want.max() - want[0])) <= 2e-11 * scale
