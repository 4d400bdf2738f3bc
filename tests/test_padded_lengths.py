"""The padded lengths of every accepted lattice (no GPU): the rules of csrc/ss_internal.h compiled for the host.

A length must hold the linear convolution (P >= 2n - 1), and a kernel of the runtime plans, whose stages are of
radix 2, 3, 4 and 8, must never be handed a length with another prime factor: the y/z kernel is the two-pass one
only where yz2p_ok takes the pair (Py, Px) and the layer count, the x kernels where t2_length takes Px.
"""
import os
import shutil
import subprocess

import pytest

from paper_1804_07135_gb300 import build as B

SOURCE = r"""
#include <cstdio>
#include <vector>
#include "ss_internal.h"
using namespace ss;
static bool smooth(int m) {
    while (m % 2 == 0) m /= 2;
    while (m % 3 == 0) m /= 3;
    return m == 1;
}
int main() {
    printf("lengths");
    for (int P = 1; P <= 4096; ++P)
        if (t2_length(P)) printf(" %d", P);
    printf("\n");
    long bad = 0, seen = 0;
    for (int nz : {1, 2, 4, 8, 9})
        for (int real : {4, 8})
            for (int pairs : {1, 13, 200}) {
                if (real == 4 && pairs != 13) continue;
                for (int nx = 1; nx <= 1024; ++nx)
                    for (int ny = 1; ny <= 1024; ++ny) {
                        int Px = 0, Py = 0;
                        padded_lengths(real, nx, ny, nz, pairs, &Px, &Py);
                        ++seen;
                        const bool ok = Px >= 2 * nx - 1 && Py >= 2 * ny - 1 && (t2_length(Px) || smooth(Px)) &&
                                        (yz2p_ok(Py, nz, Px) || smooth(Py));
                        if (!ok && bad++ < 5) printf("bad %d %d %d real %d pairs %d: %d %d\n", nx, ny, nz, real, pairs, Px, Py);
                    }
            }
    printf("shapes %d %d %d %d %d\n", x_shape_ok(true, 192, 4, 64), x_shape_ok(true, 384, 8, 64), x_shape_ok(false, 192, 4, 64),
           x_shape_ok(false, 256, 4, 64), x_shape_ok(true, 192, 4, 3));
    printf("seen %ld bad %ld\n", seen, bad);
}
"""


@pytest.fixture(scope="module")
def output(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("lengths")
    (d / "lengths.cpp").write_text(SOURCE)
    include = os.path.join(os.path.dirname(os.path.dirname(B.nvcc())), "include")
    subprocess.run([cxx, "-std=c++17", "-O2", "-I", B.CSRC, "-I", include, "-o", str(d / "lengths"), str(d / "lengths.cpp")],
                   check=True)
    return subprocess.run([str(d / "lengths")], check=True, capture_output=True, text=True).stdout.splitlines()


def test_no_length_reaches_a_kernel_that_cannot_transform_it(output):
    assert output[-1].startswith("seen ") and output[-1].endswith(" bad 0"), output


def test_the_build_compiles_every_two_pass_length(output):
    assert [int(v) for v in output[0].split()[1:]] == sorted(B.T2_LENGTHS)


def test_pinned_x_shapes(output):
    # the two-pass kernels of 128 points took any block size before they had one shape, and still do
    assert output[-2] == "shapes 1 1 0 1 0"
