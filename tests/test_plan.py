"""The tile shape and z-chunks that choose_decomposition takes on a GB300 (152 SMs, two
CTAs each), computed on the host: the grids of the GPU tests that name a shape take
it, and every plan covers its grid within the chunk limits."""
import random
import subprocess

import pytest

from paper_2009_04619_gb300 import build

PROGRAM = r"""
#include <cstdio>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include "step_config.cuh"
using namespace sgb;
int main()
{
    int kind, nb, occ;
    StepArgs a = {};
    while (scanf("%d %d %d %d %d %d", &kind, &a.Nx, &a.Ny, &a.Nz, &nb, &occ) == 6) {
        a.nb = nb;
        a.nx = a.Nx - 2 * nb, a.ny = a.Ny - 2 * nb, a.nz = a.Nz - 2 * nb;
        const StepGrid g = kind == 0 ? choose_decomposition<float>(152, occ, a)
                         : kind == 1 ? choose_decomposition<__half>(152, occ, a)
                         : kind == 2 ? choose_decomposition<__nv_bfloat16>(152, occ, a)
                         : kind == 3 ? choose_decomposition<float, true>(152, occ, a)
                         : kind == 4 ? choose_decomposition<__nv_bfloat16, true>(152, occ, a)
                                     : choose_decomposition<__half, true>(152, occ, a);
        printf("%d %d %d %d %d\n", g.square, a.tiles_x, a.tiles_y, a.zc, g.ctas);
    }
}
"""
KINDS = {"fp32": 0, "fp16": 1, "bf16": 2, "fp32_diff": 3, "bf16_diff": 4, "fp16_diff": 5}


@pytest.fixture(scope="module")
def plans(tmp_path_factory):
    """rows of (kind, Nx, Ny, Nz, nb) -> rows of (square, tiles_x, tiles_y, zc, ctas)."""
    d = tmp_path_factory.mktemp("plan")
    (d / "plan.cu").write_text(PROGRAM)
    subprocess.run([build._nvcc(), *build.ARCH, "-std=c++17", "--expt-relaxed-constexpr", "-I" + build.CSRC,
                    str(d / "plan.cu"), "-o", str(d / "plan")], check=True)

    def run(rows):
        text = "".join("%d %d %d %d %d 2\n" % (KINDS[k], *ext) for k, *ext in rows)
        out = subprocess.run([str(d / "plan")], input=text, capture_output=True, text=True, check=True).stdout
        return [tuple(map(int, line.split())) for line in out.splitlines()]
    return run


def _case(inner, nb):
    return (*(n + 2 * nb for n in inner), nb)


# grids of test_gpu_square_tiles.py, and of its rerun of the adjoint's receivers
SQUARE = [_case((121, 114, 44), 8), _case((65, 97, 120), 0), _case((128, 65, 28), 16)]
# whole shots with 16-bit wavefields against the oracle (test_gpu_precision.py)
SQUARE_16BIT = [_case((192, 192, 192), 32)]
# 134 x 38 x 48: the adjoint's receivers across the seams of 64 x 16 tiles
WIDE = [_case((126, 30, 40), 4)]


@pytest.mark.parametrize("kind", list(KINDS))
def test_grids_of_the_shape_tests(plans, kind):
    cases = SQUARE + (SQUARE_16BIT if "16" in kind else [])
    assert [p[0] for p in plans([(kind, *c) for c in cases])] == [1] * len(cases)


def test_grid_of_the_receiver_tests(plans):
    assert [p[0] for p in plans([("fp32", *c) for c in WIDE])] == [0]  # the adjoint's two kernels are planned as fp32 steps


def test_plans_cover_their_grids(plans):
    rng = random.Random(0)
    rows = []
    for _ in range(3000):
        nb = rng.choice((0, 1, 8, 16, 32))
        ext = [max(1, int(2 ** rng.uniform(0, 10))) + 2 * nb for _ in range(3)]
        rows.append((rng.choice(list(KINDS)), *ext, nb))
    shapes = set()
    for (kind, Nx, Ny, Nz, nb), (square, tx, ty, zc, ctas) in zip(rows, plans(rows)):
        bx, by = (32, 32) if square else (64, 16)
        assert (tx, ty) == (-(-Nx // bx), -(-Ny // by))
        assert 1 <= zc <= max(40, Nz // max(Nz // 4, 1) + 1)
        assert ctas == tx * ty * -(-Nz // zc)
        shapes.add((kind, square))
    assert len(shapes) == 2 * len(KINDS)
