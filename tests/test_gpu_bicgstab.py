"""BiCGStab on the block system, which serves where the Chebyshev iteration on its Schur
complement does not: here a tolerance beneath the noise of that iteration's residual.

At h = 0.5, dt = 1 cond(S) is between 1100 and 1400, and a tolerance of 5e-13 lies below 9e-16
cond(S), from which on the Chebyshev iteration is taken.  A step then errs by at most cond(S) tol =
7e-10, two by about twice that: the bound 2e-9 of the other tests on this grid.  Every test asserts
that the fused t-kernel, which the Chebyshev iteration has not, has run.
"""
import numpy as np
import pytest

import oracle as O
from oracle import picard as PC
from paper_1902_09761_gb300 import apfc as A
from paper_1902_09761_gb300 import inputs

from gpu_common import P, context, ensure_built, rel_l2_per_amp

pytestmark = pytest.mark.gpu

H, TOL, BOUND = (0.5, 0.5), 5e-13, 2e-9


@pytest.fixture(scope="module", autouse=True)
def lib():
    return ensure_built()


def _steps(shape, n=2, seed=111, **opts):
    ctx, L = context("hex", shape, H, tol=TOL, **opts)
    eta = inputs.random_amplitudes(3, shape, seed=seed, scale=0.1)
    ctx.set_amplitudes(eta)
    kernel = "fused_apinv_t" + ("_f32" if opts["precision"] == A.APFC_FP32_REFINED else "_f64")
    ctx.profile_start(kernel)
    for _ in range(n):
        ctx.step(1.0)
        if opts.get("jacobian"):
            eta, _ = PC.step_picard(eta, 1.0, P, L, H, opts["picard_iters"], jacobian=True)
        else:
            eta, zeta = O.step(eta, 1.0, P, L, H)
            assert max(rel_l2_per_amp(ctx.get_zeta(), zeta)) <= BOUND
        assert max(rel_l2_per_amp(ctx.get_amplitudes(), eta)) <= BOUND
    launches = ctx.profile_read(kernel)["launches"]
    ctx.profile_stop()
    assert launches > 0
    ctx.close()


@pytest.mark.parametrize("tile", [0, 1, 2, 3, 4, 5])
@pytest.mark.parametrize("rows", [32, 128, 179])
def test_tile_variants(tile, rows):
    # 530 columns span 3 to 5 strips, 300 rows 2 to 10 segments
    _steps((300, 530), precision=A.APFC_FP32_REFINED, tile=tile, tile_rows=rows, tile_t=-1)


@pytest.mark.parametrize("tile_t", [0, 1, 2, 4, 5])
def test_t_kernel_variants(tile_t):
    # the t-kernel's partial sums follow its own variant's block grid
    _steps((300, 530), precision=A.APFC_FP32_REFINED, tile=3, tile_t=tile_t)


@pytest.mark.parametrize("m", [2, 3, 4])
def test_degrees(m):
    _steps((130, 270), precision=A.APFC_FP32_REFINED, cheb_degree=m, tile_rows=48)


@pytest.mark.parametrize("m", [1, 2, 3, 4])
def test_fp64_over_several_strips(m):
    _steps((130, 530), n=1, precision=A.APFC_FP64, cheb_degree=m, tile_rows=48)


@pytest.mark.parametrize("prec", [A.APFC_FP64, A.APFC_FP32_REFINED])
@pytest.mark.parametrize("tile", [0, 3])
def test_jacobian_over_several_strips(prec, tile):
    # d(x) >= 0 on the triangular lattice: cond(S + d) is no larger than cond(S)
    _steps((40, 270), n=1, precision=prec, tile=tile, tile_rows=16, tile_t=-1, picard_iters=2, jacobian=1)
