"""The Chebyshev solves of the Schur complement against the oracle, at the sizes and spacings
where the kernels' edges lie.

A step stops at relative residual tol; the error of eta is at most cond(S_j) tol with
cond(S_j) <= 1 + Bx g^2 / (1/dt + dB) and g <= 2 sum_d (2/h_d^2) sqrt(1 + h_d^2) for |k_j| = 1.
At h = pi/2 that is below 25: with tol = 1e-13 the bound 1e-10 holds as in the other parity
tests.  At h = 0.5 (where the preconditioned iteration is taken) it is below 1400, and the
FP64 rounding of the residual is about 1e-13: tol = 1e-12 and the bound 2e-9.
"""
import numpy as np
import pytest

import oracle as O
from oracle import picard as PC
from paper_1902_09761_gb300 import apfc as A
from paper_1902_09761_gb300 import inputs

from gpu_common import H2, P, context, ensure_built, rel_l2_per_amp

pytestmark = pytest.mark.gpu

PRECISIONS = [A.APFC_FP64, A.APFC_FP32_REFINED]


@pytest.fixture(scope="module", autouse=True)
def lib():
    return ensure_built()


def _steps(shape, h, n, bound, dt=1.0, seed=81, **opts):
    kind = "hex" if len(shape) == 2 else "bcc"
    ctx, L = context(kind, shape, h, **opts)
    eta = inputs.random_amplitudes(L.J, shape, seed=seed, scale=0.15 if kind == "hex" else 0.1)
    ctx.set_amplitudes(eta)
    for _ in range(n):
        ctx.step(dt)
        eta, zeta = O.step(eta, dt, P, L, h)
        assert max(rel_l2_per_amp(ctx.get_amplitudes(), eta)) <= bound
        assert max(rel_l2_per_amp(ctx.get_zeta(), zeta)) <= bound
    st = ctx.stats()
    assert st["resid_last"] <= opts["tol"] and st["iters_last"] > 0
    ctx.close()


@pytest.mark.parametrize("prec", PRECISIONS)
@pytest.mark.parametrize("shape", [(3, 3), (3, 4), (4, 3), (5, 130), (131, 6), (16, 116), (40, 117), (33, 244), (29, 245)])
def test_grids_around_strip_and_halo_widths(prec, shape):
    # grids smaller than the halo wrap several times; 116 and 244 columns are one strip of 128
    # or 256 exactly, one more starts a second strip; odd rows take single-value copies
    _steps(shape, H2, 2, 1e-10, tol=1e-13, precision=prec)


@pytest.mark.parametrize("prec", PRECISIONS)
@pytest.mark.parametrize("rows", [1, 5, 70])
@pytest.mark.parametrize("tile", [3, 5])
def test_segment_heights(prec, rows, tile):
    _steps((70, 130), (1.4, 1.7), 2, 1e-10, tol=1e-13, precision=prec, tile_rows=rows, tile=tile)


@pytest.mark.parametrize("prec", PRECISIONS)
@pytest.mark.parametrize("m", [1, 2, 3, 4])
@pytest.mark.parametrize("shape", [(24, 30), (37, 131), (130, 115)])
def test_fine_grids_take_the_preconditioned_iteration(prec, m, shape):
    _steps(shape, (0.5, 0.5), 2, 2e-9, tol=1e-12, precision=prec, cheb_degree=m)


@pytest.mark.parametrize("dt", [0.01, 30.0])
@pytest.mark.parametrize("prec", PRECISIONS)
def test_small_and_large_time_steps(prec, dt):
    # cond(S) from 1.2 (dt 0.01) to 370 (dt 30): bound cond(S) tol
    _steps((48, 52), H2, 2, 1e-9, dt=dt, tol=1e-12, precision=prec)


def test_more_applications_than_max_iter_allows_fall_back_to_bicgstab():
    # the Chebyshev iteration needs about 45 applications of S for 1e-10, 10 iterations allow 20
    shape = (40, 44)
    eta = inputs.random_amplitudes(3, shape, seed=82, scale=0.15)
    ctx, L = context("hex", shape, H2, tol=1e-10, max_iter=10)
    ctx.set_amplitudes(eta)
    ctx.step(1.0)
    ref, _ = O.step(eta, 1.0, P, L, H2)
    assert max(rel_l2_per_amp(ctx.get_amplitudes(), ref)) <= 25e-10
    ctx.close()


def test_batch_on_a_fine_grid_equals_the_runs_alone():
    L = O.hex_lattice()
    shapes = [(40, 48), (33, 131), (64, 64)]
    o = A.apfc_default_opts(precision=A.APFC_FP32_REFINED, tol=1e-12)
    states = [inputs.random_amplitudes(3, s, seed=90 + r, scale=0.15) for r, s in enumerate(shapes)]
    h = (0.5, 0.5)
    with A.Batch(L.k, A.APFC_LATTICE_HEX2D, (P.dB, P.Bx, P.t, P.v), shapes, h, o) as b:
        for r, e in enumerate(states):
            b.set_amplitudes(r, e)
        b.step(1.0, 2)
        got = [b.get_amplitudes(r) for r in range(len(shapes))]
    for r, s in enumerate(shapes):
        ctx, _ = context("hex", s, h, precision=A.APFC_FP32_REFINED, tol=1e-12)
        ctx.set_amplitudes(states[r])
        ctx.step(1.0, 2)
        assert np.array_equal(ctx.get_amplitudes(), got[r]), s
        ctx.close()


@pytest.mark.parametrize("prec", PRECISIONS)
@pytest.mark.parametrize("shape", [(3, 3, 3), (4, 3, 5), (9, 16, 32), (5, 17, 33), (70, 31, 30), (21, 33, 67), (16, 40, 64)])
def test_3d_grids_around_tile_and_halo_widths(prec, shape):
    # tiles of 32 x 16 points: exact, one point more, one less; grids smaller than the halo of
    # two; odd rows take single-value copies.  cond(S) < 50 at h = pi/2 in 3D
    _steps(shape, (np.pi / 2,) * 3, 2, 1e-10, tol=1e-13, precision=prec)


@pytest.mark.parametrize("prec", PRECISIONS)
@pytest.mark.parametrize("shape", [(12, 8, 64), (20, 12, 40), (70, 13, 67)])
def test_3d_per_pass_bicgstab(prec, shape):
    # fused = 0 keeps the per-pass kernels (TMA-staged planes where nx % 64 == 0 and ny % 8 == 0)
    _steps(shape, (1.0, 1.3, 0.9), 2, 1e-10, dt=0.5, tol=1e-13, precision=prec, fused=0, cheb_degree=2)


@pytest.mark.parametrize("prec", PRECISIONS)
def test_3d_fine_grid_falls_back_to_bicgstab(prec):
    # at h = 0.35 a solve would need more than 100 terms; cond(S) < 9100 there
    _steps((10, 12, 16), (0.35,) * 3, 1, 2e-8, tol=1e-12, precision=prec)


def test_batch_beyond_the_chebyshev_iteration_steps_its_runs_alone():
    # tol below the noise of the Schur residual on this grid (kappa about 1100): BiCGStab
    L = O.hex_lattice()
    shapes, h = [(24, 28), (20, 33)], (0.5, 0.5)
    o = A.apfc_default_opts(precision=A.APFC_FP32_REFINED, tol=5e-13)
    states = [inputs.random_amplitudes(3, s, seed=95 + r, scale=0.15) for r, s in enumerate(shapes)]
    with A.Batch(L.k, A.APFC_LATTICE_HEX2D, (P.dB, P.Bx, P.t, P.v), shapes, h, o) as b:
        for r, e in enumerate(states):
            b.set_amplitudes(r, e)
        b.step(1.0, 2)
        for r, s in enumerate(shapes):
            ref = O.run(states[r], 1.0, 2, P, L, h)[-1]
            assert max(rel_l2_per_amp(b.get_amplitudes(r), ref)) <= 2e-9
            assert b.stats(r)["resid_last"] <= 5e-13 and b.stats(r)["steps"] == 2


@pytest.mark.parametrize("shape", [(56, 40), (57, 41), (55, 39), (112, 121), (23, 200), (7, 43), (331, 402)])
def test_tiles_around_their_widths(shape):
    # tiles own 40 columns of 56 rows and reach 12 further on each side: exact, one more, one less,
    # grids that the reach wraps around, several tiles a block; odd rows take single-value copies
    _steps(shape, H2, 2, 1e-10, tol=1e-13, precision=A.APFC_FP32_REFINED)


@pytest.mark.parametrize("shape", [(3, 4), (40, 117), (131, 6), (16, 116)])
def test_narrow_strips_on_small_grids(shape):
    # variant 3 takes the tiles on these, variant 0 keeps the strips of 128 columns
    _steps(shape, H2, 2, 1e-10, tol=1e-13, precision=A.APFC_FP32_REFINED, tile=0)


def test_batch_of_tiled_and_streamed_runs_equals_the_runs_alone():
    # 680 x 690 has 18 x 13 x 3 = 702 tiles (tiled), 700 x 730 has 19 x 13 x 3 = 741 (streamed)
    L = O.hex_lattice()
    shapes = [(680, 690), (40, 48), (700, 730), (33, 131)]
    o = A.apfc_default_opts(precision=A.APFC_FP32_REFINED, tol=1e-12, tile_rows=64)
    states = [inputs.random_amplitudes(3, s, seed=95 + r, scale=0.15) for r, s in enumerate(shapes)]
    with A.Batch(L.k, A.APFC_LATTICE_HEX2D, (P.dB, P.Bx, P.t, P.v), shapes, H2, o) as b:
        for r, e in enumerate(states):
            b.set_amplitudes(r, e)
        b.step(1.0, 2)
        got = [b.get_amplitudes(r) for r in range(len(shapes))]
    for r, s in enumerate(shapes):
        ctx, _ = context("hex", s, H2, precision=A.APFC_FP32_REFINED, tol=1e-12, tile_rows=64)
        ctx.set_amplitudes(states[r])
        ctx.step(1.0, 2)
        assert np.array_equal(ctx.get_amplitudes(), got[r]), s
        ctx.close()


@pytest.mark.parametrize("prec", PRECISIONS)
@pytest.mark.parametrize("shape,h", [((61, 93), H2), ((130, 41), H2), ((37, 45), (0.5, 0.5))])
def test_picard_with_the_jacobian_across_tiles(prec, shape, h):
    # d(x) >= 0 for hexagonal amplitudes and below 0.5 here: cond(S + d) is no larger than cond(S) as
    # in the bounds above.  h = 0.5 is beyond the plain iteration and keeps BiCGStab
    kind = "hex"
    ctx, L = context(kind, shape, h, precision=prec, tol=1e-12, picard_iters=2, jacobian=1)
    eta = inputs.random_amplitudes(3, shape, seed=97, scale=0.1)
    ctx.set_amplitudes(eta)
    ctx.step(1.0)
    ref, _ = PC.step_picard(eta, 1.0, P, L, h, 2, jacobian=True)
    assert max(rel_l2_per_amp(ctx.get_amplitudes(), ref)) <= 2e-9
    ctx.close()


@pytest.mark.parametrize("kind,shape", [("hex", (7, 33)), ("hex", (8, 32)), ("hex", (9, 31)), ("hex", (353, 997)),
                                        ("hex", (352, 992)), ("bcc", (3, 5, 33)), ("bcc", (60, 33, 31))])
def test_zeta_of_new_amplitudes_around_block_edges(kind, shape):
    # blocks of 32 x 8 points, of 32 x 32 from 304 blocks on.  Seven products of FP32 pairs, each
    # good to about 2^-44 of the largest term: below 1e-12 relative
    h = H2 if kind == "hex" else (np.pi / 2,) * 3
    ctx, L = context(kind, shape, h, precision=A.APFC_FP32_REFINED)
    eta = inputs.random_amplitudes(L.J, shape, seed=98, scale=0.1)
    ctx.set_amplitudes(eta)
    ref = np.stack([O.apply_G(eta[j], L.k[j], h) for j in range(L.J)])
    assert max(rel_l2_per_amp(ctx.get_zeta(), ref)) <= 1e-12
    ctx.close()


@pytest.mark.parametrize("opts", [dict(tile=0), dict(tile=5), dict(tile=0, tile_rows=9), dict(tile=0, tile_rows=1)])
@pytest.mark.parametrize("shape", [(61, 233), (40, 464)])
def test_streamed_passes_repeat_bit_for_bit(shape, opts):
    # the streamed passes (strips of 128 and 256 columns) fetch their first rows into shared memory
    # that the block has just cleared: many blocks, the same bits from every one of them each time
    ctx, L = context("hex", shape, H2, precision=A.APFC_FP32_REFINED, tol=1e-12, **opts)
    eta = inputs.random_amplitudes(3, shape, seed=99, scale=0.15)
    first = None
    for _ in range(20):
        ctx.set_amplitudes(eta)
        ctx.step(1.0, 2)
        got = ctx.get_amplitudes()
        first = got if first is None else first
        assert np.array_equal(got, first)
    ctx.close()


def test_solves_queued_ahead_do_not_change_a_converged_state():
    # Near the steady state a step's initial residual, formed pointwise from the last step's, may meet a
    # tolerance that the stencil residual of the same state misses: the two differ by about 1e-5 of
    # themselves.  An adjoint solve before a step lets the step's refinement queue solves ahead; they
    # must leave such a state alone.  Tolerances between the two residuals are found by stepping.
    shape = (24, 26)
    phi = O.uniform_solid_hex(P)
    rng = np.random.default_rng(100)
    eta0 = phi * (1.0 + 1e-9 * (rng.standard_normal((3,) + shape) + 1j * rng.standard_normal((3,) + shape)))
    lam = inputs.random_amplitudes(3, shape, seed=101, scale=0.1)

    def make(tol, **kw):
        return context("hex", shape, H2, precision=A.APFC_FP32_REFINED, tol=tol, **kw)[0]

    def stencil(eta, tol):
        with make(tol, max_refine=0) as c:
            c.set_amplitudes(eta)
            assert c.try_step(1.0) in (A.APFC_OK, A.APFC_ENOCONV)
            return c.stats()["resid_last"]

    def pointwise_ends(tol, steps=30):
        # (step, pointwise residual, stencil residual) of the steps that end at the first check
        out, solved = [], False
        with make(tol) as c:
            c.set_amplitudes(eta0)
            for n in range(steps):
                eta = c.get_amplitudes()
                c.step(1.0)
                st = c.stats()
                if st["refine_last"] == 0 and solved:
                    out.append((n, st["resid_last"], stencil(eta, tol)))
                solved = st["refine_last"] > 0
        return out

    met, tried = 0, 0
    todo = list(np.geomspace(5e-13, 5e-12, 60))
    while todo and met < 3 and tried < 400:
        tol, tried = todo.pop(0), tried + 1
        for n, p, s in pointwise_ends(tol):
            if not p <= tol < s:
                if p < s:
                    todo.append(0.5 * (p + s))
                continue
            with make(tol) as plain, make(tol) as ahead:
                plain.set_amplitudes(eta0)
                ahead.set_amplitudes(eta0)
                for _ in range(n + 1):
                    plain.step(1.0)
                    ahead.adjoint_step(1.0, eta0, eta0, lam)
                    ahead.step(1.0)
                assert np.array_equal(plain.get_amplitudes(), ahead.get_amplitudes()), (n, tol)
                assert np.array_equal(plain.get_zeta(), ahead.get_zeta()), (n, tol)
                assert plain.stats()["resid_last"] == ahead.stats()["resid_last"] == p
            met += 1
    assert met > 0, tried


def _preconditioned_bounds(k, h, dt, m, n=1024):
    # least and greatest value of the symbol of S p(D)^2 over n^2 wave numbers
    kap = float(k @ k)
    a, kt, q = 1.0 / dt + kap * P.dB, kap * P.Bx, 2.0 * np.pi * np.arange(n) / n
    sD, mu, kmax = np.sqrt(a), np.sqrt(kt), sum(4.0 / x**2 for x in h)
    K = sum(np.expand_dims(4.0 * np.sin(q / 2) ** 2 / h[d] ** 2, 1 - d) for d in range(2))
    G = -K - sum(np.expand_dims(2.0 * k[d] / h[d] * np.sin(q), 1 - d) for d in range(2))
    theta, delta = sD + 0.5 * mu * kmax, 0.5 * mu * kmax
    cheb = np.polynomial.Chebyshev.basis(m + 1)
    p = (1.0 - cheb((theta - sD - mu * K) / delta) / cheb(theta / delta)) / (sD + mu * K)
    s = (a + kt * G**2) * p**2
    return s.min(), s.max()


@pytest.mark.parametrize("h,dt,m", [(0.49, 20.0, 3), (0.475, 10.0, 3), (0.363, 10.0, 4), (0.5, 20.0, 2), (0.45, 10.0, 1)])
def test_fine_grids_with_long_steps_take_the_one_solve_planned(h, dt, m):
    # An FP64 solve is planned to end below 0.4 of the tolerance: with the spectrum's true bounds
    # (allowing 3% on their ratio) about acosh(1 / reduction) / rate terms, two to an iteration, do.
    # A bound inside the spectrum leaves modes that shrink too slowly, and further solves.
    shape, tol = (96, 100), 1e-10
    ctx, L = context("hex", shape, (h, h), precision=A.APFC_FP64, tol=tol, cheb_degree=m)
    eta = inputs.random_amplitudes(3, shape, seed=102, scale=0.15)
    b = O.rhs(eta, dt, P, L)
    most = 0.0
    for j in range(3):
        lo, hi = _preconditioned_bounds(L.k[j], (h, h), dt, m)
        r = b[j] - np.fft.ifft2(O.schur_symbol(L.k[j], dt, P, shape, (h, h)) * np.fft.fft2(eta[j]))
        reduction = 0.4 * tol * np.linalg.norm(b[j]) / np.linalg.norm(r)
        rate = np.arccosh((1.03 * hi + lo) / (1.03 * hi - lo))
        most = max(most, np.arccosh(1.0 / reduction) / rate)
    ctx.set_amplitudes(eta)
    ctx.step(dt)
    assert ctx.stats()["iters_last"] <= most / 2 + 2
    # a right-hand side with a residual spread over every mode
    lam = inputs.random_amplitudes(3, shape, seed=103, scale=0.1)
    ctx.adjoint_step(dt, eta, eta, lam)
    ctx.close()


@pytest.mark.parametrize("scale", [0.1, 1e-25])
@pytest.mark.parametrize("prec", PRECISIONS)
def test_3d_zeta_of_new_amplitudes_in_fp64(prec, scale):
    # 26 roundings of 2^-53 each (white amplitudes: the sum is as large as its terms), twice in the
    # gradient; amplitudes of any size (FP32 pairs take those below 2^-74 for zero)
    shape, h = (9, 16, 37), (np.pi / 2, 1.3, 1.1)
    ctx, L = context("bcc", shape, h, precision=prec)
    eta = inputs.random_amplitudes(6, shape, seed=104, scale=scale)
    ctx.set_amplitudes(eta)
    ref = np.stack([O.apply_G(eta[j], L.k[j], h) for j in range(6)])
    assert max(rel_l2_per_amp(ctx.get_zeta(), ref)) <= 3e-15
    ref = 2.0 * np.prod(h) * O.energy_gradient(eta, P, L, h)
    assert max(rel_l2_per_amp(ctx.energy_gradient(eta)[0], ref)) <= 6e-15
    ctx.close()


@pytest.mark.parametrize("prec", PRECISIONS)
@pytest.mark.parametrize("kind,shape", [("bcc", (11000, 3, 4)), ("hex", (530000, 3))])
def test_boxes_longer_than_a_grid_dimension(kind, shape, prec):
    # 6 x 11000 planes and 530000 / 8 rows of tiles: more than 65535
    h = (np.pi / 2,) * len(shape)
    _steps(shape, h, 1, 1e-10, tol=1e-13, precision=prec)


@pytest.mark.parametrize("kind,shape", [("hex", (128, 128)), ("hex", (190, 251)), ("bcc", (24, 30, 33))])
def test_refined_steps_end_well_below_the_tolerance(kind, shape):
    # The solve that can meet the tolerance aims at 1/16 of it, or at 0.03 tol_inner of its own
    # residual where that is more: at most 0.15 of the tolerance.  One that cannot is aimed to leave
    # at least five times the tolerance, so that none ends just beneath it.
    h, tol = (np.pi / 2,) * len(shape), 1e-10
    ctx, L = context(kind, shape, h, precision=A.APFC_FP32_REFINED, tol=tol)
    phi = O.uniform_solid_hex(P) if kind == "hex" else O.uniform_solid_bcc(P)
    for seed in range(4):
        ctx.set_amplitudes(inputs.single_grain(L.k, phi, shape, h, 0.3 * min(shape) * h[0], 5.0 + seed, seed=105 + seed, noise=1e-3))
        for _ in range(5):
            ctx.step(1.0)
            assert ctx.stats()["resid_last"] <= 0.2 * tol
    ctx.close()


@pytest.mark.parametrize("shape", [(9, 11, 59), (8, 12, 60), (9, 13, 61), (10, 27, 61), (9, 28, 60), (8, 29, 59), (97, 56, 361)])
def test_3d_boxes_around_the_tiles_of_the_passes(shape):
    # the FP32 passes own 60 columns of 12 rows, or of 28 where that gives two rounds of blocks (the
    # last box: 7 x 2 tiles x 4 chunks x 6 amplitudes, one column over, odd rows); the residual 28 x 28
    _steps(shape, (np.pi / 2,) * 3, 2, 1e-10, tol=1e-13, precision=A.APFC_FP32_REFINED)
