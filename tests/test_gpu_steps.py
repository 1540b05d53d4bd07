"""The device step loop (gradient, trial and control kernels) at the sizes
where its work planning changes: batches wider than one planning pass, and
every number of step sizes per trial pass."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def reg():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1712_02533_gb300 import _build
    _build.build()
    import paper_1712_02533_gb300 as r
    return r


@pytest.mark.parametrize("n_ops", [1, 2, 511, 512, 513, 1100])
def test_operators_of_a_wide_batch_are_those_run_alone(reg, syn, n_ops):
    """Operators of one batch are independent: whatever the batch's width, each
    result, status and iteration count is bit for bit that of the operator run
    alone (the tile records and their FP64 sums do not depend on the batch)."""
    n_fr = min(n_ops + 1, 12)
    fr = syn.series(11, n_fr, 32, spacing=8.0, sigma=1.5, peak=20.0)
    # n_ops pairs (i, i + 1), repeated, into as many slots: several series share the frames
    per = n_fr - 1
    m = -(-n_ops // per)
    p = reg.default_params(n_levels=2, iter_max=8, lam=10.0)
    ops = [(k // per, -1, -1, k % per, k % per, k % per + 1) for k in range(n_ops)]
    with reg.Series([fr] * m, p) as s:
        st, it = s.apply_operator_batch(ops)
        got = {k: s.get_slot(ops[k][3], series=ops[k][0])[0] for k in {0, n_ops // 2, n_ops - 1}}
    with reg.Series(fr, p) as s:
        for k, u in got.items():
            a, b = s.apply_operator_batch([(0, -1, -1, ops[k][3], ops[k][4], ops[k][5])])
            assert (a[0], b[0]) == (st[k], it[k])
            assert np.array_equal(s.get_slot(ops[k][3])[0], u)


@pytest.mark.parametrize("J", [1, 2, 3, 4, 5, 8])
def test_step_sizes_per_pass_do_not_change_the_accepted_steps(reg, orc, syn, J):
    """A stable pair (no shot noise, 64^2, 2 levels): for every number of step
    sizes per pass the field is within 1e-3 px of the oracle's, the bound of
    the other stable-series tests."""
    fr = syn.series(7, 2, 64, noise=False, drift_sd=1.0, dist_amp=0.0, spacing=10.0, sigma=2.5)
    want, _, _ = orc.register(orc.embed(fr[0]), orc.embed(fr[1]), orc.params(n_levels=2, iter_max=20, lam=10.0))
    with reg.Series(fr, reg.default_params(n_levels=2, iter_max=20, lam=10.0, trials_per_pass=J)) as s:
        s.apply_operator_batch([(0, -1, -1, 0, 0, 1)])
        got = s.get_slot(0)[0]
    assert np.abs(got - want * 64).max() <= 1e-3


@pytest.mark.parametrize("side", [32, 64, 512, 1024, 2048, 4096])
def test_smoothed_direction_is_the_tensor_product_solve(reg, syn, side):
    """One lockstep step of the smoothed flow from the identity moves by tau d,
    d = (T (x) T)^-1 (omega d_L2): against an FP64 solve of the library's own
    lumped direction d_L2, at every row-chunk size of the row pass (16, 8 and 4
    rows) and sides whose last chunk and column strip are partial.  Tolerance:
    the sweeps are contractions (|c'| < 1), so their FP32 rounding stays within
    a few ulp per element: 1e-5 of the largest component."""
    from scipy.linalg import solve_banded
    sg, L = 2.0, int(np.log2(side))
    fr = syn.series(3, 2, side, peak=10.0, spacing=12.0, sigma=2.0)
    n = side + 1
    with reg.Series(fr, reg.default_params(n_levels=1, lam=10.0, smooth=sg)) as s:
        d_l2, _ = s.eval_direction(0, 1, L, np.zeros((2, n, n), np.float32))
        s.set_lockstep(np.array([[1]]), np.array([1.0]))
        s.apply_operator_batch([(0, -1, -1, 0, 0, 1)])
        got = s.get_slot(0)[0]
    off, diag = 1.0 / 6.0 - 0.5 * sg * sg, np.full(n, 2.0 / 3.0 + sg * sg)
    diag[[0, -1]] = 1.0 / 3.0 + 0.5 * sg * sg
    ab = np.stack([np.full(n, off), diag, np.full(n, off)])
    w = np.ones(n)
    w[[0, -1]] = 0.5
    for c in range(2):
        f = w[:, None] * w[None, :] * d_l2[c].astype(np.float64)
        want = solve_banded((1, 1), ab, solve_banded((1, 1), ab, f).T).T
        assert np.abs(got[c] - want).max() <= 1e-5 * np.abs(want).max()


@pytest.mark.parametrize("side,rows", [(32, 4), (32, 8), (64, 16), (64, 32), (64, 64), (128, 32)])
@pytest.mark.parametrize("amp", [1e-3, 0.4, 1.6])
def test_trial_sums_against_fp64_energies(reg, orc, syn, side, rows, amp):
    """The trial pass's energy changes against the oracle's FP64 energies at tile
    heights from four rows to more than a tile holds, with moves from far below
    a cell (no node on the exact path) to beyond one (every node on it, full
    queues): 1e-4 relative, the bound of the trial parity test."""
    rng = np.random.default_rng(side + rows)
    fr = syn.series(9, 2, side, peak=20.0, spacing=9.0, sigma=1.8)
    L, n = int(np.log2(side)), side + 1
    u = (0.3 * rng.standard_normal((2, n, n))).astype(np.float32)
    with reg.Series(fr, reg.default_params(n_levels=1, lam=10.0)) as s:
        s.set_tile_rows(L, rows, rows)
        d, _ = s.eval_direction(0, 1, L, u)
        t0 = amp / np.abs(d).max()
        taus = [t0, 0.5 * t0, 0.25 * t0, 0.1 * t0]
        d, dE = s.eval_trials(0, 1, L, u, taus)
    g = [orc.embed(f) for f in fr]
    E = lambda v: orc.energy(g[0], g[1], v / side, 10.0)[0]
    e0 = E(u.astype(np.float64))
    for t, got in zip(taus, dE):
        want = E(u.astype(np.float64) + t * d.astype(np.float64)) - e0
        assert abs(got - want) <= 1e-4 * abs(want) + 1e-9 * abs(e0), (t, got, want)


@pytest.mark.parametrize("side,rows", [(32, 4), (64, 8), (128, 32), (128, 64), (256, 16)])
def test_narrow_and_wide_batches_take_the_same_steps(reg, syn, side, rows):
    """The gradient pass's two forms (a tile per warp in wide batches, a tile per
    block in narrow ones) add their sums in the same order: an operator run alone
    and in a batch wide enough for the other form ends on the same bits."""
    L, n = int(np.log2(side)), side + 1
    tiles = -(-n // 30) * -(-n // rows)
    width = 4 * 6 * 160 // tiles + 2  # more tiles than any grid of the narrow form takes
    fr = syn.series(13, 3, side, peak=20.0, spacing=9.0, sigma=1.8)
    p = reg.default_params(n_levels=2, iter_max=6, lam=10.0)
    m = -(-width // 2)
    ops = [(k // 2, -1, -1, k % 2, k % 2, k % 2 + 1) for k in range(2 * m)]
    with reg.Series([fr] * m, p) as s:
        s.set_tile_rows(L, rows, min(rows, 32))
        s.apply_operator_batch(ops)
        wide = [s.get_slot(e, series=m - 1)[0] for e in range(2)]
    with reg.Series(fr, p) as s:
        s.set_tile_rows(L, rows, min(rows, 32))
        s.apply_operator_batch([(0, -1, -1, e, e, e + 1) for e in range(2)])
        for e in range(2):
            assert np.array_equal(s.get_slot(e)[0], wide[e])
