"""GPU parity: the CUDA path (through the C ABI) against the FP64 oracle.

Tolerances (step and proxy, from the condition of the sum g_j = (1/n) sum_i
X_ij u_i): with S_j = (1/n) sum_i |X_ij u_i| and sd_j = |delta_j| + S_j/beta_j,
  |delta_gpu - delta_cpu| <= tol * sd_j,
  |phi_gpu - phi_cpu|     <= tol * sd_j * (S_j + beta_j sd_j + lambda),
tol = 1e-12 in FP64 mode and 1e-5 in FP32 mode.  Integer results (colours,
permutations, supports) are compared exactly.
"""

import numpy as np
import pytest

import oracle
import workloads
from parity_tools import (TOL, _scales, _state, _u, assert_steps_close, assert_support_matches,  # noqa: F401
                          certified_optimum)

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gb():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1206_6409_gb300 import build

    build.build()
    from paper_1206_6409_gb300 import binding

    binding.lib()
    return binding


def ragged_problem(loss="logistic", seed=0):
    """Column lengths at the kernel's edges (0, 1, 31..33, tile sizes, 4096,
    50,000), empty rows, a ragged tail."""
    rng = np.random.default_rng(seed)
    n = 60_000
    lengths = [0, 1, 2, 3, 31, 32, 33, 0, 0, 127, 128, 129, 255, 256, 257, 4096, 50_000, 5, 0, 1000,
               7, 1, 0]
    lengths += list(rng.integers(0, 40, size=300))
    lengths += [1, 0, 0, 3]
    counts = np.array(lengths, np.int64)
    col_ptr = np.zeros(counts.size + 1, np.int64)
    np.cumsum(counts, out=col_ptr[1:])
    rows = workloads.synthetic._distinct_rows(n - 100, counts, rng)  # the last 100 rows stay empty
    val = rng.lognormal(0.0, 1.0, rows.size) * np.where(rng.random(rows.size) < 0.3, -1.0, 1.0)
    y = np.where(rng.random(n) < 0.5, -1.0, 1.0) if loss == "logistic" else rng.normal(size=n)
    return workloads.Problem(n, counts.size, col_ptr, rows, val, y, loss, np.zeros(counts.size), "ragged")


PROBLEMS = {
    "cfg1-logistic": lambda: workloads.config1("logistic"),
    "cfg1-squared": lambda: workloads.config1("squared"),
    "ragged-logistic": lambda: ragged_problem("logistic"),
    "ragged-squared": lambda: ragged_problem("squared", 1),
    "zipf-logistic": lambda: workloads.config2_scaled(0.002, "logistic"),
    # several row slabs, heavy and light columns
    "zipf-slabs-squared": lambda: workloads.zipf_problem(120_000, 20_000, 400_000, cap=20_000, n_planted=10,
                                                         loss="squared", seed=5),
}


@pytest.mark.parametrize("precision", ["f64", "f32"])
@pytest.mark.parametrize("name", list(PROBLEMS))
def test_propose_matches_oracle(gb, name, precision):
    prob = PROBLEMS[name]()
    orc = oracle.Oracle(prob)
    lam = 0.05 * orc.lambda_max()
    orc.set_lambda(lam)
    w = _state(prob, 1)
    z = orc.fitted(w)
    rng = np.random.default_rng(2)
    J = np.concatenate([np.arange(prob.k), rng.integers(0, prob.k, 500)]).astype(np.int32)
    d_cpu, f_cpu = orc.propose(w, z, J)
    with gb.Problem(prob, precision=precision) as p:
        p.set_lambda(lam)
        p.set_w(w)
        d_gpu, f_gpu = p.propose_at(J)
        assert_steps_close(prob, z, w, lam, J, d_gpu, f_gpu, d_cpu, f_cpu, TOL[precision])
        # the streaming pass over all columns (Thread-Greedy's Propose)
        d_all, f_all, kkt = p.propose_all()
        Jall = np.arange(prob.k)
        assert_steps_close(prob, z, w, lam, Jall, d_all, f_all, d_cpu[:prob.k], f_cpu[:prob.k],
                           TOL[precision])
        S, _ = _scales(prob, z, lam)
        assert abs(kkt - orc.kkt(w, z)) <= TOL[precision] * (S.max() + lam) * 10


@pytest.mark.parametrize("precision", ["f64", "f32"])
def test_lambda_max_and_objective(gb, precision):
    for loss in ("logistic", "squared"):
        prob = workloads.config1(loss)
        orc = oracle.Oracle(prob)
        with gb.Problem(prob, precision=precision) as p:
            lm = p.lambda_max()
            assert lm == pytest.approx(orc.lambda_max(), rel=TOL[precision] * 10)
            lam = 0.02 * orc.lambda_max()
            orc.set_lambda(lam)
            p.set_lambda(lam)
            w = _state(prob, 5)
            p.set_w(w)
            obj, kkt = p.objective()
            assert obj == pytest.approx(orc.objective(w), rel=1e-13 if precision == "f64" else 1e-6)
            np.testing.assert_allclose(p.z(), orc.fitted(w), rtol=0,
                                       atol=1e-12 if precision == "f64" else 1e-5)


@pytest.mark.parametrize("m", [2, 3, 31, 375, 4999, 16_383, 16_384, 16_385])
def test_permutation_of_small_ranges_is_bit_exact(gb, m):
    # by rank up to 16,384 entries, by the radix sort beyond
    with gb.Problem(workloads.config1("logistic")) as p:
        np.testing.assert_array_equal(p.permutation(5, 2, m), oracle.permutation(5, 2, m))


def test_permutation_is_bit_exact(gb):
    prob = workloads.config1("logistic")
    with gb.Problem(prob) as p:
        for seed, epoch, m in [(0, 0, 1), (0, 0, 4096), (7, 3, 4097), (2**64 - 1, 11, 100_003),
                               (123, 0, 1_000_000)]:
            np.testing.assert_array_equal(p.permutation(seed, epoch, m), oracle.permutation(seed, epoch, m))


@pytest.mark.parametrize("name", ["cfg1-logistic", "ragged-squared", "zipf-logistic"])
def test_coloring_equals_first_fit(gb, name):
    prob = PROBLEMS[name]()
    colors_cpu, nc_cpu = oracle.Oracle(prob).color()
    with gb.Problem(prob) as p:
        assert p.color() == nc_cpu
        np.testing.assert_array_equal(p.colors(), colors_cpu)


@pytest.mark.parametrize("precision", ["f64"])
@pytest.mark.parametrize("loss", ["logistic", "squared"])
def test_coloring_iterations_match(gb, loss, precision):
    prob = workloads.config1(loss)
    orc = oracle.Oracle(prob)
    lam = 0.05 * orc.lambda_max()
    orc.set_lambda(lam)
    colors, C = orc.color()
    iters = C + C // 2  # crosses an epoch boundary
    w_cpu, z_cpu, _, _ = orc.run("coloring", iters, colors=colors, seed=9)
    with gb.Problem(prob, precision=precision) as p:
        p.set_lambda(lam)
        p.set_colors(colors)
        p.set_params(variant="coloring", seed=9)
        p.iterate(iters)
        w_gpu = p.w()
    np.testing.assert_array_equal(w_gpu != 0, w_cpu != 0)
    np.testing.assert_allclose(w_gpu, w_cpu, rtol=0, atol=1e-10)


@pytest.mark.parametrize("variant,B,P", [("thread_greedy", 64, 0), ("thread_greedy", 5000, 0),
                                          ("greedy", 1, 0), ("shotgun", 0, 200)])
def test_iterations_match(gb, variant, B, P):
    prob = workloads.config1("logistic")
    orc = oracle.Oracle(prob)
    lam = 0.05 * orc.lambda_max()
    orc.set_lambda(lam)
    iters = 40
    w_cpu, z_cpu, _, _ = orc.run(variant, iters, B=B or 1, P=P or 1, seed=4)
    with gb.Problem(prob) as p:
        p.set_lambda(lam)
        p.set_params(variant=variant, blocks=B, P=P, seed=4)
        r = p.iterate(iters)
        w_gpu = p.w()
        assert r.iters == iters and np.isfinite(r.objective)
    np.testing.assert_array_equal(w_gpu != 0, w_cpu != 0)
    np.testing.assert_allclose(w_gpu, w_cpu, rtol=0, atol=1e-10)


@pytest.mark.parametrize("loss", ["logistic", "squared"])
@pytest.mark.parametrize("variant", ["shotgun", "thread_greedy", "coloring"])
def test_solve_reaches_the_oracle_optimum(gb, loss, variant):
    # B = 16 partitions: Thread-Greedy has no convergence guarantee (Section 7)
    # and the oracle itself diverges on this problem for B >= 64.
    prob = workloads.uniform_problem(1000, 2000, 10, values="pm1", loss=loss, n_planted=30, seed=21)
    orc = oracle.Oracle(prob)
    lam = 0.05 * orc.lambda_max()
    orc.set_lambda(lam)
    w_opt, _, _, kkt, _ = orc.solve("ccd", tol_kkt=1e-11)
    assert kkt <= 1e-11
    P_opt = orc.objective(w_opt)
    with gb.Problem(prob) as p:
        p.set_lambda(lam)
        p.set_params(variant=variant, tol_kkt=1e-11, max_iter=400_000, check_every=50, blocks=16)
        r = p.solve()
        assert r.status == 0, r.as_dict()
        w = p.w()
    assert r.objective == pytest.approx(P_opt, rel=1e-6)
    big = (np.abs(w_opt) > 1e-6) | (np.abs(w) > 1e-6)
    np.testing.assert_array_equal(np.sign(w[big]), np.sign(w_opt[big]))
    assert_support_matches(prob, lam, w, w_opt, label=f"{variant} {loss}")


@pytest.mark.parametrize("loss", ["logistic", "squared"])
def test_config1_shotgun_solve_matches_oracle(gb, loss):
    """Plain L1 problem of n=2,000, k=5,000 (20 nnz/column, +-1 values), FP64,
    Shotgun with P* against the oracle's cyclic-CD optimum."""
    prob = workloads.config1(loss)
    orc = oracle.Oracle(prob)
    lam = 0.01 * orc.lambda_max()
    orc.set_lambda(lam)
    if loss == "logistic":  # config 1's logistic problem is config 3's +-1 one: its stored optimum
        w_opt = certified_optimum("cfg3_pm1_logistic", prob, lam)
    else:
        w_opt, _, _, kkt, _ = orc.solve("ccd", tol_kkt=1e-11, max_iter=4 * 10**8)
    P_opt = orc.objective(w_opt)
    with gb.Problem(prob) as p:
        p.set_lambda(lam)
        rho, pstar, _ = p.spectral_radius()
        rho_cpu, _ = orc.spectral_radius()
        assert rho == pytest.approx(rho_cpu, rel=1e-6)
        p.set_params(variant="shotgun", P=0, tol_kkt=1e-10, max_iter=4_000_000, check_every=200)
        r = p.solve()
        assert r.status == 0, r.as_dict()
        w = p.w()
    assert r.objective == pytest.approx(P_opt, rel=1e-6)
    assert_support_matches(prob, lam, w, w_opt, label=f"config 1 shotgun {loss}")


def test_f32_solve_reaches_the_optimum(gb):
    prob = workloads.config2_scaled(0.002, "logistic")
    orc = oracle.Oracle(prob)
    lam = 0.05 * orc.lambda_max()
    orc.set_lambda(lam)
    w_opt, _, _, _, _ = orc.solve("ccd", tol_kkt=1e-11)
    with gb.Problem(prob, precision="f32") as p:
        p.set_lambda(lam)
        p.set_params(variant="thread_greedy", blocks=128, tol_kkt=1e-8, max_iter=100_000, check_every=50)
        r = p.solve()
        assert r.status == 0, r.as_dict()
        w = p.w()
    assert r.objective == pytest.approx(orc.objective(w_opt), rel=1e-6)
    # FP32 storage rounds X: the GPU solves the problem on the stored values,
    # whose optimum is within the fragile margin of the FP64 one
    assert_support_matches(oracle.stored_problem(prob, "f32"), lam, w, w_opt, label="f32 scaled config 2")


@pytest.mark.parametrize("variant,B", [("greedy", 1), ("thread_greedy", 7), ("thread_greedy", 1024)])
def test_f32_accepts_the_best_proxy(gb, variant, B):
    # FP32 mode ranks columns with FP32 proxies and applies the winner's FP64
    # step: each partition's accepted column has the partition's best proxy up
    # to FP32 rounding, its step is the FP64 Eq. 7 step, and nothing else moves
    prob = workloads.config2_scaled(0.01, "logistic")
    orc = oracle.Oracle(prob)
    lam = 0.05 * orc.lambda_max()
    orc.set_lambda(lam)
    w = _state(prob, 11, frac=0.05, scale=0.3)
    z = orc.fitted(w)
    with gb.Problem(prob, precision="f32") as p:
        p.set_lambda(lam)
        p.set_params(variant=variant, blocks=B)
        p.set_w(w)
        _, f_all, _ = p.propose_all()
        p.iterate(1)
        w1 = p.w()
    moved = np.flatnonzero(w1 != w)
    Bp = 1 if variant == "greedy" else B
    bounds = (np.arange(Bp + 1, dtype=np.int64) * prob.k) // Bp
    part = np.searchsorted(bounds, moved, side="right") - 1
    assert moved.size > 0 and np.unique(part).size == part.size
    J = moved.astype(np.int32)
    d_cpu, _ = orc.propose(w, z, J)
    S, bj = _scales(prob, z, lam)
    for j, b, dc in zip(moved, part, d_cpu):
        fmin = f_all[bounds[b]:bounds[b + 1]].min()
        assert f_all[j] < 0 and f_all[j] <= fmin + 1e-4 * abs(fmin)
        sd = abs(dc) + (S[j] / bj[j] if bj[j] > 0 else abs(w[j]))
        assert abs((w1[j] - w[j]) - dc) <= TOL["f32"] * sd


def test_edge_cases(gb):
    # one column, one row, all-empty columns, lambda above lambda_max
    X = np.array([[2.0]])
    p1 = workloads.csc_from_dense(X, np.array([1.0]), "logistic")
    with gb.Problem(p1) as p:
        p.set_lambda(0.01)
        p.set_params(variant="greedy", tol_kkt=1e-12, max_iter=100000, check_every=1)
        r = p.solve()
        assert r.status == 0
        o = oracle.Oracle(p1, 0.01)
        w_opt, _, _, _, _ = o.solve("ccd", tol_kkt=1e-13, max_iter=10**6)
        assert p.w()[0] == pytest.approx(w_opt[0], rel=1e-9)
    empty = workloads.Problem(5, 4, np.zeros(5, np.int64), np.zeros(0, np.int32), np.zeros(0),
                              np.array([1.0, -1, 1, 1, -1]), "logistic", np.zeros(4))
    with gb.Problem(empty) as p:
        assert p.lambda_max() == 0.0
        p.set_lambda(0.1)
        p.set_params(variant="thread_greedy")
        r = p.solve()
        assert r.status == 0 and r.iters == 0
        assert (p.w() == 0).all()
        p.set_w(np.array([1.0, 0.0, -2.0, 0.0]))  # weights on empty columns go to 0 in one step
        p.iterate(1)
        assert (p.w() == 0).all()
    prob = ragged_problem("squared", 3)
    with gb.Problem(prob) as p:
        lm = p.lambda_max()
        p.set_lambda(lm * (1 + 1e-9))
        p.set_params(variant="thread_greedy", tol_kkt=0.0, max_iter=5)
        r = p.solve()
        assert (p.w() == 0).all()


def test_invalid_input_is_rejected(gb):
    good = workloads.uniform_problem(20, 10, 3, seed=1)
    cases = []
    bad = good.row_idx.copy()
    bad[0], bad[1] = bad[1], bad[0]  # unsorted rows in column 0
    cases.append(("rows", dict(row_idx=bad)))
    bad = good.row_idx.copy()
    bad[4] = bad[3]  # duplicate row in column 1
    cases.append(("rows", dict(row_idx=bad)))
    bad = good.row_idx.copy()
    bad[7] = 20  # out of range
    cases.append(("rows", dict(row_idx=bad)))
    bad = good.col_ptr.copy()
    bad[3] = bad[5]  # not monotone
    cases.append(("col_ptr", dict(col_ptr=bad)))
    bad_y = good.y.copy()
    bad_y[2] = 0.5  # logistic labels must be +-1
    cases.append(("label", dict(y=bad_y)))
    bad_v = good.val.copy()
    bad_v[2] = np.nan
    cases.append(("value", dict(val=bad_v)))
    for _, kw in cases:
        args = dict(col_ptr=good.col_ptr, row_idx=good.row_idx, val=good.val, y=good.y)
        args.update(kw)
        with pytest.raises(gb.GencdError) as e:
            gb.gencd_create(good.n, good.k, good.nnz, args["col_ptr"], args["row_idx"], args["val"], args["y"],
                            "logistic", "f64")
        assert e.value.code == gb.GENCD_EINVAL
    with pytest.raises(gb.GencdError):
        gb.gencd_create(good.n, good.k, good.nnz + 1, good.col_ptr, good.row_idx, good.val, good.y)


def test_device_inputs_match_host_inputs(gb):
    import torch

    prob = workloads.config1("logistic")
    dev = dict(col_ptr=torch.from_numpy(prob.col_ptr).cuda(), row_idx=torch.from_numpy(prob.row_idx).cuda(),
               val=torch.from_numpy(prob.val).cuda(), y=torch.from_numpy(prob.y).cuda())
    lam = 0.05 * oracle.Oracle(prob).lambda_max()
    ws = []
    for kw in (dict(prob=prob), dict(n=prob.n, k=prob.k, loss="logistic", **dev)):
        with gb.Problem(**kw) as p:
            p.set_lambda(lam)
            p.set_params(variant="thread_greedy", blocks=100)
            p.iterate(10)
            ws.append(p.w())
    # FP64 atomics combine partial sums of columns cut by lane boundaries in
    # arrival order, so two runs agree to rounding, not bit for bit
    np.testing.assert_allclose(ws[0], ws[1], rtol=1e-13, atol=1e-15)


def test_not_converged_and_diverged_are_reported(gb):
    prob = workloads.config1("logistic")
    with gb.Problem(prob) as p:
        p.set_lambda(1e-4 * p.lambda_max())
        p.set_params(variant="thread_greedy", max_iter=5, tol_kkt=1e-14, check_every=5)
        r = p.solve()
        assert r.status == gb.GENCD_NOT_CONVERGED and r.iters == 5
    # literal beta with columns of norm^2 >> n makes every step overshoot
    X = np.array([[300.0, 0.0], [0.0, 200.0], [100.0, 100.0]])
    big = workloads.csc_from_dense(X, np.array([1.0, -2.0, 0.5]), "squared")
    with gb.Problem(big) as p:
        p.set_lambda(1e-3)
        p.set_params(variant="thread_greedy", beta_mode=1, max_iter=100000, check_every=10, tol_kkt=0.0)
        r = p.solve()
        assert r.status == gb.GENCD_EDIVERGED


@pytest.mark.parametrize("precision", ["f64", "f32"])
def test_thread_greedy_backoff_converges_where_plain_thread_greedy_diverges(gb, precision):
    # config-3 shapes, squared loss: Thread-Greedy with B = 16 diverges (the
    # FP64 oracle's too); the solve's accept backoff merges partitions until
    # the iteration converges, to the oracle's cyclic CD optimum
    prob = workloads.config3("lognormal", "squared")
    orc = oracle.Oracle(prob)
    lam = 0.05 * orc.lambda_max()
    orc.set_lambda(lam)
    w_tg, _, _, _ = orc.run("thread_greedy", 200, B=16)[:4]
    assert not orc.objective(w_tg) < orc.objective(np.zeros(prob.k))  # plain Thread-Greedy diverges
    w_opt, _, _, _, _ = orc.solve("ccd", tol_kkt=1e-11)
    with gb.Problem(prob, precision=precision) as p:
        p.set_lambda(lam)
        p.set_params(variant="thread_greedy", blocks=16, tol_kkt=1e-11 if precision == "f64" else 1e-8,
                     max_iter=400_000, check_every=10)
        r = p.solve()
        assert r.status == 0, r.as_dict()
        w = p.w()
    assert r.objective == pytest.approx(orc.objective(w_opt), rel=1e-6)
    assert orc.kkt(w) <= 1e-7
    sp = prob if precision == "f64" else oracle.stored_problem(prob, "f32")
    assert_support_matches(sp, lam, w, w_opt, label=f"backoff {precision}")


@pytest.mark.parametrize("variant,B,P", [("thread_greedy", 64, 0), ("greedy", 1, 0), ("shotgun", 0, 200)])
def test_improve_steps_match_the_oracle(gb, variant, B, P):
    # Improve delta_j (Algorithm 3, reading R11): every accepted increment
    # refined on its own coordinate before the update
    prob = workloads.config1("logistic")
    orc = oracle.Oracle(prob)
    lam = 0.05 * orc.lambda_max()
    orc.set_lambda(lam)
    iters = 15
    w_plain, _, _, _ = orc.run(variant, iters, B=B or 1, P=P or 1, seed=4)
    w_cpu, _, _, _ = orc.run(variant, iters, B=B or 1, P=P or 1, seed=4, improve_steps=500)
    assert np.abs(w_cpu - w_plain).max() > 1e-6  # the step changes the trajectory
    with gb.Problem(prob) as p:
        p.set_lambda(lam)
        p.set_params(variant=variant, blocks=B, P=P, seed=4, improve_steps=500)
        p.iterate(iters)
        w_gpu = p.w()
    np.testing.assert_array_equal(w_gpu != 0, w_cpu != 0)
    np.testing.assert_allclose(w_gpu, w_cpu, rtol=0, atol=1e-9)


@pytest.mark.parametrize("B", [17, 200])
def test_top_greedy_iterations_match(gb, B):
    # Section 7's global top-|J'| Accept (reading R12): the B lowest proxies
    prob = workloads.config1("logistic")
    orc = oracle.Oracle(prob)
    lam = 0.05 * orc.lambda_max()
    orc.set_lambda(lam)
    iters = 15
    w_cpu, _, _, st = orc.run("top_greedy", iters, B=B)
    with gb.Problem(prob) as p:
        p.set_lambda(lam)
        p.set_params(variant="top_greedy", blocks=B)
        p.stats_reset()
        p.iterate(iters)
        w_gpu = p.w()
        assert p.stats().updates == st[0]
    np.testing.assert_array_equal(w_gpu != 0, w_cpu != 0)
    np.testing.assert_allclose(w_gpu, w_cpu, rtol=0, atol=1e-10)


def test_set_loss_switches_the_problem(gb):
    # +-1 labels are valid for both losses: a problem switched to the squared
    # loss equals a problem created with it, in the same state, and back
    prob = workloads.config1("logistic")
    sq = prob.with_loss("squared", prob.y)
    w = _state(prob, 21)
    J = np.arange(prob.k, dtype=np.int32)
    with gb.Problem(prob) as p, gb.Problem(sq) as q:
        lm_logistic = p.lambda_max()
        lam = 0.05 * q.lambda_max()
        for h in (p, q):
            h.set_w(w)
            h.set_lambda(lam)
        p.set_loss("squared")
        assert p.lambda_max() == pytest.approx(q.lambda_max(), rel=1e-14)
        d1, f1 = p.propose_at(J)
        d2, f2 = q.propose_at(J)
        np.testing.assert_allclose(d1, d2, rtol=1e-12, atol=1e-300)
        np.testing.assert_allclose(f1, f2, rtol=1e-12, atol=1e-300)
        assert p.objective()[0] == pytest.approx(q.objective()[0], rel=1e-14)
        p.set_loss("logistic")
        assert p.lambda_max() == pytest.approx(lm_logistic, rel=1e-14)
        orc = oracle.Oracle(prob)
        orc.set_lambda(lam)
        assert p.objective()[0] == pytest.approx(orc.objective(w), rel=1e-13)
    # real-valued labels cannot take the logistic loss; the problem is unchanged
    lasso = workloads.config1("squared")
    with gb.Problem(lasso) as p:
        lm = p.lambda_max()
        with pytest.raises(gb.GencdError) as e:
            p.set_loss("logistic")
        assert e.value.code == gb.GENCD_EINVAL and "-1/+1" in str(e.value)
        assert p.lambda_max() == lm


# --- storage modes: bfloat16 values and index-only binary columns -----------
# The oracle runs on the values the mode stores (oracle.stored_values), so the
# comparison isolates the FP32 arithmetic: the FP32 tolerance applies.

STORAGE_CASES = {
    "cfg3-lognormal-bf16": (lambda: workloads.config3("lognormal"), "bf16"),
    "cfg3-pm1-bf16": (lambda: workloads.config3("pm1", "squared"), "bf16"),
    "ragged-bf16": (lambda: ragged_problem("logistic", 2), "bf16"),
    "zipf-slabs-bf16": (PROBLEMS["zipf-slabs-squared"], "bf16"),
    "cfg3-ones-binary": (lambda: workloads.config3("ones"), "binary"),
    "ragged-binary": (lambda: workloads.binarized(ragged_problem("squared", 3)), "binary"),
    "zipf-binary": (lambda: workloads.binarized(workloads.config2_scaled(0.002, "logistic")), "binary"),
    "zipf-slabs-binary": (lambda: workloads.binarized(PROBLEMS["zipf-slabs-squared"]()), "binary"),
}


@pytest.mark.parametrize("name", list(STORAGE_CASES))
def test_storage_modes_match_oracle(gb, name):
    make, mode = STORAGE_CASES[name]
    prob = make()
    sp = oracle.stored_problem(prob, mode)
    orc = oracle.Oracle(sp)
    lam = 0.05 * orc.lambda_max()
    orc.set_lambda(lam)
    w = _state(prob, 4)
    z = orc.fitted(w)
    rng = np.random.default_rng(6)
    J = np.concatenate([np.arange(prob.k), rng.integers(0, prob.k, 300)]).astype(np.int32)
    d_cpu, f_cpu = orc.propose(w, z, J)
    with gb.Problem(prob, precision=mode) as p:
        assert p.lambda_max() == pytest.approx(orc.lambda_max(), rel=TOL["f32"] * 10)
        p.set_lambda(lam)
        p.set_w(w)
        np.testing.assert_allclose(p.z(), z, rtol=0, atol=1e-5 * max(1.0, np.abs(z).max()))
        d_gpu, f_gpu = p.propose_at(J)
        assert_steps_close(sp, z, w, lam, J, d_gpu, f_gpu, d_cpu, f_cpu, TOL["f32"])
        d_all, f_all, kkt = p.propose_all()
        assert_steps_close(sp, z, w, lam, np.arange(prob.k), d_all, f_all, d_cpu[:prob.k], f_cpu[:prob.k],
                           TOL["f32"])
        S, _ = _scales(sp, z, lam)
        assert abs(kkt - orc.kkt(w, z)) <= TOL["f32"] * (S.max() + lam) * 10
        obj, _ = p.objective()
        assert obj == pytest.approx(orc.objective(w), rel=1e-6)


@pytest.mark.parametrize("mode,values", [("bf16", "lognormal"), ("binary", "ones")])
@pytest.mark.parametrize("loss,variant", [("logistic", "thread_greedy"), ("squared", "coloring")])
def test_storage_solve_reaches_the_stored_optimum(gb, mode, values, loss, variant):
    # Thread-Greedy has no convergence guarantee (Section 7): on the squared
    # loss here the FP64 oracle diverges at B = 16 too.  Coloring converges.
    prob = workloads.config3(values, loss)
    orc = oracle.Oracle(oracle.stored_problem(prob, mode))
    lam = 0.05 * orc.lambda_max()
    orc.set_lambda(lam)
    w_opt, _, _, _, _ = orc.solve("ccd", tol_kkt=1e-11, max_iter=4 * 10**8)
    with gb.Problem(prob, precision=mode) as p:
        p.set_lambda(lam)
        p.set_params(variant=variant, blocks=16, tol_kkt=1e-9, max_iter=200_000, check_every=50)
        r = p.solve()
        assert r.status == 0, r.as_dict()
        w = p.w()
    assert r.objective == pytest.approx(orc.objective(w_opt), rel=1e-6)
    assert_support_matches(oracle.stored_problem(prob, mode), lam, w, w_opt, label=f"{mode} {values} {loss}")


def test_storage_modes_reject_what_they_cannot_hold(gb):
    pm = workloads.config3("pm1")
    with pytest.raises(ValueError) as ref:
        oracle.stored_values(pm, "binary")
    with pytest.raises(gb.GencdError) as e:
        gb.Problem(pm, precision="binary")
    assert e.value.code == gb.GENCD_EINVAL
    col = str(ref.value).split()[1]
    assert f"column {col} " in str(e.value)
    big = workloads.config3("lognormal")
    big.val[7] = 3.4e38
    with pytest.raises(gb.GencdError) as e:
        gb.Problem(big, precision="bf16")
    assert e.value.code == gb.GENCD_EINVAL and "bfloat16" in str(e.value)


# Storage error bound (reading on storage modes): a mode that rounds X
# solves the problem P' on the stored X'.  With P* = P(w*) and P'* <= P'(w*),
#   P(w) - P* = [P(w) - P'(w)] + [P'(w) - P'*] + [P'* - P(w*)]
#             <= [P(w) - P'(w)] + gap'(w) + [P'(w*) - P(w*)],
# gap' the duality gap of w on P' (weak duality bounds P'(w) - P'*).  Every
# term is evaluated by the oracle in FP64.
def _storage_bound(prob, mode, lam, w, w_opt, P_opt):
    orig = oracle.Oracle(prob, lam)
    stored = oracle.Oracle(oracle.stored_problem(prob, mode), lam)
    bound = (orig.objective(w) - stored.objective(w)) + max(stored.duality_gap(w), 0.0) + \
        (stored.objective(w_opt) - orig.objective(w_opt))
    return bound / P_opt


SWEEP = (("pm1", ["f64", "f32", "bf16"]), ("ones", ["f64", "f32", "bf16", "binary"]),
         ("lognormal", ["f64", "f32", "bf16"]))


def test_precision_sweep_config3(gb, capsys):
    # Every storage mode on config 3's shapes (logistic, lambda = 0.01
    # lambda_max), Thread-Greedy B = 16: FP64 to KKT 1e-11, the FP32-arithmetic
    # modes to 1e-9 (the floor of FP32 sums here).  Parity isolates the
    # arithmetic: each mode's w is compared with the oracle's optimum of the
    # problem it stores (objective within 1e-6, supports equal outside the
    # columns that are fragile at the compared KKT accuracy).  The storage
    # error against the original problem is reported and held to the bound
    # above (1e-6 where the mode stores X exactly).
    rows = []
    for values, modes in SWEEP:
        prob = workloads.config3(values, "logistic")
        orc = oracle.Oracle(prob)
        lam = 0.01 * orc.lambda_max()
        orc.set_lambda(lam)
        w_opt = certified_optimum(f"cfg3_{values}_logistic", prob, lam)
        P_opt = orc.objective(w_opt)
        for mode in modes:
            sp = oracle.stored_problem(prob, mode)
            exact = bool(np.array_equal(sp.val, prob.val))
            # the optimum of the stored problem: the original one where the
            # mode stores X exactly or rounds it to FP32 (a KKT perturbation of
            # ~1e-11 here, inside the compared accuracy); bfloat16 of
            # log-normal values has its own stored optimum
            if exact or mode == "f32":
                w_ref = w_opt
            else:
                w_ref = certified_optimum(f"cfg3_{values}_logistic_{mode}", sp, lam)
            o_s = oracle.Oracle(sp, lam)
            P_ref = o_s.objective(w_ref)
            with gb.Problem(prob, precision=mode) as p:
                p.set_lambda(lam)
                p.set_params(variant="thread_greedy", blocks=16, tol_kkt=1e-11 if mode == "f64" else 1e-9,
                             max_iter=3_000_000, check_every=100)
                r = p.solve()
                assert r.status == 0, (values, mode, r.as_dict())
                w = p.w()
            rel_s = (o_s.objective(w) - P_ref) / P_ref
            assert abs(rel_s) <= 1e-6, (values, mode, rel_s)
            eps, nfrag, ndiff = assert_support_matches(sp, lam, w, w_ref, label=f"{values} {mode}")
            rel = (orc.objective(w) - P_opt) / P_opt
            bound = 1e-6 if exact else max(1e-6, _storage_bound(prob, mode, lam, w, w_opt, P_opt))
            assert rel <= bound, (values, mode, rel, bound)
            supp = int(np.sum((np.abs(w) > 1e-6) != (np.abs(w_opt) > 1e-6)))
            rows.append((values, mode, rel, bound, rel_s, np.abs(w - w_opt).max(), supp, ndiff, nfrag, eps,
                         r.iters))
    with capsys.disabled():
        print("\nprecision sweep (config 3 shapes, logistic, lambda = 0.01 lambda_max; Thread-Greedy B = 16)")
        print("  values    mode   vs original: (P(w)-P*)/P*  bound     | vs stored: rel. obj.  support diff "
              "(fragile)  KKT eps   | max|w-w*|  supp diff vs original  iters")
        for values, mode, rel, bound, rel_s, dw, supp, ndiff, nfrag, eps, it in rows:
            print(f"  {values:9s} {mode:6s} {rel:+.3e}  {bound:.1e} | {rel_s:+.2e}  {ndiff:3d} ({nfrag:3d})  "
                  f"{eps:.1e} | {dw:.2e}  {supp:3d}  {it}")


@pytest.mark.parametrize("loss", ["logistic", "squared"])
def test_block_shotgun_matches_the_oracle(gb, loss):
    # Section 7's block Shotgun (reading R14): 7 uneven column blocks, each
    # with its own P*_b from the block's spectral radius; the GPU's P*_b equal
    # the oracle's and 40 iterations follow the oracle's trajectory
    prob = workloads.config1(loss)
    orc = oracle.Oracle(prob)
    lam = 0.05 * orc.lambda_max()
    orc.set_lambda(lam)
    B = 7
    Pb_cpu = orc.block_pstar(B)
    with gb.Problem(prob) as p:
        p.set_lambda(lam)
        Pb, rho = p.block_pstar(B)
        np.testing.assert_array_equal(Pb, Pb_cpu)
        p.set_params(variant="shotgun_blocks", blocks=B, seed=4)
        p.stats_reset()
        p.iterate(40)
        w_gpu = p.w()
        upd = p.stats().updates
    w_cpu, _, _, st = orc.run("shotgun_blocks", 40, B=B, block_P=Pb_cpu, seed=4)
    # the oracle counts every selected column; the library counts the applied
    # (non-zero) steps
    assert 0 < upd <= st[0]
    np.testing.assert_array_equal(w_gpu != 0, w_cpu != 0)
    np.testing.assert_allclose(w_gpu, w_cpu, rtol=0, atol=1e-10)


@pytest.mark.parametrize("between", ["shotgun", "coloring"])
def test_block_shotgun_redraws_after_another_selection(gb, between):
    # Shotgun's and Coloring's permutations take the place of the blocks' ones:
    # within the same epoch and with the same seed, block Shotgun draws its own
    # again and continues as if the other variant had not run
    prob = workloads.config1("squared")
    lam = 0.05 * oracle.Oracle(prob).lambda_max()
    with gb.Problem(prob) as p:
        p.set_lambda(lam)

        def blocks(w, t):
            p.set_params(variant="shotgun_blocks", blocks=7, seed=4)
            p.set_w(w)
            p.set_iteration(t)
            p.iterate(1)
            return p.w()

        w1 = blocks(np.zeros(prob.k), 0)
        want = blocks(w1, 1)
        blocks(np.zeros(prob.k), 0)
        p.set_params(variant=between, P=100, seed=4)
        p.iterate(1)
        got = blocks(w1, 1)
    assert np.count_nonzero(want != w1) > 0
    np.testing.assert_array_equal(got != w1, want != w1)
    np.testing.assert_allclose(got, want, rtol=0, atol=1e-10)  # FP64 sums in another order


def test_block_shotgun_solve_reaches_the_optimum(gb):
    prob = workloads.uniform_problem(1000, 2000, 10, values="pm1", loss="logistic", n_planted=30, seed=21)
    orc = oracle.Oracle(prob)
    lam = 0.05 * orc.lambda_max()
    orc.set_lambda(lam)
    w_opt, _, _, kkt, _ = orc.solve("ccd", tol_kkt=1e-11)
    with gb.Problem(prob) as p:
        p.set_lambda(lam)
        p.set_params(variant="shotgun_blocks", blocks=16, tol_kkt=1e-10, max_iter=2_000_000, check_every=100)
        r = p.solve()
        assert r.status == 0, r.as_dict()
        w = p.w()
        with pytest.raises(gb.GencdError):
            p.set_params(variant="shotgun_blocks", blocks=1025)
    assert r.objective == pytest.approx(orc.objective(w_opt), rel=1e-6)
    assert_support_matches(prob, lam, w, w_opt, label="block shotgun")


@pytest.mark.parametrize("precision", ["f64", "f32"])
@pytest.mark.parametrize("name", ["cfg1-logistic", "cfg1-squared", "ragged-logistic", "zipf-slabs-squared"])
def test_duality_gap_matches_the_oracle(gb, name, precision):
    # the device's duality gap (objective, dual point from the FP64 loss
    # derivative scaled by lambda / max |g|) against the oracle's at the same w
    prob = PROBLEMS[name]()
    orc = oracle.Oracle(prob)
    lam = 0.05 * orc.lambda_max()
    orc.set_lambda(lam)
    w = _state(prob, 31)
    with gb.Problem(prob, precision=precision) as p:
        p.set_lambda(lam)
        p.set_w(w)
        gap, primal, dual = p.duality_gap()
    sp = prob if precision == "f64" else oracle.stored_problem(prob, "f32")
    o_s = oracle.Oracle(sp, lam)
    gap_cpu = o_s.duality_gap(w)
    P = o_s.objective(w)
    assert primal == pytest.approx(P, rel=1e-13 if precision == "f64" else 1e-9)
    # P and D are each accurate to their sums' rounding; the scale of D's
    # dual point comes from max |g| in the problem's arithmetic
    tol = 1e-11 if precision == "f64" else 1e-5
    assert abs(gap - gap_cpu) <= tol * (abs(P) + abs(P - gap_cpu))
    assert gap_cpu >= 0.0


@pytest.mark.parametrize("loss", ["logistic", "squared"])
def test_solve_to_a_duality_gap_certifies_the_objective(gb, loss):
    # stopping at a relative duality gap of 1e-9 bounds (P(w) - P*) / P(w)
    prob = workloads.uniform_problem(1000, 2000, 10, values="pm1", loss=loss, n_planted=30, seed=21)
    orc = oracle.Oracle(prob)
    lam = 0.05 * orc.lambda_max()
    orc.set_lambda(lam)
    w_opt, _, _, kkt, _ = orc.solve("ccd", tol_kkt=1e-11)
    P_opt = orc.objective(w_opt)
    with gb.Problem(prob) as p:
        p.set_lambda(lam)
        p.set_params(variant="thread_greedy", blocks=16, tol_kkt=0.0, tol_gap=1e-9, max_iter=400_000,
                     check_every=50)
        r = p.solve()
        assert r.status == 0, r.as_dict()
        w = p.w()
        gap, primal, _ = p.duality_gap()
    assert gap <= 1e-9 * abs(primal) * (1 + 1e-6)
    assert orc.duality_gap(w) <= 1e-9 * abs(primal) * (1 + 1e-3)
    assert (orc.objective(w) - P_opt) / P_opt <= 1e-9 * (1 + 1e-3)


@pytest.mark.parametrize("loss", ["logistic", "squared"])
def test_top_greedy_solve_reaches_the_optimum(gb, loss):
    # the global top-|J'| Accept has no convergence guarantee either: its solve
    # backs off (|J'| / G accepted, G growing 4x on a rise of the objective)
    # and reaches the oracle's optimum
    prob = workloads.uniform_problem(1000, 2000, 10, values="pm1", loss=loss, n_planted=30, seed=21)
    orc = oracle.Oracle(prob)
    lam = 0.05 * orc.lambda_max()
    orc.set_lambda(lam)
    w_opt, _, _, kkt, _ = orc.solve("ccd", tol_kkt=1e-11)
    with gb.Problem(prob) as p:
        p.set_lambda(lam)
        p.set_params(variant="top_greedy", blocks=64, tol_kkt=1e-10, max_iter=400_000, check_every=50)
        r = p.solve()
        assert r.status == 0, r.as_dict()
        w = p.w()
    assert r.objective == pytest.approx(orc.objective(w_opt), rel=1e-6)
    assert_support_matches(prob, lam, w, w_opt, label=f"top-|J'| {loss}")


@pytest.mark.parametrize("split", [0, 20, 24, 28, 31])
def test_every_propose_schedule_matches_the_oracle(gb, split):
    # the autotuner's candidates (two kernels, or the fused kernel with each
    # split of its warps) compute the same proposals, heavy and light columns
    prob = PROBLEMS["zipf-slabs-squared"]()
    orc = oracle.Oracle(prob)
    lam = 0.05 * orc.lambda_max()
    orc.set_lambda(lam)
    w = _state(prob, 41)
    z = orc.fitted(w)
    J = np.arange(prob.k, dtype=np.int32)
    d_cpu, f_cpu = orc.propose(w, z, J)
    with gb.Problem(prob, precision="f32") as p:
        p.set_lambda(lam)
        p.set_w(w)
        gb.gencd_set_propose_schedule(p.h, split)
        assert gb.gencd_propose_schedule(p.h)[0] == split
        for _ in range(2):  # the light-tile pool's counter is reset between launches
            d_all, f_all, kkt = p.propose_all()
            assert_steps_close(prob, z, w, lam, J, d_all, f_all, d_cpu, f_cpu, TOL["f32"])
        with pytest.raises(gb.GencdError):
            gb.gencd_set_propose_schedule(p.h, 17)


@pytest.mark.parametrize("precision,tol_rel", [("f32", 1e-3), ("f64", 1e-6)])
def test_config2_at_one_percent_solves_to_a_certified_point(gb, precision, tol_rel):
    # config 2's law at 1/100 of its size (n = 10,000, k = 40,000, 2e6 nnz),
    # the benchmark's Thread-Greedy (B = 1024): solved to KKT <= tol_rel lambda,
    # the oracle's FP64 KKT value and duality gap at the GPU's w certify it
    prob = workloads.config2_scaled(0.01, "logistic")
    orc = oracle.Oracle(prob)
    lam = 0.05 * orc.lambda_max()
    orc.set_lambda(lam)
    with gb.Problem(prob, precision=precision) as p:
        p.set_lambda(lam)
        p.set_params(variant="thread_greedy", blocks=1024, tol_kkt=tol_rel * lam, max_iter=200_000, check_every=10)
        r = p.solve()
        assert r.status == 0, r.as_dict()
        w = p.w()
    sp = prob if precision == "f64" else oracle.stored_problem(prob, "f32")
    o_s = oracle.Oracle(sp, lam)
    kkt = o_s.kkt(w)
    # FP32 sums: the oracle's KKT value may exceed the device's by their rounding
    assert kkt <= tol_rel * lam * (1.0 if precision == "f64" else 1.5) + (0 if precision == "f64" else 1e-9), kkt
    P = o_s.objective(w)
    assert o_s.duality_gap(w) <= (1e-5 if precision == "f64" else 1e-2) * P
    assert r.objective == pytest.approx(P, rel=1e-9)


@pytest.mark.parametrize("precision", ["f64", "f32"])
@pytest.mark.parametrize("k,B", [(1, 1), (255, 1), (256, 2), (257, 1), (1025, 1), (1025, 4), (3000, 3000),
                                 (70_001, 3), (400_003, 1)])
def test_accept_takes_each_partitions_best_column(gb, precision, k, B):
    # partitions of one chunk of columns and of many (the last chunk short,
    # more than one round of a CTA), launched twice: the chunk counts are reset
    prob = workloads.uniform_problem(400, k, 5, values="lognormal", n_planted=20, loss="logistic", seed=k + B)
    orc = oracle.Oracle(prob)
    lam = 0.02 * orc.lambda_max()
    orc.set_lambda(lam)
    w = _state(prob, 3, frac=min(0.05, 200 / k), scale=0.3)
    bounds = (np.arange(B + 1, dtype=np.int64) * k) // B
    with gb.Problem(prob, precision=precision) as p:
        p.set_lambda(lam)
        p.set_params(variant="thread_greedy", blocks=B)
        p.set_w(w)
        for _ in range(2):
            w0 = p.w()
            _, phi = orc.propose(w0, orc.fitted(w0), np.arange(k, dtype=np.int32))
            p.iterate(1)
            moved = np.flatnonzero(p.w() != w0)
            part = np.searchsorted(bounds, moved, side="right") - 1
            best = np.minimum.reduceat(phi, bounds[:-1])
            # FP32 proxies differ from the oracle's by their rounding (1e-4 of
            # the largest bounds it: sums of 5 terms, proxies of differences)
            slack = 1e-12 if precision == "f64" else 1e-4
            assert np.unique(part).size == part.size
            assert np.isin(np.flatnonzero(best < -slack * abs(phi).max()), part).all()
            assert (best[part] < (0 if precision == "f64" else slack * abs(phi).max())).all()
            assert np.all(phi[moved] <= best[part] * (1 - slack) + slack * abs(phi).max())


@pytest.mark.parametrize("precision", ["f64", "f32"])
def test_propose_at_longer_lists_and_between_iterations(gb, precision):
    # up to k columns the call uses the iterations' lists, beyond (repeats) its
    # own memory; between iterations it changes nothing of their course
    prob = workloads.config1("logistic")
    lam = 0.05 * oracle.Oracle(prob).lambda_max()
    w = []
    for ask in (False, True):
        with gb.Problem(prob, precision=precision) as p:
            p.set_lambda(lam)
            p.set_params(variant="thread_greedy", blocks=64)
            for _ in range(5):
                p.iterate(1)
                if ask:
                    d, f = p.propose_at(np.arange(prob.k, dtype=np.int32))
                    J = np.tile(np.arange(prob.k, dtype=np.int32), 3)[: 2 * prob.k + 7]
                    d2, f2 = p.propose_at(J)
                    np.testing.assert_array_equal(d2, d[J])
                    np.testing.assert_array_equal(f2, f[J])
            w.append(p.w())
    # FP64 additions of an iteration land in any order
    np.testing.assert_allclose(w[1], w[0], rtol=0, atol=(1e-12 if precision == "f64" else 1e-6) * np.abs(w[0]).max())


@pytest.mark.parametrize("precision", ["f64", "f32"])
@pytest.mark.parametrize("frac", [0.0, 0.002, 0.3, 0.5, 1.0])
@pytest.mark.parametrize("large", [False, True])
def test_set_w_fits_sparse_and_dense_coefficients(gb, precision, frac, large):
    # below and above the size from which columns are scattered, there on both
    # sides of the line between scattering columns and summing rows, columns
    # of many segments among them; a second call starts from scratch
    prob = (workloads.zipf_problem(60_000, 8_000, 1_200_000, cap=50_000, n_planted=10, loss="squared", seed=4)
            if large else ragged_problem("squared", 4))
    longest = int(np.argmax(prob.col_nnz()))
    orc = oracle.Oracle(prob)
    rng = np.random.default_rng(8)
    with gb.Problem(prob, precision=precision) as p:
        for _ in range(2):
            w = np.where(rng.random(prob.k) < frac, rng.normal(0, 0.5, prob.k), 0.0)
            if frac == 0.002:
                w[longest] = 0.7  # a column of 50,000 non-zeros
            p.set_w(w)
            # sums of at most a few hundred terms of size 10 in FP64 (stored values rounded to FP32)
            np.testing.assert_allclose(p.z(), orc.fitted(w), rtol=0, atol=1e-11 if precision == "f64" else 2e-5)
            np.testing.assert_array_equal(p.w(), w)


@pytest.mark.parametrize("precision", ["f64", "f32"])
def test_set_w_scatters_few_columns_of_many_segments(gb, precision):
    # 100 columns of 15,000 non-zeros: 3,000 segments, 120 of them of the four
    # columns set; their scatter is three launches, without the row-major copy
    rng = np.random.default_rng(5)
    n, k, m = 60_000, 100, 15_000
    rows = np.concatenate([np.sort(rng.permutation(n)[:m]) for _ in range(k)]).astype(np.int32)
    prob = workloads.Problem(n, k, np.arange(k + 1, dtype=np.int64) * m, rows, rng.normal(size=k * m),
                             rng.normal(size=n), "squared", np.zeros(k), "long-columns")
    orc = oracle.Oracle(prob)
    w = np.zeros(k)
    w[[3, 40, 41, 99]] = [0.5, -1.0, 0.25, 2.0]
    with gb.Problem(prob, precision=precision) as p:
        before = gb.gencd_profile_read(p.h, 8)[1]
        p.set_w(w)
        assert gb.gencd_profile_read(p.h, 8)[1] - before == 3
        # sums of at most four terms of size 10 (stored values rounded to FP32)
        np.testing.assert_allclose(p.z(), orc.fitted(w), rtol=0, atol=1e-13 if precision == "f64" else 2e-6)
        w = rng.normal(size=k)  # dense: by rows
        p.set_w(w)
        np.testing.assert_allclose(p.z(), orc.fitted(w), rtol=0, atol=1e-11 if precision == "f64" else 2e-5)
        # with the row-major copy there: either form in three launches and one wait
        for w in (rng.normal(size=k), np.where(np.arange(k) == 41, 3.0, 0.0), np.zeros(k), rng.normal(size=k)):
            before = gb.gencd_profile_read(p.h, 8)[1]
            p.set_w(w)
            assert gb.gencd_profile_read(p.h, 8)[1] - before == 3
            np.testing.assert_allclose(p.z(), orc.fitted(w), rtol=0, atol=1e-11 if precision == "f64" else 2e-5)


def test_fp32_solves_to_a_gap_near_their_rounding_level_end(gb):
    # two chains of 32 warm-started solves to a gap of 8e-7, which the FP32 sums
    # barely resolve: a solve that stalls above it is decided by FP64 sums
    # instead of running to the iteration cap
    prob = workloads.config4("squared", seed=0, scale=0.1)
    fold = workloads.cv_folds(prob.n, 5, seed=0)
    for f in (3, 4):
        sub = workloads.row_subset(prob, np.flatnonzero(fold != f))
        with gb.Problem(sub, precision="f32") as p, gb.Problem(sub, precision="f64") as q:
            for lam in workloads.lambda_grid(p.lambda_max(), 32, 1e-2):
                p.set_lambda(lam)
                p.set_params(variant="thread_greedy", blocks=1024, check_every=5, max_iter=20_000, tol_kkt=0.0,
                             tol_gap=8e-7)
                r = p.solve()
                assert r.status == 0, (f, lam, r.as_dict())
                q.set_lambda(lam)
                q.set_w(p.w())
                gap, P, _ = gb.gencd_duality_gap(q.h)
                # FP32 sums of some hundred cancelling terms know max |g_j| to
                # about 1.5e-6 of lambda, and lambda |w|_1 is up to 0.9 of P
                assert gap <= (8e-7 + 1.5e-6) * P + 1e-300, (f, lam)


@pytest.mark.parametrize("start", ["few", "dense", "grown"])
def test_restarts_of_large_problems_start_from_their_w(gb, start):
    # 1.2e6 non-zeros (z = Xw from the columns): Thread-Greedy's first steps
    # overshoot, so the solve restarts, from a w of few columns, from one whose
    # columns hold more than 2/5 of the non-zeros, and from such a one that
    # iterations grew (no row-major copy yet: z by rows is decided at the next
    # check).  The solve's z belongs to its w, and its objective falls
    prob = workloads.uniform_problem(3_000, 40_000, 30, values="lognormal", loss="squared", n_planted=20, seed=6)
    assert prob.nnz > 1 << 20
    orc = oracle.Oracle(prob)
    lam = (1e-4 if start == "grown" else 0.1) * orc.lambda_max()
    orc.set_lambda(lam)
    rng = np.random.default_rng(1)
    w0 = np.where(rng.random(prob.k) < (0.7 if start == "dense" else 1e-3), rng.normal(0, 1e-4, prob.k), 0.0)
    with gb.Problem(prob, precision="f64") as p:
        p.set_lambda(lam)
        p.set_w(w0)
        if start == "grown":
            p.set_params(variant="shotgun", P=40)
            p.iterate(1000)
            w0 = p.w()
            assert prob.col_nnz()[w0 != 0].sum() > 0.4 * prob.nnz
        p.set_params(variant="thread_greedy", blocks=1024, max_iter=200, check_every=10, tol_kkt=0.0)
        before = gb.gencd_profile_read(p.h, 8)[1]
        r = p.solve()
        assert gb.gencd_profile_read(p.h, 8)[1] - before >= 3  # it restarted
        w, z = p.w(), p.z()
    assert r.iters == 200
    np.testing.assert_allclose(z, orc.fitted(w), rtol=0, atol=1e-11 * max(1.0, np.abs(z).max()))
    assert r.objective == pytest.approx(orc.objective(w), rel=1e-9)
    assert r.objective < orc.objective(w0)


@pytest.mark.parametrize("precision", ["f64", "f32"])
@pytest.mark.parametrize("name,P", [("ragged-logistic", 1), ("ragged-logistic", 326), ("cfg1-logistic", 305),
                                    ("cfg1-logistic", 4500)])
def test_shotgun_steps_match(gb, name, P, precision):
    # one and several columns a CTA, columns at the edges of one warp's share
    # (255, 256, 257) and far beyond it, empty ones, lists on both sides of
    # the 4,096 entries summed in shared memory; two steps from the same start
    prob = PROBLEMS[name]()
    orc = oracle.Oracle(prob)
    lam = 0.05 * orc.lambda_max()
    orc.set_lambda(lam)
    w0 = _state(prob, 5)
    w_cpu, z_cpu, _, st = orc.run("shotgun", 2, w=w0, P=P, seed=7)
    with gb.Problem(prob, precision=precision) as p:
        p.set_lambda(lam)
        p.set_params(variant="shotgun", P=P, seed=7)
        p.set_w(w0)
        p.stats_reset()
        p.iterate(2)
        assert 0 < p.stats().updates <= st[0]  # the oracle counts steps of 0 too
        w, z = p.w(), p.z()
    # FP64 sums in another order; FP32: u and the stored values carry 2^-24,
    # and a column's step divides its sum's error by beta_j
    tol = 1e-10 if precision == "f64" else 2e-4
    np.testing.assert_allclose(w, w_cpu, rtol=0, atol=tol * max(1.0, np.abs(w_cpu).max()))
    np.testing.assert_allclose(z, z_cpu, rtol=0, atol=tol * max(1.0, np.abs(z_cpu).max()))


def test_logistic_values_over_the_whole_range(gb):
    # X = I: z = w, and with lambda = 0 a step is -4 u_i; margins at and next to
    # the table's centres (multiples of 1/32), half way between them, at the
    # end of its range (20), beyond it, and at 0
    k = np.arange(0, 20 * 32 + 1) / 32.0
    a = np.unique(np.concatenate([k, k[:-1] + 1 / 64, np.nextafter(k[:-1] + 1 / 64, 99), np.nextafter(k[1:], 0),
                                  np.linspace(1e-9, 45.0, 3001), [1e-300, 1e-17, 700.0, 745.0, 800.0]]))
    w = np.concatenate([a, -a])
    n = w.size
    y = np.where(np.arange(n) % 2 == 0, 1.0, -1.0)
    prob = workloads.Problem(n, n, np.arange(n + 1, dtype=np.int64), np.arange(n, dtype=np.int32), np.ones(n), y,
                             "logistic", np.zeros(n), "identity")
    with gb.Problem(prob) as p:
        p.set_lambda(0.0)
        p.set_w(w)
        d, _ = p.propose_at(np.arange(n, dtype=np.int32))
        obj, _ = p.objective()
    m = y.astype(np.longdouble) * w.astype(np.longdouble)
    u = -y / (1 + np.exp(m))
    # u to about two units in the last place, then divided by n, multiplied by
    # 1/beta and n; results below the normal range carry fewer bits
    np.testing.assert_allclose(d, (-4 * u).astype(np.float64), rtol=2e-15, atol=1e-305)
    loss = np.sum(np.maximum(-m, 0) + np.log1p(np.exp(-np.abs(m)))) / n
    assert obj == pytest.approx(float(loss), rel=1e-14)


@pytest.mark.parametrize("precision", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("n", [24_576, 24_577, 49_152, 49_153, 147_457, 640_000])
def test_propose_at_the_slabs_edges(gb, n, precision):
    # rows that fill 1, 2, 3 slabs exactly or by one more (24,576 rows in FP64,
    # 49,152 in FP32), and many slabs for few CTAs each
    prob = workloads.zipf_problem(n, 1_500, 150_000, cap=n // 2, n_planted=10, loss="squared", seed=n % 89)
    if precision == "bf16":
        prob = oracle.stored_problem(prob, "bf16")
    orc = oracle.Oracle(prob)
    lam = 0.05 * orc.lambda_max()
    orc.set_lambda(lam)
    w = _state(prob, 17)
    z = orc.fitted(w)
    J = np.arange(prob.k, dtype=np.int32)
    d_cpu, f_cpu = orc.propose(w, z, J)
    with gb.Problem(prob, precision=precision) as p:
        p.set_lambda(lam)
        p.set_w(w)
        for _ in range(2):
            d, f, _ = p.propose_all()
            assert_steps_close(prob, z, w, lam, J, d, f, d_cpu, f_cpu, TOL[precision if precision == "f64" else "f32"])


@pytest.mark.parametrize("precision", ["f64", "f32", "bf16", "binary"])
def test_propose_with_light_and_heavy_columns(gb, precision):
    # columns that average less than half an entry per slab of rows keep the
    # light pass when they hold more than 2^22 non-zeros: 1.2e6 of 4 entries
    # beside 2,000 of 300 and a long one, 10 slabs in FP32 and 20 in FP64; every
    # schedule of the two passes
    rng = np.random.default_rng(12)
    n = 480_000
    counts = np.full(1_200_000, 4, np.int64)
    counts[rng.permutation(counts.size)[:2000]] = 300
    counts[77] = 100_000
    counts[[0, 5, counts.size - 1]] = 0
    col_ptr = np.zeros(counts.size + 1, np.int64)
    np.cumsum(counts, out=col_ptr[1:])
    rows = workloads.synthetic._distinct_rows(n, counts, rng)
    val = np.repeat(rng.lognormal(0.0, 0.5, counts.size), counts)
    if precision != "binary":
        val = val * rng.lognormal(0.0, 0.5, rows.size)
    prob = workloads.Problem(n, counts.size, col_ptr, rows, val, rng.normal(size=n), "squared",
                             np.zeros(counts.size), "light-heavy")
    sp = oracle.stored_problem(prob, precision) if precision in ("bf16", "binary") else prob
    orc = oracle.Oracle(sp)
    lam = 0.05 * orc.lambda_max()
    orc.set_lambda(lam)
    w = _state(prob, 17, frac=0.01)
    z = orc.fitted(w)
    J = np.arange(prob.k, dtype=np.int32)
    d_cpu, f_cpu = orc.propose(w, z, J)
    with gb.Problem(prob, precision=precision) as p:
        p.set_lambda(lam)
        p.set_w(w)
        for split in [0] if precision == "f64" else [0, 20, 31]:
            gb.gencd_set_propose_schedule(p.h, split)
            d, f, _ = p.propose_all()
            assert_steps_close(sp, z, w, lam, J, d, f, d_cpu, f_cpu, TOL["f64" if precision == "f64" else "f32"])


@pytest.mark.parametrize("slabs", [1, 2, 4, 7, 8])
@pytest.mark.parametrize("per_col", [3, 12, 100])
def test_fp32_sums_of_short_columns_keep_their_error(gb, slabs, per_col):
    # runs of few entries over 1 to 8 slabs (49,152 rows each), against 64 bits:
    # each of a sum's L products and L - 1 additions is rounded by an independent
    # c = 0.41 2^-24 of its value (rms), partial sums of i terms are sqrt(i) terms
    # large, so the error is at most c sqrt(1 + L / 2) of the norm when the terms
    # are added one after another (a lane's 8, then the lanes in a tree: 16 at
    # most here); 1.3 for the values' spread
    n, k = 49_152 * slabs - 100, 40_000
    rng = np.random.default_rng(slabs)
    counts = np.full(k, per_col, np.int64)
    counts[5] = 20_000  # a heavy column beside them
    col_ptr = np.zeros(k + 1, np.int64)
    np.cumsum(counts, out=col_ptr[1:])
    rows = workloads.synthetic._distinct_rows(n, counts, rng)
    val = rng.lognormal(0.0, 1.0, rows.size).astype(np.float32).astype(np.float64)
    y = rng.normal(size=n).astype(np.float32).astype(np.float64)
    prob = workloads.Problem(n, k, col_ptr, rows, val, y, "squared", np.zeros(k), "short")
    with gb.Problem(prob, precision="f32") as p:
        p.set_lambda(0.0)
        p.set_params(beta_mode=1)
        d, _, _ = p.propose_all()  # lambda = 0, beta = 1, w = 0: delta = -g
    g = np.add.reduceat(val * -y[rows], col_ptr[:-1]) / n
    short = np.arange(k) != 5
    err = np.linalg.norm((d + g)[short]) / np.linalg.norm(g[short])
    assert err < 1.3 * 0.41 * 2.0**-24 * np.sqrt(1 + min(per_col, 16) / 2)


@pytest.mark.parametrize("precision", ["f64", "f32"])
@pytest.mark.parametrize("n,per_col,long,passes", [
    (300_000, 3, 0, "light"), (300_000, 3, 20_000, "slabs"),  # 7 slabs in FP32, 13 in FP64
    (300_000, 60, 0, "slabs"), (40_000, 3, 0, None)])
def test_light_columns_alone_keep_their_pass(gb, n, per_col, long, passes, precision):
    # few short columns join the slabs beside heavy ones only: alone, their own
    # pass is the one kernel; either way the proposals are the oracle's
    rng = np.random.default_rng(n + per_col)
    counts = np.full(50_000, per_col, np.int64)
    if long:
        counts[777] = long
    col_ptr = np.zeros(counts.size + 1, np.int64)
    np.cumsum(counts, out=col_ptr[1:])
    rows = workloads.synthetic._distinct_rows(n, counts, rng)
    prob = workloads.Problem(n, counts.size, col_ptr, rows, rng.normal(size=rows.size), rng.normal(size=n), "squared",
                             np.zeros(counts.size), "light")
    orc = oracle.Oracle(prob)
    lam = 0.05 * orc.lambda_max()
    orc.set_lambda(lam)
    w = _state(prob, 3, frac=0.01)
    z = orc.fitted(w)
    J = np.arange(prob.k, dtype=np.int32)
    d_cpu, f_cpu = orc.propose(w, z, J)
    with gb.Problem(prob, precision=precision) as p:
        p.set_lambda(lam)
        p.set_w(w)
        gb.gencd_profile_reset(p.h)
        d, f, _ = p.propose_all()
        ran = [gb.gencd_profile_read(p.h, kernel)[1] for kernel in (9, 10, 12)]  # light, slabs, both in one
    if passes is None:
        passes = "slabs" if precision == "f32" else "light"  # one slab in FP32, two in FP64
    assert ran == ([1, 0, 0] if passes == "light" else [0, 1, 0])
    assert_steps_close(prob, z, w, lam, J, d, f, d_cpu, f_cpu, TOL[precision])


@pytest.mark.parametrize("precision", ["f64", "f32"])
@pytest.mark.parametrize("n", [3_000, 30_000])
@pytest.mark.parametrize("B", [1, 256, 257, 512, 513])
def test_update_and_refresh_on_both_sides_of_one_launch(gb, n, B, precision):
    # columns of 16: up to 256 (FP64) and 512 (FP32) partitions z and u take
    # one launch, with fewer rows than touched (all refreshed) and more; z has
    # to be X w, and u is what the proposals of the new state see
    prob = workloads.uniform_problem(n, 8_000, 16, values="lognormal", loss="logistic", n_planted=30, seed=2)
    assert prob.col_nnz().max() == 16
    orc = oracle.Oracle(prob)
    lam = 0.02 * orc.lambda_max()
    orc.set_lambda(lam)
    with gb.Problem(prob, precision=precision) as p:
        p.set_lambda(lam)
        p.set_params(variant="thread_greedy", blocks=B)
        p.iterate(3)
        w, z = p.w(), p.z()
        d, f, _ = p.propose_all()
    assert np.count_nonzero(w) > 0
    tol = TOL[precision]
    # sums of n_i terms of w_j x_ij: 2^-53 each and per partial sum (some tens of
    # columns a row, three times over); stored values carry 2^-24 in FP32
    terms = np.bincount(prob.row_idx, weights=np.abs(prob.val * np.repeat(w, prob.col_nnz())), minlength=n).max()
    np.testing.assert_allclose(z, orc.fitted(w), rtol=0, atol=(3e-14 if precision == "f64" else 1.2e-7) * terms)
    J = np.arange(prob.k, dtype=np.int32)
    d_cpu, f_cpu = orc.propose(w, z, J)
    assert_steps_close(prob, z, w, lam, J, d, f, d_cpu, f_cpu, tol)
