"""GPU: te_network_infer with the linear-Gaussian estimator against the
oracle's network inference with the same estimator.

Test decisions compare estimates, so the network path sums its
cross-covariances in FP64 (differences from the FP64 oracle are rounding
noise, far below 1e-10), and a decision can only differ where the oracle's
own decision is closer than that to a tie.  Each case first checks on the
oracle's trace that every deciding comparison (best against runner-up,
observed against each surrogate statistic) is separated by more than 1e-9;
exact ties (a surrogate whose permutation reproduces the original data) are
equal on both sides.  Then edges, selections, p-values and counts must be
identical and the omnibus estimates equal within 1e-10."""
import numpy as np
import pytest

import synth
from oracle import network as onet

pytestmark = pytest.mark.gpu

MARGIN = 1e-9      # smallest deciding gap the cases must have
TOL = 1e-10        # omnibus estimates, GPU against oracle


@pytest.fixture(scope="module")
def te():
    import paper_1902_06828_gb300 as te
    return te


@pytest.fixture(scope="module")
def ctx(te):
    c = te.Context(0)
    yield c
    c.close()


_margin = onet.decision_margin


def _compare(g, adj_o, res_o):
    np.testing.assert_array_equal(g["adjacency"], adj_o)
    for gt, o in zip(g["targets"], res_o):
        assert gt["target"] == o.target
        assert gt["sel_target"] == [tuple(v) for v in o.sel_target]
        assert gt["sel_sources"] == [tuple(v) for v in o.sel_sources]
        assert gt["omnibus_tested"] == o.omnibus_tested
        assert gt["omnibus_p"] == o.omnibus_p
        assert abs(gt["omnibus_cmi"] - o.omnibus_cmi) <= TOL
        assert gt["significant"] == o.significant
        assert gt["n_estimates"] == o.n_estimates
    assert g["theiler"] == 0


@pytest.mark.parametrize("seed,seq,fdr", [(5, False, False), (7, True, True)])
def test_gauss_network_matches_oracle(te, ctx, seed, seq, fdr):
    x, _adj, _lags = synth.var_er(n=5, p=0.35, T=1500, seed=seed, lo=0.3, hi=0.6, max_lag=3)
    s = synth.standardise_jitter(x, seed)
    kw = dict(max_lag_target=3, max_lag_sources=3, n_surr=50, alpha_max=0.1, alpha_min=0.1,
              alpha_omnibus=0.1, alpha_seq=0.1, seq_test=seq, fdr=fdr, alpha_fdr=0.1, seed=21,
              estimator="gauss")
    adj_o, res_o = onet.infer_network(s, onet.Params(**kw))
    assert _margin(res_o) > MARGIN
    g = te.te_network_infer(ctx, te.te_data_create(ctx, s), **kw)
    _compare(g, adj_o, res_o)
    assert g["n_estimates"] == sum(r.n_estimates for r in res_o)


def test_gauss_network_independent_surrogates_match_oracle(te, ctx):
    x, _adj, _lags = synth.var_er(n=4, p=0.4, T=1200, seed=6, lo=0.3, hi=0.6, max_lag=2)
    s = synth.standardise_jitter(x, 6)
    kw = dict(max_lag_target=2, max_lag_sources=2, n_surr=40, alpha_max=0.1, alpha_min=0.1,
              alpha_omnibus=0.1, alpha_seq=0.1, seq_test=True, seed=13, indep_surr=True,
              estimator="gauss")
    adj_o, res_o = onet.infer_network(s, onet.Params(**kw))
    assert _margin(res_o) > MARGIN
    g = te.te_network_infer(ctx, te.te_data_create(ctx, s), **kw)
    _compare(g, adj_o, res_o)


def _trials(R, T, seed):
    rows = []
    for r in range(R):
        x, _ = synth.var_chain3(T, seed + r, coupling=0.6)
        rows.append(synth.standardise_jitter(x, seed + r))
    return np.ascontiguousarray(np.stack(rows, axis=1).astype(np.float32))   # [3][R][T]


@pytest.mark.parametrize("seed,mode", [(1, "trials"), (2, "within")])
def test_gauss_network_trial_surrogates_match_oracle(te, ctx, seed, mode):
    s3 = _trials(5, 300, seed)
    kw = dict(max_lag_target=2, max_lag_sources=2, n_surr=40, alpha_max=0.1, alpha_min=0.1,
              alpha_omnibus=0.1, seed=seed, estimator="gauss")
    adj_o, res_o = onet.infer_network(s3, onet.Params(**kw), trials=mode)
    assert _margin(res_o) > MARGIN
    data = te.te_data_create_trials(ctx, s3, 2)
    g = te.te_network_infer(ctx, data, surr_mode=mode, **kw)
    _compare(g, adj_o, res_o)


def test_gauss_network_rejects_theiler_window(te, ctx):
    s = synth.workload_chain3(T=300, seed=1)["series"]
    data = te.te_data_create(ctx, s)
    for w in (1, -1):
        with pytest.raises(te.TEError, match="TE_EINVAL"):
            te.te_network_infer(ctx, data, theiler=w, n_surr=40, estimator="gauss")
    # k is not used by the Gaussian estimator
    g = te.te_network_infer(ctx, data, k=0, max_lag_target=2, max_lag_sources=2, n_surr=40,
                            estimator="gauss")
    assert g["adjacency"][1, 2] == 1


def test_gauss_network_full_length_target(te, ctx):
    """var10 at T = 10^4 (N = 9995), all lags up to 5, S = 100: target 3,
    whose closest deciding gap in the oracle is about 3e-8 (a split-TF32
    contraction, ~1e-7, could flip it)."""
    s = synth.workload_var10(T=10000, seed=1)["series"]
    kw = dict(max_lag_target=5, max_lag_sources=5, n_surr=100, alpha_max=0.05,
              alpha_min=0.05, alpha_omnibus=0.05, seed=3, estimator="gauss")
    r = onet.infer_target(s, 3, onet.Params(**kw))
    assert MARGIN < _margin([r]) < 1e-7
    g = te.te_network_infer(ctx, te.te_data_create(ctx, s), targets=[3], **kw)
    gt = g["targets"][0]
    assert gt["sel_target"] == [tuple(v) for v in r.sel_target]
    assert gt["sel_sources"] == [tuple(v) for v in r.sel_sources]
    assert gt["omnibus_p"] == r.omnibus_p
    assert abs(gt["omnibus_cmi"] - r.omnibus_cmi) <= TOL
    assert gt["n_estimates"] == r.n_estimates


@pytest.mark.parametrize("T,S", [(203, 31), (703, 32), (706, 33), (1031, 255), (390, 256),
                                 (1417, 300)])
def test_every_estimate_at_growing_conditioning_sets(te, ctx, T, S):
    """Every traced estimate against a plain FP64 evaluation, at surrogate
    counts on both sides of a warp and of a block of rows and at odd lengths.
    With alpha = 0.9 almost every candidate is selected, so that W grows
    column by column from 1 to over 16, through every width of the
    shared-memory contraction and into the FP64 one."""
    from oracle import ksg as oksg
    L, n = 6, 3
    x, _adj, _lags = synth.var_er(n=n, p=0.5, T=T, seed=T, lo=0.3, hi=0.6, max_lag=3)
    s = synth.standardise_jitter(x, T).astype(np.longdouble)
    N = T - L
    col = lambda v: s[v[0], L - v[1]:T - v[1]]
    sel, widths, errs = [], set(), []

    def explained(a, c):   # c^T a^-1 c by a Cholesky factor (lags are nearly collinear)
        m = len(a)
        f, v = np.zeros((m, m), np.longdouble), np.zeros_like(c)
        for j in range(m):
            f[j, j] = np.sqrt(a[j, j] - np.sum(f[j, :j] ** 2))
            f[j + 1:, j] = (a[j + 1:, j] - f[j + 1:, :j] @ f[j, :j]) / f[j, j]
        for j in range(m):
            v[:, j] = (c[:, j] - v[:, :j] @ f[j, :j]) / f[j, j]
        return np.sum(v ** 2, axis=1)

    def value(key):   # inverse of the order-preserving image
        k = key & ((1 << 64) - 1)
        k = k - (1 << 64) if k >= 1 << 63 else k
        return np.int64(k if k >= 0 else k ^ 0x7FFFFFFFFFFFFFFF).view(np.float64)

    def check(target, stage, it, vs, n_cand, n_surr, keys):
        if stage not in (1, 2):
            return
        got = np.array([[value(k) for k in row] for row in keys])
        W = np.array([col((0, 0))] + [col(v) for v in sel])
        W = W - W.mean(1, keepdims=True)
        widths.add(len(W))
        perms = [np.arange(N)] + [oksg.permutation(9, 0, stage, it, a, N)
                                  for a in range(1, n_surr + 1)]
        sww = W @ W.T / (N - 1)
        for c, v in enumerate(vs):
            xc = col(v) - col(v).mean()
            cw = np.array([xc[p] for p in perms]) @ W.T / (N - 1)
            sxx = xc @ xc / (N - 1)
            ref = 0.5 * (np.log(sxx - explained(sww[1:, 1:], cw[:, 1:]))
                         - np.log(sxx - explained(sww, cw)))
            errs.append(float(np.max(np.abs(got[c] - ref))))
        best = int(np.argmax(got[:, 0]))
        if np.sum(got[:, 1:].max(0) > got[best, 0]) / n_surr < 0.9:
            sel.append(tuple(vs[best]))

    data = te.te_data_create(ctx, s.astype(np.float32))
    ctx.set_trace(check)
    try:
        te.te_network_infer(ctx, data, max_lag_target=L, max_lag_sources=L, n_surr=S,
                            alpha_max=0.9, alpha_min=0.9, alpha_omnibus=0.9, seed=9, targets=[0],
                            estimator="gauss")
    except te.TEError as e:   # more than 8 sources left for the omnibus block
        assert "dx <= 8" in str(e)
    finally:
        ctx.set_trace(None)
    assert len(errs) > 20 and max(widths) > 4 and max(errs) <= TOL


def test_more_permutation_sets_in_a_round_than_a_grid_dimension(te, ctx):
    """Independent surrogates draw a set per candidate: 257 processes with one
    lag have 65,792 candidates in the first round of the sources stage, in
    batches that each turn their own sets.  A target's result does not depend
    on which others are analysed with it, so a few targets alone agree."""
    n, T = 257, 43
    s = synth.standardise_jitter(np.random.default_rng(4).normal(size=(n, T)), 4)
    kw = dict(max_lag_target=1, max_lag_sources=1, n_surr=3, alpha_max=0.4, alpha_min=0.4,
              alpha_omnibus=0.4, seed=6, indep_surr=True, estimator="gauss")
    data = te.te_data_create(ctx, s)
    some = [0, 16, 17, 128, 256]
    ref = te.te_network_infer(ctx, data, targets=some, **kw)
    got = te.te_network_infer(ctx, data, **kw)
    by = {t["target"]: t for t in got["targets"]}
    for r in ref["targets"]:
        g = by[r["target"]]
        assert (g["sel_target"], g["sel_sources"]) == (r["sel_target"], r["sel_sources"])
        assert g["n_estimates"] == r["n_estimates"] and g["omnibus_p"] == r["omnibus_p"]
        assert g["omnibus_cmi"] == r["omnibus_cmi"] or abs(g["omnibus_cmi"] - r["omnibus_cmi"]) <= TOL
    data.close()


@pytest.mark.parametrize("T,S", [(1501, 40), (26001, 3), (26002, 3)])
def test_every_width_of_the_conditioning_set(te, ctx, T, S):
    """A target driven by twenty sources with equal weights selects them one by
    one: W has every width from 1 to 18 (the shared-memory contraction ends
    at 16), at N = 1500 and on both sides of the N = 26,000 whose X column still
    fits shared memory; sampled estimates against FP64."""
    from oracle import ksg as oksg
    n, alpha = 21, 0.05 if S > 20 else 0.4
    rng = np.random.default_rng(T)
    s = rng.normal(size=(n, T))
    s[0, 1:] = 0.5 * s[1:, :-1].sum(0) + 0.2 * rng.normal(size=T - 1)
    s = synth.standardise_jitter(s, T).astype(np.float32)
    N = T - 1
    col = lambda v: s[v[0], 1 - v[1]:T - v[1]].astype(np.float64)
    sel, widths, errs = [], set(), []

    def value(key):   # inverse of the order-preserving image
        k = key & ((1 << 64) - 1)
        k = k - (1 << 64) if k >= 1 << 63 else k
        return np.int64(k if k >= 0 else k ^ 0x7FFFFFFFFFFFFFFF).view(np.float64)

    def check(target, stage, it, vs, n_cand, n_surr, keys):
        if stage not in (1, 2):
            return
        got = np.array([[value(k) for k in row] for row in keys])
        W = np.array([col((0, 0))] + [col(v) for v in sel])
        W -= W.mean(1, keepdims=True)
        widths.add(len(W))
        inv = np.linalg.inv(W @ W.T / (N - 1))
        inv_z = np.linalg.inv(W[1:] @ W[1:].T / (N - 1)) if sel else None
        for c in (0, len(vs) // 2, len(vs) - 1):
            for a in (0, 1, n_surr):
                x = col(vs[c]) - col(vs[c]).mean()
                if a:
                    x = x[oksg.permutation(9, 0, stage, it, a, N)]
                cw, sxx = W @ x / (N - 1), x @ x / (N - 1)
                z = cw[1:] @ inv_z @ cw[1:] if sel else 0.0
                ref = 0.5 * (np.log(sxx - z) - np.log(sxx - cw @ inv @ cw))
                errs.append(abs(got[c, a] - ref))
        best = int(np.argmax(got[:, 0]))
        if np.sum(got[:, 1:].max(0) > got[best, 0]) / n_surr < alpha:
            sel.append(tuple(vs[best]))

    data = te.te_data_create(ctx, s)
    ctx.set_trace(check)
    try:
        te.te_network_infer(ctx, data, max_lag_target=1, max_lag_sources=1, n_surr=S,
                            alpha_max=alpha, alpha_min=alpha, alpha_omnibus=alpha, seed=9,
                            targets=[0], estimator="gauss")
    except te.TEError as e:   # more than 8 sources left for the omnibus block
        assert "dx <= 8" in str(e)
    finally:
        ctx.set_trace(None)
    assert set(range(1, 19)) <= widths and max(errs) <= TOL
    data.close()
