"""The neighbour-list kernels (the default) against the member-lane kernel,
which a forced tile length selects: the keys are exact integers, so they are
equal, at the sizes where the lists can go wrong: fewer points than a step of
32 entries, one to five members (a CTA holds four, two or one), every count
of Z variables that has its own form (none, one, several), k beyond the lanes
of a member's group, several X variables, Theiler bands, tied distances (lists
that stay empty) and the largest point counts of every CTA width.  The
unpermuted estimates also equal the oracle's at the small sizes."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import paper_1902_06828_gb300 as te
    ctx = te.Context(0)
    yield te, ctx
    ctx.close()


def _both(te, ctx, jobs):
    ctx.set_option("ksg_tile", 0)
    _, got = te.cmi_ksg_batch(ctx, jobs, return_keys=True)
    try:
        ctx.set_option("ksg_tile", 256)
        _, ref = te.cmi_ksg_batch(ctx, jobs, return_keys=True)
    finally:
        ctx.set_option("ksg_tile", 0)
    return got, ref


Z = [(0, 1), (4, 2), (0, 2), (7, 1), (1, 4), (5, 3), (8, 2), (9, 1), (6, 2)]


@pytest.mark.parametrize("T,dz,dx,S,k,w", [
    (13, 2, 1, 0, 4, 0), (13, 0, 1, 3, 1, 1), (40, 1, 1, 4, 4, 0), (41, 3, 1, 2, 4, 3),
    (69, 0, 2, 1, 4, 0), (69, 2, 3, 4, 4, 2), (300, 1, 1, 5, 8, 0), (300, 1, 2, 3, 4, 5),
    (301, 2, 1, 6, 9, 0), (301, 0, 1, 6, 16, 4), (700, 9, 1, 3, 4, 0), (700, 1, 1, 7, 16, 7),
    (1203, 2, 1, 70, 4, 0), (1203, 1, 1, 66, 4, 11), (1203, 0, 1, 65, 4, 0),
    (1203, 5, 4, 9, 3, 0)])
def test_lists_equal_the_member_lane_kernel_and_the_oracle(env, T, dz, dx, S, k, w):
    from oracle import ksg as oksg
    te, ctx = env
    s = np.asarray(synth.workload_var10(T=T, seed=T + dz)["series"], dtype=np.float32)
    data = te.te_data_create(ctx, s)
    z = Z[:dz]
    xs = [[(2, 1 + a) for a in range(dx)], [(3, 1 + a) for a in range(dx)]]
    jobs = [te.Job(data, x, [(0, 0)], z, k=k, theiler=w, max_lag=5, n_surr=S, seed=4,
                   stream_tag=9) for x in xs]
    got, ref = _both(te, ctx, jobs)
    assert got == ref
    for x, keys in zip(xs, got):
        assert keys[0] == oksg.cmi_ksg(s, x, [(0, 0)], z, k=k, theiler=w, max_lag=5)["key"]
    data.close()


@pytest.mark.parametrize("dz", [0, 1, 2])
@pytest.mark.parametrize("levels", [2, 7, 40])
def test_tied_distances(env, dz, levels):
    """Few distinct values: most distances are equal, radii end at ties, lists
    hold nothing or stop short, and pairs scan all points."""
    from oracle import ksg as oksg
    te, ctx = env
    rng = np.random.default_rng(levels + dz)
    s = rng.integers(0, levels, size=(10, 2600)).astype(np.float32)
    data = te.te_data_create(ctx, s)
    jobs = [te.Job(data, [(2, 1)], [(0, 0)], Z[:dz], k=4, max_lag=5, n_surr=5, seed=1)]
    got, _ = _both(te, ctx, jobs) if dz else (te.cmi_ksg_batch(ctx, jobs, return_keys=True)[1], 0)
    perms = np.stack([oksg.permutation(1, 0, 0, 0, a, 2595) for a in range(1, 6)])
    ok, _, _ = oksg.cmi_ksg_batch(s, [[(2, 1)]] * 6, [(0, 0)], Z[:dz], perms=perms,
                                  perm_idx=[-1] + list(range(5)), k=4, max_lag=5)
    assert got[0] == ok
    data.close()


@pytest.mark.parametrize("N", [10496, 10497, 20992, 20993, 41984, 41985])
def test_largest_point_counts_of_every_width(env, N):
    """The last N at which a CTA holds four, two and one members' X values, and
    the first beyond (past the last, the member-lane kernel is the default)."""
    te, ctx = env
    rng = np.random.default_rng(N)
    s = rng.normal(size=(3, N + 1)).astype(np.float32)
    s[1, 1:] += 0.5 * s[0, :-1]
    data = te.te_data_create(ctx, s)
    for z in ([(1, 1), (2, 1)], [(1, 1)]):
        jobs = [te.Job(data, [(0, 1)], [(1, 0)], z, k=4, max_lag=1, n_surr=4, seed=2)]
        got, ref = _both(te, ctx, jobs)
        assert got == ref
    data.close()


@pytest.mark.parametrize("dz,N", [(0, 9876), (0, 9877), (0, 19756), (0, 19757), (0, 39512),
                                  (0, 39513), (1, 10332), (1, 10333), (1, 20352), (1, 20353),
                                  (1, 39512), (1, 39513)])
def test_largest_point_counts_with_a_coarse_column_beside_the_x_values(env, dz, N):
    """With one Z variable or none a CTA also holds every 16th value of the
    sorted columns, so its widths end earlier. The executed evaluations tell
    which kernel ran: equal to the member-lane kernel's past the last N only."""
    te, ctx = env
    rng = np.random.default_rng(N)
    s = rng.normal(size=(3, N + 1)).astype(np.float32)
    s[1, 1:] += 0.5 * s[0, :-1]
    data = te.te_data_create(ctx, s)
    runs = []
    for option, value in (("ksg_lists", 1), ("ksg_tile", 256)):
        try:
            ctx.set_option(option, value)
            before = ctx.stats()["pair_evals"]
            keys = te.cmi_ksg(ctx, data, [(0, 1)], [(1, 0)], [(2, 1)][:dz], k=4, max_lag=1,
                              n_surr=4, seed=2, return_keys=True)[1]
            runs.append((keys, ctx.stats()["pair_evals"] - before))
        finally:
            ctx.set_option(option, 0)
    assert runs[0][0] == runs[1][0]
    assert (runs[0][1] == runs[1][1]) == (N > 39512)
    data.close()


def test_columns_of_different_point_sets_in_one_batch(env):
    """Jobs whose maximum lags differ read the same memory as columns of
    different lengths; each sorts its own."""
    from oracle import ksg as oksg
    te, ctx = env
    s = np.asarray(synth.workload_var10(T=400, seed=8)["series"], dtype=np.float32)
    data = te.te_data_create(ctx, s)
    jobs = [te.Job(data, [(2, ml)], [(0, 0)], z, k=4, max_lag=ml, n_surr=3, seed=2)
            for ml in (2, 5) for z in ([], [(0, ml)])]
    _, got = te.cmi_ksg_batch(ctx, jobs, return_keys=True)
    for j, keys in zip(jobs, got):
        o = oksg.cmi_ksg(s, j.x, j.y, j.z, k=4, max_lag=j.max_lag)
        assert keys[0] == o["key"], (j.max_lag, j.z)
    data.close()


@pytest.mark.parametrize("N", [6, 33, 511, 513, 2048, 2049, 4099])
def test_permutations_at_every_launch_shape(env, N):
    """Surrogate keys equal the oracle's, whose permutations come from the
    sequential shuffle, at point counts on both sides of every thread count of
    the parallel one; two jobs of different length share their permutations."""
    from oracle import ksg as oksg
    te, ctx = env
    rng = np.random.default_rng(N)
    s = rng.normal(size=(3, N)).astype(np.float32)
    data = te.te_data_create(ctx, s)
    jobs = [te.Job(data, [(p, 0)], [(1, 0)], [], k=2, max_lag=0, n_surr=S, seed=5, stream_tag=6)
            for p, S in ((0, 2), (2, 5))]
    _, got = te.cmi_ksg_batch(ctx, jobs, return_keys=True)
    perms = np.stack([oksg.permutation(5, 6, 0, 0, a, N) for a in range(1, 6)])
    for j, keys in zip(jobs, got):
        ok, _, _ = oksg.cmi_ksg_batch(s, [j.x] * (j.n_surr + 1), j.y, [], perms=perms,
                                      perm_idx=[-1] + list(range(j.n_surr)), k=2, max_lag=0)
        assert keys == ok
    data.close()


@pytest.mark.parametrize("N", [20480, 20481])
def test_permutations_past_the_parallel_shuffle(env, N):
    """The largest N of the parallel shuffle and the first past it: a
    surrogate's X values, read back through the Gaussian estimate, give the
    estimate of the permuted column."""
    from oracle import ksg as oksg
    te, ctx = env
    rng = np.random.default_rng(N)
    s = rng.normal(size=(2, N)).astype(np.float32)
    data = te.te_data_create(ctx, s)
    got, _ = te.cmi_gauss(ctx, data, [(0, 0)], [(1, 0)], max_lag=0, n_surr=3, seed=8, stream_tag=1)
    for a in range(1, 4):
        x = s[0].astype(np.float64)[oksg.permutation(8, 1, 0, 0, a, N)]
        r = np.corrcoef(x, s[1].astype(np.float64))[0, 1]
        assert abs(got[a] - -0.5 * np.log1p(-r * r)) < 1e-7
    data.close()


@pytest.mark.parametrize("N", [65535, 65536, 70001])
def test_gaussian_estimates_past_16_bit_permutations(env, N):
    """The largest N whose surrogates are drawn as 16-bit rows and the first past
    it, where the contraction reads 32-bit ones: every surrogate with two Z
    variables against FP64, within the call's own bound."""
    from oracle import ksg as oksg
    te, ctx = env
    rng = np.random.default_rng(N)
    s = rng.normal(size=(4, N)).astype(np.float32)
    s[1] += 0.3 * s[0] + 0.2 * s[2]
    data = te.te_data_create(ctx, s)
    got, err = te.cmi_gauss(ctx, data, [(0, 0)], [(1, 0)], [(2, 0), (3, 0)], max_lag=0, n_surr=5,
                            seed=8, stream_tag=1)
    v = s.astype(np.float64)
    logdet = lambda rows: np.linalg.slogdet(np.cov(rows))[1]
    for a in range(6):
        x = v[0] if a == 0 else v[0][oksg.permutation(8, 1, 0, 0, a, N)]
        ref = 0.5 * (logdet(np.array([x, v[2], v[3]])) + logdet(v[1:]) - logdet(v[2:])
                     - logdet(np.array([x, v[1], v[2], v[3]])))
        assert abs(got[a] - ref) <= err[a] + 1e-12
    data.close()


@pytest.mark.parametrize("T,dz,dx,S,k", [(300, 2, 1, 6, 4), (300, 0, 1, 3, 4), (300, 1, 2, 3, 5),
                                         (6000, 2, 1, 300, 4), (6000, 1, 1, 300, 4),
                                         (9000, 2, 1, 900, 4)])
def test_static_entry_point_in_pieces(env, T, dz, dx, S, k):
    """The allocation-free call keeps the lists of as many points as its scratch
    has left: all of them, a few pieces, or (last) too few, where the
    member-lane kernel serves the call."""
    torch = pytest.importorskip("torch")
    te, ctx = env
    s = np.asarray(synth.workload_var10(T=T, seed=3)["series"], dtype=np.float32)
    data = te.te_data_create(ctx, s)
    dev = torch.from_numpy(s).cuda()
    kw = dict(k=k, max_lag=5, n_surr=S, seed=7, stream_tag=2, return_keys=True)
    x = [(2, 1 + a) for a in range(dx)]
    _, ref = te.cmi_ksg(ctx, data, x, [(0, 0)], Z[:dz], **kw)
    _, got = te.cmi_ksg_static(dev, x, [(0, 0)], Z[:dz], **kw)
    assert got == ref
    data.close()


@pytest.mark.parametrize("T,dz,dx,k,w,S,levels", [
    (38, 2, 1, 4, 0, 2, 0), (505, 0, 1, 4, 3, 9, 0), (505, 1, 1, 12, 0, 9, 0),
    (1500, 2, 1, 4, 0, 33, 0), (1500, 3, 2, 4, 5, 9, 0), (1500, 1, 4, 16, 0, 9, 0),
    (2600, 2, 1, 4, 0, 400, 7), (2600, 1, 1, 4, 0, 400, 300)])
def test_pairs_beyond_the_radii(env, T, dz, dx, k, w, S, levels):
    """Heavy tails (and, with levels, ties) put many pairs beyond their lists'
    radii: fewer than a batch of the scan and more, more than a CTA can put
    aside, and with more distances up to the bound than a pair can keep."""
    te, ctx = env
    rng = np.random.default_rng(T + dz)
    s = rng.standard_cauchy(size=(10, T)).astype(np.float32)
    if levels:
        s = np.clip(np.round(s * levels / 20), -levels, levels).astype(np.float32)
    data = te.te_data_create(ctx, s)
    jobs = [te.Job(data, [(2, 1 + a) for a in range(dx)], [(0, 0)], Z[:dz], k=k, theiler=w,
                   max_lag=5, n_surr=S, seed=3)]
    got, ref = _both(te, ctx, jobs)
    assert got == ref
    data.close()


@pytest.mark.parametrize("levels", [2, 3])
def test_member_lane_kernel_with_distances_of_zero(env, levels):
    """Empty Z and k-th distances of 0: nothing is below them, in either kernel."""
    te, ctx = env
    rng = np.random.default_rng(levels)
    s = rng.integers(0, levels, size=(3, 300)).astype(np.float32)
    data = te.te_data_create(ctx, s)
    jobs = [te.Job(data, [(2, 1)], [(0, 0)], [], k=4, max_lag=5, n_surr=5, seed=1)]
    got, ref = _both(te, ctx, jobs)
    assert got == ref
    data.close()


@pytest.mark.parametrize("dz,w", [(0, 0), (0, 3), (1, 0), (1, 3), (2, 0)])
def test_static_entry_point_with_values_that_are_not_finite(env, dz, w):
    """The allocation-free call gets a device pointer that no host check has
    read: with single and whole-column values that are not finite, in X, Y and Z,
    its keys are the member-lane kernel's (which serves the same members
    among so many surrogates that the scratch has no room for lists), and the
    next call is as good as one before."""
    torch = pytest.importorskip("torch")
    te, ctx = env
    T, many = 3300, 2500
    s = np.asarray(synth.workload_var10(T=T, seed=5)["series"], dtype=np.float32)
    dev = torch.from_numpy(s).cuda()
    kw = dict(k=4, theiler=w, max_lag=5, seed=7, return_keys=True)
    call = lambda d, n: te.cmi_ksg_static(d, [(2, 1)], [(0, 0)], Z[:dz], n_surr=n, **kw)[1]
    ref = call(dev, 3)
    assert call(dev, many)[:4] == ref
    for proc in [2, 0] + ([4] if dz > 1 else []):
        for value in (np.nan, np.inf, -np.inf):
            for where in (slice(1700, 1701), slice(0, T)):
                bad = torch.from_numpy(s.copy())
                bad[proc, where] = value
                bad = bad.cuda()
                assert call(bad, 3) == call(bad, many)[:4]
    assert call(dev, 3) == ref


@pytest.mark.parametrize("T,n_groups,S", [(360, 70, 3), (1005, 30, 20), (3005, 12, 20)])
def test_batches_whose_groups_take_both_paths(env, T, n_groups, S):
    """One batch of many groups: of few members over zero to five Z variables,
    of 201 members, of several X variables with and without Z, and (at the
    longest) of an X block past a CTA's shared memory.  Some take lists, some
    the member-lane or the fused kernel; the keys are those of the latter."""
    te, ctx = env
    s = np.asarray(synth.workload_var10(T=T, seed=T)["series"], dtype=np.float32)
    data = te.te_data_create(ctx, s)
    jobs = []
    for g in range(n_groups):
        y = [(g % 10, g // 10 % 5)] + ([((g + 1) % 10, 5)] if g >= 50 else [])
        z = [((g + 1 + d) % 10, 1 + d) for d in range(g % 6 if g % 6 < 5 else 0)]
        jobs.append(te.Job(data, [((g + 7) % 10, 1 + g % 4)], y, z, k=4, max_lag=5, n_surr=S,
                           seed=3, stream_tag=g % 3))
    for a, (dx, dz, surr) in enumerate([(1, 2, 200), (1, 0, 200), (3, 0, 70), (4, 2, 12),
                                        (16, 1, 9)]):
        jobs.append(te.Job(data, [(a, 1 + d % 5) if d < 5 else (a + 1 + d % 4, 5) for d in range(dx)],
                           [(a, 0)], Z[:dz], k=4, max_lag=5, n_surr=surr, seed=3))
    got, ref = _both(te, ctx, jobs)
    assert got == ref
    data.close()


@pytest.mark.parametrize("k", [1, 3, 8, 9, 16])
def test_batches_of_another_k_take_both_paths(env, k):
    """As above with k other than 4, whose lines lie elsewhere: many groups of
    5 and of 21 over zero, two and three Z variables, and several X variables
    with few and many members."""
    te, ctx = env
    T = 3805
    s = np.asarray(synth.workload_var10(T=T, seed=k)["series"], dtype=np.float32)
    data = te.te_data_create(ctx, s)
    kw = dict(k=k, max_lag=5, seed=3)
    jobs = [te.Job(data, [((g + 7) % 10, 2)], [(g % 10, g // 10)],
                   [((g + 1 + d) % 10, 1 + d) for d in range((0, 2, 3)[g % 3])],
                   n_surr=4 if g % 2 else 20, **kw) for g in range(18)]
    jobs += [te.Job(data, [(a, 1 + a % 5) for a in range(dx)], [(0, 0)], Z[:dz], n_surr=S, **kw)
             for dx, dz, S in ((2, 0, 11), (3, 0, 63), (3, 1, 20), (4, 1, 70))]
    got, ref = _both(te, ctx, jobs)
    assert got == ref
    data.close()


def _series(kind, T, seed=0):
    rng = np.random.default_rng(seed)
    if kind == "cauchy":
        s = rng.standard_cauchy(size=(10, T))
    elif kind == "ties":
        s = np.clip(np.round(rng.standard_cauchy(size=(10, T)) * 7 / 20), -7, 7)
    elif kind == "binary":
        s = rng.integers(0, 2, size=(10, T))
    else:   # most values zero
        s = np.where(rng.random((10, T)) < 0.7, 0.0, rng.exponential(size=(10, T)))
    return np.asarray(s, dtype=np.float32)


@pytest.mark.parametrize("kind,T,dz,dx,k,w,S", [
    ("cauchy", 38, 2, 1, 4, 0, 2), ("cauchy", 1500, 2, 1, 4, 0, 33), ("cauchy", 1500, 3, 2, 4, 5, 9),
    ("cauchy", 1500, 1, 4, 16, 0, 9), ("ties", 2600, 2, 1, 4, 0, 400), ("binary", 2600, 0, 1, 4, 0, 9),
    ("binary", 1200, 8, 1, 4, 0, 60), ("binary", 1200, 8, 3, 4, 0, 9), ("zero", 2600, 1, 1, 4, 2, 40),
    ("zero", 1200, 0, 2, 9, 0, 9)])
def test_pairs_beyond_the_radii_scanned_or_handed_over(env, kind, T, dz, dx, k, w, S):
    """Data that leave many pairs beyond their lists: scanned by the walk when
    nothing is handed over, otherwise given up and evaluated anew; one call,
    its per-point values, a batch beside ordinary groups, and as a graph."""
    te, ctx = env
    data = te.te_data_create(ctx, _series(kind, T))
    plain = te.te_data_create(ctx, synth.workload_var10(T=T, seed=3)["series"])
    x, kw = [(2, 1 + a) for a in range(dx)], dict(k=k, theiler=w, max_lag=5, seed=3)
    jobs = [te.Job(data, x, [(0, 0)], Z[:dz], n_surr=S, **kw),
            te.Job(plain, [(3, 1)], [(0, 0)], Z[:2], n_surr=7, **kw),
            te.Job(data, [(1, 2)], [(0, 0)], [(5, 1), (6, 2), (7, 3)], n_surr=2, **kw)]
    got, ref = _both(te, ctx, jobs)
    assert got == ref
    one = te.cmi_ksg(ctx, data, x, [(0, 0)], Z[:dz], n_surr=S, return_keys=True, **kw)[1]
    assert one == ref[0]
    dbg = te.cmi_ksg_debug(ctx, data, x, [(0, 0)], Z[:dz], n_surr=S, member=S // 2, **kw)
    try:
        for name in ("ksg_lists", "graph"):
            ctx.set_option(name, 1)
            assert te.cmi_ksg_batch(ctx, jobs, return_keys=True)[1] == ref
            if name == "ksg_lists":   # the scans' own per-point values
                own = te.cmi_ksg_debug(ctx, data, x, [(0, 0)], Z[:dz], n_surr=S, member=S // 2, **kw)
            ctx.set_option(name, 0)
    finally:
        ctx.set_option("ksg_lists", 0)
        ctx.set_option("graph", 0)
    for name in ("eps", "n_xz", "n_yz") + (("n_z",) if dz else ()):
        np.testing.assert_array_equal(dbg[name], own[name])
    data.close()
    plain.close()


@pytest.mark.parametrize("kind,T,dz,S", [("zero", 2600, 1, 90), ("binary", 1200, 8, 60),
                                         ("cauchy", 2600, 8, 90)])
def test_served_and_allocation_free_calls_hand_over(env, kind, T, dz, S):
    """Groups that the list walk gives up, in served batches beside others and
    in the allocation-free call: keys as everywhere."""
    torch = pytest.importorskip("torch")
    te, ctx = env
    s = _series(kind, T)
    data = te.te_data_create(ctx, s)
    plain = te.te_data_create(ctx, synth.workload_var10(T=T, seed=3)["series"])
    jobs = [te.Job(d, [(2 + a, 1)], [(0, 0)], Z[:dz], k=4, max_lag=5, n_surr=S, seed=a)
            for a in range(3) for d in (data, plain)]
    _, ref = _both(te, ctx, jobs)
    for _ in range(2):
        tickets = [te.te_serve_submit(ctx, j) for j in jobs]
        for t, j, r in zip(tickets, jobs, ref):
            assert te.te_serve_poll(ctx, t, j.n_surr, return_keys=True)[1] == r
    te.te_serve_stop(ctx)
    got = te.cmi_ksg_static(torch.from_numpy(s).cuda(), jobs[0].x, [(0, 0)], Z[:dz], k=4,
                            max_lag=5, n_surr=S, seed=0, return_keys=True)[1]
    assert got == ref[0]
    data.close()
    plain.close()


@pytest.mark.parametrize("dz,dx,w", [(8, 1, 0), (8, 1, 3), (0, 2, 0), (0, 2, 5)])
def test_work_counters_include_scans_over_all_points(env, dz, dx, w):
    """Binary values: with eight Z variables two points in 1100 share a query
    point's (Y, Z) and the rest are tied at one, so that lists end before k
    neighbours and every pair scans every point; over an empty Z a count of several X variables visits every point: at
    least one evaluation a point for each pair, no more than two scans."""
    te, ctx = env
    N, S = 1100, 4
    data = te.te_data_create(ctx, _series("binary", N + 5))
    x = [(2, 1 + a) for a in range(dx)]
    try:
        ctx.set_option("ksg_lists", 1)
        before = ctx.stats()
        te.cmi_ksg(ctx, data, x, [(0, 0)], Z[:dz], k=4, theiler=w, max_lag=5, n_surr=S)
        after = ctx.stats()
    finally:
        ctx.set_option("ksg_lists", 0)
    evals, ops = (after[n] - before[n] for n in ("pair_evals", "ksg_ops"))
    pairs = (S + 1) * N
    assert pairs * (N - 2 * w - 1) <= evals <= 5 * pairs * N
    assert 3 * evals <= ops <= 7 * evals
    data.close()
