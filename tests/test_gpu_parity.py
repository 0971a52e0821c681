"""CUDA path vs the CPU oracle: stage arrays element by element, heights bit-exact, full-size sampled checks.

Every test here calls libqfs through its C ABI (via the ctypes binding) on cuda:0.
"""
import numpy as np
import pytest
import torch

import oracle
from helpers import example_quartics
from paper_2502_12428_gb300 import inputs

pytestmark = pytest.mark.gpu

CORE_FORMS = ["int32", "dp4a", "int8tc"]


@pytest.fixture(scope="session")
def qfs():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2502_12428_gb300 import build
    build.build()
    import paper_2502_12428_gb300.qfs as q
    return q


def dev_tensor(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")


def gpu_heights(qfs, p, f, **kw):
    return qfs.heights(p, dev_tensor(f), **kw).cpu().numpy()


def find_rows(p, n, seed, want, count, gen=inputs.dense):
    f = gen(p, n, seed)
    h = oracle.heights(p, f)
    idx = [i for i in range(n) if want(h[i])][:count]
    return f[idx], h[idx]


# ------------------------------------------------------------------------------------- stage arrays
def check_stages(qfs, p, f, form, max_h=10):
    ref = oracle.stage_arrays_a(p, f, max_h=max_h)
    got = qfs.debug_stages(p, dev_tensor(f), max_h=max_h, form=form)
    assert got["h"] == ref["h"]
    assert np.array_equal(got["g"].cpu().numpy(), ref["g"]), "f^(p-1) mod p"
    if ref["h"] != 1:
        assert np.array_equal(got["G"].cpu().numpy(), ref["D"]), "lift(g)^p mod p^2"
        assert np.array_equal(got["delta"].cpu().numpy(), ref["delta"]), "Delta_1(f^(p-1))"
        rows = ref["iters"].shape[0]
        assert np.array_equal(got["iters"].cpu().numpy()[:rows], ref["iters"]), "theta iterates"
    return ref["h"]


@pytest.mark.parametrize("form", CORE_FORMS)
def test_stages_p3(qfs, form):
    f = np.concatenate([inputs.dense(3, 10, 301), inputs.sparse(3, 4, 302), inputs.fermat()[None]])
    hs = [check_stages(qfs, 3, row, form) for row in f]
    assert any(h != 1 for h in hs)


@pytest.mark.parametrize("form", CORE_FORMS)
def test_stages_p5(qfs, form):
    f, h = find_rows(5, 400, 501, lambda x: x >= 2 or x == 0, 5)
    ex = [r[3] for r in example_quartics() if r[0] == 5 and r[1] in (1, 3, 0)]
    for row in list(f) + ex:
        check_stages(qfs, 5, row, form)


def _route_a_parallel(p, rows):
    # route A releases the interpreter while it runs (ctypes), so one thread per quartic runs them side by side
    from concurrent.futures import ThreadPoolExecutor
    with ThreadPoolExecutor(max_workers=len(rows)) as ex:
        return list(ex.map(lambda r: oracle.stage_arrays_a(p, r), rows))


@pytest.mark.slow
def test_stages_p7(qfs):
    # Figure 5's rows of height 2, 3 and infinity and a sparse quartic of height >= 3, every form, every array
    ex = {r[1]: r[3] for r in example_quartics() if r[0] == 7}
    fs, hs = find_rows(7, 3000, 7070, lambda x: x >= 3, 1, gen=inputs.sparse)
    rows = [ex[2], ex[3], ex[0], fs[0]]
    refs = _route_a_parallel(7, rows)
    assert [r["h"] for r in refs[:3]] == [2, 3, 0] and refs[3]["h"] >= 3
    for row, ref in zip(rows, refs):
        for form in CORE_FORMS:
            got = qfs.debug_stages(7, dev_tensor(row), form=form)
            assert got["h"] == ref["h"]
            assert np.array_equal(got["g"].cpu().numpy(), ref["g"])
            assert np.array_equal(got["G"].cpu().numpy(), ref["D"])
            assert np.array_equal(got["delta"].cpu().numpy(), ref["delta"])
            n_it = ref["iters"].shape[0]
            assert n_it >= 1
            assert np.array_equal(got["iters"].cpu().numpy()[:n_it], ref["iters"])


@pytest.mark.slow
def test_stages_p11(qfs):
    # Figure 6's row of height 2 at p = 11 (per-CTA buffers above 15 MB): g, G and Delta against the oracle's stage
    # arrays with D formed by products with f (equal to route A's lift(g)^p, pinned on CPU), the iterate against
    # route R (equal to route A's iterates, pinned on CPU)
    row = next(r[3] for r in example_quartics() if r[0] == 11 and r[1] == 2)
    ref = oracle.stage_arrays_fchain(11, row)
    it = oracle.stage_arrays_r(11, row)
    assert not ref["h1"] and it["h"] == 2
    for form in CORE_FORMS:
        got = qfs.debug_stages(11, dev_tensor(row), form=form)
        assert got["h"] == 2
        assert np.array_equal(got["g"].cpu().numpy(), ref["g"])
        assert np.array_equal(got["G"].cpu().numpy(), ref["D"])
        assert np.array_equal(got["delta"].cpu().numpy(), ref["delta"])
        assert np.array_equal(got["iters"].cpu().numpy()[:1], it["iters"])


def _edge_quartics(p):
    """x4^4 plus each other monomial in turn (one tap beside tap (4, 4, 4): every tap position of the products'
    windows), every coefficient p - 1 (the largest sums), and two taps at the ends of one window."""
    rows = []
    for k in range(34):
        f = np.zeros(35, np.uint8)
        f[k], f[34] = p - 1, 1
        rows.append(f)
    rows.append(np.full(35, p - 1, np.uint8))
    f = np.zeros(35, np.uint8)
    f[30], f[34] = p - 1, p - 1
    rows.append(f)
    return rows


@pytest.mark.parametrize("p,step", [(3, 1), (5, 5), (7, 12)])
def test_dp4a_product_tap_positions(qfs, p, step):
    # G = f~^(p(p-1)) mod p^2 and Delta element by element, on quartics whose taps sit alone in the dp4a windows
    rows = _edge_quartics(p)
    rows = rows[:-2:step] + rows[-2:]
    seen = 0
    for f in rows:
        ref = oracle.stage_arrays_fchain(p, f)
        got = qfs.debug_stages(p, dev_tensor(f), max_h=2)
        assert np.array_equal(got["g"].cpu().numpy(), ref["g"])
        if got["h"] != 1:
            seen += 1
            assert np.array_equal(got["G"].cpu().numpy(), ref["D"])
            assert np.array_equal(got["delta"].cpu().numpy(), ref["delta"])
    assert seen >= len(rows) // 2
    assert qfs.read_status() == 0


@pytest.mark.parametrize("p", [3, 5, 7, 11, 13])
def test_dp4a_small_products(qfs, p):
    # f^(p-1) mod p by the products up to degree 4(p - 1), element by element, on quartics whose taps sit alone in the dp4a
    # windows and on random ones; and f~^p mod p^2 by the identity and reduced modes' heights
    def power(f, n):
        form = {m: int(c) for m, c in zip(oracle.form_monomials(4), f) if c}
        side = 4 * n + 1
        out = np.zeros((side,) * 3, np.int64)
        out[0, 0, 0] = 1
        for _ in range(n):
            prev, out = out, np.zeros_like(out)
            for (_, a, b, c), v in form.items():
                out[a:, b:, c:] += v * prev[:side - a, :side - b, :side - c]
            out %= p
        return np.array([out[e[1:]] for e in oracle.form_monomials(4 * n)])
    rows = _edge_quartics(p)[::3] + list(inputs.dense(p, 4, 9300 + p))
    for f in rows:
        got = qfs.debug_stages(p, dev_tensor(f), max_h=2, power="reduced")
        assert np.array_equal(got["g"].cpu().numpy(), power(f, p - 1))
    assert np.array_equal(gpu_heights(qfs, p, np.stack(rows), power="reduced"), oracle.heights(p, np.stack(rows)))
    if p >= 11:   # a light prime in the same launch: its own strips, and the first prime's again
        other = inputs.sparse(5, 50, 9310)
        outs = qfs.heights_multi([(5, dev_tensor(other), None), (p, dev_tensor(np.stack(rows)), None)], power="reduced")
        assert np.array_equal(outs[0].cpu().numpy(), oracle.heights(5, other))
        assert np.array_equal(outs[1].cpu().numpy(), oracle.heights(p, np.stack(rows)))
    assert qfs.read_status() == 0


# ------------------------------------------------------------------------------------- heights, small sets
@pytest.mark.parametrize("form", CORE_FORMS)
def test_heights_p3_64_plus_fermat(qfs, form):
    f = np.concatenate([inputs.dense(3, 64, inputs.config_seed(1)), inputs.fermat()[None]])
    want = oracle.heights(3, f, route=oracle.ROUTE_A)
    got = gpu_heights(qfs, 3, f, form=form)
    assert np.array_equal(got, want)
    assert got[-1] == 0  # Fermat quartic at p = 3: infinity


@pytest.mark.parametrize("form", CORE_FORMS)
def test_heights_paper_examples(qfs, form):
    rows = example_quartics()
    for p in (5, 7, 11, 13):
        sel = [r for r in rows if r[0] == p]
        f = np.stack([r[3] for r in sel])
        want = np.array([r[1] for r in sel], np.int8)
        assert np.array_equal(gpu_heights(qfs, p, f, form=form), want), f"p={p}"


@pytest.mark.parametrize("p,n", [(3, 2000), (5, 4096), (7, 1024), (11, 48)])
def test_heights_random_dense_and_sparse(qfs, p, n):
    f = np.concatenate([inputs.dense(p, n, 900 + p), inputs.sparse(p, n, 950 + p)])
    want = oracle.heights(p, f)
    for form in CORE_FORMS:
        assert np.array_equal(gpu_heights(qfs, p, f, form=form), want), form


def test_route_a_subset_p5(qfs):
    f = inputs.dense(5, 300, 1234)
    want = oracle.heights(5, f, route=oracle.ROUTE_A)
    assert np.array_equal(gpu_heights(qfs, 5, f), want)


# ------------------------------------------------------------------------------------- mixed primes in one launch
def test_multi_group_mixed_and_pgl4(qfs):
    groups, wants, pairs = [], [], []
    for p, n in [(5, 2048), (7, 1024), (11, 32)]:
        f = inputs.dense(p, n, 7700 + p)
        A = inputs.pgl4_matrices(p, n, 7800 + p)
        g = inputs.substitute(f, A, p)
        both = np.concatenate([f, g])
        groups.append((p, dev_tensor(both), None))
        wants.append(oracle.heights(p, both))
        pairs.append(n)
    outs = [o.cpu().numpy() for o in qfs.heights_multi(groups)]
    for out, want, n in zip(outs, wants, pairs):
        assert np.array_equal(out, want)
        assert np.array_equal(out[:n], out[n:])  # PGL_4 invariance of the height
    # one launch equals separate launches
    for (p, t, _), out in zip(groups, outs):
        assert np.array_equal(qfs.heights(p, t).cpu().numpy(), out)


def test_multi_group_with_empty_groups(qfs):
    # empty groups take no part in the launch; a call whose groups are all empty enqueues nothing
    f = inputs.dense(7, 300, 7900)
    empty = torch.zeros(0, 35, dtype=torch.uint8, device="cuda:0")
    outs = qfs.heights_multi([(5, empty, None), (7, dev_tensor(f), None), (11, empty, None)])
    assert outs[0].numel() == 0 and outs[2].numel() == 0
    assert np.array_equal(outs[1].cpu().numpy(), oracle.heights(7, f))
    outs = qfs.heights_multi([(5, empty, None), (7, empty, None)])
    assert all(o.numel() == 0 for o in outs)


# ------------------------------------------------------------------------------------- crews of CTAs
@pytest.mark.parametrize("p,n,pool", [(7, 1, 60), (7, 3, 60), (7, 40, 600), (11, 2, 60), (13, 1, 60)])
def test_few_quartics_run_by_crews_of_ctas(qfs, p, n, pool):
    # few quartics: clusters of CTAs split the products and the theta steps of each; every repetition splits
    # them differently; the caps leave one CTA per quartic
    f, h = find_rows(p, pool, 9700 + p, lambda x: x != 1, n)
    assert len(f) == n
    t = dev_tensor(f)
    for kw in [{}] * (6 if p == 7 else 2) + [{"max_ctas": 1}, {"max_ctas": 5}, {"ctas_per_sm": 1}]:
        if p == 13 and kw.get("max_ctas") == 1:
            continue
        assert np.array_equal(gpu_heights(qfs, p, f, **kw), h)
    assert qfs.read_status() == 0
    # a captured launch replays
    out = torch.empty(n, dtype=torch.int8, device="cuda:0")
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        qfs.heights(p, t, out=out)
    for _ in range(2):
        out.fill_(-5)
        g.replay()
        torch.cuda.synchronize()
        assert np.array_equal(out.cpu().numpy(), h)


def test_theta_matrix_by_crews_repeats(qfs):
    f = dev_tensor(np.concatenate([inputs.dense(7, 3, 9800), inputs.sparse(7, 2, 9801)]))
    ref = qfs.theta_matrix(7, f).cpu().numpy()
    assert np.array_equal(ref[4], oracle.theta_matrix(7, f[4].cpu().numpy()))
    for _ in range(4):
        assert np.array_equal(qfs.theta_matrix(7, f).cpu().numpy(), ref)
    assert np.array_equal(qfs.theta_matrix(7, f[:1]).cpu().numpy(), ref[:1])
    assert qfs.read_status() == 0


def _ms(fn, reps=5):
    """Milliseconds of fn() on the current stream, the least of `reps` passes after a first one."""
    best = float("inf")
    for i in range(reps + 1):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        fn()
        b.record()
        b.synchronize()
        if i:
            best = min(best, a.elapsed_time(b))
    return best


@pytest.mark.parametrize("p,n,big,past,limit", [(5, 30000, 11, False, 1.3), (5, 30000, 13, False, 1.3),
                                                (3, 60000, 7, False, 1.3), (3, 60000, 7, True, 2.0)])
def test_one_heavy_row_does_not_slow_a_mixed_launch(qfs, p, n, big, past, limit):
    # many light quartics beside one row of a large prime: the crews serve that row only, and only if it is past height 1
    # (then the launch takes as long as the row does on one CTA or a crew: 4.4 ms at most at p = 7, beside 3.5 ms)
    f, _ = find_rows(big, 60, 9760 + big, lambda x: (x != 1) == past, 1)
    light, heavy = dev_tensor(inputs.dense(p, n, 9750 + p)), dev_tensor(f)
    out, out2 = (torch.empty(k, dtype=torch.int8, device="cuda:0") for k in (n, 1))
    alone = _ms(lambda: qfs.heights(p, light, out=out))
    want, want2 = out.clone(), qfs.heights(big, heavy)
    mixed = _ms(lambda: qfs.heights_multi([(p, light, out), (big, heavy, out2)]))
    assert torch.equal(out, want) and torch.equal(out2, want2)
    assert mixed < limit * alone, (mixed, alone)
    assert qfs.read_status() == 0


@pytest.mark.parametrize("power", ["chain", "identity", "reduced"])
def test_several_groups_of_several_primes(qfs, power):
    # lists of survivors group by group: groups of one prime, empty ones, rows that are all height 1, invalid rows
    groups = []
    for p, n, gen in [(3, 900, inputs.sparse), (7, 40, inputs.dense), (5, 333, inputs.dense), (7, 1, inputs.sparse),
                      (3, 1, inputs.dense), (11, 12, inputs.dense), (5, 70, inputs.sparse)]:
        groups.append((p, gen(p, n, 9770 + n)))
    groups[2][1][5, 0] = 5
    groups.append((7, groups[1][1][oracle.heights(7, groups[1][1]) == 1]))
    outs = qfs.heights_multi([(p, dev_tensor(f), None) for p, f in groups], power=power)
    for (p, f), o in zip(groups, outs):
        assert np.array_equal(o.cpu().numpy(), oracle.heights(p, f)), p
    one = [g for g in groups if g[0] == 7]
    for (p, f), o in zip(one, qfs.heights_multi([(p, dev_tensor(f), None) for p, f in one], power=power)):
        assert np.array_equal(o.cpu().numpy(), oracle.heights(p, f))
    assert qfs.read_status() == 0


@pytest.mark.parametrize("p,n,m,k", [(11, 70, 300, 513), (251, 130, 257, 129)])
def test_matmul_mod_captured(qfs, p, n, m, k):
    # the product starts while the pack runs, also when replayed: every replay sees the operands of that moment
    rng = np.random.default_rng(p)
    A, B = (dev_tensor(rng.integers(0, p, s).astype(np.uint8)) for s in ((n, k), (k, m)))
    out = qfs.matmul_mod(p, A, B)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        qfs.matmul_mod(p, A, B, out=out)
    for _ in range(3):
        A.copy_(dev_tensor(rng.integers(0, p, (n, k)).astype(np.uint8)))
        g.replay()
        torch.cuda.synchronize()
        assert np.array_equal(out.cpu().numpy(), oracle.matmul_mod(p, A.cpu().numpy(), B.cpu().numpy()))
    assert qfs.read_status() == 0


# ------------------------------------------------------------------------------------- theta by rows
@pytest.mark.parametrize("p,n", [(3, 4000), (5, 6000)])
@pytest.mark.parametrize("form", CORE_FORMS)
def test_theta_by_rows_many_steps(qfs, p, n, form):
    # sparse quartics run up to nine theta steps; a workspace budget without room for the classes takes theta by cubes,
    # with the same heights
    f = inputs.sparse(p, n, 9900 + p)
    want = oracle.heights(p, f)
    assert len(set(want.tolist())) >= 5 and (want > 3).any()
    t = dev_tensor(f)
    assert np.array_equal(qfs.heights(p, t, form=form).cpu().numpy(), want)
    assert np.array_equal(qfs.heights(p, t, form=form, workspace_budget=1 << 20).cpu().numpy(), want)
    assert qfs.read_status() == 0


@pytest.mark.parametrize("p,n", [(3, 1), (3, 5000), (5, 1), (5, 130), (5, 140), (5, 3000)])
def test_noalloc_theta_by_rows_and_by_cubes(qfs, p, n):
    # in the fixed 64 MiB: classes by rows where every CTA's fit (p = 3; p = 5 up to about 136 quartics), cubes otherwise
    f = inputs.sparse(p, n, 9950 + p)
    want = oracle.heights(p, f)
    t = dev_tensor(f)
    for _ in range(2):
        assert np.array_equal(qfs.heights_noalloc(p, t).cpu().numpy(), want)
    assert qfs.read_status() == 0


@pytest.mark.parametrize("p,n", [(3, 3000), (5, 4000), (7, 600)])
@pytest.mark.parametrize("form", CORE_FORMS)
def test_identity_theta_by_rows(qfs, p, n, form):
    # the identity mode forms its classes by rows, with and without room for them; sparse quartics need many steps
    f = np.concatenate([inputs.dense(p, n // 2, 9920 + p), inputs.sparse(p, n // 2, 9930 + p)])
    want = oracle.heights(p, f)
    t = dev_tensor(f)
    for budget in (0, 8 << 20):
        got = qfs.heights(p, t, form=form, power="identity", workspace_budget=budget).cpu().numpy()
        assert np.array_equal(got, want), budget
    assert qfs.read_status() == 0


@pytest.mark.parametrize("p,power", [(5, "chain"), (7, "identity")])
def test_classes_first_needed_in_a_capture(qfs, p, power):
    # the workspace is prepared, the classes' buffer is not there yet: the first call is a captured one
    f = inputs.dense(p, 300, 9940 + p)
    t = dev_tensor(f)
    out = torch.empty(300, dtype=torch.int8, device="cuda:0")
    qfs.shutdown()
    qfs.plan_prepare(7, 300)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        qfs.heights(p, t, out=out, power=power)
    g.replay()
    torch.cuda.synchronize()
    assert np.array_equal(out.cpu().numpy(), oracle.heights(p, f))


# ------------------------------------------------------------------------------------- edge cases and errors
def test_edge_cases(qfs):
    p = 5
    assert qfs.heights(p, torch.zeros(0, 35, dtype=torch.uint8, device="cuda:0")).numel() == 0
    f = inputs.dense(p, 1000, 4242)
    bad = f.copy()
    bad[3, 0] = p
    bad[500, 34] = 255
    got = gpu_heights(qfs, p, bad)
    want = oracle.heights(p, f)
    assert got[3] == -1 and got[500] == -1
    keep = np.ones(1000, bool)
    keep[[3, 500]] = False
    assert np.array_equal(got[keep], want[keep])
    for n in (1, 7, 153):
        assert np.array_equal(gpu_heights(qfs, p, f[:n]), want[:n])
    # max_h caps: with max_h = 1 only the Fedder test runs
    h1 = gpu_heights(qfs, p, f, max_h=1)
    assert np.array_equal(h1, np.where(want == 1, 1, 0).astype(np.int8))
    h3 = gpu_heights(qfs, p, f, max_h=3)
    assert np.array_equal(h3, np.where((want >= 1) & (want <= 3), want, 0).astype(np.int8))
    # the all-zero form: f^(p-1) = 0, every iterate is zero -> infinity
    assert gpu_heights(qfs, p, np.zeros((1, 35), np.uint8))[0] == oracle.height_a(p, np.zeros(35, np.uint8)) == 0


def test_error_codes(qfs):
    t = dev_tensor(inputs.dense(5, 4, 1))
    with pytest.raises(qfs.QfsError) as e:
        qfs.heights(4, t)
    assert e.value.status == 1
    with pytest.raises(qfs.QfsError) as e:
        qfs.heights(5, t, max_h=11)
    assert e.value.status == 2
    with pytest.raises(qfs.QfsError) as e:
        qfs.heights(5, t, form=9)
    assert e.value.status == 7


def test_determinism_across_cta_counts(qfs):
    p = 7
    f = inputs.dense(p, 3000, 5151)
    t = dev_tensor(f)
    ref = qfs.heights(p, t).cpu().numpy()
    for cap in (1, 3, 37):
        assert np.array_equal(qfs.heights(p, t, max_ctas=cap).cpu().numpy(), ref)
    assert np.array_equal(ref, oracle.heights(p, f))


def test_device_status_clean(qfs):
    assert qfs.read_status() == 0


# ------------------------------------------------------------------------------------- height-1 screen
def test_screen_settles_whole_batches(qfs):
    # a batch that the screen settles entirely leaves the persistent launch with no survivors
    p = 5
    f, h = find_rows(p, 600, 6100, lambda x: x == 1, 300)
    qfs.read_stats()
    assert np.array_equal(gpu_heights(qfs, p, f), h)
    assert qfs.read_stats()[0] == 0
    bad = f.copy()
    bad[:, 7] = p
    assert (gpu_heights(qfs, p, bad) == -1).all()
    assert qfs.read_stats()[0] == 0
    # and a batch with no height-1 row at all: every row reaches the persistent launch
    g, hg = find_rows(p, 2000, 6150, lambda x: x != 1, 120)
    assert np.array_equal(gpu_heights(qfs, p, g), hg)
    assert qfs.read_stats()[0] == len(g)


def test_screen_survivor_count_matches_oracle(qfs):
    p = 7
    f = inputs.dense(p, 1500, 6200)
    want = oracle.heights(p, f)
    qfs.read_stats()
    assert np.array_equal(gpu_heights(qfs, p, f), want)
    assert qfs.read_stats()[0] == int((want != 1).sum())


@pytest.mark.parametrize("p", [3, 11, 13])
def test_screen_fedder_decision(qfs, p):
    # with max_h = 1 only the height-1 test decides a row: F = f^((p-1)/2) takes 0, 4 and 5 products in the warp
    f = np.concatenate([inputs.dense(p, 1200, 6300 + p), inputs.sparse(p, 400, 6400 + p)])
    want = oracle.heights(p, f, max_h=1)
    assert np.array_equal(gpu_heights(qfs, p, f, max_h=1), want)


# ------------------------------------------------------------------------------------- staged engine
@pytest.mark.parametrize("p,n", [(3, 500), (5, 3000), (7, 600)])
def test_staged_engine_matches_fused_and_oracle(qfs, p, n):
    f = np.concatenate([inputs.dense(p, n, 9100 + p), inputs.sparse(p, n // 2, 9200 + p)])
    bad = f.copy()
    bad[1, 3] = p
    t = dev_tensor(bad)
    fused = qfs.heights(p, t).cpu().numpy()
    staged = qfs.heights(p, t, engine="staged").cpu().numpy()
    assert np.array_equal(staged, fused)
    want = oracle.heights(p, f)
    want[1] = -1
    assert np.array_equal(staged, want)
    for max_h in (1, 3):
        assert np.array_equal(qfs.heights(p, t, engine="staged", max_h=max_h).cpu().numpy(),
                              qfs.heights(p, t, max_h=max_h).cpu().numpy())
    assert qfs.read_status() == 0


def test_staged_engine_small_chunks_and_multi(qfs):
    # a tiny workspace budget forces many chunks (admission by memory)
    f5 = inputs.dense(5, 5000, 9300)
    f7 = inputs.dense(7, 400, 9301)
    t5, t7 = dev_tensor(f5), dev_tensor(f7)
    outs = qfs.heights_multi([(5, t5, None), (7, t7, None)], engine="staged", workspace_budget=64 << 20)
    assert np.array_equal(outs[0].cpu().numpy(), oracle.heights(5, f5))
    assert np.array_equal(outs[1].cpu().numpy(), oracle.heights(7, f7))
    assert qfs.read_status() == 0


# ------------------------------------------------------------------------------------- identity power mode
@pytest.mark.parametrize("p,n", [(3, 6), (5, 6)])
def test_identity_power_stage_arrays(qfs, p, n):
    # the identity mode forms the same Delta_1(f^(p-1)) array as Algorithm 1, element by element
    f, h = find_rows(p, 400, 700 + p, lambda x: x >= 2 or x == 0, n)
    for row in f:
        ref = oracle.stage_arrays_a(p, row)
        for form in CORE_FORMS:
            got = qfs.debug_stages(p, dev_tensor(row), form=form, power="identity")
            assert got["h"] == ref["h"]
            assert np.array_equal(got["delta"].cpu().numpy(), ref["delta"]), form
            rows = ref["iters"].shape[0]
            assert np.array_equal(got["iters"].cpu().numpy()[:rows], ref["iters"]), form


@pytest.mark.parametrize("p,n", [(3, 1500), (5, 3000), (7, 800), (11, 24), (13, 6)])
def test_identity_power_heights(qfs, p, n):
    f = np.concatenate([inputs.dense(p, n, 7500 + p), inputs.sparse(p, n, 7600 + p)])
    t = dev_tensor(f)
    want = oracle.heights(p, f)
    for form in CORE_FORMS:
        assert np.array_equal(qfs.heights(p, t, form=form, power="identity").cpu().numpy(), want), form
    assert qfs.read_status() == 0


def test_identity_power_paper_examples(qfs):
    for p in (5, 7, 11, 13):
        sel = [r for r in example_quartics() if r[0] == p]
        f = np.stack([r[3] for r in sel])
        want = np.array([r[1] for r in sel], np.int8)
        assert np.array_equal(qfs.heights(p, dev_tensor(f), power="identity").cpu().numpy(), want), p


# ------------------------------------------------------------------------------------- tile autotuner, graphs
def test_tile_shapes_do_not_change_heights(qfs):
    p = 7
    f = inputs.dense(p, 1200, 6600)
    t = dev_tensor(f)
    want = oracle.heights(p, f)
    saved = qfs.tune_get(p)
    try:
        for rc, ring in [(256, 48 << 10), (1024, 80 << 10), (64, 32 << 10)]:
            qfs.tune_set(p, rc, ring)
            assert qfs.tune_get(p)["round_chunks"] == rc
            assert np.array_equal(qfs.heights(p, t).cpu().numpy(), want)
        with pytest.raises(qfs.QfsError):
            qfs.tune_set(p, 8, 48 << 10)
        best = qfs.autotune(p, t[:400])
        assert best["round_chunks"] >= 32 and best["ms"] > 0
        assert np.array_equal(qfs.heights(p, t).cpu().numpy(), want)
    finally:
        qfs.tune_set(p, saved["round_chunks"], saved["ring_bytes"])


@pytest.mark.parametrize("form", ["dp4a", "int32"])
def test_sweep_shapes_do_not_change_heights(qfs, form):
    # the swept chain's dense threshold decides, per quartic, between the every-pair two-slice loop and the
    # zero-pair-skipping one-slice loop; mixed dense and sparse rows take both paths under every threshold
    p = 5
    f = np.concatenate([inputs.dense(p, 700, 6610), inputs.sparse(p, 1300, 6611)])
    t = dev_tensor(f)
    want = oracle.heights(p, f)
    saved = qfs.sweep_tune_get(form, p)
    try:
        for dm, ctas in [(0, 2), (16, 1), (8, 0), (12, 1)]:
            qfs.sweep_tune_set(form, p, dm, ctas)
            assert qfs.sweep_tune_get(form, p) == {"dense_min": dm if dm else 12, "ctas_per_sm": ctas}
            assert np.array_equal(qfs.heights(p, t, form=form).cpu().numpy(), want)
        with pytest.raises(qfs.QfsError):
            qfs.sweep_tune_set(form, p, 17, 0)
        with pytest.raises(qfs.QfsError):
            qfs.sweep_tune_set("int8tc", p, 8, 0)
        best = qfs.sweep_autotune(p, t[:600], form=form)
        assert 0 <= best["dense_min"] <= 16 and best["ctas_per_sm"] >= 0 and best["ms"] > 0
        assert qfs.sweep_tune_get(form, p)["ctas_per_sm"] == best["ctas_per_sm"]
        assert np.array_equal(qfs.heights(p, t, form=form).cpu().numpy(), want)
    finally:
        qfs.sweep_tune_set(form, p, saved["dense_min"], saved["ctas_per_sm"])


def test_cuda_graph_capture_and_replay(qfs):
    # the call is stream-ordered and allocation-free once the workspace exists, so it can be captured
    p = 5
    a = inputs.dense(p, 3000, 6700)
    want = oracle.heights(p, a)
    coeffs = dev_tensor(a)
    out = torch.empty(3000, dtype=torch.int8, device="cuda:0")
    qfs.heights(p, coeffs, out=out)              # sizes the workspace before capture
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    out.zero_()
    with torch.cuda.graph(g):
        qfs.heights(p, coeffs, out=out)
    for _ in range(2):
        out.fill_(-5)
        g.replay()
        torch.cuda.synchronize()
        assert np.array_equal(out.cpu().numpy(), want)
    # new inputs in the same buffer replay through the same graph
    b = inputs.sparse(p, 3000, 6701)
    coeffs.copy_(torch.from_numpy(b))
    g.replay()
    torch.cuda.synchronize()
    assert np.array_equal(out.cpu().numpy(), oracle.heights(p, b))


# ------------------------------------------------------------------------------------- reduced theta mode
@pytest.mark.parametrize("p,n", [(3, 6), (5, 6), (7, 2)])
def test_reduced_mode_iterates(qfs, p, n):
    # the reduced step gives the same iterates g_h as u(Delta_1(f^(p-1)) g) (route A), element by element
    f, h = find_rows(p, 300, 800 + p, lambda x: x >= 2 or x == 0, n)
    for row in f:
        ref = oracle.stage_arrays_r(p, row)
        for form in CORE_FORMS:
            got = qfs.debug_stages(p, dev_tensor(row), form=form, power="reduced")
            assert got["h"] == ref["h"]
            rows = ref["iters"].shape[0]
            assert np.array_equal(got["iters"].cpu().numpy()[:rows], ref["iters"]), form


@pytest.mark.parametrize("p,n", [(3, 1500), (5, 4000), (7, 2000), (11, 200), (13, 60)])
def test_reduced_mode_heights(qfs, p, n):
    f = np.concatenate([inputs.dense(p, n, 8500 + p), inputs.sparse(p, n, 8600 + p)])
    t = dev_tensor(f)
    want = oracle.heights(p, f)
    for form in CORE_FORMS:
        assert np.array_equal(qfs.heights(p, t, form=form, power="reduced").cpu().numpy(), want), form
    for max_h in (1, 2, 4):
        assert np.array_equal(qfs.heights(p, t, power="reduced", max_h=max_h).cpu().numpy(),
                              oracle.heights(p, f, max_h=max_h))
    assert qfs.read_status() == 0


@pytest.mark.parametrize("p,n", [(3, 1), (3, 2000), (5, 1), (5, 2000), (7, 1), (7, 700)])
def test_reduced_kernel_and_general_route(qfs, p, n):
    # one prime <= 7 takes the kernel of its own; a cap on the CTAs, or another prime, the fused launch
    f = np.concatenate([inputs.dense(p, n, 9950 + p), inputs.sparse(p, n, 9960 + p)])
    f[n // 2, 3] = p
    want = oracle.heights(p, f)
    assert want[n // 2] == -1
    t = dev_tensor(f)
    for kw in ({}, {"max_ctas": 5}):
        assert np.array_equal(qfs.heights(p, t, power="reduced", **kw).cpu().numpy(), want), kw
    other = 5 if p == 7 else 7
    f2 = inputs.sparse(other, 40, 9970)
    for q, g in ((p, f[n:]), (other, f2)):
        got = qfs.heights_multi([(p, t, None), (q, dev_tensor(g), None)], power="reduced")
        assert np.array_equal(got[0].cpu().numpy(), want)
        assert np.array_equal(got[1].cpu().numpy(), oracle.heights(q, g))


@pytest.mark.parametrize("p,n", [(3, 300), (5, 300), (7, 200), (11, 150), (13, 150)])
@pytest.mark.parametrize("form", CORE_FORMS)
def test_reduced_mode_in_the_fused_kernel(qfs, p, n, form):
    # f^(p-2) waits in the second iterate's place while the product to f~^p stages in the ring
    f = np.concatenate([inputs.dense(p, n, 9980 + p), inputs.sparse(p, n, 9990 + p)])
    want = oracle.heights(p, f)
    assert len(set(want.tolist())) >= 3
    t = dev_tensor(f)
    assert np.array_equal(qfs.heights(p, t, power="reduced", form=form, max_ctas=200).cpu().numpy(), want)
    row = f[np.flatnonzero(want > 2)[0]]
    got = qfs.debug_stages(p, dev_tensor(row), form=form, power="reduced")
    assert got["h"] == want[np.flatnonzero(want > 2)[0]]
    assert qfs.read_status() == 0


def test_reduced_mode_paper_examples(qfs):
    for p in (5, 7, 11, 13):
        sel = [r for r in example_quartics() if r[0] == p]
        f = np.stack([r[3] for r in sel])
        want = np.array([r[1] for r in sel], np.int8)
        assert np.array_equal(qfs.heights(p, dev_tensor(f), power="reduced").cpu().numpy(), want), p


# ------------------------------------------------------------------------------------- theta matrix export
@pytest.mark.parametrize("p,n", [(3, 8), (5, 3), (7, 1)])
def test_theta_matrix_matches_oracle(qfs, p, n):
    # every entry of M equals the oracle's M from its definition; height-1 rows are exported too
    f = np.concatenate([inputs.dense(p, n, 8800 + p), inputs.sparse(p, 1, 8900 + p)])
    got = qfs.theta_matrix(p, dev_tensor(f)).cpu().numpy()
    for i in range(len(f)):
        assert np.array_equal(got[i], oracle.theta_matrix(p, f[i])), i
    assert qfs.read_status() == 0


def test_theta_matrix_applies_theta_and_rejects_bad_rows(qfs):
    # M g = theta(g): the device's first iterate, and an invalid row gives M = 0
    p = 5
    f, h = find_rows(p, 400, 8950, lambda x: x >= 2, 2)
    bad = f[:1].copy()
    bad[0, 7] = p
    rows = np.concatenate([f, bad])
    M = qfs.theta_matrix(p, dev_tensor(rows)).cpu().numpy().astype(np.int64)
    for i in range(len(f)):
        st = qfs.debug_stages(p, dev_tensor(f[i]))
        g = st["g"].cpu().numpy().astype(np.int64)
        assert np.array_equal(M[i] @ g % p, st["iters"].cpu().numpy()[0])
    assert not M[-1].any()
    with pytest.raises(qfs.QfsError):
        qfs.theta_matrix(4, dev_tensor(f))


# ------------------------------------------------------------------------------------- matrix multiplication mod p
@pytest.mark.parametrize("p,n,m,k", [(11, 1, 1, 1), (11, 17, 33, 65), (11, 300, 257, 129), (11, 128, 128, 64),
                                     (11, 513, 130, 1000), (2, 200, 300, 77), (251, 140, 70, 300), (256, 64, 64, 64)])
def test_matmul_mod_matches_oracle(qfs, p, n, m, k):
    rng = np.random.default_rng(p * 1000 + n + m + k)
    A = rng.integers(0, p, (n, k), dtype=np.uint8)
    B = rng.integers(0, p, (k, m), dtype=np.uint8)
    got = qfs.matmul_mod(p, dev_tensor(A), dev_tensor(B)).cpu().numpy()
    assert np.array_equal(got, oracle.matmul_mod(p, A, B))


@pytest.mark.parametrize("p,n,m,k,lo", [
    (33, 129, 257, 127, 0), (34, 129, 257, 129, 0),        # one e4m3 plane and two; edges of tiles and K steps
    (33, 130, 260, 65536, 16), (33, 5, 9, 65664, 15),      # sums up to 2^24, and past one drain
    (256, 127, 255, 896, 120), (251, 64, 300, 769, 112),   # the shortest drains, the largest plane products
    (2, 1, 700, 4097, 0)])
def test_matmul_mod_planes_and_drains(qfs, p, n, m, k, lo):
    # whole values: any lost bit of an accumulation shows
    rng = np.random.default_rng(p * 7 + k)
    A = rng.integers(lo, min(p, lo + 18), (n, k), dtype=np.uint8)
    B = rng.integers(lo, min(p, lo + 18), (k, m), dtype=np.uint8)
    got = qfs.matmul_mod(p, dev_tensor(A), dev_tensor(B)).cpu().numpy()
    want = (A.astype(np.int64) @ B.astype(np.int64)) % p
    assert np.array_equal(got, want.astype(np.uint8))
    assert qfs.read_status() == 0


def test_matmul_mod_unaligned_views(qfs):
    # row pitches and base addresses of every alignment: the pack reads and the product writes bytes then
    rng = np.random.default_rng(77)
    for off, n, m, k in [(0, 40, 16, 64), (1, 33, 24, 65), (2, 30, 20, 66), (3, 31, 37, 67)]:
        A = rng.integers(0, 11, (n, k), dtype=np.uint8)
        B = rng.integers(0, 11, (k, m), dtype=np.uint8)
        bufs = [torch.zeros(x + 8, dtype=torch.uint8, device="cuda:0") for x in (n * k, k * m, n * m)]
        a, b, c = (t[off:off + x].view(s) for t, x, s in zip(bufs, (n * k, k * m, n * m), ((n, k), (k, m), (n, m))))
        a.copy_(torch.from_numpy(A))
        b.copy_(torch.from_numpy(B))
        qfs.matmul_mod(11, a, b, out=c)
        assert np.array_equal(c.cpu().numpy(), oracle.matmul_mod(11, A, B))
        assert not bufs[2][:off].any() and not bufs[2][off + n * m:].any()


@pytest.mark.parametrize("p,top", [(33, 16), (31, 15), (29, 14), (34, 17), (101, 50), (129, 64), (251, 125), (255, 127),
                                   (256, 128)])
@pytest.mark.parametrize("steps_past", [0, 1])
@pytest.mark.parametrize("constant", [False, True])
def test_matmul_mod_at_the_float32_bound(qfs, p, top, steps_past, constant):
    # Residues are taken in the symmetric range, so operands of one sign next to p / 2 make the largest sums, up to 2^24 at
    # p = 33, and odd values next to them the ones whose last bit counts.  A drain comes after `steps` K steps of 128;
    # K is one drain, and one drain and a step.
    mag = p // 2 if p <= 33 else p // 2 + 16
    steps = 2 ** 24 // (mag * mag * 128)
    k = 128 * (steps + steps_past)
    n, m = (130, 260) if k <= 20000 else (37, 41)
    rng = np.random.default_rng(1000 * p + k)
    A, B = (np.full(s, top, np.uint8) if constant else rng.integers(top - 1, top + 1, s, dtype=np.uint8)
            for s in ((n, k), (k, m)))
    A[0, ::7] = top - 1
    drained = A[:, :128 * steps].astype(np.float64) @ B[:128 * steps].astype(np.float64)
    limit = top * top * 128 * steps
    assert limit == 2 ** 24 or p != 33
    assert drained.max() > 0.9 * limit and drained.max() <= 2 ** 24
    got = qfs.matmul_mod(p, dev_tensor(A), dev_tensor(B)).cpu().numpy()
    want = A.astype(np.float64) @ B.astype(np.float64) % p   # sums below 2^53
    assert np.array_equal(got, want.astype(np.uint8))
    assert qfs.read_status() == 0


@pytest.mark.parametrize("p,top", [(251, 125), (33, 16), (11, 5)])
def test_matmul_mod_sums_past_float32(qfs, p, top):
    # a long K whose undrained sum leaves the integers that float32 holds: 2^29 at p = 251, 2^26 at p = 33
    k = {251: 40000, 33: 300000, 11: 3000000}[p]
    rng = np.random.default_rng(p)
    A = rng.integers(max(top - 19, top // 2), top + 1, (16, k), dtype=np.uint8)
    B = rng.integers(max(top - 19, top // 2), top + 1, (k, 24), dtype=np.uint8)
    want = A.astype(np.float64) @ B.astype(np.float64)
    assert want.max() > 1.5 * 2 ** 24
    got = qfs.matmul_mod(p, dev_tensor(A), dev_tensor(B)).cpu().numpy()
    assert np.array_equal(got, (want % p).astype(np.uint8))
    assert qfs.read_status() == 0


@pytest.mark.parametrize("p", [11, 251])
@pytest.mark.parametrize("n,m", [(1, 1), (31, 3), (33, 255), (127, 257), (129, 258), (161, 511), (200, 515)])
def test_matmul_mod_rows_at_odd_addresses(qfs, p, n, m):
    # rows of C that start anywhere: first and last words of a row are shared with its neighbours, and nothing else is touched
    rng = np.random.default_rng(100 * n + m)
    k = 70
    A, B = rng.integers(0, p, (n, k), dtype=np.uint8), rng.integers(0, p, (k, m), dtype=np.uint8)
    want = (A.astype(np.int64) @ B.astype(np.int64) % p).astype(np.uint8)
    a, b = dev_tensor(A), dev_tensor(B)
    for off in range(4):
        buf = torch.full((n * m + 16,), 255, dtype=torch.uint8, device="cuda:0")
        c = buf[off + 4:off + 4 + n * m].view(n, m)
        qfs.matmul_mod(p, a, b, out=c)
        assert np.array_equal(c.cpu().numpy(), want), off
        assert (buf[:off + 4] == 255).all() and (buf[off + 4 + n * m:] == 255).all()
    assert qfs.read_status() == 0


def test_matmul_mod_odd_row_length_costs_little(qfs):
    # a short product with odd rows is bound by its stores, as is one with aligned rows
    def ms(n):
        g = torch.Generator(device="cuda").manual_seed(n)
        A = torch.randint(0, 31, (n, 129), dtype=torch.uint8, device="cuda", generator=g)
        B = torch.randint(0, 31, (129, n), dtype=torch.uint8, device="cuda", generator=g)
        out = torch.empty(n, n, dtype=torch.uint8, device="cuda")
        return _ms(lambda: [qfs.matmul_mod(31, A, B, out=out) for _ in range(10)])
    even, odd = ms(4096), ms(4097)
    assert odd < 2 * even, (odd, even)


def test_matmul_mod_long_k_reduces_between_tiles(qfs):
    # k (p-1)^2 above 2^31 at p = 251: the accumulators are reduced between K tiles
    p, n, m, k = 251, 16, 24, 40000
    rng = np.random.default_rng(9)
    A = rng.integers(p - 20, p, (n, k), dtype=np.uint8)
    B = rng.integers(p - 20, p, (k, m), dtype=np.uint8)
    got = qfs.matmul_mod(p, dev_tensor(A), dev_tensor(B)).cpu().numpy()
    assert np.array_equal(got, oracle.matmul_mod(p, A, B))


def test_matmul_mod_full_size_sampled(qfs):
    # the paper's smallest size (5,000 x 5,000 mod 11); 256 entries checked one by one
    p, n = 11, 5000
    g = torch.Generator(device="cuda").manual_seed(11)
    A = torch.randint(0, p, (n, n), dtype=torch.uint8, device="cuda", generator=g)
    B = torch.randint(0, p, (n, n), dtype=torch.uint8, device="cuda", generator=g)
    C = qfs.matmul_mod(p, A, B).cpu().numpy()
    An, Bn = A.cpu().numpy(), B.cpu().numpy()
    rng = np.random.default_rng(3)
    for i, j in zip(rng.integers(0, n, 256), rng.integers(0, n, 256)):
        assert C[i, j] == oracle.matmul_mod(p, An[i:i + 1], Bn[:, j:j + 1])[0, 0]


def test_matmul_mod_edges(qfs):
    z = torch.zeros(0, 5, dtype=torch.uint8, device="cuda")
    assert qfs.matmul_mod(11, z, torch.zeros(5, 3, dtype=torch.uint8, device="cuda")).shape == (0, 3)
    A = torch.ones(4, 0, dtype=torch.uint8, device="cuda")
    C = qfs.matmul_mod(11, A, torch.ones(0, 6, dtype=torch.uint8, device="cuda"))
    assert C.shape == (4, 6) and not C.any()
    with pytest.raises(qfs.QfsError):
        qfs.matmul_mod(1, torch.ones(2, 2, dtype=torch.uint8, device="cuda"), torch.ones(2, 2, dtype=torch.uint8,
                                                                                         device="cuda"))


# ------------------------------------------------------------------------------------- exact powering over Z
def _multinomial(es):
    from math import factorial
    out = factorial(sum(es))
    for e in es:
        out //= factorial(e)
    return out


def _eval_mod(cs, deg, pt, mod):
    pw = [[pow(x, k, mod) for k in range(deg + 1)] for x in pt]
    acc = 0
    for c, e in zip(cs, oracle.form_monomials(deg)):
        acc = (acc + c * pw[0][e[0]] * pw[1][e[1]] * pw[2][e[2]] * pw[3][e[3]]) % mod
    return acc


@pytest.mark.parametrize("d,n", [(1, 100), (16, 6)])
def test_poly_power_multinomial_closed_form(qfs, d, n):
    # (x1+x2+x3+x4)^d to the n-th power: every coefficient is a multinomial coefficient (up to 200 bits)
    f = [_multinomial(e) for e in oracle.form_monomials(d)]
    got = qfs.poly_power(d, f, n)
    assert got == [_multinomial(e) for e in oracle.form_monomials(d * n)]


# (d, n) chosen so that the transform length puts every pass size on the device: (1, 7) a one-stage column pass
# (the shared-memory stage loop), (1, 9) two, (2, 5) three, (4, 3) four, (16, 1) five, (4, 5) six, (5, 6) seven,
# (16, 2) eight; transforms of 2^13 words or more ((16, 1), (16, 2), (4, 5), (5, 6)) run the register-phase inner
# pass, the shorter ones the shared-memory one
@pytest.mark.parametrize("d,n", [(4, 3), (16, 2), (16, 1), (1, 7), (1, 9), (2, 5), (4, 5), (5, 6)])
def test_poly_power_matches_definition(qfs, d, n):
    rng = np.random.default_rng(d * 100 + n)
    f = [int(x) for x in rng.integers(0, 5, len(oracle.form_monomials(d)))]
    assert qfs.poly_power(d, f, n) == oracle.poly_power(d, f, n)


@pytest.mark.parametrize("n", [5, 15])
def test_poly_power_paper_workload_evaluation(qfs, n):
    # degree 16, coefficients in {0..4}: f^n(pt) = f(pt)^n at an integer point, modulo 2^127 - 1
    rng = np.random.default_rng(16 + n)
    f = [int(x) for x in rng.integers(0, 5, len(oracle.form_monomials(16)))]
    P = qfs.poly_power(16, f, n)
    mod = (1 << 127) - 1
    pt = (3, 5, 7, 11)
    assert _eval_mod(P, 16 * n, pt, mod) == pow(_eval_mod(f, 16, pt, mod), n, mod)


def test_poly_power_primes_in_groups(qfs):
    # five primes whose transforms of 2^23 words run two at a time, the last one alone
    rng = np.random.default_rng(28)
    f = [int(x) for x in rng.integers(0, 5, len(oracle.form_monomials(16)))]
    f[0] = 4
    P = qfs.poly_power(16, f, 12)
    mod = (1 << 127) - 1
    pt = (2, 3, 13, 17)
    assert _eval_mod(P, 16 * 12, pt, mod) == pow(_eval_mod(f, 16, pt, mod), 12, mod)


def test_poly_power_errors(qfs):
    with pytest.raises(qfs.QfsError):
        qfs.poly_power(16, [1] * 969, 16)   # degree 256
    with pytest.raises(qfs.QfsError):
        qfs.poly_power(1, [2 ** 31] * 4, 8)   # coefficients too large for 256 bits
