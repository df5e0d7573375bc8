"""k_group32 and k_group64 (one kernel for the check blocks of small instances) against the chain of
kernels: the same iterates and results, bit for bit.

The live sweep timing mode times the chain's kernels and therefore runs the chain at
every size; everything else runs k_group32 up to its size rule.  Sides of 2 and 3,
sides around a tile and a warp, several bands per slab, more tiles than CTAs, and
real-valued bin positions."""
import numpy as np
import pytest

from paper_2408_00598_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu

SIZES = [(2, 2, "white"), (3, 2, "white"), (5, 7, "gauss"), (16, 16, "shapes"), (17, 23, "white"), (33, 31, "white"),
         (64, 64, "shapes"), (65, 63, "white"), (20, 90, "white"), (96, 96, "gauss"), (129, 127, "white"),
         (200, 136, "white"), (255, 3, "white"), (3, 256, "white"), (257, 4, "white")]


def _both(ctx, mu, nu, **kw):
    got = []
    for chain in (0, 1):
        ctx.sweep_timing(chain)
        r = ctx.solve(mu, nu, tol=1e-6, max_iter=250, **kw)
        got.append((r, ctx.flows(r)))
        ctx.release(r)
    ctx.sweep_timing(0)
    return got


def _same(got):
    (a, xa), (b, xb) = got
    for key in ("ot_value", "dual_value", "rel_kkt", "abs_kkt", "sigma", "iters", "restarts", "status", "max_abs_dual"):
        assert a[key] == b[key], (key, a[key], b[key])
    np.testing.assert_array_equal(xa, xb)


@pytest.mark.parametrize("m,n,kind", SIZES)
def test_group_kernel_equals_the_chain(m, n, kind):
    from paper_2408_00598_gb300 import hot
    mu, nu = syn.make_pair(kind, m, 1, n)
    with hot.Context(precision="fp32") as ctx:
        _same(_both(ctx, mu, nu))


@pytest.mark.parametrize("m,n", [(24, 24), (45, 77), (130, 9)])
def test_group_kernel_equals_the_chain_at_real_positions(m, n):
    from paper_2408_00598_gb300 import hot
    rng = np.random.default_rng(m)
    mu, nu = syn.make_pair("white", m, 2, n)
    with hot.Context(precision="fp32") as ctx:
        _same(_both(ctx, mu, nu, xs=np.sort(rng.random(m)), ys=np.sort(rng.random(n))))


@pytest.mark.parametrize("m,n,kind", [(2, 2, "white"), (3, 2, "white"), (5, 7, "gauss"), (16, 16, "shapes"), (17, 23, "white"),
                                      (33, 31, "white"), (65, 63, "white"), (20, 90, "white"), (128, 3, "white")])
def test_fp64_group_kernel_equals_the_chain(m, n, kind):
    from paper_2408_00598_gb300 import hot
    mu, nu = syn.make_pair(kind, m, 1, n)
    with hot.Context(precision="fp64") as ctx:
        _same(_both(ctx, mu, nu))


@pytest.mark.parametrize("check_every", [2, 4, 64])
def test_group_kernel_equals_the_chain_for_other_block_lengths(check_every):
    from paper_2408_00598_gb300 import hot
    mu, nu = syn.make_pair("gauss", 40, 3)
    with hot.Context(precision="fp32", check_every=check_every) as ctx:
        _same(_both(ctx, mu, nu))


@pytest.mark.parametrize("count", [3, 40])
def test_groups_of_a_batch_equal_single_solves(count):
    """Groups of several sizes in one launch, CTAs shared by several instances among them."""
    from paper_2408_00598_gb300 import hot
    pairs = [syn.make_pair("white", 4 + (7 * q) % 23, q) for q in range(count)]
    with hot.Context(precision="fp32") as ctx:
        out = ctx.solve_batch([p[0] for p in pairs], [p[1] for p in pairs], tol=1e-6, max_iter=300)
        for (mu, nu), b in zip(pairs, out):
            a = ctx.solve(mu, nu, tol=1e-6, max_iter=300)
            ctx.release(a)
            assert (a["ot_value"], a["dual_value"], a["iters"]) == (b["ot_value"], b["dual_value"], b["iters"])


@pytest.mark.parametrize("sizes", [(128, 128), (64, 128, 256, 16)])
def test_contexts_of_several_threads_share_the_device(sizes):
    """Each thread's groups fill the device; the launches of the others take turns with them."""
    import threading
    from paper_2408_00598_gb300 import hot
    pairs = [syn.make_pair("white", S, q) for q, S in enumerate(sizes)]
    out = [[] for _ in sizes]

    def run(q, times):
        with hot.Context(precision="fp32") as ctx:
            for _ in range(times):
                r = ctx.solve(*pairs[q], tol=1e-6, max_iter=200)
                out[q].append((r["ot_value"], r["iters"], r["rel_kkt"], r["status"]))
                ctx.release(r)

    for q in range(len(sizes)):
        run(q, 1)
    threads = [threading.Thread(target=run, args=(q, 4)) for q in range(len(sizes))]
    for t in threads:
        t.start()
    for t in threads:
        t.join(120)
    for got in out:
        assert len(got) == 5 and all(g == got[0] for g in got)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_a_small_solve_runs_beside_a_kernel_of_the_caller(precision):
    """A kernel of one thread on another stream (about a second) takes one SM's place for a CTA; a small pair's
    group kernels need some of the others and do not wait for it."""
    import torch
    from paper_2408_00598_gb300 import hot
    mu, nu = syn.make_pair("white", 16, 1)
    with hot.Context(precision=precision) as ctx:
        ctx.release(ctx.solve(mu, nu, tol=0.0, max_iter=40))         # tables, pools, modules
        side, ended = torch.cuda.Stream(), torch.cuda.Event()
        with torch.cuda.stream(side):
            torch.cuda._sleep(1)
        torch.cuda.synchronize()
        with torch.cuda.stream(side):
            torch.cuda._sleep(2 * 10 ** 9)
            ended.record()
        r = ctx.solve(mu, nu, tol=0.0, max_iter=40)
        beside = not ended.query()
        ctx.release(r)
        torch.cuda.synchronize()
    assert r["iters"] == 40
    assert beside


@pytest.mark.parametrize("precision,S", [("fp32", 128), ("fp64", 64)])
def test_solves_of_two_contexts_overlap(precision, S):
    """Two threads with a context each against one thread with the same number of solves: the groups of each plan
    for a share of the device, so the two run side by side (taking turns, the times are equal)."""
    import threading
    import time
    from paper_2408_00598_gb300 import hot
    mu, nu = syn.make_pair("white", S, 1)

    def run(ctx, times):
        for _ in range(times):
            ctx.release(ctx.solve(mu, nu, tol=0.0, max_iter=400))

    with hot.Context(precision=precision) as a, hot.Context(precision=precision) as b:
        run(a, 1)
        run(b, 1)
        best = [1e9, 1e9]
        for _ in range(3):
            t0 = time.perf_counter()
            run(a, 12)
            t1 = time.perf_counter()
            threads = [threading.Thread(target=run, args=(ctx, 6)) for ctx in (a, b)]
            for t in threads:
                t.start()
            for t in threads:
                t.join()
            best = [min(best[0], t1 - t0), min(best[1], time.perf_counter() - t1)]
    assert best[1] < 0.9 * best[0], best


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_a_wait_that_runs_out_ends_the_call_with_an_error(precision):
    """With one poll per wait, the CTAs that arrive before the last one of their group give up at the first wait.
    The call says so, nothing is left behind, and the context solves again; so does the serve loop."""
    from paper_2408_00598_gb300 import hot
    mu, nu = syn.make_pair("white", 32, 1)
    with hot.Context(precision=precision) as ctx:
        a = ctx.solve(mu, nu, tol=1e-6, max_iter=200)
        ctx.release(a)
        ctx.wait_limit(1)
        for _ in range(2):
            with pytest.raises(hot.HotError, match="a wait between the CTAs of a group ran out") as e:
                ctx.solve(mu, nu, tol=1e-6, max_iter=200)
            assert e.value.status == hot.HOT_ECUDA
        with pytest.raises(hot.HotError, match="ran out"):
            ctx.solve_batch([mu] * 3, [nu] * 3, tol=1e-6, max_iter=200)
        t = ctx.submit(mu, nu, tol=1e-6, max_iter=200)
        assert ctx.wait(t)[0] == hot.HOT_ECUDA
        ctx.wait_limit(0)
        b = ctx.solve(mu, nu, tol=1e-6, max_iter=200)
        ctx.release(b)
        t = ctx.submit(mu, nu, tol=1e-6, max_iter=200)
        status, c = ctx.wait(t)
        ctx.forget(t)
    for r in (b, c):
        assert (r["ot_value"], r["iters"], r["status"]) == (a["ot_value"], a["iters"], a["status"])
    assert status == a["status"]


@pytest.mark.parametrize("S,max_iter", [(16, 10), (16, 50), (64, 3000)])
def test_blocks_of_a_solve_do_not_depend_on_the_form(S, max_iter):
    """hot_result.blocks: the check blocks that ran and the one launched ahead, though a group launch runs several."""
    from paper_2408_00598_gb300 import hot
    mu, nu = syn.make_pair("shapes", S, 1)
    with hot.Context(precision="fp32") as ctx:
        got = []
        for chain in (0, 1):
            ctx.sweep_timing(chain)
            r = ctx.solve(mu, nu, tol=1e-6, max_iter=max_iter)
            ctx.release(r)
            got.append(r["blocks"])
        ctx.sweep_timing(0)
    assert got == [r["iters"] // 10 + 1] * 2


def test_pairs_of_a_batch_report_their_own_completion():
    """25 pairs of one size and several classes, some of which end in different blocks of the same launch of the group
    kernel (four blocks): another number of iterations is another solve_ms, and 20 more of them a larger one."""
    from paper_2408_00598_gb300 import hot
    kinds = ("white", "gauss", "cauchy", "shapes", "translate")
    pairs = [syn.make_pair(kinds[q % 5], 16, q) for q in range(25)]
    with hot.Context(precision="fp32") as ctx:
        for _ in range(2):
            out = ctx.solve_batch([p[0] for p in pairs], [p[1] for p in pairs], tol=4e-3, max_iter=3000)
    got = [(r["iters"], r["solve_ms"]) for r in out]
    assert len({i for i, _ in got}) >= 3, got
    for ia, ta in got:
        assert ta > 0.0
        for ib, tb in got:
            assert ia == ib or ta != tb, got
            assert ib < ia + 20 or ta < tb, got


@pytest.mark.parametrize("precision,m,n,tiny", [("fp32", 256, 60, 150), ("fp64", 64, 64, 200)])
def test_tiny_pairs_that_share_a_cta_equal_single_solves(precision, m, n, tiny):
    """A CTA takes several instances one after the other (test_group_plan_host.py looks at this batch's plan), in one
    launch with an instance that many CTAs take."""
    from paper_2408_00598_gb300 import hot
    pairs = [syn.make_pair("white", m, 1, n)] + [syn.make_pair("white", 2, q, 2 + q % 2) for q in range(tiny)]
    with hot.Context(precision=precision) as ctx:
        out = ctx.solve_batch([p[0] for p in pairs], [p[1] for p in pairs], tol=1e-6, max_iter=80)
        # one kernel per four check blocks: the chain launches 30 or more per block
        assert out[0]["iters"] == 80 and out[0]["kernel_launches"] <= 4
        for (mu, nu), b in zip(pairs, out):
            a = ctx.solve(mu, nu, tol=1e-6, max_iter=80)
            ctx.release(a)
            for key in ("ot_value", "dual_value", "rel_kkt", "sigma", "iters", "restarts", "status"):
                assert a[key] == b[key], (key, a[key], b[key])


def test_fp64_groups_of_a_batch_equal_single_solves():
    """Groups of several sizes in one launch of k_group64."""
    from paper_2408_00598_gb300 import hot
    pairs = [syn.make_pair("white", 4 + (7 * q) % 23, q) for q in range(30)]
    with hot.Context(precision="fp64") as ctx:
        out = ctx.solve_batch([p[0] for p in pairs], [p[1] for p in pairs], tol=1e-6, max_iter=300)
        assert max(r["kernel_launches"] for r in out) <= 300 // 40 + 3
        for (mu, nu), b in zip(pairs, out):
            a = ctx.solve(mu, nu, tol=1e-6, max_iter=300)
            ctx.release(a)
            assert (a["ot_value"], a["dual_value"], a["iters"]) == (b["ot_value"], b["dual_value"], b["iters"])
