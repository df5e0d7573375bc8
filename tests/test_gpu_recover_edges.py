"""Plan recovery of FP32 solutions at its kernel's edges: sides below, at and above a
warp and a load round of 128, one long side, sparse and empty nodes, and a plan that
does not fit.  The oracle is Algorithm 1's loops on the exported flows: the same
entries, masses to 1e-13 of the total mass (FP32 flows are summed in pairs of about
48 bits: 2^-48 times a few hundred terms)."""
import numpy as np
import pytest

from oracle import recover as orec
from paper_2408_00598_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,kind", [(2, 2, "white"), (31, 3, "white"), (32, 33, "shapes"), (33, 9, "white"),
                                      (5, 129, "white"), (130, 7, "gauss"), (24, 24, "shapes"),
                                      (1023, 2, "white"), (1023, 3, "white")])      # walks of 1,024 and 1,025 steps
def test_recovery_equals_algorithm1_on_the_flows(m, n, kind):
    import torch
    from paper_2408_00598_gb300 import hot
    mu, nu = syn.make_pair(kind, m, 5, n)
    with hot.Context(precision="fp32") as ctx:
        r = ctx.solve(mu, nu, tol=0.0, max_iter=60)
        x = ctx.flows(r)
        src, dst, mass, l1 = ctx.recover_plan(r)
        # device outputs, with room to spare and with one entry too few
        k = len(mass)
        o = (torch.full((k + 5,), -1, dtype=torch.int32, device="cuda"),
             torch.full((k + 5,), -1, dtype=torch.int32, device="cuda"),
             torch.full((k + 5,), -1.0, dtype=torch.float64, device="cuda"))
        nnz, l2 = ctx.recover_plan(r, o)
        assert nnz == k and abs(l1[0] - l2[0]) <= 1e-13 and abs(l1[1] - l2[1]) <= 1e-13
        for have, want in zip(o, (src, dst, mass)):
            np.testing.assert_array_equal(have[:k].cpu().numpy(), want)
            assert (have[k:] == -1).all()
        small = tuple(torch.full((k - 1,), -7, dtype=t.dtype, device="cuda") for t in o)
        with pytest.raises(hot.HotError):
            ctx.recover_plan(r, small)
        assert all((t == -7).all() for t in small)          # nothing is written
        ctx.release(r)
    ent = orec.recover_from_x(x, m, n)
    P, Q = np.zeros((m * n, m * n)), np.zeros((m * n, m * n))
    for i, j, k_, l, p in ent:
        P[i * n + j, k_ * n + l] += p
    np.add.at(Q, (src, dst), mass)
    assert np.abs(P - Q).max() <= 1e-13
    assert abs(np.abs(Q.sum(1) - mu.ravel()).sum() - l1[0]) <= 1e-12
    assert abs(np.abs(Q.sum(0) - nu.ravel()).sum() - l1[1]) <= 1e-12


def test_offsets_of_many_nodes():
    """98,304 nodes, two steps of the scan per CTA: entries in node order without gaps."""
    import torch
    from paper_2408_00598_gb300 import hot
    m, n = 512, 192
    mu, nu = syn.make_pair("white", m, 5, n)
    with hot.Context(precision="fp32") as ctx:
        r = ctx.solve(mu, nu, tol=0.0, max_iter=30)
        nnz, l1 = ctx.recover_plan(r, ())
        o = (torch.full((nnz,), -1, dtype=torch.int32, device="cuda"), torch.full((nnz,), -1, dtype=torch.int32, device="cuda"),
             torch.full((nnz,), -1.0, dtype=torch.float64, device="cuda"))
        assert ctx.recover_plan(r, o)[0] == nnz
        ctx.release(r)
    src, dst, mass = o
    node = torch.div(dst, n, rounding_mode="floor") * n + src % n
    assert (mass > 0).all() and (src >= 0).all() and (node.diff() >= 0).all()
    for idx, hist, want in ((src, mu, l1[0]), (dst, nu, l1[1])):
        got = torch.bincount(idx, weights=mass, minlength=m * n).cpu().numpy()
        assert abs(np.abs(got - hist.ravel()).sum() - want) <= 1e-12


@pytest.mark.parametrize("nnz,D", [(1, 1), (7, 4), (255, 5), (257, 7), (2049, 8), (5000, 3)])
def test_barycentric_map_of_runs(nnz, D):
    """Runs of one source across threads, warps and CTAs, and a bin out of range inside a
    run: the run's other entries still count."""
    import torch
    from oracle import consumers
    from paper_2408_00598_gb300 import hot
    rng = np.random.default_rng(nnz)
    src = np.sort(rng.integers(0, max(1, nnz // 3), nnz)).astype(np.int32)
    dst = rng.integers(0, 50, nnz).astype(np.int32)
    mass, y = rng.uniform(0.5, 1.0, nnz), rng.standard_normal((50, D))
    nsrc = int(src.max()) + 2
    bad = np.zeros(nnz, bool)
    if nnz > 10:
        bad[[3, nnz // 2, nnz - 1]] = True
    d2 = np.where(bad, 50, dst).astype(np.int32)
    ref, wref = consumers.barycentric_map(src[~bad], dst[~bad], mass[~bad], y, nsrc)
    t = [torch.from_numpy(v).cuda() for v in (src, d2, mass, y)]
    out = torch.empty((nsrc, D), dtype=torch.float64, device="cuda")
    w = torch.empty(nsrc, dtype=torch.float64, device="cuda")
    if bad.any():
        with pytest.raises(hot.HotError) as e:
            hot.hot_barycentric_map(*t, nsrc, out=out, weight=w)
        assert e.value.status == hot.HOT_EINVAL
    else:
        hot.hot_barycentric_map(*t, nsrc, out=out, weight=w)
    np.testing.assert_allclose(w.cpu().numpy(), wref, rtol=1e-12, atol=1e-14)
    np.testing.assert_allclose(out.cpu().numpy(), ref, rtol=1e-11, atol=1e-12)
