"""Calls and inputs beside the ordinary ones: far new points, arguments that have to be refused, products captured in CUDA
graphs, non-finite right blocks, results that must not depend on what was asked before."""
import numpy as np
import pytest
import torch

import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fd():
    import __graft_entry__ as g
    g.build()
    import paper_2609_38198_b200 as fd
    assert torch.cuda.is_available()
    return fd


@pytest.fixture(scope="module")
def dev():
    return torch.device("cuda:0")


# ------------------------------------------------------------------ out-of-sample extension of far points
@pytest.mark.parametrize("path", [1, 2])
def test_extension_of_far_points(fd, dev, path):
    """New points from inside the data to exponents (base 2) of 70 from every point.  Direct differences: the formula.  Gram form: a kernel
    value carries 2^-40 absolute (one half of the last place of the 16-bit pieces), which is 2^(e - 40) of a value at exponent e and at
    most twice that of the ratio; beyond 41 every value is zero and so is the extension."""
    N, m, beta = 3000, 5, 0.8
    bp = beta * np.log2(np.e)
    rng = np.random.default_rng(7)
    X = (0.02 * rng.standard_normal((N, 3))).astype(np.float32)
    e = np.array([0.0, 4.0, 12.0, 20.0, 30.0, 36.0, 40.5, 44.0, 52.0, 66.0])
    u = rng.standard_normal((len(e), 3))
    Z = (u / np.linalg.norm(u, axis=1)[:, None] * np.sqrt(e / bp)[:, None]).astype(np.float32)
    psi = np.cos(X.astype(np.float64) @ rng.standard_normal((3, m)) * 20.0)
    lam = np.linspace(1.0, 0.4, m)
    ctx = fd.Context(torch.from_numpy(X).to(dev), b_max=16)
    ctx.set_option("path", path)
    ctx.degree(beta, 1.0)
    out = ctx.nystrom(torch.from_numpy(Z).to(dev), fd.to_colmajor(psi.astype(np.float32), dev), lam).cpu().numpy().astype(np.float64)
    X64, Z64 = X.astype(np.float64), Z.astype(np.float64)
    q = np.exp(-beta * ((X64[:, None] - X64[None]) ** 2).sum(-1)).sum(1)
    E = bp * ((Z64[:, None] - X64[None]) ** 2).sum(-1)
    K = 2.0 ** -E / q[None]
    ref = (K @ psi) / (K.sum(1)[:, None] * lam[None])
    big = np.abs(psi).max() / lam.min()
    assert np.isfinite(out).all()
    for i in range(len(e)):
        near, far = E[i].min(), E[i].max()
        if path == 1:
            assert np.abs(out[i] - ref[i]).max() <= 1e-5 * big
        elif near > 41.0:
            assert (out[i] == 0.0).all(), (e[i], out[i])
        elif far < 39.0:
            assert np.abs(out[i] - ref[i]).max() <= (1e-5 + 2.0 * 2.0 ** (far - 40.0)) * big, (e[i], out[i], ref[i])
    ctx.close()


def test_ladder_start_with_a_point_far_from_all_others(fd, dev):
    """One new point beyond the range of the Gram-form product (base-2 exponent 57 from every point) among ordinary ones: a finite
    start basis with zeros in its row, and a solve that runs."""
    n_old, N, beta, k, b = 3000, 3400, 1.0, 12, 8
    X = workloads.torus6(N, seed=13)
    X[3100] = 0.0
    X[3100, 0] = 6.9
    Xt = torch.from_numpy(X).to(dev)
    old = fd.Context(Xt[:n_old].contiguous(), b_max=b, m_max=64)
    old.set_option("path", fd.FD_PATH_TC)
    old.degree(beta, 1.0)
    lam, U, info = old.eigs(k, b)
    new = fd.Context(Xt, b_max=b, m_max=64)
    new.degree(beta, 1.0)
    Q0 = new.ladder_start(old, Xt, U, lam)
    assert old.get_option("last_path") == fd.FD_PATH_TC
    assert torch.isfinite(Q0).all() and (Q0[3100] == 0).all() and (Q0[3099] != 0).all()
    lam_w, U_w, info_w = new.eigs(k, b, Q0=Q0, max_applies=200)
    assert info_w.converged == k + 1 and np.isfinite(lam_w).all() and torch.isfinite(U_w).all()
    old.close(); new.close()


# ------------------------------------------------------------------ arguments of the extension
def _nystrom(ctx, Xn, n, psi, ldpsi, m, out, ldout):
    import ctypes
    from paper_2609_38198_b200 import binding
    lam = (ctypes.c_double * m)(*([0.5] * m))
    return binding.lib.fd_nystrom(ctx._h, Xn.data_ptr(), n, Xn.stride(0), psi, ldpsi, m, lam, out, ldout)


def _extension_problem(fd, dev, N=300, n=700, m=6):
    ctx = fd.Context(torch.from_numpy(workloads.torus6(N, seed=1)).to(dev), b_max=8)
    ctx.degree(0.6, 1.0)
    Xn = torch.from_numpy(workloads.torus6(n, seed=2)).to(dev)
    panel = torch.randn((m, N + n), device=dev)               # column-major, pitch N + n
    return ctx, Xn, panel


def test_extension_refuses_overlapping_blocks(fd, dev):
    """More new points than points: the second chunk of rows would read what the first one wrote.  Other rows of one panel do not overlap."""
    N, n, m = 300, 700, 6
    ctx, Xn, panel = _extension_problem(fd, dev, N, n, m)
    ld = N + n
    assert _nystrom(ctx, Xn, n, panel.data_ptr(), ld, m, panel.data_ptr(), ld) == fd.FD_ERR_INVALID
    assert _nystrom(ctx, Xn, n, panel.data_ptr(), ld, m, panel.data_ptr() + 4 * (N - 1), ld) == fd.FD_ERR_INVALID
    before = panel[:, :N].clone()
    want = ctx.nystrom(Xn, before.t(), [0.5] * m)
    assert _nystrom(ctx, Xn, n, panel.data_ptr(), ld, m, panel.data_ptr() + 4 * N, ld) == fd.FD_OK
    ctx.synchronize()
    assert torch.equal(panel[:, :N], before) and torch.equal(panel[:, N:].t(), want)
    ctx.close()


def test_extension_refuses_misaligned_blocks(fd, dev):
    """Found by the host's argument checks, before any launch."""
    N, n, m = 300, 50, 2
    ctx, Xn, panel = _extension_problem(fd, dev, N, n, m)
    out = torch.empty((m, n), device=dev)
    launches = fd.fd_launch_count()
    assert _nystrom(ctx, Xn, n, panel.data_ptr() + 2, N + n - 1, m, out.data_ptr(), n) == fd.FD_ERR_INVALID
    assert _nystrom(ctx, Xn, n, panel.data_ptr(), N + n, m, out.data_ptr() + 1, n - 1) == fd.FD_ERR_INVALID
    assert fd.fd_launch_count() == launches
    ctx.close()


# ------------------------------------------------------------------ results do not depend on calls in between
def _listed(fd, dev, kind):
    """A context whose products at `beta` leave out tiles: (ctx, X, beta)."""
    if kind == "direct":
        X, beta = workloads.torus2(16384, seed=1), 100.0
    else:
        X, beta = workloads.latent_torus(32768, seed=42), 5.0
    ctx = fd.Context(torch.from_numpy(X).to(dev), b_max=8)
    ctx.set_option("path", fd.FD_PATH_SIMT if kind == "direct" else fd.FD_PATH_TC)
    ctx.set_option("tc_max_mag", 1e4)
    return ctx, X, beta


@pytest.mark.parametrize("kind", ["direct", "gram"])
def test_only_degree_passes_decide_which_tiles_are_left_out(fd, dev, kind):
    """A row sum or a product at another bandwidth in between leaves the products at the degree passes' bandwidth as they were, bit for
    bit, and still without the tiles that hold only zeros."""
    ctx, X, beta = _listed(fd, dev, kind)
    V = fd.to_colmajor(workloads.block(X.shape[0], 8, seed=3), dev)
    ctx.degree(beta, 1.0)
    Y = ctx.apply(V)
    share = ctx.get_option("tile_share")
    assert share < 0.9
    for other in (0.9 * beta, 0.01 * beta):
        ctx.apply_general(other, None)
        ctx.apply_general(other, V)
        assert torch.equal(ctx.apply(V), Y)
        assert ctx.get_option("tile_share") == share
    ctx.close()


@pytest.mark.parametrize("kind", ["direct", "gram"])
def test_calls_without_lists_do_not_depend_on_the_order_of_the_points(fd, dev, kind):
    """A bandwidth so small that no two points are far apart: a context that has ordered its points for another bandwidth gives the bits
    of one that never did, in every kind of pass."""
    def passes(ctx, X, small):
        V = fd.to_colmajor(workloads.block(X.shape[0], 8, seed=3), dev)
        rows = torch.from_numpy(X[:70].copy()).to(dev)
        q, d, s, so, so2 = ctx.degree(small, 1.0)
        out = [q, d, s, ctx.apply(V), ctx.apply_general(1.5 * small, V), ctx.apply_general(small, V, Xrow=rows), ctx.nystrom(rows, V, [0.5] * 8)]
        if kind == "gram":
            out.append(ctx.apply(V, prec=fd.FD_PREC_FAST))
        return out, (so, so2)

    ctx, X, beta = _listed(fd, dev, kind)
    want, sums = passes(ctx, X, 0.01 * beta)
    ctx.close()
    ctx, X, beta = _listed(fd, dev, kind)
    V = fd.to_colmajor(workloads.block(X.shape[0], 8, seed=4), dev)
    q, d, s, _, _ = ctx.degree(beta, 1.0)
    Y = ctx.apply(V)
    assert ctx.get_option("tile_share") < 0.9
    got, sums2 = passes(ctx, X, 0.01 * beta)
    assert sums == sums2 and all(torch.equal(a, b) for a, b in zip(want, got)), [torch.equal(a, b) for a, b in zip(want, got)]
    q2, d2, s2, _, _ = ctx.degree(beta, 1.0)
    assert torch.equal(q, q2) and torch.equal(d, d2) and torch.equal(s, s2) and torch.equal(ctx.apply(V), Y)
    ctx.close()


def _notes(ctx, kind):
    """The part of the workspace with a degree pass's notes: a byte per tile, 1 for every tile that holds a point's kernel value with itself."""
    ws, N = ctx._ws[-ctx._ws.data_ptr() % 256:], ctx.N
    if kind == "direct":
        first, step, size = 1, N // 16 + 4, (N // 64) * (N // 16)        # groups of 64 rows, entries of 16 points: entry 4 g + 1 is one of group g's own
    else:
        first, step, size = 0, N // 128 + 1, 2 * (N // 128) ** 2         # tiles of 128: two planes
    at = torch.arange(0, ws.numel() - size, 256, device=ws.device)
    for k in range((N // 64) if kind == "direct" else N // 128):
        at = at[ws[at + (first + k * step)] == 1]
    found = [int(a) for a in at.cpu() if int(ws[a:a + size].max()) == 1]
    assert len(found) == 1, found
    return ws[found[0]:found[0] + size]


@pytest.mark.parametrize("kind", ["direct", "gram"])
def test_a_failed_degree_pass_leaves_no_notes(fd, dev, kind):
    """fd_degree reports a bounded wait that ran out (of the self-test here; a pass that gives up in one has not noted the tiles after it).
    What was noted is not used again: neither by products recorded afterwards nor by the next degree pass, whose results are those of a new
    context."""
    stream = torch.cuda.Stream()
    ctx, X, beta = _listed(fd, dev, kind)
    V = fd.to_colmajor(workloads.block(X.shape[0], 8, seed=3), dev)
    torch.cuda.synchronize()
    s = ctx.degree(beta, 1.0)[2]
    want = ctx.apply(V)
    ctx.close()

    def failed(stream=None):
        c = fd.Context(torch.from_numpy(X).to(dev), b_max=8, stream=stream)
        c.set_option("path", fd.FD_PATH_SIMT if kind == "direct" else fd.FD_PATH_TC)
        c.set_option("tc_max_mag", 1e4)
        c.set_option("wait_selftest", 2.0e6)
        with pytest.raises(fd.FdError) as e:
            c.degree(beta, 1.0)
        assert e.value.status == fd.FD_ERR_TIMEOUT
        torch.cuda.synchronize()
        _notes(c, kind).zero_()                                # the pass that gave up noted nothing
        torch.cuda.synchronize()
        return c

    ctx = failed()
    assert torch.equal(ctx.degree(beta, 1.0)[2], s) and torch.equal(ctx.apply(V), want)
    ctx.close()
    ctx, Y = failed(stream), torch.zeros_like(want)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):                   # (lists for itself)
        ctx.apply_general(beta, V, left=s, right=s, out=Y)
    torch.cuda.synchronize()
    g.replay()
    torch.cuda.synchronize()
    assert ((Y - want).norm() / want.norm()).item() <= 2e-6    # two orders of fp32 sums
    ctx.close()


# ------------------------------------------------------------------ products recorded into CUDA graphs
@pytest.mark.parametrize("kind,prec", [("direct", 0), ("gram", 0), ("gram", 1)])
def test_recorded_products_do_not_depend_on_calls_in_between(fd, dev, kind, prec):
    """Eager calls may come between recording and replay and between replays: external rows (which use the rows' operand buffer), degree
    passes at another bandwidth (other lists), products at a bandwidth that only a graph has seen.  Every result is that of the same
    call in a context without graphs, bit for bit."""
    stream = torch.cuda.Stream()
    if kind == "direct":
        X, beta, path = workloads.torus2(16384, seed=1), 100.0, fd.FD_PATH_SIMT
    else:
        X, beta, path = workloads.latent_torus(32768, seed=42), 5.0, fd.FD_PATH_TC
    N, b, other, unseen = X.shape[0], 8, 2.5 * beta, 0.7 * beta
    Xt = torch.from_numpy(X).to(dev)
    V = fd.to_colmajor(workloads.block(N, b, seed=3), dev)
    torch.cuda.synchronize()

    def context(s):
        ctx = fd.Context(Xt, b_max=b, stream=s)
        ctx.set_option("path", path)
        ctx.set_option("tc_max_mag", 1e4)
        return ctx

    plain = context(stream)
    s0 = plain.degree(beta, 1.0)[2].clone()

    def general(c, bt, out=None):
        Y = c.apply_general(bt, V, left=s0, right=s0, out=out, prec=prec)
        if out is None:
            torch.cuda.synchronize()                          # (compared on another stream)
        return Y

    torch.cuda.synchronize()
    want = general(plain, beta)
    assert plain.get_option("tile_share") < 0.9
    want_unseen = general(plain, unseen)
    torch.cuda.synchronize()

    ctx = context(stream)
    ctx.degree(beta, 1.0)
    general(ctx, beta)
    Y, Z = torch.zeros_like(want), torch.zeros_like(want)
    torch.cuda.synchronize()
    g1, g2 = torch.cuda.CUDAGraph(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(g1, stream=stream):
        general(ctx, beta, out=Y)
    with torch.cuda.graph(g2, stream=stream):
        general(ctx, unseen, out=Z)
    torch.cuda.synchronize()

    def replay(g, buf, expect, what):
        buf.zero_()
        torch.cuda.synchronize()
        with torch.cuda.stream(stream):
            g.replay()
        torch.cuda.synchronize()
        assert torch.equal(buf, expect), what

    assert torch.equal(general(ctx, unseen), want_unseen), "eager, recorded but never run"
    replay(g2, Z, want_unseen, "first replay")
    assert torch.equal(general(ctx, beta), want), "eager after a replay at another bandwidth"
    replay(g1, Y, want, "after an eager call")
    ctx.apply_general(beta, V, Xrow=Xt[:500].contiguous())
    ctx.nystrom(Xt[100:300].contiguous(), V, [0.5] * b)
    replay(g1, Y, want, "after external rows")
    ctx.degree(other, 1.0)
    general(ctx, other)
    replay(g1, Y, want, "after degree passes at another bandwidth")
    replay(g2, Z, want_unseen, "after degree passes at another bandwidth")
    ctx.degree(beta, 1.0)
    assert torch.equal(general(ctx, beta), want)
    ctx.synchronize()
    ctx.close(); plain.close()


def test_recorded_row_sums_do_not_wait(fd, dev):
    """A row sum over the points at a bandwidth that no degree pass has seen returns without waiting, so it can be recorded."""
    stream = torch.cuda.Stream()
    X = torch.from_numpy(workloads.torus2(16384, seed=1)).to(dev)
    torch.cuda.synchronize()
    ctx = fd.Context(X, b_max=8, stream=stream)
    ctx.set_option("path", fd.FD_PATH_SIMT)
    want = ctx.apply_general(150.0, None)
    torch.cuda.synchronize()
    ctx.apply_general(100.0, None)
    Y = torch.zeros_like(want)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        ctx.apply_general(150.0, None, out=Y)
    torch.cuda.synchronize()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(Y, want)
    ctx.close()


# ------------------------------------------------------------------ non-finite right blocks
@pytest.mark.parametrize("kind", ["direct", "gram"])
def test_entries_that_are_not_finite_reach_every_row(fd, dev, kind):
    """0 * Inf and 0 * NaN are NaN: with far tiles left out the product has NaN and Inf where the product over all tiles (a context whose
    degree passes have not seen the bandwidth) has them; the other columns are untouched.  Also in a recorded product, whose later
    replays with finite entries are as before, and in row sums with such weights."""
    ctx, X, beta = _listed(fd, dev, kind)
    N, b = X.shape[0], 24
    path = ctx.get_option("path")
    ctx.close()
    stream = torch.cuda.Stream()
    Xt = torch.from_numpy(X).to(dev)
    good = fd.to_colmajor(workloads.block(N, b, seed=3), dev)
    V = good.clone(memory_format=torch.preserve_format)
    V[100, 1] = float("nan"); V[200, 2] = float("inf"); V[300, 3] = float("-inf"); V[300, 17] = float("inf"); V[9000, 17] = float("-inf")
    V[17, 23] = float("inf"); V[18, 23] = float("nan"); V[:, 7] = 3e38                  # (finite, though its sums are not)
    w = torch.rand(N, device=dev) + 0.5
    w[12] = float("inf")
    torch.cuda.synchronize()
    ctx = fd.Context(Xt, b_max=b, stream=stream)
    ctx.set_option("path", path)
    ctx.set_option("tc_max_mag", 1e4)
    ctx.degree(beta, 1.0)
    want_good = ctx.apply(good)
    assert ctx.get_option("tile_share") < 0.9
    Y = ctx.apply(V)
    torch.cuda.synchronize()
    # every tile
    ref = fd.Context(Xt, b_max=b, stream=stream)
    ref.set_option("path", path)
    ref.set_option("tc_max_mag", 1e4)
    s = torch.empty(N, device=dev)
    s.copy_(ctx.degree(beta, 1.0)[2])
    torch.cuda.synchronize()
    Yr = ref.apply_general(beta, V, left=s, right=s)
    torch.cuda.synchronize()
    cls = lambda t: torch.where(torch.isnan(t), 3, torch.where(torch.isposinf(t), 1, torch.where(torch.isneginf(t), 2, 0)))
    assert torch.equal(cls(Y), cls(Yr))
    finite = torch.isfinite(Yr).all(0)
    assert 0 < (~finite).sum() <= 6 and ((Y[:, finite] - Yr[:, finite]).norm() / Yr[:, finite].norm()).item() <= 2e-6
    if kind == "direct":
        R, Rr = ctx.apply_general(beta, None, right=w), ref.apply_general(beta, None, right=w)
        torch.cuda.synchronize()
        assert torch.equal(cls(R), cls(Rr)) and not torch.isfinite(R).any()
    # recorded: bad entries, then finite ones in the same buffer
    buf, out = V.clone(memory_format=torch.preserve_format), torch.zeros_like(Y)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        ctx.apply(buf, out=out)
    for v, want in ((V, Y), (good, want_good), (V, Y)):
        buf.copy_(v)
        torch.cuda.synchronize()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(cls(out), cls(want)) and torch.equal(torch.nan_to_num(out), torch.nan_to_num(want))
    last = ctx.apply(good)
    torch.cuda.synchronize()
    assert torch.equal(last, want_good)
    ctx.close(); ref.close()


# ------------------------------------------------------------------ eigensolver
class _NothingNewAfterRestart:
    """A one-rank transport that turns every projection after the first thick restart into zeros, as if the basis held everything: the
    solver then finds no direction to add and leaves.  (kept = columns that a restart keeps: their projections are kept x kept.)"""
    rank, world = 0, 1

    def __init__(self, kept):
        self.kept, self.seen = kept, 0

    def allreduce_sum_host(self, arr, device, stream):
        if self.seen >= 2:
            arr[:] = 0.0
        elif arr.size == self.kept * self.kept:
            self.seen += 1

    def allgather(self, send, recv, stream):
        with torch.cuda.stream(stream):
            recv.copy_(send)


def test_vectors_of_a_solve_that_ends_right_after_a_restart(fd, dev):
    """FD_ERR_NOT_CONVERGED returns the best Ritz pairs, also where the basis has just been compressed onto them."""
    from oracle import dense
    X = workloads.torus6(600, seed=2)
    k, b, beta, cap = 4, 4, 0.5, 14
    kept = k + 1 + b                                          # every Ritz vector of a step: more than 3/5 of the capacity
    ctx = fd.Context(torch.from_numpy(X).to(dev), b_max=b, m_max=cap)
    transport = _NothingNewAfterRestart(kept)
    ctx.set_shard(fd.Shard(transport, X.shape[0], b, dev))
    ctx.degree(beta, 1.0)
    lam, U, info = ctx.eigs(k, b, tol=1e-9, max_applies=50, allow_not_converged=True)
    assert transport.seen == 2 and info.restarts == 1 and info.basis_cols == kept and info.converged < k + 1
    U = U.cpu().numpy().astype(np.float64)
    assert np.abs(U.T @ U - np.eye(k + 1)).max() <= 1e-5
    R = dense.apply(X, beta, 1.0, U) - U * lam[None, :]
    assert np.linalg.norm(R, axis=0).max() <= info.max_residual + 5e-6 and info.max_residual < 0.3
    ctx.close()


def test_reported_time_in_applies_is_the_products_time(fd, dev):
    """info.seconds_apply against the same number of products timed on their own (events; half to twice: clocks and neighbours differ)."""
    N, k, b, beta = 50021, 12, 32, 2.0
    ctx = fd.Context(torch.from_numpy(workloads.torus6(N, seed=3)).to(dev), b_max=b, m_max=3 * (k + 1) + 2 * b)
    ctx.degree(beta, 1.0)
    lam, U, info = ctx.eigs(k, b)
    V = fd.to_colmajor(workloads.block(N, b, seed=1), dev)
    ctx.apply(V)
    t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    t0.record()
    for _ in range(info.applies):
        ctx.apply(V)
    t1.record()
    torch.cuda.synchronize()
    seconds = 1e-3 * t0.elapsed_time(t1)
    assert 0.5 * seconds <= info.seconds_apply <= 2.0 * seconds, (info.seconds_apply, seconds)
    assert info.seconds_apply <= info.seconds_total
    ctx.close()


@pytest.mark.parametrize("data,N,seed,beta,k,b,cap", [
    ("torus6", 40000, 42, 2.0, 64, 32, 192), ("torus6", 40000, 42, 2.0, 64, 32, 195), ("torus6", 30000, 7, 2.0, 64, 32, 259),
    ("torus2", 16384, 42, 100.0, 32, 16, 98), ("torus2", 16384, 42, 100.0, 32, 16, 99), ("torus2", 16384, 42, 300.0, 32, 16, 131),
    ("latent", 65536, 42, 2.0, 32, 32, 98), ("latent", 65536, 42, 2.0, 32, 32, 163)])
def test_solves_at_the_accuracy_floor_on_both_sides_of_the_capacity_rule(fd, dev, data, N, seed, beta, k, b, cap):
    """Spectra whose residuals end near tol = 1e-6.  From a capacity of 3 (k + 1) on a solve that stalls above tol applies M to its basis again
    and converges.  On both sides the returned pairs' float64 residuals exceed the reported ones, which are measured with stored fp32
    images, by at most 3e-6: 1e-6 for the images' rounding, 2e-6 for the operator's own error.  (All rows: the far-out points of the
    latent torus carry most of that error, so a sample of rows would not do.)"""
    X = {"torus6": workloads.torus6, "torus2": workloads.torus2, "latent": workloads.latent_torus}[data](N, seed=seed)
    Xt = torch.from_numpy(X).to(dev)
    Xd = Xt.double()
    ctx = fd.Context(Xt, b_max=b, m_max=cap)
    s = ctx.degree(beta, 1.0)[2].double()
    lam, U, info = ctx.eigs(k, b, max_applies=600, allow_not_converged=True)
    lt, Ud = torch.tensor(lam, device=dev), U.double()
    sq = torch.zeros(k + 1, dtype=torch.float64, device=dev)
    for r in torch.arange(N, device=dev).split(1024):
        K = torch.exp(-beta * torch.cdist(Xd[r], Xd, compute_mode="donot_use_mm_for_euclid_dist") ** 2)
        sq += ((s[r, None] * (K @ (s[:, None] * Ud)) - Ud[r] * lt) ** 2).sum(0)
    est = sq.sqrt().max().item()
    print(f"{data} cap {cap}: {info.converged}/{k + 1} after {info.applies} products, reported {info.max_residual:.2e}, float64 {est:.2e}")
    assert est <= info.max_residual + 3e-6
    if cap >= 3 * (k + 1):
        assert info.converged == k + 1
    else:
        assert info.converged == k + 1 or 1e-6 < info.max_residual <= 2.5e-6
    ctx.close()


def test_c3_full_size_certificate_at_the_benchmark_capacity(fd, dev):
    """The 6-torus at N = 2^17 with the capacity the benchmark gives its solve (3 (k + 1) + 2 b, rounded up): Krylov blocks between
    Rayleigh-Ritz steps, which the smaller capacity of the other full-size certificate does not take."""
    from test_gpu_tc import full_size_certificate
    full_size_certificate(fd, dev, workloads.torus6(131072, seed=42), 2.0, 64, 32, 288, min_converged=65, sample=128)
