"""Routes chosen by size: narrow products of small sets in one launch, products over the tiles that hold near pairs, solves with blocks of
many widths."""
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


def _kernel_rows(Zd, Xd, beta):
    return torch.exp(-beta * torch.cdist(Zd, Xd, compute_mode="donot_use_mm_for_euclid_dist") ** 2)


@pytest.mark.parametrize("N,D,b", [(1, 1, 1), (3, 2, 4), (7, 5, 8), (63, 4, 16), (64, 8, 3), (65, 3, 9), (255, 2, 8), (257, 7, 16), (2047, 2, 8),
                                   (2048, 3, 16), (2049, 4, 16), (3071, 2, 1), (3072, 4, 8), (3073, 4, 8)])
def test_small_narrow_products(fd, dev, N, D, b):
    """Up to 3072 points with up to 8 coordinates and 8 columns (2048 and 16): one launch, sums inside a cluster.  Square products with scalings on both sides, a
    right block and an output with a pitch of their own, external rows, a replay from a graph with another right block in the same buffer (the bits of
    the eager call).  Gate 1e-6 of the direct-difference family."""
    rng = np.random.default_rng(N + 7 * b)
    X = torch.from_numpy(rng.standard_normal((N, D)).astype(np.float32)).to(dev)
    beta, ld = 0.7, N + 5
    V = torch.empty((b, ld), device=dev)[:, 3:3 + N].t()
    V.copy_(torch.from_numpy(rng.standard_normal((N, b)).astype(np.float32)))
    left, right = (torch.rand(N, device=dev) + 0.5 for _ in range(2))
    Xd, Vd = X.double(), V.double()
    ctx = fd.Context(X, b_max=b)
    Y = torch.zeros((b, ld), device=dev)[:, 2:2 + N].t()
    ctx.apply_general(beta, V, left=left, right=right, out=Y)
    ref = left.double()[:, None] * (_kernel_rows(Xd, Xd, beta) @ (right.double()[:, None] * Vd))
    assert ctx.get_option("last_path") == fd.FD_PATH_SIMT
    assert ((Y.double() - ref).norm() / ref.norm()).item() <= 1e-6
    for M in (1, min(N, 33), min(N, 129)):
        Z = X[:M].contiguous() + 0.01
        R = ctx.apply_general(beta, V, Xrow=Z)
        Ro = _kernel_rows(Z.double(), Xd, beta) @ Vd
        assert ((R.double() - Ro).norm() / Ro.norm()).item() <= 1e-6
    ctx.close()
    stream, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    ctx = fd.Context(X, b_max=b, stream=stream)
    ctx.apply_general(beta, V, left=left, right=right, out=Y)
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=stream):
        ctx.apply_general(beta, V, left=left, right=right, out=Y)
    V.mul_(-0.7).add_(0.2)
    torch.cuda.synchronize()
    want = ctx.apply_general(beta, V, left=left, right=right)
    Y.zero_()
    torch.cuda.synchronize()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(Y, want)
    ctx.close()


@pytest.mark.parametrize("kind", ["direct", "gram"])
@pytest.mark.parametrize("N", [16384, 33023])
def test_products_over_noted_tiles(fd, dev, kind, N):
    """The tiles that a degree pass noted: the product with them is that over all tiles (to the rounding of another order of the sums), and over
    clearly fewer than the boxes leave.  (A context in which a product has been recorded into a graph takes no notes: it lists by the boxes.)"""
    if kind == "direct":
        X, beta, path = workloads.torus2(N, seed=1), 60.0, fd.FD_PATH_SIMT
    else:
        if N < 32768:
            pytest.skip("lists of more than 8 coordinates start at 32768 points")
        X, beta, path = workloads.latent_torus(N, seed=42), 3.0, fd.FD_PATH_TC
    Xt = torch.from_numpy(X).to(dev)
    V = fd.to_colmajor(workloads.block(N, 20, seed=3), dev)
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    ctx, plain, boxes = fd.Context(Xt, b_max=20), fd.Context(Xt, b_max=20), fd.Context(Xt, b_max=20, stream=stream)
    for c in (ctx, plain, boxes):
        c.set_option("path", path)
        c.set_option("tc_max_mag", 1e4)
    s = ctx.degree(beta, 1.0)[2]
    share = ctx.get_option("tile_share")
    Y = ctx.apply_general(beta, V, left=s, right=s)
    Z = plain.apply_general(beta, V, left=s, right=s)            # (no degree pass: every tile)
    assert ((Y - Z).norm() / Z.norm()).item() <= 2e-6
    torch.cuda.synchronize()
    B = boxes.apply_general(0.01 * beta, V)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        boxes.apply_general(0.01 * beta, V, out=B)
    torch.cuda.synchronize()
    boxes.degree(beta, 1.0)
    B = boxes.apply_general(beta, V, left=s, right=s)
    torch.cuda.synchronize()
    assert ((B - Z).norm() / Z.norm()).item() <= 2e-6
    assert share < 0.9 * boxes.get_option("tile_share") and boxes.get_option("tile_share") < 0.9
    ctx.degree(0.5 * beta, 1.0)
    assert torch.equal(ctx.degree(beta, 1.0)[2], s) and ctx.get_option("tile_share") == share
    assert torch.equal(ctx.apply_general(beta, V, left=s, right=s), Y)
    ctx.close(); plain.close(); boxes.close()


@pytest.mark.parametrize("D,N,beta,kind,listed", [(4, 16384, 30.0, "direct", True), (4, 20000, 20.0, "direct", False), (6, 16384, 20.0, "direct", False),
                                                  (4, 32767, 22.0, "direct", True), (4, 32767, 10.0, "gram", True), (4, 16384, 10.0, "gram", False),
                                                  (3, 24000, 17.0, "gram", True), (3, 16384, 24.0, "gram", True)])
def test_an_order_that_would_not_stay_is_not_made(fd, dev, D, N, beta, kind, listed):
    """Below 32768 points, with 0.4 to 0.8 of the pairs far: the points of flat tori and of a sphere are ordered where lists come out of it; else the first degree pass
    launches what one without far pairs does, and the sampling of the pairs."""
    rng = np.random.default_rng(7)
    a, z = rng.random((N, D // 2)) * 2 * np.pi, rng.standard_normal((N, 3))
    X = z / np.linalg.norm(z, axis=1, keepdims=True) if D == 3 else np.concatenate([np.cos(a), np.sin(a)], 1)
    X = torch.from_numpy(X.astype(np.float32)).to(dev)
    launches = []
    for bt in (0.01 * beta, beta):
        ctx = fd.Context(X, b_max=8)
        ctx.set_option("path", fd.FD_PATH_SIMT if kind == "direct" else fd.FD_PATH_TC)
        ctx.set_option("tc_max_mag", 1e4)
        n = fd.fd_launch_count()
        ctx.degree(bt, 1.0)
        launches.append(fd.fd_launch_count() - n)
        share = ctx.get_option("tile_share")
        ctx.close()
    assert (share < 0.9) == listed
    assert listed or launches[1] <= launches[0] + (1 if kind == "direct" else 2)       # (Gram form: sampled for the product's limit and for the sums')


@pytest.mark.parametrize("N,k,b,m_max", [(24, 5, 7, 24), (65, 12, 16, 65), (300, 20, 1, 64), (300, 9, 33, 96), (700, 30, 64, 224), (900, 20, 70, 210),
                                         (512, 8, 16, 59)])
def test_solves_with_blocks_of_many_widths(fd, dev, N, k, b, m_max):
    """Blocks of one to 70 columns, bases that leave room for one block or for several beside twice the wanted pairs and bases that span everything.
    Eigenvalues to 1e-6, residuals in float64 to 5e-6, vectors orthonormal to 1e-5, against the dense matrix; the same from a warm start
    (no block ahead of the Rayleigh-Ritz step there)."""
    X = workloads.latent_torus(N, seed=42)
    beta = 0.6
    Xd = torch.from_numpy(X).to(dev).double()
    K = _kernel_rows(Xd, Xd, beta)
    q = K.sum(1)
    d = (K @ (1.0 / q)) / q
    s = 1.0 / (q * d.sqrt())
    M = s[:, None] * K * s[None]
    lam = torch.linalg.eigvalsh(M).flip(0)[:k + 1].cpu().numpy()
    ctx = fd.Context(torch.from_numpy(X).to(dev), b_max=b, m_max=m_max)
    ctx.degree(beta, 1.0)
    Q0 = None
    for _ in range(2):
        ev, U, info = ctx.eigs(k, b, Q0=Q0)
        assert np.abs(np.array(ev) - lam).max() <= 1e-6 * lam[0]
        Ud = U.double()
        assert (Ud.t() @ Ud - torch.eye(k + 1, device=dev)).abs().max().item() <= 1e-5
        assert (M @ Ud - Ud * torch.tensor(ev, device=dev)).norm(dim=0).max().item() <= 5e-6 * lam[0]
        Q0 = U
    ctx.close()


@pytest.mark.parametrize("kind,N", [("gram", 33023), ("direct", 16384), ("direct", 33000)])
def test_a_workspace_without_room_for_notes(fd, dev, kind, N, monkeypatch):
    """The smallest workspace that fd_create takes is smaller than what fd_workspace_bytes asks for where that has room for notes.  Gram form: tiles by
    the boxes, direct differences: every tile; the same results as with notes (to the rounding of another order of the sums), degrees and products
    in either precision, after a change of bandwidth too, and nothing beyond the workspace's end is touched."""
    from paper_2609_38198_b200 import binding
    if kind == "direct":
        X, beta, path = workloads.torus2(N, seed=1), 60.0, fd.FD_PATH_SIMT
    else:
        X, beta, path = workloads.latent_torus(N, seed=42), 3.0, fd.FD_PATH_TC
    Xt = torch.from_numpy(X).to(dev)
    V = fd.to_colmajor(workloads.block(N, 20, seed=3), dev)
    asked = fd.fd_workspace_bytes(N, X.shape[1], 20, 0)

    def context(size):
        monkeypatch.setattr(binding, "fd_workspace_bytes", lambda *a: size)
        ctx = fd.Context(Xt, b_max=20)
        ctx.set_option("path", path)
        ctx.set_option("tc_max_mag", 1e4)
        return ctx

    refused, taken = asked // 2, asked
    while taken - refused > 256:
        size = (refused + taken) // 512 * 256
        try:
            context(size).close()
            taken = size
        except fd.FdError as e:
            assert e.status == fd.FD_ERR_WORKSPACE
            refused = size
    assert taken < asked - N * N // 32768
    small, full = context(taken), context(asked)
    end = small._ws[-small._ws.data_ptr() % 256 + taken:]
    end.fill_(0x5A)
    for bt in (beta, 0.4 * beta, beta):
        (q, d, s, so, so2), (qf, df, sf, sof, so2f) = small.degree(bt, 1.0), full.degree(bt, 1.0)
        assert max(((a - b).abs() / b).max().item() for a, b in ((q, qf), (d, df), (s, sf))) <= 2e-6
        assert abs(so - sof) <= 1e-6 * sof and abs(so2 - so2f) <= 1e-6 * so2f
        Y, Z = small.apply(V), full.apply(V)
        assert ((Y - Z).norm() / Z.norm()).item() <= 2e-6 and torch.equal(small.apply(V), Y)
        Y, Z = small.apply(V, prec=fd.FD_PREC_FAST), full.apply(V, prec=fd.FD_PREC_FAST)
        assert ((Y - Z).norm() / Z.norm()).item() <= 2e-5
    share, noted = small.get_option("tile_share"), full.get_option("tile_share")
    assert noted < 0.8 and (share == 1.0 if kind == "direct" else noted < share < 0.9)
    assert bool((end == 0x5A).all())
    small.close(); full.close()
