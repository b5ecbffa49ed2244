"""GPU parity of the fp32-grade block product kernel at the edges of its tiles and of its work split.

The kernel cuts the sequence of (row pair, column tile) steps into equal ranges, one per CTA: sizes below, at and above one step per
CTA, ranges that start or end inside a row pair, single and several column chunks, every column tile width (16, 32, 48, 64, and
blocks split into chunks of about equal width) and two to four pipeline stages (by the dimension).
Gate: the block product's relative Frobenius error 1e-5 (the exponents carry about 2^-20 from the fp32 Gram accumulation, the
sums 2^-22); the shares of a cut row pair are added in a fixed order, so results repeat bit for bit.
"""
import numpy as np
import pytest
import torch

import workloads
from oracle import dense

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,D,b,opts", [
    (127, 12, 33, {}), (129, 12, 48, {}), (513, 12, 16, {"flush": 1}), (2177, 12, 49, {}), (2304, 30, 64, {}),
    (3000, 60, 64, {}), (3000, 44, 48, {"jt_chunk": 3}), (4481, 28, 32, {"jt_chunk": 7}), (4481, 12, 96, {"flush": 5}), (4481, 12, 130, {}),
])
def test_block_product_edges(N, D, b, opts):
    import __graft_entry__ as g
    g.build()
    import paper_2609_38198_b200 as fd
    dev = torch.device("cuda:0")
    X = workloads.latent_torus(N, seed=N, D=D) if D > 12 else workloads.torus6(N, seed=N)
    beta = 2.0 if D == 12 else 0.3
    V = workloads.block(N, b, seed=b)
    ctx = fd.Context(torch.from_numpy(X).to(dev), b_max=b)
    ctx.set_option("path", fd.FD_PATH_TC)
    for k, v in opts.items():
        ctx.set_option(k, v)
    ctx.degree(beta, 1.0)
    Vd = fd.to_colmajor(V, dev)
    Y = ctx.apply(Vd)
    Y2 = ctx.apply(Vd)
    ctx.synchronize()
    assert torch.equal(Y, Y2)
    Yo = dense.apply(X, beta, 1.0, V)
    assert np.linalg.norm(Y.cpu().numpy().astype(np.float64) - Yo) <= 1e-5 * np.linalg.norm(Yo)
    ctx.close()


@pytest.mark.parametrize("N,D,beta", [(33, 3, 1.0), (385, 12, 2.0), (6401, 30, 1.0), (6401, 60, 0.3), (40003, 12, 2.0)])
def test_symmetric_row_sums_against_every_tile(N, D, beta):
    """The half-work degree passes against the passes that evaluate every tile (sym = 0): sizes with fewer steps than CTAs, ranges that
    start inside a resident pair, more than 64 streamed tiles (a reduction inside an item), one to four K slabs (norms per slab and
    norms after the last coordinate).  Both add the same fp32 kernel values: 64-term fp32 sums (2^-24 sqrt(64) each, random) then
    fp64 / fixed point, so 1e-6 relative holds with a margin."""
    import __graft_entry__ as g
    g.build()
    import paper_2609_38198_b200 as fd
    dev = torch.device("cuda:0")
    X = workloads.latent_torus(N, seed=N, D=D) if D > 12 else workloads.torus6(N, seed=N)[:, :D].copy()
    ctx = fd.Context(torch.from_numpy(X).to(dev), b_max=8)
    ctx.set_option("path", fd.FD_PATH_TC)
    q1, d1, s1, so1, sq1 = ctx.degree(beta, 1.0)
    q3, d3, s3, so3, sq3 = ctx.degree(beta, 1.0)
    assert torch.equal(q1, q3) and torch.equal(d1, d3) and torch.equal(s1, s3) and (so1, sq1) == (so3, sq3)
    ctx.set_option("sym", 0)
    q0, d0, s0, so0, sq0 = ctx.degree(beta, 1.0)
    for a, b in ((q1, q0), (d1, d0), (s1, s0)):
        assert ((a - b).abs() / b).max().item() <= 1e-6
    assert abs(so1 - so0) <= 1e-6 * (so0 + N) and abs(sq1 - sq0) <= 1e-6 * (sq0 + N)
    ctx.close()


@pytest.mark.parametrize("N,D,b,splits", [
    (1, 2, 1, 0), (255, 3, 5, 0), (257, 4, 24, 0), (2049, 2, 8, 0), (4200, 4, 16, 1), (4200, 12, 33, 1), (4200, 16, 64, 1), (2305, 30, 48, 0), (5003, 12, 100, 0),
])
def test_direct_difference_edges(N, D, b, splits):
    """Direct-difference kernels at the edges of their row tiles (256) and column tiles (64), of the work ranges (fewer steps than CTAs,
    cuts inside row tiles; splits = 1: whole row tiles, so more than 32 column tiles are summed in two levels), of the column
    widths (4 ... 64, balanced chunks) and of the four-row / two-row layouts.  fp32 products against float64: 1e-6 relative Frobenius
    (2^-24 per operation, at most 64 x 32 terms per fp32 level, random signs)."""
    import __graft_entry__ as g
    g.build()
    import paper_2609_38198_b200 as fd
    dev = torch.device("cuda:0")
    X = workloads.gaussian_cloud(N, D, seed=N, scale=0.7)
    V = workloads.block(N, b, seed=b)
    ctx = fd.Context(torch.from_numpy(X).to(dev), b_max=b)
    ctx.set_option("path", fd.FD_PATH_SIMT)
    ctx.set_option("splits", splits)
    beta = 0.8
    q, d, s, so, so2 = ctx.degree(beta, 1.0)
    Y = ctx.apply(fd.to_colmajor(V, dev))
    Y2 = ctx.apply(fd.to_colmajor(V, dev))
    ctx.synchronize()
    assert torch.equal(Y, Y2)
    qo, do, s_o, soo, so2o = dense.degree(X, beta, 1.0)
    assert np.abs(q.cpu().numpy() / qo - 1).max() <= 1e-6 and np.abs(d.cpu().numpy() / do - 1).max() <= 2e-6
    assert abs(so2 - so2o) <= 2e-6 * (so2o + N)
    Yo = dense.apply(X, beta, 1.0, V)
    assert np.linalg.norm(Y.cpu().numpy().astype(np.float64) - Yo) <= 1e-6 * np.linalg.norm(Yo)
    ctx.close()


@pytest.mark.parametrize("path,m,b_max", [(1, 1, 16), (1, 15, 16), (1, 16, 16), (2, 33, 64), (2, 64, 64), (2, 31, 32), (2, 70, 64)])
def test_extension_column_chunks(path, m, b_max):
    """Out-of-sample extension, whose product carries the denominator as one more column: block buffers just wide enough, one column
    too narrow, several chunks.  Ratio of two products of the same kernel values: 1e-5 entrywise of the largest value."""
    import __graft_entry__ as g
    g.build()
    import paper_2609_38198_b200 as fd
    from oracle import nystrom
    dev = torch.device("cuda:0")
    X, Z = workloads.torus6(1500, seed=5), workloads.torus6(401, seed=6)
    psi, lam = workloads.block(1500, m, seed=2), np.linspace(1.0, 0.3, m)
    ctx = fd.Context(torch.from_numpy(X).to(dev), b_max=b_max)
    ctx.set_option("path", path)
    q, d, s, so, so2 = ctx.degree(1.0, 1.0)
    out = ctx.nystrom(torch.from_numpy(Z).to(dev), fd.to_colmajor(psi, dev), lam).cpu().numpy()
    qo = dense.degree(X, 1.0, 1.0)[0]
    ref = nystrom.extend(X, qo, 1.0, 1.0, psi.astype(np.float64), lam, Z)
    assert np.abs(out - ref).max() <= 1e-5 * np.abs(ref).max()
    ctx.close()


@pytest.mark.parametrize("N,path,D,const", [(700, 1, 32, 0.0), (700, 2, 32, 2.5), (700, 2, 60, -1.0), (5, 1, 20, 1.0)])
def test_coordinates_that_all_points_share(N, path, D, const):
    """Constant coordinates among the points (padding, a frozen degree of freedom) are left out of the kernels' work: same products and
    degrees, and external rows that differ from the points in such a coordinate keep their distance.  Gates: 1e-5 for the block
    products as elsewhere; degrees 1e-6 / 2e-5 (direct / Gram form)."""
    import __graft_entry__ as g
    g.build()
    import paper_2609_38198_b200 as fd
    dev = torch.device("cuda:0")
    rng = np.random.default_rng(1)
    X = np.full((N, D), const, dtype=np.float32)
    used = np.sort(rng.choice(D, 12, replace=False))
    X[:, used] = workloads.torus6(N, seed=3)
    Z = X[: min(N, 300)].copy()
    Z[:, used] += 0.1 * rng.standard_normal((len(Z), 12)).astype(np.float32)
    Z[::2, (used[0] + 1) % D if (used[0] + 1) % D not in used else [k for k in range(D) if k not in used][0]] += 0.5
    b, beta = 8, 1.0
    V = workloads.block(N, b, seed=2)
    l = rng.uniform(0.5, 2.0, len(Z)).astype(np.float32)
    ctx = fd.Context(torch.from_numpy(X).to(dev), b_max=b)
    ctx.set_option("path", path)
    q, d, s, so, so2 = ctx.degree(beta, 1.0)
    qo, do, s_o, soo, so2o = dense.degree(X, beta, 1.0)
    assert np.abs(q.cpu().numpy() / qo - 1).max() <= (1e-6 if path == 1 else 2e-5)
    Y = ctx.apply(fd.to_colmajor(V, dev)).cpu().numpy().astype(np.float64)
    Yo = dense.apply(X, beta, 1.0, V)
    assert np.linalg.norm(Y - Yo) <= 1e-5 * np.linalg.norm(Yo)
    for left in (None, l):
        R = ctx.apply_general(beta, fd.to_colmajor(V, dev), left=None if left is None else torch.from_numpy(left).to(dev), Xrow=torch.from_numpy(Z).to(dev))
        K = np.exp(-beta * ((Z[:, None, :].astype(np.float64) - X[None].astype(np.float64)) ** 2).sum(-1))
        Ro = (1.0 if left is None else left[:, None].astype(np.float64)) * (K @ V.astype(np.float64))
        assert np.linalg.norm(R.cpu().numpy().astype(np.float64) - Ro) <= 1e-5 * np.linalg.norm(Ro)
    ctx.close()


def _gpu_kernel_rows(Xd, rows, beta):
    """float64 rows of the kernel by direct differences, on the GPU."""
    return torch.exp(-beta * torch.cdist(Xd[rows], Xd, compute_mode="donot_use_mm_for_euclid_dist") ** 2)


def _gpu_degree(Xd, beta):
    """q, d, sum of q, sum of squares of the kernel, in float64 on the GPU."""
    N = Xd.shape[0]
    parts = [torch.arange(i, min(N, i + 2048), device=Xd.device) for i in range(0, N, 2048)]
    q, so2 = [], 0.0
    for r in parts:
        K = _gpu_kernel_rows(Xd, r, beta)
        q.append(K.sum(1))
        so2 += (K * K).sum().item()
    q = torch.cat(q)
    d = torch.cat([_gpu_kernel_rows(Xd, r, beta) @ (1.0 / q) for r in parts]) / q
    return q, d, q.sum().item(), so2


def _far_points(kind, N, rng):
    """Points of which many pairs are far apart, and a bandwidth for the Gram-form kernels and one for the direct ones."""
    t = rng.random((N, 2)) * 2 * np.pi
    if kind == "manifold":
        return workloads.latent_torus(N, seed=42), 5.0, None
    if kind == "torus2":
        X, bg, bd = np.concatenate([np.cos(t), np.sin(t)], 1), None, 100.0
    elif kind == "circle":
        X, bg, bd = np.concatenate([np.cos(t[:, :1]), np.sin(t[:, :1])], 1), None, 400.0
    elif kind == "clusters":                       # 5 clusters of similar size far apart, 12 coordinates (direct: 7)
        X = (rng.standard_normal((5, 12)) * 2.0)[rng.choice(5, N, p=(0.25, 0.25, 0.2, 0.15, 0.15))] + 0.1 * rng.standard_normal((N, 12))
        bg, bd = 0.8, None
    elif kind == "clusters7":
        X = (rng.standard_normal((9, 7)) * 2.0)[rng.choice(9, N)] + 0.1 * rng.standard_normal((N, 7))
        bg, bd = None, 30.0
    elif kind == "line":                           # one coordinate that matters
        X = np.concatenate([8.0 * rng.random((N, 1)), 0.01 * rng.standard_normal((N, 2))], 1)
        bg, bd = 3.4, 100.0
    else:                                          # a third of the points coincide, between two blobs
        X, bg, bd = np.zeros((N, 4)), 2.0, 40.0
        X[N // 3:] = 0.02 * rng.standard_normal((N - N // 3, 4))
        X[N // 3:, 0] += 3.9 * rng.choice((-1.0, 1.0), N - N // 3)
    return X.astype(np.float32), bg, bd


@pytest.mark.parametrize("N,kind", [(32768, "manifold"), (32769, "clusters"), (33001, "line"), (32900, "duplicates")])
def test_far_tiles_are_left_out(N, kind):
    """Data with many pairs beyond the exponent limit: the points are ordered, tiles without near pairs left out.  Same results as float64
    sums (gates of the Gram-form path: degrees 2e-5, product 1e-5; what is left out is below 2^-40 of a kernel value's
    maximum), bit-identical repeats, lists remade when the bandwidth changes, external rows against ordered columns, the same
    operator applied through other precision modes and without the symmetric passes, and a product at a bandwidth that no degree
    pass has seen, which takes every tile."""
    import __graft_entry__ as g
    g.build()
    import paper_2609_38198_b200 as fd
    dev = torch.device("cuda:0")
    X, beta, _ = _far_points(kind, N, np.random.default_rng(N))
    Xt = torch.from_numpy(X).to(dev)
    Xd = Xt.double()
    b = 20
    V = fd.to_colmajor(workloads.block(N, b, seed=2), dev)
    Vd = V.double()
    rows = torch.arange(0, N, 61, device=dev)
    ctx = fd.Context(Xt, b_max=b)
    ctx.set_option("path", fd.FD_PATH_TC)
    ctx.set_option("tc_max_mag", 1e4)
    qo, do, soo, so2o = _gpu_degree(Xd, beta)
    sd = 1.0 / (qo * do.sqrt())
    Yo = sd[rows, None] * (_gpu_kernel_rows(Xd, rows, beta) @ (sd[:, None] * Vd))
    shares = []
    for bt in (beta, 0.1 * beta, beta):
        q, d, s, so, so2 = ctx.degree(bt, 1.0)
        Y, Y2, Yf = ctx.apply(V), ctx.apply(V), ctx.apply(V, prec=fd.FD_PREC_FAST)
        shares.append(ctx.get_option("tile_share"))
        assert torch.equal(Y, Y2)
        if bt != beta:
            continue
        assert (q.double() / qo - 1).abs().max().item() <= 2e-5 and (d.double() / do - 1).abs().max().item() <= 4e-5
        assert abs(so - (soo - N)) <= 2e-5 * soo and abs(so2 - (so2o - N)) <= 4e-5 * so2o
        assert ((Y[rows].double() - Yo).norm() / Yo.norm()).item() <= 1e-5
        assert ((Yf[rows].double() - Yo).norm() / Yo.norm()).item() <= 3e-3
        R = ctx.apply_general(bt, V, Xrow=Xt[:77].contiguous()).double()
        Ro = _gpu_kernel_rows(Xd, torch.arange(77, device=dev), bt) @ Vd
        assert ((R - Ro).norm() / Ro.norm()).item() <= 1e-5
    assert shares[0] < 0.9 and shares[2] == shares[0], shares
    Z = ctx.apply_general(0.7 * beta, V)[rows].double()
    Zo = _gpu_kernel_rows(Xd, rows, 0.7 * beta) @ Vd
    assert ((Z - Zo).norm() / Zo.norm()).item() <= 1e-5
    ctx.set_option("sym", 0)
    q0, d0, s0, _, _ = ctx.degree(beta, 1.0)
    assert ((q0 - q).abs() / q0).max().item() <= 2e-6
    ctx.close()


@pytest.mark.parametrize("N,kind,b", [(16384, "torus2", 16), (16385, "circle", 5), (17001, "clusters7", 40), (33001, "duplicates", 24),
                                      (20011, "torus2", 70), (40000, "line", 3), (16400, "torus2", 1), (17000, "clusters7", 8), (16385, "clusters7", 16),
                                      (19999, "torus2", 24), (18001, "torus2", 32), (16640, "clusters7", 32), (17920, "torus2", 48), (16386, "torus2", 64),
                                      (17003, "clusters7", 64), (17100, "clusters7", 3),
                                      (16777, "circle", 4)])
def test_far_tiles_are_left_out_of_direct_passes(N, kind, b):
    """Direct-difference passes without the tiles whose kernel values are exactly zero: degrees, sums and products against float64 sums
    (gate 1e-6 of that family), bit-identical repeats, bandwidths with and without lists, and a product at a bandwidth that no
    degree pass has seen."""
    import __graft_entry__ as g
    g.build()
    import paper_2609_38198_b200 as fd
    dev = torch.device("cuda:0")
    X, _, beta = _far_points(kind, N, np.random.default_rng(N))
    Xt = torch.from_numpy(X).to(dev)
    Xd = Xt.double()
    V = fd.to_colmajor(workloads.block(N, b, seed=2), dev)
    rows = torch.arange(0, N, 97, device=dev)
    ctx = fd.Context(Xt, b_max=b)
    ctx.set_option("path", fd.FD_PATH_SIMT)
    shares = []
    for bt in (beta, 0.01 * beta, beta):
        q, d, s, so, so2 = ctx.degree(bt, 1.0)
        Y, Y2 = ctx.apply(V), ctx.apply(V)
        shares.append(ctx.get_option("tile_share"))
        assert torch.equal(Y, Y2)
        qo, do, soo, so2o = _gpu_degree(Xd, bt)
        assert (q.double() / qo - 1).abs().max().item() <= 1e-6 and (d.double() / do - 1).abs().max().item() <= 2e-6
        assert abs(so - (soo - N)) <= 1e-6 * soo and abs(so2 - (so2o - N)) <= 1e-6 * so2o
        sd = s.double()
        Yo = sd[rows, None] * (_gpu_kernel_rows(Xd, rows, bt) @ (sd[:, None] * V.double()))
        assert ((Y[rows].double() - Yo).norm() / Yo.norm()).item() <= 1e-6
    assert shares[0] < 0.8 and shares[1] == 1.0 and shares[2] == shares[0], shares
    Z = ctx.apply_general(0.7 * beta, V)[rows].double()
    Zo = _gpu_kernel_rows(Xd, rows, 0.7 * beta) @ V.double()
    assert ((Z - Zo).norm() / Zo.norm()).item() <= 1e-6
    ctx.close()


@pytest.mark.parametrize("N", [16385, 16397, 33000])
def test_listed_passes_at_any_scale_of_the_data(N):
    """Coordinates of the order of 1e18: scaled by a power of two (and beta by its inverse square), every result is that of the data of
    order one, bit for bit; the points that fill up the last tile count nowhere."""
    import __graft_entry__ as g
    g.build()
    import paper_2609_38198_b200 as fd
    dev = torch.device("cuda:0")
    X = 1.2 * torch.from_numpy(workloads.torus2(N, seed=5)).to(dev)      # (1e18 = 0.867 * 2^60: inside the data)
    V = fd.to_colmajor(workloads.block(N, 5, seed=2), dev)
    got = []
    for p in (0, 60):
        ctx = fd.Context(X * 2.0 ** p, b_max=8)
        ctx.set_option("path", fd.FD_PATH_SIMT)
        out = ctx.degree(40.0 * 2.0 ** (-2 * p), 1.0)
        got.append((*out, ctx.apply(V)))
        assert ctx.get_option("tile_share") < 0.8
        ctx.close()
    for a, b in zip(*got):
        assert torch.equal(a, b) if torch.is_tensor(a) else a == b
