"""Routes chosen by size: products over the tiles that hold near pairs."""
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


@pytest.mark.parametrize("kind", ["direct", "gram"])
@pytest.mark.parametrize("N", [16384, 33023])
def test_products_over_noted_tiles(fd, dev, kind, N):
    """The tiles that a degree pass noted: the product with them is that over all tiles (to the rounding of another order of the sums), and never
    over more of them than the boxes leave."""
    if kind == "direct":
        X, beta, path = workloads.torus2(N, seed=1), 60.0, fd.FD_PATH_SIMT
    else:
        if N < 32768:
            pytest.skip("lists of more than 8 coordinates start at 32768 points")
        X, beta, path = workloads.latent_torus(N, seed=42), 3.0, fd.FD_PATH_TC
    Xt = torch.from_numpy(X).to(dev)
    V = fd.to_colmajor(workloads.block(N, 20, seed=3), dev)
    ctx, plain = (fd.Context(Xt, b_max=20) for _ in range(2))
    for c in (ctx, plain):
        c.set_option("path", path)
        c.set_option("tc_max_mag", 1e4)
    s = ctx.degree(beta, 1.0)[2]
    share = ctx.get_option("tile_share")
    assert share < 0.8
    Y = ctx.apply_general(beta, V, left=s, right=s)
    Z = plain.apply_general(beta, V, left=s, right=s)            # (no degree pass: every tile)
    assert ((Y - Z).norm() / Z.norm()).item() <= 2e-6
    ctx.degree(0.5 * beta, 1.0)
    assert torch.equal(ctx.degree(beta, 1.0)[2], s) and ctx.get_option("tile_share") == share
    assert torch.equal(ctx.apply_general(beta, V, left=s, right=s), Y)
    ctx.close(); plain.close()
