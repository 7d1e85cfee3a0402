"""The 4d block kernels at the edges of their tiles: Gram-Schmidt and transfers of blocks of 512 and of 12 sites with
odd vector counts against the oracle, and batches whose last group of vectors is short against single solves."""
import numpy as np
import pytest

import inputs
from oracle import coarse, setup, transfer
from oracle.lattice import Lattice
from tests._util import rel_err, to_dev, to_host

pytestmark = pytest.mark.gpu

SHAPES = [((8, 4, 4, 8), (8, 4, 4, 4), 5), ((6, 4, 2, 4), (3, 2, 1, 2), 3)]


def _params(block, nv, **kw):
    import paper_0707_4018_gb300 as mg
    return mg.mg_default_params(levels=2, blocks=[block], Nv=[nv], chiral_split=1, n_pass=1, nu_setup=4, **kw)


@pytest.mark.parametrize("dims,block,nv", SHAPES)
def test_block_kernels_match_oracle(dims, block, nv):
    import torch
    import paper_0707_4018_gb300 as mg
    lat = Lattice(dims)
    U = inputs.su3_links(dims, seed=23)
    ctx = mg.Context.setup(to_dev(U), 0.1, dims, _params(block, nv))
    vecs = np.stack([inputs.gaussian_spinor(lat.volume, 12, 50, k) for k in range(nv)])
    ctx.build_level(0, to_dev(vecs))
    hier = setup.Hierarchy(coarse.WilsonOperator(U, 0.1, lat, 3),
                           setup.MGParams(levels=2, blocks=(block,), Nv=(nv,), chiral_split=True))
    hier.build_level(0, list(vecs))
    # two passes of FP64 Gram-Schmidt on independent Gaussian vectors: both sides orthonormal to a few hundred eps
    want = np.stack([transfer.from_blocks(hier.P[0][:, :, c], hier.blk[0], 12) for c in range(2 * nv)])
    assert np.abs(to_host(ctx.prolongator(0)) - want).max() < 1e-12
    n_c, k_c = ctx.level_size(1)
    r = inputs.gaussian_spinor(lat.volume, 12, 51, 0)
    rc = torch.empty((n_c, k_c), dtype=torch.complex128, device="cuda")
    ctx.restrict(0, to_dev(r), rc)
    assert rel_err(to_host(rc), hier.restrict(0, r)) < 1e-13
    e = inputs.gaussian_spinor(n_c, k_c, 52, 0)
    f = torch.empty((lat.volume, 12), dtype=torch.complex128, device="cuda")
    ctx.prolong(0, to_dev(e), f)
    assert rel_err(to_host(f), hier.prolong(0, e)) < 1e-13
    ctx.close()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("nb", [2, 5])
@pytest.mark.parametrize("dims,block,nv", SHAPES)
def test_batched_transfers_match_single_ones(dims, block, nv, nb, precision):
    # a vector whose coarse correction came from another one's block, or from none, takes the iterations of the
    # smoother alone; with the right one both forms run the same cycle up to rounding
    import torch
    import paper_0707_4018_gb300 as mg
    lat = Lattice(dims)
    U = inputs.su3_links(dims, seed=24)
    ctx = mg.Context.setup(to_dev(U), 0.05, dims, _params(block, nv, precision=precision, coarsest_tol=1e-6,
                                                          coarsest_max_iter=400, max_rhs=nb))
    chi = to_dev(np.stack([inputs.gaussian_spinor(lat.volume, 12, 53, k) for k in range(nb)]))
    psi, one = torch.empty_like(chi), torch.empty_like(chi[0])
    stats = ctx.solve_batch(chi, psi, 1e-11)
    for k in range(nb):
        st = ctx.solve(chi[k], one, 1e-11)
        assert st["converged"] and stats[k]["converged"]
        assert abs(st["iters"] - stats[k]["iters"]) <= 1
        # both residuals are below 1e-11, times the condition number (|D| <= 8.05, sigma_min > 0.02 assumed)
        assert rel_err(to_host(psi[k]), to_host(one)) < 1e-8
    ctx.close()
