"""Batches in half storage on lattices of odd volume: a field of 12 bytes per site then ends in the middle of an 8-byte
word, and the next field of the batch must not start there (a site's two components are one 8-byte load)."""
import numpy as np
import pytest

import inputs
from oracle import wilson
from oracle.lattice import Lattice
from tests._util import to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,block", [((9, 15), (3, 3)), ((25, 21), (5, 3))])
def test_odd_volume_batch_in_half_storage(dims, block):
    import torch
    import paper_0707_4018_gb300 as mg
    U = inputs.hot_links(*dims, seed=31)
    p = mg.mg_default_params(levels=2, blocks=[block], Nv=[8], n_pass=2, precision=mg.MG_FP16, max_rhs=3)
    ctx = mg.Context.setup(to_dev(U), 0.5, dims, p)
    chi = np.stack([inputs.gaussian_source(*dims, seed=32, index=v) for v in range(3)])
    psi = torch.empty((3, dims[0] * dims[1], 2), dtype=torch.complex128, device="cuda")
    many = torch.empty_like(psi)
    stats = ctx.solve_batch(to_dev(chi), psi, 1e-10)
    mg.solve_multi([ctx], [to_dev(chi)], [many], 1e-10, nrhs=[3])
    for v in range(3):
        one = torch.empty_like(psi[0])
        single = ctx.solve(to_dev(chi[v]), one, 1e-10)
        # the same cycle on the same vector: the count of a vector by itself, whose field starts the buffer
        assert stats[v]["converged"] and abs(stats[v]["iters"] - single["iters"]) <= 1
        for got in (psi[v], many[v], one):
            r = chi[v] - wilson.apply_D(U, to_host(got), 0.5, Lattice(dims))
            assert np.linalg.norm(r) <= 1.05e-10 * np.linalg.norm(chi[v])
    ctx.close()
