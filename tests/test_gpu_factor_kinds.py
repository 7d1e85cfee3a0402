"""Batched solves whose masses move the exact coarsest solve from the cyclic reduction to the dense LU and back: the
captured batched V-cycle follows. A gauge transform of unit links makes the one-dimensional operator along a line
singular at m = -1 (its eigenvalues are 2 + m - exp(+-ik)), so that the reduction has no first pivots there, while the
two-dimensional operator is regular; a full-rank prolongator carries both to the coarse level."""
import numpy as np
import pytest

import inputs
from oracle import wilson
from oracle.lattice import Lattice
from tests._util import to_dev, to_host

pytestmark = pytest.mark.gpu


def test_batches_across_the_kinds_of_factors():
    import torch
    import paper_0707_4018_gb300 as mg
    dims = (8, 12)
    V = dims[0] * dims[1]
    g = np.exp(1j * np.random.default_rng(5).uniform(0, 2 * np.pi, (dims[1], dims[0])))
    U = np.stack([(g * np.roll(g, -1, 1).conj()).reshape(-1), (g * np.roll(g, -1, 0).conj()).reshape(-1)], -1)
    p = mg.mg_default_params(levels=2, blocks=[(1, 2)], Nv=[4], n_pass=1, max_rhs=2)
    ctx = mg.Context.setup(to_dev(U), 0.5, dims, p)
    chi = np.stack([inputs.gaussian_source(*dims, seed=23, index=v) for v in range(2)])
    for masses in ([0.5, 0.7], [-1.0, 0.7], [0.6, -1.0], [0.5, 0.7], None):
        before = mg.mg_kernel_launches()
        psi = torch.empty((2, V, 2), dtype=torch.complex128, device="cuda")
        ctx.solve_batch(to_dev(chi), psi, 1e-12, masses=masses)
        if masses is not None and -1.0 in masses:  # a dense factorisation takes two launches per column
            assert mg.mg_kernel_launches() - before > 2 * (2 * V - 1)
        for v in range(2):
            want = np.linalg.solve(wilson.dense_D(U, 0.5 if masses is None else masses[v], Lattice(dims)),
                                   chi[v].reshape(-1)).reshape(-1, 2)
            # residuals of 1e-12, |D| below 5 and |D^-1| below 2 at these masses
            assert np.linalg.norm(to_host(psi)[v] - want) <= 1e-11 * np.linalg.norm(want)
    ctx.close()
