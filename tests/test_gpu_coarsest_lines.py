"""The exact coarsest solve (cyclic reduction over lattice lines, dense LU behind it) against numpy's dense solve of
the exported coarse operator, at the ring shapes where it can go wrong: odd and even rings, rings of three, lines of
one or two sites, line lengths that are no multiple of the 16 x 16 tile, both axes, and masses at which the diagonal
blocks lose the positivity that the eliminations without exchanges rely on."""
import numpy as np
import pytest

import inputs
from tests._util import to_dev, to_host

pytestmark = pytest.mark.gpu

# coarse extents, dofs per coarse site
SHAPES = [((3, 3), 3), ((4, 3), 8), ((3, 4), 8), ((5, 4), 6), ((4, 7), 5), ((1, 8), 8), ((8, 1), 4), ((2, 6), 8),
          ((6, 2), 3), ((2, 2), 8), ((1, 2), 8), ((16, 16), 8), ((9, 13), 8)]


def _dense(Y, ext):
    n, nd, N, _ = Y.shape
    assert nd == 5 and n == ext[0] * ext[1]
    A = np.zeros((n, N, n, N), dtype=np.complex128)
    for j in range(n):
        x0, x1 = j % ext[0], j // ext[0]
        for d, (o0, o1) in enumerate([(0, 0), (1, 0), (-1, 0), (0, 1), (0, -1)]):
            src = (x0 + o0) % ext[0] + ext[0] * ((x1 + o1) % ext[1])
            A[j, :, src, :] += Y[j, d]
    return A.reshape(n * N, n * N)


@pytest.mark.parametrize("m", [0.1, -1.0, -1.7])
@pytest.mark.parametrize("ext,N", SHAPES)
def test_exact_coarsest_solve(ext, N, m):
    import torch
    import paper_0707_4018_gb300 as mg
    dims = (2 * ext[0], 2 * ext[1])
    U = inputs.hot_links(*dims, seed=17)
    p = mg.mg_default_params(levels=2, blocks=[(2, 2)], Nv=[N], n_pass=1, nu_setup=2, max_rhs=5)
    ctx = mg.Context.setup(to_dev(U), m, dims, p)
    A = _dense(to_host(ctx.coarse_op(1)), ext)
    b = inputs.gaussian_spinor(ext[0] * ext[1], N, 42, 0)
    x = torch.empty((ext[0] * ext[1], N), dtype=torch.complex128, device="cuda")
    iters, _ = ctx.coarsest_solve(to_dev(b), x)
    assert iters == 0
    got = to_host(x).reshape(-1)
    # componentwise backward error of the accepted factors (1e-12 on the library's own vector; a random vector's
    # differs by no more than a small factor), which bounds the residual entry by entry
    r = np.abs(b.reshape(-1) - A @ got)
    assert (r <= 1e-11 * (np.abs(A) @ np.abs(got) + np.abs(b.reshape(-1)))).all()
    want = np.linalg.solve(A, b.reshape(-1))
    cond = np.linalg.cond(A)
    assert np.linalg.norm(got - want) <= 1e-12 * cond * np.linalg.norm(want)
    ctx.close()


def test_batched_masses_match_single_solves():
    # five vectors at five masses (a factorisation each), and five at the context mass (one shared one)
    import torch
    import paper_0707_4018_gb300 as mg
    dims = (24, 20)
    U = inputs.hot_links(*dims, seed=18)
    p = mg.mg_default_params(levels=2, blocks=[(4, 4)], Nv=[8], n_pass=2, max_rhs=5)
    ctx = mg.Context.setup(to_dev(U), 0.3, dims, p)
    chi = np.stack([inputs.gaussian_source(*dims, seed=19, index=v) for v in range(5)])
    for masses in (None, [0.3, 0.4, 0.5, 0.7, 0.9]):
        psi = torch.empty((5, dims[0] * dims[1], 2), dtype=torch.complex128, device="cuda")
        ctx.solve_batch(to_dev(chi), psi, 1e-12, masses=masses)
        for v in range(5):
            one = torch.empty((dims[0] * dims[1], 2), dtype=torch.complex128, device="cuda")
            c = ctx if masses is None else ctx.clone(masses[v])
            c.solve(to_dev(chi[v]), one, 1e-12)
            err = np.linalg.norm(to_host(psi)[v] - to_host(one)) / np.linalg.norm(to_host(one))
            assert err < 1e-10  # both residuals at 1e-12, |D^-1| below 10 at these masses
    ctx.close()
