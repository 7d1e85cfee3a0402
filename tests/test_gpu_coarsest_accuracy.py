"""The exact coarsest solve is as accurate as a dense LU with partial pivoting, also where the cyclic reduction loses
digits (indefinite operators): componentwise backward errors of random right-hand sides."""
import numpy as np
import pytest

import inputs
from tests._util import to_dev, to_host
from tests.test_gpu_coarsest_lines import _dense

pytestmark = pytest.mark.gpu

# The reduction is kept up to 2e-15 on the library's own vector, and vectors differ by a factor of a few; the LU of
# n <= 2048 columns has 1e-16 sqrt(n) times its growth, a small number for these operators (measured: up to 8e-15).
TOL = 2e-14


@pytest.mark.parametrize("m", [0.1, -1.0, -1.7])
@pytest.mark.parametrize("ext,N", [((4, 3), 8), ((5, 4), 6), ((4, 7), 5), ((9, 13), 8), ((16, 16), 8)])
def test_backward_error_of_the_exact_coarsest_solve(ext, N, m):
    import torch
    import paper_0707_4018_gb300 as mg
    dims = (2 * ext[0], 2 * ext[1])
    p = mg.mg_default_params(levels=2, blocks=[(2, 2)], Nv=[N], n_pass=1, nu_setup=2)
    ctx = mg.Context.setup(to_dev(inputs.hot_links(*dims, seed=17)), m, dims, p)
    A = _dense(to_host(ctx.coarse_op(1)), ext)
    for index in range(3):
        b = inputs.gaussian_spinor(ext[0] * ext[1], N, 43, index)
        x = torch.empty((ext[0] * ext[1], N), dtype=torch.complex128, device="cuda")
        ctx.coarsest_solve(to_dev(b), x)
        got, rhs = to_host(x).reshape(-1), b.reshape(-1)
        # the residual in extended precision: its own rounding is not counted
        r = np.abs(rhs - (A.astype(np.clongdouble) @ got.astype(np.clongdouble)))
        assert (r <= TOL * (np.abs(A) @ np.abs(got) + np.abs(rhs))).all()
    ctx.close()


def test_a_ring_of_more_lines_than_a_grid_has_rows():
    # a coarse lattice of 1 x 70000 sites with two dofs each
    import torch
    import paper_0707_4018_gb300 as mg
    dims, n, N = (2, 140000), 70000, 2
    p = mg.mg_default_params(levels=2, blocks=[(2, 2)], Nv=[N], n_pass=1, nu_setup=2, coarsest_lu_max=n * N)
    ctx = mg.Context.setup(to_dev(inputs.hot_links(*dims, seed=19)), 0.1, dims, p)
    Y = to_host(ctx.coarse_op(1))
    b = inputs.gaussian_spinor(n, N, 44, 0)
    x = torch.empty((n, N), dtype=torch.complex128, device="cuda")
    ctx.coarsest_solve(to_dev(b), x)
    x = to_host(x)
    r, size = b.astype(np.clongdouble), np.abs(b)
    for d, o in enumerate((0, 0, 0, 1, -1)):  # both hops along the extent of one lead back to the site
        v = np.roll(x, -o, 0)
        r = r - np.einsum("jab,jb->ja", Y[:, d].astype(np.clongdouble), v.astype(np.clongdouble))
        size = size + np.einsum("jab,jb->ja", np.abs(Y[:, d]), np.abs(v))
    assert (np.abs(r) <= TOL * size).all()
    ctx.close()
