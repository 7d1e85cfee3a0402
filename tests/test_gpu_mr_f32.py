"""The FP32 smoothing and coarse-apply kernels at the sizes where their launches change: lattices whose MR blocks
stride over the sites, odd coarse extents with a ragged last block, batches that are no multiple of the four vectors
a block takes, per-vector masses."""
import numpy as np
import pytest

import inputs
from tests._util import to_dev, to_host

pytestmark = pytest.mark.gpu


# (640, 512): more sites than the MR blocks of levels 0 and 1 cover in one pass; (44, 36), (20, 28): ragged blocks
@pytest.mark.parametrize("dims,blocks", [((640, 512), [(4, 4), (4, 4)]), ((44, 36), [(4, 4)]), ((20, 28), [(4, 4)])])
def test_fp32_vcycle_follows_fp64(dims, blocks):
    # the same near-null vectors in an FP64 and an FP32 context: one V-cycle agrees to FP32 accuracy (the bound of the
    # FP32 V-cycle against the oracle)
    import torch
    import paper_0707_4018_gb300 as mg
    V = dims[0] * dims[1]
    U = to_dev(inputs.hot_links(*dims, seed=23))
    b = to_dev(inputs.gaussian_source(*dims, seed=24))
    out = []
    for prec in (mg.MG_FP64, mg.MG_FP32):
        p = mg.mg_default_params(levels=len(blocks) + 1, blocks=blocks, Nv=[8] * len(blocks), n_pass=1, nu_setup=2,
                                 precision=prec, coarsest_tol=1e-12)
        ctx = mg.Context.setup(U, 0.4, dims, p)
        n, k = V, 2
        for l in range(len(blocks)):
            n, k = ctx.level_size(l)
            ctx.build_level(l, to_dev(np.stack([inputs.gaussian_spinor(n, k, 25 + l, i) for i in range(8)])))
        x = torch.empty((V, 2), dtype=torch.complex128, device="cuda")
        ctx.vcycle(b, x)
        out.append(to_host(x))
        ctx.close()
    assert np.linalg.norm(out[1] - out[0]) < 1e-5 * np.linalg.norm(out[0])


@pytest.mark.parametrize("nrhs", [3, 5, 8])
def test_fp32_batches_match_single_solves(nrhs):
    # (160, 128): the batched blocks take four vectors; each vector has its own mass
    import torch
    import paper_0707_4018_gb300 as mg
    dims = (160, 128)
    V = dims[0] * dims[1]
    p = mg.mg_default_params(levels=3, blocks=[(4, 4), (2, 2)], Nv=[8, 8], n_pass=2, precision=mg.MG_FP32, max_rhs=8,
                             coarsest_tol=0.2)
    ctx = mg.Context.setup(to_dev(inputs.hot_links(*dims, seed=26)), 0.3, dims, p)
    masses = [0.3 + 0.05 * v for v in range(nrhs)]
    chi = np.stack([inputs.gaussian_source(*dims, seed=27, index=v) for v in range(nrhs)])
    psi = torch.empty((nrhs, V, 2), dtype=torch.complex128, device="cuda")
    ctx.solve_batch(to_dev(chi), psi, 1e-12, masses=masses)
    one = torch.empty((V, 2), dtype=torch.complex128, device="cuda")
    for v in range(nrhs):
        ctx.clone(masses[v]).solve(to_dev(chi[v]), one, 1e-12)
        # both residuals at 1e-12, |D^-1| below 10 at these masses
        assert np.linalg.norm(to_host(psi)[v] - to_host(one)) < 1e-10 * np.linalg.norm(to_host(one))
    ctx.close()


@pytest.mark.parametrize("tol", [0.2, 1e-3, 1e-5])
@pytest.mark.parametrize("ext", [(41, 35), (64, 48)])
def test_fp32_large_coarsest_solve_meets_its_tolerance(ext, tol):
    # more dofs than the cluster and the shared-memory kernels take (9728), chunks of sites of uneven length
    import torch
    import paper_0707_4018_gb300 as mg
    dims = (4 * ext[0], 4 * ext[1])
    p = mg.mg_default_params(levels=2, blocks=[(4, 4)], Nv=[8], n_pass=1, precision=mg.MG_FP32, coarsest_tol=tol)
    ctx = mg.Context.setup(to_dev(inputs.hot_links(*dims, seed=28)), 0.2, dims, p)
    b = to_dev(inputs.gaussian_spinor(ext[0] * ext[1], 8, 29, 0))
    x, y = torch.empty_like(b), torch.empty_like(b)
    iters, _ = ctx.coarsest_solve(b, x)
    ctx.level_apply(1, x, y)
    # the kernel's true residual is taken in FP32: 40 products and sums per dof, rounding below 1e-5 of |A| |x|
    assert iters > 0
    assert float(torch.linalg.norm(b - y) / torch.linalg.norm(b)) <= tol + 1e-5
    ctx.close()
