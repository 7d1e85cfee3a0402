"""The FP64 smoothing kernels at the sizes where their launches change, against minimal residual steps formed from the
operator's apply: coarse extents with a ragged last block, lattices whose blocks stride over the sites."""
import pytest

import inputs
from tests._util import to_dev

pytestmark = pytest.mark.gpu


# level 1 of (640, 512): more sites than the MR blocks cover in one pass; (40, 24), (24, 8): 60 and 12 sites, ragged
@pytest.mark.parametrize("level", [0, 1])
@pytest.mark.parametrize("dims,nu", [((640, 512), 3), ((40, 24), 4), ((40, 24), 1), ((24, 8), 3)])
def test_fp64_smoothing_matches_its_definition(dims, nu, level):
    import torch
    import paper_0707_4018_gb300 as mg
    p = mg.mg_default_params(levels=3, blocks=[(4, 4), (2, 2)], Nv=[8, 8], n_pass=1, nu_setup=2)
    ctx = mg.Context.setup(to_dev(inputs.hot_links(*dims, seed=33)), 0.3, dims, p)
    n, k = (dims[0] * dims[1], 2) if level == 0 else ctx.level_size(1)
    b = to_dev(inputs.gaussian_spinor(n, k, 34, 0))
    x = torch.empty_like(b)
    want, r, Ar = torch.zeros_like(b), b.clone(), torch.empty_like(b)
    for _ in range(nu):
        ctx.level_apply(level, r, Ar)
        alpha = p.omega * torch.vdot(Ar.flatten(), r.flatten()) / torch.vdot(Ar.flatten(), Ar.flatten()).real
        want += alpha * r
        r = r - alpha * Ar
    ctx.smooth(level, b, x, nu)
    # a few hundred FP64 roundings per entry and step, the sums' below 1e-14
    assert (x - want).norm() < 1e-12 * want.norm()
    ctx.close()
