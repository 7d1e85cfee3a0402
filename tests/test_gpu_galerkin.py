"""The Galerkin operator of the second coarse level, for eight dofs per site and for other counts, in FP64 and FP32
arithmetic: applying it is prolongation, the operator of the level above and restriction."""
import pytest

import inputs
from tests._util import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("nv,dims,blocks", [([8, 8], (48, 32), [(4, 4), (2, 2)]), ([8, 5], (32, 16), [(4, 4), (2, 4)]),
                                            ([5, 8], (32, 24), [(4, 4), (4, 3)]), ([3, 3], (12, 12), [(2, 2), (3, 1)])])
def test_galerkin_is_prolong_apply_restrict(nv, dims, blocks, mixed):
    import torch
    import paper_0707_4018_gb300 as mg
    p = mg.mg_default_params(levels=3, blocks=blocks, Nv=nv, n_pass=1, nu_setup=3, coarsest_tol=0.2 if mixed else 1e-10,
                             precision=mg.MG_FP32 if mixed else mg.MG_FP64)
    base = mg.Context.setup(to_dev(inputs.hot_links(*dims, seed=51)), 0.3, dims, p)
    for ctx in (base, base.clone(0.5)):
        for l in (0, 1):
            n, k = ctx.level_size(l + 1)
            nf, kf = ctx.level_size(l) if l > 0 else (dims[0] * dims[1], 2)
            e = to_dev(inputs.gaussian_spinor(n, k, 52, l))
            f, g = (torch.empty((nf, kf), dtype=torch.complex128, device="cuda") for _ in range(2))
            want, got = torch.empty_like(e), torch.empty_like(e)
            ctx.prolong(l, e, f)
            ctx.level_apply(l, f, g)
            ctx.restrict(l, g, want)
            ctx.level_apply(l + 1, e, got)
            # sums of at most 8 x 32 products: a few hundred roundings of FP64, or of FP32 where the products use it
            assert (got - want).norm() < (1e-5 if mixed else 1e-12) * want.norm()
    base.close()
