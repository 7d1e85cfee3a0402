"""The Wilson applies whose kernel is chosen by alignment and extents: fields that start off the widest loads'
boundary take the narrower ones and give the same result as aligned copies of them."""
import numpy as np
import pytest

import inputs
from tests._util import to_dev, to_host

pytestmark = pytest.mark.gpu


def _shifted(t, n):
    """A copy of t that starts n of its elements into an allocation."""
    import torch
    buf = torch.zeros(t.numel() + n, dtype=t.dtype, device="cuda")
    buf[n:] = t.reshape(-1)
    return buf[n:].view(t.shape)


# complex64 entries: 1 is 8 bytes (links only: spinors are read in 16-byte words), 2 is 16, 4 is 32
@pytest.mark.parametrize("dims", [(8, 2, 2, 2), (16, 4, 2, 6), (8, 6, 4, 2)])
@pytest.mark.parametrize("links,spinors", [(0, 2), (1, 0), (1, 2), (2, 4)])
def test_dslash4_f32_alignments(dims, links, spinors):
    import torch
    import paper_0707_4018_gb300 as mg
    V = int(np.prod(dims))
    U = to_dev(inputs.su3_random(V * 4, 41, 0x7F).reshape(V, 4, 9), torch.complex64)
    psi = to_dev(inputs.gaussian_spinor(V, 12, 42, 0), torch.complex64)
    want = torch.empty_like(psi)
    mg.mg_dslash(U, psi, want, -0.3, dims, 1)
    out = _shifted(torch.zeros_like(psi), spinors)
    mg.mg_dslash(_shifted(U, links), _shifted(psi, spinors), out, -0.3, dims, 1)
    torch.cuda.synchronize()
    # 8 hops of 3 products and the diagonal, in another order by the gather kernel: 64 roundings of 2^-24 at most
    assert (out - want).abs().max() <= 64 * 2.0**-24 * want.abs().max()


# half fields in bytes: links start on 4, spinors (8 bytes of components and a 4-byte norm a site) on 8
@pytest.mark.parametrize("dims", [(16, 12), (130, 6), (15, 12), (2, 2)])
@pytest.mark.parametrize("links,spinors", [(4, 8), (4, 0), (8, 8), (16, 16)])
def test_half_dslash_alignments(dims, links, spinors):
    import torch
    import paper_0707_4018_gb300 as mg
    V = dims[0] * dims[1]
    U = to_dev(inputs.hot_links(*dims, seed=43))
    psi = to_dev(inputs.gaussian_complex(V * 2, 44, 0).reshape(-1, 2))
    hU, hp, want = mg.half_links(V), mg.half_spinor(V), mg.half_spinor(V)
    mg.mg_half_convert(2, U, hU, V)
    mg.mg_half_convert(0, psi, hp, V)
    mg.mg_dslash_half(hU, hp, want, 0.1, dims)
    out = _shifted(torch.zeros_like(want), spinors)
    mg.mg_dslash_half(_shifted(hU, links), _shifted(hp, spinors), out, 0.1, dims)
    torch.cuda.synchronize()
    got, ref = to_host(out), to_host(want)
    h = [a[:8 * V].view(np.float16).astype(np.float64).reshape(V, 4) for a in (got, ref)]
    n = [a[8 * V:].view(np.float32).astype(np.float64) for a in (got, ref)]
    # FP32 sums in another order move a norm by a few 2^-24 and an entry by at most one half step of its site's norm
    assert np.abs(n[0] - n[1]).max() <= 32 * 2.0**-24 * n[1].max()
    assert np.abs(h[0] * n[0][:, None] - h[1] * n[1][:, None]).max() <= 2.0**-10 * n[1].max()
