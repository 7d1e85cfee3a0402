"""The near-null network's kernels at the edges of their tiles: odd channel and vector counts, lattices that are no
multiple of a tile, against the oracle; both widths of the convolution's tile against each other."""
import numpy as np
import pytest

from oracle import nullnet
from oracle.lattice import Blocking, Lattice
from tests._util import to_dev, to_host

pytestmark = pytest.mark.gpu


def _links(dims, n):
    rng = np.random.default_rng(5)
    return np.exp(0.7j * rng.standard_normal((n, dims[0] * dims[1], 2)))


def _unpack(w, cin, ch, nv):
    out, o = [], 0
    for co, ci in nullnet.shapes(cin, ch, nv):
        n = 5 * 2 * co * 2 * ci
        out.append(w[o:o + n].astype(np.complex128).reshape(5, 2 * co, 2 * ci))
        o += n
    return out


@pytest.mark.parametrize("cin,ch,nv,dims,nf,block", [(3, 5, 3, (8, 12), 2, (4, 4)), (1, 1, 1, (4, 6), 1, (2, 2)),
                                                     (5, 16, 7, (12, 20), 3, (4, 4)), (16, 7, 8, (36, 16), 2, (4, 4))])
def test_gradient_at_odd_sizes_matches_oracle(cin, ch, nv, dims, nf, block):
    import paper_0707_4018_gb300 as mg
    lat = Lattice(dims)
    blk = Blocking(lat, block)
    Us = _links(dims, nf)
    rng = np.random.default_rng(6)
    T = 0.1 * (rng.standard_normal((nf, nv, lat.volume, 2)) + 1j * rng.standard_normal((nf, nv, lat.volume, 2)))
    net = mg.NullNet(cin, ch, nv, seed=7)
    ws = _unpack(net.get_weights(), cin, ch, nv)
    seeds = [31 + f for f in range(nf)]
    loss, grad = net.gradient(to_dev(Us), dims, seeds, to_dev(T), block)
    ref_loss, ref = 0.0, [np.zeros_like(w) for w in ws]
    for f in range(nf):
        hs, As, out = nullnet.forward(ws, nullnet.noise(lat, cin, seeds[f]), Us[f], lat, bf16=True)
        lf, gout = nullnet.loss_and_grad(out, T[f], blk)
        ref_loss += lf / nf
        for li, g in enumerate(nullnet.backward(ws, hs, As, gout / nf, Us[f], lat)):
            ref[li] += g
    # FP32 against FP64 sums, and an activation whose bfloat16 rounding lands the other way: the bounds of the
    # network's other comparisons with the oracle
    assert abs(loss - ref_loss) <= 1e-4 * ref_loss
    for li, g in enumerate(_unpack(grad, cin, ch, nv)):
        assert np.linalg.norm(g - ref[li]) <= 5e-3 * np.linalg.norm(ref[li]), li
    net.close()


@pytest.mark.parametrize("cin,ch,nv", [(8, 16, 8), (3, 5, 3), (16, 9, 1)])
def test_outputs_do_not_depend_on_the_tiling(cin, ch, nv):
    # 80 fields in one call give every SM tiles of the wide form, one field does not
    import torch
    import paper_0707_4018_gb300 as mg
    dims, nf = (32, 44), 80
    U = to_dev(_links(dims, nf))
    net = mg.NullNet(cin, ch, nv, seed=8)
    seeds = list(range(nf))
    all_at_once = net.forward(U, dims, seeds)
    for f in (0, 41, nf - 1):
        assert torch.equal(net.forward(U[f:f + 1], dims, seeds[f:f + 1])[0], all_at_once[f])
    net.close()
