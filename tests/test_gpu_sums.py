"""Where FP32 values are summed, and in what: the Krylov reductions of FP32 vectors (FP32 over a
thread's elements, one where there are threads enough, then FP64), the MR sums of the tiled 4d apply (FP32 inside a
tile of 64 sites, FP64 across) and the block loss's products (FP32, as a tree over the rows). The
inputs are integers whose products are exact in FP32 and among which one is large, so that an addition in FP32 next to
it loses the small ones. The launchers are the library's internal C++ functions."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

BIG = 2.0 ** 24  # FP32 counts in steps of two from here on


class ReduceWs(ctypes.Structure):
    _fields_ = [("partials", ctypes.c_void_p), ("ticket", ctypes.c_void_p), ("max_blocks", ctypes.c_int),
                ("capacity", ctypes.c_longlong), ("tickets", ctypes.c_longlong)]


class Geo4(ctypes.Structure):
    _fields_ = [("L", ctypes.c_int * 4), ("nsites", ctypes.c_longlong)]


class BlockGeo(ctypes.Structure):
    _fields_ = [(n, ctypes.c_int) for n in ("L0", "L1", "B0", "B1", "nb0", "nb1", "bvol", "nint", "Nb")] + [
        ("nblocks", ctypes.c_longlong)]


def _fn(name):
    import paper_0707_4018_gb300 as mg
    f = getattr(mg.load(), name)
    f.restype = None
    return f


def _p(t):
    return ctypes.c_void_p(t.data_ptr() if t is not None else 0)


def _stream():
    import torch
    return ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)


@pytest.mark.parametrize("n", [1, 7, 1000, 16384, 16385, 24576, 70000])
@pytest.mark.parametrize("batch", [False, True])
def test_krylov_reductions_of_fp32_vectors(n, batch):
    import torch
    k = 2
    rng = np.random.default_rng(n)
    W, r = rng.integers(-3, 4, (k + 1, n, 2)).astype(np.float32), rng.integers(-3, 4, (n, 2)).astype(np.float32)
    for v in (*W, r):  # an element's products are small whole numbers, in every fifth one times 2^20
        v[::5] *= 2.0 ** 10
    Wc, rc = W[..., 0] + 1j * W[..., 1].astype(np.complex128), r[..., 0] + 1j * r[..., 1].astype(np.complex128)
    want = np.array([*(np.vdot(Wc[j], Wc[k]) for j in range(k)), np.vdot(Wc[k], Wc[k]), np.vdot(Wc[k], rc),
                     np.vdot(rc, rc)])
    dW, dr = torch.from_numpy(W).cuda(), torch.from_numpy(r).cuda()
    out = torch.zeros(2 * (k + 3), dtype=torch.float64, device="cuda")
    part = torch.zeros(1 << 16, dtype=torch.float64, device="cuda")
    tick = torch.zeros(64, dtype=torch.int32, device="cuda")
    ws = ReduceWs(part.data_ptr(), tick.data_ptr(), 64, part.numel(), 64)
    if batch:
        _fn("_ZN2mg21launch_gcr_dots_batchIfEEvPKNS_2CxIT_EES5_iixPdRKNS_8ReduceWsEP11CUstream_st")(
            _p(dW), _p(dr), k, 1, ctypes.c_longlong(n), _p(out), ctypes.byref(ws), _stream())
    else:
        _fn("_ZN2mg15launch_gcr_dotsEPKNS_2CxIfEES3_S3_ixPdRKNS_8ReduceWsEP11CUstream_st")(
            _p(dW), _p(dW[k]), _p(dr), k, ctypes.c_longlong(n), _p(out), ctypes.byref(ws), _stream())
    got = out.cpu().numpy()
    # the two products of an element have few digits, the sums are whole numbers below 2^53: nothing rounds but the
    # FP32 additions of the elements that one of the 64 x 256 threads takes, each by 2^-24 of what they add up to
    adds = -(-n // (64 * 256)) - 1
    size = np.array([*(np.abs(Wc[j]) @ np.abs(Wc[k]) for j in range(k)), np.abs(Wc[k]) @ np.abs(Wc[k]),
                     np.abs(Wc[k]) @ np.abs(rc), np.abs(rc) @ np.abs(rc)])
    tol = adds * 2.0 ** -24 * size
    assert (np.abs(got[0::2] - want.real) <= tol).all() and (np.abs(got[1::2] - want.imag) <= tol).all()


@pytest.mark.parametrize("dims", [(8, 4, 4, 2), (8, 2, 2, 6)])  # four tiles of a CTA, and three
def test_mr_sums_of_the_tiled_4d_apply_are_fp64_across_tiles(dims):
    import torch
    V = int(np.prod(dims))
    U = torch.zeros((V, 4, 3, 3), dtype=torch.complex64, device="cuda")  # D r = diag r
    r = torch.zeros((V, 12), dtype=torch.complex64, device="cuda")
    r[0, 0] = 2.0 ** 12  # tile 0 sums to 2^24
    r[V - 1, 5] = 1.0    # the last tile to 1
    Ar = torch.empty_like(r)
    alpha = torch.zeros(2, dtype=torch.float32, device="cuda")
    part = torch.zeros(3 * (V // 64), dtype=torch.float64, device="cuda")
    tick = torch.zeros(1, dtype=torch.int32, device="cuda")
    f = _fn("_ZN2mg17launch_dslash4_mrEPKNS_2CxIfEES3_PS1_NS_4Geo4EdidP6float2PdxPjP11CUstream_st")
    f.restype = ctypes.c_bool
    assert f(_p(U), _p(r), _p(Ar), Geo4((ctypes.c_int * 4)(*dims), V), ctypes.c_double(1.0), 1, ctypes.c_double(0.5),
             _p(alpha), _p(part), ctypes.c_longlong(part.numel()), _p(tick), _stream())
    got = part.cpu().numpy()[:3]
    assert np.array_equal(got, [BIG + 1, 0.0, BIG + 1])
    assert alpha.cpu().numpy().tolist() == [0.5, 0.0]


@pytest.mark.parametrize("rows", [2, 8, 18, 32])
def test_block_loss_products_are_summed_as_a_tree(rows):
    import torch
    B0, B1 = {2: (1, 1), 8: (2, 2), 18: (3, 3), 32: (4, 4)}[rows]
    y = torch.ones((B0 * B1, 2, 1, 2), dtype=torch.float32, device="cuda")  # [x][2 nv] float2, one vector
    y[..., 1] = 0.0
    y.view(-1, 2)[0, 0] = 2.0 ** 12
    tgt = torch.zeros((1, B0 * B1, 2, 2), dtype=torch.float32, device="cuda")
    tgt.view(-1, 2)[0, 0] = 1.0
    gy, loss = torch.zeros_like(y), torch.zeros(1, dtype=torch.float64, device="cuda")
    bg = BlockGeo(B0, B1, B0, B1, 1, 1, B0 * B1, 2, 2 * B0 * B1, 1)
    _fn("_ZN2mg19launch_nullnet_lossEPK6float2S2_PKiiRKNS_8BlockGeoEifPS0_PdP11CUstream_st")(
        _p(y), _p(tgt), _p(None), 1, ctypes.byref(bg), 1, ctypes.c_float(1.0), _p(gy), _p(loss), _stream())
    # loss = 1 - |c|^2 / (g (1 + 1e-7)), c = 2^12 and g = 2^24 + rows - 1
    g = BIG / ((1.0 - float(loss.cpu()[0])) * (1.0 + 1e-7))
    # five additions of half a step (one above 2^24) and FP64 rounding; summed in a chain g stays at 2^24
    assert abs(g - (BIG + rows - 1)) <= 5.0 + 1e-6
