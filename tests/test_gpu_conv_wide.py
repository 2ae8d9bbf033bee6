"""Batches of 2^31 positions and more take the tensor cores like smaller ones: BF16 operands,
and every value in its place."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

CH, ROWS = 2, 4096


def _sparse(shape, seed):
    """+-(1 + 2^-9) (1 once rounded to BF16) in one place of 512, made in pieces."""
    t = torch.zeros(shape, device="cuda")
    g = torch.Generator(device="cuda").manual_seed(seed)
    flat = t.view(-1)
    for at in range(0, flat.numel(), 1 << 28):
        part = flat[at:at + (1 << 28)]
        r = torch.randint(0, 1024, part.shape, device="cuda", generator=g, dtype=torch.int16)
        part[r == 0] = 1.0 + 2.0 ** -9
        part[r == 1] = -1.0 - 2.0 ** -9
    return t


def _rows(t, n, c, r0, r1, dc):
    """Rows r0 .. r1 of a plane, BF16-rounded, shifted by dc columns; 0 outside."""
    H, Wd = t.shape[3:]
    out = torch.zeros((r1 - r0, Wd), device="cuda")
    a, b = max(r0, 0), min(r1, H)
    if a < b:
        lo, hi = max(0, -dc), min(Wd, Wd - dc)
        out[a - r0:b - r0, lo:hi] = t[n, c, 0, a:b, lo + dc:hi + dc].bfloat16().float()
    return out


# one sample of more than 2^31 values a channel; three of more than 2^31 together
@pytest.mark.parametrize("n,side", [(1, 46400), (3, 27000)])
def test_wide_batches(n, side):
    """Sums of a few small integers, exact in FP32 in any order."""
    from paper_1806_10247_gb300 import surrogate as G

    L = G._nn()
    d = 3
    shape = (n, CH, 1, side, side)
    x, gy = _sparse(shape, 1), _sparse(shape, 2)
    y, gx = torch.empty(shape, device="cuda"), torch.empty(shape, device="cuda")
    w = torch.tensor(np.random.default_rng(3).integers(-3, 4, (CH, CH, 1, 3, 3)), dtype=torch.float32, device="cuda")
    wb, b = w.to(torch.bfloat16), torch.tensor([1.0, -2.0], device="cuda")
    gw, gb = torch.empty_like(w), torch.empty(CH, device="cuda")
    s = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    tail = (G._i3(shape[2:]), G._i3((1, 3, 3)), G._i3((1, d, d)))
    G._ck(L.lbm_nn_conv3d_forward(p(x), p(wb), 1, p(b), p(y), n, CH, CH, *tail, 0, s))
    G._ck(L.lbm_nn_conv3d_backward(p(x), p(wb), 1, p(gy), p(gx), p(gw), p(gb), n, CH, CH, *tail, s))
    gwr = torch.zeros((CH, CH, 3, 3), dtype=torch.float64, device="cuda")
    for k in range(n):
        for r0 in range(0, side, ROWS):
            r1 = min(side, r0 + ROWS)
            ry = [torch.full((r1 - r0, side), float(b[o]), device="cuda") for o in range(CH)]
            rx = [torch.zeros((r1 - r0, side), device="cuda") for _ in range(CH)]
            g0 = [_rows(gy, k, o, r0, r1, 0) for o in range(CH)]
            for f in range(3):
                for e in range(3):
                    dr, dc = d * (f - 1), d * (e - 1)
                    for i in range(CH):
                        xs, gs = _rows(x, k, i, r0 + dr, r1 + dr, dc), _rows(gy, k, i, r0 - dr, r1 - dr, -dc)
                        for o in range(CH):
                            ry[o] += w[o, i, 0, f, e] * xs
                            rx[o] += w[i, o, 0, f, e] * gs
                            gwr[o, i, f, e] += (xs * g0[o]).sum(dtype=torch.float64)
            for o in range(CH):
                assert torch.equal(y[k, o, 0, r0:r1], ry[o])
                assert torch.equal(gx[k, o, 0, r0:r1], rx[o])
    assert torch.equal(gw[:, :, 0].double(), gwr)
