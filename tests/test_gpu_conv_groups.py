"""Tensor-core convolutions whose padded K has a group of eight values beyond the
channels (a channel count that is an odd multiple of eight): nothing that an earlier
kernel left in shared memory enters the result."""
import ctypes

import numpy as np
import pytest

from oracle import surrogate_ref as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _conv(ci, co, dhw, dil, x, w, b, gy):
    from paper_1806_10247_gb300 import surrogate as G

    L = G._nn()
    d = [torch.tensor(a, dtype=torch.float32, device="cuda") for a in (x, w, b, gy)]
    dw = d[1].to(torch.bfloat16)
    y, gx = torch.empty(gy.shape, device="cuda"), torch.empty(x.shape, device="cuda")
    gw, gb = torch.empty(w.shape, device="cuda"), torch.empty(co, device="cuda")
    s = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    shape = (G._i3(dhw), G._i3(w.shape[2:]), G._i3(dil), s)
    n = x.shape[0]
    G._ck(L.lbm_nn_conv3d_forward(p(d[0]), p(dw), 1, p(d[2]), p(y), n, ci, co, *shape[:3], 0, s))
    G._ck(L.lbm_nn_conv3d_backward(p(d[0]), p(dw), 1, p(d[3]), p(gx), p(gw), p(gb), n, ci, co, *shape))
    return y.cpu().numpy(), gx.cpu().numpy()


def _poison():
    """NaN operands in (nearly) all of the shared memory of every SM."""
    n, c, dhw = 8, 56, (1, 64, 64)
    x, gy = np.full((n, c) + dhw, np.nan), np.full((n, c) + dhw, np.nan)
    _conv(c, c, dhw, (1, 1, 1), x, np.ones((c, c, 1, 3, 3)), np.zeros(c), gy)


# 8 and 40: the dilation is too large for the staged form
@pytest.mark.parametrize("ch,dil,dhw", [(24, 1, (1, 40, 33)), (40, 2, (1, 40, 33)), (56, 1, (2, 17, 20)),
                                        (8, 900, (1, 3, 1000)), (40, 900, (1, 3, 1000)), (17, 1, (1, 40, 33))])
def test_padded_groups_are_zero(ch, dil, dhw):
    """Exact products of BF16 operands, FP32 sums of up to 504: 504 * 2^-24 of the sum of
    magnitudes."""
    rng = np.random.default_rng(ch)
    bf = lambda a: torch.tensor(a, dtype=torch.float32).to(torch.bfloat16).double().numpy()  # noqa: E731
    x, gy = bf(rng.standard_normal((2, ch) + dhw)), bf(rng.standard_normal((2, ch) + dhw))
    w, b = bf(rng.standard_normal((ch, ch, 1, 3, 3)) / 8), bf(rng.standard_normal(ch))
    d = (1, dil, dil)
    _poison()
    y, gx = _conv(ch, ch, dhw, d, x, w, b, gy)
    assert np.isfinite(y).all() and np.isfinite(gx).all()
    for got, ref, mag in ((y, S.conv3d(x, w, b, d), S.conv3d(abs(x), abs(w), abs(b), d)),
                          (gx, S.conv3d_backward(x, w, d, gy)[0], S.conv3d_backward(abs(x), abs(w), d, abs(gy))[0])):
        assert (np.abs(got - ref) <= 9 * ch * 2.0 ** -24 * mag.max()).all()
