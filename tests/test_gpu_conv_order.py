"""The tensor-core convolutions' forms (staged rows, gathered values) add up K in one
order: channels of zeros beyond those that the staged form takes change no bit."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1806_10247_gb300 import surrogate as G  # noqa: E402

pytestmark = pytest.mark.gpu


def _run(x, w, b, gy, dil):
    L = G._nn()
    n, ci, co, dhw = x.shape[0], x.shape[1], w.shape[0], x.shape[2:]
    d = [torch.tensor(a, dtype=torch.float32, device="cuda") for a in (x, w, b, gy)]
    dw = d[1].to(torch.bfloat16)
    y, gx = torch.empty(gy.shape, device="cuda"), torch.empty(x.shape, device="cuda")
    gw, gb = torch.empty(w.shape, device="cuda"), torch.empty(co, device="cuda")
    s = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    shape = (G._i3(dhw), G._i3(w.shape[2:]), G._i3(dil), s)
    G._ck(L.lbm_nn_conv3d_forward(p(d[0]), p(dw), 1, p(d[2]), p(y), n, ci, co, *shape[:3], 1, s))
    G._ck(L.lbm_nn_conv3d_backward(p(d[0]), p(dw), 1, p(d[3]), p(gx), p(gw), p(gb), n, ci, co, *shape))
    return y.cpu().numpy(), gx.cpu().numpy()


@pytest.mark.parametrize("dhw,dil", [((1, 24, 24), 1), ((1, 33, 47), 8), ((2, 5, 130), 2)])
@pytest.mark.parametrize("ch", [1, 5, 16])
def test_staged_and_gathered_sums_agree(ch, dhw, dil):
    rng = np.random.default_rng(ch + dil)
    wide, k, dil = 17, (1, 3, 3), (1, dil, dil)
    x, gy = rng.standard_normal((3, ch) + dhw), rng.standard_normal((3, ch) + dhw)
    w, b = rng.standard_normal((ch, ch) + k) / 3, rng.standard_normal(ch)
    X, GY = np.zeros((3, wide) + dhw), np.zeros((3, wide) + dhw)
    Wd, B = np.zeros((wide, wide) + k), np.zeros(wide)
    X[:, :ch], GY[:, :ch], Wd[:ch, :ch], B[:ch] = x, gy, w, b
    y, gx = _run(x, w, b, gy, dil)
    Y, GX = _run(X, Wd, B, GY, dil)
    assert np.array_equal(y, Y[:, :ch])
    assert np.array_equal(gx, GX[:, :ch])
