"""Tensor-core convolutions with dilations up to and beyond the image, on both sides of the
staged form's reach and of a chunk of positions, against the FP64 convolution of the
BF16-rounded operands."""
import ctypes

import numpy as np
import pytest

from oracle import surrogate_ref as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("dhw,k,dil", [
    ((1, 12, 40), (1, 3, 3), (1, 1, 16)), ((1, 12, 40), (1, 3, 3), (1, 1, 17)), ((1, 12, 40), (1, 3, 3), (1, 5, 39)),
    ((1, 12, 40), (1, 3, 3), (1, 2, 40)), ((1, 12, 40), (1, 3, 3), (1, 13, 1000)), ((1, 7, 1), (1, 3, 3), (1, 1, 1)),
    ((1, 3, 700), (1, 3, 3), (1, 1, 127)), ((1, 3, 700), (1, 3, 3), (1, 1, 128)), ((1, 3, 700), (1, 3, 3), (1, 1, 300)),
    ((1, 3, 300), (1, 1, 9), (1, 1, 60)), ((1, 3, 300), (1, 1, 9), (1, 1, 140)), ((2, 5, 6), (3, 3, 5), (1, 2, 2)),
    ((2, 5, 9), (3, 1, 5), (1, 1, 4))])
@pytest.mark.parametrize("ci,co", [(16, 16), (3, 16), (9, 5)])
def test_any_dilation(dhw, k, dil, ci, co):
    """FP32 sums of exact products: as many roundings as terms, 2^-24 of the sum of
    magnitudes each."""
    from paper_1806_10247_gb300 import surrogate as G

    rng = np.random.default_rng(dil[2])
    bf = lambda a: torch.tensor(a, dtype=torch.float32).to(torch.bfloat16).double().numpy()  # noqa: E731
    n = 2
    x, gy = bf(rng.standard_normal((n, ci) + dhw)), bf(rng.standard_normal((n, co) + dhw))
    w, b = bf(rng.standard_normal((co, ci) + k) / 4), bf(rng.standard_normal(co))
    L = G._nn()
    d = [torch.tensor(a, dtype=torch.float32, device="cuda") for a in (x, w, b, gy)]
    dw = d[1].to(torch.bfloat16)
    y, gx = torch.empty(gy.shape, device="cuda"), torch.empty(x.shape, device="cuda")
    gw, gb = torch.empty(w.shape, device="cuda"), torch.empty(co, device="cuda")
    s = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    shape = (G._i3(dhw), G._i3(k), G._i3(dil), s)
    G._ck(L.lbm_nn_conv3d_forward(p(d[0]), p(dw), 1, p(d[2]), p(y), n, ci, co, *shape[:3], 0, s))
    G._ck(L.lbm_nn_conv3d_backward(p(d[0]), p(dw), 1, p(d[3]), p(gx), p(gw), p(gb), n, ci, co, *shape))
    taps = int(np.prod(k))
    ref = (S.conv3d(x, w, b, dil), *S.conv3d_backward(x, w, dil, gy)[:2])
    mag = (S.conv3d(abs(x), abs(w), abs(b), dil), *S.conv3d_backward(abs(x), abs(w), dil, abs(gy))[:2])
    terms = (ci * taps + 1, co * taps, n * int(np.prod(dhw)))
    for got, r, m, t in zip((y, gx, gw), ref, mag, terms):
        assert (np.abs(got.cpu().numpy() - r) <= t * 2.0 ** -24 * m.max()).all()
