"""The network's tensor-core convolution and weight gradient at the sizes where their tiles end: positions are rows of
N + 1 pixels, in tiles of 128 (convolution) and stages of 64 (gradient)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

from oracle import net as ON  # noqa: E402
from paper_1506_04463_gb300 import feast_nh as F  # noqa: E402
from test_gpu_net import _case, _rel  # noqa: E402


@pytest.mark.parametrize("N,nimg", [(2, 1), (3, 70), (7, 1), (15, 8), (63, 1), (64, 2), (130, 1)])
@pytest.mark.parametrize("offset", [0, 1])
def test_one_layer(N, nimg, offset):
    # one layer: the only rounding between input and output is the operands' (BF16), so the FP32 sums of 288
    # products and of nimg N^2 products stand against the exact ones of the rounded operands; offset 1: an input
    # that does not start on a 16-byte boundary
    Ws, bs, x, t, flat = _case(L=1, N=N, nimg=nimg, seed=N)
    net = F.Net(1, N, nimg)
    net.set_params(flat)
    buf = torch.zeros(x.size + offset, dtype=torch.float32, device="cuda")
    xd = buf[offset:].view(*x.shape)
    xd.copy_(torch.from_numpy(x.astype(np.float32)))
    out = net.forward(xd).cpu().numpy().astype(np.float64)
    ref, cache = ON.forward(x, Ws, bs, quant=True)
    assert _rel(out, ref) < 288 * 2.0 ** -24
    loss, g = net.train_step(xd, torch.from_numpy(t.astype(np.float32)).cuda(), 0.0, want_grad=True)
    assert abs(loss - ON.loss(ref, t)) < 1e-5 * ON.loss(ref, t)
    dWs, dbs, _ = ON.backward(ref, t, cache, Ws, quant=True)
    g = g.cpu().numpy().astype(np.float64)
    # a gradient entry that rounds the other way in BF16 changes one of nimg N^2 terms by 2^-9
    assert _rel(g[:9 * F.NET_CH ** 2], dWs[0].reshape(-1)) < 1e-3
    assert _rel(g[9 * F.NET_CH ** 2:], dbs[0]) < 1e-3
    net.close()
