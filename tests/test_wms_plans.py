"""The training kernels at every block length's thread plan: the forward bit-exact against the oracle's
weighted BP and the backward against the oracle's reverse sweep, for odd batches, one and several
iterations, the loss on the last or on every iteration, and tensors on and off a 16-byte boundary."""
import numpy as np
import pytest

import oracle
from tests import frames as fr

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

from paper_1609_09358_gb300 import api, build  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    api.load()


def shifted(a, skip):
    """a on the device, starting `skip` floats after an allocation's start."""
    flat = torch.empty(a.size + 4, dtype=torch.float32, device="cuda")
    x = flat[skip:skip + a.size].view(a.shape)
    x.copy_(torch.from_numpy(np.ascontiguousarray(a)))
    return x


@pytest.mark.parametrize("skip", [0, 1])
@pytest.mark.parametrize("N,K,crc,T,B,all_iters", [(128, 64, 8, 1, 1, False), (128, 64, 8, 3, 5, True),
                                                   (256, 128, 16, 3, 7, False), (512, 256, 16, 2, 3, True),
                                                   (1024, 512, 16, 3, 3, False), (2048, 1024, 24, 2, 3, True)])
def test_training_kernels_match_oracle(N, K, crc, T, B, all_iters, skip):
    ocode = fr.oracle_code(N, K, crc)
    code = fr.api_code(ocode)
    _, llr = fr.frames(ocode, 1.5, B, seed=60 + N)
    rng = np.random.default_rng(N + T)
    w = rng.uniform(0.6, 1.2, (T, 2, ocode.n, N)).astype(np.float32)
    shape = (T, B, N) if all_iters else (B, N)
    dy = (rng.normal(size=shape) * (1 - ocode.frozen)).astype(np.float32)
    llr_d, w_d, dy_d = shifted(llr, skip), shifted(w, skip), shifted(dy, skip)
    out, gw = shifted(np.zeros(shape, np.float32), skip), shifted(np.full_like(w, 7.0), skip)
    need = api.wms_workspace_bytes(code, B, T)
    ws = torch.empty(need + 16, dtype=torch.uint8, device="cuda")[4 * skip:4 * skip + need]
    api.wms_forward(code, llr_d, T, 20.0, w_d, out, ws)
    api.wms_backward(code, llr_d, T, 20.0, w_d, dy_d, gw, ws)
    torch.cuda.synchronize()
    got = out.cpu().numpy()
    for t in range(T if all_iters else 1):
        its = t + 1 if all_iters else T
        ref = oracle.bp_decode(llr, ocode, its, 20.0, "f32", early_stop=False, w=w)
        assert np.array_equal(got[t] if all_iters else got, ref["llr_u"]), t
    ref_g = oracle.wms_grad(llr, ocode, T, 20.0, w, dy.astype(np.float64), "f32", all_iters=all_iters)
    g = gw.double().cpu().numpy()
    assert np.abs(ref_g).max() > 0
    # binary32 sums of at most a few hundred terms against binary64: a relative 1e-4 covers the largest
    # gradients, 1e-5 of the largest the cancelled ones
    assert np.allclose(g, ref_g, rtol=1e-4, atol=1e-5 * np.abs(ref_g).max())
