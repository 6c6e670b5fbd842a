"""The training workspace: the stored message columns (2 to n of both sweeps) of every frame and iteration,
and what it takes to start them on a 16-byte boundary.  Nothing outside it is written."""
import numpy as np
import pytest

import oracle
from paper_1609_09358_gb300 import api, build
from tests import frames as fr

CODES = pytest.mark.parametrize("N,K,crc", [(128, 64, 8), (256, 128, 16), (1024, 512, 16), (2048, 1024, 24)])


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    api.load()


@CODES
def test_size_is_the_stored_columns(N, K, crc):
    code = fr.api_code(fr.oracle_code(N, K, crc))
    n = N.bit_length() - 1
    for B, T in ((1, 1), (7, 3), (4096, 20)):
        need = api.wms_workspace_bytes(code, B, T)
        columns = B * T * 2 * (n - 1) * N * 4
        assert columns <= need <= columns + 16
    assert api.wms_workspace_bytes(code, 0, 5) == 0


@pytest.mark.gpu
@CODES
@pytest.mark.parametrize("skip", [0, 4, 8, 12])
def test_nothing_outside_is_written(N, K, crc, skip):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    ocode = fr.oracle_code(N, K, crc)
    code = fr.api_code(ocode)
    B, T = 5, 2
    _, llr = fr.frames(ocode, 1.5, B, seed=4)
    rng = np.random.default_rng(N)
    w = rng.uniform(0.6, 1.2, (T, 2, ocode.n, N)).astype(np.float32)
    dy = (rng.normal(size=(B, N)) * (1 - ocode.frozen)).astype(np.float32)
    x, wd, dyd = (torch.from_numpy(a).cuda() for a in (llr, w, dy))
    need = api.wms_workspace_bytes(code, B, T)
    flat = torch.full((need + 64,), 0x5A, dtype=torch.uint8, device="cuda")
    ws = flat[skip:skip + need]
    out, gw = torch.zeros((B, N), device="cuda"), torch.zeros_like(wd)
    api.wms_forward(code, x, T, 20.0, wd, out, ws)
    api.wms_backward(code, x, T, 20.0, wd, dyd, gw, ws)
    torch.cuda.synchronize()
    assert bool((flat[:skip] == 0x5A).all()) and bool((flat[skip + need:] == 0x5A).all())
    ref = oracle.bp_decode(llr, ocode, T, 20.0, "f32", early_stop=False, w=w)
    assert np.array_equal(out.cpu().numpy(), ref["llr_u"])
    ref_g = oracle.wms_grad(llr, ocode, T, 20.0, w, dy.astype(np.float64), "f32", all_iters=False)
    # as in the tests of the training kernels: binary32 sums of a few terms against binary64
    assert np.allclose(gw.double().cpu().numpy(), ref_g, rtol=1e-4, atol=1e-5 * np.abs(ref_g).max())
