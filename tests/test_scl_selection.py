"""CA-SCL's output path, found by the CRC of each path's codeword: batches that hold frames whose best path
fails its CRC and a later one passes, and frames on which every path fails (the best is output).  A list
without a CRC gives the best path, so the oracle tells which frames these are."""
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


@pytest.mark.parametrize("N,K,c,ebn0,B", [(128, 64, 8, -1.0, 64), (1024, 512, 16, 1.0, 60), (4096, 2048, 16, 1.0, 24)])
@pytest.mark.parametrize("L", [8, 32])
@pytest.mark.parametrize("times", [1, 60])  # a CTA per frame, and lists in warps or half-warps
def test_path_that_is_not_the_best(N, K, c, ebn0, B, L, times):
    ocode = fr.oracle_code(N, K, c)
    _, llr = fr.frames(ocode, ebn0, B, seed=900 + L)
    ref = oracle.scl_decode(llr, ocode, L, "f32")
    best = oracle.scl_decode(llr, oracle.Code(N, K, 0, 0, ocode.frozen, ocode.info_idx), L, "f32")
    other = (ref["u_hat"] != best["u_hat"]).any(axis=1)
    ok = ref["status"] == oracle.SCL_OK
    assert other.any() and not ok.all() and not (other & ~ok).any()
    dec = api.Decoder(fr.api_code(ocode), B * times, L)
    dec.scl(torch.from_numpy(np.tile(llr, (times, 1))).cuda())
    torch.cuda.synchronize()
    assert np.array_equal(dec.status.cpu().numpy(), np.tile(ref["status"], times))
    assert np.array_equal(api.unpack_bits(dec.bits.cpu().numpy(), ocode.P),
                          np.tile(oracle.payload_of(ref["u_hat"], ocode), (times, 1)))
