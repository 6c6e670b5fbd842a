"""Frames whose BP messages recur: in large batches with a high iteration limit the plain FP32 kernel at
N = 1024 recognises a repeating state and skips whole periods.  Whatever the number of iterations left
(every residue modulo the skip), bits, status and iteration count equal the oracle's, which runs them
all.  Channel values on a coarse grid make almost every failing frame periodic; unrounded ones some, and
at a low signal so few that the kernel hands the batch over to the plain one."""
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


@pytest.mark.parametrize("N,K,crc,ebn0,grid", [(1024, 512, 16, 1.5, 4.0), (1024, 512, 16, 1.5, 1.0),
                                               (1024, 512, 16, 2.5, 0.0), (1024, 512, 24, 2.0, 2.0),
                                               (1024, 512, 16, 0.5, 0.0)])
def test_skipped_periods_bit_exact(N, K, crc, ebn0, grid):
    ocode = fr.oracle_code(N, K, crc)
    code = fr.api_code(ocode)
    _, llr = fr.frames(ocode, ebn0, 900 if grid == 0.0 else 120, seed=300 + N + crc)
    if grid:
        llr = (np.round(llr / grid) * grid).astype(np.float32)
    # mostly frames that are still undecided after 20 iterations: failing ones and late successes
    first = oracle.bp_decode(llr, ocode, 20, 20.0, "f32", want_llr=False)
    llr = llr[np.concatenate([np.nonzero(first["iters"] == 20)[0][:60], [0, 1, 2]])]
    times = -(-16400 // llr.shape[0])
    x = torch.from_numpy(np.tile(llr, (times, 1))).cuda()
    dec = api.Decoder(code, x.shape[0], 2)
    for imax in (150, 151, 152, 153, 200):
        ref = oracle.hybrid_decode(llr, ocode, imax, 20.0, 2, precision="f32")
        dec.hybrid(x, imax, 20.0)
        torch.cuda.synchronize()
        assert np.array_equal(dec.iters.cpu().numpy().astype(np.int32), np.tile(ref["iters"], times))
        assert np.array_equal(dec.status.cpu().numpy(), np.tile(ref["status"], times))
        assert np.array_equal(api.unpack_bits(dec.bits.cpu().numpy(), ocode.P),
                              np.tile(oracle.payload_of(ref["u_hat"], ocode), (times, 1)))
