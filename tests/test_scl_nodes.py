"""CA-SCL's whole-node steps: aligned nodes of 32, 16, 8 and 4 bits that are all frozen or all
information are decided at once where that is exactly the bit-by-bit result.  Codes whose frozen set
mixes nodes of every size and kind, decision-aided positions inside information nodes, channel values
full of ties and zeros (where the whole-node shortcut must not be taken), rows that do not start on a
16-byte boundary and a workspace that does not either: all bit-exact against the oracle, which decides
bit by bit."""
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


def node_code(decided):
    """N = 256: 32-bit blocks all frozen, mixed at 16 / 8 / 4 / 1 bits, and all information."""
    rng = np.random.default_rng(12)
    f = np.ones(256, np.uint8)
    f[32:64] = np.repeat(rng.integers(0, 2, 2) ^ np.array([0, 1]), 16)
    f[64:96] = np.repeat(rng.integers(0, 2, 4), 8)
    f[96:160] = np.repeat(rng.integers(0, 2, 16), 4)
    f[160:192] = rng.integers(0, 2, 32)
    f[192:] = 0
    info = np.nonzero(f == 0)[0].astype(np.int32)
    mask = None
    if decided:
        mask = np.zeros(256, np.uint8)
        mask[info[rng.permutation(len(info))[:40]]] = 1
        mask[224:256] = 1
    return oracle.Code(256, len(info), 16, 0x1021, f, info, mask)


def rows(ocode, B, seed, ties):
    """Noisy codewords; ties: values on a coarse grid (many equal magnitudes, many zeros)."""
    _, llr = fr.frames(ocode, 2.0 if ocode.N == 128 else 6.0, B, seed=seed)
    return (np.round(llr / 2.0) * 2.0).astype(np.float32) if ties else llr


@pytest.mark.parametrize("L", [1, 2, 4, 8, 16, 32])
@pytest.mark.parametrize("which,ties", [("nodes", False), ("nodes", True), ("decided", False), ("short", True)])
def test_whole_nodes_bit_exact(which, ties, L):
    ocode = fr.oracle_code(128, 64, 8) if which == "short" else node_code(which == "decided")
    N = ocode.N
    some = rows(ocode, 21, 500 + L, ties)
    ref = oracle.scl_decode(some, ocode, L, "f32")
    code = api.PolarCode(N, ocode.K, ocode.crc_len, ocode.frozen.copy(), ocode.crc_poly, decided=ocode.decided)
    # rows and workspace on and off a 16-byte boundary, few frames (a CTA each) and more than any grid
    # has CTAs (a warp each, or two per warp)
    for skip, times in ((0, 1), (1, 1), (1, 60)):
        llr, B = np.tile(some, (times, 1)), 21 * times
        need = api.polar_workspace_bytes(code, B, L, api.POLAR_OP_SCL)
        flat = torch.empty(B * N + 4, dtype=torch.float32, device="cuda")
        x = flat[skip:skip + B * N].view(B, N)
        x.copy_(torch.from_numpy(llr))
        ws = torch.empty(need + 16, dtype=torch.uint8, device="cuda")[4 * skip:4 * skip + need]
        bits = torch.zeros((B, code.row_bytes), dtype=torch.uint8, device="cuda")
        status = torch.zeros(B, dtype=torch.uint8, device="cuda")
        api.scl_decode(code, x, L, bits, status, ws)
        torch.cuda.synchronize()
        assert np.array_equal(status.cpu().numpy(), np.tile(ref["status"], times))
        assert np.array_equal(api.unpack_bits(bits.cpu().numpy(), code.P),
                              np.tile(oracle.payload_of(ref["u_hat"], ocode), (times, 1)))


@pytest.mark.parametrize("L", [2, 8, 32])
@pytest.mark.parametrize("N,K,c", [(128, 64, 8), (1024, 512, 16), (4096, 2048, 16)])
def test_crc_selection_over_all_paths(N, K, c, L):
    """Frames at a signal where most fail: every path's CRC is tested before the best one is output,
    and with 8 CRC bits some frames end on a path that is not the best."""
    ocode = fr.oracle_code(N, K, c)
    B = 64 if N == 128 else 6
    _, llr = fr.frames(ocode, -1.0, B, seed=900 + L)
    ref = oracle.scl_decode(llr, ocode, L, "f32")
    assert (ref["status"] != ref["status"].min()).any() or N > 128
    code = api.PolarCode(N, K, c, ocode.frozen.copy(), ocode.crc_poly)
    ws = torch.empty(api.polar_workspace_bytes(code, B, L, api.POLAR_OP_SCL), dtype=torch.uint8, device="cuda")
    bits = torch.zeros((B, code.row_bytes), dtype=torch.uint8, device="cuda")
    status = torch.zeros(B, dtype=torch.uint8, device="cuda")
    api.scl_decode(code, torch.from_numpy(llr).cuda(), L, bits, status, ws)
    torch.cuda.synchronize()
    assert np.array_equal(status.cpu().numpy(), ref["status"])
    assert np.array_equal(api.unpack_bits(bits.cpu().numpy(), code.P), oracle.payload_of(ref["u_hat"], ocode))
