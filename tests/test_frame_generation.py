"""The encoder and the payload generator over the layouts their accesses depend on: rows of every length
modulo four bytes, buffers off their natural alignment, pad bits set in the payload rows, batches that
make the encoder's persistent grid loop, several frames per warp and several words per lane."""
import numpy as np
import pytest

import oracle
from tests import frames as fr

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

from paper_1609_09358_gb300 import api, build, inputs  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    api.load()


def bytes_at(a, skip):
    """uint8 array on the device, starting `skip` bytes after an allocation's start."""
    flat = torch.full((a.size + 8,), 0xA5, dtype=torch.uint8, device="cuda")
    x = flat[skip:skip + a.size].view(a.shape)
    x.copy_(torch.from_numpy(np.ascontiguousarray(a)))
    return x


@pytest.mark.parametrize("N,K,crc,rate,B", [(128, 64, 8, None, 9001), (256, 100, 16, 100 / 256, 203),
                                            (512, 24, 24, 24 / 512, 19), (1024, 512, 16, None, 6007),
                                            (2048, 1024, 24, None, 21), (4096, 2048, 16, None, 13)])
@pytest.mark.parametrize("skip", [0, 1, 2])
def test_encoder_layouts(N, K, crc, rate, B, skip):
    ocode = fr.oracle_code(N, K, crc) if rate is None else fr.oracle_code(N, K, crc, design_rate=rate)
    code = fr.api_code(ocode)
    pay = inputs.payload_bits(9, 3, B, ocode.P)
    packed = api.pack_bits(pay)
    if ocode.P % 8:
        packed = packed.copy()
        packed[:, -1] |= (0xFF << (ocode.P % 8)) & 0xFF  # pad bits are not payload
    cw = torch.zeros((B, N // 8), dtype=torch.uint8, device="cuda")
    api.polar_encode(code, bytes_at(packed, skip), cw)
    torch.cuda.synchronize()
    assert np.array_equal(api.unpack_bits(cw.cpu().numpy(), N), oracle.encode_batch(pay, ocode))


@pytest.mark.parametrize("P", [1, 7, 32, 127, 128, 129, 163, 240, 255, 256, 496, 2032, 6144, 6145, 20000])
@pytest.mark.parametrize("skip", [0, 1, 2])
def test_payload_rows(P, skip):
    B = 137
    out = bytes_at(np.full((B, (P + 7) // 8), 0xFF, np.uint8), skip)
    api.polar_random_payload(B, P, 4321, 2**32 - 5, out)
    torch.cuda.synchronize()
    got = out.cpu().numpy()
    assert np.array_equal(got, api.pack_bits(inputs.payload_bits(4321, 2**32 - 5, B, P)))


@pytest.mark.parametrize("N,B", [(8, 5), (128, 33), (4096, 3)])
@pytest.mark.parametrize("per_frame", [False, True])
def test_awgn_lengths(N, B, per_frame):
    x = np.random.default_rng(N).integers(0, 2, (B, N), dtype=np.uint8)
    sig = np.linspace(0.5, 1.2, B).astype(np.float32) if per_frame else np.full(B, 0.8, np.float32)
    llr = torch.zeros((B, N), dtype=torch.float32, device="cuda")
    api.polar_awgn_llr(torch.from_numpy(api.pack_bits(x)).cuda(), N, 0.8, 99, 7, llr,
                       sigma_per_frame=torch.from_numpy(sig).cuda() if per_frame else None)
    torch.cuda.synchronize()
    s = sig.astype(np.float64)[:, None]
    ref = 2.0 * ((1.0 - 2.0 * x) + s * inputs.unit_noise(99, 7, B, N)) / s ** 2
    assert np.allclose(llr.cpu().numpy(), ref, rtol=1e-4, atol=1e-4)
