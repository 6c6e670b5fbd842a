"""Frame generation at the largest batch an int32 count allows: frame indices next to 2^31."""
import numpy as np
import pytest

import oracle
from paper_1609_09358_gb300 import inputs
from tests import frames as fr

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

from paper_1609_09358_gb300 import api, build  # noqa: E402

BATCH = 2**31 - 1


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    api.load()
    if torch.cuda.mem_get_info()[0] < 64 << 30:
        pytest.skip("needs 64 GB of device memory")
    yield
    torch.cuda.empty_cache()


def test_encoder_at_the_largest_batch():
    """256 different payloads over and over; every row against its payload's codeword."""
    ocode = fr.oracle_code(128, 64, 8)
    bits = inputs.payload_bits(5, 0, 256, ocode.P)
    pay = torch.from_numpy(api.pack_bits(bits)).cuda().repeat(2**23, 1)[:BATCH]
    cw = torch.zeros((BATCH, 16), dtype=torch.uint8, device="cuda")
    api.polar_encode(fr.api_code(ocode), pay, cw)
    row = torch.from_numpy(api.pack_bits(oracle.encode_batch(bits, ocode))).cuda()
    for b in range(0, BATCH, 2**28):  # a multiple of 256 rows
        part = cw[b:b + 2**28]
        whole = part.shape[0] // 256 * 256
        assert bool((part[:whole].view(-1, 256, 16) == row).all())
        assert torch.equal(part[whole:], row[:part.shape[0] - whole])


def test_payload_at_the_largest_batch():
    out = torch.full((BATCH, 1), 0xFF, dtype=torch.uint8, device="cuda")
    api.polar_random_payload(BATCH, 7, 77, 5, out)
    for b in (0, 2**31 - 200):  # the second range ends with the last, partial block of rows
        n = min(199, BATCH - b)
        assert np.array_equal(out[b:b + n].cpu().numpy(), api.pack_bits(inputs.payload_bits(77, 5 + b, n, 7)))
