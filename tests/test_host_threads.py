"""Two host threads whose calls share a kernel but need different amounts of its shared memory: every call
succeeds and gives the result it gives alone."""
import os
import subprocess
import sys
import threading

import numpy as np
import pytest

import oracle
from tests import frames as fr

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

from paper_1609_09358_gb300 import api, build, inputs  # noqa: E402

CALLS = 3000


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    api.load()


def encoder(K):
    ocode = fr.oracle_code(4096, K, 16)
    code = fr.api_code(ocode)
    pay = inputs.payload_bits(3, 0, 3, ocode.P)
    x = torch.from_numpy(api.pack_bits(pay)).cuda()
    cw = torch.zeros((3, 512), dtype=torch.uint8, device="cuda")

    def call(stream):
        api.polar_encode(code, x, cw, stream=stream)

    def check():
        assert np.array_equal(api.unpack_bits(cw.cpu().numpy(), 4096), oracle.encode_batch(pay, ocode))
    return call, check


def lists(N, K, noalloc):
    """CA-SCL with lists of 32: levels in the workspace, or (hybrid_decode_noalloc) all in shared memory."""
    ocode = fr.oracle_code(N, K, 16)
    code = fr.api_code(ocode)
    _, llr = fr.frames(ocode, 0.0, 3, seed=8)
    x = torch.from_numpy(llr).cuda()
    dec = api.Decoder(code, 3, 32)

    def call(stream):
        if noalloc:
            api.hybrid_decode_noalloc(code, x, 1, 20.0, api.POLAR_FP32, None, 32, dec.bits, dec.status, dec.iters,
                                      stream=stream)
        else:
            dec.hybrid(x, 1, 20.0, stream=stream)

    def check():
        ref = oracle.hybrid_decode(llr, ocode, 1, 20.0, 32, precision="f32")
        assert np.array_equal(dec.status.cpu().numpy(), ref["status"])
        assert np.array_equal(api.unpack_bits(dec.bits.cpu().numpy(), ocode.P), oracle.payload_of(ref["u_hat"], ocode))
    return call, check


def two_threads(jobs):
    errors, start = [], threading.Barrier(len(jobs))

    def work(call):
        stream = torch.cuda.Stream()
        stream.wait_stream(torch.cuda.default_stream())
        try:
            call(stream)  # uploads the code
            start.wait()
            for _ in range(CALLS):
                call(stream)
        except Exception as e:  # noqa: BLE001
            errors.append(e)
            start.abort()
    threads = [threading.Thread(target=work, args=(call,)) for call, _ in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors
    for _, check in jobs:
        check()


def test_lists_from_two_threads():
    two_threads([lists(256, 128, True), lists(1024, 512, False)])


def test_encoder_from_two_threads():
    """In a process of its own, whose code table has room for two codes that no other test uses."""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    run = "import tests.test_host_threads as t; t.two_threads([t.encoder(3088), t.encoder(4096)])"
    r = subprocess.run([sys.executable, "-c", run], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
