"""The workloads whose speed this framework is judged by: what its users have it do, through its
public entry points, from one short packet burst to a full Monte-Carlo batch.

Kinds of case
  hybrid  one batch through Decoder.hybrid (BP with CRC early stop, CA-SCL on the frames it fails)
  host    the same from and to page-locked host memory (hybrid_decode_host)
  bp      a fixed number of BP iterations with both LLR outputs (BP as a soft-output stage)
  scl     CA-SCL alone on every frame
  mixed   frames of several block lengths and rates in one call (MixedDecoder.decode)
  train   a training step of the learned scales: T unrolled iterations, loss, weight gradient
  frames  the workload generator: payload bits, CRC and polar encoding, BPSK-AWGN LLRs
Codes, Eb/N0 ranges, iteration limits and list sizes are those of the repository's configurations,
benchmark and tests.
"""
import math
import os

import numpy as np
import torch

from paper_1609_09358_gb300 import api, wms

# (N, K, CRC length).  CODES: the codes of the configurations (the first four) and of the mixed
# workload, and a few whose payload is no whole number of bytes.
MIXED_CODES = [(n, n * q // 4, 16) for n in (128, 256, 512, 1024, 2048) for q in (1, 2, 3)]
CODES = [(128, 64, 8), (1024, 512, 16), (2048, 1024, 24), (4096, 2048, 16),
         (256, 101, 16), (512, 171, 8), (1024, 683, 24)] + [c for c in MIXED_CODES if c != (1024, 512, 16)]
LEARNED = {(1024, 512, 16): "wms_n1024_k512_t20.pt", (2048, 1024, 24): "wms_n2048_k1024_t20.pt"}
MESSAGES = {"fp32": api.POLAR_FP32, "fp16": api.POLAR_FP16, "exact": api.POLAR_FP32 | api.POLAR_G_EXACT,
            "reencode": api.POLAR_FP32 | api.POLAR_STOP_REENCODE}


def _case(kind, code, B, ebn0, name=None, **more):
    c = {"name": name} if name else {}
    c.update(kind=kind, N=code[0], K=code[1], crc=code[2], B=B, ebn0=ebn0)
    c.update(more)
    return c


def listed():
    prod, short, long, paper = (1024, 512, 16), (128, 64, 8), (2048, 1024, 24), (4096, 2048, 16)
    return [
        # the short-packet configuration: 1 000 frames of 128 bits, where launches and latency count
        _case("hybrid", short, 1000, 2.5, "short_packets", msg="fp32", iters=50, L=4),
        # one short burst of the production code at a poor signal: the latency of a receiver
        _case("hybrid", prod, 37, 1.5, "burst_latency", msg="fp32", iters=200, L=8),
        # the headline workload: production code, plain FP32 hybrid, a full batch
        _case("hybrid", prod, 100000, 2.5, "production_fp32", msg="fp32", iters=200, L=8),
        # the same code in its learned half2 form, an odd batch
        _case("hybrid", prod, 50001, 2.0, "production_learned", msg="fp16", iters=20, L=8, learned=True),
        # fallback-heavy stress: long code, low signal, list of 32, most frames reach CA-SCL
        _case("hybrid", long, 32768, 1.5, "stress_learned", msg="fp16", iters=20, L=32, learned=True),
        # the paper's own configuration: N = 4096, exact PE function, list of 32
        _case("hybrid", paper, 8192, 2.5, "paper_exact", msg="exact", iters=50, L=32),
        # mixed lengths and rates in one persistent launch
        _case("mixed", (0, 0, 16), 65536, 2.0, "mixed_batch", msg="fp16", iters=200, L=8),
        # a receive chain that gets its LLRs in host memory
        _case("host", prod, 30011, 2.5, "host_buffers", msg="fp32", iters=200, L=8),
        # list decoding by itself (the non-hybrid decoder), ragged batch of a mid-length code
        _case("scl", (512, 256, 16), 10007, 2.0, "scl_alone", L=8),
        # BP as a soft-output stage: both LLR outputs after a few fixed iterations
        _case("bp", (512, 171, 8), 20011, 2.0, "bp_soft_output", msg="fp32", iters=5),
        # one training step of the learned scales at the configuration's size
        _case("train", prod, 4096, 2.5, "train_step", T=20, all_iters=True),
        # frame generation of a Monte-Carlo batch
        _case("frames", prod, 100000, 2.5, "frame_generation"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["hybrid", "hybrid", "hybrid", "hybrid", "host", "bp", "scl", "scl", "mixed", "train", "frames"])
    code = rng.choice(CODES)
    N = code[0]
    ebn0 = round(rng.uniform(1.0, 3.5), 2)
    if kind == "hybrid" or kind == "host":
        msg, learned, iters = rng.choice(["fp32", "fp32", "fp16", "fp16", "exact", "reencode"]), False, rng.choice([20, 50, 200])
        if rng.random() < 0.25:
            code, msg, learned, iters = rng.choice(sorted(LEARNED)), rng.choice(["fp16", "fp16", "fp32"]), True, 20
            N = code[0]
        L = rng.choice([1, 2, 4, 8, 8, 8, 16, 32])
        top = 40_000_000 / N / (8 if msg in ("exact", "reencode") else 1) / (4 if iters == 200 and ebn0 < 2 else 1) / max(1, L / 8)
        return _case(kind, code, _log(rng, 1, top), ebn0, msg=msg, iters=iters, L=L, **({"learned": True} if learned else {}))
    if kind == "bp":
        return _case(kind, code, _log(rng, 1, 20_000_000 / N), ebn0, msg=rng.choice(["fp32", "fp16", "exact"]), iters=rng.randint(1, 6))
    if kind == "scl":
        L = rng.choice([1, 2, 4, 8, 8, 16, 32])
        return _case(kind, code, _log(rng, 1, 10_000_000 / N / max(1, L / 8)), ebn0, L=L)
    if kind == "mixed":
        return _case(kind, (0, 0, 16), _log(rng, 100, 30000), ebn0, msg=rng.choice(["fp32", "fp16"]), iters=rng.choice([20, 50, 200]), L=rng.choice([4, 8, 16]))
    if kind == "train":
        code = rng.choice([c for c in CODES if c[0] <= 2048])
        T = rng.choice([2, 5, 10, 20])
        return _case(kind, code, _log(rng, 1, 60_000_000 / code[0] / T), ebn0, T=T, all_iters=rng.random() < 0.5)
    return _case(kind, code, _log(rng, 10, 80_000_000 / N), ebn0)


# ------------------------------------------------------------------------------ inputs
def _sigma(ebn0, rate):
    return math.sqrt(1.0 / (2.0 * rate * 10.0 ** (ebn0 / 10.0)))


def _frames(code, B, ebn0, seed, spread=0.0):
    """(payload, codeword, LLRs) of B seeded frames; spread: Eb/N0 uniform in ebn0 +- spread."""
    payload = torch.empty((B, code.row_bytes), dtype=torch.uint8, device="cuda")
    cw = torch.empty((B, code.N // 8), dtype=torch.uint8, device="cuda")
    llr = torch.empty((B, code.N), dtype=torch.float32, device="cuda")
    api.polar_random_payload(B, code.P, seed, 0, payload)
    api.polar_encode(code, payload, cw)
    sig = None
    if spread:
        gen = torch.Generator(device="cuda")
        gen.manual_seed(seed)
        db = ebn0 + spread * (2.0 * torch.rand(B, generator=gen, device="cuda") - 1.0)
        sig = torch.sqrt(1.0 / (2.0 * (code.P / code.N) * torch.pow(10.0, db / 10.0))).float().contiguous()
    api.polar_awgn_llr(cw, code.N, _sigma(ebn0, code.P / code.N), seed, 0, llr, sigma_per_frame=sig)
    return payload, cw, llr


def _llr_max(msg):
    return 32.0 if msg == "fp16" else 20.0


def _weights(case, seed):
    """Scales as training meets them: between 0.5 and 1, no two alike."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed + 1)
    n = case["N"].bit_length() - 1
    return 0.5 + 0.5 * torch.rand((case["T"], 2, n, case["N"]), generator=gen, device="cuda")


def prepare(case, seed):
    kind, B = case["kind"], case["B"]
    s = dict(case)
    if kind == "mixed":
        s["codes"] = [api.make_code(*c) for c in MIXED_CODES]
        rng = np.random.default_rng(seed)
        code_of = rng.integers(0, len(s["codes"]), B)
        rows = np.array([c.N for c in s["codes"]], np.int64)[code_of]
        off = np.concatenate([np.zeros(1, np.int64), np.cumsum(rows)])
        llr = torch.empty(int(off[-1]), dtype=torch.float32, device="cuda")
        for c, code in enumerate(s["codes"]):
            idx = np.nonzero(code_of == c)[0]
            if len(idx):
                _, _, rowsc = _frames(code, len(idx), case["ebn0"], seed * 64 + c)
                at = torch.from_numpy(off[idx]).cuda()[:, None] + torch.arange(code.N, device="cuda")
                llr[at.reshape(-1)] = rowsc.reshape(-1)
        s.update(llr=llr, code_of=torch.from_numpy(code_of.astype(np.int32)).cuda(),
                 off=torch.from_numpy(off[:-1].copy()).cuda(), dec=api.MixedDecoder(s["codes"], B, case["L"]))
        return s
    code = s["code"] = api.make_code(case["N"], case["K"], case["crc"])
    if kind == "frames":
        s.update(seed=seed, payload=torch.empty((B, code.row_bytes), dtype=torch.uint8, device="cuda"),
                 cw=torch.empty((B, code.N // 8), dtype=torch.uint8, device="cuda"),
                 llr=torch.empty((B, code.N), dtype=torch.float32, device="cuda"))
        return s
    payload, cw, s["llr"] = _frames(code, B, case["ebn0"], seed, 1.5 if kind == "train" else 0.0)
    if kind == "train":
        x = (cw.unsqueeze(-1).bitwise_right_shift(torch.arange(8, device="cuda", dtype=torch.uint8)) & 1).reshape(B, code.N)
        s["info"] = torch.as_tensor(code.info_idx, dtype=torch.long, device="cuda")
        s["sign"] = 1.0 - 2.0 * wms.polar_transform_bits(x)[:, s["info"]].float()
        s["w"] = _weights(case, seed).requires_grad_(True)
        return s
    if kind == "bp":
        s.update(lu=torch.empty((B, code.N), dtype=torch.float32, device="cuda"),
                 lx=torch.empty((B, code.N), dtype=torch.float32, device="cuda"),
                 bits=torch.empty((B, code.row_bytes), dtype=torch.uint8, device="cuda"),
                 status=torch.empty(B, dtype=torch.uint8, device="cuda"),
                 its=torch.empty(B, dtype=torch.int16, device="cuda"))
        return s
    s["scales"] = None
    if case.get("learned"):
        path = os.path.join(os.path.dirname(os.path.abspath(wms.__file__)), "weights",
                            LEARNED[(case["N"], case["K"], case["crc"])])
        w, code, _, _ = wms.load(path)
        s["code"], s["scales"] = code, api.PreparedScales(code, w, MESSAGES[case["msg"]])
    if kind == "host":
        s["llr"] = s["llr"].cpu().pin_memory()
        s.update(bits=torch.empty((B, code.row_bytes), dtype=torch.uint8).pin_memory(),
                 status=torch.empty(B, dtype=torch.uint8).pin_memory(),
                 its=torch.empty(B, dtype=torch.int16).pin_memory(),
                 ws=torch.empty(api.polar_workspace_bytes(code, B, case["L"], api.POLAR_OP_HYBRID_HOST),
                                dtype=torch.uint8, device="cuda"))
        return s
    s["dec"] = api.Decoder(s["code"], B, case["L"])
    return s


# ------------------------------------------------------------------------------ one pass
def run(s):
    kind = s["kind"]
    if kind == "hybrid":
        return s["dec"].hybrid(s["llr"], s["iters"], _llr_max(s["msg"]), MESSAGES[s["msg"]], s["scales"])
    if kind == "host":
        api.hybrid_decode_host(s["code"], s["llr"], s["iters"], _llr_max(s["msg"]), MESSAGES[s["msg"]], s["scales"],
                               s["L"], s["bits"], s["status"], s["its"], s["ws"])
        return s["bits"], s["status"], s["its"]
    if kind == "scl":
        return s["dec"].scl(s["llr"])
    if kind == "bp":
        api.bp_decode(s["code"], s["llr"], s["iters"], _llr_max(s["msg"]), MESSAGES[s["msg"]] | api.POLAR_FIXED_ITERS,
                      None, s["bits"], s["status"], s["its"], s["lu"], s["lx"])
        return s["bits"], s["status"], s["its"], s["lu"], s["lx"]
    if kind == "mixed":
        return s["dec"].decode(s["code_of"], s["off"], s["llr"], s["iters"], _llr_max(s["msg"]), MESSAGES[s["msg"]])
    if kind == "train":
        s["w"].grad = None
        y = wms.wms_llr_u(s["w"], s["llr"], s["code"], s["T"], 20.0, s["all_iters"])
        loss = wms.bce_loss(y, s["sign"], s["info"])
        loss.backward()
        return loss.detach(), y.detach(), s["w"].grad
    code = s["code"]
    api.polar_random_payload(s["B"], code.P, s["seed"], 0, s["payload"])
    api.polar_encode(code, s["payload"], s["cw"])
    api.polar_awgn_llr(s["cw"], code.N, _sigma(s["ebn0"], code.P / code.N), s["seed"], 0, s["llr"])
    return s["payload"], s["cw"], s["llr"]


def work(case):
    """Inputs read once, outputs written once.  Operations: two additions, two PE functions and two
    clips per PE (6 n N per BP iteration); a frame with early stop needs at least one iteration, one
    that goes to CA-SCL as well f / g on every path, which is not counted (it depends on the noise)."""
    kind, B = case["kind"], case["B"]
    if kind == "mixed":
        n_mean = sum(c[0] for c in MIXED_CODES) / len(MIXED_CODES)
        ops = sum(6 * (c[0].bit_length() - 1) * c[0] for c in MIXED_CODES) / len(MIXED_CODES)
        return {"bytes": B * (4 * n_mean + 12 + max(c[1] - c[2] for c in MIXED_CODES) / 8 + 3), "flops": B * ops}
    N, K, P = case["N"], case["K"], case["K"] - case["crc"]
    n, row = N.bit_length() - 1, (P + 7) // 8
    if kind == "frames":  # ten rounds of the generator per four values, then about forty operations a pair
        return {"bytes": B * (2 * row + 2 * N / 8 + 4 * N), "flops": B * N * 35}
    if kind == "train":
        outs = (case["T"] if case["all_iters"] else 1) * B * N
        return {"bytes": 4 * (B * N + B * K + outs + 2 * case["T"] * 2 * n * N), "flops": B * case["T"] * n * N * (8 + 22)}
    if kind == "bp":
        return {"bytes": B * (12 * N + row + 3), "flops": B * case["iters"] * 6 * n * N}
    if kind == "scl":
        return {"bytes": B * (4 * N + row + 1), "flops": B * case["L"] * n * N}
    return {"bytes": B * (4 * N + row + 3), "flops": B * 6 * n * N}


# ------------------------------------------------------------------------------ 64-bit values
def _frozen(N, K, rate):
    """The Bhattacharyya construction at 0 dB, log domain; ties to the larger index."""
    lz = np.array([-rate])
    while len(lz) < N:
        d = -np.expm1(lz)
        small = lz <= -math.log(2.0)
        minus = np.where(small, lz + np.log(2.0 - np.exp(lz)), np.log1p(-np.where(small, 0.0, d) ** 2))
        lz = np.stack([minus, 2.0 * lz], 1).reshape(-1)
    order = sorted(range(N), key=lambda i: (lz[i], -i))
    f = np.ones(N, bool)
    f[order[:K]] = False
    return torch.from_numpy(f).cuda()


def _philox(blocks, frames, stream, seed):
    """Four 32-bit words of Philox4x32-10 for counters (block, frame, stream, 0), as int64."""
    m32 = 0xFFFFFFFF

    def mul(a, b):  # (high, low) words of a 32 x 32 bit product
        x, y = a * (b & 0xFFFF), a * (b >> 16)
        t = y + (x >> 16)
        return (t >> 16) & m32, ((t << 16) | (x & 0xFFFF)) & m32

    shape = (len(frames), len(blocks))
    c = [blocks[None, :].expand(shape), frames[:, None].expand(shape), torch.full(shape, stream, device="cuda"), torch.zeros(shape, dtype=torch.long, device="cuda")]
    k0, k1 = seed & m32, (seed >> 32) & m32
    for _ in range(10):
        h0, l0 = mul(c[0], 0xD2511F53)
        h1, l1 = mul(c[2], 0xCD9E8D57)
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
    return c


def _exact_frames(N, K, crc, B, ebn0, seed, chunk=4096):
    """[B][N] channel LLRs in 64 bits: payload, CRC, x = u G, BPSK, noise."""
    P, poly = K - crc, {8: 0x07, 16: 0x1021, 24: 0x864CFB}[crc]
    info = torch.nonzero(~_frozen(N, K, P / N))[:, 0]
    sigma = float(np.float32(_sigma(ebn0, P / N)))
    out = torch.empty((B, N), dtype=torch.float64, device="cuda")
    for b0 in range(0, B, chunk):
        f = torch.arange(b0, min(b0 + chunk, B), device="cuda")
        words = torch.stack(_philox(torch.arange((P + 127) // 128, device="cuda"), f, 0, seed), 2).reshape(len(f), -1)
        bits = ((words[:, :, None] >> torch.arange(32, device="cuda")) & 1).reshape(len(f), -1)[:, :P]
        reg = torch.zeros(len(f), dtype=torch.long, device="cuda")
        for p in range(P):
            top = ((reg >> (crc - 1)) & 1) ^ bits[:, p]
            reg = ((reg << 1) & ((1 << crc) - 1)) ^ (top * poly)
        u = torch.zeros((len(f), N), dtype=torch.long, device="cuda")
        u[:, info] = torch.cat([bits, (reg[:, None] >> torch.arange(crc - 1, -1, -1, device="cuda")) & 1], 1)
        d = 1
        while d < N:
            v = u.view(len(f), -1, 2, d)
            v[:, :, 0] ^= v[:, :, 1]
            d *= 2
        r = torch.stack(_philox(torch.arange(N // 4, device="cuda"), f, 1, seed), 2).reshape(len(f), N // 4, 2, 2)
        rad = torch.sqrt(-2.0 * torch.log(((r[..., 0] >> 8) + 1).double() / 16777216.0))
        ang = 2.0 * math.pi * ((r[..., 1] >> 8).double() / 16777216.0)
        z = torch.stack([rad * torch.cos(ang), rad * torch.sin(ang)], -1).reshape(len(f), N)
        out[b0:b0 + len(f)] = 2.0 * (1.0 - 2.0 * u + sigma * z) / sigma ** 2
    return out


def _sgn(v):
    return torch.where(v.detach() < 0, -1.0, 1.0).double()


def _g(a, b, exact=False):
    """The PE function; min-sum passes a gradient to the argument of the smaller magnitude."""
    m = torch.where(a.detach().abs() <= b.detach().abs(), a * _sgn(b), b * _sgn(a))
    if not exact:
        return m
    return m + torch.log1p(torch.exp(-(a + b).abs())) - torch.log1p(torch.exp(-(a - b).abs()))


def _clip(v, M):
    return torch.where(v.detach().abs() < M, v, M * _sgn(v))


def _exact_bp(llr, frozen, T, M, exact=False, w=None):
    """LLR(u) after each of T iterations and LLR(x) after the last, in 64 bits."""
    B, N = llr.shape
    n = N.bit_length() - 1
    R, L = [None] * (n + 2), [torch.zeros((B, N), dtype=torch.float64, device="cuda") for _ in range(n + 2)]
    R[1] = (M * frozen.double()).expand(B, N)
    L[n + 1] = llr.double().clamp(-M, M)
    lu = []

    def pe(s, ins, a, k, weights):  # ins: the sweep's own input column, a: the other one
        d = 1 << (s - 1)
        x, y, q = (t.reshape(B, -1, 2, d) for t in (ins, a, k))
        o1 = _g(x[:, :, 0], y[:, :, 1] + q[:, :, 1], exact)
        o2 = _g(y[:, :, 0], x[:, :, 0], exact)
        if weights is not None:
            ww = weights.view(-1, 2, d)
            o1, o2 = ww[:, 0] * o1, ww[:, 1] * o2
        return torch.stack([_clip(o1, M), _clip(o2 + x[:, :, 1], M)], 2).reshape(B, N)

    for t in range(T):
        for s in range(1, n + 1):
            R[s + 1] = pe(s, R[s], L[s + 1], R[s], None if w is None else w[t, 0, s - 1])
        for s in range(n, 0, -1):
            L[s] = pe(s, L[s + 1], R[s], L[s + 1], None if w is None else w[t, 1, s - 1])
        lu.append(L[1] + R[1])
    return lu, L[n + 1] + R[n + 1]


def exact(case, seed):
    kind = case["kind"]
    if kind == "frames":
        return None, None, _exact_frames(case["N"], case["K"], case["crc"], case["B"], case["ebn0"], seed)
    if kind not in ("bp", "train"):
        return None  # decided bits, statuses and iteration counts: whole numbers
    s = prepare(case, seed)
    frozen = _frozen(case["N"], case["K"], (case["K"] - case["crc"]) / case["N"])
    B, N = s["llr"].shape
    if kind == "bp":
        lu, lx = torch.empty((B, N), dtype=torch.float64, device="cuda"), torch.empty((B, N), dtype=torch.float64, device="cuda")
        for b in range(0, B, 4096):
            u, x = _exact_bp(s["llr"][b:b + 4096], frozen, case["iters"], _llr_max(case["msg"]), case["msg"] == "exact")
            lu[b:b + 4096], lx[b:b + 4096] = u[-1], x
        return None, None, None, lu, lx
    w = s["w"].detach().double().requires_grad_(True)
    every, total, ys = case["all_iters"], 0.0, []
    count = (case["T"] if every else 1) * B * len(s["info"])
    for b in range(0, B, 512):
        lu, _ = _exact_bp(s["llr"][b:b + 512], frozen, case["T"], 20.0, w=w)
        y = torch.stack(lu) if every else lu[-1]
        loss = torch.nn.functional.softplus(-s["sign"][b:b + 512].double() * y[..., s["info"]]).sum() / count
        loss.backward()
        total += float(loss)
        ys.append(y.detach())
    return total, torch.cat(ys, 1 if every else 0), w.grad
