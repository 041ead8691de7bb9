"""Performance cases: what programs that use this library have it do.

Each case is one call sequence through the public binding
(``paper_2504_14497_gb300.pcmm``) on inputs made from a seed:

  serve    an encrypted linear layer whose plaintext weights are resident as
           a plan: execute on the request's ciphertexts, normalise the result
  pcmm     a whole plaintext-ciphertext product (plan included), normalised
  batched  many uneven products in one prepared launch, each normalised
  encrypt  encryption of a message array under a resident key workspace
  decrypt  the key owner's decryption of a product's outputs

Ciphertexts are returned as canonical affine points, which are unique, so
outputs are compared as whole numbers.
"""
import math

import numpy as np
import torch

from paper_2504_14497_gb300 import inputs, pcmm


def listed():
    return [
        # The last layer of a small MLP for one encrypted vector: the
        # smallest request a server sees; launches and latency count.
        {"name": "serve_10x128_l1", "kind": "serve", "m": 10, "n": 128, "l": 1, "w": 4},
        # A wide first layer (28 x 28 inputs) for a batch of 64 encrypted
        # columns, the largest single request of the serving workload.
        {"name": "serve_256x784_l64", "kind": "serve", "m": 256, "n": 784, "l": 64, "w": 4},
        # The large product of the benchmark at its widest uint8 entries
        # (strip width 1), at 4 bits (pairs of columns) and at 1 bit (strips
        # of six columns).
        {"name": "pcmm_1024x1024x256_w8", "kind": "pcmm", "m": 1024, "n": 1024, "l": 256, "w": 8, "density": 1.0},
        {"name": "pcmm_1024x1024x256_w4", "kind": "pcmm", "m": 1024, "n": 1024, "l": 256, "w": 4, "density": 1.0},
        {"name": "pcmm_1024x1024x256_w1", "kind": "pcmm", "m": 1024, "n": 1024, "l": 256, "w": 1, "density": 1.0},
        # Pruned 8-bit weights: one entry in ten is non-zero.
        {"name": "pcmm_sparse_w8", "kind": "pcmm", "m": 1024, "n": 1024, "l": 256, "w": 8, "density": 0.1},
        # Odd sizes: a ragged last column block and an odd bit width.
        {"name": "pcmm_333x517x97_w5", "kind": "pcmm", "m": 333, "n": 517, "l": 97, "w": 5, "density": 1.0},
        # 16-bit plaintexts (the widest values the paper measures).
        {"name": "pcmm_512x512x256_w16", "kind": "pcmm", "m": 512, "n": 512, "l": 256, "w": 16, "density": 1.0},
        # A plaintext vector times many independent ciphertext scalars
        # (the vector-scalar product, amortised over a batch of scalars).
        {"name": "vector_512_x16384_w4", "kind": "pcmm", "m": 512, "n": 1, "l": 16384, "w": 4, "density": 1.0},
        # Twelve products of uneven shapes and bit widths in one launch.
        {"name": "batched_12", "kind": "batched", "count": 12, "lo": 32, "hi": 512, "shapes": 4},
        # Encrypting the 1024 x 256 input matrix of the large product.
        {"name": "encrypt_262144", "kind": "encrypt", "count": 262144},
        # Decrypting a 256 x 256 product of 8-bit matrices with an inner
        # dimension of 1024 (messages up to 1024 * 255 * 255).
        {"name": "decrypt_256x1024x256", "kind": "decrypt", "m": 256, "n": 1024, "l": 256, "w": 8},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["serve", "serve", "pcmm", "pcmm", "pcmm", "sparse", "wide", "vector", "batched", "encrypt",
                       "decrypt"])
    if kind == "serve":
        return {"kind": "serve", "m": _log_int(rng, 10, 512), "n": _log_int(rng, 32, 1024), "l": _log_int(rng, 1, 256),
                "w": rng.randint(2, 8)}
    if kind in ("pcmm", "sparse"):
        return {"kind": "pcmm", "m": _log_int(rng, 32, 1024), "n": _log_int(rng, 32, 1024), "l": _log_int(rng, 1, 256),
                "w": rng.randint(1, 8), "density": 1.0 if kind == "pcmm" else round(rng.uniform(0.02, 0.5), 3)}
    if kind == "wide":
        return {"kind": "pcmm", "m": _log_int(rng, 32, 512), "n": _log_int(rng, 32, 512), "l": _log_int(rng, 8, 256),
                "w": rng.randint(9, 16), "density": 1.0}
    if kind == "vector":
        return {"kind": "pcmm", "m": _log_int(rng, 8, 512), "n": 1, "l": _log_int(rng, 512, 16384),
                "w": rng.choice([4, 8]), "density": 1.0}
    if kind == "batched":
        return {"kind": "batched", "count": rng.randint(2, 12), "lo": 32, "hi": rng.randint(64, 320),
                "shapes": rng.randint(0, 1 << 30)}
    if kind == "encrypt":
        return {"kind": "encrypt", "count": _log_int(rng, 1, 262144)}
    return {"kind": "decrypt", "m": _log_int(rng, 16, 256), "n": _log_int(rng, 32, 1024), "l": _log_int(rng, 1, 256),
            "w": rng.choice([4, 8])}


# ------------------------------------------------------------------ inputs

def _generator(seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    return gen


def _scalars(gen, count):
    """count random nonces (quad-planar words); a top limb below 2^31
    keeps each below the group order."""
    r = torch.randint(-(1 << 31), 1 << 31, (2, count, 4), dtype=torch.int64, device="cuda", generator=gen)
    r[1, :, 3] &= (1 << 31) - 1
    r[0, :, 0] |= 1  # not zero
    return r.to(torch.int32).reshape(-1)


def _plaintext(gen, m, n, w, density=1.0):
    if density < 1.0:
        A = torch.randint(1, 1 << w, (m, n), dtype=torch.int64, device="cuda", generator=gen)
        A *= torch.rand((m, n), device="cuda", generator=gen) < density
    else:
        A = torch.randint(0, 1 << w, (m, n), dtype=torch.int64, device="cuda", generator=gen)
    if w <= 8:
        return A.to(torch.uint8)
    return torch.where(A >= 1 << 15, A - (1 << 16), A).to(torch.int16)  # the bits of a uint16


def _key(seed):
    """Secret key and public key H."""
    sk = inputs.uniform_scalars(inputs.streams(int(seed))["sk"], (1,))[0]
    return sk, pcmm.public_key(sk)


_inited = []


def _init():
    if not _inited:
        pcmm.init(torch.cuda.current_device())
        _inited.append(True)


def _encrypted(gen, H, count, ws=None):
    msg = torch.randint(0, 256, (count,), dtype=torch.uint8, device="cuda", generator=gen)
    return msg, pcmm.encrypt(H, msg, _scalars(gen, count), ws=ws)


def prepare(case, seed):
    _init()
    gen = _generator(seed)
    sk, H = _key(seed)
    kind = case["kind"]
    s = {"kind": kind}
    if kind in ("serve", "pcmm"):
        m, n, l, w = case["m"], case["n"], case["l"], case["w"]
        A = _plaintext(gen, m, n, w, case.get("density", 1.0))
        _, s["ctB"] = _encrypted(gen, H, n * l)
        s["l"], s["w"], s["count"] = l, w, m * l
        s["jac"] = torch.empty(pcmm.PCMM_JAC_WORDS * m * l, dtype=torch.int32, device="cuda")
        s["aff"] = torch.empty(pcmm.PCMM_AFF_WORDS * m * l, dtype=torch.int32, device="cuda")
        if kind == "serve":
            # The server picks the strip width once, for a full batch of 256 columns.
            s["plan"] = pcmm.Plan(A, w, pcmm.choose_k(m, n, 256, w))
            s["ws"] = torch.empty(s["plan"].exec_bytes(l), dtype=torch.uint8, device="cuda")
        else:
            s["A"] = A
            s["ws"] = pcmm.workspace(m, n, l, w)
    elif kind == "batched":
        shapes = inputs.batched_shapes(int(case["shapes"]), case["count"], case["lo"], case["hi"])
        items = []
        for m, n, l, w in shapes:
            items.append((_plaintext(gen, m, n, w), _encrypted(gen, H, n * l)[1], l, w, 0))
        s["batch"] = pcmm.Batch(items)
        s["counts"] = [m * l for m, n, l, w in shapes]
        s["affs"] = [torch.empty(pcmm.PCMM_AFF_WORDS * c, dtype=torch.int32, device="cuda") for c in s["counts"]]
    elif kind == "encrypt":
        count = case["count"]
        s["H"] = H
        s["ws"] = torch.zeros(pcmm.encrypt_workspace_bytes(), dtype=torch.uint8, device="cuda")
        s["msg"], _ = _encrypted(gen, H, count, ws=s["ws"])  # the key's table is in the workspace from here on
        s["r"] = _scalars(gen, count)
        s["ct"] = torch.empty(pcmm.PCMM_AFF_WORDS * count, dtype=torch.int32, device="cuda")
    else:
        m, n, l, w = case["m"], case["n"], case["l"], case["w"]
        A = _plaintext(gen, m, n, w)
        _, ctB = _encrypted(gen, H, n * l)
        s["ct"] = pcmm.normalize(pcmm.cussen(A, ctB, l, w), m * l)
        s["sk"], s["count"], s["mmax"] = sk, m * l, n * ((1 << w) - 1) * 255
        s["steps"] = pcmm.BabySteps.for_range(s["mmax"])
        s["out"] = torch.empty(m * l, dtype=torch.int64, device="cuda")
    return s


# --------------------------------------------------------------------- run

def run(s):
    kind = s["kind"]
    if kind == "serve":
        s["plan"].execute(s["ctB"], s["l"], ws=s["ws"], out=s["jac"])
        return pcmm.normalize(s["jac"], s["count"], out=s["aff"])
    if kind == "pcmm":
        pcmm.cussen(s["A"], s["ctB"], s["l"], s["w"], ws=s["ws"], out=s["jac"])
        return pcmm.normalize(s["jac"], s["count"], out=s["aff"])
    if kind == "batched":
        outs = s["batch"].run()
        return [pcmm.normalize(o, c, out=a) for o, c, a in zip(outs, s["counts"], s["affs"])]
    if kind == "encrypt":
        return pcmm.encrypt(s["H"], s["msg"], s["r"], ws=s["ws"], out=s["ct"])
    return pcmm.decrypt(s["sk"], s["ct"], s["count"], s["mmax"], s["steps"], out=s["out"])


def exact(case, seed):
    """Decrypted messages are the integer product; ciphertexts are exact
    whole numbers with no wider form to compare with."""
    if case["kind"] != "decrypt":
        return None
    gen = _generator(seed)
    m, n, l, w = case["m"], case["n"], case["l"], case["w"]
    A = _plaintext(gen, m, n, w).cpu().numpy().astype(np.int64)
    B = torch.randint(0, 256, (n * l,), dtype=torch.uint8, device="cuda", generator=gen).cpu().numpy()
    return (A @ B.reshape(n, l).astype(np.int64)).reshape(-1)


# -------------------------------------------------------------------- work

# 32 x 32 limb products of the cheapest known group operations: an affine
# addition inside a batch (5 multiplications of 64 products and a squaring of
# 36) and a doubling (3 and 5).
_ADD = 5 * 64 + 36
_DBL = 3 * 64 + 5 * 36


def _product_work(m, n, l, w, density=1.0, plan=False):
    """Strips of floor(8 / w) columns: one table entry per distinct non-zero
    code and one addition per row, strip and chain with a non-zero code."""
    k = max(1, 8 // w)
    strips = -(-n // k)
    codes = 2.0 ** (w * k) - 1
    nz = m * (1.0 - (1.0 - density * (1.0 - 2.0 ** -w)) ** k)
    entries = codes * -math.expm1(nz * math.log1p(-1.0 / codes)) if codes > 1 else 1.0
    adds = 2.0 * l * strips * (nz + entries)
    size = 1 if w <= 8 else 2
    bytes_ = (0 if plan else m * n * size) + 4 * pcmm.PCMM_AFF_WORDS * (n * l + m * l)
    return bytes_, 2.0 * _ADD * adds


def work(case):
    kind = case["kind"]
    if kind in ("serve", "pcmm"):
        b, f = _product_work(case["m"], case["n"], case["l"], case["w"], case.get("density", 1.0), kind == "serve")
    elif kind == "batched":
        b = f = 0.0
        for shape in inputs.batched_shapes(int(case["shapes"]), case["count"], case["lo"], case["hi"]):
            x, y = _product_work(*shape)
            b, f = b + x, f + y
    elif kind == "encrypt":
        # One addition per byte of the nonce and base point, one for the message.
        b, f = case["count"] * (1 + 32 + 128.0), case["count"] * 65 * 2.0 * _ADD
    else:
        # A 256-bit scalar multiplication (256 doublings, 51 additions) and
        # one table probe per ciphertext.
        count = case["m"] * case["l"]
        b, f = count * (128 + 8 + 8.0), count * 2.0 * (256 * _DBL + 52 * _ADD)
    return {"bytes": float(b), "flops": float(f)}
