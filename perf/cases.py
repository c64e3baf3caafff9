"""The work that a program has this framework do, as cases that can be timed and compared.

A case names an operation ("op") and its sizes in 16-byte blocks ("blocks") or messages.  Every operation goes
through the package's public calls with the caller's own buffers, as the README shows them.  All results are
bytes and unique (AES is a permutation for each key), so every comparison is exact.
"""
import math

import numpy as np
import torch

import paper_1201_0398_gb300 as gbaes

MIB = 1 << 16  # blocks
NR = {128: 10, 192: 12, 256: 14}


def listed():
    return [
        # One database page or record, into memory that the call itself takes ("fresh"): what a call costs when
        # the cipher is next to nothing.
        {"name": "ecb_enc128_4k", "op": "ecb", "bits": 128, "decrypt": False, "blocks": 256, "fresh": True},
        # A stored object of 1 MiB, written and read back: encryption, then decryption of what it gave.
        {"name": "ecb_roundtrip128_1m", "op": "roundtrip", "bits": 128, "blocks": MIB},
        # A file of odd length, read with the middle key size.
        {"name": "ecb_dec192_9m_odd", "op": "ecb", "bits": 192, "decrypt": True, "blocks": 9 * MIB + 4321,
         "fresh": False},
        # Bulk encryption and decryption of a buffer far larger than the caches.
        {"name": "ecb_enc128_1g", "op": "ecb", "bits": 128, "decrypt": False, "blocks": 1024 * MIB,
         "fresh": False},
        {"name": "ecb_dec256_1g", "op": "ecb", "bits": 256, "decrypt": True, "blocks": 1024 * MIB, "fresh": False},
        # A piece in the middle of a long stream (12-byte nonce, 32-bit block counter), of odd length.
        {"name": "ctr128_be_256m_odd", "op": "ctr", "bits": 128, "kind": gbaes.CTR_BE128, "first": 1_000_003,
         "blocks": 256 * MIB - 77},
        # A short piece of a stream with the little-endian counter of the paper's listing.
        {"name": "ctr256_le_300k", "op": "ctr", "bits": 256, "kind": gbaes.CTR_LE32_CARRY, "first": 0,
         "blocks": 19_201},
        # A large CBC archive, read.
        {"name": "cbc_dec256_256m", "op": "cbc", "bits": 256, "blocks": 256 * MIB},
        # Thousands of messages of uneven length, each with its own key, in one launch of a kept plan.
        {"name": "batch_plan_10k", "op": "batch_plan", "messages": 10_000, "max_bytes": 4 << 20, "keys": 10_000,
         "threads": 512, "bpt": 8},
        # Short messages gathered and sent off at once, with no plan kept.
        {"name": "batch_once_2k_short", "op": "batch_once", "messages": 2_000, "max_bytes": 16 << 10, "keys": 256},
        # Data that lives in page-locked host memory.
        {"name": "pipeline_direct128_64m", "op": "pipeline", "bits": 128, "decrypt": False, "blocks": 64 * MIB},
        # A burst of requests that reach a running server together.
        {"name": "server_burst_256", "op": "server", "messages": 256, "max_bytes": 1 << 20, "keys": 1024},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    op = rng.choice(["ecb", "ecb", "ecb", "roundtrip", "ctr", "ctr", "cbc", "cbc", "batch_plan", "batch_once",
                     "pipeline", "server"])
    bits = rng.choice([128, 192, 256])
    if op == "ecb":
        return {"op": op, "bits": bits, "decrypt": rng.random() < 0.5, "blocks": _log_int(rng, 1, 1024 * MIB),
                "fresh": rng.random() < 0.5}
    if op == "roundtrip":
        return {"op": op, "bits": bits, "blocks": _log_int(rng, 256, 64 * MIB)}
    if op == "ctr":
        return {"op": op, "bits": bits, "kind": rng.choice([gbaes.CTR_BE128, gbaes.CTR_LE32_CARRY]),
                "first": rng.choice([0, rng.randrange(1 << 32)]), "blocks": _log_int(rng, 1, 1024 * MIB)}
    if op == "cbc":
        return {"op": op, "bits": bits, "blocks": _log_int(rng, 1, 1024 * MIB)}
    if op == "batch_plan":
        threads, bpt = rng.choice([(0, 0), (512, 8)])
        n = _log_int(rng, 16, 10_000)
        return {"op": op, "messages": n, "max_bytes": _log_int(rng, 1 << 10, 3 << 20),
                "keys": rng.choice([n, min(n, 64)]), "threads": threads, "bpt": bpt}
    if op == "batch_once":
        n = _log_int(rng, 1, 4_000)
        return {"op": op, "messages": n, "max_bytes": _log_int(rng, 64, 256 << 10), "keys": min(n, 256)}
    if op == "pipeline":
        return {"op": op, "bits": bits, "decrypt": rng.random() < 0.5, "blocks": _log_int(rng, 4096, 64 * MIB)}
    return {"op": "server", "messages": _log_int(rng, 16, 512), "max_bytes": 1 << 20, "keys": 1024}


# ------------------------------------------------------------------- inputs


def _rng(seed):
    return np.random.default_rng([seed, 1201])


def _device_bytes(seed, nbytes):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.randint(0, 256, (nbytes,), dtype=torch.uint8, device="cuda", generator=g)


def _iv(case, rng):
    """16 bytes; for the big-endian counter a random nonce followed by a block counter that starts at 0."""
    iv = rng.integers(0, 256, 16, dtype=np.uint8)
    if case["op"] == "ctr" and case["kind"] == gbaes.CTR_BE128:
        iv[12:] = 0
    return iv.tobytes()


def _messages(case, seed):
    """(raw keys, key size of each, blocks, offset, key index and direction of each message): lengths
    log-uniform from 16 bytes (the case's own, whatever the seed), key sizes 128/192/256 in ratio 2:1:1,
    directions a fair coin."""
    n, nkeys = case["messages"], case["keys"]
    lo = 64 if case["op"] == "server" else 16
    size = np.exp(_rng(n * nkeys).uniform(math.log(lo), math.log(case["max_bytes"]), n))
    blocks = np.maximum(1, np.round(size / 16)).astype(np.int64)
    offset = (np.cumsum(blocks) - blocks) * 16
    rng = _rng(seed)
    bits = rng.permutation(np.resize([128, 192, 128, 256], nkeys))
    keys = [rng.integers(0, 256, b // 8, dtype=np.uint8).tobytes() for b in bits]
    index = rng.permutation(n) if nkeys == n else rng.integers(0, nkeys, n)
    decrypt = rng.integers(0, 2, n)
    return keys, bits, blocks, offset, index, decrypt


def prepare(case, seed):
    op = case["op"]
    s = {"op": op, "case": case}
    if op in ("batch_plan", "batch_once", "server"):
        raw, _, blocks, offset, index, decrypt = _messages(case, seed)
        s["keys"] = [gbaes.Key(k) for k in raw]
        s["in"] = _device_bytes(seed, 16 * int(blocks.sum()))
        s["out"] = torch.zeros_like(s["in"])
        if op == "server":
            r = np.zeros(len(blocks), gbaes.REQUEST)
            r["id"] = np.arange(len(blocks))
            r["in_ptr"] = s["in"].data_ptr() + offset
            r["out_ptr"] = s["out"].data_ptr() + offset
            r["nblocks"], r["key_index"], r["decrypt"] = blocks, index, decrypt
            s["requests"] = r
            s["done"] = np.zeros(len(blocks), gbaes.COMPLETION)
            s["server"] = gbaes.Server(s["keys"])
            torch.cuda.synchronize()  # the server's streams read the inputs as soon as requests arrive
        else:
            s["descs"] = gbaes.make_descs(offset, offset, blocks, index, decrypt)
            if op == "batch_plan":
                s["plan"] = gbaes.BatchPlan(s["descs"], s["keys"], case["threads"], case["bpt"])
        return s
    rng = _rng(seed)
    s["key"] = gbaes.Key(rng.integers(0, 256, case["bits"] // 8, dtype=np.uint8).tobytes())
    s["iv"] = _iv(case, rng)
    s["in"] = _device_bytes(seed, 16 * case["blocks"])
    s["out"] = torch.zeros_like(s["in"])
    if op == "roundtrip":
        s["back"] = torch.zeros_like(s["in"])
    if op == "pipeline":
        s["in"] = s["in"].cpu().pin_memory()
        s["out"] = s["out"].cpu().pin_memory()
        s["pipe"] = gbaes.Pipeline(mode=gbaes.PIPE_DIRECT)
    return s


def run(s):
    op, c = s["op"], s["case"]
    if op == "ecb":
        call = gbaes.decrypt_ecb if c["decrypt"] else gbaes.encrypt_ecb
        return call(s["key"], s["in"]) if c["fresh"] else call(s["key"], s["in"], s["out"])
    if op == "roundtrip":
        out = gbaes.encrypt_ecb(s["key"], s["in"], s["out"])
        return out, gbaes.decrypt_ecb(s["key"], out, s["back"])
    if op == "ctr":
        return gbaes.ctr_xcrypt(s["key"], s["iv"], s["in"], s["out"], kind=c["kind"], first_block=c["first"])
    if op == "cbc":
        return gbaes.cbc_decrypt(s["key"], s["iv"], s["in"], s["out"])
    if op == "batch_plan":
        return s["plan"].launch(s["in"], s["out"])
    if op == "batch_once":
        return gbaes.ecb_batch(s["descs"], s["keys"], s["in"], s["out"])
    if op == "pipeline":
        return s["pipe"].ecb(s["key"], s["in"], s["out"], decrypt=c["decrypt"])
    server = s["server"]
    server.replay(s["requests"])
    server.replay_join()
    server.drain()
    done = server.poll(out=s["done"])
    return s["out"], np.sort(done["id"]).astype(np.int64), done["status"].copy()


def work(case):
    """Each input byte read once, each output byte written once, and each schedule and descriptor once."""
    op = case["op"]
    if op in ("batch_plan", "batch_once", "server"):
        lo, hi, n = (64 if op == "server" else 16), case["max_bytes"], case["messages"]
        mean = (hi - lo) / math.log(hi / lo) if hi > lo else lo
        return {"bytes": 2 * n * mean + 32 * n + 188 * min(n, case["keys"]), "flops": 0}
    return {"bytes": 32 * case["blocks"] * (2 if op == "roundtrip" else 1) + 16 * (NR[case["bits"]] + 1), "flops": 0}


def tolerance(case):
    return "exact"


# ----------------------------------------------------- the same, byte by byte


def _sbox():
    """The S-box and its inverse: inverses in GF(2^8) found by search, then the affine map bit by bit."""
    def mul(a, b):
        p = 0
        while b:
            p ^= a if b & 1 else 0
            a = (a << 1) ^ (0x11B if a & 0x80 else 0)
            b >>= 1
        return p

    box = np.zeros(256, np.uint8)
    for x in range(256):
        inv = next((y for y in range(256) if mul(x, y) == 1), 0)
        v = 0x63
        for i in range(8):
            v ^= (sum((inv >> ((i + k) % 8)) & 1 for k in (0, 4, 5, 6, 7)) & 1) << i
        box[x] = v
    back = np.zeros(256, np.uint8)
    back[box] = np.arange(256, dtype=np.uint8)
    return box, back


def _schedules(keys, box):
    """Round keys [keys, rounds + 1, 16] of keys of one size."""
    k = np.array([list(x) for x in keys], np.uint8)
    nk = k.shape[1] // 4
    w = [k[:, 4 * i:4 * i + 4] for i in range(nk)]
    rcon = 1
    for i in range(nk, 4 * (nk + 7)):
        t = w[-1]
        if i % nk == 0:
            t = box[np.roll(t, -1, 1)]
            t[:, 0] ^= rcon
            rcon = (rcon << 1) ^ (0x11B if rcon & 0x80 else 0)
        elif nk == 8 and i % nk == 4:
            t = box[t]
        w.append(w[i - nk] ^ t)
    return np.concatenate(w, 1).reshape(len(keys), nk + 7, 16)


class _Plain:
    """The cipher on uint8 tensors [blocks, 16], one byte at a time by index, on the GPU."""

    def __init__(self):
        self.np_box, back = _sbox()
        dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
        self.box, self.back = dev(self.np_box), dev(back)
        self.shift = dev(np.array([4 * ((c + r) % 4) + r for c in range(4) for r in range(4)]))
        self.unshift = dev(np.array([4 * ((c - r) % 4) + r for c in range(4) for r in range(4)]))

    @staticmethod
    def twice(x):
        return (x << 1) ^ ((x >> 7) * 0x1B)

    def mix(self, s, inverse):
        s = s.view(-1, 4, 4)
        if inverse:  # as the forward map after adding 4 * (a0 + a2), 4 * (a1 + a3)
            u = self.twice(self.twice(s ^ s.roll(-2, 2)))
            s = s ^ u
        total = s[..., 0] ^ s[..., 1] ^ s[..., 2] ^ s[..., 3]
        return (s ^ total.unsqueeze(-1) ^ self.twice(s ^ s.roll(-1, 2))).view(-1, 16)

    def cipher(self, s, rk, decrypt):
        """rk: [rounds + 1, 16], or [blocks, rounds + 1, 16] for a schedule of its own for each block."""
        key = lambda r: rk[..., r, :]  # noqa: E731
        nr = rk.shape[-2] - 1
        if decrypt:
            s = s ^ key(nr)
            for r in range(nr - 1, -1, -1):
                s = self.back[s[:, self.unshift].int()] ^ key(r)
                s = self.mix(s, True) if r else s
            return s
        s = s ^ key(0)
        for r in range(1, nr + 1):
            s = self.box[s[:, self.shift].int()]
            s = (self.mix(s, False) if r < nr else s) ^ key(r)
        return s


def _counters(case, iv, start, count):
    """Counter blocks start .. start + count - 1 of a stream, mod 2^128, as bytes."""
    order = "big" if case["kind"] == gbaes.CTR_BE128 else "little"
    base = (int.from_bytes(iv, order) + case["first"] + start) % (1 << 128)
    lo = np.uint64(base & (2**64 - 1)) + np.arange(count, dtype=np.uint64)
    hi = np.full(count, base >> 64, np.uint64) + (lo < np.uint64(base & (2**64 - 1))).astype(np.uint64)
    words = [hi.astype(">u8"), lo.astype(">u8")] if order == "big" else [lo.astype("<u8"), hi.astype("<u8")]
    return torch.from_numpy(np.stack([w.view(np.uint8).reshape(-1, 8) for w in words], 1).reshape(-1, 16).copy()).cuda()


def exact(case, seed):
    plain, step, op = _Plain(), 1 << 20, case["op"]
    if op in ("batch_plan", "batch_once", "server"):
        raw, bits, blocks, offset, index, decrypt = _messages(case, seed)
        if int(blocks.sum()) > 64 * MIB:
            return None
        x = _device_bytes(seed, 16 * int(blocks.sum())).view(-1, 16)
        out = torch.zeros_like(x)
        for b in NR:
            of = np.flatnonzero(bits == b)
            if not of.size:
                continue
            place = np.zeros(len(raw), np.int64)
            place[of] = np.arange(of.size)
            rk = torch.from_numpy(_schedules([raw[i] for i in of], plain.np_box)).cuda()
            for d in (0, 1):
                m = np.flatnonzero((bits[index] == b) & (decrypt == d))
                at = np.repeat(offset[m] // 16 - (np.cumsum(blocks[m]) - blocks[m]), blocks[m]) + np.arange(blocks[m].sum())
                which = np.repeat(place[index[m]], blocks[m])
                for i in range(0, len(at), step):
                    rows = torch.from_numpy(at[i:i + step]).cuda()
                    own = rk[torch.from_numpy(which[i:i + step]).cuda()]
                    out[rows] = plain.cipher(x[rows], own, bool(d))
        out = out.view(-1)
        return (out, np.arange(len(blocks)), np.zeros(len(blocks), np.int32)) if op == "server" else out
    rng = _rng(seed)
    key = rng.integers(0, 256, case["bits"] // 8, dtype=np.uint8).tobytes()
    iv = _iv(case, rng)
    rk = torch.from_numpy(_schedules([key], plain.np_box)[0]).cuda()
    x = _device_bytes(seed, 16 * case["blocks"]).view(-1, 16)
    out = torch.zeros_like(x)
    for i in range(0, len(x), step):
        part = x[i:i + step]
        if op == "ctr":
            out[i:i + step] = part ^ plain.cipher(_counters(case, iv, i, len(part)), rk, False)
        elif op == "cbc":
            first = torch.from_numpy(np.frombuffer(iv, np.uint8).copy()).cuda().view(1, 16) if i == 0 else x[i - 1:i]
            out[i:i + step] = plain.cipher(part, rk, True) ^ torch.cat([first, part[:-1]])
        else:
            out[i:i + step] = plain.cipher(part, rk, case.get("decrypt", False))
    out = out.view(-1)
    if op == "roundtrip":
        return out, x.reshape(-1)
    return out.cpu() if op == "pipeline" else out
