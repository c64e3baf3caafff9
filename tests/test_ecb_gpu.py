"""GPU parity: the T-table kernels against the CPU oracle, bit for bit.

AES is a permutation per key, so the result is unique and the tolerance is zero
(Section 2.1's cipher; Eq. 1 is a re-arrangement of the same arithmetic).
"""
import ctypes
import json
import os

import numpy as np
import pytest

import oracle
from paper_1201_0398_gb300 import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BITS = (128, 192, 256)


def dev(a: np.ndarray):
    a = np.ascontiguousarray(a)
    return torch.from_numpy(a if a.flags.writeable else a.copy()).cuda()


def host(t) -> np.ndarray:
    torch.cuda.synchronize()
    return t.cpu().numpy()


def sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


def test_small_workload_encrypt_then_decrypt(gbaes):
    key, data = workloads.small_workload()
    k = gbaes.Key(key)
    x = dev(data)
    c = gbaes.encrypt_ecb(k, x)
    p = gbaes.decrypt_ecb(k, c)
    want_c = oracle.ecb(key, 128, data)
    assert np.array_equal(host(c), want_c)
    assert np.array_equal(host(p), data)
    assert np.array_equal(host(p), oracle.ecb(key, 128, want_c, decrypt=True))
    assert gbaes.device_status() == 0


def edge_sizes():
    tile = 1024 * 2
    full = sms() * tile
    return sorted({1, 2, 3, 31, 32, 33, 1023, 1024, 1025, tile - 1, tile, tile + 1, full - 1, full, full + 1,
                   3 * full + 17})


@pytest.mark.parametrize("bits", BITS)
@pytest.mark.parametrize("decrypt", (False, True))
def test_edge_sizes_vs_oracle(gbaes, bits, decrypt):
    rng = np.random.default_rng(bits + 7 * decrypt)
    key = rng.integers(0, 256, bits // 8, dtype=np.uint8).tobytes()
    k = gbaes.Key(key)
    for n in edge_sizes():
        data = rng.integers(0, 256, 16 * n, dtype=np.uint8)
        out = (gbaes.decrypt_ecb if decrypt else gbaes.encrypt_ecb)(k, dev(data))
        assert np.array_equal(host(out), oracle.ecb(key, bits, data, decrypt=decrypt)), n


@pytest.mark.parametrize("threads", (64, 256, 512, 768, 1024))
@pytest.mark.parametrize("bpt", (1, 2, 4))
def test_every_launch_shape(gbaes, threads, bpt):
    rng = np.random.default_rng(threads * 10 + bpt)
    n = sms() * threads * bpt + threads + 5  # all CTAs busy, a second pass, a ragged tail
    for bits in (128, 256):
        key = rng.integers(0, 256, bits // 8, dtype=np.uint8).tobytes()
        k = gbaes.Key(key)
        data = rng.integers(0, 256, 16 * n, dtype=np.uint8)
        for decrypt in (False, True):
            out = gbaes.ecb_ex(k, dev(data), decrypt=decrypt, threads=threads, blocks_per_thread=bpt)
            assert np.array_equal(host(out), oracle.ecb(key, bits, data, decrypt=decrypt))


def test_in_place_and_side_stream(gbaes):
    rng = np.random.default_rng(5)
    key = rng.integers(0, 256, 32, dtype=np.uint8).tobytes()
    k = gbaes.Key(key)
    data = rng.integers(0, 256, 16 * 100_003, dtype=np.uint8)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        x = dev(data)
        gbaes.encrypt_ecb(k, x, out=x)
        s.synchronize()
    assert np.array_equal(host(x), oracle.ecb(key, 256, data))
    gbaes.decrypt_ecb(k, x, out=x, stream=s)
    s.synchronize()
    assert np.array_equal(host(x), data)


def test_golden_known_answers(gbaes):
    path = os.path.join(os.path.dirname(__file__), "golden", "ecb_kat.json")
    for v in json.load(open(path))["vectors"]:
        k = gbaes.Key(bytes.fromhex(v["key"]))
        pt = np.frombuffer(bytes.fromhex(v["plaintext"]), np.uint8)
        ct = np.frombuffer(bytes.fromhex(v["ciphertext"]), np.uint8)
        assert host(gbaes.encrypt_ecb(k, dev(pt))).tobytes() == ct.tobytes()
        assert host(gbaes.decrypt_ecb(k, dev(ct))).tobytes() == pt.tobytes()


def test_argument_errors(gbaes):
    k = gbaes.Key(bytes(16))
    buf = torch.zeros(16 * 64 + 16, dtype=torch.uint8, device="cuda")
    with pytest.raises(gbaes.AesError) as e:  # misaligned
        gbaes.encrypt_ecb(k, buf[1:1 + 16 * 8], out=buf[32:32 + 16 * 8].clone())
    assert e.value.name == "AES_ERR_ALIGN"
    with pytest.raises(gbaes.AesError) as e:  # partial overlap
        gbaes.encrypt_ecb(k, buf[0:16 * 8], out=buf[16:16 * 9])
    assert e.value.name == "AES_ERR_ARG"
    lib = gbaes.load()
    import ctypes

    base = ctypes.c_void_p(buf.data_ptr())
    # a range running past the end of its allocation is rejected on the host
    big = torch.zeros(16 * 4, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    rc = lib.aes_encrypt_ecb(k.handle, ctypes.c_void_p(big.data_ptr()), ctypes.c_void_p(big.data_ptr()),
                             1 << 40, None)
    assert rc == -1
    assert lib.aes_encrypt_ecb(k.handle, base, base, 0, None) == 0  # empty input: no-op
    with pytest.raises(gbaes.AesError):
        gbaes.ecb_ex(k, buf[:16 * 8], threads=100)
    with pytest.raises(gbaes.AesError):
        gbaes.ecb_ex(k, buf[:16 * 8], blocks_per_thread=3)
    assert gbaes.device_status() == 0


@pytest.mark.parametrize("bits", BITS)
def test_ctr_vs_oracle(gbaes, bits):
    rng = np.random.default_rng(600 + bits)
    key = rng.integers(0, 256, bits // 8, dtype=np.uint8).tobytes()
    k = gbaes.Key(key)
    n = 3 * sms() * 2048 + 77
    data = rng.integers(0, 256, 16 * n, dtype=np.uint8)
    ivs = [rng.integers(0, 256, 16, dtype=np.uint8).tobytes(), b"\xff" * 16,
           (0xFFFFFF00).to_bytes(4, "little") + b"\xff" * 4 + bytes(8)]
    for iv in ivs:
        for kind in (oracle.CTR_BE128, oracle.CTR_LE32_CARRY):
            out = gbaes.ctr_xcrypt(k, iv, dev(data), kind=kind)
            assert np.array_equal(host(out), oracle.ctr(key, bits, iv, data, kind)), (iv.hex(), kind)
    # a message processed in two pieces equals one call (first_block offsets the counter)
    iv = ivs[0]
    x = dev(data)
    half = (n // 2) * 16
    a = gbaes.ctr_xcrypt(k, iv, x[:half])
    b = gbaes.ctr_xcrypt(k, iv, x[half:], first_block=n // 2)
    assert np.array_equal(np.concatenate([host(a), host(b)]), oracle.ctr(key, bits, iv, data))
    # in place
    gbaes.ctr_xcrypt(k, iv, x, out=x)
    assert np.array_equal(host(x), oracle.ctr(key, bits, iv, data))


@pytest.mark.parametrize("bits", BITS)
@pytest.mark.parametrize("passes", (0, 1, 2))
def test_full_passes_and_shares_of_the_rest(gbaes, bits, passes):
    """The table kernel takes full passes of all CTAs, then equal shares of the rest:
    sizes at and around whole passes of two CTAs of 512 threads per SM, a block or
    two per thread, in every mode and, for ECB, in every launch shape that divides
    the rest differently."""
    rng = np.random.default_rng(bits + passes)
    key = rng.integers(0, 256, bits // 8, dtype=np.uint8).tobytes()
    k = gbaes.Key(key)
    iv = rng.integers(0, 256, 16, dtype=np.uint8).tobytes()
    base = 2 * sms() * 512
    sizes = [max(passes, 1) * base + d for d in (-33, 0, 1, 545)] + ([2 * passes * base + 31] if passes else [257, 9728])
    data = rng.integers(0, 256, 16 * max(sizes), dtype=np.uint8)
    enc, dec = oracle.ecb(key, bits, data), oracle.ecb(key, bits, data, decrypt=True)
    ctr, cbc = oracle.ctr(key, bits, iv, data), oracle.cbc_decrypt(key, bits, iv, data)
    x = dev(data)
    for n in sizes:
        for threads, bpt in ((0, 0), (512, 1), (512, 2), (512, 4), (1024, 1), (96, 2), (64, 4)):
            for d, want in ((False, enc), (True, dec)):
                y = gbaes.ecb_ex(k, x[:16 * n], decrypt=d, kernel=gbaes.KERNEL_TABLE_REPLICATED, threads=threads,
                                 blocks_per_thread=bpt)
                assert np.array_equal(host(y), want[:16 * n]), (n, threads, bpt, d)
        assert np.array_equal(host(gbaes.ctr_xcrypt(k, iv, x[:16 * n])), ctr[:16 * n]), n
        assert np.array_equal(host(gbaes.cbc_decrypt(k, iv, x[:16 * n])), cbc[:16 * n]), n
    assert gbaes.device_status() == 0


@pytest.mark.parametrize("bits", BITS)
@pytest.mark.parametrize("kind", ("CTR_BE128", "CTR_LE32_CARRY"))
def test_ctr_long_inputs_share_their_first_rounds(gbaes, bits, kind):
    """Inputs from the length at which rows of 256 counters share the first two
    rounds (one block below it, at it, and with ragged last rows), from first
    counters at the edges of a row, of the 2^16 counters that agree in their
    upper bytes, of a 64-bit half and of 2^128, and with a block index: as the
    oracle computes them from the counter that comes out, and in place."""
    rng = np.random.default_rng(bits)
    key = rng.integers(0, 256, bits // 8, dtype=np.uint8).tobytes()
    k = gbaes.Key(key)
    least = sms() * 2 * 256 * 5
    order = "big" if kind == "CTR_BE128" else "little"
    nonce = int.from_bytes(rng.integers(0, 256, 16, dtype=np.uint8).tobytes(), "big") & ~((1 << 64) - 1)
    firsts = (nonce, nonce | 0xFF, nonce | 0x100, nonce | 0xFFFF, nonce | 0x12FFE1, nonce | ((1 << 64) - 70_000),
              (1 << 128) - 1)
    data = rng.integers(0, 256, 16 * (least + 9001), dtype=np.uint8)
    x = dev(data)
    for j, first in enumerate(firsts):
        n = least + (0, 1, -1, 255, 9001, 31, 4096)[j]
        index = (0, 3, 1 << 40, 65_537, 0, (1 << 64) - n - 1, 12_345)[j]
        iv = ((first - index) % (1 << 128)).to_bytes(16, order)
        got = gbaes.ctr_xcrypt(k, iv, x[:16 * n], kind=getattr(gbaes, kind), first_block=index)
        want = oracle.ctr(key, bits, first.to_bytes(16, order), data[:16 * n], getattr(oracle, kind))
        assert np.array_equal(host(got), want), (hex(first), n, index)
    gbaes.ctr_xcrypt(k, iv, x[:16 * n], out=x[:16 * n], kind=getattr(gbaes, kind), first_block=index)
    assert np.array_equal(host(x[:16 * n]), want) and np.array_equal(host(x[16 * n:]), data[16 * n:])
    assert gbaes.device_status() == 0


@pytest.mark.parametrize("bits", BITS)
def test_cbc_decrypt_vs_oracle(gbaes, bits):
    rng = np.random.default_rng(700 + bits)
    key = rng.integers(0, 256, bits // 8, dtype=np.uint8).tobytes()
    iv = rng.integers(0, 256, 16, dtype=np.uint8).tobytes()
    k = gbaes.Key(key)
    for n in (1, 2, 33, 2 * sms() * 2048 + 5):
        data = rng.integers(0, 256, 16 * n, dtype=np.uint8)
        out = gbaes.cbc_decrypt(k, iv, dev(data))
        assert np.array_equal(host(out), oracle.cbc_decrypt(key, bits, iv, data)), n
    x = dev(data)
    with pytest.raises(gbaes.AesError):
        gbaes.cbc_decrypt(k, iv, x, out=x)
    # two pieces chained through the iv argument
    h = (n // 2) * 16
    a = gbaes.cbc_decrypt(k, iv, x[:h])
    b = gbaes.cbc_decrypt(k, data[h - 16:h].tobytes(), x[h:])
    assert np.array_equal(np.concatenate([host(a), host(b)]), oracle.cbc_decrypt(key, bits, iv, data))


def sampled_parity(key, bits, x, out, decrypt, nsample=1 << 15, seed=0):
    """Compares out against the oracle on nsample random blocks of x."""
    nblocks = x.numel() // 16
    idx = np.random.default_rng(seed).choice(nblocks, size=min(nsample, nblocks), replace=False)
    idx = np.concatenate([idx, [0, nblocks - 1]])
    ti = torch.from_numpy(idx).cuda()
    xs = host(x.view(-1, 16)[ti]).reshape(-1)
    os_ = host(out.view(-1, 16)[ti]).reshape(-1)
    assert np.array_equal(os_, oracle.ecb(key, bits, xs, decrypt=decrypt))


@pytest.mark.parametrize("bits", BITS)
def test_one_gib_single_launch(gbaes, bits):
    """1 GiB device-resident buffer per key size, one launch per direction:
    sampled blocks against the oracle, and decrypt(encrypt(x)) == x everywhere."""
    key = workloads.random_key(workloads.SEED_BULK[bits], bits)
    k = gbaes.Key(key)
    x = workloads.device_bytes(workloads.SEED_BULK[bits], workloads.GiB)
    c = gbaes.encrypt_ecb(k, x)
    sampled_parity(key, bits, x, c, False)
    p = gbaes.decrypt_ecb(k, c)
    sampled_parity(key, bits, c, p, True, seed=1)
    assert torch.equal(p, x)
    del c, p, x
    torch.cuda.empty_cache()


@pytest.mark.parametrize("bits", (128, 256))
@pytest.mark.parametrize("kind", (oracle.CTR_BE128, oracle.CTR_LE32_CARRY))
def test_ctr_and_cbc_one_gib(gbaes, bits, kind):
    """The modes at the bench's size (1 GiB, 2^26 blocks, one launch each): the
    CTR keystream (output XOR input) on 2^14 sampled blocks equals the oracle's
    encryption of those blocks' counter blocks, and CTR applied twice gives the
    input back everywhere; CBC decryption on sampled blocks (the first, whose
    predecessor is the IV, and the last included) equals the oracle's
    decryption of the block XOR the previous ciphertext block."""
    key = workloads.random_key(90 + bits, bits)
    k = gbaes.Key(key)
    x = workloads.device_bytes(91 + bits, workloads.GiB)
    n = x.numel() // 16
    iv = bytes(range(0xF0, 0x100))  # low bytes near a carry
    rng = np.random.default_rng(bits + kind)
    idx = np.concatenate([[0, 1, n - 1], rng.choice(n, 1 << 14, replace=False)])
    ti = torch.from_numpy(idx).cuda()
    xb = host(x.view(-1, 16)[ti])
    c = gbaes.ctr_xcrypt(k, iv, x, kind=kind)
    ks = host(c.view(-1, 16)[ti]) ^ xb
    ctrs = np.frombuffer(b"".join(oracle.counter_block(iv, int(i), kind) for i in idx), np.uint8)
    assert np.array_equal(ks.reshape(-1), oracle.ecb(key, bits, ctrs))
    assert torch.equal(gbaes.ctr_xcrypt(k, iv, c, kind=kind), x)
    del c
    if kind == oracle.CTR_BE128:
        d = gbaes.cbc_decrypt(k, iv, x)
        prev_idx = torch.from_numpy(np.maximum(idx - 1, 0)).cuda()
        prev = host(x.view(-1, 16)[prev_idx])
        prev[idx == 0] = np.frombuffer(iv, np.uint8)
        want = oracle.ecb(key, bits, xb.reshape(-1), decrypt=True).reshape(-1, 16) ^ prev
        assert np.array_equal(host(d.view(-1, 16)[ti]), want)
        del d
    del x
    torch.cuda.empty_cache()


@pytest.mark.parametrize("gib", (4, 16))
def test_sweep_top_sizes_sampled(gbaes, gib):
    """The largest sweep points (4 and 16 GiB; 2^28 and 2^30 blocks): 64-bit
    block indices.  AES-128 and AES-256 encryption against the oracle on 2^20
    sampled blocks (plus the first and last), and the whole output against the
    bitsliced kernel's, which shares no table, round or indexing code."""
    free, _ = torch.cuda.mem_get_info()
    if free < 3 * gib * workloads.GiB + workloads.GiB:
        pytest.skip("not enough device memory")
    x = workloads.device_bytes(11, gib * workloads.GiB)
    for bits in (128, 256):
        key = workloads.random_key(20 + bits, bits)
        k = gbaes.Key(key)
        c = gbaes.encrypt_ecb(k, x)
        sampled_parity(key, bits, x, c, False, nsample=1 << 20, seed=bits)
        b = gbaes.ecb_ex(k, x, kernel=gbaes.KERNEL_BITSLICED)
        assert torch.equal(b, c)
        del b, c
    del x
    torch.cuda.empty_cache()


@pytest.mark.parametrize("bits", BITS)
def test_bitsliced_kernel_vs_oracle(gbaes, bits):
    """The Boolean-circuit kernel (a lane pair holds 32 blocks as bit planes, split
    by state columns; a warp takes 512 blocks, a CTA 2,048): edge sizes around a
    pair's, a warp's and a CTA's tile, and more than one pass of the full grid
    (152 SMs x 4 CTAs for decryption, x 5 for encryption, x 2,048 blocks) with a
    ragged tail."""
    rng = np.random.default_rng(900 + bits)
    key = rng.integers(0, 256, bits // 8, dtype=np.uint8).tobytes()
    k = gbaes.Key(key)
    for n in (1, 15, 16, 17, 31, 33, 511, 512, 513, 2047, 2049, 4097, sms() * 5 * 2048 + 2048 * 3 + 5):
        data = rng.integers(0, 256, 16 * n, dtype=np.uint8)
        for decrypt in (False, True):
            out = gbaes.ecb_ex(k, dev(data), decrypt=decrypt, kernel=gbaes.KERNEL_BITSLICED)
            assert np.array_equal(host(out), oracle.ecb(key, bits, data, decrypt=decrypt)), (n, decrypt)


def test_bitsliced_equals_table_kernel_large(gbaes):
    x = workloads.device_bytes(77, 256 << 20)
    for bits in BITS:
        k = gbaes.Key(workloads.random_key(70 + bits, bits))
        for decrypt in (False, True):
            a = gbaes.ecb_ex(k, x, decrypt=decrypt, kernel=gbaes.KERNEL_TABLE)
            b = gbaes.ecb_ex(k, x, decrypt=decrypt, kernel=gbaes.KERNEL_BITSLICED)
            assert torch.equal(a, b)


def test_ctr_counter_index_limit(gbaes):
    """Block indices are 64-bit: a call whose last index would pass 2^64 - 1 is
    refused on the host; one ending exactly at 2^64 - 1 runs, its counters
    taken as IV + index modulo 2^128 (checked against plain integer arithmetic
    and ECB of those counter blocks)."""
    key = bytes(range(16))
    k = gbaes.Key(key)
    iv = bytes(16)
    x = torch.zeros(16 * 4, dtype=torch.uint8, device="cuda")
    with pytest.raises(gbaes.AesError):
        gbaes.ctr_xcrypt(k, iv, x, first_block=(1 << 64) - 3)
    first = (1 << 64) - 4
    out = host(gbaes.ctr_xcrypt(k, iv, x, first_block=first))
    ctrs = b"".join((first + i).to_bytes(16, "big") for i in range(4))
    assert out.tobytes() == oracle.ecb(key, 128, np.frombuffer(ctrs, np.uint8)).tobytes()


def test_default_kernel_switch(gbaes):
    """aes_set_kernel changes what aes_encrypt_ecb / aes_decrypt_ecb run; the
    result is the same bytes either way."""
    rng = np.random.default_rng(55)
    key = rng.integers(0, 256, 24, dtype=np.uint8).tobytes()
    k = gbaes.Key(key)
    data = rng.integers(0, 256, 16 * 5000, dtype=np.uint8)
    want = oracle.ecb(key, 192, data)
    prev = gbaes.set_kernel(gbaes.KERNEL_BITSLICED)
    try:
        assert np.array_equal(host(gbaes.encrypt_ecb(k, dev(data))), want)
        assert np.array_equal(host(gbaes.decrypt_ecb(k, dev(want))), data)
    finally:
        gbaes.set_kernel(prev)
    assert np.array_equal(host(gbaes.encrypt_ecb(k, dev(data))), want)


@pytest.mark.parametrize("shape", __import__("paper_1201_0398_gb300.autotune", fromlist=["x"]).ECB_CANDIDATES)
def test_one_gib_every_tuner_shape(gbaes, shape):
    """The 1 GiB single-launch workload in every launch shape the autotuner may
    pick for the bench: sampled blocks against the oracle, AES-128 encryption and
    AES-256 decryption (the bench's dominant launch)."""
    threads, bpt = shape
    x = workloads.device_bytes(workloads.SEED_BULK[128], workloads.GiB)
    for bits, dec in ((128, False), (256, True)):
        key = workloads.random_key(workloads.SEED_BULK[bits], bits)
        k = gbaes.Key(key)
        out = gbaes.ecb_ex(k, x, decrypt=dec, threads=threads, blocks_per_thread=bpt)
        sampled_parity(key, bits, x, out, dec, nsample=1 << 13, seed=threads + bpt)
        del out
    del x
    torch.cuda.empty_cache()


def compact_sizes():
    """Sizes around the compact kernel's shapes: one warp, warps spread one per
    SM, 8 warps per CTA, the grid cap (8 CTAs per SM) with a grid-stride tail."""
    w = 32
    return sorted({1, 2, 31, 32, 33, 255, 256, 257, sms() * w - 1, sms() * w, sms() * w + 1,
                   sms() * 8 * w + 3, 8 * sms() * 8 * w - 1, 8 * sms() * 8 * w + 1000})


@pytest.mark.parametrize("bits", BITS)
def test_compact_tables_vs_oracle(gbaes, bits):
    """The compact-table kernel (each table stored once), and short CTR and CBC calls."""
    rng = np.random.default_rng(1300 + bits)
    key = rng.integers(0, 256, bits // 8, dtype=np.uint8).tobytes()
    iv = rng.integers(0, 256, 16, dtype=np.uint8).tobytes()
    k = gbaes.Key(key)
    for n in compact_sizes():
        data = rng.integers(0, 256, 16 * n, dtype=np.uint8)
        x = dev(data)
        for decrypt in (False, True):
            out = gbaes.ecb_ex(k, x, decrypt=decrypt, kernel=gbaes.KERNEL_TABLE_COMPACT)
            assert np.array_equal(host(out), oracle.ecb(key, bits, data, decrypt=decrypt)), (n, decrypt)
        if n <= 128 * sms():  # (CTR and CBC decryption have the replicated table only)
            for kind in (oracle.CTR_BE128, oracle.CTR_LE32_CARRY):
                assert np.array_equal(host(gbaes.ctr_xcrypt(k, iv, x, kind=kind)),
                                      oracle.ctr(key, bits, iv, data, kind)), (n, kind)
            assert np.array_equal(host(gbaes.cbc_decrypt(k, iv, x)), oracle.cbc_decrypt(key, bits, iv, data)), n
    assert gbaes.device_status() == 0


@pytest.mark.parametrize("decrypt", (False, True))
def test_size_dispatch_and_balanced_shapes_vs_oracle(gbaes, decrypt):
    """AES_KERNEL_TABLE runs one CTA per SM for short calls and two above, and shrinks
    its CTAs so that calls of a few tiles per SM spread evenly.  Sizes on both sides
    of the switch and across the shrinking range, through the default call and both variants forced."""
    rng = np.random.default_rng(1400 + decrypt)
    s = sms()
    for bits in (128, 256):
        key = rng.integers(0, 256, bits // 8, dtype=np.uint8).tobytes()
        k = gbaes.Key(key)
        for n in (128 * s - 1, 128 * s, 128 * s + 1, 65536, 3 * s * 1024 + 7, 262144, (1 << 20) + 13):
            data = rng.integers(0, 256, 16 * n, dtype=np.uint8)
            want = oracle.ecb(key, bits, data, decrypt=decrypt)
            x = dev(data)
            out = (gbaes.decrypt_ecb if decrypt else gbaes.encrypt_ecb)(k, x)
            assert np.array_equal(host(out), want), n
            for kid in (gbaes.KERNEL_TABLE_REPLICATED, gbaes.KERNEL_TABLE_COMPACT):
                for bpt in (1, 2, 4):
                    out = gbaes.ecb_ex(k, x, decrypt=decrypt, kernel=kid, blocks_per_thread=bpt)
                    assert np.array_equal(host(out), want), (n, kid, bpt)
    assert gbaes.device_status() == 0


@pytest.mark.parametrize("captured", (False, True))
@pytest.mark.parametrize("n", (1, 4096, 19_456, 19_457, 65_536, 400_000))
def test_dependent_calls_back_to_back(gbaes, n, captured):
    """Calls that each take the one before's output, in place and without a wait
    between them, mixed with torch's own kernels and batches: each must see the
    finished output of its predecessor (a kernel may start while the one before
    it in the stream still runs).  Undoing every step gives the input back, and
    the state in the middle is the oracle's."""
    rng = np.random.default_rng(n)
    raw = [rng.integers(0, 256, b // 8, dtype=np.uint8).tobytes() for b in BITS]
    ks = [gbaes.Key(r) for r in raw]
    data = rng.integers(0, 256, 16 * n, dtype=np.uint8)
    iv = bytes(range(16))
    cut = n // 2
    descs = [gbaes.make_descs([0, 16 * cut], [0, 16 * cut], [cut, n - cut], [0, 2], [d, 1 - d]) for d in (0, 1)]
    plans = [gbaes.BatchPlan(d, ks) for d in descs]
    steps = 6
    x = dev(data)
    mid = torch.empty_like(x)

    def chain():
        for i in range(steps):
            gbaes.encrypt_ecb(ks[i % 3], x, x)
            gbaes.ctr_xcrypt(ks[(i + 1) % 3], iv, x, x, first_block=i)
            plans[0].launch(x, x)
            x.bitwise_xor_(i + 1)
        mid.copy_(x)
        for i in reversed(range(steps)):
            x.bitwise_xor_(i + 1)
            plans[1].launch(x, x)
            gbaes.ctr_xcrypt(ks[(i + 1) % 3], iv, x, x, first_block=i)
            gbaes.decrypt_ecb(ks[i % 3], x, x)

    if captured:
        s = torch.cuda.Stream()
        torch.cuda.synchronize()
        with torch.cuda.stream(s):
            chain()
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            chain()
        g.replay()
        g.replay()
    else:
        chain()
    assert np.array_equal(host(x), data)
    want = data
    for i in range(steps):
        want = oracle.ecb(raw[i % 3], BITS[i % 3], want)
        shifted = ((int.from_bytes(iv, "big") + i) % (1 << 128)).to_bytes(16, "big")
        want = oracle.ctr(raw[(i + 1) % 3], BITS[(i + 1) % 3], shifted, want)
        parts = [oracle.ecb(raw[0], 128, want[:16 * cut])] if cut else []
        want = np.concatenate(parts + [oracle.ecb(raw[2], 256, want[16 * cut:], decrypt=True)]) ^ np.uint8(i + 1)
    assert np.array_equal(host(mid), want)
    assert gbaes.device_status() == 0


@pytest.mark.parametrize("n", (9728, 30_001, 155_649, 400_003))
def test_dependent_calls_on_buffers_off_by_a_block(gbaes, n):
    """Buffers that begin 16 bytes into a 32-byte sector, so that warps (and CTAs)
    share sectors: calls that follow one another without a wait, in place and from
    buffer to buffer, must not see a half that a cache kept from before."""
    rng = np.random.default_rng(n)
    raw = [rng.integers(0, 256, b // 8, dtype=np.uint8).tobytes() for b in BITS]
    ks = [gbaes.Key(r) for r in raw]
    iv = bytes(range(16))
    bufs = [torch.zeros(16 * (n + 2), dtype=torch.uint8, device="cuda") for _ in range(2)]
    x, y = (b[16:16 * (n + 1)] for b in bufs)
    data = rng.integers(0, 256, 16 * n, dtype=np.uint8)
    x.copy_(torch.from_numpy(data))
    plan = gbaes.BatchPlan(gbaes.make_descs([0], [0], [n], [1], [0]), ks)
    steps = 12
    for i in range(steps):
        gbaes.encrypt_ecb(ks[i % 3], x, x)
        gbaes.cbc_decrypt(ks[(i + 1) % 3], iv, x, y)
        gbaes.ctr_xcrypt(ks[(i + 2) % 3], iv, y, x)
        plan.launch(x, x)
        gbaes.decrypt_ecb(ks[i % 3], x, y)
        gbaes.cbc_decrypt(ks[i % 3], iv, y, x)
    want = data
    for i in range(steps):
        want = oracle.ecb(raw[i % 3], BITS[i % 3], want)
        want = oracle.cbc_decrypt(raw[(i + 1) % 3], BITS[(i + 1) % 3], iv, want)
        want = oracle.ctr(raw[(i + 2) % 3], BITS[(i + 2) % 3], iv, want)
        want = oracle.ecb(raw[1], BITS[1], want)
        want = oracle.ecb(raw[i % 3], BITS[i % 3], want, decrypt=True)
        want = oracle.cbc_decrypt(raw[i % 3], BITS[i % 3], iv, want)
    assert np.array_equal(host(x), want)
    for b in bufs:  # nothing before or after the blocks
        assert not host(b[:16]).any() and not host(b[16 * (n + 1):]).any()
    assert gbaes.device_status() == 0


@pytest.mark.parametrize("n", (1, 4097, 65_536, 300_001))
def test_dependent_calls_of_other_kernels_and_streams(gbaes, n):
    """The bitsliced kernel, the allocation-free batch and the direct host pipeline
    in chains of calls without a wait on the host, each on its predecessor's output,
    and the chain handed to the other of two streams by events at every step."""
    rng = np.random.default_rng(n)
    raw = [rng.integers(0, 256, b // 8, dtype=np.uint8).tobytes() for b in BITS]
    ks = [gbaes.Key(r) for r in raw]
    data = rng.integers(0, 256, 16 * n, dtype=np.uint8)
    lib = gbaes.load()
    ctxs = gbaes._ctx_array(ks)
    cut = n // 3
    descs = gbaes.make_descs([0, 16 * cut], [0, 16 * cut], [cut, n - cut], [1, 2], [1, 0])
    x = dev(data)
    h = torch.empty(16 * n, dtype=torch.uint8, pin_memory=True)
    pipe = gbaes.Pipeline(mode=gbaes.PIPE_DIRECT)
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    torch.cuda.synchronize()
    steps = 6
    for i in range(steps):
        s = streams[i % 2]
        s.wait_stream(streams[1 - i % 2])
        with torch.cuda.stream(s):
            gbaes.encrypt_ecb(ks[i % 3], x, x)
            gbaes.ecb_ex(ks[(i + 1) % 3], x, x, kernel=gbaes.KERNEL_BITSLICED)
            gbaes.ecb_ex(ks[(i + 2) % 3], x, x, decrypt=True, kernel=gbaes.KERNEL_BITSLICED)
            rc = lib.aes_ecb_batch_noalloc(ctypes.c_void_p(descs.ctypes.data), 2, ctxs, 3,
                                           ctypes.c_void_p(x.data_ptr()), 16 * n, ctypes.c_void_p(x.data_ptr()), 16 * n,
                                           ctypes.c_void_p(s.cuda_stream))
            assert rc == 0
            h.copy_(x, non_blocking=True)
            pipe.ecb(ks[i % 3], h, h)
            pipe.ecb(ks[(i + 1) % 3], h, h, decrypt=True)
            x.copy_(h, non_blocking=True)
    got = host(x)
    want = data
    for i in range(steps):
        want = oracle.ecb(raw[i % 3], BITS[i % 3], want)
        want = oracle.ecb(raw[(i + 1) % 3], BITS[(i + 1) % 3], want)
        want = oracle.ecb(raw[(i + 2) % 3], BITS[(i + 2) % 3], want, decrypt=True)
        parts = [oracle.ecb(raw[1], 192, want[:16 * cut], decrypt=True)] if cut else []
        want = np.concatenate(parts + [oracle.ecb(raw[2], 256, want[16 * cut:])])
        want = oracle.ecb(raw[i % 3], BITS[i % 3], want)
        want = oracle.ecb(raw[(i + 1) % 3], BITS[(i + 1) % 3], want, decrypt=True)
    assert np.array_equal(got, want)
    assert gbaes.device_status() == 0


@pytest.mark.parametrize("bits", BITS)
@pytest.mark.parametrize("captured", (False, True))
def test_short_calls_in_both_orders(gbaes, bits, captured):
    """A plain launch (a captured call) loads its first blocks before it fills its
    table, an overlapped one after: short calls of every mode, table variant and
    number of fill steps per thread (CTAs of 64 to 1024 threads), at one block, at
    whole and ragged shares of a CTA, and on both sides of the lines by size."""
    rng = np.random.default_rng(2100 + bits)
    key = rng.integers(0, 256, bits // 8, dtype=np.uint8).tobytes()
    iv = rng.integers(0, 256, 16, dtype=np.uint8).tobytes()
    k = gbaes.Key(key)
    s = sms()
    shapes = [(gbaes.KERNEL_TABLE, 0, 0), (gbaes.KERNEL_TABLE_COMPACT, 0, 0)]
    shapes += [(gbaes.KERNEL_TABLE_REPLICATED, t, b) for t, b in ((64, 1), (96, 2), (128, 4), (256, 1), (512, 2), (1024, 4))]
    sizes = (1, 33, 32 * s, 64 * s - 1, 64 * s + 1, 128 * s, 128 * s + 1, 256 * s + 31)
    data = rng.integers(0, 256, 16 * max(sizes), dtype=np.uint8)
    x = dev(data)
    iv_c = (ctypes.c_uint8 * 16)(*iv)
    lib = gbaes.load()
    calls = [(oracle.ecb(key, bits, data, decrypt=d),
              lambda n, y, s, d=d, v=v: lib.aes_ecb_ex(k.handle, int(d), x.data_ptr(), y.data_ptr(), n, *v, s))
             for d in (False, True) for v in shapes]
    calls += [(oracle.ctr(key, bits, iv, data),
               lambda n, y, s: lib.aes_ctr_xcrypt(k.handle, iv_c, 0, 0, x.data_ptr(), y.data_ptr(), n, s)),
              (oracle.cbc_decrypt(key, bits, iv, data),
               lambda n, y, s: lib.aes_cbc_decrypt(k.handle, iv_c, x.data_ptr(), y.data_ptr(), n, s))]
    stream = torch.cuda.Stream()
    outs = [torch.zeros_like(x) for _ in calls]
    torch.cuda.synchronize()
    for n in sizes:
        def go():
            for (_, call), y in zip(calls, outs):
                assert call(n, y, stream.cuda_stream) == 0

        if captured:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=stream):
                go()
            g.replay()
        else:
            go()
        torch.cuda.synchronize()
        for i, ((want, _), y) in enumerate(zip(calls, outs)):
            assert np.array_equal(host(y[:16 * n]), want[:16 * n]), (n, i)
            assert not y[16 * n:].any(), (n, i)
            y.zero_()
    assert gbaes.device_status() == 0
