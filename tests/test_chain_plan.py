"""Which drafters the one-sequence chain kernel takes: the plan of its shared memory, which needs no device."""
import ctypes as C

import pytest

SMS, LIMIT = 148, 227 * 1024


class Phase(C.Structure):
    _fields_ = [("W", C.c_void_p), ("N", C.c_int), ("K", C.c_int)]


class ChainArgs(C.Structure):
    """The head of the launch arguments (hivis_internal.cuh); the plan reads nothing behind it."""
    _fields_ = [("ph", Phase * 6)] + [(n, C.c_int) for n in ("k", "d", "qw", "kvw", "F", "V", "Hq", "Hkv", "dh", "max_len")] + [("rest", C.c_char * 1024)]


def planned_bytes(d, hq, hkv, dh, ffn, vocab, bf16):
    from paper_2509_23928_b200 import lib
    f = lib._Z16chain_smem_bytesRK9ChainArgsii
    f.restype, f.argtypes = C.c_size_t, [C.POINTER(ChainArgs), C.c_int, C.c_int]
    a = ChainArgs()
    shapes = [(d, 2 * d), ((hq + 2 * hkv) * dh, d), (d, hq * dh), (2 * ffn, d), (d, ffn), (vocab, d)]
    for p, (n, k) in enumerate(shapes):
        a.ph[p].N, a.ph[p].K = n, k
    a.dh = dh
    return f(C.byref(a), int(bf16), SMS)


def taken(d, hq, hkv, dh, ffn, vocab, bf16):
    """A ring of 128 KB with its barriers, the longest input vector in fp32 (or what the attention keeps there), a partial sum for every
    chunk of 4 KB of a CTA's rows, and 280 bytes of bookkeeping."""
    es, longest, slots = 2 if bf16 else 4, 0, 0
    for n, k in [(d, 2 * d), ((hq + 2 * hkv) * dh, d), (d, hq * dh), (2 * ffn, d), (d, ffn), (vocab, d)]:
        longest = max(longest, k)
        slots = max(slots, ((n + SMS - 1) // SMS + 2) * ((k * es + 4095) // 4096))
    attn = 4 * (3 * dh + 2 * 16 + 16 * dh + 1)
    up = lambda x, m: (x + m - 1) // m * m
    return 131072 + up(max(4 * longest, attn), 128) + up(4 * slots, 128) + 256 + 280 <= LIMIT


# the widest feed-forward layer that fits beside the dimensions of the two full-size drafters and of one with heads of 64
@pytest.mark.parametrize("bf16,d,hq,hkv,dh,vocab,ffn", [
    (True, 4096, 32, 32, 128, 32000, 24512), (False, 4096, 32, 32, 128, 32000, 23872), (True, 3584, 28, 4, 128, 152064, 23104),
    (False, 3584, 28, 4, 128, 152064, 21056), (True, 1024, 16, 16, 64, 32000, 24832),
])
def test_widest_feed_forward_layer(bf16, d, hq, hkv, dh, vocab, ffn):
    assert 0 < planned_bytes(d, hq, hkv, dh, ffn, vocab, bf16) <= LIMIT
    assert planned_bytes(d, hq, hkv, dh, ffn + 8, vocab, bf16) == 0


@pytest.mark.parametrize("bf16", [True, False])
@pytest.mark.parametrize("d", [256, 1000, 2560, 3584, 4096, 8192])
def test_which_drafters_are_taken(d, bf16):
    heads = max(1, d // 128)
    for vocab in (1024, 32000, 50257, 152064, 300001):
        for ffn in range(8, 26000, 8):
            assert (planned_bytes(d, heads, 1, 128, ffn, vocab, bf16) != 0) == taken(d, heads, 1, 128, ffn, vocab, bf16), (vocab, ffn)
