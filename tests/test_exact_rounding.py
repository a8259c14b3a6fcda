"""The exact decisions of the Hadamard encoder that replace divisions, on the CPU.

A code is rint(fl(d / s)) with an fp16 scale s and an fp32 difference d. Near a half-integer B the
encoder compares d with the product B s, which is exact in fp32, instead of dividing: d > B s means
the rounded quotient lies above B, d < B s below, equality is the tie. Checked for every B of 8-bit
codes, scales over the fp16 range (its subnormals and the values at the ends of a binade among
them) and the fp32 neighbours of B s. Likewise a scale is fp16(fl(d / qmax)), decided by comparing
the range d with M qmax at the midpoint M of two neighbouring fp16 values: every such pair, every
code width.
"""
import numpy as np


def test_side_of_half_integer():
    rng = np.random.default_rng(3)
    bits = np.concatenate([np.arange(1, 64), np.arange(0x03F0, 0x0410), 0x0400 * np.arange(1, 31), 0x0400 * np.arange(1, 31) + 0x3FF,
                           rng.integers(1, 0x7C00, 400)]).astype(np.uint16)
    s = np.unique(bits).view(np.float16).astype(np.float32)[:, None]
    B = (np.arange(0, 256, dtype=np.float32) + np.float32(0.5))[None, :]
    p = s * B
    np.testing.assert_array_equal(p.astype(np.float64), s.astype(np.float64) * B.astype(np.float64))
    np.testing.assert_array_equal((p / s), np.broadcast_to(B, p.shape))
    for k in range(1, 4):
        up, dn = p, p
        for _ in range(k):
            up, dn = np.nextafter(up, np.float32(np.inf)), np.nextafter(dn, np.float32(-np.inf))
        assert ((up / s) > B).all()
        assert ((dn / s) < B).all()


def test_side_of_scale_midpoint():
    h = np.arange(0, 0x7C00, dtype=np.uint16).view(np.float16).astype(np.float32)
    M = np.append((h[:-1] + h[1:]) * np.float32(0.5), np.float32(65520.0))[None, :]
    q = np.array([3, 7, 15, 63, 255], np.float32)[:, None]
    p = M * q
    np.testing.assert_array_equal(p.astype(np.float64), M.astype(np.float64) * q.astype(np.float64))
    np.testing.assert_array_equal(p / q, np.broadcast_to(M, p.shape))
    for k in range(1, 4):
        up, dn = p, p
        for _ in range(k):
            up, dn = np.nextafter(up, np.float32(np.inf)), np.nextafter(dn, np.float32(-np.inf))
        assert ((up / q) > M).all()
        assert ((dn / q) < M).all()
