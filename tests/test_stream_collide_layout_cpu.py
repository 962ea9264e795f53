"""Addresses of the stream-collide kernels, restated for two nodes a thread in
every storage and node bits in place of flag bytes: the reads past a row's end
against the buffers' tail pads, and the staged kernel's bulk copies (planes, node
bits, announced bytes).  The constants are read from the sources, so a change
there is noticed here."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2308_16597_gb300", "csrc")


def const(name, pattern):
    with open(os.path.join(CSRC, name)) as f:
        return int(re.search(pattern, f.read()).group(1))


V = const("lbm_internal.cuh", r"constexpr int kScNodes = (\d+);")
THREADS = const("k_fluid.cu", r"constexpr int kSCThreads = (\d+);")
PAD = const("lbm_api.cu", r"constexpr size_t kDistTailPad = (\d+);")
EX = [0, 1, 0, -1, 0, 1, -1, -1, 1]
EY = [0, 0, 1, 0, -1, 1, 1, -1, -1]
PDX, PDY = EX + EX[:5], EY + EY[:5]


def test_reads_past_the_last_row_fit_the_tail_pad():
    """A warp that starts below the pitch reads its lanes' V-vectors and one
    element right of the last; on the last row of the last plane what lies past
    the pitch must fit the pad, and past the row's start one element at most
    (the previous plane: every plane with e_x = 1 has index p >= 1)."""
    assert V == 2
    for es in (4, 2):
        worst = 0
        for nx in range(4, 2100):
            pitch = (nx + 31) // 32 * 32
            tx = pitch // V
            bx = min((tx + 31) // 32 * 32, THREADS)
            for xw in range(0, (tx + bx - 1) // bx * bx * V, 32 * V):
                if xw < pitch:  # else the warp returns before its first load
                    worst = max(worst, xw + 32 * V + 1 - pitch)
        assert worst == 33 and worst * es <= PAD


def test_vectors_are_aligned():
    """V elements at an even column of rows and planes that are whole multiples
    of 32 and 64 elements; the word pair of a thread's node bits (8 bytes)."""
    for nx in (4, 31, 33, 257, 4000):
        pitch = (nx + 31) // 32 * 32
        ps = (pitch * 5 + 63) // 64 * 64
        bpitch = (pitch // 32 + 7) // 8 * 8
        for es in (4, 2):
            assert pitch * es % (V * es) == 0 and ps * es % (V * es) == 0
        for x in range(0, pitch, V):
            assert x // 32 == (x + V - 1) // 32  # both nodes in one word
            assert ((3 * bpitch + x // 32) * 2) * 4 % 8 == 0


def test_staged_copies_are_aligned_in_bounds_and_announced():
    """16-bit storage, tiles of W = V x threads nodes, H = 16 bytes of elements
    more on the side a plane pulls from, source rows clamped at walls; node bits:
    both parities' words of the whole tile, from rows padded to whole tiles."""
    es, W, H = 2, V * THREADS, 8
    bits_b = W // 32 * 8
    seg_b = (W + 2 * H) * es
    shifted = sum(d != 0 for d in PDX)
    assert bits_b == 64 and bits_b % 16 == 0 and 14 * seg_b % 16 == 0
    for nx in list(range(4, 700, 7)) + [4000, 4001, 2047]:
        for ny in (4, 5, 37):
            pitch = (nx + 31) // 32 * 32
            bpitch = (pitch // 32 + 7) // 8 * 8
            ps = (pitch * ny + 63) // 64 * 64
            a_bytes, bits_bytes = 14 * ps * es + PAD, ny * bpitch * 8
            ntx = (pitch + W - 1) // W
            assert ntx * bits_b <= bpitch * 8  # a row's tiles stay in the row
            for per_y in (0, 1):
                for it in range(ntx * ny):
                    y, cx = divmod(it, ntx)
                    xs, xe = cx * W, min(cx * W + W, pitch)
                    start = (y * bpitch + (xs >> 5)) * 8
                    assert start % 16 == 0 and start + bits_b <= bits_bytes
                    got = bits_b
                    for p in range(14):
                        ys = y - PDY[p]
                        if ys < 0 or ys >= ny:
                            ys = ys % ny if per_y else min(max(ys, 0), ny - 1)
                        lo, hi = xs - (H if PDX[p] == 1 else 0), xe + (H if PDX[p] == -1 else 0)
                        start, size = (p * ps + ys * pitch + lo) * es, (hi - lo) * es
                        assert 0 <= start and start + size <= a_bytes
                        assert start % 16 == 0 and size % 16 == 0
                        dst = (lo - xs + H) * es
                        assert dst % 16 == 0 and 0 <= dst and dst + size <= seg_b
                        got += size
                    # the bytes announced on the stage's barrier
                    assert got == (xe - xs) * 14 * es + bits_b + shifted * 16


def test_a_threads_bits_lie_in_its_tiles_copy():
    """Thread t of a tile reads the word pair t V / 32 of the copy: the word of
    its node x = xs + t V."""
    for xs in (0, 256, 512):
        for t in range(THREADS):
            x = xs + t * V
            assert (t * V >> 5) * 8 + 8 <= V * THREADS // 32 * 8
            assert (xs >> 5) + (t * V >> 5) == x >> 5
