"""The corner a tracer interpolates from lies inside its leaf's padded block wherever
the tracer is: unchanged for one inside its leaf, the outermost cells else."""
import ctypes


def test_corner_stays_inside_the_block():
    from paper_1810_01319_gb300 import build
    hc = ctypes.CDLL(build.build_hostcheck())
    g = 4
    for n in (8, 16, 32):
        N = n + 2 * g
        for v in range(-1, n):                               # cells of the leaf and half a cell around
            assert hc.cello_hc_corner_index(v, g, N) == v + g
        for v in (-2**31, 2**31 - 1, -2**31 + 3, 2**31 - 4, -g - 1, -g, N - g - 2, N - g - 1, N):
            i = hc.cello_hc_corner_index(v, g, N)
            assert 0 <= i <= N - 2 and i == min(max(v + g, 0), N - 2)
