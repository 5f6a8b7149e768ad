"""Host check of the N = 2048 exchange that trades two bits through TMEM and one
by shuffles (tx11s in ols_fft_passes.cuh), with the shape layouts and helpers of
test_tmem_exchange_maps: the register assignment of the kernel, restated, must
end in the pass-2 layout, and the relabelled shared exchange must be a
bijection without bank conflicts."""
from .test_tmem_exchange_maps import L32, L256, Tmem, bits, final_check, pos

LANES, REGS = (2, 7, 8, 0, 1), (3, 4, 5, 6)      # pass 1


def test_n2048_one_round_trip_and_shuffles():
    m = Tmem()
    x1 = [[[(pos(LANES, REGS, T, k), e) for e in (0, 1)] for k in range(16)] for T in range(32)]
    for T in range(32):
        odd, v = T & 1, [None] * 32
        for i in range(8):
            o = 2 * ((i >> 1) + 8 * (i & 1))
            for e in (0, 1):
                c, d = x1[T][i][e], x1[T][i + 8][e]
                r = x1[T ^ 1][i][e] if (T ^ 1) & 1 else x1[T ^ 1][i + 8][e]
                v[o + e] = r if odd else c
                v[o + 8 + e] = d if odd else r
        m.st(L32, T, v)
    x = [[[None, None] for _ in range(16)] for _ in range(32)]
    for T in range(32):
        w = [m.ld(L256, T, 16, lb=16 * h) for h in range(2)]
        for k in range(16):
            p0, p1, _, _ = bits(k, 4)
            p23 = k >> 2
            x[T][k] = [w[p1][4 * p23 + 2 * p0], w[p1][4 * p23 + 2 * p0 + 1]]
    final_check(x)


def test_n2048_relabelled_shared_exchange():
    def A(q):
        return (q & 127) + 130 * ((q >> 7) & 1) + 264 * ((q >> 8) & 1) + 528 * (q >> 9)

    def pos1(t, k):
        return pos(LANES, REGS, t & 31, k) | ((t >> 5) << 9)

    assert len({A(q) for q in range(2048)}) == 2048 and max(A(q) for q in range(2048)) < 2048 + 128
    for t in range(128):
        for k in range(16):
            assert t + 130 * (k & 1) + 264 * ((k >> 1) & 1) + 528 * (k >> 2) == A(t + 128 * k)
            a1 = (((t >> 3) & 3) + 4 * (t & 1) + 130 * ((t >> 1) & 1) + 264 * ((t >> 2) & 1) + 528 * (t >> 5) + 8 * k)
            assert a1 == A(pos1(t, k))
        assert ((t >> 3) & 3) + 4 * (t & 1) == pos1(t, 0) % 8          # twiddle index
    for h in range(8):
        for k in range(16):
            ts = range(16 * h, 16 * h + 16)
            assert len({A(pos1(t, k)) % 16 for t in ts}) == 16 and len({A(t + 128 * k) % 16 for t in ts}) == 16
