"""The products for up to 8 tokens as a stream of weights (sq_gemm_stream.cu): layouts on the CPU, edges of tiles and rings on the GPU."""
import numpy as np
import pytest

import csrc_util
from gpu_util import Guarded, dev, torch_mod
from oracle import singlequant_oracle as ora


def _layout_code():
    src = csrc_util.source("sq_gemm_stream.cu")
    return (csrc_util.lines(src, r"^constexpr int SM_.*$") + "\n" + csrc_util.block(src, "struct StreamLayout")
            + csrc_util.block(src, "__host__ __device__ inline StreamLayout stream_layout(")
            + csrc_util.block(src, "int stream_blocks("))                # and stream_rows, up to its closing brace


def test_layouts_fit_and_their_rings_can_be_followed():
    """Every warp meets every phase of its stages (the depth is a multiple of the stages worked on side by side), the loads in
    flight are whole laps and no more than there are stages, and ring, sums and barriers lie apart inside a block's shared memory."""
    rows = csrc_util.run(_layout_code() + """
void show(int kind, StreamLayout L, int red) {
  printf("%d %d %d %d %d %d %d %d %d %d %d %d\\n", kind, L.rows, L.wr, L.nb, L.stages, L.flight, L.w_st, L.x_st, L.off_x,
         L.off_red, L.off_bar, L.total - 3 * SM_MAX_STAGES * 8);
}
int main() {
  for (int r = 8; r <= SM_MAX_ROWS; r += 2) {
    show(0, stream_layout(r, SM_NT * 128, SM_NT * SM_RP8 * 4, false), 0);
    for (int o = 0; o < 2; ++o) show(1 + o, stream_layout(r, SM_NT * 512, 8 / (r > 32 ? 2 : 1) * SM_PART * 4, o), 0);
  }
}""")
    assert len(rows) == 61 * 3
    for kind, r, wr, nb, stages, flight, w_st, x_st, off_x, off_red, off_bar, end in (map(int, x) for x in rows):
        lap = 16 // wr // 2
        assert stages >= lap and stages % lap == 0 and stages <= 32 and lap <= flight <= stages and flight % lap == 0, r
        assert nb <= 4 and nb * wr * 16 >= r and off_x == stages * w_st and w_st >= 128 * r
        ring = off_x + stages * x_st
        sums = 8 * 136 * 4 if kind == 0 else (4 if wr == 2 else 8) * 8 * 132 * 4
        assert (off_red == 0 and kind == 2) or off_red >= ring
        assert off_bar >= max(ring, off_red + sums) and off_bar % 8 == 0 and end == off_bar
        assert end + 768 + 1024 <= 227 * 1024
        assert (nb * wr * 16 - r) * 128 <= stages * x_st        # a ragged last block is read past its stage, never past the ring


def test_what_the_stream_kernels_leave_to_the_others():
    """The lines that the measurements beside them draw, both sides of each, on 148 SMs."""
    cases = [(1, 4736, 4096, 1), (1, 4738, 4096, 0), (1, 9472, 4096, 0), (1, 9474, 4096, 1), (1, 8192, 2016, 1), (1, 8192, 2048, 0),
             (1, 8192, 7168, 0), (1, 8192, 7200, 1), (1, 7104, 16416, 0), (1, 7106, 16416, 1), (1, 6144, 16384, 1), (1, 6144, 32800, 1),
             (2, 8192, 3040, 1), (2, 8192, 3072, 0), (2, 8192, 4096, 0), (2, 8192, 4128, 1), (2, 9474, 4096, 1), (2, 6144, 28672, 0),
             (3, 8192, 4096, 1), (3, 1024, 12288, 1), (3, 1024, 12416, 0), (8, 1032, 12416, 1), (8, 8192, 16512, 0), (8, 8200, 16512, 1),
             (8, 8192, 16416, 1), (9, 4096, 4096, 0), (4, 126, 4096, 0), (4, 129, 4096, 0), (4, 4096, 224, 0), (4, 4096, 4112, 0)]
    assert [w4a4 for w4a4, _ in csrc_util.stream_takes([c[:3] for c in cases])] == [bool(c[3]) for c in cases]
    assert [wo for _, wo in csrc_util.stream_takes([(1, 4096, 2048), (1, 3900, 2048), (1, 128, 2080)])] == [True, False, True]


def _rows(rows, M):
    """Channels that make a tile of `rows` on 148 SMs."""
    return (148 - M) * rows


# One and several stages, a ragged last one; the tile heights at which warps are split and blocks are added; several tiles per
# block; ragged last tiles; one token and a full tile of eight.
SHAPES = [(1, 128, 256), (8, 130, 288), (3, 200, 544), (8, 2048, 14336), (5, 4106, 1312)] + [
    (8, _rows(r, 8), 800) for r in (16, 18, 32, 34, 48, 50, 64, 66, 96, 98, 128)] + [(8, _rows(128, 8) + 6, 576), (2, 40002, 288)]
# A ring that wraps with fewer loads in flight than it has stages: one tile per block, two, and two of nearly full height.
SHAPES += [(1, 14336, 4096), (8, 28672, 8192), (8, 32000, 4096)]


@pytest.mark.parametrize("kernel", ["w4a4", "weight-only"])
def test_the_shapes_wrap_their_rings_with_a_limited_flight(kernel):
    """Among the products below: rings that wrap while the loads in flight are limited, with one tile per block and with several."""
    wide = [s for s in SHAPES if s[1] > 74 * 128]                 # more channels than a cluster per two SMs takes: K is not split
    rows = csrc_util.run(_layout_code() + """
int main(int n, char** v) {
  for (int i = 1; i + 2 < n; i += 3) {
    const int M = atoi(v[i]), N = atoi(v[i + 1]), K = atoi(v[i + 2]), blocks = stream_blocks(148, M), rows = stream_rows(N, blocks);
    const int tiles = (N + rows - 1) / rows, waves = (tiles + blocks - 1) / blocks;
    const StreamLayout L = W4A4 ? stream_layout(rows, SM_NT * 128, SM_NT * SM_RP8 * 4, false)
                                : stream_layout(rows, SM_NT * 512, 8 / (rows > 32 ? 2 : 1) * SM_PART * 4, tiles <= blocks);
    printf("%d %d %d %d\\n", waves, waves * ((K + 255) / 256), L.stages, L.flight);
  }
}""".replace("W4A4", "1" if kernel == "w4a4" else "0"), *(v for s in wide for v in s))
    limited = {waves > 1 for waves, blocks, stages, flight in (map(int, r) for r in rows) if blocks > stages > flight}
    assert limited == {False, True}


def _codes(rng, n, K):
    return rng.integers(-8, 8, size=(n, K), dtype=np.int8)


# Beside the lines of stream_yields, on the side of the other kernels.
YIELDED = [(1, 4738, 4096), (1, 9472, 2048), (1, 7104, 16416), (2, 8192, 3072), (2, 4738, 32768), (3, 1024, 12416), (8, 1032, 16512)]
# The last tokens of a batch that the decode kernel begins.
BEGUN = [(65, 1024, 1024), (72, 512, 4096)]


@pytest.mark.gpu
@pytest.mark.parametrize("M,N,K", SHAPES + YIELDED + BEGUN)
def test_w4a4_stream_is_bit_exact(M, N, K):
    from paper_2511_22316_b200 import binding as sq
    rng = np.random.default_rng(M * 131 + N + K)
    Xc, Wc = _codes(rng, M, K), _codes(rng, N, K)
    Xc[0], Wc[0] = -8, -8
    sx, sw = rng.uniform(0.01, 2.0, size=M).astype(np.float16), rng.uniform(0.001, 0.1, size=N).astype(np.float16)
    y, acc = Guarded(M * N * 2), Guarded(M * N * 4)
    sq.sq_w4a4_gemm(dev(ora.pack_int4(Xc)), dev(sx), dev(ora.pack_int4(Wc)), dev(sw), M, N, K, y, acc)
    torch_mod().cuda.synchronize()
    assert sq.sq_last_device_status() == sq.SQ_OK
    y.check(), acc.check()
    want = Xc.astype(np.float64) @ Wc.astype(np.float64).T                   # integers below 2^53
    assert np.array_equal(acc.numpy(np.int32, (M, N)), want.astype(np.int32))
    apart = y.numpy(np.float16, (M, N)).view(np.int16).astype(int) - ora.dequant(want.astype(np.int32), sx, sw).view(np.int16)
    assert np.abs(apart).max() <= 1       # its product with the steps is rounded to fp32 before fp16


# The same, and K over clusters of 2, 4 and 8 (few channels, long K).
@pytest.mark.gpu
@pytest.mark.parametrize("M,N,K", [s for s in SHAPES if s[0] > 1] + [(1, 5128, 4096), (8, 136, 8192), (8, 1024, 8192), (7, 4098, 14336),
                                                                  (8, 8192, 28672), (8, 136, 65536), (3, 2050, 65536)])
def test_weight_only_stream_is_bit_exact_on_integers(M, N, K):
    """Tokens in [-8, 8], steps powers of two: every partial sum is an integer below 2^24, so that any order gives the same."""
    from paper_2511_22316_b200 import binding as sq
    rng = np.random.default_rng(M * 137 + N + K)
    Z, Wc = rng.integers(-8, 9, size=(M, K)).astype(np.float16), _codes(rng, N, K)
    Z[0], Wc[0] = -8, -8
    sw = (2.0 ** rng.integers(-12, -6, size=N)).astype(np.float16)
    y = Guarded(M * N * 2)
    sq.sq_w4a16_gemm(dev(Z), dev(ora.pack_int4_interleaved(Wc)), dev(sw), M, N, K, y)
    torch_mod().cuda.synchronize()
    assert sq.sq_last_device_status() == sq.SQ_OK
    y.check()
    want = (Z.astype(np.float32) @ Wc.astype(np.float32).T) * sw.astype(np.float32)         # exact: see above
    assert np.array_equal(y.numpy(np.float16, (M, N)), want.astype(np.float16))


@pytest.mark.gpu
@pytest.mark.parametrize("M,K", [(1, 14336), (8, 4096), (8, 28672)])
def test_weight_only_stream_stays_within_the_fp32_accumulation_bound(M, K):
    """fp32 sums of K products, each addition off by at most one unit in the last place of a sum bounded by the sum of the
    magnitudes, then one rounding to fp16; the same bits again on a second call.  And few outputs are off the rounded exact value:
    a chain adds K / 128 times (8 shares of K, 16 products at a time), so its error is some sqrt(K / 128) 2^-24 of the sum, and a rounding
    to fp16 (spacing 2^-11 of the value or more) comes out otherwise for a share of twice that over 2^-11, at most."""
    from paper_2511_22316_b200 import binding as sq
    N = 1024
    rng = np.random.default_rng(K + M)
    Z, Wc = rng.standard_normal((M, K)).astype(np.float16), _codes(rng, N, K)
    sw = rng.uniform(0.001, 0.1, size=N).astype(np.float16)
    y, y2 = Guarded(M * N * 2), Guarded(M * N * 2)
    args = (dev(Z), dev(ora.pack_int4_interleaved(Wc)), dev(sw), M, N, K)
    sq.sq_w4a16_gemm(*args, y)
    sq.sq_w4a16_gemm(*args, y2)
    torch_mod().cuda.synchronize()
    got, again = (g.numpy(np.float16, (M, N)) for g in (y, y2))
    assert np.array_equal(got, again)
    z, w, s = Z.astype(np.float64), Wc.astype(np.float64), sw.astype(np.float64)
    want, mag = z @ w.T * s, np.abs(z) @ np.abs(w).T * s
    assert np.all(np.abs(got - want) <= 2.0 ** -10 * np.abs(want) + K * 2.0 ** -23 * mag + 2.0 ** -24)
    assert np.mean(got != want.astype(np.float16)) <= (K / 128) ** 0.5 * 2.0 ** -12 + 4.0 / want.size


@pytest.mark.gpu
@pytest.mark.parametrize("M,N,K", [(3, 130, 288), (8, 1024, 8192), (5, 4106, 1312)])
def test_infinities_and_nan_stay_with_their_token_and_channel(M, N, K):
    """An infinity or NaN among the tokens or in a step spoils its own row or column and no other bit."""
    from paper_2511_22316_b200 import binding as sq
    rng = np.random.default_rng(N + K)
    Z, Wc = rng.standard_normal((M, K)).astype(np.float16), _codes(rng, N, K)
    Xc = _codes(rng, M, K)
    sx, sw = rng.uniform(0.01, 2.0, size=M).astype(np.float16), rng.uniform(0.001, 0.1, size=N).astype(np.float16)
    wq, wi, xq = dev(ora.pack_int4(Wc)), dev(ora.pack_int4_interleaved(Wc)), dev(ora.pack_int4(Xc))

    def both(z, steps_x, steps_w):
        y, yw = Guarded(M * N * 2), Guarded(M * N * 2)
        sq.sq_w4a4_gemm(xq, dev(steps_x), wq, dev(steps_w), M, N, K, y)
        sq.sq_w4a16_gemm(dev(z), wi, dev(steps_w), M, N, K, yw)
        torch_mod().cuda.synchronize()
        assert sq.sq_last_device_status() == sq.SQ_OK
        y.check(), yw.check()
        return y.numpy(np.float16, (M, N)), yw.numpy(np.float16, (M, N))

    clean = both(Z, sx, sw)
    Z[1, K - 1], Z[2, 0], sx[1], sw[N - 1] = np.inf, np.nan, np.inf, np.nan
    spoilt = both(Z, sx, sw)
    rows = [np.arange(M) != 1, (np.arange(M) != 1) & (np.arange(M) != 2)]
    for a, b, keep in zip(clean, spoilt, rows):
        assert np.array_equal(a[keep, :-1], b[keep, :-1]) and np.all(np.isnan(b[:, -1]))
        assert not np.any(np.isfinite(b[~keep]))


@pytest.mark.gpu
@pytest.mark.parametrize("bits", [0, 4])
def test_a_product_right_behind_the_packing_reads_the_new_weights(bits):
    """Queued without a wait, on a buffer that held other weights: the product asks for its first weights ahead of the kernel
    before it, and must not be let go before they are written."""
    from paper_2511_22316_b200 import binding as sq
    torch = torch_mod()
    n1, n2, M, N = 16, 64, 4, 4096
    K = n1 * n2
    rng = np.random.default_rng(bits)
    rot = sq.sq_build_rotation(rng.standard_normal((8, K)).astype(np.float32), n1, n2, seed=1)
    W = [dev(rng.standard_normal((N, K)).astype(np.float16)) for _ in range(2)]
    x = dev(rng.standard_normal((M, K)).astype(np.float16)) if bits else dev(ora.pack_int4(_codes(rng, M, K)))
    sx = dev(np.ones(M, np.float16))
    Wq, sw = torch.empty(N * K // 2, dtype=torch.uint8, device="cuda"), torch.empty(N, dtype=torch.float16, device="cuda")
    y = [torch.empty(M, N, dtype=torch.float16, device="cuda") for _ in range(4)]

    def pack(w):
        if bits:
            sq.sq_pack_weight_wo(rot, w, N, K, bits, Wq, sw)
        else:
            sq.sq_pack_weight(rot, w, N, K, Wq, sw)

    def product(out):
        if bits:
            sq.sq_w4a16_gemm(x, Wq, sw, M, N, K, out)
        else:
            sq.sq_w4a4_gemm(x, sx, Wq, sw, M, N, K, out)

    for w, out in zip(W, y):                       # with a wait
        pack(w)
        torch.cuda.synchronize()
        product(out)
        torch.cuda.synchronize()
    assert not torch.equal(y[0], y[1])
    for turn in range(20):                         # without
        for w, out in zip(W, y[2:]):
            pack(w)
            product(out)
        torch.cuda.synchronize()
        assert sq.sq_last_device_status() == sq.SQ_OK
        assert torch.equal(y[0], y[2]) and torch.equal(y[1], y[3]), turn
    rot.close()


@pytest.mark.gpu
def test_grouped_experts_of_few_rows_with_ragged_channels():
    """K % 128 != 0: experts one by one, their steps and outputs at odd rows.  Same bits as expert by expert on its own."""
    from paper_2511_22316_b200 import binding as sq
    torch = torch_mod()
    n1, n2, N = 33, 32, 136
    K, offsets = n1 * n2, [0, 3, 4, 4, 9, 17]
    M, E = offsets[-1], len(offsets) - 1
    rng = np.random.default_rng(7)
    X = dev(rng.standard_normal((M, K)).astype(np.float16))
    rot = sq.sq_build_rotation(rng.standard_normal((8, K)).astype(np.float32), n1, n2, seed=1)
    Wq = [dev(ora.pack_int4(_codes(rng, N, K))) for _ in range(E)]
    sw = [dev(rng.uniform(0.001, 0.1, size=N).astype(np.float16)) for _ in range(E)]
    nbytes = sq.sq_linear_workspace_bytes(M, K)
    ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    y, one = Guarded(M * N * 2), Guarded(M * N * 2)
    sq.sq_linear_grouped([rot] * E, offsets, X, Wq, sw, N, K, ws, nbytes, y)
    out = one.view.view(torch.float16).view(M, N)
    for e in range(E):
        r0, r1 = offsets[e], offsets[e + 1]
        if r1 > r0:
            sq.sq_linear(rot, X[r0:r1], r1 - r0, Wq[e], sw[e], N, K, ws, nbytes, out[r0:r1])
    torch.cuda.synchronize()
    assert sq.sq_last_device_status() == sq.SQ_OK
    y.check(), one.check()
    assert np.array_equal(y.numpy(np.uint16, (M, N)), one.numpy(np.uint16, (M, N)))
    rot.close()
