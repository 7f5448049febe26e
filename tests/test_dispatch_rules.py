"""Host-side rules and layouts of the kernels, compiled out of the sources and checked without a GPU."""
import pytest

import csrc_util


def test_weight_only_pair_widths_are_instruction_shapes():
    """The width is the N of a cta_group::2 MMA with M = 256 and A in tensor memory: 32, 64, ... 256."""
    shapes = [(M, N) for M in range(65, 2100, 37) for N in (256, 264, 1024, 4096, 5120, 9480, 11008, 14336, 18944, 32000)]
    widths = csrc_util.wo_pair_widths(shapes)
    assert set(widths) == set(range(64, 257, 32))


def test_rotate_layouts_hold_all_that_the_kernel_writes():
    """The forms with eight warps per accumulator slot swap a maximum per lane, 1024 bytes a slot, 512 bytes behind the
    start of the barrier area; 1024 bytes on top of the layout belong to its alignment."""
    tc = csrc_util.source("sq_rotate_quant_tc.cu")
    rows = csrc_util.run(
        csrc_util.lines(tc, r"^constexpr int k(?:Max|Half)DynSmem.*$") + "\n" + csrc_util.block(tc, "struct RqLayout")
        + csrc_util.block(tc, "__host__ __device__ inline RqLayout rq_layout(") + """
int main() {
  for (int n2 = 64; n2 <= 128; n2 *= 2)
    for (int n1 = 1; n1 <= 128; ++n1)
      for (int few = 0; few < 2; ++few) {
        const RqLayout L = rq_layout(n1, n2, kMaxDynSmem, few);
        const int swap_slots = few ? 1 : (n2 == 128 ? 2 : 0);          // slots of eight warps
        printf("%d %d %d %d %d %d\\n", n1, n2, few, L.off_misc + 512 + 1024 * swap_slots, L.total, L.XS);
      }
}""")
    assert len(rows) == 2 * 128 * 2
    for n1, n2, few, end, total, stages in (map(int, r) for r in rows):
        assert end <= total and total + 1024 <= 227 * 1024 and stages >= 2, (n1, n2, few)


@pytest.mark.parametrize("rows,ncta", [(1, 1), (5, 5), (1300, 1184), (2 ** 31 - 1, 1184), (2 ** 31 - 1, 444), (2 ** 31 - 100, 740)])
def test_warp_level_rotation_counts_its_tokens_beyond_32_bits(rows, ncta):
    """n = 32 fits 2^31 - 1 rows on one GPU; the counts of all blocks add up to the rows, and no block's is negative."""
    code = csrc_util.block(csrc_util.source("sq_rotate_quant_mma.cu"), "__host__ __device__ inline int rm_tokens(")
    got = csrc_util.run(code + """
int main(int, char** v) { for (int c = 0; c < atoi(v[1]); ++c) printf("%d\\n", rm_tokens(c, atoi(v[1]), atoi(v[2]))); }
""", ncta, rows)
    counts = [int(r[0]) for r in got]
    assert counts == [(rows - c + ncta - 1) // ncta for c in range(ncta)] and sum(counts) == rows
