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


def test_no_kernel_can_take_the_tensor_memory_that_its_predecessor_still_needs():
    """A kernel launched as a programmatic dependent may come up beside a block of its predecessor that has not allocated its
    tensor memory yet, take what that block needs, and then wait for it for good.  So any two kernels in a row, one of them
    a rotation, either do not fit the SM's 228 KB together or need no more than the 512 columns."""
    tc, pair_rot, dec, pair, wo, gemm = (csrc_util.source(f) for f in (
        "sq_rotate_quant_tc.cu", "sq_rotate_quant_pair.cu", "sq_gemm_decode.cu", "sq_gemm_pair.cu", "sq_gemm_wo.cu", "sq_gemm.cu"))
    rows = csrc_util.run(
        csrc_util.lines(tc, r"^constexpr int k(?:Max|Half)DynSmem.*$") + "\n" + csrc_util.block(tc, "struct RqLayout")
        + csrc_util.block(tc, "__host__ __device__ inline RqLayout rq_layout(") + "\n"
        + csrc_util.lines(tc, r"^constexpr int kAloneSmem.*$|^inline int rq_smem.*$") + "\n"
        + csrc_util.block(pair_rot, "struct RqPairLayout") + csrc_util.block(pair_rot, "__host__ __device__ inline RqPairLayout") + "\n"
        + csrc_util.block(pair, "template <int S_OP_, int S_ST_") + csrc_util.lines(pair, r"^using Pair\w+ = .*$") + "\n"
        + csrc_util.lines(dec, r"^constexpr int D_.*$") + "\n" + csrc_util.block(dec, "template <int NT>\nstruct DecSmem") + "\n"
        + csrc_util.lines(wo, r"^constexpr int (?:WO_|WOD_|WP_).*$") + "\n"
        + csrc_util.block(wo, "template <int NT, int ST, int SS>\nstruct WoDecSmem") + csrc_util.block(wo, "template <int SS>\nstruct WoPairSmem")
        + "\nconstexpr int BM = 128;\n" + csrc_util.block(gemm, "template <int BN, int S_OP, int S_ST>\nstruct GemmSmem") + """
int main() {
  printf("gemm %d 512\\ngemm %d 512\\n", PairWide::DYN_BYTES, PairNarrow::DYN_BYTES);
  printf("gemm %d 512\\ngemm %d 512\\ngemm %d 512\\n", DecSmem<16>::DYN_BYTES, DecSmem<32>::DYN_BYTES, DecSmem<64>::DYN_BYTES);
  printf("gemm %d 512\\ngemm %d 512\\n", WoDecSmem<16, 4, 8>::DYN_BYTES, WoDecSmem<32, 4, 8>::DYN_BYTES);
  printf("gemm %d 512\\ngemm %d 512\\n", WoDecSmem<64, 3, 6>::DYN_BYTES, WoDecSmem<128, 2, 4>::DYN_BYTES);
  printf("gemm %d 512\\ngemm %d 256\\n", WoPairSmem<4>::DYN_BYTES, GemmSmem<128, 3, 3>::DYN_BYTES);
  for (int n2 = 64; n2 <= 128; n2 *= 2) {
    for (int n1 = 1; n1 <= 128; ++n1) {
      const RqLayout few = rq_layout(n1, n2, kMaxDynSmem, true), half = rq_layout(n1, n2, kHalfDynSmem);
      printf("rotate %d %d\\nrotate %d %d\\n", rq_smem(few, 1), 2 * n2, rq_smem(few, 2), 2 * n2);      // codes, fp16 rows
      if (n2 == 64 && half.XS >= 2) printf("rotate %d 256\\n", rq_smem(half, 2));
      else printf("rotate %d 512\\n", rq_smem(rq_layout(n1, n2), 1));
    }
    for (int n1 = 129; n1 <= 256; ++n1) printf("rotate %d 512\\n", rq_pair_layout(n1, n2).total + 1024);
  }
}""")
    forms = {(r[0], int(r[1]), int(r[2])) for r in rows}
    rotations = [f for f in forms if f[0] == "rotate"]
    assert len(rotations) > 20 and len(forms) > len(rotations) + 5
    for kind, smem, columns in forms:
        for _, smem_2, columns_2 in rotations:
            assert smem + smem_2 + 2 * 1024 > 228 * 1024 or columns + columns_2 <= 512, (kind, smem, columns, smem_2, columns_2)
