"""The rings of the W4A4 products, explored on the CPU.

Two groups of converter warps take the blocks of a ring in turn and tell the phases of a stage apart by their parity
(mbarrier.try_wait.parity).  Loads that are in flight together may land in any order.  The model below walks every
interleaving of loads, groups and MMAs for a ring of given depth and reports whether a group can be let through to a
block whose load has not landed.  The depths are taken out of the sources by compiling the kernels' layout structs.
"""
import pytest

from csrc_util import block, lines, run, source


def let_through_too_early(stages, op_stages, groups, operand_first=False, blocks=None):
    """The first (block, blocks landed) at which a group passes its wait for a load that is still in flight, else None.
    `operand_first`: the group waits for its operand stage before the load, else after it.

    State: loads issued, the set of loads landed, each group's next block and whether it holds that block's stage, MMAs
    retired.  A stage's barrier has completed as many phases as loads of it have landed; a wait for parity p passes when
    the last completed phase has parity p (none completed: parity 1)."""
    blocks = blocks or 2 * stages + 2
    start = (0, frozenset(), tuple((g, False) for g in range(groups)), 0)
    seen, todo = {start}, [start]

    def landed_of(landed, s):
        return sum(1 for it in landed if it % stages == s)

    def done(state_groups, it):                        # block `it` has been converted
        nxt, _ = state_groups[it % groups]
        return nxt > it

    while todo:
        issued, landed, grp, mma = state = todo.pop()
        nxt = []
        if issued < blocks and (issued < stages or done(grp, issued - stages)):
            nxt.append((issued + 1, landed, grp, mma))
        for it in range(issued):
            # the loads of one stage follow one another; those of different stages land in any order
            if it not in landed and (it < stages or it - stages in landed):
                nxt.append((issued, landed | {it}, grp, mma))
        for g, (it, held) in enumerate(grp):
            if it >= blocks:
                continue
            if not held:                                # full[it % stages], parity (it / stages) & 1
                if operand_first and it >= op_stages and mma <= it - op_stages:
                    continue
                phases = landed_of(landed, it % stages)
                if (phases - 1) & 1 == (it // stages) & 1:
                    if it not in landed:
                        return it, sorted(landed)
                    nxt.append((issued, landed, grp[:g] + ((it, True),) + grp[g + 1:], mma))
            elif it < op_stages or mma > it - op_stages:  # empty[it % op_stages]: the MMAs of block it - op_stages
                nxt.append((issued, landed, grp[:g] + ((it + groups, False),) + grp[g + 1:], mma))
        if mma < blocks and done(grp, mma):
            nxt.append((issued, landed, grp, mma + 1))
        for s in nxt:
            if s not in seen:
                seen.add(s)
                todo.append(s)
    return None


def test_the_model_tells_sound_rings_from_unsound_ones():
    assert let_through_too_early(5, 4, 2) is not None         # a group meets every other phase of a stage
    assert let_through_too_early(3, 2, 2) is not None
    assert let_through_too_early(3, 4, 2, operand_first=True) is not None
    assert let_through_too_early(5, 4, 2, operand_first=True) is None
    assert let_through_too_early(4, 4, 2) is None
    assert let_through_too_early(3, 3, 1) is None


@pytest.fixture(scope="module")
def rings():
    pair, dec = source("sq_gemm_pair.cu"), source("sq_gemm_decode.cu")
    rows = run(block(pair, "template <int S_OP_, int S_ST_") + lines(pair, r"^using Pair\w+ = .*$") + "\n"
               + lines(dec, r"^constexpr int D_.*$") + "\n" + block(dec, "template <int NT>\nstruct DecSmem") + """
template <class P> void pair(const char* n) { printf("%s %d %d %d 0\\n", n, P::S_ST, P::S_OP, P::GROUPS); }
template <int NT> void dec() {
  using L = DecSmem<NT>;
  printf("decode_w%d %d %d %d %d\\n", NT, L::S_W, L::S_OP, D_CONV_GROUPS, L::OPERAND_FIRST);
  printf("decode_x%d %d %d %d 1\\n", NT, L::S_X, L::S_OP, D_CONV_GROUPS);      // its two waits cost nothing in this order
}
int main() { pair<PairWide>("wide"); pair<PairNarrow>("narrow"); dec<16>(); dec<32>(); dec<64>(); }
""")
    return {row[0]: tuple(int(v) for v in row[1:]) for row in rows}


@pytest.mark.parametrize("name", ["wide", "narrow", "decode_w16", "decode_x16", "decode_w32", "decode_x32", "decode_w64",
                                  "decode_x64"])
def test_no_group_is_let_through_before_its_load_has_landed(rings, name):
    stages, op_stages, groups, operand_first = rings[name]
    assert let_through_too_early(stages, op_stages, groups, bool(operand_first)) is None
