"""The rings of the products, explored on the CPU.

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


def left_waiting(stages, flight, pairs, blocks, held):
    """The loading warp of the stream kernels (stream_loads): lane s owns stage s, block `it` is requested when its stage is free and
    block it - flight has been seen landed; `pairs` pairs of warps take the blocks in turn.  Pair `held` does nothing until all the
    others have come to a stop, then it goes on too.  Returns the pairs that do not come to their end."""
    first = min(flight, blocks)
    nxt = [s + stages if s < first else s for s in range(stages)]
    landed, freed = [int(s < first) for s in range(stages)], [0] * stages              # phases completed per stage
    seen, at = [False] * stages, list(range(pairs))

    def passes(phases, parity):
        return (phases - 1) & 1 == parity

    def turn(active):
        moved, go = False, []
        for s, it in enumerate(nxt):
            if it >= blocks:
                continue
            f = it - flight
            if not seen[s] and passes(landed[f % stages], (f // stages) & 1):
                seen[s] = moved = True
            if seen[s] and (it < stages or passes(freed[s], (it // stages - 1) & 1)):
                go.append(s)
        for s in go:                                            # requested, and landed at once
            landed[s], nxt[s], seen[s], moved = landed[s] + 1, nxt[s] + stages, False, True
        for p in active:
            s = at[p] % stages
            if at[p] < blocks and landed[s] == at[p] // stages + 1:
                freed[s], at[p], moved = freed[s] + 1, at[p] + pairs, True
        return moved

    for active in (set(range(pairs)) - {held}, range(pairs)):
        while turn(active):
            pass
    return [p for p in range(pairs) if at[p] < blocks]


def test_a_flight_of_parts_of_a_lap_can_leave_a_lane_waiting():
    assert all(left_waiting(12, 9, 4, 64, held) for held in range(4))
    assert left_waiting(28, 21, 4, 112, 0) and left_waiting(32, 25, 4, 200, 0)
    assert not left_waiting(12, 8, 4, 64, 0) and not left_waiting(12, 12, 4, 64, 0)


def test_no_lane_of_a_stream_ring_is_left_waiting():
    src = source("sq_gemm_stream.cu")
    rows = run(lines(src, r"^constexpr int SM_.*$") + "\n" + block(src, "struct StreamLayout")
               + block(src, "__host__ __device__ inline StreamLayout stream_layout(") + """
void show(const StreamLayout& L) { printf("%d %d %d\\n", L.stages, L.flight, SM_WARPS / L.wr / 2); }
int main() {
  for (int r = 8; r <= SM_MAX_ROWS; r += 2) {
    show(stream_layout(r, SM_NT * 128, SM_NT * SM_RP8 * 4, false));
    for (int o = 0; o < 2; ++o) show(stream_layout(r, SM_NT * 512, 8 / (r > 32 ? 2 : 1) * SM_PART * 4, o));
  }
}""")
    rings = {tuple(int(v) for v in r) for r in rows}
    assert len(rings) > 10
    for stages, flight, pairs in rings:
        for held in range(pairs):
            assert left_waiting(stages, flight, pairs, 8 * stages, held) == [], (stages, flight, pairs, held)
