"""Hand-over of the TMA-staged step's stages, for every block shape the step launches: a warp
never reads a stage before the copies of its tile have landed, in whatever order tiles land.

The kernel's protocol (mbarriers with a parity each, slices claimed from a shared counter or
taken in turn) is run on the CPU with the shapes that the header compiles.  mbarrier
semantics: a wait for parity P returns once the phase before the current one has parity P."""
import os
import subprocess

import pytest

from paper_2301_07684_gb300 import build as B

SHAPES = ([("float", "FK_SOA", cw) for cw in (8, 16, 20)] + [("float", "FK_PW", cw) for cw in (8, 15, 16, 20)] +
          [("double", "FK_SOA", cw) for cw in (8, 16, 20)] + [("double", "FK_PW", cw) for cw in (8, 15, 16, 20)])


@pytest.fixture(scope="module")
def stages(tmp_path_factory):
    """(slices per tile, stages) of every shape, from the header itself."""
    d = tmp_path_factory.mktemp("tma")
    rows = "\n".join(f'    row<{t}, {fk}, {cw}>();' for t, fk, cw in SHAPES)
    (d / "p.cu").write_text(f"""#include <cstdio>
#include "sfq_step_tma.cuh"
template <typename T, int FK, int CW> void row() {{
    using C = sfq::TmaCfg<T, FK, CW>;
    printf("%d %d\\n", sfq::TmaStage<T, FK, CW>::TILE / (32 * C::PPL), C::NSTAGE);
}}
int main() {{
    using namespace sfq;
{rows}
}}
""")
    exe = os.path.join(d, "p")
    subprocess.run([B.NVCC, *B.ARCH, "-std=c++17", "-I", B.INCLUDE, "-I", B.CSRC, "-o", exe, os.path.join(d, "p.cu")],
                   check=True, capture_output=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()
    return {s: (int(out[2 * k]), int(out[2 * k + 1])) for k, s in enumerate(SHAPES)}


class Bar:
    """An mbarrier: `done` completed phases, `want` arrivals each."""

    def __init__(self, want):
        self.want, self.left, self.done = want, want, 0

    def arrive(self):
        self.left -= 1
        if self.left == 0:
            self.left, self.done = self.want, self.done + 1

    def passed(self, parity):
        return (self.done & 1) != parity


def _run(slices, warps, nstage, claim, ntiles, last):
    """Everything moves as far as it can before tile `last` lands.  Returns the first read of a
    stage that does not hold the reader's tile, or None; every slice has then been read once."""
    full, empty = [Bar(1) for _ in range(nstage)], [Bar(slices) for _ in range(nstage)]
    held = [None] * nstage                               # the tile whose copies have landed in the stage
    issued, flying, counter, turn = 0, [], 0, [0] * warps
    want, read = [None] * warps, set()
    while True:
        moved = False
        if issued < ntiles:
            s = issued % nstage
            if issued < nstage or empty[s].passed((issued // nstage - 1) & 1):
                flying.append(issued)
                held[s] = None
                issued += 1
                moved = True
        for t in [t for t in flying if t != last]:
            flying.remove(t)
            held[t % nstage] = t
            full[t % nstage].arrive()
            moved = True
        for w in range(warps):
            if want[w] is None:
                g = counter if claim else turn[w] * warps + w
                if g // slices >= ntiles:
                    continue
                counter += 1
                turn[w] += 1
                want[w] = g
                moved = True
            t = want[w] // slices
            s = t % nstage
            if full[s].passed((t // nstage) & 1):
                if held[s] != t:
                    return w, t, held[s]
                read.add(want[w])
                want[w] = None
                empty[s].arrive()
                moved = True
        if not moved:
            # one more chance for the tile held back, which lands when nothing else can move
            if not flying:
                break
            t = flying.pop(0)
            held[t % nstage] = t
            full[t % nstage].arrive()
    assert read == set(range(ntiles * slices))
    return None


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "-".join(map(str, s)))
def test_no_warp_reads_a_stage_before_its_tile(stages, shape):
    slices, nstage = stages[shape]
    warps, claim = shape[2], shape[1] == "FK_SOA"
    for ntiles in (1, 2, 3, 4, 7, 12):
        for last in range(-1, ntiles):
            assert _run(slices, warps, nstage, claim, ntiles, last) is None, (ntiles, last)


def test_more_warps_than_slices_need_tiles_in_order():
    """What the shapes must not be: warps to spare run round the ring past a late tile."""
    assert _run(16, 19, 3, True, 12, -1) is None
    assert any(_run(16, 19, 3, True, 12, k) is not None for k in range(12))
