"""The barriers that W1's 8-bit codes land on in the leaf kernel's ring: no role passes a wait before what it waits for, in whatever
order the copies land and the roles run (no GPU work).

LeafCodeRing, compiled for the host, says for every visit of the ring which stage, barrier, phase and expanding warp it has.  A model of
the roles around it (gather warp, copy engine, two expanding warps, MMA issuer) is run through all its interleavings."""
import os
import re
import subprocess

import pytest

from paper_2308_14711_b200 import build

VISITS = 14
PROGRAM = r"""
#include <cstdio>
#include "kernels/leaf_umma.cuh"
template <int LP> void stages() {
    using L = fff::LeafUmmaLayout<LP, true>;
    std::printf("stages %d %d %d\n", LP, L::smem_bytes(0), L::kStageBytes);
}
int main() {
    stages<16>(); stages<32>(); stages<64>();
    for (int n = 2; n <= fff::kLUMaxStages; ++n) {
        fff::LeafCodeRing r(n);
        for (int v = 0; v < VISITS; ++v, r.next()) std::printf("visit %d %d %d %d %u\n", n, r.stage(), r.at, r.owner(), r.phase);
    }
}
""".replace("VISITS", str(VISITS))


@pytest.fixture(scope="module")
def rings(tmp_path_factory):
    """Visits of rings of 2 to 8 stages, as (stage, barrier, owner, phase), and the stages that each padded width runs with."""
    d = tmp_path_factory.mktemp("code_ring")
    (d / "ring.cu").write_text(PROGRAM)
    subprocess.check_call([build.NVCC, "-std=c++17", "--expt-relaxed-constexpr", "-gencode", "arch=compute_100a,code=sm_100a",
                           "-I", build.CSRC, "-o", str(d / "ring"), str(d / "ring.cu")])
    lines = [line.split() for line in subprocess.check_output([str(d / "ring")], text=True).splitlines()]
    api = open(os.path.join(build.CSRC, "fff_api.cu")).read()
    budget = eval(re.search(r"constexpr int kSmemBudget = ([0-9 *-]+);", api).group(1))
    stages = {int(lp): min(8, (budget - int(fixed)) // int(stage)) for key, lp, fixed, stage in (l for l in lines if l[0] == "stages")}
    visits = {}
    for line in lines:
        if line[0] == "visit":
            visits.setdefault(int(line[1]), []).append(tuple(int(v) for v in line[2:]))
    return visits, stages


def first_fault(n_stages, visits):
    """None, or what goes wrong first.  A barrier is the number of its phases that have ended; waiting for parity p passes unless p is
    that number's, as the hardware has it."""
    n = len(visits)
    n_codes = 1 + max(v[1] for v in visits)
    turns = [[v for v in range(n) if visits[v][2] == w] for w in (0, 1)]
    passed = lambda ended, parity: ended % 2 != parity
    # state: visits gathered, set in flight, turns taken per warp, MMAs done, ended phases of the codes', full and empty barriers
    start = (0, frozenset(), (0, 0), 0, (0,) * n_codes, (0,) * n_stages, (0,) * n_stages)
    seen, todo = {start}, [start]
    up = lambda t, i: t[:i] + (t[i] + 1,) + t[i + 1:]
    while todo:
        sent, flying, taken, done, codes, full, empty = todo.pop()
        steps = []
        if sent < n and passed(empty[sent % n_stages], (sent // n_stages) % 2 ^ 1):
            if sent - n_stages >= done:
                return f"visit {sent} is gathered over visit {sent - n_stages}"
            steps.append((sent + 1, flying | {sent}, taken, done, codes, full, empty))
        for v in flying:
            steps.append((sent, flying - {v}, taken, done, up(codes, visits[v][1]), full, empty))
        for w in (0, 1):
            if taken[w] == len(turns[w]):
                continue
            v = turns[w][taken[w]]
            stage, barrier, _, phase = visits[v]
            if passed(codes[barrier], phase):
                if v >= sent or v in flying:
                    return f"visit {v} is expanded before its codes have landed"
                steps.append((sent, flying, up(taken, w), done, codes, up(full, stage), empty))
        if done < n and passed(full[done % n_stages], (done // n_stages) % 2):
            w = visits[done][2]
            if turns[w].index(done) >= taken[w]:
                return f"visit {done} is multiplied before it is expanded"
            steps.append((sent, flying, taken, done + 1, codes, full, up(empty, done % n_stages)))
        if not steps and done < n:
            return "all roles wait"
        for s in steps:
            if s not in seen:
                seen.add(s)
                todo.append(s)
    return None


@pytest.mark.parametrize("LP", [16, 32, 64])
def test_no_wait_passes_early(rings, LP):
    visits, stages = rings
    n = stages[LP]
    assert n >= 2
    ring = visits[n]
    assert [v[0] for v in ring] == [v % n for v in range(VISITS)] and [v[2] for v in ring] == [v % 2 for v in range(VISITS)]
    assert first_fault(n, ring) is None


@pytest.mark.parametrize("n", range(2, 6))
def test_a_barrier_per_stage_would_not_do_for_odd_rings(rings, n):
    """The model sees the fault that the second barrier is for."""
    shared = [(v % n, v % n, v % 2, v // n % 2) for v in range(VISITS)]
    assert first_fault(n, rings[0][n]) is None
    assert (first_fault(n, shared) is None) == (n % 2 == 0)
