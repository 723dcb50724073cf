"""How the many-steps kernel shares out a lattice, with the functions that it
and the library compile (lbm_multi_plan.h, built here by the C++ compiler)."""
from tests.test_pair_plan import compiled

MAIN = r"""
#include "lbm_multi_plan.h"
#include <cstdio>
#include <vector>
using namespace tlv;
int main()
{
    for (int sms : {4, 148, 152})
        for (int per_sm : {1, 2, 3})
            for (int nx : {1, 31, 32, 33, 64, 65, 97, 129, 225, 249, 1749, 4000})
                for (int ny : {1, 2, 3, 5, 87, 250, 502, 4533}) {
                    const int nseg = (nx + 31) / 32, ntask = ny * nseg;
                    const MultiGrid g = multi_grid(ntask, sms, per_sm);
                    bool once = true, fits = g.warps >= 1 && g.warps <= MULTI_WARPS && g.blocks >= 1 && g.blocks <= per_sm * sms;
                    std::vector<char> seen(ntask, 0);
                    std::vector<int> load(sms, 0);
                    int heaviest = 0, lightest = 1 << 30;
                    const bool twist = per_sm == 2 || multi_twist(nseg, g.warps * g.blocks);
                    for (int t = 0; t < ntask; ++t) {
                        int y = -1, seg = -1;
                        multi_coords(t, nseg, ny, twist, y, seg);
                        once = once && y >= 0 && y < ny && seg >= 0 && seg < nseg && !seen[y * nseg + seg];
                        if (once) seen[y * nseg + seg] = 1;
                    }
                    for (int b = 0; b < g.blocks; ++b) load[b % sms] += g.warps;
                    for (int l : load) heaviest = std::max(heaviest, l), lightest = std::min(lightest, l);
                    std::printf("%d %d %d %d %d %d\n", nx, ny, (int)once, (int)fits, heaviest - lightest, g.warps);
                }
}
"""


def test_every_segment_once(tmp_path):
    """Each row and segment is one task; blocks lie within the resident ones, and
    the SMs' warps differ by one block at most."""
    rows = [tuple(map(int, ln.split())) for ln in compiled(tmp_path, MAIN)().splitlines()]
    assert len(rows) == 3 * 3 * 12 * 8
    for r in rows:
        assert r[2] and r[3], r
        assert r[4] <= r[5], r


SIDES = r"""
#include "lbm_multi_plan.h"
#include <cstdio>
#include <vector>
using namespace tlv;
int main()
{
    int nx, ny, nw;
    while (std::scanf("%d %d %d", &nx, &ny, &nw) == 3) {
        const int nseg = (nx + 31) / 32;
        std::vector<int> sides(nw, 0);
        int most = 0;
        const bool twist = multi_twist(nseg, nw);
        for (int t = 0; t < ny * nseg; ++t) {
            int y, seg;
            multi_coords(t, nseg, ny, twist, y, seg);
            if (seg == 0 || seg == nseg - 1) most = std::max(most, ++sides[t % nw]);
        }
        std::printf("%d\n", most);
    }
}
"""


def test_side_edges_do_not_meet_in_few_warps(tmp_path):
    """Warp counts that are multiples of the segments per row squared: the
    side-edge segments that one warp gets, at most twice an even share, rounded up."""
    cases = [(225, 4533, 2432), (225, 4533, 1216), (249, 250, 1216), (254, 1021, 2432), (480, 2000, 2025),
             (1000, 1000, 2048)]
    out = compiled(tmp_path, SIDES)("".join("%d %d %d\n" % c for c in cases)).split()
    for (nx, ny, nw), most in zip(cases, map(int, out)):
        assert most <= 2 * -(-2 * ny // nw), (nx, ny, nw, most)
