"""The layout of a batch in the cluster kernel (plan_groups, csrc/host.h), without
a GPU: a small program made with the library's own header prints the groups of
given batches on a device of 152 SMs that holds 76, 36 and 15 clusters of 2, 4
and 8 CTAs."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "host.h"
using namespace hac;
using namespace hac::host;
// stdin: one batch a line: ants_per_warp cluster_log2 {count n m k local_search}...
// with arguments count and step_apw: the autotuner's candidates instead
int main(int argc, char **argv)
{
    if (argc == 3) {
        for (const hac_exec &e : tune_candidates(std::atoi(argv[1]), std::atoi(argv[2])))
            std::printf("%d,%d,%d,%d,%d,%d,%d,%d ", e.ants_per_warp, e.warps_per_block, e.use_graph, e.fused,
                        e.fallback_list, e.profile, e.cluster_log2, e.parts);
        return 0;
    }
    char line[4096];
    while (std::fgets(line, sizeof line, stdin)) {
        int apw, clog, used, off = 0, c, n, m, k, ls;
        if (std::sscanf(line, "%d %d%n", &apw, &clog, &off) != 2) continue;
        std::vector<Sizes> zs;
        while (std::sscanf(line + off, "%d %d %d %d %d%n", &c, &n, &m, &k, &ls, &used) == 5) {
            Sizes z{};
            z.n = n; z.m = m; z.kp = 4 * ((k + 3) / 4); z.k_eff = k; z.iters = 10; z.ls = ls;
            zs.insert(zs.end(), c, z);
            off += used;
        }
        std::vector<int> mem(zs.size());
        for (size_t q = 0; q < mem.size(); ++q) mem[q] = (int)q;
        std::vector<FusedGroup> g;
        std::vector<int32_t> order;
        const int st = plan_groups(zs, mem, apw, clog, 32, DeviceShape(), g, order);
        std::printf("%d", st);
        for (const FusedGroup &G : g)
            std::printf(" %d,%d,%d,%d,%d,%zu", G.count, G.clog, G.apw, G.warps, G.block_warps,
                        fused_smem_bytes(G.rows_cap, G.kp_cap, G.warps, G.apw, G.stride, G.xy_cap, G.list_rows));
        std::printf("\n");
    }
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    """plan(apw, clog, [(count, n, m, k, ls), ...]) -> status, [(count, clog, apw, warps, block_warps, smem), ...]"""
    from paper_2601_19041_gb300 import build as B
    cc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(cc):
        pytest.skip("no nvcc")
    lib = B.build()
    d = tmp_path_factory.mktemp("plan")
    src, exe = d / "plan.cu", d / "plan"
    src.write_text(PROGRAM)
    subprocess.run([cc, *B.ARCH, "-O1", "-std=c++17", "--expt-relaxed-constexpr", "-I", os.path.join(ROOT, "include"),
                    "-I", B.CSRC, str(src), "-o", str(exe), lib, "-Xlinker", f"-rpath={os.path.dirname(lib)}"], check=True)

    def call(apw, clog, parts=None):
        if parts is None:      # the autotuner's candidates for apw instances, clog ants per warp if left open
            out = subprocess.run([str(exe), str(apw), str(clog)], capture_output=True, text=True, check=True).stdout
            return [tuple(int(v) for v in c.split(",")) for c in out.split()]
        text = " ".join(map(str, [apw, clog] + [x for p in parts for x in p])) + "\n"
        out = subprocess.run([str(exe)], input=text, capture_output=True, text=True, check=True).stdout.split()
        return int(out[0]), [tuple(int(v) for v in g.split(",")) for g in out[1:]]
    return call


# An SM holds 16 warps of the cluster kernel and 228 KB of shared memory.
@pytest.mark.parametrize("apw,clog,parts,block", [
    (0, 0, [(128, 500, 32, 20, 0)], 16),                             # an SM each
    (0, 0, [(256, 500, 32, 20, 0)], 8),                              # two share an SM
    (0, 0, [(256, 1000, 64, 20, 0)], 16),                            # too large to share one
    (0, 0, [(100, 500, 32, 20, 0), (100, 500, 32, 20, 1)], 8),       # two groups side by side
    (0, 1, [(76, 500, 32, 20, 0)], 16),
    (0, 2, [(36, 1000, 64, 20, 0)], 16),
    (0, 3, [(16, 1000, 64, 20, 0)], 8),                              # 15 clusters of 8 fit
    (2, 3, [(128, 500, 32, 20, 0)], 4),
    (0, 0, [(1000, 12, 4, 8, 0)], 2),                                # seven share an SM
    (0, 0, [(3000, 40, 10, 8, 0)], 1),
    (16, 0, [(600, 30, 8, 8, 0)], 4),
    (32, 0, [(100, 500, 32, 20, 1)], 16),
])
def test_block_width(plan, apw, clog, parts, block):
    st, groups = plan(apw, clog, parts)
    assert st == 0 and sum(g[0] for g in groups) == sum(p[0] for p in parts)
    for count, cl, a, warps, bw, smem in groups:
        assert bw == max(block, warps), groups
        assert smem <= 226 * 1024


# On a cluster, as few ants per warp (2, 4, 8) as leave at most 8 warps on an SM.
@pytest.mark.parametrize("clog,part,apw", [
    (3, (8, 1000, 64, 20, 0), 2),        # 8 ants per CTA
    (2, (32, 1000, 64, 20, 0), 2),       # 16
    (1, (32, 1000, 64, 20, 0), 4),       # 32
    (1, (60, 1000, 128, 20, 0), 8),      # 64
    (1, (128, 1000, 64, 20, 0), 8),      # 32, two CTAs to an SM
    (0, (32, 6000, 32, 10, 0), 2),       # too large for one SM: 2 CTAs
    (0, (128, 4000, 64, 20, 0), 2),      # 4 CTAs, room for one on an SM
    (0, (128, 2000, 64, 20, 0), 4),      # 2 CTAs
    (0, (128, 1000, 64, 20, 0), 8),      # one SM
])
def test_ants_per_warp_on_clusters(plan, clog, part, apw):
    st, groups = plan(0, clog, [part])
    assert st == 0 and [(g[0], g[2]) for g in groups] == [(part[0], apw)], groups


# More than 64 ants on one SM, or more than 32 on a CTA of a cluster: the largest
# cluster of which all fit on the device at once.
@pytest.mark.parametrize("parts,clogs", [
    ([(15, 500, 128, 20, 0)], [3]), ([(16, 500, 128, 20, 0)], [2]), ([(36, 500, 65, 20, 0)], [2]),
    ([(37, 500, 65, 20, 0)], [1]), ([(76, 500, 65, 20, 0)], [1]), ([(77, 500, 65, 20, 0)], [0]),
    ([(1, 500, 64, 20, 0)], [0]), ([(1, 500, 1000, 20, 0)], [3]), ([(1, 500, 256, 20, 0)], [3]),
    ([(32, 2000, 64, 20, 0)], [1]), ([(32, 2000, 65, 20, 0)], [2]), ([(37, 2000, 128, 20, 0)], [1]),
    ([(10, 500, 100, 20, 0), (80, 500, 32, 20, 0)], [0, 2]), ([(10, 500, 100, 20, 0), (140, 500, 32, 20, 0)], [0]),
])
def test_crowded_instances_spread_over_idle_sms(plan, parts, clogs):
    st, groups = plan(0, 0, parts)
    assert st == 0 and sorted(set(g[1] for g in groups)) == clogs, groups


# The tuner times what a per-step call with the layout left open runs, and only
# layouts that a batch accepts.
@pytest.mark.parametrize("count,step_apw", [(1, 1), (3, 2), (4, 4), (60, 3), (100, 6), (500, 8)])
def test_autotuner_candidates(plan, count, step_apw):
    cands = plan(count, step_apw)
    assert len(set(cands)) == len(cands)
    for parts in (1, 4):
        mine = [c for c in cands if not c[3] and c[7] == parts]
        if parts > count:
            assert not mine
            continue
        assert (0, 0, 1, 0, 32, 0, 0, parts) in mine
        for wpb in (4, 8):
            assert ((0, wpb, 1, 0, 32, 0, 0, parts) in mine) == (step_apw not in (1, 2, 4))
    for apw, wpb, graph, fused, fbl, prof, clog, parts in cands:
        assert apw in (0, 1, 2, 4, 16, 32) and 0 <= wpb <= 8 and graph == 1 and fbl in (0, 32) and prof == 0
        assert fused == 0 or (apw != 1 and 0 <= clog <= 3)


def test_members_that_do_not_fit_together_are_placed_one_by_one(plan):
    # spread over clusters of 8, the ten with many ants would share a group with
    # the one whose table takes a CTA's shared memory: masks of both do not fit
    st, groups = plan(0, 0, [(1, 14000, 64, 20, 0), (10, 500, 128, 20, 0)])
    assert st == 0 and sorted((g[0], g[1], g[2]) for g in groups) == [(1, 3, 8), (10, 0, 8)], groups
    st, groups = plan(0, 0, [(1, 14000, 64, 20, 0)])
    assert st == 0 and [(g[0], g[1], g[2]) for g in groups] == [(1, 3, 2)], groups
    st, groups = plan(0, 0, [(1, 60000, 64, 20, 0)])
    assert st != 0 and not groups


# What fits in some layout of its own is taken by the open layout, alone and in a
# batch, and every group stays inside the limits of a block.
@pytest.mark.parametrize("n", [3, 40, 1000, 1700, 5000, 9000, 13000])
def test_open_layout_takes_what_fits(plan, n):
    for m in (1, 8, 33, 64, 65, 130, 600, 1024):
        for k in (4, 20, 32):
            named = [plan(a, 0, [(1, n, m, k, 0)])[0] == 0 for a in (2, 4)]
            st, groups = plan(0, 0, [(1, n, m, k, 0)])
            assert st == 0 or not any(named), (n, m, k)
            for count in (1, 20, 200):
                st2, groups = plan(0, 0, [(count, n, m, k, 0), (2, 100, 10, k, 1)])
                assert st2 == st
                for g in groups:
                    assert g[3] <= g[4] <= 16 and g[5] <= 226 * 1024 and g[2] in (2, 4, 8), groups
