"""How batches of one direction at several observer times are cut into time
groups: a small C++ program calls the library's grouping rule on views that differ
only in observer time, and its groups are held to the rule stated here.

A group's members are consecutive, at most `gmax` of them, and span at most
min(3, (M + 1) / 2) snapshots; a batch takes as few groups as that allows, or none
where they would hold less than 7/4 views on average."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2609_09322_gb300 import build, gbdart

CUDA = os.path.dirname(os.path.dirname(build.nvcc()))

PROGRAM = r"""
#include <cstdio>
#include <cstring>
#include <memory>
#include "gbd_internal.h"
namespace gbd { void group_views(MarchArgs &a, int gmax); }
int main()
{
    int m, gmax, n;
    while (std::scanf("%d %d %d", &m, &gmax, &n) == 3) {
        auto a = std::make_unique<gbd::MarchArgs>();
        std::memset(a.get(), 0, sizeof(*a));
        a->vol.M = m;
        a->n_views = n;
        for (int v = 0; v < n; ++v) {
            double u;
            if (std::scanf("%lf", &u) != 1) return 1;
            a->views[v].u_obs = static_cast<long long>(u * 4294967296.0);
            a->views[v].win_lo = static_cast<float>(u - m);
            a->views[v].win_hi = static_cast<float>(u + 1.0);
        }
        gbd::group_views(*a, gmax);
        const int units = a->n_groups > 0 ? a->n_groups : n;
        std::printf("%d %d", a->n_groups > 0 ? a->group_snaps : 0, a->n_groups > 0 ? a->group_size : 0);
        for (int g = 0; g < units; ++g) std::printf(" %d", a->n_groups > 0 ? a->group_first[g + 1] - a->group_first[g] : 1);
        std::printf("\n");
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    gbdart.load_library()
    d = tmp_path_factory.mktemp("groups")
    (d / "groups.cpp").write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-I", build.CSRC, "-I", os.path.join(CUDA, "include"), str(d / "groups.cpp"),
                    build.lib_path(), "-Wl,-rpath," + build.BUILD, "-Wl,--allow-shlib-undefined", "-o",
                    str(d / "groups")], check=True, capture_output=True)

    def run(cases):
        text = "\n".join(f"{m} {gmax} {len(t)} " + " ".join(repr(float(x)) for x in t) for m, gmax, t in cases)
        env = dict(os.environ)
        env["LD_LIBRARY_PATH"] = os.path.join(CUDA, "lib64") + ":" + env.get("LD_LIBRARY_PATH", "")
        out = subprocess.run([str(d / "groups")], input=text, check=True, capture_output=True, text=True, env=env).stdout
        return [[int(x) for x in line.split()] for line in out.splitlines()]

    return run


def fewest(m, gmax, times):
    """The fewest groups that hold the views in order."""
    lim, n, best = min(3.0, 0.5 * (m + 1)), len(times), [0]
    for e in range(1, n + 1):
        best.append(min(best[b] + 1 for b in range(max(0, e - gmax), e)
                        if e == b + 1 or max(times[b:e]) - min(times[b:e]) <= lim))
    return best[n]


EVEN = list(np.arange(24) * 0.125)
SERIES = [
    EVEN,                                            # evenly spaced and close
    EVEN[:-1] + [EVEN[-1] + 8.0],                    # the last one late
    [0.0] + [t + 8.0 for t in EVEN[1:]],             # a gap after the first
    EVEN[:5] + [t + 8.0 for t in EVEN[5:]],          # and after the fifth
    [0.0, 0.125, 0.25, 0.375, 0.5, 0.625, 0.75, 20.0],
    [0.0, 2.5, 2.75, 3.0, 5.75, 6.0, 6.25],          # cut where equal parts would not be
    list(np.arange(127) * 0.0625) + [40.0],
    list(np.arange(12) * 4.0),                       # no two close enough
    list(np.arange(9) * 1.0), list(np.arange(11) * 1.5),
    list(np.random.default_rng(1).uniform(0.0, 9.0, 40)), sorted(np.random.default_rng(2).uniform(0.0, 60.0, 128)),
]


@pytest.mark.parametrize("m", [1, 2, 5, 16])
@pytest.mark.parametrize("gmax", [2, 3, 4, 8])
def test_groups_are_the_fewest_and_close(rule, m, gmax):
    lim = min(3.0, 0.5 * (m + 1))
    for times, (snaps, size, *lens) in zip(SERIES, rule([(m, gmax, t) for t in SERIES])):
        at, widest = 0, 0.0
        for k in lens:
            span = max(times[at:at + k]) - min(times[at:at + k])
            assert 1 <= k <= gmax and (k == 1 or span <= lim), (times, lens)
            widest, at = max(widest, span), at + k
        assert at == len(times)
        n, few = len(times), fewest(m, gmax, times)
        assert len(lens) == (few if 4 * n >= 7 * few else n), (times, lens)
        if max(lens) > 1:
            assert snaps == (3 if widest <= 1.0 else 5) and size == (4 if max(lens) <= 4 else 8)


def test_one_late_view_leaves_the_others_grouped(rule):
    assert [len(x) - 2 for x in rule([(16, 4, t) for t in SERIES[:4]])] == [6, 7, 7, 7]


RUNS_PROGRAM = r"""
#include <cstdio>
#include <cstring>
#include <memory>
#include <vector>
#include "runtime.h"
int main()
{
    int w, h, n;
    while (std::scanf("%d %d %d", &w, &h, &n) == 3) {
        std::vector<gbd::ViewDev> hv(n);
        std::memset(hv.data(), 0, sizeof(gbd::ViewDev) * n);
        for (int v = 0; v < n; ++v) {
            int dir;
            double u;
            if (std::scanf("%d %lf", &dir, &u) != 2) return 1;
            hv[v].g0[0] = dir;
            hv[v].u_obs = static_cast<long long>(u * 4294967296.0);
        }
        gbd::Volume vol;
        vol.grid.n[0] = vol.grid.n[1] = vol.grid.n[2] = 4;
        vol.grid.n_epochs = 4;
        gbd_image_spec s{};
        s.width = w;
        s.height = h;
        auto a = std::make_unique<gbd::MarchArgs>();
        gbd::fill_args(*a, vol, hv.data(), n, 0, s, nullptr, nullptr, gbd::LaunchCfg{8, 4, 4, 2, 1, 1, 0, 4}, nullptr);
        std::printf("%d", a->near_units);
        for (int v = 0; v < n; ++v) std::printf(" %d:%d", a->run_first[v], a->run_len[v]);
        std::printf("\n");
    }
    std::fflush(stdout);
    std::_Exit(0);
}
"""


@pytest.fixture(scope="module")
def runs(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    gbdart.load_library()
    d = tmp_path_factory.mktemp("runs")
    (d / "runs.cpp").write_text(RUNS_PROGRAM.replace("#include <cstdio>", "#include <cstdio>\n#include <cstdlib>"))
    subprocess.run([cxx, "-std=c++17", "-I", build.CSRC, "-I", os.path.join(CUDA, "include"), str(d / "runs.cpp"),
                    build.lib_path(), "-Wl,-rpath," + build.BUILD, "-Wl,--allow-shlib-undefined", "-o",
                    str(d / "runs")], check=True, capture_output=True)

    def run(w, h, views):
        text = f"{w} {h} {len(views)} " + " ".join(f"{d} {u}" for d, u in views) + "\n"
        env = dict(os.environ)
        env["LD_LIBRARY_PATH"] = os.path.join(CUDA, "lib64") + ":" + env.get("LD_LIBRARY_PATH", "")
        out = subprocess.run([str(d / "runs")], input=text, check=True, capture_output=True, text=True, env=env).stdout
        near, *pairs = out.split()
        first = [tuple(int(x) for x in p.split(":")) for p in pairs]
        # runs are whole: every unit names the run it is in
        at = 0
        lens = []
        while at < len(views):
            f, k = first[at]
            assert f == at and k >= 1 and first[at:at + k] == [(f, k)] * k
            lens.append(k)
            at += k
        return int(near), lens

    return run


def test_which_views_go_side_by_side(runs):
    dirs = [(k, 1.0) for k in range(24)]
    assert runs(256, 256, dirs[:16]) == (0, [16])                       # 2^20 pixels at a time
    assert runs(256, 256, dirs) == (0, [12, 12])                        # in equal parts
    assert runs(1024, 1024, dirs[:3]) == (0, [1, 1, 1])
    assert runs(16384, 16384, dirs[:2]) == (0, [1, 1])
    assert runs(1, 1, [(k, 0.0) for k in range(128)]) == (0, [128])
    same = [(0, 0.5 * k) for k in range(9)]
    assert runs(512, 512, same) == (8, [9])                             # whatever their size
    assert runs(512, 512, [(0, 1.5 * k) for k in range(5)]) == (0, [5])
    assert runs(512, 512, [(0, 2.0 * k) for k in range(5)]) == (0, [1] * 5)
    # two other directions, a series, and one more direction
    assert runs(64, 64, [(1, 0.0), (2, 0.0)] + same + [(3, 0.0)]) == (8, [2, 9, 1])
