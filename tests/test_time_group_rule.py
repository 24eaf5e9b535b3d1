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
