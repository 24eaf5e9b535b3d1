"""Serving on the host: requests can be submitted while a wave is being launched, and
the next wave takes all of them.

A C++ program runs the library's server over its own stand-ins for the CUDA calls
and for the wave's launch, which it holds until the other requests are in."""
import os
import shutil
import subprocess

import pytest

from paper_2609_09322_gb300 import build, gbdart

CUDA = os.path.dirname(os.path.dirname(build.nvcc()))

PROGRAM = r"""
#include <chrono>
#include <condition_variable>
#include <cstdio>
#include <cstdlib>
#include <mutex>
#include <thread>
#include <vector>
#include "runtime.h"

static std::mutex g_mu;
static std::condition_variable g_cv;
static int g_entered = 0, g_released = 0;
static std::vector<int> g_waves;  // requests of each
static bool g_fail = false;

namespace gbd {
cudaError_t launch_wave(const WaveArgs &a, const LaunchCfg &, cudaStream_t)
{
    std::unique_lock<std::mutex> lock(g_mu);
    g_waves.push_back(a.n_reqs);
    ++g_entered;
    g_cv.notify_all();
    // bounded: a server that keeps submissions out meanwhile goes on after 2 s
    g_cv.wait_for(lock, std::chrono::seconds(2), [] { return g_released >= g_entered; });
    return g_fail ? cudaErrorUnknown : cudaSuccess;
}
}
extern "C" {
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { *s = nullptr; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = 1.f; return cudaSuccess; }
cudaError_t cudaLaunchHostFunc(cudaStream_t, cudaHostFn_t fn, void *p) { std::thread(fn, p).detach(); return cudaSuccess; }
}

static gbd_request request(float *out)
{
    gbd_request r{};
    r.volume = 7;
    r.view.dir[2] = 1.0;
    r.view.up[1] = 1.0;
    r.view.c = 1.0;
    r.view.nu_ratio = 1.0;
    r.spec.width = r.spec.height = 8;
    r.spec.fov_u = r.spec.fov_v = 8.0;
    r.spec.out = out;
    return r;
}

static void enter(int n)  // wait until the n-th launch has begun
{
    std::unique_lock<std::mutex> lock(g_mu);
    if (!g_cv.wait_for(lock, std::chrono::seconds(10), [&] { return g_entered >= n; })) std::exit(2);
}
static void release()
{
    std::lock_guard<std::mutex> lock(g_mu);
    ++g_released;
    g_cv.notify_all();
}

int main(int argc, char **)
{
    g_fail = argc > 1;
    gbd_ctx *ctx = new gbd_ctx;
    ctx->budget = 1 << 30;
    auto vol = std::make_unique<gbd::Volume>();
    vol->grid.n[0] = vol->grid.n[1] = vol->grid.n[2] = 4;
    vol->grid.dx[0] = vol->grid.dx[1] = vol->grid.dx[2] = 1.0;
    vol->grid.n_epochs = 1;
    vol->grid.dt = 1.0;
    gbd::Volume *v = vol.get();
    ctx->volumes[7] = std::move(vol);
    gbd_serve_config cfg{};
    cfg.max_waves = 2;
    if (gbd_serve_start(ctx, &cfg)) return 3;
    float out[64];
    uint64_t t[6];
    gbd_request r = request(out);
    if (gbd_submit(ctx, &r, &t[0])) return 4;
    enter(1);
    const auto t0 = std::chrono::steady_clock::now();
    for (int k = 1; k < 6; ++k)
        if (gbd_submit(ctx, &r, &t[k])) return 5;
    gbd_serve_summary s;
    if (gbd_serve_stats(ctx, 0, &s)) return 6;
    const double held = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
    std::printf("held %d running %d pending %d pinned %d\n", held > 1.0, s.in_flight, s.pending, v->pinned_by_requests.load());
    if (gbd_cancel(ctx, t[0]) || gbd_unload(ctx, 7) != GBD_ERR_BUSY) return 7;
    release();
    enter(2);
    release();
    int rc[6];
    for (int k = 0; k < 6; ++k) rc[k] = gbd_wait(ctx, t[k], 10000, nullptr);
    std::printf("codes %d %d %d %d %d %d\n", rc[0], rc[1], rc[2], rc[3], rc[4], rc[5]);
    std::printf("waves");
    for (int n : g_waves) std::printf(" %d", n);
    gbd_serve_stats(ctx, 0, &s);
    std::printf("\nleft %d %d %d\n", s.in_flight, s.pending, v->pinned_by_requests.load());
    gbd_serve_stop(ctx);
    std::fflush(stdout);
    std::_Exit(0);
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    gbdart.load_library()
    d = tmp_path_factory.mktemp("serve")
    (d / "serve.cpp").write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-rdynamic", "-pthread", "-I", build.CSRC, "-I", os.path.join(CUDA, "include"),
                    str(d / "serve.cpp"), build.lib_path(), "-Wl,-rpath," + build.BUILD,
                    "-Wl,--allow-shlib-undefined", "-o", str(d / "serve")], check=True, capture_output=True)

    def run(*args):
        env = dict(os.environ)
        env["LD_LIBRARY_PATH"] = os.path.join(CUDA, "lib64") + ":" + env.get("LD_LIBRARY_PATH", "")
        out = subprocess.run([str(d / "serve"), *args], check=True, capture_output=True, text=True, env=env, timeout=60)
        return dict(line.split(" ", 1) for line in out.stdout.splitlines())

    return run


def test_submissions_get_through_during_a_launch(program):
    r = program()
    assert r["held"] == "0 running 1 pending 5 pinned 6"
    assert r["waves"] == "1 5"
    assert r["codes"] == f"{gbdart.ERR_CANCELLED} 0 0 0 0 0"
    assert r["left"] == "0 0 0"


def test_a_launch_that_fails_gives_everything_back(program):
    r = program("fail")
    assert r["waves"] == "1 5"
    assert r["codes"] == " ".join([str(gbdart.ERR_CUDA)] * 6)
    assert r["left"] == "0 0 0"
