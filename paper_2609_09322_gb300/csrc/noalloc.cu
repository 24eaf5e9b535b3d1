// noalloc.cu -- batch render that allocates no memory.
//
// gbd_render_batch keeps a cached graph per batch, and a table of the order in
// which a single view's blocks are taken.  Some
// callers cannot let a library allocate device memory while they render:
// applications that hand the whole device to their own allocator or memory
// pool up front (a cudaMalloc inside the library would fail, or break their
// accounting), and latency-critical loops where cudaMalloc / cudaFree, which
// may synchronise the device, are not acceptable.  This entry point serves
// them: the march needs no device memory of its own.
#include <cuda_runtime.h>

#include <cstring>
#include <mutex>

#include "runtime.h"

namespace gbd {
namespace {

constexpr int kNoAllocMaxViews = GBD_NOALLOC_MAX_VIEWS;
std::mutex g_mu;                          // guards the arrays below
ViewDev g_host_views[kNoAllocMaxViews];   // the views, set up on the host
MarchArgs g_args;                         // launch arguments (about 31 KB: not on the stack)

}  // namespace
}  // namespace gbd

using namespace gbd;

extern "C" int gbd_render_batch_noalloc(gbd_ctx *ctx, gbd_volume vid, const gbd_view *views, int32_t n,
                                        const gbd_image_spec *spec, const gbd_launch *launch, void *stream)
{
    if (!ctx || !views || !spec) return fail(GBD_ERR_INVALID, "NULL argument");
    if (n < 1 || n > kNoAllocMaxViews)
        return fail(GBD_ERR_INVALID, "gbd_render_batch_noalloc takes 1 to %d views per call (got %d)",
                    kNoAllocMaxViews, n);
    if (spec->width < 1 || spec->height < 1 || spec->width > 16384 || spec->height > 16384)
        return fail(GBD_ERR_INVALID, "image: width/height must be in [1, 16384]");
    if (!spec->out || spec->out_on_host)
        return fail(GBD_ERR_INVALID, "gbd_render_batch_noalloc needs a device output buffer");
    LaunchCfg cfg = resolve_launch(launch);
    int rc = check_launch(cfg);
    if (rc) return rc;
    // The region schedule needs partial-sum slots in device memory.
    if (cfg.region != 0)
        return fail(GBD_ERR_INVALID, "gbd_render_batch_noalloc has no region schedule (launch.region must be 0)");
    std::lock_guard<std::mutex> lock(ctx->mu);
    Volume *vol = ctx->find(vid);
    if (!vol) return fail(GBD_ERR_NOTFOUND, "unknown volume %llu", static_cast<unsigned long long>(vid));
    if (!launch) {
        // a tuned region schedule is replaced by the whole-ray march (the
        // tuned packet, CTA and group shapes are kept)
        lookup_tuned(*ctx, tune_key(*vol, spec->width, spec->height, n, views[0].flags), cfg);
        cfg.region = 0;
    }
    DeviceGuard guard(ctx->device);

    std::lock_guard<std::mutex> slock(g_mu);
    for (int k = 0; k < n; ++k)
        if ((rc = make_view(*vol, views[k], spec->width, spec->height, spec->fov_u, spec->fov_v, g_host_views[k])))
            return rc;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    cudaError_t e = cudaSuccess;
    const int chunks = march_chunks(n);
    for (int c = 0; c < chunks && e == cudaSuccess; ++c) {
        fill_args(g_args, *vol, g_host_views, n, c, *spec, spec->out, spec->samples, cfg, ctx->err_word);
        group_views(g_args, cfg.group);
        e = launch_march(g_args, cfg, st);
    }
    if (e != cudaSuccess) return cuda_fail(e, "no-alloc batch launch");
    set_launch_count(chunks);
    return GBD_OK;
}
