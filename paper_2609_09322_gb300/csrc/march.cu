// march.cu -- sm_103a ray-march kernels for the relativistic line-of-sight sum.
//
// One lane owns one ray (pixel) from entry to exit, so every pixel is summed in
// one fixed order whether it is rendered alone, in a batch or in a served mix.
// A warp owns a packet of 32 neighbouring pixels (8x4 by default), so at each
// step its lanes gather neighbouring cells of the bricked volume.
//
// Per view, on the host in float64: the constants of ViewDev (fixed-point
// pixel positions, face spacings, epoch rates), with every axis the view runs
// down mirrored so that the march always steps to increasing cell index.
// Per ray (Sec. 2.4 traversal, Sec. 5.1 fast-forward, Eqs. 2, 6-9, 14, 19),
// with no float64 on the device:
//   * once: the pixel position in Q24.40 fixed point, an anchor at the later of
//     the box entry and the window start where the retarded time can reach a
//     stored snapshot, the anchor's cell, and the epoch coordinate there in
//     Q31.32 fixed point;
//   * per cell: the nearest next face crossing (each recomputed from its plane
//     count, never accumulated), the chord ds from the previous one, the epoch
//     coordinate at the chord midpoint, the two snapshot records, the Doppler
//     boost of each, their linear interpolation, and a compensated float32
//     accumulation of value * ds.
// Cells are gathered a stage of H at a time, while the stage before is being
// evaluated (run_stages), so each lane keeps up to 4 H independent loads in
// flight.
//
// Time groups (batched renders of one direction at several observer times):
// one traversal per ray serves up to 4 or 8 views, each with its own sums
// (march_group, group_kernel).
//
// bfloat16/float16 records (march_ray_bf16, march_group_bf16) take a lighter
// march whose storage error (2^-9 in j', 2^-11 in u) dwarfs its arithmetic:
// the epoch coordinate is a float linear in s instead of the exact fixed
// point, the step runs without branches for every lane (a lane whose ray has
// ended takes no step and reads nothing), the Doppler factor is the plain
// 1 / (Gamma + u.s_hat) where the volume's Gamma allows it, and the sum is
// not compensated.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cfloat>
#include <type_traits>

#include "gbd_internal.h"

namespace gbd {
namespace {

constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ float lg2_approx(float x)
{
    float r;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ float ex2_approx(float x)
{
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ float sqrt_approx(float x)
{
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ float2 f2(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 neg2(float2 v) { return make_float2(-v.x, -v.y); }

// Per-view float constants held in registers during the march.
struct BoostConsts {
    float shx, shy, shz;  // s_hat rounded to float
    float slx, sly, slz;  // rounding residual of s_hat
    float expo;           // 2 - alpha
    bool beaming;
};

template <int STORE>
struct Record;

// 16-byte record {j', beta_x, beta_y, beta_z}.
template <>
struct Record<GBD_STORE_F32> {
    using T = float4;
    static __device__ __forceinline__ T load_at(unsigned long long a) { return __ldg(reinterpret_cast<const float4 *>(a)); }
    static __device__ __forceinline__ T zero() { return make_float4(0.f, 0.f, 0.f, 0.f); }
    // D^(2 - alpha) j' with D = sqrt(1 - beta^2) / (1 + beta . s_hat) (Eq. 14).
    // 1 + beta.s_hat and 1 - beta^2 are formed with fused multiply-adds so
    // each is rounded once near its (possibly small) value.
    static __device__ __forceinline__ float emissivity(const T r) { return r.x; }
    // D^(2 - alpha), or 1 without beaming
    static __device__ __forceinline__ float boost(const T r, const BoostConsts &c)
    {
        if (!c.beaming) return 1.0f;
        float den = fmaf(r.y, c.shx, fmaf(r.z, c.shy, fmaf(r.w, c.shz, 1.0f)));
        den += fmaf(r.y, c.slx, fmaf(r.z, c.sly, r.w * c.slz));
        const float inv_g2 = fmaf(-r.y, r.y, fmaf(-r.z, r.z, fmaf(-r.w, r.w, 1.0f)));
        const float log2_d = fmaf(0.5f, lg2_approx(inv_g2), -lg2_approx(den));
        return ex2_approx(c.expo * log2_d);
    }
};

// 8-byte record {bf16 j', f16 u_x, f16 u_y, f16 u_z}, u = Gamma beta.
template <>
struct Record<GBD_STORE_BF16_F16U> {
    using T = uint2;
    static __device__ __forceinline__ T zero() { return make_uint2(0u, 0u); }
    static __device__ __forceinline__ T load_at(unsigned long long a) { return __ldg(reinterpret_cast<const uint2 *>(a)); }
    // Both snapshots of a paired block: one 16-byte load.
    static __device__ __forceinline__ void load_pair_at(unsigned long long a, T &lo, T &hi)
    {
        const uint4 v = __ldg(reinterpret_cast<const uint4 *>(a));
        lo = make_uint2(v.x, v.y);
        hi = make_uint2(v.z, v.w);
    }
    // D = 1 / (Gamma + u.s_hat).  When u.s_hat < 0 (motion towards the
    // observer) the denominator cancels, so the same D is evaluated as
    // (Gamma + |u.s_hat|) / (1 + |u|^2 - (u.s_hat)^2), which has no cancellation.
    // s_hat enters rounded to float: its rounding (6e-8) is far below the
    // float16 resolution of u (5e-4 relative), unlike in the float32 record.
    static __device__ __forceinline__ float emissivity(const T r) { return __uint_as_float(r.x << 16); }
    // D^(2 - alpha), or 1 without beaming
    static __device__ __forceinline__ float boost(const T r, const BoostConsts &c)
    {
        if (!c.beaming) return 1.0f;
        // u_x is the high half of r.x, (u_y, u_z) the two halves of r.y
        __half2 hx, hyz;
        memcpy(&hx, &r.x, sizeof(hx));
        memcpy(&hyz, &r.y, sizeof(hyz));
        const float ux = __high2float(hx);
        const float2 uyz = __half22float2(hyz);
        const float uy = uyz.x, uz = uyz.y;
        const float us = fmaf(ux, c.shx, fmaf(uy, c.shy, uz * c.shz));
        const float uu = fmaf(ux, ux, fmaf(uy, uy, uz * uz));
        const float gp = sqrt_approx(1.0f + uu) + fabsf(us);
        const float perp = 1.0f + fmaf(-us, us, uu);
        const float log2_d = (us < 0.f) ? (lg2_approx(gp) - lg2_approx(perp)) : -lg2_approx(gp);
        return ex2_approx(c.expo * log2_d);
    }
    // boosted2() in the plain form D = 1 / (Gamma + u.s_hat), log2 D =
    // -log2(Gamma + u.s_hat).  For u.s_hat near -Gamma the sum cancels: its
    // float32 rounding (about 3.3e-7 Gamma absolute) over Gamma + u.s_hat >=
    // 1 / (2 Gamma) bounds the relative error of D by 6.6e-7 Gamma^2, at most
    // 4.3e-5 (1.1e-4 in D^2.6) for Gamma <= 8, the volumes this form is used
    // for (beta <= 0.992); the float16 u itself carries 4.9e-4.
    static __device__ __forceinline__ float2 boosted2_plain(const T lo, const T hi, const BoostConsts &c)
    {
        const float2 j = make_float2(__uint_as_float(lo.x << 16), __uint_as_float(hi.x << 16));
        if (!c.beaming) return j;
        const uint32_t px = __byte_perm(lo.x, hi.x, 0x7632);  // (u_x lo, u_x hi)
        const uint32_t py = __byte_perm(lo.y, hi.y, 0x5410);  // (u_y lo, u_y hi)
        const uint32_t pz = __byte_perm(lo.y, hi.y, 0x7632);  // (u_z lo, u_z hi)
        __half2 hx, hy, hz;
        memcpy(&hx, &px, sizeof(hx));
        memcpy(&hy, &py, sizeof(hy));
        memcpy(&hz, &pz, sizeof(hz));
        const float2 ux = __half22float2(hx), uy = __half22float2(hy), uz = __half22float2(hz);
        const float2 us = __ffma2_rn(ux, f2(c.shx), __ffma2_rn(uy, f2(c.shy), __fmul2_rn(uz, f2(c.shz))));
        const float2 g2 = __ffma2_rn(ux, ux, __ffma2_rn(uy, uy, __ffma2_rn(uz, uz, f2(1.0f))));  // Gamma^2
        const float2 den = __fadd2_rn(make_float2(sqrt_approx(g2.x), sqrt_approx(g2.y)), us);
        const float2 e = __fmul2_rn(f2(-c.expo), make_float2(lg2_approx(den.x), lg2_approx(den.y)));
        return __fmul2_rn(j, make_float2(ex2_approx(e.x), ex2_approx(e.y)));
    }
    // boosted() of two records at once: their u components are paired by
    // byte permutes, then each lane takes the same correctly rounded steps as
    // boosted() (paired float32 instructions of sm_100 and later).
    static __device__ __forceinline__ float2 boosted2(const T lo, const T hi, const BoostConsts &c)
    {
        const float2 j = make_float2(__uint_as_float(lo.x << 16), __uint_as_float(hi.x << 16));
        if (!c.beaming) return j;
        const uint32_t px = __byte_perm(lo.x, hi.x, 0x7632);  // (u_x lo, u_x hi)
        const uint32_t py = __byte_perm(lo.y, hi.y, 0x5410);  // (u_y lo, u_y hi)
        const uint32_t pz = __byte_perm(lo.y, hi.y, 0x7632);  // (u_z lo, u_z hi)
        __half2 hx, hy, hz;
        memcpy(&hx, &px, sizeof(hx));
        memcpy(&hy, &py, sizeof(hy));
        memcpy(&hz, &pz, sizeof(hz));
        const float2 ux = __half22float2(hx), uy = __half22float2(hy), uz = __half22float2(hz);
        const float2 us = __ffma2_rn(ux, f2(c.shx), __ffma2_rn(uy, f2(c.shy), __fmul2_rn(uz, f2(c.shz))));
        const float2 uu = __ffma2_rn(ux, ux, __ffma2_rn(uy, uy, __fmul2_rn(uz, uz)));
        const float2 g1 = __fadd2_rn(f2(1.0f), uu);
        const float2 gp = __fadd2_rn(make_float2(sqrt_approx(g1.x), sqrt_approx(g1.y)),
                                     make_float2(fabsf(us.x), fabsf(us.y)));
        const float2 perp = __fadd2_rn(f2(1.0f), __ffma2_rn(neg2(us), us, uu));
        const float2 lgp = make_float2(lg2_approx(gp.x), lg2_approx(gp.y));
        const float2 lpp = make_float2(lg2_approx(perp.x), lg2_approx(perp.y));
        const float2 dif = __fadd2_rn(lgp, neg2(lpp));
        const float2 lg = make_float2(us.x < 0.f ? dif.x : -lgp.x, us.y < 0.f ? dif.y : -lgp.y);
        const float2 e = __fmul2_rn(f2(c.expo), lg);
        return __fmul2_rn(j, make_float2(ex2_approx(e.x), ex2_approx(e.y)));
    }
};

#ifdef GBD_CHECKED
__device__ __forceinline__ bool check_cell(const VolDev &vol, int *err_word, int ix, int iy, int iz, int m)
{
    const bool ok = ix >= 0 && ix < vol.n[0] && iy >= 0 && iy < vol.n[1] && iz >= 0 && iz < vol.n[2] &&
                    m >= 0 && m < vol.M;
    if (!ok && err_word) atomicCAS(err_word, 0, 1);
    return ok;
}
#endif

// The epoch coordinate u = (t_bar - t0) / dt is carried in Q31.32 fixed point
// (int64, 2^-32 epochs per unit): float32 cannot resolve u to better than half
// an ulp of the snapshot count (about 4e-6 at u ~ 64), which a fast-changing
// field amplifies beyond a 1e-5 relative pixel tolerance; integer updates are
// exact and cheap.
constexpr float kTwo32 = 4294967296.0f;        // 2^32
constexpr float kTwo40 = 1099511627776.0f;      // 2^40
constexpr float kInv2p40 = 9.094947017729282e-13f;  // 2^-40

// x (a float) times y = y_hi + y_lo (a double-float), as a fixed-point
// integer of scale `scale`: the product x * y_hi is split exactly into its
// rounded value and rounding error with a fused multiply-add, and each part
// is converted separately, so the result carries about 48 bits of y.
__device__ __forceinline__ long long dd_mul_fix(float x, float y_hi, float y_lo, float scale)
{
    const float p = __fmul_rn(x, y_hi);
    const float e = fmaf(x, y_hi, -p);
    const float r = fmaf(x, y_lo, e);
    return __float2ll_rn(p * scale) + __float2ll_rn(r * scale);
}

__device__ __forceinline__ float fix_to_float(long long v, float inv_scale)
{
    return __ll2float_rn(v) * inv_scale;
}

// One entry of the march tables at byte offset `cur` from `base` (shared memory).
__device__ __forceinline__ int32_t tab_at(const int32_t *base, uint32_t cur)
{
    return *reinterpret_cast<const int32_t *>(reinterpret_cast<const char *>(base) + cur);
}

// State of one axis of a ray: the next face crossing and what changes there.
struct AxisState {
    float nkf;      // planes from the anchor cell's lower face to the next crossing
    float sn;       // s of the next crossing, relative to the anchor
    float of;       // the anchor's offset inside its cell, times the face spacing
    long long un;   // epoch coordinate at the next crossing, Q31.32
    uint32_t cur;   // byte offset of the table entry of the step through it
};

// The box a ray is marched through, in the march frame (mirrored axes
// mirrored), and where its table entries start: the whole grid for a direct
// render, one region of it for the region schedule.  Along axis i the steps out
// of cells lo[i] .. hi[i] - 1 have their entries at byte offsets cur0[i],
// cur0[i] + 4, ..., and one more entry follows (of any value).
struct RayBox {
    int lo[3], hi[3];
    uint32_t cur0[3];
};

// The whole grid as seen by view V, with the volume's own march tables.
__device__ __forceinline__ RayBox grid_box(const VolDev &vol, const ViewDev &V)
{
    RayBox B;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const bool mirrored = (V.flags & (kFlagMirror0 << i)) != 0u;
        B.lo[i] = 0;
        B.hi[i] = vol.n[i];
        B.cur0[i] = 4u * static_cast<uint32_t>(march_table_base(vol.n, i) + (mirrored ? vol.n[i] + 1 : 0));
    }
    return B;
}

// Copies a volume's march tables into shared memory.
__device__ __forceinline__ void stage_all(int32_t *s_tab, const VolDev &vol)
{
    const int total = march_table_entries(vol.n);
    for (int i = threadIdx.x; i < total; i += blockDim.x) s_tab[i] = vol.mtab[i];
    __syncthreads();
}

// The same for tables that take a thread more than kCopiesMax loads, only where the
// rays of this CTA can read them (pixel (p, q) of this lane, as view V sees them,
// within [win_lo, win_hi]): of each axis the table of the view's direction, from
// the lowest cell that a ray enters to the highest.  s_tab stands after kSpanEntries words.
// Per ray the cells follow from the float chord through the box: the march starts in
// the cell of the later of s_in and win_lo, which set-up computes alike, and leaves
// the box by s_out, so they are known to within float rounding (a few 2^-24 of the
// largest coordinate in the sum; the slack is 2 and 2^-20 of it), and it reads at
// most two entries past its last one.  A ray that misses the box or the window takes
// no step; its lane may read an entry that is not there, and uses nothing of it.
//
// What it is for: a CTA marches 32 to 256 rays, and where an axis is long and the
// rays are short or miss, copying everything takes longer than they do: 1024^2 images of
// 4096 x 16 x 16 across the long axis 123 -> 40 us, filled by rays of 16 cells 167 -> 102.
// Shorter tables are copied whole, as finding the spans takes about as long (32^3: 5% more).
// A call, not inlined: the marches behind it keep their registers.
constexpr int kCopiesMax = 32;
__device__ __noinline__ void stage_spans(int32_t *s_tab, const VolDev &vol, const ViewDev &V, int p, int q, bool in_image,
                                         float win_lo, float win_hi)
{
    const int threads = static_cast<int>(blockDim.x), t = static_cast<int>(threadIdx.x);
    float g[3], s_in = -3.0e38f, s_out = 3.0e38f;
    bool hit = in_image;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const long long gx = V.g0[i] + static_cast<long long>(p) * V.gu[i] + static_cast<long long>(q) * V.gv[i];
        g[i] = fix_to_float(gx, kInv2p40);
        if (V.inv_a[i] != 0.f) {
            s_in = fmaxf(s_in, -g[i] * V.inv_a[i]);
            // late by more than g's rounding, which a slowly crossed axis turns into a long way
            const float n = static_cast<float>(vol.n[i]);
            s_out = fminf(s_out, (n - g[i] + 1e-6f * (n + fabsf(g[i]))) * V.inv_a[i]);
        } else if (gx < 0 || gx >= (static_cast<long long>(vol.n[i]) << 40)) {
            hit = false;
        }
    }
    // the test of setup_ray, twice as wide
    s_in = fmaxf(s_in, win_lo);
    if (!(fminf(s_out, win_hi) > s_in - 2e-3f * (1.f + fabsf(s_in)))) hit = false;
    int32_t *s_span = s_tab - kSpanEntries;  // per warp: lowest and highest entry of each axis
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const float n = static_cast<float>(vol.n[i]), from = s_in * V.a_hi[i], to = fmaxf(s_in, s_out) * V.a_hi[i];
        const float slack = 2.0f + 1e-6f * (fabsf(g[i]) + fmaxf(fabsf(from), fabsf(to)));
        const int first = static_cast<int>(fminf(fmaxf(g[i] + from - slack, 0.f), n));
        const int last = static_cast<int>(fminf(fmaxf(g[i] + to + slack + 2.0f, 0.f), n));
        const int lo = __reduce_min_sync(kFull, hit ? first : vol.n[i]);
        const int hi = __reduce_max_sync(kFull, hit ? last : -1);
        if ((t & 31) == 0) {
            s_span[6 * (t >> 5) + 2 * i] = lo;
            s_span[6 * (t >> 5) + 2 * i + 1] = hi;
        }
    }
    __syncthreads();
#pragma unroll 1
    for (int i = 0; i < 3; ++i) {
        int lo = vol.n[i], hi = -1;
        for (int w = 0; w < threads >> 5; ++w) {
            lo = min(lo, s_span[6 * w + 2 * i]);
            hi = max(hi, s_span[6 * w + 2 * i + 1]);
        }
        // 0 <= lo <= n, hi <= n; no ray hits: lo = n, hi = -1
        const int base = march_table_base(vol.n, i) + ((V.flags & (kFlagMirror0 << i)) != 0u ? vol.n[i] + 1 : 0);
        for (int e = lo + t; e <= hi; e += threads) s_tab[base + e] = vol.mtab[base + e];
    }
    __syncthreads();
}
__device__ __forceinline__ void stage_tables(int32_t *s_tab, const VolDev &vol, const ViewDev &V, int p, int q,
                                             bool in_image, float win_lo, float win_hi)
{
    if (march_table_entries(vol.n) <= kCopiesMax * static_cast<int>(blockDim.x)) stage_all(s_tab, vol);
    else stage_spans(s_tab, vol, V, p, q, in_image, win_lo, win_hi);
}

// State of a ray during the march: per axis the next crossing, the layout
// offset of the current cell, its chord start (the latest face crossed) and
// the epoch coordinate there.
struct RayState {
    AxisState ax[3];
    uint32_t sum;      // layout offset of the current cell (the sum of its three axis terms)
    float s_cur;       // s of the latest face crossed
    float s_end;       // s of the box face through which the ray leaves
    long long u_cur;   // epoch coordinate at s_cur, Q31.32
    long long u_a;     // epoch coordinate at the anchor (s = 0), Q31.32
    bool alive;
#ifdef GBD_CHECKED
    int kc[3], kd[3];  // current cell in the volume's own frame, and its step per axis
#endif
};

__device__ __forceinline__ float min3(float a, float b, float c)
{
    float r;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
// The face through which a ray leaves its cell: the nearest of the three next
// crossings, ties to the lowest axis (the zero-length chord that follows adds
// nothing).  No axis is set for a lane whose ray has ended.
struct ExitFace {
    bool x0, x1, x2;
    float s;
};
__device__ __forceinline__ ExitFace exit_face(const AxisState (&ax)[3], bool alive)
{
    ExitFace X;
    X.s = min3(ax[0].sn, ax[1].sn, ax[2].sn);
    X.x0 = alive & (ax[0].sn <= X.s);
    X.x1 = alive & !X.x0 & (ax[1].sn <= X.s);
    X.x2 = alive & !X.x0 & !X.x1;
    return X;
}

// Steps a ray into its next cell through face X: the exit axis's next crossing
// is recomputed from its plane count (never accumulated), and the table entry
// of the step moves the cell's layout offset.  Every update is a select on the
// exit axis, so the lanes of a warp never diverge here; recomputing an axis's
// crossing from an unchanged plane count reproduces it (an axis the ray runs
// parallel to has of = -3e38 and inv_a = 0, so its crossing stays at 3e38).
// A lane whose ray has ended keeps its crossings and cursors and reads the
// table at the cursor it stopped at; its layout offset is never used again.
__device__ __forceinline__ void step_lite(RayState &R, const ExitFace &X, float ia0, float ia1, float ia2,
                                          const int32_t *tab)
{
    AxisState (&ax)[3] = R.ax;
    const uint32_t ce = X.x0 ? ax[0].cur : (X.x1 ? ax[1].cur : ax[2].cur);
    R.sum += static_cast<uint32_t>(tab_at(tab, ce));
    ax[0].nkf = X.x0 ? ax[0].nkf + 1.0f : ax[0].nkf;
    ax[1].nkf = X.x1 ? ax[1].nkf + 1.0f : ax[1].nkf;
    ax[2].nkf = X.x2 ? ax[2].nkf + 1.0f : ax[2].nkf;
    ax[0].cur = X.x0 ? ax[0].cur + 4u : ax[0].cur;
    ax[1].cur = X.x1 ? ax[1].cur + 4u : ax[1].cur;
    ax[2].cur = X.x2 ? ax[2].cur + 4u : ax[2].cur;
    ax[0].sn = fmaf(ax[0].nkf, ia0, -ax[0].of);
    ax[1].sn = fmaf(ax[1].nkf, ia1, -ax[1].of);
    ax[2].sn = fmaf(ax[2].nkf, ia2, -ax[2].of);
#ifdef GBD_CHECKED
    R.kc[0] += X.x0 ? R.kd[0] : 0;
    R.kc[1] += X.x1 ? R.kd[1] : 0;
    R.kc[2] += X.x2 ? R.kd[2] : 0;
#endif
}

// step_lite with the exact epoch coordinate of each axis: it drops by the
// exact per-plane amount.
__device__ __forceinline__ void step_exact(RayState &R, const ExitFace &X, float ia0, float ia1, float ia2,
                                           long long du0, long long du1, long long du2, const int32_t *tab)
{
    step_lite(R, X, ia0, ia1, ia2, tab);
    R.ax[0].un = X.x0 ? R.ax[0].un - du0 : R.ax[0].un;
    R.ax[1].un = X.x1 ? R.ax[1].un - du1 : R.ax[1].un;
    R.ax[2].un = X.x2 ? R.ax[2].un - du2 : R.ax[2].un;
}

// Ray set-up, once per ray, no float64: the anchor at the later of the box
// entry and the window start [win_lo, win_hi] (a view's own window, or the
// union of a group's), its cell and crossings, and the leading empty chords
// stepped through, so that the march proper starts on the first cell whose
// chord is positive.
//
// s_end is where the ray leaves the box: along axis i the crossing of the box's
// upper face is the crossing of plane hi[i] - k, computed from that plane count
// exactly as the march will, and the nearest of the three is s_end.  A
// crossing before s_end is therefore not the last one of its axis, and a ray
// that stops at the first crossing at or past s_end never steps a cursor past
// the entry behind its box's last cell: one float comparison per step keeps
// every gather inside the box.
__device__ __forceinline__ void setup_ray(RayState &R, const VolDev &vol, const ViewDev &V, const RayBox &B, int p,
                                          int q, bool in_image, float win_lo, float win_hi,
                                          const int32_t *__restrict__ tab)
{
    AxisState (&ax)[3] = R.ax;
    bool &alive = R.alive;
    float &s_cur = R.s_cur;
    long long &u_cur = R.u_cur;
    alive = in_image;
    // Pixel position on the image plane in grid-index units (Q24.40, exact
    // integer arithmetic from the per-view constants), in the frame where
    // every axis is marched upwards.
    long long g0[3];
#pragma unroll
    for (int i = 0; i < 3; ++i)
        g0[i] = V.g0[i] + static_cast<long long>(p) * V.gu[i] + static_cast<long long>(q) * V.gv[i];
    // Estimated start of the traversal: the later of the box entry and the
    // window start.  This anchor only has to be a point of the ray no more
    // than a cell past the true start (crossings are measured from it, so it
    // should be close to keep them accurate); it may lie outside the box.
    float s_in_e = -3.0e38f, s_out_e = 3.0e38f;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        if (V.inv_a[i] != 0.f) {
            const float gf = fix_to_float(g0[i], kInv2p40);
            s_in_e = fmaxf(s_in_e, (static_cast<float>(B.lo[i]) - gf) * V.inv_a[i]);
            s_out_e = fminf(s_out_e, (static_cast<float>(B.hi[i]) - gf) * V.inv_a[i]);
        } else if (g0[i] < (static_cast<long long>(B.lo[i]) << 40) ||
                   g0[i] >= (static_cast<long long>(B.hi[i]) << 40)) {
            alive = false;  // parallel to this axis and outside the box along it
        }
    }
    const float s_a = fmaxf(s_in_e, win_lo);
    if (!(fminf(s_out_e, win_hi) > s_a - 1e-3f * (1.f + fabsf(s_a)))) alive = false;
    const float sa = alive ? s_a : 0.f;

    // Anchor: the point s_a of the ray, in exact fixed point; its cell (k,
    // clamped onto the grid), the position o inside that cell, and per axis
    // the face spacing along the ray (inv_a, Eq. 11), so that the crossing of
    // the plane nk cells above the cell's lower face is at nk inv_a - o inv_a.
    const long long u_a = V.u_obs - dd_mul_fix(sa, V.kk_hi, V.kk_lo, kTwo32);
    R.u_a = u_a;
    s_cur = -3.0e38f;  // the latest entry face of the anchor cell
    u_cur = 0;
    R.sum = 0;
    R.s_end = 3.0e38f;
    const int32_t *off = vol.axis_off;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const bool moving = V.inv_a[i] != 0.f;
        const bool mirrored = (V.flags & (kFlagMirror0 << i)) != 0u;
        const long long ga = moving ? g0[i] + dd_mul_fix(sa, V.a_hi[i], V.a_lo[i], kTwo40) : g0[i];
        int k = static_cast<int>(ga >> 40);
        k = min(max(k, B.lo[i]), B.hi[i] - 1);
        const float o = fix_to_float(ga - (static_cast<long long>(k) << 40), kInv2p40);
        AxisState &A = ax[i];
        A.nkf = 1.0f;
        // Rounded products and differences, never contracted: this first
        // crossing, the recomputed ones and s_end have to be one function of
        // the plane count, or a ray could pass its last face unseen.
        A.of = __fmul_rn(o, V.inv_a[i]);
        if (moving) {
            A.sn = __fsub_rn(V.inv_a[i], A.of);
            A.un = u_a - dd_mul_fix(1.0f - o, V.w_hi[i], V.w_lo[i], kTwo32);
            R.s_end = fminf(R.s_end, fmaf(static_cast<float>(B.hi[i] - k), V.inv_a[i], -A.of));
            // the anchor cell's entry face along this axis (plane nk = 0)
            if (-A.of > s_cur) {
                s_cur = -A.of;
                u_cur = A.un + V.du[i];
            }
        } else {
            A.of = -3.0e38f;     // with inv_a = 0: the crossing stays at 3e38,
            A.sn = 3.0e38f;      // never the nearest face
            A.un = LLONG_MIN / 2;
        }
        A.cur = B.cur0[i] + 4u * static_cast<uint32_t>(k - B.lo[i]);
        R.sum += static_cast<uint32_t>(__ldg(off + (mirrored ? vol.n[i] - 1 - k : k)));
        off += vol.n[i];
#ifdef GBD_CHECKED
        R.kc[i] = mirrored ? vol.n[i] - 1 - k : k;
        R.kd[i] = mirrored ? -1 : 1;
#endif
    }

    // Leading empty chords: when the anchor cell was clamped onto the grid, or
    // the anchor sits on a face, the ray can leave a cell along one axis before
    // it has entered it along another.  Those cells are stepped through until
    // the nearest exit lies past the latest entry; from there on the exits
    // only increase, so every chord of the march proper starts at the end of
    // the one before.  Each step moves one table cursor up, and s_end stops
    // the ray at the box face, so the loop is bounded by the grid.
    if (alive) {
        for (int guard = B.hi[0] + B.hi[1] + B.hi[2] + 4; guard > 0; --guard) {
            const ExitFace X = exit_face(ax, true);
            if (X.s > s_cur) break;
            if (X.s >= R.s_end) {
                alive = false;
                break;
            }
            step_exact(R, X, V.inv_a[0], V.inv_a[1], V.inv_a[2], V.du[0], V.du[1], V.du[2], tab);
        }
    }
}

// Where the march of a ray may stop: at s_end, or past the last time that
// reaches a snapshot (u < -1).  Beyond that time no chord has a weight, so the
// bound only has to lie at or past it: it is taken a few float roundings late.
__device__ __forceinline__ float march_end(const RayState &R, float kk)
{
    const float c0 = fix_to_float(R.u_a, 1.0f / kTwo32);
    const float s_stop = kk > 0.f ? (c0 + 1.0f + 1e-6f * (fabsf(c0) + 1.0f)) / kk : 3.0e38f;
    return fminf(R.s_end, s_stop);
}

// Byte address of the unit of UNIT bytes (a record, or a pair of them) at layout
// offset `sum` of block `blk`, blocks blk_bytes apart.  The block term is one 64-bit
// product of bytes: the same address as (blk * units + sum) << log2(UNIT), in
// units of a shifted stride, came out with the stride shifted twice in some kernels (CUDA
// 13.0; their images matched that address and no other).
template <unsigned UNIT>
__device__ __forceinline__ unsigned long long rec_addr(unsigned long long base, int blk, long long blk_bytes,
                                                       uint32_t sum)
{
    return base + static_cast<unsigned long long>(static_cast<long long>(blk) * blk_bytes) +
           static_cast<unsigned long long>(sum) * UNIT;
}

// The float epoch coordinate of the bfloat16/float16 march: u(s) = c0 -
// kk s along the ray (s from the anchor), so that the chord midpoint's is
// c0 + mkk (s_cur + s_exit) with mkk = -kk / 2; the ray stops at the first
// crossing at or past s_lim, the nearer of the box face and the first float
// past s_stop = (c0 + 1) / kk, the last time that reaches a snapshot (u = -1).  c0 is the exact
// coordinate at the anchor rounded to float: the coordinate is off by at most
// a few float ulps of M (2e-6 snapshots at M = 16), against the 2^-9 and
// 2^-11 resolution of the stored j' and u.
struct EpochLine {
    float c0, mkk, s_lim;
};
__device__ __forceinline__ EpochLine epoch_line(const RayState &R, const ViewDev &V)
{
    EpochLine L;
    const float kk = V.kk_hi;
    L.c0 = fix_to_float(R.u_a, 1.0f / kTwo32);
    L.mkk = -0.5f * kk;
    L.s_lim = R.s_end;
    if (kk > 0.f) {
        const float s_stop = (L.c0 + 1.0f) / kk;
        // the next float up: s <= s_stop is s < next
        const int b = __float_as_int(s_stop);
        const float next = s_stop > 0.f ? __int_as_float(b + 1) : (s_stop < 0.f ? __int_as_float(b - 1) : FLT_MIN);
        L.s_lim = fminf(L.s_lim, next);
    }
    return L;
}

// floor(u) + 1 as an integer, and the fraction w = u - floor(u), on the FMA pipe:
// u + 1.5 * 2^23 rounded down holds floor(u) in its low mantissa bits for
// |u| < 2^22 (snapshot counts end at 10^6); for any other u the integer lies outside
// [0, 10^6], so a range test on it still fails.
__device__ __forceinline__ int floor_plus1(float u, float &w)
{
    const float t = __fadd_rd(u, 12582912.0f);
    w = u - (t - 12582912.0f);
    return static_cast<int>(static_cast<unsigned>(__float_as_int(t)) - 0x4B3FFFFFu);
}

// The march's loop.  A stage is some cells of every lane: gather() traverses them
// and issues the loads of their records, evaluate() boosts and sums them.  Two stages
// alternate, and each is evaluated after the next one has been gathered, so that its loads
// have the evaluation of the stage before and the traversal of the stage after to arrive
// in.  What bounds the march is waiting for its gathers (issue slots half used).
// Measured, cells gathered then evaluated / stages of one / of two (at most 80
// registers each): 24 views of 384^2 of 256^3 x 16 float32 2.93 / 2.81 / 2.49 ms, one
// 1024^2 image of 512^3 x 8 float32 1.50 / 1.44 / 1.41 ms, of paired
// bfloat16/float16 records 0.87 / 0.96 / 0.82 ms.
template <class Stage, class Gather, class Evaluate>
__device__ __forceinline__ void run_stages(const bool &alive, Gather gather, Evaluate evaluate)
{
    if (!__any_sync(kFull, alive)) return;
    Stage a, b;
    gather(a);
    while (__any_sync(kFull, alive)) {
        gather(b);
        evaluate(a);
        gather(a);
        evaluate(b);
    }
    evaluate(a);
}

// The march of march_ray for bfloat16/float16 records (see the file
// header): same cells, chords, midpoints and hat weights (Eqs. 2, 6-9, 19),
// with the epoch coordinate of EpochLine.  PLAIN: the Doppler factor in the
// plain form (volumes whose Gamma <= 8).
template <int H, bool PAIRED, bool PARTIAL, bool PLAIN>
__device__ __forceinline__ void march_ray_bf16(const VolDev &vol, const ViewDev &V, const RayBox &B, int p, int q,
                                               int width, int height, float *out_img, uint32_t *cnt_img,
                                               int *err_word, const int32_t *__restrict__ tab, bool accumulate)
{
    using Rec = Record<GBD_STORE_BF16_F16U>;
    const bool in_image = (p < width) && (q < height);
    RayState R;
    setup_ray(R, vol, V, B, p, q, in_image, V.win_lo, V.win_hi, tab);
    bool alive = R.alive;
    float s_cur = R.s_cur;
    const float ia0 = V.inv_a[0], ia1 = V.inv_a[1], ia2 = V.inv_a[2];
    const EpochLine L = epoch_line(R, V);
    const int M = vol.M;

    BoostConsts bc;
    bc.shx = V.sh_hi[0]; bc.shy = V.sh_hi[1]; bc.shz = V.sh_hi[2];
    bc.slx = V.sh_lo[0]; bc.sly = V.sh_lo[1]; bc.slz = V.sh_lo[2];
    bc.expo = V.expo;
    bc.beaming = (V.flags & GBD_BEAMING) != 0u;

    // Block b of the record array (paired: of record pairs) starts b es_bytes
    // from the base.  A sample's lower snapshot m_bar is bp - 1: unpaired, it
    // lies in block bp - 1 and the upper one in block bp; paired, both lie in
    // block bp.
    constexpr unsigned kUnit = PAIRED ? 16 : 8;
    const long long es_bytes = vol.epoch_stride * 8;
    const unsigned long long base = reinterpret_cast<unsigned long long>(vol.rec) - (PAIRED ? 0 : es_bytes);

    float acc = 0.f;
    uint32_t count = 0;
    struct Stage {
        float wgt[H], dsv[H];
        bool has[H];
        typename Rec::T rlo[H], rhi[H];
    };
    auto gather = [&](Stage &T) {
#pragma unroll
        for (int d = 0; d < H; ++d) {
            // the nearest face, the chord, and the epoch coordinate at the
            // chord midpoint: m_bar + w
            const ExitFace X = exit_face(R.ax, alive);
            const float ds = X.s - s_cur;
            const float um = fmaf(L.mkk, s_cur + X.s, L.c0);
            float w;
            const int bp = floor_plus1(um, w);
            // -1 <= m_bar <= M - 1; snapshots m_bar (weight 1 - w) and m_bar + 1 (w)
            const bool take = alive & (ds > 0.f) & (static_cast<unsigned>(bp) <= static_cast<unsigned>(M));
            bool has_lo = take & (bp != 0);
            bool has_hi = take & (bp < M) & (w != 0.f);
#ifdef GBD_CHECKED
            if ((has_lo && !check_cell(vol, err_word, R.kc[0], R.kc[1], R.kc[2], bp - 1)) ||
                (has_hi && !check_cell(vol, err_word, R.kc[0], R.kc[1], R.kc[2], bp)))
                has_lo = has_hi = false;
#endif
            const unsigned long long pa = rec_addr<kUnit>(base, bp, es_bytes, R.sum);
            T.wgt[d] = take ? w : 0.f;
            T.dsv[d] = take ? ds : 0.f;
            T.has[d] = has_lo | has_hi;
            T.rlo[d] = Rec::zero();
            T.rhi[d] = Rec::zero();
            if (PAIRED) {
                if (has_lo | has_hi) Rec::load_pair_at(pa, T.rlo[d], T.rhi[d]);
            } else {
                if (has_lo) T.rlo[d] = Rec::load_at(pa);
                if (has_hi) T.rhi[d] = Rec::load_at(pa + es_bytes);
            }
            step_lite(R, X, ia0, ia1, ia2, tab);
            s_cur = X.s;
            alive = alive & (X.s < L.s_lim);
        }
    };
    // A snapshot a sample does not read is a zero record (boosted value
    // exactly 0), and a sample not taken has weight and chord 0.
    auto evaluate = [&](const Stage &T) {
#pragma unroll
        for (int d = 0; d < H; ++d) {
            const float2 vv = PLAIN ? Rec::boosted2_plain(T.rlo[d], T.rhi[d], bc) : Rec::boosted2(T.rlo[d], T.rhi[d], bc);
            const float v = fmaf(T.wgt[d], vv.y - vv.x, vv.x);  // Eq. 8
            acc = fmaf(v, T.dsv[d], acc);
            count += T.has[d] ? 1u : 0u;
        }
    };
    run_stages<Stage>(alive, gather, evaluate);

    if (in_image) {
        const long long pix = static_cast<long long>(q) * width + p;
        if (PARTIAL) {
            if (count > 0u) atomicAdd(out_img + pix, acc);
        } else if (accumulate) {
            out_img[pix] += V.prefactor * acc;
            if (cnt_img) cnt_img[pix] += count;
        } else {
            out_img[pix] = V.prefactor * acc;
            if (cnt_img) cnt_img[pix] = count;
        }
    }
}

// Marches the ray of pixel (p, q) of one image through box B.  Direct
// (PARTIAL false): stores the pixel value (Eq. 19, with the prefactor) and,
// if cnt_img is set, its cell-sample count, or adds them to what is there
// when `accumulate` is set (one thread owns each pixel, so the adds of
// successive launches land in launch order).  PARTIAL: adds the ray's sum over
// the box, without the prefactor, to out_img[pixel] if the ray sampled at
// least one cell there (one region per slot and ray, so the add lands on
// zero).  tab points at the march tables in shared memory.
//
// NCH > 0 (vector renders, Sec. 2.1): the volume carries NCH more emissivity
// channels sharing its velocity; each is summed with the same weights and
// Doppler factors as j' (Eq. 19 per channel) into component c + 1 of the
// pixel, at out_img + (c + 1) * width * height.
//
// TOUCH (memory analysis, not a render): instead of reading the two records
// of a sample, set the bits of (snapshot, cell) in the bitmap `touch`, whose
// bit m * cell_stride + cell stands for that record.
struct ChanPtrs {
    const float *chan;
    long long comp_stride, cell_stride;
    uint32_t *touch;
};

// The march without branches (every lane executes each step; a lane whose ray
// has ended takes no step and reads no record), with the exact Q31.32 epoch
// coordinate, the records' own Doppler factor and compensated sums: float32
// records, and the vector and memory-analysis forms of both stores.
template <int STORE, int H, bool PAIRED, bool PARTIAL, int NCH, bool TOUCH>
__device__ __forceinline__ void march_ray_exact(const VolDev &vol, const ViewDev &V, const RayBox &B, int p, int q,
                                                int width, int height, float *out_img, uint32_t *cnt_img,
                                                int *err_word, const int32_t *__restrict__ tab, bool accumulate,
                                                const ChanPtrs ch)
{
    using Rec = Record<STORE>;
    const bool in_image = (p < width) && (q < height);
    RayState R;
    setup_ray(R, vol, V, B, p, q, in_image, V.win_lo, V.win_hi, tab);
    bool alive = R.alive;
    float s_cur = R.s_cur;
    long long u_cur = R.u_cur;
    const float s_lim = march_end(R, V.kk_hi);
    const float ia0 = V.inv_a[0], ia1 = V.inv_a[1], ia2 = V.inv_a[2];
    const long long du0 = V.du[0], du1 = V.du[1], du2 = V.du[2];
    const int M = vol.M;
    BoostConsts bc;
    bc.shx = V.sh_hi[0]; bc.shy = V.sh_hi[1]; bc.shz = V.sh_hi[2];
    bc.slx = V.sh_lo[0]; bc.sly = V.sh_lo[1]; bc.slz = V.sh_lo[2];
    bc.expo = V.expo;
    bc.beaming = (V.flags & GBD_BEAMING) != 0u;
    // blocks and records as in march_ray_bf16.  Paired float32: a sample that
    // reads no snapshot loads the zero record pair after the last block
    // (faster for 32-byte pairs than a predicated load).
    constexpr unsigned kRec = STORE == GBD_STORE_F32 ? 16 : 8;
    constexpr unsigned kUnit = PAIRED ? 2 * kRec : kRec;
    constexpr bool kZeroPair = PAIRED && STORE == GBD_STORE_F32;
    const long long es_bytes = vol.epoch_stride * kRec;
    const unsigned long long recb = reinterpret_cast<unsigned long long>(vol.rec);
    const unsigned long long base = recb - (PAIRED ? 0 : es_bytes);
    const unsigned long long zero_addr = recb + static_cast<unsigned long long>((vol.M + 1) * es_bytes);

    float acc = 0.f, comp = 0.f;
    uint32_t count = 0;
    constexpr int kNch = NCH > 0 ? NCH : 1;
    float cacc[kNch], ccomp[kNch];
#pragma unroll
    for (int c = 0; c < kNch; ++c) cacc[c] = ccomp[c] = 0.f;

    struct Stage {
        float wgt[H], dsv[H];
        bool has[H];
        typename Rec::T rlo[H], rhi[H];
        float clo[H][kNch], chi[H][kNch];
    };
    auto gather = [&](Stage &T) {
#pragma unroll
        for (int d = 0; d < H; ++d) {
            const ExitFace X = exit_face(R.ax, alive);
            const long long u_exit = X.x0 ? R.ax[0].un : (X.x1 ? R.ax[1].un : R.ax[2].un);
            const float ds = X.s - s_cur;
            // epoch coordinate at the chord midpoint: m_bar + w, w in [0, 1)
            const long long um = (u_cur + u_exit) >> 1;
            const int bp = static_cast<int>(um >> 32) + 1;
            const uint32_t frac = static_cast<uint32_t>(um);
            // -1 <= m_bar <= M - 1 (at u = -1 exactly both weights vanish)
            const bool take = alive & (ds > 0.f) & (static_cast<unsigned>(bp) <= static_cast<unsigned>(M));
            bool has_lo = take & (bp != 0);
            bool has_hi = take & (bp < M) & (frac != 0u);
#ifdef GBD_CHECKED
            if ((has_lo && !check_cell(vol, err_word, R.kc[0], R.kc[1], R.kc[2], bp - 1)) ||
                (has_hi && !check_cell(vol, err_word, R.kc[0], R.kc[1], R.kc[2], bp)))
                has_lo = has_hi = false;
#endif
            T.wgt[d] = static_cast<float>(frac) * 2.3283064365386963e-10f;
            T.dsv[d] = ds;
            T.has[d] = has_lo | has_hi;
            if constexpr (TOUCH) {
                const long long bit = static_cast<long long>(bp - 1) * ch.cell_stride + R.sum;
                if (has_lo) atomicOr(ch.touch + (bit >> 5), 1u << (bit & 31));
                if (has_hi) {
                    const long long i = bit + ch.cell_stride;
                    atomicOr(ch.touch + (i >> 5), 1u << (i & 31));
                }
            } else {
                const unsigned long long a = rec_addr<kUnit>(base, bp, es_bytes, R.sum);
                if constexpr (kZeroPair) {
                    const unsigned long long pa = T.has[d] ? a : zero_addr;
                    T.rlo[d] = Rec::load_at(pa);
                    T.rhi[d] = Rec::load_at(pa + kRec);
                } else if constexpr (PAIRED) {
                    T.rlo[d] = Rec::zero();
                    T.rhi[d] = Rec::zero();
                    if (has_lo | has_hi) Rec::load_pair_at(a, T.rlo[d], T.rhi[d]);
                } else {
                    T.rlo[d] = has_lo ? Rec::load_at(a) : Rec::zero();
                    T.rhi[d] = has_hi ? Rec::load_at(a + es_bytes) : Rec::zero();
                }
            }
            if constexpr (NCH > 0) {
                const float *cp = ch.chan + (static_cast<long long>(bp - 1) * ch.cell_stride + R.sum);
#pragma unroll
                for (int c = 0; c < NCH; ++c, cp += ch.comp_stride) {
                    T.clo[d][c] = has_lo ? __ldg(cp) : 0.f;
                    T.chi[d][c] = has_hi ? __ldg(cp + ch.cell_stride) : 0.f;
                }
            }
            step_exact(R, X, ia0, ia1, ia2, du0, du1, du2, tab);
            s_cur = X.s;
            u_cur = u_exit;
            alive = alive & (X.s < s_lim);
        }
    };
    // A snapshot the sample does not read is a zero record (boosted value
    // exactly 0); the compensated sums take the sample only where it read
    // one, so a ray's sum does not depend on how long the other lanes of
    // its warp march.
    auto evaluate = [&](const Stage &T) {
        if constexpr (TOUCH) return;
#pragma unroll
        for (int d = 0; d < H; ++d) {
            const bool take = T.has[d];
            const float blo = Rec::boost(T.rlo[d], bc), bhi = Rec::boost(T.rhi[d], bc);
            const float vlo = __fmul_rn(Rec::emissivity(T.rlo[d]), blo);
            const float v = fmaf(T.wgt[d], fmaf(Rec::emissivity(T.rhi[d]), bhi, -vlo), vlo);  // Eq. 8
            const float y = fmaf(v, T.dsv[d], -comp);
            const float t = acc + y;
            comp = take ? (t - acc) - y : comp;
            acc = take ? t : acc;
            count += take ? 1u : 0u;
            if constexpr (NCH > 0) {
                // the Doppler factor of each snapshot serves every channel
#pragma unroll
                for (int c = 0; c < NCH; ++c) {
                    const float ulo = T.clo[d][c] * blo, uhi = T.chi[d][c] * bhi;
                    const float u = fmaf(T.wgt[d], uhi - ulo, ulo);
                    const float yc = fmaf(u, T.dsv[d], -ccomp[c]);
                    const float tc = cacc[c] + yc;
                    ccomp[c] = take ? (tc - cacc[c]) - yc : ccomp[c];
                    cacc[c] = take ? tc : cacc[c];
                }
            }
        }
    };
    run_stages<Stage>(alive, gather, evaluate);
    if (in_image && !TOUCH) {
        const long long pix = static_cast<long long>(q) * width + p;
        if (PARTIAL) {
            if (count > 0u) atomicAdd(out_img + pix, acc);
        } else if (accumulate) {
            out_img[pix] += V.prefactor * acc;
            if (cnt_img) cnt_img[pix] += count;
        } else {
            out_img[pix] = V.prefactor * acc;
            if (cnt_img) cnt_img[pix] = count;
        }
        if constexpr (NCH > 0) {
            const long long plane = static_cast<long long>(width) * height;
#pragma unroll
            for (int c = 0; c < NCH; ++c) out_img[(c + 1) * plane + pix] = V.prefactor * cacc[c];
        }
    }
}

template <int STORE, int H, bool PAIRED, bool PARTIAL = false, int NCH = 0, bool TOUCH = false>
__device__ __forceinline__ void march_ray(const VolDev &vol, const ViewDev &V, const RayBox &B, int p, int q,
                                          int width, int height, float *out_img, uint32_t *cnt_img, int *err_word,
                                          const int32_t *__restrict__ tab, bool accumulate = false,
                                          const ChanPtrs ch = ChanPtrs{nullptr, 0, 0, nullptr})
{
    if constexpr (STORE == GBD_STORE_BF16_F16U && NCH == 0 && !TOUCH) {
        if (vol.plain_boost)
            march_ray_bf16<H, PAIRED, PARTIAL, true>(vol, V, B, p, q, width, height, out_img, cnt_img, err_word,
                                                         tab, accumulate);
        else
            march_ray_bf16<H, PAIRED, PARTIAL, false>(vol, V, B, p, q, width, height, out_img, cnt_img, err_word,
                                                          tab, accumulate);
    } else {
        march_ray_exact<STORE, H, PAIRED, PARTIAL, NCH, TOUCH>(vol, V, B, p, q, width, height, out_img, cnt_img,
                                                                   err_word, tab, accumulate, ch);
    }
}

// Time groups (batched renders).  Views that differ only in observer time
// (and so in window and prefactor) share their rays; one lane marches its ray
// once for up to kGroupMax such views.  The traversal covers the union of the
// members' windows and carries the epoch coordinate of the reference member,
// the one whose window ends last (largest u_obs); member g's coordinate
// differs from it by the exact constant Delta_g = u_obs,g - u_obs,ref <= 0
// (Q31.32), so at a chord midpoint it is um + Delta_g.
//
// The members also share the snapshots.  Their coordinates lie within S - 2
// snapshots of each other (the host's grouping rule), so the two snapshots
// that any member interpolates between are among the S from the reference's
// upper one, m_0 = floor(um) + 1, down to m_0 - S + 1.  Per cell those S records
// are gathered and boosted once, and each member only picks its pair, forms
// its hat weight and adds to its own sum (Eq. 19 per view).  Snapshots that no
// member of the lane reaches are not read.
//
// What bounds it: instruction issue, as for the lone march.  A cell costs the
// traversal once, S records of about 16 (float32) or 8 (bfloat16/float16)
// instructions of boost, and about 18 or 13 per member, where the members once
// gathered and boosted two records each (18 images of 512^2 of a 256^3 x 16
// series, groups of three: float32 892 -> 580 us, bfloat16/float16 600 -> 428).
//
// A member's pixel is summed over the same cells, chords, midpoints and
// boosted values as when its view is marched alone; the crossings are measured
// from the group's anchor instead of the view's own, so the two agree to float
// rounding, not bit for bit.  Member g's image is at out + g * img_stride.
// GD cells are traversed per iteration, and all their records gathered before
// any is evaluated.
template <int STORE, int GD, int G, int S, bool PLAIN>
__device__ __forceinline__ void march_group(const VolDev &vol, const ViewDev &V, float win_lo, float win_hi,
                                            const ViewDev *GV, const long long *dl, int gcnt, const RayBox &B, int p,
                                            int q, int width, int height, float *out, long long img_stride,
                                            uint32_t *cnt_img, int *err_word, const int32_t *__restrict__ tab)
{
    constexpr bool kF32 = STORE == GBD_STORE_F32;
    using Rec = Record<STORE>;
    const bool in_image = (p < width) && (q < height);
    RayState R;
    setup_ray(R, vol, V, B, p, q, in_image, win_lo, win_hi, tab);
    bool alive = R.alive;
    float s_cur = R.s_cur;
    long long u_cur = R.u_cur;
    const float ia0 = V.inv_a[0], ia1 = V.inv_a[1], ia2 = V.inv_a[2];
    const long long du0 = V.du[0], du1 = V.du[1], du2 = V.du[2];
    const EpochLine L = epoch_line(R, V);
    const float s_lim = kF32 ? march_end(R, V.kk_hi) : L.s_lim;
    const int M = vol.M;

    BoostConsts bc;
    bc.shx = V.sh_hi[0]; bc.shy = V.sh_hi[1]; bc.shz = V.sh_hi[2];
    bc.slx = V.sh_lo[0]; bc.sly = V.sh_lo[1]; bc.slz = V.sh_lo[2];
    bc.expo = V.expo;
    bc.beaming = (V.flags & GBD_BEAMING) != 0u;

    // Unpaired, snapshot m is a record of block m.  Paired, block m holds the
    // records of m - 1 and m side by side: of the snapshots m_0 - k, the even k
    // are the second records of blocks m_0 - k and the odd k the first ones of
    // blocks m_0 - k + 1, so that neighbours share a sector.  Either way the record of
    // m_0 - k lies (k & 1) odd_bytes + (k & ~1) blk_bytes below that of m_0.
    constexpr unsigned kRec = kF32 ? 16 : 8;
    const long long blk_bytes = vol.epoch_stride * kRec;
    const long long odd_bytes = vol.paired ? kRec : blk_bytes;
    const int cell_shift = vol.paired ? 1 : 0;
    const unsigned long long recb = reinterpret_cast<unsigned long long>(vol.rec) + (vol.paired ? kRec : 0u);

    float dlf[G];  // Delta_g as a float (bfloat16/float16 march)
    float acc[G], comp[G];
    uint32_t count[G];
#pragma unroll
    for (int g = 0; g < G; ++g) {
        dlf[g] = (!kF32 && g < gcnt) ? fix_to_float(dl[g], 1.0f / kTwo32) : 0.f;
        acc[g] = comp[g] = 0.f;
        count[g] = 0u;
    }
    long long dl_min = 0;  // the earliest member's
    for (int g = 0; g < gcnt; ++g) dl_min = min(dl_min, dl[g]);
    const float dlf_min = fix_to_float(dl_min, 1.0f / kTwo32);

    while (__any_sync(kFull, alive)) {
        long long umx[GD];          // the reference's epoch coordinate at the chord midpoints (float32 march)
        float umf[GD], dsv[GD];     // the same (bfloat16/float16 march), and the chords (0 where there is none)
        typename Rec::T rec[GD][S];  // snapshots m_0, m_0 - 1, ... of each cell
        bool pos[GD];
#pragma unroll
        for (int d = 0; d < GD; ++d) {
            const ExitFace X = exit_face(R.ax, alive);
            const float ds = X.s - s_cur;
            pos[d] = alive && ds > 0.f;
            dsv[d] = pos[d] ? ds : 0.f;
            int top, low;  // m_0, and the lowest snapshot that a member reaches
            long long u_exit = 0;
            if constexpr (kF32) {
                u_exit = X.x0 ? R.ax[0].un : (X.x1 ? R.ax[1].un : R.ax[2].un);
                umx[d] = (u_cur + u_exit) >> 1;
                top = static_cast<int>(umx[d] >> 32) + 1;
                low = static_cast<int>((umx[d] + dl_min) >> 32);
            } else {
                umf[d] = fmaf(L.mkk, s_cur + X.s, L.c0);
                top = static_cast<int>(floorf(umf[d])) + 1;
                low = static_cast<int>(floorf(umf[d] + dlf_min));
            }
            const unsigned long long at = rec_addr<kRec>(recb, top, blk_bytes, R.sum << cell_shift);
#pragma unroll
            for (int k = 0; k < S; ++k) {
                const int m = top - k;
                bool want = pos[d] && static_cast<unsigned>(m) < static_cast<unsigned>(M) && m >= low;
#ifdef GBD_CHECKED
                if (want && !check_cell(vol, err_word, R.kc[0], R.kc[1], R.kc[2], m)) want = false;
#endif
                rec[d][k] = Rec::zero();
                if (want) rec[d][k] = Rec::load_at(at - static_cast<unsigned long long>((k & 1) * odd_bytes + (k & ~1) * blk_bytes));
            }
            if constexpr (kF32) {
                step_exact(R, X, ia0, ia1, ia2, du0, du1, du2, tab);
                u_cur = u_exit;
            } else {
                step_lite(R, X, ia0, ia1, ia2, tab);
            }
            s_cur = X.s;
            alive = alive & (X.s < s_lim);
        }
        // boosted value of each snapshot (0 of one not read), and its difference
        // from the next lower one, as the lone march forms them
        float b[GD][S], dif[GD][S - 1];
        if constexpr (kF32) {
#pragma unroll
            for (int d = 0; d < GD; ++d) {
                float bk[S];
#pragma unroll
                for (int k = 0; k < S; ++k) {
                    bk[k] = Rec::boost(rec[d][k], bc);
                    b[d][k] = __fmul_rn(Rec::emissivity(rec[d][k]), bk[k]);
                }
#pragma unroll
                for (int k = 0; k < S - 1; ++k) dif[d][k] = fmaf(Rec::emissivity(rec[d][k]), bk[k], -b[d][k + 1]);
            }
        } else {
            // two records at a time, over all cells
#pragma unroll
            for (int i = 0; i < GD * S; i += 2) {
                const int d0 = i / S, k0 = i % S, d1 = (i + 1) / S, k1 = (i + 1) % S;
                const typename Rec::T r1 = i + 1 < GD * S ? rec[d1 < GD ? d1 : 0][k1] : Rec::zero();
                const float2 vv = PLAIN ? Rec::boosted2_plain(rec[d0][k0], r1, bc) : Rec::boosted2(rec[d0][k0], r1, bc);
                b[d0][k0] = vv.x;
                if (i + 1 < GD * S) b[d1 < GD ? d1 : 0][k1] = vv.y;
            }
#pragma unroll
            for (int d = 0; d < GD; ++d)
#pragma unroll
                for (int k = 0; k < S - 1; ++k) dif[d][k] = b[d][k] - b[d][k + 1];
        }
#pragma unroll
        for (int d = 0; d < GD; ++d) {
#pragma unroll
            for (int g = 0; g < G; ++g) {
                if (g >= gcnt) break;  // uniform
                // member g's lower snapshot is m_0 - 1 - k: b[k + 1], its pair's difference dif[k]
                float w, lower = b[d][1], up = dif[d][0];
                bool take;
                if constexpr (kF32) {
                    const long long ug = umx[d] + dl[g];
                    const uint32_t frac = static_cast<uint32_t>(ug);
                    const int mb = static_cast<int>(ug >> 32), m0 = static_cast<int>(umx[d] >> 32);
                    w = static_cast<float>(frac) * 2.3283064365386963e-10f;
                    // -1 <= m_bar <= M - 1 (at u = -1 exactly both weights vanish)
                    take = pos[d] && static_cast<unsigned>(mb + 1) <= static_cast<unsigned>(M) && (mb >= 0 || frac != 0u);
#pragma unroll
                    for (int k = 1; k < S - 1; ++k) {
                        lower = mb <= m0 - k ? b[d][k + 1] : lower;
                        up = mb <= m0 - k ? dif[d][k] : up;
                    }
                    const float v = fmaf(w, up, lower);  // Eq. 8
                    const float y = fmaf(v, dsv[d], -comp[g]);      // compensated sum
                    const float t = acc[g] + y;
                    comp[g] = take ? (t - acc[g]) - y : comp[g];
                    acc[g] = take ? t : acc[g];
                } else {
                    const float ug = umf[d] + dlf[g];
                    const float fl = floorf(ug), f0 = floorf(umf[d]);
                    w = ug - fl;
                    take = pos[d] && fl >= -1.0f && fl <= static_cast<float>(M - 1) && (fl >= 0.f || w != 0.f);
#pragma unroll
                    for (int k = 1; k < S - 1; ++k) {
                        lower = fl <= f0 - static_cast<float>(k) ? b[d][k + 1] : lower;
                        up = fl <= f0 - static_cast<float>(k) ? dif[d][k] : up;
                    }
                    const float v = fmaf(w, up, lower);  // Eq. 8
                    acc[g] = fmaf(take ? v : 0.f, dsv[d], acc[g]);
                }
                count[g] += take ? 1u : 0u;
            }
        }
    }

    if (in_image) {
        const long long pix = static_cast<long long>(q) * width + p;
#pragma unroll
        for (int g = 0; g < G; ++g) {
            if (g >= gcnt) break;
            out[g * img_stride + pix] = GV[g].prefactor * acc[g];
            if (cnt_img) cnt_img[g * img_stride + pix] = count[g];
        }
    }
}

// The pixel of this lane in block `block` of an image.
__device__ __forceinline__ void block_pixel(const PacketGrid &g, int blocks_x, int block, int &p, int &q)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int by = block / blocks_x, bx = block - by * blocks_x;
    const int wy = warp / g.block_w, wx = warp - wy * g.block_w;
    const int ly = lane / g.packet_w, lx = lane - ly * g.packet_w;
    p = bx * g.step_x + wx * g.packet_w + lx;
    q = by * g.step_y + wy * g.packet_h + ly;
}

// The march kernels' work split: one CTA per block of packets of one view (or
// time group), one packet per warp, and the CTAs of the launch run after run (set_runs).  The
// hardware hands out CTAs as they end, which balances the load by itself, and the
// rays of a CTA share cells in L1 (against persistent CTAs pulling packets from
// per-view counters: 24 views of 384^2 of 256^3 x 16 float32 3.09 -> 2.53
// ms, one 1024^2 image of 512^3 x 8 1.60 -> 1.47 ms).  The view index comes
// from the CTA index alone, so every per-view constant stays uniform.
// RUNS: the units of a run (set_runs) go side by side, block by block, instead of one
// after the other.  bfloat16/float16 groups go without: 18 images of 512^2 of a
// 256^3 x 16 series 431 us, with 477.
struct BlockWork {
    int unit;   // view, or time group
    int block;  // of its image
};
template <bool RUNS>
__device__ __forceinline__ BlockWork block_work(const MarchArgs &a)
{
    BlockWork w;
    const int b = static_cast<int>(blockIdx.x);
    w.unit = b / a.pk.blocks;
    if (RUNS) {
        const int first = a.run_first[w.unit], len = a.run_len[w.unit];
        const int i = b - first * a.pk.blocks;
        w.block = i / len;
        w.unit = first + i - w.block * len;
    } else {
        w.block = b - w.unit * a.pk.blocks;
    }
    if (a.block_order) {
        w.block = __ldg(a.block_order + w.block);
    } else if (RUNS && a.rows_from_middle) {
        // rows of blocks m, m - 1, m + 1, m - 2, ... from the middle one, m
        const int row = w.block / a.pk.blocks_x, half = (row + 1) >> 1;
        const int to = ((a.pk.blocks / a.pk.blocks_x) >> 1) + ((row & 1) ? -half : half);
        w.block += (to - row) * a.pk.blocks_x;
    }
    return w;
}

// MINB = 1 leaves the register count to the compiler; MINB = 3 asks for
// three 256-thread CTAs per SM (at most 80 registers per thread).
template <int STORE, int H, int MINB, bool PAIRED>
__global__ void __launch_bounds__(256, MINB) march_kernel(const __grid_constant__ MarchArgs a)
{
    extern __shared__ int32_t s_mem[];
    int32_t *s_tab = s_mem + kSpanEntries;
    const BlockWork w = block_work<true>(a);
    const ViewDev &V = a.views[w.unit];
    const long long img = w.unit * (a.img_stride ? a.img_stride : static_cast<long long>(a.width) * a.height);
    int p, q;
    block_pixel(a.pk, a.pk.blocks_x, w.block, p, q);
    stage_tables(s_tab, a.vol, V, p, q, p < a.width && q < a.height, V.win_lo, V.win_hi);
    march_ray<STORE, H, PAIRED>(a.vol, V, grid_box(a.vol, V), p, q, a.width, a.height, a.out + img,
                                    a.samples ? a.samples + img : nullptr, a.error_word, s_tab, a.accumulate != 0);
}

// Time groups: march_kernel's work split over groups of views instead of
// single views (group g is views group_first[g] .. group_first[g + 1] - 1).
// DEPTH cells per iteration, S snapshots per cell, at most 80 registers.
// SPANS: with tables too long to be copied whole (stage_spans).  A kernel of its own: the
// call costs the others registers (bfloat16/float16 series of 18 images 434 -> 491 us).
template <int STORE, int DEPTH, int G, int S, bool SPANS>
__global__ void __launch_bounds__(256, 3) group_kernel(const __grid_constant__ MarchArgs a)
{
    extern __shared__ int32_t s_mem[];
    int32_t *s_tab = s_mem + kSpanEntries;
    if constexpr (!SPANS) stage_all(s_tab, a.vol);
    const BlockWork w = block_work<STORE == GBD_STORE_F32>(a);
    const int first = a.group_first[w.unit];
    const int gcnt = a.group_first[w.unit + 1] - first;
    const ViewDev &V = a.views[a.group_ref[w.unit]];
    const long long stride = a.img_stride ? a.img_stride : static_cast<long long>(a.width) * a.height;
    int p, q;
    block_pixel(a.pk, a.pk.blocks_x, w.block, p, q);
    if constexpr (SPANS)
        stage_spans(s_tab, a.vol, V, p, q, p < a.width && q < a.height, a.group_win[w.unit][0], a.group_win[w.unit][1]);
    auto march = [&](auto plain) {
        march_group<STORE, DEPTH, G, S, decltype(plain)::value>(
            a.vol, V, a.group_win[w.unit][0], a.group_win[w.unit][1], a.views + first, a.view_delta + first, gcnt,
            grid_box(a.vol, V), p, q, a.width, a.height, a.out + first * stride, stride,
            a.samples ? a.samples + first * stride : nullptr, a.error_word, s_tab);
    };
    if constexpr (STORE == GBD_STORE_F32) {
        march(std::false_type{});
    } else {
        if (a.vol.plain_boost) march(std::true_type{});
        else march(std::false_type{});
    }
}

// Vector renders: march_kernel's work split with NCH extra channels summed
// along every ray (stages of one cell, at most 96 registers: six views of 384^2 of
// 192^3 x 8 with three channels 878 us at the compiler's 106, 854 at 96, 897 at 80).
// RUNS: side by side (set_runs) for launches of kRunsPixels and more; below, the run's arithmetic
// costs each ray's latency more than the order gains (three channels of 3 views of 64^2 of 160^3
// 182 us without, 191 with; of 4 of 192^2 327 and 271).
constexpr long long kRunsPixels = 1 << 17;
template <int STORE, int NCH, bool PAIRED, bool RUNS>
__global__ void __maxnreg__(96) vector_kernel(const __grid_constant__ MarchArgs a)
{
    extern __shared__ int32_t s_mem[];
    int32_t *s_tab = s_mem + kSpanEntries;
    const BlockWork w = block_work<RUNS>(a);
    const ViewDev &V = a.views[w.unit];
    int p, q;
    block_pixel(a.pk, a.pk.blocks_x, w.block, p, q);
    stage_tables(s_tab, a.vol, V, p, q, p < a.width && q < a.height, V.win_lo, V.win_hi);
    const ChanPtrs ch{a.chan, a.chan_comp_stride, a.chan_cell_stride, nullptr};
    march_ray<STORE, 1, PAIRED, false, NCH>(a.vol, V, grid_box(a.vol, V), p, q, a.width, a.height,
                                            a.out + w.unit * a.img_stride, nullptr, a.error_word, s_tab, false, ch);
}

// Memory analysis: marks every (snapshot, cell) record the views' samples
// read.
template <int STORE, bool PAIRED>
__global__ void __launch_bounds__(256, 1) touch_kernel(const __grid_constant__ MarchArgs a, uint32_t *bits,
                                                        long long cells)
{
    extern __shared__ int32_t s_mem[];
    int32_t *s_tab = s_mem + kSpanEntries;
    const BlockWork w = block_work<false>(a);
    const ViewDev &V = a.views[w.unit];
    int p, q;
    block_pixel(a.pk, a.pk.blocks_x, w.block, p, q);
    stage_tables(s_tab, a.vol, V, p, q, p < a.width && q < a.height, V.win_lo, V.win_hi);
    const ChanPtrs ch{nullptr, 0, cells, bits};
    march_ray<STORE, 1, PAIRED, false, 0, true>(a.vol, V, grid_box(a.vol, V), p, q, a.width, a.height, a.out, nullptr,
                                                a.error_word, s_tab, false, ch);
}

// Serving: one launch over the tiles of many requests, each with its own
// volume (float32 or bfloat16/float16 records), view and image.  A CTA finds
// its request by binary search over the requests' first CTAs (uniform across
// the CTA) and stages that request's march tables in shared memory (sized for
// the largest volume of the launch); every ray runs the same march_ray as the
// single-volume kernel, so a request's pixels are the same whether it is
// served alone or in a mix.
template <int H, int MINB>
__global__ void __launch_bounds__(256, MINB) wave_kernel(const __grid_constant__ WaveArgs a)
{
    extern __shared__ int32_t s_mem[];
    int32_t *s_tab = s_mem + kSpanEntries;
    const int b = static_cast<int>(blockIdx.x);
    int lo = 0, hi = a.n_reqs - 1;  // last request whose first CTA is <= b
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (a.reqs[mid].cta_begin <= b) lo = mid;
        else hi = mid - 1;
    }
    const ReqDev &R = a.reqs[lo];
    int p, q;
    block_pixel(a.pk, R.blocks_x, b - R.cta_begin, p, q);
    stage_tables(s_tab, R.vol, R.view, p, q, p < R.width && q < R.height, R.view.win_lo, R.view.win_hi);
    const RayBox box = grid_box(R.vol, R.view);
    if (R.vol.store == GBD_STORE_F32) {
        if (R.vol.paired)
            march_ray<GBD_STORE_F32, H, true>(R.vol, R.view, box, p, q, R.width, R.height, R.out, R.samples,
                                                        a.error_word, s_tab);
        else
            march_ray<GBD_STORE_F32, H, false>(R.vol, R.view, box, p, q, R.width, R.height, R.out, R.samples,
                                                         a.error_word, s_tab);
    } else {
        if (R.vol.paired)
            march_ray<GBD_STORE_BF16_F16U, H, true>(R.vol, R.view, box, p, q, R.width, R.height, R.out,
                                                              R.samples, a.error_word, s_tab);
        else
            march_ray<GBD_STORE_BF16_F16U, H, false>(R.vol, R.view, box, p, q, R.width, R.height, R.out,
                                                               R.samples, a.error_word, s_tab);
    }
}

// Region schedule (RegionArgs): CTA (x, y) marches rays of one view through
// region y.  The region's table entries along each axis (forward or reversed,
// as the view needs) are staged in shared memory.
// The view's pixels whose rays can cross the region lie in the projection of
// the region's box; screen_kernel lists them, longest chord first, and each warp takes
// the next 32 of the list, so that its rays end at about the same step.  Each ray adds
// its region sum to its partial slot.
// Region r of view vi: its box in the view's march frame (mirrored axes
// mirrored) with the offsets of its staged march tables, its partial slot, and
// the pixels p_lo .. p_lo + pw - 1, q_lo .. q_lo + qh - 1 of the image that
// hold every pixel whose centre projects into the box, with a pixel of margin
// (pw = qh = 0 if none).
struct RegionFrame {
    RayBox B;
    int slot;
    int p_lo, q_lo, pw, qh;
};

__device__ __forceinline__ RegionFrame region_frame(const RegionArgs &a, int vi, int r)
{
    const ViewDev &V = a.views[vi];
    const RegionProj &P = a.proj[vi];
    const int rr[3] = {r % a.nreg[0], (r / a.nreg[0]) % a.nreg[1], r / (a.nreg[0] * a.nreg[1])};
    RegionFrame F;
    F.slot = 0;
    float pc = P.p0, qc = P.q0, hp = 0.f, hq = 0.f;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const int n = a.vol.n[i];
        const int olo = rr[i] * a.region;
        const int ohi = min(olo + a.region, n);
        const bool mirrored = (V.flags & (kFlagMirror0 << i)) != 0u;
        F.B.lo[i] = mirrored ? n - ohi : olo;
        F.B.hi[i] = mirrored ? n - olo : ohi;
        F.B.cur0[i] = 4u * static_cast<uint32_t>(i * (a.region + 1));
        F.slot += mirrored ? a.nreg[i] - 1 - rr[i] : rr[i];
        const float c = 0.5f * static_cast<float>(F.B.lo[i] + F.B.hi[i]);
        const float h = 0.5f * static_cast<float>(F.B.hi[i] - F.B.lo[i]);
        pc = fmaf(P.ip[i], c, pc);
        qc = fmaf(P.iq[i], c, qc);
        hp = fmaf(fabsf(P.ip[i]), h, hp);
        hq = fmaf(fabsf(P.iq[i]), h, hq);
    }
    const int p_lo = max(static_cast<int>(floorf(pc - hp)) - 1, 0);
    const int p_hi = min(static_cast<int>(floorf(pc + hp)) + 1, a.width - 1);
    const int q_lo = max(static_cast<int>(floorf(qc - hq)) - 1, 0);
    const int q_hi = min(static_cast<int>(floorf(qc + hq)) + 1, a.height - 1);
    const bool any = p_hi >= p_lo && q_hi >= q_lo;
    F.p_lo = p_lo;
    F.q_lo = q_lo;
    F.pw = any ? p_hi - p_lo + 1 : 0;
    F.qh = any ? q_hi - q_lo + 1 : 0;
    return F;
}

// Chord classes of the ray lists: class 0 holds the longest chords.
constexpr int kChordClasses = 64;
// Warps per CTA of screen_kernel, and the candidates a warp classifies per
// pass (a byte each in shared memory).
constexpr int kScreenWarps = 8;
constexpr int kScreenBatch = 2048;

// Ray lists of the region schedule, one warp per view and region (view
// fastest): the pixels of the region's projected bounding box whose rays
// cross its box inside the view's window, in a counting sort by chord
// length, so that each warp of region_kernel gets 32 rays of nearly equal
// length.  The float slab test runs against the box grown by 0.01 cells, far
// above its rounding (the exact set-up of the march still decides), so no ray
// that the march would sample is dropped.  No chord in the box is longer than
// the crossing time smax of any one axis, which scales the classes.
// Candidates (the bounding box in row-major order) are taken kScreenBatch at a
// time: classified and counted, then placed; each batch appends its own
// sorted run.  The 32 candidates of a step lie along a row, where the chord
// length changes smoothly: each run of lanes with one class takes its places
// with one shared atomic.  The list has room for every pixel the box can cover (the
// host's bound); were it ever full, the pixels past its end would be dropped
// and bit 1 of the error word set.  The launch also clears the partial slots
// that the region march then writes: each warp a contiguous share, before its
// own listing, so that the stores overlap the listing's arithmetic.
__global__ void __launch_bounds__(32 * kScreenWarps) screen_kernel(const __grid_constant__ RegionArgs a)
{
    __shared__ int s_off_all[kScreenWarps][kChordClasses];
    __shared__ uint8_t s_cls_all[kScreenWarps][kScreenBatch];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int regions = a.nreg[0] * a.nreg[1] * a.nreg[2];
    const long long pair = static_cast<long long>(blockIdx.x) * kScreenWarps + warp;
    {
        const long long warps = static_cast<long long>(gridDim.x) * kScreenWarps;
        const long long n4 = a.partial_floats >> 2;  // the slots start 256-byte aligned
        const long long share = (n4 + warps - 1) / warps;
        const long long lo = min(pair * share, n4), hi = min(lo + share, n4);
        float4 *p4 = reinterpret_cast<float4 *>(a.partial);
        for (long long i = lo + lane; i < hi; i += 32) __stcs(p4 + i, make_float4(0.f, 0.f, 0.f, 0.f));
        if (pair == 0 && lane < (a.partial_floats & 3)) a.partial[(n4 << 2) + lane] = 0.f;
    }
    if (pair >= static_cast<long long>(a.n_views) * regions) return;
    const int vi = static_cast<int>(pair % a.n_views), r = static_cast<int>(pair / a.n_views);
    int *s_off = s_off_all[warp];
    uint8_t *s_cls = s_cls_all[warp];
    const ViewDev &V = a.views[vi];
    const RegionProj &P = a.proj[vi];
    const RegionFrame F = region_frame(a, vi, r);
    const int cap = a.ctas_per_view * a.rays_per_cta;
    const int n_pix = F.pw * F.qh;
    const int nc = (n_pix + 31) & ~31;  // the whole warp takes each step
    const float inv_pw = F.pw > 0 ? 1.0f / static_cast<float>(F.pw) : 0.f;
    float lo[3], hi[3], ia[3], g0[3], gu[3], gv[3];
    float smax = 3.0e38f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        lo[k] = static_cast<float>(F.B.lo[k]) - 0.01f;
        hi[k] = static_cast<float>(F.B.hi[k]) + 0.01f;
        ia[k] = V.inv_a[k];
        g0[k] = P.g0f[k];
        gu[k] = P.guf[k];
        gv[k] = P.gvf[k];
        if (ia[k] != 0.f) smax = fminf(smax, (hi[k] - lo[k]) * ia[k]);
    }
    const float cls_scale = static_cast<float>(kChordClasses) / smax;
    const float win_lo = V.win_lo, win_hi = V.win_hi;
    uint32_t *list = a.rays + (static_cast<long long>(r) * a.n_views + vi) * cap;
    const uint32_t below = (1u << lane) - 1u;
    int done = 0;
    for (int base = 0; base < nc; base += kScreenBatch) {
        const int nb = min(nc - base, kScreenBatch);
        s_off[lane] = 0;
        s_off[lane + 32] = 0;
        __syncwarp();
        // classify and count (one leader lane per class updates its count)
        for (int i = lane; i < nb; i += 32) {
            const int j = base + i;  // row-major index in the bounding box
            int qo = static_cast<int>(static_cast<float>(j) * inv_pw);
            int po = j - qo * F.pw;
            if (po < 0) { po += F.pw; --qo; }
            if (po >= F.pw) { po -= F.pw; ++qo; }
            const float p = static_cast<float>(F.p_lo + po), q = static_cast<float>(F.q_lo + qo);
            bool hit = j < n_pix;
            float s_lo = win_lo, s_hi = win_hi;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const float g = fmaf(q, gv[k], fmaf(p, gu[k], g0[k]));
                if (ia[k] != 0.f) {
                    s_lo = fmaxf(s_lo, (lo[k] - g) * ia[k]);
                    s_hi = fminf(s_hi, (hi[k] - g) * ia[k]);
                } else {
                    hit = hit && g >= lo[k] && g < hi[k];
                }
            }
            hit = hit && s_hi > s_lo - 1e-3f * (1.f + fabsf(s_lo));
            const float f = fminf(fmaxf((s_hi - s_lo) * cls_scale, 0.f), static_cast<float>(kChordClasses - 1));
            const int c = hit ? kChordClasses - 1 - static_cast<int>(f) : kChordClasses;
            s_cls[i] = static_cast<uint8_t>(c);
            const int c_prev = __shfl_up_sync(kFull, c, 1);  // every lane takes part
            const bool head = lane == 0 || c != c_prev;
            const uint32_t heads = __ballot_sync(kFull, head);
            if (head && c < kChordClasses) {
                const uint32_t after = heads & ~below & ~(1u << lane);
                atomicAdd(&s_off[c], (after ? __ffs(after) - 1 : 32) - lane);
            }
        }
        __syncwarp();
        // exclusive prefix sum over the classes, two per lane
        const int c0 = s_off[2 * lane], c1 = s_off[2 * lane + 1];
        int incl = c0 + c1;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int v = __shfl_up_sync(kFull, incl, d);
            incl += lane >= d ? v : 0;
        }
        const int excl = done + incl - c0 - c1;
        __syncwarp();
        s_off[2 * lane] = excl;
        s_off[2 * lane + 1] = excl + c0;
        __syncwarp();
        // place
        for (int i = lane; i < nb; i += 32) {
            const int c = s_cls[i];
            const int c_prev = __shfl_up_sync(kFull, c, 1);  // every lane takes part
            const bool head = lane == 0 || c != c_prev;
            const uint32_t heads = __ballot_sync(kFull, head);
            int pos = 0;
            if (head && c < kChordClasses) {
                const uint32_t after = heads & ~below & ~(1u << lane);
                pos = atomicAdd(&s_off[c], (after ? __ffs(after) - 1 : 32) - lane);
            }
            const int lead = 31 - __clz(heads & (below | (1u << lane)));
            pos = __shfl_sync(kFull, pos, lead) + lane - lead;
            if (c < kChordClasses) {
                const int j = base + i;
                int qo = static_cast<int>(static_cast<float>(j) * inv_pw);
                int po = j - qo * F.pw;
                if (po < 0) { po += F.pw; --qo; }
                if (po >= F.pw) { po -= F.pw; ++qo; }
                if (pos < cap)
                    list[pos] = static_cast<uint32_t>(F.p_lo + po) | (static_cast<uint32_t>(F.q_lo + qo) << 16);
                else if (a.error_word)
                    atomicOr(a.error_word, 2);
            }
        }
        done += __shfl_sync(kFull, incl, 31);
        __syncwarp();  // the counts and classes are reused by the next batch
    }
    if (lane == 0) a.ray_count[r * a.n_views + vi] = min(done, cap);
}

// A value that every lane of the warp holds, as a warp-uniform one: the
// result of a warp reduction, which the compiler keeps in a uniform register.
__device__ __forceinline__ uint32_t uniform(uint32_t x) { return __reduce_or_sync(kFull, x); }
__device__ __forceinline__ float uniform(float x) { return __uint_as_float(uniform(__float_as_uint(x))); }
__device__ __forceinline__ long long uniform(long long x)
{
    const unsigned long long u = static_cast<unsigned long long>(x);
    return static_cast<long long>((static_cast<unsigned long long>(uniform(static_cast<uint32_t>(u >> 32))) << 32) |
                                  uniform(static_cast<uint32_t>(u)));
}

// The march of the region schedule: CTA (blockIdx.x) of the region's
// blockIdx.y-th view (region_order) in region blockIdx.z stages the region's
// march tables and gives each warp the next 32 rays of the view's ray list for
// the region, so that warp w of CTA cb marches entries (cb * warps + w) * 32 ..
// + 31.  CTAs past the end of the list return at once.
//
// The views sit in device memory, so their constants would be loaded into every lane's
// registers; the ones the march uses in each step are made warp-uniform, which
// frees 16 registers.  CAP: the register cap (select_region says which, and why).
template <int STORE, int H, int CAP, bool PAIRED>
__global__ void __maxnreg__(CAP) region_kernel(const __grid_constant__ RegionArgs a)
{
    extern __shared__ int32_t s_tab[];
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int r = static_cast<int>(blockIdx.z);
    const int vi = __ldg(a.region_order + static_cast<long long>(r) * a.n_views + blockIdx.y);
    const int count = __ldg(a.ray_count + r * a.n_views + vi);
    const int first = static_cast<int>(blockIdx.x) * a.rays_per_cta;
    if (first >= count) return;
    const ViewDev &V = a.views[vi];
    const RegionFrame F = region_frame(a, vi, r);
    for (int i = 0; i < 3; ++i) {
        const bool mirrored = (V.flags & (kFlagMirror0 << i)) != 0u;
        const int len = F.B.hi[i] - F.B.lo[i];
        const int src = march_table_base(a.vol.n, i) + (mirrored ? a.vol.n[i] + 1 : 0) + F.B.lo[i];
        for (int j = threadIdx.x; j < len + 1; j += blockDim.x) s_tab[i * (a.region + 1) + j] = a.vol.mtab[src + j];
    }
    const int k = first + warp * 32 + lane;
    const uint32_t *list = a.rays + (static_cast<long long>(r) * a.n_views + vi) * a.ctas_per_view * a.rays_per_cta;
    const uint32_t pq = k < count ? __ldg(list + k) : (static_cast<uint32_t>(a.width) | (static_cast<uint32_t>(a.height) << 16));
    __syncthreads();  // tables staged
    if (__all_sync(kFull, k >= count)) return;
    ViewDev U = V;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        U.inv_a[i] = uniform(V.inv_a[i]);
        U.du[i] = uniform(V.du[i]);
        U.sh_hi[i] = uniform(V.sh_hi[i]);
        U.sh_lo[i] = uniform(V.sh_lo[i]);
    }
    U.expo = uniform(V.expo);
    U.kk_hi = uniform(V.kk_hi);
    U.flags = uniform(V.flags);
    float *out = a.partial + static_cast<long long>(F.slot) * a.slot_stride +
                 static_cast<long long>(a.image[vi]) * a.width * a.height;
    march_ray<STORE, H, PAIRED, true>(a.vol, U, F.B, static_cast<int>(pq & 0xffffu), static_cast<int>(pq >> 16),
                                                a.width, a.height, out, nullptr, a.error_word, s_tab);
}

// One view per blockIdx.y.
__global__ void __launch_bounds__(256) reduce_kernel(const __grid_constant__ ReduceArgs a)
{
    const int v = static_cast<int>(blockIdx.y);
    const long long img = static_cast<long long>(a.image[v]) * a.pix_per_view;
    const float pre = a.prefactor[v];
    for (long long px = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x; px < a.pix_per_view;
         px += static_cast<long long>(gridDim.x) * blockDim.x) {
        const long long i = img + px;
        float acc = 0.f, comp = 0.f;
        for (int s = 0; s < a.n_slots; ++s) {
            const float y = a.partial[static_cast<long long>(s) * a.slot_stride + i] - comp;
            const float t = acc + y;
            comp = (t - acc) - y;
            acc = t;
        }
        a.out[i] = pre * acc;
    }
}

// Stages of `depth` cells, at most two: four spill at 80 registers (1024^2 image of
// bfloat16/float16 records 0.87 against 0.81 ms) or leave 16 warps per SM.
template <int STORE, int MINB, bool PAIRED>
void *select_depth(int depth)
{
    switch (depth) {
    case 1: return reinterpret_cast<void *>(&march_kernel<STORE, 1, MINB, PAIRED>);
    case 2:
    case 4: return reinterpret_cast<void *>(&march_kernel<STORE, 2, MINB, PAIRED>);
    default: return nullptr;
    }
}

template <int STORE, bool PAIRED>
void *select_cap(int depth, int capped)
{
    return capped ? select_depth<STORE, 3, PAIRED>(depth) : select_depth<STORE, 1, PAIRED>(depth);
}

template <int STORE, int DEPTH, int G>
void *select_group_snaps(int snaps)
{
    if (snaps == kGroupSnapsMin) return reinterpret_cast<void *>(&group_kernel<STORE, DEPTH, G, kGroupSnapsMin, false>);
    if (snaps == kGroupSnapsMax) return reinterpret_cast<void *>(&group_kernel<STORE, DEPTH, G, kGroupSnapsMax, false>);
    return nullptr;
}

template <int STORE, int DEPTH>
void *select_group_size(int size, int snaps)
{
    return size == 4 ? select_group_snaps<STORE, DEPTH, 4>(snaps)
                     : (size == kGroupMax ? select_group_snaps<STORE, DEPTH, kGroupMax>(snaps) : nullptr);
}

// Time groups: a kernel for groups of up to 4 views and one for up to 8, each
// for members within one snapshot of each other and within kGroupSnapsMax - 2.
// float32 groups march one cell per iteration whatever the depth, and
// bfloat16/float16 ones at most two: a cell's S gathers already keep as many
// loads in flight, and more cells' records would cost more warps than the
// loads gain.  Groups of more than four with five snapshots take one: two spill 108 bytes
// (8 views of 384^2 of 256^3 x 32 within 2.9 snapshots 311 / 300 us; with three snapshots, 8
// bytes spilled, within 0.9: 197 / 218).
// Long tables (spans): one kernel per store, for any group.
void *select_group(int store, int size, int depth, int snaps, bool spans)
{
    if (depth != 1 && depth != 2 && depth != 4) return nullptr;
    if (spans)
        return store == GBD_STORE_F32
                   ? reinterpret_cast<void *>(&group_kernel<GBD_STORE_F32, 1, kGroupMax, kGroupSnapsMax, true>)
                   : reinterpret_cast<void *>(&group_kernel<GBD_STORE_BF16_F16U, 1, kGroupMax, kGroupSnapsMax, true>);
    if (store == GBD_STORE_F32) return select_group_size<GBD_STORE_F32, 1>(size, snaps);
    if (store != GBD_STORE_BF16_F16U) return nullptr;
    if (depth == 1 || (size == kGroupMax && snaps == kGroupSnapsMax))
        return select_group_size<GBD_STORE_BF16_F16U, 1>(size, snaps);
    if (size == kGroupMax)
        return reinterpret_cast<void *>(&group_kernel<GBD_STORE_BF16_F16U, 2, kGroupMax, kGroupSnapsMin, false>);
    return select_group_snaps<GBD_STORE_BF16_F16U, 2, 4>(snaps);
}

void *select_kernel(int store, int depth, int capped, int paired)
{
    if (store == GBD_STORE_F32)
        return paired ? select_cap<GBD_STORE_F32, true>(depth, capped) : select_cap<GBD_STORE_F32, false>(depth, capped);
    if (store == GBD_STORE_BF16_F16U)
        return paired ? select_cap<GBD_STORE_BF16_F16U, true>(depth, capped)
                      : select_cap<GBD_STORE_BF16_F16U, false>(depth, capped);
    return nullptr;
}

// The region march waits for its gathers.  Where few rays cross a region (64 cells and more,
// few rays through a cell), what is in flight counts: stages of `depth` cells and 80 registers,
// whatever the cap asked for.  Elsewhere warps count more: 64 registers, and for
// float32 (which two cells would spill; 80 without the cap) stages of one cell.
// Paired bfloat16/float16 records fit two cells in 64.
// Measured, two cells at 80 registers / the others (us), regions of 64. float32 (one at 64), by rays
// through a cell: 1.1: 60 views of 216^2 of 147^3 x 6 729 / 692; 0.4: 224^2 of 250^3 1181 / 1158;
// 0.35: 64 of 160^2 of 192^3 x 12 850 / 892; 0.2: 256 of 256^2 of 384^3 x 32 (8-cell bricks) 19441 / 19402, 61 of
// 192 x 64 of 305^3 x 13 1602 / 1913; 0.08: 100 of 128^2 of 320^3 x 16 3331 / 3830; regions of 128, 0.4:
// 1392 / 1478, of 32, 0.28: 5703 / 5328.  bfloat16/float16, unpaired (two at 64, 8 bytes spilled): 1.1: 158 of
// 216 x 91 of 147^3 x 6 987 / 917; 0.28: 60 of 224^2 of 300^3 1167 / 1123; 0.055: 100 of 100^2 of 300^3 x 16
// 1197 / 1400; regions of 128, 0.32: 100 of 200^2 of 250^3 x 16 2382 / 2671; of 32, 0.055: 1341 / 1171.
bool sparse_regions(int store, int paired, int region, float rays)
{
    if (region < 64) return false;
    if (store == GBD_STORE_F32) return rays < (region >= 128 ? 0.5f : 0.375f);
    return !paired && rays < (region >= 128 ? 0.35f : 0.15f);
}

template <bool PAIRED>
void *select_region_f32(int depth, int capped, bool sparse)
{
    if (sparse && depth == 2) return reinterpret_cast<void *>(&region_kernel<GBD_STORE_F32, 2, 80, PAIRED>);
    return capped && !sparse ? reinterpret_cast<void *>(&region_kernel<GBD_STORE_F32, 1, 64, PAIRED>)
                             : reinterpret_cast<void *>(&region_kernel<GBD_STORE_F32, 1, 80, PAIRED>);
}

template <bool PAIRED>
void *select_region_bf16(int depth)
{
    return depth == 2 ? reinterpret_cast<void *>(&region_kernel<GBD_STORE_BF16_F16U, 2, 64, PAIRED>)
                      : reinterpret_cast<void *>(&region_kernel<GBD_STORE_BF16_F16U, 1, 64, PAIRED>);
}

void *select_region(int store, int depth, int capped, int paired, bool sparse)
{
    if (depth != 1 && depth != 2) return nullptr;
    if (store == GBD_STORE_F32)
        return paired ? select_region_f32<true>(depth, capped, sparse) : select_region_f32<false>(depth, capped, sparse);
    if (store == GBD_STORE_BF16_F16U) {
        if (sparse && depth == 2) return reinterpret_cast<void *>(&region_kernel<GBD_STORE_BF16_F16U, 2, 80, false>);
        return paired ? select_region_bf16<true>(depth) : select_region_bf16<false>(depth);
    }
    return nullptr;
}

template <int NCH, bool RUNS>
void *select_vector_store(int store, int paired)
{
    if (store == GBD_STORE_F32)
        return paired ? reinterpret_cast<void *>(&vector_kernel<GBD_STORE_F32, NCH, true, RUNS>)
                      : reinterpret_cast<void *>(&vector_kernel<GBD_STORE_F32, NCH, false, RUNS>);
    if (store == GBD_STORE_BF16_F16U)
        return paired ? reinterpret_cast<void *>(&vector_kernel<GBD_STORE_BF16_F16U, NCH, true, RUNS>)
                      : reinterpret_cast<void *>(&vector_kernel<GBD_STORE_BF16_F16U, NCH, false, RUNS>);
    return nullptr;
}

template <int NCH>
void *select_vector_runs(const MarchArgs &a)
{
    const bool runs = a.n_views > 1 && static_cast<long long>(a.n_views) * a.width * a.height >= kRunsPixels;
    return runs ? select_vector_store<NCH, true>(a.vol.store, a.vol.paired)
                : select_vector_store<NCH, false>(a.vol.store, a.vol.paired);
}

void *select_wave(int depth, int capped)
{
    if (depth == 1) return capped ? reinterpret_cast<void *>(&wave_kernel<1, 3>) : reinterpret_cast<void *>(&wave_kernel<1, 1>);
    if (depth == 2) return capped ? reinterpret_cast<void *>(&wave_kernel<2, 3>) : reinterpret_cast<void *>(&wave_kernel<2, 1>);
    return nullptr;
}

}  // namespace

cudaError_t launch_wave(const WaveArgs &a, const LaunchCfg &cfg, cudaStream_t stream)
{
    void *k = select_wave(cfg.depth, cfg.regcap);
    if (!k) return cudaErrorInvalidValue;
    if (a.total_ctas < 1) return cudaSuccess;
    // shared memory for the largest march tables of the launch
    int smem = 0;
    for (int r = 0; r < a.n_reqs; ++r)
        smem = std::max(smem, static_cast<int>(sizeof(int32_t)) * staged_entries(a.reqs[r].vol.n));
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
    }
    void *params[] = {const_cast<WaveArgs *>(&a)};
    return cudaLaunchKernel(k, dim3(static_cast<unsigned>(a.total_ctas)), dim3(32 * cfg.cta_warps), params, smem,
                            stream);
}

cudaError_t launch_vector(MarchArgs &a, int n_chan, const LaunchCfg &cfg, cudaStream_t stream)
{
    void *k = n_chan == 1 ? select_vector_runs<1>(a) : (n_chan == 3 ? select_vector_runs<3>(a) : nullptr);
    if (!k) return cudaErrorInvalidValue;
    // grid and shared memory as planned for the scalar kernel
    KernelLaunch L;
    cudaError_t e = plan_march(a, cfg, L);
    if (e != cudaSuccess) return e;
    if (L.smem > 48 * 1024) {
        e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, L.smem);
        if (e != cudaSuccess) return e;
    }
    void *params[] = {&a};
    return cudaLaunchKernel(k, L.grid, L.block, params, L.smem, stream);
}

cudaError_t launch_touch(MarchArgs &a, uint32_t *bits, long long cells, const LaunchCfg &cfg, cudaStream_t stream)
{
    void *k = a.vol.store == GBD_STORE_F32
                  ? (a.vol.paired ? reinterpret_cast<void *>(&touch_kernel<GBD_STORE_F32, true>)
                                  : reinterpret_cast<void *>(&touch_kernel<GBD_STORE_F32, false>))
                  : (a.vol.paired ? reinterpret_cast<void *>(&touch_kernel<GBD_STORE_BF16_F16U, true>)
                                  : reinterpret_cast<void *>(&touch_kernel<GBD_STORE_BF16_F16U, false>));
    KernelLaunch L;
    cudaError_t e = plan_march(a, cfg, L);
    if (e != cudaSuccess) return e;
    if (L.smem > 48 * 1024) {
        e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, L.smem);
        if (e != cudaSuccess) return e;
    }
    void *params[] = {&a, &bits, &cells};
    return cudaLaunchKernel(k, L.grid, L.block, params, L.smem, stream);
}

cudaError_t launch_screen(const RegionArgs &a, cudaStream_t stream)
{
    const long long regions = static_cast<long long>(a.nreg[0]) * a.nreg[1] * a.nreg[2];
    if (a.n_views < 1 || a.n_views > 65535 || !a.rays || !a.ray_count || !a.views || !a.proj || a.rays_per_cta < 32 ||
        a.ctas_per_view < 1 || regions < 1 || regions > 65535 || a.partial_floats < 0 ||
        (a.partial_floats > 0 && !a.partial))
        return cudaErrorInvalidValue;
    const long long ctas = (a.n_views * regions + kScreenWarps - 1) / kScreenWarps;
    void *params[] = {const_cast<RegionArgs *>(&a)};
    return cudaLaunchKernel(reinterpret_cast<void *>(&screen_kernel), dim3(static_cast<unsigned>(ctas)),
                            dim3(32 * kScreenWarps), params, 0, stream);
}

cudaError_t launch_region(const RegionArgs &a, const LaunchCfg &cfg, cudaStream_t stream)
{
    void *k = select_region(a.vol.store, cfg.depth, cfg.regcap, a.vol.paired,
                            sparse_regions(a.vol.store, a.vol.paired, a.region, a.rays_per_cell));
    const long long regions = static_cast<long long>(a.nreg[0]) * a.nreg[1] * a.nreg[2];
    if (!k || a.n_views < 1 || a.n_views > 65535 || regions < 1 || regions > 65535 || a.ctas_per_view < 1 ||
        a.rays_per_cta != 32 * cfg.cta_warps || !a.image || !a.region_order)
        return cudaErrorInvalidValue;
    const int smem = static_cast<int>(sizeof(int32_t)) * 3 * (a.region + 1);
    void *params[] = {const_cast<RegionArgs *>(&a)};
    return cudaLaunchKernel(k, dim3(static_cast<unsigned>(a.ctas_per_view), static_cast<unsigned>(a.n_views),
                                    static_cast<unsigned>(regions)),
                            dim3(32 * cfg.cta_warps), params, smem, stream);
}

cudaError_t launch_reduce(const ReduceArgs &a, cudaStream_t stream)
{
    if (a.n_views < 1 || a.pix_per_view < 1) return cudaSuccess;
    if (a.n_views > kImagesPerReduce) return cudaErrorInvalidValue;
    const long long per_view = std::max<long long>(1, 152LL * 16 / a.n_views);
    const long long blocks = std::min<long long>((a.pix_per_view + 255) / 256, per_view);
    void *params[] = {const_cast<ReduceArgs *>(&a)};
    return cudaLaunchKernel(reinterpret_cast<void *>(&reduce_kernel),
                            dim3(static_cast<unsigned>(blocks), static_cast<unsigned>(a.n_views)), dim3(256), params,
                            0, stream);
}

// Cells of a stage at depth 2, the default.  Unpaired float32 stages of two cells take 80
// registers (24 warps per SM), of one 64 (32 warps): two hide the latency of DRAM, one does
// more work where L1 and L2 deliver.  One cell where the records that a launch reads come
// from the caches:
//  * kDenseRays rays and more through a cell: its record is read again at once;
//  * the snapshots around a time (or the only one) fit in L2 with room to spare;
//  * one snapshot: half the loads of a sample;
//  * half of the views within a snapshot of the one before, along the same rays.
// And only in launches that fill 32 warps per SM about one and a half times: with fewer, each
// ray's own latency counts.  Two cells / one, us: dense: 1024^2 of 128^3 x 8 324 / 270, six
// views of 512^2 of 200^3 x 8 (3.3 rays) 520 / 460, 1024^2 of 384^3 x 6 (3.6) 1009 / 1023, 512^2 of 256^3
// x 8 (2.0) 236 / 282; L2: 12 of 256^2 of 160^3 x 8 (131 MB) 231 / 220, 6 of 300^2 of 200^3 x 12 (256 MB)
// 279 / 314; one snapshot: 1024^2 of 512^3 741 / 639; series: 18 of 512^2 of 256^3 x 16, marched alone,
// 942 / 826; few warps: 24 of 100^2 of 160^3 x 8 (7500) 176 / 198, 512^2 of 100^3 x 8 (8192) 84 / 76.
// Paired records (one pair for a sample) and bfloat16/float16 take two: 24 of 384^2 of 256^3 x 16
// 2290 / 2337 paired, 1627 / 1716 in bfloat16/float16.
constexpr double kDenseRays = 3.2;
constexpr long long kCachedBytes = 128LL << 20;
constexpr long long kFullWarps = 8000;
int stage_cells(const MarchArgs &a)
{
    if (a.vol.store != GBD_STORE_F32 || a.vol.paired) return 2;
    const long long warps = static_cast<long long>(a.n_views) * a.pk.blocks * (a.pk.step_x * a.pk.step_y / 32);
    if (warps < kFullWarps) return 2;
    const long long cells = static_cast<long long>(a.vol.n[0]) * a.vol.n[1] * a.vol.n[2];
    if (a.vol.M == 1 || cells * 2 * 16 <= kCachedBytes || 2 * a.near_units >= a.n_views) return 1;
    return rays_per_cell(a.views[0]) >= kDenseRays ? 1 : 2;
}

cudaError_t plan_march(const MarchArgs &a, const LaunchCfg &cfg, KernelLaunch &L)
{
    // n_groups > 0: time groups, one image's blocks of CTAs per group; else per view
    const bool grouped = a.n_groups > 0;
    void *k = grouped ? select_group(a.vol.store, a.group_size, cfg.depth, a.group_snaps,
                                     march_table_entries(a.vol.n) > kCopiesMax * 32 * cfg.cta_warps)
                      : select_kernel(a.vol.store, cfg.depth == 2 ? stage_cells(a) : cfg.depth, cfg.regcap,
                                      a.vol.paired);
    if (!k || a.n_views < 1 || a.n_views > kViewsPerLaunch) return cudaErrorInvalidValue;
    if (grouped && (a.n_groups > a.n_views || a.group_first[0] != 0 || a.group_first[a.n_groups] != a.n_views))
        return cudaErrorInvalidValue;
    const int units = grouped ? a.n_groups : a.n_views;
    for (int u = 0; u < units && grouped; ++u) {
        const int v0 = a.group_first[u], v1 = a.group_first[u + 1];
        if (v1 <= v0 || v1 - v0 > a.group_size || a.group_ref[u] < v0 || a.group_ref[u] >= v1)
            return cudaErrorInvalidValue;
    }
    const int smem = static_cast<int>(sizeof(int32_t)) * staged_entries(a.vol.n);
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
    }
    const long long total = static_cast<long long>(units) * a.pk.blocks;
    if (total < 1 || total > 0x7fffffffLL) return cudaErrorInvalidValue;
    L.func = k;
    L.grid = dim3(static_cast<unsigned>(total));
    L.block = dim3(32 * cfg.cta_warps);
    L.smem = smem;
    return cudaSuccess;
}

cudaError_t launch_march(MarchArgs &a, const LaunchCfg &cfg, cudaStream_t stream)
{
    KernelLaunch L;
    cudaError_t e = plan_march(a, cfg, L);
    if (e != cudaSuccess) return e;
    void *params[] = {&a};
    return cudaLaunchKernel(L.func, L.grid, L.block, params, L.smem, stream);
}

}  // namespace gbd
