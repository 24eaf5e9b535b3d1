// pack.cu -- converts one snapshot epoch from C-ordered input arrays into the
// packed record layout of the march kernels, validating every value.
//
// The method's inputs are the rest-frame emissivity j' and the velocity beta
// of every cell (Sec. 2.5).  Records are written at the per-axis offset sum
// described in gbd_internal.h; padding cells are left as the caller cleared
// them.
//
// GBD_STORE_F32 keeps {j', beta} as float32 (rounded to nearest).
// GBD_STORE_BF16_F16U keeps j' rounded to float32 then to bfloat16, and the
// four-velocity u = Gamma beta as computed in float64 with explicitly rounded
// operations (b2 = (bx*bx + by*by) + bz*bz, Gamma = 1/sqrt(1 - b2),
// u_i = beta_i * Gamma) and rounded once to float16, so that the stored value
// is a fixed function of the input.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>

#include "gbd_internal.h"

namespace gbd {
namespace {

// |beta|^2 <= 1 - 2^-20 for stored float32 components, decided as in float64.
// The float32 sum is off by less than 2^-22, so below 1 - 2^-19 the answer is known.
__device__ __forceinline__ bool below_limit(float x, float y, float z)
{
    if (fmaf(x, x, fmaf(y, y, z * z)) < 1.0f - 1.0f / 524288.0f) return true;
    const double b2 = static_cast<double>(x) * x + static_cast<double>(y) * y + static_cast<double>(z) * z;
    return b2 <= 1.0 - 1.0 / 1048576.0;
}

// u = Gamma beta in float64, rounded once to float16; false if |beta| >= 1 or not a number.
__device__ __forceinline__ bool velocity_f64(double bx, double by, double bz, __half (&u)[3])
{
    const double b2 = __dadd_rn(__dadd_rn(__dmul_rn(bx, bx), __dmul_rn(by, by)), __dmul_rn(bz, bz));
    const bool ok = b2 < 1.0;
    const double g = ok ? __ddiv_rn(1.0, __dsqrt_rn(__dadd_rn(1.0, -b2))) : 1.0;
    u[0] = __double2half(__dmul_rn(bx, g));
    u[1] = __double2half(__dmul_rn(by, g));
    u[2] = __double2half(__dmul_rn(bz, g));
    return ok;
}

__device__ __forceinline__ bool velocity_f16(double bx, double by, double bz, __half (&u)[3])
{
    return velocity_f64(bx, by, bz, u);
}

// The same for float32 input, without float64 where float32 can decide it:
// 1 - |beta|^2 from a double-float |beta|^2, its inverse root to a few 2^-24, and u to
// within 2^-21.  Where u (1 +- 2^-20) round to one float16, so does the
// float64 value between them; the few cells beside a rounding boundary, and those with
// Gamma > 64, take float64.
__device__ __forceinline__ bool velocity_f16(float bx, float by, float bz, __half (&u)[3])
{
    const float px = __fmul_rn(bx, bx), py = __fmul_rn(by, by), pz = __fmul_rn(bz, bz);
    const float ex = fmaf(bx, bx, -px), ey = fmaf(by, by, -py), ez = fmaf(bz, bz, -pz);
    const float s = __fadd_rn(px, py), sb = __fsub_rn(s, px);
    const float se = __fadd_rn(__fsub_rn(px, __fsub_rn(s, sb)), __fsub_rn(py, sb));
    const float t = __fadd_rn(s, pz), tb = __fsub_rn(t, s);
    const float te = __fadd_rn(__fsub_rn(s, __fsub_rn(t, tb)), __fsub_rn(pz, tb));
    const float om = __fsub_rn(1.0f - t, (ex + ey) + (ez + (se + te)));
    if (om > 1.0f / 4096.0f) {
        float g = rsqrtf(om);
        g = fmaf(0.5f * g, fmaf(-om * g, g, 1.0f), g);
        const float v[3] = {bx * g, by * g, bz * g};
        bool sure = true;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            u[i] = __float2half_rn(v[i] * (1.0f + 1.0f / 1048576.0f));
            sure = sure && __half_as_ushort(u[i]) == __half_as_ushort(__float2half_rn(v[i] * (1.0f - 1.0f / 1048576.0f)));
        }
        if (sure) return true;
    }
    return velocity_f64(bx, by, bz, u);
}

// One thread per cell.  What bounds it: HBM (a cell's 16 or 32 input bytes read and its
// records written once).  The float64 arithmetic that decides limits and
// rounds u ran on every cell before (FP64 pipe 87% busy, 618 us for a 256^3 float32
// epoch); now it runs only where float32 cannot decide, with 32-bit
// indices (an epoch has fewer than 2^31 records): 89 us, 0.89 of the measured copy rate.
template <typename TIN, int STORE>
__global__ void __launch_bounds__(256) pack_kernel(const PackArgs a)
{
    const uint32_t nx = a.n[0], ny = a.n[1];
    const uint32_t ncell = nx * ny * static_cast<uint32_t>(a.n[2]);
    const TIN *jin = static_cast<const TIN *>(a.j);
    const TIN *vin = static_cast<const TIN *>(a.vel);
    const int32_t *offx = a.axis_off;
    const int32_t *offy = a.axis_off + nx;
    const int32_t *offz = a.axis_off + nx + ny;
    float g2max = 0.f;  // largest Gamma^2 of this thread's stored bfloat16/float16 records
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < ncell; i += gridDim.x * blockDim.x) {
        const uint32_t r = i / nx, ix = i - r * nx;
        const uint32_t iz = r / ny, iy = r - iz * ny;
        const uint32_t cell = static_cast<uint32_t>(offx[ix] + offy[iy] + offz[iz]);
        // paired blocks: snapshot m is the second record of block m and the
        // first record of block m + 1
        const long long off = a.paired ? static_cast<long long>(a.m) * a.stride + 2 * static_cast<long long>(cell) + 1
                                       : static_cast<long long>(a.m) * a.stride + cell;
        const long long off2 = off + a.stride - 1;
        const TIN j = jin[i];
        const TIN *v = vin + 3 * static_cast<size_t>(i);
        const TIN bx = v[0], by = v[1], bz = v[2];
        bool ok = isfinite(j) && j >= TIN(0) && isfinite(bx) && isfinite(by) && isfinite(bz);
        const float jf = static_cast<float>(j);
        if constexpr (STORE == GBD_STORE_F32) {
            const float fx = static_cast<float>(bx), fy = static_cast<float>(by), fz = static_cast<float>(bz);
            // |beta| as stored must stay below 1 with room for float32
            // rounding of 1 - beta^2.
            ok = ok && isfinite(jf) && below_limit(fx, fy, fz);
            const float4 rec = ok ? make_float4(jf, fx, fy, fz) : make_float4(0.f, 0.f, 0.f, 0.f);
            reinterpret_cast<float4 *>(a.dst)[off] = rec;
            if (a.paired) reinterpret_cast<float4 *>(a.dst)[off2] = rec;
        } else {
            __half u[3];
            ok = velocity_f16(bx, by, bz, u) && ok;
            const __nv_bfloat16 jb = __float2bfloat16_rn(jf);
            ok = ok && isfinite(__bfloat162float(jb)) && __hisinf(u[0]) == 0 && __hisinf(u[1]) == 0 && __hisinf(u[2]) == 0;
            uint2 rec;
            rec.x = static_cast<uint32_t>(__bfloat16_as_ushort(jb)) | (static_cast<uint32_t>(__half_as_ushort(u[0])) << 16);
            rec.y = static_cast<uint32_t>(__half_as_ushort(u[1])) | (static_cast<uint32_t>(__half_as_ushort(u[2])) << 16);
            if (!ok) rec = make_uint2(0u, 0u);
            // Gamma^2 of the stored u, as the march computes it from the
            // float16 values
            const float fx = __half2float(u[0]), fy = __half2float(u[1]), fz = __half2float(u[2]);
            if (ok) g2max = fmaxf(g2max, fmaf(fx, fx, fmaf(fy, fy, fmaf(fz, fz, 1.0f))));
            reinterpret_cast<uint2 *>(a.dst)[off] = rec;
            if (a.paired) reinterpret_cast<uint2 *>(a.dst)[off2] = rec;
        }
        if (!ok) atomicExch(a.bad, 1);
    }
    if (STORE != GBD_STORE_F32 && a.gamma2_max) {
        // one atomic per warp (non-negative floats order as their bits)
        for (int o = 16; o > 0; o >>= 1) g2max = fmaxf(g2max, __shfl_xor_sync(0xffffffffu, g2max, o));
        if ((threadIdx.x & 31) == 0 && g2max > 0.f) atomicMax(a.gamma2_max, __float_as_uint(g2max));
    }
}

// One epoch of one extra emissivity channel (vector renders): a float per
// cell at the cell's layout offset; any finite value (a channel may be a
// signed component).
template <typename TIN>
__global__ void chan_pack_kernel(const ChanPackArgs a)
{
    const int nx = a.n[0], ny = a.n[1], nz = a.n[2];
    const long long ncell = static_cast<long long>(nx) * ny * nz;
    const TIN *in = static_cast<const TIN *>(a.src);
    for (long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x; i < ncell;
         i += static_cast<long long>(gridDim.x) * blockDim.x) {
        const int ix = static_cast<int>(i % nx);
        const long long r = i / nx;
        const int iy = static_cast<int>(r % ny);
        const int iz = static_cast<int>(r / ny);
        const long long cell = static_cast<long long>(a.axis_off[ix]) + a.axis_off[nx + iy] + a.axis_off[nx + ny + iz];
        const float v = __double2float_rn(static_cast<double>(in[i]));
        const bool ok = isfinite(v);
        a.dst[cell] = ok ? v : 0.f;
        if (!ok) atomicExch(a.bad, 1);
    }
}

// Copies every record of one epoch from one layout to another (the tables of
// both layouts have the same n_x + n_y + n_z entries).
template <typename R>
__global__ void relayout_kernel(const RelayoutArgs a)
{
    const int nx = a.n[0], ny = a.n[1], nz = a.n[2];
    const long long ncell = static_cast<long long>(nx) * ny * nz;
    const R *src = static_cast<const R *>(a.src);
    R *dst = static_cast<R *>(a.dst);
    for (long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x; i < ncell;
         i += static_cast<long long>(gridDim.x) * blockDim.x) {
        const int ix = static_cast<int>(i % nx);
        const long long r = i / nx;
        const int iy = static_cast<int>(r % ny);
        const int iz = static_cast<int>(r / ny);
        const long long cs = static_cast<long long>(a.src_off[ix]) + a.src_off[nx + iy] + a.src_off[nx + ny + iz];
        const long long cd = static_cast<long long>(a.dst_off[ix]) + a.dst_off[nx + iy] + a.dst_off[nx + ny + iz];
        const long long from = a.src_paired ? static_cast<long long>(a.m) * a.src_stride + 2 * cs + 1
                                            : static_cast<long long>(a.m) * a.src_stride + cs;
        const R v = src[from];
        if (a.dst_paired) {
            dst[static_cast<long long>(a.m) * a.dst_stride + 2 * cd + 1] = v;
            dst[static_cast<long long>(a.m + 1) * a.dst_stride + 2 * cd] = v;
        } else {
            dst[static_cast<long long>(a.m) * a.dst_stride + cd] = v;
        }
    }
}

}  // namespace

cudaError_t launch_relayout(const RelayoutArgs &a, cudaStream_t stream)
{
    const long long ncell = static_cast<long long>(a.n[0]) * a.n[1] * a.n[2];
    long long blocks = (ncell + 255) / 256;
    if (blocks > 65535LL * 16) blocks = 65535LL * 16;
    if (blocks < 1) return cudaSuccess;
    RelayoutArgs args = a;
    void *params[] = {&args};
    void *k = a.record_bytes == 16 ? reinterpret_cast<void *>(&relayout_kernel<uint4>)
                                   : (a.record_bytes == 8 ? reinterpret_cast<void *>(&relayout_kernel<uint2>)
                                                          : reinterpret_cast<void *>(&relayout_kernel<float>));
    return cudaLaunchKernel(k, dim3(static_cast<unsigned>(blocks)), dim3(256), params, 0, stream);
}

cudaError_t launch_pack(const PackArgs &a, cudaStream_t stream)
{
    const long long ncell = static_cast<long long>(a.n[0]) * a.n[1] * a.n[2];
    if (ncell < 1) return cudaSuccess;
    if (ncell >= (1LL << 31)) return cudaErrorInvalidValue;  // the layout takes fewer
    // at most 2^16 CTAs, so that the 32-bit cell index cannot wrap in the kernel's stride
    const unsigned blocks = static_cast<unsigned>(std::min<long long>((ncell + 255) / 256, 65536));
    PackArgs args = a;
    void *params[] = {&args};
    const bool f64 = a.dtype_in == GBD_IN_F64;
    void *k = a.store == GBD_STORE_F32
                  ? (f64 ? reinterpret_cast<void *>(&pack_kernel<double, GBD_STORE_F32>)
                         : reinterpret_cast<void *>(&pack_kernel<float, GBD_STORE_F32>))
                  : (f64 ? reinterpret_cast<void *>(&pack_kernel<double, GBD_STORE_BF16_F16U>)
                         : reinterpret_cast<void *>(&pack_kernel<float, GBD_STORE_BF16_F16U>));
    return cudaLaunchKernel(k, dim3(blocks), dim3(256), params, 0, stream);
}

cudaError_t launch_chan_pack(const ChanPackArgs &a, cudaStream_t stream)
{
    const long long ncell = static_cast<long long>(a.n[0]) * a.n[1] * a.n[2];
    long long blocks = (ncell + 255) / 256;
    if (blocks > 65535LL * 16) blocks = 65535LL * 16;
    if (blocks < 1) return cudaSuccess;
    ChanPackArgs args = a;
    void *params[] = {&args};
    void *k = a.dtype_in == GBD_IN_F64 ? reinterpret_cast<void *>(&chan_pack_kernel<double>)
                                       : reinterpret_cast<void *>(&chan_pack_kernel<float>);
    return cudaLaunchKernel(k, dim3(static_cast<unsigned>(blocks)), dim3(256), params, 0, stream);
}

}  // namespace gbd
