// gravity_noalloc.cu -- softened direct-sum gravity of one set of spheres
// that allocates no memory at all.
//
// Who needs it: code that may not call cudaMalloc or any allocator -- for
// example a caller running inside someone else's memory pool or arena with a
// fixed budget, a real-time or safety-certified host loop where allocation
// after start-up is forbidden, or a plugin whose host application owns every
// device allocation.  Such a caller cannot create a dem_world (a world
// obtains its buffers at add time), but it can hand this entry point device
// buffers it already owns for the inputs and the output.
//
// The formula is the world's gravity formula (FP32 pair terms, FP64 sums;
// results agree with the world's within the mixed-precision tolerance, not
// bitwise, since the world sums symmetric tile pairs), with the j range split
// into parts: each part writes an FP64 partial sum per sphere, and a second
// kernel adds the parts in a fixed order.  Those partial sums are the only
// scratch memory, and here they live in the file-scope array
// g_na_scratch below (16 MiB), which the CUDA runtime places in device memory
// when the library is loaded; every GPU that loads the library keeps it until
// the process exits.  Host code cannot use g_na_scratch's name as a device
// address: the host-side symbol is only a stand-in, and a kernel handed it
// would fault or, where the GPU can reach host memory, silently use the wrong
// memory.  The device address is therefore looked up with
// cudaGetSymbolAddress, once per device, with that device current, on the
// first call made on it.
#include <algorithm>
#include <cstdio>
#include <mutex>

#include "dem_internal.h"

namespace {

constexpr int kNAMaxSpheres = 131072;        // largest n accepted
constexpr int kNAScratch = 4 * kNAMaxSpheres;   // partial sums: 4 parts of the largest n, more of fewer spheres
constexpr int kNABlock = 128;
constexpr int kNAFlush = 1024;
constexpr int kNAMaxDevices = 64;

// 524,288 x 32 B = 16 MiB of partial sums.
static __device__ __align__(256) dem::dbl4 g_na_scratch[kNAScratch];

std::mutex g_na_mutex;
dem::dbl4 *g_na_addr[kNAMaxDevices] = {nullptr};
int g_na_sms[kNAMaxDevices] = {0};

// Packed FP32 pairs without flushing denormals.
typedef unsigned long long na_f2;
__device__ __forceinline__ na_f2 pack2(float lo, float hi)
{
    na_f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(na_f2 v, float &lo, float &hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ na_f2 sub2(na_f2 a, na_f2 b)
{
    na_f2 d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ na_f2 mul2(na_f2 a, na_f2 b)
{
    na_f2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ na_f2 fma2(na_f2 a, na_f2 b, na_f2 c)
{
    na_f2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
// for arguments in the normal range (the softening keeps them there)
__device__ __forceinline__ float rsqrt_normal(float x)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Block (b, c): the PER x kNABlock i-spheres of block b against part c of the
// j-spheres, 128 at a time from shared memory, packed two by two (j and j + 64).
// A tile none of whose aggregate ids lies in the range of the block's takes the
// packed loop (each i-sphere duplicated into both halves: 12 f32x2 operations
// and two rsqrt for two pairs), any other the loop that compares ids (and, with
// eps = 0, looks for coincident spheres; a sphere that is not finite counts as
// every id, so that its pairs are treated as there).  Ids in any order are
// correct; contiguous aggregates leave all but one or two tiles of a block to
// the packed loop.  Measured per call, one sphere per thread, every pair
// compared and always 4 parts -> this: 10,000 spheres 129 -> 72 us, 20,001
// 390 -> 200 us, 131,072 11.9 -> 6.7 ms (below 3,000 the launches, 29 us).
template <int PER>
__global__ void __launch_bounds__(kNABlock)
k_na_partial(const float4 *__restrict__ pm, const int32_t *__restrict__ agg, int n, int jc,
             float eps2, bool softened, dem::dbl4 *scratch)
{
    constexpr int kHalf = kNABlock / 2;
    __shared__ ulonglong2 sxy[kHalf], szm[kHalf];   // (xa, xb, ya, yb), (za, zb, ma, mb)
    __shared__ int sa[kNABlock];
    __shared__ int lohi[2][kNABlock / 32][2];
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    const int i0 = blockIdx.x * (kNABlock * PER) + t;
    const int c = blockIdx.y;
    const int j0 = c * jc;
    const int j1 = min(n, j0 + jc);
    const unsigned FULL = 0xffffffffu;
    float4 xi[PER];
    int ai[PER];
    int lo = 0x7fffffff, hi = (int)0x80000000;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        const int i = i0 + k * kNABlock;
        xi[k] = i < n ? pm[i] : make_float4(0.f, 0.f, 0.f, 0.f);
        ai[k] = i < n ? agg[i] : 0;
        if (i < n) {
            const bool fin = isfinite((xi[k].x + xi[k].y) + xi[k].z);
            lo = min(lo, fin ? ai[k] : (int)0x80000000);
            hi = max(hi, fin ? ai[k] : 0x7fffffff);
        }
    }
    // range of values over the block: w is one of two buffers used in turn
    auto block_range = [&](int l, int h, int w, int &bl, int &bh) {
        l = __reduce_min_sync(FULL, l);
        h = __reduce_max_sync(FULL, h);
        if (lane == 0) {
            lohi[w][wid][0] = l;
            lohi[w][wid][1] = h;
        }
        __syncthreads();
        bl = lohi[w][0][0];
        bh = lohi[w][0][1];
        for (int k = 1; k < kNABlock / 32; ++k) {
            bl = min(bl, lohi[w][k][0]);
            bh = max(bh, lohi[w][k][1]);
        }
    };
    int ilo, ihi;
    block_range(lo, hi, 0, ilo, ihi);
    const na_f2 e2 = pack2(eps2, eps2);
    na_f2 ax[PER] = {}, ay[PER] = {}, az[PER] = {};
    double d[PER][3] = {};
    auto flush = [&] {
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            float u, v;
            unpack2(ax[k], u, v);
            d[k][0] += u + v;
            unpack2(ay[k], u, v);
            d[k][1] += u + v;
            unpack2(az[k], u, v);
            d[k][2] += u + v;
            ax[k] = ay[k] = az[k] = 0;
        }
    };
    int since = 0, buf = 1;
    for (int jt = j0; jt < j1; jt += kNABlock) {
        const int j = jt + t;
        const bool in = j < j1;
        const float4 v = in ? pm[j] : make_float4(1.0e18f, 1.0e18f, 1.0e18f, 0.f);
        const int ag = in ? agg[j] : 0;
        const bool fin = isfinite((v.x + v.y) + v.z);
        __syncthreads();   // the previous tile has been used
        float *q = (float *)(sxy + (t & (kHalf - 1))) + t / kHalf, *r = (float *)(szm + (t & (kHalf - 1))) + t / kHalf;
        q[0] = v.x; q[2] = v.y; r[0] = v.z; r[2] = v.w;
        sa[t] = ag;
        int jlo, jhi;
        block_range(!in ? 0x7fffffff : fin ? ag : (int)0x80000000, !in ? (int)0x80000000 : fin ? ag : 0x7fffffff, buf,
                    jlo, jhi);   // (synchronises)
        buf ^= 1;
        const int nj = min(kNABlock, j1 - jt), np = min(kHalf, nj);   // j-spheres, pairs of the tile
        if (softened && (jlo > ihi || jhi < ilo)) {
            na_f2 px[PER], py[PER], pz[PER];
#pragma unroll
            for (int k = 0; k < PER; ++k) {
                px[k] = pack2(xi[k].x, xi[k].x);
                py[k] = pack2(xi[k].y, xi[k].y);
                pz[k] = pack2(xi[k].z, xi[k].z);
            }
#pragma unroll 8
            for (int jj = 0; jj < np; ++jj) {
                const ulonglong2 xy = sxy[jj], zm = szm[jj];
#pragma unroll
                for (int k = 0; k < PER; ++k) {
                    const na_f2 dx = sub2(xy.x, px[k]), dy = sub2(xy.y, py[k]), dz = sub2(zm.x, pz[k]);
                    float ra, rb;
                    unpack2(fma2(dz, dz, fma2(dy, dy, fma2(dx, dx, e2))), ra, rb);
                    const na_f2 inv = pack2(rsqrt_normal(ra), rsqrt_normal(rb));
                    const na_f2 s = mul2(mul2(zm.y, inv), mul2(inv, inv));
                    ax[k] = fma2(dx, s, ax[k]);
                    ay[k] = fma2(dy, s, ay[k]);
                    az[k] = fma2(dz, s, az[k]);
                }
            }
        } else {
#pragma unroll 2
            for (int jj = 0; jj < np; ++jj) {
                const ulonglong2 xy = sxy[jj], zm = szm[jj];
                float jx[2], jy[2], jz[2], jm[2];
                unpack2(xy.x, jx[0], jx[1]);
                unpack2(xy.y, jy[0], jy[1]);
                unpack2(zm.x, jz[0], jz[1]);
                unpack2(zm.y, jm[0], jm[1]);
                const int aj[2] = {sa[jj], sa[jj + kHalf]};
#pragma unroll
                for (int k = 0; k < PER; ++k) {
                    float s[2], ex[2], ey[2], ez[2];
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        ex[h] = jx[h] - xi[k].x;
                        ey[h] = jy[h] - xi[k].y;
                        ez[h] = jz[h] - xi[k].z;
                        const float r2 = fmaf(ez[h], ez[h], fmaf(ey[h], ey[h], fmaf(ex[h], ex[h], eps2)));
                        const float inv = rsqrtf(r2);
                        // same aggregate (and i itself): skipped; with eps = 0 two coincident
                        // spheres of different aggregates exert no force on each other
                        s[h] = (aj[h] == ai[k] || !(r2 > 0.f)) ? 0.f : (jm[h] * inv) * (inv * inv);
                    }
                    const na_f2 sv = pack2(s[0], s[1]);
                    ax[k] = fma2(pack2(ex[0], ex[1]), sv, ax[k]);
                    ay[k] = fma2(pack2(ey[0], ey[1]), sv, ay[k]);
                    az[k] = fma2(pack2(ez[0], ez[1]), sv, az[k]);
                }
            }
        }
        since += kNABlock;
        if (since >= kNAFlush) {
            since = 0;
            flush();
        }
    }
    flush();
    // every (part, sphere) slot read by k_na_combine is written here in the
    // same call, so nothing left over from an earlier call is ever read
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        const int i = i0 + k * kNABlock;
        if (i < n) scratch[(size_t)c * n + i] = dem::make_dbl4(d[k][0], d[k][1], d[k][2], 0.0);
    }
}

__global__ void k_na_combine(const double *__restrict__ mass, int n, int parts, double G,
                             const dem::dbl4 *__restrict__ scratch, dem::dbl4 *out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double sx = 0.0, sy = 0.0, sz = 0.0;
#pragma unroll 4
    for (int c = 0; c < parts; ++c) {
        const dem::dbl4 v = scratch[(size_t)c * n + i];
        sx += v.x; sy += v.y; sz += v.z;
    }
    const double gm = G * mass[i];
    out[i] = dem::make_dbl4(gm * sx, gm * sy, gm * sz, 0.0);
}

// i-spheres per thread: 2 share the shared-memory reads of the j-spheres; 1
// where that leaves too few blocks (us per call with 1 / 2: 10,000 spheres 72 /
// 78, 20,001 197 / 190, 131,072 7,370 / 6,740; 4 spilled, 252 at 20,001).
constexpr int kNAPer = 2, kNASmall = 16384;

// Parts of the j range: enough that the blocks fill the GPU twice over
// (kNABlocksPerSM resident on each SM), as many as the scratch holds, none
// shorter than 32 spheres, and at most kNAMaxParts, since k_na_combine reads
// them one after the other (3,000 spheres in 94 parts 43 us, in 20 29 us).
constexpr int kNABlocksPerSM = 10, kNAMaxParts = 24;
int na_parts(int n, int per, int sms)
{
    const int iblocks = (n + kNABlock * per - 1) / (kNABlock * per);
    const int want = 2 * kNABlocksPerSM * sms / iblocks;
    const int most = std::min({kNAScratch / n, (n + 31) / 32, kNAMaxParts});
    return std::max(1, std::min(want, most));
}

void set_msg(char *msg, size_t len, const char *text)
{
    if (msg && len) snprintf(msg, len, "%s", text);
}

}  // namespace

extern "C" dem_status dem_gravity_noalloc(const void *pos_mass, const double *mass,
                                          const int32_t *agg_id, int32_t n, double G,
                                          double eps_soft, double *force_out, void *cuda_stream,
                                          char *msg, size_t msg_len)
{
    set_msg(msg, msg_len, "");
    if (!pos_mass || !mass || !agg_id || !force_out) {
        set_msg(msg, msg_len, "dem_gravity_noalloc: NULL pointer argument");
        return DEM_ERR_ARG;
    }
    if (n < 1 || n > kNAMaxSpheres) {
        char buf[160];
        snprintf(buf, sizeof buf,
                 "dem_gravity_noalloc: n = %d outside 1..%d (the fixed scratch holds %d spheres)",
                 n, kNAMaxSpheres, kNAMaxSpheres);
        set_msg(msg, msg_len, buf);
        return DEM_ERR_ARG;
    }
    if (!(G >= 0.0) || !(eps_soft >= 0.0) || !(G < 1e300) || !(eps_soft < 1e300)) {
        set_msg(msg, msg_len, "dem_gravity_noalloc: G and eps_soft must be finite and >= 0");
        return DEM_ERR_ARG;
    }
    if ((((uintptr_t)pos_mass) & 15) || (((uintptr_t)force_out) & 31) || (((uintptr_t)mass) & 7) ||
        (((uintptr_t)agg_id) & 3)) {
        set_msg(msg, msg_len, "dem_gravity_noalloc: pos_mass must be 16-byte, force_out 32-byte, "
                              "mass 8-byte and agg_id 4-byte aligned");
        return DEM_ERR_ARG;
    }
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess || dev < 0 || dev >= kNAMaxDevices) {
        set_msg(msg, msg_len, "dem_gravity_noalloc: no usable current CUDA device");
        return DEM_ERR_CUDA;
    }
    dem::dbl4 *scratch = nullptr;
    int sms = 0;
    {
        std::lock_guard<std::mutex> lock(g_na_mutex);
        if (!g_na_addr[dev]) {
            void *p = nullptr;
            e = cudaGetSymbolAddress(&p, g_na_scratch);
            if (e != cudaSuccess || !p) {
                char buf[200];
                snprintf(buf, sizeof buf, "dem_gravity_noalloc: cudaGetSymbolAddress failed: %s",
                         cudaGetErrorString(e));
                set_msg(msg, msg_len, buf);
                return DEM_ERR_CUDA;
            }
            if (cudaDeviceGetAttribute(&g_na_sms[dev], cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
                cudaGetLastError();
                g_na_sms[dev] = 1;   // still correct, with fewer parts
            }
            g_na_addr[dev] = (dem::dbl4 *)p;
        }
        scratch = g_na_addr[dev];
        sms = g_na_sms[dev];
    }
    cudaStream_t st = (cudaStream_t)cuda_stream;
    const float eps2 = (float)(eps_soft * eps_soft);
    const int per = n <= kNASmall ? 1 : kNAPer;
    const int parts = na_parts(n, per, sms);
    const int jc = (n + parts - 1) / parts;
    const dim3 grid((n + kNABlock * per - 1) / (kNABlock * per), parts);
    const auto kernel = per == 1 ? k_na_partial<1> : k_na_partial<kNAPer>;
    kernel<<<grid, kNABlock, 0, st>>>((const float4 *)pos_mass, agg_id, n, jc, eps2, eps2 >= 1.0e-30f, scratch);
    k_na_combine<<<(n + 127) / 128, 128, 0, st>>>(mass, n, parts, G, scratch, (dem::dbl4 *)force_out);
    e = cudaGetLastError();
    if (e != cudaSuccess) {
        char buf[200];
        snprintf(buf, sizeof buf, "dem_gravity_noalloc: launch failed: %s", cudaGetErrorString(e));
        set_msg(msg, msg_len, buf);
        return DEM_ERR_CUDA;
    }
    return DEM_OK;
}
