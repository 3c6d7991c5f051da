// tf_stats.cu -- field statistics for the watchdog: sum of squares, largest
// magnitude and count of non-finite values of one stored field array.
//
// Two passes: CTAs reduce a range of rows of a z plane each to a partial (FP64
// sum of squares, FP32 max |v|, 64-bit non-finite count) in scratch memory;
// one CTA reduces the partials.  Values are scaled to SI units on the way.
#include <math.h>

#include "tf_internal.cuh"

namespace tf {

namespace {
constexpr int kStatThreads = 256;
constexpr int kStatCtas = 1216;

__device__ void block_reduce(double& s, float& m, unsigned long long& nf) {
    __shared__ double ss[kStatThreads / 32];
    __shared__ float sm[kStatThreads / 32];
    __shared__ unsigned long long sn[kStatThreads / 32];
    for (int o = 16; o > 0; o >>= 1) {
        s += __shfl_down_sync(0xffffffffu, s, o);
        m = fmaxf(m, __shfl_down_sync(0xffffffffu, m, o));
        nf += __shfl_down_sync(0xffffffffu, nf, o);
    }
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) {
        ss[w] = s;
        sm[w] = m;
        sn[w] = nf;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int i = 1; i < kStatThreads / 32; ++i) {
            s += ss[i];
            m = fmaxf(m, sm[i]);
            nf += sn[i];
        }
    }
}
}  // namespace

// the FP64 value of a float, conversions kept off the FP64 pipe (2 lanes per
// cycle and SM on this part) but for subnormal numbers
__device__ __forceinline__ double widen(float f) {
    const unsigned b = __float_as_uint(f), m = b & 0x7fffffffu;
    if (m - 0x00800000u < 0x7f000000u)
        return __hiloint2double((int)((b & 0x80000000u) | ((m >> 3) + 0x38000000u)), (int)(b << 29));
    return m == 0u ? 0.0 : (double)f;
}

// Pass 1: blockIdx.y = plane k of an (n0, n1, n2) array with row pitch `pitch`,
// blockIdx.x = a share of its rows; a warp per row (rows shorter than a warp:
// several rows per warp).  Bound by the FP64 pipe: one multiply-add per point.
// (One CTA per plane with a division and a conversion per point took 45 us on
// the 256 x 128 x 64 grid's 65 planes; now 9.)
__global__ void __launch_bounds__(kStatThreads) k_stats_planes(const float* f, int n0, int n1, int pitch,
                                                               long long plane, double scale, StatPartial* part) {
    const int k = blockIdx.y;
    const float* p = f + (long long)k * plane;
    const int j0 = (int)((long long)n1 * blockIdx.x / gridDim.x), j1 = (int)((long long)n1 * (blockIdx.x + 1) / gridDim.x);
    // 2^b >= n0 threads to a row, a warp at most
    int b = 0;
    while (b < 5 && (1 << b) < n0) ++b;
    const int i0 = threadIdx.x & ((1 << b) - 1), jr = threadIdx.x >> b, rows = kStatThreads >> b;
    double s = 0.0;
    float m = 0.f;
    unsigned long long nf = 0;
    for (int j = j0 + jr; j < j1; j += rows) {
        // 64-bit offset: a caller's row pitch may make pitch * n1 exceed 2^31
        const float* r = p + (long long)j * pitch;
        for (int i = i0; i < n0; i += 4 << b) {
            float v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int x = i + (u << b);
                v[u] = x < n0 ? r[x] : 0.f;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (!isfinite(v[u])) {
                    ++nf;
                } else {
                    const double d = widen(v[u]);
                    s = fma(d, d, s);
                    m = fmaxf(m, fabsf(v[u]));
                }
            }
        }
    }
    block_reduce(s, m, nf);
    if (threadIdx.x == 0) {
        StatPartial& o = part[(long long)k * gridDim.x + blockIdx.x];
        o.sumsq = s * scale * scale;
        o.maxabs = (double)m * fabs(scale);
        o.nonfinite = nf;
    }
}

// pass 2: one CTA reduces n partials into out
__global__ void __launch_bounds__(kStatThreads) k_stats_final(const StatPartial* part, int n, StatPartial* out) {
    __shared__ double ssum[kStatThreads], smax[kStatThreads];
    __shared__ unsigned long long snf[kStatThreads];
    double s = 0.0, mx = 0.0;
    unsigned long long nf = 0;
    for (int t = threadIdx.x; t < n; t += kStatThreads) {
        s += part[t].sumsq;
        mx = fmax(mx, part[t].maxabs);
        nf += part[t].nonfinite;
    }
    ssum[threadIdx.x] = s;
    smax[threadIdx.x] = mx;
    snf[threadIdx.x] = nf;
    __syncthreads();
    for (int o = kStatThreads / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) {
            ssum[threadIdx.x] += ssum[threadIdx.x + o];
            smax[threadIdx.x] = fmax(smax[threadIdx.x], smax[threadIdx.x + o]);
            snf[threadIdx.x] += snf[threadIdx.x + o];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        out->sumsq = ssum[0];
        out->maxabs = smax[0];
        out->nonfinite = snf[0];
    }
}

// capacity: partials that fit the scratch (at least n2).  A plane is shared
// among as many CTAs as there are partials for, up to some eight CTAs per SM of
// the largest device over all planes and no fewer than eight rows each.
cudaError_t launch_field_stats(const float* f, int n0, int n1, int n2, int pitch, long long plane, double scale,
                               StatPartial* partials, int capacity, StatPartial* out, cudaStream_t st) {
    if (n2 < 1 || capacity < n2) return cudaErrorInvalidValue;
    int share = kStatCtas / n2;
    if (share > capacity / n2) share = capacity / n2;
    if (share > n1 / 8) share = n1 / 8;
    if (share < 1) share = 1;
    for (int k = 0; k < n2; k += 65535) {   // (blockIdx.y ends there)
        const int nk = n2 - k < 65535 ? n2 - k : 65535;
        k_stats_planes<<<dim3(share, nk), kStatThreads, 0, st>>>(f + (long long)k * plane, n0, n1, pitch, plane, scale,
                                                                  partials + (long long)k * share);
    }
    k_stats_final<<<1, kStatThreads, 0, st>>>(partials, n2 * share, out);
    return cudaGetLastError();
}

}  // namespace tf

// ---------------------------------------------------------------------------
// Allocation-free variant.
//
// Some callers cannot allocate device memory at the moment they want the
// statistics: a monitoring thread that checks a running simulation for
// blow-ups must not take the CUDA allocator's lock or trigger the device-wide
// synchronisation that cudaFree implies, and a host application whose memory
// pool has already reserved (nearly) all of the device cannot get more.  For
// them the per-plane partials live in a fixed array of this file, sized for
// kNoAllocMaxPlanes planes, which every GPU that loads the library holds
// until the process exits.
// ---------------------------------------------------------------------------
#include <mutex>

namespace {

constexpr int kNoAllocMaxPlanes = 4096;
constexpr int kMaxDevices = 64;

// partials of one call followed by its result; shared by every call on a device
static __device__ __align__(256) tf::StatPartial g_stats_scratch[kNoAllocMaxPlanes + 1];

tf::StatPartial* g_scratch_addr[kMaxDevices] = {nullptr};
std::mutex g_scratch_mu;

// device address of g_stats_scratch on the current device (looked up once per device)
cudaError_t scratch_address(tf::StatPartial** out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_scratch_mu);
    if (!g_scratch_addr[dev]) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_stats_scratch);
        if (e != cudaSuccess) return e;
        g_scratch_addr[dev] = (tf::StatPartial*)p;
    }
    *out = g_scratch_addr[dev];
    return cudaSuccess;
}

}  // namespace

extern "C" tf_status tf_field_stats_noalloc(const float* field, int nx_pts, int ny_pts, int nz_pts, int pitch,
                                            double scale, double* sumsq, double* maxabs, int64_t* nonfinite,
                                            void* stream) {
    if (!field || nx_pts < 1 || ny_pts < 1 || nz_pts < 1 || pitch < nx_pts) return TF_EINVAL;
    if ((long long)nx_pts * ny_pts >= (1LL << 31)) return TF_EINVAL;
    if (nz_pts > kNoAllocMaxPlanes) return TF_EINVAL;   // beyond the fixed scratch
    tf::StatPartial* scratch = nullptr;
    if (scratch_address(&scratch) != cudaSuccess) return TF_ECUDA;
    cudaStream_t st = (cudaStream_t)stream;
    const long long plane = (long long)pitch * ny_pts;
    if (tf::launch_field_stats(field, nx_pts, ny_pts, nz_pts, pitch, plane, scale, scratch,
                               kNoAllocMaxPlanes, scratch + kNoAllocMaxPlanes, st) != cudaSuccess)
        return TF_ECUDA;
    tf::StatPartial r;
    if (cudaMemcpyAsync(&r, scratch + kNoAllocMaxPlanes, sizeof(r), cudaMemcpyDeviceToHost, st) != cudaSuccess)
        return TF_ECUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return TF_ECUDA;
    if (sumsq) *sumsq = r.sumsq;
    if (maxabs) *maxabs = r.maxabs;
    if (nonfinite) *nonfinite = (int64_t)r.nonfinite;
    return TF_OK;
}
