// tf_kernels.cu -- CUDA kernels of the two-fluid Yee library for sm_103a.
//
// The per-step kernels besides the fused step of tf_step.cu:
// set-up and read-back kernels (material scaling, level-0 priming
// B^{-1/2} = B^0 + dt/2 curl E^0 and Js^{-1/2} = Js^0 - dt/2 kappa E^0, and
// integer-level read-back B^n = B^{n-1/2} - dt/2 curl E^n,
// Js^n = Js^{n-1/2} + dt/2 kappa E^n).
#include <math.h>

#include "tf_internal.cuh"

namespace tf {

namespace {

constexpr int BX = 32, BY = 4, BZ = 2;  // 256-thread blocks, x rows coalesced

__device__ __forceinline__ bool point_of(const Params& P, int& i, int& j, int& k) {
    i = blockIdx.x * BX + threadIdx.x;
    j = blockIdx.y * BY + threadIdx.y;
    k = blockIdx.z * BZ + threadIdx.z;
    return i < P.N[0] && j < P.N[1] && k < P.N[2];
}

inline dim3 grid_of(const Params& P) {
    return dim3((P.N[0] + BX - 1) / BX, (P.N[1] + BY - 1) / BY, (P.N[2] + BZ - 1) / BZ);
}

// the term of axis a in component cb of curl E at point p, from its difference dE
// (scaled units, r_a folded in), with the CPML memory advanced to the current E
// without storing it.  Every rounding is spelled out, so that a value does not
// depend on the kernel that reads it.
__device__ __forceinline__ float curl_term(const Params& P, int cb, int a, int pa, long long q, float dE) {
    const float t = __fmul_rn(P.r[a], dE);
    if (!P.psiB[cb][a] || !in_slab(P, a, pa)) return t;
    return __fadd_rn(t, __fmaf_rn(P.pbB[a][pa], P.psiB[cb][a][q], __fmul_rn(P.pcB[a][pa], dE)));
}
// component cb of curl E at the B_cb position of p
__device__ __forceinline__ float curl_E_peek(const Params& P, int cb, const int p[3], long long q) {
    float acc = 0.f;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (a == cb) continue;
        const int e = 3 - cb - a;
        int pn[3] = {p[0], p[1], p[2]};
        pn[a] = nxt(P, a, p[a]);
        const float dE = P.E[e][lin(P, pn[0], pn[1], pn[2])] - P.E[e][q];
        acc = __fadd_rn(acc, curl_sign(cb, a) * curl_term(P, cb, a, p[a], q, dE));
    }
    return acc;
}

}  // namespace

// ------------------------------------------------------------ set-up
__global__ void k_fill(float* p, long long n, float v) {
    long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    for (; t < n; t += (long long)gridDim.x * blockDim.x) p[t] = v;
}

__global__ void k_convert_materials(Params P, const float* eps_r, const float* mu_r, const float* lam,
                                    const float* sigma, double dt, float* eps, float* sig, float* kap,
                                    float* mu, unsigned* mm) {
    const long long ncell = (long long)P.n[0] * P.n[1] * P.n[2];
    const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    unsigned a_bits = 0, b_bits = 0, nonuni = 0;
    if (t < ncell) {
        const int i = (int)(t % P.n[0]);
        const long long r = t / P.n[0];
        const int j = (int)(r % P.n[1]);
        const int k = (int)(r / P.n[1]);
        const double e = eps_r ? (double)eps_r[t] : 1.0, u = mu_r ? (double)mu_r[t] : 1.0;
        const double l = lam ? (double)lam[t] : 0.0, s = sigma ? (double)sigma[t] : 0.0;
        if (!(e > 0.0) || !(u > 0.0) || !(s >= 0.0) || !(l >= 0.0) || isinf(e) || isinf(u) || isinf(s))
            atomicOr(P.status, kStatusBadMaterial);
        const double c0dt = kC0 * dt;
        // first London equation: kt = dt^2/(eps0 lambda^2 mu0 mu_r) = (c0 dt / lambda)^2 / mu_r
        const double kt = (l > 0.0 && isfinite(l)) ? (c0dt / l) * (c0dt / l) / u : 0.0;
        const long long q = lin(P, i, j, k);
        eps[q] = (float)e;
        sig[q] = (float)(s * dt / kEps0);
        kap[q] = (float)kt;
        mu[q] = (float)u;
        if (e > 0.0 && u > 0.0) {
            a_bits = __float_as_uint((float)(1.0 / (e * u)));
            b_bits = __float_as_uint((float)(kt / (4.0 * e)));
        }
        nonuni = (u != 1.0);
    }
    // non-negative floats order like their bit patterns
    a_bits = __reduce_max_sync(0xffffffffu, a_bits);
    b_bits = __reduce_max_sync(0xffffffffu, b_bits);
    nonuni = __reduce_or_sync(0xffffffffu, nonuni);
    if ((threadIdx.x & 31) == 0) {
        atomicMax(mm + 0, a_bits);
        atomicMax(mm + 1, b_bits);
        if (nonuni) atomicOr(mm + 2, 1u);
    }
}

__global__ void k_set_field(Params P, int comp, const float* dense, float* dst, double scale) {
    const long long tot = (long long)P.N[0] * P.N[1] * P.N[2];
    const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (t >= tot) return;
    const int i = (int)(t % P.N[0]);
    const long long r = t / P.N[0];
    const int p[3] = {i, (int)(r % P.N[1]), (int)(r / P.N[1])};
    bool keep;
    if (comp < 3) {
        keep = upd_E(P, comp, p) || mur_E(P, comp, p);
    } else if (comp < 6) {
        keep = upd_B(P, comp - 3, p);
    } else {   // Js lives on superconducting edges only
        keep = upd_E(P, comp - 6, p);
        if (keep) {
            float eps, st, kt;
            edge_material(P, comp - 6, p, eps, st, kt);
            keep = kt > 0.f;
        }
    }
    dst[lin(P, p[0], p[1], p[2])] = keep ? (float)((double)dense[t] * scale) : 0.f;
}

// after new materials: Js is zero on every edge that is not superconducting
__global__ void k_mask_js(Params P) {
    int i, j, k;
    if (!point_of(P, i, j, k)) return;
    const int p[3] = {i, j, k};
    const long long q = lin(P, i, j, k);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        bool keep = upd_E(P, c, p);
        if (keep) {
            float eps, st, kt;
            edge_material(P, c, p, eps, st, kt);
            keep = kt > 0.f;
        }
        if (!keep) P.J[c][q] = 0.f;
    }
}

__global__ void k_prime(Params P) {
    int i, j, k;
    if (!point_of(P, i, j, k)) return;
    const int p[3] = {i, j, k};
    const long long q = lin(P, i, j, k);
#pragma unroll
    for (int cb = 0; cb < 3; ++cb)
        if (upd_B(P, cb, p)) P.B[cb][q] += 0.5f * curl_E_peek(P, cb, p, q);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        float jt = 0.f;
        if (upd_E(P, c, p)) {
            float eps, st, kt;
            edge_material(P, c, p, eps, st, kt);
            if (kt > 0.f) jt = P.J[c][q] - 0.5f * kt * P.E[c][q];
        }
        P.J[c][q] = jt;
    }
}

// (float)(v * scale) of FP64 arithmetic, whose pipe takes 48 cycles per warp, with
// FP32's: the scale as an unevaluated sum sh + sl, the product as p + t.  t is off
// by less than 2^-20 of itself, but where it is too small to matter; if p + t
// rounds to the same number either side of that, so does the FP64 product.  The
// others (some four in ten million), and what is no normal number or has too few
// bits below it for t, take the FP64 pipe.
struct Scale {
    float sh, sl;
    double s;
};
__device__ __forceinline__ float scaled(float v, const Scale& S) {
    const float p = __fmul_rn(v, S.sh), t = __fmaf_rn(v, S.sl, __fmaf_rn(v, S.sh, -p));
    const float lo_ = __fmaf_rn(t, 1.f - 0x1p-20f, p), hi_ = __fmaf_rn(t, 1.f + 0x1p-20f, p);
    const bool sure = lo_ == hi_ && fabsf(p) > 0x1p-100f && fabsf(p) < 0x1p127f;
    return sure ? hi_ : v == 0.f ? p : (float)((double)v * S.s);
}

// integer-level value of component c of E (kKind 0), B (1) or Js (2) at a point
template <int kKind>
__device__ __forceinline__ float read_point(const Params& P, int c, int primed, const float4* tilemat, int ntx,
                                            const int p[3], const Scale& S) {
    const int q = (int)lin(P, p[0], p[1], p[2]);
    if constexpr (kKind == 0) {
        return P.E[c][q];
    } else if constexpr (kKind == 1) {
        float b = P.B[c][q];
        if (primed && upd_B(P, c, p)) b = __fmaf_rn(-0.5f, curl_E_peek(P, c, p, q), b);
        return scaled(b, S);
    } else {
        // Js lives on superconducting edges only: none on a tile-plane
        // without a superconducting cell, nor off the tiles (walls)
        if (p[0] >= (P.per[0] ? P.N[0] : P.n[0]) || p[1] >= (P.per[1] ? P.N[1] : P.n[1])) return 0.f;
        const float4 rec = __ldg(tilemat + (long long)((p[1] / kSY) * ntx + p[0] / kSX) * P.N[2] + p[2]);
        if (!(rec.z > 0.f)) return 0.f;
        const float kt = __ldg(P.cj[c] + q);   // zero on the other edges and on edges no step advances
        if (!(kt > 0.f)) return 0.f;
        return scaled(P.J[c][q] + (primed ? 0.5f * kt * P.E[c][q] : 0.f), S);
    }
}

// four points of a row of B_c (32 apart, from i0): every load that all points
// need before the first use, at positions kept inside the row
template <int kC>
__device__ __forceinline__ void read_b_row(const Params& P, int primed, int i0, int j, int k, const Scale& S, float v[4]) {
    constexpr int a1 = kC == 0 ? 1 : 0, a2 = kC == 2 ? 1 : 2;
    const float *e1 = P.E[3 - kC - a1], *e2 = P.E[3 - kC - a2];
    const int row = (int)lin(P, 0, j, k);
    const int rows[3] = {row, (int)lin(P, 0, nxt(P, 1, j), k), (int)lin(P, 0, j, nxt(P, 2, k))};
    auto past = [&](int a, int x) { return a == 0 ? row + nxt(P, 0, x) : rows[a] + x; };
    float d1[4], d2[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int x = min(i0 + 32 * u, P.N[0] - 1);
        v[u] = P.B[kC][row + x];
        d1[u] = e1[past(a1, x)] - e1[row + x];
        d2[u] = e2[past(a2, x)] - e2[row + x];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int p[3] = {min(i0 + 32 * u, P.N[0] - 1), j, k}, q = row + p[0];
        if (primed && upd_B(P, kC, p)) {   // curl_E_peek of the loaded differences
            const float t1 = curl_sign(kC, a1) * curl_term(P, kC, a1, p[a1], q, d1[u]);
            const float t2 = curl_sign(kC, a2) * curl_term(P, kC, a2, p[a2], q, d2[u]);
            v[u] = __fmaf_rn(-0.5f, __fadd_rn(__fadd_rn(0.f, t1), t2), v[u]);
        }
        v[u] = scaled(v[u], S);
    }
}

// Read-back.  Bound by memory: a warp takes 128 points of a row, four loads of
// each array in flight per thread, the component a constant.  Nine fields of the
// 1024 x 512 x 256 CPW take 2.6 ms: E 0.18 each (5.9 TB/s), Js 0.20, B 0.46 to
// 0.51 (four arrays' worth at 4.4 TB/s), whose 0.83 were bound by instructions
// and by loads one after the other while the component was an argument and each
// point formed its curl by itself.  (9.3 ms with one thread per point, 64-bit
// divisions and three FP64 operations a point, 2 FP64 lanes per cycle and SM.)
// kRows = false: rows shorter than a warp, points in sequence.
template <int kKind, int kC, bool kRows>
__global__ void __launch_bounds__(256) k_read_field(Params P, int primed, const float4* tilemat, int ntx,
                                                    float* dense, Scale S) {
    if constexpr (kRows) {
        const int j = blockIdx.y * 8 + threadIdx.y, k = blockIdx.z, i0 = blockIdx.x * 128 + threadIdx.x;
        if (j >= P.N[1]) return;
        float* const out = dense + ((long long)k * P.N[1] + j) * P.N[0];
        float v[4];
        if constexpr (kKind == 1) {
            read_b_row<kC>(P, primed, i0, j, k, S, v);
        } else {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int p[3] = {i0 + 32 * u, j, k};
                if (p[0] < P.N[0]) v[u] = read_point<kKind>(P, kC, primed, tilemat, ntx, p, S);
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (i0 + 32 * u < P.N[0]) out[i0 + 32 * u] = v[u];
    } else {
        const unsigned t = blockIdx.x * 256u + threadIdx.x, row = t / (unsigned)P.N[0];
        const int p[3] = {(int)(t - row * (unsigned)P.N[0]), (int)(row % (unsigned)P.N[1]), (int)(row / (unsigned)P.N[1])};
        if (p[2] < P.N[2]) dense[t] = read_point<kKind>(P, kC, primed, tilemat, ntx, p, S);
    }
}

// ------------------------------------------------------------ copies
// Every part of a state in one launch (a checkpoint has up to 24), each read
// once for up to three targets: memory bound, four float4 in flight a thread's
// loop.  A gradient of 384 steps on 96 x 64 x 40 cells, whose checkpoints were
// up to 63 copies of ~2.5 us each on the host: 4.36 -> 3.6 ms.  blockIdx.y = part.
__global__ void __launch_bounds__(256) k_copy_parts(const __grid_constant__ CopyParts C) {
    const CopyParts::Part& p = C.part[blockIdx.y];
    const float4* const src = (const float4*)p.src;
    const long long step = (long long)gridDim.x * 256;
    for (long long i = (long long)blockIdx.x * 256 + threadIdx.x; i < p.n16; i += step) {
        const float4 v = src[i];
#pragma unroll
        for (int d = 0; d < 3; ++d)
            if (p.dst[d]) ((float4*)p.dst[d])[i] = v;
    }
}

// ------------------------------------------------------------ launchers
static inline unsigned blocks_for(long long n, int bs) { return (unsigned)((n + bs - 1) / bs); }

cudaError_t launch_convert_materials(const Params& P, const float* eps_r, const float* mu_r,
                                     const float* lam, const float* sigma, double dt, float* eps,
                                     float* sig, float* kap, float* mu, unsigned* mm, cudaStream_t st) {
    const long long tot = P.plane * P.N[2];
    k_fill<<<1024, 256, 0, st>>>(eps, tot, 1.f);
    k_fill<<<1024, 256, 0, st>>>(sig, tot, 0.f);
    k_fill<<<1024, 256, 0, st>>>(kap, tot, 0.f);
    k_fill<<<1024, 256, 0, st>>>(mu, tot, 1.f);
    const long long ncell = (long long)P.n[0] * P.n[1] * P.n[2];
    k_convert_materials<<<blocks_for(ncell, 256), 256, 0, st>>>(P, eps_r, mu_r, lam, sigma, dt, eps,
                                                                 sig, kap, mu, mm);
    return cudaGetLastError();
}

cudaError_t launch_copy_parts(const CopyParts& C, int sms, cudaStream_t st) {
    if (C.n < 1) return cudaSuccess;
    long long most = 1;
    for (int k = 0; k < C.n; ++k) most = C.part[k].n16 > most ? C.part[k].n16 : most;
    const long long want = (most + 1023) / 1024, cap = 8LL * sms;   // four a thread, or all CTA places for each part
    k_copy_parts<<<dim3((unsigned)(want < cap ? want : cap), C.n), 256, 0, st>>>(C);
    return cudaGetLastError();
}

cudaError_t launch_set_field(const Params& P, int comp, const float* dense, float* dst, double scale,
                             cudaStream_t st) {
    const long long tot = (long long)P.N[0] * P.N[1] * P.N[2];
    k_set_field<<<blocks_for(tot, 256), 256, 0, st>>>(P, comp, dense, dst, scale);
    return cudaGetLastError();
}

cudaError_t launch_mask_js(const Params& P, cudaStream_t st) {
    k_mask_js<<<grid_of(P), dim3(BX, BY, BZ), 0, st>>>(P);
    return cudaGetLastError();
}

cudaError_t launch_prime(const Params& P, cudaStream_t st) {
    k_prime<<<grid_of(P), dim3(BX, BY, BZ), 0, st>>>(P);
    return cudaGetLastError();
}

template <int kKind, int kC>
static void read_kernel(const Params& P, int primed, const float4* tilemat, int ntx, float* dense, const Scale& S,
                        cudaStream_t st) {
    if (P.N[0] >= 32 && P.N[1] <= 8 * 65535 && P.N[2] <= 65535) {   // (blockIdx.y and z end there)
        k_read_field<kKind, kC, true><<<dim3((P.N[0] + 127) / 128, (P.N[1] + 7) / 8, P.N[2]), dim3(32, 8), 0, st>>>(
            P, primed, tilemat, ntx, dense, S);
    } else {
        const long long tot = (long long)P.N[0] * P.N[1] * P.N[2];
        k_read_field<kKind, kC, false><<<blocks_for(tot, 256), 256, 0, st>>>(P, primed, tilemat, ntx, dense, S);
    }
}
template <int kKind>
static void read_kernel_of(const Params& P, int c, int primed, const float4* tilemat, int ntx, float* dense,
                           const Scale& S, cudaStream_t st) {
    if (c == 0)
        read_kernel<kKind, 0>(P, primed, tilemat, ntx, dense, S, st);
    else if (c == 1)
        read_kernel<kKind, 1>(P, primed, tilemat, ntx, dense, S, st);
    else
        read_kernel<kKind, 2>(P, primed, tilemat, ntx, dense, S, st);
}

cudaError_t launch_read_field(const Params& P, int comp, int primed, const float4* tilemat, int ntx, float* dense,
                              double scale, cudaStream_t st) {
    const float sh = (float)scale;
    const Scale S = {sh, (float)(scale - (double)sh), scale};
    if (comp < 3)
        read_kernel_of<0>(P, comp, primed, tilemat, ntx, dense, S, st);
    else if (comp < 6)
        read_kernel_of<1>(P, comp - 3, primed, tilemat, ntx, dense, S, st);
    else
        read_kernel_of<2>(P, comp - 6, primed, tilemat, ntx, dense, S, st);
    return cudaGetLastError();
}

}  // namespace tf
