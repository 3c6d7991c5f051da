// tf_quad.cuh -- four x-adjacent points of a thread (tf_pass.cu, tf_narrow.cu):
// 128-bit accesses, packed FP32x2 arithmetic, the lanes that each component
// advances.
#pragma once

#include "tf_device.cuh"
#include "tf_internal.cuh"

namespace tf {
namespace dev {


// four x-adjacent values: lanes 0, 1 in v[0], lanes 2, 3 in v[1]
struct Q4 {
    f2 v[2];
};
__device__ __forceinline__ Q4 ld4(const float* p) {
    const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(p);
    return {{t.x, t.y}};
}
__device__ __forceinline__ void st4(float* p, const Q4& q) {
    *reinterpret_cast<ulonglong2*>(p) = make_ulonglong2(q.v[0], q.v[1]);
}
// lanes whose bit is set in m take nv, the others ov
__device__ __forceinline__ Q4 sel4(const Q4& nv, const Q4& ov, unsigned m) {
    return {{sel2(nv.v[0], ov.v[0], m & 3u), sel2(nv.v[1], ov.v[1], m >> 2)}};
}
// products rounded on their own
__device__ __forceinline__ Q4 rnd4(const Q4& a, const Q4& b) {
    return {{pk(__fmul_rn(lo(a.v[0]), lo(b.v[0])), __fmul_rn(hi(a.v[0]), hi(b.v[0]))),
             pk(__fmul_rn(lo(a.v[1]), lo(b.v[1])), __fmul_rn(hi(a.v[1]), hi(b.v[1])))}};
}
// store the lanes of m over the old values (the whole quad is this thread's)
__device__ __forceinline__ void st4m(float* p, const Q4& nv, const Q4& ov, unsigned m) {
    if (m == 15u)
        st4(p, nv);
    else if (m)
        st4(p, sel4(nv, ov, m));
}
// lanes shifted by one: the next higher / lower x neighbour of each lane
__device__ __forceinline__ Q4 up4(const Q4& q, float next) {
    return {{pk(hi(q.v[0]), lo(q.v[1])), pk(hi(q.v[1]), next)}};
}
__device__ __forceinline__ Q4 dn4(const Q4& q, float prev) {
    return {{pk(prev, lo(q.v[0])), pk(hi(q.v[0]), lo(q.v[1]))}};
}
__device__ __forceinline__ float lane(const Q4& q, int p) {
    const f2 v = p < 2 ? q.v[0] : q.v[1];
    return p & 1 ? hi(v) : lo(v);
}
__device__ __forceinline__ Q4 set_lane(const Q4& q, int p, float x) {
    Q4 r = q;
#pragma unroll
    for (int u = 0; u < 4; ++u)
        if (u == p) r.v[u >> 1] = u & 1 ? pk(lo(r.v[u >> 1]), x) : pk(x, hi(r.v[u >> 1]));
    return r;
}
__device__ __forceinline__ Q4 sub4(const Q4& a, const Q4& b) { return {{sub2(a.v[0], b.v[0]), sub2(a.v[1], b.v[1])}}; }
__device__ __forceinline__ Q4 add4(const Q4& a, const Q4& b) { return {{add2(a.v[0], b.v[0]), add2(a.v[1], b.v[1])}}; }
__device__ __forceinline__ Q4 mul4(const Q4& a, const Q4& b) { return {{mul2(a.v[0], b.v[0]), mul2(a.v[1], b.v[1])}}; }
__device__ __forceinline__ Q4 fma4(const Q4& a, const Q4& b, const Q4& c) {
    return {{fma2(a.v[0], b.v[0], c.v[0]), fma2(a.v[1], b.v[1], c.v[1])}};
}
__device__ __forceinline__ Q4 neg4(const Q4& a) {
    const f2 s = 0x8000000080000000ull;
    return {{a.v[0] ^ s, a.v[1] ^ s}};
}
__device__ __forceinline__ Q4 all4(float x) {
    const f2 v = pk(x, x);
    return {{v, v}};
}

// the quad of a thread: its points and the lanes each component advances
struct Quad {
    int x, j, k;
    unsigned o;          // byte offset in a field array
    unsigned hv, in;     // lanes with a half / an integer position off the walls along x
    unsigned sx;         // lanes inside the CPML slabs of the x axis
    bool iny, inz;       // the row / plane is off the low walls
    bool sy, sz;         // the row / plane is inside a CPML slab
    bool full;           // every lane of every component advances
};
__device__ __forceinline__ Quad quad_of(const Params& P, int x, int j, int k) {
    Quad u;
    u.x = x;
    u.j = j;
    u.k = k;
    u.o = 4u * (unsigned)(k * (int)P.plane + j * P.pitch + x);
    const int hx = P.per[0] ? P.N[0] : P.n[0];   // points advanced along x: [lo, hx)
    u.hv = x + 4 <= hx ? 15u : x < hx ? (1u << (hx - x)) - 1u : 0u;
    u.in = (!P.per[0] && x == 0) ? u.hv & 14u : u.hv;
    u.sx = 0u;
    const int L = P.L[0];
    if (L > 0 && (x < L || x + 3 >= P.n[0] - L)) {
#pragma unroll
        for (int p = 0; p < 4; ++p) u.sx |= (x + p < L || x + p >= P.n[0] - L) ? 1u << p : 0u;
        u.sx &= u.hv;
    }
    u.iny = P.per[1] || j >= 1;
    u.inz = P.per[2] || k >= 1;
    u.sy = in_slab(P, 1, j);
    u.sz = in_slab(P, 2, k);
    u.full = u.in == 15u && u.iny && u.inz;
    return u;
}

// soft sources of step t at a quad
__device__ __forceinline__ void add_src(const Sources& S, const PassAmps& W, int x, int j, int k, Q4& nx, Q4& ny, Q4& nz) {
    Q4 ax = {{0, 0}}, ay = ax, az = ax;
    for (int s = 0; s < S.n; ++s) {
        if (j < S.lo[s][1] || j >= S.hi[s][1] || k < S.lo[s][2] || k >= S.hi[s][2]) continue;
        const float v = W.a[s];
        const int x0 = S.lo[s][0], x1 = S.hi[s][0];
        const Q4 a = {{pk(x >= x0 && x < x1 ? v : 0.f, x + 1 >= x0 && x + 1 < x1 ? v : 0.f),
                       pk(x + 2 >= x0 && x + 2 < x1 ? v : 0.f, x + 3 >= x0 && x + 3 < x1 ? v : 0.f)}};
        if (S.comp[s] == 0)
            ax = add4(ax, a);
        else if (S.comp[s] == 1)
            ay = add4(ay, a);
        else
            az = add4(az, a);
    }
    nx = add4(nx, ax);
    ny = add4(ny, ay);
    nz = add4(nz, az);
}

// accesses at a 32-bit byte offset from a uniform base
__device__ __forceinline__ Q4 ldo(const float* base, unsigned o) { return ld4((const float*)((const char*)base + o)); }
__device__ __forceinline__ void sto(float* base, unsigned o, const Q4& q) { st4((float*)((char*)base + o), q); }
__device__ __forceinline__ float ldf(const float* base, unsigned o) { return *(const float*)((const char*)base + o); }

// own values that a pass needs and that nobody else writes: read past L1, so
// that they may be fetched while the pass before is still running elsewhere
__device__ __forceinline__ Q4 own4(const float* base, unsigned o) {
    Q4 q;
    asm volatile("ld.global.cg.v2.u64 {%0, %1}, [%2];" : "=l"(q.v[0]), "=l"(q.v[1]) : "l"((const char*)base + o) : "memory");
    return q;
}

// running DFT of probe pr at its frequency f over the samples of `steps` steps
// from `level`, in step order (the accumulation of probe_update), by one warp:
// a step per lane for the phase factors, then the two sums, one lane each, in
// sequence (a chain of 32 dependent FP64 additions; the FP64 pipe takes 16
// cycles per warp instruction)
__device__ __forceinline__ void probe_dft(const Probes& R, const float* samples, int pr, int f, long long level,
                                          int steps) {
    const int ln = threadIdx.x & 31;
    const long long n = level + ln;
    double s = 0.0, sc = 0.0, ss = 0.0;
    const bool live = ln < steps;
    if (live) {
        s = (double)samples[ln * TF_MAX_PROBES + pr];
        if (f == 0 && n < R.cap) R.series[(long long)pr * R.cap + n] = s;
    }
    if (f >= R.nfreq[pr]) return;
    const bool on = live && n >= R.n0[pr];
    if (on) {
        double ph = R.fdt[pr * TF_MAX_FREQS + f] * (double)n;
        ph -= floor(ph);
        double sn, cs;
        sincospi(2.0 * ph, &sn, &cs);
        sc = s * cs;
        ss = -(s * sn);
    }
    const unsigned who = __ballot_sync(0xffffffffu, on);
    double* const to = (ln == 0 ? R.re : R.im) + pr * TF_MAX_FREQS + f;
    double acc = ln < 2 ? *to : 0.0;
#pragma unroll
    for (int u = 0; u < 32; ++u) {
        const double a = __shfl_sync(0xffffffffu, sc, u), b = __shfl_sync(0xffffffffu, ss, u);
        if (who >> u & 1u) acc += (ln == 0 ? a : b) * R.dt;
    }
    if (ln < 2) *to = acc;
}

}  // namespace dev
}  // namespace tf
