// tf_pass.cu -- the fused leapfrog in place, two passes per step (sm_103a).
//
// Algorithm 1 (arXiv 2305.13419, Sec. 3) in its fused leapfrog form is
//   B pass  Bt^{n+1/2} = Bt^{n-1/2} - curl(E^n)                    (CPML psi_B)
//   E pass  Jt^{n+1/2} = Jt^{n-1/2} + kt_e E^n,
//           E^{n+1}    = ca E^n + cb (curl(Bt/mu) - Jt^{n+1/2})      (CPML psi_E)
// each of which may run in place: the B pass reads its neighbours' E and only
// its own B, the E pass its neighbours' B and only its own E.
//
// A thread owns four x-adjacent points (128-bit accesses); its arithmetic is
// the packed FP32x2 add / sub / mul / fma of the single-step kernel in the
// same order, so the two give the same bits.  There is no staging, no barrier
// and no ring to fill: a pass is a launch of independent threads, each with
// one round of loads in flight.  That moves 72 bytes per point and step where
// the staged kernel moves 48, but in place (24 bytes of E and B per point
// where that one keeps two buffers), so that up to a few million points it
// all stays in the L2 cache, and a small grid is not held up by a chain of
// planes per CTA.
#include <math.h>

#include "tf_quad.cuh"

namespace tf {

namespace {

using namespace dev;

constexpr int kFT = kPassThreads;
// resident CTAs per SM: 24 warps of 80 registers (B), 20 of 96 (E), 16 of 128 (kEarly), no spills
constexpr int kBMin = 6, kEMin = 5, kEarlyMin = 4;

// profile of the x axis at a quad, zero off its slab lanes
__device__ __forceinline__ Q4 prof_x(const float* pf, const Quad& u) {
    const Q4 z = {{0, 0}};
    return sel4(ld4(pf + u.x), z, u.sx);
}

struct PreB {
    Q4 ox, oy, oz;       // B
    Q4 p0, p1;                   // psi_B pair of the first slab axis of z, x, y
    Q4 x0, x1, y0, y1, fb, fc;   // kEarly: the pairs of x and y and the x profiles (else when they are used)
    float bz, cz, by, cy;        // CPML coefficients of the plane and the row
};
template <bool kEarly>
__device__ __forceinline__ void pre_b(const Params& P, const Quad& u, PreB& r) {
    r.ox = own4(P.B[0], u.o);
    r.oy = own4(P.B[1], u.o);
    r.oz = own4(P.B[2], u.o);
    if (u.sz) {
        r.p0 = own4(P.psiB[0][2], u.o);
        r.p1 = own4(P.psiB[1][2], u.o);
        r.bz = __ldg(P.pbB[2] + u.k);
        r.cz = __ldg(P.pcB[2] + u.k);
    } else if (u.sx) {
        r.p0 = own4(P.psiB[1][0], u.o);
        r.p1 = own4(P.psiB[2][0], u.o);
    } else if (u.sy) {
        r.p0 = own4(P.psiB[0][1], u.o);
        r.p1 = own4(P.psiB[2][1], u.o);
    }
    if (u.sy) {
        r.by = __ldg(P.pbB[1] + u.j);
        r.cy = __ldg(P.pcB[1] + u.j);
    }
    if (kEarly) {
        if (u.sx) {
            r.fb = prof_x(P.pbB[0], u);
            r.fc = prof_x(P.pcB[0], u);
            if (u.sz) {
                r.x0 = own4(P.psiB[1][0], u.o);
                r.x1 = own4(P.psiB[2][0], u.o);
            }
        }
        if (u.sy && (u.sz || u.sx)) {
            r.y0 = own4(P.psiB[0][1], u.o);
            r.y1 = own4(P.psiB[2][1], u.o);
        }
    }
}
// CPML memory pair: n = b psi + c d, stored on the lanes of m
__device__ __forceinline__ void psi_new(float* w1, float* w2, unsigned o, const Q4& b, const Q4& c, const Q4& o1,
                                        const Q4& o2, const Q4& d1, const Q4& d2, unsigned m1, unsigned m2, Q4& n1,
                                        Q4& n2) {
    n1 = fma4(b, o1, mul4(c, d1));
    n2 = fma4(b, o2, mul4(c, d2));
    st4m((float*)((char*)w1 + o), n1, o1, m1);
    st4m((float*)((char*)w2 + o), n2, o2, m2);
}

template <bool kEarly>
__device__ __forceinline__ void post_b(const Params& P, const Quad& u, const PreB& r) {
    const unsigned o = u.o, row = 4u * (unsigned)P.pitch, pl = 4u * (unsigned)P.plane;
    unsigned oy1 = o + row, oz1 = o + pl, on = o + 16u;
    if (u.j + 1 == P.N[1]) oy1 = o - (unsigned)u.j * row;
    if (u.k + 1 == P.N[2]) oz1 = o - (unsigned)u.k * pl;
    // the point past the quad; at the row's end the wrap to x = 0 (on a walled axis: nothing keeps it)
    if (u.x + 4 >= P.N[0]) on = o - 4u * (unsigned)u.x;
    const bool wrap = P.per[0] && u.x + 4 > P.N[0];
    const Q4 ex = ldo(P.E[0], o), ey = ldo(P.E[1], o), ez = ldo(P.E[2], o);
    const Q4 ex_y = ldo(P.E[0], oy1), ez_y = ldo(P.E[2], oy1);
    const Q4 ex_z = ldo(P.E[0], oz1), ey_z = ldo(P.E[1], oz1);
    const float ey_n = ldf(P.E[1], on), ez_n = ldf(P.E[2], on);
    Q4 ey_x = up4(ey, ey_n), ez_x = up4(ez, ez_n);
    if (wrap) {   // the row ends inside the quad: its last point wraps
        ey_x = set_lane(ey_x, P.N[0] - 1 - u.x, ey_n);
        ez_x = set_lane(ez_x, P.N[0] - 1 - u.x, ez_n);
    }
    const Q4 r0 = all4(P.r[0]), r1 = all4(P.r[1]), r2 = all4(P.r[2]);
    const Q4 dEz_y = sub4(ez_y, ez), dEx_y = sub4(ex_y, ex), dEy_z = sub4(ey_z, ey), dEx_z = sub4(ex_z, ex);
    const Q4 dEz_x = sub4(ez_x, ez), dEy_x = sub4(ey_x, ey);
    Q4 bx = fma4(r2, dEy_z, sub4(r.ox, mul4(r1, dEz_y)));
    Q4 by = fma4(r0, dEz_x, sub4(r.oy, mul4(r2, dEx_z)));
    Q4 bz = fma4(r1, dEx_y, sub4(r.oz, mul4(r0, dEy_x)));
    const unsigned mx = u.in, my = u.iny ? u.hv : 0u, mz = u.inz ? u.hv : 0u;
    Q4 n1, n2;
    if (u.sz) {
        psi_new(P.psiB[0][2], P.psiB[1][2], o, all4(r.bz), all4(r.cz), r.p0, r.p1,
                dEy_z, dEx_z, mx, my, n1, n2);
        bx = add4(bx, n1);
        by = sub4(by, n2);
    }
    if (u.sx) {
        const Q4 o1 = !u.sz ? r.p0 : kEarly ? r.x0 : ldo(P.psiB[1][0], o);
        const Q4 o2 = !u.sz ? r.p1 : kEarly ? r.x1 : ldo(P.psiB[2][0], o);
        const Q4 fb = kEarly ? r.fb : prof_x(P.pbB[0], u), fc = kEarly ? r.fc : prof_x(P.pcB[0], u);
        psi_new(P.psiB[1][0], P.psiB[2][0], o, fb, fc, o1, o2, dEz_x, dEy_x,
                u.sx & my, u.sx & mz, n1, n2);
        by = add4(by, n1);
        bz = sub4(bz, n2);
    }
    if (u.sy) {
        const bool late = u.sz || u.sx;
        const Q4 o1 = !late ? r.p0 : kEarly ? r.y0 : ldo(P.psiB[0][1], o);
        const Q4 o2 = !late ? r.p1 : kEarly ? r.y1 : ldo(P.psiB[2][1], o);
        psi_new(P.psiB[0][1], P.psiB[2][1], o, all4(r.by), all4(r.cy), o1, o2,
                dEz_y, dEx_y, mx, mz, n1, n2);
        bx = sub4(bx, n1);
        bz = add4(bz, n2);
    }
    if (!u.full) {
        bx = sel4(bx, r.ox, mx);
        by = sel4(by, r.oy, my);
        bz = sel4(bz, r.oz, mz);
    }
    sto(P.B[0], o, bx);
    sto(P.B[1], o, by);
    sto(P.B[2], o, bz);
}

struct PreE {
    Q4 ex, ey, ez;               // E
    Q4 p0, p1;                   // psi_E pair of the first slab axis of z, x, y
    Q4 x0, x1, y0, y1, fb, fc;   // kEarly: the pairs of x and y, the x profiles, Js (else when they are used)
    Q4 jx, jy, jz;
    float bz, cz, by, cy;        // CPML coefficients of the plane and the row
    float4 rec;
};
template <bool kEarly>
__device__ __forceinline__ void pre_e(const PassArgs& A, const Quad& u, PreE& r) {
    const Params& P = A.P;
    r.rec = __ldg(A.tilemat + (long long)((u.j / kSY) * A.ntx + u.x / kSX) * P.N[2] + u.k);
    // Ex and Ey of the low z wall are held, or a Mur update's, by the threads of
    // the plane above during this very pass: none of this one's business
    const Q4 z = {{0, 0}};
    r.ex = u.inz ? own4(P.E[0], u.o) : z;
    r.ey = u.inz ? own4(P.E[1], u.o) : z;
    r.ez = own4(P.E[2], u.o);
    if (u.sz) {
        r.p0 = own4(P.psiE[0][2], u.o);
        r.p1 = own4(P.psiE[1][2], u.o);
        r.bz = __ldg(P.pbE[2] + u.k);
        r.cz = __ldg(P.pcE[2] + u.k);
    } else if (u.sx) {
        r.p0 = own4(P.psiE[1][0], u.o);
        r.p1 = own4(P.psiE[2][0], u.o);
    } else if (u.sy) {
        r.p0 = own4(P.psiE[0][1], u.o);
        r.p1 = own4(P.psiE[2][1], u.o);
    }
    if (u.sy) {
        r.by = __ldg(P.pbE[1] + u.j);
        r.cy = __ldg(P.pcE[1] + u.j);
    }
    if (kEarly) {
        if (u.sx) {
            r.fb = prof_x(P.pbE[0], u);
            r.fc = prof_x(P.pcE[0], u);
            if (u.sz) {
                r.x0 = own4(P.psiE[1][0], u.o);
                r.x1 = own4(P.psiE[2][0], u.o);
            }
        }
        if (u.sy && (u.sz || u.sx)) {
            r.y0 = own4(P.psiE[0][1], u.o);
            r.y1 = own4(P.psiE[2][1], u.o);
        }
        if (r.rec.z > 0.f) {
            r.jx = own4(P.J[0], u.o);
            r.jy = own4(P.J[1], u.o);
            r.jz = own4(P.J[2], u.o);
        }
    }
}

template <bool kEarly>
__device__ __forceinline__ void post_e(const PassArgs& A, const Quad& u, const PreE& r, const PassAmps& W) {
    const Params& P = A.P;
    const unsigned o = u.o, row = 4u * (unsigned)P.pitch, pl = 4u * (unsigned)P.plane;
    unsigned oy1 = o - row, oz1 = o - pl, op = o - 4u;
    // below a low wall: the own value, whose difference nothing keeps
    if (u.j == 0) oy1 = P.per[1] ? o + (unsigned)(P.N[1] - 1) * row : o;
    if (u.k == 0) oz1 = P.per[2] ? o + (unsigned)(P.N[2] - 1) * pl : o;
    if (u.x == 0) op = P.per[0] ? o + 4u * (unsigned)(P.N[0] - 1) : o;
    const Q4 hx = ldo(P.B[0], o), hy = ldo(P.B[1], o), hz = ldo(P.B[2], o);
    const Q4 hx_zm = ldo(P.B[0], oz1), hy_zm = ldo(P.B[1], oz1);
    const Q4 hx_ym = ldo(P.B[0], oy1), hz_ym = ldo(P.B[2], oy1);
    const float hy_p = ldf(P.B[1], op), hz_p = ldf(P.B[2], op);
    // (the first use of the record: every load above is on its way by now)
    const bool coef = isnan(r.rec.x), sc = r.rec.z > 0.f;   // per-point coefficients; Js advances on the tile-plane
    Q4 dHz_y, dHy_z, dHx_z, dHz_x, dHy_x, dHx_y;
    if (P.uniform_mu) {
        dHz_y = sub4(hz, hz_ym);
        dHy_z = sub4(hy, hy_zm);
        dHx_z = sub4(hx, hx_zm);
        dHz_x = sub4(hz, dn4(hz, hz_p));
        dHy_x = sub4(hy, dn4(hy, hy_p));
        dHx_y = sub4(hx, hx_ym);
    } else {
        // differences of H = B / mu, rounded as the single-step kernel's: both
        // products on their own (rnd4: no product may move into a fused
        // multiply-add), but for dHx_y where the tile-plane's material varies
        const Q4 wx = ldo(A.imu[0], o), wy = ldo(A.imu[1], o), wz = ldo(A.imu[2], o);
        auto diff = [&](const Q4& h, const Q4& w, const Q4& hm, const Q4& wm) { return sub4(rnd4(h, w), rnd4(hm, wm)); };
        dHz_y = diff(hz, wz, hz_ym, ldo(A.imu[2], oy1));
        const Q4 wx_y = ldo(A.imu[0], oy1);
        dHx_y = coef ? fma4(neg4(hx_ym), wx_y, rnd4(hx, wx)) : diff(hx, wx, hx_ym, wx_y);
        dHy_z = diff(hy, wy, hy_zm, ldo(A.imu[1], oz1));
        dHx_z = diff(hx, wx, hx_zm, ldo(A.imu[0], oz1));
        dHz_x = diff(hz, wz, dn4(hz, hz_p), dn4(wz, ldf(A.imu[2], op)));
        dHy_x = diff(hy, wy, dn4(hy, hy_p), dn4(wy, ldf(A.imu[1], op)));
    }
    const Q4 r0 = all4(P.r[0]), r1 = all4(P.r[1]), r2 = all4(P.r[2]);
    Q4 cx = sub4(mul4(r1, dHz_y), mul4(r2, dHy_z));
    Q4 cy = sub4(mul4(r2, dHx_z), mul4(r0, dHz_x));
    Q4 cz = sub4(mul4(r0, dHy_x), mul4(r1, dHx_y));
    const unsigned mx = u.iny && u.inz ? u.hv : 0u, my = u.inz ? u.in : 0u, mz = u.iny ? u.in : 0u;
    Q4 n1, n2;
    if (u.sz) {
        psi_new(P.psiE[0][2], P.psiE[1][2], o, all4(r.bz), all4(r.cz), r.p0, r.p1,
                dHy_z, dHx_z, mx, my, n1, n2);
        cx = sub4(cx, n1);
        cy = add4(cy, n2);
    }
    if (u.sx) {
        const Q4 o1 = !u.sz ? r.p0 : kEarly ? r.x0 : ldo(P.psiE[1][0], o);
        const Q4 o2 = !u.sz ? r.p1 : kEarly ? r.x1 : ldo(P.psiE[2][0], o);
        const Q4 fb = kEarly ? r.fb : prof_x(P.pbE[0], u), fc = kEarly ? r.fc : prof_x(P.pcE[0], u);
        psi_new(P.psiE[1][0], P.psiE[2][0], o, fb, fc, o1, o2, dHz_x, dHy_x,
                u.sx & my, u.sx & mz, n1, n2);
        cy = sub4(cy, n1);
        cz = add4(cz, n2);
    }
    if (u.sy) {
        const bool late = u.sz || u.sx;
        const Q4 o1 = !late ? r.p0 : kEarly ? r.y0 : ldo(P.psiE[0][1], o);
        const Q4 o2 = !late ? r.p1 : kEarly ? r.y1 : ldo(P.psiE[2][1], o);
        psi_new(P.psiE[0][1], P.psiE[2][1], o, all4(r.by), all4(r.cy), o1, o2,
                dHz_y, dHx_y, mx, mz, n1, n2);
        cx = add4(cx, n1);
        cz = sub4(cz, n2);
    }
    if (sc) {
        const Q4 ojx = kEarly ? r.jx : ldo(P.J[0], o), ojy = kEarly ? r.jy : ldo(P.J[1], o),
                 ojz = kEarly ? r.jz : ldo(P.J[2], o);
        Q4 jx, jy, jz;
        if (coef) {
            jx = fma4(ldo(P.cj[0], o), r.ex, ojx);
            jy = fma4(ldo(P.cj[1], o), r.ey, ojy);
            jz = fma4(ldo(P.cj[2], o), r.ez, ojz);
        } else {
            const Q4 cj = all4(r.rec.z);
            jx = fma4(cj, r.ex, ojx);
            jy = fma4(cj, r.ey, ojy);
            jz = fma4(cj, r.ez, ojz);
        }
        cx = sub4(cx, jx);
        cy = sub4(cy, jy);
        cz = sub4(cz, jz);
        st4m((float*)((char*)P.J[0] + o), jx, ojx, mx);
        st4m((float*)((char*)P.J[1] + o), jy, ojy, my);
        st4m((float*)((char*)P.J[2] + o), jz, ojz, mz);
    }
    Q4 nx, ny, nz;
    if (coef) {
        const Q4 bx = ldo(P.cb[0], o), by = ldo(P.cb[1], o), bz = ldo(P.cb[2], o);
        if (r.rec.y > 0.f) {   // no conductor on the tile-plane: ca = 1
            nx = fma4(bx, cx, r.ex);
            ny = fma4(by, cy, r.ey);
            nz = fma4(bz, cz, r.ez);
        } else {
            nx = fma4(bx, cx, mul4(ldo(P.ca[0], o), r.ex));
            ny = fma4(by, cy, mul4(ldo(P.ca[1], o), r.ey));
            nz = fma4(bz, cz, mul4(ldo(P.ca[2], o), r.ez));
        }
    } else {
        const Q4 ca = all4(r.rec.x), cb = all4(r.rec.y);
        nx = fma4(cb, cx, mul4(ca, r.ex));
        ny = fma4(cb, cy, mul4(ca, r.ey));
        nz = fma4(cb, cz, mul4(ca, r.ez));
    }
    const Sources& S = A.S;
    float* const* hist = W.hist;
    if (S.n > 0 && u.x + 3 >= S.bb_lo[0] && u.x < S.bb_hi[0] && u.j >= S.bb_lo[1] && u.j < S.bb_hi[1] &&
        u.k >= S.bb_lo[2] && u.k < S.bb_hi[2])
        add_src(S, W, u.x, u.j, u.k, nx, ny, nz);
    if (u.full) {
        sto(P.E[0], o, nx);
        sto(P.E[1], o, ny);
        sto(P.E[2], o, nz);
    } else {   // (a component held on a low z wall plane is not stored: a Mur update of that wall is another thread's)
        nx = sel4(nx, r.ex, mx);
        ny = sel4(ny, r.ey, my);
        nz = sel4(nz, r.ez, mz);
        if (mx) sto(P.E[0], o, nx);
        if (my) sto(P.E[1], o, ny);
        if (mz) sto(P.E[2], o, nz);
    }
    if (hist[0]) {   // (what the adjoint reads of it: the advanced edges)
        sto(hist[0], o, nx);
        sto(hist[1], o, ny);
        sto(hist[2], o, nz);
    }
    const Q4 sum = add4(add4(nx, ny), nz);
    if (!isfinite(lo(sum.v[0]) + hi(sum.v[0])) || !isfinite(lo(sum.v[1]) + hi(sum.v[1])))
        atomicOr(P.status, kStatusNonFinite);
    // first-order Mur on the z walls: E_w^{n+1} = E_i^n + M (E_i^{n+1} - E_w^n)
    if (P.bc[2] == TF_BC_MUR && (u.k == 1 || u.k == P.n[2] - 1)) {
        const unsigned wx = u.iny ? u.hv : 0u, wy = u.in;
#pragma unroll
        for (int w = 0; w < 2; ++w) {
            if (u.k != (w ? P.n[2] - 1 : 1)) continue;
            const unsigned ow = w ? o + pl : o - pl;
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                float* e0 = (float*)((char*)P.E[0] + ow) + p;
                float* e1 = (float*)((char*)P.E[1] + ow) + p;
                if (wx >> p & 1u) *e0 = lane(r.ex, p) + P.mur_M * (lane(nx, p) - *e0);
                if (wy >> p & 1u) *e1 = lane(r.ey, p) + P.mur_M * (lane(ny, p) - *e1);
            }
        }
    }
}

struct Item {
    bool live;
    Quad u;
};
// the thread's quad in a launch over planes [k0, k1)
__device__ __forceinline__ Item item_at(const PassArgs& A, int k0, int k1) {
    Item it;
    const int tid = threadIdx.x;
    const int iq = tid & ((1 << A.sa) - 1), jr = (tid >> A.sa) & ((1 << A.sb) - 1), kr = tid >> (A.sa + A.sb);
    const int x0 = 4 * (blockIdx.x << A.sa), y0 = blockIdx.y << A.sb, z0 = k0 + (blockIdx.z << A.sc);
    const int x = x0 + 4 * iq, j = y0 + jr, k = z0 + kr;
    it.live = x < A.cx && j < A.cy && k < k1;
    it.u = quad_of(A.P, x, j, k);
    return it;
}
__device__ __forceinline__ void sample(const PassArgs& A, int t, int k0, int k1) {
    const int p = threadIdx.x;
    if (p < A.nprobe && A.pr_item[p] == (int)(blockIdx.y * A.nbx + blockIdx.x) && A.pr_k[p] >= k0 && A.pr_k[p] < k1 &&
        (A.pr_k[p] - k0) >> A.sc == (int)blockIdx.z)
        A.samples[t * TF_MAX_PROBES + p] = A.P.E[A.pr_comp[p]][A.pr_q[p]];
}

}  // namespace

// One pass of one step over the planes [k0, k1) (kE: the E pass).  Bound by the latency
// of its one round of loads on small grids (two launches, 7.5 us a step on the
// 128 x 64 x 40 CPW) and by memory on large ones: over the whole 512 x 256 x 128
// CPW it takes 234 us a step (6.2 TB/s of 72 bytes per point plus the CPML
// memories), 189 in windows of planes (below: L2 to SM traffic and the
// launches' ends), on the 256 x 128 x 64 CPW, whose 90 MB nearly stay in L2, 31.  What is spilled goes to
// L2 and back: with all three slab axes' memories and Js fetched up front the E
// pass spilled 170 bytes a thread (252 and 43 us); now the first slab axis is
// fetched early, the others and Js where they are used.  A step of the latter
// grid took 41 us while its random substrate read ca, cj and Js as well; the
// tile-planes' records say where ca is 1 and where nothing superconducts.
// Columns of 4 planes per thread were slower (55 against 52 us then).
// kEarly fetches every slab axis' memories and Js before the launch before is
// done; it takes 128 registers, and is used where all CTAs are resident at
// once all the same: 6.5 against 7.5 us a step on the 96 x 64 x 48 CPW (576
// items), but 9.2 against 7.6 on the 128 x 64 x 40 one (640 on 608 places).
// Items off the walls, seams and slabs take the same code: a variant without
// its tests was no faster.
// Launches overlap (programmatic dependent launch): a thread fetches what
// only its own pass writes -- two launches ago or more -- before it waits
// for the launch before.  That launch lets the next one start only once its
// own wait is over, so the launch before it is complete by then.
template <bool kE, bool kEarly>
__global__ void __launch_bounds__(kFT, kEarly ? kEarlyMin : kE ? kEMin : kBMin)
    k_pass(const __grid_constant__ PassArgs A, const __grid_constant__ PassAmps W, int t, int k0, int k1) {
    const Item it = item_at(A, k0, k1);
    if constexpr (kE) {
        PreE r;
        if (it.live) pre_e<kEarly>(A, it.u, r);
        asm volatile("griddepcontrol.wait;" ::: "memory");
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        if (it.live) post_e<kEarly>(A, it.u, r, W);
    } else {
        PreB r;
        if (it.live) pre_b<kEarly>(A.P, it.u, r);
        asm volatile("griddepcontrol.wait;" ::: "memory");
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        if (it.live) post_b<kEarly>(A.P, it.u, r);
        sample(A, t, k0, k1);
    }
}

// running DFTs over the samples of a group of steps, a warp per (probe, frequency)
__global__ void __launch_bounds__(32) k_pass_probes(Probes R, const float* samples, long long level, int steps) {
    probe_dft(R, samples, blockIdx.x, blockIdx.y, level, steps);
}

// per-face 1/mu of the three components on the padded grid
__global__ void __launch_bounds__(kFT) k_face_imu(Params P, float* w0, float* w1, float* w2) {
    const long long t = (long long)blockIdx.x * kFT + threadIdx.x;
    if (t >= P.plane * P.N[2]) return;
    const int p[3] = {(int)(t % P.pitch), (int)(t / P.pitch % P.N[1]), (int)(t / P.plane)};
    const bool in = p[0] < P.N[0];
    w0[t] = in ? inv_mu_face(P, 0, p) : 0.f;
    w1[t] = in ? inv_mu_face(P, 1, p) : 0.f;
    w2[t] = in ? inv_mu_face(P, 2, p) : 0.f;
}

cudaError_t launch_face_imu(const Params& P, float* const w[3], cudaStream_t st) {
    const long long n = P.plane * P.N[2];
    k_face_imu<<<(unsigned)((n + kFT - 1) / kFT), kFT, 0, st>>>(P, w[0], w[1], w[2]);
    return cudaGetLastError();
}

cudaError_t launch_pass_probes(const Probes& R, const float* samples, long long level, int steps, cudaStream_t st) {
    k_pass_probes<<<dim3(R.n, TF_MAX_FREQS), 32, 0, st>>>(R, samples, level, steps);
    return cudaGetLastError();
}

// Windows of planes, each stepped `depth` times before the next one, so that
// what a pass reads is still in L2 from the passes before (over a whole grid
// beyond L2 every pass streams 36 bytes per point from DRAM).  The planes go up
// and a window's step u works on it shifted u planes down: the B pass of a
// plane needs E of that plane and the one above at the same level, the E pass
// B of that plane and the one below, and neither is a level ahead.  Every value
// is the one of whole passes, whatever the windows.  (A periodic z axis would
// need the last plane's neighbour before its own step.)
// us per step of CPW grids, whole / in windows of some million points, 16 steps,
// items of 2 to 4 planes:
//   512 x 256 x 128   234 / 1.5: 208, 2: 199, 2.5: 205, 3: 220, 4: 242
//   256 x 256 x 128   127 / 1: 120, 1.5: 105, 2: 102, 2.5: 105, 3: 118
//   700 x 300 x 150   (421 in two-step passes) / 1.5: 387, 1.9: 368, 2.5: 372, 3: 398
//   160 x 160 x 128    53 / 1: 48, 1.4: 44, 1.8: 42;   128^3  30 / 1: 38, 1.4: 30
// smaller windows leave the last wave of each launch emptier, larger ones leave
// L2.  8 steps instead of 16 are 1 to 3 % slower, 4 steps 4 to 7 %; one step alone
// takes the grid whole (512 x 256 x 128 CPW 268 us in windows, 640 x 640 x 190 1044).
// Items of one plane: with items of 2 or 4 planes a window of 5 leaves a fifth to
// two fifths of the threads idle (1024 x 400 x 180: 756 us a step against 900).
constexpr int kWindowSteps = 16;
// steps of a window, of `steps` in all: groups of one size
int window_steps(int win, const PassArgs& A, int steps) {
    if (win == A.kend) return 1;
    const int groups = (steps + kWindowSteps - 1) / kWindowSteps;
    return (steps + groups - 1) / groups;
}

// `steps` steps from `level`, two launches per step and window of planes, with
// the amplitudes amp[step]; a launch may start while the one before drains (it
// waits for it before it reads what that one writes: what it fetches earlier
// was last written by a launch of its own kind, two launches ago or more)
cudaError_t launch_passes(const PassArgs& A, const Probes& R, const PassAmps* amp, long long level, int steps,
                          cudaStream_t st) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(A.nbx, A.nby, A.nbz);
    cfg.blockDim = dim3(kFT);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    const bool early = A.nbx * A.nby * A.nbz <= kEarlyMin * A.sms;
    const int win = steps > 1 ? A.win : A.kend, depth = window_steps(win, A, steps);
    cfg.numAttrs = 0;   // the first launch waits for whatever the stream holds
    cudaError_t e = cudaSuccess;
    for (int t0 = 0; t0 < steps; t0 += depth) {
        const int m = steps - t0 < depth ? steps - t0 : depth;
        for (int z = 0; z < A.kend + m - 1; z += win)
            for (int u = 0; u < m && e == cudaSuccess; ++u) {
                const int k0 = z > u ? z - u : 0, k1 = z + win - u < A.kend ? z + win - u : A.kend;
                if (k0 >= k1) continue;
                const PassAmps& W = amp[t0 + u];
                cfg.gridDim.z = ((k1 - k0 - 1) >> A.sc) + 1;
                e = early ? cudaLaunchKernelEx(&cfg, k_pass<false, true>, A, W, t0 + u, k0, k1)
                          : cudaLaunchKernelEx(&cfg, k_pass<false, false>, A, W, t0 + u, k0, k1);
                cfg.numAttrs = 1;
                if (e == cudaSuccess)
                    e = early ? cudaLaunchKernelEx(&cfg, k_pass<true, true>, A, W, t0 + u, k0, k1)
                              : cudaLaunchKernelEx(&cfg, k_pass<true, false>, A, W, t0 + u, k0, k1);
            }
    }
    if (e == cudaSuccess && R.n > 0) e = launch_pass_probes(R, A.samples, level, steps, st);
    return e;
}

}  // namespace tf
