// tf_adjoint.cu -- discrete adjoint of the fused step (sm_103a).
//
// With sources fixed, one fused step of Algorithm 1 (arXiv 2305.13419,
// Sec. 3) is a linear map of the state (E, Bt, Jt, psi_B, psi_E):
//   psi_B' = bB psi_B + cB dE              (CPML slabs, updated faces)
//   Bt'    = Bt - curl_r E - sB psi_B'      (sB(c, a) = -curl_sign(c, a))
//   Jt'    = Jt + cj E
//   psi_E' = bE psi_E + cE dH(Bt'/mu)      (CPML slabs, updated edges)
//   E'     = ca E + cb (curl_r (Bt'/mu) + sE psi_E' - Jt')   (sE = curl_sign)
// (curl_r: the Yee curls with the r_a = c0 dt / d_a weights; ca, cb, cj the
// per-edge coefficients, 1, 0, 0 on edges the step leaves alone).  Its
// transpose, applied to the adjoint state (Eh, Bh, Jh, psi_Bh, psi_Eh), is
//   e          = cb Eh'
//   psi_Eh'tot = psi_Eh' + sE e
//   Bh'tot     = Bh' + (1/mu) [transposed backward differences of
//                sE r e + cE psi_Eh'tot]                     (face pass)
//   psi_Bh'tot = bB-scaled psi_Bh' + sB Bh'tot
//   Jh         = Jh' - e
//   psi_Eh     = bE psi_Eh'tot
//   Eh         = ca Eh' + cj Jh + [transposed forward differences of
//                -curl_sign r Bh'tot + cB psi_Bh'tot]         (edge pass)
// and the gradient of the objective collects, per edge,
//   dJ/d eps_e += Eh' cb (E^n - E'_no-source)     (Alg. 1 step 3, theta scheme)
//   dJ/d kt_e  += Jh E^n                           (steps 4 + 2)
// Off the slabs the transposed differences are curls again: the face pass is
// the step's B pass with the other sign and e in the place of E, the edge
// pass its E pass with the other sign.  So both are laid out like the passes
// of tf_pass.cu (in place, four x-adjacent points per thread, overlapping
// launches); only e = cb Eh is kept between them (three arrays, zero on edges
// the step leaves alone), the weights of either pass are formed again from
// it, Bh and the CPML memories.  Jh is read where a superconducting edge is,
// and nowhere else.
#include <math.h>

#include "tf_quad.cuh"

namespace tf {

namespace {

using namespace dev;

constexpr int kAT = kPassThreads;
constexpr int kAMin = 4;   // resident CTAs per SM: 16 warps of 128 registers

// the FP64 value of a float without the FP64 pipe (2 lanes per cycle and SM
// here) but for what is no normal number
__device__ __forceinline__ double widen(float f) {
    const unsigned b = __float_as_uint(f), m = b & 0x7fffffffu;
    if (m - 0x00800000u < 0x7f000000u)
        return __hiloint2double((int)((b & 0x80000000u) | ((m >> 3) + 0x38000000u)), (int)(b << 29));
    return m == 0u ? 0.0 : (double)f;
}
__device__ __forceinline__ bool any4(const Q4& q) {
    return ((q.v[0] | q.v[1]) & 0x7fffffff7fffffffull) != 0ull;
}

// does an item keep all it reads -- its points and their neighbours on both
// sides -- off the walls, the seams and the CPML slabs?
__device__ __forceinline__ bool plain_adj(const Params& P, int x0, int x1, int y0, int y1, int z0, int z1) {
    const int a0[3] = {x0, y0, z0}, a1[3] = {x1, y1, z1};
    bool ok = P.uniform_mu;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const int lo_ = P.L[a] + 1, hi_ = P.per[a] ? P.N[a] - 1 : P.n[a] - P.L[a];
        ok = ok && a0[a] >= lo_ && a1[a] <= hi_;
    }
    return ok;
}

struct Item {
    bool live, plain;
    Quad u;
};
__device__ __forceinline__ Item item_at(const AdjArgs& A) {
    const PassArgs& G = A.G;
    Item it;
    const int tid = threadIdx.x;
    const int iq = tid & ((1 << G.sa) - 1), jr = (tid >> G.sa) & ((1 << G.sb) - 1), kr = tid >> (G.sa + G.sb);
    const int x0 = 4 * (blockIdx.x << G.sa), y0 = blockIdx.y << G.sb, z0 = blockIdx.z << G.sc;
    const int x = x0 + 4 * iq, j = y0 + jr, k = z0 + kr;
    it.live = x < G.cx && j < G.cy && k < G.kend;
    it.plain = plain_adj(G.P, x0, x0 + (4 << G.sa), y0, y0 + (1 << G.sb), z0, z0 + (1 << G.sc));
    it.u = quad_of(G.P, x, j, k);
    return it;
}

__device__ __forceinline__ void yield_launch() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// cE (psi_Eh' + sE e) at a position; neg: sE = -1
__device__ __forceinline__ Q4 wpsi(const Q4& c, const Q4& psi, const Q4& e, bool neg) {
    return mul4(c, neg ? sub4(psi, e) : add4(psi, e));
}

template <bool kPlain>
__device__ __forceinline__ void faces(const AdjArgs& A, const Quad& u) {
    const Params& P = A.G.P;
    const AdjState& S = A.S;
    const unsigned o = u.o, row = 4u * (unsigned)P.pitch, pl = 4u * (unsigned)P.plane;
    unsigned oy1 = o + row, oz1 = o + pl, on = o + 16u;
    bool wrap = false;
    if (!kPlain) {
        if (u.j + 1 == P.N[1]) oy1 = o - (unsigned)u.j * row;
        if (u.k + 1 == P.N[2]) oz1 = o - (unsigned)u.k * pl;
        if (u.x + 4 >= P.N[0]) on = o - 4u * (unsigned)u.x;
        wrap = P.per[0] && u.x + 4 > P.N[0];
    }
    const Q4 bx0 = own4(S.B[0], o), by0 = own4(S.B[1], o), bz0 = own4(S.B[2], o);
    yield_launch();
    const Q4 vx = ldo(S.V[0], o), vy = ldo(S.V[1], o), vz = ldo(S.V[2], o);
    const Q4 vx_y = ldo(S.V[0], oy1), vz_y = ldo(S.V[2], oy1);
    const Q4 vx_z = ldo(S.V[0], oz1), vy_z = ldo(S.V[1], oz1);
    const float vy_n = ldf(S.V[1], on), vz_n = ldf(S.V[2], on);
    Q4 vy_x = up4(vy, vy_n), vz_x = up4(vz, vz_n);
    if (!kPlain && wrap) {
        vy_x = set_lane(vy_x, P.N[0] - 1 - u.x, vy_n);
        vz_x = set_lane(vz_x, P.N[0] - 1 - u.x, vz_n);
    }
    const Q4 r0 = all4(P.r[0]), r1 = all4(P.r[1]), r2 = all4(P.r[2]);
    Q4 hx = sub4(mul4(r1, sub4(vz_y, vz)), mul4(r2, sub4(vy_z, vy)));
    Q4 hy = sub4(mul4(r2, sub4(vx_z, vx)), mul4(r0, sub4(vz_x, vz)));
    Q4 hz = sub4(mul4(r0, sub4(vy_x, vy)), mul4(r1, sub4(vx_y, vx)));
    if (kPlain) {
        sto(S.B[0], o, add4(bx0, hx));
        sto(S.B[1], o, add4(by0, hy));
        sto(S.B[2], o, add4(bz0, hz));
        return;
    }
    // CPML memories of the edges on both sides of the face along each slab
    // axis (past the slab's inner end the profile is zero)
    if (u.sz) {
        const Q4 c0 = all4(__ldg(P.pcE[2] + u.k)), c1 = all4(__ldg(P.pcE[2] + u.k + 1));
        hy = add4(hy, sub4(wpsi(c0, ldo(S.psiE[0][2], o), vx, true), wpsi(c1, ldo(S.psiE[0][2], oz1), vx_z, true)));
        hx = add4(hx, sub4(wpsi(c0, ldo(S.psiE[1][2], o), vy, false), wpsi(c1, ldo(S.psiE[1][2], oz1), vy_z, false)));
    }
    if (u.sx) {
        const Q4 c0 = ld4(P.pcE[0] + u.x);
        const bool next = u.x + 4 < P.N[0];
        const float cn = next ? __ldg(P.pcE[0] + u.x + 4) : 0.f;
        const float p1 = next ? ldf(S.psiE[1][0], on) : 0.f, p2 = next ? ldf(S.psiE[2][0], on) : 0.f;
        const Q4 wy = wpsi(c0, ldo(S.psiE[1][0], o), vy, true), wz = wpsi(c0, ldo(S.psiE[2][0], o), vz, false);
        hz = add4(hz, sub4(wy, up4(wy, cn * (p1 - vy_n))));
        hy = add4(hy, sub4(wz, up4(wz, cn * (p2 + vz_n))));
    }
    if (u.sy) {
        const Q4 c0 = all4(__ldg(P.pcE[1] + u.j)), c1 = all4(__ldg(P.pcE[1] + u.j + 1));
        hx = add4(hx, sub4(wpsi(c0, ldo(S.psiE[2][1], o), vz, true), wpsi(c1, ldo(S.psiE[2][1], oy1), vz_y, true)));
        hz = add4(hz, sub4(wpsi(c0, ldo(S.psiE[0][1], o), vx, false), wpsi(c1, ldo(S.psiE[0][1], oy1), vx_y, false)));
    }
    if (!P.uniform_mu) {
        hx = mul4(hx, ldo(A.G.imu[0], o));
        hy = mul4(hy, ldo(A.G.imu[1], o));
        hz = mul4(hz, ldo(A.G.imu[2], o));
    }
    const unsigned mx = u.in, my = u.iny ? u.hv : 0u, mz = u.inz ? u.hv : 0u;
    const Q4 bx = sel4(add4(bx0, hx), bx0, mx), by = sel4(add4(by0, hy), by0, my), bz = sel4(add4(bz0, hz), bz0, mz);
    sto(S.B[0], o, bx);
    sto(S.B[1], o, by);
    sto(S.B[2], o, bz);
    // psi_Bh' = bB psi_Bh' - curl_sign Bh'
    auto psi = [&](float* w, const Q4& b, const Q4& bh, bool neg, unsigned m) {
        const Q4 old = ldo(w, o), t = mul4(b, old);
        st4m((float*)((char*)w + o), neg ? sub4(t, bh) : add4(t, bh), old, m);
    };
    if (u.sz) {
        const Q4 b = all4(__ldg(P.pbB[2] + u.k));
        psi(S.psiB[0][2], b, bx, false, mx);
        psi(S.psiB[1][2], b, by, true, my);
    }
    if (u.sx) {
        const Q4 b = ld4(P.pbB[0] + u.x);
        psi(S.psiB[1][0], b, by, false, u.sx & my);
        psi(S.psiB[2][0], b, bz, true, u.sx & mz);
    }
    if (u.sy) {
        const Q4 b = all4(__ldg(P.pbB[1] + u.j));
        psi(S.psiB[0][1], b, bx, true, mx);
        psi(S.psiB[2][1], b, bz, false, mz);
    }
}

// one component of the edge pass: Jh, Eh, e and the gradient sums on the lanes of m
__device__ __forceinline__ void edge(const AdjArgs& A, const Quad& u, int e, const Q4& ep, const Q4& en, Q4 e1,
                                     const Q4& d, const Q4& ca, const Q4& cb, const Q4& cj, const Q4& ev, unsigned m) {
    const AdjState& S = A.S;
    const Sources& R = A.G.S;
    const unsigned o = u.o;
    if (R.n > 0 && u.x + 3 >= R.bb_lo[0] && u.x < R.bb_hi[0] && u.j >= R.bb_lo[1] && u.j < R.bb_hi[1] &&
        u.k >= R.bb_lo[2] && u.k < R.bb_hi[2])   // E^{n+1} without this step's soft sources
        for (int s = 0; s < R.n; ++s) {
            if (R.comp[s] != e || u.j < R.lo[s][1] || u.j >= R.hi[s][1] || u.k < R.lo[s][2] || u.k >= R.hi[s][2])
                continue;
            const float v = A.W.a[s];
            const int x0 = R.lo[s][0], x1 = R.hi[s][0];
            const Q4 a = {{pk(u.x >= x0 && u.x < x1 ? v : 0.f, u.x + 1 >= x0 && u.x + 1 < x1 ? v : 0.f),
                           pk(u.x + 2 >= x0 && u.x + 2 < x1 ? v : 0.f, u.x + 3 >= x0 && u.x + 3 < x1 ? v : 0.f)}};
            e1 = sub4(e1, a);
        }
    const Q4 de = sub4(en, e1);
    const Q4 z = {{0, 0}};
    const Q4 epm = sel4(ep, z, m);
    // dJ/d eps_e += Eh' cb (E^n - E'): FP64 sums of FP64 products; nothing to add where a factor is zero
    if (any4(epm) && any4(de)) {
        double2* const g = reinterpret_cast<double2*>(S.gE[e] + o / 4u);
        double2 g0 = g[0], g1 = g[1];
        g0.x = fma(widen(lane(epm, 0)) * widen(lane(cb, 0)), widen(lane(de, 0)), g0.x);
        g0.y = fma(widen(lane(epm, 1)) * widen(lane(cb, 1)), widen(lane(de, 1)), g0.y);
        g1.x = fma(widen(lane(epm, 2)) * widen(lane(cb, 2)), widen(lane(de, 2)), g1.x);
        g1.y = fma(widen(lane(epm, 3)) * widen(lane(cb, 3)), widen(lane(de, 3)), g1.y);
        g[0] = g0;
        g[1] = g1;
    }
    Q4 sum = d;   // Eh = ca Eh' + (cj Jh + d): one rounding of Eh's size
    const Q4 cjm = sel4(cj, z, m);
    if (any4(cjm)) {   // a superconducting edge
        const Q4 jo = ldo(S.J[e], o), jh = sub4(jo, ev);
        sto(S.J[e], o, sel4(jh, jo, m));
        sum = fma4(cj, jh, d);
        double* const g = S.gK[e] + o / 4u;
#pragma unroll
        for (int p = 0; p < 4; ++p)
            if ((m >> p & 1u) && lane(cj, p) > 0.f) g[p] = fma(widen(lane(jh, p)), widen(lane(en, p)), g[p]);
    }
    Q4 en1 = fma4(ca, ep, sum);
    if (e == A.probe_comp && A.probe_o - o < 16u) {   // the objective's derivative at the probe
        const int p = (int)(A.probe_o - o) >> 2;
        const float v = p == 0 ? lane(en1, 0) : p == 1 ? lane(en1, 1) : p == 2 ? lane(en1, 2) : lane(en1, 3);
        en1 = set_lane(en1, p, v + A.probe_src);
    }
    sto(S.E[e], o, sel4(en1, ep, m));
    sto(S.V[e], o, sel4(mul4(cb, en1), z, m));   // e of the next step back
}

template <bool kPlain>
__device__ __forceinline__ void edges(const AdjArgs& A, const Quad& u) {
    const Params& P = A.G.P;
    const AdjState& S = A.S;
    const unsigned o = u.o, row = 4u * (unsigned)P.pitch, pl = 4u * (unsigned)P.plane;
    unsigned oy1 = o - row, oz1 = o - pl, op = o - 4u;
    if (!kPlain) {   // below a low wall: nothing that an advanced edge reads
        if (u.j == 0) oy1 = P.per[1] ? o + (unsigned)(P.N[1] - 1) * row : o;
        if (u.k == 0) oz1 = P.per[2] ? o + (unsigned)(P.N[2] - 1) * pl : o;
        if (u.x == 0) op = P.per[0] ? o + 4u * (unsigned)(P.N[0] - 1) : o;
    }
    const float4 rec = __ldg(A.G.tilemat + (long long)((u.j / kSY) * A.G.ntx + u.x / kSX) * P.N[2] + u.k);
    const Q4 ex = own4(S.E[0], o), ey = own4(S.E[1], o), ez = own4(S.E[2], o);
    const Q4 nx = own4(A.En[0], o), ny = own4(A.En[1], o), nz = own4(A.En[2], o);
    const Q4 qx = own4(A.En1[0], o), qy = own4(A.En1[1], o), qz = own4(A.En1[2], o);
    yield_launch();
    const Q4 bx = ldo(S.B[0], o), by = ldo(S.B[1], o), bz = ldo(S.B[2], o);
    const Q4 bx_z = ldo(S.B[0], oz1), by_z = ldo(S.B[1], oz1);
    const Q4 bx_y = ldo(S.B[0], oy1), bz_y = ldo(S.B[2], oy1);
    const float by_p = ldf(S.B[1], op), bz_p = ldf(S.B[2], op);
    const Q4 r0 = all4(P.r[0]), r1 = all4(P.r[1]), r2 = all4(P.r[2]);
    Q4 dx = sub4(mul4(r1, sub4(bz_y, bz)), mul4(r2, sub4(by_z, by)));
    Q4 dy = sub4(mul4(r2, sub4(bx_z, bx)), mul4(r0, sub4(dn4(bz, bz_p), bz)));
    Q4 dz = sub4(mul4(r0, sub4(dn4(by, by_p), by)), mul4(r1, sub4(bx_y, bx)));
    const unsigned mx = kPlain ? 15u : u.iny && u.inz ? u.hv : 0u, my = kPlain ? 15u : u.inz ? u.in : 0u,
                   mz = kPlain ? 15u : u.iny ? u.in : 0u;
    if (!kPlain) {   // CPML memories of the faces on both sides of the edge: cB psi_Bh
        const bool sz = u.sz || (u.k > 0 && in_slab(P, 2, u.k - 1)), sy = u.sy || (u.j > 0 && in_slab(P, 1, u.j - 1));
        const int L = P.L[0];
        const bool sx = L > 0 && (u.x <= L || u.x + 3 >= P.n[0] - L);
        if (sz) {
            const Q4 c0 = all4(__ldg(P.pcB[2] + u.k)), c1 = all4(u.k > 0 ? __ldg(P.pcB[2] + u.k - 1) : 0.f);
            dx = add4(dx, sub4(mul4(c1, ldo(S.psiB[1][2], oz1)), mul4(c0, ldo(S.psiB[1][2], o))));
            dy = add4(dy, sub4(mul4(c1, ldo(S.psiB[0][2], oz1)), mul4(c0, ldo(S.psiB[0][2], o))));
        }
        if (sx) {
            const Q4 c0 = ld4(P.pcB[0] + u.x);
            const float cp = u.x > 0 ? __ldg(P.pcB[0] + u.x - 1) : 0.f;
            const Q4 w1 = mul4(c0, ldo(S.psiB[1][0], o)), w2 = mul4(c0, ldo(S.psiB[2][0], o));
            dy = add4(dy, sub4(dn4(w2, cp * ldf(S.psiB[2][0], op)), w2));
            dz = add4(dz, sub4(dn4(w1, cp * ldf(S.psiB[1][0], op)), w1));
        }
        if (sy) {
            const Q4 c0 = all4(__ldg(P.pcB[1] + u.j)), c1 = all4(u.j > 0 ? __ldg(P.pcB[1] + u.j - 1) : 0.f);
            dx = add4(dx, sub4(mul4(c1, ldo(S.psiB[2][1], oy1)), mul4(c0, ldo(S.psiB[2][1], o))));
            dz = add4(dz, sub4(mul4(c1, ldo(S.psiB[0][1], oy1)), mul4(c0, ldo(S.psiB[0][1], o))));
        }
    }
    // the coefficients that the forward step used
    const bool coef = isnan(rec.x);
    auto ca = [&](int e) { return coef ? (rec.y > 0.f ? all4(1.f) : ldo(P.ca[e], o)) : all4(rec.x); };
    auto cb = [&](int e) { return coef ? ldo(P.cb[e], o) : all4(rec.y); };
    auto cj = [&](int e) { return coef && rec.z > 0.f ? ldo(P.cj[e], o) : all4(rec.z); };
    const Q4 cbx = cb(0), cby = cb(1), cbz = cb(2);
    const Q4 vx = mul4(cbx, ex), vy = mul4(cby, ey), vz = mul4(cbz, ez);
    if (!kPlain) {   // psi_Eh = bE (psi_Eh' + sE e)
        auto psi = [&](float* w, const Q4& b, const Q4& v, bool neg, unsigned m) {
            const Q4 old = ldo(w, o);
            st4m((float*)((char*)w + o), mul4(b, neg ? sub4(old, v) : add4(old, v)), old, m);
        };
        if (u.sz) {
            const Q4 b = all4(__ldg(P.pbE[2] + u.k));
            psi(S.psiE[0][2], b, vx, true, mx);
            psi(S.psiE[1][2], b, vy, false, my);
        }
        if (u.sx) {
            const Q4 b = ld4(P.pbE[0] + u.x);
            psi(S.psiE[1][0], b, vy, true, u.sx & my);
            psi(S.psiE[2][0], b, vz, false, u.sx & mz);
        }
        if (u.sy) {
            const Q4 b = all4(__ldg(P.pbE[1] + u.j));
            psi(S.psiE[0][1], b, vx, false, mx);
            psi(S.psiE[2][1], b, vz, true, mz);
        }
    }
    if (mx) edge(A, u, 0, ex, nx, qx, dx, ca(0), cbx, cj(0), vx, mx);
    if (my) edge(A, u, 1, ey, ny, qy, dy, ca(1), cby, cj(1), vy, my);
    if (mz) edge(A, u, 2, ez, nz, qz, dz, ca(2), cbz, cj(2), vz, mz);
}

}  // namespace

// Face pass: Bh'tot and psi_Bh'tot.  Edge pass: Jh, psi_Eh, Eh, e; per-edge
// gradients; the objective's derivative at the probe.  Bound by memory: 36
// bytes a point for the faces (e; Bh read and written); 72 for the edges (Bh, Eh, E^n, E^{n+1}, e) and 48
// for the FP64 sums, with the per-point coefficients where the material
// varies.  On the 256 x 128 x 64 CPW an adjoint step (both passes; no
// recompute) takes 85 us; it took 125 with twelve stored weight arrays and
// one thread per point, most of the edge pass's 89 us on the FP64 pipe
// (five operations per edge: conversions run there too; two are left).
__global__ void __launch_bounds__(kAT, kAMin) k_adj_faces(const __grid_constant__ AdjArgs A) {
    const Item it = item_at(A);
    if (it.plain)
        faces<true>(A, it.u);
    else if (it.live)
        faces<false>(A, it.u);
    else
        yield_launch();
}

__global__ void __launch_bounds__(kAT, kAMin) k_adj_edges(const __grid_constant__ AdjArgs A) {
    const Item it = item_at(A);
    if (it.plain)
        edges<true>(A, it.u);
    else if (it.live)
        edges<false>(A, it.u);
    else
        yield_launch();
}

// per cell: dJ/d eps_r and dJ/d lambda_L from the per-edge sums, with the
// weights of the edge rule (eps: mean of 4 cells; kt: mean over the 4 cells
// or over the superconducting ones); `unscale` undoes the seed's scaling
__global__ void __launch_bounds__(256) k_adj_cells(Params P, AdjState A, float dt_c0, double unscale, float* g_eps,
                                                   float* g_lam) {
    const long long t = (long long)blockIdx.x * 256 + threadIdx.x;
    const long long nc = (long long)P.n[0] * P.n[1] * P.n[2];
    if (t >= nc) return;
    const int cell[3] = {(int)(t % P.n[0]), (int)((t / P.n[0]) % P.n[1]), (int)(t / ((long long)P.n[0] * P.n[1]))};
    const long long m = lin(P, cell[0], cell[1], cell[2]);
    const float kc = __ldg(P.kap + m);
    double ge = 0.0, gk = 0.0;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const int b1 = (c + 1) % 3, b2 = (c + 2) % 3;
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
            for (int v = 0; v < 2; ++v) {
                // edge E_c whose cell (p[c], p[b1] - u, p[b2] - v) is this cell
                int x[3];
                x[c] = cell[c];
                x[b1] = cell[b1] + u;
                x[b2] = cell[b2] + v;
                if (x[b1] >= P.N[b1]) { if (!P.per[b1]) continue; x[b1] -= P.N[b1]; }
                if (x[b2] >= P.N[b2]) { if (!P.per[b2]) continue; x[b2] -= P.N[b2]; }
                if (!upd_E(P, c, x)) continue;
                const long long q = lin(P, x[0], x[1], x[2]);
                ge += 0.25 * A.gE[c][q];
                if (kc > 0.f) {
                    float wgt = 0.25f;
                    if (P.edge_rule != TF_EDGE_PLAIN_MEAN) {
                        int nk = 0;
#pragma unroll
                        for (int uu = 0; uu < 2; ++uu)
#pragma unroll
                            for (int vv = 0; vv < 2; ++vv) {
                                int cc[3];
                                cc[c] = x[c];
                                cc[b1] = uu ? prv(P, b1, x[b1]) : x[b1];
                                cc[b2] = vv ? prv(P, b2, x[b2]) : x[b2];
                                nk += __ldg(P.kap + lin(P, cc[0], cc[1], cc[2])) > 0.f;
                            }
                        wgt = nk ? 1.f / (float)nk : 0.f;
                    }
                    gk += (double)wgt * A.gK[c][q];
                }
            }
    }
    g_eps[t] = (float)(ge * unscale);
    float gl = 0.f;
    if (kc > 0.f) {   // kt = (c0 dt / lambda)^2 / mu_r: d kt / d lambda = -2 kt / lambda
        const float lam = dt_c0 / sqrtf(kc * __ldg(P.mu + m));
        gl = (float)(gk * unscale * (-2.0 * (double)kc / (double)lam));
    }
    g_lam[t] = gl;
}

// E^n of the three components into the adjoint's history (16-byte aligned
// arrays of n4 float4 each), grid-stride
__global__ void __launch_bounds__(256) k_copy3(float4* d0, float4* d1, float4* d2, const float4* s0, const float4* s1,
                                               const float4* s2, long long n4) {
    for (long long i = (long long)blockIdx.x * 256 + threadIdx.x; i < n4; i += (long long)gridDim.x * 256) {
        const float4 a = __ldg(s0 + i), b = __ldg(s1 + i), c = __ldg(s2 + i);
        d0[i] = a;
        d1[i] = b;
        d2[i] = c;
    }
}

cudaError_t launch_copy3(float* const dst[3], float* const src[3], long long n, cudaStream_t stream) {
    if (n % 4 != 0) return cudaErrorInvalidValue;
    int sms = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, 0) != cudaSuccess || sms < 1) sms = 1;
    k_copy3<<<4 * sms, 256, 0, stream>>>((float4*)dst[0], (float4*)dst[1], (float4*)dst[2], (const float4*)src[0],
                                          (const float4*)src[1], (const float4*)src[2], n / 4);
    return cudaGetLastError();
}

// one step back; `chained`: the launch before in the stream is the edge pass of the step after
cudaError_t launch_adjoint_step(const AdjArgs& A, bool chained, cudaStream_t stream) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(A.G.nbx, A.G.nby, A.G.nbz);
    cfg.blockDim = dim3(kAT);
    cfg.stream = stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = chained ? 1 : 0;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, k_adj_faces, A);
    if (e != cudaSuccess) return e;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_adj_edges, A);
}

cudaError_t launch_adjoint_cells(const Params& P, const AdjState& A, float dt_c0, double unscale, float* g_eps,
                                 float* g_lam, cudaStream_t stream) {
    const long long nc = (long long)P.n[0] * P.n[1] * P.n[2];
    k_adj_cells<<<(unsigned)((nc + 255) / 256), 256, 0, stream>>>(P, A, dt_c0, unscale, g_eps, g_lam);
    return cudaGetLastError();
}

}  // namespace tf
