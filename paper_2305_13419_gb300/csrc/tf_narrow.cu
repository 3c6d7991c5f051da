// tf_narrow.cu -- many steps per launch on grids with a small x-y cross
// section: 1-D columns and quasi-1-D slabs (sm_103a).
//
// A CTA takes a window of whole planes: the planes it owns and, on either
// side, one plane per step of the launch.  A step reaches one plane up and
// one down (Bt at plane k reads E at k and k + 1, E reads Bt at k and k - 1),
// so what the window's ends lack spoils one plane per step and the owned
// planes come out right after all of them, without a word between CTAs.
// (A Mur wall takes up the new E of the plane next to it and is right only as
// long as that plane is: the CTA that owns that plane owns the wall as well.)
// A thread keeps four x-adjacent points -- E, Bt, Js, their coefficients and
// CPML memories -- in registers for the whole launch; neighbours meet in
// shared memory, two barriers per step.  The launch reads one buffer and
// writes the other.  The arithmetic is that of the passes (tf_pass.cu), in
// the same order: the same bits.
#include <type_traits>

#include "tf_quad.cuh"

namespace tf {

namespace {

using namespace dev;

constexpr int kNT = kNarrowThreads;

__device__ __forceinline__ Q4 all0() { return {{0, 0}}; }

// a quad in shared memory: both halves, or (rows of one or two points) the
// first alone -- the arithmetic of a half that nothing keeps is not compiled
template <bool kHalf>
struct Cell {
    f2 v[kHalf ? 1 : 2];
};
template <bool kHalf>
__device__ __forceinline__ void put(Cell<kHalf>& c, const Q4& q) {
    c.v[0] = q.v[0];
    if constexpr (!kHalf) c.v[1] = q.v[1];
}
template <>
__device__ __forceinline__ void put<false>(Cell<false>& c, const Q4& q) {
    *reinterpret_cast<ulonglong2*>(&c) = make_ulonglong2(q.v[0], q.v[1]);
}
template <bool kHalf>
__device__ __forceinline__ Q4 get(const Cell<kHalf>& c) {
    if constexpr (kHalf) {
        return {{c.v[0], 0}};
    } else {
        const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(&c);
        return {{t.x, t.y}};
    }
}
// lane l of a cell (l a run-time value)
template <bool kHalf>
__device__ __forceinline__ float at(const Cell<kHalf>& c, int l) {
    return reinterpret_cast<const float*>(&c)[l];
}
template <bool kHalf>
__device__ __forceinline__ void keep(float* base, unsigned o, const Q4& q) {
    if constexpr (kHalf)
        *(f2*)((char*)base + o) = q.v[0];
    else
        sto(base, o, q);
}

}  // namespace

// Bound by the latency of a step's instruction chain (two warps per scheduler,
// two barriers, shared-memory round trips): 0.25 us a step in a 1 x 1 column's
// CTAs, 0.5 in a 4 x 4 slab's, and half as much again in the CTAs with a
// source or a wall; plus some 4 us per launch to load, store and hand over.
// The 1 x 1 x 4480 column takes 0.6 us a step in launches of 32 (7 us by two
// passes per step, 74 by staged planes), the 4 x 4 x 2048 slab 1.0 in launches
// of 20 (7 and 47).  Windows of 128 threads: 0.82 against 0.86 us on the column,
// 1.65 against 1.29 on the slab; of 64: slower on both.
// The CTAs past the `blocks` windows add the launch before's samples to the
// running DFTs meanwhile (8 us for one probe, a launch of its own before).
// kHalf: rows of one or two points.  kLine: a column, periodic along x and y:
// differences along x and y are zero.
template <bool kHalf, bool kLine>
__global__ void __launch_bounds__(kNT, 1) k_narrow(const __grid_constant__ NarrowArgs A, const __grid_constant__ Probes R,
                                                   int blocks) {
    const Params& P = A.P;
    __shared__ __align__(16) Cell<kHalf> sE[3][kNT], sB[3][kNT];
    if ((int)blockIdx.x >= blocks) {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        const int w = ((int)blockIdx.x - blocks) * (kNT / 32) + (int)threadIdx.x / 32;
        if (w < R.n * TF_MAX_FREQS)
            probe_dft(R, A.samples_before, w / TF_MAX_FREQS, w % TF_MAX_FREQS, A.level - A.steps_before, A.steps_before);
        return;
    }
    const int tid = threadIdx.x, per = A.nq * P.N[1];
    const int kl = tid / per, r = tid % per, j = r / A.nq, iq = r % A.nq, x = 4 * iq;
    const int kw = blockIdx.x * A.own - A.steps + kl;   // the plane, before wrapping
    int k = kw;
    const bool seat = kl < A.window;   // the last threads may have no plane
    bool live = seat;
    if (P.per[2]) {
        k %= P.N[2];
        if (k < 0) k += P.N[2];
    } else {
        live = live && k >= 0 && k < P.N[2];
    }
    if (!live) k = 0;
    // a Mur wall goes with the plane next to it (with N[2] - 1 a multiple of `own`,
    // or own = 1, it would be another CTA's, where that plane is spoiled by then)
    const bool mur = P.bc[2] == TF_BC_MUR;
    const int ko = (mur ? min(max(kw, 1), P.n[2] - 1) : kw) - (int)blockIdx.x * A.own;
    const bool mine = live && ko >= 0 && ko < A.own && kw < P.N[2];
    // lanes that each component advances
    const Quad u = quad_of(P, x, j, k);
    const bool adv = live && (P.per[1] || j < P.n[1]) && (P.per[2] || k < P.n[2]);
    const unsigned hv = adv ? u.hv : 0u, in = adv ? u.in : 0u;
    const unsigned mbx = in, mby = u.iny ? hv : 0u, mbz = u.inz ? hv : 0u;
    const unsigned mex = u.iny && u.inz ? hv : 0u, mey = u.inz ? in : 0u, mez = u.iny ? in : 0u;
    // neighbours' threads; past the window, a wall or a seam that does not wrap: the own one
    const int ty1 = !seat ? tid : j + 1 < P.N[1] ? tid + A.nq : P.per[1] ? tid - j * A.nq : tid;
    const int ty0 = !seat ? tid : j > 0 ? tid - A.nq : P.per[1] ? tid + (P.N[1] - 1) * A.nq : tid;
    const int tz1 = live && kl + 1 < A.window && (P.per[2] || k + 1 < P.N[2]) ? tid + per : tid;
    const int tz0 = live && kl > 0 && (P.per[2] || k > 0) ? tid - per : tid;
    const bool xlast = x + 4 >= P.N[0];
    const int tx1 = !seat ? tid : !xlast ? tid + 1 : P.per[0] ? tid - iq : tid;
    const int tx0 = !seat ? tid : x > 0 ? tid - 1 : P.per[0] ? tid + A.nq - 1 : tid;
    const int lx0 = x > 0 ? 3 : (P.N[0] - 1) & 3;   // lane of the neighbour below
    const bool wrap = P.per[0] && x + 4 > P.N[0];
    // First-order Mur: E of a wall plane comes from the plane next to it, whose
    // threads hold that plane's old and new E: they write the wall's as well,
    // its own threads only take it up
    const bool wall = mur && live && (k == 0 || k == P.n[2]);
    const bool lo_wall = mur && live && k == 1 && kl > 0, hi_wall = mur && live && k == P.n[2] - 1 && kl + 1 < A.window;
    const bool by_wall = lo_wall || hi_wall;
    const unsigned mwx = adv && u.iny ? u.hv : 0u, mwy = in;
    // every lane of the row's points advances in every component: no selects
    const unsigned row = x + 4 <= P.N[0] ? 15u : (1u << (P.N[0] - x)) - 1u;
    const bool full = (mbx & mby & mbz & mex & mey & mez) == row;
    const bool one_row = P.N[1] == 1;

    // everything above is the launch's own; what follows reads the launch before's results
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    Q4 ex = all0(), ey = ex, ez = ex, bx = ex, by = ex, bz = ex, jx = ex, jy = ex, jz = ex;
    Q4 ca0 = ex, ca1 = ex, ca2 = ex, cb0 = ex, cb1 = ex, cb2 = ex, cj0 = ex, cj1 = ex, cj2 = ex;
    Q4 pb0 = ex, pb1 = ex, pe0 = ex, pe1 = ex;
    float bB = 0.f, cB = 0.f, bE = 0.f, cE = 0.f;
    const bool sz = live && u.sz;
    bool sc = false;
    if (live) {
        ex = ldo(P.E[0], u.o);
        ey = ldo(P.E[1], u.o);
        ez = ldo(P.E[2], u.o);
        bx = ldo(P.B[0], u.o);
        by = ldo(P.B[1], u.o);
        bz = ldo(P.B[2], u.o);
        if (sz) {
            pb0 = ldo(P.psiB[0][2], u.o);
            pb1 = ldo(P.psiB[1][2], u.o);
            pe0 = ldo(P.psiE[0][2], u.o);
            pe1 = ldo(P.psiE[1][2], u.o);
            bB = __ldg(P.pbB[2] + k);
            cB = __ldg(P.pcB[2] + k);
            bE = __ldg(P.pbE[2] + k);
            cE = __ldg(P.pcE[2] + k);
        }
        if (adv && u.hv) {
            const float4 rec = __ldg(A.tilemat + (long long)((j / kSY) * A.ntx + x / kSX) * P.N[2] + k);
            if (isnan(rec.x)) {
                ca0 = ldo(P.ca[0], u.o);
                ca1 = ldo(P.ca[1], u.o);
                ca2 = ldo(P.ca[2], u.o);
                cb0 = ldo(P.cb[0], u.o);
                cb1 = ldo(P.cb[1], u.o);
                cb2 = ldo(P.cb[2], u.o);
                cj0 = ldo(P.cj[0], u.o);
                cj1 = ldo(P.cj[1], u.o);
                cj2 = ldo(P.cj[2], u.o);
                sc = true;
            } else {
                ca0 = ca1 = ca2 = all4(rec.x);
                cb0 = cb1 = cb2 = all4(rec.y);
                cj0 = cj1 = cj2 = all4(rec.z);
                sc = rec.z > 0.f;
            }
            if (sc) {
                jx = ldo(P.J[0], u.o);
                jy = ldo(P.J[1], u.o);
                jz = ldo(P.J[2], u.o);
            }
        }
    }
    unsigned probes = 0;   // probes inside the own quad
    if (mine)
        for (int p = 0; p < A.nprobe; ++p)
            if (A.pr[p][2] == k && A.pr[p][1] == j && A.pr[p][0] >= x && A.pr[p][0] < x + 4) probes |= 1u << p;
    const Sources& S = A.S;
    // soft sources inside the quad: a bit per source, its lanes four bits each
    unsigned hit = 0;
    unsigned long long hit_lanes = 0;
    const bool src = adv && S.n > 0 && x + 3 >= S.bb_lo[0] && x < S.bb_hi[0] && j >= S.bb_lo[1] && j < S.bb_hi[1] &&
                     k >= S.bb_lo[2] && k < S.bb_hi[2];
    if (src)
        for (int q = 0; q < S.n; ++q) {
            if (j < S.lo[q][1] || j >= S.hi[q][1] || k < S.lo[q][2] || k >= S.hi[q][2]) continue;
            unsigned m = 0;
            for (int p = 0; p < 4; ++p) m |= x + p >= S.lo[q][0] && x + p < S.hi[q][0] ? 1u << p : 0u;
            if (m) {
                hit |= 1u << q;
                hit_lanes |= (unsigned long long)m << (4 * q);
            }
        }
    put(sE[0][tid], ex);
    put(sE[1][tid], ey);
    put(sE[2][tid], ez);
    __syncthreads();

    const int hit0 = hit ? __ffs(hit) - 1 : 0;   // the first one's amplitude: fetched a pass ahead
    const Q4 r0 = all4(P.r[0]), r1 = all4(P.r[1]), r2 = all4(P.r[2]);
    // one plane of differences and updates; kFull: without selects
    auto pass_b = [&](auto full_tag) {
        constexpr bool kFull = decltype(full_tag)::value;
        const Q4 ex_z = get(sE[0][tz1]), ey_z = get(sE[1][tz1]);
        const Q4 dEy_z = sub4(ey_z, ey), dEx_z = sub4(ex_z, ex);
        Q4 nx, ny, nz;
        if constexpr (kLine) {   // a column: nothing varies along x and y, Bz stays
            nx = fma4(r2, dEy_z, bx);
            ny = sub4(by, mul4(r2, dEx_z));
            nz = bz;
        } else {
            Q4 ex_y = ex, ez_y = ez;
            if (!one_row) {
                ex_y = get(sE[0][ty1]);
                ez_y = get(sE[2][ty1]);
            }
            const float ey_n = at(sE[1][tx1], 0), ez_n = at(sE[2][tx1], 0);
            Q4 ey_x = up4(ey, ey_n), ez_x = up4(ez, ez_n);
            if (wrap) {   // the row ends inside the quad: its last point wraps
                ey_x = set_lane(ey_x, P.N[0] - 1 - x, ey_n);
                ez_x = set_lane(ez_x, P.N[0] - 1 - x, ez_n);
            }
            const Q4 dEz_y = sub4(ez_y, ez), dEx_y = sub4(ex_y, ex), dEz_x = sub4(ez_x, ez), dEy_x = sub4(ey_x, ey);
            nx = fma4(r2, dEy_z, sub4(bx, mul4(r1, dEz_y)));
            ny = fma4(r0, dEz_x, sub4(by, mul4(r2, dEx_z)));
            nz = fma4(r1, dEx_y, sub4(bz, mul4(r0, dEy_x)));
        }
        if (sz) {
            const Q4 n1 = fma4(all4(bB), pb0, mul4(all4(cB), dEy_z)), n2 = fma4(all4(bB), pb1, mul4(all4(cB), dEx_z));
            nx = add4(nx, n1);
            ny = sub4(ny, n2);
            pb0 = kFull ? n1 : sel4(n1, pb0, mbx);
            pb1 = kFull ? n2 : sel4(n2, pb1, mby);
        }
        bx = kFull ? nx : sel4(nx, bx, mbx);
        by = kFull ? ny : sel4(ny, by, mby);
        bz = kFull ? nz : sel4(nz, bz, mbz);
        put(sB[0][tid], bx);
        put(sB[1][tid], by);
        if (!kLine) put(sB[2][tid], bz);
    };
    auto pass_e = [&](auto full_tag, int t, float amp0) {
        constexpr bool kFull = decltype(full_tag)::value;
        const Q4 hx_zm = get(sB[0][tz0]), hy_zm = get(sB[1][tz0]);
        const Q4 dHy_z = sub4(by, hy_zm), dHx_z = sub4(bx, hx_zm);
        Q4 cx, cy, cz;
        if constexpr (kLine) {
            cx = sub4(all0(), mul4(r2, dHy_z));
            cy = mul4(r2, dHx_z);
            cz = all0();
        } else {
            Q4 hx_ym = bx, hz_ym = bz;
            if (!one_row) {
                hx_ym = get(sB[0][ty0]);
                hz_ym = get(sB[2][ty0]);
            }
            const float hy_p = at(sB[1][tx0], lx0), hz_p = at(sB[2][tx0], lx0);
            const Q4 dHz_y = sub4(bz, hz_ym), dHz_x = sub4(bz, dn4(bz, hz_p)), dHy_x = sub4(by, dn4(by, hy_p));
            const Q4 dHx_y = sub4(bx, hx_ym);
            cx = sub4(mul4(r1, dHz_y), mul4(r2, dHy_z));
            cy = sub4(mul4(r2, dHx_z), mul4(r0, dHz_x));
            cz = sub4(mul4(r0, dHy_x), mul4(r1, dHx_y));
        }
        if (sz) {
            const Q4 n1 = fma4(all4(bE), pe0, mul4(all4(cE), dHy_z)), n2 = fma4(all4(bE), pe1, mul4(all4(cE), dHx_z));
            cx = sub4(cx, n1);
            cy = add4(cy, n2);
            pe0 = kFull ? n1 : sel4(n1, pe0, mex);
            pe1 = kFull ? n2 : sel4(n2, pe1, mey);
        }
        if (sc) {
            const Q4 ux = fma4(cj0, ex, jx), uy = fma4(cj1, ey, jy), uz = fma4(cj2, ez, jz);
            cx = sub4(cx, ux);
            cy = sub4(cy, uy);
            cz = sub4(cz, uz);
            jx = kFull ? ux : sel4(ux, jx, mex);
            jy = kFull ? uy : sel4(uy, jy, mey);
            jz = kFull ? uz : sel4(uz, jz, mez);
        }
        Q4 nx = fma4(cb0, cx, mul4(ca0, ex));
        Q4 ny = fma4(cb1, cy, mul4(ca1, ey));
        Q4 nz = fma4(cb2, cz, mul4(ca2, ez));
        if (hit) {   // the sums of add_src, in its order
            Q4 ax = all0(), ay = ax, az = ax;
            for (unsigned m = hit; m; m &= m - 1) {
                const int q = __ffs(m) - 1;
                const Q4 a = sel4(all4(q == hit0 ? amp0 : A.amp[q][t]), all0(), (unsigned)(hit_lanes >> (4 * q)) & 15u);
                if (S.comp[q] == 0)
                    ax = add4(ax, a);
                else if (S.comp[q] == 1)
                    ay = add4(ay, a);
                else
                    az = add4(az, a);
            }
            nx = add4(nx, ax);
            ny = add4(ny, ay);
            nz = add4(nz, az);
        }
        if (!kFull) {
            nx = sel4(nx, ex, mex);
            ny = sel4(ny, ey, mey);
            nz = sel4(nz, ez, mez);
        }
        if (by_wall) {   // E_w^{n+1} = E_i^n + M (E_i^{n+1} - E_w^n)
#pragma unroll
            for (int w = 0; w < 2; ++w) {
                if (!(w ? hi_wall : lo_wall)) continue;
                const int tw = w ? tid + per : tid - per;
                float* const e0 = reinterpret_cast<float*>(&sE[0][tw]);
                float* const e1 = reinterpret_cast<float*>(&sE[1][tw]);
#pragma unroll
                for (int p = 0; p < (kHalf ? 2 : 4); ++p) {
                    if (mwx >> p & 1u) e0[p] = lane(ex, p) + P.mur_M * (lane(nx, p) - e0[p]);
                    if (mwy >> p & 1u) e1[p] = lane(ey, p) + P.mur_M * (lane(ny, p) - e1[p]);
                }
            }
        }
        ex = nx;
        ey = ny;
        ez = nz;
        if (!wall) {
            put(sE[0][tid], ex);
            put(sE[1][tid], ey);
        }
        if (!kLine) put(sE[2][tid], ez);
    };
    const bool wfull = __all_sync(0xffffffffu, full);
    for (int t = 0; t < A.steps; ++t) {
        if (wall) {   // as the plane next to it left it
            ex = get(sE[0][tid]);
            ey = get(sE[1][tid]);
        }
        for (unsigned m = probes; m; m &= m - 1) {
            const int p = __ffs(m) - 1;
            const Q4 v = A.pr_comp[p] == 0 ? ex : A.pr_comp[p] == 1 ? ey : ez;
            const int l = A.pr[p][0] & 3;
            A.samples[t * TF_MAX_PROBES + p] =
                l == 0 ? lane(v, 0) : l == 1 ? lane(v, 1) : kHalf ? 0.f : l == 2 ? lane(v, 2) : lane(v, 3);
        }
        const float amp0 = hit ? A.amp[hit0][t] : 0.f;
        if (wfull)
            pass_b(std::true_type{});
        else
            pass_b(std::false_type{});
        __syncthreads();
        if (wfull)
            pass_e(std::true_type{}, t, amp0);
        else
            pass_e(std::false_type{}, t, amp0);
        __syncthreads();
    }
    if (wall) {
        ex = get(sE[0][tid]);
        ey = get(sE[1][tid]);
    }
    if (mine) {
        // the watchdog, once per launch: a non-finite E stays non-finite
        // (E' = ca E + ..), and what lies past the row's points may run wild
        const Q4 sum = sel4(add4(add4(ex, ey), ez), all0(), row);
        const bool bad = !isfinite(lo(sum.v[0]) + hi(sum.v[0])) || (!kHalf && !isfinite(lo(sum.v[1]) + hi(sum.v[1])));
        const Q4 z = all0();   // past the row's end: zeros
        keep<kHalf>(A.E[0], u.o, sel4(ex, z, row));
        keep<kHalf>(A.E[1], u.o, sel4(ey, z, row));
        keep<kHalf>(A.E[2], u.o, sel4(ez, z, row));
        keep<kHalf>(A.B[0], u.o, sel4(bx, z, row));
        keep<kHalf>(A.B[1], u.o, sel4(by, z, row));
        keep<kHalf>(A.B[2], u.o, sel4(bz, z, row));
        if (sc) {
            keep<kHalf>(A.J[0], u.o, sel4(jx, z, row));
            keep<kHalf>(A.J[1], u.o, sel4(jy, z, row));
            keep<kHalf>(A.J[2], u.o, sel4(jz, z, row));
        }
        if (sz) {
            keep<kHalf>(A.psiB[0], u.o, pb0);
            keep<kHalf>(A.psiB[1], u.o, pb1);
            keep<kHalf>(A.psiE[0], u.o, pe0);
            keep<kHalf>(A.psiE[1], u.o, pe1);
        }
        if (bad) atomicOr(P.status, kStatusNonFinite);
    }
}

cudaError_t launch_narrow(const NarrowArgs& A, const Probes& R, cudaStream_t st) {
    const int blocks = narrow_blocks(A.P, A.own);
    const int dft = A.steps_before > 0 ? (R.n * TF_MAX_FREQS + kNT / 32 - 1) / (kNT / 32) : 0;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(blocks + dft);
    cfg.blockDim = dim3(kNT);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = A.chained ? 1 : 0;
    if (A.P.N[0] == 1 && A.P.N[1] == 1 && A.P.per[0] && A.P.per[1]) return cudaLaunchKernelEx(&cfg, k_narrow<true, true>, A, R, blocks);
    if (A.P.N[0] <= 2) return cudaLaunchKernelEx(&cfg, k_narrow<true, false>, A, R, blocks);
    return cudaLaunchKernelEx(&cfg, k_narrow<false, false>, A, R, blocks);
}

}  // namespace tf
