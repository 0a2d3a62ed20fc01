// K_LINE: the fused BR2 Navier-Stokes stage of FP32 solvers, one thread per
// element line (included by fr_kernels.cuh).
//
// Same method and exchange as K_STAGE (every element sends its partners its
// face state and the gradient part of its viscous normal flux; the next stage
// forms both sides' BR2 fluxes locally), with another split of the work.  A
// thread owns one line of every direction of its element, so everything
// one-dimensional - derivative, interpolation to the line's two faces,
// divergence with its correction - runs on registers with operator entries
// from the constant bank, and a value goes through shared memory once per
// direction instead of N times.  The threads of an element sit in one warp
// (25-line hexes: one CTA): no CTA barrier separates the phases.
//
// 2-D, measured (GB300, p = 3, 259,298 curved quads, one stage): gradient + flux
// kernels 306 us (1,500 instructions per point, issue slots and phase barriers
// the bound); one thread per line 193 us (777 instructions; the L1 data stage,
// 36 % of its cycles on 64-byte-step row accesses); rows and face data fetched
// by asynchronous copies 164 us; packed FP32 pairs in the contractions 144 us
// (95.5 M warp instructions, 52 % of the issue slots).  243,854 quads of eight
// airfoils: 142 us and 658 MB of DRAM traffic per stage, 4.65 TB/s = 0.68 of a
// copy.  What is left: 12 warps per SM (shared memory), each stalled 4.2 cycles
// per instruction, on shared-memory, global and instruction latency most.
#pragma once

namespace frk {

// values per flux point of the packed face geometry, in parts of four: 2-D
// normal (outward, scaled by |dS|) and own lifting coefficients (times eta),
// then the partner's and its index as bits; 3-D normal and partner index, own
// lifting coefficients, the partner's
__host__ __device__ constexpr int face_geo(int dim) { return 4 * dim; }

// NV contiguous values of a row at a multiple of NV values (so 16-byte aligned
// where NV is a multiple of 4, 8-byte aligned where it is even)
template <int NV, typename real>
__device__ __forceinline__ void ld_row(const real *p, real *o) {
    if constexpr (NV % 4 == 0 && sizeof(real) == 4) {
#pragma unroll
        for (int i = 0; i < NV / 4; ++i) {
            const float4 t = reinterpret_cast<const float4 *>(p)[i];
            o[4 * i] = t.x; o[4 * i + 1] = t.y; o[4 * i + 2] = t.z; o[4 * i + 3] = t.w;
        }
    } else if constexpr (NV % 2 == 0 && sizeof(real) == 4) {
#pragma unroll
        for (int i = 0; i < NV / 2; ++i) {
            const float2 t = reinterpret_cast<const float2 *>(p)[i];
            o[2 * i] = t.x; o[2 * i + 1] = t.y;
        }
    } else {
#pragma unroll
        for (int i = 0; i < NV; ++i) o[i] = p[i];
    }
}
template <int NV, typename real>
__device__ __forceinline__ void st_row(real *p, const real *o) {
    if constexpr (NV % 4 == 0 && sizeof(real) == 4) {
#pragma unroll
        for (int i = 0; i < NV / 4; ++i)
            reinterpret_cast<float4 *>(p)[i] = make_float4(o[4 * i], o[4 * i + 1], o[4 * i + 2], o[4 * i + 3]);
    } else if constexpr (NV % 2 == 0 && sizeof(real) == 4) {
#pragma unroll
        for (int i = 0; i < NV / 2; ++i) reinterpret_cast<float2 *>(p)[i] = make_float2(o[2 * i], o[2 * i + 1]);
    } else {
#pragma unroll
        for (int i = 0; i < NV; ++i) p[i] = o[i];
    }
}

// geometry of one flux point
template <int D, typename real>
struct FaceGeo {
    real n[D], lf[D], lfp[D];
    int32_t pt;
};
// The element's flux reference (LocalRef) in the few values the main path
// reads: u_c = u_r + du, the rest follows from it.
template <int D, typename real>
struct LineRef {
    real rho, m[D], v[D], p, H, du[D + 2];
};

template <int D, typename real>
__device__ __forceinline__ void line_ref(const RefState<real> &g, const real *u0, bool local, real gamma,
                                         LineRef<D, real> &L) {
    constexpr int V = D + 2;
    if (!local) {
        L.rho = g.rho;
        L.p = g.p;
        L.H = g.H;
#pragma unroll
        for (int i = 0; i < D; ++i) { L.m[i] = g.m[i]; L.v[i] = g.v[i]; }
#pragma unroll
        for (int v = 0; v < V; ++v) L.du[v] = 0;
        return;
    }
    L.rho = g.rho + u0[0];
    L.du[0] = L.rho - g.rho;
    const real E = g.E + u0[V - 1];
    L.du[V - 1] = E - g.E;
    real ke = 0;
#pragma unroll
    for (int i = 0; i < D; ++i) {
        L.m[i] = g.m[i] + u0[1 + i];
        L.du[1 + i] = L.m[i] - g.m[i];
        L.v[i] = L.m[i] / L.rho;
        ke += real(0.5) * L.m[i] * L.v[i];
    }
    L.p = (gamma - real(1)) * (E - ke);
    L.H = E + L.p;
}

// Boundary points and the Roe flux are calls, so that their functions neither
// widen the main path's registers nor repeat per face; the full reference is
// rebuilt there (u_r + du is exact).
template <int D, typename real>
struct BcPair { real ug[D + 2], ub[D + 2]; };
template <int D, typename real>
struct BcIn { real u[D + 2], du[D + 2], n[D]; };
template <int D, typename real>
__device__ __forceinline__ void full_ref(const KArgs<real> *a, const real *du, bool local, LocalRef<D, real> &R) {
    if (local) make_local_ref<D>(a->ref, du, a->gamma, R);
    else global_ref<D>(a->ref, R);
}
template <int D, typename real>
__device__ __noinline__ BcPair<D, real> bc_call(const KArgs<real> *a, const int b, const BcIn<D, real> in) {
    LocalRef<D, real> R;
    full_ref<D>(a, in.du, a->local_ref && !a->DIVREF, R);
    real bv[D];
#pragma unroll
    for (int d = 0; d < D; ++d) bv[d] = a->BVREF[(int64_t)b * D + d] - R.bv[d];
    BcPair<D, real> o;
    bc_states_pert<D>(a->BTAG[b], in.u, in.n, bv, R.r, a->gamma, o.ug, o.ub);
    return o;
}
template <int D, typename real>
struct RoeIn { real uL[D + 2], uR[D + 2], n[D], du[D + 2]; };
template <int D, typename real>
struct RoeOut { real F[D + 2]; };
template <int D, typename real>
__device__ __noinline__ RoeOut<D, real> roe_call(const KArgs<real> *a, const RoeIn<D, real> in) {
    LocalRef<D, real> R;
    full_ref<D>(a, in.du, a->local_ref && !a->DIVREF, R);
    RoeOut<D, real> o;
    roe_pert<D>(in.uL, in.uR, in.n, R.r, a->gamma, o.F);
    return o;
}

// F(u).n - F(u_r).n from the primitive perturbations; returns the wave-speed
// bound |v.n| + c |n|
template <int D, typename real>
__device__ __forceinline__ real normal_flux_prim(const real *up, const real *vp, const real *v, real pp, real p,
                                                 real ir, const real *n, real vnr, real nn, const LineRef<D, real> &r,
                                                 real gamma, real *F) {
    real vnp = 0, mn = 0;
#pragma unroll
    for (int j = 0; j < D; ++j) {
        vnp += vp[j] * n[j];
        mn += up[1 + j] * n[j];
    }
    const real vn = vnr + vnp;
    F[0] = mn;
#pragma unroll
    for (int i = 0; i < D; ++i) F[1 + i] = up[1 + i] * vn + r.m[i] * vnp + pp * n[i];
    F[D + 1] = (up[D + 1] + pp) * vn + r.H * vnp;
    return fabs(vn) + sqrt(nn * (gamma * p * ir));
}

// rho, 1/rho, v' = v - v_r, v, p', p from the perturbation u' (prim_pert with
// the reciprocal kept)
template <int D, typename real>
__device__ __forceinline__ void prim_line(const real *up, const LineRef<D, real> &r, real gm1, real &ir, real *vp,
                                          real *v, real &pp, real &p) {
    ir = real(1) / (r.rho + up[0]);
    real kep = 0;
#pragma unroll
    for (int i = 0; i < D; ++i) {
        vp[i] = (up[1 + i] - r.v[i] * up[0]) * ir;
        v[i] = r.v[i] + vp[i];
        kep += r.m[i] * vp[i] + up[1 + i] * v[i];
    }
    pp = gm1 * (up[D + 1] - real(0.5) * kep);
    p = r.p + pp;
}

// visc_normal for the rank-one gradient lf (x) dd (the lifting of a jump)
template <int D, typename real>
__device__ __forceinline__ void visc_lift(const real *lf, const real *dd, const real *v, real Es, real mi, real ki,
                                          const real *n, real *out) {
    constexpr int V = D + 2;
    real w[D], ln = 0, lw = 0, wn = 0, vw = 0;
#pragma unroll
    for (int i = 0; i < D; ++i) {
        w[i] = dd[1 + i] - dd[0] * v[i];
        ln += lf[i] * n[i];
        lw += lf[i] * w[i];
        wn += w[i] * n[i];
        vw += v[i] * w[i];
    }
    real en = 0;
    const real l3 = real(2.0 / 3.0) * lw;
    out[0] = 0;
#pragma unroll
    for (int i = 0; i < D; ++i) {
        out[1 + i] = mi * (w[i] * ln + lf[i] * wn - l3 * n[i]);
        en += v[i] * out[1 + i];
    }
    out[V - 1] = en + ki * ln * (dd[V - 1] - dd[0] * Es - vw);
}

// common normal flux (inviscid - BR2 viscous) and face jump of one flux point
template <int D, int N, typename real>
__device__ __forceinline__ void line_face(const KArgs<real> &a, const LineRef<D, real> &R, const FaceGeo<D, real> &g,
                                          const real *uL, const real (*Q)[D + 2], real *uR, const real *fvp, real kq,
                                          real *Fs, real *dd) {
    constexpr int V = D + 2;
    const real gm1 = a.gamma - real(1);
    const bool inner = g.pt >= 0;
    if (inner && g.pt >= (int32_t)a.fp_real) {
        // mortar point: the common flux was formed on the mortar, relative to
        // n . F(u_r); take n . (F(u_c) - F(u_r)) off
        real Fc[V], vn, c2;
        ldg_v<V>(a.MFLUX + (int64_t)(g.pt - (int32_t)a.fp_real) * V, Fs);
        flux_normal_pert<D>(R.du, g.n, a.ref, gm1, a.gamma, Fc, vn, c2);
#pragma unroll
        for (int v = 0; v < V; ++v) {
            Fs[v] -= Fc[v];
            dd[v] = real(0.5) * (uR[v] - uL[v]);
        }
        return;
    }
    real uLl[V], uRl[V], ub[V];
#pragma unroll
    for (int v = 0; v < V; ++v) uLl[v] = uL[v] - R.du[v];
    bool wall = false;
    if (!inner) {
        const int b = -1 - g.pt;
        wall = a.BTAG[b] == BC_WALL;
        BcIn<D, real> in;
#pragma unroll
        for (int v = 0; v < V; ++v) { in.u[v] = uLl[v]; in.du[v] = R.du[v]; }
#pragma unroll
        for (int d = 0; d < D; ++d) in.n[d] = g.n[d];
        const BcPair<D, real> o = bc_call<D, real>(&a, b, in);
#pragma unroll
        for (int v = 0; v < V; ++v) {
            uRl[v] = o.ug[v];
            uR[v] = o.ug[v] + R.du[v];
            ub[v] = o.ub[v] + R.du[v];
        }
    } else {
#pragma unroll
        for (int v = 0; v < V; ++v) uRl[v] = uR[v] - R.du[v];
    }
    real irL, vpL[D], vL[D], ppL, pL, irR, vpR[D], vR[D], ppR, pR;
    prim_line<D>(uLl, R, gm1, irL, vpL, vL, ppL, pL);
    prim_line<D>(uRl, R, gm1, irR, vpR, vR, ppR, pR);
    if (a.flux == 1) {
        RoeIn<D, real> in;
#pragma unroll
        for (int v = 0; v < V; ++v) { in.uL[v] = uLl[v]; in.uR[v] = uRl[v]; in.du[v] = R.du[v]; }
#pragma unroll
        for (int d = 0; d < D; ++d) in.n[d] = g.n[d];
        const RoeOut<D, real> o = roe_call<D, real>(&a, in);
#pragma unroll
        for (int v = 0; v < V; ++v) Fs[v] = o.F[v];
    } else {
        real nn = 0, vnr = 0;
#pragma unroll
        for (int d = 0; d < D; ++d) {
            nn += g.n[d] * g.n[d];
            vnr += R.v[d] * g.n[d];
        }
        real FL[V], FR[V];
        const real sL = normal_flux_prim<D>(uLl, vpL, vL, ppL, pL, irL, g.n, vnr, nn, R, a.gamma, FL);
        const real sR = normal_flux_prim<D>(uRl, vpR, vR, ppR, pR, irR, g.n, vnr, nn, R, a.gamma, FR);
        const real lam = real(0.5) * fmax(sL, sR);
#pragma unroll
        for (int v = 0; v < V; ++v) Fs[v] = real(0.5) * (FL[v] + FR[v]) - lam * (uR[v] - uL[v]);
    }
    const real eL = (a.ref.E + uL[V - 1]) * irL;
    real fvo[V], Ql[D][V];
    if (inner) {
#pragma unroll
        for (int v = 0; v < V; ++v) dd[v] = real(0.5) * (uR[v] - uL[v]);
#pragma unroll
        for (int d = 0; d < D; ++d)
#pragma unroll
            for (int v = 0; v < V; ++v) Ql[d][v] = Q[d][v] + g.lf[d] * dd[v];
        visc_normal<D>(Ql, vL, eL, a.mu * irL, kq * irL, g.n, fvo);
        // partner: its gradient part plus its lifting of the jump -dd along
        // its normal -n; common flux 1/2 (own - partner) along n
        real fl[V];
        const real eR = (a.ref.E + uR[V - 1]) * irR;
        visc_lift<D>(g.lfp, dd, vR, eR, a.mu * irR, kq * irR, g.n, fl);
#pragma unroll
        for (int v = 1; v < V; ++v) Fs[v] -= real(0.5) * (fvo[v] - (fvp[v] + fl[v]));
    } else {
        real full[V], vb[D];
        add_ref<V>(a.ref, ub, full);
        const real ib = real(1) / full[0];
#pragma unroll
        for (int d = 0; d < D; ++d) vb[d] = full[1 + d] * ib;
#pragma unroll
        for (int v = 0; v < V; ++v) dd[v] = ub[v] - uL[v];
#pragma unroll
        for (int d = 0; d < D; ++d)
#pragma unroll
            for (int v = 0; v < V; ++v) Ql[d][v] = Q[d][v] + g.lf[d] * dd[v];
        visc_normal<D>(Ql, vb, full[V - 1] * ib, a.mu * ib, kq * ib, g.n, fvo);
        if (wall) fvo[V - 1] = 0;   // adiabatic wall
#pragma unroll
        for (int v = 1; v < V; ++v) Fs[v] -= fvo[v];
    }
}

// F(u) - F(u_c) - F_v(u, grad u) in every direction (u: perturbation)
template <int D, typename real>
__device__ __forceinline__ void line_flux(const KArgs<real> &a, const LineRef<D, real> &R, const real *u,
                                          const real (*gr)[D + 2], real gm1, real kq, real (*F)[D + 2]) {
    constexpr int V = D + 2;
    real ul[V], ir, vp[D], v_[D], pp, p;
#pragma unroll
    for (int v = 0; v < V; ++v) ul[v] = u[v] - R.du[v];
    prim_line<D>(ul, R, gm1, ir, vp, v_, pp, p);
    const real Es = (a.ref.E + u[V - 1]) * ir, mi = a.mu * ir, ki = kq * ir;
    const real Hp = ul[V - 1] + pp;
    real gv[D][D], div = 0;
#pragma unroll
    for (int d = 0; d < D; ++d) {
#pragma unroll
        for (int c = 0; c < D; ++c) gv[d][c] = gr[d][1 + c] - gr[d][0] * v_[c];
        div += gv[d][d];
    }
    const real d3 = real(2.0 / 3.0) * div;
#pragma unroll
    for (int d = 0; d < D; ++d) {
        F[d][0] = ul[1 + d];
        real wk = 0, va = 0;
#pragma unroll
        for (int c = 0; c < D; ++c) {
            const real tau = mi * (gv[d][c] + gv[c][d] - (c == d ? d3 : real(0)));
            F[d][1 + c] = ul[1 + c] * v_[d] + R.m[c] * vp[d] + (c == d ? pp : real(0)) - tau;
            wk += v_[c] * tau;
            va += v_[c] * gv[d][c];
        }
        F[d][V - 1] = Hp * v_[d] + R.H * vp[d] - (wk + ki * (gr[d][V - 1] - gr[d][0] * Es - va));
    }
}

// Four variables as two packed FP32 pairs: one fma.f32x2 issues two FMAs, and
// the kernel is bound by issue slots, not by the FMA pipe.  The coefficients
// come as pairs (c, c) from the constant bank.
struct V4 {
    uint64_t a, b;
    __device__ __forceinline__ void set(const float *x) {
        asm("mov.b64 %0, {%1, %2};" : "=l"(a) : "f"(x[0]), "f"(x[1]));
        asm("mov.b64 %0, {%1, %2};" : "=l"(b) : "f"(x[2]), "f"(x[3]));
    }
    __device__ __forceinline__ void get(float *x) const {
        asm("mov.b64 {%0, %1}, %2;" : "=f"(x[0]), "=f"(x[1]) : "l"(a));
        asm("mov.b64 {%0, %1}, %2;" : "=f"(x[2]), "=f"(x[3]) : "l"(b));
    }
};
__device__ __forceinline__ V4 fma4(const float2 c, const float *x, const V4 &t) {
    V4 q, o;
    q.set(x);
    uint64_t k;
    asm("mov.b64 %0, {%1, %2};" : "=l"(k) : "f"(c.x), "f"(c.y));
    asm("fma.rn.ftz.f32x2 %0, %1, %2, %3;" : "=l"(o.a) : "l"(k), "l"(q.a), "l"(t.a));
    asm("fma.rn.ftz.f32x2 %0, %1, %2, %3;" : "=l"(o.b) : "l"(k), "l"(q.b), "l"(t.b));
    return o;
}
__device__ __forceinline__ V4 mul4(const float2 c, const float *x) {
    V4 q, o;
    q.set(x);
    uint64_t k;
    asm("mov.b64 %0, {%1, %2};" : "=l"(k) : "f"(c.x), "f"(c.y));
    asm("mul.rn.ftz.f32x2 %0, %1, %2;" : "=l"(o.a) : "l"(k), "l"(q.a));
    asm("mul.rn.ftz.f32x2 %0, %1, %2;" : "=l"(o.b) : "l"(k), "l"(q.b));
    return o;
}

// --------------------------------------------------------------------------
// 2-D line kernel.  A warp owns EPW elements (8 of p = 3), a thread one row
// (xi line) and one column (eta line) of its element.  Everything the warp
// reads is contiguous in memory, so it is fetched at the start with 16-byte
// asynchronous copies into the warp's part of shared memory (two groups:
// geometry + state, partners' face data) and read from there; the new state and
// register go back as whole sectors.  Lanes reading rows or columns directly
// (64-byte steps) took more cycles of the L1 data stage than the shared
// memory traffic of the whole kernel.
// --------------------------------------------------------------------------
__device__ __forceinline__ void cp16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp4(void *dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp8(void *dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void prefetch_l2(const void *src) {
    asm volatile("prefetch.global.L2 [%0];" ::"l"(src));
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int K>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(K) : "memory"); }

// Shared layout of one warp's elements, in 16-byte slots.  Four-point rows
// are swizzled so that the eight lanes of a 128-bit access phase (two elements
// x four rows, or columns, or face points) fall in different banks; the other
// degrees use the natural order (rows of odd length are free of conflicts).
template <int N>
struct Line2 {
    static constexpr int NSP = N * N, NFP = 4 * N, MS = 5;
    static constexpr int EPW = 32 / N, WARPS = 4, TH = 32 * WARPS, EPB = EPW * WARPS;
    static constexpr bool FULL = EPW * N == 32;
    static constexpr int NP = EPW * NSP, NF = EPW * NFP;       // points, flux points of a warp
    static constexpr int NR = NP > NF ? NP : NF;               // partners' fluxes, later the RK register
    static constexpr int oU = 0, oG = NP, oUF = 3 * NP, oFV = oUF + NF, oGEO = oFV + NR, oM = oGEO + 2 * NF;
    static constexpr int SLOTS = oM + (NP * MS + 3) / 4;       // slots of a warp
    static constexpr size_t BYTES = (size_t)SLOTS * 16 * WARPS;
    // slot of point (row r, column c) of element j, of point l of group q (face
    // or face part) of element j with NG groups
    __device__ __forceinline__ static int pt(int j, int r, int c) {
        if (N == 4) return j * NSP + ((r ^ (j & 1)) << 2) + (c ^ r);
        return j * NSP + r * N + c;
    }
    template <int NG>
    __device__ __forceinline__ static int fp(int j, int q, int l) {
        if (N == 4) return j * (NG * N) + ((q ^ (j & 1)) << 2) + l;
        return j * (NG * N) + q * N + l;
    }
};

template <int N, int RL>
struct Line2Blocks {
    // CTAs per SM asked of the register allocator (shared memory holds 3 of
    // p = 3, 4: there level 2 has fewer registers and no CTA more)
    static constexpr int value = RL == 1 ? 2 : RL == 2 ? 4 : 3;
};

template <int N, int RL = 0>
__global__ void __launch_bounds__((Line2<N>::TH), (Line2Blocks<N, RL>::value))
k_line2(const __grid_constant__ KArgs<float> a) {
    using L = Line2<N>;
    using real = float;
    constexpr int D = 2, V = 4, NSP = L::NSP, NFP = L::NFP, MS = L::MS;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    float4 *sm = reinterpret_cast<float4 *>(smem_raw) + wid * L::SLOTS;
    const int64_t e0 = a.elem0 + (int64_t)blockIdx.x * L::EPB + wid * L::EPW;
    const int64_t e_end = a.elem0 + a.n_elem;
    if (e0 >= e_end) return;                       // whole warps: only warp barriers below
    const int ne = (int)min((int64_t)L::EPW, e_end - e0);
    const int mode = a.mode;
    const bool faces_only = mode == M_FACES;

    auto copy_points = [&](int o, const real *src) {
#pragma unroll
        for (int i = 0; i < (L::NP + 31) / 32; ++i) {
            const int it = lane + 32 * i;
            if (it < ne * NSP) {
                const int j = it / NSP, s = it % NSP;
                cp16(sm + o + L::pt(j, s / N, s % N), src + (e0 * NSP + it) * V);
            }
        }
    };
    {
        const real *src = a.MET + e0 * (NSP * MS);
        real *dst = reinterpret_cast<real *>(sm + L::oM);
        constexpr int per = NSP * MS;
        if (per % 4 == 0) {
#pragma unroll
            for (int i = 0; i < (L::EPW * per / 4 + 31) / 32; ++i) {
                const int it = lane + 32 * i;
                if (it < ne * (per / 4)) cp16(dst + 4 * it, src + 4 * it);
            }
        } else {
            for (int it = lane; it < ne * per; it += 32) cp4(dst + it, src + it);
        }
    }
#pragma unroll
    for (int i = 0; i < (2 * L::NF + 31) / 32; ++i) {
        const int it = lane + 32 * i;
        if (it < ne * 2 * NFP) {
            const int j = it / (2 * NFP), q = it % (2 * NFP);
            cp16(sm + L::oGEO + L::template fp<8>(j, q / N, q % N), a.FGEO + (e0 * 2 * NFP + it) * 4);
        }
    }
    pdl_wait();
    copy_points(L::oU, a.U);
    cp_commit();
    if (!faces_only) {
#pragma unroll
        for (int i = 0; i < (L::NF + 31) / 32; ++i) {
            const int it = lane + 32 * i;
            if (it < ne * NFP) {
                const int j = it / NFP, q = it % NFP, sl = L::template fp<4>(j, q / N, q % N);
                cp16(sm + L::oUF + sl, a.UFin + (e0 * NFP + it) * V);
                cp16(sm + L::oFV + sl, a.FVin + (e0 * NFP + it) * V);
            }
        }
    }
    cp_commit();

    // lanes without an element of their own repeat the last one and store nothing
    const bool live = lane < ne * N;
    const int j = min(lane / N, ne - 1), l = lane % N;
    const int64_t e = e0 + j;
    int ro[N], co[N];                              // slots of this thread's row and column
#pragma unroll
    for (int m = 0; m < N; ++m) {
        ro[m] = L::pt(j, l, m);
        co[m] = L::pt(j, m, l);
    }
    auto ld = [&](int slot, real *o) {
        const float4 t = sm[slot];
        o[0] = t.x; o[1] = t.y; o[2] = t.z; o[3] = t.w;
    };
    auto st = [&](int slot, const real *o) {
        if (live) sm[slot] = make_float4(o[0], o[1], o[2], o[3]);
    };
    const real *gM = reinterpret_cast<const real *>(sm + L::oM) + (j * N + l) * (N * MS);
    const real gm1 = a.gamma - real(1), kq = a.kq;

    auto deriv = [&](const real (*x)[V], real (*d)[V]) {
#pragma unroll
        for (int i = 0; i < N; ++i) {
            V4 t = mul4(a.rD2[i * kMaxN], x[0]);
#pragma unroll
            for (int m = 1; m < N; ++m) t = fma4(a.rD2[i * kMaxN + m], x[m], t);
            t.get(d[i]);
        }
    };
    auto ends = [&](const real (*x)[V], real (*o)[V]) {
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            V4 t = mul4(a.rL2[s * kMaxN], x[0]);
#pragma unroll
            for (int m = 1; m < N; ++m) t = fma4(a.rL2[s * kMaxN + m], x[m], t);
            t.get(o[s]);
        }
    };
    // uncorrected physical gradient of the state (row x, all of it in field U)
    // at every point into the fields G, its values at the row's ends into Q0
    auto gradient = [&](const real (*x)[V], real (*Q0)[D][V]) {
        {
            real y[N][V], d[N][V];
#pragma unroll
            for (int m = 0; m < N; ++m) ld(L::oU + co[m], y[m]);
            deriv(y, d);
#pragma unroll
            for (int m = 0; m < N; ++m) st(L::oG + co[m], d[m]);
        }
        __syncwarp();
        real M[N * MS], dx[N][V];
        ld_row<N * MS>(gM, M);
        deriv(x, dx);
#pragma unroll
        for (int s = 0; s < 2; ++s)
#pragma unroll
            for (int d = 0; d < D; ++d)
#pragma unroll
                for (int v = 0; v < V; ++v) Q0[s][d][v] = 0;
#pragma unroll
        for (int i = 0; i < N; ++i) {
            real dy[V];
            ld(L::oG + ro[i], dy);
            const real *m = M + i * MS;
#pragma unroll
            for (int d = 0; d < D; ++d) {
                const real c0 = m[d] * m[4], c1 = m[2 + d] * m[4];
                real g[V];
#pragma unroll
                for (int v = 0; v < V; ++v) g[v] = c0 * dx[i][v] + c1 * dy[v];
                st(L::oG + d * L::NP + ro[i], g);
#pragma unroll
                for (int s = 0; s < 2; ++s) {
                    V4 t;
                    t.set(Q0[s][d]);
                    fma4(a.rL2[s * kMaxN + i], g, t).get(Q0[s][d]);
                }
            }
        }
        __syncwarp();
    };
    auto ends_grad = [&](real (*Q)[D][V]) {        // at the column's ends
#pragma unroll
        for (int d = 0; d < D; ++d) {
            real x[N][V], o[2][V];
#pragma unroll
            for (int m = 0; m < N; ++m) ld(L::oG + d * L::NP + co[m], x[m]);
            ends(x, o);
#pragma unroll
            for (int s = 0; s < 2; ++s)
#pragma unroll
                for (int v = 0; v < V; ++v) Q[s][d][v] = o[s][v];
        }
    };
    auto geo = [&](int f, FaceGeo<D, real> &g) {
        const float4 A = sm[L::oGEO + L::template fp<8>(j, 2 * f, l)], B = sm[L::oGEO + L::template fp<8>(j, 2 * f + 1, l)];
        g.n[0] = A.x; g.n[1] = A.y; g.lf[0] = A.z; g.lf[1] = A.w;
        g.lfp[0] = B.x; g.lfp[1] = B.y; g.pt = __float_as_int(B.z);
    };

    real u[N][V];
    cp_wait<1>();
    __syncwarp();
#pragma unroll
    for (int m = 0; m < N; ++m) ld(L::oU + ro[m], u[m]);

    if (!faces_only) {
        real Fs[D][2][V], dd0[2][V];
        LineRef<D, real> R;      // the element's flux reference, its own or the global one
        {
            real u0[V];
            ld(L::oU + L::pt(j, 0, 0), u0);
            line_ref<D>(a.ref, u0, a.local_ref && !a.DIVREF, a.gamma, R);
        }
        // 1) common normal fluxes and jumps at the ends of this thread's row and column
        real Q[2][D][V], uf[2][V];
        gradient(u, Q);
        ends(u, uf);
        cp_wait<0>();
        __syncwarp();
        auto face_pair = [&](int k) {
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                FaceGeo<D, real> g;
                real uR[V], fvp[V], dd[V];
                const int sl = L::template fp<4>(j, 2 * k + s, l);
                geo(2 * k + s, g);
                ld(L::oUF + sl, uR);
                ld(L::oFV + sl, fvp);
                line_face<D, N>(a, R, g, uf[s], Q[s], uR, fvp, kq, Fs[k][s], dd);
                if (k == 0) {
#pragma unroll
                    for (int v = 0; v < V; ++v) dd0[s][v] = dd[v];
                } else {
                    st(L::oUF + sl, dd);           // the jump takes the partner state's slot
                }
            }
        };
        face_pair(0);
        {
            real y[N][V];
#pragma unroll
            for (int m = 0; m < N; ++m) ld(L::oU + co[m], y[m]);
            ends(y, uf);
        }
        ends_grad(Q);
        face_pair(1);
        __syncwarp();
        // the register array of the RK update comes in over the partners' viscous fluxes
        const bool lsrk = mode == M_LSRK;
        if (lsrk) copy_points(L::oFV, a.R1);
        cp_commit();

        // 2) transformed flux at the row's points, corrected gradient
        real f0[N][V], iJ[N];
        {
            real M[N * MS];
            ld_row<N * MS>(gM, M);
            const real cgl = a.rGL[l], cgr = a.rGR[l];
#pragma unroll
            for (int i = 0; i < N; ++i) {
                const real *m = M + i * MS;
                iJ[i] = m[4];
                real gr[D][V], c0[V], c1[V], dm[V], dp[V];
                ld(L::oUF + L::template fp<4>(j, 2, i), dm);
                ld(L::oUF + L::template fp<4>(j, 3, i), dp);
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    c0[v] = a.rGL[i] * dd0[0][v] + a.rGR[i] * dd0[1][v];
                    c1[v] = cgl * dm[v] + cgr * dp[v];
                }
#pragma unroll
                for (int d = 0; d < D; ++d) {
                    ld(L::oG + d * L::NP + ro[i], gr[d]);
                    const real k0 = m[d] * m[4], k1 = m[2 + d] * m[4];
#pragma unroll
                    for (int v = 0; v < V; ++v) gr[d][v] += k0 * c0[v] + k1 * c1[v];
                }
                real F[D][V];
                line_flux<D>(a, R, u[i], gr, gm1, kq, F);
                real t[V];
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    f0[i][v] = m[0] * F[0][v] + m[1] * F[1][v];
                    t[v] = m[2] * F[0][v] + m[3] * F[1][v];
                }
                st(L::oG + ro[i], t);
            }
        }
        __syncwarp();

        // 3) divergence + correction along the column and the row (the flux
        // polynomial's end values are folded into DT), then the RK update
        auto line_div = [&](const real (*x)[V], const real (*F2)[V], real (*o)[V]) {
#pragma unroll
            for (int i = 0; i < N; ++i) {
                V4 t = fma4(a.rGLm2[i], F2[0], mul4(a.rGR2[i], F2[1]));
#pragma unroll
                for (int m = 0; m < N; ++m) t = fma4(a.rDT2[i * kMaxN + m], x[m], t);
                t.get(o[i]);
            }
        };
        {
            real y[N][V], o[N][V];
#pragma unroll
            for (int m = 0; m < N; ++m) ld(L::oG + co[m], y[m]);
            line_div(y, Fs[1], o);
#pragma unroll
            for (int m = 0; m < N; ++m) st(L::oG + co[m], o[m]);
        }
        real dv[N][V];
        line_div(f0, Fs[0], dv);
        cp_wait<0>();
        __syncwarp();
        const int64_t row = (e * NSP + l * N) * V;
#pragma unroll
        for (int i = 0; i < N; ++i) {
            real x[V];
            ld(L::oG + ro[i], x);
#pragma unroll
            for (int v = 0; v < V; ++v) dv[i][v] += x[v];
        }
        if (a.DIVREF) {
            // the constant reference flux's share of the divergence
            real dr[N][V];
            ld_row<N * V>(a.DIVREF + row, &dr[0][0]);
#pragma unroll
            for (int i = 0; i < N; ++i)
#pragma unroll
                for (int v = 0; v < V; ++v) dv[i][v] += dr[i][v];
        }
#pragma unroll
        for (int i = 0; i < N; ++i)
#pragma unroll
            for (int v = 0; v < V; ++v) dv[i][v] *= -iJ[i];
        // shared field o back to memory, whole sectors
        auto write_points = [&](int o, real *dst) {
#pragma unroll
            for (int i = 0; i < (L::NP + 31) / 32; ++i) {
                const int it = lane + 32 * i;
                if (it < ne * NSP) {
                    const int jj = it / NSP, s = it % NSP;
                    reinterpret_cast<float4 *>(dst)[e0 * NSP + it] = sm[o + L::pt(jj, s / N, s % N)];
                }
            }
        };
        if (mode == M_LSRK_FIRST || mode == M_LSRK) {
#pragma unroll
            for (int i = 0; i < N; ++i) {
                real r[V];
                if (lsrk) {
                    ld(L::oFV + ro[i], r);
#pragma unroll
                    for (int v = 0; v < V; ++v) r[v] = a.rk_a * r[v] + a.dt * dv[i][v];
                } else {
#pragma unroll
                    for (int v = 0; v < V; ++v) r[v] = a.dt * dv[i][v];
                }
#pragma unroll
                for (int v = 0; v < V; ++v) u[i][v] += a.rk_b * r[v];
                st(L::oFV + ro[i], r);
                st(L::oU + ro[i], u[i]);
            }
            __syncwarp();
            write_points(L::oFV, a.R1);
            write_points(L::oU, a.U);
        } else {
            if (mode == M_RK4_1) {
                if (live) {
                    st_row<N * V>(a.R1 + row, &u[0][0]);
                    st_row<N * V>(a.R2 + row, &dv[0][0]);
                }
#pragma unroll
                for (int i = 0; i < N; ++i)
#pragma unroll
                    for (int v = 0; v < V; ++v) u[i][v] += a.rk_c * dv[i][v];
            } else {
                real r1[N][V], r2[N][V];
                ld_row<N * V>(a.R1 + row, &r1[0][0]);
                ld_row<N * V>(a.R2 + row, &r2[0][0]);
                const bool last = mode == M_RK4_4;
#pragma unroll
                for (int i = 0; i < N; ++i)
#pragma unroll
                    for (int v = 0; v < V; ++v) {
                        const real acc = last ? r2[i][v] + dv[i][v] : r2[i][v] + real(2) * dv[i][v];
                        u[i][v] = r1[i][v] + a.rk_c * (last ? acc : dv[i][v]);
                        r2[i][v] = acc;
                    }
                if (live && !last) st_row<N * V>(a.R2 + row, &r2[0][0]);
            }
#pragma unroll
            for (int i = 0; i < N; ++i) st(L::oU + ro[i], u[i]);
            __syncwarp();
            write_points(L::oU, a.U);
        }
    } else {
        cp_wait<0>();
        __syncwarp();
    }

    // 4) the new state's gradient, then face state + gradient flux part to the
    // partners' inbound slots for the next stage
    real Q[2][D][V], uf[2][V];
    gradient(u, Q);
    auto send = [&](int k) {
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            FaceGeo<D, real> g;
            geo(2 * k + s, g);
            if (!live || g.pt < 0) continue;
            real full[V], v[D], fv[V];
            add_ref<V>(a.ref, uf[s], full);
            const real ir = real(1) / full[0];
#pragma unroll
            for (int d = 0; d < D; ++d) v[d] = full[1 + d] * ir;
            visc_normal<D>(Q[s], v, full[V - 1] * ir, a.mu * ir, kq * ir, g.n, fv);
            st_v<V>(a.UFout + (int64_t)g.pt * V, uf[s]);
            st_v<V>(a.FVout + (int64_t)g.pt * V, fv);
        }
    };
    ends(u, uf);
    send(0);
    {
        real y[N][V];
#pragma unroll
        for (int m = 0; m < N; ++m) ld(L::oU + co[m], y[m]);
        ends(y, uf);
    }
    ends_grad(Q);
    send(1);
}

// --------------------------------------------------------------------------
// LDG on 2-D lines.  An LDG face needs both sides' corrected gradients, so a
// stage stays two kernels, in the layout and with the exchange of K_GRAD and
// K_FLUX (own viscous normal fluxes in FV, the partner's gathered): FLUX false
// the corrected gradient and the own viscous normal flux of every flux point,
// FLUX true the rest of the stage.  The work is split as in k_line2: the
// corrections of a row or column are its own thread's jumps, so nothing but
// the lines themselves passes through shared memory.  Bound as k_line2 (and by
// the call of the Roe flux); 20 steps of 26,568 quads of p = 4 with Roe 6.62 ->
// 4.47 ms against K_GRAD + K_FLUX.
// --------------------------------------------------------------------------
template <int D, typename real>
__device__ __forceinline__ void ldg_face(const KArgs<real> &a, const LineRef<D, real> &R, const FaceGeo<D, real> &g,
                                         int64_t gf, const real *uL, real *uR, const real *fvo, const real *fvp,
                                         real *Fs, real *dd) {
    constexpr int V = D + 2;
    const real gm1 = a.gamma - real(1);
    const bool inner = g.pt >= 0;
    real uLl[V], uRl[V], ub[V];
#pragma unroll
    for (int v = 0; v < V; ++v) uLl[v] = uL[v] - R.du[v];
    if (!inner) {
        BcIn<D, real> in;
#pragma unroll
        for (int v = 0; v < V; ++v) { in.u[v] = uLl[v]; in.du[v] = R.du[v]; }
#pragma unroll
        for (int d = 0; d < D; ++d) in.n[d] = g.n[d];
        const BcPair<D, real> o = bc_call<D, real>(&a, -1 - g.pt, in);
#pragma unroll
        for (int v = 0; v < V; ++v) {
            uRl[v] = o.ug[v];
            uR[v] = o.ug[v] + R.du[v];
            ub[v] = o.ub[v] + R.du[v];
        }
    } else {
#pragma unroll
        for (int v = 0; v < V; ++v) uRl[v] = uR[v] - R.du[v];
    }
    real nn = 0, vnr = 0;
#pragma unroll
    for (int d = 0; d < D; ++d) {
        nn += g.n[d] * g.n[d];
        vnr += R.v[d] * g.n[d];
    }
    if (a.flux == 1) {
        RoeIn<D, real> in;
#pragma unroll
        for (int v = 0; v < V; ++v) { in.uL[v] = uLl[v]; in.uR[v] = uRl[v]; in.du[v] = R.du[v]; }
#pragma unroll
        for (int d = 0; d < D; ++d) in.n[d] = g.n[d];
        const RoeOut<D, real> o = roe_call<D, real>(&a, in);
#pragma unroll
        for (int v = 0; v < V; ++v) Fs[v] = o.F[v];
    } else {
        real ir, vp[D], vel[D], pp, p, FL[V], FR[V];
        prim_line<D>(uLl, R, gm1, ir, vp, vel, pp, p);
        const real sL = normal_flux_prim<D>(uLl, vp, vel, pp, p, ir, g.n, vnr, nn, R, a.gamma, FL);
        prim_line<D>(uRl, R, gm1, ir, vp, vel, pp, p);
        const real sR = normal_flux_prim<D>(uRl, vp, vel, pp, p, ir, g.n, vnr, nn, R, a.gamma, FR);
        const real lam = real(0.5) * fmax(sL, sR);
#pragma unroll
        for (int v = 0; v < V; ++v) Fs[v] = real(0.5) * (FL[v] + FR[v]) - lam * (uR[v] - uL[v]);
    }
    if (inner) {
        // the side with the smaller point index is the left one
        const real bs = gf < g.pt ? a.ldg_beta : -a.ldg_beta, pen = a.ldg_tau * sqrt(nn);
#pragma unroll
        for (int v = 0; v < V; ++v) {
            dd[v] = (real(0.5) - bs) * (uR[v] - uL[v]);
            Fs[v] += pen * (uL[v] - uR[v]) - ((real(0.5) - bs) * fvo[v] - (real(0.5) + bs) * fvp[v]);
        }
    } else {
#pragma unroll
        for (int v = 0; v < V; ++v) {
            dd[v] = ub[v] - uL[v];
            Fs[v] -= fvo[v];
        }
    }
}

template <int N, bool FLUX>
__global__ void __launch_bounds__((Line2<N>::TH), 3)
k_ldg2(const __grid_constant__ KArgs<float> a) {
    using L = Line2<N>;
    using real = float;
    constexpr int D = 2, V = 4, NSP = L::NSP, NFP = L::NFP, MS = L::MS;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    float4 *sm = reinterpret_cast<float4 *>(smem_raw) + wid * L::SLOTS;
    const int64_t e0 = a.elem0 + (int64_t)blockIdx.x * L::EPB + wid * L::EPW;
    const int64_t e_end = a.elem0 + a.n_elem;
    if (e0 >= e_end) return;                       // whole warps: only warp barriers below
    const int ne = (int)min((int64_t)L::EPW, e_end - e0);
    const int mode = a.mode;

    auto copy_points = [&](int o, const real *src) {
#pragma unroll
        for (int i = 0; i < (L::NP + 31) / 32; ++i) {
            const int it = lane + 32 * i;
            if (it < ne * NSP) {
                const int j = it / NSP, s = it % NSP;
                cp16(sm + o + L::pt(j, s / N, s % N), src + (e0 * NSP + it) * V);
            }
        }
    };
    {
        const real *src = a.MET + e0 * (NSP * MS);
        real *dst = reinterpret_cast<real *>(sm + L::oM);
        constexpr int per = NSP * MS;
        if (per % 4 == 0) {
#pragma unroll
            for (int i = 0; i < (L::EPW * per / 4 + 31) / 32; ++i) {
                const int it = lane + 32 * i;
                if (it < ne * (per / 4)) cp16(dst + 4 * it, src + 4 * it);
            }
        } else {
            for (int it = lane; it < ne * per; it += 32) cp4(dst + it, src + it);
        }
    }
#pragma unroll
    for (int i = 0; i < (2 * L::NF + 31) / 32; ++i) {
        const int it = lane + 32 * i;
        if (it < ne * 2 * NFP) {
            const int j = it / (2 * NFP), q = it % (2 * NFP);
            cp16(sm + L::oGEO + L::template fp<8>(j, q / N, q % N), a.FGEO + (e0 * 2 * NFP + it) * 4);
        }
    }
    pdl_wait();
    copy_points(L::oU, a.U);
    cp_commit();
    {
#pragma unroll
        for (int i = 0; i < (L::NF + 31) / 32; ++i) {
            const int it = lane + 32 * i;
            if (it < ne * NFP) {
                const int j = it / NFP, q = it % NFP, sl = L::template fp<4>(j, q / N, q % N);
                cp16(sm + L::oUF + sl, a.UFin + (e0 * NFP + it) * V);
                if (FLUX) cp16(sm + L::oFV + sl, a.FV + (e0 * NFP + it) * V);
            }
        }
    }
    cp_commit();

    // lanes without an element of their own repeat the last one and store nothing
    const bool live = lane < ne * N;
    const int j = min(lane / N, ne - 1), l = lane % N;
    const int64_t e = e0 + j;
    int ro[N], co[N];                              // slots of this thread's row and column
#pragma unroll
    for (int m = 0; m < N; ++m) {
        ro[m] = L::pt(j, l, m);
        co[m] = L::pt(j, m, l);
    }
    auto ld = [&](int slot, real *o) {
        const float4 t = sm[slot];
        o[0] = t.x; o[1] = t.y; o[2] = t.z; o[3] = t.w;
    };
    auto st = [&](int slot, const real *o) {
        if (live) sm[slot] = make_float4(o[0], o[1], o[2], o[3]);
    };
    const real *gM = reinterpret_cast<const real *>(sm + L::oM) + (j * N + l) * (N * MS);
    const real gm1 = a.gamma - real(1), kq = a.kq;

    auto ends = [&](const real (*x)[V], real (*o)[V]) {
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            V4 t = mul4(a.rL2[s * kMaxN], x[0]);
#pragma unroll
            for (int m = 1; m < N; ++m) t = fma4(a.rL2[s * kMaxN + m], x[m], t);
            t.get(o[s]);
        }
    };
    // derivative of a line with the correction of its jumps
    auto corrected = [&](const real (*x)[V], const real (*dd)[V], real (*d)[V]) {
#pragma unroll
        for (int i = 0; i < N; ++i) {
            V4 t = mul4(a.rD2[i * kMaxN], x[0]);
#pragma unroll
            for (int m = 1; m < N; ++m) t = fma4(a.rD2[i * kMaxN + m], x[m], t);
            fma4(a.rGL2[i], dd[0], fma4(a.rGR2[i], dd[1], t)).get(d[i]);
        }
    };
    auto columns = [&](const real (*dd)[V]) {      // the column's corrected derivative into field G
        real y[N][V], d[N][V];
#pragma unroll
        for (int m = 0; m < N; ++m) ld(L::oU + co[m], y[m]);
        corrected(y, dd, d);
#pragma unroll
        for (int m = 0; m < N; ++m) st(L::oG + co[m], d[m]);
    };
    // physical gradient at point i of the row from its corrected derivatives
    auto grad_pt = [&](const real *m, const real *dx, const real *dy, real (*g)[V]) {
#pragma unroll
        for (int d = 0; d < D; ++d) {
            const real c0 = m[d] * m[4], c1 = m[2 + d] * m[4];
#pragma unroll
            for (int v = 0; v < V; ++v) g[d][v] = c0 * dx[v] + c1 * dy[v];
        }
    };
    auto ends_grad = [&](real (*Q)[D][V]) {        // at the column's ends
#pragma unroll
        for (int d = 0; d < D; ++d) {
            real x[N][V], o[2][V];
#pragma unroll
            for (int m = 0; m < N; ++m) ld(L::oG + d * L::NP + co[m], x[m]);
            ends(x, o);
#pragma unroll
            for (int s = 0; s < 2; ++s)
#pragma unroll
                for (int v = 0; v < V; ++v) Q[s][d][v] = o[s][v];
        }
    };
    auto geo = [&](int f, FaceGeo<D, real> &g) {
        const float4 A = sm[L::oGEO + L::template fp<8>(j, 2 * f, l)], B = sm[L::oGEO + L::template fp<8>(j, 2 * f + 1, l)];
        g.n[0] = A.x; g.n[1] = A.y; g.lf[0] = A.z; g.lf[1] = A.w;
        g.lfp[0] = B.x; g.lfp[1] = B.y; g.pt = __float_as_int(B.z);
    };

    real u[N][V], ufr[2][V], ufc[2][V];
    cp_wait<0>();
    __syncwarp();
#pragma unroll
    for (int m = 0; m < N; ++m) ld(L::oU + ro[m], u[m]);
    ends(u, ufr);
    {
        real y[N][V];
#pragma unroll
        for (int m = 0; m < N; ++m) ld(L::oU + co[m], y[m]);
        ends(y, ufc);
    }
    auto face_of = [&](int f) { return e * NFP + f * N + l; };

    if constexpr (!FLUX) {
        // jumps u_c - u_f and the state of the viscous flux (in place of u_f)
        real ddr[2][V], ddc[2][V];
        auto jumps = [&](int k, real (*uf)[V], real (*dd)[V]) {
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                FaceGeo<D, real> g;
                geo(2 * k + s, g);
                if (g.pt >= 0) {
                    real uR[V];
                    ld(L::oUF + L::template fp<4>(j, 2 * k + s, l), uR);
                    const real c = real(0.5) - (face_of(2 * k + s) < g.pt ? a.ldg_beta : -a.ldg_beta);
#pragma unroll
                    for (int v = 0; v < V; ++v) dd[s][v] = c * (uR[v] - uf[s][v]);
                } else {
                    BcIn<D, real> in;
#pragma unroll
                    for (int v = 0; v < V; ++v) { in.u[v] = uf[s][v]; in.du[v] = 0; }
#pragma unroll
                    for (int d = 0; d < D; ++d) in.n[d] = g.n[d];
                    const BcPair<D, real> o = bc_call<D, real>(&a, -1 - g.pt, in);
#pragma unroll
                    for (int v = 0; v < V; ++v) {
                        dd[s][v] = o.ub[v] - uf[s][v];
                        uf[s][v] = o.ub[v];
                    }
                }
            }
        };
        jumps(0, ufr, ddr);
        jumps(1, ufc, ddc);
        columns(ddc);
        __syncwarp();
        real Q[2][D][V];
        {
            real M[N * MS], dx[N][V];
            ld_row<N * MS>(gM, M);
            corrected(u, ddr, dx);
#pragma unroll
            for (int s = 0; s < 2; ++s)
#pragma unroll
                for (int d = 0; d < D; ++d)
#pragma unroll
                    for (int v = 0; v < V; ++v) Q[s][d][v] = 0;
#pragma unroll
            for (int i = 0; i < N; ++i) {
                real dy[V], g[D][V];
                ld(L::oG + ro[i], dy);
                grad_pt(M + i * MS, dx[i], dy, g);
#pragma unroll
                for (int d = 0; d < D; ++d) {
                    st(L::oG + d * L::NP + ro[i], g[d]);
#pragma unroll
                    for (int s = 0; s < 2; ++s) {
                        V4 t;
                        t.set(Q[s][d]);
                        fma4(a.rL2[s * kMaxN + i], g[d], t).get(Q[s][d]);
                    }
                }
            }
        }
        __syncwarp();
        auto own_flux = [&](int k, const real (*uf)[V]) {
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                FaceGeo<D, real> g;
                geo(2 * k + s, g);
                real full[V], vel[D], fv[V];
                add_ref<V>(a.ref, uf[s], full);
                const real ir = real(1) / full[0];
#pragma unroll
                for (int d = 0; d < D; ++d) vel[d] = full[1 + d] * ir;
                visc_normal<D>(Q[s], vel, full[V - 1] * ir, a.mu * ir, kq * ir, g.n, fv);
                if (g.pt < 0 && a.BTAG[-1 - g.pt] == BC_WALL) fv[V - 1] = 0;   // adiabatic wall
                if (live) st_v<V>(a.FV + face_of(2 * k + s) * V, fv);
            }
        };
        own_flux(0, ufr);
        ends_grad(Q);
        own_flux(1, ufc);
    } else {
        real Fs[D][2][V], ddr[2][V];
        LineRef<D, real> R;      // the element's flux reference, its own or the global one
        {
            real u0[V];
            ld(L::oU + L::pt(j, 0, 0), u0);
            line_ref<D>(a.ref, u0, a.local_ref && !a.DIVREF, a.gamma, R);
        }
        // 1) common normal fluxes and jumps at the ends of this thread's row and column
        auto face_pair = [&](int k, const real (*uf)[V], real (*dd)[V]) {
            FaceGeo<D, real> g[2];
            real fvp[2][V] = {};
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                geo(2 * k + s, g[s]);
                if (g[s].pt >= 0) ld_v<V>(a.FV + (int64_t)g[s].pt * V, fvp[s]);
            }
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                real uR[V], fvo[V];
                const int sl = L::template fp<4>(j, 2 * k + s, l);
                ld(L::oUF + sl, uR);
                ld(L::oFV + sl, fvo);
                ldg_face<D>(a, R, g[s], face_of(2 * k + s), uf[s], uR, fvo, fvp[s], Fs[k][s], dd[s]);
            }
        };
        {
            real ddc[2][V];
            face_pair(1, ufc, ddc);
            columns(ddc);
        }
        face_pair(0, ufr, ddr);
        __syncwarp();
        // the register array of the RK update comes in over the viscous fluxes
        const bool lsrk = mode == M_LSRK;
        if (lsrk) copy_points(L::oFV, a.R1);
        cp_commit();

        // 2) transformed flux at the row's points
        real f0[N][V], iJ[N];
        {
            real M[N * MS], dx[N][V];
            ld_row<N * MS>(gM, M);
            corrected(u, ddr, dx);
#pragma unroll
            for (int i = 0; i < N; ++i) {
                const real *m = M + i * MS;
                iJ[i] = m[4];
                real dy[V], gr[D][V], F[D][V], t[V];
                ld(L::oG + ro[i], dy);
                grad_pt(m, dx[i], dy, gr);
                line_flux<D>(a, R, u[i], gr, gm1, kq, F);
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    f0[i][v] = m[0] * F[0][v] + m[1] * F[1][v];
                    t[v] = m[2] * F[0][v] + m[3] * F[1][v];
                }
                st(L::oG + ro[i], t);
            }
        }
        __syncwarp();

        // 3) divergence + correction along the column and the row (the flux
        // polynomial's end values are folded into DT), then the RK update
        auto line_div = [&](const real (*x)[V], const real (*F2)[V], real (*o)[V]) {
#pragma unroll
            for (int i = 0; i < N; ++i) {
                V4 t = fma4(a.rGLm2[i], F2[0], mul4(a.rGR2[i], F2[1]));
#pragma unroll
                for (int m = 0; m < N; ++m) t = fma4(a.rDT2[i * kMaxN + m], x[m], t);
                t.get(o[i]);
            }
        };
        {
            real y[N][V], o[N][V];
#pragma unroll
            for (int m = 0; m < N; ++m) ld(L::oG + co[m], y[m]);
            line_div(y, Fs[1], o);
#pragma unroll
            for (int m = 0; m < N; ++m) st(L::oG + co[m], o[m]);
        }
        real dv[N][V];
        line_div(f0, Fs[0], dv);
        cp_wait<0>();
        __syncwarp();
        const int64_t row = (e * NSP + l * N) * V;
#pragma unroll
        for (int i = 0; i < N; ++i) {
            real x[V];
            ld(L::oG + ro[i], x);
#pragma unroll
            for (int v = 0; v < V; ++v) dv[i][v] += x[v];
        }
        if (a.DIVREF) {
            // the constant reference flux's share of the divergence
            real dr[N][V];
            ld_row<N * V>(a.DIVREF + row, &dr[0][0]);
#pragma unroll
            for (int i = 0; i < N; ++i)
#pragma unroll
                for (int v = 0; v < V; ++v) dv[i][v] += dr[i][v];
        }
#pragma unroll
        for (int i = 0; i < N; ++i)
#pragma unroll
            for (int v = 0; v < V; ++v) dv[i][v] *= -iJ[i];
        // shared field o back to memory, whole sectors
        auto write_points = [&](int o, real *dst) {
#pragma unroll
            for (int i = 0; i < (L::NP + 31) / 32; ++i) {
                const int it = lane + 32 * i;
                if (it < ne * NSP) {
                    const int jj = it / NSP, s = it % NSP;
                    reinterpret_cast<float4 *>(dst)[e0 * NSP + it] = sm[o + L::pt(jj, s / N, s % N)];
                }
            }
        };
        if (mode == M_LSRK_FIRST || mode == M_LSRK) {
#pragma unroll
            for (int i = 0; i < N; ++i) {
                real r[V];
                if (lsrk) {
                    ld(L::oFV + ro[i], r);
#pragma unroll
                    for (int v = 0; v < V; ++v) r[v] = a.rk_a * r[v] + a.dt * dv[i][v];
                } else {
#pragma unroll
                    for (int v = 0; v < V; ++v) r[v] = a.dt * dv[i][v];
                }
#pragma unroll
                for (int v = 0; v < V; ++v) u[i][v] += a.rk_b * r[v];
                st(L::oFV + ro[i], r);
                st(L::oU + ro[i], u[i]);
            }
            __syncwarp();
            write_points(L::oFV, a.R1);
            write_points(L::oU, a.U);
        } else {
            if (mode == M_RK4_1) {
                if (live) {
                    st_row<N * V>(a.R1 + row, &u[0][0]);
                    st_row<N * V>(a.R2 + row, &dv[0][0]);
                }
#pragma unroll
                for (int i = 0; i < N; ++i)
#pragma unroll
                    for (int v = 0; v < V; ++v) u[i][v] += a.rk_c * dv[i][v];
            } else {
                real r1[N][V], r2[N][V];
                ld_row<N * V>(a.R1 + row, &r1[0][0]);
                ld_row<N * V>(a.R2 + row, &r2[0][0]);
                const bool last = mode == M_RK4_4;
#pragma unroll
                for (int i = 0; i < N; ++i)
#pragma unroll
                    for (int v = 0; v < V; ++v) {
                        const real acc = last ? r2[i][v] + dv[i][v] : r2[i][v] + real(2) * dv[i][v];
                        u[i][v] = r1[i][v] + a.rk_c * (last ? acc : dv[i][v]);
                        r2[i][v] = acc;
                    }
                if (live && !last) st_row<N * V>(a.R2 + row, &r2[0][0]);
            }
#pragma unroll
            for (int i = 0; i < N; ++i) st(L::oU + ro[i], u[i]);
            __syncwarp();
            write_points(L::oU, a.U);
        }
        // 4) the new face states to the partners' inbound slots
        auto send = [&](int k, const real (*uf)[V]) {
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                FaceGeo<D, real> g;
                geo(2 * k + s, g);
                if (live && g.pt >= 0) st_v<V>(a.UFout + (int64_t)g.pt * V, uf[s]);
            }
        };
        ends(u, ufr);
        send(0, ufr);
        real y[N][V];
#pragma unroll
        for (int m = 0; m < N; ++m) ld(L::oU + co[m], y[m]);
        ends(y, ufc);
        send(1, ufc);
    }
}

// --------------------------------------------------------------------------
// 3-D line kernel.  A thread owns line l of each of the three directions of
// its element.  A state or flux of five variables is one 128-bit vector (rho,
// rho v) and one word (rho E), in shared memory as in the face buffers.
// Loops over directions and points stay rolled where their bodies are long:
// unrolled, the kernel is 7,200 instructions that every warp runs once, and
// instruction fetch was the largest stall (p = 4: 4 of 10 cycles per issue).
// Metric terms come in an order of their own, so that neighbouring lanes read
// neighbouring vectors; they, the partners' states and viscous fluxes are
// fetched at the start by asynchronous copies, the face geometry and the RK
// register prefetched into L2.  Shared memory then holds two CTAs per SM,
// which leaves 255 registers a thread (three CTAs at 168 spill 260 bytes and
// measured 8 % slower).
//
// Measured (GB300, ms per LSRK45 step), gradient + flux kernels at their best
// register level -> this kernel: 48^3 hexes of p = 3 5.32 -> 3.12, 57,120 of
// p = 4 6.62 -> 4.59.  On the way (p = 3): unrolled, one plane per variable
// 4.56; loops rolled 3.90; vectors 3.43; staged inputs 3.29; prefetches 3.12.
// Bound by latency at 8 warps per SM: 45 % of the issue slots, 57 % of the L1
// data stage, 37 % of DRAM at p = 3.
// --------------------------------------------------------------------------
template <int N>
struct Line3 {
    static constexpr int V = 5, MS = 10, NSP = N * N * N, LPE = N * N, NFP = 6 * LPE;
    static constexpr int TH = 128;
    static constexpr bool WARP = LPE <= 16;             // an element's lines fit a warp
    static constexpr int EPW = WARP ? 32 / LPE : 1;
    static constexpr int EPB = WARP ? EPW * (TH / 32) : TH / LPE;
    // slot of point (i, j, k): i + SJ j + SK k, SE per element.  N = 4: with a
    // row of 5 slots every 128-bit phase of a row or column view and every
    // 32-bit access of them falls in different banks (the zeta view: one
    // conflict in eight lanes)
    static constexpr int SJ = N == 4 ? 5 : N, SK = N * SJ, SE = N * SK;
    static constexpr int NS = EPB * SE;                 // slots of a field
    static constexpr int ND = EPB * LPE;                // face jumps of one (direction, side)
    // fields: 0 state, 1..3 gradient / transformed flux; then the jumps of
    // directions 1, 2.  Vectors first, the fifth variable behind them
    static constexpr int SLOTS = 4 * NS + 4 * ND;
    // staged inputs: metric terms (two vectors and a pair per point), then the
    // partners' states and viscous fluxes (a vector and a word per flux point)
    static constexpr int NF = EPB * NFP, NM = EPB * NSP;
    static constexpr int oM = SLOTS, oUF = oM + 2 * NM, oFV = oUF + NF, VECS = oFV + NF;      // vectors
    static constexpr int oMC = (SLOTS + 1) / 2 * 2, oUE = oMC + 2 * NM, oFE = oUE + NF, TAILS = oFE + NF;   // words
    static constexpr size_t BYTES = (size_t)VECS * 16 + (size_t)TAILS * 4;
    static_assert(BYTES <= 115712, "two CTAs per SM");
    __device__ __forceinline__ static int step(int k) { return k == 0 ? 1 : (k == 1 ? SJ : SK); }
    __device__ __forceinline__ static int base(int k, int l) {
        return k == 0 ? (l % N) * SJ + (l / N) * SK : l % N + (l / N) * (k == 1 ? SK : SJ);
    }
};
// word of metric term c at point i of xi line `line` of element e of n_elem:
// [element][point of the line][two vectors of all lines], then [element][point]
// [one pair of all lines]
__host__ __device__ constexpr int64_t metl_word(int N, int64_t n_elem, int64_t e, int i, int c, int line) {
    return c < 8 ? (((e * N + i) * 2 + c / 4) * (N * N) + line) * 4 + c % 4
                 : n_elem * N * N * N * 8 + ((e * N + i) * (N * N) + line) * 2 + c - 8;
}

// Five variables, four of them as packed pairs (see V4)
struct V5 {
    V4 p;
    float c;
    __device__ __forceinline__ void get(float *x) const {
        p.get(x);
        x[4] = c;
    }
};
__device__ __forceinline__ V5 fma5(const float2 k, const float *x, const V5 &t) {
    return V5{fma4(k, x, t.p), fmaf(k.x, x[4], t.c)};
}
__device__ __forceinline__ V5 mul5(const float2 k, const float *x) { return V5{mul4(k, x), k.x * x[4]}; }

// face data of the 3-D line kernel: the vectors of all nf flux points, then
// their fifth variables
__device__ __forceinline__ void st_face3(float *buf, int64_t nf, int32_t pt, const float *o) {
    reinterpret_cast<float4 *>(buf)[pt] = make_float4(o[0], o[1], o[2], o[3]);
    buf[4 * nf + pt] = o[4];
}

template <int N>
__global__ void __launch_bounds__((Line3<N>::TH), 2)
k_line3(const __grid_constant__ KArgs<float> a) {
    using L = Line3<N>;
    using real = float;
    constexpr int D = 3, V = 5, NSP = L::NSP, LPE = L::LPE, MS = L::MS, NS = L::NS;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float4 *sv = reinterpret_cast<float4 *>(smem_raw);
    real *se = reinterpret_cast<real *>(sv + L::VECS);
    const int tid = threadIdx.x;
    const int64_t e_end = a.elem0 + a.n_elem, eb = a.elem0 + (int64_t)blockIdx.x * L::EPB;
    const int ne = (int)min((int64_t)L::EPB, e_end - eb);
    // element slot and line of this thread; threads without an element of
    // their own repeat another one's line and store nothing
    int j, l;
    bool live;
    if (L::WARP) {
        const int w = (tid >> 5) * L::EPW, x = (tid & 31) / LPE;
        if (w >= ne) return;                       // whole warps: only warp barriers below
        l = (tid & 31) % LPE;
        live = x < L::EPW && w + x < ne;
        j = live ? w + x : w;
    } else {
        j = tid / LPE;
        l = tid % LPE;
        live = j < ne;
        j = live ? j : 0;
    }
    auto sync = [] {
        if (L::WARP) __syncwarp();
        else __syncthreads();
    };
    const int64_t e = eb + j;
    const int la = l % N, lb = l / N;
    const int mode = a.mode;
    const real gm1 = a.gamma - real(1), kq = a.kq;
    const int64_t nf = a.fp_real;                  // flux points of the group
    {
        // the group's inputs (a warp's or the CTA's elements g0 .. g0 + gn)
        const int t0 = L::WARP ? tid & 31 : tid, nt = L::WARP ? 32 : L::TH;
        const int g0 = L::WARP ? (tid >> 5) * L::EPW : 0, gn = min(L::WARP ? L::EPW : L::EPB, ne - g0);
        const float4 *mA = reinterpret_cast<const float4 *>(a.METL) + (eb + g0) * (2 * NSP);
        const float2 *mC = reinterpret_cast<const float2 *>(a.METL + nf / L::NFP * NSP * 8) + (eb + g0) * NSP;
        for (int i = t0; i < gn * 2 * NSP; i += nt) cp16(sv + L::oM + g0 * 2 * NSP + i, mA + i);
        for (int i = t0; i < gn * NSP; i += nt) cp8(se + L::oMC + 2 * (g0 * NSP + i), mC + i);
        cp_commit();
        if (mode != M_FACES) {
            const int64_t f0 = (eb + g0) * L::NFP;
            for (int i = t0; i < gn * L::NFP; i += nt) {
                cp16(sv + L::oUF + g0 * L::NFP + i, a.UFin + 4 * (f0 + i));
                cp16(sv + L::oFV + g0 * L::NFP + i, a.FVin + 4 * (f0 + i));
                cp4(se + L::oUE + g0 * L::NFP + i, a.UFin + 4 * nf + f0 + i);
                cp4(se + L::oFE + g0 * L::NFP + i, a.FVin + 4 * nf + f0 + i);
            }
        }
        cp_commit();
        // what is read later from memory: into L2 meanwhile (128-byte lines)
        const char *pg = reinterpret_cast<const char *>(a.FGEO) + (eb + g0) * (L::NFP * 48);
        for (int i = t0 * 128; i < gn * L::NFP * 48; i += nt * 128) prefetch_l2(pg + i);
        if (mode == M_LSRK) {
            const char *pr = reinterpret_cast<const char *>(a.R1 + (eb + g0) * (NSP * V));
            for (int i = t0 * 128; i < gn * NSP * V * 4; i += nt * 128) prefetch_l2(pr + i);
        }
    }
    const float4 *mA = sv + L::oM + j * 2 * NSP + l;
    const float2 *mC = reinterpret_cast<const float2 *>(se + L::oMC) + j * NSP + l;
    auto met = [&](int i, real *M) {
        const float4 A = mA[2 * i * LPE], B = mA[(2 * i + 1) * LPE];
        const float2 C = mC[i * LPE];
        M[0] = A.x; M[1] = A.y; M[2] = A.z; M[3] = A.w; M[4] = B.x; M[5] = B.y; M[6] = B.z; M[7] = B.w;
        M[8] = C.x; M[9] = C.y;
    };
    auto ld = [&](int slot, real *o) {
        const float4 t = sv[slot];
        o[0] = t.x; o[1] = t.y; o[2] = t.z; o[3] = t.w;
        o[4] = se[slot];
    };
    auto st = [&](int slot, const real *o) {
        if (!live) return;
        sv[slot] = make_float4(o[0], o[1], o[2], o[3]);
        se[slot] = o[4];
    };
    auto deriv = [&](int i, const real (*x)[V], real *o) {
        V5 t = mul5(a.rD2[i * kMaxN], x[0]);
#pragma unroll
        for (int m = 1; m < N; ++m) t = fma5(a.rD2[i * kMaxN + m], x[m], t);
        t.get(o);
    };
    auto ends = [&](const real (*x)[V], real (*o)[V]) {
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            V5 t = mul5(a.rL2[s * kMaxN], x[0]);
#pragma unroll
            for (int m = 1; m < N; ++m) t = fma5(a.rL2[s * kMaxN + m], x[m], t);
            t.get(o[s]);
        }
    };
    const int ju = j * L::SE, jr = ju + L::base(0, l);     // the element's first slot, the row's
    const int64_t row = (e * NSP + l * N) * V;
    real u[N][V];
    ld_row<N * V>(a.U + row, &u[0][0]);
#pragma unroll
    for (int m = 0; m < N; ++m) st(jr + m, u[m]);
    cp_wait<1>();
    sync();

#pragma unroll 1
    for (int pass = mode == M_FACES ? 1 : 0; pass < 2; ++pass) {
        // uncorrected physical gradient of the state (u, field U) at every point into the fields G
#pragma unroll 1
        for (int k = 1; k < D; ++k) {
            const int o = ju + L::base(k, l), so = L::step(k);
            real x[N][V];
#pragma unroll
            for (int m = 0; m < N; ++m) ld(o + m * so, x[m]);
#pragma unroll
            for (int i = 0; i < N; ++i) {
                real d[V];
                deriv(i, x, d);
                st(k * NS + o + i * so, d);
            }
        }
        sync();
#pragma unroll
        for (int i = 0; i < N; ++i) {
            real M[MS], dk[D][V];
            met(i, M);
            deriv(i, u, dk[0]);
            ld(NS + jr + i, dk[1]);
            ld(2 * NS + jr + i, dk[2]);
#pragma unroll
            for (int d = 0; d < D; ++d) {
                real g[V];
                const real c0 = M[d] * M[9], c1 = M[3 + d] * M[9], c2 = M[6 + d] * M[9];
#pragma unroll
                for (int v = 0; v < V; ++v) g[v] = c0 * dk[0][v] + c1 * dk[1][v] + c2 * dk[2][v];
                st((1 + d) * NS + jr + i, g);
            }
        }
        sync();

        if (pass == 1) {
            // 4) face state + gradient flux part of the (new) state to the
            // partners' inbound slots for the next stage
#pragma unroll 1
            for (int k = 0; k < D; ++k) {
                const int o = ju + L::base(k, l), so = L::step(k);
                const int64_t face = e * 6 + 2 * k;
                float4 geo[2];
#pragma unroll
                for (int s = 0; s < 2; ++s)
                    geo[s] = __ldg(reinterpret_cast<const float4 *>(a.FGEO) + (face + s) * (3 * LPE) + l);
                real uf[2][V], Q[2][D][V];
                {
                    real x[N][V];
#pragma unroll
                    for (int m = 0; m < N; ++m) ld(o + m * so, x[m]);
                    ends(x, uf);
                }
#pragma unroll
                for (int d = 0; d < D; ++d) {
                    real x[N][V], q[2][V];
#pragma unroll
                    for (int m = 0; m < N; ++m) ld((1 + d) * NS + o + m * so, x[m]);
                    ends(x, q);
#pragma unroll
                    for (int s = 0; s < 2; ++s)
#pragma unroll
                        for (int v = 0; v < V; ++v) Q[s][d][v] = q[s][v];
                }
#pragma unroll
                for (int s = 0; s < 2; ++s) {
                    const int32_t pt = __float_as_int(geo[s].w);
                    if (!live || pt < 0) continue;
                    const real n[D] = {geo[s].x, geo[s].y, geo[s].z};
                    real full[V], v[D], fv[V];
                    add_ref<V>(a.ref, uf[s], full);
                    const real ir = real(1) / full[0];
#pragma unroll
                    for (int d = 0; d < D; ++d) v[d] = full[1 + d] * ir;
                    visc_normal<D>(Q[s], v, full[V - 1] * ir, a.mu * ir, kq * ir, n, fv);
                    st_face3(a.UFout, nf, pt, uf[s]);
                    st_face3(a.FVout, nf, pt, fv);
                }
            }
            return;
        }

        LineRef<D, real> R;      // the element's flux reference, its own or the global one
        {
            real u0[V];
            ld(ju, u0);
            line_ref<D>(a.ref, u0, a.local_ref && !a.DIVREF, a.gamma, R);
        }
        // 1) common normal fluxes and jumps at the ends of this thread's lines
        cp_wait<0>();
        sync();
        real F0[2][V], F1[2][V], F2[2][V], dd0[2][V];
#pragma unroll 1
        for (int k = 0; k < D; ++k) {
            const int64_t face = e * 6 + 2 * k;
            FaceGeo<D, real> g[2];
            real uR[2][V], fvp[2][V];
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                const float4 *p = reinterpret_cast<const float4 *>(a.FGEO) + (face + s) * (3 * LPE) + l;
                const float4 A = __ldg(p), B = __ldg(p + LPE), C = __ldg(p + 2 * LPE);
                g[s].n[0] = A.x; g[s].n[1] = A.y; g[s].n[2] = A.z; g[s].pt = __float_as_int(A.w);
                g[s].lf[0] = B.x; g[s].lf[1] = B.y; g[s].lf[2] = B.z;
                g[s].lfp[0] = C.x; g[s].lfp[1] = C.y; g[s].lfp[2] = C.z;
                const int q = j * L::NFP + (2 * k + s) * LPE + l;
                const float4 U = sv[L::oUF + q], W = sv[L::oFV + q];
                uR[s][0] = U.x; uR[s][1] = U.y; uR[s][2] = U.z; uR[s][3] = U.w; uR[s][4] = se[L::oUE + q];
                fvp[s][0] = W.x; fvp[s][1] = W.y; fvp[s][2] = W.z; fvp[s][3] = W.w; fvp[s][4] = se[L::oFE + q];
            }
            const int o = ju + L::base(k, l), so = L::step(k);
            real uf[2][V], Q[2][D][V];
            {
                real x[N][V];
#pragma unroll
                for (int m = 0; m < N; ++m) ld(o + m * so, x[m]);
                ends(x, uf);
            }
#pragma unroll
            for (int d = 0; d < D; ++d) {
                real x[N][V], q[2][V];
#pragma unroll
                for (int m = 0; m < N; ++m) ld((1 + d) * NS + o + m * so, x[m]);
                ends(x, q);
#pragma unroll
                for (int s = 0; s < 2; ++s)
#pragma unroll
                    for (int v = 0; v < V; ++v) Q[s][d][v] = q[s][v];
            }
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                real F[V], dd[V];
                line_face<D, N>(a, R, g[s], uf[s], Q[s], uR[s], fvp[s], kq, F, dd);
                if (k == 0) {
#pragma unroll
                    for (int v = 0; v < V; ++v) { F0[s][v] = F[v]; dd0[s][v] = dd[v]; }
                } else {
                    st(4 * NS + ((k - 1) * 2 + s) * L::ND + j * LPE + l, dd);
#pragma unroll
                    for (int v = 0; v < V; ++v) {
                        if (k == 1) F1[s][v] = F[v];
                        else F2[s][v] = F[v];
                    }
                }
            }
        }
        sync();

        // 2) transformed flux at the points of the xi line, corrected gradient
        {
            const real g1l = a.rGL[la], g1r = a.rGR[la], g2l = a.rGL[lb], g2r = a.rGR[lb];
            const int jd = 4 * NS + j * LPE;
#pragma unroll 1
            for (int i = 0; i < N; ++i) {
                real M[MS], ui[V], gr[D][V], d1m[V], d1p[V], d2m[V], d2p[V];
                met(i, M);
                ld(jr + i, ui);
#pragma unroll
                for (int d = 0; d < D; ++d) ld((1 + d) * NS + jr + i, gr[d]);
                ld(jd + i + N * lb, d1m);
                ld(jd + L::ND + i + N * lb, d1p);
                ld(jd + 2 * L::ND + i + N * la, d2m);
                ld(jd + 3 * L::ND + i + N * la, d2p);
                const real g0l = a.rGL[i], g0r = a.rGR[i];
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    const real c0 = M[9] * (g0l * dd0[0][v] + g0r * dd0[1][v]);
                    const real c1 = M[9] * (g1l * d1m[v] + g1r * d1p[v]);
                    const real c2 = M[9] * (g2l * d2m[v] + g2r * d2p[v]);
#pragma unroll
                    for (int d = 0; d < D; ++d) gr[d][v] += M[d] * c0 + M[3 + d] * c1 + M[6 + d] * c2;
                }
                real F[D][V];
                line_flux<D>(a, R, ui, gr, gm1, kq, F);
#pragma unroll
                for (int k = 0; k < D; ++k) {
                    real t[V];
#pragma unroll
                    for (int v = 0; v < V; ++v) t[v] = M[3 * k] * F[0][v] + M[3 * k + 1] * F[1][v] + M[3 * k + 2] * F[2][v];
                    st((1 + k) * NS + jr + i, t);
                }
            }
        }
        sync();

        // 3) divergence + correction along every line (the flux polynomial's
        // end values are folded into DT), then the RK update of the xi line
        auto div_pt = [&](int i, const real (*x)[V], const real (*F)[V], real *o) {
            V5 t = fma5(a.rGLm2[i], F[0], mul5(a.rGR2[i], F[1]));
#pragma unroll
            for (int m = 0; m < N; ++m) t = fma5(a.rDT2[i * kMaxN + m], x[m], t);
            t.get(o);
        };
        real r1[N][V];           // issued here: its latency passes under the divergence
        if (mode == M_LSRK) ld_row<N * V>(a.R1 + row, &r1[0][0]);
#pragma unroll 1
        for (int k = 1; k < D; ++k) {
            const int o = (1 + k) * NS + ju + L::base(k, l), so = L::step(k);
            real x[N][V], F[2][V];
#pragma unroll
            for (int m = 0; m < N; ++m) ld(o + m * so, x[m]);
#pragma unroll
            for (int s = 0; s < 2; ++s)
#pragma unroll
                for (int v = 0; v < V; ++v) F[s][v] = k == 1 ? F1[s][v] : F2[s][v];
#pragma unroll
            for (int i = 0; i < N; ++i) {
                real d[V];
                div_pt(i, x, F, d);
                st(o + i * so, d);
            }
        }
        real dv[N][V];
        {
            real x[N][V];
#pragma unroll
            for (int m = 0; m < N; ++m) ld(NS + jr + m, x[m]);
#pragma unroll
            for (int i = 0; i < N; ++i) div_pt(i, x, F0, dv[i]);
        }
        sync();
#pragma unroll
        for (int i = 0; i < N; ++i) {
            real x[V], y[V];
            ld(2 * NS + jr + i, x);
            ld(3 * NS + jr + i, y);
#pragma unroll
            for (int v = 0; v < V; ++v) dv[i][v] += x[v] + y[v];
        }
        if (a.DIVREF) {
            // the constant reference flux's share of the divergence
            real dr[N][V];
            ld_row<N * V>(a.DIVREF + row, &dr[0][0]);
#pragma unroll
            for (int i = 0; i < N; ++i)
#pragma unroll
                for (int v = 0; v < V; ++v) dv[i][v] += dr[i][v];
        }
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const real iJ = mC[i * LPE].y;
#pragma unroll
            for (int v = 0; v < V; ++v) dv[i][v] *= -iJ;
        }
        if (mode == M_LSRK_FIRST || mode == M_LSRK) {
#pragma unroll
            for (int i = 0; i < N; ++i)
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    r1[i][v] = mode == M_LSRK ? a.rk_a * r1[i][v] + a.dt * dv[i][v] : a.dt * dv[i][v];
                    u[i][v] += a.rk_b * r1[i][v];
                }
            if (live) st_row<N * V>(a.R1 + row, &r1[0][0]);
        } else if (mode == M_RK4_1) {
            if (live) {
                st_row<N * V>(a.R1 + row, &u[0][0]);
                st_row<N * V>(a.R2 + row, &dv[0][0]);
            }
#pragma unroll
            for (int i = 0; i < N; ++i)
#pragma unroll
                for (int v = 0; v < V; ++v) u[i][v] += a.rk_c * dv[i][v];
        } else {
            real r2[N][V];
            ld_row<N * V>(a.R1 + row, &r1[0][0]);
            ld_row<N * V>(a.R2 + row, &r2[0][0]);
            const bool last = mode == M_RK4_4;
#pragma unroll
            for (int i = 0; i < N; ++i)
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    const real acc = last ? r2[i][v] + dv[i][v] : r2[i][v] + real(2) * dv[i][v];
                    u[i][v] = r1[i][v] + a.rk_c * (last ? acc : dv[i][v]);
                    r2[i][v] = acc;
                }
            if (live && !last) st_row<N * V>(a.R2 + row, &r2[0][0]);
        }
        if (live) st_row<N * V>(a.U + row, &u[0][0]);
#pragma unroll
        for (int i = 0; i < N; ++i) st(jr + i, u[i]);
        sync();
    }
}

// --------------------------------------------------------------------------
// Mortar faces of 2-D line-kernel batches, once per stage, after the line
// kernels have put every mortar side's trace and gradient flux part into its
// outbox rows.  Eight lanes per face: carry the traces across (T, P; see
// K_MORTAR), then form the common flux of the next stage on the mortar: both
// sides' own viscous normal fluxes are their gradient part plus the lifting of
// their jump, the lower side's carried by T; the lower side takes minus the
// projection of the common flux.  (The gradient + flux pair needs two mortar
// launches per stage, around the flux kernel.)  Latency-bound, some thousand
// faces per launch; with it an 8-candidate poll of degrees 3 to 0 runs its
// stages in line kernels, 1.80 -> 0.87 ms per step.
// --------------------------------------------------------------------------
struct MortarLineArgs {
    float *UF[5];                  // face states of the pass, per degree group
    const float *FV[5];            // gradient flux parts of the pass
    const float *FGEO[5];
    float *MFLUX[5];
    int64_t fp_real[5];
    const struct MortarFace *faces;
    int64_t n_faces;
    const float *mats;
    float gamma, mu, kq;
    int flux;
    RefState<float> ref;
};

}  // namespace frk
