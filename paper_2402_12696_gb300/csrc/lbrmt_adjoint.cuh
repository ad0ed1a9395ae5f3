// lbrmt_adjoint.cuh -- reverse (adjoint) kernels of one LBRMT step and the
// centroid loss, for FP32 or FP64 arithmetic with full-precision storage.
//
// The forward step n -> n+1 (Algorithm 1) maps
//   K2: xi^{n+1} = advect(xi^n, u^n) on S^n = {phi(xi^n) < 0} (Eqs. 3_1_refmap_adv,
//       3_1_eno), then the layered weighted least-squares extrapolation of the band
//       (Sec. 3.2) whose weights for layers 1-2 use the normal of phi(xi^n);
//   K3: F^(n) = div tau(xi^{n+1}) + blended solid acceleration + body force
//       (Eqs. 3_3_refmap_jacobian, 3_3_solid_stress, 3_6_global_stress,
//       3_6_collision_stress, 3_3_div_solid_stress), Delta rho^(n) (Eq. 2_3_drho);
//   K1: f^{n+1}(x + c_q) = BGK collision of f^n with f^eq,SFC(rho^n, u^n, Delta rho)
//       and the Guo term (Eqs. 2_2_bgk_force, 2_3_feq_sfc, 3_4_Fi), with halfway
//       bounce-back (Sec. 3.5); u^n = (sum c f^n + rho^{n-1} F^(n-1) / 2) / rho^n.
// The kernels below apply the transposed Jacobians in the reverse order
// (K1, K3, K2), with the branch decisions of the forward step (solid set,
// layers, windows, upwind directions, contact pairs) recomputed from the
// recorded state; the adjoint of the populations is that of the absolute f_q.
#pragma once

#include "lbrmt_kernels.cuh"

namespace lbrmt {

template <class R> __device__ __forceinline__ R rcos(R x);
template <> __device__ __forceinline__ float rcos<float>(float x) { return cosf(x); }
template <> __device__ __forceinline__ double rcos<double>(double x) { return cos(x); }

// dH/dphi of the smoothed Heaviside.
template <class R> __device__ __forceinline__ R dheaviside(R phi, R eps) {
    if (phi <= -eps || phi >= eps) return R(0);
    const R pi = R(3.14159265358979323846);
    return R(0.5) * (R(1) + rcos<R>(pi * phi / eps)) / eps;
}

// d phi / d eta at a tile node: phi = |p + eta| - R with p = l + off.
template <class R>
__device__ __forceinline__ void dphi_deta(R ex, R ey, int lx, int ly, const Frame &fr, R &gx, R &gy) {
    const R X = (R(lx) + R(fr.offx)) + ex, Y = (R(ly) + R(fr.offy)) + ey;
    const R r = rsqrt_<R>(X * X + Y * Y);
    if (r > R(0)) { gx = X / r; gy = Y / r; }
    else { gx = R(0); gy = R(0); }
}

// ---------------------------------------------------------------------------
// K1 reverse: one node per thread.
// ---------------------------------------------------------------------------
template <class R>
struct LbAdjArgs {
    const R *tape;     // rho^n, ux^n, uy^n, Fx^(n), Fy^(n) (5 planes)
    const R *fb_next;  // adjoint of f^{n+1} (9 planes)
    const R *cb_next;  // adjoint of the stored half-force rho^n F^(n) / 2 (2 planes)
    R *fb, *cb;        // adjoint of f^n, of the half-force read at step n
    R *Fb, *Db;        // adjoint of F^(n) (2 planes) and Delta rho^(n)
    double *bodyb;     // adjoint of the body force field, accumulated (2 planes) or null
    R *zero;           // cleared besides: the adjoint of xi^n, before the reverse K2 adds to it
    long long nzero;
};

template <class R>
__global__ void __launch_bounds__(256) lb_adjoint_kernel(SimParams sp, LbAdjArgs<R> a) {
    const long long P = sp.P;
    const int nx = sp.nx, ny = sp.ny;
    const R omega = pick<R>(sp.omega, sp.omega_f), kf = pick<R>(sp.kf, sp.kf_f);
    const R lid = pick<R>(sp.lid_u, sp.lid_u_f);
    for (long long k = blockIdx.x * 256ll + threadIdx.x; k < a.nzero; k += (long long)gridDim.x * 256) a.zero[k] = R(0);
    for (long long c = blockIdx.x * 256ll + threadIdx.x; c < P; c += (long long)gridDim.x * 256) {
        const int i = (int)(c % nx), j = (int)(c / nx);
        const R rho = a.tape[c], ux = a.tape[P + c], uy = a.tape[2 * P + c];
        const R Fx = a.tape[3 * P + c], Fy = a.tape[4 * P + c];
        // adjoint of the post-collision populations: pull of the push, bounce-back at walls
        R am[9];
        R rhob = R(0);
        am[0] = a.fb_next[c];
#pragma unroll
        for (int q = 1; q < 9; q++) {
            int di = i + cxq(q), dj = j + cyq(q);
            const bool ox = di < 0 || di >= nx, oy = dj < 0 || dj >= ny;
            if ((ox && sp.wall_x) || (oy && sp.wall_y)) {
                const R g = a.fb_next[oppq(q) * P + c];
                am[q] = g;
                const R uw = (oy && sp.wall_y && dj >= ny) ? lid : R(0);
                rhob -= R(6) * wq<R>(q) * R(cxq(q)) * uw * g;
            } else {
                if (ox) di = di < 0 ? di + nx : di - nx;
                if (oy) dj = dj < 0 ? dj + ny : dj - ny;
                am[q] = a.fb_next[q * P + (long long)dj * nx + di];
            }
        }
        const R cbx = a.cb_next[c], cby = a.cb_next[P + c];
        // f^eq_q = w rho A + Delta rho (delta_q0 - w), A = 1 + 3 cu + 4.5 cu^2 - 1.5 u^2, and the Guo term
        // rho w (3 (cF - uF) + 9 cu cF) enter through the adjoint's moments with the weights 36 w_q
        // = 16, 4, 1.  Opposite directions meet first: their adjoints are nearly c.j and cancel
        // exactly, where sums over all directions left the rounding of the large ones in the
        // small moments; the 36th at the end in parts (weights rounded at 1/9 scale every step's adjoint
        // by 1 + 7e-9).  (Errors against FP64 on
        // 256^2, 160 steps, 40 problems: ratio gradient 3.4e-6 -> 6.8e-7, body force field 7.3e-7 -> 4.3e-7.)
        const R s1 = am[1] + am[3], s2 = am[2] + am[4], s5 = am[5] + am[7], s6 = am[6] + am[8], sd = s5 + s6;
        const R d1 = am[1] - am[3], d2 = am[2] - am[4], d5 = am[5] - am[7], d6 = am[6] - am[8];
        const R T0 = R(16) * am[0] + (R(4) * (s1 + s2) + sd);
        const R mx = R(4) * d1 + (d5 - d6), my = R(4) * d2 + (d5 + d6);
        const R Qxx = R(4) * s1 + sd, Qyy = R(4) * s2 + sd, Qxy = s5 - s6;
        const R Qux = Qxx * ux + Qxy * uy, Quy = Qxy * ux + Qyy * uy;
        const R QFx = Qxx * Fx + Qxy * Fy, QFy = Qxy * Fx + Qyy * Fy;
        const R hx = omega * ux + kf * Fx, hy = omega * uy + kf * Fy;
        auto by36 = [](R v) { return third<R>(third<R>(R(0.25) * v)); };
        const R rs = (omega * (R(1) - R(1.5) * (ux * ux + uy * uy)) - R(3) * kf * (ux * Fx + uy * Fy)) * T0 +
                     (R(4.5) * omega * (ux * Qux + uy * Quy) + R(9) * kf * (ux * QFx + uy * QFy) + R(3) * (hx * mx + hy * my));
        rhob += by36(rs) + R(0.5) * (Fx * cbx + Fy * cby);
        const R r12 = rho * R(0.25);  // by36(3 v) = third(v / 4)
        const R ubx = third<R>(r12 * (omega * mx + R(3) * (omega * Qux + kf * QFx) - hx * T0));
        const R uby = third<R>(r12 * (omega * my + R(3) * (omega * Quy + kf * QFy) - hy * T0));
        const R Fbx = R(0.5) * rho * cbx + third<R>(r12 * kf * (mx + R(3) * Qux - ux * T0));
        const R Fby = R(0.5) * rho * cby + third<R>(r12 * kf * (my + R(3) * Quy - uy * T0));
        const R Dbv = omega * (am[0] - by36(T0));
        // u = (sum c f + half-force) / rho
        const R inv = R(1) / rho;
        const R jbx = ubx * inv, jby = uby * inv;
        rhob -= (ubx * ux + uby * uy) * inv;
        a.cb[c] = jbx;
        a.cb[P + c] = jby;
#pragma unroll
        for (int q = 0; q < 9; q++) a.fb[q * P + c] = (R(1) - omega) * am[q] + rhob + R(cxq(q)) * jbx + R(cyq(q)) * jby;
        a.Fb[c] = Fbx;
        a.Fb[P + c] = Fby;
        a.Db[c] = Dbv;
        if (a.bodyb) {
            a.bodyb[c] += (double)Fbx;
            a.bodyb[P + c] += (double)Fby;
        }
    }
}

// ---------------------------------------------------------------------------
// K3 reverse: one registered tile per CTA iteration.
// ---------------------------------------------------------------------------
template <class R>
struct ForceAdjArgs {
    const R *xi;            // xi^{n+1} tiles
    const Frame *frame;     // their frames
    const int *reg_count, *reg_solids, *reg_active, *reg_nactive;  // registry of step n
    const SolidDesc *solids;
    const R *Fb;            // adjoint of F^(n) (2 planes); null: zero (node terms only)
    const R *Db;            // adjoint of Delta rho^(n) (1 plane)
    R *xib;                 // adjoint of xi^{n+1}, accumulated (same tiles and frames)
    double *Gb, *Rb;        // per-solid adjoints of G and of rho_s / rho_f, accumulated
};

__host__ __device__ __forceinline__ int force_adj_smem_elems(int tx, int ty) {
    return 4 * KMAX * force_patch_n(tx, ty) + 9 * ((tx + 1) * ty + tx * (ty + 1)) + 3 * TILE_N;
}
__host__ __device__ __forceinline__ int force_adj_smem_max() {
    int m = 0;
    for (int tx = 16; tx <= 128; tx *= 2) m = force_adj_smem_elems(tx, TILE_N / tx) > m ? force_adj_smem_elems(tx, TILE_N / tx) : m;
    return m;
}

// Reverse of stress_from_grad: given the adjoint of (txx, txy, tyy), add the
// adjoint of (Axx, Axy, Ayx, Ayy).
template <class R>
__device__ __forceinline__ void stress_adjoint(R Axx, R Axy, R Ayx, R Ayy, R G, R tbxx, R tbxy, R tbyy, R &Abxx,
                                               R &Abxy, R &Abyx, R &Abyy) {
    const R dl = (Axx + Ayy) + (Axx * Ayy - Axy * Ayx);
    const R inv = R(1) / (R(1) + dl);
    const R Dxx = (Ayy - dl) * inv, Dxy = -Axy * inv, Dyx = -Ayx * inv, Dyy = (Axx - dl) * inv;
    const R Ebxx = G * (R(2) * tbxx - tbyy) / R(3), Ebyy = G * (R(2) * tbyy - tbxx) / R(3), Ebxy = G * tbxy;
    const R Dbxx = Ebxx * (R(2) + R(2) * Dxx) + Ebxy * Dyx;
    const R Dbxy = Ebxx * R(2) * Dxy + Ebxy * (R(1) + Dyy);
    const R Dbyx = Ebxy * (R(1) + Dxx) + Ebyy * R(2) * Dyx;
    const R Dbyy = Ebxy * Dxy + Ebyy * (R(2) + R(2) * Dyy);
    R dlb = -(Dbxx + Dbyy) * inv;
    const R invb = Dbxx * (Ayy - dl) - Dbxy * Axy - Dbyx * Ayx + Dbyy * (Axx - dl);
    dlb += -invb * inv * inv;
    Abyy += Dbxx * inv + dlb * (R(1) + Axx);
    Abxx += Dbyy * inv + dlb * (R(1) + Ayy);
    Abxy += -Dbxy * inv - dlb * Ayx;
    Abyx += -Dbyx * inv - dlb * Axy;
}

// Sum of v over the warp into *s (shared), one addition per warp.
__device__ __forceinline__ void warp_add_to(double *s, double v) {
    if (__ballot_sync(0xffffffffu, __double_as_longlong(v) != 0ll) == 0u) return;  // (an FP64 compare would cost as an addition)
    for (int d = 16; d > 0; d >>= 1) v += __shfl_down_sync(0xffffffffu, v, d);
    if ((threadIdx.x & 31) == 0) atomicAdd(s, v);
}

// One registered tile.  Each half-edge's adjoints (of one solid's edge derivatives and edge
// phi) go to shared memory, and each patch node gathers those of the half-edges whose
// stencil holds it; the solids' sums meet once per warp.
// Bound by latency: a tile or two per SM, in a chain of loads, edge terms and the gather.
// (Scattered from the half-edges with atomics -- compare-and-swap loops on shared floats, and
// on doubles with every thread of the tile at one address -- a disk of radius 39 took 55 us; gathered, 16;
// 256 disks of radius 16 on 2048^2: 300 us less a step.)
template <class R>
__device__ void force_adjoint_tile(const SimParams &sp, const ForceAdjArgs<R> &a, const int tile, ForceShared<R> &fs,
                                   double *sGb, double *sRb, double *sRc, R *dyn, bool node_only) {
    const int TX = sp.tx, TY = sp.ty, PX = TX + 2, PN = force_patch_n(TX, TY);
    const int NXE = (TX + 1) * TY, NE = NXE + TX * (TY + 1);
    R *sX = dyn, *sY = sX + KMAX * PN, *sP = sY + KMAX * PN, *bP = sP + KMAX * PN;
    R *eS = bP + KMAX * PN;  // [4][NE]: adjoint of the half-edge's solid stress, and of its sum of lambda
    R *eG = eS + 4 * NE;     // [5][NE]: of one solid's edge derivatives Xn, Xt, Yn, Yt and of its edge phi
    R *nF = eG + 5 * NE;     // [3 * TILE_N]: F_x, F_y, Delta rho adjoints of the tile nodes
    const R eps = pick<R>(sp.eps, sp.eps_f), eta = pick<R>(sp.eta, sp.eta_f);
    const int i0 = tile % sp.ntx * TX, j0 = tile / sp.ntx * TY;
    __syncthreads();  // the previous tile's shared state is no longer read
    if (threadIdx.x < 32) {  // slot = rank of the id, as the forward
        const int k = threadIdx.x, n = min(a.reg_count[tile], sp.kmax);
        const int id = k < n ? a.reg_solids[tile * KMAX + k] : 0x7fffffff;
        int rank = 0;
#pragma unroll
        for (int m = 0; m < KMAX; m++) rank += __shfl_sync(0xffffffffu, id, m) < id ? 1 : 0;
        if (k < n) {
            const SolidDesc &sd = a.solids[id];
            fs.ids[rank] = id;
            fs.sfr[rank] = a.frame[id];
            fs.sG[rank] = pick<R>(sd.G, sd.G_f);
            fs.sD[rank] = pick<R>(sd.drho, sd.drho_f);
            fs.sA[rank] = pick<R>(sd.accel, sd.accel_f);
            fs.srq[rank] = Rsq<R>(sd);
            fs.sT[rank] = sd.T;
            fs.soff[rank] = sd.off;
            sGb[rank] = 0.0;
            sRb[rank] = 0.0;
            // drho_s = rho_f (r - 1), a_s = -(1 - 1/r) g with r = rho_s / rho_f
            const double ir = sp.rho_f / sd.rho_s;
            sRc[rank] = sp.gravity * ir * ir;
        }
        if (k == 0) fs.nk = n;
    }
    {
        const int lt = threadIdx.x;
        const int i = i0 + (lt & (TX - 1)), j = j0 + (lt >> sp.lx);
        const bool in = i < sp.nx && j < sp.ny;
        const long long c = (long long)j * sp.nx + i;
        nF[lt] = (in && a.Fb) ? a.Fb[c] : R(0);
        nF[TILE_N + lt] = (in && a.Fb) ? a.Fb[sp.P + c] : R(0);
        nF[2 * TILE_N + lt] = in ? a.Db[c] : R(0);
    }
    __syncthreads();
    const int n = fs.nk;
    for (int ks = 0; ks < n; ks++) {
        const Frame fr = fs.sfr[ks];
        const int T = fs.sT[ks];
        const R *Xs = a.xi + fs.soff[ks];
        BoxWalk wk(PX);
        for (int p = threadIdx.x; p < PN; p += blockDim.x, wk.next()) {
            const int gx = i0 - 1 + wk.c, gy = j0 - 1 + wk.r;
            const int lx = sp.wall_x ? gx - fr.ox : wrapi(gx - fr.ox, sp.nx);
            const int ly = sp.wall_y ? gy - fr.oy : wrapi(gy - fr.oy, sp.ny);
            R X = nanv<R>(), Y = nanv<R>(), Pv = nanv<R>();
            if (in_box(fr, lx, ly)) {
                X = Xs[ly * T + lx];
                Y = Xs[T * T + ly * T + lx];
                if (X == X) Pv = phi_eta(X, Y, lx, ly, fr, fs.srq[ks]);
            }
            sX[ks * PN + p] = X; sY[ks * PN + p] = Y; sP[ks * PN + p] = Pv;
            bP[ks * PN + p] = R(0);
        }
    }
    __syncthreads();
    // Node terms: Delta rho = sum lam drho_s / max(1, L), A_y = sum lam a_s / max(1, L).
    {
        const int lt = threadIdx.x, p = ((lt >> sp.lx) + 1) * PX + (lt & (TX - 1)) + 1;
        const R Dbar = nF[2 * TILE_N + lt], Aybar = nF[TILE_N + lt];
        R L = 0, D = 0, Ay = 0;
        for (int ks = 0; ks < n; ks++) {
            const R ph = sP[ks * PN + p];
            if (!(ph == ph)) continue;
            const R lam = R(1) - heaviside<R>(ph, eps);
            L += lam; D += lam * fs.sD[ks]; Ay += lam * fs.sA[ks];
        }
        R Dr = Dbar, Ar = Aybar, Lb = R(0);
        if (L > R(1)) {
            Dr = Dbar / L; Ar = Aybar / L;
            Lb = -(Dbar * (D / L) + Aybar * (Ay / L)) / L;
        }
        for (int ks = 0; ks < n; ks++) {  // uniform over the CTA
            const R ph = sP[ks * PN + p];
            double rb = 0.0;
            if (ph == ph && (Dbar != R(0) || Aybar != R(0))) {
                const R lam = R(1) - heaviside<R>(ph, eps);
                bP[ks * PN + p] = -dheaviside<R>(ph, eps) * (Dr * fs.sD[ks] + Ar * fs.sA[ks] + Lb);
                if (lam != R(0)) rb = (double)lam * ((double)Dr * sp.rho_f - (double)Ar * sRc[ks]);
            }
            warp_add_to(&sRb[ks], rb);
        }
    }
    if (node_only) {
        __syncthreads();
        if (threadIdx.x < n) atomicAdd(&a.Rb[fs.ids[threadIdx.x]], sRb[threadIdx.x]);
        return;
    }
    const unsigned xdiv = 0xffffffffu / (unsigned)(TX + 1) + 1u;  // e / (TX + 1) = umulhi(e, xdiv)
    // The stencil of half-edge e: patch node p0 of its low side's first column (row), the
    // steps along and across it, and whether its normal is x.
    auto stencil = [&](int e, int &p0, int &al, int &ac) {
        const bool xe = e < NXE;
        const int f = e - NXE, ey = xe ? (int)__umulhi((unsigned)e, xdiv) : f >> sp.lx;
        p0 = ey * PX + (xe ? e - ey * (TX + 1) : f & (TX - 1));
        al = xe ? PX : 1;
        ac = xe ? 1 : PX;
        return xe;
    };
    // Solid ks on it: derivatives in x and y, edge phi; false where its stress does not enter.
    auto edge = [&](int ks, int p0, int al, int ac, bool xe, R &Axx, R &Axy, R &Ayx, R &Ayy, R &ph) {
        const R *P = sP + ks * PN + p0, *X = sX + ks * PN + p0, *Y = sY + ks * PN + p0;
        ph = R(0.5) * (P[al] + P[ac + al]);
        if (!(ph < eps)) return false;  // lambda = 0 and dlambda/dphi = 0: as the forward, no terms
        R Xn, Xt, Yn, Yt;
        edge_grad<R>(X[0], X[al], X[2 * al], X[ac], X[ac + al], X[ac + 2 * al], Xn, Xt);
        if (!(Xt == Xt)) return false;
        edge_grad<R>(Y[0], Y[al], Y[2 * al], Y[ac], Y[ac + al], Y[ac + 2 * al], Yn, Yt);
        Axx = xe ? Xn : Xt; Axy = xe ? Xt : Xn; Ayx = xe ? Yn : Yt; Ayy = xe ? Yt : Yn;
        return true;
    };
    if (n > 1) __syncthreads();  // the contact terms add to the node terms
    // Each half-edge's stress adjoint from the tile's nodes (F_x = d_x tau_xx + d_y tau_xy, F_y =
    // d_x tau_xy + d_y tau_yy), and through the blend; contact pairs.
    for (int e = threadIdx.x; e < NE; e += blockDim.x) {
        int p0, al, ac;
        const bool xe = stencil(e, p0, al, ac);
        R bxx = 0, bxy = 0, byy = 0;
        if (xe) {
            const int ey = (int)__umulhi((unsigned)e, xdiv), ex = e - ey * (TX + 1), r = ey * TX + ex;
            if (ex >= 1) { bxx += nF[r - 1]; bxy += nF[TILE_N + r - 1]; }
            if (ex < TX) { bxx -= nF[r]; bxy -= nF[TILE_N + r]; }
        } else {
            const int t = e - NXE;  // ey TX + ex
            if (t >= TX) { bxy += nF[t - TX]; byy += nF[TILE_N + t - TX]; }
            if (t < TX * TY) { bxy -= nF[t]; byy -= nF[TILE_N + t]; }
        }
        R Lb = R(0), Sbxx = bxx, Sbxy = bxy, Sbyy = byy;
        if (n > 1 && (bxx != R(0) || bxy != R(0) || byy != R(0))) {
            R Sxx = 0, Sxy = 0, Syy = 0, L = 0;
            unsigned okm = 0;
            for (int ks = 0; ks < n; ks++) {
                R Axx, Axy, Ayx, Ayy, ph, txx, txy, tyy;
                if (!edge(ks, p0, al, ac, xe, Axx, Axy, Ayx, Ayy, ph) ||
                    !stress_from_grad<R>(Axx, Axy, Ayx, Ayy, fs.sG[ks], txx, txy, tyy))
                    continue;
                const R lam = R(1) - heaviside<R>(ph, eps);
                okm |= 1u << ks;
                Sxx += lam * txx; Sxy += lam * txy; Syy += lam * tyy; L += lam;
            }
            if (L > R(1)) {
                Sbxx /= L; Sbxy /= L; Sbyy /= L;
                Lb = -(bxx * Sxx + bxy * Sxy + byy * Syy) / (L * L);
            }
            // contact pairs (Eq. 3_6_collision_stress), not normalised
            for (unsigned ms = okm; ms; ms &= ms - 1u) {
                const int ks = __ffs(ms) - 1;
                const R *Ps = sP + ks * PN + p0;
                const R phs = R(0.5) * (Ps[al] + Ps[ac + al]);
                for (unsigned mt = ms & (ms - 1u); mt; mt &= mt - 1u) {
                    const int kt = __ffs(mt) - 1;
                    const R *Pt = sP + kt * PN + p0;
                    const R pht = R(0.5) * (Pt[al] + Pt[ac + al]);
                    const R fsv = R(0.5) * (R(1) - phs / eps), ftv = R(0.5) * (R(1) - pht / eps);
                    const bool take_s = fsv < ftv;
                    const R fm = take_s ? fsv : ftv;
                    R gn, gt;
                    edge_grad<R>(Ps[0] - Pt[0], Ps[al] - Pt[al], Ps[2 * al] - Pt[2 * al], Ps[ac] - Pt[ac],
                                 Ps[ac + al] - Pt[ac + al], Ps[ac + 2 * al] - Pt[ac + 2 * al], gn, gt);
                    const R gxx = xe ? gn : gt, gyy = xe ? gt : gn;
                    const R nrm = rsqrt_<R>(gxx * gxx + gyy * gyy);
                    if (nrm == R(0)) continue;
                    const R nx_ = gxx / nrm, ny_ = gyy / nrm;
                    const R Gst = fs.sG[ks] + fs.sG[kt];
                    const R kk = -eta * fm * Gst;
                    const R kkb = bxx * (nx_ * nx_ - R(0.5)) + bxy * (nx_ * ny_) + byy * (ny_ * ny_ - R(0.5));
                    const R nbx = kk * (R(2) * bxx * nx_ + bxy * ny_), nby = kk * (bxy * nx_ + R(2) * byy * ny_);
                    const R gG = -eta * fm * kkb;
                    atomicAdd(&sGb[ks], (double)gG);
                    atomicAdd(&sGb[kt], (double)gG);
                    const R phw = eta * Gst * kkb / (R(2) * eps);  // f = (1 - phi / eps) / 2
                    R *const w = bP + (take_s ? ks : kt) * PN + p0;
                    atomicAdd(&w[al], R(0.5) * phw);
                    atomicAdd(&w[ac + al], R(0.5) * phw);
                    const R nd = nx_ * nbx + ny_ * nby;
                    const R gbx = (nbx - nx_ * nd) / nrm, gby = (nby - ny_ * nd) / nrm;
                    const R gbn = xe ? gbx : gby, gbt = (xe ? gby : gbx) * R(0.25);
                    for (int v = 0; v < 2; v++) {  // (gn, gt) = edge_grad(P_s - P_t)
                        const R sn = v == 0 ? gbn : -gbn, st = v == 0 ? gbt : -gbt;
                        R *const g = bP + (v == 0 ? ks : kt) * PN + p0;
                        atomicAdd(&g[ac + al], sn); atomicAdd(&g[al], -sn);
                        atomicAdd(&g[ac + 2 * al], st); atomicAdd(&g[2 * al], st);
                        atomicAdd(&g[ac], -st); atomicAdd(&g[0], -st);
                    }
                }
            }
        }
        eS[e] = Sbxx; eS[NE + e] = Sbxy; eS[2 * NE + e] = Sbyy; eS[3 * NE + e] = Lb;
    }
    for (int ks = 0; ks < n; ks++) {
        const R G = fs.sG[ks];
        double gb = 0.0;
        bool any = false;
        for (int e = threadIdx.x; e < NE; e += blockDim.x) {  // the half-edges of the loop above
            const R Sbxx = eS[e], Sbxy = eS[NE + e], Sbyy = eS[2 * NE + e], Lb = eS[3 * NE + e];
            R g[5] = {0, 0, 0, 0, 0}, Axx, Axy, Ayx, Ayy, ph, hxx, hxy, hyy;
            int p0, al, ac;
            const bool xe = stencil(e, p0, al, ac);
            if ((Sbxx != R(0) || Sbxy != R(0) || Sbyy != R(0)) && edge(ks, p0, al, ac, xe, Axx, Axy, Ayx, Ayy, ph) &&
                stress_from_grad<R>(Axx, Axy, Ayx, Ayy, R(1), hxx, hxy, hyy)) {  // stress per unit G
                const R lam = R(1) - heaviside<R>(ph, eps), tau = Sbxx * hxx + Sbxy * hxy + Sbyy * hyy;
                gb += (double)(lam * tau);
                R bxx = 0, bxy = 0, byx = 0, byy = 0;
                stress_adjoint<R>(Axx, Axy, Ayx, Ayy, G, lam * Sbxx, lam * Sbxy, lam * Sbyy, bxx, bxy, byx, byy);
                // of dn = b1 - a1 and dt = (b2 + a2 - b0 - a0) / 4 of both components
                g[0] = xe ? bxx : bxy; g[1] = R(0.25) * (xe ? bxy : bxx);
                g[2] = xe ? byx : byy; g[3] = R(0.25) * (xe ? byy : byx);
                g[4] = R(-0.5) * dheaviside<R>(ph, eps) * (G * tau + Lb);
                any = true;
            }
#pragma unroll
            for (int k = 0; k < 5; k++) eG[k * NE + e] = g[k];
        }
        warp_add_to(&sGb[ks], gb);
        any = __syncthreads_or(any);
        // Patch node (px, py) and the half-edges around it: x-edge (ex, ey) lies between the
        // patch columns ex and ex + 1, along the rows ey .. ey + 2; y-edges with x and y exchanged.
        const Frame fr = fs.sfr[ks];
        const int T = fs.sT[ks];
        R *Xb = a.xib + fs.soff[ks];
        BoxWalk wk(PX);
        for (int p = threadIdx.x; p < PN; p += blockDim.x, wk.next()) {
            const int px = wk.c, py = wk.r;
            const R X = sX[ks * PN + p], Y = sY[ks * PN + p];
            if (!(X == X)) continue;
            R gx = 0, gy = 0, gp = bP[ks * PN + p];
            if (any) {
#pragma unroll
                for (int dir = 0; dir < 2; dir++) {
                    const int pn = dir == 0 ? px : py, pt = dir == 0 ? py : px;      // across and along the edges
                    const int nn = dir == 0 ? TX + 1 : TY + 1, nt = dir == 0 ? TY : TX;  // their number
#pragma unroll
                    for (int side = 0; side < 2; side++) {  // the node on the low (0) or the high side of the edge
                        const int en = pn - side;
                        if (en < 0 || en >= nn) continue;
#pragma unroll
                        for (int k = 0; k < 3; k++) {  // its place along the edge
                            const int et = pt - k;
                            if (et < 0 || et >= nt) continue;
                            const R *q = eG + (dir == 0 ? et * (TX + 1) + en : NXE + en * TX + et);
                            if (k == 1) {
                                gx += side ? q[0] : -q[0];
                                gy += side ? q[2 * NE] : -q[2 * NE];
                                gp += q[4 * NE];
                            } else {
                                gx += k == 2 ? q[NE] : -q[NE];
                                gy += k == 2 ? q[3 * NE] : -q[3 * NE];
                            }
                        }
                    }
                }
            }
            // phi = phi_0(xi): push the level-set adjoint onto xi, and to the solid's adjoint tile
            const int gxg = i0 - 1 + px, gyg = j0 - 1 + py;
            const int lx = sp.wall_x ? gxg - fr.ox : wrapi(gxg - fr.ox, sp.nx);
            const int ly = sp.wall_y ? gyg - fr.oy : wrapi(gyg - fr.oy, sp.ny);
            if (gp != R(0)) {
                R dx_, dy_;
                dphi_deta<R>(X, Y, lx, ly, fr, dx_, dy_);
                gx += gp * dx_;
                gy += gp * dy_;
            }
            if (gx == R(0) && gy == R(0)) continue;
            atomicAdd(&Xb[ly * T + lx], gx);
            atomicAdd(&Xb[T * T + ly * T + lx], gy);
        }
        __syncthreads();  // eG is free again
    }
    if (threadIdx.x < n) {
        atomicAdd(&a.Gb[fs.ids[threadIdx.x]], sGb[threadIdx.x]);
        atomicAdd(&a.Rb[fs.ids[threadIdx.x]], sRb[threadIdx.x]);
    }
}

template <class R>
__global__ void __launch_bounds__(TILE_N) force_adjoint_kernel(SimParams sp, ForceAdjArgs<R> a, int node_only) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ ForceShared<R> fs;
    __shared__ double sGb[KMAX], sRb[KMAX], sRc[KMAX];
    const int nact = *a.reg_nactive;
    for (int it = blockIdx.x; it < nact; it += gridDim.x)
        force_adjoint_tile<R>(sp, a, a.reg_active[it], fs, sGb, sRb, sRc, reinterpret_cast<R *>(smem), node_only != 0);
}

// ---------------------------------------------------------------------------
// K2 reverse: a cluster of CTAs per solid.
// ---------------------------------------------------------------------------
template <class R>
struct RmtAdjArgs {
    const R *xi_in, *xi_out;            // xi^n and xi^{n+1} tiles
    const Frame *frame_in, *frame_out;  // their frames
    const R *tape;                      // rho^n, ux^n, uy^n (first 3 of 5 planes)
    R *xib_out;                         // adjoint of xi^{n+1}: complete on entry, passed down the layers
    R *xib_in;                          // adjoint of xi^n, accumulated
    R *fb, *cb;                         // adjoint of f^n and of the half-force of step n, accumulated
    const SolidDesc *solids;
    // workspace, per tile node: its layer (-1: none), and the strips' lists of targets
    signed char *labels;
    int *lists;
};

// Weight of valid node (dx, dy) relative to the target (0 if the node is not used).
template <class R>
__device__ __forceinline__ R adj_weight(const signed char *lab, int k, int l, int dx, int dy, bool use_n, R nhx,
                                        R nhy, R &dn) {
    const int L = lab[k];
    dn = R(0);
    if (!(L >= 0 && L < l)) return R(0);
    R wt = pow2neg<R>(abs(dx) + abs(dy));
    if (use_n) {
        dn = (R(-dx) * nhx + R(-dy) * nhy) * rinv_tab<R>(dx, dy);
        wt = dn > R(COS_TIE) ? dn * wt : R(0);
    }
    return wt;
}

// Reverse of one extrapolated target (tx, ty) of layer l with any window: pass its
// adjoint (xb, yb) to the nodes of its fit and, for the directional weights, return
// the adjoint of the unit normal.  One thread; only for the rare windows beyond 5x5.
template <class R>
__device__ __noinline__ void extrapolate_adjoint(const SimParams &sp, const signed char *lab, const R *X, const R *Y, R *Xb,
                                    int T, int tx, int ty, int l, bool use_n, R nhx, R nhy, R xb, R yb, R &nbx,
                                    R &nby) {
    nbx = R(0);
    nby = R(0);
    // the same window growth as the forward fit
    int nvalid = 0, n = 0, sx = 0, sy = 0, sxx = 0, syy = 0, sxy = 0;
    R a = 0, b = 0, c = 0, d = 0, e = 0, fw = 0;
    int rsel = -1;
    for (int r = 2; r <= sp.rmax && rsel < 0; r++) {
        for (int dy = -r; dy <= r; dy++)
            for (int dx = -r; dx <= r; dx++) {
                if (r > 2 && abs(dx) != r && abs(dy) != r) continue;  // only the new ring
                if (tx + dx < 0 || ty + dy < 0 || tx + dx >= T || ty + dy >= T) continue;
                const int k = (ty + dy) * T + tx + dx;
                const int L = lab[k];
                if (!(L >= 0 && L < l)) continue;
                nvalid++;
                R dn;
                const R wt = adj_weight<R>(lab, k, l, dx, dy, use_n, nhx, nhy, dn);
                if (!(wt > R(0))) continue;
                n++; sx += dx; sy += dy; sxx += dx * dx; syy += dy * dy; sxy += dx * dy;
                const R x = R(dx), y = R(dy), wx = wt * x, wy = wt * y;
                a += wx * x; b += wx * y; c += wx; d += wy * y; e += wy; fw += wt;
            }
        if (nvalid < 3 || n < 3) continue;
        const long long g1 = (long long)n * sxx - (long long)sx * sx;
        const long long g2 = (long long)n * syy - (long long)sy * sy;
        const long long g3 = (long long)n * sxy - (long long)sx * sy;
        if (g1 * g2 - g3 * g3 == 0) continue;
        const R det = a * (d * fw - e * e) - b * (b * fw - c * e) + c * (b * e - c * d);
        if (!(det != R(0))) continue;
        rsel = r;
    }
    if (rsel < 0) return;  // the forward flagged it and wrote NaN
    // full inverse of the symmetric normal matrix M = [[a b c],[b d e],[c e fw]]
    const R C11 = d * fw - e * e, C12 = c * e - b * fw, C13 = b * e - c * d;
    const R C22 = a * fw - c * c, C23 = b * c - a * e, C33 = a * d - b * b;
    const R det = a * C11 + b * C12 + c * C13;
    const R id = R(1) / det;
    const R g0 = C13 * id, g1v = C23 * id, g2 = C33 * id;  // M^-1 e3
    // fit coefficients (needed for the residuals of the weight derivatives)
    R cX[3] = {0, 0, 0}, cY[3] = {0, 0, 0}, xref = 0, yref = 0;
    if (use_n) {
        R bx0 = 0, bx1 = 0, bx2 = 0, by0 = 0, by1 = 0, by2 = 0;
        bool have = false;
        for (int dy = -rsel; dy <= rsel; dy++)
            for (int dx = -rsel; dx <= rsel; dx++) {
                if (tx + dx < 0 || ty + dy < 0 || tx + dx >= T || ty + dy >= T) continue;
                const int k = (ty + dy) * T + tx + dx;
                R dn;
                const R wt = adj_weight<R>(lab, k, l, dx, dy, use_n, nhx, nhy, dn);
                if (!(wt > R(0))) continue;
                if (!have) { xref = X[k]; yref = Y[k]; have = true; }
                const R Xv = X[k] - xref, Yv = Y[k] - yref;
                const R wx = wt * R(dx), wy = wt * R(dy);
                bx0 += wx * Xv; bx1 += wy * Xv; bx2 += wt * Xv;
                by0 += wx * Yv; by1 += wy * Yv; by2 += wt * Yv;
            }
        cX[0] = (C11 * bx0 + C12 * bx1 + C13 * bx2) * id;
        cX[1] = (C12 * bx0 + C22 * bx1 + C23 * bx2) * id;
        cX[2] = (C13 * bx0 + C23 * bx1 + C33 * bx2) * id;
        cY[0] = (C11 * by0 + C12 * by1 + C13 * by2) * id;
        cY[1] = (C12 * by0 + C22 * by1 + C23 * by2) * id;
        cY[2] = (C13 * by0 + C23 * by1 + C33 * by2) * id;
    }
    for (int dy = -rsel; dy <= rsel; dy++)
        for (int dx = -rsel; dx <= rsel; dx++) {
            if (tx + dx < 0 || ty + dy < 0 || tx + dx >= T || ty + dy >= T) continue;
            const int k = (ty + dy) * T + tx + dx;
            R dn;
            const R wt = adj_weight<R>(lab, k, l, dx, dy, use_n, nhx, nhy, dn);
            if (!(wt > R(0))) continue;
            const R gp = g0 * R(dx) + g1v * R(dy) + g2;  // (M^-1 e3) . (dx, dy, 1)
            const R al = wt * gp;
            atomicAdd(&Xb[k], al * xb);
            atomicAdd(&Xb[T * T + k], al * yb);
            if (use_n) {
                // d value / d w_k = gp * residual_k; w_k = 2^-(|dx|+|dy|) * dn
                const R rx = (X[k] - xref) - (cX[0] * R(dx) + cX[1] * R(dy) + cX[2]);
                const R ry = (Y[k] - yref) - (cY[0] * R(dx) + cY[1] * R(dy) + cY[2]);
                const R wb = gp * (xb * rx + yb * ry);
                const R dnb = wb * pow2neg<R>(abs(dx) + abs(dy)) * rinv_tab<R>(dx, dy);
                nbx += -R(dx) * dnb;
                nby += -R(dy) * dnb;
            }
        }
}

// A target's fit in reverse, as RMT_ADJ_LANES lanes hold it: everything that does not
// depend on its adjoint.
constexpr int RMT_ADJ_LANES = 8;
template <class R>
struct AdjPlan {
    static constexpr int NW = (25 + RMT_ADJ_LANES - 1) / RMT_ADJ_LANES;
    int e;       // lx | ly << 16; -1: no target
    bool plane;  // false: a window beyond 5x5 (extrapolate_adjoint)
    R al[NW];    // d value / d node for the lane's window nodes sub + j RMT_ADJ_LANES
    // layers 1 and 2, lanes 0-3: the adjoint (px, py) . (xb, yb) of phi^n at the lane's neighbour, d phi / d eta there
    R px, py, dx, dy;
};

// K2 reverse of solid s, its band spread over the nc CTAs of a cluster in strips of
// rows.  The layers of the forward step are formed anew (S from phi^n as bit masks, of
// the rows that the strip can be reached from) and listed.  Then, in reverse order, eight lanes to a target: its adjoint goes to the nodes of its fit by
// atomics at L2, one cluster barrier per layer; last the advection of the strip's nodes of S.
// Bound by that chain's latency: per layer a load, the atomics and the barrier (2 K cycles); the
// next layer's fits are planned before the barrier's wait.
// A disk of radius 39 on 256^2 (16 CTAs) takes, in cycles, S 5 K, the layers and lists 11 K,
// layers 11-3 27 K, layers 2-1 14 K, the advection 7 K: 120 -> 34 us against one CTA of 1024 threads
// with byte labels, a target per thread and a window walked three times.
template <class R>
__global__ void __launch_bounds__(RMT_ADJ_THREADS, 1) rmt_adjoint_kernel(SimParams sp, RmtAdjArgs<R> a) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int loff[24];  // a layer's targets: list[loff[l] .. loff[l + 1])
    __shared__ int fill[24];  // their number
    __shared__ int lut[32];
    __shared__ R rd[25], wd[25];  // 1 / |d| of the window's nodes, times 2^-(|dx|+|dy|)
    const int nc = cluster_size(), rank = cluster_rank(), s = (int)blockIdx.x / nc;
    const SolidDesc &sd = a.solids[s];
    const int NL = sp.n_layers, T = sd.T, TT = T * T, rw = mask_row_words(T), mw = mask_words(T, nc, NL);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = RMT_ADJ_THREADS / 32;
    const Frame fo = a.frame_out[s], fi = a.frame_in[s];
    const int2 oo = make_int2(fo.ox, fo.oy);
    const int shx = fo.ox - fi.ox, shy = fo.oy - fi.oy;
    const R *Xi = a.xi_in + sd.off, *Yi = Xi + TT, *Pi = Yi + TT;
    const R *Xo = a.xi_out + sd.off, *Yo = Xo + TT;
    R *XbO = a.xib_out + sd.off;
    R *XbI = a.xib_in + sd.off;
    const long long P = sp.P, node0 = sd.off / xi_planes<R>();
    signed char *lab = a.labels + node0;
    // the band's box and this CTA's rows of it (the forward recorded the box)
    const int x0 = fo.bx0, x1 = fo.bx1, y0 = fo.by0, y1 = fo.by1;
    if (x0 > x1 || y0 > y1) return;  // uniform over the cluster
    const Strips st = {y0, y1, 31 - __clz(nc), NL};
    const int yr0 = st.first(rank), yr1 = st.first(rank + 1);
    const int my0 = st.set_first(rank);
    const RowMask mS = {reinterpret_cast<unsigned *>(smem), rw, st.set_first(rank)};
    // layers of the strip and two halo rows and columns (NL + 1: none): node (x, y) at slab[(y - yr0 + 2) ls + x - x0 + 2]
    const int ls = x1 - x0 + 5, lh = yr1 - yr0 + 4;
    int *const slist = reinterpret_cast<int *>(mS.p + mw);  // the layers' targets, where they fit
    unsigned char *slab = reinterpret_cast<unsigned char *>(slist + RMT_ADJ_LIST), *srow = slab + ls * lh;
    if (tid < 24) loff[tid] = 0;
    if (tid < 24) fill[tid] = 0;
    if (tid < 32) lut[tid] = row_moments(tid);
    if (tid >= 32 && tid < 57) {
        const int dx = (tid - 32) % 5 - 2, dy = (tid - 32) / 5 - 2;
        rd[tid - 32] = rinv_tab<R>(dx, dy);
        wd[tid - 32] = pow2neg<R>(abs(dx) + abs(dy)) * rinv_tab<R>(dx, dy);
    }
    for (int k = tid; k < mw / 4; k += RMT_ADJ_THREADS) reinterpret_cast<int4 *>(smem)[k] = make_int4(0, 0, 0, 0);
    {  // labels for a fit beyond its 5x5 window (extrapolate_adjoint): this CTA's rows, free
        const int c0 = rank == 0 ? 0 : yr0 * T, c1 = rank == nc - 1 ? TT : yr1 * T;  // T: a multiple of 8
        for (int k = c0 + 8 * tid; k < c1; k += 8 * RMT_ADJ_THREADS) *reinterpret_cast<int2 *>(lab + k) = make_int2(-1, -1);
    }
    __syncthreads();
    const int wa = (x0 + 32) >> 5, wn = ((x1 + 32) >> 5) - wa + 1;
    const unsigned wdiv = wn > 1 ? 0xffffffffu / (unsigned)wn + 1u : 0u;  // k / wn = umulhi(k, wdiv) for k wn < 2^32
    {  // S: a warp per mask word, of the rows that the strip and its halo can be reached from
        const int r0 = max(yr0 - NL - 2, y0), n = (min(yr1 + NL + 1, y1) - r0 + 1) * wn;
        // the input box, within the domain
        const int ax = max(fi.bx0 - shx, sp.wall_x ? -oo.x : 0), ay = max(fi.by0 - shy, sp.wall_y ? -oo.y : 0);
        const int ex = min(min(fi.bx1 - shx, T - 1), sp.wall_x ? sp.nx - 1 - oo.x : T - 1);
        const int ey = min(min(fi.by1 - shy, T - 1), sp.wall_y ? sp.ny - 1 - oo.y : T - 1);
        for (int k0 = warp; k0 < n; k0 += 4 * nw) {
            R ph[4];
            int at[4];
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const int k = k0 + q * nw, row = wn > 1 ? (int)__umulhi((unsigned)k, wdiv) : k, w = wa + k - row * wn;
                const int ly = r0 + row, lx = 32 * w - 32 + lane;
                at[q] = k < n ? (ly - mS.y0) * rw + w : -1;  // uniform over the warp
                ph[q] = R(0);
                if (k < n && lx >= max(ax, 0) && lx <= ex && ly >= ay && ly <= ey) ph[q] = Pi[(ly + shy) * T + lx + shx];
            }
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const unsigned m = __ballot_sync(0xffffffffu, ph[q] < -R(PHI_TIE));
                if (lane == 0 && at[q] >= 0) mS.p[at[q]] = m;
            }
        }
    }
    __syncthreads();
    // The layer of each node of the strip and its halo, the number of 4-neighbour steps to S:
    // the steps along its row to the nearest set bit (from a window of the row's mask, 2 NL
    // + 1 bits), then the least over the rows around it, nearest first.
    const int hr0 = yr0 - 2 - NL;
    {
        BoxWalk wl(ls);
        for (int k = tid; k < ls * (lh + 2 * NL); k += RMT_ADJ_THREADS, wl.next()) {
            const int x = x0 - 2 + wl.c, y = hr0 + wl.r;
            int d = 64;
            if (x >= x0 && x <= x1 && y >= y0 && y <= y1) {
                const int sh = (x - NL + 64) & 31, wi = ((x - NL + 64) >> 5) - 1;  // bit 0 of the window: node x - NL
                const unsigned *r = mS.p + (y - mS.y0) * rw + wi;
                const unsigned a0 = r[0], a1 = wi + 1 < rw ? r[1] : 0u, lo = __funnelshift_r(a0, a1, sh);
                if (NL <= 15) {
                    d = min(__clz(__brev(lo >> NL)), __clz(lo << (31 - NL)));
                } else {
                    const unsigned hi = __funnelshift_r(a1, wi + 2 < rw ? r[2] : 0u, sh);
                    const unsigned long long m = ((unsigned long long)hi << 32) | lo;
                    d = min(__clzll(__brevll(m >> NL)), __clzll(m << (63 - NL)));
                }
            }
            srow[k] = (unsigned char)d;
        }
    }
    __syncthreads();
    {
        BoxWalk wl(ls);
        for (int k = tid; k < ls * lh; k += RMT_ADJ_THREADS, wl.next()) {
            const int x = x0 - 2 + wl.c, y = yr0 - 2 + wl.r;
            const unsigned char *r = srow + k + NL * ls;
            int l = NL + 1;
            if (x >= x0 && x <= x1 && y >= y0 && y <= y1) {
                l = min(l, (int)r[0]);
                for (int dy = 1; dy < l; dy++) l = min(l, dy + min((int)r[-dy * ls], (int)r[dy * ls]));
            }
            slab[k] = (unsigned char)l;
        }
    }
    __syncthreads();
    // The lists, a layer per warp (counters in shared memory would take an atomic per node on
    // as few addresses as there are layers).
    const int ns = (yr1 - yr0) * ls;  // the strip's rows, with their free halo columns
    const unsigned char *strip = slab + 2 * ls;
    const unsigned lsdiv = 0xffffffffu / (unsigned)ls + 1u;  // k / ls = umulhi(k, lsdiv) for k ls < 2^32
    for (int l = warp + 1; l <= NL; l += nw) {
        int c = 0;
        for (int k = lane; k < ns; k += 32) c += strip[k] == l ? 1 : 0;
        c = __reduce_add_sync(0xffffffffu, c);
        if (lane == 0) fill[l] = c;
    }
    __syncthreads();
    if (warp == 0) {  // ends of the layers
        int e = lane >= 1 && lane <= NL ? fill[lane] : 0;
        for (int d = 1; d < 32; d *= 2) {
            const int v = __shfl_up_sync(0xffffffffu, e, d);
            if (lane >= d) e += v;
        }
        if (lane >= 1 && lane <= NL) loff[lane + 1] = e;
    }
    __syncthreads();
    int *const list = loff[NL + 1] <= RMT_ADJ_LIST ? slist : a.lists + node0 + (long long)yr0 * T;
    for (int l = warp; l <= NL; l += nw) {
        int at = loff[max(l, 1)];
        for (int k0 = 0; k0 < ns; k0 += 128) {
            unsigned m[4];
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const int k = k0 + 32 * q + lane;
                m[q] = __ballot_sync(0xffffffffu, k < ns && strip[min(k, ns - 1)] == l);
            }
#pragma unroll
            for (int q = 0; q < 4; q++) {
                if ((m[q] >> lane) & 1u) {
                    const int k = k0 + 32 * q + lane, r = (int)__umulhi((unsigned)k, lsdiv), x = x0 - 2 + k - r * ls, y = yr0 + r;
                    lab[y * T + x] = (signed char)l;
                    if (l > 0) list[at + __popc(m[q] & ((1u << lane) - 1u))] = x | (y << 16);
                }
                at += __popc(m[q]);
            }
        }
    }
    __syncthreads();
    constexpr int L = RMT_ADJ_LANES, NW = AdjPlan<R>::NW, G = RMT_ADJ_THREADS / L;
    const int sub = lane % L;
    const unsigned gm = (0xffffffffu >> (32 - L)) << (lane & ~(L - 1));
    auto sum = [&](R v) {
#pragma unroll
        for (int d = L / 2; d > 0; d >>= 1) v += __shfl_xor_sync(gm, v, d);
        return v;
    };
    // layers 1 and 2: the normal of phi^n from central differences, as the forward
    auto normal = [&](int l, int lx, int ly, R &nhx, R &nhy, R &nn) {
        const int ix = lx + shx, iy = ly + shy, k0 = iy * T + ix;
        nhx = nhy = nn = R(0);
        if (l > 2 || !(ix > fi.bx0 && iy > fi.by0 && ix < fi.bx1 && iy < fi.by1)) return false;
        const R Xe = Xi[k0 + 1], Xw = Xi[k0 - 1], Xn = Xi[k0 + T], Xs = Xi[k0 - T];
        const R gx = (Pi[k0 + 1] - Pi[k0 - 1]) * R(0.5), gy = (Pi[k0 + T] - Pi[k0 - T]) * R(0.5);
        nn = rsqrt_<R>(gx * gx + gy * gy);
        nhx = gx / nn;
        nhy = gy / nn;
        return Xe == Xe && Xw == Xw && Xn == Xn && Xs == Xs && nn > R(0);
    };
    // the neighbour of lane sub (< 4) in the central differences
    auto nbr = [&](int sb, int &ox, int &oy) {
        ox = sb < 2 ? 1 - 2 * sb : 0;
        oy = sb < 2 ? 0 : 5 - 2 * sb;
    };
    auto make = [&](int l, int k) {  // uniform over the lanes of a target
        AdjPlan<R> p;
        p.e = -1;
        p.plane = true;
        p.px = p.py = p.dx = p.dy = R(0);
        if (k >= loff[l + 1]) return p;
        p.e = list[k];
        const int lx = p.e & 0xffff, ly = p.e >> 16, t = ly * T + lx;
        unsigned own = 0;  // the fit's nodes among the lane's, of earlier layers
#pragma unroll
        for (int j = 0; j < NW; j++) {
            const int w = sub + j * L;
            if (w < 25 && slab[(ly - yr0 + w / 5) * ls + lx - x0 + w % 5] < l) own |= 1u << w;
        }
        const unsigned bits = __reduce_or_sync(gm, own);
        R nhx, nhy, nn;
        const bool use_n = normal(l, lx, ly, nhx, nhy, nn);
        int c13, c23, c33;
        if (!use_n) {
            const int det = window_moments(lut, bits, c13, c23, c33);
            p.plane = det != 0;
            const R id = R(16) / whole<R>(det);  // the moments carry powers of 16: (c / 16^2) / (det / 16^3)
            const R g0 = whole<R>(c13) * id, g1 = whole<R>(c23) * id, g2 = whole<R>(c33) * id;  // M^-1 e3
#pragma unroll
            for (int j = 0; j < NW; j++) {
                const int w = sub + j * L, dx = w % 5 - 2, dy = w / 5 - 2;
                p.al[j] = w < 25 && ((bits >> w) & 1u) ? pow2neg<R>(abs(dx) + abs(dy)) * (g0 * R(dx) + g1 * R(dy) + g2) : R(0);
            }
            return p;
        }
        // directional weights 2^-(|dx|+|dy|) dn; the inverse of M = [[a b c],[b d e],[c e f]]
        R wt[NW], m[6] = {R(0), R(0), R(0), R(0), R(0), R(0)}, Xv[NW], Yv[NW];
        unsigned mine = 0;
        const R xref = Xo[t], yref = Yo[t];  // the fit's value at the target
#pragma unroll
        for (int j = 0; j < NW; j++) {
            const int w = sub + j * L, q = t + (w / 5 - 2) * T + w % 5 - 2;
            const bool on = w < 25 && ((bits >> w) & 1u);
            Xv[j] = on ? Xo[q] : xref;
            Yv[j] = on ? Yo[q] : yref;
            const R x = R(w % 5 - 2), y = R(w / 5 - 2);
            R v = R(0);
            if (on) {
                const R dn = (-x * nhx - y * nhy) * rd[w];
                if (dn > R(COS_TIE)) v = dn * pow2neg<R>(abs(w % 5 - 2) + abs(w / 5 - 2));
            }
            if (v > R(0)) mine |= 1u << w;
            wt[j] = v;
            const R wx = v * x, wy = v * y;
            m[0] += wx * x; m[1] += wx * y; m[2] += wx; m[3] += wy * y; m[4] += wy; m[5] += v;
        }
        const unsigned pos = __reduce_or_sync(gm, mine);  // nodes of positive weight
        p.plane = window_moments(lut, pos, c13, c23, c33) != 0;
#pragma unroll
        for (int j = 0; j < 6; j++) m[j] = sum(m[j]);
        const R C11 = m[3] * m[5] - m[4] * m[4], C12 = m[2] * m[4] - m[1] * m[5], C13 = m[1] * m[4] - m[2] * m[3];
        const R C22 = m[0] * m[5] - m[2] * m[2], C23 = m[1] * m[2] - m[0] * m[4], C33 = m[0] * m[3] - m[1] * m[1];
        const R det = m[0] * C11 + m[1] * C12 + m[2] * C13;
        p.plane = p.plane && det != R(0);
        const R id = R(1) / det, g0 = C13 * id, g1 = C23 * id, g2 = C33 * id;
        // d value / d w_k = (M^-1 e3 . (dx, dy, 1)) residual_k
        R b[6] = {R(0), R(0), R(0), R(0), R(0), R(0)}, nb[4] = {R(0), R(0), R(0), R(0)};
#pragma unroll
        for (int j = 0; j < NW; j++) {
            const int w = sub + j * L;
            const R x = R(w % 5 - 2), y = R(w / 5 - 2), wx = wt[j] * x, wy = wt[j] * y;
            p.al[j] = wt[j] * (g0 * x + g1 * y + g2);
            Xv[j] -= xref;
            Yv[j] -= yref;
            b[0] += wx * Xv[j]; b[1] += wy * Xv[j]; b[2] += wt[j] * Xv[j];
            b[3] += wx * Yv[j]; b[4] += wy * Yv[j]; b[5] += wt[j] * Yv[j];
        }
#pragma unroll
        for (int j = 0; j < 6; j++) b[j] = sum(b[j]);
        const R cX0 = (C11 * b[0] + C12 * b[1] + C13 * b[2]) * id, cX1 = (C12 * b[0] + C22 * b[1] + C23 * b[2]) * id;
        const R cX2 = (C13 * b[0] + C23 * b[1] + C33 * b[2]) * id;
        const R cY0 = (C11 * b[3] + C12 * b[4] + C13 * b[5]) * id, cY1 = (C12 * b[3] + C22 * b[4] + C23 * b[5]) * id;
        const R cY2 = (C13 * b[3] + C23 * b[4] + C33 * b[5]) * id;
#pragma unroll
        for (int j = 0; j < NW; j++) {
            const int w = sub + j * L;
            if (!(wt[j] > R(0))) continue;
            const R x = R(w % 5 - 2), y = R(w / 5 - 2), g = (g0 * x + g1 * y + g2) * wd[w];
            const R rx = (Xv[j] - (cX0 * x + cX1 * y + cX2)) * g, ry = (Yv[j] - (cY0 * x + cY1 * y + cY2)) * g;
            nb[0] -= x * rx; nb[1] -= y * rx; nb[2] -= x * ry; nb[3] -= y * ry;
        }
#pragma unroll
        for (int j = 0; j < 4; j++) nb[j] = sum(nb[j]);
        if (sub < 4) {
            // n = g / |g|, g = central differences of phi^n
            const R n1 = nhx * nb[0] + nhy * nb[1], n2 = nhx * nb[2] + nhy * nb[3];
            const R h = (sub & 1) ? R(-0.5) / nn : R(0.5) / nn;
            p.px = h * (sub < 2 ? nb[0] - nhx * n1 : nb[1] - nhy * n1);
            p.py = h * (sub < 2 ? nb[2] - nhx * n2 : nb[3] - nhy * n2);
            int ox, oy;
            nbr(sub, ox, oy);
            const int ix = lx + shx + ox, iy = ly + shy + oy, q = iy * T + ix;
            dphi_deta<R>(Xi[q], Yi[q], ix, iy, fi, p.dx, p.dy);
        }
        return p;
    };
    auto apply = [&](int l, const AdjPlan<R> &p) {
        if (p.e < 0) return;
        const int lx = p.e & 0xffff, ly = p.e >> 16, t = ly * T + lx;
        const R xb = __ldcg(XbO + t), yb = __ldcg(XbO + TT + t);
        if (xb == R(0) && yb == R(0)) return;
        if (!p.plane) {
            if (sub) return;
            R nhx, nhy, nn, nbx, nby;
            const bool use_n = normal(l, lx, ly, nhx, nhy, nn);
            extrapolate_adjoint<R>(sp, lab, Xo, Yo, XbO, T, lx, ly, l, use_n, nhx, nhy, xb, yb, nbx, nby);
            if (!use_n || (nbx == R(0) && nby == R(0))) return;
            const R nd = nhx * nbx + nhy * nby;
            for (int m = 0; m < 4; m++) {
                int ox, oy;
                nbr(m, ox, oy);
                const int ix = lx + shx + ox, iy = ly + shy + oy, q = iy * T + ix;
                const R pb = (m < 2 ? nbx - nhx * nd : nby - nhy * nd) * ((m & 1) ? R(-0.5) : R(0.5)) / nn;
                R dx, dy;
                dphi_deta<R>(Xi[q], Yi[q], ix, iy, fi, dx, dy);
                atomicAdd(&XbI[q], pb * dx);
                atomicAdd(&XbI[TT + q], pb * dy);
            }
            return;
        }
#pragma unroll
        for (int j = 0; j < NW; j++) {
            const int w = sub + j * L, q = t + (w / 5 - 2) * T + w % 5 - 2;
            if (p.al[j] == R(0)) continue;
            atomicAdd(&XbO[q], p.al[j] * xb);
            atomicAdd(&XbO[TT + q], p.al[j] * yb);
        }
        const R pb = p.px * xb + p.py * yb;
        if (pb != R(0)) {
            int ox, oy;
            nbr(sub, ox, oy);
            const int q = (ly + shy + oy) * T + lx + shx + ox;
            atomicAdd(&XbI[q], pb * p.dx);
            atomicAdd(&XbI[TT + q], pb * p.dy);
        }
    };
    // An advected node: eta^{n+1} = eta - (u - dd) - u d_x eta - v d_y eta (one-sided, upwind).
    struct Adv {
        int t, kk;  // output and input tile node; t < 0: none
        long long c;
        R rho, u, v, dXdx, dYdx, dXdy, dYdy;
    };
    const int nadv = (x1 - x0 + 1) * (yr1 - yr0);
    BoxWalk wk(x1 - x0 + 1);
    auto adv_load = [&](int k) {  // wk stands at node k
        Adv n;
        const int lx = x0 + wk.c, ly = yr0 + wk.r;
        n.t = -1;
        if (k >= nadv || !mS.bit(lx, ly)) return n;
        const int ix = lx + shx, iy = ly + shy, kk = iy * T + ix;
        n.kk = kk;
        n.c = (long long)wrapi(oo.y + ly, sp.ny) * sp.nx + wrapi(oo.x + lx, sp.nx);
        n.rho = a.tape[n.c];
        n.u = a.tape[P + n.c];
        n.v = a.tape[2 * P + n.c];
        const int sx = (n.u >= R(0)) ? -1 : 1, sy = (n.v >= R(0)) ? -1 : 1;
        const int x2 = ix + 2 * sx, y2 = iy + 2 * sy;
        if (x2 < fi.bx0 || x2 > fi.bx1 || y2 < fi.by0 || y2 > fi.by1) return n;  // the forward flagged it
        n.t = ly * T + lx;
        const int k1 = kk + sx, k2 = kk + 2 * sx, k3 = kk + sy * T, k4 = kk + 2 * sy * T;
        const R hx = R(-sx) * R(0.5), hy = R(-sy) * R(0.5), ex = Xi[kk], ey = Yi[kk];
        n.dXdx = hx * (R(3) * ex - R(4) * Xi[k1] + Xi[k2]);
        n.dYdx = hx * (R(3) * ey - R(4) * Yi[k1] + Yi[k2]);
        n.dXdy = hy * (R(3) * ex - R(4) * Xi[k3] + Xi[k4]);
        n.dYdy = hy * (R(3) * ey - R(4) * Yi[k3] + Yi[k4]);
        return n;
    };
    auto adv_apply = [&](const Adv &n) {
        if (n.t < 0) return;
        const R Xb = __ldcg(XbO + n.t), Yb = __ldcg(XbO + TT + n.t), u = n.u, v = n.v;
        if (Xb == R(0) && Yb == R(0)) return;
        const int sx = (u >= R(0)) ? -1 : 1, sy = (v >= R(0)) ? -1 : 1;
        const int kk = n.kk, k1 = kk + sx, k2 = kk + 2 * sx, k3 = kk + sy * T, k4 = kk + 2 * sy * T;
        const R hx = R(-sx) * R(0.5), hy = R(-sy) * R(0.5);
        const R c0 = R(1) - R(3) * (u * hx + v * hy);
        atomicAdd(&XbI[kk], Xb * c0); atomicAdd(&XbI[TT + kk], Yb * c0);
        atomicAdd(&XbI[k1], Xb * R(4) * u * hx); atomicAdd(&XbI[TT + k1], Yb * R(4) * u * hx);
        atomicAdd(&XbI[k2], -Xb * u * hx); atomicAdd(&XbI[TT + k2], -Yb * u * hx);
        atomicAdd(&XbI[k3], Xb * R(4) * v * hy); atomicAdd(&XbI[TT + k3], Yb * R(4) * v * hy);
        atomicAdd(&XbI[k4], -Xb * v * hy); atomicAdd(&XbI[TT + k4], -Yb * v * hy);
        const R ub = -Xb * (R(1) + n.dXdx) - Yb * n.dYdx;
        const R vb = -Xb * n.dXdy - Yb * (R(1) + n.dYdy);
        // u = (sum c f + half-force) / rho
        const R inv = R(1) / n.rho;
#pragma unroll
        for (int q = 0; q < 9; q++)
            atomicAdd(&a.fb[q * P + n.c], ((R(cxq(q)) - u) * ub + (R(cyq(q)) - v) * vb) * inv);
        atomicAdd(&a.cb[n.c], ub * inv);
        atomicAdd(&a.cb[P + n.c], vb * inv);
    };
    // One layer after the other, G targets at a time; the next ones' plan is made between
    // the arrival at a layer's barrier and the wait (the first barrier: the labels).  One
    // place for each of the pieces: a launch runs through its code but once, and every line of it
    // is fetched anew.
    AdjPlan<R> p;
    p.e = -1;
    int l = NL + 1, k = 0, rounds = 1;  // rounds of the layer left
    while (true) {
        apply(l, p);
        const bool last = --rounds == 0;
        if (last) {
            cluster_arrive();
            if (--l == 0) break;
            k = loff[l] + tid / L;
            rounds = max((loff[l + 1] - loff[l] + G - 1) / G, 1);
        } else {
            k += G;
        }
        p = make(l, k);
        if (last) cluster_wait();
    }
    // advected nodes
    for (int i = tid;; i += RMT_ADJ_THREADS, wk.next()) {
        const Adv n = adv_load(i);
        if (i == tid) cluster_wait();  // layer 1's
        if (i >= nadv) break;
        adv_apply(n);
    }
}

// ---------------------------------------------------------------------------
// Centroid c_s = sum lambda x / sum lambda (lambda = 1 - H(phi), domain nodes
// of the solid's tile) and the adjoint of xi for a given dL/dc_s.
// ---------------------------------------------------------------------------
template <class R>
__global__ void centroid_seed_kernel(SimParams sp, const R *xi, const Frame *frames, const SolidDesc *solids,
                                     const double *dLdc, R *xib) {
    __shared__ double red[32 * 3];
    __shared__ double tot[3];
    const int s = blockIdx.x;
    const SolidDesc sd = solids[s];
    const Frame fr = frames[s];
    const Rsq<R> rq(sd);
    const int T = sd.T, TT = T * T;
    const R eps = pick<R>(sp.eps, sp.eps_f);
    const R *X = xi + sd.off, *Y = X + TT;
    double st[3] = {0, 0, 0};
    for (int t = threadIdx.x; t < TT; t += blockDim.x) {
        const int lx = t % T, ly = t / T;
        if (!in_box(fr, lx, ly) || !domain_cell(sp, fr.ox + lx, fr.oy + ly)) continue;
        if (!(X[t] == X[t])) continue;
        const R phi = phi_eta(X[t], Y[t], lx, ly, fr, rq);
        if (!(phi < eps)) continue;
        const double lam = 1.0 - (double)heaviside<R>(phi, eps);
        st[0] += lam; st[1] += lam * (fr.ox + lx); st[2] += lam * (fr.oy + ly);
    }
    block_sum<double, 3>(st, red);
    if (threadIdx.x == 0) { tot[0] = st[0]; tot[1] = st[1]; tot[2] = st[2]; }
    __syncthreads();
    const double lsum = tot[0];
    if (lsum <= 0.0) return;
    const double cx = tot[1] / lsum, cy = tot[2] / lsum;
    const double gx = dLdc[2 * s], gy = dLdc[2 * s + 1];
    R *Xb = xib + sd.off;
    for (int t = threadIdx.x; t < TT; t += blockDim.x) {
        const int lx = t % T, ly = t / T;
        if (!in_box(fr, lx, ly) || !domain_cell(sp, fr.ox + lx, fr.oy + ly)) continue;
        if (!(X[t] == X[t])) continue;
        const R phi = phi_eta(X[t], Y[t], lx, ly, fr, rq);
        if (!(phi < eps) || phi <= -eps) continue;  // dH/dphi = 0 inside
        const R lamb = R((gx * (fr.ox + lx - cx) + gy * (fr.oy + ly - cy)) / lsum);
        const R phb = -dheaviside<R>(phi, eps) * lamb;
        R dx_, dy_;
        dphi_deta<R>(X[t], Y[t], lx, ly, fr, dx_, dy_);
        Xb[t] += phb * dx_;
        Xb[TT + t] += phb * dy_;
    }
}

}  // namespace lbrmt
