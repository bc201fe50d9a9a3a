// Register-streaming adjoint step (the transpose of the forward step; the algebra is in bte_adjoint.cu)
// for 2-D and 3-D grids of any shape with at least kRows rows, any storage, any wall; included by the
// instantiation units bte_adjoint_stream_<storage>.cu.
//
// A thread owns two neighbouring cells of a row and kRows rows of one slice, and loops over a part of one
// band's directions, reading e^n and lambda^{n+1} straight from global memory.  In natural (not stream)
// order the transpose needs no sign in its stencil: with the differences a = u_p - u_{p-1}, b = u_{p+1} -
// u_p of the face whose upwind cell is p, G_a and G_b the partials of the symmetric limiter, and
//   theta_p = |nu|/2 (lambda_{p+1} - lambda_p)   for nu > 0,   |nu|/2 (lambda_p - lambda_{p-1})   for nu < 0,
//   U_p = theta_p G_a, V_p = theta_p G_b,
// cell p collects  2 sign(nu) theta_p + U_p - V_p - U_{p+1} + V_{p-1}  along each axis: the sign only picks
// which lambda differences are read.  A face is taken when its three values lie in the domain or wrap;
// those that read a ghost value have weight 0 here and belong to k_adj_walls, so positions outside the
// domain may read any cell and there are no wall rules and no barriers.  Faces are shared along the rows
// (1 + 2 / kRows a cell); 2 x faces and 3 z faces a cell are evaluated, two at a time (packed FP32).
//
// 16-bit codes are worked on as e / s_k = h + rho (the partials are of degree 0); the references of every
// cell a thread reads, and mu^{n+1} and C_k T_L^n of its own, do not depend on the direction: they stay in
// shared memory, in slots no other thread reads.
//
// What bounds it: issue and the FMA pipe (58 and 57 % busy, 16 warps an SM), 166 thread instructions an update
// in 3-D, 91 in 2-D.  A launch, against the tiled step (k_adj_tiled, whose blocks stage a box, wait, and
// exchange z faces between barriers): 96^3, 32 x 96, FP16 40.6 -> 19.2 ms (floor at the copy rate 4.0); 128^2,
// 20 x 64, FP32 107 -> 92 us (37).
#pragma once

#include "bte_adjoint.h"
#include "bte_tiled_kernel.cuh"

namespace bte {
namespace adjs {

using tiled::St;
constexpr int kThreads = 256, kRows = 4;

// the arguments of the adjoint launch beside the step's
struct AdjStreamArgs {
    const float *lam_in;
    float *lam_out;
    const float *mu_in;
    float *P;   // [nb nchunk][ncell] sums of lambda^n over a part's directions
    float *Ps;  // [nb nchunk blocks][2] sum lambda^{n+1} (C_k T_L/W - e), sum w_d mu^{n+1} e
    const float *w;
    int nchunk, nys, G, blocks;  // parts of a band's directions; strips a slice, pairs a row; blocks a part
};

// shared slots (float2 a thread): mu, C_k T_L, and for 16-bit storage the references of the rows y0-2 ..
// y0+kRows+1, of the pairs left and right of each row and of the four slices around it
template <int S, int DIM> constexpr int slots() {
    return 2 * kRows + (St<S>::kRef ? (kRows + 4) + 2 * kRows + (DIM == 3 ? 4 * kRows : 0) : 0);
}

__device__ __forceinline__ float2 f2(float x) { return make_float2(x, x); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, f2(-1.f), a); }

// A pair of cells: at p and p + o1 - o0 in general, 8 (4) bytes where rows are even (VEC).
template <bool VEC> __device__ __forceinline__ float2 ld2(const float *p, int o0, int o1) {
    if constexpr (VEC) return __ldg(reinterpret_cast<const float2 *>(p + o0));
    else return make_float2(__ldg(p + o0), __ldg(p + o1));
}
template <int S, bool VEC> __device__ __forceinline__ float2 lde(const typename St<S>::T *p, int o0, int o1, const float2 *rho) {
    if constexpr (!St<S>::kRef) {
        return ld2<VEC>(p, o0, o1);
    } else {
        uint32_t lo, hi;
        if constexpr (VEC) {
            const uint32_t q = __ldg(reinterpret_cast<const uint32_t *>(p + o0));
            lo = q & 0xffffu;
            hi = q >> 16;
        } else {
            lo = __ldg(reinterpret_cast<const unsigned short *>(p + o0));
            hi = __ldg(reinterpret_cast<const unsigned short *>(p + o1));
        }
        return __fadd2_rn(*rho, make_float2(St<S>::val(lo), St<S>::val(hi)));
    }
}

// U = th dL/da and V = th dL/db at the differences a, b (sa, sb: their squares plus half of kTiny)
constexpr float kTiny = 1e-30f;
__device__ __forceinline__ float2 square(float2 a) { return __ffma2_rn(a, a, f2(0.5f * kTiny)); }
template <int LIM>
__device__ __forceinline__ void grads(float2 a, float2 sa, float2 b, float2 sb, float2 th, bool up, float2 &U, float2 &V) {
    if constexpr (LIM == kLimFirst) {
        U = V = f2(0.f);
    } else if constexpr (LIM == kLimMinmod) {
        const float2 ab = __fmul2_rn(a, b);
        // equal slopes: the downwind one counts
        const bool pa0 = up ? fabsf(a.x) < fabsf(b.x) : fabsf(a.x) <= fabsf(b.x);
        const bool pa1 = up ? fabsf(a.y) < fabsf(b.y) : fabsf(a.y) <= fabsf(b.y);
        const float t0 = ab.x > 0.f ? th.x : 0.f, t1 = ab.y > 0.f ? th.y : 0.f;
        U = make_float2(pa0 ? t0 : 0.f, pa1 ? t1 : 0.f);
        V = make_float2(pa0 ? 0.f : t0, pa1 ? 0.f : t1);
    } else {
        // L = ab(a+b)/(a^2+b^2): dL/da = b^2 (2ab + b^2 - a^2)/(a^2+b^2)^2, symmetric in b
        const float2 ab = __fmul2_rn(a, b), den = __fadd2_rn(sa, sb);
        const float2 rq = make_float2(tiled::rcp_approx(den.x), tiled::rcp_approx(den.y));
        const float2 df = sub2(sb, sa);
        const float2 u = __fmul2_rn(__ffma2_rn(f2(2.f), ab, df), rq), v = __fmul2_rn(sub2(__fadd2_rn(ab, ab), df), rq);
        const float2 t = make_float2(ab.x > kTiny ? th.x : 0.f, ab.y > kTiny ? th.y : 0.f);
        // (sb / den) (t u): the bounded factors first, so that 1/den cannot overflow a product
        U = __fmul2_rn(__fmul2_rn(sb, rq), __fmul2_rn(t, u));
        V = __fmul2_rn(__fmul2_rn(sa, rq), __fmul2_rn(t, v));
    }
}

// position pos along an axis of n cells: wrapped on a periodic axis, else the nearest cell
__device__ __forceinline__ int clip(int pos, int n, bool per) {
    if (per) return pos < 0 ? pos + n : (pos >= n ? pos - n : pos);
    return min(max(pos, 0), n - 1);
}
// weight of the face with upwind cell pos
__device__ __forceinline__ float face_on(int pos, int n, bool per) { return per || (pos >= 1 && pos + 1 < n) ? 1.f : 0.f; }

template <int S, int LIM, int DIM, bool VEC>
__global__ void __launch_bounds__(kThreads, 2) k_adj_stream(const __grid_constant__ StepArgs a,
                                                            const __grid_constant__ AdjStreamArgs g) {
    using T = typename St<S>::T;
    constexpr bool REF = St<S>::kRef;
    extern __shared__ float2 shm[];
    __shared__ float red[2][kThreads / 32];
    float2 *mus = shm + threadIdx.x, *ckt = mus + kRows * kThreads;
    float2 *ry = ckt + kRows * kThreads, *rx = ry + (kRows + 4) * kThreads, *rz = rx + 2 * kRows * kThreads;
    const int row = blockIdx.x / g.blocks, bi = blockIdx.x - row * g.blocks;
    const int k = row / g.nchunk, c = row - k * g.nchunk;
    const int d0 = (int)((long long)c * a.nd / g.nchunk), d1 = (int)((long long)(c + 1) * a.nd / g.nchunk);
    const int nx = a.n[0], ny = a.n[1], nz = DIM == 3 ? a.n[2] : 1;
    const int tid = bi * kThreads + (int)threadIdx.x;
    const int strip = tid / g.G, pr = tid - strip * g.G;
    const bool active = strip < g.nys * nz;
    const BandConst b = a.band[k];
    float2 s1 = f2(0.f), s2 = f2(0.f);
    if (active) {
        // strip index: slices first, so that a block's strips share rows with their neighbours
        const int z = strip / g.nys, ys = strip - z * g.nys;
        const int x0 = min(2 * pr, nx - 2), y0 = min(ys * kRows, ny - kRows);
        // cells a shifted pair or strip shares with its neighbour count once in the scalar sums
        const float2 ownx = make_float2(2 * pr == x0 ? 1.f : 0.f, 1.f);
        const int jown = ys * kRows - y0;
        const bool px = a.bc[0] == kBcPeriodic, py = a.bc[2] == kBcPeriodic, pz = DIM == 3 && a.bc[4] == kBcPeriodic;
        const int nxy = nx * ny, idx0 = (z * ny + y0) * nx + x0;
        // x: cells x0-2, x0-1, x0+2, x0+3 (even rows: where the pairs start)
        const int l0 = VEC && !px && x0 < 2 ? 0 : clip(x0 - 2, nx, px) - x0, l1 = clip(x0 - 1, nx, px) - x0;
        const int h0 = VEC && !px && x0 + 2 >= nx ? 0 : clip(x0 + 2, nx, px) - x0, h1 = clip(x0 + 3, nx, px) - x0;
        const float2 mxA = make_float2(face_on(x0 - 1, nx, px), face_on(x0, nx, px));
        const float2 mxB = make_float2(face_on(x0 + 1, nx, px), face_on(x0 + 2, nx, px));
        // y: rows -2, -1, kRows, kRows + 1 of the strip
        const int ym2 = (clip(y0 - 2, ny, py) - y0) * nx, ym1 = (clip(y0 - 1, ny, py) - y0) * nx;
        const int yp0 = (clip(y0 + kRows, ny, py) - y0) * nx, yp1 = (clip(y0 + kRows + 1, ny, py) - y0) * nx;
        const float myA = face_on(y0 - 1, ny, py), my0 = face_on(y0, ny, py);
        const float my1 = face_on(y0 + kRows - 1, ny, py), myB = face_on(y0 + kRows, ny, py);
        int zm2 = 0, zm1 = 0, zp1 = 0, zp2 = 0;
        float mz0 = 0.f, mz1 = 0.f, mz2 = 0.f;
        if constexpr (DIM == 3) {
            zm2 = (clip(z - 2, nz, pz) - z) * nxy;
            zm1 = (clip(z - 1, nz, pz) - z) * nxy;
            zp1 = (clip(z + 1, nz, pz) - z) * nxy;
            zp2 = (clip(z + 2, nz, pz) - z) * nxy;
            mz0 = face_on(z - 1, nz, pz);
            mz1 = face_on(z, nz, pz);
            mz2 = face_on(z + 1, nz, pz);
        }
        #pragma unroll
        for (int j = 0; j < kRows; ++j) {
            const int i = idx0 + j * nx;
            mus[j * kThreads] = ld2<VEC>(g.mu_in + i, 0, 1);
            ckt[j * kThreads] = __fmul2_rn(f2(b.ck), ld2<VEC>(a.TL + i, 0, 1));
            if constexpr (REF) {
                auto ref = [&](int o0, int o1) { return __fmul2_rn(f2(a.invTs), ld2<VEC>(a.R + i, o0, o1)); };
                ry[(j + 2) * kThreads] = ref(0, 1);
                rx[(2 * j) * kThreads] = ref(l0, l1);
                rx[(2 * j + 1) * kThreads] = ref(h0, h1);
                if constexpr (DIM == 3) {
                    rz[(4 * j) * kThreads] = ref(zm2, zm2 + 1);
                    rz[(4 * j + 1) * kThreads] = ref(zm1, zm1 + 1);
                    rz[(4 * j + 2) * kThreads] = ref(zp1, zp1 + 1);
                    rz[(4 * j + 3) * kThreads] = ref(zp2, zp2 + 1);
                }
            }
        }
        if constexpr (REF) {
            const int yo[4] = {ym2, ym1, yp0, yp1};
            #pragma unroll
            for (int m = 0; m < 4; ++m)
                ry[(m < 2 ? m : kRows + m) * kThreads] = __fmul2_rn(f2(a.invTs), ld2<VEC>(a.R + idx0, yo[m], yo[m] + 1));
        }
        float2 acc[kRows];
        #pragma unroll
        for (int j = 0; j < kRows; ++j) acc[j] = f2(0.f);
        const float diag = 1.f - b.dtinv, sc = REF ? b.scale : 1.f;
        for (int d = d0; d < d1; ++d) {
            const int plane = k * a.nd + d;
            const long long base = (long long)plane * a.ncell + idx0;
            const T *e = static_cast<const T *>(a.e_in) + base;
            const float *lam = g.lam_in + base;
            float *out = g.lam_out + base;
            const float *nu = a.nu + 3 * (long long)plane;
            const float nux = __ldg(nu), nuy = __ldg(nu + 1), nuz = DIM == 3 ? __ldg(nu + 2) : 0.f;
            const bool ux = nux > 0.f, uy = nuy > 0.f, uz = nuz > 0.f;
            const float hx = 0.5f * fabsf(nux), hy = 0.5f * fabsf(nuy), hz = 0.5f * fabsf(nuz);
            const float2 hA = __fmul2_rn(f2(hx), mxA), hB = __fmul2_rn(f2(hx), mxB);
            const float sx = ux ? 2.f : -2.f, sy = uy ? 2.f : -2.f, sz = uz ? 2.f : -2.f;
            const float wmD = __ldg(a.wmom + plane) * a.invD;
            if (d + 1 < d1) {  // the same cells of the next direction, towards L2
                #pragma unroll
                for (int j = 0; j < kRows; ++j) {
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(e + a.ncell + j * nx));
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(lam + a.ncell + j * nx));
                }
            }
            // y: lambda rows q_r = lambda_r (nu > 0) or lambda_{r-1}, r = -1 .. kRows + 1, so that
            // theta_p = hy (q_{p+1} - q_p)
            const float *lq = lam + (uy ? 0 : -nx);
            auto ldq = [&](int r) {
                if (r == -1) return ld2<VEC>(lam, uy ? ym1 : ym2, (uy ? ym1 : ym2) + 1);
                if (r == 0) return ld2<VEC>(lam, uy ? 0 : ym1, (uy ? 0 : ym1) + 1);
                if (r == kRows) return ld2<VEC>(lam, uy ? yp0 : (kRows - 1) * nx, (uy ? yp0 : (kRows - 1) * nx) + 1);
                if (r == kRows + 1) return ld2<VEC>(lam, uy ? yp1 : yp0, (uy ? yp1 : yp0) + 1);
                return ld2<VEC>(lq, r * nx, r * nx + 1);
            };
            auto ldrow = [&](int r) {
                const int o = r == -2 ? ym2 : (r == -1 ? ym1 : (r == kRows ? yp0 : (r == kRows + 1 ? yp1 : r * nx)));
                return lde<S, VEC>(e, o, o + 1, ry + (r + 2) * kThreads);
            };
            float2 w = ldrow(0), wn = ldrow(1);
            // differences and squares of the running face; V of the face before, theta, U, V of this one
            float2 dn, sn, qn, Vp, th, U, V;
            {
                const float2 um1 = ldrow(-1);
                const float2 dm = sub2(um1, ldrow(-2)), d0_ = sub2(w, um1), s0_ = square(d0_);
                const float2 qm = ldq(-1), q0 = ldq(0);
                qn = ldq(1);
                dn = sub2(wn, w);
                sn = square(dn);
                float2 dead;
                grads<LIM>(dm, square(dm), d0_, s0_, __fmul2_rn(f2(hy * myA), sub2(q0, qm)), uy, dead, Vp);
                th = __fmul2_rn(f2(hy * my0), sub2(qn, q0));
                grads<LIM>(d0_, s0_, dn, sn, th, uy, U, V);
            }
            float2 s2d = f2(0.f);
            #pragma unroll
            for (int j = 0; j < kRows; ++j) {
                const int o = j * nx;
                const float2 lv = ld2<VEC>(lam, o, o + 1);
                const float2 wnn = ldrow(j + 2), qnn = ldq(j + 2);
                const float2 eL = lde<S, VEC>(e + o, l0, l1, rx + (2 * j) * kThreads);
                const float2 eH = lde<S, VEC>(e + o, h0, h1, rx + (2 * j + 1) * kThreads);
                const float2 lL = ld2<VEC>(lam + o, l0, l1), lH = ld2<VEC>(lam + o, h0, h1);
                float2 v = __ffma2_rn(f2(wmD), mus[j * kThreads], __fmul2_rn(f2(diag), lv));
                {  // y: the face of the next row
                    const float2 db = sub2(wnn, wn), sb = square(db);
                    const float2 tn = __fmul2_rn(f2(j + 1 == kRows - 1 ? hy * my1 : (j + 1 == kRows ? hy * myB : hy)), sub2(qnn, qn));
                    float2 Un, Vn;
                    grads<LIM>(dn, sn, db, sb, tn, uy, Un, Vn);
                    v = __fadd2_rn(v, __ffma2_rn(f2(sy), th, __fadd2_rn(sub2(U, V), sub2(Vp, Un))));
                    Vp = V;
                    th = tn;
                    U = Un;
                    V = Vn;
                    dn = db;
                    sn = sb;
                    qn = qnn;
                }
                {  // x: the faces of cells x0-1, x0 (A) and x0+1, x0+2 (B)
                    const float2 a0 = make_float2(__fadd_rn(eL.y, -eL.x), __fadd_rn(w.x, -eL.y));
                    const float m1 = __fadd_rn(w.y, -w.x);
                    const float2 b1 = make_float2(__fadd_rn(eH.x, -w.y), __fadd_rn(eH.y, -eH.x));
                    const float2 sa0 = square(a0), sb1 = square(b1);
                    const float sm = fmaf(m1, m1, 0.5f * kTiny);
                    const float t0 = __fadd_rn(lL.y, -lL.x), t1 = __fadd_rn(lv.x, -lL.y), t2 = __fadd_rn(lv.y, -lv.x);
                    const float t3 = __fadd_rn(lH.x, -lv.y), t4 = __fadd_rn(lH.y, -lH.x);
                    const float2 tA = __fmul2_rn(hA, make_float2(ux ? t1 : t0, ux ? t2 : t1));
                    const float2 tB = __fmul2_rn(hB, make_float2(ux ? t3 : t2, ux ? t4 : t3));
                    float2 UA, VA, UB, VB;
                    grads<LIM>(a0, sa0, make_float2(a0.y, m1), make_float2(sa0.y, sm), tA, ux, UA, VA);
                    grads<LIM>(make_float2(m1, b1.x), make_float2(sm, sb1.x), b1, sb1, tB, ux, UB, VB);
                    const float2 own = __ffma2_rn(f2(sx), make_float2(tA.y, tB.x), sub2(make_float2(UA.y, UB.x), make_float2(VA.y, VB.x)));
                    v = __fadd2_rn(v, __fadd2_rn(own, sub2(VA, UB)));
                }
                if constexpr (DIM == 3) {  // z: the faces of slices z-1, z, z+1
                    const float2 e0 = lde<S, VEC>(e + o, zm2, zm2 + 1, rz + (4 * j) * kThreads);
                    const float2 e1 = lde<S, VEC>(e + o, zm1, zm1 + 1, rz + (4 * j + 1) * kThreads);
                    const float2 e3 = lde<S, VEC>(e + o, zp1, zp1 + 1, rz + (4 * j + 2) * kThreads);
                    const float2 e4 = lde<S, VEC>(e + o, zp2, zp2 + 1, rz + (4 * j + 3) * kThreads);
                    const float2 q1 = ld2<VEC>(lam + o, zm1, zm1 + 1), q3 = ld2<VEC>(lam + o, zp1, zp1 + 1);
                    const int zf = uz ? zp2 : zm2;
                    const float2 qf = ld2<VEC>(lam + o, zf, zf + 1);
                    const float2 up = sub2(lv, q1), dw = sub2(q3, lv), far = uz ? sub2(qf, q3) : sub2(q1, qf);
                    const float2 t0 = __fmul2_rn(f2(hz * mz0), uz ? up : far);
                    const float2 t1 = __fmul2_rn(f2(hz * mz1), uz ? dw : up);
                    const float2 t2 = __fmul2_rn(f2(hz * mz2), uz ? far : dw);
                    const float2 d1 = sub2(e1, e0), d2 = sub2(w, e1), d3 = sub2(e3, w), d4 = sub2(e4, e3);
                    const float2 q2s = square(d2), q3s = square(d3);
                    float2 dead, Vz, Uz, Wz, Ud;
                    grads<LIM>(d1, square(d1), d2, q2s, t0, uz, dead, Vz);
                    grads<LIM>(d2, q2s, d3, q3s, t1, uz, Uz, Wz);
                    grads<LIM>(d3, q3s, d4, square(d4), t2, uz, Ud, dead);
                    v = __fadd2_rn(v, __ffma2_rn(f2(sz), t1, __fadd2_rn(sub2(Uz, Wz), sub2(Vz, Ud))));
                }
                if constexpr (VEC) __stcs(reinterpret_cast<float2 *>(out + o), v);
                else {
                    __stcs(out + o, v.x);
                    __stcs(out + o + 1, v.y);
                }
                acc[j] = __fadd2_rn(acc[j], v);
                const float2 own = j >= jown ? ownx : f2(0.f);
                s1 = __ffma2_rn(__fmul2_rn(own, lv), __ffma2_rn(f2(-sc), w, ckt[j * kThreads]), s1);
                s2d = __ffma2_rn(__fmul2_rn(own, mus[j * kThreads]), w, s2d);
                w = wn;
                wn = wnn;
            }
            s2 = __ffma2_rn(f2(__ldg(g.w + d) * sc), s2d, s2);
        }
        float *P = g.P + (long long)row * a.ncell + idx0;
        #pragma unroll
        for (int j = 0; j < kRows; ++j) {
            if constexpr (VEC) *reinterpret_cast<float2 *>(P + j * nx) = acc[j];
            else {
                P[j * nx] = acc[j].x;
                P[j * nx + 1] = acc[j].y;
            }
        }
    }
    // the part's scalars: warp sums, then warp 0 adds the warps in order
    float t1 = s1.x + s1.y, t2 = s2.x + s2.y;
    #pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        t1 += __shfl_xor_sync(0xffffffffu, t1, o);
        t2 += __shfl_xor_sync(0xffffffffu, t2, o);
    }
    if ((threadIdx.x & 31) == 0) {
        red[0][threadIdx.x >> 5] = t1;
        red[1][threadIdx.x >> 5] = t2;
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        float t = 0.f;
        for (int i = 0; i < kThreads / 32; ++i) t += red[threadIdx.x][i];
        g.Ps[2 * (long long)blockIdx.x + threadIdx.x] = t;
    }
}

template <int S, int LIM, int DIM, bool VEC>
cudaError_t launch_one(const StepArgs &a, const AdjStreamArgs &g, cudaStream_t s) {
    const int smem = slots<S, DIM>() * kThreads * (int)sizeof(float2);
    cudaError_t e = cudaFuncSetAttribute(k_adj_stream<S, LIM, DIM, VEC>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    k_adj_stream<S, LIM, DIM, VEC><<<(unsigned)(a.nb * g.nchunk * g.blocks), kThreads, smem, s>>>(a, g);
    return cudaGetLastError();
}
template <int S, int DIM, bool VEC>
cudaError_t launch_lim(const StepArgs &a, const AdjStreamArgs &g, int limiter, cudaStream_t s) {
    if (limiter == kLimFirst) return launch_one<S, kLimFirst, DIM, VEC>(a, g, s);
    if (limiter == kLimMinmod) return launch_one<S, kLimMinmod, DIM, VEC>(a, g, s);
    return launch_one<S, kLimVanAlbada, DIM, VEC>(a, g, s);
}
template <int S>
cudaError_t launch_storage(const StepArgs &a, const AdjStreamArgs &g, int limiter, cudaStream_t s) {
    const bool vec = a.n[0] % 2 == 0;
    if (a.dim == 3) return vec ? launch_lim<S, 3, true>(a, g, limiter, s) : launch_lim<S, 3, false>(a, g, limiter, s);
    return vec ? launch_lim<S, 2, true>(a, g, limiter, s) : launch_lim<S, 2, false>(a, g, limiter, s);
}
// one definition per instantiation unit
cudaError_t launch_f32(const StepArgs &a, const AdjStreamArgs &g, int limiter, cudaStream_t s);
cudaError_t launch_f16(const StepArgs &a, const AdjStreamArgs &g, int limiter, cudaStream_t s);
cudaError_t launch_bf16(const StepArgs &a, const AdjStreamArgs &g, int limiter, cudaStream_t s);

}  // namespace adjs
}  // namespace bte
