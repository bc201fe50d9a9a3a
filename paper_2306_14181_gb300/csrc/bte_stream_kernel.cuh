// Register-streaming forward step of the explicit DOM scheme (arXiv 2306.14181, Sec. 4, Eq.
// disretized_transientBTE) for 2-D and 3-D grids of any shape, any wall, with
// FP32 states (small grids are faster on the generic kernel and run it); included by the instantiation
// units bte_stream_<dim>d.cu.
//
// A thread owns two neighbouring cells of a row and KR rows, and loops over a part of one band's
// directions.  Per direction it streams the rows from upwind to downwind straight from global memory:
// the y difference and slope of a row come from the row before it, and the two cells share the face
// between them (1.5 x, 1 + 1/KR y and 2 z limited slopes a cell).  The T_L moment partials of the
// thread's cells stay in registers for the whole part (in stream order, reversed when the y sign of the
// directions changes, which their order makes rare) and the relaxation targets in shared memory, which
// no other thread reads, so nothing but the state moves and no barrier is needed.
//
// What bounds it: issue and latency, not DRAM.  FP32, 256^2 x 40 x 128, interior threads alone: 0.61 ms
// (41 instructions an update, issue slots 53 % busy, FMA pipes 47 %), 66 % of the measured copy rate; with
// the threads next to the walls 0.77 to 0.80 ms.  The kernel it replaced (one thread a cell and band,
// ghost rules per neighbour) took 4.0 ms.  Odd grids, that kernel before, this one after: 203 x 157, 24 x
// 96: 817 -> 191 us; 97 x 75 x 41, 10 x 96: 1.21 ms.  16-bit states keep the generic kernel: a last-bit
// change of the sums before a code is rounded flips codes, and the heat flux and the gradients taken from
// coded states show it.  Tried and slower: two or four slices a thread (their code no
// longer fits the instruction cache: 2.3 ms against 2.1 on 128^2 x 64 x 8 x 96), relaxation targets in
// registers (3-8 %), no L2 prefetch of the next direction (8-10 %), x ghosts by general sources in
// every warp (3.9 ms).
//
// Strips and groups that do not fit are shifted back to overlap their neighbour: the cells of the
// overlap are computed twice by the same operations and stored twice with the same bits, and no
// loop carries a ragged end.  Rows and slices outside the domain that hold cells of the same plane
// (the wrapped row, the wall row itself for directions leaving through it) are plain offsets
// worked out once per sign; the remaining ghost values (Sec. 2.2) come by a thread's sources, pointers
// by kind worked out once per sign too.  Threads next to an x wall (whose loads touch a line a lane)
// and, in 3-D, next to a y or z wall run in blocks of their own.
#pragma once

#include "bte_internal.h"
#include "bte_stream.h"

namespace bte {
namespace stream {

constexpr int kThreads = 256;
constexpr float kVaTiny = 0x1p-125f;

__device__ __forceinline__ float rcp_approx(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float2 f2(float x) { return make_float2(x, x); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, f2(-1.f), a); }

// The limited slope L(a, b) of the upwind and downwind differences a, b; a face's value is e_m + L/2.
// Van Albada: max(ab, 0) (a + b) / (a^2 + b^2 + 2^-125) with the approximate reciprocal of a denominator
// that is always a normal number; the constant is below the last bit of the squares wherever the products of
// the numerator are normal numbers, so slopes are limited alike in any units.
template <int LIM> __device__ __forceinline__ float slope(float a, float b);
template <> __device__ __forceinline__ float slope<kLimFirst>(float, float) { return 0.f; }
template <> __device__ __forceinline__ float slope<kLimMinmod>(float a, float b) {
    const float m = fabsf(a) < fabsf(b) ? a : b;
    return __fmul_rn(a, b) > 0.f ? m : 0.f;
}
template <> __device__ __forceinline__ float slope<kLimVanAlbada>(float a, float b) {
    const float num = __fmul_rn(fmaxf(__fmul_rn(a, b), 0.f), __fadd_rn(a, b));
    return __fmul_rn(num, rcp_approx(fmaf(a, a, fmaf(b, b, kVaTiny))));
}
template <int LIM> __device__ __forceinline__ float2 slope2(float2 a, float2 b) {
    if constexpr (LIM == kLimVanAlbada) {
        const float2 ab = __fmul2_rn(a, b);
        const float2 num = __fmul2_rn(make_float2(fmaxf(ab.x, 0.f), fmaxf(ab.y, 0.f)), __fadd2_rn(a, b));
        const float2 den = __ffma2_rn(a, a, __ffma2_rn(b, b, f2(kVaTiny)));
        return __fmul2_rn(num, make_float2(rcp_approx(den.x), rcp_approx(den.y)));
    } else {
        return make_float2(slope<LIM>(a.x, b.x), slope<LIM>(a.y, b.y));
    }
}
// Twice the difference of a cell's out-face and in-face, 2 (e_i - e_up) + (L_i - L_up), from its upwind
// difference a: no face value is formed, so nothing is rounded at the size of e but the final sum.
__device__ __forceinline__ float2 outflow(float2 a, float2 L, float2 Lup) { return __ffma2_rn(f2(2.f), a, sub2(L, Lup)); }

// A pair of neighbouring cells: 8 bytes where rows are even (VEC), else cell by cell.
template <bool VEC> __device__ __forceinline__ float2 two(const float *p) {
    if constexpr (VEC) return __ldg(reinterpret_cast<const float2 *>(p));
    else return make_float2(__ldg(p), __ldg(p + 1));
}
template <bool VEC> __device__ __forceinline__ void put(float *p, float2 v) {
    if constexpr (VEC) __stcs(reinterpret_cast<float2 *>(p), v);
    else {
        __stcs(p, v.x);
        __stcs(p + 1, v.y);
    }
}

// What a stencil position along axis ax holds for a direction of sign sg on that axis (Sec. 2.2).
enum : int {
    kCell = 0,   // a cell of the same plane: itself, the wrapped cell, or the wall cell for
                 // directions leaving through a thermalizing or diffuse wall
    kMirror = 1, // specular wall: the mirrored direction at the mirrored cell
    kDiff = 2,   // diffuse wall, entering: the wall's value
    kConst = 3,  // thermalizing wall, entering: the emission, a constant of the band
    kJump = 4,   // periodic wall with a temperature jump: the wrapped cell plus a constant
};
// kind of position pos, and in `at` the cell's position along the axis
__device__ __forceinline__ int position(const StepArgs &a, int ax, int pos, int sg, bool jump, int &at) {
    const int n = a.n[ax];
    at = pos;
    if (pos >= 0 && pos < n) return kCell;
    const int side = pos < 0 ? 0 : 1, bc = a.bc[2 * ax + side];
    if (bc == kBcPeriodic) {
        at = side ? pos - n : pos + n;
        return jump ? kJump : kCell;
    }
    if (bc == kBcSpecular) {
        at = side ? 2 * n - 1 - pos : -pos - 1;
        return kMirror;
    }
    at = side ? n - 1 : 0;
    if (side == 0 ? sg <= 0 : sg >= 0) return kCell;
    return bc == kBcDiffuse ? kDiff : kConst;
}

// Where a stencil value around a thread's cells comes from: the array (of the plane, of the mirrored
// direction, of the wall's values) by kind, and row 0's index in it with its step with the row.
struct Src {
    int kind;
    int at;    // index of row 0's value in its array
    int step;  // of `at` with the row
    float c;   // kConst: the value; kJump: the offset
};
// a thread's sources: x neighbours m2, m1, p1 (scalars), rows -2, -1, KR and slices -2, -1, 1 (pairs)
enum : int { kX = 0, kY = 3, kZ = 6, kSources = 9 };

// A thread's cells and, for the current direction signs, where its rows and slices lie.
struct Place {
    int x0, y0, z;         // first cell of the group, first row of the strip, slice
    int sy, sz;            // signs of the current directions
    int idx0, dy;          // cell index of stream row 0; step downwind
    int ym2, ym1, yp;      // cell offsets from row 0 of rows -2, -1 and KR
    int zm2, zm1, zp;      // cell offsets of slices -2, -1 and 1
    bool yspec, zspec;     // some row / slice holds no plain cells
};

template <int DIM, int KR>
__device__ __forceinline__ void aim(const StepArgs &a, Place &t, int sy, int sz, int jump) {
    const int nx = a.n[0], nxy = a.n[0] * a.n[1];
    t.sy = sy;
    t.sz = sz;
    const int ys = sy > 0 ? t.y0 : t.y0 + KR - 1;
    t.dy = sy * nx;
    t.idx0 = t.z * nxy + ys * nx + t.x0;
    t.ym2 = t.ym1 = t.yp = t.zm2 = t.zm1 = t.zp = 0;
    t.yspec = t.zspec = false;
    int p2, p1, pd;
    {
        const int k2 = position(a, 1, ys - 2 * sy, sy, jump >> 1 & 1, p2);
        const int k1 = position(a, 1, ys - sy, sy, jump >> 1 & 1, p1);
        const int kd = position(a, 1, ys + KR * sy, sy, jump >> 1 & 1, pd);
        t.ym2 = (p2 - ys) * nx;
        t.ym1 = (p1 - ys) * nx;
        t.yp = (pd - ys) * nx;
        t.yspec = (k2 | k1 | kd) != kCell;
    }
    if constexpr (DIM == 3) {
        const int k2 = position(a, 2, t.z - 2 * sz, sz, jump >> 2 & 1, p2);
        const int k1 = position(a, 2, t.z - sz, sz, jump >> 2 & 1, p1);
        const int kd = position(a, 2, t.z + sz, sz, jump >> 2 & 1, pd);
        t.zm2 = (p2 - t.z) * nxy;
        t.zm1 = (p1 - t.z) * nxy;
        t.zp = (pd - t.z) * nxy;
        t.zspec = (k2 | k1 | kd) != kCell;
    }
}

// The thread's sources for the current signs, to its own memory (kept out of the registers of the
// plain sweep).
template <int DIM, int KR>
__device__ __noinline__ void fill_sources(const StepArgs &a, const Place &t, int k, int sx, int jump, Src *src) {
    const int ys = t.sy > 0 ? t.y0 : t.y0 + KR - 1;
    for (int s = 0; s < 3 * DIM; ++s) {
        const int ax = s / 3, m = s - 3 * ax;
        const int sg = ax == 0 ? sx : (ax == 1 ? t.sy : t.sz), ref = ax == 0 ? t.x0 : (ax == 1 ? ys : t.z);
        int off = m == 0 ? -2 * sg : (m == 1 ? -sg : (ax == 1 ? KR * sg : sg));
        if (ax == 0) off = sx > 0 ? (m == 0 ? -2 : (m == 1 ? -1 : 2)) : (m == 0 ? 3 : (m == 1 ? 2 : -1));
        const int pos = ref + off;
        Src q;
        int at;
        q.kind = position(a, ax, pos, sg, (jump >> ax & 1) != 0, at);
        const int stride = ax == 0 ? 1 : (ax == 1 ? a.n[0] : a.n[0] * a.n[1]);
        q.at = t.idx0 + (at - ref) * stride;
        q.step = t.dy;
        q.c = 0.f;
        const int wall = 2 * ax + (pos < 0 ? 0 : 1);
        if (q.kind == kDiff) {
            // wall cells: x walls z ny + y, y walls z nx + x, z walls y nx + x
            q.at = (wall * a.nb + k) * a.wc_max +
                   (ax == 0 ? t.z * a.n[1] + ys : (ax == 1 ? t.z * a.n[0] + t.x0 : ys * a.n[0] + t.x0));
            if (ax == 0) q.step = t.sy;
        } else if (q.kind == kConst) {
            q.c = __ldg(a.iso + wall * a.nb + k);
        } else if (q.kind == kJump) {
            q.c = (pos < 0 ? 1.f : -1.f) * __ldg(a.jmp + ax * a.nb + k);
        }
        src[s] = q;
    }
}

// x neighbours of a pair in stream order (m2, m1 upwind, p1 downwind) and z neighbours.
struct Xn { float m2, m1, p1; };
struct Zn { float2 m2, m1, p1; };

// The update of one row: e^{n+1} of the pair w from its neighbours (wn: the next row downwind; ya, Ly: the
// difference and slope upwind in y, replaced by those downwind), bt the relaxation target.  The increment
// is summed first and added to e once.
template <int LIM, int DIM, int SX>
__device__ __forceinline__ float2 update(float2 w, float2 wn, const Xn &x, const Zn &z, float2 bt, float dtinv, float hx,
                                         float hy, float hz, float2 &ya, float2 &Ly) {
    const float c0 = SX > 0 ? w.x : w.y, c1 = SX > 0 ? w.y : w.x;  // upwind, downwind cell
    const float d0 = __fadd_rn(x.m1, -x.m2), d1 = __fadd_rn(c0, -x.m1), d2 = __fadd_rn(c1, -c0), d3 = __fadd_rn(x.p1, -c1);
    const float Lm = slope<LIM>(d0, d1);
    // differences and slopes of the pair in its own order
    const float2 xa = SX > 0 ? make_float2(d1, d2) : make_float2(d2, d1);
    const float2 Lx = slope2<LIM>(xa, SX > 0 ? make_float2(d2, d3) : make_float2(d3, d2));
    float2 inc = __ffma2_rn(f2(-dtinv), w, bt);
    inc = __ffma2_rn(f2(-hx), outflow(xa, Lx, SX > 0 ? make_float2(Lm, Lx.x) : make_float2(Lx.y, Lm)), inc);
    {
        const float2 yb = sub2(wn, w), Ln = slope2<LIM>(ya, yb);
        inc = __ffma2_rn(f2(-hy), outflow(ya, Ln, Ly), inc);
        ya = yb;
        Ly = Ln;
    }
    if constexpr (DIM == 3) {
        const float2 e1 = sub2(w, z.m1);
        const float2 Li = slope2<LIM>(sub2(z.m1, z.m2), e1), Lo = slope2<LIM>(e1, sub2(z.p1, w));
        inc = __ffma2_rn(f2(-hz), outflow(e1, Lo, Li), inc);
    }
    return __fadd2_rn(w, inc);
}

// Half the Courant numbers of a plane (the face differences are doubled) and its moment weight.
struct Dir {
    float hx, hy, hz, wm;
};
template <int DIM> __device__ __forceinline__ Dir direction(const StepArgs &a, int plane) {
    const float *nu = a.nu + 3 * (long long)plane;
    Dir d;
    d.hx = 0.5f * fabsf(__ldg(nu));
    d.hy = 0.5f * fabsf(__ldg(nu + 1));
    d.hz = DIM == 3 ? 0.5f * fabsf(__ldg(nu + 2)) : 0.f;
    d.wm = __ldg(a.wmom + plane);
    return d;
}

// One direction over the thread's cells.  XG: a group next to an x wall, the x
// neighbours come by their sources; ZG: the z neighbours come by theirs (next to a z wall).
template <int LIM, int DIM, int KR, bool VEC, int SX, bool XG, bool ZG>
__device__ __forceinline__ void sweep(const StepArgs &a, const Place &t, int plane, float dtinv, int next, float2 (&acc)[KR],
                                      const float2 *bts, const Src *src) {
    const float *e = static_cast<const float *>(a.e_in) + (long long)plane * a.ncell;
    float *eo = static_cast<float *>(a.e_out) + (long long)plane * a.ncell;
    const Dir dr = direction<DIM>(a, plane);
    auto base = [&](const Src &q, int ax) {
        const float *p = e;
        if (q.kind == kMirror) {
            const int k = plane / a.nd, d = plane - k * a.nd;
            p = static_cast<const float *>(a.e_in) + (long long)(k * a.nd + __ldg(a.mirror + ax * a.nd + d)) * a.ncell;
        }
        if (q.kind == kDiff) p = static_cast<const float *>(a.ediff_in);
        return p + q.at;
    };
    auto pair = [&](const Src &q, const float *p, int j) {
        float2 v = two<VEC>(p + j * q.step);
        if (q.kind >= kConst) v = q.kind == kConst ? f2(q.c) : __fadd2_rn(v, f2(q.c));
        return v;
    };
    auto yval = [&](int m, int off) {
        if (!t.yspec) return two<VEC>(e + (t.idx0 + off));
        const Src q = src[kY + m];
        return pair(q, base(q, 1), 0);
    };
    // x neighbours by their sources: pointers of row 0
    const float *xp[3];
    int xstep[3], xkind = 0;
    if constexpr (XG) {
        #pragma unroll
        for (int m = 0; m < 3; ++m) {
            const Src q = src[kX + m];
            xp[m] = base(q, 0);
            xstep[m] = q.step;
            xkind |= (q.kind >= kConst ? q.kind - kConst + 1 : 0) << (2 * m);
        }
    }
    auto ldx = [&](int j, int id) {
        Xn x;
        if constexpr (XG) {
            float v[3];
            #pragma unroll
            for (int m = 0; m < 3; ++m) v[m] = __ldg(xp[m] + j * xstep[m]);
            if (xkind != 0) {
                #pragma unroll
                for (int m = 0; m < 3; ++m) {
                    const int q = xkind >> (2 * m) & 3;
                    if (q) v[m] = q == 1 ? src[kX + m].c : __fadd_rn(v[m], src[kX + m].c);
                }
            }
            x.m2 = v[0];
            x.m1 = v[1];
            x.p1 = v[2];
        } else {
            const float2 q = two<VEC>(e + (SX > 0 ? id - 2 : id + 2));
            x.m2 = SX > 0 ? q.x : q.y;
            x.m1 = SX > 0 ? q.y : q.x;
            x.p1 = __ldg(e + (SX > 0 ? id + 2 : id - 1));
        }
        return x;
    };
    Src zq[3];
    const float *zb[3];
    if constexpr (ZG) {
        #pragma unroll
        for (int m = 0; m < 3; ++m) {
            zq[m] = src[kZ + m];
            zb[m] = base(zq[m], 2);
        }
    }
    auto ldz = [&](int j, int id) {
        if constexpr (ZG) return Zn{pair(zq[0], zb[0], j), pair(zq[1], zb[1], j), pair(zq[2], zb[2], j)};
        else return Zn{two<VEC>(e + (id + t.zm2)), two<VEC>(e + (id + t.zm1)), two<VEC>(e + (id + t.zp))};
    };
    auto ldrow = [&](int j) { return j < KR ? two<VEC>(e + (t.idx0 + j * t.dy)) : yval(2, t.yp); };
    const float2 m2 = yval(0, t.ym2), m1 = yval(1, t.ym1);
    float2 w = two<VEC>(e + t.idx0), wn = ldrow(1);
    float2 ya = sub2(w, m1), Ly = slope2<LIM>(sub2(m1, m2), ya);
    Xn xc = ldx(0, t.idx0);
    Zn zc = {};
    if constexpr (DIM == 3) zc = ldz(0, t.idx0);
    // the same cells of the next direction, towards L2
    if (next >= 0) {
        const float *en = static_cast<const float *>(a.e_in) + (long long)next * a.ncell;
        #pragma unroll
        for (int j = 0; j < KR; ++j) asm volatile("prefetch.global.L2 [%0];" ::"l"(en + (t.idx0 + j * t.dy)));
    }
    #pragma unroll
    for (int j = 0; j < KR; ++j) {
        const int id = t.idx0 + j * t.dy;
        // the next row's loads go out before this row's arithmetic
        float2 wnn = f2(0.f);
        Xn xn = xc;
        Zn zn = {};
        if (j + 1 < KR) {
            wnn = ldrow(j + 2);
            xn = ldx(j + 1, id + t.dy);
            if constexpr (DIM == 3) zn = ldz(j + 1, id + t.dy);
        }
        const float2 en = update<LIM, DIM, SX>(w, wn, xc, zc, bts[(t.sy > 0 ? j : KR - 1 - j) * kThreads], dtinv, dr.hx,
                                               dr.hy, dr.hz, ya, Ly);
        put<VEC>(eo + id, en);
        acc[j] = __ffma2_rn(f2(dr.wm), en, acc[j]);
        w = wn;
        wn = wnn;
        xc = xn;
        zc = zn;
    }
}

// Blocks an SM the register budget aims at: 24 warps of 80 registers in 2-D, 16 of 128 in 3-D.
template <int DIM> constexpr int min_blocks() { return DIM == 3 ? 2 : 3; }

template <int LIM, int DIM, int KR, bool VEC>
__global__ void __launch_bounds__(kThreads, min_blocks<DIM>()) k_step_stream(const __grid_constant__ StepArgs a,
                                                                  const __grid_constant__ StreamArgs p) {
    __shared__ float2 bts[KR * kThreads];
    // Blocks of a (band, part): sb of them hold the threads next to a wall (the groups next to an x wall,
    // then the other groups of the special strips), which wait on latencies.  Spread evenly among the
    // others, whose arithmetic on the same SM covers them (mixed), or first of the whole launch.
    const int nblk = p.blocks[0] + p.blocks[1] + p.blocks[2], sb = p.blocks[0] + p.blocks[1];
    int row, bi, cls;  // row: of P
    if (p.mixed) {
        row = blockIdx.x / nblk;
        const int i = blockIdx.x - row * nblk;
        const int s0 = (int)((long long)i * sb / nblk), s1 = (int)((long long)(i + 1) * sb / nblk);
        cls = s1 > s0 ? (s0 < p.blocks[0] ? 0 : 1) : 2;
        bi = cls == 2 ? i - s0 : (cls == 1 ? s0 - p.blocks[0] : s0);
    } else {
        bi = blockIdx.x;
        cls = 0;
        while (cls < 2 && bi >= p.blocks[cls] * a.nb * p.nchunk) bi -= p.blocks[cls++] * a.nb * p.nchunk;
        row = bi / p.blocks[cls];
        bi -= row * p.blocks[cls];
    }
    const bool edge = cls == 0;
    const int per = edge ? p.E : p.G - p.E;  // groups a strip
    const int tid = bi * kThreads + (int)threadIdx.x;
    int strip = tid / per;
    const int gi = tid - strip * per;
    if (cls == 2) strip += p.nspecial;
    if (strip >= (cls == 1 ? p.nspecial : p.nys * p.nz)) return;
    strip = __ldg(p.strips + strip);
    // group: the E next to the walls are the row's first and its last E - 1
    const int g = edge ? (gi == 0 ? 0 : p.G - p.E + gi) : gi + 1;
    Place t;
    t.x0 = min(2 * g, a.n[0] - 2);
    const int ys = DIM == 3 ? strip / p.nz : strip;
    t.z = DIM == 3 ? strip - ys * p.nz : 0;
    t.y0 = min(ys * KR, a.n[1] - KR);
    const int k = row / p.nchunk, c = row - k * p.nchunk;
    const int d0 = (int)((long long)c * a.nd / p.nchunk), d1 = (int)((long long)(c + 1) * a.nd / p.nchunk);
    const BandConst b = a.band[k];
    float2 acc[KR];
    float2 *bt = bts + threadIdx.x;
    int tsx = 0;
    t.sz = 0;
    t.sy = 1;
    Src src[kSources];
    // relaxation target and source, dt/tau C T_L / W + a dt C Q/(sum C W)
    const int id0 = (t.z * a.n[1] + t.y0) * a.n[0] + t.x0;
    #pragma unroll
    for (int j = 0; j < KR; ++j) {
        const int id = id0 + j * a.n[0];
        float v[2];
        #pragma unroll
        for (int x = 0; x < 2; ++x) {
            const float src = a.Q ? __fmul_rn(b.srck, __fmul_rn(a.amp, __ldg(a.Q + id + x))) : 0.f;
            v[x] = fmaf(b.dtinv, __fmul_rn(b.ck, __ldg(a.TL + id + x)), src);
        }
        bt[j * kThreads] = make_float2(v[0], v[1]);
        acc[j] = f2(0.f);
    }
    int dn = __ldg(p.dord + d0);
    for (int o = d0; o < d1; ++o) {
        const int d = dn, plane = k * a.nd + d;
        dn = o + 1 < d1 ? __ldg(p.dord + o + 1) : -1;
        const int next = dn < 0 ? -1 : k * a.nd + dn;
        const float *nu = a.nu + 3 * (long long)plane;
        const int sx = __ldg(nu) < 0.f ? -1 : 1;
        const int sy = __ldg(nu + 1) < 0.f ? -1 : 1, sz = DIM == 3 && __ldg(nu + 2) < 0.f ? -1 : 1;
        if (sx != tsx || sy != t.sy || sz != t.sz) {
            if (sy != t.sy) {
                #pragma unroll
                for (int j = 0; j < KR / 2; ++j) {
                    const float2 u = acc[j];
                    acc[j] = acc[KR - 1 - j];
                    acc[KR - 1 - j] = u;
                }
            }
            aim<DIM, KR>(a, t, sy, sz, p.jump);
            tsx = sx;
            if (edge || t.zspec || t.yspec) fill_sources<DIM, KR>(a, t, k, sx, p.jump, src);
        }
#define BTE_SWEEP(SX_, X_, Z_) sweep<LIM, DIM, KR, VEC, SX_, X_, Z_>(a, t, plane, b.dtinv, next, acc, bt, src)
        if (edge) {
            if (sx > 0) BTE_SWEEP(1, true, DIM == 3); else BTE_SWEEP(-1, true, DIM == 3);
        } else if (DIM == 3 && t.zspec) {
            if (sx > 0) BTE_SWEEP(1, false, DIM == 3); else BTE_SWEEP(-1, false, DIM == 3);
        } else {
            if (sx > 0) BTE_SWEEP(1, false, false); else BTE_SWEEP(-1, false, false);
        }
#undef BTE_SWEEP
    }
    // moment partials of this part: sum w/tau e
    float *P = a.P + (long long)row * a.ncell;
    #pragma unroll
    for (int j = 0; j < KR; ++j) {
        const int id = id0 + (t.sy > 0 ? j : KR - 1 - j) * a.n[0];
        if constexpr (VEC) *reinterpret_cast<float2 *>(P + id) = acc[j];
        else {
            P[id] = acc[j].x;
            P[id + 1] = acc[j].y;
        }
    }
}

typedef void (*StreamKernel)(const StepArgs, const StreamArgs);

// rows a thread; fewer on small grids
constexpr int kRows = 4, kRowsSmall = 2;

template <int DIM, int KR, bool VEC>
StreamKernel pick_lim(int lim) {
    if (lim == kLimFirst) return k_step_stream<kLimFirst, DIM, KR, VEC>;
    if (lim == kLimMinmod) return k_step_stream<kLimMinmod, DIM, KR, VEC>;
    return k_step_stream<kLimVanAlbada, DIM, KR, VEC>;
}

template <int DIM>
StreamKernel pick_instance(int lim, bool vec, int kr) {
    if (kr == kRows) return vec ? pick_lim<DIM, kRows, true>(lim) : pick_lim<DIM, kRows, false>(lim);
    return vec ? pick_lim<DIM, kRowsSmall, true>(lim) : pick_lim<DIM, kRowsSmall, false>(lim);
}

// one definition per instantiation unit
StreamKernel pick_2d(int lim, bool vec, int kr);
StreamKernel pick_3d(int lim, bool vec, int kr);

}  // namespace stream
}  // namespace bte
