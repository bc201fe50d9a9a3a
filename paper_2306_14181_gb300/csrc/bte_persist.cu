// Persistent forward step for small 1-D problems (the cross-plane film of Sec. 3.6): the whole
// FP32 state lives in the shared memory of one thread-block cluster for all the steps of one
// bte_step call, so a step costs block barriers and one cluster barrier instead of launches.  Each step follows
// Eq. (disretized_transientBTE) with the limited face value of Sec. 4.1 and the wall ghosts of
// Sec. 2.2 (periodic wrap, thermalizing emission, diffuse value Eq. diff_bound, specular
// mirror), then forms T_L of Eq. (BTE_get_e0) from the new state.  At the end the state, T_L
// and the diffuse-wall values are written back, so the context continues as after bte_step.
#include <cooperative_groups.h>

#include "bte_device.cuh"

namespace bte {

// Value of plane (band lb of this CTA, global band kg, direction d) at position p of the 1-D
// line (p in [-2, n+1]); eps: the CTA's state [nbl*nd][n]; ed: its diffuse-wall values [2][nbl].
__device__ __forceinline__ float p1_ext(const StepArgs &a, const float *eps, const float *ed, int lb, int kg, int d,
                                       int p, float nu, int nbl) {
    const int n = a.n[0];
    const float *row = eps + (lb * a.nd + d) * n;
    if (p >= 0 && p < n) return row[p];
    const int side = p < 0 ? 0 : 1;
    const int bc = a.bc[side];
    if (bc == kBcPeriodic) return row[side ? p - n : p + n];
    if (bc == kBcSpecular) {
        const int layer = side ? p - n + 1 : -p;
        return eps[(lb * a.nd + a.mirror[d]) * n + (side ? n - layer : layer - 1)];
    }
    const bool incoming = side == 0 ? nu > 0.f : nu < 0.f;
    if (!incoming) return row[side ? n - 1 : 0];
    if (bc == kBcIsothermal) return a.iso[side * a.nb + kg];
    return ed[side * nbl + lb];
}

// Persistent kernel: a thread-block cluster of C CTAs, CTA r owning bands r, r + C, ...; each
// holds its bands' state in shared memory for all the steps.  Per step a CTA updates its planes,
// forms its bands' share of the T_L numerator per cell (fixed plane order) in a double-buffered
// shared array, the cluster synchronises once, and every CTA adds the C shares in rank order
// from distributed shared memory.  C = 1 is the single-CTA case.
template <int LIM>
__global__ void __launch_bounds__(1024, 1) k_persist_1d(const StepArgs a, int nsteps, const float *amps, float *e_io,
                                                        float *tl_out, float *ediff_out) {
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    const int C = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    extern __shared__ __align__(16) float sm[];
    const int n = a.n[0], nd = a.nd;
    const int nbl = (a.nb - rank + C - 1) / C;  // bands of this CTA: rank, rank + C, ...
    const int npl = nbl * nd, nel = npl * n;
    // laid out for rank 0's bands (the most): peers read one another's part at the same place
    const int nelm = (a.nb + C - 1) / C * nd * n;
    float *e0 = sm, *e1 = sm + nelm, *tl = e1 + nelm;
    float *part = tl + n;  // [2][n] this CTA's share of the T_L numerator, read by the cluster
    float *ed = part + 2 * n;  // [2][nbl] diffuse-wall values of this CTA's bands
    float *pnu = ed + 2 * nbl, *pwm = pnu + npl, *pdt = pwm + npl, *pck = pdt + npl, *psr = pck + npl;
    // local plane lp = lb * nd + d is global plane (rank + lb C) nd + d
    auto gplane = [&](int lp) { return (rank + (lp / nd) * C) * nd + lp % nd; };
    for (int j = threadIdx.x; j < nel; j += blockDim.x) e0[j] = e_io[(long long)gplane(j / n) * n + j % n];
    for (int lp = threadIdx.x; lp < npl; lp += blockDim.x) {
        const int pl = gplane(lp);
        const BandConst b = a.band[pl / nd];
        pnu[lp] = a.nu[3 * pl];
        pwm[lp] = a.wmom[pl];
        pdt[lp] = b.dtinv;
        pck[lp] = b.ck;
        psr[lp] = b.srck;
    }
    __syncthreads();
    // this CTA's diffuse-wall values and share of the T_L numerator, from the state es
    auto walls_and_share = [&](const float *es, float *pt) {
        for (int j = threadIdx.x; j < 2 * nbl; j += blockDim.x) {
            const int side = j / nbl, lb = j % nbl;
            float v = 0.f;
            if (a.bc[side] == kBcDiffuse) {
                const int x = side ? n - 1 : 0;
                for (int d = 0; d < nd; ++d) v = fmaf(a.wdiff[side * nd + d], es[(lb * nd + d) * n + x], v);
                v *= a.inv_den[side];
            }
            ed[j] = v;
        }
        for (int x = threadIdx.x; x < n; x += blockDim.x) {
            float v = 0.f;
            for (int lp = 0; lp < npl; ++lp) v = fmaf(pwm[lp], es[lp * n + x], v);
            pt[x] = v;
        }
    };
    auto gather_tl = [&](int buf) {
        for (int x = threadIdx.x; x < n; x += blockDim.x) {
            float v = 0.f;
            for (int r = 0; r < C; ++r) v += cl.map_shared_rank(part + buf * n, r)[x];
            tl[x] = v * a.invD;
        }
    };
    int buf = 0;
    walls_and_share(e0, part + buf * n);
    cl.sync();
    gather_tl(buf);
    __syncthreads();
    const int bx = blockDim.x % n, bp = blockDim.x / n;
    const int x00 = threadIdx.x % n, p00 = threadIdx.x / n;
    for (int s = 0; s < nsteps; ++s) {
        const float amp = amps[s];
        int x = x00, lp = p00;
        for (int j = threadIdx.x; j < nel; j += blockDim.x) {
            const int lb = lp / nd, d = lp - lb * nd;
            const float nu = pnu[lp];
            const float u0 = e0[j];
            float div = 0.f;
            if (nu != 0.f) {
                const int sg = nu > 0.f ? 1 : -1;
                // interior cells read the row directly; the two cells next to each wall use the
                // ghost rules (the mirrored direction is in the same band, so in this CTA)
                float um2, um1, up1;
                if (x >= 2 && x + 2 < n) {
                    um2 = e0[j - 2 * sg];
                    um1 = e0[j - sg];
                    up1 = e0[j + sg];
                } else {
                    const int kg = rank + lb * C;
                    um2 = p1_ext(a, e0, ed, lb, kg, d, x - 2 * sg, nu, nbl);
                    um1 = p1_ext(a, e0, ed, lb, kg, d, x - sg, nu, nbl);
                    up1 = p1_ext(a, e0, ed, lb, kg, d, x + sg, nu, nbl);
                }
                const float fo = u0 + 0.5f * limit<LIM>(u0 - um1, up1 - u0);
                const float fi = um1 + 0.5f * limit<LIM>(um1 - um2, u0 - um1);
                div = fabsf(nu) * (fo - fi);
            }
            const float src = a.Q ? psr[lp] * (amp * a.Q[x]) : 0.f;
            e1[j] = u0 - div + pdt[lp] * (pck[lp] * tl[x] - u0) + src;
            x += bx;
            lp += bp;
            if (x >= n) {
                x -= n;
                ++lp;
            }
        }
        __syncthreads();
        buf ^= 1;
        walls_and_share(e1, part + buf * n);
        cl.sync();  // every CTA's share of this step is written; the previous buffer is free
        gather_tl(buf);
        __syncthreads();
        float *t = e0;
        e0 = e1;
        e1 = t;
    }
    for (int j = threadIdx.x; j < nel; j += blockDim.x) e_io[(long long)gplane(j / n) * n + j % n] = e0[j];
    if (rank == 0)
        for (int x = threadIdx.x; x < n; x += blockDim.x) tl_out[x] = tl[x];
    // the diffuse-wall values in the layout the other kernels read: [wall][k][wall cell 0]
    for (int j = threadIdx.x; j < 2 * nbl; j += blockDim.x) {
        const int side = j / nbl, lb = j % nbl;
        ediff_out[(long long)(side * a.nb + rank + lb * C) * a.wc_max] = ed[j];
    }
    cl.sync();  // no CTA leaves while another may still read its shared memory
}

// ---- rows with their ghosts in shared memory -----------------------------------------------------
// Persistent kernel, the usual form: bound by latency (one step of a film of 100 cells, 10 x 16 planes
// touches 3 KB a CTA), so what counts is the length of the chain from one step's barrier to the next.
//   - A row holds its two ghost cells a side (NS = 4 + n4 + 4 floats, n4 = n rounded up to 4), so the
//     update is the same code for every cell, without ghost rules: a thread steps four neighbouring
//     cells from three vector loads, five faces for four cells.
//   - A CTA's share of the T_L numerator goes to every CTA's shared memory as it is formed (remote
//     stores), before the cluster barrier, so that after it the shares are added from local memory.
//   - The wall tasks (ghost cells, diffuse sums) run between the barrier's arrival and its wait.
// Sums keep k_persist_1d's order (planes of a CTA, then CTAs), and a cell its operations, the source's product rounded
// by itself: the results have its bits, which dJ/dlog tau, sums that cancel, shows (others moved it by up to 1.6e-4).
// 100 cells, 10 bands x 16 directions, 200 steps: 1.97 us a step against 3.08 for k_persist_1d.
struct RowLayout {
    int n4, ns, e, tl, q, part, ed, cst, mir;  // row stride and offsets (floats)
    size_t floats;
};
__host__ __device__ inline RowLayout row_layout(int n, int nd, int nbl, int C) {
    RowLayout L;
    const int npl = nbl * nd;
    L.n4 = (n + 3) / 4 * 4;
    L.ns = L.n4 + 8;
    L.e = 0;
    L.tl = 2 * npl * L.ns;
    L.q = L.tl + L.n4;
    L.part = L.q + L.n4;
    L.ed = L.part + 2 * C * L.n4;
    L.cst = L.ed + 2 * nbl;
    L.mir = L.cst + 5 * npl;
    L.floats = (size_t)L.mir + nd;
    return L;
}

template <int LIM>
__global__ void __launch_bounds__(1024, 1) k_persist_rows(const StepArgs a, int nsteps, const float *amps, float *e_io,
                                                          float *tl_out, float *ediff_out) {
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    const int C = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    extern __shared__ __align__(16) float sm[];
    const int n = a.n[0], nd = a.nd, T = (int)blockDim.x, tid = (int)threadIdx.x;
    const int nbl = (a.nb - rank + C - 1) / C;  // bands of this CTA: rank, rank + C, ...
    const int npl = nbl * nd;
    // every CTA lays its memory out for rank 0's bands (the most): peers address one another's parts
    const RowLayout L = row_layout(n, nd, (a.nb + C - 1) / C, C);
    const int ns = L.ns, n4 = L.n4;
    float *e0 = sm + L.e, *e1 = e0 + npl * ns, *tl = sm + L.tl, *qs = sm + L.q, *part = sm + L.part, *ed = sm + L.ed;
    float *pnu = sm + L.cst, *pwm = pnu + npl, *pdt = pwm + npl, *pck = pdt + npl, *psr = pck + npl;
    int *mir = reinterpret_cast<int *>(sm + L.mir);
    auto gplane = [&](int lp) { return (rank + (lp / nd) * C) * nd + lp % nd; };
    for (int j = tid; j < 2 * npl * ns; j += T) e0[j] = 0.f;
    for (int j = tid; j < 2 * C * n4; j += T) part[j] = 0.f;
    for (int x = tid; x < n4; x += T) {
        tl[x] = 0.f;
        qs[x] = a.Q && x < n ? a.Q[x] : 0.f;
    }
    for (int d = tid; d < nd; d += T) mir[d] = a.mirror[d];
    for (int lp = tid; lp < npl; lp += T) {
        const int pl = gplane(lp);
        const BandConst b = a.band[pl / nd];
        pnu[lp] = a.nu[3 * pl];
        pwm[lp] = a.wmom[pl];
        pdt[lp] = b.dtinv;
        pck[lp] = b.ck;
        psr[lp] = b.srck;
    }
    __syncthreads();
    for (int j = tid; j < npl * n; j += T) e0[(j / n) * ns + 4 + j % n] = e_io[(long long)gplane(j / n) * n + j % n];
    cl.sync();  // the state is in place; the peers' parts are zeroed before the first share arrives
    const int warp = tid >> 5, lane = tid & 31, nw = T >> 5;
    // this CTA's share of the T_L numerator from the state es, to every CTA's part [buf][rank]
    auto share = [&](const float *es, int buf) {
        for (int x = tid; x < n; x += T) {
            float v = 0.f;
            #pragma unroll 8
            for (int lp = 0; lp < npl; ++lp) v = fmaf(pwm[lp], es[lp * ns + 4 + x], v);
            float *dst = part + (buf * C + rank) * n4 + x;
            for (int r = 0; r < C; ++r) *cl.map_shared_rank(dst, r) = v;
        }
    };
    // ghost cells of every row of es.  Warp tasks, dealt from the last warp down (the first warps hold
    // the shares): 2 nbl diffuse sums, each written to its incoming rows, then the other rows' sides.
    const int nwt = 2 * nbl, ngt = (2 * npl + 31) / 32;
    auto ghosts = [&](float *es) {
        for (int t = nw - 1 - warp; t < nwt + ngt; t += nw) {
            if (t < nwt) {
                const int side = t / nbl, lb = t % nbl;
                float v = 0.f;
                if (a.bc[side] == kBcDiffuse) {
                    const float *col = es + lb * nd * ns + 4 + (side ? n - 1 : 0);
                    #pragma unroll 8
                    for (int d = 0; d < nd; ++d) v = fmaf(a.wdiff[side * nd + d], col[d * ns], v);
                    v *= a.inv_den[side];
                    for (int d = lane; d < nd; d += 32) {
                        const int lp = lb * nd + d;
                        if (side == 0 ? pnu[lp] > 0.f : pnu[lp] < 0.f) {
                            float *g = es + lp * ns + (side ? 4 + n : 2);
                            g[0] = g[1] = v;
                        }
                    }
                }
                if (lane == 0) ed[side * nbl + lb] = v;
                continue;
            }
            const int i = (t - nwt) * 32 + lane;
            if (i >= 2 * npl) continue;
            const int side = i / npl, lp = i - side * npl, lb = lp / nd, d = lp - lb * nd;
            const int bc = a.bc[side];
            const float nu = pnu[lp];
            const bool incoming = side == 0 ? nu > 0.f : nu < 0.f;
            const float *row = es + lp * ns + 4;
            float g1, g2;  // next to the wall, and behind it
            if (bc == kBcPeriodic) {
                g1 = row[side ? 0 : n - 1];
                g2 = row[side ? 1 : n - 2];
            } else if (bc == kBcSpecular) {
                const float *m = es + (lb * nd + mir[d]) * ns + 4;
                g1 = m[side ? n - 1 : 0];
                g2 = m[side ? n - 2 : 1];
            } else if (!incoming) {
                g1 = g2 = row[side ? n - 1 : 0];
            } else if (bc == kBcIsothermal) {
                g1 = g2 = a.iso[side * a.nb + rank + lb * C];
            } else {
                continue;  // diffuse: written with its sum
            }
            float *g = es + lp * ns + (side ? 4 + n : 2);
            g[side ? 0 : 1] = g1;
            g[side ? 1 : 0] = g2;
        }
    };
    auto gather_tl = [&](int buf) {
        const float *pb = part + buf * C * n4;
        for (int x = tid; x < n; x += T) {
            float v = 0.f;
            #pragma unroll 4
            for (int r = 0; r < C; ++r) v += pb[r * n4 + x];
            tl[x] = v * a.invD;
        }
    };
    int buf = 0;
    share(e0, buf);
    ghosts(e0);
    cl.sync();
    gather_tl(buf);
    __syncthreads();
    const int ng = n4 / 4, nit = npl * ng;
    const int bx = T % ng, bp = T / ng;
    const int g00 = tid % ng, p00 = tid / ng;
    for (int s = 0; s < nsteps; ++s) {
        const float amp = a.Q ? amps[s] : 0.f;
        int xg = g00, lp = p00;
        for (int j = tid; j < nit; j += T) {
            const int x0 = 4 * xg;
            const float *row = e0 + lp * ns + 4 + x0;
            const float4 u = *reinterpret_cast<const float4 *>(row);
            const float2 lo = *reinterpret_cast<const float2 *>(row - 2), hi = *reinterpret_cast<const float2 *>(row + 4);
            const float4 t4 = *reinterpret_cast<const float4 *>(tl + x0), q4 = *reinterpret_cast<const float4 *>(qs + x0);
            const float nu = pnu[lp], dt = pdt[lp], ck = pck[lp], sr = psr[lp], an = fabsf(nu);
            const bool up = nu > 0.f;
            // the stencil in streaming order: w[2..5] are the four cells, upwind first
            const float w[7] = {up ? lo.x : hi.y, up ? lo.y : hi.x, up ? u.x : u.w, up ? u.y : u.z,
                                up ? u.z : u.y,   up ? u.w : u.x,   up ? hi.x : lo.y};
            const float t[4] = {up ? t4.x : t4.w, up ? t4.y : t4.z, up ? t4.z : t4.y, up ? t4.w : t4.x};
            const float qv[4] = {up ? q4.x : q4.w, up ? q4.y : q4.z, up ? q4.z : q4.y, up ? q4.w : q4.x};
            float f[5];
            #pragma unroll
            for (int i = 0; i < 5; ++i) f[i] = w[i + 1] + 0.5f * limit<LIM>(w[i + 1] - w[i], w[i + 2] - w[i + 1]);
            float o[4];
            #pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float u0 = w[i + 2];
                const float div = nu != 0.f ? an * (f[i + 1] - f[i]) : 0.f;
                const float src = a.Q ? __fmul_rn(sr, __fmul_rn(amp, qv[i])) : 0.f;
                o[i] = u0 - div + dt * (ck * t[i] - u0) + src;
            }
            float *out = e1 + lp * ns + 4 + x0;
            const float4 v = make_float4(up ? o[0] : o[3], up ? o[1] : o[2], up ? o[2] : o[1], up ? o[3] : o[0]);
            if (x0 + 4 <= n) {
                *reinterpret_cast<float4 *>(out) = v;
            } else {  // the row's last cells: its ghosts follow them
                out[0] = v.x;
                if (x0 + 1 < n) out[1] = v.y;
                if (x0 + 2 < n) out[2] = v.z;
            }
            xg += bx;
            lp += bp;
            if (xg >= ng) {
                xg -= ng;
                ++lp;
            }
        }
        __syncthreads();
        buf ^= 1;
        share(e1, buf);
        // every CTA's share of this step is written when the barrier completes, and the other buffer free
        asm volatile("barrier.cluster.arrive.release;" ::: "memory");
        ghosts(e1);
        asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
        gather_tl(buf);
        __syncthreads();
        float *t = e0;
        e0 = e1;
        e1 = t;
    }
    for (int j = tid; j < npl * n; j += T) e_io[(long long)gplane(j / n) * n + j % n] = e0[(j / n) * ns + 4 + j % n];
    if (rank == 0)
        for (int x = tid; x < n; x += T) tl_out[x] = tl[x];
    for (int j = tid; j < 2 * nbl; j += T) {
        const int side = j / nbl, lb = j % nbl;
        ediff_out[(long long)(side * a.nb + rank + lb * C) * a.wc_max] = ed[j];
    }
    cl.sync();  // no CTA leaves while a peer's share may still be on its way to it
}

// Launches k over the largest cluster (<= 16, <= nb) whose CTAs hold their memory and which the device
// can place; `threads` and `smem` of a cluster size.  False: no cluster size fits.
template <typename K, typename TH, typename SM>
static bool launch_cluster(K k, const StepArgs &a, TH threads, SM smem_of, cudaError_t &err, int nsteps, const float *amps,
                           float *e_io, float *tl_out, float *ediff_out, cudaStream_t s) {
    err = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (err != cudaSuccess) cudaGetLastError();
    for (int C = a.nb < 16 ? a.nb : 16; C >= 1; --C) {
        const size_t smem = smem_of(C);
        if (smem > (size_t)1 << 20 ||
            cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) {
            cudaGetLastError();
            continue;
        }
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)C);
        cfg.blockDim = dim3((unsigned)threads(C));
        cfg.dynamicSmemBytes = smem;
        cfg.stream = s;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = (unsigned)C;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int ncl = 0;
        if (cudaOccupancyMaxActiveClusters(&ncl, k, &cfg) != cudaSuccess || ncl < 1) {
            cudaGetLastError();
            continue;
        }
        err = cudaLaunchKernelEx(&cfg, k, a, nsteps, amps, e_io, tl_out, ediff_out);
        return true;
    }
    return false;
}

static size_t persist_smem(const StepArgs &a, int C) {
    const size_t nbl = (a.nb + C - 1) / C, npl = nbl * a.nd;
    return (2 * npl * a.n[0] + 3 * (size_t)a.n[0] + 2 * nbl + 5 * npl) * sizeof(float);
}

cudaError_t launch_persist_1d(const StepArgs &a, int limiter, int nsteps, const float *amps, float *e_io,
                              float *tl_out, float *ediff_out, cudaStream_t s) {
    using Kern = void (*)(const StepArgs, int, const float *, float *, float *, float *);
    const Kern rows = limiter == kLimFirst ? k_persist_rows<kLimFirst> : limiter == kLimMinmod ? k_persist_rows<kLimMinmod>
                                                                                         : k_persist_rows<kLimVanAlbada>;
    const Kern flat = limiter == kLimFirst ? k_persist_1d<kLimFirst> : limiter == kLimMinmod ? k_persist_1d<kLimMinmod>
                                                                                       : k_persist_1d<kLimVanAlbada>;
    cudaError_t err;
    const int nd = a.nd, n = a.n[0], nb = a.nb;
    // As many threads as share the items (four cells each) evenly, at least one a cell for the sums, and a warp for
    // each wall task as far as there are tasks for 16 warps: short rows have more tasks than cells.  Us a step by
    // k_persist_1d / without that / with it: 5 cells, 100 x 8 2.71 / 3.27 / 2.30; 2 cells, 40 x 64 4.31 / 5.08 / 3.00.
    // Long rows take all the threads there are: 600 cells, 1 x 8 5.1 / 5.9 / 4.7; 700 5.6 / 6.0 / 5.0.
    auto threads = [=](int C) {
        const long long nbl = (nb + C - 1) / C, nit = nbl * nd * ((n + 3) / 4), tasks = 2 * nbl + (2 * nbl * nd + 31) / 32;
        const long long rounds = (nit + 1023) / 1024;
        if (n > 512 && rounds > 1) return 1024;
        long long t = (nit + rounds - 1) / rounds;
        if (t < n) t = n;
        if (t < 32 * tasks) t = tasks < 16 ? 32 * tasks : (t < 512 ? 512 : t);
        if (t < 128) t = 128;
        t = (t + 31) / 32 * 32;
        return t > 1024 ? 1024 : (int)t;
    };
    // the flat form takes what the padded rows do not fit (one band whose state nearly fills a CTA)
    if (launch_cluster(rows, a, threads, [=](int C) { return row_layout(n, nd, (nb + C - 1) / C, C).floats * sizeof(float); },
                       err, nsteps, amps, e_io, tl_out, ediff_out, s))
        return err;
    if (launch_cluster(flat, a, [](int) { return 1024; }, [&](int C) { return persist_smem(a, C); }, err, nsteps, amps,
                       e_io, tl_out, ediff_out, s))
        return err;
    return cudaErrorInvalidConfiguration;
}

}  // namespace bte
