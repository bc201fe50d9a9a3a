// Steady state by the implicit discrete-ordinates method, sequential iterative scheme
// (Sec. 3.3-3.5 of arXiv 2306.14181, Eq. disretized_BTE in delta form).
//
// One iteration: the forward step computes e^n + dt R (R: the steady equation's right-hand side
// with the step's limited second-order faces, walls and source), then this sweep solves, for
// every band k and direction d, the first-order upwind system of the increment
//     (dt/tau_k + sum_a |nu_a|) De_i - sum_a |nu_a| De_{up_a(i)} = dt R_i,
// nu_a = dt v_k s_{d,a} / h_a being the step's own Courant numbers and up_a(i) the upwind
// neighbour of cell i along axis a; across a wall (periodic pairs included) the upwind De is 0,
// so each plane's system is lower triangular in upwind order and one sweep solves it:
// z, y and x each run from the upwind side.
//
// One warp a plane.  A row is cut into chunks of 128 cells in upwind order, 4 consecutive cells
// a lane.  Along x the recurrence De_u = a_u + b De_{u-1} (b = |nu_x| / diag, a_u the cell's
// right-hand side with its y and z upwind terms, over diag) is a composition of affine maps:
// each lane folds its 4 cells into one map, a warp scan of maps (Kogge-Stone, 5 shuffle steps)
// gives every lane the De entering its cells, and the lanes then run their 4 cells again.  The
// y upwind De is the previous row's, kept in registers for rows of up to CH chunks; the z upwind
// De (3-D) is read back from the slice the same lane wrote before (e_io - e_in at the same x), so a
// lane only ever reads its own stores.
//
// Bound by latency along a row and by the memory of the 33 warps an SM that the hot spot's 5120 planes
// give: the next row's (longer rows: the next chunk's) own values are loaded, 16 bytes a lane where rows allow,
// before this row's scan, and a row's z values with them.
// An iteration on 256^2, 40 x 128: 2.41 -> 1.54 ms with this and k_moment_rows (the sweep alone was 1.11
// ms with the y term read back and no loads ahead).  Few planes, us an iteration without the loads ahead of long
// rows and of the z values / with them: 20001 cells, 2 x 64 216 / 140; 130 x 16 x 16, 3 x 48 522 / 342, 20 x 96 1102 /
// 878; 100^2, 1 x 8 93 / 79.
#include <cuda_runtime.h>

#include "bte_internal.h"

namespace bte {
namespace {

constexpr int kSweepWarps = 4;
constexpr int kCellsPerLane = 4;

// Chunks of a row held in registers: rows of up to CH * 128 cells (CH = 0: any length, the y term read
// back like the z term).  VEC: rows are multiples of four cells, which move 16 bytes a lane.  Z: 3-D, whose z values
// take registers of their own, on their way together with the next loads.
template <int CH, bool VEC, bool Z>
__global__ void __launch_bounds__(kSweepWarps * 32, Z ? 6 : 9) k_sis_sweep(const StepArgs a, const float *__restrict__ e_in,
                                                                           float *e_io) {
    const int lane = threadIdx.x & 31;
    const long long plane = (long long)blockIdx.x * kSweepWarps + (threadIdx.x >> 5);
    if (plane >= (long long)a.nb * a.nd) return;
    const int k = (int)(plane / a.nd);
    const int nx = a.n[0], ny = a.n[1], nz = a.n[2];
    const float nux = fabsf(a.nu[3 * plane]), nuy = fabsf(a.nu[3 * plane + 1]), nuz = fabsf(a.nu[3 * plane + 2]);
    const int sx = a.nu[3 * plane] >= 0.f ? 1 : -1;
    const int sy = a.nu[3 * plane + 1] >= 0.f ? 1 : -1;
    const int sz = a.nu[3 * plane + 2] >= 0.f ? 1 : -1;
    const float diag = a.band[k].dtinv + nux + nuy + nuz;
    const float inv = 1.f / diag;
    const float b = nux * inv;
    const float *ei = e_in + plane * a.ncell;
    float *eo = e_io + plane * a.ncell;
    const long long dyg = (long long)sy * nx, dzg = (long long)sz * nx * ny;
    constexpr int NC = CH > 0 ? CH : 1, V = kCellsPerLane;
    // this lane's cells of chunk c of a row, upwind order: x of the first and how many lie in the row
    auto xof = [&](int u) { return sx > 0 ? u : nx - 1 - u; };
    auto load = [&](long long row, int u0, float (&vo)[V], float (&vi)[V]) {
        const int u = u0 + lane * V;
        if constexpr (VEC) {
            if (u < nx) {
                const long long i = row + (sx > 0 ? u : nx - V - u);
                const float4 o = *reinterpret_cast<const float4 *>(eo + i), q = *reinterpret_cast<const float4 *>(ei + i);
                vo[0] = sx > 0 ? o.x : o.w; vo[1] = sx > 0 ? o.y : o.z; vo[2] = sx > 0 ? o.z : o.y; vo[3] = sx > 0 ? o.w : o.x;
                vi[0] = sx > 0 ? q.x : q.w; vi[1] = sx > 0 ? q.y : q.z; vi[2] = sx > 0 ? q.z : q.y; vi[3] = sx > 0 ? q.w : q.x;
            }
        } else {
            #pragma unroll
            for (int v = 0; v < V; ++v)
                if (u + v < nx) {
                    const long long i = row + xof(u + v);
                    vo[v] = eo[i];
                    vi[v] = ei[i];
                }
        }
    };
    // the next chunks' values; De of the row upwind in y (CH = 0: its stored values dp and yi)
    float no[NC][V], ni[NC][V], dp[NC][V], yi[V];
    #pragma unroll
    for (int c = 0; c < NC; ++c)
        #pragma unroll
        for (int v = 0; v < V; ++v) no[c][v] = ni[c][v] = dp[c][v] = yi[v] = 0.f;
    auto row_of = [&](int uz, int uy) {
        return ((long long)(sz > 0 ? uz : nz - 1 - uz) * ny + (sy > 0 ? uy : ny - 1 - uy)) * nx;
    };
    #pragma unroll
    for (int c = 0; c < NC; ++c) load(row_of(0, 0), c * 32 * V, no[c], ni[c]);
    for (int uz = 0; uz < nz; ++uz) {
        for (int uy = 0; uy < ny; ++uy) {
            const long long row = row_of(uz, uy);
            float carry = 0.f;  // De of the cell before the chunk (0 at the upwind wall)
            const int nch = CH > 0 ? CH : (nx + 32 * V - 1) / (32 * V);
            const int my = uy + 1 < ny ? uy + 1 : 0, mz = uy + 1 < ny ? uz : uz + 1;  // the next row
            float av[NC][V], vi[NC][V];
            // right-hand sides of the NC chunks at c0, their z term in step with the next chunks' loads
            auto rhs = [&](int c0) {
                float zo[NC][V], zi[NC][V];
                if constexpr (Z) {
                    if (uz > 0) {
                        #pragma unroll
                        for (int c = 0; c < NC; ++c) load(row - dzg, (c0 + c) * 32 * V, zo[c], zi[c]);
                    }
                }
                if constexpr (CH == 0) {
                    if (uy > 0) load(row - dyg, c0 * 32 * V, dp[0], yi);
                }
                #pragma unroll
                for (int c = 0; c < NC; ++c)
                    #pragma unroll
                    for (int v = 0; v < V; ++v) {
                        vi[c][v] = ni[c][v];
                        av[c][v] = no[c][v] - ni[c][v];  // dt R
                    }
                const bool last = c0 + NC >= nch;
                if (!last || mz < nz) {
                    #pragma unroll
                    for (int c = 0; c < NC; ++c) load(last ? row_of(mz, my) : row, last ? c * 32 * V : (c0 + 1) * 32 * V, no[c], ni[c]);
                }
                #pragma unroll
                for (int c = 0; c < NC; ++c)
                    #pragma unroll
                    for (int v = 0; v < V; ++v) {
                        if (uy > 0) av[c][v] = fmaf(nuy, CH > 0 ? dp[c][v] : dp[c][v] - yi[v], av[c][v]);
                        if (Z && uz > 0) av[c][v] = fmaf(nuz, zo[c][v] - zi[c][v], av[c][v]);
                    }
            };
            if constexpr (CH > 0) rhs(0);
            #pragma unroll(NC)
            for (int c = 0; c < nch; ++c) {
                if constexpr (CH == 0) rhs(c);
                const int q = CH > 0 ? c : 0;
                const int u = c * 32 * V + lane * V;
                // the lane's map De_out = A + B De_in over its cells of the row
                float A = 0.f, B = 1.f;
                #pragma unroll
                for (int v = 0; v < V; ++v) {
                    const bool in = u + v < nx;
                    av[q][v] *= inv;
                    A = in ? fmaf(b, A, av[q][v]) : A;
                    B = in ? B * b : B;
                }
                // inclusive scan of the maps over the lanes: lane l composes lanes 0..l
                #pragma unroll
                for (int off = 1; off < 32; off <<= 1) {
                    const float Au = __shfl_up_sync(0xffffffffu, A, off);
                    const float Bu = __shfl_up_sync(0xffffffffu, B, off);
                    if (lane >= off) {
                        A = fmaf(B, Au, A);
                        B *= Bu;
                    }
                }
                const float Ain = __shfl_up_sync(0xffffffffu, A, 1);
                const float Bin = __shfl_up_sync(0xffffffffu, B, 1);
                float d = lane == 0 ? carry : fmaf(Bin, carry, Ain);
                float out[V];
                #pragma unroll
                for (int v = 0; v < V; ++v) {
                    d = fmaf(b, d, av[q][v]);
                    // De as the stored values give it, which is what the next row's reads gave
                    out[v] = vi[q][v] + d;
                    if constexpr (CH > 0) dp[q][v] = out[v] - vi[q][v];
                }
                if constexpr (VEC) {
                    if (u < nx)
                        *reinterpret_cast<float4 *>(eo + row + (sx > 0 ? u : nx - V - u)) =
                            sx > 0 ? make_float4(out[0], out[1], out[2], out[3]) : make_float4(out[3], out[2], out[1], out[0]);
                } else {
                    #pragma unroll
                    for (int v = 0; v < V; ++v)
                        if (u + v < nx) eo[row + xof(u + v)] = out[v];
                }
                // De of the chunk's last cell: the composed map of all 32 lanes applied to carry
                carry = __shfl_sync(0xffffffffu, fmaf(B, carry, A), 31);
            }
        }
    }
}

template <bool VEC, bool Z>
void launch_sweep(const StepArgs &a, const float *e_in, float *e_io, unsigned blocks, cudaStream_t s) {
    const int chunks = (a.n[0] + 127) / 128;
    if (chunks == 1) k_sis_sweep<1, VEC, Z><<<blocks, kSweepWarps * 32, 0, s>>>(a, e_in, e_io);
    else if (chunks == 2) k_sis_sweep<2, VEC, Z><<<blocks, kSweepWarps * 32, 0, s>>>(a, e_in, e_io);
    else k_sis_sweep<0, VEC, Z><<<blocks, kSweepWarps * 32, 0, s>>>(a, e_in, e_io);
}

}  // namespace

cudaError_t launch_sis_sweep(const StepArgs &a, const float *e_in, float *e_io, cudaStream_t s) {
    const long long planes = (long long)a.nb * a.nd;
    const unsigned blocks = (unsigned)((planes + kSweepWarps - 1) / kSweepWarps);
    const bool vec = a.n[0] % kCellsPerLane == 0;
    if (a.n[2] > 1) {
        if (vec) launch_sweep<true, true>(a, e_in, e_io, blocks, s);
        else launch_sweep<false, true>(a, e_in, e_io, blocks, s);
    } else {
        if (vec) launch_sweep<true, false>(a, e_in, e_io, blocks, s);
        else launch_sweep<false, false>(a, e_in, e_io, blocks, s);
    }
    return cudaGetLastError();
}

}  // namespace bte
