// Plan, dispatch and finalize pass of the register-streaming forward kernel
// (bte_stream_kernel.cuh).
#include <algorithm>
#include <climits>
#include <cstring>

#include "bte_stream_kernel.cuh"

namespace bte {

namespace stream {

// Finalize pass of a step: a block is 64 items by 4 groups; group g takes rows (or directions) g,
// g + 4, ... and group 0 adds the four sums in order, so the result is fixed for a given plan.
// The first tblocks blocks form T_L_i = (sum of the moment partials of cell i) / sum_k C_k/tau_k.
// The others form the diffuse-wall values, Eq. (diff_bound), from the stored state: sum over
// the leaving directions of w |s.n| e / sum_in w|s.n|.
// Bound by latency: kBatch loads are in flight together, the last ones too (a loop's remainder would wait for
// them one by one).  Grating (1000 cells, 512 directions, the
// same in k_finalize_1d): 9.5 -> 7.5 us a step.
constexpr int kItems = 64, kGroups = 4, kBatch = 8;

struct WallList {
    int n;
    int w[6];
    int first[7];  // first wall item (wall cell) of each wall, in multiples of kItems
};

__global__ void __launch_bounds__(kItems * kGroups) k_finalize_stream(const StepArgs a, int rows, int tblocks,
                                                                      const WallList wl, const float *state, float *TL_out) {
    __shared__ float part[kGroups][kItems];
    const int lane = threadIdx.x % kItems, grp = threadIdx.x / kItems;
    if ((int)blockIdx.x < tblocks) {
        const long long i = (long long)blockIdx.x * kItems + lane;
        float s = 0.f;
        if (i < a.ncell) {
            const float *P = a.P + i;
            for (int r = grp; r < rows; r += kBatch * kGroups) {
                float v[kBatch];
                #pragma unroll
                for (int m = 0; m < kBatch; ++m)
                    v[m] = r + m * kGroups < rows ? __ldcs(P + (long long)(r + m * kGroups) * a.ncell) : 0.f;
                #pragma unroll
                for (int m = 0; m < kBatch; ++m)
                    if (r + m * kGroups < rows) s += v[m];
            }
        }
        part[grp][lane] = s;
        __syncthreads();
        if (grp == 0 && i < a.ncell) {
            #pragma unroll
            for (int g = 1; g < kGroups; ++g) s += part[g][lane];
            TL_out[i] = s * a.invD;
        }
        return;
    }
    const int per_band = wl.first[wl.n] / kItems;
    const int b0 = blockIdx.x - tblocks, k = b0 / per_band;
    const int item = (b0 - k * per_band) * kItems;
    int wi = 0;
    while (item >= wl.first[wi + 1]) ++wi;
    const int wall = wl.w[wi], ax = wall >> 1, side = wall & 1;
    const int n0 = ax == 0 ? a.n[1] : a.n[0], n1 = ax == 2 ? a.n[1] : a.n[2];
    const int j = item - wl.first[wi] + lane;
    const bool valid = j < n0 * n1;
    float s = 0.f;
    if (valid) {
        const int ja = j % n0, jb = j / n0;
        const int x = ax == 0 ? (side ? a.n[0] - 1 : 0) : ja;
        const int y = ax == 0 ? ja : (ax == 1 ? (side ? a.n[1] - 1 : 0) : jb);
        const int z = ax == 2 ? (side ? a.n[2] - 1 : 0) : jb;
        const long long i = ((long long)z * a.n[1] + y) * a.n[0] + x;
        const float *e = state + (long long)k * a.nd * a.ncell + i;
        const float *wd = a.wdiff + wall * a.nd;
        for (int d = grp; d < a.nd; d += kBatch * kGroups) {
            float w[kBatch], v[kBatch];
            #pragma unroll
            for (int m = 0; m < kBatch; ++m) w[m] = d + m * kGroups < a.nd ? __ldg(wd + d + m * kGroups) : 0.f;
            #pragma unroll
            for (int m = 0; m < kBatch; ++m) v[m] = w[m] != 0.f ? e[(long long)(d + m * kGroups) * a.ncell] : 0.f;
            #pragma unroll
            for (int m = 0; m < kBatch; ++m)
                if (w[m] != 0.f) s = fmaf(w[m], v[m], s);
        }
    }
    part[grp][lane] = s;
    __syncthreads();
    if (grp == 0 && valid) {
        #pragma unroll
        for (int g = 1; g < kGroups; ++g) s += part[g][lane];
        static_cast<float *>(a.ediff_out)[((long long)wall * a.nb + k) * a.wc_max + j] = s * a.inv_den[wall];
    }
}

}  // namespace stream

using namespace stream;

bool stream_plan(int dim, const int n[3], int nb, int nd, const double *s, const int bc[6], const double jump[3], int storage,
                 int limiter, StreamPlan &plan, std::string &why) {
    plan = StreamPlan();
    if (dim < 2 || storage != kStoreF32) {
        why = "the streaming kernel takes 2-D and 3-D grids with FP32 states";
        return false;
    }
    const long long ncell = (long long)n[0] * n[1] * n[2];
    if (ncell > INT_MAX / 4 || 6LL * nb * (ncell / std::min(n[0], dim > 2 ? std::min(n[1], n[2]) : n[1]) + 8) > INT_MAX) {
        why = "the streaming kernel indexes the cells of a plane and of the walls with 32 bits";
        return false;
    }
    plan.dim = dim;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        cudaGetLastError();
        why = "no CUDA device";
        return false;
    }
    // rows a thread: fewer where the grid has fewer rows, or where all directions of all bands would not
    // give every SM a few blocks
    plan.kr = n[1] < kRows || ncell * nb * nd < 2LL * kRows * kThreads * 4 * sms ? kRowsSmall : kRows;
    plan.nys = (n[1] + plan.kr - 1) / plan.kr;
    plan.nz = n[2];
    plan.G = (n[0] + 1) / 2;
    for (int a = 0; a < dim; ++a)
        if (jump[a] != 0.0) plan.jump |= 1 << a;
    plan.E = std::min(plan.G, n[0] % 2 ? 3 : 2);  // the last group of an odd row overlaps the one before it
    const long long strips = (long long)plan.nys * plan.nz;
    if (strips * plan.G > INT_MAX) {
        why = "too many strips";
        return false;
    }
    // strips that touch a y or z wall whose ghosts are more than wrapped rows
    auto walled = [&](int a) { return a < dim && (bc[2 * a] != kBcPeriodic || jump[a] != 0.0); };
    std::vector<int> rest;
    for (int ys = 0; ys < plan.nys; ++ys)
        for (int z = 0; z < plan.nz; ++z) {
            const bool sp = dim == 3 && ((walled(1) && (ys == 0 || (ys + 1) * plan.kr >= n[1])) ||
                                         (walled(2) && (z < 2 || z >= plan.nz - 2)));
            (sp ? plan.h_strips : rest).push_back(ys * plan.nz + z);
        }
    plan.nspecial = (int)plan.h_strips.size();
    plan.h_strips.insert(plan.h_strips.end(), rest.begin(), rest.end());
    auto nblk = [](long long threads) { return (int)((threads + kThreads - 1) / kThreads); };
    plan.blocks[0] = nblk(strips * plan.E);
    plan.blocks[1] = nblk((long long)plan.nspecial * (plan.G - plan.E));
    plan.blocks[2] = nblk((strips - plan.nspecial) * (plan.G - plan.E));
    const long long blocks = (long long)plan.blocks[0] + plan.blocks[1] + plan.blocks[2];
    plan.mixed = dim == 3;
    // Parts of a band's directions: enough blocks to fill the GPU many times over (in 3-D also short ones,
    // so that the slow blocks leave no tail), but no more than a row of moment partials (4 bytes a cell
    // written and read) for every 12 directions where the blocks suffice, 4 where they then give every SM 8.
    const long long have = blocks * nb, want = (dim == 3 ? 64LL : 16LL) * sms, least = 4LL * sms;
    int nc = 1;
    while (have * nc < want && nd / (2 * nc) >= 12) nc *= 2;
    while (have * nc < 2 * least && nd / (2 * nc) >= 4) nc *= 2;
    while (have * nc < least && nc < nd) nc *= 2;
    plan.nchunk = nc = std::min(nc, nd);
    if (blocks * nb * nc > INT_MAX) {
        why = "too many blocks";
        return false;
    }
    // directions in the order of their signs
    plan.h_dord.resize(nd);
    for (int d = 0; d < nd; ++d) plan.h_dord[d] = d;
    auto key = [&](int d) {
        int q = 0;
        for (int a = dim - 1; a >= 0; --a) q = 2 * q + (s[3 * d + a] < 0.0 ? 1 : 0);
        return q;
    };
    std::stable_sort(plan.h_dord.begin(), plan.h_dord.end(), [&](int u, int v) { return key(u) < key(v); });
    plan.kernel = (void *)(dim == 2 ? pick_2d(limiter, n[0] % 2 == 0, plan.kr) : pick_3d(limiter, n[0] % 2 == 0, plan.kr));
    plan.valid = 1;
    return true;
}

bool stream_setup(StreamPlan &plan, std::string &why) {
    auto up = [](int **d, const std::vector<int> &h) {
        return cudaMalloc((void **)d, h.size() * sizeof(int)) == cudaSuccess &&
               cudaMemcpy(*d, h.data(), h.size() * sizeof(int), cudaMemcpyHostToDevice) == cudaSuccess;
    };
    if (!up(&plan.dord, plan.h_dord) || !up(&plan.strips, plan.h_strips)) {
        cudaGetLastError();
        why = "cudaMalloc failed";
        return false;
    }
    return true;
}

void stream_free(StreamPlan &plan) {
    if (plan.dord) cudaFree(plan.dord);
    if (plan.strips) cudaFree(plan.strips);
    plan.dord = plan.strips = nullptr;
}

cudaError_t launch_step_stream(const StepArgs &a, const StreamPlan &plan, cudaStream_t s) {
    StreamArgs p;
    p.dord = plan.dord;
    p.nchunk = plan.nchunk;
    p.nys = plan.nys;
    p.nz = plan.nz;
    p.G = plan.G;
    p.E = plan.E;
    p.strips = plan.strips;
    p.nspecial = plan.nspecial;
    p.mixed = plan.mixed;
    for (int c = 0; c < 3; ++c) p.blocks[c] = plan.blocks[c];
    p.jump = plan.jump;
    const unsigned blocks = (unsigned)(plan.blocks[0] + plan.blocks[1] + plan.blocks[2]) * (unsigned)(a.nb * plan.nchunk);
    ((StreamKernel)plan.kernel)<<<blocks, kThreads, 0, s>>>(a, p);
    return cudaGetLastError();
}

cudaError_t launch_finalize_stream(const StepArgs &a, const StreamPlan &plan, float *TL_out, cudaStream_t s) {
    WallList wl;
    wl.n = 0;
    wl.first[0] = 0;
    for (int w = 0; w < 2 * a.dim; ++w) {
        if (a.bc[w] != kBcDiffuse) continue;
        const int cells = (int)(a.ncell / a.n[w >> 1]);
        wl.w[wl.n] = w;
        wl.first[wl.n + 1] = wl.first[wl.n] + (cells + kItems - 1) / kItems * kItems;
        ++wl.n;
    }
    const int tblocks = (int)((a.ncell + kItems - 1) / kItems);
    const unsigned blocks = (unsigned)tblocks + (unsigned)(wl.first[wl.n] / kItems) * (unsigned)a.nb;
    k_finalize_stream<<<blocks, kItems * kGroups, 0, s>>>(a, a.nb * plan.nchunk, tblocks, wl,
                                                           static_cast<const float *>(a.e_out), TL_out);
    return cudaGetLastError();
}

}  // namespace bte
