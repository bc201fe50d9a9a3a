// Register-streaming forward kernel of the explicit DOM step for 2-D and 3-D grids of any shape, FP32 states:
// launch interface (the kernel is described in bte_stream_kernel.cuh).
#pragma once

#include <string>
#include <vector>

#include "bte_internal.h"

namespace bte {

// Device-side view of the plan, passed by value.
struct StreamArgs {
    const int *dord;  // [nd] directions ordered by the signs of their components
    int nchunk;       // parts of dord; part c of band k writes row k nchunk + c of the moment partials
    int nys, nz;      // strips of KR rows a slice, slices
    int G, E;         // groups of two cells a row, of which E next to an x wall
    const int *strips;  // [nys nz] strips ys nz + z, the nspecial next to a y or z wall first
    int nspecial;
    int blocks[3];    // blocks a (band, part): groups next to an x wall, the other groups of the
                      // special strips, the rest
    int mixed;        // the slow blocks spread among the others, else first
    int jump;         // bit a: a periodic temperature jump on axis a
};

struct StreamPlan {
    int valid = 0;
    int dim = 0;
    int kr = 1, nchunk = 1;
    int nys = 1, nz = 1, G = 0, E = 0, nspecial = 0, mixed = 0, blocks[3] = {0, 0, 0};
    int jump = 0;
    void *kernel = nullptr;
    int *dord = nullptr, *strips = nullptr;
    std::vector<int> h_dord, h_strips;
};

// Strip shape, direction order and launch shape (queries the current device for its SM count).
// s: [nd][3] directions.  false + reason where the kernel does not apply.
bool stream_plan(int dim, const int n[3], int nb, int nd, const double *s, const int bc[6], const double jump[3], int storage,
                 int limiter, StreamPlan &plan, std::string &why);
bool stream_setup(StreamPlan &plan, std::string &why);
void stream_free(StreamPlan &plan);
cudaError_t launch_step_stream(const StepArgs &a, const StreamPlan &plan, cudaStream_t s);
// T_L from the rows of moment partials and the diffuse-wall values (a.ediff_out) of the state it wrote, in one
// launch.
cudaError_t launch_finalize_stream(const StepArgs &a, const StreamPlan &plan, float *TL_out, cudaStream_t s);

}  // namespace bte
