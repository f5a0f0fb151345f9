// The fused 3-D kernel (jacobi3d_fused.cu) as jacobi3d.cu launches it.
#pragma once

#include "runtime.h"

namespace sdfg {

struct J3FGeo {
    int D, R, C, ld;
    long long plane;        // plane pitch (elements) = R * ld
    int tiles_x, tiles_y;   // tiles per plane
    int zseg, n_zseg;       // planes per CTA, CTAs along z
};

constexpr int J3F_MAX_K = 3;  // fused steps per launch: 2 or 3
int j3_fused_rows(int K);     // TMA box
int j3_fused_cols();
J3FGeo j3_fused_plan(int K, int D, int R, int C, int ld, int dtype, int sm_count);
// K steps, interior points only; dst holds the shell already.
int launch_j3_fused(const CUtensorMap &tm, void *dst, const J3FGeo &g, int K, int dtype, int *err, cudaStream_t s);
// The shell of box src into d0 and, unless null, d1.
int j3_shell_copy(const void *src, void *d0, void *d1, int D, int R, int C, int ld, int dtype, cudaStream_t s);

}  // namespace sdfg
