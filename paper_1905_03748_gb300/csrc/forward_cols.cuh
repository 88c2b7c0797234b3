// The column projector (forward_cols.cu).
#pragma once

#include "common.cuh"

namespace tigre {

// Column quads of a whole volume: element (y, x, s), s fastest, of the
// zero-bordered volume (padded_elems of them).
template <typename T>
tigre_status build_quad_columns(const tigre_geometry_desc& d, const T* vol, float4* out,
                                cudaStream_t st);
// The angles of a launch's blocks: with `four`, block row i projects the angles
// table[4 i .. 4 i + 3] (relative to the launch's first one, -1 for none), or
// with a null table 4 i .. 4 i + 3 themselves; otherwise angle i alone.
struct ColGroups {
    bool four;
    const int* table;
    int64_t count;
};
// Projection of the angles [a_first, a_first + na).  A batch's members lie
// vol_stride quads and proj_stride elements apart.
template <typename TP>
tigre_status launch_forward_columns(tigre_geometry* g, const float4* quads, TP* proj, int a_first,
                                    int64_t na, const ColGroups& groups, int batch,
                                    int64_t vol_stride, int64_t proj_stride, cudaStream_t st);

// Exact transpose of the projection of the angles [a0, a0 + na) (adjoint_cols.cu)
// through padded_elems accumulator quads, zeroed by the caller.
template <typename TP, typename TV>
tigre_status launch_adjoint_columns(tigre_geometry* g, const TP* proj, float4* acc, TV* vol,
                                    int64_t a0, int64_t na, cudaStream_t st);

// Whether warps of detector rows suit a call of na angles (forward.cu).
bool column_warps_pay(const tigre_geometry* g, int64_t na);

}  // namespace tigre
