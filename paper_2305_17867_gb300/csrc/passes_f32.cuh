// Warp-per-box kernels of the upward and downward passes of 3D trees
// (passes_f32.cu).  Each launcher returns false, launching nothing, for what its
// kernel is not built for: d != 3, no box-relative point copy (uniform P2M, L2P), or
// an order other than 4, 6, 8, 10, 12, 16 (P2M, L2P, float M2M), 4, 6, 8 (float
// L2L), 4 (double-word M2M and L2L), 4 to 12 and 16 (L2P of adaptive trees).
#pragma once

#include "fmm_internal.cuh"

bool passes_f32_order(int p);
bool launch_p2m_f32(const fmm_plan_s* P, const Workspace& ws, cudaStream_t st);
// the same for the leaves (level >= 2) of an adaptive tree, from its FP64 points
struct ATree;
bool launch_ap2m_f32(const fmm_plan_s* P, const Workspace& ws, const ATree& t, cudaStream_t st);
// M2M from level l + 1 into level l, L2L from level l into level l + 1, in
// float or double-word float (dwf.cuh); FP64 shifts always run by blocks
enum ShiftArith { kShiftF32, kShiftDW, kShiftF64 };
// whether a level's M2M (up) or L2L runs by a warp per parent (else a block)
bool shift_by_warp(int p, int64_t parents, ShiftArith a, bool up);
bool launch_m2m_warp(const fmm_plan_s* P, const Workspace& ws, int l, ShiftArith a,
                     cudaStream_t st);
bool launch_l2l_warp(const fmm_plan_s* P, const Workspace& ws, int l, ShiftArith a,
                     cudaStream_t st);
// far field at the targets of the leaves, added to phi (and grad)
bool launch_l2p_f32(const fmm_plan_s* P, const Workspace& ws, double* phi, double* grad,
                    cudaStream_t st);
// the same for the leaves (level >= 2) of an adaptive tree; false: order not built
bool launch_al2p_f32(const fmm_plan_s* P, const Workspace& ws, const ATree& t, double* phi,
                     cudaStream_t st);
