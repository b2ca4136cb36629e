// gf_m2l.cuh -- the multipole-to-local stage (Sec. 2.3: an ME is turned
// into an LE for every box of the interaction list).
#pragma once

#include "gf_fmm.cuh"

namespace gf {

gf_status m2l_upload_offsets(const signed char h_il[8][189][3]);
gf_status m2l_prepare_tables(Tables *T, cudaStream_t st);
// LE_l[t] = sum over the interaction list of box t of T_o * ME_l[t + o],
// for every observer box t of every level (overwrites each LE_l).  Mixed
// precision runs on the tensor cores (tcgen05, FP16 parts) unless the plan asks
// for the SIMT kernel; FP64 forwards run on the tensor cores from BF16 digits
// where m2l_oz_prepare chose so, the rest of FP64 on the SIMT kernel.
// adj: the transpose, MEdual_l[s] = sum_{o in IL(class of s)} T_{-o}^T LEdual_l[s + o]
// over every source box s (observer boxes found through the level's map).
// fork: when non-null, recorded on st right before the M2L kernels are
// launched (after the input split).
template <class T>
gf_status m2l_run(gf_plan_s *plan, int B, bool adj, cudaStream_t st, cudaEvent_t fork = nullptr);
// Whether a block of the forward M2L leaves no room for others on its SM (tensor
// cores: its shared memory).
bool m2l_fills_sms(const gf_plan_s *plan, int B);

// Translations between levels (gf_xlate.cu; Ts = storage, Tc = arithmetic):
//   kind 0  M2M into `level` from level + 1 (store)
//   kind 1  L2L into `level` from level - 1 (update)
//   kind 2  M2M^T into `level` from level - 1 (update), over source boxes
//   kind 3  L2L^T into `level` from level + 1 (store), over observer boxes
template <class Ts, class Tc>
gf_status translate_run(gf_plan_s *plan, int level, int kind, int B, cudaStream_t st);

// The tables that the translations read beside the operators themselves, and
// any FP32 matrix [rows][K] in their component order (allocated here).
gf_status xlate_prepare_tables(Tables *T, cudaStream_t st);
gf_status xlate_quad_table(const Tables *T, const float *src, int rows, float **dst, cudaStream_t st);

// P2M of 4^3-voxel leaves under a mirror-symmetric rule (p2m_fold_ok): the
// leaves [first, first + count) from their leaf-blocked masses, and every box
// of level L - 1 straight from the density grid.
bool p2m_fold_ok(const gf_plan_s *plan);
bool rule_mirrors(const QuadRule &q);
template <class T>
gf_status p2m_leaf_run(gf_plan_s *plan, int B, int64_t first, int64_t count, cudaStream_t st);
template <class T>
gf_status p2m_up_run(gf_plan_s *plan, const void *rho, int rho_f32, int B, cudaStream_t st);
// Plans with shift tables: the expansions that the two above left in tc_split, of
// boxes [first, first + count) of a level, shifted by the rule's nodes into ME.
gf_status p2m_shift_run(gf_plan_s *plan, int B, int level, int64_t first, int64_t count, cudaStream_t st);
// The rows of a level in the M2L's split inputs, as FP32 rows (mixed precision).
float *tc_split_rows(const FmmPlan *F, int level);

// Upper bound of the partial rows of the tensor-core M2L's cut tiles (fp64: of the
// digit M2L's).
size_t m2l_tc_bytes(int p, bool fp64);
// Plan-time set-up of the tensor-core path (level descriptors on the device).
gf_status m2l_tc_prepare(gf_plan_s *plan);
// FP64 plans: workspaces of the M2L on the tensor cores by BF16 digits, where
// that is the faster one.
gf_status m2l_oz_prepare(gf_plan_s *plan);
// The adjoint's level tables (built on the plan's first adjoint call).
gf_status m2l_tc_prepare_adj(gf_plan_s *plan);

}  // namespace gf
