// router_fwd.cu -- SMoES router forward on sm_103a.
//
// One pass over X computes, per token: the gate logits z = W x (Sec. 3.1) on tcgen05 tensor
// cores (TMA-fed, accumulators in TMEM), the Gaussian modality score of eqs. (8)-(9) from the
// same shared-memory X tiles, softmax, top-k, bin sums p_k = sum_{e in B_k} g_e, and the
// per-(128-token tile, sample) partial sums of the joint table of eq. (12). The reducer warp of the
// CTA that completes the last partial of a sample reduces that sample's joint to P (eq. 13),
// I (eq. 14) and the backward coefficient table; the one that completes the last sample writes
// the loss of eq. (15). All reductions run in a fixed order: results are bitwise reproducible.
//
// Code that runs once per tile is kept in compact loops: a kernel that streams one or two tiles
// per SM spends most of its epilogue fetching instructions and waiting on dependent latency,
// not issuing arithmetic.
//
// The tensor-core kernel and the epilogue it shares with the fp32 kernel are in router_fwd_tc.cuh, the
// fp32 kernel in router_fwd_f32.cuh; this file holds the launchers (router_fwd_var.cu instantiates
// both kernels with the router variants).
#include "router_fwd_f32.cuh"

namespace smoes {

// Plans without router variants run kernels compiled without their code (the epilogue of a
// kernel that streams one or two tiles per SM is bound by instruction fetch and latency, and
// the variant branches lengthen it); plans with a variant run those of router_fwd_var.cu.
cudaError_t launch_router_fwd_bf16(const FwdParams& p, const CUtensorMap& tmX,
                                   const CUtensorMap& tmW, const CUtensorMap* tmG, int n_sms,
                                   cudaStream_t s) {
  if (p.dm.gate || p.dm.mask) return launch_router_fwd_bf16_var(p, tmX, tmW, tmG, n_sms, s);
  return launch_fwd_tc<false>(p, tmX, tmW, tmG, n_sms, s);
}

cudaError_t launch_router_fwd_f32(const FwdParams& p, cudaStream_t s) {
  if (p.dm.gate || p.dm.mask) return launch_router_fwd_f32_var(p, s);
  return launch_fwd_f32<false>(p, s);
}

int f32_chunks(int d) { return (d + kF32Cols - 1) / kF32Cols; }

}  // namespace smoes
