// Launchers of the compile-time-geometry FP32 passes for edge HFX_CT_N (one translation unit per
// edge, so the sizes compile in parallel).
#include "hfx_ct.cuh"
#include "hfx_ct_diag.cuh"
#include "hfx_ct_plane.cuh"
#include "hfx_internal.h"

namespace hfx {
namespace {

constexpr int kN = HFX_CT_N;
constexpr int kB = 8;
// the forward and x passes of this edge: the plane passes of hfx_ct_plane.cuh where they exist
template <int N, bool PLANE = N % 4 == 0> struct PlanePasses;
template <int N> struct PlanePasses<N, true> {
  using G = ct::PlaneGeo<N>;
  using K = ct::PlaneCfg<N>;
  static constexpr int fwd_threads = K::fnt, x_threads = K::xnt;
  static constexpr size_t fwd_smem = G::smem_fwd, x_smem = G::smem_x;
  static constexpr auto fwd = ct::k_fwd_plane<N, K::fnt, K::fmb, K::un>;
  static constexpr auto x = ct::k_x_plane<N, K::xnt, K::xmb>;
};
template <int N> struct PlanePasses<N, false> {
  static constexpr int fwd_threads = ct::PlaneThreads<N>::value, x_threads = fwd_threads;
  static constexpr size_t fwd_smem = (N * (N + 1) + ct::Plan<N>::p.twtotal) * sizeof(float2), x_smem = fwd_smem;
  static constexpr auto fwd = ct::k_fwd_yz_ct<float, N>;
  static constexpr auto x = ct::k_x_coulomb_ct<float, N>;
};
using PP = PlanePasses<kN>;

cudaError_t prepare(int max_dynamic_smem, int* blocks_fwd, int* blocks_x) {
  const void* ks[] = {(const void*)PP::fwd, (const void*)PP::x, (const void*)ct::k_y_acc_dense_ct<float, kN, kB>,
                      (const void*)ct::k_y_acc_dense_tma<float, kN, kB>, (const void*)ct::k_y_acc_diag_ct<float, kN, kB>};
  for (const void* k : ks) {
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, max_dynamic_smem);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (e != cudaSuccess) return e;
  }
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_fwd, PP::fwd, PP::fwd_threads, PP::fwd_smem);
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_x, PP::x, PP::x_threads, PP::x_smem);
}

void fwd_yz(int grid, cudaStream_t st, const float* orb, long long Ntot, const int4* couples, int c0, int c1, float2* W,
            const float2* tw, int prefetch) {
  PP::fwd<<<grid, PP::fwd_threads, PP::fwd_smem, st>>>(orb, Ntot, couples, c0, c1, W, tw, prefetch);
}

void x_coulomb(int grid, cudaStream_t st, const int4* couples, int c0, int c1, float2* W, const float* vtab,
               const float2* tw, double* epart, int energy_only, int prefetch) {
  PP::x<<<grid, PP::x_threads, PP::x_smem, st>>>(couples, c0, c1, W, vtab, tw, epart, energy_only, prefetch);
}

void y_acc_dense(dim3 grid, size_t smem, cudaStream_t st, const float* orb, long long Ntot, const int4* couples,
                 const int* slot_list, const int* slot_couple_base, const int2* slot_blocks, int c0, const float2* W,
                 const float2* tw, float* V, double vscale) {
  ct::k_y_acc_dense_ct<float, kN, kB><<<grid, ct::DenseGeo<float, kN>::NT, smem, st>>>(
      orb, Ntot, couples, slot_list, slot_couple_base, slot_blocks, c0, W, tw, V, vscale);
}

void y_acc_dense_tma(dim3 grid, size_t smem, cudaStream_t st, const CUtensorMap& tmW, const CUtensorMap& tmOrb,
                     const CUtensorMap& tmV, const unsigned* dead_words, int n_orb, const int* slot_list,
                     const int* slot_couple_base, const int2* slot_blocks, int c0, const float2* tw, double vscale, int* err, int stall) {
  ct::k_y_acc_dense_tma<float, kN, kB><<<grid, ct::DenseGeo<float, kN>::NT, smem, st>>>(
      tmW, tmOrb, tmV, dead_words, n_orb, slot_list, slot_couple_base, slot_blocks, c0, tw, vscale, err, stall);
}

void y_acc_diag(dim3 grid, size_t smem, cudaStream_t st, const float* orb, long long Ntot, const int4* couples,
                const int* slot_list, const int* slot_couple_base, const int2* slot_blocks, int c0, const float2* W,
                const float2* tw, float* V, double vscale, const CUtensorMap& tmV, int tma_flush) {
  ct::k_y_acc_diag_ct<float, kN, kB><<<grid, ct::DenseGeo<float, kN>::NT, smem, st>>>(
      orb, Ntot, couples, slot_list, slot_couple_base, slot_blocks, c0, W, tw, V, vscale, tmV, tma_flush);
}

const CtFns kFns = {kN, ct::DenseGeo<float, kN>::NT, PP::fwd_smem > PP::x_smem ? PP::fwd_smem : PP::x_smem, &prepare, &fwd_yz, &x_coulomb, &y_acc_dense,
                    &y_acc_dense_tma, &y_acc_diag};

}  // namespace

#define HFX_CT_JOIN2(a, b) a##b
#define HFX_CT_JOIN(a, b) HFX_CT_JOIN2(a, b)
const CtFns* HFX_CT_JOIN(ct_fns_, HFX_CT_N)() { return &kFns; }

}  // namespace hfx
