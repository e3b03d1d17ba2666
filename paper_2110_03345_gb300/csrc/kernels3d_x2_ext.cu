// 3D step kernels of the extended schemes of Sec. 2.4 on the two-point
// TMA-staged plane ring of the leapfrog (step3d_x2.cuh): the fourth-order
// time scheme's two passes (EXT_KW, EXT_T4) and the attenuation terms (y = 0:
// EXT_ATT0; y = 2: EXT_ATT2, in the adjoint after EXT_LC).  The plane ring
// holds the pass's stencil input (u^n, lambda^k, the k w / k L^T lambda scratch,
// or att lambda); 64 x 8 columns in z chunks, one shot per CTA.
//
// The y = 2 adjoint needs lap(att lambda) beside L^T lambda.  A second ring and
// queue for the product would leave one CTA per SM, so each step also writes
// att lambda^{k-1} and a Laplacian pass without density terms (EXT_LC) runs
// ahead of the next one.
#include "step3d_x2.cuh"

namespace fwi {

namespace {

constexpr int EXT3_BY = 8;

template <int R, bool VD, bool ADJ, int MODE, bool PP = false>
cudaError_t launch_e3(const StepParams& p, const CUtensorMap* const* m, cudaStream_t st) {
  constexpr size_t smem = smem_bytes_x2<R, VD, ADJ, EXT3_BY, MODE>();
  static DeviceOnce once;
  const cudaError_t attr = allow_smem(once, k_step3d_x2<R, VD, ADJ, EXT3_BY, MODE, false, PP>, (int)smem, true);
  if (attr != cudaSuccess) return attr;
  dim3 grid((p.nx + 63) / 64, (p.ny + EXT3_BY - 1) / EXT3_BY, p.B * p.nzc);
  return launch_pdl(k_step3d_x2<R, VD, ADJ, EXT3_BY, MODE, false, PP>, grid, dim3(32, EXT3_BY), smem, st, p,
                    *m[0], *m[1], *m[2], *m[3], *m[4], *m[5], *m[6]);
}

template <int R, bool VD, bool ADJ>
cudaError_t launch_mode3(const StepParams& p, const CUtensorMap* const* m, int mode,
                         cudaStream_t st) {
  switch (mode) {
    case EXT_KW: return launch_e3<R, VD, ADJ, EXT_KW>(p, m, st);
    case EXT_T4: return launch_e3<R, VD, ADJ, EXT_T4>(p, m, st);
    case EXT_ATT2:
      if (VD && p.bflag) return launch_e3<R, VD, ADJ, EXT_ATT2, VD>(p, m, st);
      return launch_e3<R, VD, ADJ, EXT_ATT2>(p, m, st);
    default: return launch_e3<R, VD, ADJ, EXT_ATT0>(p, m, st);
  }
}

}  // namespace

cudaError_t launch_step3d_x2_ext(const StepParams& p, const CUtensorMap& xm, const CUtensorMap& bxm,
                                 const CUtensorMap& bym, const CUtensorMap& upm,
                                 const CUtensorMap& kfm, const CUtensorMap& gm,
                                 const CUtensorMap& hm, int R, bool vd, bool adj, int mode,
                                 cudaStream_t st) {
  const CUtensorMap* m[7] = {&xm, &bxm, &bym, &upm, &kfm, &gm, &hm};
  if (mode == EXT_LC)
    return R == 4 ? launch_e3<4, false, false, EXT_LC>(p, m, st) : launch_e3<5, false, false, EXT_LC>(p, m, st);
  if (R == 4) {
    if (vd) return adj ? launch_mode3<4, true, true>(p, m, mode, st) : launch_mode3<4, true, false>(p, m, mode, st);
    return adj ? launch_mode3<4, false, true>(p, m, mode, st) : launch_mode3<4, false, false>(p, m, mode, st);
  }
  if (vd) return adj ? launch_mode3<5, true, true>(p, m, mode, st) : launch_mode3<5, true, false>(p, m, mode, st);
  return adj ? launch_mode3<5, false, true>(p, m, mode, st) : launch_mode3<5, false, false>(p, m, mode, st);
}

}  // namespace fwi
