// 3D perfectly matched layer (the scheme of kernels_pml.cu's header) on the
// two-point plane ring: CTAs of 32 x 8 threads stream 64 x 8 columns along z,
// two x points per thread in packed FP32x2 arithmetic.  The stencil input's
// planes arrive by TMA with their halo; the fields whose derivative is taken
// along one axis only (phi_x, phi_y; their adjoints; b_x, b_y) arrive as row
// and column tiles of one plane, and the z ones as values of the own column.
//
// What the one-point kernels spent on every point is spent where it matters:
//  * phi and its adjoints are zero outside the layer, so planes of tiles away
//    from it neither load nor differentiate them;
//  * q and its adjoint enter only where two axes are damped (f and g_j hold
//    products of two or three A): elsewhere they are left at zero, and the
//    derivatives of q are taken from global memory by the rows that need them;
//  * with t_j = phibar_j / (1 + A_j) and S_j = A_k + A_l, constant along j,
//      D1_j(b_j phibar_j) = 2 (S_j D1_j t_j - D1_j(A_j t_j)),
//      D1_j(g_j phibar_j) = (4 A_k A_l / dt) D1_j t_j,
//    so the adjoint keeps t_j and needs no quotient per staged value.
// The adjoint's first pass stores k c (the second pass's stencil input) and
// adds (2 - e) c to ubar^n itself; the second pass then adds L^T(k c) only.
//
// The one-point kernels before spent 632 / 466 / 949 / 557 instructions per
// point in the four passes (10-14% of DRAM peak).  us per pass before -> now at
// 160 x 144 x 168, order 10 with density: PML_U 204 -> 79, PML_PHI 103 -> 48,
// PML_A 230 -> 76, PML_B 238 -> 85; now bound by the latency of a plane (two
// CTAs per SM at 128 registers).  Reciprocals in place of the update's and the
// memory factors' quotients were 7% faster and lost precision in the layer
// (gradient error 1.2e-6 -> 1.8e-6 against 64 bits).
#include "step3d_x2.cuh"

namespace fwi {

namespace {

constexpr int PB = 8;                       // thread rows
constexpr int PNT = 32 * PB;
constexpr int PSTG = 4;                     // row / column stages (two loop trips)

template <int R>
struct GeoP : GeoX2<R, PB, true> {
  using G = GeoX2<R, PB, true>;
  static constexpr int SROW = G::BXB, SCOL = G::BYB, STAGE = SROW + SCOL;
};

template <int R, bool VD, int MODE>
constexpr bool pml_stage() { return MODE == PML_U || MODE == PML_A || (MODE == PML_B && VD); }
template <int R, bool VD, int MODE>
constexpr size_t pml_smem() {
  using G = GeoP<R>;
  return ((MODE != PML_A ? (size_t)G::NSU * G::PLANE : 0) +
          (pml_stage<R, VD, MODE>() ? (size_t)PSTG * G::STAGE : 0)) * sizeof(float);
}

// D1 of a register queue around entry c (unscaled weights).
template <int R>
__device__ __forceinline__ float2 d1q(const float2* q) {
  float2 s = make_float2(0.f, 0.f);
#pragma unroll
  for (int j = 1; j <= R; ++j)
    s = __ffma2_rn(bc2(w1c<R>(j)), __fadd2_rn(q[R + j], neg2(q[R - j])), s);
  return s;
}
// D1 along x of a pair from the pairs X[0 .. 2M] around it.
template <int R>
__device__ __forceinline__ float2 d1x(const float2* X) {
  constexpr int M = (R + 1) / 2;
  auto at = [&](int d) {
    const int e = d + 2 * M;
    return (e & 1) ? X[e >> 1].y : X[e >> 1].x;
  };
  float2 s = make_float2(0.f, 0.f);
#pragma unroll
  for (int j = 1; j <= R; ++j)
    s = __ffma2_rn(bc2(w1c<R>(j)), __fadd2_rn(make_float2(at(j), at(j + 1)),
                                              neg2(make_float2(at(-j), at(1 - j)))), s);
  return s;
}

template <int R, bool VD, int MODE>
__global__ void __launch_bounds__(PNT, MODE == PML_PHI ? 3 : 2)
k_pml3x(const StepParams p, const __grid_constant__ CUtensorMap xmap,
        const __grid_constant__ CUtensorMap rmap, const __grid_constant__ CUtensorMap cmap) {
  pdl_trigger();
  using G = GeoP<R>;
  constexpr int Q = 2 * R + 1, NSU = G::NSU, M = G::M, BXW = G::BXW, TXP = G::TXP;
  constexpr bool RING = MODE != PML_A;
  constexpr bool STG = pml_stage<R, VD, MODE>();
  constexpr bool QC = STG;                    // a z queue beside the ring's
  extern __shared__ __align__(128) float smp[];
  float* ring = smp;
  float* stg = smp + (RING ? NSU * G::PLANE : 0);   // [PSTG][row tile 8 x 80, column tile (8 + 2R) x 64]
  __shared__ uint64_t bar[NSU];
  __shared__ uint64_t sbar[PSTG];
  __shared__ int s_pe[MAX_ZCHUNK + 1];
  __shared__ __align__(16) float s_ax[BXW];         // A along the row and column tiles
  __shared__ float s_ay[PB + 2 * R];

  const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * 32 + tx;
  const int b = blockIdx.z / p.nzc, zc = blockIdx.z - b * p.nzc;
  const int x0 = blockIdx.x * TXP, y0 = blockIdx.y * PB;
  const int z0 = zc * p.zchunk, z1 = min(z0 + p.zchunk, p.nz), nz_c = z1 - z0;
  const int nplanes = nz_c + 2 * R;
  const size_t fo = (size_t)b * p.fstride;
  const int xg = x0 + 2 * tx, yg = y0 + ty;
  const long long col = (long long)(yg + p.oy) * p.sx + (xg + p.ox);
  const int nb = p.nb;
  // layer contact of the tile's points, and of what lies within R of them
  const bool layx = x0 < nb || x0 + TXP > p.nx - nb, layy = y0 < nb || y0 + PB > p.ny - nb;
  const bool nearxy = x0 < nb + R || x0 + TXP > p.nx - nb - R || y0 < nb + R || y0 + PB > p.ny - nb - R;
  auto layz = [&](int z) { return z < nb || z >= p.nz - nb; };
  auto nearz = [&](int z) { return z < nb + R || z >= p.nz - nb - R; };
  if (MODE == PML_PHI && !(layx || layy || z0 < nb || z1 > p.nz - nb)) {
    pdl_wait();
    return;   // phi changes only inside the layer
  }
  const unsigned long long bon = VD && (MODE == PML_U || MODE == PML_B) ? density_planes(p, z0, nz_c) : 0ull;
  auto b_on = [&](int z) { return ((bon >> (z - z0)) & 1) != 0; };   // plane z has density gradients
  // planes whose row / column tiles matter
  auto staged = [&](int z) { return MODE == PML_B ? b_on(z) : (nearxy || nearz(z)); };

  const int tmx = x0 + p.ox - G::XOFF, tmy = y0 + p.oy - R, pz0 = z0 - R + p.oz;
  if (tid == 0) {
    for (int k = 0; k < NSU; ++k) mbar_init(&bar[k], 1);
    for (int k = 0; k < PSTG; ++k) mbar_init(&sbar[k], 1);
    fence_mbar_init();
  }
  auto a_at = [](const float* sp, int i, int n) { return (i >= 0 && i < n) ? __ldg(sp + i) : 0.f; };
  if (MODE == PML_A) {
    for (int i = tid; i < BXW; i += PNT) s_ax[i] = a_at(p.spx, x0 - G::XOFF + i, p.nx);
    for (int i = tid; i < PB + 2 * R; i += PNT) s_ay[i] = a_at(p.spy, y0 - R + i, p.ny);
  }
  bool has_inj = false;
  if ((MODE == PML_U || MODE == PML_A) && p.inj_off) {
    const int t = b * p.ntiles + (zc * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
    has_inj = p.inj_off[t + 1] > p.inj_off[t];
    if (has_inj) plane_entries(p, t, nz_c, PB * TXP, tid, PNT, s_pe);
  }
  pdl_wait();   // the previous pass's fields are complete from here on
  if (MODE == PML_U && p.nrec > 0) {
    const long long blk = ((long long)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
    sample_receivers(p, blk * PNT + tid);
  }
  if (nz_c <= 0) return;
  __syncthreads();
  auto issue_plane = [&](int lp) {
    const int k = lp % NSU;
    mbar_arrive_expect_tx(&bar[k], G::PLANE_BYTES);
    tma_load_4d(ring + k * G::PLANE, &xmap, &bar[k], tmx, tmy, pz0 + lp, b);
  };
  auto issue_stage = [&](int i) {   // the tiles of plane i of the chunk
    const int k = i % PSTG;
    if (!staged(z0 + i)) {   // nothing to fetch: the stage's phase completes by itself
      mbar_arrive(&sbar[k]);
      return;
    }
    float* s = stg + k * G::STAGE;
    const int slot = MODE == PML_B ? 0 : b;
    mbar_arrive_expect_tx(&sbar[k], (uint32_t)G::STAGE * 4u);
    tma_load_4d(s, &rmap, &sbar[k], tmx, y0 + p.oy, z0 + i + p.oz, slot);
    tma_load_4d(s + G::SROW, &cmap, &sbar[k], x0 + p.ox, tmy, z0 + i + p.oz, slot);
  };
  if (tid == 0) {
    if (RING)
      for (int lp = 0; lp < NSU && lp < nplanes; ++lp) issue_plane(lp);
    if (STG)
      for (int i = 0; i < PSTG && i < nz_c; ++i) issue_stage(i);
  }

  auto ldg2 = [](const float* a) { return __ldg(reinterpret_cast<const float2*>(a)); };
  auto ld2 = [](const float* a) { return *reinterpret_cast<const float2*>(a); };
  const float2 z2 = make_float2(0.f, 0.f);
  const int c0 = G::XOFF + 2 * tx, own = (ty + R) * BXW + c0;
  bool timed_out = false;
  constexpr int U = 2;
  float2 q[RING ? Q + U - 1 : 1];             // the ring's values of this column
  float2 qc[QC ? Q + U - 1 : 1];              // phi_z, t_z or b_z k c
  // staged-z value of padded plane lp (plane z0 - R + lp) beside the ring's value u
  auto qc_val = [&](int lp, const float2& u) {
    const int z = z0 - R + lp;
    const long long id = (long long)(pz0 + lp) * p.sxy + col;
    if (MODE == PML_B) return lp < 2 * R || b_on(z - R) ? __fmul2_rn(ldg2(p.bz + id), u) : z2;
    if (!(layx || layy || layz(z)) || z < 0 || z >= p.nz) return z2;
    return ld2(p.ph[2] + fo + id);
  };
  auto take = [&](int lp, int at) {           // plane lp into queue entry `at`
    if (RING) {
      if (!mbar_wait_bounded(&bar[lp % NSU], (uint32_t)((lp / NSU) & 1))) timed_out = true;
      q[at] = lds2(ring + (lp % NSU) * G::PLANE + own);
    }
    if (QC) qc[at] = qc_val(lp, RING ? q[at] : z2);
  };
#pragma unroll
  for (int lp = 0; lp < R; ++lp) take(lp, lp);
  if (RING) {
    __syncthreads();   // their slots take planes NSU .. NSU + R - 1
    if (tid == 0)
      for (int lp = NSU; lp < NSU + R && lp < nplanes; ++lp) {
        fence_proxy_async_smem();
        issue_plane(lp);
      }
  }
#pragma unroll
  for (int lp = R; lp < 2 * R; ++lp) take(lp, lp);

  const float2 Ax = make_float2(a_at(p.spx, xg, p.nx), a_at(p.spx, xg + 1, p.nx));
  const float Ay = a_at(p.spy, yg, p.ny);
  const float2 rx = make_float2(__frcp_rn(1.f + Ax.x), __frcp_rn(1.f + Ax.y));
  const float ry = __frcp_rn(1.f + Ay);
  // the memory factors p_j act on every step: quotients rounded once
  auto p_of = [](float A) { return (1.f - A) / (1.f + A); };
  const float2 pxf = make_float2(p_of(Ax.x), p_of(Ax.y));
  const float pyf = p_of(Ay);
  const bool anyx = __any_sync(0xffffffffu, Ax.x != 0.f || Ax.y != 0.f);
  const bool in_y = yg < p.ny, in0 = in_y && xg < p.nx, in1 = in_y && xg + 1 < p.nx;
  const int loc0 = ty * TXP + 2 * tx;

  struct Ops {
    float2 k, up, q, h, g, xc, bx, by, bz, f[3];
  };
  // planes where two axes can be damped: q (and its adjoint) live there
  auto edge = [&](int z) { return (int)layx + (int)layy + (int)layz(z) >= 2; };
  auto in_layer = [&](int z) { return layx || layy || layz(z); };
  auto load_ops = [&](int i) {
    Ops o;
    o.k = o.up = o.q = o.h = o.g = o.xc = o.bx = o.by = o.bz = z2;
#pragma unroll
    for (int j = 0; j < 3; ++j) o.f[j] = z2;
    const int z = z0 + i;
    const long long id = (long long)(z + p.oz) * p.sxy + col;
    if (MODE == PML_U || MODE == PML_A) {
      o.k = ldg2(p.kf + id);
      if (edge(z)) o.q = ld2(p.q + fo + id);
    }
    if (MODE != PML_PHI) o.up = ld2(p.up + fo + id);
    if (MODE == PML_U && VD && b_on(z)) {
      o.bx = ldg2(p.bx + id);
      o.by = ldg2(p.by + id);
      o.bz = ldg2(p.bz + id);
    }
    if (MODE == PML_A) {
      o.h = __ldcs(reinterpret_cast<const float2*>(p.hist + fo + id));
      o.g = ld2(p.g + fo + id);
      o.xc = ld2(p.hist2 + fo + id);
    }
    if ((MODE == PML_PHI || MODE == PML_B) && in_layer(z)) {
#pragma unroll
      for (int j = 0; j < 3; ++j) o.f[j] = ld2(p.ph[j] + fo + id);
    }
    return o;
  };
  Ops nxt = load_ops(0);
  auto put = [&](float* f, long long id, const float2& v) {
    if (in1) *reinterpret_cast<float2*>(f + fo + id) = v;
    else if (in0) f[fo + id] = v.x;
  };

  for (int i0 = 0; i0 < nz_c; i0 += U) {
#pragma unroll
    for (int s = 0; s < U; ++s) {
      const int i = i0 + s;
      if (i < nz_c) {
        const int z = z0 + i;
        const long long idx = (long long)(z + p.oz) * p.sxy + col;
        const Ops cur = nxt;
        if (i + 1 < nz_c) nxt = load_ops(i + 1);
        take(i + 2 * R, s + 2 * R);
        const float* st = stg + (i % PSTG) * G::STAGE;
        const bool stz = STG && staged(z);
        if (stz && !mbar_wait_bounded(&sbar[i % PSTG], (uint32_t)((i / PSTG) & 1))) timed_out = true;
        const float Az = __ldg(p.spz + z);
        const bool lay = in_layer(z);
        const float* cp = ring + ((i + R) % NSU) * G::PLANE;

        float2 acc = z2, dx = z2, dy = z2, dz = z2;   // L u (lap), D1 u (unscaled)
        const float2 cen = RING ? q[RING ? s + R : 0] : z2;
        constexpr bool LAP = MODE == PML_U || MODE == PML_B;
        const bool d1 = MODE == PML_PHI || (MODE == PML_U && VD && b_on(z)) || (MODE == PML_B && lay);
        float2 X[2 * M + 1], Yp[R + 1], Ym[R + 1];
        if (RING) {
#pragma unroll
          for (int k = 0; k <= 2 * M; ++k) X[k] = lds2(cp + (ty + R) * BXW + c0 - 2 * M + 2 * k);
#pragma unroll
          for (int j = 1; j <= R; ++j) {
            Yp[j] = lds2(cp + (ty + R + j) * BXW + c0);
            Ym[j] = lds2(cp + (ty + R - j) * BXW + c0);
          }
          auto ux = [&](int d) {
            const int e = d + 2 * M;
            return (e & 1) ? X[e >> 1].y : X[e >> 1].x;
          };
          if (LAP) {
            const float2 n2 = make_float2(-(cen.x + cen.x), -(cen.y + cen.y));
            float2 ax = z2, ay = z2, az = z2;
#pragma unroll
            for (int j = 1; j <= R; ++j) {
              ax = __ffma2_rn(bc2(w2c<R>(j)), __fadd2_rn(__fadd2_rn(make_float2(ux(j), ux(j + 1)),
                                                                    make_float2(ux(-j), ux(1 - j))), n2), ax);
              ay = __ffma2_rn(bc2(w2c<R>(j)), __fadd2_rn(__fadd2_rn(Yp[j], Ym[j]), n2), ay);
              az = __ffma2_rn(bc2(w2c<R>(j)), __fadd2_rn(__fadd2_rn(q[s + R + j], q[s + R - j]), n2), az);
            }
            acc = __fmul2_rn(ax, bc2(p.ih2[0]));
            acc = __ffma2_rn(ay, bc2(p.ih2[1]), acc);
            acc = __ffma2_rn(az, bc2(p.ih2[2]), acc);
          }
          if (d1) {
            dx = d1x<R>(X);
#pragma unroll
            for (int j = 1; j <= R; ++j) dy = __ffma2_rn(bc2(w1c<R>(j)), __fadd2_rn(Yp[j], neg2(Ym[j])), dy);
            dz = d1q<R>(q + s);
            dx = __fmul2_rn(dx, bc2(p.ih1[0]));
            dy = __fmul2_rn(dy, bc2(p.ih1[1]));
            dz = __fmul2_rn(dz, bc2(p.ih1[2]));
          }
          if (MODE == PML_U && VD && b_on(z)) {
            float2 t = __fmul2_rn(cur.bx, dx);
            t = __ffma2_rn(cur.by, dy, t);
            t = __ffma2_rn(cur.bz, dz, t);
            acc = __fadd2_rn(acc, neg2(t));
          }
        }
        // D1 of the row tile, the column tile and the z queue
        float2 sx = z2, sy = z2, sz = z2;             // PML_A: D1_j t_j
        float2 ax_ = z2, ay_ = z2, az_ = z2;          // PML_A: D1_j(A_j t_j)
        if (stz) {
          float2 P[2 * M + 1];
#pragma unroll
          for (int k = 0; k <= 2 * M; ++k) {
            P[k] = lds2(st + ty * BXW + c0 - 2 * M + 2 * k);
            if (MODE == PML_B) P[k] = __fmul2_rn(P[k], X[k]);
          }
          sx = d1x<R>(P);
          const float* cs = st + G::SROW + (ty + R) * TXP + 2 * tx;
#pragma unroll
          for (int j = 1; j <= R; ++j) {
            float2 up = lds2(cs + j * TXP), um = lds2(cs - j * TXP);
            if (MODE == PML_B) {
              up = __fmul2_rn(up, Yp[j]);
              um = __fmul2_rn(um, Ym[j]);
            }
            sy = __ffma2_rn(bc2(w1c<R>(j)), __fadd2_rn(up, neg2(um)), sy);
            if (MODE == PML_A) {
              const float ap = s_ay[ty + R + j], am = s_ay[ty + R - j];
              ay_ = __ffma2_rn(bc2(w1c<R>(j)), __ffma2_rn(bc2(ap), up, neg2(__fmul2_rn(bc2(am), um))), ay_);
            }
          }
          sz = d1q<R>(qc + s);
          if (MODE == PML_A) {
#pragma unroll
            for (int k = 0; k <= 2 * M; ++k) P[k] = __fmul2_rn(P[k], lds2(s_ax + c0 - 2 * M + 2 * k));
            ax_ = d1x<R>(P);
            if (nearz(z))
#pragma unroll
              for (int j = 1; j <= R; ++j) {
                const float ap = a_at(p.spz, z + j, p.nz), am = a_at(p.spz, z - j, p.nz);
                az_ = __ffma2_rn(bc2(w1c<R>(j)),
                                 __ffma2_rn(bc2(ap), qc[s + R + j], neg2(__fmul2_rn(bc2(am), qc[s + R - j]))), az_);
              }
          }
          sx = __fmul2_rn(sx, bc2(p.ih1[0]));
          sy = __fmul2_rn(sy, bc2(p.ih1[1]));
          sz = __fmul2_rn(sz, bc2(p.ih1[2]));
        }
        float2 inj = z2;
        if (has_inj) {
          const int lz = z - z0, l0 = lz * (PB * TXP) + loc0;
          int e = s_pe[lz], e1 = s_pe[lz + 1];
          if (e1 - e > 32) {   // crowded (sinc points): this pair's entries by two bisections
            auto first = [&](int a, int z_, int lim) {
              while (a < z_) {
                const int m = (a + z_) >> 1;
                if (__ldg(p.inj_loc + m) < lim) a = m + 1;
                else z_ = m;
              }
              return a;
            };
            const int a = first(e, e1, l0);
            e1 = first(a, e1, l0 + 2);
            e = a;
          }
          for (; e < e1; ++e) {
            const int l = __ldg(p.inj_loc + e);
            if (l == l0) inj.x = fmaf(p.inj_w[e], p.vals[p.inj_vidx[e] + p.step_off], inj.x);
            else if (l == l0 + 1) inj.y = fmaf(p.inj_w[e], p.vals[p.inj_vidx[e] + p.step_off], inj.y);
          }
        }
        // ---- the pass's update
        const float syz = Ay + Az;
        const float2 a = make_float2(Ax.x + syz, Ax.y + syz);
        auto ef = [&](float A) { return 4.f * fmaf(A, syz, Ay * Az); };   // e
        const float2 e2 = lay ? make_float2(ef(Ax.x), ef(Ax.y)) : z2;
        if (MODE == PML_U) {
          float2 E = __fadd2_rn(acc, inj);
          if (stz) E = __fadd2_rn(E, __fadd2_rn(__fadd2_rn(sx, sy), sz));
          const float2 hv = __fmul2_rn(cur.k, E);
          float2 r = make_float2(2.f * cen.x - cur.up.x, 2.f * cen.y - cur.up.y);
          if (lay) {
            const float yz8 = edge(z) ? 8.f * Ay * Az / p.dt : 0.f;
            auto upd = [&](float A, float a_, float e, float c, float uo, float qv, float h) {
              return (2.f * c - (1.f - a_) * uo - e * c - (yz8 * A) * qv + h) / (1.f + a_);
            };
            r = make_float2(upd(Ax.x, a.x, e2.x, cen.x, cur.up.x, cur.q.x, hv.x),
                            upd(Ax.y, a.y, e2.y, cen.y, cur.up.y, cur.q.y, hv.y));
          } else {
            r = __fadd2_rn(r, hv);
          }
          put(p.up, idx, r);
          if (edge(z)) put(p.q, idx, __ffma2_rn(bc2(p.dt), r, cur.q));
          if (p.hist) {
            if (in1) __stcs(reinterpret_cast<float2*>(p.hist + fo + idx), hv);
            else if (in0) __stcs(p.hist + fo + idx, hv.x);
          }
        } else if (MODE == PML_PHI) {
          if (lay) {
            const float rz = __frcp_rn(1.f + Az), pzf = p_of(Az);
            const float2 sxz = make_float2(Ax.x + Az, Ax.y + Az), sxy = make_float2(Ax.x + Ay, Ax.y + Ay);
            auto one = [](float pj, float A, float S, float r, float f, float d) {
              return pj * f + (2.f * (S - A) * r) * d;
            };
            float2 nx = make_float2(one(pxf.x, Ax.x, syz, rx.x, cur.f[0].x, dx.x),
                                    one(pxf.y, Ax.y, syz, rx.y, cur.f[0].y, dx.y));
            float2 ny = make_float2(one(pyf, Ay, sxz.x, ry, cur.f[1].x, dy.x),
                                    one(pyf, Ay, sxz.y, ry, cur.f[1].y, dy.y));
            float2 nz = make_float2(one(pzf, Az, sxy.x, rz, cur.f[2].x, dz.x),
                                    one(pzf, Az, sxy.y, rz, cur.f[2].y, dz.y));
            // + g_j D1_j q where two other axes are damped
            const float* qf = p.q + fo + idx;
            const float c4 = 4.f / p.dt;
            if (Ay != 0.f && Az != 0.f) {
              float2 Z[2 * M + 1];
#pragma unroll
              for (int k = 0; k <= 2 * M; ++k) Z[k] = ld2(qf - 2 * M + 2 * k);
              const float2 d = d1x<R>(Z);
              const float g = c4 * Ay * Az * p.ih1[0];
              nx = make_float2(fmaf(g * rx.x, d.x, nx.x), fmaf(g * rx.y, d.y, nx.y));
            }
            auto line = [&](long long step) {
              float2 d = z2;
#pragma unroll
              for (int j = 1; j <= R; ++j)
                d = __ffma2_rn(bc2(w1c<R>(j)), __fadd2_rn(ld2(qf + j * step), neg2(ld2(qf - j * step))), d);
              return d;
            };
            if (anyx && Az != 0.f) {
              const float2 d = line(p.sx);
              const float g = c4 * Az * ry * p.ih1[1];
              ny = make_float2(fmaf(g * Ax.x, d.x, ny.x), fmaf(g * Ax.y, d.y, ny.y));
            }
            if (anyx && Ay != 0.f) {
              const float2 d = line(p.sxy);
              const float g = c4 * Ay * rz * p.ih1[2];
              nz = make_float2(fmaf(g * Ax.x, d.x, nz.x), fmaf(g * Ax.y, d.y, nz.y));
            }
            put(p.ph[0], idx, nx);
            put(p.ph[1], idx, ny);
            put(p.ph[2], idx, nz);
          }
        } else if (MODE == PML_A) {
          float2 c = cur.up, un, xc, qb = cur.q;
          if (stz) {
            ax_ = __fmul2_rn(ax_, bc2(p.ih1[0]));
            ay_ = __fmul2_rn(ay_, bc2(p.ih1[1]));
            az_ = __fmul2_rn(az_, bc2(p.ih1[2]));
            const float c4 = 4.f / p.dt;
            auto upd = [&](float A, float ub, float& qv, float t1x, float t1y, float t1z, float t2x, float t2y,
                           float t2z) {
              const float ds = (syz * t1x - t2x) + ((A + Az) * t1y - t2y) + ((A + Ay) * t1z - t2z);
              qv = qv - c4 * ((Ay * Az) * t1x + (A * Az) * t1y + (A * Ay) * t1z);
              return (ub - 2.f * ds) + p.dt * qv;
            };
            c.x = upd(Ax.x, c.x, qb.x, sx.x, sy.x, sz.x, ax_.x, ay_.x, az_.x);
            c.y = upd(Ax.y, c.y, qb.y, sx.y, sy.y, sz.y, ax_.y, ay_.y, az_.y);
          }
          if (lay) {
            c = make_float2(c.x / (1.f + a.x), c.y / (1.f + a.y));
            un = make_float2(inj.x - (1.f - a.x) * c.x, inj.y - (1.f - a.y) * c.y);
            xc = make_float2(cur.xc.x + (2.f - e2.x) * c.x, cur.xc.y + (2.f - e2.y) * c.y);
          } else {
            un = __fadd2_rn(inj, neg2(c));
            xc = __ffma2_rn(bc2(2.f), c, cur.xc);
          }
          const float2 kc = __fmul2_rn(cur.k, c);
          put(p.out, idx, kc);
          put(p.up, idx, un);
          put(p.hist2, idx, xc);
          put(p.g, idx, __ffma2_rn(neg2(kc), cur.h, cur.g));
          if (edge(z)) {
            const float yz8 = 8.f * Ay * Az / p.dt;
            put(p.q, idx, make_float2(qb.x - (yz8 * Ax.x) * c.x, qb.y - (yz8 * Ax.y) * c.y));
          }
        } else {   // PML_B
          if (VD && stz) acc = __fadd2_rn(acc, __fadd2_rn(__fadd2_rn(sx, sy), sz));
          put(p.up, idx, __fadd2_rn(cur.up, acc));
          if (lay) {
            const float rz = __frcp_rn(1.f + Az), pzf = p_of(Az);
            auto one = [](float pj, float r, float f, float d) { return pj * f - r * d; };
            put(p.ph[0], idx, make_float2(one(pxf.x, rx.x, cur.f[0].x, dx.x), one(pxf.y, rx.y, cur.f[0].y, dx.y)));
            put(p.ph[1], idx, make_float2(one(pyf, ry, cur.f[1].x, dy.x), one(pyf, ry, cur.f[1].y, dy.y)));
            put(p.ph[2], idx, make_float2(one(pzf, rz, cur.f[2].x, dz.x), one(pzf, rz, cur.f[2].y, dz.y)));
          }
        }
      }
    }
    // one barrier per trip: every thread is done with the trip's centre planes
    // and stages, whose slots take the planes R + NSU and PSTG ahead
    __syncthreads();
    if (tid == 0) {
#pragma unroll
      for (int s = 0; s < U; ++s) {
        const int i = i0 + s;
        if (i < nz_c) {
          if (RING && i + R + NSU < nplanes) {
            fence_proxy_async_smem();
            issue_plane(i + R + NSU);
          }
          if (STG && i + PSTG < nz_c) {
            fence_proxy_async_smem();
            issue_stage(i + PSTG);
          }
        }
      }
    }
#pragma unroll
    for (int j = 0; j < Q - 1; ++j) {
      if (RING) q[j] = q[j + U];
      if (QC) qc[j] = qc[j + U];
    }
  }
  if (timed_out && p.flags) atomicOr(p.flags, 2);
}

template <int R, bool VD, int MODE>
cudaError_t launch_p(const StepParams& p, const CUtensorMap& xm, const CUtensorMap& rm, const CUtensorMap& cm,
                     cudaStream_t st) {
  constexpr size_t smem = pml_smem<R, VD, MODE>();
  static DeviceOnce once;
  const cudaError_t attr = allow_smem(once, k_pml3x<R, VD, MODE>, (int)smem, true);
  if (attr != cudaSuccess) return attr;
  dim3 grid((p.nx + 63) / 64, (p.ny + PB - 1) / PB, p.B * p.nzc);
  return launch_pdl(k_pml3x<R, VD, MODE>, grid, dim3(32, PB), smem, st, p, xm, rm, cm);
}

template <int R, bool VD>
cudaError_t launch_mode(const StepParams& p, const CUtensorMap& xm, const CUtensorMap& rm, const CUtensorMap& cm,
                        int mode, cudaStream_t st) {
  switch (mode) {
    case PML_U: return launch_p<R, VD, PML_U>(p, xm, rm, cm, st);
    case PML_PHI: return launch_p<R, VD, PML_PHI>(p, xm, rm, cm, st);
    case PML_A: return launch_p<R, VD, PML_A>(p, xm, rm, cm, st);
    default: return launch_p<R, VD, PML_B>(p, xm, rm, cm, st);
  }
}

}  // namespace

cudaError_t launch_pml3d(const StepParams& p, const CUtensorMap& xm, const CUtensorMap& rm, const CUtensorMap& cm,
                         int R, bool vd, int mode, cudaStream_t st) {
  if (R == 4) return vd ? launch_mode<4, true>(p, xm, rm, cm, mode, st) : launch_mode<4, false>(p, xm, rm, cm, mode, st);
  return vd ? launch_mode<5, true>(p, xm, rm, cm, mode, st) : launch_mode<5, false>(p, xm, rm, cm, mode, st);
}

}  // namespace fwi
