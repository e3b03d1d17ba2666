// Perfectly matched layer (Sec. 2.4 offers a PML next to the sponge): the
// unsplit second-order form from the coordinate stretching
// d_j -> d_j / (1 + z_j / p), with the sponge's per-axis profiles z_j.  With
// A_j = z_j dt / 2 (the sponge arrays), k = (vp dt)^2,
//   a = sum A,  e = 4 (A_x A_y + A_x A_z + A_y A_z),  f = 8 A_x A_y A_z / dt,
//   p_j = (1 - A_j) / (1 + A_j),  b_j = 2 (A_k + A_l - A_j) / (1 + A_j),
//   g_j = 4 A_k A_l / (dt (1 + A_j))      (k, l the other axes; A_z = 0 in 2D)
// one time step is
//   PML_U:   E = L u^n + s^n + sum_j D1_j phi_j^n,
//            (1+a) u^{n+1} = 2u^n - (1-a) u^{n-1} - e u^n - f q^n + k E,
//            q^{n+1} = q^n + dt u^{n+1}   (3D),   h^n = k E stored;
//   PML_PHI: phi_j^{n+1} = p_j phi_j^n + b_j D1_j u^{n+1} + g_j D1_j q^{n+1},
// (D1 the solver's first-derivative stencil; outside the layer every A is 0,
// phi stays 0 and PML_U is the leapfrog, so PML_PHI skips tiles that do not
// touch the layer).  The exact discrete adjoint runs backwards, per step n:
//   PML_A:   ub = ubar^{n+1} - sum_j D1_j(b_j phibar_j) + dt qb,
//            qb = qbar^{n+1} - sum_j D1_j(g_j phibar_j),  c^n = ub / (1+a),
//            qbar^n = qb - f c^n,  ubar^{n-1} = P^T r^{n-1} - (1-a) c^n,
//            g -= (k c^n) h^n   (the imaging condition of Sec. 2.2, Eq. 8);
//   PML_B:   ubar^n += (2 - e) c^n + L^T(k c^n),
//            phibar_j^n = p_j phibar_j^{n+1} - D1_j(k c^n).
// 3D: kernels_pml3d.cu.  2D: PML_U and PML_B run on the TMA shot-loop tiles
// (EXT_PML of tma2d_tile.cuh); this file holds PML_PHI and PML_A, on the frame of
// points that need them.
//
// Away from the layer the scheme is the leapfrog, and with lambda^n = k c^n so
// is its adjoint: lambda^{n-1} = 2 lambda^n - lambda^{n+1} + k (L^T lambda^n +
// P^T r^n).  So points farther than the layer width plus R from every face
// (pml_near) take the leapfrog's update, and only the others PML_A and PML_B, with
// three fields for both: `cur` holds lambda^n everywhere (near points: ubar^{n+1}
// before PML_A), `other` lambda^{n+1}, then lambda^{n-1} (near: ubar^n), and a
// third the near points' share of ubar^{n-1}.  The phi adjoints are kept as
// psi_j = b_j phibar_j, so that PML_A needs no b_j at its stencil's points.
#include "fwi_internal.cuh"

namespace fwi {

namespace {

__device__ __forceinline__ float4 ldg4(const float* q) {
  return __ldg(reinterpret_cast<const float4*>(q));
}
__device__ __forceinline__ float4 ld4(const float* q) { return *reinterpret_cast<const float4*>(q); }
__device__ __forceinline__ void st4(float* q, const float4& v) { *reinterpret_cast<float4*>(q) = v; }
__device__ __forceinline__ void unpack(const float4& t, float* v) {
  v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
__device__ __forceinline__ float4 pack(const float* v) { return make_float4(v[0], v[1], v[2], v[3]); }

// The frame of points within W of a face, as float4 groups: row strips of
// 32 groups x 8 rows per CTA (top, bottom), then the groups at both ends of the
// rows between, 256 per CTA in linear order.
struct Frame {
  int ngx, yt, yb, gl, gr;   // rows [0, yt) and [yb, ny) whole, groups [0, gl) and [gr, ngx) else
  int bx, nrow, ncol;        // CTAs per strip of 8 rows, of the row strips, of the rest
  __host__ __device__ Frame(int nx, int ny, int W) {
    ngx = (nx + 3) / 4;
    yt = W < ny ? W : ny;
    yb = ny - W > yt ? ny - W : yt;
    gl = (W + 3) / 4 < ngx ? (W + 3) / 4 : ngx;
    gr = (nx - W) / 4 > gl ? (nx - W) / 4 : gl;
    bx = (ngx + 31) / 32;
    nrow = bx * ((yt + 7) / 8 + (ny - yb + 7) / 8);
    ncol = ((yb - yt) * (gl + ngx - gr) + 255) / 256;
  }
  // group and row of thread t of CTA b; false: none
  __device__ __forceinline__ bool at(int b, int t, int ny, int* g, int* y) const {
    if (b < nrow) {
      const int strip = b / bx, top = (yt + 7) / 8;
      *g = (b - strip * bx) * 32 + (t & 31);
      *y = (strip < top ? 8 * strip : yb + 8 * (strip - top)) + (t >> 5);
      return *g < ngx && *y < (strip < top ? yt : ny);
    }
    const int i = (b - nrow) * 256 + t, n = gl + ngx - gr;
    *y = yt + i / n;
    *g = i % n;
    if (*g >= gl) *g += gr - gl;
    return *y < yb;
  }
};

// PML_PHI on the layer, or PML_A on the points within the stencil's reach of it.
//
// Bound by latency and L2: a thread has some 13 float4 loads in flight and little
// else.  A frame of groups instead of the 128 x 16 tiles that touch it (1024 x
// 1024, a 20-point layer, 6 shots: PML_PHI 20.5 -> 9.0 us, PML_A 36 -> 10 us; the
// tiles hold three times the frame's points).  With U and B on the shot-loop tiles
// a time step of the gradient takes 111 us where four passes over one-shot tiles
// of the whole grid took 195.
template <int R, int MODE>
__global__ void __launch_bounds__(256, 4) k_pml2d(const StepParams p) {
  constexpr int NL = (R <= 4) ? 1 : 2;
  constexpr int NV = 4 + 8 * NL;
  const Frame F(p.nx, p.ny, MODE == PML_PHI ? p.nb : p.nb + R);
  int g, yg;
  if (!F.at(blockIdx.x, threadIdx.x, p.ny, &g, &yg)) return;
  const int b = blockIdx.y;
  const int xg = 4 * g;
  const int pix = (yg + p.oy) * p.sx + (xg + p.ox);
  const long long pi = (long long)b * p.fstride + pix;
  bool in[4];
#pragma unroll
  for (int l = 0; l < 4; ++l) in[l] = xg + l < p.nx;

  // D1x and D1y of u^{n+1}, or of psi_x = b_x phibar_x and psi_y = b_y phibar_y
  const float* row = (MODE == PML_PHI ? p.x : p.ph[0]) + pi;
  const float* col = (MODE == PML_PHI ? p.x : p.ph[1]) + pi;
  float d1x[4] = {0.f, 0.f, 0.f, 0.f}, d1y[4] = {0.f, 0.f, 0.f, 0.f};
  float v[NV];
#pragma unroll
  for (int q = 0; q <= 2 * NL; ++q) unpack(ld4(row + 4 * (q - NL)), v + 4 * q);
#pragma unroll
  for (int l = 0; l < 4; ++l)
#pragma unroll
    for (int j = 1; j <= R; ++j) d1x[l] = fmaf(p.wx.w1[j], v[4 * NL + l + j] - v[4 * NL + l - j], d1x[l]);
#pragma unroll
  for (int j = 1; j <= R; ++j) {
    float a[4], c[4];
    unpack(ld4(col - j * p.sx), a);
    unpack(ld4(col + j * p.sx), c);
#pragma unroll
    for (int l = 0; l < 4; ++l) d1y[l] = fmaf(p.wy.w1[j], c[l] - a[l], d1y[l]);
  }
  float Ax[4];
  unpack(ldg4(p.spx + xg), Ax);
  const float Ay = p.spy[yg];
  if (MODE == PML_PHI) {
    float fx[4], fy[4];
    unpack(ld4(p.ph[0] + pi), fx);
    unpack(ld4(p.ph[1] + pi), fy);
#pragma unroll
    for (int l = 0; l < 4; ++l) {
      fx[l] = in[l] ? ((1.f - Ax[l]) * fx[l] + 2.f * (Ay - Ax[l]) * d1x[l]) / (1.f + Ax[l]) : 0.f;
      fy[l] = in[l] ? ((1.f - Ay) * fy[l] + 2.f * (Ax[l] - Ay) * d1y[l]) / (1.f + Ay) : 0.f;
    }
    st4(p.ph[0] + pi, pack(fx));
    st4(p.ph[1] + pi, pack(fy));
    return;
  }
  // PML_A: the residual of step n-1 (this row's entries)
  float inj[4] = {0.f, 0.f, 0.f, 0.f};
  if (p.inj_off) {
    const int t = b * p.ntiles + (yg / EXT_TY2) * ((p.nx + EXT_TX2 - 1) / EXT_TX2) + xg / EXT_TX2;
    if (p.inj_off[t + 1] > p.inj_off[t]) {
      const int ly = yg % EXT_TY2, tx = (xg % EXT_TX2) / 4;
      const int* rr = p.inj_row + (size_t)t * (EXT_TY2 + 1) + ly;
      const int r1 = rr[1];
      for (int e = rr[0]; e < r1; ++e) {
        const int elx = p.inj_loc[e] - ly * EXT_TX2;
        if ((elx >> 2) == tx) {
          const float val = p.inj_w[e] * p.vals[p.inj_vidx[e] + p.step_off];
          const int l = elx & 3;
#pragma unroll
          for (int q = 0; q < 4; ++q) inj[q] += (q == l) ? val : 0.f;
        }
      }
    }
  }
  float k[4], xn[4], xc[4], un[4], lam[4];
  unpack(ldg4(p.kf + pix), k);
  unpack(ld4(p.up + pi), xn);
  unpack(ld4(p.hist2 + pi), xc);
#pragma unroll
  for (int l = 0; l < 4; ++l) {
    const float a = Ax[l] + Ay, e = 4.f * Ax[l] * Ay;
    const float c = (xn[l] - (d1x[l] + d1y[l])) / (1.f + a);
    lam[l] = in[l] ? k[l] * c : 0.f;
    un[l] = in[l] ? inj[l] - (1.f - a) * c : 0.f;
    xc[l] = in[l] ? xc[l] + (2.f - e) * c : 0.f;
  }
  st4(p.up + pi, pack(lam));
  st4(p.hist2 + pi, pack(un));
  st4(p.out + pi, pack(xc));
  if (p.image) {
    float h[4], gr[4];
    unpack(__ldcs(reinterpret_cast<const float4*>(p.hist + pi)), h);
    unpack(ld4(p.g + pi), gr);
#pragma unroll
    for (int l = 0; l < 4; ++l)
      if (in[l]) gr[l] = fmaf(-lam[l], h[l], gr[l]);
    st4(p.g + pi, pack(gr));
  }
}

template <int R, int MODE>
cudaError_t launch_m(const StepParams& p, cudaStream_t st) {
  const Frame F(p.nx, p.ny, MODE == PML_PHI ? p.nb : p.nb + R);
  if (F.nrow + F.ncol == 0) return cudaSuccess;   // (no layer)
  k_pml2d<R, MODE><<<dim3(F.nrow + F.ncol, p.B), 256, 0, st>>>(p);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_pml2d(const StepParams& p, int R, int mode, cudaStream_t st) {
  if (mode == PML_PHI) return R == 4 ? launch_m<4, PML_PHI>(p, st) : launch_m<5, PML_PHI>(p, st);
  if (mode == PML_A) return R == 4 ? launch_m<4, PML_A>(p, st) : launch_m<5, PML_A>(p, st);
  return cudaErrorInvalidValue;   // (PML_U and PML_B: EXT_PML of kernels2d_tma_ext.cu)
}

namespace {

// field[slot][node] += w val for every entry of every (slot, tile) bucket, one
// thread per bucket in its entries' order (no two tiles share a node): the
// receiver residuals of one step spread onto an adjoint field.
__global__ void k_inject_buckets(const StepParams p, float* __restrict__ field, int tx, int ty,
                                 int zc, int gx, int gy, int reach, int nbuckets) {
  const int bk = blockIdx.x * blockDim.x + threadIdx.x;
  if (bk >= nbuckets) return;
  const int slot = bk / p.ntiles, t = bk - slot * p.ntiles;
  const int bx = t % gx, by = (t / gx) % gy, bz = t / (gx * gy);
  float* f = field + (long long)slot * p.fstride;
  for (int e = p.inj_off[bk]; e < p.inj_off[bk + 1]; ++e) {
    const int loc = p.inj_loc[e];
    const int lx = loc % tx, ly = (loc / tx) % ty, lz = loc / (tx * ty);
    if (reach > 0 && !pml_near((bx * tx + lx) & ~3, by * ty + ly, reach, p.nx, p.ny)) continue;
    const long long idx = (long long)(bz * zc + lz + p.oz) * p.sxy +
                          (long long)(by * ty + ly + p.oy) * p.sx + (bx * tx + lx + p.ox);
    f[idx] += p.inj_w[e] * p.vals[p.inj_vidx[e] + p.step_off];
  }
}

}  // namespace

cudaError_t launch_inject_buckets(const StepParams& p, float* field, int tx, int ty, int zc, int gx,
                                  int gy, int reach, cudaStream_t st) {
  const int n = p.B * p.ntiles;
  if (n <= 0 || !p.inj_off) return cudaSuccess;
  k_inject_buckets<<<(n + 127) / 128, 128, 0, st>>>(p, field, tx, ty, zc, gx, gy, reach, n);
  return cudaGetLastError();
}

}  // namespace fwi
