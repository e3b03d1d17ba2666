// 2D leapfrog kernels that keep a whole shot on chip (damped leapfrog of
// Eq. 10, Sec. 2.4; exact discrete adjoint with the imaging condition of
// Sec. 2.2, Eq. 8).
//
// The per-step kernels (kernels2d_tma.cu) read and write u^n, u^{n-1} in
// global memory and pay a launch per step.  All 152 SMs together hold 34 MB of
// shared memory, so a 2D wavefield pair of up to about a million points fits
// there: one launch advances a shot by many steps.
//
//  * A CTA owns a tile of 128 x TH points of one shot for the whole launch, one
//    CTA per SM; several shots run side by side when their tiles fit.  u^n and
//    u^{n-1} live in two shared tiles with halos and u^{n+1} overwrites u^{n-1}
//    in place; global memory sees the history (4 bytes per point and step), the
//    halo exchange and the receiver samples.
//  * A thread owns a float4 of x points in RY consecutive rows and slides a
//    window of 2R+1 rows down its strip, so the y taps cost (RY + 2R) / RY
//    shared loads per row instead of 2R.
//  * Neighbours exchange the R outermost rows / columns of u^{n+1} through
//    global memory (L2) as 8-byte words {value, step tag}: a word whose tag
//    matches carries its value, so neither fences nor flags are needed, and a
//    step costs one store -> load trip to L2 (about 2000 cycles) and a CTA
//    barrier.  Two parities suffice: a CTA overwrites a word only after it has
//    received the neighbour's data of the following step, which the neighbour
//    sends after reading that word.
//  * Tiles above 16 rows advance in two halves (PH = 2), so that the trip of one
//    half's edges overlaps the other half's arithmetic.
//  * Rows whose density gradient is zero (water, the inside of a homogeneous
//    tissue) leave its terms out: they add an exact zero.
//  * All CTAs of a launch must be resident together: the launch is
//    cooperative, with at most one CTA per SM.  Every wait is bounded; on
//    time-out the CTA flags the step and the launch ends.
//
// What bounds it (ncu, one 1024 x 1024 shot with density, TH = 56): the L1 /
// shared data pipe is busy 56% of the time and the FMA pipe 40% at 14 warps of
// 128 registers; every CTA keeps step with the slowest, so a step costs the
// slowest tile's arithmetic plus about 1200 cycles of exchange and barriers.
// One shot, 64 receivers, 8th order, time of a call of 1000 steps per step, per-step kernels
// -> resident, forward / forward and adjoint with imaging, in us: 256 x 256 with density
// 3.6 -> 2.0 / 8.0 -> 4.2, without 3.5 -> 1.7 / 7.2 -> 3.7; 700 x 748 with 4.0 -> 2.7 / 9.1 -> 7.5,
// without 3.9 -> 2.4 / 8.3 -> 5.4; 1024 x 1024 with 5.7 -> 3.7 / 15.2 -> 9.1, without 5.1 -> 3.2 /
// 12.4 -> 7.0.
// Tried and slower: 28 warps of 72 registers with one row each (shared loads
// and spills), four rows in one phase (the exchange is exposed), scalar
// weights in place of packed ones, the outer columns sent by every warp.
#include "fwi_internal.cuh"
#include "tma_util.cuh"

namespace fwi {

namespace {

constexpr int RES_TX = 128;
constexpr int RES_WARPS = 16;             // thread rows of a CTA at most (128 registers a thread)
constexpr unsigned RES_POLLS = 1u << 21;  // about a second of L2 round trips

template <int R>
struct ResGeo {
  static constexpr int XH = (R <= 4) ? 4 : 8;   // halo floats staged left and right
  static constexpr int NL = XH / 4;
  static constexpr int SW = RES_TX / 4 + 2 * NL;  // float4 per staged row
  __host__ __device__ static constexpr int cells(int TH) { return 2 * R * 32 + 2 * TH * NL; }
};

// Four words {value, tag}, where `on` is set (predicated, no branch).
__device__ __forceinline__ void st_tagged(bool on, unsigned long long* q, const float4& v, unsigned tag) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 a, b, c, d;\n\t"
      "setp.ne.u32 p, %6, 0;\n\t"
      "mov.b64 a, {%1, %5};\n\tmov.b64 b, {%2, %5};\n\t"
      "mov.b64 c, {%3, %5};\n\tmov.b64 d, {%4, %5};\n\t"
      "@p st.relaxed.gpu.global.v2.b64 [%0], {a, b};\n\t"
      "@p st.relaxed.gpu.global.v2.b64 [%0 + 16], {c, d};\n\t}"
      ::"l"(q), "r"(__float_as_uint(v.x)), "r"(__float_as_uint(v.y)), "r"(__float_as_uint(v.z)),
      "r"(__float_as_uint(v.w)), "r"(tag), "r"((unsigned)on)
      : "memory");
}
struct Words {
  unsigned long long w[4];
};
__device__ __forceinline__ void ld_words(const unsigned long long* q, Words& x) {
  asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(x.w[0]), "=l"(x.w[1]) : "l"(q) : "memory");
  asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2 + 16];" : "=l"(x.w[2]), "=l"(x.w[3]) : "l"(q) : "memory");
}
__device__ __forceinline__ bool tagged(const Words& x, unsigned tag) {
  return (unsigned)(x.w[0] >> 32) == tag && (unsigned)(x.w[1] >> 32) == tag &&
         (unsigned)(x.w[2] >> 32) == tag && (unsigned)(x.w[3] >> 32) == tag;
}
__device__ __forceinline__ float4 words4(const Words& x) {
  return make_float4(__uint_as_float((unsigned)x.w[0]), __uint_as_float((unsigned)x.w[1]),
                     __uint_as_float((unsigned)x.w[2]), __uint_as_float((unsigned)x.w[3]));
}
__device__ __forceinline__ void cp_async16(float4* dst, const float* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(tma::smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ float4 ldf4(const float* q) { return *reinterpret_cast<const float4*>(q); }
__device__ __forceinline__ float4 ldg4(const float* q) { return __ldg(reinterpret_cast<const float4*>(q)); }
__device__ __forceinline__ float2 lo2(const float4& v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 hi2(const float4& v) { return make_float2(v.z, v.w); }
__device__ __forceinline__ float2 add2(const float2& a, const float2& b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float4 mul4(const float4& a, const float4& b) {
  const float2 p = __fmul2_rn(lo2(a), lo2(b)), q = __fmul2_rn(hi2(a), hi2(b));
  return make_float4(p.x, p.y, q.x, q.y);
}
__device__ __forceinline__ void axpy2(float2& acc, float w, const float2& s) {
  acc = __ffma2_rn(make_float2(w, w), s, acc);
}
__device__ __forceinline__ void put4(const float4& t, float* v) {
  v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}

// PH: the tile's rows are advanced in one phase, or in two halves one after
// the other, so that the halo of one half travels while the other half is
// computed.  Tiles of odd rows take their lower half first: the edges that two
// neighbours exchange then belong to the same phase on both sides.
// RY: rows per thread and phase.
template <int R, bool VD, bool ADJ, int PH, int RY>
__global__ void __launch_bounds__(32 * RES_WARPS, 1) k_res2d(const ResParams p) {
  using G = ResGeo<R>;
  constexpr int NL = G::NL, SW = G::SW, XH = G::XH;
  constexpr int NV = 4 + 8 * NL;
  constexpr int C = 4 * NL;                // own first point in the x window
  constexpr int NTASK = PH == 2 ? 1 : 3;   // halo cells a thread receives per phase, at most
  constexpr bool GREG = !VD;               // adjoint: the gradient in registers
  constexpr bool KREG = PH * RY <= 2;      // k in registers
  extern __shared__ __align__(128) float4 sm[];
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int NT = 32 * blockDim.y, tid = ty * 32 + tx;
  const int TH = p.TH, SH = TH + 2 * R;
  const int cta = blockIdx.x;
  const int byi = cta / p.gx, bxi = cta - byi * p.gx;
  const int slot = blockIdx.y;
  const int x0 = bxi * RES_TX, y0 = byi * TH;
  const size_t fo = (size_t)slot * p.fstride;

  float4* const s_u0 = sm;
  float4* const s_u1 = sm + SH * SW;
  float4* const s_x = sm + 2 * SH * SW;
  float4* const s_h = s_x;                                   // adjoint: h^k of the own points [TH][32]
  float4* const s_bx = ADJ ? s_x + TH * 32 : s_x;            // -b_x of the own points, or b_x rows with x halo
  float4* const s_by = s_bx + (ADJ ? TH * SW : TH * 32);     // -b_y of the own points, or b_y columns with y halo
  float4* const s_g = s_by + SH * 32;                        // adjoint with density: the gradient [TH][32]
  float4* const s_end = VD ? (ADJ ? s_g + TH * 32 : s_by + TH * 32) : (ADJ ? s_x + TH * 32 : s_x);
  unsigned* const s_cell = reinterpret_cast<unsigned*>(s_end);   // injection entries of each float4 cell
  float* const s_val = reinterpret_cast<float*>(s_cell + TH * 32);   // their values, two parities
  unsigned char* const s_ix = reinterpret_cast<unsigned char*>(s_val + 2 * p.nval);   // and lane of the float4

  // ---- tile state: u^n with halo, u^{n-1}, model
  const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
  const float2 m1 = make_float2(-1.f, -1.f), m2 = make_float2(-2.f, -2.f);
  // a - b, and s - 2 c, rounded once (a packed multiply-add takes no operand
  // negation from elsewhere, a packed add would)
  auto dif2 = [&](const float2& a, const float2& b) { return __ffma2_rn(b, m1, a); };
  auto sec2 = [&](const float2& sum, const float2& c) { return __ffma2_rn(c, m2, sum); };
  const int gbase = (y0 + p.oy - R) * p.sx + (x0 + p.ox - XH);
  for (int i = tid; i < SH * SW; i += NT) {
    const int r = i / SW, c = i - r * SW;
    const bool in = y0 - R + r < p.ny;
    s_u0[i] = in ? ldf4(p.u + fo + gbase + r * p.sx + 4 * c) : z4;
    s_u1[i] = (in && r >= R && r < SH - R && c >= NL && c < SW - NL)
                  ? ldf4(p.up + fo + gbase + r * p.sx + 4 * c) : z4;
  }
  if (VD && ADJ) {
    for (int i = tid; i < TH * SW; i += NT) {
      const int r = i / SW, c = i - r * SW;
      s_bx[i] = (y0 + r < p.ny) ? ldg4(p.bx + gbase + (r + R) * p.sx + 4 * c) : z4;
    }
    for (int i = tid; i < SH * 32; i += NT) {
      const int r = i / 32, c = i - r * 32;
      s_by[i] = (y0 - R + r < p.ny) ? ldg4(p.by + gbase + r * p.sx + 4 * (c + NL)) : z4;
    }
  }
  const int xg = x0 + 4 * tx;
  const float4 ax4 = ldg4(p.spx + xg);
  const bool dampx = __any_sync(0xffffffffu, ax4.x != 0.f || ax4.y != 0.f || ax4.z != 0.f || ax4.w != 0.f);
  const int flip = PH == 2 ? (byi & 1) : 0;
  const int pixc = (y0 + p.oy) * p.sx + (xg + p.ox);      // padded index of tile row 0
  // first row of this thread's strip in phase ph
  auto strip = [&](int ph) { return (PH == 2 ? (ph ^ flip) * (TH / 2) : 0) + ty * RY; };
  // offsets of the own rows (rows beyond the grid stand on the zero padding row)
  int off[PH * RY];
  float4 kk[KREG ? PH * RY : 1], gg[(ADJ && GREG) ? PH * RY : 1];
  // own rows (alike in a warp) where the density gradient is not zero: elsewhere,
  // in water or within a homogeneous tissue, its terms vanish and are left out
  unsigned bxm = 0, bym = 0;
  unsigned inb = 0;                        // own rows inside the grid
  unsigned spm = 0;                        // and those with points in the sponge (alike in a warp)
#pragma unroll
  for (int i = 0; i < PH * RY; ++i) {
    const int row = strip(i / RY) + i % RY;
    const int yg = y0 + row;
    const bool in = yg < p.ny;
    off[i] = (min(yg, p.ny) - y0) * p.sx;
    const int pix = pixc + off[i];
    if (in) inb |= 1u << i;
    if (in && (dampx || __ldg(p.spy + yg) != 0.f)) spm |= 1u << i;
    if (KREG) kk[i] = ldg4(p.kf + pix);
    if (ADJ) {
      const float4 g = in ? ldf4(p.g + fo + pix) : z4;
      if (GREG) gg[i] = g;
      else s_g[row * 32 + tx] = g;
    }
    if (VD && !ADJ) {
      const float4 bx = in ? ldg4(p.bx + pix) : z4, by = in ? ldg4(p.by + pix) : z4;
      if (__any_sync(0xffffffffu, bx.x != 0.f || bx.y != 0.f || bx.z != 0.f || bx.w != 0.f || by.x != 0.f ||
                                      by.y != 0.f || by.z != 0.f || by.w != 0.f))
        bxm |= 1u << i;
      s_bx[row * 32 + tx] = make_float4(-bx.x, -bx.y, -bx.z, -bx.w);
      s_by[row * 32 + tx] = make_float4(-by.x, -by.y, -by.z, -by.w);
    }
  }


  if (VD && ADJ) {
    __syncthreads();   // the b_x and b_y tiles
    auto any4 = [](const float4& b) { return b.x != 0.f || b.y != 0.f || b.z != 0.f || b.w != 0.f; };
#pragma unroll
    for (int i = 0; i < PH * RY; ++i) {
      const int row = strip(i / RY) + i % RY;
      bool x = false, y = false;
      for (int q = 0; q <= 2 * NL; ++q) x = x || any4(s_bx[row * SW + tx + q]);
      for (int r = 0; r <= 2 * R; ++r) y = y || any4(s_by[(row + r) * 32 + tx]);
      if (__any_sync(0xffffffffu, x)) bxm |= 1u << i;
      if (__any_sync(0xffffffffu, y)) bym |= 1u << i;
    }
  }

  // ---- injection entries (sorted by position): first and count per cell
  const int eb = p.inj_off ? p.inj_off[slot * p.P + cta] : 0;
  const int ne = p.inj_off ? min(p.inj_off[slot * p.P + cta + 1] - eb, p.nval) : 0;
  unsigned injm = 0;                       // own rows whose cell has entries
  if (ne > 0) {
#pragma unroll
    for (int i = 0; i < PH * RY; ++i) {
      const int row = strip(i / RY) + i % RY;
      const int lo = row * RES_TX + 4 * tx;
      int a = 0, b = ne;
      while (a < b) {
        const int m = (a + b) >> 1;
        if (__ldg(p.inj_loc + eb + m) < lo) a = m + 1;
        else b = m;
      }
      int n = 0;
      while (a + n < ne && __ldg(p.inj_loc + eb + a + n) < lo + 4) ++n;
      s_cell[row * 32 + tx] = (unsigned)a | ((unsigned)n << 16);
      if (n) injm |= 1u << i;
    }
    for (int e = tid; e < ne; e += NT) {
      s_ix[e] = (unsigned char)(__ldg(p.inj_loc + eb + e) & 3);
      s_val[e] = __ldg(p.inj_w + eb + e) * p.vals[p.inj_vidx[eb + e] + p.voff];
    }
  }
  const int sb = p.smp_off ? p.smp_off[(size_t)slot * p.smp_slot + cta] : 0;
  const int nsmp = p.smp_off ? p.smp_off[(size_t)slot * p.smp_slot + cta + 1] - sb : 0;

  // ---- halo exchange: own area, and the cells this thread receives in each phase
  const int ncell = G::cells(TH);
  const unsigned par = (unsigned)ncell * 4;    // words per parity
  unsigned long long* const ex0 = p.ex + (size_t)slot * p.P * 2 * par;
  unsigned long long* const exo = ex0 + (size_t)cta * 2 * par;
  const bool hasN = byi > 0, hasS = byi + 1 < p.gy, hasW = bxi > 0, hasE = bxi + 1 < p.gx;
  unsigned nsm = 0;                            // own rows among the tile's outer rows
#pragma unroll
  for (int i = 0; i < PH * RY; ++i) {
    const int row = strip(i / RY) + i % RY;
    if ((hasN && row < R) || (hasS && row >= TH - R)) nsm |= 1u << i;
  }
  const unsigned rare = injm | spm | nsm;      // own rows that take the longer way
  // The outer columns.  One phase: lanes of each warp send their cells with the
  // row.  Two phases: those of a phase are sent after the next barrier, one
  // cell per thread (staged index and word of the upper half).
  const bool ew = (hasW && tx < NL) || (hasE && tx >= 32 - NL);
  int ewi = -1;
  unsigned ewc = 4u * (2 * R * 32 + (tx < NL ? tx : TH * NL + tx - (32 - NL)));
  if (PH == 2) {
    const int n = TH / 2 * NL;
    const bool east = tid >= n;
    const int row = (tid - (east ? n : 0)) / NL, q = (tid - (east ? n : 0)) % NL;
    if (tid < 2 * n && (east ? hasE : hasW)) ewi = (row + R) * SW + NL + (east ? 32 - NL : 0) + q;
    ewc = 4u * (2 * R * 32 + (east ? TH * NL : 0) + row * NL + q);
  }
  // columns of phase ph's rows of staged tile t, under `tag`
  auto send_columns = [&](int ph, const float4* t, unsigned parity, unsigned tag) {
    const int half = ph ^ flip;
    if (ewi >= 0)
      st_tagged(true, exo + parity * par + (ewc + half * (TH / 2 * NL * 4)), t[ewi + half * (TH / 2 * SW)], tag);
  };
  unsigned src[PH * NTASK];
  int dst[PH * NTASK];                         // < 0: none
#pragma unroll
  for (int i = 0; i < PH * NTASK; ++i) {
    const int half = (i / NTASK) ^ flip;       // phase -> half (PH = 2)
    int t = tid + (i % NTASK) * NT;
    const int rows = PH == 2 ? TH / 2 : TH, rlo = PH == 2 ? half * rows : 0;
    const int nns = PH == 2 ? R * 32 : 2 * R * 32;   // north / south cells of the phase
    int nb = -1, cell = 0, d = -1;
    if (t < nns) {
      const bool north = PH == 2 ? half == 0 : t < R * 32;
      if (PH == 1 && !north) t -= R * 32;
      if (north) {                             // the northern tile's last rows
        if (hasN) nb = cta - p.gx;
        cell = R * 32 + t;
        d = (t >> 5) * SW + NL + (t & 31);
      } else {                                 // the southern tile's first rows
        if (hasS) nb = cta + p.gx;
        cell = t;
        d = (TH + R + (t >> 5)) * SW + NL + (t & 31);
      }
    } else if (t < nns + 2 * rows * NL) {
      t -= nns;
      const bool west = t < rows * NL;
      if (!west) t -= rows * NL;
      const int row = rlo + t / NL, q = t % NL;
      if (west) {                              // the western tile's last columns
        if (hasW) nb = cta - 1;
        cell = 2 * R * 32 + TH * NL + row * NL + q;
        d = (row + R) * SW + q;
      } else {                                 // the eastern tile's first columns
        if (hasE) nb = cta + 1;
        cell = 2 * R * 32 + row * NL + q;
        d = (row + R) * SW + NL + 32 + q;
      }
    }
    dst[i] = nb >= 0 ? d : -1;
    src[i] = nb >= 0 ? (unsigned)nb * 2 * par + 4u * cell : 0u;
  }
  // Cells of phase ph carrying `tag` into tile t; false when they never come.
  // `ahead`: the first cell's words were requested earlier.
  auto receive = [&](int ph, float4* t, unsigned parity, unsigned tag, Words& ahead, bool asked) {
    bool ok = true;
#pragma unroll
    for (int q = 0; q < NTASK; ++q) {
      const int i = ph * NTASK + q;
      if (dst[i] < 0) continue;
      const unsigned long long* w = ex0 + src[i] + parity * par;
      Words x = ahead;
      unsigned polls = 0;
      if (!(asked && q == 0)) ld_words(w, x);
      while (!tagged(x, tag)) {
        if (++polls > RES_POLLS) {
          ok = false;
          break;
        }
        ld_words(w, x);
      }
      t[dst[i]] = words4(x);
    }
    return ok;
  };
  if (ADJ) {   // h of the first imaged step
#pragma unroll
    for (int ph = 0; ph < PH; ++ph) {
      if (p.nimg > 0 && p.img0 == 0)
#pragma unroll
        for (int iy = 0; iy < RY; ++iy)
          cp_async16(s_h + (strip(ph) + iy) * 32 + tx, p.hist + fo + pixc + off[ph * RY + iy]);
      asm volatile("cp.async.commit_group;" ::: "memory");
    }
  }
  Words ahead;
  ahead.w[0] = ahead.w[1] = ahead.w[2] = ahead.w[3] = 0;

  for (int it = 0; it < p.steps; ++it) {
    float4* const su = (it & 1) ? s_u1 : s_u0;
    float4* const so = (it & 1) ? s_u0 : s_u1;
    unsigned long long* const exw = exo + ((it + 1) & 1) * par;
    const unsigned tag = p.tag0 + it + 1;
    const bool img = ADJ && it >= p.img0;
    const float* const sval = s_val + (it & 1) * p.nval;
    float nval = 0.f;
    float* const hrow = p.hist + (size_t)it * p.hstride + fo + pixc;   // forward: tile row 0 of h
#pragma unroll
    for (int ph = 0; ph < PH; ++ph) {
      // the halo of u^n of this phase's rows (the first step's came from global memory)
      bool ok = true;
      if (it > 0) ok = receive(ph, su, it & 1, tag - 1, ahead, PH == 2);
      if (__syncthreads_or(!ok)) {   // a neighbour's data never came: flag and end the launch
        if (tid == 0 && p.flags) atomicOr(p.flags, 2);
        asm volatile("cp.async.wait_all;" ::: "memory");
        return;
      }
      if (PH == 2) {
        if (ph == 1) send_columns(0, so, (it + 1) & 1, tag);
        else if (it > 0) send_columns(1, su, it & 1, tag - 1);
      }
      if (ph == 0) {
        // the next step's injected value of this thread's entry, a step ahead
        if (tid < ne && it + 1 < p.steps)
          nval = __ldg(p.inj_w + eb + tid) * p.vals[p.inj_vidx[eb + tid] + p.voff + (it + 1) * p.vstep];
        // samples of u^n (lambda^k): the raw nodes, weighted by k_res_combine
        if (nsmp > 0) {
          float* raw = p.raw + ((size_t)it * gridDim.y + slot) * p.nraw + sb;
          const float* sf = reinterpret_cast<const float*>(su);
          for (int e = tid; e < nsmp; e += NT) raw[e] = sf[__ldg(p.smp_loc + (size_t)slot * p.smp_locslot + sb + e)];
        }
      }
      const int r0 = strip(ph);
      // the y taps come from a window of 2R + 1 rows that slides down the strip
      const float4* col = su + r0 * SW + NL + tx;     // row r0 - R of the column
      float4 W[RY + 2 * R];
#pragma unroll
      for (int r = 0; r < 2 * R; ++r) W[r] = col[r * SW];
#pragma unroll
      for (int iy = 0; iy < RY; ++iy) {
        const int i = ph * RY + iy;
        const int row = r0 + iy;
        W[iy + 2 * R] = col[(iy + 2 * R) * SW];
        float4 kq;
        if (KREG) kq = kk[i];
        else kq = ldg4(p.kf + pixc + off[i]);
        float4 inv = z4;   // 1 / (1 + a) in the sponge
        float ay = 0.f;
        if (spm >> i & 1) {
          inv = ldg4(p.inv + pixc + off[i]);
          ay = __ldg(p.spy + y0 + row);
        }
        const float4 cen = W[iy + R];
        const float2 c0 = lo2(cen), c1 = hi2(cen);
        const float4* xr = su + (row + R) * SW + tx;
        float v[NV];
#pragma unroll
        for (int q = 0; q <= 2 * NL; ++q) put4(q == NL ? cen : xr[q], v + 4 * q);
        // second derivatives in the zero-sum form sum_j w_j (u_{+j} + u_{-j} - 2 u_0);
        // the sums of even x taps fall on aligned pairs and run packed
        float2 a0 = make_float2(0.f, 0.f), a1 = a0;
#pragma unroll
        for (int j = 1; j <= R; ++j) {
          const float w2 = p.wx.w2[j];
          if (j & 1) {
            a0.x = fmaf(w2, fmaf(-2.f, v[C], v[C + j] + v[C - j]), a0.x);
            a0.y = fmaf(w2, fmaf(-2.f, v[C + 1], v[C + 1 + j] + v[C + 1 - j]), a0.y);
            a1.x = fmaf(w2, fmaf(-2.f, v[C + 2], v[C + 2 + j] + v[C + 2 - j]), a1.x);
            a1.y = fmaf(w2, fmaf(-2.f, v[C + 3], v[C + 3 + j] + v[C + 3 - j]), a1.y);
          } else {
            axpy2(a0, w2, sec2(add2(make_float2(v[C + j], v[C + 1 + j]), make_float2(v[C - j], v[C + 1 - j])), c0));
            axpy2(a1, w2, sec2(add2(make_float2(v[C + 2 + j], v[C + 3 + j]), make_float2(v[C + 2 - j], v[C + 3 - j])), c1));
          }
        }
        if (VD && (bxm >> i & 1)) {
          // forward: - b_x D1x u; adjoint: D1x(b_x lambda)
          float px[ADJ ? NV : 1];
          if (ADJ) {
            const float4* br = s_bx + row * SW + tx;
#pragma unroll
            for (int q = 0; q <= 2 * NL; ++q)
              put4(mul4(br[q], make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3])), px + 4 * q);
          }
          const float* dw = ADJ ? px : v;
          float2 d0 = make_float2(0.f, 0.f), d1 = d0;
#pragma unroll
          for (int j = 1; j <= R; ++j) {
            const float w1 = p.wx.w1[j];
            if (j & 1) {
              d0.x = fmaf(w1, dw[C + j] - dw[C - j], d0.x);
              d0.y = fmaf(w1, dw[C + 1 + j] - dw[C + 1 - j], d0.y);
              d1.x = fmaf(w1, dw[C + 2 + j] - dw[C + 2 - j], d1.x);
              d1.y = fmaf(w1, dw[C + 3 + j] - dw[C + 3 - j], d1.y);
            } else {
              axpy2(d0, w1, dif2(make_float2(dw[C + j], dw[C + 1 + j]), make_float2(dw[C - j], dw[C + 1 - j])));
              axpy2(d1, w1, dif2(make_float2(dw[C + 2 + j], dw[C + 3 + j]), make_float2(dw[C + 2 - j], dw[C + 3 - j])));
            }
          }
          if (ADJ) {
            a0 = add2(a0, d0);
            a1 = add2(a1, d1);
          } else {
            const float4 b = s_bx[row * 32 + tx];
            a0 = __ffma2_rn(lo2(b), d0, a0);
            a1 = __ffma2_rn(hi2(b), d1, a1);
          }
        }
#pragma unroll
        for (int j = 1; j <= R; ++j) {
          const float4 a = W[iy + R - j], c = W[iy + R + j];
          axpy2(a0, p.wy.w2[j], sec2(add2(lo2(a), lo2(c)), c0));
          axpy2(a1, p.wy.w2[j], sec2(add2(hi2(a), hi2(c)), c1));
        }
        if (VD && ((ADJ ? bym : bxm) >> i & 1)) {
          // forward: - b_y D1y u; adjoint: D1y(b_y lambda)
          float2 e0 = make_float2(0.f, 0.f), e1 = e0;
          const float4* bcol = s_by + (row + R) * 32 + tx;   // adjoint: row 0 of the column
#pragma unroll
          for (int j = 1; j <= R; ++j) {
            float4 a = W[iy + R - j], c = W[iy + R + j];
            if (ADJ) {
              a = mul4(bcol[-j * 32], a);
              c = mul4(bcol[j * 32], c);
            }
            axpy2(e0, p.wy.w1[j], dif2(lo2(c), lo2(a)));
            axpy2(e1, p.wy.w1[j], dif2(hi2(c), hi2(a)));
          }
          if (ADJ) {
            a0 = add2(a0, e0);
            a1 = add2(a1, e1);
          } else {
            const float4 b = s_by[row * 32 + tx];
            a0 = __ffma2_rn(lo2(b), e0, a0);
            a1 = __ffma2_rn(hi2(b), e1, a1);
          }
        }
        // the update; u^{n+1} replaces u^{n-1}
        float4* own = so + (row + R) * SW + NL + tx;
        const float4 uo = *own;
        const float2 c20 = add2(c0, c0), c21 = add2(c1, c1);
        float2 h0, h1;
        if (rare >> i & 1) {
          if (injm >> i & 1) {   // this cell's sources (residuals), in the table's order
            float acc[4] = {a0.x, a0.y, a1.x, a1.y};
            const unsigned ce = s_cell[row * 32 + tx];
            const int last = (int)(ce & 0xffffu) + (int)(ce >> 16);
            for (int e = (int)(ce & 0xffffu); e < last; ++e) {
              const int ix = s_ix[e];
              const float val = sval[e];
#pragma unroll
              for (int q = 0; q < 4; ++q) acc[q] += (q == ix) ? val : 0.f;
            }
            a0 = make_float2(acc[0], acc[1]);
            a1 = make_float2(acc[2], acc[3]);
          }
          h0 = __fmul2_rn(lo2(kq), a0);
          h1 = __fmul2_rn(hi2(kq), a1);
          float4 r4;
          if (spm >> i & 1) {   // sponge
            auto upd = [&](float a, float u, float c2, float h, float r) {
              return __fadd_rn(fmaf(-(1.f - a), u, c2), h) * r;
            };
            r4 = make_float4(upd(ax4.x + ay, uo.x, c20.x, h0.x, inv.x), upd(ax4.y + ay, uo.y, c20.y, h0.y, inv.y),
                             upd(ax4.z + ay, uo.z, c21.x, h1.x, inv.z), upd(ax4.w + ay, uo.w, c21.y, h1.y, inv.w));
          } else {
            const float2 q0 = add2(dif2(c20, lo2(uo)), h0), q1 = add2(dif2(c21, hi2(uo)), h1);
            r4 = make_float4(q0.x, q0.y, q1.x, q1.y);
          }
          *own = r4;
          if (nsm >> i & 1) {   // the tile's outer rows
            st_tagged(hasN && row < R, exw + (size_t)(row * 32 + tx) * 4, r4, tag);
            st_tagged(hasS && row >= TH - R, exw + (size_t)((2 * R + row - TH) * 32 + tx) * 4, r4, tag);
          }
        } else {
          h0 = __fmul2_rn(lo2(kq), a0);
          h1 = __fmul2_rn(hi2(kq), a1);
          const float2 q0 = add2(dif2(c20, lo2(uo)), h0), q1 = add2(dif2(c21, hi2(uo)), h1);
          *own = make_float4(q0.x, q0.y, q1.x, q1.y);
        }
        if (PH == 1) st_tagged(ew, exw + (ewc + row * (4 * NL)), so[(row + R) * SW + NL + tx], tag);
        if (!ADJ) {
          if (p.hist) __stcs(reinterpret_cast<float4*>(hrow + off[i]), make_float4(h0.x, h0.y, h1.x, h1.y));
        } else if (img) {
          // this phase's h was requested a step ago (two phases: one younger group is in flight)
          if (iy == 0) asm volatile("cp.async.wait_group %0;" ::"n"(PH - 1) : "memory");
          const float4 h = s_h[row * 32 + tx];
          float4 g = GREG ? gg[i] : s_g[row * 32 + tx];
          g.x = fmaf(-cen.x, h.x, g.x);
          g.y = fmaf(-cen.y, h.y, g.y);
          g.z = fmaf(-cen.z, h.z, g.z);
          g.w = fmaf(-cen.w, h.w, g.w);
          if (GREG) gg[i] = g;
          else s_g[row * 32 + tx] = g;
        }
        if (PH == 2 && iy == 0) {   // ask for the next phase's halo words
          const int np = ph ^ 1;
          const unsigned pr = ph == 0 ? (it & 1) : ((it + 1) & 1);
          if (dst[np * NTASK] >= 0) ld_words(ex0 + src[np * NTASK] + pr * par, ahead);
        }
      }
      if (ADJ) {   // h of the next step into the same (own) cells
        const int nx_ = it + 1;
        if (nx_ < p.steps && nx_ >= p.img0) {
          const float* h = p.hist + fo - (long long)(nx_ - p.img0) * p.hstride;
#pragma unroll
          for (int iy = 0; iy < RY; ++iy)
            cp_async16(s_h + (r0 + iy) * 32 + tx, h + pixc + off[ph * RY + iy]);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
      }
    }
    if (it + 1 < p.steps) {
      float* nv = s_val + ((it + 1) & 1) * p.nval;
      if (tid < ne) nv[tid] = nval;
      for (int e = tid + NT; e < ne; e += NT)
        nv[e] = __ldg(p.inj_w + eb + e) * p.vals[p.inj_vidx[eb + e] + p.voff + (it + 1) * p.vstep];
    }
  }
  // A launch of one step has received nothing yet: wait for the neighbours' words,
  // so that no tile is written back before its neighbours have read it (a word is
  // sent after its tile is staged).  Each thread waits for its own cells only, hence
  // the barrier; longer launches have passed one behind the receive of their steps.  (On
  // time-out the flag makes the call an error; an early return here cost one instantiation
  // 5% of its step.)
  if (p.steps == 1) {
    bool ok = true;
    if (PH == 2) {
      __syncthreads();
      send_columns(1, s_u1, 1u, p.tag0 + 1);
    }
#pragma unroll
    for (int ph = 0; ph < PH; ++ph) ok = receive(ph, s_u1, 1u, p.tag0 + 1, ahead, false) && ok;
    if (!ok && p.flags) atomicOr(p.flags, 2);
    __syncthreads();
  }
  // ---- state back to global memory: u^{n+steps} and u^{n+steps-1}
  const float4* fu = (p.steps & 1) ? s_u1 : s_u0;
  const float4* fp = (p.steps & 1) ? s_u0 : s_u1;
#pragma unroll
  for (int i = 0; i < PH * RY; ++i) {
    if (!(inb >> i & 1)) continue;
    const int row = strip(i / RY) + i % RY;
    const int si = (row + R) * SW + NL + tx;
    const size_t gi = fo + pixc + row * p.sx;
    *reinterpret_cast<float4*>(p.u_out + gi) = fu[si];
    *reinterpret_cast<float4*>(p.up_out + gi) = fp[si];
    if (ADJ) *reinterpret_cast<float4*>(p.g + gi) = GREG ? gg[i] : s_g[row * 32 + tx];
  }
}

// inv = 1 / (1 + a), a the sponge's damping of the leapfrog update.
__global__ void k_res_inv(const float* __restrict__ spx, const float* __restrict__ spy, int nx, int ny, int sx,
                          int ox, int oy, float* __restrict__ inv) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
  if (x < nx && y < ny) inv[(size_t)(y + oy) * sx + x + ox] = __frcp_rn(1.f + (spx[x] + spy[y]));
}

// Weighted samples of `steps` time steps from the raw node values: the
// arithmetic of sample_receivers (one thread per linear point, a warp with
// shuffles per sinc point).
__global__ void k_res_combine(const float* __restrict__ raw, int nraw, int nslots, int steps,
                              const int* __restrict__ node, const float* __restrict__ w, int slot_nodes,
                              int npt, int nc, int grp, float* __restrict__ out, long long out_step,
                              long long out_slot) {
  const long long gid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long pt = gid / grp;
  const int lane = (int)(gid - pt * grp);
  const bool on = pt < (long long)steps * nslots * npt;
  float acc = 0.f;
  int r = 0, s = 0, n = 0;
  if (on) {
    r = (int)(pt % npt);
    const long long q = pt / npt;
    s = (int)(q % nslots);
    n = (int)(q / nslots);
    const float* rb = raw + ((long long)n * nslots + s) * nraw;
    const int* nd = node + (long long)s * slot_nodes + (long long)r * nc;
    const float* wr = w + (long long)s * slot_nodes + (long long)r * nc;
    for (int c = lane; c < nc; c += grp) acc = fmaf(wr[c], rb[nd[c]], acc);
  }
  if (grp > 1)
    for (int o = grp / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (on && lane == 0) out[(long long)n * out_step + (long long)s * out_slot + r] = acc;
}

template <int R, bool VD, bool ADJ, int PH, int RY>
cudaError_t launch_t(const ResParams& p, int nty, int nslots, cudaStream_t st) {
  const size_t smem = res2d_smem(R, VD, ADJ, p.TH, p.nval);
  // the most a CTA may have: a plan's own size here would lower the limit under
  // another thread's launch of a larger one
  static DeviceOnce once;
  const cudaError_t attr = allow_smem(once, k_res2d<R, VD, ADJ, PH, RY>, 0);
  if (attr != cudaSuccess) return attr;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(p.P, nslots);
  cfg.blockDim = dim3(32, nty);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_res2d<R, VD, ADJ, PH, RY>, p);
}

template <int R, bool VD, bool ADJ>
cudaError_t launch_ry(const ResParams& p, int ph, int ry, int nty, int nslots, cudaStream_t st) {
  if (ph == 1) return launch_t<R, VD, ADJ, 1, 1>(p, nty, nslots, st);
  return ry == 1 ? launch_t<R, VD, ADJ, 2, 1>(p, nty, nslots, st)
                 : launch_t<R, VD, ADJ, 2, 2>(p, nty, nslots, st);
}

}  // namespace

int res2d_warps() { return RES_WARPS; }

int res2d_cells(int R, int TH) { return R <= 4 ? ResGeo<4>::cells(TH) : ResGeo<5>::cells(TH); }

size_t res2d_smem(int R, bool vd, bool adj, int TH, int nval) {
  const int NL = R <= 4 ? 1 : 2, SW = 32 + 2 * NL, SH = TH + 2 * R;
  size_t n = 2 * (size_t)SH * SW;
  if (adj) n += (size_t)TH * 32 + (vd ? (size_t)TH * SW + (size_t)SH * 32 + (size_t)TH * 32 : 0);
  else if (vd) n += 2 * (size_t)TH * 32;
  return n * 16 + (size_t)TH * 32 * 4 + 2 * (size_t)nval * 4 + ((size_t)nval + 15) / 16 * 16;
}

cudaError_t launch_res2d(const ResParams& p, int R, bool vd, bool adj, int ph, int ry, int nty, int nslots,
                         cudaStream_t st) {
  if (R == 4) {
    if (vd) return adj ? launch_ry<4, true, true>(p, ph, ry, nty, nslots, st)
                       : launch_ry<4, true, false>(p, ph, ry, nty, nslots, st);
    return adj ? launch_ry<4, false, true>(p, ph, ry, nty, nslots, st)
               : launch_ry<4, false, false>(p, ph, ry, nty, nslots, st);
  }
  if (vd) return adj ? launch_ry<5, true, true>(p, ph, ry, nty, nslots, st)
                     : launch_ry<5, true, false>(p, ph, ry, nty, nslots, st);
  return adj ? launch_ry<5, false, true>(p, ph, ry, nty, nslots, st)
             : launch_ry<5, false, false>(p, ph, ry, nty, nslots, st);
}

cudaError_t launch_res_inv(const Layout& L, const float* spx, const float* spy, float* inv, cudaStream_t st) {
  k_res_inv<<<dim3((L.nx_r + 127) / 128, L.ny), 128, 0, st>>>(spx, spy, L.nx_r, L.ny, L.sx, L.ox, L.oy, inv);
  return cudaGetLastError();
}

cudaError_t launch_res_combine(const float* raw, int nraw, int nslots, int steps, const int* node,
                               const float* w, int slot_nodes, int npt, int nc, int grp, float* out,
                               long long out_step, long long out_slot, cudaStream_t st) {
  const long long n = (long long)steps * nslots * npt * grp;
  if (n <= 0) return cudaSuccess;
  k_res_combine<<<(unsigned)((n + 127) / 128), 128, 0, st>>>(raw, nraw, nslots, steps, node, w, slot_nodes,
                                                             npt, nc, grp, out, out_step, out_slot);
  return cudaGetLastError();
}

}  // namespace fwi
