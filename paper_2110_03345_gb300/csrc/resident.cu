// Host side of the resident 2D kernels (kernels2d_res.cu): the choice of tile
// and shots per launch, the sampling lists, and the runs of steps.
#include "fwi_plan.cuh"

namespace fwi {

namespace {

constexpr size_t RES_SMEM = 232448;        // shared memory of one CTA (227 KB)
constexpr size_t RES_RAW = 8u << 20;       // floats of raw samples held at most
constexpr int RES_CHUNK = 512;             // steps per launch at most

// Most injection entries of one tile of 128 x TH: every point's w x w nodes,
// w = 2 (linear) or 8 (sinc), from its first node.
int most_entries(const fwi_plan* P, const double* xyz, long long n, int TH, int gx, int gy) {
  const int w = P->opt.interp == FWI_INTERP_SINC ? 2 * FWI_SINC_RADIUS : 2;
  const int back = w / 2 - 1;
  std::vector<int> cnt((size_t)gx * gy, 0);
  int most = 0;
  for (long long i = 0; i < n; ++i) {
    const int y = (int)std::floor(xyz[2 * i] / P->h[1]) - back;
    const int x = (int)std::floor(xyz[2 * i + 1] / P->h[0]) - back;
    for (int by = std::max(y - 1, 0) / TH; by <= (y + w) / TH && by < gy; ++by)
      for (int bx = std::max(x - 1, 0) / TILE_X; bx <= (x + w) / TILE_X && bx < gx; ++bx) {
        const int rows = std::min(y + w + 1, (by + 1) * TH) - std::max(y - 1, by * TH);
        const int cols = std::min(x + w + 1, (bx + 1) * TILE_X) - std::max(x - 1, bx * TILE_X);
        if (rows > 0 && cols > 0) {
          int& c = cnt[(size_t)by * gx + bx];
          c += std::min(rows, w) * std::min(cols, w);
          most = std::max(most, c);
        }
      }
  }
  return most;
}

}  // namespace

// Whether a call of B shots may run resident.  A resident shot costs the same
// whatever the number of shots; the per-step kernels' cost per shot falls as CTAs
// of several shots fill the SMs (one and two shots: the figures of kernels2d_res.cu;
// two shots of 1024 x 1024 with density 8.4 -> 7.1 us per forward step and 22.0 -> 18.0 per
// step pair).  Above 8 tile-shots (128 x 16 points) per SM for forward runs and 12.5 for
// gradients the per-step kernels are as good in most calls (per-step / resident there
// 0.77 - 1.14); below, choose_res compares the two (resident_pays).
bool res_eligible(const fwi_plan* P, bool grad, int B, const Scheme& sc) {
  if (P->grid.ndim != 2 || sc.ext() || P->fixed_memory || P->per_step || P->opt.tile != 0 ||
      P->opt.shots_per_cta != 0 || B < 1 || P->nt < 2)
    return false;
  int id = 0, shape = 0;
  bool tma = false;
  return resolve_tile(P, 0, &id, &shape, &tma) &&
         2LL * tile_geo(P, shape, true).ntiles() * B <= (grad ? 25LL : 16LL) * P->nsm;
}

namespace {

// Floats of raw samples kept for B shots: all steps of the shots side by side
// (each has one CTA at least), or what the limit allows.
size_t raw_floats(const fwi_plan* P, const fwi_geometry* g, int B) {
  const size_t ne = (size_t)std::max(g->nrec, g->nsrc) * interp_nodes(P->opt.interp, 2) * std::min(B, P->nsm);
  return std::min(RES_RAW, ne * (size_t)P->nt);
}

// Words of the halo exchange of all CTAs of a launch (two parities).
size_t exchange_words(const fwi_plan* P) {
  return (size_t)P->nsm * 2 * res2d_cells(P->R, 4 * res2d_warps()) * 4;
}

}  // namespace

size_t res_buffers(const fwi_plan* P, const fwi_geometry* g, int B) {
  return raw_floats(P, g, B) * 4 + exchange_words(P) * 8 + (size_t)P->L.fstride * 4 + 1024;
}

// Tile height: a step takes about t0 + t1 TH (t0: the exchange and the
// barriers; t1: a row of 128 points on one SM; in units of 18 ns), and B shots
// take ceil(B / conc) launches of conc shots each.
void choose_res(const fwi_plan* P, const fwi_geometry* g, bool vd, bool grad, int B, int K, const Scheme& sc,
                ResPlan* out) {
  *out = ResPlan();
  if (!res_eligible(P, grad, B, sc) || !resident_run(P->nt, K, grad)) return;
  const int gx = (P->L.nx + TILE_X - 1) / TILE_X;
  const int nc = interp_nodes(P->opt.interp, 2);
  double best = 0.0;
  ResPlan r;
  const struct { int ph, ry; double t0, t1; } var[3] = {{1, 1, 70.0, 1.0}, {2, 1, 90.0, 1.5}, {2, 2, 75.0, 1.85}};
  for (const auto& v : var)
    for (int nty = 1; nty <= res2d_warps(); ++nty) {
      const int TH = v.ph * v.ry * nty;
      if (TH < v.ph * P->R) continue;   // the outer rows lie within a phase's half
      const int gy = (P->L.ny + TH - 1) / TH;
      if ((long long)gx * gy > P->nsm) continue;
      if (res2d_smem(P->R, vd, grad, TH, 64) > RES_SMEM || res2d_smem(P->R, vd, false, TH, 64) > RES_SMEM) continue;
      // every thread receives at most three halo cells (one per phase of two)
      const int cells = res2d_cells(P->R, TH);
      if (v.ph == 1 ? cells > 3 * 32 * nty : cells > 2 * 32 * nty) continue;
      const int conc = std::min(B, P->nsm / (gx * gy));
      const double t = (double)((B + conc - 1) / conc) * (v.t0 + v.t1 * TH);
      if (!r.on || t < best) {
        best = t;
        r.on = true;
        r.gx = gx;
        r.gy = gy;
        r.ph = v.ph;
        r.ry = v.ry;
        r.nty = nty;
        r.TH = TH;
        r.P = gx * gy;
        r.conc = conc;
      }
    }
  if (!r.on) return;
  int id = 0, shape = 0;
  bool tma = false;
  double shot_times = 0.0;
  if (!resolve_tile(P, 0, &id, &shape, &tma)) return;
  shot_group(P->nsm, {{tile_geo(P, shape, true).ntiles(), B}}, GROUP_TAIL, &shot_times);
  if (!resident_pays(best, shot_times, grad, vd)) return;
  int nval = 0;
  for (int s = 0; s < g->nshots; ++s)
    nval = std::max(nval, most_entries(P, g->src_xyz + (size_t)s * g->nsrc * 2, g->nsrc, r.TH, r.gx, r.gy));
  if (grad) nval = std::max(nval, most_entries(P, g->rec_xyz, g->nrec, r.TH, r.gx, r.gy));
  r.nval = nval;
  if (nval > 65535 || res2d_smem(P->R, vd, grad, r.TH, nval) > RES_SMEM ||
      res2d_smem(P->R, vd, false, r.TH, nval) > RES_SMEM)
    return;
  // raw samples: at least 16 steps of every concurrent shot
  r.raw = raw_floats(P, g, B);
  if ((size_t)std::max(g->nrec, g->nsrc) * nc * r.conc * std::min(P->nt, 16) > r.raw) return;
  r.ex = exchange_words(P);
  r.inv = (size_t)P->L.fstride;
  *out = r;
}

// Lists of the nodes each CTA samples (nodes3: x, y, z of `slots` equal sets
// of nodes) and their places in a raw row.
fwi_status res_sample_table(Call& c, const std::vector<int>& nodes3, int slots, Carve& C, ResSamples* out) {
  fwi_plan* P = c.P;
  const ResPlan& r = c.pl.res;
  const int n = (int)(nodes3.size() / 3) / slots;   // nodes of one slot
  const int XH = P->R <= 4 ? 4 : 8, sw = TILE_X + 2 * XH;
  std::vector<int> off((size_t)slots * (r.P + 1), 0), loc((size_t)slots * n), pos((size_t)slots * n);
  for (int s = 0; s < slots; ++s) {
    int* o = off.data() + (size_t)s * (r.P + 1);
    auto cta = [&](int i) {
      const int* q = &nodes3[3 * ((size_t)s * n + i)];
      return (q[1] / r.TH) * r.gx + q[0] / TILE_X;
    };
    for (int i = 0; i < n; ++i) o[cta(i) + 1]++;
    for (int t = 0; t < r.P; ++t) o[t + 1] += o[t];
    std::vector<int> at(o, o + r.P);
    for (int i = 0; i < n; ++i) {
      const int* q = &nodes3[3 * ((size_t)s * n + i)];
      const int k = at[cta(i)]++;
      pos[(size_t)s * n + i] = k;
      loc[(size_t)s * n + k] = (q[1] % r.TH + P->R) * sw + XH + q[0] % TILE_X;
    }
  }
  int* d_off = C.take<int>(off.size());
  int* d_loc = C.take<int>(loc.size());
  int* d_pos = C.take<int>(pos.size());
  CUDA_TRY(cudaMemcpyAsync(d_off, off.data(), off.size() * 4, cudaMemcpyHostToDevice, P->st));
  CUDA_TRY(cudaMemcpyAsync(d_loc, loc.data(), loc.size() * 4, cudaMemcpyHostToDevice, P->st));
  CUDA_TRY(cudaMemcpyAsync(d_pos, pos.data(), pos.size() * 4, cudaMemcpyHostToDevice, P->st));
  out->off = d_off;
  out->loc = d_loc;
  out->pos = d_pos;
  out->nraw = n;
  return FWI_OK;
}

namespace {

ResParams res_params(const Call& c) {
  const fwi_plan* P = c.P;
  const ResPlan& r = c.pl.res;
  ResParams p{};
  p.kf = c.W.kf;
  p.bx = c.W.bx;
  p.by = c.W.by;
  p.spx = P->spx;
  p.spy = P->spy;
  p.inv = c.W.INV;
  p.fstride = P->L.fstride;
  p.hstride = P->L.fstride * c.pl.B;
  p.wx = P->wx;
  p.wy = P->wy;
  p.sx = P->L.sx;
  p.nx = P->L.nx;
  p.ny = P->L.ny;
  p.ox = P->L.ox;
  p.oy = P->L.oy;
  p.gx = r.gx;
  p.gy = r.gy;
  p.P = r.P;
  p.TH = r.TH;
  p.nval = r.nval;
  p.ex = c.W.EX;
  p.flags = P->d_flags + 1;
  return p;
}

// Steps [m0, m0 + n) of the running count that profile = every times.
int64_t timed_steps(int64_t m0, int n, int every) {
  auto upto = [&](int64_t m) { return (m + every - 1) / every; };   // multiples of `every` below m
  return upto(m0 + n) - upto(m0);
}

fwi_status res_launch(Call& c, ResParams& p, bool adj, int slots) {
  fwi_plan* P = c.P;
  p.tag0 = c.tag;
  c.tag += (unsigned)p.steps;
  const bool prof = P->opt.profile > 0;
  if (prof) FWI_TRY(record_event(P, adj ? 1 : 0));
  cudaError_t e = launch_res2d(p, P->R, c.vd, adj, c.pl.res.ph, c.pl.res.ry, c.pl.res.nty, slots, P->st);
  if (e != cudaSuccess) return fail(FWI_ERR_CUDA, std::string("resident launch: ") + cudaGetErrorString(e));
  if (prof) FWI_TRY(record_event(P, adj ? 1 : 0));
  c.launches++;
  return FWI_OK;
}

void res_count(Call& c, bool adj, int nb, int steps) {
  const int64_t pts = (int64_t)nb * c.P->L.nx * c.P->L.ny * steps;
  const int64_t timed = c.P->opt.profile > 0
                            ? timed_steps(c.fwd_launches + c.adj_launches, steps, c.P->opt.profile) : 0;
  (adj ? c.adj_timed : c.fwd_timed) += timed;
  (adj ? c.adj_launches : c.fwd_launches) += steps;
  (adj ? c.adj_points : c.fwd_points) += pts;
}

}  // namespace

fwi_status res_forward_steps(Call& c, int nb, const DevTable& src, float* A, float* Bf, int n0, int n1,
                             float* hist, bool sample) {
  fwi_plan* P = c.P;
  const ResPlan& r = c.pl.res;
  const size_t fs = (size_t)P->L.fstride;
  const int nraw = c.rsmp.nraw;
  const int most = sample ? (int)std::min<size_t>(RES_CHUNK, r.raw / ((size_t)nraw * r.conc)) : RES_CHUNK;
  for (int n = n0; n < n1;) {
    const int steps = std::min(n1 - n, std::max(most, 1));
    for (int s0 = 0; s0 < nb; s0 += r.conc) {
      const int m = std::min(r.conc, nb - s0);
      ResParams p = res_params(c);
      p.u = p.u_out = A + s0 * fs;
      p.up = p.up_out = Bf + s0 * fs;
      p.hist = hist ? hist + (size_t)(n - n0) * p.hstride + s0 * fs : nullptr;
      p.inj_off = src.off + (size_t)s0 * r.P;
      p.inj_loc = src.loc;
      p.inj_vidx = src.vidx;
      p.inj_w = src.w;
      p.vals = c.wavelet;
      p.voff = n;
      p.vstep = 1;
      p.steps = steps;
      if (sample) {
        p.smp_off = c.rsmp.off;
        p.smp_loc = c.rsmp.loc;
        p.raw = c.W.RAW;
        p.nraw = nraw;
      }
      FWI_TRY(res_launch(c, p, false, m));
      if (sample) {
        const long long row = (long long)c.pl.B * c.geom->nrec;
        cudaError_t e = launch_res_combine(c.W.RAW, nraw, m, steps, c.rsmp.pos, c.smp_w, 0, c.geom->nrec,
                                           c.ncorner, sample_group(c.ncorner),
                                           c.D + n * row + (long long)s0 * c.geom->nrec, row, c.geom->nrec,
                                           P->st);
        if (e != cudaSuccess) return fail(FWI_ERR_CUDA, cudaGetErrorString(e));
        c.launches++;
      }
    }
    n += steps;
  }
  res_count(c, false, nb, n1 - n0);
  return FWI_OK;
}

fwi_status res_adjoint_steps(Call& c, int nb, float* LA, float* LB, int k0, int k1, bool image_first,
                             float* hist) {
  fwi_plan* P = c.P;
  const ResPlan& r = c.pl.res;
  const size_t fs = (size_t)P->L.fstride;
  const int nsrc = c.geom->nsrc, nrec = c.geom->nrec;
  const int nraw = c.wsmp.nraw;
  const int most = c.Dw ? (int)std::min<size_t>(RES_CHUNK, r.raw / ((size_t)nraw * r.conc)) : RES_CHUNK;
  const long long row = (long long)c.pl.B * nrec;
  bool img = image_first;
  for (int k = k0; k >= k1;) {
    const int steps = std::min(k - k1 + 1, std::max(most, 1));
    const int img0 = img ? 0 : 1;
    for (int s0 = 0; s0 < nb; s0 += r.conc) {
      const int m = std::min(r.conc, nb - s0);
      ResParams p = res_params(c);
      p.u = p.u_out = LA + s0 * fs;
      p.up = p.up_out = LB + s0 * fs;
      p.g = c.W.G + s0 * fs;
      p.img0 = img0;
      p.nimg = hist ? steps - img0 : 0;
      p.hist = hist ? hist + s0 * fs : nullptr;
      p.inj_off = c.rec_tab.off + (size_t)s0 * r.P;
      p.inj_loc = c.rec_tab.loc;
      p.inj_vidx = c.rec_tab.vidx;
      p.inj_w = c.rec_tab.w;
      p.vals = c.D;
      p.voff = (long long)k * row;
      p.vstep = -row;
      p.steps = steps;
      if (c.Dw) {   // lambda^k at the sources
        p.smp_off = c.wsmp.off + (size_t)s0 * (r.P + 1);
        p.smp_loc = c.wsmp.loc + (size_t)s0 * nraw;
        p.smp_slot = r.P + 1;
        p.smp_locslot = nraw;
        p.raw = c.W.RAW;
        p.nraw = nraw;
      }
      FWI_TRY(res_launch(c, p, true, m));
      if (c.Dw) {
        const long long wrow = (long long)c.pl.B * nsrc;
        cudaError_t e = launch_res_combine(c.W.RAW, nraw, m, steps, c.wsmp.pos + (size_t)s0 * nraw,
                                           c.ws_w + (size_t)s0 * nraw, nraw, nsrc, c.ncorner,
                                           sample_group(c.ncorner), c.Dw + k * wrow + (long long)s0 * nsrc,
                                           -wrow, nsrc, P->st);
        if (e != cudaSuccess) return fail(FWI_ERR_CUDA, cudaGetErrorString(e));
        c.launches++;
      }
    }
    if (hist) hist -= (long long)(steps - img0) * P->L.fstride * c.pl.B;
    img = true;
    k -= steps;
  }
  res_count(c, true, nb, k0 - k1 + 1);
  return FWI_OK;
}

}  // namespace fwi
