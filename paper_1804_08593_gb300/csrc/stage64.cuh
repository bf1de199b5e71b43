// The FP64 operator stage: the same operation as stage.cuh's stage kernel (out = hop_scale *
// [Post * Dh(in)] + [Loc * in2], optional residual update and norm) for FP64 storage.
//
// What bounds it.  GB300 issues two FP64 lanes per clock and SM (1.255 TFLOP/s measured with
// independent FMAs; a quarter of an SM takes 64 cycles per warp-wide FP64 instruction), so a
// site and slice's ~900 FP64 instructions are the time of a stage: memory, shared memory and
// integer work hide behind a handful of warps.  Two things follow.
//
//  * The number of FP64 instructions is what counts.  Projections and reconstructions multiply
//    by +-1 inside the FMA that adds; which component, real or imaginary part, and sign a
//    direction needs is selected by integer moves, so that one piece of code serves the four
//    directions.  The fifth-dimension recurrence runs with its constant factors folded on the
//    host (4 instructions per element instead of 7), scalings by 1 are left out.  (Taking
//    g_f + g_b and g_b - g_f from one FMA chain would save another 12 of 216 instructions per
//    direction pair and 5 % of the time, but turns infinite inputs into NaNs.)
//  * Work has to reach every quarter of every SM.  A CTA is 2^lst sites x Ls slices, x DS = 16
//    groups of threads (direction and half-spinor component) on lattices too small to fill
//    the chip with whole hops; lst and DS are chosen at launch (stage64_shape).
//
// Measured, us per launch of the stage with the recurrence post (before: one CTA per 32 sites,
// every instruction above): 4^4 x 8 74 -> 7, 8^3x16 x 8 74 -> 59, 12^4 x 12 325 -> 224,
// 16^4 x 16 1020 -> 870 (92 % of the FP64 rate on the instructions left), 16^3x32 x 12
// 1498 -> 1298.
#pragma once

#include "stage.cuh"

namespace dwf {

__device__ __forceinline__ double2 sel_swap(double2 v, bool swap) {
  return swap ? make_double2(v.y, v.x) : v;
}

// Component i of the projected half-spinor in direction mu: (1 + sg gamma_mu) =
// [[1, sg B], [sg B^dag, 1]]; (B psi_dn)_i takes spin 3 - i (x and y) or 2 + i (z and t), whose
// first component is kp, with real and imaginary part swapped for x and z, times the signs m.
// B^dag feeds the product g_i to spin 2 (`two`) or 3, swapped alike, times the signs n.
struct HalfSpin {
  int kp;
  bool swap, two;
  double mx, my, nx, ny;
};
__device__ __forceinline__ HalfSpin half_spin(int mu, int i) {
  HalfSpin h;
  h.swap = (mu & 1) == 0;
  h.kp = mu < 2 ? 9 - 3 * i : 6 + 3 * i;
  h.mx = i == 0 ? (mu == 1 ? -1.0 : 1.0) : (mu == 2 ? -1.0 : 1.0);
  h.my = i == 0 ? (mu == 3 ? 1.0 : -1.0) : (mu == 0 ? -1.0 : 1.0);
  h.two = (mu < 2) == (i == 1);
  h.nx = h.two ? (h.swap ? -1.0 : 1.0) : (mu < 2 ? -1.0 : 1.0);
  h.ny = h.two ? 1.0 : ((mu == 1 || mu == 2) ? -1.0 : 1.0);
  return h;
}

// h = the projected component of the neighbour at q (site stride v), sg the sign of gamma; zero
// where the neighbour is absent.
__device__ __forceinline__ void project64(cx<double> (&h)[3], const HalfSpin& f, int i,
                                          const double2* q, long v, bool has, double sg) {
#pragma unroll
  for (int a = 0; a < 3; a++) {
    h[a] = {0.0, 0.0};
    if (has) {
      const double2 p = __ldg(q + (3 * i + a) * v);
      const double2 b = sel_swap(__ldg(q + (f.kp + a) * v), f.swap);
      h[a] = {fma(sg * f.mx, b.x, p.x), fma(sg * f.my, b.y, p.y)};
    }
  }
}

// The hop in the directions +mu and -mu at one site and slice for both components:
// up[i] += g_f + g_b (spin i), lo[i] += B^dag (g_b - g_f) (spin 3 - i for x and y, 2 + i for z
// and t).  qf, qb: the slice's first chunk of the neighbour in the two directions, site stride
// vf, vb (the blocked operators' halo neighbours live in another array); has: the neighbour
// takes part; L: the link of direction 2 mu at this site, chunk stride vl.
template <bool DAG>
__device__ __forceinline__ void hop64_pair(cx<double> (&up)[2][3], cx<double> (&lo)[2][3],
                                           int mu, const double2* qf, long vf, bool has_f,
                                           const double2* qb, long vb, bool has_b,
                                           const double2* L, long vl) {
  const HalfSpin f[2] = {half_spin(mu, 0), half_spin(mu, 1)};
  constexpr double F = DAG ? 1.0 : -1.0;   // sign of gamma in the forward hop
  cx<double> h[2][3], gf[2][3];
#pragma unroll
  for (int n = 0; n < 2; n++) project64(h[n], f[n], n, qf, vf, has_f, F);
#pragma unroll
  for (int a = 0; a < 3; a++) {
#pragma unroll
    for (int n = 0; n < 2; n++) gf[n][a] = {0.0, 0.0};
#pragma unroll
    for (int b = 0; b < 3; b++) {
      const double2 u = __ldg(L + (a * 3 + b) * vl);
#pragma unroll
      for (int n = 0; n < 2; n++) cfma(gf[n][a], cx<double>{u.x, u.y}, h[n][b]);
    }
  }
#pragma unroll
  for (int n = 0; n < 2; n++) project64(h[n], f[n], n, qb, vb, has_b, -F);
  L += 9 * vl;
  constexpr double G = DAG ? -1.0 : 1.0;   // lower spins: B^dag D, D = g_b - g_f (DAG: -D)
#pragma unroll
  for (int a = 0; a < 3; a++) {
    cx<double> gb[2];
#pragma unroll
    for (int n = 0; n < 2; n++) gb[n] = {0.0, 0.0};
#pragma unroll
    for (int b = 0; b < 3; b++) {
      const double2 u = __ldg(L + (a * 3 + b) * vl);
#pragma unroll
      for (int n = 0; n < 2; n++) cfma(gb[n], cx<double>{u.x, u.y}, h[n][b]);
    }
#pragma unroll
    for (int n = 0; n < 2; n++) {
      up[n][a] = cadd(up[n][a], cadd(gf[n][a], gb[n]));
      const cx<double> d = csub(gb[n], gf[n][a]);
      const double2 l = sel_swap(make_double2(d.x, d.y), f[n].swap);
      lo[n][a].x = fma(G * f[n].nx, l.x, lo[n][a].x);
      lo[n][a].y = fma(G * f[n].ny, l.y, lo[n][a].y);
    }
  }
}

// Threads: site (tid mod 2^lst), slice, group (direction, half-spinor component);
// LS * 2^lst * DS is a multiple of 32 and at most stage64_threads(DS).
__host__ __device__ constexpr int stage64_threads(int ds) { return ds == 1 ? 192 : 256; }
constexpr int STAGE64_DS = 16;   // direction groups where a site and slice is split

// Shared memory: the results, [24 reals][LS][st], or the half-spinor products of the direction
// groups, [16][6 reals][LS][st] (then the results); for the dense post its matrices.
__host__ __device__ constexpr int stage64_hop_doubles(int ds) { return ds > 1 ? 96 : 24; }
inline size_t stage64_smem(int Ls, int post, int st, int ds) {
  size_t b = 0;
  if (post || ds > 1) b = (size_t)stage64_hop_doubles(ds) * Ls * st * sizeof(double);
  if (post == 1) b += (size_t)2 * Ls * Ls * sizeof(double);
  return b;
}

// Whole hops: two CTAs' worth of registers (168 a thread) keep three warps per SM quarter
// resident (12^4 x 12: 964 us a CG iteration; with the 186 that the compiler takes freely 1028).
template <int LS, bool DAG, bool BLOCKED, int POST, int DS>
__global__ void __launch_bounds__(stage64_threads(DS), DS == 1 ? 2 : 1)
    stage64_kernel(const StageArgs a, const int lst) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ double red_scratch[32];
  programmatic_start();
  const int st = 1 << lst, tid = threadIdx.x, nt = blockDim.x;
  const long tile = blockIdx.x;
  const int sl = tid & (st - 1), rest = tid >> lst;
  const int s = DS == 1 ? rest : rest % LS, dg = DS == 1 ? 0 : rest / LS;
  const long site = (tile << lst) + sl;
  const int per = 32 >> lst;   // CTAs per 32-site tile, the unit of the segments' sizes
  int seg, ntl, jl, vh;
  long first;
  const void* post = a.post;
  Coef5<double> C;
  if (a.tile_seg) {
    seg = __ldg(a.tile_seg + (tile << lst >> 5));
    if (a.stop && a.stop[seg]) return;
    const BatchSeg& S = a.segp[seg];
    first = (long)S.first_tile * per;
    ntl = S.ntiles * per;
    jl = (int)(site - (long)S.first_tile * 32);
    vh = S.Vh;
    if (POST) post = S.mat[a.post_which];
    C = S.k64;
  } else {
    if (a.stop && *a.stop) return;
    ntl = a.seg_cps * per;
    seg = (int)tile / ntl;
    first = (long)seg * ntl;
    jl = (int)site % a.Vhb_pad;
    vh = a.Vhb;
    C = a.k64;
  }
  const bool valid = jl < vh;

  // this thread's share of the results: all 12 components, or (direction groups) component dg,
  // for the first twelve groups
  constexpr int NC = DS == 1 ? 12 : 1;
  const bool owner = DS == 1 || dg < 12;
  cx<double> v[NC];
  double* buf = reinterpret_cast<double*>(smem_raw);
  const int vol = LS << lst;            // one real component of the CTA
  const int me = (s << lst) + sl;
  if constexpr (DS == 1) {
    cx<double> up[2][3], lo[2][3];   // spins 0, 1 and their lower partners
#pragma unroll
    for (int n = 0; n < 2; n++)
#pragma unroll
      for (int k = 0; k < 3; k++) up[n][k] = lo[n][k] = {0.0, 0.0};
#pragma unroll 1
    for (int mu = 0; mu < 4; mu++) {
      if (mu == 2) {   // x and y feed the lower spins crosswise, z and t straight
#pragma unroll
        for (int k = 0; k < 3; k++) {
          const cx<double> t = lo[0][k];
          lo[0][k] = lo[1][k];
          lo[1][k] = t;
        }
      }
      if (!valid) continue;
      const void* src[2];
      long vs[2], j[2];
      bool has[2];
#pragma unroll
      for (int f = 0; f < 2; f++) {
        const uint32_t nb = __ldg(a.nbr + (long)(2 * mu + f) * a.Vp + site);
        has[f] = nbr_source<BLOCKED>(a, nb, src[f], vs[f]);
        j[f] = (long)(nb & NBR_IDX);
      }
      if (BLOCKED && !has[0] && !has[1]) continue;
      hop64_pair<DAG>(up, lo, mu, reinterpret_cast<const double2*>(src[0]) + s * 12 * vs[0] + j[0],
                      vs[0], has[0],
                      reinterpret_cast<const double2*>(src[1]) + s * 12 * vs[1] + j[1], vs[1],
                      has[1],
                      reinterpret_cast<const double2*>(a.links) + (long)mu * 18 * a.Vp_link + site,
                      a.Vp_link);
    }
#pragma unroll
    for (int k = 0; k < 3; k++) {
      v[k] = up[0][k];
      v[3 + k] = up[1][k];
      v[6 + k] = lo[0][k];
      v[9 + k] = lo[1][k];
    }
  } else {
    // group dg: direction dg & 7, half-spinor component dg >> 3; its product g goes to shared
    // memory, [direction][component][colour][re, im][vol]
    const int d = dg & 7, i = dg >> 3, mu = d >> 1;
    const double back = (d & 1) ? 1.0 : -1.0, sg = DAG ? -back : back;
    cx<double> g[3] = {{0.0, 0.0}, {0.0, 0.0}, {0.0, 0.0}};
    if (valid) {
      const uint32_t nb = __ldg(a.nbr + (long)d * a.Vp + site);
      const void* src;
      long vs;
      if (nbr_source<BLOCKED>(a, nb, src, vs)) {
        cx<double> h[3];
        project64(h, half_spin(mu, i), i,
                  reinterpret_cast<const double2*>(src) + s * 12 * vs + (long)(nb & NBR_IDX), vs,
                  true, sg);
        const double2* L = reinterpret_cast<const double2*>(a.links) + (long)d * 9 * a.Vp_link +
                           site;
#pragma unroll
        for (int c = 0; c < 3; c++)
#pragma unroll
          for (int b = 0; b < 3; b++) {
            const double2 u = __ldg(L + (c * 3 + b) * a.Vp_link);
            cfma(g[c], cx<double>{u.x, u.y}, h[b]);
          }
      }
    }
    double* mine = buf + (d * 2 + i) * 6 * vol + me;
#pragma unroll
    for (int c = 0; c < 3; c++) {
      mine[2 * c * vol] = g[c].x;
      mine[(2 * c + 1) * vol] = g[c].y;
    }
    __syncthreads();
    v[0] = {0.0, 0.0};
    if (owner) {
      const int sp = dg / 3, c = dg - 3 * sp;   // spin and colour of component dg
#pragma unroll
      for (int e = 0; e < 8; e++) {
        const int m = e >> 1;
        if (sp < 2) {
          const double* p = buf + ((e * 2 + sp) * 6 + 2 * c) * vol + me;
          v[0].x += p[0];
          v[0].y += p[vol];
        } else {   // sg B^dag g of the component that feeds this spin
          const int src_i = (m < 2) == (sp == 2) ? 1 : 0;
          const HalfSpin f = half_spin(m, src_i);
          const double se = ((e & 1) != 0) != DAG ? 1.0 : -1.0;
          const double* p = buf + ((e * 2 + src_i) * 6 + 2 * c) * vol + me;
          const double2 l = sel_swap(make_double2(p[0], p[vol]), f.swap);
          v[0].x = fma(se * f.nx, l.x, v[0].x);
          v[0].y = fma(se * f.ny, l.y, v[0].y);
        }
      }
    }
    if constexpr (POST != 0) __syncthreads();   // the buffer is written again below
  }
  const int k0 = DS == 1 ? 0 : dg * NC;   // first component of the share

  if constexpr (POST != 0) {
    if (owner) {
#pragma unroll
      for (int c = 0; c < NC; c++) {
        buf[2 * (k0 + c) * vol + me] = v[c].x;
        buf[(2 * (k0 + c) + 1) * vol + me] = v[c].y;
      }
    }
    if constexpr (POST == 1) {
      double* mat = buf + stage64_hop_doubles(DS) * vol;
      const double* pm = reinterpret_cast<const double*>(post);
      for (int i = tid; i < 2 * LS * LS; i += nt) mat[i] = pm[i];
    }
    __syncthreads();
  }
  if (POST == 3 && owner) {
    // hop_scale D+^dag h at s = b h_s + c (P+ h_{s+1} + P- h_{s-1}), walls -mf
    const double b_ = a.hop_scale * C.db, c_ = a.hop_scale * C.dc;
    const double wall = -C.mf * c_;
    const int su = s + 1 < LS ? s + 1 : 0, sd = s > 0 ? s - 1 : LS - 1;
    const double cu = s + 1 < LS ? c_ : wall, cd = s > 0 ? c_ : wall;
#pragma unroll
    for (int c = 0; c < NC; c++) {
      const bool up = k0 + c < 6;
      const int o = ((up ? su : sd) << lst) + sl;
      const double f = up ? cu : cd;
      v[c].x = fma(f, buf[2 * (k0 + c) * vol + o], b_ * v[c].x);
      v[c].y = fma(f, buf[(2 * (k0 + c) + 1) * vol + o], b_ * v[c].y);
    }
  }
  if constexpr (POST == 4) {
    // hop_scale D+ M5op^-1 (DAG: M5op^-dag D+^dag), column by column: K restricted to one
    // chirality is a cyclic shift with a -mf corner, M5op = alpha (1 + r S); a one-sided
    // sweep and the Sherman-Morrison correction of the corner, the constants folded
    // on the host (Post5)
    const double mr = -C.r;
    for (int col = tid; col < (24 << lst); col += nt) {
      const int c = col >> lst, l = col & (st - 1);
      const bool lower = ((c < 12) != DAG);
      double* q = buf + c * vol + l;
      double w[LS];
      // the lower form in memory order; the upper form is its mirror image in s
#pragma unroll
      for (int t = 0; t < LS; t++) w[t] = q[(lower ? t : LS - 1 - t) << lst];
      auto post = [&](const Post5& p) {
        auto dplus = [&]() {
          const double wrap = w[LS - 1];
#pragma unroll
          for (int t = LS - 1; t > 0; t--) w[t] = fma(p.pc, w[t - 1], p.pb * w[t]);
          w[0] = fma(p.pcw, wrap, p.pb * w[0]);
        };
        if (DAG) dplus();
#pragma unroll
        for (int t = 1; t < LS; t++) w[t] = fma(mr, w[t - 1], w[t]);
        const double e = w[LS - 1];
#pragma unroll
        for (int t = 0; t < LS; t++) w[t] = fma(p.cor[t], e, w[t]);
        if (!DAG) dplus();
      };
      if (a.tile_seg) post(a.segp[seg].post5);
      else post(a.post5);
#pragma unroll
      for (int t = 0; t < LS; t++) q[(lower ? t : LS - 1 - t) << lst] = w[t];
    }
  }
  if constexpr (POST == 1) {
    const double* mat = buf + stage64_hop_doubles(DS) * vol;
    for (int col = tid; col < (24 << lst); col += nt) {
      const int c = col >> lst, l = col & (st - 1);
      const double* m = mat + (c >= 12 ? LS * LS : 0);
      double* q = buf + c * vol + l;
      double w[LS];
#pragma unroll
      for (int t = 0; t < LS; t++) w[t] = q[t << lst];
#pragma unroll
      for (int u = 0; u < LS; u++) {
        double o = 0.0;
#pragma unroll
        for (int t = 0; t < LS; t++) o = fma(m[u * LS + t], w[t], o);
        q[u << lst] = a.hop_scale * o;
      }
    }
  }
  if constexpr (POST == 1 || POST == 4) {
    __syncthreads();
    if (owner) {
#pragma unroll
      for (int c = 0; c < NC; c++)
        v[c] = {buf[2 * (k0 + c) * vol + me], buf[(2 * (k0 + c) + 1) * vol + me]};
    }
  }
  if constexpr (POST == 0) {
    if (owner && a.hop_scale != 1.0) {
#pragma unroll
      for (int c = 0; c < NC; c++) v[c] = cscale(a.hop_scale, v[c]);
    }
  }

  if (owner && a.local_mode != LOC_NONE && valid) {
    // M5op x at s = alpha x_s + beta (P- x_{s+1} + P+ x_{s-1}) (dagger: P+ and P- swapped),
    // walls -mf; each component needs one of the two neighbouring slices only
    const bool dagm = (a.local_mode == LOC_M5DAG);
    const double wall = -C.mf * C.lb;
    const int su = s + 1 < LS ? s + 1 : 0, sd = s > 0 ? s - 1 : LS - 1;
    const double fu = s + 1 < LS ? C.lb : wall, fd = s > 0 ? C.lb : wall;
    const double2* x = reinterpret_cast<const double2*>(a.in2) + site;
#pragma unroll
    for (int c = 0; c < NC; c++) {
      const int k = k0 + c;
      const bool up = dagm == (k < 6);
      const double2 x0 = __ldg(x + (s * 12 + k) * a.Vp);
      const double2 xn = __ldg(x + ((up ? su : sd) * 12 + k) * a.Vp);
      const double f = up ? fu : fd;
      // the largest term last: its sum is rounded once
      v[c].x = fma(C.la, x0.x, fma(f, xn.x, v[c].x));
      v[c].y = fma(C.la, x0.y, fma(f, xn.y, v[c].y));
    }
  }
  double nrm = 0.0;
  if (!owner) {
    // the first twelve groups hold the components
  } else if (a.epi == EPI_CG_R) {
    const double al = a.alpha[seg];
    double2* r = reinterpret_cast<double2*>(a.r) + site;
#pragma unroll
    for (int c = 0; c < NC; c++) {
      double2* q = r + (s * 12 + k0 + c) * a.Vp;
      double2 x = *q;
      x.x = fma(-al, v[c].x, x.x);
      x.y = fma(-al, v[c].y, x.y);
      *q = x;
      nrm = fma(x.x, x.x, fma(x.y, x.y, nrm));
    }
  } else {
    double2* o = reinterpret_cast<double2*>(a.out) + site;
#pragma unroll
    for (int c = 0; c < NC; c++) {
      if (a.epi != EPI_NORM_ONLY) o[(s * 12 + k0 + c) * a.Vp] = make_double2(v[c].x, v[c].y);
      if (a.epi != EPI_STORE) nrm = fma(v[c].x, v[c].x, fma(v[c].y, v[c].y, nrm));
    }
  }
  if (a.epi != EPI_STORE) {
    double n[1] = {nrm};
    grid_reduce_seg<1, double>(a.red, n, red_scratch, tile, seg, first, ntl);
  }
}

// The launch shape (sites per CTA 2^lst, direction groups ds) whose busiest SM quarter has the
// least FP64 work: a quarter takes 64 cycles per warp-wide FP64 instruction, so its work is
// its warps times their FP64 instructions, about 1000 with whole hops and 110 with a direction
// and half-spinor component per thread.  Among equals the smaller CTA, whose warps spread more
// evenly, unless a load would fetch less than 64 contiguous bytes.  Measured per launch of the
// stage with the recurrence post, whole hops: 16^4 x 16, 2 / 4 (chosen) / 8 sites: 898 / 870 /
// 866 us; 12^4 x 12, 8 (chosen) / 16: 224 / 243; 8^3x16 x 8, 4 (chosen) / 8 / 16: 59 / 67 / 67, with
// direction groups 70 to 73.
struct Stage64Shape {
  int lst, ds;
};
inline Stage64Shape stage64_shape(long sites, int Ls, int nsm, bool split) {
  Stage64Shape best{5, 1};
  double cost = -1.0;
  for (int ds = 1; ds <= (split ? STAGE64_DS : 1); ds += STAGE64_DS - 1)
    for (int lst = 5; lst >= 0; lst--) {
      const int threads = (Ls << lst) * ds;
      if (threads % 32 != 0 || threads > stage64_threads(ds)) continue;
      const int warps = threads / 32;
      const long per_sm = ((sites >> lst) + nsm - 1) / nsm;
      double c = (double)((per_sm * warps + 3) / 4) * (ds == 1 ? 1000.0 : 110.0);
      for (int w = warps; w > 1; w >>= 1) c *= 1.02;
      if (lst < 2) c *= 1.05;
      if (cost < 0.0 || c < cost) {
        cost = c;
        best = {lst, ds};
      }
    }
  return best;
}

}  // namespace dwf
