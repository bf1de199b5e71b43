// Pseudofermion action S = phi^dag (Mpc^dag Mpc)^-1 phi and its gradient with respect to the
// links (PyTorch complex convention dS/dRe U + i dS/dIm U).
//
// With X = A^-1 phi, Y = Mpc X, V = D+ X (even), W = D+ M5op^-1 Dh_oe V (odd) and
// Z = M5op^-dag D+^dag Dh^dag_oe Y (odd):  dS = 1/2 Re(<Y, dDh W> + <Z, dDh V>).
// U_mu(x) enters Dh as (1 - gamma_mu) U_mu(x) b(x+mu) at output x and as
// (1 + gamma_mu) U_mu(x)^dag b(x) at output x+mu, so for full-lattice fields a, b the gradient
// of Re <a, Dh b> at link (x, mu) is
//   sum_s sum_spin [(1 - gamma_mu) a(x,s)] b(x+mu,s)^dag + b(x,s) [(1 + gamma_mu) a(x+mu,s)]^dag.
// For an even site x only Y(x), V(x) and W(x+mu), Z(x+mu) are non-zero; for an odd site only
// Z(x), W(x) and V(x+mu), Y(x+mu).
#include <cmath>

#include "engine.h"

namespace dwf {

// acc[a][b] += sum_spin ((1 + sgn gamma_mu) u)_{spin,a} conj(v_{spin,b}).  With (1 + sgn gamma) =
// R R^dag, R = [1; sgn B^dag], the sum over four spins is one over the two components of the
// projected half-spinors R^dag u and R^dag v: 24 additions and 72 FMAs instead of 168
// instructions, and either factor may be the one the projector stands at.
template <int MU>
__device__ __forceinline__ void projected_outer(cx<double> (&acc)[9], const Spinor<double>& u,
                                                const Spinor<double>& v, double sgn) {
  cx<double> hu[2][3], hv[2][3];
  project_half<double, MU>(hu, u, sgn);
  project_half<double, MU>(hv, v, sgn);
#pragma unroll
  for (int i = 0; i < 2; i++)
#pragma unroll
    for (int a = 0; a < 3; a++)
#pragma unroll
      for (int b = 0; b < 3; b++) {
        cx<double>& c = acc[a * 3 + b];
        const cx<double> x = hu[i][a], y = hv[i][b];
        c.x = fma(x.x, y.x, fma(x.y, y.y, c.x));
        c.y = fma(x.y, y.x, fma(-x.x, y.y, c.y));
      }
}

struct ForceArgs {
  const void *Ye, *Ve, *Wo, *Zo;  // FP64 internal fields
  const uint32_t* nbr[2];
  const int* lex[2];
  double2* out;                    // caller layout [V][4][9]
  long Vp;
  int Ls;
};

// This thread's slices (s0, s0 + ds, ...) of the gradient of one link.
template <int MU>
__device__ __forceinline__ void force_link(const ForceArgs& a, int p, long idx, int s0, int ds,
                                           cx<double> (&acc)[9]) {
  // x even: (1-g) Y(x) W(x+mu)^dag + V(x) [(1+g) Z(x+mu)]^dag
  // x odd : (1-g) Z(x) V(x+mu)^dag + W(x) [(1+g) Y(x+mu)]^dag
  const void* A = p == 0 ? a.Ye : a.Zo;
  const void* B = p == 0 ? a.Wo : a.Ve;
  const void* C = p == 0 ? a.Ve : a.Wo;
  const void* D = p == 0 ? a.Zo : a.Ye;
  const long nidx = (long)(a.nbr[p][(long)(2 * MU) * a.Vp + idx] & NBR_IDX);
#pragma unroll 1
  for (int s = s0; s < a.Ls; s += ds) {
    Spinor<double> x, y;
    load_spinor<P64>(x, A, a.Vp, idx, s);
    load_spinor<P64>(y, B, a.Vp, nidx, s);
    projected_outer<MU>(acc, x, y, -1.0);
    load_spinor<P64>(x, C, a.Vp, idx, s);
    load_spinor<P64>(y, D, a.Vp, nidx, s);
    projected_outer<MU>(acc, x, y, 1.0);
  }
}

// Thread (lane, group): one link of 32 sites, every blockDim.y-th slice; the groups' sums are
// added in order through shared memory.  FP64 instructions bound it (64 cycles per warp and
// SM quarter): 192 per link and slice.  16^4 x 16: 3.60 ms before with four spins (336), now
// 1.4 ms; the slices are split only where the links alone leave SM quarters without a warp
// (force_groups).
__global__ void force_kernel(const ForceArgs a) {
  extern __shared__ double force_smem[];   // [groups - 1][18][32]
  const long idx = (long)blockIdx.x * 32 + threadIdx.x;
  const int mu = blockIdx.y, p = blockIdx.z, g = threadIdx.y, ng = blockDim.y;
  const int lx = idx < a.Vp ? a.lex[p][idx] : -1;
  cx<double> acc[9];
#pragma unroll
  for (int k = 0; k < 9; k++) acc[k] = {0.0, 0.0};
  if (lx >= 0) switch (mu) {
    case 0: force_link<0>(a, p, idx, g, ng, acc); break;
    case 1: force_link<1>(a, p, idx, g, ng, acc); break;
    case 2: force_link<2>(a, p, idx, g, ng, acc); break;
    default: force_link<3>(a, p, idx, g, ng, acc);
  }
  if (g > 0) {
#pragma unroll
    for (int k = 0; k < 9; k++) {
      force_smem[((g - 1) * 18 + 2 * k) * 32 + threadIdx.x] = acc[k].x;
      force_smem[((g - 1) * 18 + 2 * k + 1) * 32 + threadIdx.x] = acc[k].y;
    }
  }
  __syncthreads();
  if (g > 0 || lx < 0) return;
  for (int j = 0; j < ng - 1; j++)
#pragma unroll
    for (int k = 0; k < 9; k++) {
      acc[k].x += force_smem[(j * 18 + 2 * k) * 32 + threadIdx.x];
      acc[k].y += force_smem[(j * 18 + 2 * k + 1) * 32 + threadIdx.x];
    }
  double2* o = a.out + ((long)lx * 4 + mu) * 9;
#pragma unroll
  for (int k = 0; k < 9; k++) o[k] = make_double2(0.5 * acc[k].x, 0.5 * acc[k].y);
}

// Slice groups per CTA: enough that every SM quarter has several warps (a warp works through
// its slices alone), at most 8 and at least two slices each.
static int force_groups(long Vp, int Ls) {
  const long warps = Vp / 32 * 8, want = (long)sm_count() * 4 * 6;
  int g = 1;
  while (g < 8 && warps * g < want && Ls / (2 * g) >= 2) g *= 2;
  return g;
}

}  // namespace dwf

using namespace dwf;

// Solve to tol into a workspace buffer when the caller gives no X.
static dwf_status solution(dwf_t h, Layout* lay, const void* dphi, const void* X, double tol,
                           const void** dX) {
  const size_t ub = (size_t)h->Ls * (lay->g.V / 2) * 12 * 16;
  if (X) {
    void* p;
    DWF_TRY(stage_buffer(h, "force_X", X, ub, true, &p));
    *dX = p;
    return DWF_OK;
  }
  void* p;
  DWF_TRY(h->ws->get("force_X", ub, &p));
  DWF_CUDA(cudaMemsetAsync(p, 0, ub, h->stream));
  dwf_stats st{};
  dwf_status s = dwf_cg(h, dphi, p, tol, 1000000, DWF_F64, &st);
  if (s != DWF_OK) return s;
  *dX = p;
  return DWF_OK;
}

extern "C" dwf_status dwf_force(dwf_t h, const void* phi, const void* X, void* dSdU,
                                double tol) {
  if (!h || !phi || !dSdU) return set_error(DWF_ERR_ARG, "null argument");
  Layout* lay;
  DWF_TRY(get_layout(h, h->dims, &lay));
  const Geom& g = lay->g;
  const size_t ub = (size_t)h->Ls * (g.V / 2) * 12 * 16;
  void* dphi;
  DWF_TRY(stage_buffer(h, "force_phi", phi, ub, true, &dphi));
  const void* dX;
  DWF_TRY(solution(h, lay, dphi, X, tol, &dX));
  OpEngine E;
  DWF_TRY(E.init(h, lay, P64, false));
  const size_t fb = field_bytes(g, P64);
  void *x, *u, *w, *y, *z;
  DWF_TRY(h->ws->get("force_x", fb, &x));
  DWF_TRY(h->ws->get("force_u", fb, &u));
  DWF_TRY(h->ws->get("force_w", fb, &w));
  DWF_TRY(h->ws->get("force_y", fb, &y));
  DWF_TRY(h->ws->get("force_z", fb, &z));
  DWF_TRY(pack_even(h, lay, dX, x, P64));
  // Y = Mpc X; the first stage leaves W = D+ M5op^-1 Dh_oe D+ X in w and D+ X in u
  DWF_TRY(E.mpc(x, u, w, y, EPI_STORE, RedArgs{}, nullptr));
  const void* V = x;
  if (!E.trivial()) {
    V = u;
  } else if (h->b != 1.0) {
    // D+ = b: V = b X
    VopArgs a{};
    a.op = VOP_ZERO;
    a.y = u;
    a.Vp = g.Vp;
    a.Vhb = g.Vhb;
    a.Vhb_pad = g.Vhb_pad;
    DWF_CUDA(launch_vop(P64, P64, a, h->Ls, h->stream));
    a.op = VOP_AXPY;
    a.x = x;
    a.sa = h->b;
    DWF_CUDA(launch_vop(P64, P64, a, h->Ls, h->stream));
    V = u;
  }
  // Z = M5op^-dag D+^dag Dh^dag_oe Y: first stage of Mpc^dag
  {
    StageArgs a = E.base(1);
    a.in = y;
    a.out = z;
    a.post = h->mats.d_m5idpt[0];
    E.set_struct(a);   // by recurrence where it is stable (the dense matrices: 1.20 ms against
                       // 0.88 ms on 16^4 x 16)
    a.epi = EPI_STORE;
    DWF_TRY(E.launch(a, true));
  }
  void* dout;
  const size_t lb = (size_t)g.V * 4 * 9 * 16;
  DWF_TRY(stage_buffer(h, "force_out", dSdU, lb, false, &dout));
  ForceArgs fa{};
  fa.Ye = y;
  fa.Ve = V;
  fa.Wo = w;
  fa.Zo = z;
  fa.nbr[0] = lay->nbr[0];
  fa.nbr[1] = lay->nbr[1];
  fa.lex[0] = lay->lex[0];
  fa.lex[1] = lay->lex[1];
  fa.out = reinterpret_cast<double2*>(dout);
  fa.Vp = g.Vp;
  fa.Ls = h->Ls;
  const int ng = force_groups(g.Vp, h->Ls);
  dim3 grid((unsigned)(g.Vp / 32), 4, 2), block(32, ng);
  force_kernel<<<grid, block, (size_t)(ng - 1) * 18 * 32 * sizeof(double), h->stream>>>(fa);
  DWF_CUDA(cudaGetLastError());
  return finish_output(h, dSdU, dout, lb);
}

extern "C" dwf_status dwf_action(dwf_t h, const void* phi, const void* X, double tol, double* S) {
  if (!h || !phi || !S) return set_error(DWF_ERR_ARG, "null argument");
  Layout* lay;
  DWF_TRY(get_layout(h, h->dims, &lay));
  const Geom& g = lay->g;
  const size_t ub = (size_t)h->Ls * (g.V / 2) * 12 * 16;
  void* dphi;
  DWF_TRY(stage_buffer(h, "force_phi", phi, ub, true, &dphi));
  const void* dX;
  DWF_TRY(solution(h, lay, dphi, X, tol, &dX));
  OpEngine E;
  DWF_TRY(E.init(h, lay, P64, false));
  const size_t fb = field_bytes(g, P64);
  void *x, *f, *u, *t, *y;
  double* d;
  DWF_TRY(h->ws->get("force_x", fb, &x));
  DWF_TRY(h->ws->get("force_f", fb, &f));
  DWF_TRY(h->ws->get("force_u", fb, &u));
  DWF_TRY(h->ws->get("force_w", fb, &t));
  DWF_TRY(h->ws->get("force_y", fb, &y));
  DWF_TRY(h->ws->get("force_d", 4 * sizeof(double), (void**)&d));
  DWF_TRY(pack_even(h, lay, dX, x, P64));
  DWF_TRY(pack_even(h, lay, dphi, f, P64));
  // S = Re(2 <phi, X> - ||Mpc X||^2): equals phi^dag A^-1 phi at the exact solution, with an
  // error quadratic in the solve residual.
  DWF_TRY(E.mpc(x, u, t, y, EPI_NORM, E.red(FIN_STORE, d), nullptr));
  VopArgs a{};
  a.op = VOP_DOT;
  a.x = f;
  a.y = x;
  a.Vp = g.Vp;
  a.Vhb = g.Vhb;
  a.Vhb_pad = g.Vhb_pad;
  a.red = E.red(FIN_STORE, d + 1);
  DWF_CUDA(launch_vop(P64, P64, a, h->Ls, h->stream));
  double hv[2];
  DWF_CUDA(cudaMemcpyAsync(hv, d, 2 * sizeof(double), cudaMemcpyDeviceToHost, h->stream));
  DWF_CUDA(cudaStreamSynchronize(h->stream));
  *S = 2.0 * hv[1] - hv[0];
  return DWF_OK;
}
