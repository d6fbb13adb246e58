// Linear feasibility projection (Sec. II, eq. linfeas; the initial feasibility step of Alg. 1): the
// current iterate x0 of every instance is replaced by the nearest point, in
// the Euclidean norm, that satisfies the NLP's linear constraints -- the bus
// power balances (eq. opfc5, opfc6 with the flows of eq. acopf_pf, linear in
// w, wR, wI) and the bounds on pg, qg, w and theta (opfc1-4), theta_ref = 0.
//
// It is solved by the same component decomposition as the QP (Alg. 2), in
// FP64:
//   generator g   min (pg - pg0)^2 + (qg - qg0)^2 + ADMM terms, box: closed form;
//   branch l      variables v = (w_i, wR, wI, w_j): its own wR, wI and copies of
//                 the end-bus voltages, flows F v; min (wR - wR0)^2 + (wI - wI0)^2
//                 + ADMM terms on the 4 flows and 2 voltage copies, box on the
//                 copies;
//   bus i         the 2x2 system of its balance rows (right-hand side pd, qd)
//                 with its own voltage term (w - w0)^2 added to the voltage row;
//                 multiplier update and residuals.
// theta does not appear in any balance row, so its projection is the clamp
// into [-2 pi, 2 pi] (0 at the reference bus).
//
// What bounds an iteration on GB300 is the count of FP64 instructions (a warp
// instruction takes about 16 cycles of an SM's FP64 pipe: one instruction per
// branch of 128 2,000-bus scenarios is 0.55 us) and the bytes of the state, so
// both are kept small by algebra that leaves the iterates the same up to
// rounding:
//   - The branch's 4x4 matrix rho F'F + diag(rho, 2, 2, rho) does not change
//     from one iteration to the next, and its (wR, wI) block is a multiple of
//     the identity.  wR and wI have no bounds, so they are eliminated once per
//     call; what is left per iteration is a 2-variable box QP in closed form
//     (linfeas_qp.cuh).
//   - A coupling's multiplier after the bus update is -nu (branch flow) or +nu
//     (generator) of its bus, so flows carry no multiplier of their own; the
//     primal residual of a flow is |nu - nu_old| / rho, a bus quantity.
//   - The bus side hands the components y = lambda - rho z, the only way z and
//     lambda enter their updates: one 32-byte vector per branch end instead of
//     two, and the dual residual follows from x, nu and the previous y.
//   - The residuals are formed only in the iterations whose residuals are read.
//   - Each window of 1,024 buses is processed in order of degree, so that the
//     lanes of a warp loop equally often.
// 128 scenarios of the 2,000-bus grid (345,600 branches): 469 -> 82 us per iteration, 504 -> 92 ms per call.
#include <math.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "common.cuh"
#include "linfeas_qp.cuh"

namespace acopf {

typedef V4<double> D4;  // 32-byte aligned (p, q, w, -) of a branch end

__device__ __forceinline__ D4 d4(double a, double b, double c, double e) {
  D4 v;
  v.x = a; v.y = b; v.z = c; v.w = e;
  return v;
}

constexpr int kLfBus = 7;  // per bus: inverse of the 2x2 matrix (3), 1/Qw, M, 2 w0, Qw
constexpr int kLfWindow = 1024;

struct LfState {
  D4* X;        // [2L] per branch end (p, q, w, wR at end 0 or wI at end 1)
  D4* Y;        // [2L] per branch end lambda - rho z of (p, q, w), and lambda of w
  double2* XG;  // [G] (p, q)
  double2* YG;  // [G] lambda - rho z
  double* cb;   // [kLfBranch][L] constants of the branch QPs
  double* cu;   // [kLfBus][B] constants of the bus systems
  double2* N;   // [B] multipliers of the balance rows
  double* WB;   // [B] bus voltage w
  double* g0;   // [2][G] 2 pg0, 2 qg0
  int* order;   // [B] buses, by degree within windows
  unsigned long long* res;  // [2K]: per-instance max r, s (bits of non-negative doubles)
};

// Start of the iteration (x = z = x0, lambda = 0) and the constants
__global__ void k_lf_init(Dev d, LfState s, double rho) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  const int G = d.G, B = d.B;
  const size_t L = d.L;
  if (n < G) {
    s.g0[n] = 2.0 * d.pg[n];
    s.g0[G + n] = 2.0 * d.qg[n];
    s.YG[n] = make_double2(-rho * d.pg[n], -rho * d.qg[n]);
  }
  if (n < B) {
    const double ne = d.end_ptr[n + 1] - d.end_ptr[n], ng = d.gen_ptr[n + 1] - d.gen_ptr[n];
    const double Qw = 2.0 + rho * ne, M = (ne + ng) / rho, g = d.gs[n], b = d.bs[n];
    const double M11 = M + g * g / Qw, M22 = M + b * b / Qw, M12 = -g * b / Qw, det = M11 * M22 - M12 * M12;
    double* c = s.cu + n;
    c[0 * (size_t)B] = M22 / det;
    c[1 * (size_t)B] = -M12 / det;
    c[2 * (size_t)B] = M11 / det;
    c[3 * (size_t)B] = 1.0 / Qw;
    c[4 * (size_t)B] = M;
    c[5 * (size_t)B] = 2.0 * d.w[n];
    c[6 * (size_t)B] = Qw;
    s.WB[n] = d.w[n];
    s.N[n] = make_double2(0.0, 0.0);
  }
  if (n < d.L) {
    const double* Y = d.Y + n;
    const double gii = Y[0], bii = Y[L], gij = Y[2 * L], bij = Y[3 * L];
    const double gji = Y[4 * L], bji = Y[5 * L], gjj = Y[6 * L], bjj = Y[7 * L];
    const int fi = d.f[n], ti = d.t[n];
    const double wi = d.w[fi], wj = d.w[ti], wr = d.wr[n], wim = d.wi[n];
    s.Y[2 * n] = d4(-rho * (gii * wi + gij * wr + bij * wim), -rho * (-bii * wi - bij * wr + gij * wim), -rho * wi, 0.0);
    s.Y[2 * n + 1] =
        d4(-rho * (gjj * wj + gji * wr - bji * wim), -rho * (-bjj * wj - bji * wr - gji * wim), -rho * wj, 0.0);
    double c[kLfBranch] = {};
    const double Yn[8] = {gii, bii, gij, bij, gji, bji, gjj, bjj};
    lf_constants(Yn, rho, c);
    c[8] = 2.0 * wr;
    c[9] = 2.0 * wim;
    c[10] = d.wmin[fi];
    c[11] = d.wmax[fi];
    c[12] = d.wmin[ti];
    c[13] = d.wmax[ti];
#pragma unroll
    for (int k = 0; k < kLfBranch; ++k) s.cb[k * L + n] = c[k];
  }
}

// order: the buses of each window of kLfWindow by entry count (a counting sort
// in shared memory; equal counts in any order, every bus is independent).  A
// warp of k_lf_buses takes as long as its largest bus: in bus order 3-4 times
// the mean, sorted about the mean.
__global__ void __launch_bounds__(kLfWindow) k_lf_order(Dev d, int* order) {
  __shared__ int cnt[32];
  const int i = blockIdx.x * kLfWindow + threadIdx.x;
  if (threadIdx.x < 32) cnt[threadIdx.x] = 0;
  __syncthreads();
  int key = 0;
  if (i < d.B) {
    key = d.end_ptr[i + 1] - d.end_ptr[i] + d.gen_ptr[i + 1] - d.gen_ptr[i];
    key = key < 31 ? key : 31;
    atomicAdd(&cnt[key], 1);
  }
  __syncthreads();
  if (threadIdx.x == 0)
    for (int k = 0, at = 0; k < 32; ++k) {
      const int n = cnt[k];
      cnt[k] = at;
      at += n;
    }
  __syncthreads();
  if (i < d.B) order[blockIdx.x * kLfWindow + atomicAdd(&cnt[key], 1)] = i;
}

// Out of line: few branches need it.
__device__ __noinline__ void lf_edges_call(double l, double i1, double i2, double si, double sj, double li, double hi,
                                           double lj, double hj, double& wi, double& wj) {
  lf_edges(l, i1, i2, si, sj, li, hi, lj, hj, wi, wj);
}

// generators and branches (one thread each): x from y
__global__ void __launch_bounds__(128) k_lf_components(Dev d, LfState s, double gen_div,
                                                       double gen_inv) {
  const int u = blockIdx.x * blockDim.x + threadIdx.x;
  const int G = d.G;
  const size_t L = d.L;
  if (u < G) {
    const double2 y = s.YG[u];
    s.XG[u] = make_double2(clampv(quot_kept(s.g0[u] - y.x, gen_div, gen_inv), d.pmin[u], d.pmax[u]),
                           clampv(quot_kept(s.g0[G + u] - y.y, gen_div, gen_inv), d.qmin[u], d.qmax[u]));
    return;
  }
  const int l = u - G;
  if (l >= d.L) return;
  const D4 yi = s.Y[2 * l], yj = s.Y[2 * l + 1];
  const double* Y = d.Y + l;
  const double gii = Y[0], bii = Y[L], gij = Y[2 * L], bij = Y[3 * L];
  const double gji = Y[4 * L], bji = Y[5 * L], gjj = Y[6 * L], bjj = Y[7 * L];
  double c[kLfBranch];
#pragma unroll
  for (int k = 0; k < kLfBranch; ++k) c[k] = s.cb[k * L + l];
  const double Yl[8] = {gii, bii, gij, bij, gji, bji, gjj, bjj}, ei[3] = {yi.x, yi.y, yi.z}, ej[3] = {yj.x, yj.y, yj.z};
  double v[4];
  lf_branch(Yl, c, ei, ej, v, lf_edges_call);
  const double wi = v[0], wj = v[1], wr = v[2], wm = v[3];
  s.X[2 * l] = d4(gii * wi + gij * wr + bij * wm, gij * wm - bii * wi - bij * wr, wi, wr);
  s.X[2 * l + 1] = d4(gjj * wj + gji * wr - bji * wm, -bjj * wj - bji * wr - gji * wm, wj, wm);
}

// buses (one thread each): balance rows with right-hand side (pd, qd), the
// voltage row with the bus's own term (w - w0)^2, then y and lambda of every
// coupling; with RES also the residuals
template <bool RES>
__global__ void __launch_bounds__(128) k_lf_buses(Dev d, LfState s, double rho) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  const size_t B = d.B;
  double rm = 0.0, sm = 0.0;
  bool nan = false;
  int k = -1;
  if (n < d.B) {
    const int i = s.order[n];
    k = d.bus_inst[i];
    const int g0 = d.gen_ptr[i], g1 = d.gen_ptr[i + 1], e0 = d.end_ptr[i], e1 = d.end_ptr[i + 1];
    const double* c = s.cu + i;
    const double2 no = s.N[i];
    const double M = c[4 * B];
    // sums of (lambda + rho x) / rho = x -+ nu_old / rho, generators entering with +, flows with -
    double v1 = no.x * M - d.pd[i], v2 = no.y * M - d.qd[i], cw = c[5 * B];
    for (int g = g0; g < g1; ++g) {
      const double2 x = s.XG[g];
      v1 += x.x;
      v2 += x.y;
    }
    for (int e = e0; e < e1; ++e) {
      const int le = d.end_idx[e];
      const D4 x = s.X[le];
      v1 -= x.x;
      v2 -= x.y;
      cw += s.Y[le].w + rho * x.z;
    }
    const double gsh = d.gs[i], bsh = d.bs[i], iq = c[3 * B];
    const double t = cw * iq;
    v1 -= gsh * t;
    v2 += bsh * t;
    const double n1 = c[0] * v1 + c[1 * B] * v2, n2 = c[1 * B] * v1 + c[2 * B] * v2;
    const double w = quot_kept(cw + gsh * n1 - bsh * n2, c[6 * B], iq), rw = rho * w;
    // y = lambda - rho z = -+(2 nu - nu_old) - rho x
    const double a1 = no.x - 2.0 * n1, a2 = no.y - 2.0 * n2;
    if (RES) {
      const double ir = 1.0 / rho;
      if (e1 > e0 || g1 > g0) rm = fmax(fabs(n1 - no.x), fabs(n2 - no.y)) * ir;
      if (e1 > e0) sm = rho * fabs(w - s.WB[i]);
      nan = !(rm + sm == rm + sm);
    }
    for (int g = g0; g < g1; ++g) {
      const double2 x = s.XG[g];
      if (RES) {
        const double2 y = s.YG[g];
        const double sp = fabs(rho * x.x - n1 + y.x), sq = fabs(rho * x.y - n2 + y.y);
        sm = fmax(sm, fmax(sp, sq));
        nan = nan || !(sp + sq == sp + sq);
      }
      s.YG[g] = make_double2(-a1 - rho * x.x, -a2 - rho * x.y);
    }
    for (int e = e0; e < e1; ++e) {
      const int le = d.end_idx[e];
      const D4 x = s.X[le], y = s.Y[le];
      const double a = y.w + rho * x.z;
      if (RES) {
        const double sp = fabs(rho * x.x + n1 + y.x), sq = fabs(rho * x.y + n2 + y.y), rp = fabs(x.z - w);
        sm = fmax(sm, fmax(sp, sq));
        rm = fmax(rm, rp);
        nan = nan || !(sp + sq + rp == sp + sq + rp);
      }
      s.Y[le] = d4(a1 - rho * x.x, a2 - rho * x.y, a - 2.0 * rw, a - rw);
    }
    s.N[i] = make_double2(n1, n2);
    s.WB[i] = w;
  }
  if (RES) {  // one atomic per warp where its buses belong to one instance
    if (nan) rm = sm = kBig;
    const unsigned FULL = 0xffffffffu;
    if (__all_sync(FULL, k == __shfl_sync(FULL, k, 0))) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        rm = fmax(rm, __shfl_xor_sync(FULL, rm, o));
        sm = fmax(sm, __shfl_xor_sync(FULL, sm, o));
      }
      if ((threadIdx.x & 31) != 0) k = -1;
    }
    if (k >= 0) {
      atomicMax(&s.res[k], (unsigned long long)__double_as_longlong(rm));
      atomicMax(&s.res[d.K + k], (unsigned long long)__double_as_longlong(sm));
    }
  }
}

// the projection into the iterate: generators from their (box-feasible)
// update, w from the bus values (clamped), theta clamped, wR and wI from the
// branches
__global__ void k_lf_finish(Dev d, LfState s) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n < d.G) {
    d.pg[n] = s.XG[n].x;
    d.qg[n] = s.XG[n].y;
  }
  if (n < d.B) {
    d.w[n] = clampv(s.WB[n], d.wmin[n], d.wmax[n]);
    d.th[n] = d.isref[n] ? 0.0 : clampv(d.th[n], -kTwoPi, kTwoPi);
  }
  if (n < d.L) {
    d.wr[n] = s.X[2 * n].w;
    d.wi[n] = s.X[2 * n + 1].w;
  }
}

acopf_status project_linear(Ctx& c, double rho, double eps, int max_iter, int check, int* iters, double* rs) {
  Dev& d = c.d;
  LfState s{};
  // one block of scratch for the call, the arrays 256-byte aligned inside it
  size_t bytes = 0;
  auto place = [&](size_t n) {
    const size_t at = bytes;
    bytes += (n + 255) & ~(size_t)255;
    return at;
  };
  const size_t L = d.L, G = d.G, B = d.B;
  const size_t oX = place(sizeof(D4) * 2 * L), oY = place(sizeof(D4) * 2 * L), oXG = place(sizeof(double2) * G),
               oYG = place(sizeof(double2) * G), ocb = place(sizeof(double) * kLfBranch * L),
               ocu = place(sizeof(double) * kLfBus * B), oN = place(sizeof(double2) * B),
               oWB = place(sizeof(double) * B), og0 = place(sizeof(double) * 2 * G), oord = place(sizeof(int) * B),
               ores = place(sizeof(unsigned long long) * 2 * d.K);
  void* block = nullptr;
  cudaError_t e = ctx_alloc(c, &block, bytes);
  if (e != cudaSuccess) {
    c.last_error = std::string("acopf_project_linear: ") + cudaGetErrorString(e);
    return e == cudaErrorMemoryAllocation ? ACOPF_ENOMEM : ACOPF_ECUDA;
  }
  unsigned char* base = (unsigned char*)block;
  s.X = (D4*)(base + oX); s.Y = (D4*)(base + oY);
  s.XG = (double2*)(base + oXG); s.YG = (double2*)(base + oYG);
  s.cb = (double*)(base + ocb); s.cu = (double*)(base + ocu);
  s.N = (double2*)(base + oN); s.WB = (double*)(base + oWB); s.g0 = (double*)(base + og0);
  s.order = (int*)(base + oord); s.res = (unsigned long long*)(base + ores);
  const long m = d.G + d.L > d.B ? d.G + d.L : d.B;
  k_lf_init<<<nblk(m, 256), 256, 0, c.stream>>>(d, s, rho);
  k_lf_order<<<nblk(d.B, kLfWindow), kLfWindow, 0, c.stream>>>(d, s.order);
  c.launches += 2;
  std::vector<double> h(2 * (size_t)d.K, 0.0);
  int it = 0;
  bool done = false;
  while (it < max_iter && !done) {
    const int n = max_iter - it < check ? max_iter - it : check;
    cudaMemsetAsync(s.res, 0, sizeof(unsigned long long) * 2 * d.K, c.stream);
    for (int k = 0; k < n; ++k) {
      k_lf_components<<<nblk(d.G + d.L, 128), 128, 0, c.stream>>>(d, s, 2.0 + rho, 1.0 / (2.0 + rho));
      if (k == n - 1) k_lf_buses<true><<<nblk(d.B, 128), 128, 0, c.stream>>>(d, s, rho);
      else k_lf_buses<false><<<nblk(d.B, 128), 128, 0, c.stream>>>(d, s, rho);
      c.launches += 2;
    }
    it += n;
    e = cudaMemcpyAsync(h.data(), s.res, sizeof(double) * 2 * d.K, cudaMemcpyDeviceToHost, c.stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c.stream);
    if (e != cudaSuccess) break;
    done = true;
    for (int k = 0; k < 2 * d.K; ++k) done = done && h[k] <= eps;
  }
  if (e == cudaSuccess) {
    k_lf_finish<<<nblk(m, 256), 256, 0, c.stream>>>(d, s);
    c.launches++;
    e = cudaStreamSynchronize(c.stream);
  }
  ctx_free(c, block);
  if (e != cudaSuccess) {
    c.last_error = std::string("acopf_project_linear: ") + cudaGetErrorString(e);
    return ACOPF_ECUDA;
  }
  if (iters) *iters = it;
  if (rs) {
    double r = 0.0, sv = 0.0;
    for (int k = 0; k < d.K; ++k) {
      r = fmax(r, h[k]);
      sv = fmax(sv, h[d.K + k]);
    }
    rs[0] = r;
    rs[1] = sv;
  }
  return ACOPF_OK;
}

}  // namespace acopf
