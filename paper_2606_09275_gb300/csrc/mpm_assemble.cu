// Per-Newton-iteration assembly of Eq. (MPMweak) (static part): point
// kinematics, the Hencky / return-map constitutive update with its consistent
// spatial tangent (Sec. 2.2), the internal force, the tangent gathered row by
// row into the 3x3 block matrix, the ghost term (Sec. 4), the penalty contact
// (Sec. 2.3) and the strong Dirichlet rows (Sec. 2.4).
#include <algorithm>

#include "mpm_internal.cuh"
#include "mpm_law.cuh"
#include "mpm_sliced.cuh"

namespace mpm {
namespace {

// ------------------------------------------------------------------ kinematics

// dF = I + sum_v du_v (x) grad S_vp, four lanes per point.  Bound by the FP64
// rate: an FP64 instruction takes 16 SM cycles whatever the number of active
// lanes, so a warp costs the longest support of its points (8, 12, 18 or 27
// nodes in the interior, mixed within a cell).  Each block therefore deals its
// points to the warps in order of support size (counted in shared memory, in
// integers).  Per point 6 FP64 instructions instead of 10.5 with eight lanes
// in point order; indentation, 1.9 M points: 1.35 -> 0.65 ms.
constexpr int KIN_T = 256, KIN_P = KIN_T / 4;  // threads and points of a block
__global__ void __launch_bounds__(KIN_T)
    k_kinematics(int P, const int* __restrict__ nsup, const int* __restrict__ sidx, const double* __restrict__ dS,
                 const double* __restrict__ du, double* dF) {
  __shared__ int size[KIN_P], order[KIN_P];
  const int w0 = blockIdx.x * KIN_P, np = min(KIN_P, P - w0), t = threadIdx.x;
  if (t < np) size[t] = nsup[w0 + t];
  __syncthreads();
  {
    // rank of point t / 4 among the block's, its four threads comparing a quarter each
    int p = t >> 2, rank = 0;
    if (p < np) {
      int n = size[p];
      for (int j = t & 3; j < np; j += 4) rank += size[j] < n || (size[j] == n && j < p);
    }
    rank += __shfl_xor_sync(0xffffffffu, rank, 1);
    rank += __shfl_xor_sync(0xffffffffu, rank, 2);
    if (p < np && (t & 3) == 0) order[rank] = p;
  }
  __syncthreads();
  const int sub = t & 3;
  bool in = (t >> 2) < np;
  int p = in ? order[t >> 2] : 0, n = in ? size[p] : 0;
  size_t w = (size_t)w0 + p;
  double a[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) a[i] = 0.0;
  for (int k = sub; k < n; k += 4) {
    size_t o = w * MAXS + k;
    int j = sidx[o];
    double u0 = du[3 * (size_t)j], u1 = du[3 * (size_t)j + 1], u2 = du[3 * (size_t)j + 2];
    double g0 = dS[3 * o], g1 = dS[3 * o + 1], g2 = dS[3 * o + 2];
    a[0] += u0 * g0; a[1] += u0 * g1; a[2] += u0 * g2;
    a[3] += u1 * g0; a[4] += u1 * g1; a[5] += u1 * g2;
    a[6] += u2 * g0; a[7] += u2 * g1; a[8] += u2 * g2;
  }
  // reduce-scatter of a[0..7] over the 4 lanes (lane sub ends with the sums of
  // a[2 sub'], a[2 sub' + 1] in bit-reversed order), a[8] by a butterfly
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    bool up = sub & 2;
    double send = up ? a[i] : a[i + 4];
    double keep = up ? a[i + 4] : a[i];
    a[i] = keep + __shfl_xor_sync(0xffffffffu, send, 2);
  }
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    bool up = sub & 1;
    double send = up ? a[i] : a[i + 2];
    double keep = up ? a[i + 2] : a[i];
    a[i] = keep + __shfl_xor_sync(0xffffffffu, send, 1);
  }
  a[8] += __shfl_xor_sync(0xffffffffu, a[8], 2);
  a[8] += __shfl_xor_sync(0xffffffffu, a[8], 1);
  if (in) {
    int e = 2 * sub;  // entries e and e + 1; 0 and 4 lie on the diagonal
    dF[9 * w + e] = a[0] + ((e & 3) == 0 ? 1.0 : 0.0);
    dF[9 * w + e + 1] = a[1];
    if (sub == 0) dF[9 * w + 8] = a[8] + 1.0;
  }
}

// ------------------------------------------------------------------ constitutive

// Full per-point update.  in: dF, b_e,n (6); out: tau (6: xx yy zz xy yz xz),
// b_e (6), V0 A' (tangent_rotate)
// The consistent spatial tangent from the spectral state: theta_ab =
// (tau_a - tau_b)/(lam_a - lam_b) = g/2 * divided difference of ln (in FP64),
// then the eigenbasis rotation of the 81 entries in the precision the tangent
// is stored in (FP32 for the mixed path, where it runs on the FP32 pipe).
// Layout [(i*9 + k*3 + m)*4 + j] = V0 (A_ijkm - tau_im delta_jk), the fourth
// entry of each term unused: a lane of the row gather loads one term's three
// factors in one 16-byte word (FP32).
template <class TA>
__device__ void tangent_rotate(const double* Q, const double* lam, const double* dd, double gr,
                               const double* tau6, double V0, TA* Aout) {
  // theta_ab = (tau_a - tau_b)/(lam_a - lam_b) = g/2 * divided difference of ln
  // (in FP64), then the eigenbasis rotation of the 81 entries in the
  // precision the tangent is stored in: FP32 for the mixed path, where it
  // runs on the FP32 pipe
  typedef TA R;
  double th01 = 0.5 * gr * ln_divdiff(lam[0], lam[1]);
  double th02 = 0.5 * gr * ln_divdiff(lam[0], lam[2]);
  double th12 = 0.5 * gr * ln_divdiff(lam[1], lam[2]);
  R th[9] = {(R)0, (R)th01, (R)th02, (R)th01, (R)0, (R)th12, (R)th02, (R)th12, (R)0};
  R q[9], d[9], lr[3];
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    q[i] = (R)Q[i];
    d[i] = (R)dd[i];
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) lr[a] = (R)lam[a];
  const R v0 = (R)V0;
  R taum[9];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      int s = (i == j) ? i : (i + j == 1 ? 3 : (i + j == 3 ? 4 : 5));
      taum[3 * i + j] = v0 * (R)tau6[s];
    }
  // A_ijkm for a pair (k, m) is Q B Q^T, B symmetric in the eigenbasis: B_aa =
  // sum_c d_ac q_kc q_mc, B_ac = theta_ac (lam_c q_ka q_mc + lam_a q_kc q_ma).
  // Some 80 multiply-adds a pair, where the sums written out entry by entry took
  // 750 (FP64: the law and this for the punch of depths 3 to 6 50 us, 96 so;
  // this alone for the rolling sphere 28 and 71 us)
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      R B[3][3];
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        R s = d[3 * a] * (q[3 * k] * q[3 * m]);
        s += d[3 * a + 1] * (q[3 * k + 1] * q[3 * m + 1]);
        s += d[3 * a + 2] * (q[3 * k + 2] * q[3 * m + 2]);
        B[a][a] = v0 * s;
      }
#pragma unroll
      for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int c = a + 1; c < 3; ++c)
          B[a][c] = B[c][a] = v0 * (th[3 * a + c] * (lr[c] * (q[3 * k + a] * q[3 * m + c]) +
                                                     lr[a] * (q[3 * k + c] * q[3 * m + a])));
      R o[3][4];
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        R t[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) t[c] = q[3 * i] * B[0][c] + q[3 * i + 1] * B[1][c] + q[3 * i + 2] * B[2][c];
#pragma unroll
        for (int j = i; j < 3; ++j)
          o[i][j] = o[j][i] = t[0] * q[3 * j] + t[1] * q[3 * j + 1] + t[2] * q[3 * j + 2];
        o[i][3] = (R)0;
      }
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        o[i][k] -= taum[3 * i + m];
        st4(Aout + (i * 9 + k * 3 + m) * 4, o[i]);
      }
    }
}

template <bool TANGENT, class TA, bool SAVE = false>
__device__ bool point_update_law(const Law& L, double E, double ys, const double* be, const double* dF,
                                 double* tau6, double* be_new, double V0, TA* Aout, double* save = nullptr) {
  double b[9] = {be[0], be[3], be[5], be[3], be[1], be[4], be[5], be[4], be[2]};
  double t[9], bt[9];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j)
      t[3 * i + j] = dF[3 * i] * b[j] + dF[3 * i + 1] * b[3 + j] + dF[3 * i + 2] * b[6 + j];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j)
      bt[3 * i + j] = t[3 * i] * dF[3 * j] + t[3 * i + 1] * dF[3 * j + 1] + t[3 * i + 2] * dF[3 * j + 2];
  // symmetrise before the rotations
  bt[1] = bt[3] = 0.5 * (bt[1] + bt[3]);
  bt[2] = bt[6] = 0.5 * (bt[2] + bt[6]);
  bt[5] = bt[7] = 0.5 * (bt[5] + bt[7]);
  double lam[3], Q[9];
  jacobi3(bt, lam, Q);
  if (!(lam[0] > 0.0 && lam[1] > 0.0 && lam[2] > 0.0) || !isfinite(lam[0] + lam[1] + lam[2]))
    return false;
  double eps[3] = {0.5 * log_stretch(lam[0]), 0.5 * log_stretch(lam[1]), 0.5 * log_stretch(lam[2])};
  double ta[3], dd[9], gr;
  principal_return(L, E, ys, eps, ta, dd, &gr);
  double mu = E * L.cmu, lm = E * L.clm;
  double tt = ta[0] + ta[1] + ta[2], tm = lm * tt / (3.0 * lm + 2.0 * mu), imu = 1.0 / mu;
  double bw[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) bw[a] = exp((ta[a] - tm) * imu);
  // tau = Q diag(ta) Q^T, b_e = Q diag(bw) Q^T
  const int ii[6] = {0, 1, 2, 0, 1, 0}, jj[6] = {0, 1, 2, 1, 2, 2};
#pragma unroll
  for (int s = 0; s < 6; ++s) {
    int i = ii[s], j = jj[s];
    tau6[s] = Q[3 * i] * ta[0] * Q[3 * j] + Q[3 * i + 1] * ta[1] * Q[3 * j + 1] + Q[3 * i + 2] * ta[2] * Q[3 * j + 2];
    be_new[s] = Q[3 * i] * bw[0] * Q[3 * j] + Q[3 * i + 1] * bw[1] * Q[3 * j + 1] + Q[3 * i + 2] * bw[2] * Q[3 * j + 2];
  }
  if (TANGENT) tangent_rotate<TA>(Q, lam, dd, gr, tau6, V0, Aout);
  if constexpr (SAVE) {
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      save[i] = Q[i];
      save[12 + i] = dd[i];
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) save[9 + a] = lam[a];
    save[21] = gr;
  }
  return true;
}

__device__ inline double det3(const double* a) {
  return a[0] * (a[4] * a[8] - a[5] * a[7]) - a[1] * (a[3] * a[8] - a[5] * a[6]) +
         a[2] * (a[3] * a[7] - a[4] * a[6]);
}

// also M = V0 tau dF^-T (row-major, 12 per point, the last 3 unused), so that
// the internal force of support k is M grad S_k (k_residual_rows).  SAVE: the
// spectral state for a tangent at the same increment (k_tangent_state), of use
// to a Newton iteration only.  Bound by FP64 issue, some
// 550 instructions a point: 1.9 M points take 1.88 ms (1.71 elastic ones), with
// the FP32 tangent 2.23 (2.51 with its entries summed term by term).
template <bool TANGENT, class TA, bool SAVE>
__global__ void k_constitutive(int P, Law L, const double* __restrict__ E, const double* __restrict__ ys,
                               const double* __restrict__ be, const double* __restrict__ dF,
                               const double* __restrict__ V0, double* tau, double* dFinv,
                               double* Mf, TA* Aalg, double* lawst, int* err) {
  int w = blockIdx.x * blockDim.x + threadIdx.x;
  if (w >= P) return;
  double f[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) f[i] = dF[9 * (size_t)w + i];
  double det = det3(f);
  double t6[6], bn[6];
  bool ok = det > 0.0 && isfinite(det) &&
            point_update_law<TANGENT, TA, SAVE>(L, E[w], ys[w], be + 6 * (size_t)w, f, t6, bn, V0[w],
                                                Aalg + 108 * (size_t)w, lawst + 22 * (size_t)w);
  if (!ok) {
    atomicOr(err, EB_NAN);
#pragma unroll
    for (int s = 0; s < 6; ++s) t6[s] = 0.0;
    det = 1.0;
  }
#pragma unroll
  for (int s = 0; s < 6; ++s) tau[6 * (size_t)w + s] = t6[s];
  double id = 1.0 / det;
  double* o = dFinv + 9 * (size_t)w;
  o[0] = (f[4] * f[8] - f[5] * f[7]) * id;
  o[1] = (f[2] * f[7] - f[1] * f[8]) * id;
  o[2] = (f[1] * f[5] - f[2] * f[4]) * id;
  o[3] = (f[5] * f[6] - f[3] * f[8]) * id;
  o[4] = (f[0] * f[8] - f[2] * f[6]) * id;
  o[5] = (f[2] * f[3] - f[0] * f[5]) * id;
  o[6] = (f[3] * f[7] - f[4] * f[6]) * id;
  o[7] = (f[1] * f[6] - f[0] * f[7]) * id;
  o[8] = (f[0] * f[4] - f[1] * f[3]) * id;
  // M_il = V0 sum_j tau_ij (dF^-1)_lj
  double fi[9];
#pragma unroll
  for (int e = 0; e < 9; ++e) fi[e] = o[e];
  double v0 = V0[w], u6[6];
#pragma unroll
  for (int s = 0; s < 6; ++s) u6[s] = v0 * t6[s];
  double tm[9] = {u6[0], u6[3], u6[5], u6[3], u6[1], u6[4], u6[5], u6[4], u6[2]};
  double* M = Mf + 12 * (size_t)w;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int l = 0; l < 3; ++l)
      M[3 * i + l] = tm[3 * i] * fi[3 * l] + tm[3 * i + 1] * fi[3 * l + 1] + tm[3 * i + 2] * fi[3 * l + 2];
}

// the tangent of the state the last residual evaluation left (same increment):
// no second eigen-decomposition or return map
template <class TA>
__global__ void k_tangent_state(int P, const double* __restrict__ lawst, const double* __restrict__ tau,
                                const double* __restrict__ V0, TA* Aalg) {
  int w = blockIdx.x * blockDim.x + threadIdx.x;
  if (w >= P) return;
  const double* st = lawst + 22 * (size_t)w;
  double Q[9], lam[3], dd[9], t6[6];
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    Q[i] = st[i];
    dd[i] = st[12 + i];
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) lam[a] = st[9 + a];
#pragma unroll
  for (int i = 0; i < 6; ++i) t6[i] = tau[6 * (size_t)w + i];
  tangent_rotate<TA>(Q, lam, dd, st[21], t6, V0[w], Aalg + 108 * (size_t)w);
}

// grad_x S = grad S . dF^{-1} for the tangent gather (in its precision), one
// 4-vector per support node at gx[4 (w pw + k)]: the gather loads a node's in
// one 16-byte word (FP32).  Eight lanes per point.  A conversion from FP64
// occupies the FP64 pipe as long as an FMA, for a whole warp instruction:
// dF^-1 is converted one entry per lane and shared by shuffles, and the FP32
// path reads grad S from its FP32 copy (TS = float), made once per mesh build.
template <class TG, class TS>
__global__ void k_gx(int P, int pw, const int* __restrict__ nsup, const TS* __restrict__ dS,
                     const double* __restrict__ dFinv, TG* gx) {
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  int w = (int)(t >> 3), sub = (int)(t & 7);
  bool in = w < P;
  TG mine = in ? (TG)dFinv[9 * (size_t)w + sub] : (TG)0, last = in ? (TG)dFinv[9 * (size_t)w + 8] : (TG)0;
  TG fi[9];
#pragma unroll
  for (int i = 0; i < 8; ++i) fi[i] = __shfl_sync(0xffffffffu, mine, i, 8);
  fi[8] = last;
  int n = in ? nsup[w] : 0;
  for (int k = sub; k < n; k += 8) {
    size_t o = (size_t)w * MAXS + k;
    TG a0 = (TG)dS[3 * o], a1 = (TG)dS[3 * o + 1], a2 = (TG)dS[3 * o + 2];
    TG g[4] = {a0 * fi[0] + a1 * fi[3] + a2 * fi[6], a0 * fi[1] + a1 * fi[4] + a2 * fi[7],
               a0 * fi[2] + a1 * fi[5] + a2 * fi[8], (TG)0};
    st4(gx + 4 * ((size_t)w * pw + k), g);
  }
}

// the FP32 copy of the basis gradients (the used slots of every point)
__global__ void k_dS_to_float(int P, const int* __restrict__ nsup, const double* __restrict__ dS,
                              float* dS32) {
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  int w = (int)(t / (3 * MAXS)), e = (int)(t - (long long)w * 3 * MAXS);
  if (w >= P || e >= 3 * nsup[w]) return;
  dS32[t] = (float)dS[t];
}

// ------------------------------------------------------------------ internal force and residual

// R = f_int - load f_ext + K_G du, one warp per row r, where f_int,r is the sum
// over the point sources (p, k) of the row (the pattern's sorted source keys)
// of M_p grad S_pk, M_p = V0 tau dF^-T from k_constitutive.  A fixed-order
// gather: every lane sums a fixed set of sources in key order and the lanes
// are combined by a fixed shuffle tree, so f_int and R are the same bit for
// bit on every run (no floating-point atomics).
// Bound by the FP64 rate and the L2: per row 9 multiply-adds per 32 sources,
// 6 additions for the three sums over the lanes, and the ghost term only where
// the row has one (its coefficients are tested as integers).  Indentation,
// 1.9 M points: 1.85 ms with six shuffle trees of 5 additions and an FP64
// compare per block, 1.20 so, 1.03 with the loads of two sources of a lane under
// way at once (of four 1.17).
__device__ inline double sum3_scatter(double f0, double f1, double f2, int lane) {
  // lane 0 ends with the sum of f0 over the warp, lane 16 of f1, lane 8 of f2
  bool up = lane & 16;
  double a = (up ? f1 : f0) + __shfl_xor_sync(0xffffffffu, up ? f0 : f1, 16);
  f2 += __shfl_xor_sync(0xffffffffu, f2, 16);
  up = lane & 8;
  a = (up ? f2 : a) + __shfl_xor_sync(0xffffffffu, up ? a : f2, 8);
  a += __shfl_xor_sync(0xffffffffu, a, 4);
  a += __shfl_xor_sync(0xffffffffu, a, 2);
  return a + __shfl_xor_sync(0xffffffffu, a, 1);
}

constexpr int RS = 2;

__global__ void k_residual_rows(int nd, int P, double load, const long long* __restrict__ sptr,
                                const uint64_t* __restrict__ skeys, const double* __restrict__ M,
                                const double* __restrict__ dS, const int* __restrict__ rp,
                                const int* __restrict__ col, const double* __restrict__ kg,
                                const double* __restrict__ du, const double* __restrict__ fext,
                                double* fint, double* R) {
  int r = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (r >= nd) return;
  double f0 = 0.0, f1 = 0.0, f2 = 0.0;
  long long q1 = sptr[r + 1];
  // RS sources of a lane at a time, all their loads under way before the sums
  for (long long q = sptr[r] + lane; q < q1; q += 32 * RS) {
    double2 m[RS][5];
    double a[RS][3];
    bool on[RS];
#pragma unroll
    for (int u = 0; u < RS; ++u) {
      uint32_t sid = q + 32 * u < q1 ? (uint32_t)skeys[q + 32 * u] : 0xffffffffu;
      int w = (int)(sid >> 6), k = (int)(sid & 63);
      on[u] = w < P;  // else a ghost-face source
      if (!on[u]) continue;
      const double2* mp = reinterpret_cast<const double2*>(M + 12 * (size_t)w);
      const double* ap = dS + 3 * ((size_t)w * MAXS + k);
#pragma unroll
      for (int i = 0; i < 5; ++i) m[u][i] = mp[i];
#pragma unroll
      for (int i = 0; i < 3; ++i) a[u][i] = ap[i];
    }
#pragma unroll
    for (int u = 0; u < RS; ++u) {
      if (!on[u]) continue;
      f0 = fma(m[u][1].x, a[u][2], fma(m[u][0].y, a[u][1], fma(m[u][0].x, a[u][0], f0)));
      f1 = fma(m[u][2].y, a[u][2], fma(m[u][2].x, a[u][1], fma(m[u][1].y, a[u][0], f1)));
      f2 = fma(m[u][4].x, a[u][2], fma(m[u][3].y, a[u][1], fma(m[u][3].x, a[u][0], f2)));
    }
  }
  double g0 = 0.0, g1 = 0.0, g2 = 0.0;
  bool ghost = false;
  for (int s = rp[r] + lane; s < rp[r + 1]; s += 32) {
    double k = kg[s];
    if (__double_as_longlong(k) << 1) {
      int c = col[s];
      ghost = true;
      g0 += k * du[3 * (size_t)c];
      g1 += k * du[3 * (size_t)c + 1];
      g2 += k * du[3 * (size_t)c + 2];
    }
  }
  double f = sum3_scatter(f0, f1, f2, lane), g = 0.0;
  if (__any_sync(0xffffffffu, ghost)) g = sum3_scatter(g0, g1, g2, lane);
  if (lane == 0 || lane == 8 || lane == 16) {
    size_t i = 3 * (size_t)r + (lane == 16 ? 1 : lane == 8 ? 2 : 0);
    fint[i] = f;
    R[i] = f - load * fext[i] + g;
  }
}

// ------------------------------------------------------------------ tangent (row gather)

constexpr int TW = 4;  // warps per block of the tangent gather (at most)
constexpr int TSMEM = 220 * 1024;  // shared memory of a block of it (at most)
constexpr int CSMEM = 200 * 1024;  // and of the contact rows
constexpr int TANGENT_FEW_ROWS = 20000;  // below: a block per row (tangent_passes)

// open-addressing table of a row's columns (dof -> position in the row), in
// shared memory: a power of two at least twice the longest row
constexpr int tangent_hash_size(int mr) {
  int h = 64;
  while (h < 2 * mr) h <<= 1;
  return h;
}

__device__ inline unsigned tangent_hash(int c, int hmask) {
  return ((unsigned)c * 2654435761u >> 7) & (unsigned)hmask;
}

// row position of every (source, support node) pair, pw per source (0xffff
// beyond the source's support, and for ghost faces): made at a mesh's first
// tangent, 2.45 ms on the indentation block, so that the gather (6.3 ms, every
// Newton iteration) needs no lookup.  A hash table
// of the row's columns in shared memory; a warp per row, or (SHARED, meshes of
// few rows) a block per row, its warps taking the sources 32 at a time in turn.
template <bool SHARED>
__global__ void k_src_pos(int nd, int P, int pw, int hs, const int* __restrict__ rp, const int* __restrict__ col,
                          const long long* __restrict__ sptr, const uint64_t* __restrict__ skeys,
                          const int* __restrict__ nsup, const int* __restrict__ sidx, unsigned short* pos) {
  extern __shared__ int smh[];
  const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int t = SHARED ? threadIdx.x : lane, nt = SHARED ? blockDim.x : 32;
  int *hkey = smh + (SHARED ? 0 : wi * 2 * hs), *hval = hkey + hs, hmask = hs - 1;
  int r = SHARED ? blockIdx.x : blockIdx.x * nw + wi;
  if (r >= nd) return;
  auto sync = [] {
    if (SHARED)
      __syncthreads();
    else
      __syncwarp();
  };
  int s0 = rp[r], nb = rp[r + 1] - s0;
  for (int i = t; i < hs; i += nt) hkey[i] = -1;
  sync();
  for (int i = t; i < nb; i += nt) {
    int c = col[s0 + i];
    unsigned h = tangent_hash(c, hmask);
    while (atomicCAS(hkey + h, -1, c) != -1) h = (h + 1) & hmask;
    hval[h] = i;
  }
  sync();
  long long q1 = sptr[r + 1];
  for (long long qb = sptr[r] + (SHARED ? 32 * wi : 0); qb < q1; qb += SHARED ? 32 * nw : 32) {
    int cnt = (int)min(32LL, q1 - qb);
    uint32_t kb = lane < cnt ? (uint32_t)skeys[qb + lane] : 0u;
    for (int u = 0; u < cnt; ++u) {
      int w = (int)(__shfl_sync(0xffffffffu, kb, u) >> 6);
      int n = w < P ? nsup[w] : 0;
      for (int l = lane; l < pw; l += 32) {
        int v = 0xffff;
        if (l < n) {
          int c = sidx[(size_t)w * MAXS + l], key;
          unsigned h = tangent_hash(c, hmask);
          while ((key = hkey[h]) != c && key != -1) h = (h + 1) & hmask;
          if (key == c) v = hval[h];
        }
        pos[(size_t)(qb + u) * pw + l] = (unsigned short)v;
      }
    }
  }
}

template <class T>
__device__ inline T dot3(const T* t, const T* g) {
  return fma(t[2], g[2], fma(t[1], g[1], t[0] * g[0]));
}
template <class T>
__device__ inline T dot3_add(const T* t, const T* g, T a) {
  return fma(t[2], g[2], fma(t[1], g[1], fma(t[0], g[0], a)));
}

// ---- FP32: a column of the support per lane

constexpr int TF_AS = 12;  // a block's 9 accumulators, padded for 16-byte accesses

// shared memory of one row: the accumulators, then the 32 terms of two sources
// (the rows of a warp 16 bytes apart in the banks)
constexpr size_t tangent_row_bytes_f32(int mr) { return ((size_t)mr * TF_AS + 64) * sizeof(float) + 16; }

// the 27 terms (grad_x S_k)^T A'_p of a source, 16-byte aligned, 32 entries
__device__ inline void tangent_terms(const float* Tt, float* t) {
  const float4* v = reinterpret_cast<const float4*>(Tt);
#pragma unroll
  for (int i = 0; i < 7; ++i) {
    float4 a = v[i];
    t[4 * i] = a.x;
    if (4 * i + 1 < 27) t[4 * i + 1] = a.y;
    if (4 * i + 2 < 27) t[4 * i + 2] = a.z;
    if (4 * i + 3 < 27) t[4 * i + 3] = a.w;
  }
}

// acc[0..8] += the block t (x) g of one (source, column) pair, with vector
// shared-memory accesses.  An entry of the block is summed first: one rounding of
// the long sum a source, not three (FMAs nested into it: 2.6e-7 of |K| in the rms
// against the FP64 tangent at 248 k rows, 1.4e-7 so, for 0.8 % of the time)
__device__ inline void tangent_add(float* a, const float* t, const float* g) {
  float4* v = reinterpret_cast<float4*>(a);
  float4 x = v[0], y = v[1];
  float z = a[8];
  x.x += dot3(t, g);
  x.y += dot3(t + 3, g);
  x.z += dot3(t + 6, g);
  x.w += dot3(t + 9, g);
  y.x += dot3(t + 12, g);
  y.y += dot3(t + 15, g);
  y.z += dot3(t + 18, g);
  y.w += dot3(t + 21, g);
  z += dot3(t + 24, g);
  v[0] = x;
  v[1] = y;
  a[8] = z;
}

// the loads of one source (point w, local index k) of a row, issued together:
// lane l of the row's HL lanes holds the grad_x S and row positions of support
// nodes l, l + HL, ... < 32 and the three A'_p factors of terms l, l + HL, ...
template <int HL>
struct TangentSrcF {
  static constexpr int NP = 32 / HL;
  float gk[4], a[NP][4], g[NP][4];
  unsigned pos[NP];
};

template <int HL>
__device__ inline void tangent_fetch_f(TangentSrcF<HL>& s, uint32_t sid, long long q, int pw, int l,
                                       const float* gx, const float* Aalg, const unsigned short* pos) {
  const float* gw = gx + 4 * (size_t)pw * (sid >> 6);
  const float* aw = Aalg + 108 * (size_t)(sid >> 6);
  const unsigned short* pq = pos + (size_t)q * pw;
  ld4(gw + 4 * (sid & 63), s.gk);
#pragma unroll
  for (int j = 0; j < 32 / HL; ++j) {
    int lj = l + HL * j;
    if (lj < 27) ld4(aw + 4 * lj, s.a[j]);
    s.pos[j] = 0xffffu;
    if (lj < pw) {  // (beyond the support: a position of 0xffff, nothing is added)
      ld4(gw + 4 * lj, s.g[j]);
      s.pos[j] = pq[lj];
    }
  }
}

// Block row r: for every point p with r in its support (local index k),
// K_{r,w} += V0_p (grad_x S_k)^T A'_p (grad_x S_w) for all w in the support of
// p, accumulated in shared memory in source order, free of atomics, and
// written out, coalesced, in the sliced layout, with the ghost coefficients and
// the Dirichlet identity (mr = longest row, a multiple of 4).
// HL lanes work on a source.  HL = 16: a warp takes two rows (16 nodes is the
// mean support), one per half, so that a warp instruction serves two sources.
// Bound by shared-memory wavefronts: the accumulators' round trip at random
// 48-byte slots, 37 of them per source, and 15 of the loads (ncu, LSU data
// pipe 72 % busy).  Indentation, 1.9 M points, 28.8 M sources: 7.6 ms with a
// hash lookup per pair and 13 loads per source, 6.4 with the precomputed
// positions and 16-byte loads, 6.0 with two rows per warp (the long rows' pass
// 1.2 -> 0.36 of it); an entry of the block per lane, as in FP64, 7.0.
// HL = 32, WPR > 1: the warps of a block share a row, each taking a contiguous
// part of its sources with a copy of the accumulators, added up in warp order:
// for rows whose serial chain of sources would be the time (few rows, and the
// long rows near hanging nodes).
template <int HL, int WPR>
__global__ void __launch_bounds__(32 * TW)
    k_tangent_rows_f32(int nd, int P, int pw, int minlen, int mr, int last, const int* __restrict__ rp,
                   const int* __restrict__ col, Sliced S, const long long* __restrict__ sptr,
                   const uint64_t* __restrict__ skeys, const unsigned short* __restrict__ spos,
                   const float* __restrict__ gx, const float* __restrict__ Aalg, const double* __restrict__ kg,
                   const int* __restrict__ mask, float* K, int* err) {
  static_assert(HL == 32 || WPR == 1, "shared rows take whole warps");
  constexpr int AS = TF_AS, RPW = 32 / HL, NP = 32 / HL;
  extern __shared__ __align__(16) unsigned char smraw[];
  const unsigned FULL = 0xffffffffu;
  int wi = threadIdx.x >> 5, lane = threadIdx.x & 31, l = lane % HL, part = wi % WPR;
  const size_t rsz = (size_t)mr * AS + 68;
  float* acc = (float*)smraw + (wi * RPW + lane / HL) * rsz;
  float* Tt = acc + AS * (size_t)mr;
  // rows in storage order: the two rows of a warp have about the same length
  int sr = (blockIdx.x * ((blockDim.x >> 5) / WPR) + wi / WPR) * RPW + lane / HL;
  int r = sr < nd ? S.row[sr] : nd, s0 = 0, nb = 0;
  bool live = r < nd;
  if (live) {
    s0 = rp[r];
    nb = rp[r + 1] - s0;
    if (nb > mr && last && l == 0) atomicOr(err, EB_ROW);
    live = nb > minlen && nb <= mr;  // else done by the other pass
  }
  if (WPR == 1 && !__any_sync(FULL, live)) return;
  int n = 0;  // this row's (part's) sources
  long long q0 = 0;
  if (live) {
    for (int i = l; i < AS * nb; i += HL) acc[i] = 0.f;
    // the point sources come first in the row's key order, the ghost faces last
    long long lo = sptr[r], hi = sptr[r + 1];
    q0 = lo;
    while (lo < hi) {
      long long mid = (lo + hi) >> 1;
      if ((int)((uint32_t)skeys[mid] >> 6) < P)
        lo = mid + 1;
      else
        hi = mid;
    }
    n = (int)(lo - q0);
    if (WPR > 1) {
      int e = (int)((long long)n * (part + 1) / WPR);
      n = (int)((long long)n * part / WPR);
      q0 += n;
      n = e - n;
    }
  }
  int nmax = HL == 32 ? n : (int)__reduce_max_sync(FULL, n);
  __syncwarp();
  // the source keys HL at a time (one coalesced load, then broadcast); a row
  // with no source left repeats a source of its own without adding it
  if (nmax > 0) {
    auto keys = [&](int u0) { return u0 + l < n ? (uint32_t)skeys[q0 + u0 + l] : 0u; };
    uint32_t kb = keys(0), sid = __shfl_sync(FULL, kb, 0, HL);
    TangentSrcF<HL> s;
    tangent_fetch_f<HL>(s, sid, q0, pw, l, gx, Aalg, spos);
    for (int u = 0; u < nmax; ++u) {
      TangentSrcF<HL> nx;
      uint32_t nsid = 0;
      if (u + 1 < nmax) {
        if ((u + 1) % HL == 0) kb = keys(u + 1);
        nsid = __shfl_sync(FULL, kb, (u + 1) % HL, HL);
        tangent_fetch_f<HL>(nx, nsid, u + 1 < n ? q0 + u + 1 : 0, pw, l, gx, Aalg, spos);
      }
      // two sets of terms in turn: one __syncwarp per source separates both
      // the terms' writes from their reads and the row's updates
      float* tt = Tt + 32 * (u & 1);
#pragma unroll
      for (int j = 0; j < NP; ++j)
        if (l + HL * j < 27) tt[l + HL * j] = dot3(s.a[j], s.gk);
      __syncwarp();
      float t[27];
      tangent_terms(tt, t);
      const bool on = u < n;
#pragma unroll
      for (int j = 0; j < NP; ++j)
        if (on && s.pos[j] != 0xffffu) tangent_add(acc + AS * s.pos[j], t, s.g[j]);
      // supports of more than 32 nodes (deep hanging chains)
      if (pw > 32)
        for (int i = l + 32; on && i < pw; i += HL) {
          unsigned pl = spos[(size_t)(q0 + u) * pw + i];
          if (pl == 0xffffu) continue;
          float g[4];
          ld4(gx + 4 * ((size_t)(sid >> 6) * pw + i), g);
          tangent_add(acc + AS * pl, t, g);
        }
      s = nx;
      sid = nsid;
    }
  }
  if (WPR > 1) {
    __syncthreads();
    acc = (float*)smraw + (wi - part) * rsz;
  } else {
    __syncwarp();
  }
  if (!live) return;
  // ghost, then the Dirichlet identity, then the row (and its padding slots,
  // zero) into the sliced storage
  int mr_ = mask[r];
  int sl = sr >> 5, W = S.w[sl];
  long long b0 = S.base[sl];
  for (int i = l + HL * part; i < W; i += HL * WPR) {
    long long slot = sliced_slot(b0, sr, i);
    if (i >= nb) {
#pragma unroll
      for (int e = 0; e < 9; ++e) K[sliced_entry(b0, W, slot, e)] = 0.f;
      continue;
    }
    // the ghost coefficient is zero away from the cut cells: convert only
    // where some lane of the warp has one
    double kd = kg[s0 + i];
    float kv = __any_sync(__activemask(), kd != 0.0) ? (float)kd : 0.f;
    int c = col[s0 + i];
    int mc = mask[c];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        int e = 3 * a + b;
        float v = acc[AS * i + e];
#pragma unroll
        for (int w = 1; w < WPR; ++w) v += acc[w * rsz + AS * i + e];
        if (a == b) v += kv;
        if (((mr_ >> a) & 1) || ((mc >> b) & 1)) v = (c == r && a == b) ? 1.f : 0.f;
        K[sliced_entry(b0, W, slot, e)] = v;
      }
  }
}

// ---- FP64: an entry of the block per lane

// shared memory of one warp: the gradients (and, in their fourth component,
// row positions) of the support nodes of two sources, then the row's 9
// accumulators per block
inline size_t tangent_warp_bytes_f64(int mr) { return (9 * (size_t)mr + 256) * sizeof(double); }

// the loads of one source (point w, local index k) of a row, issued together:
// lane l holds the l-th support node's grad_x S and row position, lanes < 27
// the three A'_p factors of one of the 27 terms
struct TangentSrcD {
  double gk[4], a[4], g[4];
  unsigned pos;
};

__device__ inline void tangent_fetch_d(TangentSrcD& s, uint32_t sid, long long q, int pw, int lane, const double* gx,
                                       const double* Aalg, const unsigned short* pos) {
  const double* gw = gx + 4 * (size_t)pw * (sid >> 6);
  ld4(gw + 4 * (sid & 63), s.gk);
  if (lane < 27) ld4(Aalg + 108 * (size_t)(sid >> 6) + 4 * lane, s.a);
  s.pos = 0xffffu;
  if (lane < pw) {  // (beyond the support: a position of 0xffff)
    ld4(gw + 4 * lane, s.g);
    s.pos = pos[(size_t)q * pw + lane];
  }
}

// Block row r: for every point p with r in its support (local index k),
// K_{r,w} += V0_p (grad_x S_k)^T A'_p (grad_x S_w) for all w in the support of
// p, accumulated in shared memory in source order, free of atomics, and
// written out, coalesced, in the sliced layout, with the ghost coefficients and
// the Dirichlet identity (mr = longest row, a multiple of 4).
// The 27 working lanes of a warp are the 9 entries of a block times three
// columns: a lane keeps the three terms (grad_x S_k)^T A'_p of its entry in
// registers and walks the support three columns at a time.  Bound by the FP64
// rate (an FP64 instruction takes 16 SM cycles however many lanes are active),
// which this spends on ceil(n / 3) times 3 FMAs for n columns, or half of them
// in the upper triangle; a column per lane takes 27 (36 before the sums were
// nested FMAs) whatever n.  Punch, 17.8 k points: 2.47 ms with a column per
// lane and a warp per row, 0.75 with four warps per row, 0.52 so.
// WPR > 1: the warps of a block share a row, each taking a contiguous part of
// its sources with a copy of the accumulators, added up in warp order.
// UPPER (a symmetric tangent: Hencky, von Mises, frictionless contact): only
// the blocks of columns c >= r are formed and written; k_tangent_mirror then
// copies each into its transposed place.
template <bool UPPER, int WPR>
__global__ void __launch_bounds__(32 * TW)
    k_tangent_rows_f64(int nd, int P, int pw, int minlen, int mr, int last, const int* __restrict__ rp,
                   const int* __restrict__ col, Sliced S, const long long* __restrict__ sptr,
                   const uint64_t* __restrict__ skeys, const unsigned short* __restrict__ spos,
                   const double* __restrict__ gx, const double* __restrict__ Aalg, const double* __restrict__ kg,
                   const int* __restrict__ mask, double* K, int* err) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const unsigned FULL = 0xffffffffu;
  int wi = threadIdx.x >> 5, lane = threadIdx.x & 31, part = wi % WPR;
  const int e = lane % 9, cg = lane < 27 ? lane / 9 : 1 << 20;  // (idle lanes: no column)
  const size_t wsz = 9 * (size_t)mr + 256;
  double* sg = (double*)smraw + wi * wsz;  // [2][32][4]
  double* acc = sg + 256;
  int r = blockIdx.x * ((blockDim.x >> 5) / WPR) + wi / WPR;
  int s0 = 0, nb = 0;
  bool live = r < nd;
  if (live) {
    s0 = rp[r];
    nb = rp[r + 1] - s0;
    if (nb > mr && last && lane == 0) atomicOr(err, EB_ROW);
    live = nb > minlen && nb <= mr;  // else done by the other pass
  }
  if (WPR == 1 && !live) return;
  if (live) {
    for (int i = lane; i < 9 * nb; i += 32) acc[i] = 0.0;
    // the point sources come first in the row's key order, the ghost faces last
    long long q0 = sptr[r], q1 = sptr[r + 1];
    {
      long long lo = q0;
      while (lo < q1) {
        long long mid = (lo + q1) >> 1;
        if ((int)((uint32_t)skeys[mid] >> 6) < P)
          lo = mid + 1;
        else
          q1 = mid;
      }
    }
    if (WPR > 1) {
      long long n = q1 - q0;
      q1 = q0 + n * (part + 1) / WPR;
      q0 += n * part / WPR;
    }
    int n = (int)(q1 - q0);
    if (n > 0) {
      // the row's source keys 32 at a time (one coalesced load, then broadcast)
      uint32_t kb = lane < n ? (uint32_t)skeys[q0 + lane] : 0u, sid = __shfl_sync(FULL, kb, 0);
      TangentSrcD s;
      tangent_fetch_d(s, sid, q0, pw, lane, gx, Aalg, spos);
      for (int u = 0; u < n; ++u) {
        double tv = dot3(s.a, s.gk), t[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) t[j] = __shfl_sync(FULL, tv, 3 * e + j);
        s.g[3] = __longlong_as_double((long long)s.pos);
        double* sb = sg + 128 * (u & 1);  // two sets in turn: one __syncwarp per source
        st4(sb + 4 * lane, s.g);
        int ns = __popc(__ballot_sync(FULL, s.pos != 0xffffu));
        // (UPPER: the supports are sorted, so the columns c >= r are the nodes
        // from the source's own on)
        const int k0 = UPPER ? (int)(sid & 63) : 0;
        const uint32_t w = sid >> 6;
        if (u + 1 < n) {
          if (((u + 1) & 31) == 0) kb = u + 1 + lane < n ? (uint32_t)skeys[q0 + u + 1 + lane] : 0u;
          sid = __shfl_sync(FULL, kb, (u + 1) & 31);
          tangent_fetch_d(s, sid, q0 + u + 1, pw, lane, gx, Aalg, spos);
        }
        __syncwarp();
        // three trips at a time: their columns are distinct
        for (int c = k0 + cg; c < ns; c += 9) {
          double v[3][4], x[3];
          double* a[3];
#pragma unroll
          for (int j = 0; j < 3; ++j) {
            int cj = min(c + 3 * j, 31);
            ld4(sb + 4 * cj, v[j]);
            a[j] = acc + 9 * (unsigned)__double_as_longlong(v[j][3]) + e;
          }
#pragma unroll
          for (int j = 0; j < 3; ++j)
            if (c + 3 * j < ns) x[j] = *a[j];
#pragma unroll
          for (int j = 0; j < 3; ++j)
            if (c + 3 * j < ns) *a[j] = dot3_add(t, v[j], x[j]);
        }
        // supports of more than 32 nodes (deep hanging chains)
        if (pw > 32) {
          const unsigned short* pq = spos + (size_t)(q0 + u) * pw;
          for (int i = max(32, k0) + cg; i < pw && pq[i] != 0xffffu; i += 3) {
            double g[4];
            ld4(gx + 4 * ((size_t)w * pw + i), g);
            double* a = acc + 9 * (unsigned)pq[i] + e;
            *a = dot3_add(t, g, *a);
          }
        }
      }
    }
  }
  if (WPR > 1) {
    __syncthreads();
    if (!live) return;
    acc -= part * (ptrdiff_t)wsz;
  } else {
    __syncwarp();
  }
  // ghost, then the Dirichlet identity, then the row (and its padding slots,
  // zero) into the sliced storage
  int mr_ = mask[r];
  int sr = S.pos[r], sl = sr >> 5, W = S.w[sl];
  long long b0 = S.base[sl];
  for (int i = lane + 32 * part; i < W; i += 32 * WPR) {
    long long slot = sliced_slot(b0, sr, i);
    if (i >= nb) {
#pragma unroll
      for (int k = 0; k < 9; ++k) K[sliced_entry(b0, W, slot, k)] = 0.0;
      continue;
    }
    // the ghost coefficient is zero away from the cut cells: convert only
    // where some lane of the warp has one
    double kd = kg[s0 + i];
    double kv = __any_sync(__activemask(), kd != 0.0) ? kd : 0.0;
    int c = col[s0 + i];
    if (UPPER && c < r) continue;  // written by k_tangent_mirror
    int mc = mask[c];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        int k = 3 * a + b;
        double v = acc[9 * i + k];
#pragma unroll
        for (int u = 1; u < WPR; ++u) v += acc[u * wsz + 9 * i + k];
        if (a == b) v += kv;
        if (((mr_ >> a) & 1) || ((mc >> b) & 1)) v = (c == r && a == b) ? 1.0 : 0.0;
        K[sliced_entry(b0, W, slot, k)] = v;
      }
  }
}

// the lower blocks of a symmetric tangent: block (r, c), c < r, is the
// transpose of block (c, r), found by binary search in row c (one warp per row)
__global__ void k_tangent_mirror(int nd, const int* __restrict__ rp, const int* __restrict__ col,
                                 Sliced S, double* K) {
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  int r = (int)(t >> 5), lane = (int)(t & 31);
  if (r >= nd) return;
  int s0 = rp[r], nb = rp[r + 1] - s0;
  int sr = S.pos[r], sl = sr >> 5, W = S.w[sl];
  long long b0 = S.base[sl];
  for (int i = lane; i < nb; i += 32) {
    int c = col[s0 + i];
    if (c >= r) break;  // columns sorted: the rest is the upper part
    int lo = rp[c], hi = rp[c + 1] - 1, j = -1;
    while (lo <= hi) {
      int mid = (lo + hi) >> 1, v = col[mid];
      if (v == r) {
        j = mid;
        break;
      }
      if (v < r)
        lo = mid + 1;
      else
        hi = mid - 1;
    }
    if (j < 0) continue;  // (the pattern is symmetric: never)
    int src = S.pos[c], slc = src >> 5, Wc = S.w[slc];
    long long bc = S.base[slc], sc = sliced_slot(bc, src, j - rp[c]);
    double v[9];
#pragma unroll
    for (int e = 0; e < 9; ++e) v[e] = K[sliced_entry(bc, Wc, sc, e)];
    long long slot = sliced_slot(b0, sr, i);
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int b = 0; b < 3; ++b) K[sliced_entry(b0, W, slot, 3 * a + b)] = v[3 * b + a];
  }
}

// rows beyond ndof in the last slice (stored in place): zero padding slots
template <class T>
__global__ void k_zero_pad_rows(int nd, int npad, Sliced S, T* K) {
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  int r = nd + (int)(t >> 5), lane = (int)(t & 31);
  if (r >= npad) return;
  int sl = r >> 5, W = S.w[sl];
  long long b0 = S.base[sl];
  for (int i = lane; i < W; i += 32) {
    long long slot = sliced_slot(b0, r, i);
    for (int e = 0; e < 9; ++e) K[sliced_entry(b0, W, slot, e)] = (T)0;
  }
}

// sliced values -> plain [nnzb][3][3] blocks (FP64)
template <class T>
__global__ void k_blocks_export(int nd, const int* __restrict__ rp, Sliced S, const T* __restrict__ K,
                                double* out) {
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  int r = (int)(t >> 5), lane = (int)(t & 31);
  if (r >= nd) return;
  int sr = S.pos[r], sl = sr >> 5, W = S.w[sl];
  long long b0 = S.base[sl];
  for (int i = lane; i < rp[r + 1] - rp[r]; i += 32) {
    long long slot = sliced_slot(b0, sr, i);
    for (int e = 0; e < 9; ++e) out[9 * (size_t)(rp[r] + i) + e] = (double)K[sliced_entry(b0, W, slot, e)];
  }
}

// ------------------------------------------------------------------ contact (Sec. 2.3)

__device__ inline int find_slot(const int* __restrict__ rp, const int* __restrict__ col, int r, int c) {
  int lo = rp[r], hi = rp[r + 1] - 1;
  while (lo <= hi) {
    int mid = (lo + hi) >> 1;
    int v = col[mid];
    if (v == c) return mid;
    if (v < c)
      lo = mid + 1;
    else
      hi = mid - 1;
  }
  return -1;
}

// [a]x, the matrix of b -> a x b (row-major)
__device__ inline void cross_mat(const double* a, double* C) {
  C[0] = 0.0;
  C[1] = -a[2];
  C[2] = a[1];
  C[3] = a[2];
  C[4] = 0.0;
  C[5] = -a[0];
  C[6] = -a[1];
  C[7] = a[0];
  C[8] = 0.0;
}

__device__ inline void mul33(const double* A, const double* B, double* C) {
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) C[3 * i + j] = A[3 * i] * B[j] + A[3 * i + 1] * B[3 + j] + A[3 * i + 2] * B[6 + j];
}

// one thread per candidate domain corner: the gap against the body at the moved
// corner; in contact the force on the material f (normal f_N n with
// f_N = -eps_N phi, plus Coulomb friction) and k_c = -d f / d y are stored for
// the row gather below (zeros and on = 0 otherwise), and with `reac` the
// force on the body, -sum f, is summed in a fixed order (every thread of the
// grid takes part).  The body sits at its given pose moved by bi.shift; the
// friction measures the node's slip against the body's own displacement at
// the node, qt + qr x d (d = y - X, X the body's reference point); with
// `ct` the derivative of f in the body's rotation ([d]x through the slip) and
// d are stored per corner for the body's equations.
__global__ void k_contact_corner(int nc8, const int* __restrict__ cand, const int* __restrict__ cb_n,
                                 const int* __restrict__ cb_idx, const double* __restrict__ cb_phi,
                                 const double* __restrict__ cb_y0, const double* __restrict__ pE,
                                 const double* __restrict__ pV0, Body body, double L, double pf,
                                 double pt, double mu, BodyInc bi,
                                 const double* __restrict__ du, double* cf, double* ck, int* con,
                                 double* ct, double* cdv, double* reac, GridRed gr) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  double f[3] = {0.0, 0.0, 0.0};
  if (i < nc8) {
    int w = cand[i >> 3], n = cb_n[i];
    const int* ids = cb_idx + (size_t)i * MAXCB;
    const double* ph = cb_phi + (size_t)i * MAXCB;
    double y[3] = {cb_y0[3 * (size_t)i], cb_y0[3 * (size_t)i + 1], cb_y0[3 * (size_t)i + 2]};
    for (int e = 0; e < n; ++e)
      for (int d = 0; d < 3; ++d) y[d] += ph[e] * du[3 * (size_t)ids[e] + d];
    double phi, nv[3], H[9], yb[3], dv[3];
    for (int d = 0; d < 3; ++d) yb[d] = y[d] - bi.shift[d];
    bool on = body_sdf(body, L, yb, &phi, nv, H) && phi < 0.0;
    dv[0] = y[0] - (body.b.cx + bi.shift[0]);
    dv[1] = y[1] - (body.b.cy + bi.shift[1]);
    dv[2] = y[2] - (body.b.z + bi.shift[2]);
    double Fy[9], Ft[9];
    for (int e = 0; e < 9; ++e) Fy[e] = Ft[e] = 0.0;
    if (on) {
      double A0 = pow(pV0[w], 2.0 / 3.0);
      double epsN = pf * pE[w] * A0, fN = -epsN * phi;
      for (int d = 0; d < 3; ++d) f[d] = fN * nv[d];
      for (int a = 0; a < 3; ++a)
        for (int b = 0; b < 3; ++b) Fy[3 * a + b] = -epsN * (nv[a] * nv[b] + phi * H[3 * a + b]);
      if (mu > 0.0) {
        // Coulomb friction: the slip g = (y - y0) - (qt + qr x d) on the
        // tangent plane; trial force t = -eps_T (I - n n^T) g, stick while
        // |t| <= mu f_N, else slip with mu f_N t / |t|; Jd, Jg its
        // derivatives in d (through n, H, f_N) and in g
        double epsT = pt * pE[w] * A0;
        double g[3], t[3], Hg[3], Td[9], Tg[9], Jd[9], Jg[9];
        for (int d = 0; d < 3; ++d) {
          double rot = bi.qr[(d + 1) % 3] * dv[(d + 2) % 3] - bi.qr[(d + 2) % 3] * dv[(d + 1) % 3];
          g[d] = (y[d] - cb_y0[3 * (size_t)i + d]) - (bi.qt[d] + rot);
        }
        double ng = nv[0] * g[0] + nv[1] * g[1] + nv[2] * g[2];
        for (int a = 0; a < 3; ++a) Hg[a] = H[3 * a] * g[0] + H[3 * a + 1] * g[1] + H[3 * a + 2] * g[2];
        for (int d = 0; d < 3; ++d) t[d] = -epsT * (g[d] - nv[d] * ng);
        for (int a = 0; a < 3; ++a)
          for (int b = 0; b < 3; ++b) {
            Td[3 * a + b] = epsT * (ng * H[3 * a + b] + nv[a] * Hg[b]);
            Tg[3 * a + b] = -epsT * ((a == b ? 1.0 : 0.0) - nv[a] * nv[b]);
          }
        double tn = sqrt(t[0] * t[0] + t[1] * t[1] + t[2] * t[2]);
        if (tn <= mu * fN) {
          for (int d = 0; d < 3; ++d) f[d] += t[d];
          for (int e = 0; e < 9; ++e) {
            Jd[e] = Td[e];
            Jg[e] = Tg[e];
          }
        } else {
          double u[3] = {t[0] / tn, t[1] / tn, t[2] / tn};
          for (int d = 0; d < 3; ++d) f[d] += mu * fN * u[d];
          for (int a = 0; a < 3; ++a)
            for (int b = 0; b < 3; ++b) {
              double sd = 0.0, sg = 0.0;
              for (int c = 0; c < 3; ++c) {
                double P = (a == c ? 1.0 : 0.0) - u[a] * u[c];
                sd += P * Td[3 * c + b];
                sg += P * Tg[3 * c + b];
              }
              Jd[3 * a + b] = mu * u[a] * (-epsN * nv[b]) + mu * fN * sd / tn;
              Jg[3 * a + b] = mu * fN * sg / tn;
            }
        }
        // d f / d y = N + Jd + Jg (I - [qr]x); d f / d qr = Jg [d]x
        double Qr[9], IQ[9], T[9], Dx[9];
        cross_mat(bi.qr, Qr);
        for (int e = 0; e < 9; ++e) IQ[e] = (e % 4 == 0 ? 1.0 : 0.0) - Qr[e];
        mul33(Jg, IQ, T);
        for (int e = 0; e < 9; ++e) Fy[e] += Jd[e] + T[e];
        cross_mat(dv, Dx);
        mul33(Jg, Dx, Ft);
      }
    }
    for (int d = 0; d < 3; ++d) cf[3 * (size_t)i + d] = f[d];
    for (int e = 0; e < 9; ++e) ck[9 * (size_t)i + e] = -Fy[e];
    con[i] = on ? 1 : 0;
    if (ct) {
      for (int e = 0; e < 9; ++e) ct[9 * (size_t)i + e] = Ft[e];
      for (int d = 0; d < 3; ++d) cdv[3 * (size_t)i + d] = dv[d];
    }
  }
  if (reac) {
    double v[3] = {-f[0], -f[1], -f[2]};
    double* o[3] = {reac, reac + 1, reac + 2};
    grid_sum<3>(v, o, gr);
  }
}

// the set entries of a chunk of NPER blockDim.x, in order, in list (shared
// memory): on(i) tells whether entry i of the chunk is set, its value goes in;
// returns their number.  Every thread of the block calls; ends with a
// __syncthreads.
template <int NPER, class F, class G>
__device__ inline int block_compact(F on, G value, int* list, int* wsum) {
  int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  unsigned m[NPER];
  int mine = 0;
#pragma unroll
  for (int u = 0; u < NPER; ++u) {
    m[u] = __ballot_sync(0xffffffffu, on((w * NPER + u) * 32 + lane));
    mine += __popc(m[u]);
  }
  if (lane == 0) wsum[w] = mine;
  __syncthreads();
  int base = 0, n = 0;
  for (int i = 0; i < (int)(blockDim.x >> 5); ++i) {
    if (i < w) base += wsum[i];
    n += wsum[i];
  }
#pragma unroll
  for (int u = 0; u < NPER; ++u) {
    if ((m[u] >> lane) & 1) list[base + __popc(m[u] & ((1u << lane) - 1u))] = value((w * NPER + u) * 32 + lane);
    base += __popc(m[u]);
  }
  __syncthreads();
  return n;
}

// The rigid body's sums over the contact corners, in a fixed order (one
// block): the corners in contact, a few of the candidates, are listed in order
// and dealt to the threads in turn; the threads' 42 sums are added up through
// shared memory, a warp per value.  out[0..5] the residual terms f and d x f,
// out[6..41] their derivative in the body's increment q (row-major 6 x 6):
// [d f / d qt, d f / d qr; [f]x + [d]x d f / d qt, [d]x d f / d qr] with
// d f / d qt = -d f / d y.  (A tree of shuffles per value and warp, 5 FP64
// additions at 16 SM cycles each, made this 51 us on the rolling sphere's 2.4 k
// candidates; 47 so, most of it the scan.)
constexpr int BSUM_T = 256, BSUM_N = 8;
__global__ void __launch_bounds__(BSUM_T)
    k_body_sums(int nc8, const double* __restrict__ cf, const double* __restrict__ ck, const double* __restrict__ ct,
                const double* __restrict__ cdv, const int* __restrict__ con, double* out) {
  __shared__ int list[BSUM_N * BSUM_T], wsum[BSUM_T / 32];
  __shared__ double sh[14][BSUM_T];
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  double acc[42];
  for (int e = 0; e < 42; ++e) acc[e] = 0.0;
  int busy = 0, next = 0;  // threads with a sum; thread of the next corner
  for (int base = 0; base < nc8; base += BSUM_N * BSUM_T) {
    int n = block_compact<BSUM_N>([&](int i) { return base + i < nc8 && con[base + i] != 0; },
                                  [&](int i) { return base + i; }, list, wsum);
    // corner j of the list goes to thread (next + j) % BSUM_T
    for (int j = (t - next + BSUM_T) % BSUM_T; j < n; j += BSUM_T) {
      int i = list[j];
      const double* f = cf + 3 * (size_t)i;
      const double* d = cdv + 3 * (size_t)i;
      const double* Ft = ct + 9 * (size_t)i;
      double FX[9], Dx[9], Fx[9], DF[9], DT[9];
      for (int e = 0; e < 9; ++e) FX[e] = ck[9 * (size_t)i + e];  // -d f / d y
      cross_mat(d, Dx);
      cross_mat(f, Fx);
      mul33(Dx, FX, DF);
      mul33(Dx, Ft, DT);
      for (int a = 0; a < 3; ++a) {
        acc[a] += f[a];
        acc[3 + a] += d[(a + 1) % 3] * f[(a + 2) % 3] - d[(a + 2) % 3] * f[(a + 1) % 3];
        for (int b = 0; b < 3; ++b) {
          acc[6 + 6 * a + b] += FX[3 * a + b];
          acc[6 + 6 * a + 3 + b] += Ft[3 * a + b];
          acc[6 + 6 * (3 + a) + b] += Fx[3 * a + b] + DF[3 * a + b];
          acc[6 + 6 * (3 + a) + 3 + b] += DT[3 * a + b];
        }
      }
    }
    busy = min(BSUM_T, busy + n);
    next = (next + n) % BSUM_T;
    __syncthreads();
  }
#pragma unroll
  for (int h = 0; h < 3; ++h) {
    if (t < busy)
      for (int e = 0; e < 14; ++e) sh[e][t] = acc[14 * h + e];
    __syncthreads();
    for (int e = w; e < 14; e += BSUM_T / 32) {
      double v = lane < busy ? sh[e][lane] : 0.0;
      for (int u = lane + 32; u < busy; u += 32) v += sh[e][u];
      v = warp_sum(v);
      if (lane == 0) out[14 * h + e] = v;
    }
    __syncthreads();
  }
}

// the body's coupling columns and rows at the rows of the contact list (one
// block of 64 per row, a thread per output value, the row's corner entries in
// contact in list order): Kgb[j][3r + a] = d R_{r,a} / d q_j = sum phi (d f /
// d y)[a][j] for the translation (j < 3) and -sum phi (d f / d qr)[a][j - 3]
// for the rotation; Kbg[j][3r + b] = d Rb_j / d du_{r,b} = sum phi (d f / d
// y)[j][b] (j < 3) and sum phi ([d]x d f / d y - [f]x)[j - 3][b]
__global__ void __launch_bounds__(64)
    k_body_rows(const int* __restrict__ crow, const int* __restrict__ cptr, const int* __restrict__ cent,
                const double* __restrict__ cb_phi, const double* __restrict__ cf, const double* __restrict__ ck,
                const double* __restrict__ ct, const double* __restrict__ cdv, const int* __restrict__ con,
                long long n3, double* Kgb, double* Kbg) {
  __shared__ int list[64], wsum[2];
  const int t = blockIdx.x, o = threadIdx.x;
  int r = crow[t], e0 = cptr[t], e1 = cptr[t + 1];
  // o < 18: Kgb, component a = o / 6 of row r, body column j = o % 6;
  // o >= 18: Kbg, body row j = (o - 18) / 3, component b = (o - 18) % 3
  bool gb = o < 18;
  int a = gb ? o / 6 : (o - 18) % 3, j = gb ? o % 6 : (o - 18) / 3;
  double s = 0.0;
  for (int base = e0; base < e1; base += 64) {
    int pk0 = base + o < e1 ? cent[base + o] : 0;
    int n = block_compact<1>([&](int) { return base + o < e1 && con[pk0 >> 5] != 0; }, [&](int) { return pk0; }, list,
                             wsum);
    if (o < 36)
      for (int u = 0; u < n; ++u) {
        int pk = list[u], i = pk >> 5;
        double ph = cb_phi[(size_t)i * MAXCB + (pk & 31)];
        const double* Fm = ck + 9 * (size_t)i;  // -d f / d y
        double v;
        if (gb) {
          v = j < 3 ? -Fm[3 * a + j] : -ct[9 * (size_t)i + 3 * a + (j - 3)];
        } else if (j < 3) {
          v = -Fm[3 * j + a];
        } else {
          const double* d = cdv + 3 * (size_t)i;
          const double* f = cf + 3 * (size_t)i;
          int jr = j - 3, j1 = (jr + 1) % 3, j2 = (jr + 2) % 3;
          // ([d]x (d f / d y))[jr][a] - ([f]x)[jr][a]
          double dF = -(d[j1] * Fm[3 * j2 + a] - d[j2] * Fm[3 * j1 + a]);
          double fx = (a == j2 ? f[j1] : 0.0) - (a == j1 ? f[j2] : 0.0);
          v = dF - fx;
        }
        s += ph * v;
      }
    __syncthreads();
  }
  if (o >= 36) return;
  if (gb)
    Kgb[(size_t)j * n3 + 3 * (size_t)r + a] = s;
  else
    Kbg[(size_t)j * n3 + 3 * (size_t)r + a] = s;
}

// Newmark inertia of each point (time steps): m_p a_p with
// a_p = (2 / dt^2) (sum_v S_vp du_v - dt v_p)
__global__ void k_point_inertia(int P, const int* __restrict__ nsup, const int* __restrict__ sidx,
                                const double* __restrict__ S, const double* __restrict__ du,
                                const double* __restrict__ v, const double* __restrict__ mass,
                                double dt, double* ma) {
  int w = blockIdx.x * blockDim.x + threadIdx.x;
  if (w >= P) return;
  double u[3] = {0.0, 0.0, 0.0};
  int n = nsup[w];
  for (int k = 0; k < n; ++k) {
    size_t o = (size_t)w * MAXS + k;
    int j = sidx[o];
    for (int d = 0; d < 3; ++d) u[d] += S[o] * du[3 * (size_t)j + d];
  }
  double c2 = 2.0 / (dt * dt);
  for (int d = 0; d < 3; ++d) ma[3 * (size_t)w + d] = mass[w] * (c2 * (u[d] - dt * v[3 * (size_t)w + d]));
}

// the inertia term of Eq. (MPMweak), sum_p S_vp m_p a_p, gathered per row over
// the row's point sources (warp per row): added to R and stored in finert
__global__ void k_inertia_rows(int nd, int P, const long long* __restrict__ sptr,
                               const uint64_t* __restrict__ skeys, const double* __restrict__ S,
                               const double* __restrict__ ma, double* R, double* finert) {
  int r = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (r >= nd) return;
  double a0 = 0.0, a1 = 0.0, a2 = 0.0;
  for (long long q = sptr[r] + lane; q < sptr[r + 1]; q += 32) {
    uint32_t sid = (uint32_t)skeys[q];
    int w = (int)(sid >> 6), k = (int)(sid & 63);
    if (w >= P) continue;  // ghost-face source
    double sv = S[(size_t)w * MAXS + k];
    a0 += sv * ma[3 * (size_t)w];
    a1 += sv * ma[3 * (size_t)w + 1];
    a2 += sv * ma[3 * (size_t)w + 2];
  }
  a0 = warp_sum(a0);
  a1 = warp_sum(a1);
  a2 = warp_sum(a2);
  if (lane < 3) {
    double a = lane == 0 ? a0 : (lane == 1 ? a1 : a2);
    R[3 * (size_t)r + lane] += a;
    finert[3 * (size_t)r + lane] = a;
  }
}

// the consistent mass of a time step, (2 / dt^2) m_p S_vp S_wp I, added to the
// tangent's diagonal entries: one block per row r, its warps taking a
// contiguous part of the row's point sources each (the lanes over the source
// point's support) into their own copy of the row's sums in shared memory, by
// the row positions of the tangent gather; the copies added in warp order,
// the Dirichlet components skipped
template <class T>
__global__ void k_mass_rows(int P, int pw, int mr, const long long* __restrict__ sptr,
                            const uint64_t* __restrict__ skeys, const unsigned short* __restrict__ spos,
                            const double* __restrict__ S, const double* __restrict__ mass, double c2,
                            const int* __restrict__ rp, const int* __restrict__ col, Sliced SL,
                            const int* __restrict__ mask, T* K) {
  extern __shared__ double smm[];
  const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5, nw = blockDim.x >> 5, r = blockIdx.x;
  double* acc = smm + (size_t)wi * mr;
  int s0 = rp[r], nb = rp[r + 1] - s0;
  for (int i = lane; i < nb; i += 32) acc[i] = 0.0;
  __syncwarp();
  long long q0 = sptr[r], n = sptr[r + 1] - q0;
  for (long long q = q0 + n * wi / nw; q < q0 + n * (wi + 1) / nw; ++q) {
    uint32_t sid = (uint32_t)skeys[q];
    int w = (int)(sid >> 6), k = (int)(sid & 63);
    if (w >= P) continue;
    double sk = c2 * mass[w] * S[(size_t)w * MAXS + k];
    for (int l = lane; l < pw; l += 32) {
      unsigned p = spos[(size_t)q * pw + l];
      if (p != 0xffffu) acc[p] += sk * S[(size_t)w * MAXS + l];
    }
    __syncwarp();
  }
  __syncthreads();
  int ma = mask[r], srr = SL.pos[r], slc = srr >> 5, W = SL.w[slc];
  long long b0 = SL.base[slc];
  for (int i = threadIdx.x; i < nb; i += blockDim.x) {
    double v = smm[i];
    for (int u = 1; u < nw; ++u) v += smm[(size_t)u * mr + i];
    int m = ma | mask[col[s0 + i]];
    long long slot = sliced_slot(b0, srr, i);
    for (int a = 0; a < 3; ++a)
      if (!((m >> a) & 1)) {
        T* kv = K + sliced_entry(b0, W, slot, 4 * a);
        *kv += (T)v;
      }
  }
}

// One block per row r of the contact list (the rows that the background basis
// of some candidate corner touches; entries (corner, basis entry) in sorted
// order).  RES: R_r -= sum of phi_e f and f_c,r += the same sum, threads strided
// over the entries, each warp's by the fixed shuffle tree, the warps in order.
// TANGENT: K_{r,b} += phi_e phi_b k_c over the basis entries b of each corner
// in contact, the Dirichlet components skipped.  Each warp takes the entries
// 32 at a time in turn, looks which of their corners are in contact (most are
// not) in one step, and adds into its own copy of the row in shared memory, 9
// lanes per column as in the FP64 tangent gather; the copies are added in warp
// order.  No atomics: the same sums on every run.  (A warp per row that walked
// the list entry by entry, a flag and a binary search in memory per corner,
// took 346 us on the punch's 81 k corners; 240 on the cone's.)
template <class T, bool RES, bool TANGENT>
__global__ void __launch_bounds__(128)
    k_contact_rows(int mr, const int* __restrict__ crow, const int* __restrict__ cptr, const int* __restrict__ cent,
                   const int* __restrict__ cb_n, const int* __restrict__ cb_idx, const double* __restrict__ cb_phi,
                   const double* __restrict__ cf, const double* __restrict__ ck, const int* __restrict__ con,
                   double* R, double* fc, const int* __restrict__ rp, const int* __restrict__ col, Sliced S,
                   const int* __restrict__ mask, T* K) {
  extern __shared__ double smc[];
  __shared__ double fs[3][4];
  __shared__ int touched;
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5, nw = blockDim.x >> 5;
  int t = blockIdx.x, r = crow[t], e0 = cptr[t], e1 = cptr[t + 1];
  if (RES) {
    double s0 = 0.0, s1 = 0.0, s2 = 0.0;
    for (int e = e0 + threadIdx.x; e < e1; e += blockDim.x) {
      int pk = cent[e], i = pk >> 5;
      if (!con[i]) continue;  // (no force)
      double ph = cb_phi[(size_t)i * MAXCB + (pk & 31)];
      s0 += ph * cf[3 * (size_t)i];
      s1 += ph * cf[3 * (size_t)i + 1];
      s2 += ph * cf[3 * (size_t)i + 2];
    }
    if (__any_sync(FULL, s0 != 0.0 || s1 != 0.0 || s2 != 0.0)) {
      s0 = warp_sum(s0);
      s1 = warp_sum(s1);
      s2 = warp_sum(s2);
    }
    if (lane < 3) fs[lane][wi] = lane == 0 ? s0 : (lane == 1 ? s1 : s2);
    __syncthreads();
    if (threadIdx.x < 3) {
      double v = 0.0;
      for (int w = 0; w < nw; ++w) v += fs[threadIdx.x][w];
      R[3 * (size_t)r + threadIdx.x] -= v;
      fc[3 * (size_t)r + threadIdx.x] += v;
    }
  }
  if (!TANGENT) return;
  const size_t wsz = 9 * (size_t)mr + 64;
  double* sph = smc + wi * wsz;  // phi_e phi_b of the current entry's columns, then their positions
  int* spo = (int*)(sph + 32);
  double* acc = sph + 64;
  int s0r = rp[r], nb = rp[r + 1] - s0r;
  if (threadIdx.x == 0) touched = 0;
  bool mine = false;
  const int k = lane % 9, cg = lane < 27 ? lane / 9 : 1 << 20;
  for (int base = e0 + 32 * wi; base < e1; base += 32 * nw) {
    int pk0 = base + lane < e1 ? cent[base + lane] : 0;
    unsigned on = __ballot_sync(FULL, base + lane < e1 && con[pk0 >> 5] != 0);
    if (on && !mine) {
      for (int i = lane; i < 9 * nb; i += 32) acc[i] = 0.0;
      mine = true;
    }
    while (on) {
      int pk = __shfl_sync(FULL, pk0, __ffs(on) - 1), i = pk >> 5;
      on &= on - 1;
      int n = cb_n[i];
      double kc = lane < 27 ? ck[9 * (size_t)i + k] : 0.0;
      __syncwarp();
      if (lane < n) {
        spo[lane] = find_slot(rp, col, r, cb_idx[(size_t)i * MAXCB + lane]) - s0r;
        sph[lane] = cb_phi[(size_t)i * MAXCB + (pk & 31)] * cb_phi[(size_t)i * MAXCB + lane];
      }
      __syncwarp();
      for (int c = cg; c < n; c += 3)
        if (spo[c] >= 0) acc[9 * spo[c] + k] += sph[c] * kc;
    }
  }
  // (the copies of the warps that met no corner in contact count as zero)
  __syncthreads();
  if (mine && lane == 0) atomicOr(&touched, 1 << wi);
  __syncthreads();
  int used = touched;
  if (!used) return;
  int ma = mask[r], srr = S.pos[r], slc = srr >> 5, W = S.w[slc];
  long long b0 = S.base[slc];
  for (int i = threadIdx.x; i < nb; i += blockDim.x) {
    int mb = mask[col[s0r + i]];
    long long slot = sliced_slot(b0, srr, i);
    for (int a = 0; a < 3; ++a)
      for (int b = 0; b < 3; ++b) {
        double v = 0.0;
        for (int w = 0; w < nw; ++w)
          if ((used >> w) & 1) v += smc[w * wsz + 64 + 9 * i + 3 * a + b];
        if (v == 0.0 || ((ma >> a) & 1) || ((mb >> b) & 1)) continue;
        T* kv = K + sliced_entry(b0, W, slot, 3 * a + b);
        *kv += (T)v;
      }
  }
}

// ------------------------------------------------------------------ norms

// slots: 0 ||R_free||^2, 1 ||f_int||^2, 2 ||load f_ext + f_c||^2, 3
// ||f_inert||^2 (time steps) (fixed-order grid sums: the norms, and so
// Newton's convergence test and line search, are the same on every run)
__global__ void k_norms(int n3, const double* __restrict__ R, const double* __restrict__ fint,
                        const double* __restrict__ fext, const double* __restrict__ fc, double load,
                        const double* __restrict__ finert, const int* __restrict__ mask, double* out,
                        GridRed gr) {
  double a = 0.0, b = 0.0, c = 0.0, e2 = 0.0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n3; i += gridDim.x * blockDim.x) {
    if (!((mask[i / 3] >> (i % 3)) & 1)) a += R[i] * R[i];
    if (fint) b += fint[i] * fint[i];
    if (fext) {
      double e = load * fext[i] + (fc ? fc[i] : 0.0);
      c += e * e;
    }
    if (finert) e2 += finert[i] * finert[i];
  }
  double v[4] = {a, b, c, e2};
  double* o[4] = {out, out + 1, out + 2, out + 3};
  grid_sum<4>(v, o, gr);
}

}  // namespace


double norm_free(mpm_ctx* c, const mpm_mesh* m, const double* R) {
  double* slot = c->d_red + 16;
  MPM_CUDA(cudaMemsetAsync(slot, 0, 4 * sizeof(double), c->stream));
  MPM_LAUNCH(k_norms<<<grid_strided(3 * m->ndof), 256, 0, c->stream>>>(3 * m->ndof, R, nullptr, nullptr, nullptr, 0.0,
                                          nullptr, ptr<int>(m->dof_mask), slot, grid_red(c, 4, 4 * 152)));
  MPM_CUDA(cudaMemcpyAsync(c->h_red + 16, slot, sizeof(double), cudaMemcpyDeviceToHost, c->stream));
  MPM_CUDA(cudaStreamSynchronize(c->stream));
  return sqrt(c->h_red[16]);
}

namespace {

// the penalty contact of one assembly: per-corner forces and stiffness (and
// the reaction when `reac` is given), then the row gather; with a free body
// (dyn->body) also the body's sums (bsum, device [42]: k_body_sums) and, with
// the tangent, the coupling blocks
template <class T, bool RES, bool TANGENT>
void contact_terms(mpm_ctx* c, mpm_mesh* m, const mpm_material& mat, const mpm_rigid& body,
                   const double* du, double* R, double* fc, double* reac, T* K, const Dyn* dyn,
                   double* bsum) {
  cudaStream_t st = c->stream;
  int n8 = 8 * m->ncand;
  double* cf = grow<double>(c, m->cc_f, 3 * (size_t)n8);
  double* ck = grow<double>(c, m->cc_k, 9 * (size_t)n8);
  int* con = grow<int>(c, m->cc_on, n8);
  bool couple = dyn && dyn->body;
  double* ct = couple ? grow<double>(c, m->cc_t, 9 * (size_t)n8) : nullptr;
  double* cdv = couple ? grow<double>(c, m->cc_d, 3 * (size_t)n8) : nullptr;
  BodyInc bi{};
  for (int d = 0; d < 3; ++d) {
    bi.qt[d] = dyn ? dyn->q[d] : body.step_d[d];
    bi.qr[d] = dyn ? dyn->q[3 + d] : 0.0;
    bi.shift[d] = body.free ? bi.qt[d] : 0.0;
  }
  MPM_LAUNCH_P(MPM_PROF_CONTACT, k_contact_corner<<<grid_for(n8, 128), 128, 0, st>>>(
      n8, ptr<int>(m->cand), ptr<int>(m->cb_n), ptr<int>(m->cb_idx), ptr<double>(m->cb_phi),
      ptr<double>(m->cb_y0), ptr<double>(m->pE), ptr<double>(m->pV0), body_view(m, body), m->g.L,
      mat.pf, mat.pt, mat.mu, bi, du, cf, ck, con, ct, cdv, reac,
      grid_red(c, 3, grid_for(n8, 128))));
  if (couple && bsum)
    MPM_LAUNCH_P(MPM_PROF_CONTACT, k_body_sums<<<1, BSUM_T, 0, st>>>(n8, cf, ck, ct, cdv, con, bsum));
  if (!m->nct) return;
  Sliced S = sliced_view(m);
  // 128 threads per row, fewer where four copies of the longest row do not fit
  size_t wb = TANGENT ? sizeof(double) * (9 * (size_t)m->maxrow + 64) : 0;
  int nw = TANGENT ? (int)std::min<size_t>(4, CSMEM / wb) : 4;
  auto kern = k_contact_rows<T, RES, TANGENT>;
  dynamic_smem(kern, CSMEM);
  MPM_LAUNCH_P(MPM_PROF_CONTACT, kern<<<m->nct, 32 * nw, nw * wb, st>>>(
      m->maxrow, ptr<int>(m->ct_row), ptr<int>(m->ct_ptr), ptr<int>(m->ct_ent), ptr<int>(m->cb_n),
      ptr<int>(m->cb_idx), ptr<double>(m->cb_phi), cf, ck, con, R, fc, ptr<int>(m->row_ptr),
      ptr<int>(m->col), S, ptr<int>(m->dof_mask), K));
  if (TANGENT && couple && dyn->Kgb && dyn->Kbg)
    MPM_LAUNCH_P(MPM_PROF_CONTACT, k_body_rows<<<m->nct, 64, 0, st>>>(
        ptr<int>(m->ct_row), ptr<int>(m->ct_ptr), ptr<int>(m->ct_ent),
        ptr<double>(m->cb_phi), cf, ck, ct, cdv, con, 3LL * m->ndof, dyn->Kgb, dyn->Kbg));
}

}  // namespace

namespace {

// one pass of the tangent gather (rows of lo < length <= hi blocks): rpw rows
// per warp, or wpr warps per row
template <class T, class F>
void tangent_launch(mpm_ctx* c, mpm_mesh* m, F kern, size_t row_bytes, int rpw, int wpr, int pw, int lo, int hi,
                    int last, const void* gx, const void* Aalg, void* K) {
  size_t wb = rpw * row_bytes;
  int tw = (int)std::min<size_t>(TW, TSMEM / wb) / wpr * wpr;
  if (tw < 1) throw CudaError(MPM_ERR_SUPPORT, "stiffness row too long for the tangent gather");
  size_t smem = wb * tw;
  Sliced S = sliced_view(m);
  dynamic_smem(kern, TSMEM);
  MPM_LAUNCH_P(MPM_PROF_TANGENT, kern<<<grid_for(m->ndof, tw / wpr * rpw), 32 * tw, smem, c->stream>>>(
      m->ndof, m->np, pw, lo, hi, last, ptr<int>(m->row_ptr), ptr<int>(m->col), S, ptr<long long>(m->src_ptr),
      ptr<uint64_t>(m->src_key), ptr<unsigned short>(m->src_pos), (const T*)gx, (const T*)Aalg, ptr<double>(m->kg),
      ptr<int>(m->dof_mask), (T*)K, c->d_err));
}

// two passes: rows up to 128 blocks (the 5^3 interior stencil and below) with
// a small shared-memory footprint per row, for occupancy, then the longer rows
// near hanging nodes, which are few and have many sources.  The block's four
// warps share a row there, and everywhere on meshes of few rows, where a
// row's serial chain of sources is the time: below 20,000 rows a warp per row
// leaves most of the 152 x 24 resident warps idle (the cone at 2.4 k rows:
// 0.68 -> 0.16 ms).
void tangent_passes(mpm_ctx* c, mpm_mesh* m, bool mixed, bool upper, int pw, const void* gx, const void* Aalg,
                    void* K) {
  const int SHORT = 128;
  int mr = (m->maxrow + 3) & ~3;
  int passes[2][2] = {{-1, std::min(mr, SHORT)}, {SHORT, mr}};
  int np_ = mr > SHORT ? 2 : 1;
  for (int ps = 0; ps < np_; ++ps) {
    int lo = passes[ps][0], hi = passes[ps][1], last = ps == np_ - 1;
    size_t rb = mixed ? tangent_row_bytes_f32(hi) : tangent_warp_bytes_f64(hi);
    bool share = (ps > 0 || m->ndof < TANGENT_FEW_ROWS) && 4 * rb <= TSMEM;
    if (mixed) {
      // (four FP32 copies of the longest row fit: every long row is shared)
      static_assert(4 * tangent_row_bytes_f32(MAXROW) <= TSMEM, "long rows of the FP32 tangent");
      if (share)
        tangent_launch<float>(c, m, k_tangent_rows_f32<32, 4>, rb, 1, 4, pw, lo, hi, last, gx, Aalg, K);
      else
        tangent_launch<float>(c, m, k_tangent_rows_f32<16, 1>, rb, 2, 1, pw, lo, hi, last, gx, Aalg, K);
    } else {
      auto kern = upper ? (share ? k_tangent_rows_f64<true, 4> : k_tangent_rows_f64<true, 1>)
                        : (share ? k_tangent_rows_f64<false, 4> : k_tangent_rows_f64<false, 1>);
      tangent_launch<double>(c, m, kern, rb, 1, share ? 4 : 1, pw, lo, hi, last, gx, Aalg, K);
    }
  }
}

}  // namespace

namespace {

// the free body's equations on the host from the contact sums (bsum, device
// [42]): Rb = m (2 / dt^2) (qt - dt v) - m load g + sum f,
// J (2 / dt^2) (qr - dt w) + sum d x f, and (with the tangent) Kbb = the
// sums' derivative plus the inertia's m (2 / dt^2) I, J (2 / dt^2) I
void body_out(mpm_ctx* c, const mpm_material& mat, const mpm_rigid& body, double load, const Dyn* dyn,
              const double* bsum, AsmOut* out, bool tangent) {
  double h[42];
  MPM_CUDA(cudaMemcpyAsync(h, bsum, sizeof(h), cudaMemcpyDeviceToHost, c->stream));
  MPM_CUDA(cudaStreamSynchronize(c->stream));
  double dt = dyn->dt, c2 = dt > 0.0 ? 2.0 / (dt * dt) : 0.0;
  for (int d = 0; d < 3; ++d) {
    out->Rb[d] = h[d];
    out->Rb[3 + d] = h[3 + d];
    if (dt > 0.0) {
      out->Rb[d] += body.mass * (c2 * (dyn->q[d] - dt * body.v[d]) - load * mat.g[d]);
      out->Rb[3 + d] += body.inertia * c2 * (dyn->q[3 + d] - dt * body.w[d]);
    }
  }
  if (!tangent) return;
  for (int e = 0; e < 36; ++e) out->Kbb[e] = h[6 + e];
  if (dt > 0.0)
    for (int d = 0; d < 3; ++d) {
      out->Kbb[7 * d] += body.mass * c2;
      out->Kbb[7 * (3 + d)] += body.inertia * c2;
    }
}

}  // namespace

void assemble(mpm_ctx* c, const mpm_mesh* mc, const mpm_material& mat, const mpm_rigid& body,
              const double* du, double load, int precision, double* R, void* K, AsmOut* out,
              bool want_norms, bool reuse, const Dyn* dyn, bool save_state) {
  mpm_mesh* m = const_cast<mpm_mesh*>(mc);
  cudaStream_t st = c->stream;
  int P = m->np, nd = m->ndof;
  Law L = make_law(mat);
  double* dF = grow<double>(c, m->dF, 9 * (size_t)P);
  double* dFinv = grow<double>(c, m->dFinv, 9 * (size_t)P);
  double* tau = grow<double>(c, m->tau, 6 * (size_t)P);
  double* lawst = save_state || reuse ? grow<double>(c, m->lawst, 22 * (size_t)P) : nullptr;
  double* Mf = grow<double>(c, m->Mf, 12 * (size_t)P);
  const int* nsup = ptr<int>(m->nsup);
  const int* sidx = ptr<int>(m->sidx);
  const double* dS = ptr<double>(m->dS);
  const double* V0 = ptr<double>(m->pV0);
  const int* rp = ptr<int>(m->row_ptr);
  const int* col = ptr<int>(m->col);
  Sliced S = sliced_view(m);
  bool mixed = precision == MPM_MIXED;
  size_t asz = mixed ? sizeof(float) : sizeof(double);
  int pw = (std::max(m->maxs, 1) + 3) & ~3;  // support nodes stored per point by the gather's arrays
  void* Aalg = K ? grow_bytes(c, m->Aalg, 108 * (size_t)P * asz) : nullptr;
  void* gx = K ? grow_bytes(c, m->gx, 4 * (size_t)P * pw * asz) : nullptr;
  if (K && m->src_pos_gen != m->gen) {
    int hs = tangent_hash_size(m->maxrow);
    unsigned short* sp = grow<unsigned short>(c, m->src_pos, (size_t)m->nsrc_used * pw);
    bool few = nd < TANGENT_FEW_ROWS;
    size_t smem = (few ? 1 : 4) * 2 * sizeof(int) * (size_t)hs;
    auto kern = few ? k_src_pos<true> : k_src_pos<false>;
    dynamic_smem(kern, 4 * 2 * (int)sizeof(int) * tangent_hash_size(MAXROW));
    MPM_LAUNCH_P(MPM_PROF_PATTERN, kern<<<grid_for(nd, few ? 1 : 4), 128, smem, st>>>(
        nd, P, pw, hs, rp, col, ptr<long long>(m->src_ptr), ptr<uint64_t>(m->src_key), nsup, sidx, sp));
    m->src_pos_gen = m->gen;
  }
  const float* dS32 = nullptr;
  if (K && mixed) {
    float* d32 = grow<float>(c, m->dS32, 3 * (size_t)P * MAXS);
    if (m->dS32_gen != m->gen) {
      MPM_LAUNCH_P(MPM_PROF_FORCE, k_dS_to_float<<<grid_for(3LL * MAXS * P, 256), 256, 0, st>>>(P, nsup, dS, d32));
      m->dS32_gen = m->gen;
    }
    dS32 = d32;
  }
  double* fint = grow<double>(c, c->v[0], 3 * (size_t)nd);
  double* fc = grow<double>(c, c->v[1], 3 * (size_t)nd);
  bool contact = m->ncand && mat.contact_on && body.kind != 0;
  bool inertia = dyn && dyn->dt > 0.0;
  if (inertia && !m->has_v) throw CudaError(MPM_ERR_ARG, "a time step needs point velocities");
  double* finert = inertia ? grow<double>(c, c->v[2], 3 * (size_t)nd) : nullptr;
  bool couple = dyn && dyn->body;
  double* bsum = couple ? grow<double>(c, m->cc_b, 42) : nullptr;
  if (couple) MPM_CUDA(cudaMemsetAsync(bsum, 0, 42 * sizeof(double), st));
  if (couple && K && dyn->Kgb && dyn->Kbg) {
    MPM_CUDA(cudaMemsetAsync(dyn->Kgb, 0, sizeof(double) * 18 * (size_t)nd, st));
    MPM_CUDA(cudaMemsetAsync(dyn->Kbg, 0, sizeof(double) * 18 * (size_t)nd, st));
  }
  // grid-sum partials for every reduction below, sized once; a clean ticket,
  // norms and reaction (slots 14 to 22)
  grid_red(c, 4, std::max(4096, grid_for(8LL * m->ncand, 128)));
  MPM_CUDA(cudaMemsetAsync(c->d_red + 14, 0, 9 * sizeof(double), st));
  if (out) out->clean = false;
  if (K && reuse) {
    // Newton's tangent at the increment of the last residual evaluation: its
    // dF, dF^-1, tau and spectral state are still in place, R is complete
    if (mixed) {
      MPM_LAUNCH_P(MPM_PROF_CONSTITUTIVE, k_tangent_state<float><<<grid_for(P, 128), 128, 0, st>>>(P, lawst, tau, V0, (float*)Aalg));
      MPM_LAUNCH_P(MPM_PROF_FORCE, k_gx<float, float><<<grid_for(8LL * P, 256), 256, 0, st>>>(P, pw, nsup, dS32, dFinv, (float*)gx));
    } else {
      MPM_LAUNCH_P(MPM_PROF_CONSTITUTIVE, k_tangent_state<double><<<grid_for(P, 128), 128, 0, st>>>(P, lawst, tau, V0, (double*)Aalg));
      MPM_LAUNCH_P(MPM_PROF_FORCE, k_gx<double, double><<<grid_for(8LL * P, 256), 256, 0, st>>>(P, pw, nsup, dS, dFinv, (double*)gx));
    }
  } else {
    MPM_LAUNCH_P(MPM_PROF_KINEMATICS, k_kinematics<<<grid_for(P, KIN_P), KIN_T, 0, st>>>(P, nsup, sidx, dS, du, dF));
    if (!K) {
      auto kern = save_state ? k_constitutive<false, double, true> : k_constitutive<false, double, false>;
      MPM_LAUNCH_P(MPM_PROF_CONSTITUTIVE, kern<<<grid_for(P, 128), 128, 0, st>>>(
          P, L, ptr<double>(m->pE), ptr<double>(m->pys), ptr<double>(m->pbe), dF, V0, tau, dFinv, Mf,
          nullptr, lawst, c->d_err));
    }
    else if (mixed)
      MPM_LAUNCH_P(MPM_PROF_CONSTITUTIVE, (k_constitutive<true, float, false><<<grid_for(P, 128), 128, 0, st>>>(
          P, L, ptr<double>(m->pE), ptr<double>(m->pys), ptr<double>(m->pbe), dF, V0, tau, dFinv, Mf,
          (float*)Aalg, nullptr, c->d_err)));
    else
      MPM_LAUNCH_P(MPM_PROF_CONSTITUTIVE, (k_constitutive<true, double, false><<<grid_for(P, 128), 128, 0, st>>>(
          P, L, ptr<double>(m->pE), ptr<double>(m->pys), ptr<double>(m->pbe), dF, V0, tau, dFinv, Mf,
          (double*)Aalg, nullptr, c->d_err)));
    if (contact) MPM_CUDA(cudaMemsetAsync(fc, 0, sizeof(double) * 3 * nd, st));
    MPM_LAUNCH_P(MPM_PROF_RESIDUAL, k_residual_rows<<<grid_for(nd, 8), 256, 0, st>>>(
        nd, P, load, ptr<long long>(m->src_ptr), ptr<uint64_t>(m->src_key), Mf, dS, rp, col,
        ptr<double>(m->kg), du, ptr<double>(m->fext), fint, R));
    if (inertia) {
      double* ma = grow<double>(c, m->pma, 3 * (size_t)P);
      MPM_LAUNCH_P(MPM_PROF_RESIDUAL, k_point_inertia<<<grid_for(P, 128), 128, 0, st>>>(
          P, nsup, sidx, ptr<double>(m->S), du, ptr<double>(m->pv), ptr<double>(m->pmass), dyn->dt, ma));
      MPM_LAUNCH_P(MPM_PROF_RESIDUAL, k_inertia_rows<<<grid_for(nd, 8), 256, 0, st>>>(
          nd, P, ptr<long long>(m->src_ptr), ptr<uint64_t>(m->src_key), ptr<double>(m->S), ma, R, finert));
    }
    if (K) {
      if (mixed)
        MPM_LAUNCH_P(MPM_PROF_FORCE, k_gx<float, float><<<grid_for(8LL * P, 256), 256, 0, st>>>(P, pw, nsup, dS32, dFinv, (float*)gx));
      else
        MPM_LAUNCH_P(MPM_PROF_FORCE, k_gx<double, double><<<grid_for(8LL * P, 256), 256, 0, st>>>(P, pw, nsup, dS, dFinv, (double*)gx));
    }
  }
  if (K) {
    // a symmetric FP64 tangent forms only its upper blocks and mirrors them:
    // its pairs are bound by the FP64 FMA rate, which the halving pays for; the
    // FP32 gather is bound by its shared-memory traffic, and the mirror pass
    // would cost more than the halved pairs save
    bool upper = !mixed && (mat.model == 0 || mat.model == 1) && !(mat.mu > 0.0 && contact);
    tangent_passes(c, m, mixed, upper, pw, gx, Aalg, K);
    if (upper)
      MPM_LAUNCH_P(MPM_PROF_TANGENT, k_tangent_mirror<<<grid_for(32LL * nd, 256), 256, 0, st>>>(nd, rp, col, S, (double*)K));
    if (inertia) {
      double c2 = 2.0 / (dyn->dt * dyn->dt);
      size_t smem = 4 * sizeof(double) * (size_t)m->maxrow;
      auto launch = [&](auto kern, auto* Kt) {
        MPM_LAUNCH_P(MPM_PROF_TANGENT, kern<<<nd, 128, smem, st>>>(
            P, pw, m->maxrow, ptr<long long>(m->src_ptr), ptr<uint64_t>(m->src_key),
            ptr<unsigned short>(m->src_pos), ptr<double>(m->S), ptr<double>(m->pmass), c2, rp, col, S,
            ptr<int>(m->dof_mask), Kt));
      };
      if (mixed)
        launch(k_mass_rows<float>, (float*)K);
      else
        launch(k_mass_rows<double>, (double*)K);
    }
    int npad = 32 * m->nslice;
    if (npad > nd) {
      if (mixed)
        MPM_LAUNCH(k_zero_pad_rows<float><<<grid_for(32LL * (npad - nd), 256), 256, 0, st>>>(nd, npad, S, (float*)K));
      else
        MPM_LAUNCH(k_zero_pad_rows<double><<<grid_for(32LL * (npad - nd), 256), 256, 0, st>>>(nd, npad, S, (double*)K));
    }
  }
  double* reac = c->d_red + 20;
  if (K && reuse) {
    // contact stiffness only: its forces are already in R
    if (contact) {
      if (mixed)
        contact_terms<float, false, true>(c, m, mat, body, du, R, fc, nullptr, (float*)K, dyn, bsum);
      else
        contact_terms<double, false, true>(c, m, mat, body, du, R, fc, nullptr, (double*)K, dyn, bsum);
    }
    if (couple) body_out(c, mat, body, load, dyn, bsum, out, true);
    return;
  }
  if (contact) {
    if (!K)
      contact_terms<double, true, false>(c, m, mat, body, du, R, fc, reac, (double*)nullptr, dyn, bsum);
    else if (mixed)
      contact_terms<float, true, true>(c, m, mat, body, du, R, fc, reac, (float*)K, dyn, bsum);
    else
      contact_terms<double, true, true>(c, m, mat, body, du, R, fc, reac, (double*)K, dyn, bsum);
  }
  if (want_norms) {
    double* slot = c->d_red + 16;
    MPM_LAUNCH(k_norms<<<grid_strided(3 * nd), 256, 0, st>>>(3 * nd, R, fint, ptr<double>(m->fext), contact ? fc : nullptr, load, finert,
                                     ptr<int>(m->dof_mask), slot, grid_red(c, 4, 4 * 152)));
    MPM_CUDA(cudaMemcpyAsync(c->h_red + 16, slot, 8 * sizeof(double), cudaMemcpyDeviceToHost, st));
    MPM_CUDA(cudaStreamSynchronize(st));
    out->clean = *(const int*)(c->h_red + 23) == 0;
    out->fint_norm = sqrt(c->h_red[17]);
    out->fextc_norm = sqrt(c->h_red[18]);
    out->finert_norm = sqrt(c->h_red[19]);
    for (int d = 0; d < 3; ++d) out->reaction[d] = c->h_red[20 + d];
  }
  if (couple) body_out(c, mat, body, load, dyn, bsum, out, K != nullptr);
}

void blocks_export(mpm_ctx* c, const mpm_mesh* m, const void* K, int precision, double* out) {
  Sliced S = sliced_view(m);
  int nd = m->ndof;
  if (precision == MPM_MIXED)
    MPM_LAUNCH(k_blocks_export<float><<<grid_for(32LL * nd, 256), 256, 0, c->stream>>>(nd, ptr<int>(m->row_ptr), S, (const float*)K, out));
  else
    MPM_LAUNCH(k_blocks_export<double><<<grid_for(32LL * nd, 256), 256, 0, c->stream>>>(nd, ptr<int>(m->row_ptr), S, (const double*)K, out));
}

// ------------------------------------------------------------------ point update helpers (used by mpm_step.cu)

namespace {

// end-of-step update, one thread per (sorted) point: x += sum S du, F <- dF F,
// b_e from the converged return, l = l0 diag(U), U = sqrt(F^T F)
__global__ void k_point_update(int P, Law L, const int* __restrict__ perm,
                               const int* __restrict__ nsup, const int* __restrict__ sidx,
                               const double* __restrict__ S, const double* __restrict__ dS,
                               const double* __restrict__ du, const double* __restrict__ pE,
                               const double* __restrict__ pys, const double* __restrict__ pbe,
                               const double* __restrict__ pF, const double* __restrict__ px,
                               const double* __restrict__ pl0, const double* __restrict__ pv,
                               double dt, mpm_points pts, int* err) {
  int w = blockIdx.x * blockDim.x + threadIdx.x;
  if (w >= P) return;
  double dF[9] = {1, 0, 0, 0, 1, 0, 0, 0, 1}, dx[3] = {0, 0, 0};
  int n = nsup[w];
  for (int k = 0; k < n; ++k) {
    size_t o = (size_t)w * MAXS + k;
    int j = sidx[o];
    double u[3] = {du[3 * (size_t)j], du[3 * (size_t)j + 1], du[3 * (size_t)j + 2]};
    for (int i = 0; i < 3; ++i) {
      dx[i] += S[o] * u[i];
      for (int jj = 0; jj < 3; ++jj) dF[3 * i + jj] += u[i] * dS[3 * o + jj];
    }
  }
  double t6[6], bn[6];
  if (!point_update_law<false, double>(L, pE[w], pys[w], pbe + 6 * (size_t)w, dF, t6, bn, 0.0, nullptr)) {
    atomicOr(err, EB_NAN);
    return;
  }
  const double* Fo = pF + 9 * (size_t)w;
  double Fn[9];
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j)
      Fn[3 * i + j] = dF[3 * i] * Fo[j] + dF[3 * i + 1] * Fo[3 + j] + dF[3 * i + 2] * Fo[6 + j];
  double C[9];
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j)
      C[3 * i + j] = Fn[i] * Fn[j] + Fn[3 + i] * Fn[3 + j] + Fn[6 + i] * Fn[6 + j];
  double lam[3], Q[9];
  jacobi3(C, lam, Q);
  size_t p = perm[w];
  for (int d = 0; d < 3; ++d) {
    double u = 0.0;
    for (int a = 0; a < 3; ++a) u += sqrt(lam[a]) * Q[3 * d + a] * Q[3 * d + a];
    pts.x[3 * p + d] = px[3 * (size_t)w + d] + dx[d];
    pts.lp[3 * p + d] = pl0[3 * (size_t)w + d] * u;
    // a time step's velocity: v + dt a, a = (2 / dt^2) (du_p - dt v)
    if (dt > 0.0) {
      double v = pv[3 * (size_t)w + d];
      pts.v[3 * p + d] = v + dt * ((2.0 / (dt * dt)) * (dx[d] - dt * v));
    }
  }
  for (int i = 0; i < 9; ++i) pts.F[9 * p + i] = Fn[i];
  for (int s = 0; s < 6; ++s) pts.be[6 * p + s] = bn[s];
}

}  // namespace

void point_update(mpm_ctx* c, const mpm_mesh* mc, const mpm_material& mat, const double* du,
                  mpm_points* pts, double dt) {
  mpm_mesh* m = const_cast<mpm_mesh*>(mc);
  int P = m->np;
  if (dt > 0.0 && !(m->has_v && pts->v)) throw CudaError(MPM_ERR_ARG, "a time step needs point velocities");
  MPM_LAUNCH(k_point_update<<<grid_for(P, 128), 128, 0, c->stream>>>(
      P, make_law(mat), ptr<int>(m->perm), ptr<int>(m->nsup), ptr<int>(m->sidx), ptr<double>(m->S),
      ptr<double>(m->dS), du, ptr<double>(m->pE), ptr<double>(m->pys), ptr<double>(m->pbe),
      ptr<double>(m->pF), ptr<double>(m->px), ptr<double>(m->pl0), dt > 0.0 ? ptr<double>(m->pv) : nullptr,
      dt, *pts, c->d_err));
}

}  // namespace mpm
