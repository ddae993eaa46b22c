// Once-per-load-step mesh build: octree adaptivity and 2:1 balance (Sec. 5),
// nodes, hanging classification and constraints (Sec. 3.1), GIMP refinement
// (Sec. 5), the discrete GIMP basis (Sec. 3.2, Eq. GIMP numerical), ghost
// faces and the ghost matrix (Sec. 4), the 3x3 block pattern, the gravity
// force and the contact candidates.  Compiled with --fmad=false so that the
// box and grid arithmetic that decides discrete events rounds like the plain
// IEEE expressions of the method.
#include <algorithm>
#include <vector>

#include "mpm_internal.cuh"

namespace mpm {
namespace {

// ------------------------------------------------------------------ octree

__global__ void k_tree_uniform(int n, int shift, int lev, uint64_t* key, int* levs) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  key[i] = (uint64_t)i << shift;
  levs[i] = lev;
}

// Sec. 5, Steps 1-2: mark leaves meeting the body or with a corner within dx_region
__global__ void k_mark_refine(int n, const uint64_t* __restrict__ key, const int* __restrict__ lev,
                              Geo g, Body b, double dxr, int dmax, int* flag, int* any) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  int f = 0;
  if (lev[i] < dmax) {
    int a[3];
    demorton(key[i], a);
    int s = 1 << (g.D - lev[i]);
    double lo[3], hi[3];
    for (int d = 0; d < 3; ++d) {
      lo[d] = (double)a[d] * g.unit;
      hi[d] = (double)(a[d] + s) * g.unit;
    }
    if (body_meets_box(b, lo, hi)) {
      f = 1;
    } else {
      for (int c = 0; c < 8 && !f; ++c) {
        double xc[3] = {(c & 1) ? hi[0] : lo[0], (c & 2) ? hi[1] : lo[1], (c & 4) ? hi[2] : lo[2]};
        if (body_distance(b, xc, dxr) <= dxr) f = 1;
      }
    }
  }
  flag[i] = f;
  if (f) *any = 1;
}

__global__ void k_child_count(int n, const int* flag, int* cnt) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) cnt[i] = flag[i] ? 8 : 1;
}

// children of a leaf are contiguous in Morton order: the sorted order survives
__global__ void k_refine_write(int n, const uint64_t* __restrict__ key, const int* __restrict__ lev,
                               const int* __restrict__ flag, const int* __restrict__ pos, int D,
                               uint64_t* okey, int* olev) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  int p = pos[i];
  if (flag[i]) {
    int sh = 3 * (D - lev[i] - 1);
    for (int c = 0; c < 8; ++c) {
      okey[p + c] = key[i] + ((uint64_t)c << sh);
      olev[p + c] = lev[i] + 1;
    }
  } else {
    okey[p] = key[i];
    olev[p] = lev[i];
  }
}

// 2:1 balance across faces and edges (Sec. 5: one hanging node per edge/face)
__global__ void k_balance_mark(int n, const uint64_t* __restrict__ key, const int* __restrict__ lev,
                               Geo g, int* flag, int* any) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  int a[3];
  demorton(key[i], a);
  int s = 1 << (g.D - lev[i]);
  for (int dz = -1; dz <= 1; ++dz)
    for (int dy = -1; dy <= 1; ++dy)
      for (int dx = -1; dx <= 1; ++dx) {
        int nz = (dx != 0) + (dy != 0) + (dz != 0);
        if (nz == 0 || nz == 3) continue;
        int dd[3] = {dx, dy, dz}, q[3];
        bool ok = true;
        for (int d = 0; d < 3; ++d) {
          q[d] = dd[d] == 1 ? a[d] + s : (dd[d] == -1 ? a[d] - 1 : a[d]);
          ok = ok && q[d] >= 0 && q[d] < g.N;
        }
        if (!ok) continue;
        int nb = locate(key, n, q[0], q[1], q[2]);
        if (lev[nb] < lev[i] - 1) {
          flag[nb] = 1;
          *any = 1;
        }
      }
}

// ------------------------------------------------------------------ nodes

__global__ void k_corner_keys(int n, const uint64_t* __restrict__ key, const int* __restrict__ lev,
                              int D, uint64_t* ck) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  int a[3];
  demorton(key[i], a);
  int s = 1 << (D - lev[i]);
  for (int c = 0; c < 8; ++c)
    ck[8 * (size_t)i + c] = morton(a[0] + (c & 1) * s, a[1] + ((c >> 1) & 1) * s, a[2] + ((c >> 2) & 1) * s);
}

__device__ inline int find_exact(const uint64_t* __restrict__ key, int n, uint64_t k) {
  int lo = 0, hi = n - 1;
  while (lo <= hi) {
    int mid = (lo + hi) >> 1;
    uint64_t v = key[mid];
    if (v == k) return mid;
    if (v < k)
      lo = mid + 1;
    else
      hi = mid - 1;
  }
  return -1;
}

__global__ void k_corner_ids(int n, const uint64_t* __restrict__ key, const int* __restrict__ lev,
                             int D, const uint64_t* __restrict__ nkey, int nn, int* corner) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  int a[3];
  demorton(key[i], a);
  int s = 1 << (D - lev[i]);
  for (int c = 0; c < 8; ++c)
    corner[8 * (size_t)i + c] = find_exact(
        nkey, nn, morton(a[0] + (c & 1) * s, a[1] + ((c >> 1) & 1) * s, a[2] + ((c >> 2) & 1) * s));
}

// Sec. 3.1: n hangs when it lies on the boundary of a leaf without being one of
// its vertices; K_n is the largest such leaf (ties: lowest Morton key)
__global__ void k_hang(int nn, const uint64_t* __restrict__ nkey, const uint64_t* __restrict__ lkey,
                       const int* __restrict__ llev, int nl, Geo g, int* hang, int* owner,
                       int* nhang) {
  int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= nn) return;
  int X[3];
  demorton(nkey[n], X);
  int best = -1;
  for (int sc = 0; sc < 8; ++sc) {
    int q[3];
    bool ok = true;
    for (int d = 0; d < 3; ++d) {
      q[d] = X[d] - 1 + ((sc >> d) & 1);
      ok = ok && q[d] >= 0 && q[d] < g.N;
    }
    if (!ok) continue;
    int K = locate(lkey, nl, q[0], q[1], q[2]);
    int s = 1 << (g.D - llev[K]);
    int a[3];
    demorton(lkey[K], a);
    bool corner = true;
    for (int d = 0; d < 3; ++d) {
      int r = X[d] - a[d];
      corner = corner && (r == 0 || r == s);
    }
    if (corner) continue;
    if (best < 0 || llev[K] < llev[best] || (llev[K] == llev[best] && lkey[K] < lkey[best])) best = K;
  }
  hang[n] = best >= 0 ? 1 : 0;
  owner[n] = best;
  unsigned on = __activemask(), hs = __ballot_sync(on, best >= 0);
  if (hs && (threadIdx.x & 31) == __ffs(on) - 1) atomicAdd(nhang, __popc(hs));
}

struct NodeView {
  const uint64_t* nkey;
  const uint64_t* lkey;
  const int* llev;
  const int* corner;
  const int* hang;
  const int* owner;
  int D;
};

// Eq. (constraint equation reduced): weights phi_{i,K_n}(x_n) of the owner's corners
__device__ int direct_constraint(const NodeView& v, int h, int* ids, double* ws) {
  int K = v.owner[h];
  int s = 1 << (v.D - v.llev[K]);
  int a[3], X[3];
  demorton(v.lkey[K], a);
  demorton(v.nkey[h], X);
  double xi[3];
  for (int d = 0; d < 3; ++d) {
    int t = 2 * (X[d] - a[d]);
    if (t != 0 && t != s && t != 2 * s) return -1;
    xi[d] = (double)t / (2.0 * s);
  }
  int cnt = 0;
  for (int c = 0; c < 8; ++c) {
    double w = 1.0;
    for (int d = 0; d < 3; ++d) w *= ((c >> d) & 1) ? xi[d] : 1.0 - xi[d];
    if (w != 0.0) {
      ids[cnt] = v.corner[8 * (size_t)K + c];
      ws[cnt] = w;
      ++cnt;
    }
  }
  return cnt;
}

// transitive substitution of hanging supports; returns the count or -1
__device__ int resolve_node(const NodeView& v, int n, int* ids, double* ws) {
  int cnt = 1;
  ids[0] = n;
  ws[0] = 1.0;
  for (int round = 0; round < 128; ++round) {
    int i = -1;
    for (int k = 0; k < cnt; ++k)
      if (v.hang[ids[k]]) {
        i = k;
        break;
      }
    if (i < 0) {
      for (int a = 1; a < cnt; ++a)
        for (int b = a; b > 0 && ids[b - 1] > ids[b]; --b) {
          int t = ids[b]; ids[b] = ids[b - 1]; ids[b - 1] = t;
          double tw = ws[b]; ws[b] = ws[b - 1]; ws[b - 1] = tw;
        }
      return cnt;
    }
    int h = ids[i];
    double wh = ws[i];
    ids[i] = ids[cnt - 1];
    ws[i] = ws[cnt - 1];
    --cnt;
    int dids[8];
    double dws[8];
    int nd = direct_constraint(v, h, dids, dws);
    if (nd < 0) return -2;
    for (int k = 0; k < nd; ++k) {
      int slot = -1;
      for (int q = 0; q < cnt; ++q)
        if (ids[q] == dids[k]) slot = q;
      if (slot >= 0) {
        ws[slot] += wh * dws[k];
      } else {
        if (cnt >= MAXC) return -1;
        ids[cnt] = dids[k];
        ws[cnt] = wh * dws[k];
        ++cnt;
      }
    }
  }
  return -2;
}

__global__ void k_con_count(int nn, NodeView v, int* cnt, int* err) {
  int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= nn) return;
  int ids[MAXC];
  double ws[MAXC];
  int c = resolve_node(v, n, ids, ws);
  if (c < 0) {
    atomicOr(err, c == -1 ? EB_SUPPORT : EB_BALANCE);
    c = 0;
  }
  cnt[n] = c;
}

__global__ void k_con_fill(int nn, NodeView v, const int* __restrict__ cptr, int* cidx, double* cw) {
  int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= nn) return;
  int ids[MAXC];
  double ws[MAXC];
  int c = resolve_node(v, n, ids, ws);
  int b = cptr[n], e = cptr[n + 1];
  for (int k = 0; k < c && b + k < e; ++k) {
    cidx[b + k] = ids[k];
    cw[b + k] = ws[k];
  }
}

// ------------------------------------------------------------------ GIMP domains and split

// GIMP domain in finest-grid units: bounds snapped, clipped; returns V_p (unclipped)
__device__ inline double domain_box(const double* x, const double* l, const Geo& g, double* Lo,
                                    double* Hi) {
  double V = 1.0, N = (double)g.N;
  for (int d = 0; d < 3; ++d) {
    double lo = snap_grid((x[d] - l[d]) * g.scale);
    double hi = snap_grid((x[d] + l[d]) * g.scale);
    V *= hi - lo;
    Lo[d] = lo < 0.0 ? 0.0 : lo;
    Hi[d] = hi > N ? N : hi;
  }
  return V;
}

// Sec. 5: split if some overlapped leaf has l_K < beta l_p (l_p: largest reference
// half-length); the leaf-by-leaf cutting stops at the first such leaf, and a
// work list overflow counts as a split
__global__ void k_split_flag(int P, const double* __restrict__ x, const double* __restrict__ lp,
                             const double* __restrict__ l0, const uint64_t* __restrict__ lkey,
                             const int* __restrict__ llev, int nl, Geo g, double beta, int* flag,
                             int* err) {
  int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= P) return;
  double Lo[3], Hi[3];
  domain_box(x + 3 * (size_t)p, lp + 3 * (size_t)p, g, Lo, Hi);
  if (!(Hi[0] > Lo[0]) || !(Hi[1] > Lo[1]) || !(Hi[2] > Lo[2])) {
    atomicOr(err, EB_DOMAIN);
    flag[p] = 0;
    return;
  }
  double lm = l0[3 * (size_t)p];
  if (l0[3 * (size_t)p + 1] > lm) lm = l0[3 * (size_t)p + 1];
  if (l0[3 * (size_t)p + 2] > lm) lm = l0[3 * (size_t)p + 2];
  double lim = beta * lm * g.scale;
  // 0.5 s < lim for a leaf of s grid units: s below the next integer of 2 lim
  int slim = 2.0 * lim < 1e9 ? (int)ceil(2.0 * lim) : 0x7fffffff;
  if (!(lim > 0.0)) slim = 0;
  // the walk in integers (as the basis kernel's): FP64 on this part is slow, and
  // the work list half as long (0.55 -> 0.34 ms at 1.9 M points)
  DomainCells dc;
  for (int d = 0; d < 3; ++d) {
    double fh = floor(Hi[d]);
    dc.lo[d] = (int)floor(Lo[d]);
    dc.hi[d] = (int)fh;
    dc.whole[d] = Hi[d] == fh;
  }
  int st[SPLIT_STACK][6];
  int ns = 1;
  for (int d = 0; d < 6; ++d) st[0][d] = -1;
  int f = 0;
  while (ns > 0) {
    --ns;
    int a[3], b[3];
    for (int d = 0; d < 3; ++d) {
      a[d] = st[ns][d];
      b[d] = st[ns][3 + d];
    }
    LeafCut l;
    l.cut(g, lkey, llev, nl, dc, a, b);
    if (l.s < slim || ns + 3 > SPLIT_STACK) {
      f = 1;
      break;
    }
    for (int d = 0; d < 3; ++d)
      if (l.gt[d]) l.child(d, a, b, st[ns++]);
  }
  flag[p] = f;
}

// children: child 0 keeps the parent slot, children 1..7 go to P + 7 rank + c - 1
__global__ void k_split_write(int P, const int* __restrict__ flag, const int* __restrict__ rank,
                              mpm_points pts) {
  int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= P || !flag[p]) return;
  double xc[3], lc[3], l0c[3];
  for (int d = 0; d < 3; ++d) {
    xc[d] = pts.x[3 * (size_t)p + d];
    lc[d] = pts.lp[3 * (size_t)p + d];
    l0c[d] = pts.l0[3 * (size_t)p + d];
  }
  for (int c = 0; c < 8; ++c) {
    size_t q = c == 0 ? (size_t)p : (size_t)P + 7 * (size_t)rank[p] + (c - 1);
    for (int d = 0; d < 3; ++d) {
      double sg = ((c >> d) & 1) ? 0.5 : -0.5;
      pts.x[3 * q + d] = xc[d] + sg * lc[d];
      pts.lp[3 * q + d] = 0.5 * lc[d];
      pts.l0[3 * q + d] = 0.5 * l0c[d];
    }
    if (c) {
      for (int i = 0; i < 9; ++i) pts.F[9 * q + i] = pts.F[9 * (size_t)p + i];
      for (int i = 0; i < 6; ++i) pts.be[6 * q + i] = pts.be[6 * (size_t)p + i];
      pts.V0[q] = pts.V0[p] / 8.0;
      pts.mass[q] = pts.mass[p] / 8.0;
      pts.E[q] = pts.E[p];
      pts.ys[q] = pts.ys[p];
      if (pts.v)
        for (int d = 0; d < 3; ++d) pts.v[3 * q + d] = pts.v[3 * (size_t)p + d];
    }
  }
  pts.V0[p] /= 8.0;
  pts.mass[p] /= 8.0;
}

// ------------------------------------------------------------------ cell sort

__global__ void k_point_cell(int P, const double* __restrict__ x, Geo g,
                             const uint64_t* __restrict__ lkey, int nl, int* cell, int* idx) {
  int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= P) return;
  int q[3];
  for (int d = 0; d < 3; ++d) {
    double v = floor(x[3 * (size_t)p + d] * g.scale);
    q[d] = v < 0 ? 0 : (v > g.N - 1 ? g.N - 1 : (int)v);
  }
  cell[p] = locate(lkey, nl, q[0], q[1], q[2]);
  idx[p] = p;
}

__global__ void k_gather_points(int P, const int* __restrict__ perm, mpm_points pts, double* x,
                                double* lp, double* l0, double* F, double* be, double* V0,
                                double* mass, double* E, double* ys, double* v) {
  int w = blockIdx.x * blockDim.x + threadIdx.x;
  if (w >= P) return;
  size_t p = perm[w];
  for (int d = 0; d < 3; ++d) {
    x[3 * (size_t)w + d] = pts.x[3 * p + d];
    lp[3 * (size_t)w + d] = pts.lp[3 * p + d];
    l0[3 * (size_t)w + d] = pts.l0[3 * p + d];
    if (v) v[3 * (size_t)w + d] = pts.v[3 * p + d];
  }
  for (int i = 0; i < 9; ++i) F[9 * (size_t)w + i] = pts.F[9 * p + i];
  for (int i = 0; i < 6; ++i) be[6 * (size_t)w + i] = pts.be[6 * p + i];
  V0[w] = pts.V0[p];
  mass[w] = pts.mass[p];
  E[w] = pts.E[p];
  ys[w] = pts.ys[p];
}

// ------------------------------------------------------------------ discrete GIMP basis

struct SubBox {
  double xi[3];  // centroid in the leaf's local coordinates
  double w;      // V_Kp / V_p
  double is;     // 1 / leaf size (a power of two, exact)
  int K;
};

constexpr int BW = 4;  // warps per block of the basis kernel

constexpr int BH = 256;  // per-warp hash set of the basis kernel's node ids (at most MAXS distinct)

constexpr int BT = 16;  // sub-boxes whose corner values are tabulated at a time

__device__ inline unsigned basis_hash(int j) { return ((unsigned)j * 2654435761u) >> 24; }

// a positive normal float as a double, in integer instructions
__device__ inline double widen(float f) {
  unsigned b = __float_as_uint(f);
  return __hiloint2double((int)((b >> 3) + 0x38000000u), (int)(b << 29));
}

// scratch of one warp of the basis kernel: the open boxes of the leaf walk,
// then the node set, then the corner values
union BasisTmp {
  int open[MAXK][6];
  struct {
    int node[MAXE];  // node of an entry, then its rank
    int hkey[BH];
    int uid[MAXS], cnt[MAXS], next[MAXS];
    unsigned char hslot[BH], rank[MAXS];
  } set;
  double val[BT * 8 * 4];
};

// Eq. (GIMP numerical), one warp per point (cell-sorted order):
//  1. the domain is cut into its leaf intersections (centre, volume), the open
//     boxes of a round one per lane;
//  2. the (leaf corner, constraint entry) pairs are listed in a fixed order;
//  3. the distinct independent nodes are found by a shared-memory hash set and
//     ranked by id (support sorted by node id); the entries are grouped by
//     node, each group keeping list order;
//  4. every (sub-box, corner) value and gradient is computed once, by one lane,
//     into shared memory; a lane then owns one of the four numbers of a support
//     node and adds its weighted entries in list order, so the result does not
//     depend on scheduling.
// What bounds it: FP64 issue.  A warp's FP64 instruction takes its quarter of
// the SM for 64 cycles whatever the number of active lanes, so each stage
// spreads its FP64 work over the lanes: a bound of the domain, an axis of a
// sub-box, a corner, a (node, number) pair.  A lane per node that recomputed its entries'
// products took 20 instructions an entry, the longest group of 32 nodes long;
// here an entry takes one fma, the longest group of 8 nodes long.  1.9 M points:
// 26.1 ms so, 10.4 ms with the table and a lane per open box, sub-box and axis
// of the domain, 8.8 ms with a lane per bound and per axis of a sub-box (some
// 75 FP64 instructions a point, 7.5 ms of the FP64 pipe).
__global__ void __launch_bounds__(32 * BW)
    k_basis(int P, Geo g, const double* __restrict__ px, const double* __restrict__ plp,
            const double* __restrict__ pE, const uint64_t* __restrict__ lkey,
            const int* __restrict__ llev, int nl, const int* __restrict__ corner,
            const int* __restrict__ cptr, const int* __restrict__ cidx,
            const double* __restrict__ cw, int* nsup, int* sidx, double* S, double* dS,
            int* active, int* populated, unsigned long long* betaK, int* err) {
  __shared__ SubBox sb_s[BW][MAXK];
  __shared__ __align__(16) BasisTmp tmp_s[BW];
  __shared__ float e_w_s[BW][MAXE];  // constraint weights are sums of products of 1/2 and 1/4: exact
  __shared__ unsigned short e_ord_s[BW][MAXE];
  __shared__ unsigned short ustart_s[BW][MAXS + 1];
  __shared__ unsigned char e_q_s[BW][MAXE];  // 8 sub-box + corner, below 8 MAXK = 216
  __shared__ int nu_s[BW];
  int wi = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int w = blockIdx.x * BW + wi;
  if (w >= P) return;
  SubBox* sb = sb_s[wi];
  BasisTmp& tmp = tmp_s[wi];
  float* e_w = e_w_s[wi];
  unsigned char* e_q = e_q_s[wi];
  unsigned short *e_ord = e_ord_s[wi], *ustart = ustart_s[wi];
  const unsigned all = 0xffffffffu;
  // 1. the domain's bounds, one of the six per lane (lanes beyond the sixth
  // repeat them), then its leaf intersections
  double bd, Vp;  // lane 2 d + side: bound of axis d
  DomainCells dc;
  {
    int d = (lane % 6) >> 1, side = lane & 1;
    double x = px[3 * (size_t)w + d], l = plp[3 * (size_t)w + d];
    double v = snap_grid((side ? x + l : x - l) * g.scale), N = (double)g.N;
    double len = __shfl_xor_sync(all, v, 1) - v;  // of use in the even lanes
    bd = side ? (v > N ? N : v) : (v < 0.0 ? 0.0 : v);
    double fl = floor(bd);
    int f = (int)fl;
    unsigned whole = __ballot_sync(all, bd == fl);
    bool empty = !(__shfl_xor_sync(all, bd, 1) > bd) && !side;
    for (int i = 0; i < 3; ++i) {
      dc.lo[i] = __shfl_sync(all, f, 2 * i);
      dc.hi[i] = __shfl_sync(all, f, 2 * i + 1);
      dc.whole[i] = (whole >> (2 * i + 1)) & 1u;
    }
    Vp = __shfl_sync(all, len, 0) * __shfl_sync(all, len, 2) * __shfl_sync(all, len, 4);
    if (__any_sync(all, empty)) {
      if (lane == 0) {
        atomicOr(err, EB_DOMAIN);
        nsup[w] = 0;
      }
      return;
    }
  }
  int nsub = warp_cut_domain(g, lkey, llev, nl, dc, tmp.open, lane, [&](int n, int K, const int* a, const int* e) {
    int* cd = reinterpret_cast<int*>(sb[n].xi);  // bound codes until step 1b
    for (int d = 0; d < 3; ++d) {
      cd[d] = a[d];
      cd[3 + d] = e[d];
    }
    sb[n].K = K;
  });
  if (nsub < 0) {
    if (lane == 0) {
      atomicOr(err, EB_SUPPORT);
      nsup[w] = 0;
    }
    return;
  }
  // 1b. a sub-box and axis per lane, ten sub-boxes at a time: the sides'
  // lengths and the centroid in leaf coordinates; then a sub-box per lane: its
  // volume fraction
  for (int s0 = 0; s0 < nsub; s0 += 10) {
    int i = s0 + lane / 3, d = lane % 3;
    bool on = lane < 30 && i < nsub;
    SubBox& o = sb[on ? i : 0];
    const int* cd = reinterpret_cast<const int*>(o.xi);
    double lo = __shfl_sync(all, bd, 2 * d), hi = __shfl_sync(all, bd, 2 * d + 1);
    int ca = cd[d], ce = cd[3 + d], K = o.K, ka[3];
    demorton(lkey[K], ka);
    // the leaf size is a power of two: multiplying by its exact reciprocal
    // equals the division
    double is = __hiloint2double((1023 + llev[K] - g.D) << 20, 0);
    double a = ca < 0 ? lo : (double)ca, e = ce < 0 ? hi : (double)ce;
    double xi = (0.5 * (a + e) - (double)(d == 0 ? ka[0] : (d == 1 ? ka[1] : ka[2]))) * is;
    double len = e - a;
    double v1 = __shfl_down_sync(all, len, 1), v2 = __shfl_down_sync(all, len, 2);
    __syncwarp();
    if (on) o.xi[d] = xi;
    if (on && d == 0) {
      o.is = is;
      o.w = len * v1 * v2 / Vp;
      populated[K] = 1;
      atomicMax(betaK + K, (unsigned long long)__double_as_longlong(pE[w]));
    }
  }
  __syncwarp();
  // 2. list the (corner, constraint) entries in pair order
  int npair = 8 * nsub;
  int per = (npair + 31) / 32;
  int q0 = lane * per, q1 = min(q0 + per, npair);
  int len = 0;
  for (int q = q0; q < q1; ++q) {
    int node = corner[8 * (size_t)sb[q >> 3].K + (q & 7)];
    len += cptr[node + 1] - cptr[node];
  }
  int off = warp_excl_scan(len, lane);
  int total = __shfl_sync(all, off + len, 31);
  if (total > MAXE) {
    if (lane == 0) {
      atomicOr(err, EB_SUPPORT);
      nsup[w] = 0;
    }
    return;
  }
  int pos = off;
  for (int q = q0; q < q1; ++q) {
    int node = corner[8 * (size_t)sb[q >> 3].K + (q & 7)];
    for (int t = cptr[node]; t < cptr[node + 1]; ++t) {
      tmp.set.node[pos] = cidx[t];
      e_q[pos] = (unsigned char)q;
      e_w[pos] = (float)cw[t];
      ++pos;
    }
  }
  // 3. distinct nodes (hash set), ranked by id, entries grouped by node
  for (int i = lane; i < BH; i += 32) tmp.set.hkey[i] = -1;
  for (int u = lane; u < MAXS; u += 32) tmp.set.cnt[u] = 0;
  if (lane == 0) nu_s[wi] = 0;
  __syncwarp();
  for (int e = lane; e < total; e += 32) {
    int j = tmp.set.node[e];
    unsigned h = basis_hash(j);
    for (int probe = 0; probe < BH; ++probe) {
      int prev = atomicCAS(&tmp.set.hkey[h], -1, j);
      if (prev == -1) {
        int slot = atomicAdd(&nu_s[wi], 1);
        if (slot < MAXS) tmp.set.uid[slot] = j;
        tmp.set.hslot[h] = (unsigned char)min(slot, 255);
        break;
      }
      if (prev == j) break;
      h = (h + 1) & (BH - 1);
    }
  }
  __syncwarp();
  int ns = nu_s[wi];
  if (ns > MAXS) {
    if (lane == 0) {
      atomicOr(err, EB_SUPPORT);
      nsup[w] = 0;
    }
    return;
  }
  for (int u = lane; u < ns; u += 32) {
    int j = tmp.set.uid[u], r = 0;
    for (int u2 = 0; u2 < ns; ++u2) r += tmp.set.uid[u2] < j ? 1 : 0;
    tmp.set.rank[u] = (unsigned char)r;
    sidx[(size_t)w * MAXS + r] = j;
    active[j] = 1;
  }
  __syncwarp();
  // rank of every entry (hash lookup) and the count per rank
  for (int e = lane; e < total; e += 32) {
    int j = tmp.set.node[e];
    unsigned h = basis_hash(j);
    while (tmp.set.hkey[h] != j) h = (h + 1) & (BH - 1);
    int r = tmp.set.rank[tmp.set.hslot[h]];
    tmp.set.node[e] = r;
    atomicAdd(&tmp.set.cnt[r], 1);
  }
  __syncwarp();
  {
    int c0 = lane < ns ? tmp.set.cnt[lane] : 0, c1 = lane + 32 < ns ? tmp.set.cnt[lane + 32] : 0;
    int x0 = warp_excl_scan(c0, lane), x1 = warp_excl_scan(c1, lane);
    int t0 = __shfl_sync(all, x0 + c0, 31);
    if (lane < ns) tmp.set.next[lane] = ustart[lane] = x0;
    if (lane + 32 < ns) tmp.set.next[lane + 32] = ustart[lane + 32] = t0 + x1;
    if (lane == 0) ustart[ns] = total;
  }
  __syncwarp();
  // stable grouping: chunks of 32 entries in list order, positions inside a
  // chunk by lane order among the lanes of the same rank
  for (int c0 = 0; c0 < total; c0 += 32) {
    int e = c0 + lane;
    bool valid = e < total;
    int r = valid ? tmp.set.node[e] : -1 - lane;
    unsigned grp = __match_any_sync(all, r);
    int before = __popc(grp & ((1u << lane) - 1u));
    int at = valid ? tmp.set.next[r] + before : 0;
    __syncwarp();
    if (valid) {
      e_ord[at] = (unsigned short)e;
      if (before == 0) tmp.set.next[r] += __popc(grp);
    }
    __syncwarp();
  }
  // 4. values and gradients of S_vp
  for (int b0 = 0; b0 < nsub; b0 += BT) {
    int b1 = min(b0 + BT, nsub);
    __syncwarp();
    for (int i = lane; i < 8 * (b1 - b0); i += 32) {
      const SubBox& o = sb[b0 + (i >> 3)];
      int c = i & 7;
      double f0 = (c & 1) ? o.xi[0] : 1.0 - o.xi[0];
      double f1 = (c & 2) ? o.xi[1] : 1.0 - o.xi[1];
      double f2 = (c & 4) ? o.xi[2] : 1.0 - o.xi[2];
      double v = o.w, vs = v * o.is;
      double f01 = f0 * f1, f02 = f0 * f2, f12 = f1 * f2;
      double* t = tmp.val + 4 * i;
      t[0] = v * (f01 * f2);
      t[1] = ((c & 1) ? vs : -vs) * f12;
      t[2] = ((c & 2) ? vs : -vs) * f02;
      t[3] = ((c & 4) ? vs : -vs) * f01;
    }
    __syncwarp();
    int n = lane & 3;  // S and the three components of dS
    for (int k = lane >> 2; k < ns; k += 8) {
      size_t o = (size_t)w * MAXS + k;
      double* out = n == 0 ? S + o : dS + 3 * o + (n - 1);
      double a = b0 ? *out : 0.0;
      for (int t = ustart[k]; t < ustart[k + 1]; ++t) {
        int e = e_ord[t], q = (int)e_q[e] - 8 * b0;
        if (nsub > BT && (q < 0 || q >= 8 * BT)) continue;
        a = fma(widen(e_w[e]), tmp.val[4 * q + n], a);
      }
      *out = n > 0 && b1 == nsub ? a * g.scale : a;
    }
  }
  if (lane == 0) nsup[w] = ns;
}

__global__ void k_number_dofs(int nn, const int* __restrict__ active, const int* __restrict__ pos,
                              int* node_dof, int* dof_node) {
  int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= nn) return;
  if (active[n]) {
    node_dof[n] = pos[n];
    dof_node[pos[n]] = n;
  } else {
    node_dof[n] = -1;
  }
}

struct Planes {
  int n;
  int axis[8];
  int pos[8];
  int mask[8];
};

__global__ void k_dof_mask(int nd, const int* __restrict__ dof_node, const uint64_t* __restrict__ nkey,
                           Planes pl, int* mask) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nd) return;
  int X[3];
  demorton(nkey[dof_node[i]], X);
  int m = 0;
  for (int b = 0; b < pl.n; ++b)
    if (X[pl.axis[b]] == pl.pos[b]) m |= pl.mask[b];
  mask[i] = m;
}

// ------------------------------------------------------------------ ghost faces (Sec. 4)

__device__ inline int across(const uint64_t* lkey, const int* llev, int nl, const Geo& g, int K,
                             int axis, int sign, int o1, int o2) {
  int a[3];
  demorton(lkey[K], a);
  int s = 1 << (g.D - llev[K]);
  a[axis] = sign > 0 ? a[axis] + s : a[axis] - 1;
  if (a[axis] < 0 || a[axis] >= g.N) return -1;
  a[(axis + 1) % 3] += o1;
  a[(axis + 2) % 3] += o2;
  return locate(lkey, nl, a[0], a[1], a[2]);
}

// T^B: populated leaves sharing a face with an unpopulated leaf
__global__ void k_boundary_elements(int nl, const uint64_t* __restrict__ lkey,
                                    const int* __restrict__ llev, Geo g,
                                    const int* __restrict__ pop, int* isB) {
  int K = blockIdx.x * blockDim.x + threadIdx.x;
  if (K >= nl) return;
  int b = 0;
  if (pop[K]) {
    int s = 1 << (g.D - llev[K]);
    for (int f = 0; f < 6 && !b; ++f) {
      int axis = f >> 1, sign = (f & 1) ? 1 : -1;
      int nb = across(lkey, llev, nl, g, K, axis, sign, 0, 0);
      if (nb < 0) continue;
      if (llev[nb] <= llev[K]) {
        if (!pop[nb]) b = 1;
      } else {
        for (int o = 0; o < 4; ++o) {
          int nb2 = across(lkey, llev, nl, g, K, axis, sign, (o & 1) * (s >> 1), ((o >> 1) & 1) * (s >> 1));
          if (!pop[nb2]) b = 1;
        }
      }
    }
  }
  isB[K] = b;
}

// F_B: both leaves populated and one of them in T^B; each face once, from its
// smaller leaf (equal leaves: from the lower one)
__global__ void k_ghost_face_flag(int nl, const uint64_t* __restrict__ lkey,
                                  const int* __restrict__ llev, Geo g, const int* __restrict__ pop,
                                  const int* __restrict__ isB, int* flag) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 6 * nl) return;
  int K = i / 6, f = i % 6;
  int axis = f >> 1, sign = (f & 1) ? 1 : -1;
  int ok = 0;
  if (pop[K]) {
    int nb = across(lkey, llev, nl, g, K, axis, sign, 0, 0);
    if (nb >= 0 && llev[nb] <= llev[K] && !(llev[nb] == llev[K] && sign < 0) && pop[nb] &&
        (isB[K] || isB[nb]))
      ok = 1;
  }
  flag[i] = ok;
}

__global__ void k_ghost_face_write(int nl, const uint64_t* __restrict__ lkey,
                                   const int* __restrict__ llev, Geo g, const int* __restrict__ flag,
                                   const int* __restrict__ pos, int* face) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 6 * nl || !flag[i]) return;
  int K = i / 6, f = i % 6;
  int axis = f >> 1, sign = (f & 1) ? 1 : -1;
  int p = pos[i];
  face[4 * p] = K;
  face[4 * p + 1] = across(lkey, llev, nl, g, K, axis, sign, 0, 0);
  face[4 * p + 2] = axis;
  face[4 * p + 3] = sign;
}

// dofs of I(K+) u I(K-) of each ghost face
__global__ void k_ghost_face_dofs(int nf, const int* __restrict__ face, const int* __restrict__ corner,
                                  const int* __restrict__ cptr, const int* __restrict__ cidx,
                                  const int* __restrict__ node_dof, int* gdof, int* gn, int* err) {
  int f = blockIdx.x * blockDim.x + threadIdx.x;
  if (f >= nf) return;
  int n = 0;
  int* out = gdof + (size_t)f * MAXG;
  for (int side = 0; side < 2; ++side) {
    int K = face[4 * f + side];
    for (int c = 0; c < 8; ++c) {
      int node = corner[8 * (size_t)K + c];
      for (int t = cptr[node]; t < cptr[node + 1]; ++t) {
        int j = node_dof[cidx[t]];
        bool have = false;
        for (int q = 0; q < n; ++q) have = have || out[q] == j;
        if (have) continue;
        if (n >= MAXG || j < 0) {
          atomicOr(err, EB_SUPPORT);
          continue;
        }
        out[n++] = j;
      }
    }
  }
  gn[f] = n;
}

__device__ inline int find_slot(const int* __restrict__ row_ptr, const int* __restrict__ col, int r,
                                int c) {
  int lo = row_ptr[r], hi = row_ptr[r + 1] - 1;
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

// Eq. (ghost): 2x2 Gauss points on the smaller face, mapped into the larger
// leaf; k_G(i,j) = sum over faces and Gauss points of w (h_F beta_F / kappa)
// J_i J_j with J the normal-derivative jump.  One warp per face stores the
// face's coefficient w h_F beta_F / kappa and its jumps J (4 x MAXG); the
// rows are summed by k_ghost_rows.  The 64 corner derivatives (Gauss point,
// side, corner) are computed once, two a lane, into shared memory; then the
// warp goes over the constraint entries of the 16 corners, and the lane of an
// entry's dof adds them at the four Gauss points.  A lane that looked through
// the entries of both leaves for its dof at every Gauss point, the derivatives
// with it, was bound by FP64 and the chains of lookups (1.06 ms for the
// indentation block's faces at 1.9 M points, 0.10 now).
__global__ void __launch_bounds__(128)
    k_ghost_jumps(int nf, Geo g, double kappa, const int* __restrict__ face,
                              const uint64_t* __restrict__ lkey, const int* __restrict__ llev,
                              const double* __restrict__ betaK, const int* __restrict__ gdof,
                              const int* __restrict__ gn, const int* __restrict__ corner,
                              const int* __restrict__ cptr, const int* __restrict__ cidx,
                              const double* __restrict__ cw, const int* __restrict__ node_dof,
                              double* gJ, double* gcoef) {
  __shared__ double dphi[4][16][4];  // [warp][side, corner][Gauss point]
  const unsigned all = 0xffffffffu;
  int wi = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int f = blockIdx.x * 4 + wi;
  if (f >= nf) return;
  int K = face[4 * f], Nb = face[4 * f + 1], axis = face[4 * f + 2], sign = face[4 * f + 3];
  int lK = llev[K], lN = llev[Nb];
  int sK = 1 << (g.D - lK), sN = 1 << (g.D - lN);
  // the entries of corner `lane` (side lane >> 3): the first one's dof and weight at once
  int t0 = 0, nt = 0, j0 = -1;
  double w0 = 0.0;
  if (lane < 16) {
    int node = corner[8 * (size_t)(lane < 8 ? K : Nb) + (lane & 7)];
    t0 = cptr[node];
    nt = cptr[node + 1] - t0;
    if (nt > 0) {
      j0 = node_dof[cidx[t0]];
      w0 = cw[t0];
    }
  }
  {
    int aK[3], aL[3];
    demorton(lkey[K], aK);
    int side = (lane >> 3) & 1, c = lane & 7;
    demorton(lkey[side ? Nb : K], aL);
    // leaf sizes are powers of two: their reciprocals are exact
    double is = __hiloint2double((1023 + (side ? lN : lK) - g.D) << 20, 0);
    const double gq = 0.5 / sqrt(3.0);
    int t1 = (axis + 1) % 3, t2 = (axis + 2) % 3;
    int ak1 = t1 == 0 ? aK[0] : (t1 == 1 ? aK[1] : aK[2]), ak2 = t2 == 0 ? aK[0] : (t2 == 1 ? aK[1] : aK[2]);
    int al1 = t1 == 0 ? aL[0] : (t1 == 1 ? aL[1] : aL[2]), al2 = t2 == 0 ? aL[0] : (t2 == 1 ? aL[1] : aL[2]);
    double d0 = ((c >> axis) & 1) ? is : -is;
    for (int gp = lane >> 4; gp < 4; gp += 2) {
      double x1 = (double)ak1 + (double)sK * ((gp & 1) ? 0.5 + gq : 0.5 - gq);
      double x2 = (double)ak2 + (double)sK * ((gp & 2) ? 0.5 + gq : 0.5 - gq);
      double xi1 = (x1 - (double)al1) * is, xi2 = (x2 - (double)al2) * is;
      double f1 = ((c >> t1) & 1) ? xi1 : 1.0 - xi1, f2 = ((c >> t2) & 1) ? xi2 : 1.0 - xi2;
      dphi[wi][lane & 15][gp] = d0 * f1 * f2;
    }
  }
  if (lane == 0) {
    double hF = (double)(sK > sN ? sK : sN) * g.unit;
    double bF = betaK[K] > betaK[Nb] ? betaK[K] : betaK[Nb];
    double area = ((double)sK * g.unit) * ((double)sK * g.unit);
    gcoef[f] = hF * bF / kappa * area / 4.0;
  }
  __syncwarp();
  int n = gn[f];
  const int* ids = gdof + (size_t)f * MAXG;
  for (int e0 = 0; e0 < n; e0 += 32) {
    int e = e0 + lane, j = e < n ? ids[e] : -2;
    double jk[4] = {0.0, 0.0, 0.0, 0.0}, jn[4] = {0.0, 0.0, 0.0, 0.0};
    for (int q = 0; q < 16; ++q) {
      int m = __shfl_sync(all, nt, q), t = __shfl_sync(all, t0, q);
      for (int k = 0; k < m; ++k) {
        int jq = k ? node_dof[cidx[t + k]] : __shfl_sync(all, j0, q);
        double w = k ? cw[t + k] : __shfl_sync(all, w0, q);
        if (jq != j) continue;
#pragma unroll
        for (int gp = 0; gp < 4; ++gp) {
          if (q < 8)
            jk[gp] = fma(w, dphi[wi][q][gp], jk[gp]);
          else
            jn[gp] = fma(w, dphi[wi][q][gp], jn[gp]);
        }
      }
    }
    if (e < n)
      for (int gp = 0; gp < 4; ++gp)
        gJ[((size_t)f * 4 + gp) * MAXG + e] = (double)sign * (jk[gp] - jn[gp]) * g.scale;
  }
}

// k_G row r: one warp; the row's ghost-face sources (face f, local index a of
// r in the face's dofs) in key order, and for each the face's dofs b over the
// lanes: k_G(r, b) += coef_f sum over Gauss points of J_a J_b.  The lanes of
// one source write distinct columns and the sources follow one another, so
// every entry is summed in a fixed order (no atomics).  The faces are the last
// of a row's sources; the warp looks for the first of them from the end, 32 keys
// at a time (passing over some 200 points one by one took 0.62 ms for 248 k
// rows, most of them without a face; 0.21 now).
__global__ void k_ghost_rows(int nd, int P, const long long* __restrict__ sptr,
                             const uint64_t* __restrict__ skeys, const int* __restrict__ gdof,
                             const int* __restrict__ gn, const double* __restrict__ gJ,
                             const double* __restrict__ gcoef, const int* __restrict__ row_ptr,
                             const int* __restrict__ col, double* kg) {
  int r = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (r >= nd) return;
  long long q0 = sptr[r], q1 = sptr[r + 1], first = q1;
  while (first > q0) {
    long long q = first - 1 - lane;
    unsigned faces = __ballot_sync(0xffffffffu, q >= q0 && (int)((uint32_t)skeys[q] >> 6) >= P);
    first -= __popc(faces);  // the faces of the 32 keys are the last of them
    if (faces != 0xffffffffu) break;
  }
  for (long long q = first; q < q1; ++q) {
    uint32_t sid = (uint32_t)skeys[q];
    int f = (int)(sid >> 6) - P, a = (int)(sid & 63);
    double cf = gcoef[f];
    const double* J = gJ + (size_t)f * 4 * MAXG;
    double ja[4] = {J[a], J[MAXG + a], J[2 * MAXG + a], J[3 * MAXG + a]};
    int n = gn[f];
    for (int b = lane; b < n; b += 32) {
      double v = cf * (ja[0] * J[b] + ja[1] * J[MAXG + b] + ja[2] * J[2 * MAXG + b] +
                       ja[3] * J[3 * MAXG + b]);
      if (v == 0.0) continue;
      int sl = find_slot(row_ptr, col, r, gdof[(size_t)f * MAXG + b]);
      if (sl >= 0) kg[sl] += v;
    }
    __syncwarp();
  }
}

// ------------------------------------------------------------------ block pattern

// Counts of a mesh kept on the device until the build's last synchronisation:
// the sum over the points of (support size)^2, i.e. the (source, column) pairs
// of the tangent gather, for the benchmark's operation counts (integer, exact);
// the largest support, the longest row and the number of hanging nodes.
struct MeshCounts {
  unsigned long long npair;
  int maxs, maxrow, nhang;
};

// one warp per point: its support from node ids to dofs, and the point's
// source keys: row dof << 32 | source << 6 | local index (points, then ghost
// faces).  With these bits the keys of the points, and of the faces after them,
// are listed in ascending order of their lower 32 bits: a stable sort by the
// row alone (3 passes of 8 bits at 248 k rows instead of 8) orders them fully.
__global__ void k_point_sources(int P, const int* __restrict__ nsup, const int* __restrict__ node_dof,
                                const int* __restrict__ off, int* sidx, uint64_t* keys,
                                MeshCounts* mc) {
  __shared__ int ns[32];
  int wi = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  int w = blockIdx.x * nw + wi;
  int n = w < P ? nsup[w] : 0;
  int o = n ? off[w] : 0;
  for (int k = lane; k < n; k += 32) {
    size_t i = (size_t)w * MAXS + k;
    int r = node_dof[sidx[i]];
    sidx[i] = r;
    keys[o + k] = ((uint64_t)(uint32_t)r << 32) | ((uint64_t)(uint32_t)w << 6) | (uint32_t)k;
  }
  if (lane == 0) ns[wi] = n;
  __syncthreads();
  if (wi == 0) {
    n = lane < nw ? ns[lane] : 0;
    int mx = __reduce_max_sync(0xffffffffu, n), sq = warp_sum_int(n * n);
    if (lane == 0 && sq) {
      atomicAdd(&mc->npair, (unsigned long long)sq);
      if (mx > *(volatile int*)&mc->maxs) atomicMax(&mc->maxs, mx);
    }
  }
}

__global__ void k_src_keys_faces(int nf, int P, const int* __restrict__ gn, const int* __restrict__ gdof,
                                 long long base, uint64_t* keys) {
  long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (long long)nf * MAXG) return;
  int f = (int)(i / MAXG), k = (int)(i % MAXG);
  if (k >= gn[f]) return;
  keys[base + (long long)f * MAXG + k] =
      ((uint64_t)(uint32_t)gdof[i] << 32) | ((uint64_t)(uint32_t)(P + f) << 6) | (uint32_t)k;
}

__global__ void k_src_ptr(long long n, const uint64_t* __restrict__ keys, int ndof, long long* ptr) {
  long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  uint32_t r = (uint32_t)(keys[i] >> 32);
  if (r >= (uint32_t)ndof) return;  // unused padding keys sort last
  if (i == 0 || (uint32_t)(keys[i - 1] >> 32) != r) ptr[r] = i;
  if (i == n - 1 || (uint32_t)(keys[i + 1] >> 32) != r) ptr[r + 1] = i + 1;
}

// Block pattern: the columns of row r are the union of the supports of every
// source (point or ghost face) touching r.  One warp per row collects them in
// a hash set in shared memory and ranks them.  Taken source by source it
// waits on the chain key -> support -> insertion, some 200 times a row; so a warp
// takes 32 keys and support sizes
// at once, 8 supports in flight, and reads a slot before it tries to claim it
// (some 40 of 41 insertions find their column there).  Rows of at most PSHORT
// columns (125 where the leaf size does not change) use a set of 512 slots
// (3 KB a warp, 44 warps to the SM; 2048 slots leave room for 18) and leave
// their sorted columns in a staging row, which a copy takes to its place once
// the row lengths are known; the others are collected again then, by the kernel
// with the large set.  Two traversals, source by source, of a 2048-slot set took
// 2 x 5.63 ms for 248 k rows and 29 M sources; now 2.10 ms, bound by
// instruction issue (87 % of the slots), and the copy 0.08 ms.
constexpr int PSHORT = 256;            // longest row of the small set, and a staging row
constexpr int PHASH = 2 * PSHORT;      // its slots
constexpr int PPROBE = 64;             // its longest probe sequence; a row beyond it is a long one
constexpr int PW = 4;                  // warps per block of the pattern kernels
constexpr int PLW = 2;                 // the same of the long rows' kernel

struct PatternSrc {
  int P;
  const long long* sptr;
  const uint64_t* keys;
  const int *nsup, *sidx, *gn, *gdof;
};

// 1: added, 0: there already, -1: no slot within `probes`
template <int H>
__device__ inline int set_insert(volatile int* h, int key, int probes) {
  unsigned s = ((unsigned)key * 2654435761u) >> 16 & (H - 1);
  for (int i = 0; i < probes; ++i) {
    int v = h[s];
    if (v == -1) v = atomicCAS((int*)h + s, -1, key);
    if (v == -1) return 1;
    if (v == key) return 0;
    s = (s + 1) & (H - 1);
  }
  return -1;
}

// the set of row r's columns in h[H]; their number, or -1 when more than `limit`
// or out of slots
template <int H>
__device__ int pattern_collect(const PatternSrc& p, int r, int* h, int limit, int probes, int lane) {
  const unsigned all = 0xffffffffu;
  for (int i = lane; i < H; i += 32) h[i] = -1;
  __syncwarp();
  int cnt = 0;
  bool bad = false;
  long long s1 = p.sptr[r + 1];
  for (long long s0 = p.sptr[r]; s0 < s1; s0 += 32) {
    int m = (int)min(32LL, s1 - s0), n = 0;
    long long base = 0;  // of the lane's source, in sidx or (from P on) gdof
    if (lane < m) {
      int sid = (int)((uint32_t)p.keys[s0 + lane] >> 6);
      n = sid < p.P ? p.nsup[sid] : p.gn[sid - p.P];
      base = sid < p.P ? (long long)sid * MAXS : -1 - (long long)(sid - p.P) * MAXG;
    }
    for (int t = 0; t < m; t += 8) {
      int v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        int nu = __shfl_sync(all, n, (t + u) & 31);  // 0 past the last source
        long long b = __shfl_sync(all, base, (t + u) & 31);
        const int* q = b >= 0 ? p.sidx + b : p.gdof + (-1 - b);
        v[u] = lane < nu ? q[lane] : -1;
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        if (v[u] < 0) continue;
        int rv = set_insert<H>(h, v[u], probes);
        cnt += rv > 0;
        bad |= rv < 0;
      }
    }
    // supports of more than 32 nodes
    for (unsigned more = __ballot_sync(all, n > 32); more; more &= more - 1) {
      int t = __ffs(more) - 1;
      int nu = __shfl_sync(all, n, t);
      long long b = __shfl_sync(all, base, t);
      const int* q = b >= 0 ? p.sidx + b : p.gdof + (-1 - b);
      for (int l = lane + 32; l < nu; l += 32) {
        int rv = set_insert<H>(h, q[l], probes);
        cnt += rv > 0;
        bad |= rv < 0;
      }
      __syncwarp();
    }
    if (__any_sync(all, bad) || __reduce_add_sync(all, cnt) > limit) return -1;
  }
  __syncwarp();
  return warp_sum_int(cnt);
}

// the set's cnt members in ascending order to out, by way of the list lst (its
// length a multiple of 4, 16-byte aligned)
template <int H>
__device__ void pattern_sorted(const int* h, int cnt, int* lst, int* out, int lane) {
  int at = 0;
  for (int i = lane; i < H; i += 32) {
    int v = h[i];
    unsigned b = __ballot_sync(0xffffffffu, v >= 0);
    if (v >= 0) lst[at + __popc(b & ((1u << lane) - 1u))] = v;
    at += __popc(b);
  }
  if (lane < ((4 - (cnt & 3)) & 3)) lst[cnt + lane] = 0x7fffffff;
  __syncwarp();
  for (int e0 = 0; e0 < cnt; e0 += 128) {
    int v[4], rk[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      int e = e0 + 32 * j + lane;
      v[j] = e < cnt ? lst[e] : 0;
      rk[j] = 0;
    }
    for (int t = 0; t < cnt; t += 4) {
      int4 x = *reinterpret_cast<const int4*>(lst + t);
#pragma unroll
      for (int j = 0; j < 4; ++j)
        rk[j] += (x.x < v[j]) + (x.y < v[j]) + (x.z < v[j]) + (x.w < v[j]);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (e0 + 32 * j + lane < cnt) out[rk[j]] = v[j];
  }
}

// lengths of the rows and the sorted columns of the short ones in their staging
// rows; -1 for a long row
__global__ void __launch_bounds__(32 * PW)
    k_pattern_rows(int ndof, PatternSrc p, int* rowcnt, int* stage) {
  __shared__ int h[PW][PHASH];
  __shared__ __align__(16) int lst[PW][PSHORT];
  int wi = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int r = blockIdx.x * PW + wi;
  if (r >= ndof) return;
  int cnt = pattern_collect<PHASH>(p, r, h[wi], PSHORT, PPROBE, lane);
  if (lane == 0) rowcnt[r] = cnt;
  if (cnt > 0) pattern_sorted<PHASH>(h[wi], cnt, lst[wi], stage + (size_t)r * PSHORT, lane);
}

// the long rows.  row_ptr null: their lengths (columns to the staging row where
// they fit it after all); else the columns of those that did not fit it
__global__ void __launch_bounds__(32 * PLW)
    k_pattern_long(int ndof, PatternSrc p, int* rowcnt, int* stage, const int* __restrict__ row_ptr,
                   int* col, int* err) {
  __shared__ int h[PLW][HASH];
  __shared__ __align__(16) int lst[PLW][MAXROW];
  int wi = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int r0 = 32 * (blockIdx.x * PLW + wi); r0 < ndof; r0 += 32 * PLW * gridDim.x) {
    int n = r0 + lane < ndof ? rowcnt[r0 + lane] : 0;
    unsigned todo = __ballot_sync(0xffffffffu, row_ptr ? n > PSHORT : n < 0);
    for (; todo; todo &= todo - 1) {
      int r = r0 + __ffs(todo) - 1;
      int cnt = pattern_collect<HASH>(p, r, h[wi], MAXROW, HASH, lane);
      if (!row_ptr && lane == 0) {
        rowcnt[r] = max(cnt, 0);
        if (cnt < 0) atomicOr(err, EB_ROW);
      }
      if (row_ptr && cnt > 0)
        pattern_sorted<HASH>(h[wi], cnt, lst[wi], col + row_ptr[r], lane);
      else if (!row_ptr && cnt > 0 && cnt <= PSHORT)
        pattern_sorted<HASH>(h[wi], cnt, lst[wi], stage + (size_t)r * PSHORT, lane);
      __syncwarp();
    }
  }
}

// staging rows to their place, one warp per row
__global__ void k_pattern_write(int ndof, const int* __restrict__ row_ptr, const int* __restrict__ stage,
                                int* col) {
  int r = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (r >= ndof) return;
  int b = row_ptr[r], n = row_ptr[r + 1] - b;
  if (n > PSHORT) return;
  for (int i = lane; i < n; i += 32) col[b + i] = stage[(size_t)r * PSHORT + i];
}

// ------------------------------------------------------------------ gravity, contact candidates

// f_ext,r = sum over the point sources (p, k) of row r of S_pk m_p g: one warp
// per row, lanes strided over the sources in key order, then the fixed
// shuffle tree (the same sums on every run)
__global__ void k_fext_rows(int nd, int P, const long long* __restrict__ sptr,
                            const uint64_t* __restrict__ skeys, const double* __restrict__ S,
                            const double* __restrict__ mass, double g0, double g1, double g2,
                            double* fext) {
  int r = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (r >= nd) return;
  double a = 0.0;
  for (long long q = sptr[r] + lane; q < sptr[r + 1]; q += 32) {
    uint32_t sid = (uint32_t)skeys[q];
    int w = (int)(sid >> 6), k = (int)(sid & 63);
    if (w >= P) continue;
    a += S[(size_t)w * MAXS + k] * mass[w];
  }
  a = warp_sum(a);
  if (lane < 3) fext[3 * (size_t)r + lane] = a * (lane == 0 ? g0 : (lane == 1 ? g1 : g2));
}

__global__ void k_cand_flag(int P, const double* __restrict__ px, const double* __restrict__ plp,
                            Body b, double margin, int* flag) {
  int w = blockIdx.x * blockDim.x + threadIdx.x;
  if (w >= P) return;
  int f = 0;
  // the distance to the body changes by no more than the step: a domain whose
  // centre lies farther off than the margin and its half-diagonal (at most the
  // sum of its half-lengths; with room for rounding) has no corner within the
  // margin.  One distance for most points, not eight: 1.17 -> 0.19 ms, 1.9 M
  const double *xp = px + 3 * (size_t)w, *lp = plp + 3 * (size_t)w;
  double far = 1.000001 * (margin + (fabs(lp[0]) + fabs(lp[1]) + fabs(lp[2])));
  if (body_distance(b, xp, far) > far) {
    flag[w] = 0;
    return;
  }
  for (int c = 0; c < 8 && !f; ++c) {
    double y[3];
    for (int d = 0; d < 3; ++d)
      y[d] = px[3 * (size_t)w + d] + (((c >> d) & 1) ? 1.0 : -1.0) * plp[3 * (size_t)w + d];
    if (body_distance(b, y, margin) <= margin) f = 1;
  }
  flag[w] = f;
}

__global__ void k_cand_write(int P, const int* __restrict__ flag, const int* __restrict__ pos,
                             int* cand) {
  int w = blockIdx.x * blockDim.x + threadIdx.x;
  if (w < P && flag[w]) cand[pos[w]] = w;
}

// background basis of each candidate corner, in the leaf on the inside of the domain
__global__ void k_cand_basis(int nc, const int* __restrict__ cand, Geo g,
                             const double* __restrict__ px, const double* __restrict__ plp,
                             const uint64_t* __restrict__ lkey, const int* __restrict__ llev, int nl,
                             const int* __restrict__ corner, const int* __restrict__ cptr,
                             const int* __restrict__ cidx, const double* __restrict__ cw,
                             const int* __restrict__ node_dof, int* cb_n, int* cb_idx,
                             double* cb_phi, double* cb_y0, int* err) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 8 * nc) return;
  int w = cand[i >> 3], c = i & 7;
  double Lo[3], Hi[3];
  domain_box(px + 3 * (size_t)w, plp + 3 * (size_t)w, g, Lo, Hi);
  int q[3];
  double X[3];
  for (int d = 0; d < 3; ++d) {
    int side = (c >> d) & 1;
    X[d] = side ? Hi[d] : Lo[d];
    int v = side ? (int)ceil(X[d]) - 1 : (int)floor(X[d]);
    q[d] = v < 0 ? 0 : (v > g.N - 1 ? g.N - 1 : v);
    cb_y0[3 * (size_t)i + d] = px[3 * (size_t)w + d] + (side ? 1.0 : -1.0) * plp[3 * (size_t)w + d];
  }
  int K = locate(lkey, nl, q[0], q[1], q[2]);
  int s = 1 << (g.D - llev[K]);
  int a[3];
  demorton(lkey[K], a);
  double xi[3];
  for (int d = 0; d < 3; ++d) xi[d] = (X[d] - (double)a[d]) / (double)s;
  int n = 0;
  int* ids = cb_idx + (size_t)i * MAXCB;
  double* ph = cb_phi + (size_t)i * MAXCB;
  for (int cc = 0; cc < 8; ++cc) {
    double f = 1.0;
    for (int d = 0; d < 3; ++d) f *= ((cc >> d) & 1) ? xi[d] : 1.0 - xi[d];
    int node = corner[8 * (size_t)K + cc];
    for (int t = cptr[node]; t < cptr[node + 1]; ++t) {
      int j = node_dof[cidx[t]];
      int slot = -1;
      for (int e = 0; e < n; ++e)
        if (ids[e] == j) slot = e;
      if (slot < 0) {
        if (n >= MAXCB || j < 0) {
          atomicOr(err, EB_SUPPORT);
          continue;
        }
        slot = n++;
        ids[slot] = j;
        ph[slot] = 0.0;
      }
      ph[slot] += cw[t] * f;
    }
  }
  cb_n[i] = n;
}

// the transpose of the corner basis: keys (dof << 32 | corner << 5 | entry),
// unused entries last
__global__ void k_ct_keys(int nc8, const int* __restrict__ cb_n, const int* __restrict__ cb_idx,
                          uint64_t* keys) {
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (long long)nc8 * MAXCB) return;
  int i = (int)(t / MAXCB), e = (int)(t % MAXCB);
  keys[t] = e < cb_n[i] ? ((uint64_t)(uint32_t)cb_idx[t] << 32) | ((uint64_t)i << 5) | (uint64_t)e
                        : ~0ULL;
}

// first entry of each row in the sorted keys
__global__ void k_ct_flag(long long n, const uint64_t* __restrict__ keys, int* flag) {
  long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= n) return;
  uint64_t k = keys[q];
  flag[q] = k != ~0ULL && (q == 0 || (keys[q - 1] >> 32) != (k >> 32));
}

__global__ void k_ct_write(long long n, const uint64_t* __restrict__ keys, const int* __restrict__ flag,
                           const int* __restrict__ pos, int nrow, int* crow, int* cptr, int* cent) {
  long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= n) return;
  uint64_t k = keys[q];
  if (k == ~0ULL) return;
  cent[q] = (int)(k & 0xffffffffULL);
  if (flag[q]) {
    crow[pos[q]] = (int)(k >> 32);
    cptr[pos[q]] = (int)q;
  }
  if (q == n - 1 || keys[q + 1] == ~0ULL) cptr[nrow] = (int)(q + 1);
}

// ------------------------------------------------------------------ triangulated body

// unit normal of every triangle (body frame)
__global__ void k_tri_fn(int nt, const double* __restrict__ v, const int* __restrict__ t, double* fn) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nt) return;
  const double *a = v + 3 * (size_t)t[3 * i], *b = v + 3 * (size_t)t[3 * i + 1],
               *c = v + 3 * (size_t)t[3 * i + 2];
  double u[3] = {b[0] - a[0], b[1] - a[1], b[2] - a[2]};
  double w[3] = {c[0] - a[0], c[1] - a[1], c[2] - a[2]};
  double n[3] = {u[1] * w[2] - u[2] * w[1], u[2] * w[0] - u[0] * w[2], u[0] * w[1] - u[1] * w[0]};
  double l = sqrt(n[0] * n[0] + n[1] * n[1] + n[2] * n[2]);
  for (int d = 0; d < 3; ++d) fn[3 * (size_t)i + d] = n[d] / l;
}

// edge pseudo-normals: the face normal plus that of the first other triangle
// (in index order) holding both ends of the edge
__global__ void k_tri_en(int nt, const int* __restrict__ t, const double* __restrict__ fn, double* en) {
  int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= 3 * nt) return;
  int i = e / 3, k = e % 3;
  int a = t[3 * i + k], b = t[3 * i + (k + 1) % 3];
  double N[3] = {fn[3 * (size_t)i], fn[3 * (size_t)i + 1], fn[3 * (size_t)i + 2]};
  for (int u = 0; u < nt; ++u) {
    if (u == i) continue;
    int ha = 0, hb = 0;
    for (int q = 0; q < 3; ++q) {
      ha |= t[3 * u + q] == a;
      hb |= t[3 * u + q] == b;
    }
    if (ha && hb) {
      for (int d = 0; d < 3; ++d) N[d] += fn[3 * (size_t)u + d];
      break;
    }
  }
  for (int d = 0; d < 3; ++d) en[3 * (size_t)e + d] = N[d];
}

// vertex pseudo-normals: angle-weighted sum of the face normals around the
// vertex (triangles in index order)
__global__ void k_tri_vn(int nv, int nt, const double* __restrict__ v, const int* __restrict__ t,
                         const double* __restrict__ fn, double* vn) {
  int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= nv) return;
  double N[3] = {0.0, 0.0, 0.0};
  const double* a = v + 3 * (size_t)p;
  for (int u = 0; u < nt; ++u)
    for (int k = 0; k < 3; ++k) {
      if (t[3 * u + k] != p) continue;
      const double* b = v + 3 * (size_t)t[3 * u + (k + 1) % 3];
      const double* c = v + 3 * (size_t)t[3 * u + (k + 2) % 3];
      double e1[3] = {b[0] - a[0], b[1] - a[1], b[2] - a[2]};
      double e2[3] = {c[0] - a[0], c[1] - a[1], c[2] - a[2]};
      double cs = (e1[0] * e2[0] + e1[1] * e2[1] + e1[2] * e2[2]) /
                  sqrt((e1[0] * e1[0] + e1[1] * e1[1] + e1[2] * e1[2]) *
                       (e2[0] * e2[0] + e2[1] * e2[1] + e2[2] * e2[2]));
      double ang = acos(fmin(fmax(cs, -1.0), 1.0));
      for (int d = 0; d < 3; ++d) N[d] += ang * fn[3 * (size_t)u + d];
    }
  for (int d = 0; d < 3; ++d) vn[3 * (size_t)p + d] = N[d];
}

// ------------------------------------------------------------------ sliced storage

// storage order: one block per window of SLICE_WINDOW storage rows, a thread
// per dof row of the window; the window's dof rows by decreasing length, ties
// by dof (a rank by counting, so the order is the same on every run); rows at
// or beyond nd stay in place
__global__ void k_slice_order(int nd, int npad, const int* __restrict__ rp, int* row, int* pos) {
  __shared__ int len[SLICE_WINDOW];
  int w0 = blockIdx.x * SLICE_WINDOW, t = threadIdx.x, r = w0 + t;
  int n = min(SLICE_WINDOW, max(0, nd - w0));
  len[t] = t < n ? rp[r + 1] - rp[r] : -1;
  __syncthreads();
  if (r >= npad) return;
  if (t >= n) {
    row[r] = r;
    pos[r] = r;
    return;
  }
  int L = len[t], rank = 0;
  for (int j = 0; j < n; ++j) rank += (len[j] > L) || (len[j] == L && j < t);
  pos[r] = w0 + rank;
  row[w0 + rank] = r;
}

// width of each slice of 32 storage rows: longest row, rounded up to 4 blocks;
// the longest row of all
__global__ void k_slice_width(int nd, int ns, const int* __restrict__ rp, const int* __restrict__ row, int* w,
                              int* maxrow) {
  int s = blockIdx.x * blockDim.x + threadIdx.x;
  int m = 0;
  if (s < ns) {
    for (int sr = 32 * s; sr < 32 * s + 32; ++sr) {
      int r = row[sr];
      if (r < nd) m = max(m, rp[r + 1] - rp[r]);
    }
    w[s] = (m + 3) & ~3;
  }
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) atomicMax(maxrow, m);
}

__global__ void k_slice_slots(int ns, const int* __restrict__ w, int* slots) {
  int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s < ns) slots[s] = 32 * w[s];
}

__global__ void k_slice_base64(int ns, const int* __restrict__ pos, long long* base) {
  int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s < ns) base[s] = pos[s];
}

// slot columns of each storage row: its dof row's sorted columns, then padding
// slots pointing at that row
__global__ void k_slice_cols(int nd, int ns, const int* __restrict__ rp, const int* __restrict__ col,
                             const int* __restrict__ w, const long long* __restrict__ base,
                             const int* __restrict__ row, int* scol) {
  long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  int sr = (int)(t >> 5), lane = (int)(t & 31);
  if (sr >= 32 * ns) return;
  int s = sr >> 5, r = row[sr];
  int nb = r < nd ? rp[r + 1] - rp[r] : 0;
  for (int idx = lane; idx < w[s]; idx += 32)
    scol[sliced_slot(base[s], sr, idx)] = idx < nb ? col[rp[r] + idx] : (r < nd ? r : 0);
}

// ------------------------------------------------------------------ host helpers

int read_total(mpm_ctx* c, const int* scan_out, const int* cnt, int n) {
  if (n == 0) return 0;
  MPM_CUDA(cudaMemcpyAsync(c->h_int + 2, scan_out + n - 1, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
  MPM_CUDA(cudaMemcpyAsync(c->h_int + 3, cnt + n - 1, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
  MPM_CUDA(cudaStreamSynchronize(c->stream));
  return c->h_int[2] + c->h_int[3];
}

int read_flag(mpm_ctx* c, int* d_any) {
  MPM_CUDA(cudaMemcpyAsync(c->h_int + 4, d_any, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
  MPM_CUDA(cudaStreamSynchronize(c->stream));
  return c->h_int[4];
}

void tree_refine(mpm_ctx* c, mpm_mesh* m, const int* flag) {
  int n = m->nleaf;
  int* cnt = grow<int>(c, c->tmp[0], n);
  int* pos = grow<int>(c, m->scan, n);
  MPM_LAUNCH(k_child_count<<<grid_for(n, 256), 256, 0, c->stream>>>(n, flag, cnt));
  cub_exclusive_sum_int(c, cnt, pos, n);
  int total = read_total(c, pos, cnt, n);
  uint64_t* okey = grow<uint64_t>(c, m->leaf_tmp_key, total);
  int* olev = grow<int>(c, m->leaf_tmp_lev, total);
  MPM_LAUNCH(k_refine_write<<<grid_for(n, 256), 256, 0, c->stream>>>(n, ptr<uint64_t>(m->leaf_key),
                                                          ptr<int>(m->leaf_lev), flag, pos, m->g.D,
                                                          okey, olev));
  std::swap(m->leaf_key, m->leaf_tmp_key);
  std::swap(m->leaf_lev, m->leaf_tmp_lev);
  m->nleaf = total;
}

void tree_balance(mpm_ctx* c, mpm_mesh* m) {
  int* any = (int*)(c->d_red + 8);
  for (int it = 0; it < 4 * m->g.D + 8; ++it) {
    int n = m->nleaf;
    int* flag = grow<int>(c, m->flag, n);
    MPM_CUDA(cudaMemsetAsync(flag, 0, sizeof(int) * n, c->stream));
    MPM_CUDA(cudaMemsetAsync(any, 0, sizeof(int), c->stream));
    MPM_LAUNCH(k_balance_mark<<<grid_for(n, 256), 256, 0, c->stream>>>(n, ptr<uint64_t>(m->leaf_key),
                                                            ptr<int>(m->leaf_lev), m->g, flag, any));
    if (!read_flag(c, any)) return;
    tree_refine(c, m, flag);
  }
  throw CudaError(MPM_ERR_BALANCE, "octree balance did not settle");
}

}  // namespace

// ------------------------------------------------------------------ the build

// a triangulated body: check its arrays, then its pseudo-normals and bounding box
void tri_setup(mpm_ctx* c, mpm_mesh* m, const mpm_rigid& b) {
  cudaStream_t st = c->stream;
  if (b.ntri <= 0 || b.nvert <= 0 || !b.tri_v || !b.tri_t)
    throw CudaError(MPM_ERR_ARG, "triangulated body: need ntri > 0, nvert > 0 and both arrays");
  std::vector<double> v(3 * (size_t)b.nvert);
  std::vector<int> t(3 * (size_t)b.ntri);
  MPM_CUDA(cudaMemcpyAsync(v.data(), b.tri_v, sizeof(double) * v.size(), cudaMemcpyDeviceToHost, st));
  MPM_CUDA(cudaMemcpyAsync(t.data(), b.tri_t, sizeof(int) * t.size(), cudaMemcpyDeviceToHost, st));
  MPM_CUDA(cudaStreamSynchronize(st));
  for (int i : t)
    if (i < 0 || i >= b.nvert) throw CudaError(MPM_ERR_ARG, "triangulated body: vertex index out of range");
  for (int d = 0; d < 3; ++d) {
    m->tri_lo[d] = 1e300;
    m->tri_hi[d] = -1e300;
  }
  for (int i = 0; i < b.nvert; ++i)
    for (int d = 0; d < 3; ++d) {
      m->tri_lo[d] = std::min(m->tri_lo[d], v[3 * (size_t)i + d]);
      m->tri_hi[d] = std::max(m->tri_hi[d], v[3 * (size_t)i + d]);
    }
  double* fn = grow<double>(c, m->tri_fn, 3 * (size_t)b.ntri);
  double* en = grow<double>(c, m->tri_en, 9 * (size_t)b.ntri);
  double* vn = grow<double>(c, m->tri_vn, 3 * (size_t)b.nvert);
  MPM_LAUNCH(k_tri_fn<<<grid_for(b.ntri, 128), 128, 0, st>>>(b.ntri, b.tri_v, b.tri_t, fn));
  MPM_LAUNCH(k_tri_en<<<grid_for(3LL * b.ntri, 128), 128, 0, st>>>(b.ntri, b.tri_t, fn, en));
  MPM_LAUNCH(k_tri_vn<<<grid_for(b.nvert, 128), 128, 0, st>>>(b.nvert, b.ntri, b.tri_v, b.tri_t, fn, vn));
}

void build_mesh(mpm_ctx* c, mpm_mesh* m, const mpm_domain& dom, const mpm_rigid& body,
                const mpm_adapt& ad, const mpm_material& mat, mpm_points* pts, int flags,
                double cand_extra) {
  cudaStream_t st = c->stream;
  m->built = 0;
  ++m->gen;
  m->dom = dom;
  m->body = body;
  m->ad = ad;
  m->mat = mat;
  Geo& g = m->g;
  g.D = dom.depth_max;
  g.N = 1 << g.D;
  g.L = dom.L;
  g.unit = dom.L / ldexp(1.0, g.D);
  g.scale = ldexp(1.0, g.D) / dom.L;
  int* d_err = c->d_err;
  if (body.kind == 3) tri_setup(c, m, body);
  const Body bv = body_view(m, body);
  MeshCounts* mc = (MeshCounts*)(c->d_red + 50);
  MPM_CUDA(cudaMemsetAsync(mc, 0, sizeof(MeshCounts), st));

  // ---- a1: uniform tree at depth_min, then Sec. 5 refinement + balance
  {
    int n = 1 << (3 * dom.depth_min);
    grow<uint64_t>(c, m->leaf_key, n);
    grow<int>(c, m->leaf_lev, n);
    MPM_LAUNCH(k_tree_uniform<<<grid_for(n, 256), 256, 0, st>>>(n, 3 * (g.D - dom.depth_min), dom.depth_min,
                                                     ptr<uint64_t>(m->leaf_key), ptr<int>(m->leaf_lev)));
    m->nleaf = n;
    if (body.kind != 0 && dom.depth_max > dom.depth_min) {
      int* any = (int*)(c->d_red + 8);
      bool settled = false;
      for (int it = 0; it < 4 * g.D + 8; ++it) {
        int nl = m->nleaf;
        int* flag = grow<int>(c, m->flag, nl);
        MPM_CUDA(cudaMemsetAsync(any, 0, sizeof(int), st));
        MPM_LAUNCH(k_mark_refine<<<grid_for(nl, 256), 256, 0, st>>>(nl, ptr<uint64_t>(m->leaf_key),
                                                         ptr<int>(m->leaf_lev), g, bv, ad.dx_region,
                                                         dom.depth_max, flag, any));
        if (!read_flag(c, any)) {
          settled = true;
          break;
        }
        tree_refine(c, m, flag);
        tree_balance(c, m);
      }
      if (!settled) throw CudaError(MPM_ERR_BALANCE, "octree refinement did not settle");
    }
  }
  int nl = m->nleaf;
  const uint64_t* lkey = ptr<uint64_t>(m->leaf_key);
  const int* llev = ptr<int>(m->leaf_lev);

  // ---- a3: GIMP refinement, in the caller's arrays
  for (SplitRound& r : m->split_log) {
    free_buf(c, r.flag);
    free_buf(c, r.rank);
  }
  m->split_log.clear();
  if (!(flags & 1)) {
    for (int round = 0; round < 32; ++round) {
      int P = pts->count;
      int* flag = grow<int>(c, c->tmp[1], P);
      int* rank = grow<int>(c, c->tmp[2], P);
      MPM_LAUNCH(k_split_flag<<<grid_for(P, 128), 128, 0, st>>>(P, pts->x, pts->lp, pts->l0, lkey, llev, nl, g,
                                                     ad.beta, flag, d_err));
      cub_exclusive_sum_int(c, flag, rank, P);
      int cnt = read_total(c, rank, flag, P);
      if (cnt == 0) break;
      long long np = (long long)P + 7LL * cnt;
      if (np > pts->capacity)
        throw CudaError(MPM_ERR_CAPACITY, "GIMP split needs " + std::to_string(np) +
                                              " points, capacity is " + std::to_string(pts->capacity));
      MPM_LAUNCH(k_split_write<<<grid_for(P, 128), 128, 0, st>>>(P, flag, rank, *pts));
      if (m->record_splits) {
        m->split_log.emplace_back();
        SplitRound& r = m->split_log.back();
        r.P = P;
        r.cnt = cnt;
        MPM_CUDA(cudaMemcpyAsync(grow<int>(c, r.flag, P), flag, sizeof(int) * P, cudaMemcpyDeviceToDevice, st));
        MPM_CUDA(cudaMemcpyAsync(grow<int>(c, r.rank, P), rank, sizeof(int) * P, cudaMemcpyDeviceToDevice, st));
      }
      pts->count = (int)np;
      if (round == 31) throw CudaError(MPM_ERR_SUPPORT, "GIMP split did not settle");
    }
  }
  int P = pts->count;
  m->np = P;

  // ---- a2: nodes, hanging classification, constraints
  {
    uint64_t* ck = grow<uint64_t>(c, c->tmp[3], 8 * (size_t)nl);
    uint64_t* alt = grow<uint64_t>(c, c->tmp[4], 8 * (size_t)nl);
    MPM_LAUNCH(k_corner_keys<<<grid_for(nl, 256), 256, 0, st>>>(nl, lkey, llev, g.D, ck));
    ck = cub_sort_u64(c, ck, alt, 8 * nl, 0, 3 * (g.D + 1));
    uint64_t* nkey = grow<uint64_t>(c, m->node_key, 8 * (size_t)nl);
    int nn = cub_unique_u64(c, ck, nkey, 8 * nl);
    m->nnode = nn;
    int* corner = grow<int>(c, m->corner, 8 * (size_t)nl);
    MPM_LAUNCH(k_corner_ids<<<grid_for(nl, 256), 256, 0, st>>>(nl, lkey, llev, g.D, nkey, nn, corner));
    int* hang = grow<int>(c, m->hang, nn);
    int* owner = grow<int>(c, m->owner, nn);
    MPM_LAUNCH(k_hang<<<grid_for(nn, 256), 256, 0, st>>>(nn, nkey, lkey, llev, nl, g, hang, owner, &mc->nhang));
    NodeView v{nkey, lkey, llev, corner, hang, owner, g.D};
    int* cnt = grow<int>(c, c->tmp[0], nn + 1);
    int* cptr = grow<int>(c, m->cptr, nn + 1);
    MPM_LAUNCH(k_con_count<<<grid_for(nn, 128), 128, 0, st>>>(nn, v, cnt, d_err));
    MPM_CUDA(cudaMemsetAsync(cnt + nn, 0, sizeof(int), st));
    cub_exclusive_sum_int(c, cnt, cptr, nn + 1);
    int ncon = read_total(c, cptr, cnt, nn + 1);
    m->ncon = ncon;
    int* cidx = grow<int>(c, m->cidx, ncon);
    double* cw = grow<double>(c, m->cw, ncon);
    MPM_LAUNCH(k_con_fill<<<grid_for(nn, 128), 128, 0, st>>>(nn, v, cptr, cidx, cw));
    int st2 = check_device_error(c, "node constraints");
    if (st2) throw CudaError(st2, c->err);
  }
  const int* corner = ptr<int>(m->corner);
  const int* cptr = ptr<int>(m->cptr);
  const int* cidx = ptr<int>(m->cidx);
  const double* cw = ptr<double>(m->cw);
  int nn = m->nnode;

  // ---- points: sort by leaf of the centre, gather the step-start state
  {
    int* cell = grow<int>(c, c->tmp[1], P);
    int* idx = grow<int>(c, c->tmp[2], P);
    int* perm = grow<int>(c, m->perm, P);
    int* pcell = grow<int>(c, m->pcell, P);
    MPM_LAUNCH(k_point_cell<<<grid_for(P, 256), 256, 0, st>>>(P, pts->x, g, lkey, nl, cell, idx));
    cub_sort_pairs_int(c, cell, pcell, idx, perm, P, bits_for(nl));
    MPM_LAUNCH(k_gather_points<<<grid_for(P, 256), 256, 0, st>>>(
        P, perm, *pts, grow<double>(c, m->px, 3 * (size_t)P), grow<double>(c, m->plp, 3 * (size_t)P),
        grow<double>(c, m->pl0, 3 * (size_t)P), grow<double>(c, m->pF, 9 * (size_t)P),
        grow<double>(c, m->pbe, 6 * (size_t)P), grow<double>(c, m->pV0, P),
        grow<double>(c, m->pmass, P), grow<double>(c, m->pE, P), grow<double>(c, m->pys, P),
        pts->v ? grow<double>(c, m->pv, 3 * (size_t)P) : nullptr));
    m->has_v = pts->v != nullptr;
  }

  // ---- a4: discrete GIMP basis
  int* nsup = grow<int>(c, m->nsup, P);
  int* sidx = grow<int>(c, m->sidx, (size_t)P * MAXS);
  double* S = grow<double>(c, m->S, (size_t)P * MAXS);
  double* dS = grow<double>(c, m->dS, (size_t)P * MAXS * 3);
  int* pop = grow<int>(c, m->populated, nl);
  double* betaK = grow<double>(c, m->betaK, nl);
  MPM_CUDA(cudaMemsetAsync(pop, 0, sizeof(int) * nl, st));
  MPM_CUDA(cudaMemsetAsync(betaK, 0, sizeof(double) * nl, st));
  int* active = grow<int>(c, c->tmp[0], nn);
  MPM_CUDA(cudaMemsetAsync(active, 0, sizeof(int) * nn, st));
  MPM_LAUNCH_P(MPM_PROF_BASIS, k_basis<<<grid_for(P, BW), 32 * BW, 0, st>>>(P, g, ptr<double>(m->px), ptr<double>(m->plp),
                                               ptr<double>(m->pE), lkey, llev, nl, corner, cptr, cidx,
                                               cw, nsup, sidx, S, dS, active, pop,
                                               (unsigned long long*)betaK, d_err));
  {
    int e = check_device_error(c, "GIMP basis");
    if (e) throw CudaError(e, c->err);
  }
  // active nodes -> dofs (Morton order)
  {
    int* pos = grow<int>(c, c->tmp[1], nn);
    cub_exclusive_sum_int(c, active, pos, nn);
    int nd = read_total(c, pos, active, nn);
    m->ndof = nd;
    int* node_dof = grow<int>(c, m->node_dof, nn);
    int* dof_node = grow<int>(c, m->dof_node, nd);
    MPM_LAUNCH(k_number_dofs<<<grid_for(nn, 256), 256, 0, st>>>(nn, active, pos, node_dof, dof_node));
    Planes pl{};
    pl.n = dom.nbc;
    for (int b = 0; b < dom.nbc; ++b) {
      pl.axis[b] = dom.bc_axis[b];
      pl.pos[b] = (int)floor(dom.bc_pos[b] * g.scale + 0.5);
      pl.mask[b] = dom.bc_mask[b];
    }
    MPM_LAUNCH(k_dof_mask<<<grid_for(nd, 256), 256, 0, st>>>(nd, dof_node, ptr<uint64_t>(m->node_key), pl,
                                                  grow<int>(c, m->dof_mask, nd)));
  }
  int nd = m->ndof;
  const int* node_dof = ptr<int>(m->node_dof);

  // ---- a6 (faces): boundary elements and ghost faces
  int nf = 0;
  {
    int* isB = grow<int>(c, m->isB, nl);
    MPM_LAUNCH(k_boundary_elements<<<grid_for(nl, 256), 256, 0, st>>>(nl, lkey, llev, g, pop, isB));
    if (mat.ghost_on) {
      int* flag = grow<int>(c, c->tmp[0], 6 * (size_t)nl);
      int* pos = grow<int>(c, c->tmp[1], 6 * (size_t)nl);
      MPM_LAUNCH(k_ghost_face_flag<<<grid_for(6LL * nl, 256), 256, 0, st>>>(nl, lkey, llev, g, pop, isB, flag));
      cub_exclusive_sum_int(c, flag, pos, 6 * nl);
      nf = read_total(c, pos, flag, 6 * nl);
      int* face = grow<int>(c, m->gface, 4 * (size_t)nf);
      MPM_LAUNCH(k_ghost_face_write<<<grid_for(6LL * nl, 256), 256, 0, st>>>(nl, lkey, llev, g, flag, pos, face));
      MPM_LAUNCH(k_ghost_face_dofs<<<grid_for(nf, 128), 128, 0, st>>>(nf, face, corner, cptr, cidx, node_dof,
                                                          grow<int>(c, m->gdof, (size_t)nf * MAXG),
                                                          grow<int>(c, m->gn, nf), d_err));
    }
    m->nghost = nf;
  }

  // ---- a5: sources of every row, then the pattern
  {
    int* off = grow<int>(c, c->tmp[0], P + 1);
    MPM_CUDA(cudaMemsetAsync(off + P, 0, sizeof(int), st));
    // nsup[P] is not defined: scan P entries and read the total
    cub_exclusive_sum_int(c, nsup, off, P);
    long long npt = read_total(c, off, nsup, P);
    long long total = npt + (long long)nf * MAXG;
    uint64_t* keys = grow<uint64_t>(c, m->src_key, total);
    uint64_t* alt = grow<uint64_t>(c, c->tmp[3], total);
    // rows below 2^bits - 1: the unused face slots' row of ones sorts last.  An
    // odd number of passes starts in the scratch buffer, to end in the keys
    int bits = bits_for(nd);
    bool odd = ((bits + 7) / 8) & 1;
    uint64_t *first = odd ? alt : keys, *second = odd ? keys : alt;
    MPM_LAUNCH(k_point_sources<<<grid_for(P, 8), 256, 0, st>>>(P, nsup, node_dof, off, sidx, first, mc));
    if (nf) {
      // unused face slots keep an out-of-range row so that they sort last
      MPM_CUDA(cudaMemsetAsync(first + npt, 0xff, sizeof(uint64_t) * (size_t)nf * MAXG, st));
      MPM_LAUNCH(k_src_keys_faces<<<grid_for((long long)nf * MAXG, 256), 256, 0, st>>>(
          nf, P, ptr<int>(m->gn), ptr<int>(m->gdof), npt, first));
    }
    uint64_t* sorted = cub_sort_u64(c, first, second, (int)total, 32, 32 + bits);
    if (sorted != keys)
      MPM_CUDA(cudaMemcpyAsync(keys, sorted, sizeof(uint64_t) * (size_t)total, cudaMemcpyDeviceToDevice, st));
    long long* sptr = grow<long long>(c, m->src_ptr, nd + 1);
    MPM_CUDA(cudaMemsetAsync(sptr, 0, sizeof(long long) * (nd + 1), st));
    MPM_LAUNCH(k_src_ptr<<<grid_for(total, 256), 256, 0, st>>>(total, keys, nd, sptr));
    m->nsrc = total;
    int* rowcnt = grow<int>(c, m->rowcnt, nd + 1);
    int* rp = grow<int>(c, m->row_ptr, nd + 1);
    MPM_CUDA(cudaMemsetAsync(rowcnt + nd, 0, sizeof(int), st));
    PatternSrc ps{P, sptr, keys, nsup, sidx, ptr<int>(m->gn), ptr<int>(m->gdof)};
    int* stage = grow<int>(c, c->tmp[3], (size_t)nd * PSHORT);  // the sort's scratch is free again
    int lblocks = std::min(grid_for(nd, 32 * PLW), 152 * 9);
    MPM_LAUNCH_P(MPM_PROF_PATTERN, k_pattern_rows<<<grid_for(nd, PW), 32 * PW, 0, st>>>(nd, ps, rowcnt, stage));
    MPM_LAUNCH_P(MPM_PROF_PATTERN, k_pattern_long<<<lblocks, 32 * PLW, 0, st>>>(nd, ps, rowcnt, stage, nullptr,
                                                                               nullptr, d_err));
    cub_exclusive_sum_int(c, rowcnt, rp, nd + 1);
    int nnzb = read_total(c, rp, rowcnt, nd + 1);
    {
      int e = check_device_error(c, "block pattern");
      if (e) throw CudaError(e, c->err);
    }
    m->nnzb = nnzb;
    int* col = grow<int>(c, m->col, nnzb);
    MPM_LAUNCH_P(MPM_PROF_PATTERN, k_pattern_write<<<grid_for(nd, 8), 256, 0, st>>>(nd, rp, stage, col));
    MPM_LAUNCH_P(MPM_PROF_PATTERN, k_pattern_long<<<lblocks, 32 * PLW, 0, st>>>(nd, ps, rowcnt, stage, rp, col,
                                                                               d_err));
    // sliced storage of the stiffness
    int ns = (nd + 31) / 32;
    m->nslice = ns;
    int* sw = grow<int>(c, m->slice_w, ns + 1);
    int* slots = grow<int>(c, c->tmp[1], ns + 1);
    int* spos = grow<int>(c, c->tmp[2], ns + 1);
    int* srow = grow<int>(c, m->srow, 32 * (size_t)ns);
    int* rpos = grow<int>(c, m->spos, 32 * (size_t)ns);
    MPM_LAUNCH(k_slice_order<<<(32 * ns + SLICE_WINDOW - 1) / SLICE_WINDOW, SLICE_WINDOW, 0, st>>>(nd, 32 * ns, rp, srow, rpos));
    MPM_LAUNCH(k_slice_width<<<grid_for(ns, 256), 256, 0, st>>>(nd, ns, rp, srow, sw, &mc->maxrow));
    MPM_LAUNCH(k_slice_slots<<<grid_for(ns, 256), 256, 0, st>>>(ns, sw, slots));
    MPM_CUDA(cudaMemsetAsync(slots + ns, 0, sizeof(int), st));
    cub_exclusive_sum_int(c, slots, spos, ns + 1);
    // the widths of a small mesh on the host, where the resident Krylov solves
    // divide the rows among the SMs
    m->slice_w_host.resize(ns <= RESIDENT_SLICES ? ns : 0);
    if (!m->slice_w_host.empty())
      MPM_CUDA(cudaMemcpyAsync(m->slice_w_host.data(), sw, sizeof(int) * ns, cudaMemcpyDeviceToHost, st));
    m->nslot = read_total(c, spos, slots, ns + 1);
    long long* sb = grow<long long>(c, m->slice_base, ns + 1);
    MPM_LAUNCH(k_slice_base64<<<grid_for(ns + 1, 256), 256, 0, st>>>(ns + 1, spos, sb));
    int* scol = grow<int>(c, m->scol, m->nslot);
    MPM_LAUNCH(k_slice_cols<<<grid_for(32LL * 32 * ns, 256), 256, 0, st>>>(nd, ns, rp, col, sw, sb, srow, scol));
  }
  const int* rp = ptr<int>(m->row_ptr);
  const int* col = ptr<int>(m->col);

  // ---- a6 (matrix): ghost coefficients
  {
    double* kg = grow<double>(c, m->kg, m->nnzb);
    MPM_CUDA(cudaMemsetAsync(kg, 0, sizeof(double) * m->nnzb, st));
    if (nf) {
      double* gJ = grow<double>(c, m->gJ, 4 * (size_t)nf * MAXG);
      double* gco = grow<double>(c, m->gcoef, nf);
      MPM_LAUNCH(k_ghost_jumps<<<grid_for(nf, 4), 128, 0, st>>>(nf, g, mat.kappa, ptr<int>(m->gface), lkey, llev,
                                                               betaK, ptr<int>(m->gdof), ptr<int>(m->gn),
                                                               corner, cptr, cidx, cw, node_dof, gJ, gco));
      MPM_LAUNCH(k_ghost_rows<<<grid_for(nd, 8), 256, 0, st>>>(nd, P, ptr<long long>(m->src_ptr),
                                                              ptr<uint64_t>(m->src_key), ptr<int>(m->gdof),
                                                              ptr<int>(m->gn), gJ, gco, rp, col, kg));
    }
  }

  // ---- gravity force at load 1: f_ext,v = sum_p S_vp m_p g
  {
    double* fext = grow<double>(c, m->fext, 3 * (size_t)nd);
    MPM_CUDA(cudaMemsetAsync(fext, 0, sizeof(double) * 3 * nd, st));
    if (mat.g[0] != 0.0 || mat.g[1] != 0.0 || mat.g[2] != 0.0)
      MPM_LAUNCH(k_fext_rows<<<grid_for(nd, 8), 256, 0, st>>>(nd, P, ptr<long long>(m->src_ptr),
                                                             ptr<uint64_t>(m->src_key), S,
                                                             ptr<double>(m->pmass), mat.g[0], mat.g[1],
                                                             mat.g[2], fext));
  }

  // ---- contact candidates: domains with a corner within 4 finest cells of the
  // body (plus cand_extra: a free body's motion over the step)
  m->ncand = 0;
  m->nct = 0;
  if (mat.contact_on && body.kind != 0) {
    int* flag = grow<int>(c, c->tmp[0], P);
    int* pos = grow<int>(c, c->tmp[1], P);
    MPM_LAUNCH(k_cand_flag<<<grid_for(P, 256), 256, 0, st>>>(P, ptr<double>(m->px), ptr<double>(m->plp), bv,
                                                  4.0 * g.unit + cand_extra, flag));
    cub_exclusive_sum_int(c, flag, pos, P);
    int nc = read_total(c, pos, flag, P);
    m->ncand = nc;
    if (nc) {
      int* cand = grow<int>(c, m->cand, nc);
      MPM_LAUNCH(k_cand_write<<<grid_for(P, 256), 256, 0, st>>>(P, flag, pos, cand));
      MPM_LAUNCH(k_cand_basis<<<grid_for(8LL * nc, 128), 128, 0, st>>>(
          nc, cand, g, ptr<double>(m->px), ptr<double>(m->plp), lkey, llev, nl, corner, cptr, cidx,
          cw, node_dof, grow<int>(c, m->cb_n, 8 * (size_t)nc),
          grow<int>(c, m->cb_idx, 8 * (size_t)nc * MAXCB),
          grow<double>(c, m->cb_phi, 8 * (size_t)nc * MAXCB),
          grow<double>(c, m->cb_y0, 24 * (size_t)nc), d_err));
      // the transpose of the corner basis, rows with their (corner, entry)
      // lists in sorted order, for the contact row gather
      long long nk = 8LL * nc * MAXCB;
      uint64_t* keys = grow<uint64_t>(c, c->tmp[4], nk);
      uint64_t* alt = grow<uint64_t>(c, c->tmp[5], nk);
      MPM_LAUNCH(k_ct_keys<<<grid_for(nk, 256), 256, 0, st>>>(8 * nc, ptr<int>(m->cb_n), ptr<int>(m->cb_idx), keys));
      // listed in ascending order of the lower 32 bits: sorted by the row alone
      keys = cub_sort_u64(c, keys, alt, (int)nk, 32, 32 + bits_for(nd));
      int* cflag = grow<int>(c, c->tmp[6], nk + 1);
      int* cpos = grow<int>(c, c->tmp[7], nk + 1);
      MPM_LAUNCH(k_ct_flag<<<grid_for(nk, 256), 256, 0, st>>>(nk, keys, cflag));
      cub_exclusive_sum_int(c, cflag, cpos, (int)nk);
      int nrow = read_total(c, cpos, cflag, (int)nk);
      m->nct = nrow;
      MPM_LAUNCH(k_ct_write<<<grid_for(nk, 256), 256, 0, st>>>(
          nk, keys, cflag, cpos, nrow, grow<int>(c, m->ct_row, nrow + 1), grow<int>(c, m->ct_ptr, nrow + 1),
          grow<int>(c, m->ct_ent, nk)));
    }
  }

  // FP32 copies of the basis for the mixed-precision path are made on demand
  // by the assembly
  MeshCounts* h = (MeshCounts*)c->h_red;
  long long* used = (long long*)(c->h_red + 8);
  MPM_CUDA(cudaMemcpyAsync(h, mc, sizeof(MeshCounts), cudaMemcpyDeviceToHost, st));
  MPM_CUDA(cudaMemcpyAsync(used, ptr<long long>(m->src_ptr) + m->ndof, sizeof(long long), cudaMemcpyDeviceToHost, st));
  MPM_CUDA(cudaStreamSynchronize(st));
  m->nsrc_used = *used;
  m->npair = (long long)h->npair;
  m->maxs = h->maxs;
  m->maxrow = h->maxrow;
  m->nhang = h->nhang;
  m->built = 1;
}

Body body_view(const mpm_mesh* m, const mpm_rigid& b) {
  Body v{};
  v.b = b;
  if (b.kind == 3) {
    v.fn = ptr<double>(m->tri_fn);
    v.en = ptr<double>(m->tri_en);
    v.vn = ptr<double>(m->tri_vn);
    for (int d = 0; d < 3; ++d) {
      v.lo[d] = m->tri_lo[d];
      v.hi[d] = m->tri_hi[d];
    }
  }
  return v;
}

}  // namespace mpm
