// Whole Krylov solves in one cooperative launch, for meshes whose iteration is
// bound by latency and not by HBM.  A launch per vector update and per SpMV
// costs 2 to 4 us each, and the row-per-thread SpMV of the large meshes puts
// 2,000 rows on 8 of the 152 SMs (one 256-row block each, FP64 at 2 lanes per
// clock).  Here every worker block owns a fixed, balanced range of storage
// rows for the whole solve and keeps their state (and, where it fits, their
// blocks of K) in shared memory; only the vector that K multiplies goes
// through the L2.  The blocks meet twice (PCG) or five times (BiCGStab) per
// iteration in a grid-wide sum taken by the last block, the coordinator, which
// also forms the solve's scalars and decides when it ends.  The sums run in a
// fixed order for a given device, so a solve is the same bit for bit on every
// run.  Bound by: the sums (2.4 us, 3.1 us where a vector is published too) on
// small meshes, the FP64 rate (9 FMAs a block) or the L2 above.
//
// us per iteration, launches per iteration -> resident (up to 10 k rows the
// launches as they were before this file, then as they are):
//   rows (blocks)      PCG FP64       PCG FP32       BiCGStab FP64    FP32
//      858 (67 k)      128 -> 13       50 -> 9         275 -> 27      104 -> 20
//    2,026 (178 k)     144 -> 15       51 -> 10        308 -> 32      101 -> 21
//   10,446 (1.04 M)    146 -> 36       52 -> 16        320 -> 74      102 -> 35
//   36,935 (3.99 M)    173 -> 103      97 -> 55        271 -> 206     125 -> 114
//   58,052 (6.29 M)    202 -> 150     103 -> 69        376 -> 299     155 -> 144
//   78,044 (8.57 M)    212 -> 194     110 -> 84        408 -> 410     188 -> 178
//   96,364 (10.7 M)    267 -> 230     117 -> 100       530 (state     209 -> 207
//  110,690 (12.3 M)    278 (281)      123 (129)        550  too       230 (264)
//  121,837 (13.6 M)    345 (342)      131 (137)        646  large)    277 (423)
// (in brackets: resident, beyond the limit RESIDENT_SLICES)
#pragma once
#include "mpm_sliced.cuh"

namespace mpm {

constexpr int RK_T = 512;           // threads per block, one block per SM
constexpr int RK_QUADS = RK_T / 4;  // quads of storage rows worked on at a time
constexpr int RK_NBUF = 6;          // rotating sets of sum slots and messages
constexpr int RK_NV = 2;            // values per grid sum
constexpr int RK_COPY = 16;         // copies of a message, a line each
constexpr int RK_POLLS = 1 << 21;   // bound of a wait unless the context sets another (about a second)
constexpr int RK_SMEM = 200 * 1024;  // dynamic shared memory of a block (at most)
constexpr int RK_ROW = 64;          // slots' worth of a quad's own vector work

// slots of a launch of G blocks: the sums' partials, then the messages
__host__ __device__ constexpr size_t rk_slot_words(int G) {
  return (size_t)RK_NBUF * (RK_NV * (size_t)G + 16 * RK_COPY);
}

// A slot that holds no value yet.  All bits set is a NaN that rk_pack never
// writes, so a slot's 8 bytes carry the value and the fact that it is there;
// two more NaNs tell the workers to stop.
constexpr unsigned long long RK_EMPTY = ~0ULL, RK_STOP = 0xfff8000000000010ULL;

__device__ inline unsigned long long rk_pack(double v) {
  return v != v ? 0x7ff8000000000000ULL : (unsigned long long)__double_as_longlong(v);
}
__device__ inline unsigned long long rk_ld(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ inline unsigned long long rk_ld_acquire(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ inline void rk_st(unsigned long long* p, unsigned long long v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ inline void rk_fence() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }

// loads of a vector that other SMs write during the launch (past the L1)
__device__ inline void ld4_cg(const float* p, float* v) {
  float4 t = __ldcg(reinterpret_cast<const float4*>(p));
  v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
__device__ inline void ld4_cg(const double* p, double* v) {
  double2 a = __ldcg(reinterpret_cast<const double2*>(p)), b = __ldcg(reinterpret_cast<const double2*>(p) + 1);
  v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}

// what a launch works with (host side: resident_plan)
struct RkPlan {
  int G;              // blocks: G - 1 workers and the coordinator
  int rows;           // most rows of a worker
  int groups;         // most groups of 4 blocks x 4 rows of a worker, if K is kept in shared memory (else 0)
  int smem;           // dynamic shared memory
  int polls;          // bound of a wait; one that runs out sets Scal::late, and the call fails
};

// elements of a group of 16 blocks in shared memory, padded so that the quad
// lanes of a warp, which read neighbouring groups, meet no bank twice
template <class T>
__host__ __device__ constexpr int rk_group() {
  return sizeof(T) == 8 ? 146 : 144;
}

// An FP64 instruction occupies the quarter of the SM that its warp runs on for
// 64 cycles (76 for an addition) here, whatever the number of active lanes and
// whatever it depends on.  So FP64 work is packed into as few warps'
// instructions as possible and laid on warps of different quarters.
struct RkShared {
  double red[RK_NV][RK_T];
  double scal[2];  // the scalars the block's threads use next
  int stop;
  int q0, q1;
};

// One block's side of the grid sums.  A worker posts its partial sums in its
// own slots; the coordinator reads them all, and answers with two scalars or
// a stop in a message (RK_COPY copies, so that the waiting workers do not all
// poll one line; with every block reading every slot the polls alone slowed
// the L2 down fivefold).  Slots and messages rotate through RK_NBUF sets.  A
// worker empties its slots two sums later (its answer to the sum between
// shows that they were read), the coordinator its message when the next sum
// is complete; a set comes round again RK_NBUF sums later, and at least every
// third sum is fenced, so nobody meets a stale value.
//
// A fenced sum hands the vectors that the blocks stored before it to all of
// them: every worker fences and posts slot 0 (release); the coordinator's lanes
// that saw the slots fence (acquire) and meet at its barrier; each lane that
// answers fences again and stores its message (release), which covers what the
// other lanes saw; the workers load its second word with acquire and meet at
// their barrier.
struct RkGrid {
  unsigned long long* slot;
  int* late;
  int G, me, polls, k;
  __device__ unsigned long long* part(int k_) const {
    return slot + (size_t)(k_ % RK_NBUF) * RK_NV * G;
  }
  __device__ unsigned long long* msg(int k_, int copy) const {
    return slot + (size_t)RK_NBUF * RK_NV * G + ((size_t)(k_ % RK_NBUF) * RK_COPY + copy) * 16;
  }
};

// finite and positive, at most thr (both not negative), finite: on the bits
__device__ inline bool rk_positive(double v) {
  long long b = __double_as_longlong(v);
  return b > 0 && b < 0x7ff0000000000000LL;
}
__device__ inline bool rk_at_most(double v, double thr) {
  return (unsigned long long)__double_as_longlong(v) <= (unsigned long long)__double_as_longlong(thr);
}
__device__ inline bool rk_finite(double v) {
  return (__double_as_longlong(v) & 0x7ff0000000000000LL) != 0x7ff0000000000000LL;
}

// s f / d for the factor inv = f / d, formed ahead of the sum s (a division in
// line takes some 0.3 us); for a d so small that inv overflows the quotient first
__device__ inline double rk_quotient(double s, double d, double f, double inv) {
  return rk_finite(inv) ? s * inv : s / d * f;
}

// worker: posts the block's sums of v[0..NV) (one value per thread t < n; a
// warp per value adds them up from shared memory) and waits for the answer,
// left in sh.scal and sh.stop.  fence: the block's global stores before the
// call are seen by every block's loads after it.  Ends with a __syncthreads.
template <int NV>
__device__ inline void rk_sum(RkGrid& g, RkShared& sh, const double* v, int n, bool fence) {
  const int t = threadIdx.x, w = t >> 5, l = t & 31;
  if (t < n) {
#pragma unroll
    for (int i = 0; i < NV; ++i) sh.red[i][t] = v[i];
  }
  __syncthreads();
  if (w < NV) {
    if (fence && t == 0) rk_fence();
    double s = l < n ? sh.red[w][l] : 0.0;
    for (int j = l + 32; j < n; j += 32) s += sh.red[w][j];
    for (int o = n > 16 ? 16 : n > 8 ? 8 : n > 4 ? 4 : n > 2 ? 2 : n > 1 ? 1 : 0; o > 0; o >>= 1)
      s += __shfl_xor_sync(0xffffffffu, s, o);
    if (l == 0) {
      rk_st(g.part(g.k) + (size_t)w * g.G + g.me, rk_pack(s));
      if (w == 0) {
        if (g.k > 1) {
#pragma unroll
          for (int i = 0; i < RK_NV; ++i) rk_st(g.part(g.k + RK_NBUF - 2) + (size_t)i * g.G + g.me, RK_EMPTY);
        }
        const unsigned long long* m = g.msg(g.k, g.me % RK_COPY);
        unsigned long long a = RK_EMPTY, b = RK_EMPTY;
        for (int p = 0; p < g.polls; ++p) {
          a = rk_ld(m);
          b = fence ? rk_ld_acquire(m + 1) : rk_ld(m + 1);
          if (a != RK_EMPTY && b != RK_EMPTY) break;
        }
        sh.scal[0] = __longlong_as_double((long long)a);
        sh.scal[1] = __longlong_as_double((long long)b);
        bool none = a == RK_EMPTY || b == RK_EMPTY;
        if (none) *g.late = 1;  // this block leaves with its rows as they are
        sh.stop = none ? 1 : (b >> 4) == (RK_STOP >> 4) ? (int)(b & 15) : 0;
      }
    }
  }
  __syncthreads();
  ++g.k;
}

constexpr int RK_CT = 32 * RK_NV;  // threads of the coordinator, a warp per value

// coordinator: the sums of the workers' slots, in slot order per lane and by a
// fixed tree over the lanes, in every thread; false when a wait ran out
template <int NV>
__device__ inline bool rk_collect(const RkGrid& g, RkShared& sh, double* s, bool fence) {
  const int t = threadIdx.x, w = t >> 5, l = t & 31, W = g.G - 1;
  constexpr int PU = 5;  // slots of a lane whose loads are in flight together
  bool late = false;
  double x = 0.0;
  if (w < NV) {
    const unsigned long long* set = g.part(g.k) + (size_t)w * g.G;
    for (int j0 = l; j0 < W; j0 += 32 * PU) {
      unsigned long long u[PU];
#pragma unroll
      for (int h = 0; h < PU; ++h) u[h] = j0 + 32 * h < W ? RK_EMPTY : 0ULL;
      for (int n = 0;; ++n) {
        bool all = true;
#pragma unroll
        for (int h = 0; h < PU; ++h)
          if (u[h] == RK_EMPTY) u[h] = rk_ld(set + j0 + 32 * h);
#pragma unroll
        for (int h = 0; h < PU; ++h) all = all && u[h] != RK_EMPTY;
        if (all) break;
        if (n >= g.polls) {
          late = true;
          break;
        }
      }
#pragma unroll
      for (int h = 0; h < PU; ++h)
        if (h == 0 || 32 * h < W) x += __longlong_as_double((long long)u[h]);
    }
    if (fence && w == 0) rk_fence();
    x = warp_sum(x);
    late = __any_sync(0xffffffffu, late);
    if (l == 0) {
      sh.red[w][g.k & 1] = x;
      sh.red[w][2 + (g.k & 1)] = late ? 1.0 : 0.0;
    }
  }
  asm volatile("bar.sync 1, %0;" ::"n"(RK_CT) : "memory");
  bool ok = true;
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    s[i] = sh.red[i][g.k & 1];
    ok = ok && __double_as_longlong(sh.red[i][2 + (g.k & 1)]) == 0;
  }
  if (!ok && t == 0) *g.late = 1;
  return ok;
}

// coordinator: the answer to the sum just collected, `fence` as there (stop: 0
// go on, else the code the workers find in sh.stop)
__device__ inline void rk_tell(RkGrid& g, double a, double b, int stop, bool fence) {
  const int t = threadIdx.x;
  if (t < RK_COPY) {
    unsigned long long* m = g.msg(g.k, t);
    if (fence) rk_fence();  // (no store of this warp is under way: some 0.1 us)
    rk_st(m, rk_pack(a));
    rk_st(m + 1, stop ? RK_STOP | (unsigned long long)stop : rk_pack(b));
    if (g.k > 0) {
      unsigned long long* o = g.msg(g.k + RK_NBUF - 1, t);
      rk_st(o, RK_EMPTY);
      rk_st(o + 1, RK_EMPTY);
    }
  }
  __syncwarp();
  ++g.k;
}

// The quads (4 storage rows) are dealt out to the W workers by their block
// slots plus a constant for the rows' own vector work, so that every worker
// gets about the same time.  Worker b starts at rk_start(b) (the search for
// the slice is given: `lo` is the last slice whose cost before it, the sum of
// 32 w + 8 RK_ROW over the slices, is at most total b / W).
__host__ __device__ inline int rk_start(long long want, int lo, long long before, int w) {
  long long per = 4LL * w + RK_ROW, off = (want - before + per - 1) / per;
  return 8 * lo + (int)(off < 8 ? off : 8);
}
__device__ inline void rk_range(const Sliced& S, int ns, int W, int me, RkShared& sh) {
  if (threadIdx.x < 2) {
    int b = me + threadIdx.x;
    auto before = [&](int s) { return S.base[s] + 8LL * RK_ROW * s; };
    long long want = before(ns) * b / W;
    int lo = 0, hi = ns;
    while (hi - lo > 1) {
      int mid = (lo + hi) >> 1;
      if (before(mid) <= want)
        lo = mid;
      else
        hi = mid;
    }
    int q = b >= W ? 8 * ns : rk_start(want, lo, before(lo), S.w[lo]);
    if (threadIdx.x == 0)
      sh.q0 = q;
    else
      sh.q1 = q;
  }
  __syncthreads();
}

// A worker's rows: their dof rows, their blocks (in shared memory or in place)
// and the product with a vector.
template <class T>
struct RkRows {
  static constexpr int KLM = 32;
  Sliced S;
  const T* Kg;
  int nd, q0, nr, R;    // first quad, rows, stride of the shared vectors
  bool keep;
  int* id;              // dof row of each row (-1: padding)
  int* gb;              // first group of each quad (kept K)
  T* Ks;
  int* Cs;
  T (*sy)[RK_T];

  // carves the shared memory: nv vectors of R x 3 and the 3x3 inverses follow
  __device__ T* init(const Sliced& S_, const T* K_, int nd_, const RkPlan& pl, const RkShared& sh, T (*sy_)[RK_T],
                     unsigned char* mem, int nv) {
    S = S_;
    Kg = K_;
    nd = nd_;
    q0 = sh.q0;
    nr = 4 * (sh.q1 - q0);
    R = pl.rows;
    sy = sy_;
    keep = pl.groups > 0;
    Ks = (T*)mem;
    T* vec = Ks + (size_t)pl.groups * rk_group<T>();
    Cs = (int*)(vec + (size_t)R * (3 * nv + 9));
    id = Cs + 16 * (size_t)pl.groups;
    gb = id + R;
    const int t = threadIdx.x;
    for (int i = t; i < nr; i += RK_T) {
      int row = S.row[4 * q0 + i];
      id[i] = row < nd ? row : -1;
    }
    if (keep) {
      // (a serial count over at most R / 4 quads of few slices)
      if (t == 0) {
        int n = 0;
        for (int q = 0; 4 * q < nr; ++q) {
          gb[q] = n;
          n += S.w[(q0 + q) >> 3] >> 2;
        }
      }
      __syncthreads();
      for (int q = t >> 5; 4 * q < nr; q += RK_T / 32) {
        int qq = q0 + q, s = qq >> 3, ln = 4 * (qq & 7), W = S.w[s];
        long long b0 = S.base[s];
        size_t plane = (size_t)32 * W;
        // a lane per block of the group's 16: 9 planes of 16 consecutive entries
        for (int u = t & 31; u < 16 * (W >> 2); u += 32) {
          int k4 = u >> 4, e16 = u & 15;
          size_t off = ((size_t)k4 * 32 + ln) * 4 + e16;
          T* d = Ks + (size_t)(gb[q] + k4) * rk_group<T>() + e16;
          for (int e = 0; e < 9; ++e) d[16 * e] = Kg[9 * b0 + e * plane + off];
          Cs[16 * (gb[q] + k4) + e16] = S.scol[b0 + off];
        }
      }
    }
    __syncthreads();
    return vec;
  }

  // rows [c0, c0 + 4 nq) of K x (nq <= RK_QUADS): the quad lanes (4 threads,
  // one per row) of a quad take its groups in turn; `get` adds them up.
  // Contains one __syncthreads; the caller separates two calls.
  __device__ void mul(const T* x, int c0, int nq) const {
    const int t = threadIdx.x, KL = min(KLM, RK_QUADS / nq), ql = t >> 2, q = ql / KL, kl = ql - q * KL;
    if (q < nq) {
      T a[3] = {(T)0, (T)0, (T)0};
      int qq = (c0 >> 2) + q, gq = q0 + qq, s = gq >> 3, ln = 4 * (gq & 7) + (t & 3), W = S.w[s];
      long long b0 = S.base[s];
      const T* Kb = Kg + 9 * b0;
      const int* cb = S.scol + b0;
      size_t plane = (size_t)32 * W;
      for (int k4 = kl; k4 < (W >> 2); k4 += KL) {
        int4 c;
        T v[9][4];
        if (keep) {
          size_t o = (size_t)(gb[qq] + k4);
          c = reinterpret_cast<const int4*>(Cs)[4 * o + (t & 3)];
          const T* d = Ks + o * rk_group<T>() + 4 * (t & 3);
#pragma unroll
          for (int e = 0; e < 9; ++e) ld4(d + 16 * e, v[e]);
        } else {
          size_t off = ((size_t)k4 * 32 + ln) * 4;
          c = *reinterpret_cast<const int4*>(cb + off);
#pragma unroll
          for (int e = 0; e < 9; ++e) ld4(Kb + e * plane + off, v[e]);
        }
        int cc[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          T xv[4];
          ld4_cg(x + 4 * (size_t)cc[j], xv);
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            // (FP64 nested: its rate is the bound; FP32 with one rounding of the
            // long sum a block, as sliced_row)
            if constexpr (sizeof(T) == 8)
              a[d] = fma(v[3 * d + 2][j], xv[2], fma(v[3 * d + 1][j], xv[1], fma(v[3 * d][j], xv[0], a[d])));
            else
              a[d] += fma(v[3 * d + 2][j], xv[2], fma(v[3 * d + 1][j], xv[1], v[3 * d][j] * xv[0]));
          }
        }
      }
#pragma unroll
      for (int d = 0; d < 3; ++d) sy[d][t] = a[d];
    }
    __syncthreads();
  }
  // Adds up the last product: f(i, c, y) with component c of row i (of the
  // 4 nq), on thread (4 i + c) % RK_T.  With few rows, up to 8 threads of a
  // warp add the quad lanes of one value.
  template <class F>
  __device__ void each(int nq, F f) const {
    const int t = threadIdx.x, KL = min(KLM, RK_QUADS / nq), SL = nq <= 4 ? 8 : nq <= 8 ? 4 : nq <= 16 ? 2 : 1;
    if (SL > 1) {
      // value v of the 16 nq, its SL threads neighbours
      int v = t / SL, sub = t - v * SL, i = v >> 2, c = min(v & 3, 2);
      T y = (T)0;
      if (v < 16 * nq) {
        const T* p = sy[c] + 4 * (i >> 2) * KL + (i & 3);
        for (int k = sub; k < KL; k += SL) y += p[4 * k];
      }
      for (int o = SL >> 1; o > 0; o >>= 1) y += __shfl_xor_sync(0xffffffffu, y, o);
      __syncthreads();
      if (v < 16 * nq && sub == 0) sy[0][v] = y;
      __syncthreads();
      if (t < 16 * nq && (t & 3) < 3) f(t >> 2, t & 3, sy[0][t]);
    } else {
      for (int u = t; u < 16 * nq; u += RK_T) {
        int i = u >> 2, c = u & 3;
        if (c == 3) continue;
        const T* p = sy[c] + 4 * (i >> 2) * KL + (i & 3);
        T y = p[0];
        for (int k = 1; k < KL; ++k) y += p[4 * k];
        f(i, c, y);
      }
    }
  }
};

// component c of D r, r held component by component by the threads 4 i + c of
// row i (entry e of the row's inverse at D[e R]); every lane of the warp calls
template <class T>
__device__ inline T rk_dinv(const T* D, int R, int c, T r) {
  T r0 = __shfl_sync(0xffffffffu, r, 0, 4), r1 = __shfl_sync(0xffffffffu, r, 1, 4), r2 = __shfl_sync(0xffffffffu, r, 2, 4);
  const T* d = D + 3 * min(c, 2) * R;
  return fma(d[2 * R], r2, fma(d[R], r1, d[0] * r0));
}

// f(u, i, c, row) for the values u = 4 i + c of the rows, on thread u % RK_T
// (every lane of a warp calls; row = -1 where there is nothing to do)
template <class T, class F>
__device__ inline void rk_values(const RkRows<T>& A, F f) {
  const int l = threadIdx.x & 31;
  for (int u0 = threadIdx.x & ~31; u0 < 4 * A.nr; u0 += RK_T) {
    int u = u0 + l, i = u >> 2, c = u & 3;
    bool in = u < 4 * A.nr;
    f(in ? i : 0, c, in && c < 3 ? A.id[i] : -1);
  }
}

// PCG with the block-Jacobi inverses Dinv, from x = 0 to ||b - K x|| <= tol
// ||b|| or maxit iterations: the recurrences of k_pcg_a and k_pcg_b.  z is the
// vector the blocks exchange (4-component rows, padding rows zero).  The
// scalars in sc as the host reads them (rr of the last iteration at
// rr[iters % 3]).
constexpr int RK_PCG_VECS = 5;
template <class T>
__global__ void __launch_bounds__(RK_T, 1)
    k_pcg_resident(int nd, int ns, Sliced S, const T* __restrict__ K, const T* __restrict__ Dinv,
                   const int* __restrict__ mask, const double* __restrict__ b, T* x, T* z, double tol, int maxit,
                   Scal* sc, unsigned long long* slots, RkPlan pl) {
  extern __shared__ __align__(16) unsigned char mem[];
  __shared__ RkShared sh;
  __shared__ T sy[3][RK_T];
  const int t = threadIdx.x;
  RkGrid g{slots, &sc->late, pl.G, (int)blockIdx.x, pl.polls, 0};
  if (g.me == g.G - 1) {
    // the coordinator
    if (t >= RK_CT) return;
    double s[2];
    bool ok = rk_collect<2>(g, sh, s, true);
    double rz = s[0], rr = s[1], bb = s[1], thr = tol * tol * bb;
    bool conv = bb == 0.0, bad = !ok;
    int iters = 0;
    rk_tell(g, 0.0, 0.0, conv || bad, true);
    while (!conv && !bad && iters < maxit) {
      double irz = 1.0 / rz;  // ready before the sum it divides
      ok = rk_collect<1>(g, sh, s, false);
      bad = !ok || !rk_positive(s[0]);
      rk_tell(g, rz / s[0], 0.0, bad, false);
      if (bad) break;
      ok = rk_collect<2>(g, sh, s, true);
      rr = s[1];
      ++iters;
      bad = !ok || !rk_finite(rr);
      conv = rk_at_most(rr, thr);
      rk_tell(g, rk_quotient(s[0], rz, 1.0, irz), 0.0, conv || bad || iters >= maxit, true);
      rz = s[0];
    }
    if (t == 0) {
      sc->bb = bb;
      sc->thr = thr;
      sc->rr[iters % 3] = rr;
      sc->iters = iters;
      sc->done = conv || bad;
      sc->breakdown = bad;
    }
    return;
  }
  rk_range(S, ns, g.G - 1, g.me, sh);
  RkRows<T> A;
  T* vr = A.init(S, K, nd, pl, sh, sy, mem, RK_PCG_VECS);
  const int R = A.R, nr = A.nr, n4 = min(4 * nr, RK_T);
  T *vx = vr + 3 * R, *vp = vx + 3 * R, *vq = vp + 3 * R, *vz = vq + 3 * R, *vd = vz + 3 * R;
  double s2[2] = {0.0, 0.0};
  for (int u = t; u < 4 * nr; u += RK_T) z[4 * (size_t)S.row[4 * A.q0 + (u >> 2)] + (u & 3)] = (T)0;
  rk_values(A, [&](int i, int c, int row) {
    T rv = (T)0;
    if (row >= 0) {
      rv = ((mask[row] >> c) & 1) ? (T)0 : (T)b[3 * (size_t)row + c];
      for (int e = 0; e < 3; ++e) vd[(3 * c + e) * R + i] = Dinv[12 * (size_t)row + 4 * c + e];
    }
    T zv = rk_dinv(vd + i, R, c, rv);
    if (row < 0) return;
    int o = c * R + i;
    z[4 * (size_t)row + c] = vz[o] = zv;
    vr[o] = rv;
    vx[o] = vp[o] = vq[o] = (T)0;
    s2[0] += (double)rv * (double)zv;
    s2[1] += (double)rv * (double)rv;
  });
  rk_sum<2>(g, sh, s2, n4, true);
  while (!sh.stop) {
    // p = z + beta p, q = K z + beta q, p.q
    const T be = (T)sh.scal[0];
    double part = 0.0;
    for (int c0 = 0; c0 < nr; c0 += 4 * RK_QUADS) {
      int nq = min(RK_QUADS, (nr - c0) >> 2);
      if (c0) __syncthreads();
      A.mul(z, c0, nq);
      A.each(nq, [&](int i, int c, T y) {
        int o = c * R + c0 + i;
        if (A.id[c0 + i] < 0) return;
        T pv = vz[o] + be * vp[o], qv = y + be * vq[o];
        vp[o] = pv;
        vq[o] = qv;
        part += (double)pv * (double)qv;
      });
    }
    rk_sum<1>(g, sh, &part, n4, false);
    if (sh.stop) break;
    // x += alpha p, r -= alpha q, z = Dinv r, r.z, r.r
    const T alpha = (T)sh.scal[0];
    s2[0] = s2[1] = 0.0;
    rk_values(A, [&](int i, int c, int row) {
      int o = c * R + i;
      T rv = row >= 0 ? vr[o] - alpha * vq[o] : (T)0;
      T zv = rk_dinv(vd + i, R, c, rv);
      if (row < 0) return;
      z[4 * (size_t)row + c] = vz[o] = zv;
      vr[o] = rv;
      vx[o] += alpha * vp[o];
      s2[0] += (double)rv * (double)zv;
      s2[1] += (double)rv * (double)rv;
    });
    rk_sum<2>(g, sh, s2, n4, true);
  }
  rk_values(A, [&](int i, int c, int row) {
    if (row >= 0) x[3 * (size_t)row + c] = vx[c * R + i];
  });
}

// BiCGStab, right preconditioned by the block-Jacobi inverses: the recurrences
// of k_bicg_p / _s / _x / _rotate, the products of k_spmv_dot.  ph and sp are
// the vectors the blocks exchange.  Scalars for the host as there: iters,
// done, breakdown, rr[0].
constexpr int RK_BICG_VECS = 9;
template <class T>
__global__ void __launch_bounds__(RK_T, 1)
    k_bicg_resident(int nd, int ns, Sliced S, const T* __restrict__ K, const T* __restrict__ Dinv,
                    const int* __restrict__ mask, const double* __restrict__ b, T* x, T* ph, T* sp, double tol,
                    int maxit, Scal* sc, unsigned long long* slots, RkPlan pl) {
  extern __shared__ __align__(16) unsigned char mem[];
  __shared__ RkShared sh;
  __shared__ T sy[3][RK_T];
  const int t = threadIdx.x;
  RkGrid g{slots, &sc->late, pl.G, (int)blockIdx.x, pl.polls, 0};
  if (g.me == g.G - 1) {
    // the coordinator
    if (t >= RK_CT) return;
    double s[2];
    bool ok = rk_collect<1>(g, sh, s, true);
    double bb = s[0], rr = bb, thr = tol * tol * bb, rho1 = bb;
    bool conv = bb == 0.0, bad = !ok;
    int it = 0;
    // beta (times p - omega v = 0 at the start) and omega
    rk_tell(g, bb, 1.0, conv || bad, true);
    while (!conv && !bad && it < maxit) {
      ++it;
      ok = rk_collect<1>(g, sh, s, true);  // ph is there
      bad = !ok;
      rk_tell(g, 0.0, 0.0, bad, true);
      if (bad) break;
      double irho = 1.0 / rho1;
      ok = rk_collect<1>(g, sh, s, false);  // r0.v
      bad = !ok || !rk_finite(s[0]) || s[0] == 0.0;
      double alpha = rho1 / s[0];
      rk_tell(g, alpha, 0.0, bad, false);
      if (bad) break;
      ok = rk_collect<1>(g, sh, s, true);  // s.s
      conv = ok && rk_at_most(s[0], thr);
      bad = !ok;
      rk_tell(g, alpha, 0.0, bad ? 1 : conv ? 2 : 0, true);
      if (conv) rr = s[0];
      if (bad || conv) break;
      ok = rk_collect<2>(g, sh, s, false);  // t.s, t.t
      double omega = rk_positive(s[1]) ? s[0] / s[1] : 0.0;
      bad = !ok;
      rk_tell(g, alpha, omega, bad, false);
      if (bad) break;
      double ao = alpha / omega, f = irho * ao;
      ok = rk_collect<2>(g, sh, s, false);  // r.r, r0.r
      rr = s[0];
      conv = rk_at_most(rr, thr);
      bad = !ok || (!conv && (!(omega != 0.0) || !rk_finite(rr)));
      rk_tell(g, rk_quotient(s[1], rho1, ao, f), omega, conv || bad || it >= maxit, false);
      rho1 = s[1];
    }
    if (t == 0) {
      sc->bb = bb;
      sc->thr = thr;
      sc->rr[0] = rr;
      sc->iters = it;
      sc->done = conv || bad;
      sc->breakdown = bad;
    }
    return;
  }
  rk_range(S, ns, g.G - 1, g.me, sh);
  RkRows<T> A;
  T* vr = A.init(S, K, nd, pl, sh, sy, mem, RK_BICG_VECS);
  const int R = A.R, nr = A.nr, n4 = min(4 * nr, RK_T);
  T *vx = vr + 3 * R, *r0 = vx + 3 * R, *vp = r0 + 3 * R, *vv = vp + 3 * R, *vs = vv + 3 * R, *vt = vs + 3 * R,
    *vph = vt + 3 * R, *vsp = vph + 3 * R, *vd = vsp + 3 * R;
  double part = 0.0;
  for (int u = t; u < 4 * nr; u += RK_T) {
    size_t o = 4 * (size_t)S.row[4 * A.q0 + (u >> 2)] + (u & 3);
    ph[o] = sp[o] = (T)0;
  }
  rk_values(A, [&](int i, int c, int row) {
    if (row < 0) return;
    int o = c * R + i;
    T rv = ((mask[row] >> c) & 1) ? (T)0 : (T)b[3 * (size_t)row + c];
    for (int e = 0; e < 3; ++e) vd[(3 * c + e) * R + i] = Dinv[12 * (size_t)row + 4 * c + e];
    vr[o] = r0[o] = rv;
    vx[o] = vp[o] = vv[o] = (T)0;
    part += (double)rv * (double)rv;
  });
  rk_sum<1>(g, sh, &part, n4, true);
  while (!sh.stop) {
    // p = r + beta (p - omega v), ph = Dinv p
    const T be = (T)sh.scal[0], om1 = (T)sh.scal[1];
    rk_values(A, [&](int i, int c, int row) {
      int o = c * R + i;
      T pv = row >= 0 ? vr[o] + be * (vp[o] - om1 * vv[o]) : (T)0;
      T zv = rk_dinv(vd + i, R, c, pv);
      if (row < 0) return;
      ph[4 * (size_t)row + c] = vph[o] = zv;
      vp[o] = pv;
    });
    part = 0.0;
    rk_sum<1>(g, sh, &part, 1, true);
    if (sh.stop) break;
    // v = K ph, r0.v
    for (int c0 = 0; c0 < nr; c0 += 4 * RK_QUADS) {
      int nq = min(RK_QUADS, (nr - c0) >> 2);
      if (c0) __syncthreads();
      A.mul(ph, c0, nq);
      A.each(nq, [&](int i, int c, T y) {
        int o = c * R + c0 + i;
        if (A.id[c0 + i] < 0) return;
        vv[o] = y;
        part += (double)r0[o] * (double)y;
      });
    }
    rk_sum<1>(g, sh, &part, n4, false);
    if (sh.stop) break;
    // s = r - alpha v, sp = Dinv s, s.s
    const T al = (T)sh.scal[0];
    part = 0.0;
    rk_values(A, [&](int i, int c, int row) {
      int o = c * R + i;
      T sv = row >= 0 ? vr[o] - al * vv[o] : (T)0;
      T zv = rk_dinv(vd + i, R, c, sv);
      if (row < 0) return;
      sp[4 * (size_t)row + c] = vsp[o] = zv;
      vs[o] = sv;
      part += (double)sv * (double)sv;
    });
    rk_sum<1>(g, sh, &part, n4, true);
    if (sh.stop) {
      if (sh.stop == 2) {
        // converged on s: x += alpha ph
        const double a = sh.scal[0];
        rk_values(A, [&](int i, int c, int row) {
          if (row >= 0) vx[c * R + i] += (T)(a * (double)vph[c * R + i]);
        });
      }
      break;
    }
    // t = K sp, t.s, t.t
    double s2[2] = {0.0, 0.0};
    for (int c0 = 0; c0 < nr; c0 += 4 * RK_QUADS) {
      int nq = min(RK_QUADS, (nr - c0) >> 2);
      if (c0) __syncthreads();
      A.mul(sp, c0, nq);
      A.each(nq, [&](int i, int c, T y) {
        int o = c * R + c0 + i;
        if (A.id[c0 + i] < 0) return;
        vt[o] = y;
        s2[0] += (double)vs[o] * (double)y;
        s2[1] += (double)y * (double)y;
      });
    }
    rk_sum<2>(g, sh, s2, n4, false);
    if (sh.stop) break;
    // x += alpha ph + omega sp, r = s - omega t, r.r, r0.r
    const double a = sh.scal[0], om = sh.scal[1];
    const T omt = (T)om;
    s2[0] = s2[1] = 0.0;
    rk_values(A, [&](int i, int c, int row) {
      if (row < 0) return;
      int o = c * R + i;
      T rv = vs[o] - omt * vt[o];
      vr[o] = rv;
      s2[0] += (double)rv * (double)rv;
      s2[1] += (double)r0[o] * (double)rv;
      vx[o] += (T)(a * (double)vph[o] + om * (double)vsp[o]);
    });
    rk_sum<2>(g, sh, s2, n4, false);
  }
  rk_values(A, [&](int i, int c, int row) {
    if (row >= 0) x[3 * (size_t)row + c] = vx[c * R + i];
  });
}

}  // namespace mpm
