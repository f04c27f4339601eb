// Step 1 of §4.1 for blocks that stay in L2: the whole block CG in one cooperative launch.
//
// What bounds a small solve is not memory but the sequence itself: four or five launches of
// 3 to 10 us an iteration and a host synchronisation every other one, for passes that take a
// microsecond or two.  Here one grid of at most one CTA per SM runs the start and every
// iteration: each CTA owns a contiguous range of grid points (its stencil neighbours are
// mostly its own, so they come from L1), the dot products meet in a grid-wide barrier, and
// every CTA sums the partials of all CTAs itself, in the same order, so alpha, beta and the
// active columns need no second pass and no host.  The arithmetic per element is that of the
// row kernels (stencil_cg.cu): FP32 recomputes P = R + beta P at the stencil points and takes
// two barriers an iteration; FP64 stores Q and P and takes three (recomputing would cost six
// more FP64 operations per element, and GB300 runs two a clock and SM).
//
// What is left of an iteration: tiny solves 4.9 us of shuffles, barriers and latency (32 x 32 x 8,
// FP32, one cluster; 37 us by kernels), FP64 the FP64 pipe (199 x 199 x 16: 31 us with the Jacobi
// preconditioner, of which 11 for its 10 operations an element; 58 us by kernels), FP32 the L2 latency
// of its stencil loads (200 x 200 x 16 15 us, 39 by kernels).
//
// Every wait of the barrier is bounded; a CTA that gives up sets the error word and returns.
#include <string.h>

#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "kernels.cuh"
#include "sums.cuh"
#include "tc.cuh"

namespace opevo {

namespace {

constexpr int kCoopThreads = 512;
// Largest block of a cooperative solve; microseconds an iteration here and by the general kernels
// (Jacobi).  FP32: the four blocks of an iteration have to stay in the 126 MB L2, and on 3-D grids the
// TMA direction kernel takes over: 48^3 x 80 (34 MB) 88 and 97, 36^3 x 200 (36 MB) 111 and 118,
// 56^3 x 56 (38 MB) 97 and 94, 56^3 x 64 (43 MB) 112 and 100.  2-D grids: 700 x 700 x 24 (45 MB) 99 and
// 114, and 127 against 141 at 61 MB, 208 against 196 at 92 MB, beyond the line.  FP64, bound by the FP64
// pipe either way: 64^3 x 64 (128 MB) 568 and 645; the line is not a crossing (72^3 x 128, 365 MB: 1581
// and 1721).
template <typename T> constexpr long long coop_bytes(int dim) {
  return (sizeof(T) == 8 ? 140ll : (dim == 3 ? 36ll : 48ll)) << 20;
}
// Dynamic shared memory a launch may ask for (the largest any size below takes is 140 KB).  The
// limit belongs to the kernel on the device, so every call sets this one value: a limit of the
// call's own size could be lowered by another thread's solve between setting it and the launch.
constexpr int kCoopSmem = 224 * 1024;
// polls of the barrier (several hundred clocks each) before a CTA gives up: some seconds
constexpr int kBarrierPolls = 1 << 23;
// ctl words (256 bytes): 2 iterations, 3 error, 32 the barrier's arrivals
constexpr int kCtlBar = 32;

// Grid-wide barrier: `target` is the number of arrivals (mod 2^32: some 10^7 iterations of a full
// grid) that completes it.  False when the
// wait gave up (the error word is set and every CTA gives up in turn).
__device__ __forceinline__ bool grid_barrier(int *ctl, unsigned target, int *ok_sh) {
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned *cnt = reinterpret_cast<unsigned *>(ctl + kCtlBar);
    int ok = 1;
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(cnt) : "memory");
    // (no clock is read here: %globaltimer alone costs more than a poll)
    int left = kBarrierPolls;
    for (;;) {
      unsigned v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(cnt) : "memory");
      if (count_reached(v, target)) break;
      if (--left == 0) {
        atomicExch(ctl + 3, 1);
        ok = 0;
        break;
      }
    }
    *ok_sh = ok;
  }
  __syncthreads();
  return *ok_sh != 0;
}

// Barrier of the CTAs of one cluster (in hardware: every CTA of a cluster is resident).
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Running sum across threads and CTAs.  FP64 blocks: a double.  FP32 blocks: a triple of floats
// (sums.cuh: with FP64 additions the reductions were half of an iteration).  A sum that leaves the
// FP32 range is formed again in FP64 (`total` below) and held as the double's bits in h and m,
// marked by l = NaN.  WIDE: the sums are such doubles.
template <typename T> struct Sum;
// Threads that share the sums of the columns: all of them for FP32 blocks, one warp a scheduler
// for FP64 (its additions queue on the one FP64 pipe, and idle lanes cost as much as busy ones).
template <typename T> constexpr int kSumThreads = sizeof(T) == 4 ? kCoopThreads : 128;
template <> struct Sum<double> {
  double h = 0.0;
  __device__ __forceinline__ void add(double x) { h += x; }
  __device__ __forceinline__ void add(const Sum &o) { h += o.h; }
  __device__ __forceinline__ bool finite() const { return true; }  // (nothing to form again)
  __device__ __forceinline__ double value() const { return h; }
  __device__ __forceinline__ Sum over(int o) const {
    Sum s;
    s.h = __shfl_xor_sync(0xffffffffu, h, o);
    return s;
  }
  __device__ __forceinline__ static Sum load(const Sum *p) {
    Sum s;
    s.h = __ldcg(&p->h);
    return s;
  }
  // q = a / b, 0 where b <= 0; false: for WIDE
  template <bool WIDE>
  __device__ __forceinline__ static bool quotient(const Sum &a, const Sum &b, double *q) {
    *q = b.h > 0.0 ? a.h / b.h : 0.0;
    return true;
  }
  // 1 or 0: a sum of squares is above t or not (tf: t in the block's type); -1: for WIDE
  template <bool WIDE> __device__ __forceinline__ int above(double t, double) const { return h > t; }
};
template <> struct __align__(16) Sum<float> : Sum3 {
  __device__ __forceinline__ static Sum of(double d) {
    Sum s;
    s.h = __int_as_float(__double2loint(d));
    s.m = __int_as_float(__double2hiint(d));
    s.l = __int_as_float(0x7fffffff);
    return s;
  }
  __device__ __forceinline__ double value() const {
    return finite() ? Sum3::value() : __hiloint2double(__float_as_int(m), __float_as_int(h));
  }
  __device__ __forceinline__ Sum over(int o) const {
    Sum s;
    s.h = __shfl_xor_sync(0xffffffffu, h, o);
    s.m = __shfl_xor_sync(0xffffffffu, m, o);
    s.l = __shfl_xor_sync(0xffffffffu, l, o);
    return s;
  }
  __device__ __forceinline__ static Sum load(const Sum *p) {
    const float4 v = __ldcg(reinterpret_cast<const float4 *>(p));
    Sum s;
    s.h = v.x;
    s.m = v.y;
    s.l = v.z;
    return s;
  }
  template <bool WIDE>
  __device__ __forceinline__ static bool quotient(const Sum &a, const Sum &b, float *q) {
    if constexpr (WIDE) {
      const double d = b.value();
      *q = d > 0.0 ? (float)(a.value() / d) : 0.f;
      return true;
    }
    return opevo::quotient(a, b, q);
  }
  // (the FP32 parts decide unless they are within 2^-12: a sum of n squares has |m| < n 2^-24 h)
  template <bool WIDE> __device__ __forceinline__ int above(double t, float tf) const {
    if constexpr (WIDE) return value() > t;
    if (!(tf < 1e30f)) return -1;
    if (h > fmaxf(tf, 1e-30f) * 1.000245f) return 1;
    return tf > 1e-30f && h < tf * 0.999755f ? 0 : -1;
  }
};

// v into CTA `rank`'s copy of the shared-memory slot p.
template <typename S> __device__ __forceinline__ void store_cluster(S *p, int rank, const S &v) {
  uint32_t a;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(tc::smem_u32(p)), "r"(rank));
  unsigned long long bits[2] = {0, 0};
  static_assert(sizeof(S) == 8 || sizeof(S) == 16, "one store");
  memcpy(bits, &v, sizeof(S));
  if constexpr (sizeof(S) == 8)
    asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(a), "l"(bits[0]) : "memory");
  else
    asm volatile("st.shared::cluster.v2.u64 [%0], {%1, %2};" ::"r"(a), "l"(bits[0]), "l"(bits[1])
                 : "memory");
}

struct CoopArgs {
  Geom g;
  const void *Vt, *U;
  void *W, *R, *P, *Q;
  int p, ld, max_iter, rows_per_cta, inv_rows, cluster;
  double rtol2, shift;
  double *part;
  int *ctl;
};

template <typename T>
__device__ __forceinline__ Pack<T> ldp(const T *x) {  // plain load: other CTAs write the blocks
  return Pack<T>::load_rw(x);
}

// Row i of (H + sigma) applied to the values at(offset): the point's and its neighbours'.  A
// neighbour outside the grid is read at the point itself and counted as zero, so the loads of
// all points are issued together, without branches between them.
template <typename T, typename F>
__device__ __forceinline__ Pack<T> stencil_sum(const Geom &g, int i, int ld, T diag,
                                               const Pack<T> &xc, F &&at) {
  constexpr int N = Pack<T>::N;
  const unsigned r = (unsigned)i / (unsigned)g.nx;
  const int ix = i - (int)r * g.nx;
  const unsigned iz = r / (unsigned)g.ny;
  const int iy = (int)r - (int)iz * g.ny;
  const int sy = g.nx * ld, sz = g.nx * g.ny * ld;
  const bool bx0 = ix > 0, bx1 = ix < g.nx - 1, by0 = iy > 0, by1 = iy < g.ny - 1;
  const T cx = (T)g.c[0], cy = (T)g.c[1], cz = (T)g.c[2];
  const Pack<T> x0 = at(bx0 ? -ld : 0), x1 = at(bx1 ? ld : 0);
  const Pack<T> y0 = at(by0 ? -sy : 0), y1 = at(by1 ? sy : 0);
  Pack<T> y;
  if (g.dim == 3) {
    const bool bz0 = iz > 0, bz1 = (int)iz < g.nz - 1;
    const Pack<T> z0 = at(bz0 ? -sz : 0), z1 = at(bz1 ? sz : 0);
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const T s0 = (bx0 ? x0.v[k] : T(0)) + (bx1 ? x1.v[k] : T(0));
      const T s1 = (by0 ? y0.v[k] : T(0)) + (by1 ? y1.v[k] : T(0));
      const T s2 = (bz0 ? z0.v[k] : T(0)) + (bz1 ? z1.v[k] : T(0));
      y.v[k] = diag * xc.v[k] - cx * s0 - cy * s1 - cz * s2;
    }
  } else {
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const T s0 = (bx0 ? x0.v[k] : T(0)) + (bx1 ? x1.v[k] : T(0));
      const T s1 = (by0 ? y0.v[k] : T(0)) + (by1 ? y1.v[k] : T(0));
      y.v[k] = diag * xc.v[k] - cx * s0 - cy * s1;
    }
  }
  return y;
}

// Sums of the CTAs' partials in shared memory: at most 512 or one row of 3 ld, at an odd pitch.
__host__ __device__ constexpr int tot_len(int ld) { return kCoopThreads + 3 * ld + 64; }

// L: neighbouring lanes that reduce one column
template <typename T, bool JAC, int L>
__global__ void __launch_bounds__(kCoopThreads, 1) k_cg_coop(const CoopArgs A) {
  constexpr int N = Pack<T>::N;
  constexpr bool kFused = std::is_same<T, float>::value;
  extern __shared__ __align__(16) double sm[];
  __shared__ int ok_sh, nact_sh, wide_sh;
  const Geom &g = A.g;
  const int ld = A.ld, nv = ld / N, nr = kCoopThreads / nv;
  const int tx = threadIdx.x % nv, ty = threadIdx.x / nv;
  const bool on = ty < nr;
  const int nra = min(nr, A.rows_per_cta);  // rows of threads that hold points
  const int col = tx * N, G = gridDim.x;
  const int r0 = blockIdx.x * A.rows_per_cta;
  const int r1 = min(r0 + A.rows_per_cta, (int)g.n);
  const T *Vt = (const T *)A.Vt, *U = (const T *)A.U;
  T *W = (T *)A.W, *R = (T *)A.R;
  const T shift = (T)A.shift;
  // shared memory: per-column state, 1 / diag of the CTA's points, the cluster's partials
  // [2][CTA][3 ld] (odd pitch), sums of the CTAs' partials, the threads' sums
  using S = Sum<T>;
  double *target = sm;
  S *rho = reinterpret_cast<S *>(target + ld);
  T *al = reinterpret_cast<T *>(rho + ld), *be = al + ld, *target_t = be + ld;
  int *act = reinterpret_cast<int *>(target_t + ld), *wide = act + ld;
  T *inv_sh = reinterpret_cast<T *>(wide + ld);
  S *xch = reinterpret_cast<S *>(inv_sh + A.inv_rows);
  S *tot = xch + (A.cluster ? 2 * G * (3 * ld + 1) : 0);
  T *rows = reinterpret_cast<T *>(tot + tot_len(ld));
  constexpr int jstep = kCoopThreads / L;
  const int lane = threadIdx.x & (L - 1);
  const int jw = (int)(threadIdx.x & ~31u) / L, jl = (int)(threadIdx.x & 31) / L;
  unsigned epoch = 0;
  int odd = 0;

  if (JAC && A.inv_rows) {
    for (int i = r0 + (int)threadIdx.x; i < r1; i += kCoopThreads)
      inv_sh[i - r0] = T(1) / (__ldg(Vt + i) + shift);
    __syncthreads();
  }
  auto inv_of = [&](int i, T dg) -> T { return A.inv_rows ? inv_sh[i - r0] : T(1) / dg; };

  // All CTAs arrive, and see what the others wrote before.
  auto meet = [&]() -> bool {
    if (G == 1) {
      __syncthreads();
      return true;
    }
    if (A.cluster) {
      cluster_barrier();
      return true;
    }
    epoch += G;
    return grid_barrier(A.ctl, epoch, &ok_sh);
  };

  // Totals over the grid of the per-thread sums acc[c][k] (column col + k): over the CTA's rows,
  // then over the CTAs, in the same order in every CTA; one lane a column gets fin(j, sums, WIDE).
  // A cluster's partials go straight into every member's shared memory.  A column that fin refuses
  // (a sum outside the FP32 range, or a quotient or comparison that takes FP64: rare) is summed
  // again in FP64 from the threads' sums: every CTA has the same partials, so all refuse alike.
  auto total = [&](auto &acc, auto &&fin) -> bool {
    constexpr int NC = sizeof(acc) / sizeof(acc[0]);
    const int w = NC * ld, pitch = w | 1, pm = w | 1;
    __syncthreads();
    if (ty < nra) {
#pragma unroll
      for (int c = 0; c < NC; ++c)
#pragma unroll
        for (int k = 0; k < N; ++k) rows[ty * pitch + c * ld + col + k] = acc[c][k];
    }
    __syncthreads();
    auto last = [&](int j, S *s) {
      if (!fin(j, s, std::false_type{})) wide[j] = wide_sh = 1;
    };
    // alternate buffers: a CTA may still read the last totals' partials
    S *part = reinterpret_cast<S *>(A.part) + odd * 3 * G * ld;
    S *mine = xch + odd * G * (3 * ld + 1);
    odd ^= 1;
    for (int jb = jw; jb < ld; jb += jstep) {  // (whole warps)
      const int j = jb + jl;
      S s[NC];
      if (j < ld)
#pragma unroll 4
        for (int y = lane; y < nra; y += L)
#pragma unroll
          for (int c = 0; c < NC; ++c) s[c].add(rows[y * pitch + c * ld + j]);
#pragma unroll
      for (int o = L >> 1; o > 0; o >>= 1)
#pragma unroll
        for (int c = 0; c < NC; ++c) s[c].add(s[c].over(o));
      if (j >= ld) continue;
      if (G == 1) {
        if (lane == 0) last(j, s);
      } else if (A.cluster) {
#pragma unroll
        for (int c = 0; c < NC; ++c)
          for (int r = lane; r < G; r += L) store_cluster(mine + blockIdx.x * pm + c * ld + j, r, s[c]);
      } else if (lane == 0) {
#pragma unroll
        for (int c = 0; c < NC; ++c) part[blockIdx.x * w + c * ld + j] = s[c];
      }
    }
    if (G > 1) {
      if (!meet()) return false;
      // the CTAs' partials: a cluster's are here; a grid's come from L2 as whole lines, summed
      // in `gg` interleaved groups first
      const S *from = mine;
      int terms = G;
      if (!A.cluster) {
        const int gg = max(1, min(G, max(kSumThreads<T>, min(kCoopThreads, 4 * w)) / w));
        for (int t = threadIdx.x; t < gg * w; t += kCoopThreads) {
          const int q = t / w, e = t - q * w;
          S s;
#pragma unroll 8
          for (int b = q; b < G; b += gg) s.add(S::load(part + b * w + e));
          tot[q * pm + e] = s;
        }
        __syncthreads();
        from = tot;
        terms = gg;
      }
      for (int jb = jw; jb < ld; jb += jstep) {  // (whole warps)
        const int j = jb + jl;
        S s[NC];
        if (j < ld)
#pragma unroll 4
          for (int b = lane; b < terms; b += L)
#pragma unroll
            for (int c = 0; c < NC; ++c) s[c].add(from[b * pm + c * ld + j]);
#pragma unroll
        for (int o = L >> 1; o > 0; o >>= 1)
#pragma unroll
          for (int c = 0; c < NC; ++c) s[c].add(s[c].over(o));
        if (lane == 0 && j < ld) last(j, s);
      }
    }
    __syncthreads();
    if constexpr (kFused) {
      if (wide_sh) {
        part = reinterpret_cast<S *>(A.part) + odd * 3 * G * ld;
        mine = xch + odd * G * (3 * ld + 1);
        odd ^= 1;
#pragma unroll 1
        for (int e = threadIdx.x; e < w; e += kCoopThreads) {
          double d = 0.0;
#pragma unroll 1
          for (int y = 0; y < nra; ++y) d += (double)rows[y * pitch + e];
          const S v = S::of(d);
          if (G == 1) {
            tot[e] = v;
          } else if (A.cluster) {
#pragma unroll 1
            for (int r = 0; r < G; ++r) store_cluster(mine + blockIdx.x * pm + e, r, v);
          } else {
            part[blockIdx.x * w + e] = v;
          }
        }
        if (G > 1) {
          if (!meet()) return false;
#pragma unroll 1
          for (int e = threadIdx.x; e < w; e += kCoopThreads) {
            double d = 0.0;
#pragma unroll 1
            for (int b = 0; b < G; ++b)
              d += (A.cluster ? mine[b * pm + e] : S::load(part + b * w + e)).value();
            tot[e] = S::of(d);
          }
        }
        __syncthreads();
        for (int j = threadIdx.x; j < ld; j += kCoopThreads)
          if (wide[j]) {
            S s[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) s[c] = tot[c * ld + j];
            fin(j, s, std::true_type{});
            wide[j] = 0;
          }
        if (threadIdx.x == 0) wide_sh = 0;
        __syncthreads();
      }
    }
    return true;
  };
  for (int j = threadIdx.x; j < ld; j += kCoopThreads) wide[j] = 0;
  if (threadIdx.x == 0) wide_sh = 0;
  if (A.cluster) cluster_barrier();  // every member runs before its shared memory is written

  // start: R = U - (H + sigma) W (Z = R / d with the Jacobi preconditioner); FP64: P = R
  bool ok;
  {
    T acc[3][N] = {};
    if (on)
      for (int i = r0 + ty; i < r1; i += nr) {
        const long long o = (long long)i * ld + col;
        const T dg = __ldg(Vt + i) + shift;
        const Pack<T> wc = ldp(W + o), u = ldp(U + o);
        const Pack<T> aw = stencil_sum<T>(g, i, ld, dg, wc, [&](int d) { return ldp(W + o + d); });
        const T inv = JAC ? inv_of(i, dg) : T(1);
        Pack<T> r;
#pragma unroll
        for (int k = 0; k < N; ++k) {
          const T rk = u.v[k] - aw.v[k];
          r.v[k] = JAC ? rk * inv : rk;
          acc[0][k] += rk * r.v[k];
          acc[1][k] += u.v[k] * u.v[k];
          acc[2][k] += rk * rk;
        }
        r.store(R + o);
        if (!kFused) r.store((T *)A.P + o);
      }
    if (threadIdx.x == 0) nact_sh = 0;
    ok = total(acc, [&](int j, S *s, auto wd) {
      if (!decltype(wd)::value && !(s[0].finite() && s[1].finite() && s[2].finite())) return false;
      const double bb = s[1].value();
      rho[j] = s[0];
      target[j] = A.rtol2 * bb;
      target_t[j] = (T)target[j];
      al[j] = be[j] = T(0);
      const int a = (j < A.p) && (s[2].value() > A.rtol2 * bb) && (bb > 0.0);
      act[j] = a;
      if (a) atomicAdd(&nact_sh, 1);
      return true;
    });
  }
  int it = 0;
  while (ok && nact_sh > 0 && it < A.max_iter) {
    // FP32 alternates the two direction buffers; FP64 keeps P and stores Q = (H + sigma) P
    const T *Po = (const T *)((kFused && (it & 1)) ? A.Q : A.P);
    T *Pn = (T *)((kFused && !(it & 1)) ? A.Q : A.P);
    T *Q = (T *)A.Q;
    {
      T acc[1][N] = {};
      if (on) {
        T b[N];
#pragma unroll
        for (int k = 0; k < N; ++k) b[k] = be[col + k];
        const bool first = it == 0;
        for (int i = r0 + ty; i < r1; i += nr) {
          const long long o = (long long)i * ld + col;
          const T dg = __ldg(Vt + i) + shift;
          Pack<T> pc, q;
          if (kFused) {
            auto dir = [&](int d) {
              Pack<T> r = ldp(R + o + d);
              if (!first) {
                const Pack<T> x = ldp(Po + o + d);
#pragma unroll
                for (int k = 0; k < N; ++k) r.v[k] += b[k] * x.v[k];
              }
              return r;
            };
            pc = dir(0);
            q = stencil_sum<T>(g, i, ld, dg, pc, dir);
            pc.store(Pn + o);
          } else {
            pc = ldp(Po + o);
            q = stencil_sum<T>(g, i, ld, dg, pc, [&](int d) { return ldp(Po + o + d); });
            q.store(Q + o);
          }
#pragma unroll
          for (int k = 0; k < N; ++k) acc[0][k] += pc.v[k] * q.v[k];
        }
      }
      ok = total(acc, [&](int j, S *s, auto wd) {
        T q = T(0);
        if (act[j] && !S::template quotient<decltype(wd)::value>(rho[j], s[0], &q)) return false;
        al[j] = q;
        return true;
      });
      if (!ok) break;
      if (threadIdx.x == 0) nact_sh = 0;  // (every thread has read it for this iteration)
    }
    {
      constexpr int NC = JAC ? 2 : 1;
      T acc[NC][N] = {};
      if (on) {
        T a[N];
#pragma unroll
        for (int k = 0; k < N; ++k) a[k] = al[col + k];
        for (int i = r0 + ty; i < r1; i += nr) {
          const long long o = (long long)i * ld + col;
          const T dg = __ldg(Vt + i) + shift;
          const Pack<T> pc = ldp(Pn + o);
          Pack<T> q, w = ldp(W + o), r = ldp(R + o);
          if (kFused)
            q = stencil_sum<T>(g, i, ld, dg, pc, [&](int d) { return ldp(Pn + o + d); });
          else
            q = ldp(Q + o);
          const T inv = JAC ? inv_of(i, dg) : T(1);
#pragma unroll
          for (int k = 0; k < N; ++k) {
            w.v[k] += a[k] * pc.v[k];
            if (JAC) {
              r.v[k] -= a[k] * (q.v[k] * inv);
              const T rk = dg * r.v[k];
              acc[0][k] += rk * r.v[k];
              acc[NC - 1][k] += rk * rk;
            } else {
              r.v[k] -= a[k] * q.v[k];
              acc[0][k] += r.v[k] * r.v[k];
            }
          }
          w.store(W + o);
          r.store(R + o);
        }
      }
      ok = total(acc, [&](int j, S *s, auto wd) {
        constexpr bool kWide = decltype(wd)::value;
        T q = T(0);
        if (act[j]) {
          const int a = s[NC - 1].template above<kWide>(target[j], target_t[j]);
          if (a < 0 || !S::template quotient<kWide>(s[0], rho[j], &q)) return false;
          rho[j] = s[0];
          act[j] = a;
          if (a) atomicAdd(&nact_sh, 1);
        }
        be[j] = q;
        return true;
      });
      if (!ok) break;
      ++it;
    }
    if (!kFused && nact_sh > 0 && it < A.max_iter) {
      if (on) {
        T b[N];
#pragma unroll
        for (int k = 0; k < N; ++k) b[k] = be[col + k];
        for (int i = r0 + ty; i < r1; i += nr) {
          const long long o = (long long)i * ld + col;
          const Pack<T> r = ldp(R + o);
          Pack<T> pp = ldp(Pn + o);
#pragma unroll
          for (int k = 0; k < N; ++k) pp.v[k] = r.v[k] + b[k] * pp.v[k];
          pp.store(Pn + o);
        }
      }
      ok = meet();
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) A.ctl[2] = it;
}

// CTAs of a solve and their grid points (*rows).  Up to a few vectors a thread in one cluster of
// 16 CTAs (their barrier is in hardware and the partials stay in shared memory); FP64 only up
// to one, since 16 SMs run 32 FP64 operations a clock.  Larger ones take at most one CTA per SM:
// FP32 as many as give every thread the same number of vectors, FP64 all of them.
constexpr int kCluster = 16;
template <typename T> int coop_ctas(long long n, int ld, int *rows) {
  const bool f32 = sizeof(T) == 4;
  const long long nr = kCoopThreads / (ld / Pack<T>::N), sms = num_sms();
  if (n > nr && n <= (f32 ? 4 : 1) * nr * kCluster && ld <= 64) {
    *rows = (int)((n + kCluster - 1) / kCluster);
    return kCluster;
  }
  const long long k = (n + nr * sms - 1) / (nr * sms);
  *rows = (int)(f32 || k == 1 ? nr * k : (n + sms - 1) / sms);
  return (int)((n + *rows - 1) / *rows);
}

// Lanes a column: FP32 blocks have at most 256 columns for 512 threads, FP64 ones at least 8 for 128.
// FP32 no more than 8: a level of the shuffle tree (three shuffles, two dependent two-sums) takes
// as long as five terms summed in turn (20 steps of 32 x 32 x 8 in FP64: 24.0 ms by up
// to 32 lanes, 23.7 by 16, 22.9 by 8, 23.3 by 4).
template <typename T> constexpr int kMinLanes = sizeof(T) == 4 ? 2 : 1;
template <typename T> constexpr int kMaxLanes = sizeof(T) == 4 ? 8 : 16;
template <typename T, bool JAC, int L = kMinLanes<T>> const void *coop_kernel(int lanes) {
  if constexpr (L < kMaxLanes<T>)
    if (lanes > L) return coop_kernel<T, JAC, 2 * L>(lanes);
  return (const void *)k_cg_coop<T, JAC, L>;
}

}  // namespace

template <typename T> bool cg_coop_eligible(const Geom &g, int ld) {
  return ld / Pack<T>::N <= 64 && g.n * ld * (long long)sizeof(T) <= coop_bytes<T>(g.dim);
}

template <typename T>
op_status cg_coop(const Geom &g, const T *Vt, double sigma, const T *U, T *W, int p, int ld,
                  double rtol, int max_iter, CGWork &w, int *iters, bool *ran, cudaStream_t st) {
  constexpr int N = Pack<T>::N;
  int rows = 0;
  const int G = coop_ctas<T>(g.n, ld, &rows);
  const bool cluster = G == kCluster && ld <= 64;  // (wider partials leave no room beside them)
  CoopArgs a{};
  a.g = g;
  a.Vt = Vt;
  a.U = U;
  a.W = W;
  a.R = w.R;
  a.P = w.P;
  a.Q = w.Q;
  a.p = p;
  a.ld = ld;
  a.max_iter = max_iter;
  a.rows_per_cta = rows;
  a.inv_rows = w.jacobi && rows <= 8192 ? (rows + 3) / 4 * 4 : 0;  // (16-byte alignment after it)
  a.rtol2 = rtol * rtol;
  a.shift = g.cdiag + sigma;
  a.part = w.part;
  a.ctl = w.ctl;
  a.cluster = cluster;
  // as laid out in the kernel; the threads' sums have an odd pitch
  const size_t sum = sizeof(Sum<T>);
  const size_t smem = (size_t)ld * (sizeof(double) + sum + 3 * sizeof(T) + 2 * sizeof(int)) +
                      (size_t)a.inv_rows * sizeof(T) +
                      (cluster ? (size_t)2 * G * (3 * ld + 1) * sum : 0) + tot_len(ld) * sum +
                      ((size_t)kCoopThreads * N * 3 + kCoopThreads / (ld / N) + 1) * sizeof(T);
  OP_CUDA(cudaMemsetAsync(w.ctl, 0, 256, st));
  void *args[] = {&a};
  int lanes = kMinLanes<T>;
  while (lanes < kMaxLanes<T> && 2 * lanes * ld <= kSumThreads<T>) lanes *= 2;
  const void *fn = w.jacobi ? coop_kernel<T, true>(lanes) : coop_kernel<T, false>(lanes);
  OP_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kCoopSmem));
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(G);
  cfg.blockDim = dim3(kCoopThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  if (cluster) {
    OP_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = kCluster;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  } else {
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
  }
  cfg.attrs = at;
  cfg.numAttrs = 1;
  prof_begin(w.prof, PK_CG_SOLVE, st);
  const cudaError_t e =
      w.route == 2 ? cudaErrorCooperativeLaunchTooLarge : cudaLaunchKernelExC(&cfg, fn, args);
  // a process confined to a few SMs may not hold the CTAs together: the general path needs no such thing
  *ran = e != cudaErrorCooperativeLaunchTooLarge && e != cudaErrorInvalidClusterSize &&
         e != cudaErrorLaunchOutOfResources;
  if (!*ran) {
    (void)cudaGetLastError();
    return OP_OK;
  }
  OP_CUDA(e);
  prof_end(w.prof, st);
  count_launch();
  OP_CUDA(cudaMemcpyAsync(w.host_ctl, w.ctl, 4 * sizeof(int), cudaMemcpyDeviceToHost, st));
  OP_CUDA(cudaStreamSynchronize(st));
  prof_harvest(w.prof);
  if (w.host_ctl[3]) {
    set_error("the cooperative CG gave up a bounded wait of its grid barrier");
    return OP_ERR_TIMEOUT;
  }
  *iters = w.host_ctl[2];
  w.expect_iters = *iters;
  return OP_OK;
}

#define OPEVO_INST(T)                                                                          \
  template bool cg_coop_eligible<T>(const Geom &, int);                                        \
  template op_status cg_coop<T>(const Geom &, const T *, double, const T *, T *, int, int,     \
                                double, int, CGWork &, int *, bool *, cudaStream_t);
OPEVO_INST(float)
OPEVO_INST(double)
#undef OPEVO_INST

}  // namespace opevo
