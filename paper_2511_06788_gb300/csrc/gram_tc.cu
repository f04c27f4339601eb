// Inner matrices of [U W] for FP32 blocks on the 5th-generation tensor cores:
// C = W^T U, S = W^T W, D = U^T U (§2.1; the matrices of Steps 2-3 and of
// Theorem 4.1) with tcgen05.mma kind::tf32 and FP32 accumulation in TMEM.
//
// FP32 accuracy from TF32 units (split = 1): every operand value x is split as
// x = hi + lo (hi = tf32(x), lo = tf32(x - hi)) and each product uses four
// MMAs, hi*hi + hi*lo + lo*hi + lo*lo (the lo*lo term would otherwise leave a
// one-signed error of ~2^-22 in the squared norms of <U,U> and <W,W>).  With
// split = 0 (the TF32 mixed mode) one MMA per product on tf32(x) is used.
//
// Work split: items of (output tile of 128 x 128, chunk of grid points), one persistent CTA per
// SM.  The contraction index is the grid point (the row of the n x ld blocks), so the operand
// tiles are transposed while they are staged: each thread loads a 4 x 4 patch (4 grid points x
// 4 columns) with 16-byte loads, splits it, and writes 16-byte K-chunks into the 128B-swizzled
// K-major layout the MMA reads.
//
// Accumulation: the tensor core adds into its FP32 accumulator with truncation, so a long run of
// additions drifts by about (run length) x 2^-24 of the accumulated value (for <U,U> = I that is
// a systematic error of the orthogonality).  Each 32-point slab therefore starts a fresh
// accumulator (four TMEM accumulators in turn), which is drained into FP32 registers
// (round-to-nearest additions); a chunk's FP32 sums are its partial tile, and the partials are
// added over the chunks in a fixed order as triples of floats (sums.cuh).
//
// Roles (k_gram_ws), meeting only at mbarriers: eight warps stage slabs into a ring of three,
// one thread issues the MMAs (16 a slab, 74 clocks each: the bound), eight warps drain.  With
// every warp staging, waiting and draining in lockstep (one CTA per item) a slab took 3050
// clocks, 1190 of them the MMAs.  262144 x 128, C, S and D: 216 us, 301 before (an MMA takes 111
// clocks beside the staging: both load shared memory).
#include <type_traits>

#include "common.cuh"
#include "kernels.cuh"
#include "sums.cuh"
#include "tc.cuh"

namespace opevo {

namespace {

constexpr int kTM = 128;                      // output tile (rows and columns)
constexpr int kRedLanes = 64, kRedGroups = 4;  // reduce: elements x split groups of a CTA
constexpr int kReduceSlices = kTM * kTM / kRedLanes;
constexpr int kKS = 32;                       // grid points per slab (one 128-byte K row)
constexpr int kPiece = kTM * 128;             // bytes of one operand piece (128 rows x 128 B)
constexpr int kStage = 4 * kPiece;            // A_hi, A_lo, B_hi, B_lo
constexpr int kRing = 3;                        // staged slabs
constexpr int kAcc = 4;                         // TMEM accumulators
constexpr int kSmem = kRing * kStage + 1024;    // + alignment slack
constexpr int kStageWarps = 8, kDrainWarps = 8;
constexpr int kThreadsWs = 32 * (kStageWarps + kDrainWarps + 1);
constexpr uint64_t kWaitNs = 2000000000ull;
constexpr uint32_t kIdesc = tc::idesc_tf32(kTM, kTM);

enum { PROD_C = 0, PROD_S = 1, PROD_D = 2 };

__device__ __forceinline__ void decode_job(int idx, int mask, int nt, int *prod, int *ti, int *tj) {
  int pr = 0;
  for (; pr < 3; ++pr) {
    if (!((mask >> pr) & 1)) continue;
    const int cnt = pr == PROD_C ? nt * nt : nt * (nt + 1) / 2;
    if (idx < cnt) break;
    idx -= cnt;
  }
  *prod = pr;
  if (pr == PROD_C) {
    *ti = idx / nt;
    *tj = idx % nt;
  } else {
    int i = 0;
    while (idx >= nt - i) {
      idx -= nt - i;
      ++i;
    }
    *ti = i;
    *tj = i + idx;
  }
}

// 4 grid points x 4 columns of X starting at (row, col); zero outside [r1) x [ld).
__device__ __forceinline__ void load_patch(const float *__restrict__ X, long long row, long long r1,
                                           int col, int ld, float (&v)[4][4]) {
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
    if (row + r < r1 && col < ld) x = __ldg(reinterpret_cast<const float4 *>(X + (row + r) * ld + col));
    v[r][0] = x.x;
    v[r][1] = x.y;
    v[r][2] = x.z;
    v[r][3] = x.w;
  }
}

// The patch at p (row pitch ld) of a slab that lies inside the chunk; `in`: its columns exist.
__device__ __forceinline__ void load_patch_in(const float *__restrict__ p, int ld, bool in,
                                              float (&v)[4][4]) {
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
    if (in) x = __ldg(reinterpret_cast<const float4 *>(p + r * ld));
    v[r][0] = x.x;
    v[r][1] = x.y;
    v[r][2] = x.z;
    v[r][3] = x.w;
  }
}

// Split the patch and store it transposed: operand row m = 4q + e gets the
// K-chunk kq = (v[0][e], .., v[3][e]).  Without `split` only tf32(x) is stored.
__device__ __forceinline__ void store_patch(uint8_t *hi, uint8_t *lo, int q, int kq,
                                            const float (&v)[4][4], bool split) {
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    float4 h, l;
    tc::split_tf32(v[0][e], h.x, l.x);
    tc::split_tf32(v[1][e], h.y, l.y);
    tc::split_tf32(v[2][e], h.z, l.z);
    tc::split_tf32(v[3][e], h.w, l.w);
    const uint32_t off = tc::sw128_offset(4 * q + e, kq);
    *reinterpret_cast<float4 *>(hi + off) = h;
    if (split) *reinterpret_cast<float4 *>(lo + off) = l;
  }
}

// One item: output tile of A^T B over grid points [r0, r1), rows ca .., columns cb ..; its partial
// tile is written column by column (element (i, j) at j 128 + i: the drain threads own rows, so a
// warp writes 128 consecutive bytes) as FP32, or added to an FP64 tile with atomics.
struct GramTask {
  const float *A, *B;
  int ld, ca, cb, nslab;
  bool same;  // A and B are the same columns: staged once
  long long r0, r1;
  float *part;
  double *sum;  // not null: atomics instead of `part`
  int *err;
};

__device__ __forceinline__ void set_task(GramTask *t, long long n, int ld, const float *U,
                                         const float *W, int prod, int ti, int tj, long long r0,
                                         long long r1) {
  t->A = (prod == PROD_D) ? U : W;
  t->B = (prod == PROD_S) ? W : U;
  t->ld = ld;
  t->ca = ti * kTM;
  t->cb = tj * kTM;
  t->same = (t->A == t->B) && ti == tj;
  t->r0 = r0;
  t->r1 = r1 < n ? r1 : n;
  t->nslab = t->r1 > r0 ? (int)((t->r1 - r0 + kKS - 1) / kKS) : 0;
}

// Items of one problem: split s of job j is item s njobs + j.
struct GramSrc {
  long long n, rps, items;
  int ld, mask, nt, njobs;
  const float *U, *W;
  float *part;
  double *sum;
  int *err;
  __device__ __forceinline__ bool get(long long i, GramTask *t) const {
    const int job = (int)(i % njobs);
    const long long r0 = i / njobs * rps;
    int prod, ti, tj;
    decode_job(job, mask, nt, &prod, &ti, &tj);
    set_task(t, n, ld, U, W, prod, ti, tj, r0, r0 + rps);
    t->part = part + i * (kTM * kTM);
    t->sum = sum ? sum + (long long)job * (kTM * kTM) : nullptr;
    t->err = err;
    return true;
  }
};
// Items of a batch (problem, job, chunk), all three products; a frozen problem's are skipped.
struct GramBatchSrc {
  long long items;
  const BatchProb *B;
  const GramItem *list;
  int parity;
  __device__ __forceinline__ bool get(long long i, GramTask *t) const {
    const GramItem it = list[i];
    const BatchProb &pb = B[it.prob];
    if (*pb.frozen) return false;
    int prod, ti, tj;
    decode_job(it.job, 7, (pb.ld + kTM - 1) / kTM, &prod, &ti, &tj);
    set_task(t, pb.g.n, pb.ld, pb.U[parity], pb.W, prod, ti, tj, it.r0, it.r1);
    t->part = pb.gram_part + ((long long)it.split * pb.gram_jobs + it.job) * (kTM * kTM);
    t->sum = nullptr;
    t->err = pb.err;
    return true;
  }
};

__device__ __forceinline__ bool warp_wait(uint64_t *bar, uint32_t parity, volatile int *abort) {
  int ok = 0;
  if ((threadIdx.x & 31) == 0) ok = tc::wait_or_abort(bar, parity, abort, kWaitNs) ? 1 : 0;
  return __shfl_sync(0xffffffffu, ok, 0) != 0;
}

template <typename Src>
__global__ void __launch_bounds__(kThreadsWs, 1) k_gram_ws(const Src src, int split) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ uint64_t full[kRing], empty[kRing], done[kAcc], freed[kAcc];
  __shared__ uint32_t tmem_sh;
  __shared__ int abort_sh;
  uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  constexpr int kMma = kStageWarps + kDrainWarps;
  if (warp == kMma) tc::tmem_alloc(&tmem_sh, kAcc * kTM);
  if (t == 0) {
    for (int i = 0; i < kRing; ++i) {
      tc::mbar_init(&full[i], kStageWarps);
      tc::mbar_init(&empty[i], 1);
    }
    for (int i = 0; i < kAcc; ++i) {
      tc::mbar_init(&done[i], 1);
      tc::mbar_init(&freed[i], kDrainWarps);
    }
    tc::fence_mbar_init();
    abort_sh = 0;
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = tmem_sh;
  volatile int *abort = &abort_sh;
  int *err = nullptr;  // of the last item this thread saw

  if (warp < kStageWarps) {
    // ---- staging: points 4 kq .. of a slab, columns 4 q .. of the tile
    const int kq = t & 7, q = t >> 3;
    uint32_t slot = 0, phase = 1, g = 0;  // phase of the slot's last release
    bool ok = true;
    for (long long i = blockIdx.x; i < src.items && ok; i += gridDim.x) {
      GramTask k;
      if (!src.get(i, &k)) continue;
      err = k.err;
      float va[4][4], vb[4][4];
      if (k.nslab > 0) {
        load_patch(k.A, k.r0 + 4 * kq, k.r1, k.ca + 4 * q, k.ld, va);
        if (!k.same) load_patch(k.B, k.r0 + 4 * kq, k.r1, k.cb + 4 * q, k.ld, vb);
      }
      // lines of slab kAhead on (row t / 4, 32 columns t % 4): A by the first 128 threads, B by the
      // others; the loads of a slab then come from L2
      constexpr int kAhead = 3;
      const int pcol = (t < 128 ? k.ca : k.cb) + 32 * (t & 3), prow = (t & 127) >> 2;
      const bool pin = pcol < k.ld && (t < 128 || !k.same);
      const float *pf = (t < 128 ? k.A : k.B) + (k.r0 + kAhead * kKS + prow) * k.ld + pcol;
      const int pslabs = pin ? (int)((k.r1 - k.r0 - prow + kKS - 1) / kKS) - kAhead : 0;
      // this thread's patches of the next slab
      const bool ina = k.ca + 4 * q < k.ld, inb = k.cb + 4 * q < k.ld;
      const float *pa = k.A + (k.r0 + kKS + 4 * kq) * k.ld + k.ca + 4 * q;
      const float *pb = k.B + (k.r0 + kKS + 4 * kq) * k.ld + k.cb + 4 * q;
      const int inside = (int)((k.r1 - k.r0) / kKS), step = kKS * k.ld;
      for (int s = 0; s < k.nslab; ++s, ++g) {
        if (g >= kRing && !warp_wait(&empty[slot], phase, abort)) {
          ok = false;
          break;
        }
        uint8_t *stage = smem + slot * kStage;
        store_patch(stage, stage + kPiece, q, kq, va, split != 0);
        if (!k.same) store_patch(stage + 2 * kPiece, stage + 3 * kPiece, q, kq, vb, split != 0);
        // (the loads of the next slab come after the fence, which waits for every access before it)
        tc::fence_async_smem();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&full[slot]);
        if (s + 1 < inside) {
          load_patch_in(pa, k.ld, ina, va);
          if (!k.same) load_patch_in(pb, k.ld, inb, vb);
        } else if (s + 1 < k.nslab) {  // the chunk's ragged last slab
          const long long r = k.r0 + (long long)(s + 1) * kKS + 4 * kq;
          load_patch(k.A, r, k.r1, k.ca + 4 * q, k.ld, va);
          if (!k.same) load_patch(k.B, r, k.r1, k.cb + 4 * q, k.ld, vb);
        }
        if (s < pslabs) asm volatile("prefetch.global.L2 [%0];" ::"l"(pf) : "memory");
        pa += step;
        pb += step;
        pf += step;
        if (++slot == kRing) {
          slot = 0;
          phase ^= 1;
        }
      }
    }
  } else if (warp == kMma) {
    if (lane == 0) {
      uint32_t slot = 0, phase = 0, g = 0;
      bool ok = true;
      for (long long i = blockIdx.x; i < src.items && ok; i += gridDim.x) {
        GramTask k;
        if (!src.get(i, &k)) continue;
        err = k.err;
        for (int s = 0; s < k.nslab; ++s, ++g) {
          const uint32_t a = g % kAcc;
          if ((g >= kAcc && !tc::wait_or_abort(&freed[a], (g / kAcc - 1) & 1, abort, kWaitNs)) ||
              !tc::wait_or_abort(&full[slot], phase, abort, kWaitNs)) {
            ok = false;
            break;
          }
          tc::tc_fence_after();
          const uint32_t base = tc::smem_u32(smem + slot * kStage);
          const uint32_t bbase = k.same ? base : base + 2 * kPiece;
          const uint32_t d = tmem + a * kTM;
#pragma unroll
          for (int kk = 0; kk < kKS / 8; ++kk) {
            const uint64_t ah = tc::desc_sw128(base + kk * 32);
            const uint64_t al = tc::desc_sw128(base + kPiece + kk * 32);
            const uint64_t bh = tc::desc_sw128(bbase + kk * 32);
            const uint64_t bl = tc::desc_sw128(bbase + kPiece + kk * 32);
            tc::mma_tf32(d, ah, bh, kIdesc, kk > 0 ? 1u : 0u);
            if (split) {
              tc::mma_tf32(d, ah, bl, kIdesc, 1u);
              tc::mma_tf32(d, al, bh, kIdesc, 1u);
              tc::mma_tf32(d, al, bl, kIdesc, 1u);
            }
          }
          tc::mma_commit(&empty[slot]);
          tc::mma_commit(&done[a]);
          if (++slot == kRing) {
            slot = 0;
            phase ^= 1;
          }
        }
      }
      // MMAs issued but not drained finish before the TMEM is freed
      if (!ok && g > 0) (void)tc::mbar_wait(&done[(g - 1) % kAcc], ((g - 1) / kAcc) & 1);
    }
  } else {
    // ---- drain: accumulator row (TMEM lane) 32 (warp % 4) + lane, columns 64 half ..
    const int quarter = warp & 3, half = (warp - kStageWarps) >> 2, row = quarter * 32 + lane;
    const uint32_t tb = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(half * 64);
    uint32_t g = 0;
    bool ok = true;
    for (long long i = blockIdx.x; i < src.items && ok; i += gridDim.x) {
      GramTask k;
      if (!src.get(i, &k)) continue;
      err = k.err;
      float acc[64];
#pragma unroll
      for (int e = 0; e < 64; ++e) acc[e] = 0.f;
      for (int s = 0; s < k.nslab; ++s, ++g) {
        const uint32_t a = g % kAcc;
        if (!warp_wait(&done[a], (g / kAcc) & 1, abort)) {
          ok = false;
          break;
        }
        tc::tc_fence_after();
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          float v[16];
          tc::tmem_ld16(tb + a * kTM + (uint32_t)(c * 16), v);
#pragma unroll
          for (int e = 0; e < 16; ++e) acc[c * 16 + e] += v[e];
        }
        tc::tc_fence_before();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&freed[a]);
      }
      if (!ok) break;
      const int at = half * 64 * kTM + row;
      if (k.sum) {
#pragma unroll
        for (int e = 0; e < 64; ++e) atomicAdd(k.sum + at + e * kTM, (double)acc[e]);
      } else {
#pragma unroll
        for (int e = 0; e < 64; ++e) k.part[at + e * kTM] = acc[e];
      }
    }
  }
  tc::tc_fence_before();
  __syncthreads();
  if (warp == kMma) {
    tc::tc_fence_after();
    tc::tmem_dealloc(tmem, kAcc * kTM);
  }
  if (lane == 0 && abort_sh && err) atomicExch(err, 1);
}

// ---- BF16 variants -------------------------------------------------------------------
// The same tiling with BF16 operands: every value is split in three BF16 pieces
// (x = b0 + b1 + b2 to 2^-24), and each product takes the six MMAs (kind::f16) whose
// pieces have index sum <= 2 (one piece and one MMA in the plain BF16 mode); a slab is
// 64 grid points (one 128-byte row of BF16 K values).  The staging patch is 8 grid points x 4 columns; the register buffer runs
// one slab ahead.
constexpr int kKSb = 64;
constexpr int kStageB16 = 6 * kPiece;  // A0 A1 A2 B0 B1 B2
constexpr int kSmemB16 = 2 * kStageB16 + 1024;
constexpr uint32_t kIdescB16 = tc::idesc_bf16(kTM, kTM);

__device__ __forceinline__ void load_patch8(const float *__restrict__ X, long long row,
                                            long long r1, int col, int ld, float (&v)[8][4]) {
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
    if (row + r < r1 && col < ld) x = __ldg(reinterpret_cast<const float4 *>(X + (row + r) * ld + col));
    v[r][0] = x.x;
    v[r][1] = x.y;
    v[r][2] = x.z;
    v[r][3] = x.w;
  }
}

// operand row m = 4q + e gets the K-chunk kq (8 BF16 values) of each of the three pieces
// (of the first piece, bf16(x), only, when three == false)
__device__ __forceinline__ void store_patch8(uint8_t *piece0, int q, int kq, const float (&v)[8][4],
                                             bool three) {
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    float col[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) col[r] = v[r][e];
    uint4 c0, c1, c2;
    tc::split8_bf16x3(col, c0, c1, c2);
    const uint32_t off = tc::sw128_offset(4 * q + e, kq);
    *reinterpret_cast<uint4 *>(piece0 + off) = c0;
    if (three) {
      *reinterpret_cast<uint4 *>(piece0 + kPiece + off) = c1;
      *reinterpret_cast<uint4 *>(piece0 + 2 * kPiece + off) = c2;
    }
  }
}

__device__ __forceinline__ void gram_bf16_body(long long n, int ld, const float *__restrict__ U,
                                               const float *__restrict__ W, int prod, int ti,
                                               int tj, long long r0, long long r1,
                                               float *__restrict__ dst_tile, int *err,
                                               bool three) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ uint64_t mbar[2];
  __shared__ uint32_t tmem_base_sh;
  __shared__ int abort_sh;
  uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);

  const float *A = (prod == PROD_D) ? U : W;
  const float *B = (prod == PROD_S) ? W : U;
  const int ca = ti * kTM, cb = tj * kTM;
  const bool same = (A == B) && (ca == cb);
  if (r1 > n) r1 = n;
  const int nslab = r1 > r0 ? (int)((r1 - r0 + kKSb - 1) / kKSb) : 0;

  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int kq = t & 7, q = t >> 3;
  const int row = (warp & 3) * 32 + lane;
  const int half = warp >> 2;

  if (warp == 0) tc::tmem_alloc(&tmem_base_sh, 2 * kTM);
  if (t == 0) {
    tc::mbar_init(&mbar[0], 1);
    tc::mbar_init(&mbar[1], 1);
    tc::fence_mbar_init();
    abort_sh = 0;
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = tmem_base_sh;
  const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;

  float acc[64];
#pragma unroll
  for (int i = 0; i < 64; ++i) acc[i] = 0.f;

  auto drain = [&](int s) -> bool {
    const int a = s & 1;
    if (t == 0 && !tc::mbar_wait(&mbar[a], (uint32_t)((s >> 1) & 1))) abort_sh = 1;
    __syncthreads();
    if (abort_sh) return false;
    tc::tc_fence_after();
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      float v[32];
      tc::tmem_ld32(tmem + lane_base + (uint32_t)(a * kTM + half * 64 + c * 32), v);
#pragma unroll
      for (int i = 0; i < 32; ++i) acc[c * 32 + i] += v[i];
    }
    tc::tc_fence_before();
    return true;
  };

  float va[8][4], vb[8][4];
  if (nslab > 0) {
    load_patch8(A, r0 + 8 * kq, r1, ca + 4 * q, ld, va);
    if (!same) load_patch8(B, r0 + 8 * kq, r1, cb + 4 * q, ld, vb);
  }
  bool ok = true;
  for (int s = 0; s < nslab && ok; ++s) {
    const int st = s & 1;
    uint8_t *stage = smem + st * kStageB16;
    // stage st was read by the MMAs of slab s-2, which the drain of slab s-2 waited for
    store_patch8(stage, q, kq, va, three);
    if (!same) store_patch8(stage + 3 * kPiece, q, kq, vb, three);
    tc::fence_async_smem();
    tc::tc_fence_before();
    __syncthreads();
    // (after the fence, which waits for every access before it)
    if (s + 1 < nslab) {
      const long long r = r0 + (long long)(s + 1) * kKSb + 8 * kq;
      load_patch8(A, r, r1, ca + 4 * q, ld, va);
      if (!same) load_patch8(B, r, r1, cb + 4 * q, ld, vb);
    }
    if (t == 0) {
      tc::tc_fence_after();
      const uint32_t base = tc::smem_u32(stage);
      const uint32_t bbase = same ? base : base + 3 * kPiece;
      const uint32_t d = tmem + (uint32_t)(st * kTM);
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) {
        uint64_t a[3], b[3];
#pragma unroll
        for (int r = 0; r < 3; ++r) {
          a[r] = tc::desc_sw128(base + r * kPiece + kk * 32);
          b[r] = tc::desc_sw128(bbase + r * kPiece + kk * 32);
        }
        tc::mma_bf16(d, a[0], b[0], kIdescB16, kk > 0 ? 1u : 0u);
        if (three) {
          tc::mma_bf16(d, a[0], b[1], kIdescB16, 1u);
          tc::mma_bf16(d, a[1], b[0], kIdescB16, 1u);
          tc::mma_bf16(d, a[0], b[2], kIdescB16, 1u);
          tc::mma_bf16(d, a[1], b[1], kIdescB16, 1u);
          tc::mma_bf16(d, a[2], b[0], kIdescB16, 1u);
        }
      }
      tc::mma_commit(&mbar[st]);
    }
    if (s >= 1) ok = drain(s - 1);
  }
  if (ok && nslab > 0) ok = drain(nslab - 1);
  __syncthreads();
  if (!ok || abort_sh) {
    if (t == 0) atomicExch(err, 1);
  } else {
    float *dst = dst_tile + half * 64 * kTM + row;  // column by column
#pragma unroll
    for (int i = 0; i < 64; ++i) dst[i * kTM] = acc[i];
  }
  tc::tc_fence_before();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, 2 * kTM);
}

__global__ void __launch_bounds__(256, 1)
    k_gram_bf16(long long n, int ld, const float *__restrict__ U, const float *__restrict__ W,
                int mask, int nt, int njobs, long long rows_per_split, float *__restrict__ part,
                int *err, int three) {
  int prod, ti, tj;
  decode_job(blockIdx.x, mask, nt, &prod, &ti, &tj);
  const long long r0 = (long long)blockIdx.y * rows_per_split;
  gram_bf16_body(n, ld, U, W, prod, ti, tj, r0, r0 + rows_per_split,
                 part + ((long long)blockIdx.y * njobs + blockIdx.x) * (kTM * kTM), err,
                 three != 0);
}

// A running sum of partials: FP32 ones as a triple of floats (sums.cuh; the FP64 pipe would take
// longer than reading them), or FP64.
template <typename P> struct SplitSum;
template <> struct SplitSum<float> : Sum3 {};
template <> struct SplitSum<double> {
  double s = 0.0;
  __device__ __forceinline__ void add(double v) { s += v; }
  __device__ __forceinline__ void add(const SplitSum &o) { s += o.s; }
  __device__ __forceinline__ double value() const { return s; }
};

// out(i, j) = the summed tile element, zero outside p x p, both triangles of S and D.
// A CTA of kRedLanes x kRedGroups threads: group g sums every kRedGroups-th split, the first
// group adds the sums up.  One thread per element and all its splits was a serial chain of up to
// 228 loads and two-sums: 24 us at 262144 x 128, now 15 (13 with pairs of floats).  An element whose sum leaves the FP32 range
// is summed in FP64.
template <typename P>
__device__ __forceinline__ void reduce_tile(int prod, int ti, int tj, int slice, int slices,
                                            const P *part, long long stride, int nsplit, int p,
                                            int ld, double *out) {
  __shared__ SplitSum<P> sh[kRedGroups - 1][kRedLanes];
  const int lane = threadIdx.x % kRedLanes, g = threadIdx.x / kRedLanes;
  for (int e0 = slice * kRedLanes; e0 < kTM * kTM; e0 += slices * kRedLanes) {
    const int e = e0 + lane, i = ti * kTM + e % kTM, j = tj * kTM + e / kTM;
    SplitSum<P> s;
    if (i < p && j < p) {
#pragma unroll 8
      for (int sp = g; sp < nsplit; sp += kRedGroups) s.add(part[e + sp * stride]);
    }
    if (g) sh[g - 1][lane] = s;
    __syncthreads();
    if (g == 0 && i < ld && j < ld) {
#pragma unroll
      for (int q = 0; q < kRedGroups - 1; ++q) s.add(sh[q][lane]);
      double v = (i < p && j < p) ? s.value() : 0.0;
      if constexpr (std::is_same<P, float>::value)
        if (!s.finite()) v = sum64(part + e, stride, nsplit);
      out[(long long)i * ld + j] = v;
      if (prod != PROD_C && ti != tj) out[(long long)j * ld + i] = v;
    }
    __syncthreads();
  }
}

// Batched reduce: grid (jobs, problems, element slices).
// (eight CTAs an SM: the sums are a chain of loads)
__global__ void __launch_bounds__(kRedLanes * kRedGroups, 8)
    k_b_gram_tc_reduce(const BatchProb *__restrict__ Bp) {
  const BatchProb &pb = Bp[blockIdx.y];
  if (*pb.frozen || (int)blockIdx.x >= pb.gram_jobs) return;
  int prod, ti, tj;
  decode_job(blockIdx.x, 7, (pb.ld + kTM - 1) / kTM, &prod, &ti, &tj);
  reduce_tile(prod, ti, tj, blockIdx.z, gridDim.z,
              pb.gram_part + (long long)blockIdx.x * (kTM * kTM),
              (long long)pb.gram_jobs * (kTM * kTM), pb.n_gram_splits, pb.p, pb.ld,
              prod == PROD_C ? pb.C : (prod == PROD_S ? pb.S : pb.D));
}

template <typename P>
__global__ void __launch_bounds__(kRedLanes * kRedGroups, 8)
    k_gram_tc_reduce(int mask, int nt, int njobs, int nsplit, const P *__restrict__ part, int p,
                     int ld, double *C, double *S, double *D) {
  int prod, ti, tj;
  decode_job(blockIdx.x, mask, nt, &prod, &ti, &tj);
  reduce_tile(prod, ti, tj, blockIdx.y, gridDim.y, part + (long long)blockIdx.x * (kTM * kTM),
              (long long)njobs * (kTM * kTM), nsplit, p, ld,
              prod == PROD_C ? C : (prod == PROD_S ? S : D));
}

template <typename Src> op_status launch_gram_ws(const Src &src, int split, cudaStream_t st) {
  OP_CUDA(cudaFuncSetAttribute(k_gram_ws<Src>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem));
  const long long grid = src.items < num_sms() ? src.items : num_sms();
  if (grid < 1) return OP_OK;
  k_gram_ws<Src><<<(unsigned)grid, kThreadsWs, kSmem, st>>>(src, split);
  count_launch();
  OP_LAUNCH("k_gram_ws");
  return OP_OK;
}

int tc_jobs(int nt, int mask) {
  return ((mask & 1) ? nt * nt : 0) + ((mask & 2) ? nt * (nt + 1) / 2 : 0) +
         ((mask & 4) ? nt * (nt + 1) / 2 : 0);
}

}  // namespace

// Splits: about three CTAs per SM over all jobs, at least 512 grid points each.
static void plan_tc(long long n, int njobs, int *nsplit, long long *rps) {
  long long ns = (3 * num_sms() + njobs - 1) / njobs;
  const long long maxs = (n + 511) / 512;
  if (ns > maxs) ns = maxs;
  if (ns < 1) ns = 1;
  long long r = (n + ns - 1) / ns;
  r = (r + kKS - 1) / kKS * kKS;
  *rps = r;
  *nsplit = (int)((n + r - 1) / r);
}

size_t gram_tc_workspace_bytes(long long n, int ld) {
  (void)n;
  // plan_tc gives nj * nsplit <= 3 * num_sms() + nj for every subset of the products
  const int nt = (ld + kTM - 1) / kTM;
  return (size_t)(3 * num_sms() + tc_jobs(nt, 7)) * kTM * kTM * sizeof(double) + 256;
}

op_status gram_tc(long long n, int p, int ld, const float *U, const float *W, double *C, double *S,
                  double *D, void *ws, size_t ws_bytes, int *err, cudaStream_t st, int split) {
  if (ld % 8 != 0 || p > ld || n < 1) {
    set_error("gram_tc: bad sizes n=%lld p=%d ld=%d", n, p, ld);
    return OP_ERR_ARG;
  }
  const int nt = (ld + kTM - 1) / kTM;
  const int mask = (C ? 1 : 0) | (S ? 2 : 0) | (D ? 4 : 0);
  const int nj = tc_jobs(nt, mask);
  if (nj == 0) return OP_OK;
  int nsplit;
  long long rps;
  plan_tc(n, nj, &nsplit, &rps);
  const size_t need = (size_t)nj * nsplit * kTM * kTM * sizeof(double);
  if (!ws || ws_bytes < need) {
    set_error("gram_tc: workspace too small (%zu < %zu)", ws_bytes, need);
    return OP_ERR_ARG;
  }
  float *part = (float *)ws;
  if (split >= 2) {  // BF16: 2 three pieces, 3 one piece
    OP_CUDA(cudaFuncSetAttribute(k_gram_bf16, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 kSmemB16));
    k_gram_bf16<<<dim3(nj, nsplit), 256, kSmemB16, st>>>(n, ld, U, W, mask, nt, nj, rps, part,
                                                          err, split == 2 ? 1 : 0);
    count_launch();
    OP_LAUNCH("k_gram_bf16");
  } else {
    OP_TRY(launch_gram_ws(GramSrc{n, rps, (long long)nj * nsplit, ld, mask, nt, nj, U, W, part,
                                  nullptr, err}, split, st));
  }
  k_gram_tc_reduce<float><<<dim3(nj, kReduceSlices), kRedLanes * kRedGroups, 0, st>>>(mask, nt, nj, nsplit, part, p, ld,
                                                             C, S, D);
  count_launch();
  OP_LAUNCH("k_gram_tc_reduce");
  return OP_OK;
}

// As gram_tc() (the same chunks of grid points, so the same FP32 runs and rounding
// bound), but the chunk partials of each output tile are added into one FP64 tile with
// atomics: part_bytes must hold one 128 x 128 FP64 tile per output tile.  The FP64
// chunk sums are taken in whatever order the CTAs finish.
op_status gram_tc_fixed_scratch(long long n, int p, int ld, const float *U, const float *W,
                                double *C, double *S, double *D, void *part, size_t part_bytes,
                                int *err, cudaStream_t st) {
  if (ld % 8 != 0 || p > ld || n < 1) {
    set_error("gram_tc: bad sizes n=%lld p=%d ld=%d", n, p, ld);
    return OP_ERR_ARG;
  }
  const int nt = (ld + kTM - 1) / kTM;
  const int mask = (C ? 1 : 0) | (S ? 2 : 0) | (D ? 4 : 0);
  const int nj = tc_jobs(nt, mask);
  if (nj == 0) return OP_OK;
  const size_t tile_bytes = (size_t)kTM * kTM * sizeof(double);
  if (part_bytes < (size_t)nj * tile_bytes) {
    set_error("gram_tc: %d output tiles need %zu bytes of partials, the fixed scratch holds %zu",
              nj, (size_t)nj * tile_bytes, part_bytes);
    return OP_ERR_ARG;
  }
  int nsplit;
  long long rps;
  plan_tc(n, nj, &nsplit, &rps);
  OP_CUDA(cudaMemsetAsync(part, 0, (size_t)nj * tile_bytes, st));
  OP_TRY(launch_gram_ws(GramSrc{n, rps, (long long)nj * nsplit, ld, mask, nt, nj, U, W, nullptr,
                                (double *)part, err}, 1, st));
  k_gram_tc_reduce<double><<<dim3(nj, kReduceSlices), kRedLanes * kRedGroups, 0, st>>>(mask, nt, nj, 1, (const double *)part,
                                                             p, ld, C, S, D);
  count_launch();
  OP_LAUNCH("k_gram_tc_reduce");
  return OP_OK;
}

op_status launch_b_gram(const BatchProb *B, const GramItem *items, int nitems, int nprob,
                        int parity, cudaStream_t st) {
  OP_TRY(launch_gram_ws(GramBatchSrc{nitems, B, items, parity}, 1, st));
  // at most 3 * 8 * 8 + ... jobs for ld <= 1024: grid x covers the largest job count
  k_b_gram_tc_reduce<<<dim3(tc_jobs(8, 7), nprob, 8), kRedLanes * kRedGroups, 0, st>>>(B);
  count_launch();
  OP_LAUNCH("k_b_gram_tc_reduce");
  return OP_OK;
}

size_t gram_tc_tile_bytes() { return (size_t)kTM * kTM * sizeof(double); }
int gram_tc_jobs_all(int ld) { return tc_jobs((ld + kTM - 1) / kTM, 7); }

}  // namespace opevo
