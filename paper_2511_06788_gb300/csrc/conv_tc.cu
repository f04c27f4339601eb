// Forward convolution of the learned warm start (opnet.h) on the tensor cores: an
// implicit GEMM with BF16 operands and FP32 accumulation in TMEM (tcgen05.mma
// kind::f16), bias and SiLU in the epilogue.
//
//   out[m][co] = b[co] + sum_k A[m][k] W[k][co],   A[m][t Cin + ci] = X[m + off_t][ci]
//
// with X channels-last [point][ci] on an N^3 grid, taps t = (dz+1) 9 + (dy+1) 3 + (dx+1)
// (27 taps, zero outside the grid) or the point itself (1 tap).
//
// Tiling: tiles of 128 grid points (the MMA's M), all output channels at once
// (N = Cout rounded up to 16, at most 128), one FP32 accumulator a tile, K in order.  Two kernels with
// the same products in the same order (bit-identical results):
//
// k_conv_tma (Cin a multiple of 8, or few K values).  A first pass rounds X to BF16 once, into a copy with one
// point of zeros around the grid, so a tap of a run of points is the same run shifted by a
// constant number of rows: TMA loads A as boxes of 128 rows, 64, 32 or 16 channels wide, and two
// 8-wide boxes for a K step that straddles two taps.  A narrow box takes as long as a wide one, so
// where it saves a third of them the copy holds the three taps along x of a point side by side
// (merge_x).  No value is gathered or converted again; the tiles run over the padded points
// between the first and the last grid point (about 9 % more at 48^3).  Up to three persistent
// CTAs an SM: one thread loads A, one B (a box of 64 K values a stage, whatever pieces A comes
// in), one issues the MMAs into two accumulators in turn, four warps write the outputs of the
// other.  With one CTA a tile the first loads and the outputs stood beside nothing, and 937 tiles
// made four waves where three and a bit were work.  Bound by the copies: 27 taps of narrow rows.
// The 11 layers at 48^3, widths 24, 48, 96, p = 64: 0.39 ms and 0.12 ms for the BF16 copies; one
// CTA a tile and a box per tap 0.51 and 0.10, by k_conv_tc 1.37 ms.
//
// k_conv_tc (other layers, and scratch without room for the copy).  K in slabs of 64; the 256 threads gather a slab of A from FP32 (27
// taps, zero padding) and convert it, one thread issues the slab's MMAs; the gather of slab
// s + 1 runs while the tensor core works on slab s.
//
// Every wait is bounded; a wait that gives up sets the error word and the CTA writes nothing.
#include <cuda_bf16.h>

#include <algorithm>

#include "common.cuh"
#include "kernels.cuh"
#include "tc.cuh"
#include "tma.cuh"

namespace opevo {
namespace {

constexpr int kCM = 128;                 // points per CTA (MMA M)
constexpr int kCK = 64;                  // K per slab (BF16: 128 bytes per operand row)
constexpr int kAPiece = kCM * 128;       // 16 KB
constexpr int kBMax = 128 * 128;         // up to 128 output channels x 128 bytes
constexpr int kCStage = kAPiece + kBMax;
constexpr int kCSmem = 2 * kCStage + 1024;

__device__ __forceinline__ uint32_t bf16_bits(float x) {
  return (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(x));
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float (&v)[8]) {
  uint32_t r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                 "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}

// Wt[co][k] = bf16(W[k][co]) for co < cout, k < K; zero in the padding (co < coutp, k < Kp).
__global__ void k_conv_wt(const float *__restrict__ W, int K, int cout, int Kp, int coutp,
                          uint16_t *__restrict__ Wt) {
  const long long total = (long long)coutp * Kp;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const int co = (int)(e / Kp), k = (int)(e % Kp);
    const float w = (co < cout && k < K) ? W[(long long)k * cout + co] : 0.f;
    Wt[e] = (uint16_t)bf16_bits(w);
  }
}

struct ConvTc {
  const float *X;       // [n][cin]
  const uint16_t *Wt;   // [coutp][Kp] BF16
  const float *bias;    // [cout] or null
  float *Z, *A;         // [n][cout] each, or null
  int N, taps, cin, cout, coutp, K, Kp;
  int *err;
};

// Eight consecutive K values k0 .. k0 + 7 of operand row (point) m, as four BF16 pairs.
__device__ __forceinline__ uint4 gather8(const ConvTc &a, int x, int y, int z, bool in, int k0) {
  float v[8];
  if (in && a.cin % 8 == 0 && k0 < a.K) {
    // one tap, eight consecutive channels (k0 and cin are multiples of 8)
    const int t = k0 / a.cin, ci = k0 - t * a.cin;
    int dx = 0, dy = 0, dz = 0;
    if (a.taps == 27) {
      dx = t % 3 - 1;
      dy = (t / 3) % 3 - 1;
      dz = t / 9 - 1;
    }
    const int xx = x + dx, yy = y + dy, zz = z + dz;
    if (xx >= 0 && xx < a.N && yy >= 0 && yy < a.N && zz >= 0 && zz < a.N) {
      const float4 *src = reinterpret_cast<const float4 *>(
          a.X + (((long long)zz * a.N + yy) * a.N + xx) * a.cin + ci);
      const float4 p = __ldg(src), q = __ldg(src + 1);
      v[0] = p.x; v[1] = p.y; v[2] = p.z; v[3] = p.w;
      v[4] = q.x; v[5] = q.y; v[6] = q.z; v[7] = q.w;
    } else {
#pragma unroll
      for (int e = 0; e < 8; ++e) v[e] = 0.f;
    }
  } else {
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int k = k0 + e;
      float w = 0.f;
      if (in && k < a.K) {
        const int t = k / a.cin, ci = k - t * a.cin;
        int dx = 0, dy = 0, dz = 0;
        if (a.taps == 27) {
          dx = t % 3 - 1;
          dy = (t / 3) % 3 - 1;
          dz = t / 9 - 1;
        }
        const int xx = x + dx, yy = y + dy, zz = z + dz;
        if (xx >= 0 && xx < a.N && yy >= 0 && yy < a.N && zz >= 0 && zz < a.N)
          w = __ldg(a.X + (((long long)zz * a.N + yy) * a.N + xx) * a.cin + ci);
      }
      v[e] = w;
    }
  }
  return make_uint4(bf16_bits(v[0]) | (bf16_bits(v[1]) << 16), bf16_bits(v[2]) | (bf16_bits(v[3]) << 16),
                    bf16_bits(v[4]) | (bf16_bits(v[5]) << 16), bf16_bits(v[6]) | (bf16_bits(v[7]) << 16));
}

__global__ void __launch_bounds__(256) k_conv_tc(const ConvTc a) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ uint64_t mbar[2];
  __shared__ uint32_t tmem_sh;
  __shared__ int abort_sh;
  uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const long long n = (long long)a.N * a.N * a.N;
  const long long m0 = (long long)blockIdx.x * kCM;
  const uint32_t ncols = a.coutp <= 32 ? 32u : (a.coutp <= 64 ? 64u : 128u);

  if (warp == 0) tc::tmem_alloc(&tmem_sh, ncols);
  if (t == 0) {
    tc::mbar_init(&mbar[0], 1);
    tc::mbar_init(&mbar[1], 1);
    tc::fence_mbar_init();
    abort_sh = 0;
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = tmem_sh;
  const uint32_t idesc = tc::idesc_bf16(kCM, a.coutp);

  // this thread's four A chunks: rows r = (t + 256 i) / 8, 16-byte chunk kc = t % 8
  const int kc = t & 7;
  int px[4], py[4], pz[4];
  bool pin[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = (t >> 3) + 32 * i;
    const long long m = m0 + r;
    pin[i] = m < n;
    const long long mm = pin[i] ? m : 0;
    px[i] = (int)(mm % a.N);
    py[i] = (int)((mm / a.N) % a.N);
    pz[i] = (int)(mm / ((long long)a.N * a.N));
  }
  const int nslab = a.Kp / kCK;
  bool ok = true;
  for (int s = 0; s < nslab && ok; ++s) {
    const int b = s & 1;
    uint8_t *As = smem + b * kCStage, *Bs = As + kAPiece;
    if (s >= 2) {
      // the MMAs of slab s - 2 read this buffer
      if (t == 0 && !tc::mbar_wait(&mbar[b], (uint32_t)(((s - 2) >> 1) & 1))) abort_sh = 1;
      __syncthreads();
      if (abort_sh) {
        ok = false;
        break;
      }
    }
    const int k0 = s * kCK;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = (t >> 3) + 32 * i;
      const uint4 c = gather8(a, px[i], py[i], pz[i], pin[i], k0 + 8 * kc);
      *reinterpret_cast<uint4 *>(As + tc::sw128_offset(r, kc)) = c;
    }
    for (int c = t; c < a.coutp * 8; c += 256) {
      const int co = c >> 3, kk = c & 7;
      const uint4 w = __ldg(reinterpret_cast<const uint4 *>(a.Wt + (long long)co * a.Kp + k0 + 8 * kk));
      *reinterpret_cast<uint4 *>(Bs + tc::sw128_offset(co, kk)) = w;
    }
    tc::fence_async_smem();
    tc::tc_fence_before();
    __syncthreads();
    if (t == 0) {
      tc::tc_fence_after();
      const uint32_t ab = tc::smem_u32(As), bb = tc::smem_u32(Bs);
#pragma unroll
      for (int ks = 0; ks < kCK / 16; ++ks)
        tc::mma_bf16(tmem, tc::desc_sw128(ab + ks * 32), tc::desc_sw128(bb + ks * 32), idesc,
                     (s > 0 || ks > 0) ? 1u : 0u);
      tc::mma_commit(&mbar[b]);
    }
  }
  // the last slab's MMAs complete after all the others
  if (ok && nslab > 0) {
    const int s = nslab - 1;
    if (t == 0 && !tc::mbar_wait(&mbar[s & 1], (uint32_t)((s >> 1) & 1))) abort_sh = 1;
  }
  __syncthreads();
  if (ok && !abort_sh) {
    tc::tc_fence_after();
    // epilogue: warp w reads TMEM lanes 32 (w % 4) .. (rows), columns of its half
    const int q = warp & 3, h = warp >> 2, half = a.coutp / 2;
    const long long m = m0 + q * 32 + lane;
    for (int c0 = h * half; c0 < (h + 1) * half; c0 += 8) {
      float v[8];
      tmem_ld8(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)c0, v);
      if (m < n) {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int co = c0 + j;
          if (co >= a.cout) continue;
          const float z = v[j] + (a.bias ? a.bias[co] : 0.f);
          if (a.Z) a.Z[m * a.cout + co] = z;
          if (a.A) a.A[m * a.cout + co] = z / (1.0f + expf(-z));
        }
      }
    }
  } else if (t == 0) {
    atomicExch(a.err, 1);
  }
  tc::tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc::tc_fence_after();
    tc::tmem_dealloc(tmem, ncols);
  }
}

// ---- TMA-fed kernel -------------------------------------------------------------------
constexpr int kTmaThreads = 224;           // A copies, MMA, four epilogue warps, B copies
constexpr int kMaxStages = 8;
// Limit of the dynamic shared memory (a ring of (227 - 9) KB at most and 1 KB of alignment slack),
// the same at every call: it belongs to the kernel on the device, where another thread's call
// with a smaller ring could lower it between setting it and the launch.
constexpr int kTmaSmem = 219 * 1024;
constexpr uint64_t kWaitNs = 2000000000ull;

// BF16 weights as k_conv_wt, and the BF16 copy of X: rows of cin values, the grid points with
// one point of zeros around them (pad = 1, row ((z + 1) Np + y + 1) Np + x + 1, Np = N + 2) or
// as they are (pad = 0), with the xcin = cin channels of the point or (cin = 3 xcin) those of the
// point and its neighbours along x; or (gcin > 0) the gathered rows themselves, cin = K rounded up
// values of the taps of gcin channels.  One thread per 8 values.
__global__ void k_conv_prep(const float *__restrict__ W, int K, int cout, int Kp, int coutp,
                            uint16_t *__restrict__ Wt, const float *__restrict__ X, int N, int cin,
                            int xcin, int pad, int gcin, uint16_t *__restrict__ Xb) {
  const long long wtot = (long long)coutp * Kp, step = (long long)gridDim.x * blockDim.x;
  const long long e0 = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  for (long long e = e0; e < wtot; e += step) {
    const int co = (int)(e / Kp), k = (int)(e % Kp);
    Wt[e] = (uint16_t)bf16_bits((co < cout && k < K) ? W[(long long)k * cout + co] : 0.f);
  }
  const unsigned Np = (unsigned)(N + 2 * pad), nv = (unsigned)cin / 8;
  const long long total = (long long)Np * Np * Np * nv;
  for (long long e = e0; e < total; e += step) {
    const unsigned q = (unsigned)(e / nv), v = (unsigned)(e - (long long)q * nv);
    const unsigned r = q / Np;
    const int x = (int)(q - r * Np) - pad, y = (int)(r % Np) - pad, z = (int)(r / Np) - pad;
    uint4 o = make_uint4(0, 0, 0, 0);
    if (gcin > 0) {
      ConvTc a;
      a.X = X;
      a.N = N;
      a.taps = K == gcin ? 1 : 27;
      a.cin = gcin;
      a.K = K;
      o = gather8(a, x, y, z, true, 8 * (int)v);
    } else if (x >= 0 && x < N && y >= 0 && y < N && z >= 0 && z < N) {
      const int d = 8 * (int)v / xcin, xx = xcin < cin ? x + d - 1 : x;
      if (xx >= 0 && xx < N) {
        const float4 *src = reinterpret_cast<const float4 *>(
            X + (((long long)z * N + y) * N + xx) * xcin + (8 * (int)v - d * xcin));
        const float4 a = __ldg(src), b = __ldg(src + 1);
        o = make_uint4(bf16_bits(a.x) | (bf16_bits(a.y) << 16), bf16_bits(a.z) | (bf16_bits(a.w) << 16),
                       bf16_bits(b.x) | (bf16_bits(b.y) << 16), bf16_bits(b.z) | (bf16_bits(b.w) << 16));
      }
    }
    *reinterpret_cast<uint4 *>(Xb + e * 8) = o;
  }
}

// The K axis as pieces: `width` values (64, 32 or 16) of one tap from channel `off`, or (width 8)
// the last 8 channels of a tap and the first 8 of the next.  Consecutive pieces share a stage
// while they are at most 64 K values together.  The host lists them: a single thread walking the
// channels took longer per piece (some 500 clocks) than the copies.
struct __align__(16) KPiece {
  int row, row2;        // the tap's row shift; of the next tap (width 8)
  uint16_t off;
  uint8_t width, stage;  // stage: K values of the stage that starts here, 0: the same stage
};
constexpr int kMaxPieces = 320;  // (27 taps of at most 512 channels: at most 11 pieces a tap)
struct KPieces {
  int count;
  KPiece p[kMaxPieces];
};

struct ConvTma {
  const float *bias;
  float *Z, *A;
  int N, pad, cout, coutp, stages, tiles;
  int q0, q1;            // first output row and one past the last
  int *err;
};

// Shared-memory descriptors of K-major operands: rows of 64 or 32 bytes swizzled over 8 rows,
// and core matrices of 8 rows x 16 bytes without swizzle (the next 8 rows 128 bytes on, the
// next 8 K values 2048 bytes on).
__device__ __forceinline__ uint64_t desc_kmajor(uint32_t saddr, int lead, int stride, int layout) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(lead >> 4) << 16) |
         ((uint64_t)(stride >> 4) << 32) | ((uint64_t)1 << 46) | ((uint64_t)layout << 61);
}

__global__ void __launch_bounds__(kTmaThreads)
    k_conv_tma(const __grid_constant__ CUtensorMap a64, const __grid_constant__ CUtensorMap a32,
               const __grid_constant__ CUtensorMap a16, const __grid_constant__ CUtensorMap a8,
               const __grid_constant__ CUtensorMap b64, const __grid_constant__ KPieces pc,
               const ConvTma c) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ uint64_t full[kMaxStages], empty[kMaxStages], fin[2], freed[2];
  __shared__ uint32_t tmem_sh;
  __shared__ int abort_sh;
  __shared__ KPiece piece[kMaxPieces];
  for (int i = threadIdx.x; i < pc.count; i += kTmaThreads) piece[i] = pc.p[i];
  uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t ncols = c.coutp <= 32 ? 32u : (c.coutp <= 64 ? 64u : 128u);
  const int stage_bytes = kAPiece + c.coutp * 128;
  if (warp == 1) tc::tmem_alloc(&tmem_sh, 2 * ncols);
  if (threadIdx.x == 0) {
    for (int s = 0; s < c.stages; ++s) {
      tc::mbar_init(&full[s], 2);
      tc::mbar_init(&empty[s], 1);
    }
    for (int i = 0; i < 2; ++i) {
      tc::mbar_init(&fin[i], 1);
      tc::mbar_init(&freed[i], 4);
    }
    tc::fence_mbar_init();
    abort_sh = 0;
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = tmem_sh;
  volatile int *abort = &abort_sh;

  if (warp == 0) {
    if (lane == 0) {
      int it = 0, slot = 0, o = 0;
      uint32_t phase = 1;  // of the slot's last release (the first use of a slot passes)
      uint8_t *as = smem;
      bool ok = true;
      for (int tile = blockIdx.x; tile < c.tiles && ok; tile += gridDim.x) {
        const int q0 = c.q0 + tile * kCM;
        for (int i = 0; i < pc.count; ++i) {
          const KPiece s = piece[i];
          if (s.stage) {  // a new stage
            if (it > 0 && ++slot == c.stages) {
              slot = 0;
              phase ^= 1;
            }
            if (it >= c.stages && !tc::wait_or_abort(&empty[slot], phase, abort, kWaitNs)) {
              ok = false;
              break;
            }
            as = smem + slot * stage_bytes;
            o = 0;
            tma::bar_expect(&full[slot], (uint32_t)(s.stage * 2 * kCM));
            ++it;
          }
          uint64_t *bar = &full[slot];
          uint8_t *ap = as + o * 2 * kCM;
          const int r = q0 + s.row;
          if (s.width == 64) {
            tma::load_2d(ap, &a64, s.off, r, bar);
          } else if (s.width == 32) {
            tma::load_2d(ap, &a32, s.off, r, bar);
          } else if (s.width == 16) {
            tma::load_2d(ap, &a16, s.off, r, bar);
          } else {
            tma::load_2d(ap, &a8, s.off, r, bar);
            tma::load_2d(ap + 16 * kCM, &a8, 0, q0 + s.row2, bar);
          }
          o += s.width == 8 ? 16 : s.width;
        }
      }
      // the copies issued last land before the CTA may exit
      for (int u = it - 1; u >= 0 && u >= it - c.stages; --u)
        tma::bar_wait(&full[u % c.stages], (uint32_t)((u / c.stages) & 1), kWaitNs);
    }
  } else if (warp == kTmaThreads / 32 - 1) {
    if (lane == 0) {  // B: one box of 64 K values a stage, whatever pieces its A comes in
      int it = 0, slot = 0;
      uint32_t phase = 1;
      bool ok = true;
      for (int tile = blockIdx.x; tile < c.tiles && ok; tile += gridDim.x) {
        int k = 0;
        for (int i = 0; i < pc.count; ++i) {
          const int len = piece[i].stage;
          if (!len) continue;
          if (it > 0 && ++slot == c.stages) {
            slot = 0;
            phase ^= 1;
          }
          if (it >= c.stages && !tc::wait_or_abort(&empty[slot], phase, abort, kWaitNs)) {
            ok = false;
            break;
          }
          tma::bar_expect(&full[slot], (uint32_t)(kCK * 2 * c.coutp));
          tma::load_2d(smem + slot * stage_bytes + kAPiece, &b64, k, 0, &full[slot]);
          k += len;
          ++it;
        }
      }
      for (int u = it - 1; u >= 0 && u >= it - c.stages; --u)
        tma::bar_wait(&full[u % c.stages], (uint32_t)((u / c.stages) & 1), kWaitNs);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t idesc = tc::idesc_bf16(kCM, c.coutp);
      int slot = 0, o = 0, j = 0;  // j: tiles begun
      uint32_t phase = 0, as = 0;
      uint64_t bs = 0;
      bool ok = true, open = false;  // open: a stage whose MMAs are not committed yet
      for (int tile = blockIdx.x; tile < c.tiles && ok; tile += gridDim.x, ++j) {
        // two accumulators in turn: the read-out of a tile runs beside the next one
        if (j >= 2 && !tc::wait_or_abort(&freed[j & 1], (uint32_t)((j >> 1) - 1) & 1, abort, kWaitNs))
          break;
        const uint32_t d = tmem + (uint32_t)(j & 1) * ncols;
        uint32_t acc = 0;
        for (int i = 0; i < pc.count; ++i) {
          const KPiece s = piece[i];
          if (s.stage) {
            if (open) {
              tc::mma_commit(&empty[slot]);
              if (++slot == c.stages) {
                slot = 0;
                phase ^= 1;
              }
            }
            if (!tc::wait_or_abort(&full[slot], phase, abort, kWaitNs)) {
              ok = false;
              break;
            }
            tc::tc_fence_after();
            as = tc::smem_u32(smem + slot * stage_bytes);
            bs = desc_kmajor(as + kAPiece, 16, 1024, 2);
            o = 0;
            open = true;
          }
          const uint32_t ap = as + o * 2 * kCM;
          const uint64_t bd = bs + (uint64_t)(o / 8);  // o K values along the 128-byte rows
          if (s.width == 64) {
            const uint64_t ad = desc_kmajor(ap, 16, 1024, 2);
#pragma unroll
            for (int ks = 0; ks < 4; ++ks, acc = 1)
              tc::mma_bf16(d, ad + 2 * ks, bd + 2 * ks, idesc, acc);
            o += 64;
          } else if (s.width == 32) {
            const uint64_t ad = desc_kmajor(ap, 16, 512, 4);
#pragma unroll
            for (int ks = 0; ks < 2; ++ks, acc = 1)
              tc::mma_bf16(d, ad + 2 * ks, bd + 2 * ks, idesc, acc);
            o += 32;
          } else {
            const uint64_t ad =
                s.width == 16 ? desc_kmajor(ap, 16, 256, 6) : desc_kmajor(ap, 16 * kCM, 128, 0);
            tc::mma_bf16(d, ad, bd, idesc, acc);
            acc = 1;
            o += 16;
          }
        }
        tc::mma_commit(&fin[j & 1]);  // (also after a failed wait: the MMAs end before the CTA does)
      }
      if (j > 0) tma::bar_wait(&fin[(j - 1) & 1], (uint32_t)((j - 1) >> 1) & 1, kWaitNs);
    }
  } else {
    int j = 0;
    for (int tile = blockIdx.x; tile < c.tiles; tile += gridDim.x, ++j) {
      int ok = 0;
      if (lane == 0)
        ok = tc::wait_or_abort(&fin[j & 1], (uint32_t)(j >> 1) & 1, abort, kWaitNs) && !*abort;
      if (!__shfl_sync(0xffffffffu, ok, 0)) break;
      tc::tc_fence_after();
      const int quarter = warp & 3, q = c.q0 + tile * kCM + quarter * 32 + lane;
      long long m = q;
      bool in = q < c.q1;
      if (c.pad) {
        const unsigned Np = (unsigned)c.N + 2, r = (unsigned)q / Np;
        const int x = (int)((unsigned)q - r * Np) - 1, y = (int)(r % Np) - 1, z = (int)(r / Np) - 1;
        in = in && x >= 0 && x < c.N && y >= 0 && y < c.N && z >= 0 && z < c.N;
        m = ((long long)z * c.N + y) * c.N + x;
      }
      const uint32_t tb = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(j & 1) * ncols;
      for (int c0 = 0; c0 < c.coutp; c0 += 8) {
        float v[8];
        tmem_ld8(tb + (uint32_t)c0, v);
        if (!in) continue;
        if (c.cout % 4 == 0) {
#pragma unroll
          for (int h = 0; h < 8; h += 4) {
            if (c0 + h >= c.cout) continue;
            float4 z, y;
            const float *bi = c.bias ? c.bias + c0 + h : nullptr;
            z.x = v[h] + (bi ? __ldg(bi) : 0.f);
            z.y = v[h + 1] + (bi ? __ldg(bi + 1) : 0.f);
            z.z = v[h + 2] + (bi ? __ldg(bi + 2) : 0.f);
            z.w = v[h + 3] + (bi ? __ldg(bi + 3) : 0.f);
            if (c.Z) *reinterpret_cast<float4 *>(c.Z + m * c.cout + c0 + h) = z;
            if (c.A) {
              y.x = z.x / (1.0f + expf(-z.x));
              y.y = z.y / (1.0f + expf(-z.y));
              y.z = z.z / (1.0f + expf(-z.z));
              y.w = z.w / (1.0f + expf(-z.w));
              *reinterpret_cast<float4 *>(c.A + m * c.cout + c0 + h) = y;
            }
          }
        } else {
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const int co = c0 + j;
            if (co >= c.cout) continue;
            const float z = v[j] + (c.bias ? __ldg(c.bias + co) : 0.f);
            if (c.Z) c.Z[m * c.cout + co] = z;
            if (c.A) c.A[m * c.cout + co] = z / (1.0f + expf(-z));
          }
        }
      }
      tc::tc_fence_before();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&freed[j & 1]);
    }
  }
  tc::tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc::tc_fence_after();
    tc::tmem_dealloc(tmem, 2 * ncols);
  }
  if (threadIdx.x == 0 && abort_sh) atomicExch(c.err, 1);
}

// Copies of 128 rows that a group of `cin` K values takes.
int boxes(int cin) { return cin / 64 + ((cin & 32) != 0) + ((cin & 16) != 0) + ((cin & 8) != 0); }
// Whether the copy holds the three taps along x side by side (rows of 3 cin values, 9 groups of
// taps): where that takes at most two thirds of the boxes and the copy stays within 8 GiB.  The K
// order, and so every sum, is the same.  48^3, one CTA a tile: 24 -> 24 channels 70 -> 51 us,
// 48 -> 48 97 -> 83; for 72 channels (5 boxes instead of 6) the three times larger copy would
// cost what it saves.
bool merge_x(int N, int taps, int cin) {
  const long long m = N + 2;
  return taps == 27 && cin % 8 == 0 && boxes(3 * cin) <= 2 * boxes(cin) &&
         m * m * m * 3 * cin * 2 <= (8ll << 30);
}

// Rows and row length of the BF16 copy (0: the layer is left to k_conv_tc).  Channels in 16-byte
// groups: the padded points.  Other layers with few K values (the 4-channel first one): the
// gathered rows, written once (at 48^3, 4 -> 24: 64 us in all, by k_conv_tc 73).  At most 8 GiB
// beside the FP32 activations.
long long copy_rows(int N, int taps, int cin) {
  const long long m = taps == 27 && cin % 8 == 0 ? N + 2 : N;
  return m * m * m;
}
int copy_len(int N, int taps, int cin) {
  if (merge_x(N, taps, cin)) return 3 * cin;
  const int len = cin % 8 == 0 ? cin : (taps * cin <= 256 ? (taps * cin + 15) / 16 * 16 : 0);
  return copy_rows(N, taps, cin) * len * 2 <= (8ll << 30) ? len : 0;
}
// Pieces of taps x cin K values over a copy of `rows` rows (Np points an axis with the padding).
void list_pieces(int taps, int cin, int Np, long long rows, KPieces *out) {
  auto shift = [&](int t) -> int {
    if (t >= taps) return (int)rows;  // past the last row: zeros
    if (taps == 9) return ((t / 3 - 1) * Np + t % 3 - 1) * Np;
    return taps == 1 ? 0 : ((t / 9 - 1) * Np + (t / 3) % 3 - 1) * Np + t % 3 - 1;
  };
  int n = 0, used = kCK, first = 0, off = 0;
  for (int t = 0; t < taps;) {
    KPiece &p = out->p[n];
    const int rem = cin - off;
    p.width = (uint8_t)(rem >= 64 ? 64 : (rem >= 32 ? 32 : (rem >= 16 ? 16 : 8)));
    p.off = (uint16_t)off;
    p.row = shift(t);
    p.row2 = shift(t + 1);
    p.stage = 0;
    const int len = p.width == 8 ? 16 : p.width;
    if (used + len > kCK) {
      first = n;
      used = 0;
    }
    used += len;
    out->p[first].stage = (uint8_t)used;
    ++n;
    off += p.width;
    if (p.width == 8) {  // the first 8 channels of the next tap came along
      ++t;
      off = 8;
    }
    if (off >= cin) {
      off = 0;
      ++t;
    }
  }
  out->count = n;
}
size_t weight_bytes(int taps, int cin, int cout) {
  const long long Kp = ((long long)taps * cin + kCK - 1) / kCK * kCK;
  return (size_t)(Kp * ((cout + 15) / 16 * 16) * 2 + 255) / 256 * 256;
}

}  // namespace

size_t conv_tc_scratch_min(int taps, int cin, int cout) { return weight_bytes(taps, cin, cout); }
size_t conv_tc_scratch_bytes(int N, int taps, int cin, int cout) {
  return weight_bytes(taps, cin, cout) +
         (size_t)copy_rows(N, taps, cin) * copy_len(N, taps, cin) * 2;
}

op_status conv_bf16_tc(const float *X, int N, int taps, int cin, int cout, const float *W,
                       const float *bias, float *Z, float *A, void *scratch, size_t scratch_bytes,
                       int *err, cudaStream_t st) {
  if (!X || !W || !scratch || !err || N < 1 || (taps != 1 && taps != 27) || cin < 1 ||
      cout < 1 || cout > 128 || scratch_bytes < conv_tc_scratch_min(taps, cin, cout) ||
      ((uintptr_t)scratch & 15) != 0) {
    set_error("conv_bf16_tc: bad arguments (N=%d taps=%d cin=%d cout=%d)", N, taps, cin, cout);
    return OP_ERR_ARG;
  }
  if (cin % 8 == 0 && ((uintptr_t)X & 15) != 0) {
    set_error("conv_bf16_tc: X must be 16-byte aligned");
    return OP_ERR_ARG;
  }
  const int K = taps * cin, coutp = (cout + 15) / 16 * 16, Kp = (K + kCK - 1) / kCK * kCK;
  const int clen = copy_len(N, taps, cin);
  if (clen > 0 && scratch_bytes >= conv_tc_scratch_bytes(N, taps, cin, cout) &&
      (!Z || ((uintptr_t)Z & 15) == 0) && (!A || ((uintptr_t)A & 15) == 0)) {
    uint16_t *Wt = (uint16_t *)scratch;
    uint16_t *Xb = (uint16_t *)((char *)scratch + weight_bytes(taps, cin, cout));
    const int gcin = cin % 8 == 0 ? 0 : cin, pad = taps == 27 && !gcin ? 1 : 0;
    const long long rows = copy_rows(N, taps, cin);
    const long long work = std::max(rows * (clen / 8), (long long)coutp * Kp);
    k_conv_prep<<<(unsigned)std::min<long long>((work + 255) / 256, 16LL * num_sms()), 256, 0, st>>>(
        W, K, cout, Kp, coutp, Wt, X, N, clen, gcin ? clen : cin, pad, gcin, Xb);
    count_launch();
    OP_LAUNCH("k_conv_prep");
    ConvTma c;
    c.bias = bias;
    c.Z = Z;
    c.A = A;
    c.N = N;
    c.pad = pad;
    c.cout = cout;
    c.coutp = coutp;
    c.err = err;
    const int Np = N + 2;
    c.q0 = pad ? Np * Np + Np + 1 : 0;
    c.q1 = (int)rows - c.q0;
    const int tiles = (c.q1 - c.q0 + kCM - 1) / kCM, stage = kAPiece + coutp * 128;
    KPieces pc;
    list_pieces(gcin ? 1 : (clen > cin ? 9 : taps), clen, Np, rows, &pc);
    const int ncols = coutp <= 32 ? 32 : (coutp <= 64 ? 64 : 128);
    // with no more tiles than SMs a CTA has the SM to itself and is bound by the latency of its
    // loads: as many stages as fit; else CTAs that cover each other's first loads and waits (the
    // 11 layers by one CTA an SM 0.698 ms, two 0.619, three 0.615, four 0.617)
    int per_sm = tiles <= num_sms() ? 1 : std::min(3, 256 / ncols);
    auto ring = [&](int ctas) { return std::min(kMaxStages, (227 / ctas - 9) * 1024 / stage); };
    while (per_sm > 1 && ring(per_sm) < 2) --per_sm;
    c.stages = ring(per_sm);
    c.tiles = tiles;
    CUtensorMap ma[4], mb;
    const int wid[4] = {64, 32, 16, 8};
    for (int i = 0; i < 4; ++i)
      OP_TRY(tma_map_2d_bf16(&ma[i], Xb, (uint64_t)clen, (uint64_t)rows, wid[i], kCM));
    OP_TRY(tma_map_2d_bf16(&mb, Wt, (uint64_t)Kp, (uint64_t)coutp, kCK, coutp));
    // (room for no more CTAs than their TMEM allows)
    const int smem = std::max(c.stages * stage, 228 * 1024 / (256 / ncols + 1)) + 1024;
    OP_CUDA(cudaFuncSetAttribute(k_conv_tma, cudaFuncAttributeMaxDynamicSharedMemorySize, kTmaSmem));
    k_conv_tma<<<(unsigned)std::min(tiles, per_sm * num_sms()), kTmaThreads, smem, st>>>(
        ma[0], ma[1], ma[2], ma[3], mb, pc, c);
    count_launch();
    OP_LAUNCH("k_conv_tma");
    return OP_OK;
  }
  ConvTc a;
  a.X = X;
  a.Wt = (const uint16_t *)scratch;
  a.bias = bias;
  a.Z = Z;
  a.A = A;
  a.N = N;
  a.taps = taps;
  a.cin = cin;
  a.cout = cout;
  a.coutp = coutp;
  a.K = K;
  a.Kp = Kp;
  a.err = err;
  const long long wt = (long long)a.coutp * a.Kp;
  k_conv_wt<<<(unsigned)std::min<long long>((wt + 255) / 256, 4LL * num_sms()), 256, 0, st>>>(
      W, a.K, cout, a.Kp, a.coutp, (uint16_t *)scratch);
  count_launch();
  OP_LAUNCH("k_conv_wt");
  // per device, so set on every call (cheap)
  OP_CUDA(cudaFuncSetAttribute(k_conv_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, kCSmem));
  const long long n = (long long)N * N * N;
  k_conv_tc<<<(unsigned)((n + kCM - 1) / kCM), 256, kCSmem, st>>>(a);
  count_launch();
  OP_LAUNCH("k_conv_tc");
  return OP_OK;
}

}  // namespace opevo
