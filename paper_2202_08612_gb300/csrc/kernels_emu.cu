// FP64-accurate contractions on the BF16 tensor cores (sm_103a), after the
// error-free splitting of Ozaki, Ogita, Oishi and Rump: an operand is an
// integer of up to 63 bits per element (its value over a power of two that its
// row or the whole operand shares), held as S balanced base-256 digits, each
// exact in bfloat16.  Products of digits are integers of at most 2^14, which
// FP32 sums exactly over 256 of them for the digit degrees t + u <= 3.  Kept are
// the degrees up to S - 1, and with S = 8 (the FP64 mode) up to 8, which leaves
// out terms below 2^-69 of full scale per product.
//
// GB300 retires about two FP64 operations per clock and SM (1.1 TFLOP/s in
// all), and BF16 on the tensor cores about 1.7 PFLOP/s, so even the 43 digit
// products of S = 8 leave room for a factor of some twenty over the FP64 pipe.
#include <cudaTypedefs.h>

#include <algorithm>
#include <cstdint>

#include "kernels_emu.cuh"
#include "tc_ptx.cuh"

namespace mlcc3 {

namespace {

// chunks per TMEM accumulation chain
template <int S> constexpr int kChainOf = S == kEmuSlices ? kEmuChain : 256 / kEmuKB;
constexpr int kRowB = 2 * kEmuKB;     // bytes of a shared-memory operand row

__device__ __forceinline__ void tma_load_5d(uint32_t dst, const CUtensorMap *map, int c0, int c1,
                                            int c2, int c3, int c4, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4, %5, %6}], [%7];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "r"(bar)
      : "memory");
}

// K-major operand, 64-byte rows with the 64-byte swizzle, 8-row groups 512 bytes apart.
__device__ __forceinline__ uint64_t smem_desc64(uint32_t addr) {
  uint64_t d = 0;
  d |= (uint64_t)((addr >> 4) & 0x3FFF);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)((8 * kRowB) >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)4 << 61;  // SWIZZLE_64B
  return d;
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t *r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                 "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}

// T 2^e (+-), rounded to binary64 on the integer pipe (an FP64 conversion costs
// one of the two FP64 operations an SM retires per clock).
__device__ __forceinline__ double int_to_double(long long T, int e) {
  if (T == 0) return 0.0;
  const unsigned long long sgn = (unsigned long long)T & (1ULL << 63);
  unsigned long long u = T < 0 ? 0ULL - (unsigned long long)T : (unsigned long long)T;
  const int lz = __clzll(u);
  u <<= lz;
  const int ex = e - lz + 63 + 1023;  // biased exponent of the leading bit
  if (ex < 1 || ex > 2045) return ldexp((double)T, e);
  const unsigned long long m = (u >> 11) + ((u >> 10) & 1);
  return __longlong_as_double((long long)((((unsigned long long)(ex - 1) << 52) + m) | sgn));
}

// (T + M 2^-32) 2^e, rounded to binary64 once (to nearest, ties to even).
__device__ __forceinline__ double sum_to_double(long long T, long long M, int e) {
  unsigned long long h = (unsigned long long)(T + (M >> 32)), l = (unsigned long long)M << 32;
  const unsigned long long sgn = h & (1ULL << 63);
  if (sgn) {
    h = ~h + (l == 0 ? 1 : 0);
    l = 0ULL - l;
  }
  if (h == 0) {
    if (l == 0) return 0.0;
    h = l;
    l = 0;
    e -= 64;
  }
  const int lz = __clzll((long long)h);
  if (lz) {
    h = (h << lz) | (l >> (64 - lz));
    l <<= lz;
  }
  const int ex = e - lz + 63 + 1023;
  if (ex < 1 || ex > 2045) {
    const double v = ldexp((double)h, e - lz);
    return sgn ? -v : v;
  }
  unsigned long long m = h >> 11;
  const unsigned rest = (unsigned)h & 2047u;
  if (rest > 1024u || (rest == 1024u && (l != 0 || (m & 1)))) ++m;
  return __longlong_as_double((long long)((((unsigned long long)(ex - 1) << 52) + m) | sgn));
}

__device__ __forceinline__ int scale_exp(EmuScale s) {
  return (int)(((s + (1ULL << 46)) >> 52) & 0x7ff) - 1022;
}

}  // namespace

// One 128 x n tile of C = sum_segments A_seg B_seg^T per item, persistent (one
// CTA per SM, item i to CTA i mod gridDim.x).
//
// A stage holds 32 K elements of all S slices of both operands.  The slices of
// B lie one below the other in shared memory, so the MMA of A's slice t with
// the stacked slices of B (N = their number times n, in pieces of at most 256)
// puts digit pair (t, u) into TMEM columns (t + u) n: one accumulator per digit
// degree and wide MMAs instead of narrow ones per pair.
//
// S = 8, the FP64 mode: degrees 0..8 and, in a tenth group of columns, the product of the
// operands' magnitudes (a ninth slice), which an item accumulates from its first chunk to
// its last and which says whether the digits hold its outputs to FP64 accuracy
// (kStatusSpread).  If they do not, the caller runs the call on the FP64 pipe.  With n = 48, 480 of TMEM's 512
// columns; a stage is 101 KB, two are in flight.
//
// After each chain of K elements eight epilogue warps add the degrees, weighted by 2^-8d,
// into 64-bit integers in registers (degrees 0..4 in units of 2^-32, below 2^60 for
// kEmuMaxK products; degrees 5..8 in units of 2^-64, below 2^54; S = 6: degree 5 in FP32)
// and hand TMEM back, so the next chain's MMAs wait only for the reads.  An
// item's sums are rounded to binary64 once, at its end, on the integer pipe.
//   warp 0 lane 0: TMA producer; warp 1: TMEM, lane 0 issues; warps 2..9: epilogue
// C = A B^T with M = N = K = 4096 and S = 5, slicing included: 1.77 ms, against
// 8.26 ms with one launch of the split mode's kernel per digit degree (two of its
// three products on zeros, and an FP64 reduction per output, pair and 1024 products).
// AMN: A's rows are the contiguous index of its map (boxes of 64 rows x 32 K of
// every slice, two per stage).
template <int S, int N, bool AMN>
__global__ void __launch_bounds__(320, 1)
    emu_gemm_kernel(const __grid_constant__ TcMaps maps, const TcItem *__restrict__ items,
                    const TcSeg *__restrict__ segs, int nitems, int stages, const EmuEpi epi,
                    int *__restrict__ status) {
  constexpr bool FULL = S == kEmuSlices;       // the FP64 mode
  constexpr int SL = FULL ? kEmuStored : S;    // slices of a stage
  constexpr int DG = FULL ? S + 1 : S;         // digit degrees
  constexpr int GR = FULL ? DG + 1 : S;        // groups of n columns in TMEM
  constexpr int kChain = kChainOf<S>;
  constexpr int NG = N / 16;  // 8-column groups per epilogue thread
  constexpr int A_SL = 128 * kRowB;         // bytes of one slice of A
  constexpr uint32_t IDESC =
      (1u << 4) | (1u << 7) | (1u << 10) | (AMN ? 1u << 15 : 0u) | ((uint32_t)(128 >> 4) << 24);
  extern __shared__ unsigned char smem_raw[];
  unsigned char *smem = reinterpret_cast<unsigned char *>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  constexpr int n = N;
  constexpr int stage_bytes = SL * (A_SL + n * kRowB);
  uint64_t *bars = reinterpret_cast<uint64_t *>(smem + stages * stage_bytes);
  const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + 8);
  const uint32_t tfull = smem_u32(bars + 16), tempty = smem_u32(bars + 17);
  const uint32_t done = smem_u32(bars + 18);
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 19);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  constexpr uint32_t ncols = GR * n <= 128 ? 128u : GR * n <= 256 ? 256u : 512u;
  static_assert(GR * n <= 512, "TMEM columns");

  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    mbar_init(tfull, 1);
    mbar_init(tempty, 8);
    mbar_init(done, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 0 && lane == 0) {
    // ---- TMA producer ----
    int stage = 0;
    uint32_t phase = 0, last = 0, pending = 0;
    for (int i = blockIdx.x; i < nitems && !*abort_flag; i += gridDim.x) {
      const int s0 = items[i].seg_begin, s1 = s0 + items[i].seg_count;
      TcSeg next = segs[s0];  // read one segment ahead of its loads
      for (int q = s0; q < s1 && !*abort_flag; ++q) {
        const TcSeg sg = next;
        if (q + 1 < s1) next = segs[q + 1];
        for (int kc = 0; kc < sg.nk; ++kc) {
          if (!mbar_wait(empty0 + 8 * stage, phase ^ 1u, status, epi.wait)) {
            *abort_flag = 1;
            break;
          }
          const uint32_t st = smem_u32(smem + stage * stage_bytes), fb = full0 + 8 * stage;
          mbar_expect_tx(fb, (uint32_t)stage_bytes);
          if constexpr (AMN) {
            for (int h = 0; h < 2; ++h)
              tma_load_5d(st + h * (SL * A_SL / 2), &maps.m[sg.amap], sg.ac[1] + 64 * h,
                          sg.ac[0] + kEmuKB * kc, sg.ac[2], sg.ac[3], 0, fb);
          } else {
            tma_load_5d(st, &maps.m[sg.amap], sg.ac[0] + kEmuKB * kc, sg.ac[1], sg.ac[2], sg.ac[3], 0, fb);
          }
          tma_load_5d(st + SL * A_SL, &maps.m[sg.bmap], sg.bc[0] + kEmuKB * kc, sg.bc[1], sg.bc[2],
                      sg.bc[3], 0, fb);
          last = (last & ~(1u << stage)) | (phase << stage);
          pending |= 1u << stage;
          if (++stage == stages) {
            stage = 0;
            phase ^= 1u;
          }
        }
      }
    }
    // the shared memory must outlive every copy issued into it
    for (int s = 0; s < stages; ++s)
      if ((pending >> s) & 1u) mbar_wait(full0 + 8 * s, (last >> s) & 1u, status, kTcWaitDefault);
  } else if (warp == 1) {
    // ---- MMA issuer: the warp goes through the loops together, one lane issues.  An
    // MMA of N = 64 takes 32 clocks, so the loop around it has to be short: with the
    // tile width a constant its descriptors are a stage's plus constants (with a
    // runtime width the issue took about 100 clocks per MMA, and the tensor pipe ran 59%
    // of the time) ----
    const bool leader = elect_one();
    int stage = 0;
    uint32_t phase = 0;
    int t = 0;  // accumulation chains so far
    bool ok = true;
    for (int i = blockIdx.x; i < nitems && ok; i += gridDim.x) {
      if (__shfl_sync(0xffffffffu, *abort_flag, 0)) break;
      const int s0 = items[i].seg_begin, s1 = s0 + items[i].seg_count;
      int cc = 0;  // chunk of the accumulation chain
      int nk1 = segs[s0].nk, tail1 = segs[s0].tail;
      for (int q = s0; q < s1 && ok; ++q) {
        const int nk = nk1, tail = tail1;
        if (q + 1 < s1) {
          nk1 = segs[q + 1].nk;
          tail1 = segs[q + 1].tail;
        }
        for (int kc = 0; kc < nk; ++kc) {
          if (cc == 0) ok = mbar_wait(tempty, ((uint32_t)t & 1u) ^ 1u, status, epi.wait);
          ok = __all_sync(0xffffffffu, ok && mbar_wait(full0 + 8 * stage, phase, status, epi.wait));
          if (!ok) {
            *abort_flag = 1;
            break;
          }
          tc_fence_after();
          const bool last = q == s1 - 1 && kc == nk - 1;
          if (leader) {
            const uint32_t a0 = smem_u32(smem) + stage * stage_bytes;
            const uint64_t ad = AMN ? smem_desc_mn(a0, SL * A_SL / 2) : smem_desc64(a0);
            const uint64_t bd = smem_desc64(a0 + SL * A_SL);
            const int steps = kc == nk - 1 && tail > 0 ? tail : kEmuKB / 16;
#pragma unroll
            for (int kk = 0; kk < kEmuKB / 16; ++kk) {
              if (kk < steps) {  // zeros to the end of the reduction
                const uint32_t add = kk > 0 || cc > 0 ? 1u : 0u;  // 0: first of the chain
                // A's slice t with B's slices [u0, u1) into the degrees t + u0 .. t + u1 - 1
                auto mmas = [&](int t, int u0, int u1, int group, uint32_t acc) {
                  constexpr int W = 256 / n * n, a_slice = AMN ? A_SL / 2 : A_SL, a_step = AMN ? 2048 : 32;
#pragma unroll
                  for (int c0 = u0 * n; c0 < u1 * n; c0 += W) {
                    const int nn = u1 * n - c0 < W ? u1 * n - c0 : W;
                    mma_bf16(tmem + (uint32_t)((group - u0) * n + c0),
                             ad + (uint64_t)((t * a_slice + kk * a_step) >> 4),
                             bd + (uint64_t)((c0 * kRowB + kk * 32) >> 4), IDESC | ((uint32_t)(nn >> 3) << 17), acc);
                  }
                };
#pragma unroll
                for (int d = 0; d < S; ++d) {
                  // the first MMA of a chain (d = 0) covers every degree up to S - 1 and
                  // clears them; degree S (FULL) first comes up in the last slice of d = 1
                  const int u1 = DG - d < S ? DG - d : S;
                  if (FULL && d == 1 && add == 0) {
                    mmas(1, 0, S - 1, 1, 1u);
                    mmas(1, S - 1, S, S, 0u);
                  } else {
                    mmas(d, 0, u1, d, d > 0 ? 1u : add);
                  }
                }
                if constexpr (FULL)  // magnitudes, over the whole item
                  mmas(S, S, S + 1, DG, q > s0 || kc > 0 || kk > 0 ? 1u : 0u);
              }
            }
            mma_commit(empty0 + 8 * stage);
            if (cc == kChain - 1 || last) mma_commit(tfull);
          }
          __syncwarp();
          if (++stage == stages) {
            stage = 0;
            phase ^= 1u;
          }
          if (++cc == kChain || last) {
            ++t;
            cc = 0;
          }
        }
      }
    }
    if (leader) mma_commit(done);
  } else if (warp >= 2) {
    // ---- epilogue ----
    const int lg = warp & 3, half = (warp - 2) >> 2;
    const int row = lg * 32 + lane, hn = n / 2;
    const uint32_t tm = tmem + ((uint32_t)(lg * 32) << 16) + (uint32_t)(half * hn);
    int e0 = epi.ebias - 32;
    if (epi.sa && !epi.ra) e0 += scale_exp(*epi.sa);
    if (epi.sb && !epi.rb) e0 += scale_exp(*epi.sb);
    int t = 0;
    bool ok = true;
    for (int i = blockIdx.x; i < nitems && ok; i += gridDim.x) {
      if (__shfl_sync(0xffffffffu, *abort_flag, 0)) break;
      const TcItem it = items[i];
      const int chains = (it.chunks + kChain - 1) / kChain;
      const int c0 = it.c0 + half * hn;
      int r1 = 0, r2 = 0, cmax = 0;
      auto place = [&] {
        if (epi.linear) {
          const int m = it.r2_0 + row;
          r1 = m / epi.R2;
          r2 = m % epi.R2;
        } else {
          r1 = it.r1_0 + row / epi.R2;
          r2 = it.r2_0 + row % epi.R2;
        }
        cmax = r1 < epi.lim1 && r2 < epi.lim2 ? epi.nlim : 0;
      };
      if (FULL) place();
      long long T[NG * 8];
      long long U[FULL ? NG * 8 : 1];  // degrees 5..8
      float L[S == 6 ? NG * 8 : 1];    // degree 5
      unsigned nan[NG];
      bool weak = false;
#pragma unroll
      for (int g = 0; g < NG; ++g) {
        nan[g] = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          T[g * 8 + j] = 0;
          if constexpr (FULL) U[g * 8 + j] = 0;
          if constexpr (S == 6) L[g * 8 + j] = 0.f;
        }
      }
      for (int ch = 0; ch < chains; ++ch, ++t) {
        // the whole warp goes on or leaves: the TMEM reads are warp collectives
        if (!__all_sync(0xffffffffu, mbar_wait(tfull, (uint32_t)t & 1u, status, epi.wait))) {
          *abort_flag = 1;
          ok = false;
          break;
        }
        tc_fence_after();
#pragma unroll
        for (int g = 0; g < NG; ++g) {
          if (g * 8 < hn) {
            constexpr int D1 = FULL ? 5 : S;  // degrees read at a time (registers)
            uint32_t r[D1][8];
#pragma unroll
            for (int d = 0; d < D1; ++d) tmem_ld8(tm + (uint32_t)(d * n + g * 8), r[d]);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const float f0 = __uint_as_float(r[0][j]);
              if (!FULL && !(f0 == f0)) nan[g] |= 1u << j;
              long long x = T[g * 8 + j];
              x += (long long)((unsigned long long)(uint32_t)__float2int_rn(f0) << 32);
#pragma unroll
              for (int d = 1; d < (S < 5 ? S : 5); ++d)
                x += (long long)__float2int_rn(__uint_as_float(r[d][j])) * (1LL << (32 - 8 * d));
              T[g * 8 + j] = x;
              if constexpr (S == 6) L[g * 8 + j] += __uint_as_float(r[5][j]);
            }
            if constexpr (FULL) {
#pragma unroll
              for (int d = 0; d < 4; ++d) tmem_ld8(tm + (uint32_t)((5 + d) * n + g * 8), r[d]);
              asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                long long x = U[g * 8 + j];
#pragma unroll
                for (int d = 0; d < 4; ++d)
                  x += (long long)__float2int_rn(__uint_as_float(r[d][j])) * (1LL << (24 - 8 * d));
                U[g * 8 + j] = x;
              }
              if (ch == chains - 1) {
                const float least = (float)it.chunks * (kEmuKB * kEmuLeast);
                tmem_ld8(tm + (uint32_t)(DG * n + g * 8), r[4]);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                  const float m = __uint_as_float(r[4][j]);
                  weak = weak || (c0 + g * 8 + j < cmax && !(m >= least) && m != 0.f);
                }
              }
            }
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(tempty);
      }
      if (!ok) break;
      if (!FULL) place();  // (registers)
      if (FULL && __any_sync(0xffffffffu, weak) && lane == 0) atomicOr(status, kStatusSpread);
      int er = e0;
      if (FULL && epi.ra && cmax) er += scale_exp(epi.sa[it.ea + it.r2_0 + row]);
      if (!FULL && epi.ea && cmax) er += epi.ea[it.r2_0 + row];
      double *o = epi.out + it.out_off + (long long)r1 * epi.s1 + (long long)r2 * epi.s2 + (long long)c0 * epi.sn;
#pragma unroll
      for (int g = 0; g < NG; ++g) {
        if (g * 8 >= hn) continue;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int c = g * 8 + j;
          if (c0 + c >= cmax) break;
          long long x = T[c];
          int ex = er;
          if (FULL && epi.rb) ex += scale_exp(epi.sb[it.eb + c0 + c]);
          if (!FULL && epi.eb) ex += epi.eb[c0 + c];
          double v;
          if constexpr (FULL) {
            v = sum_to_double(x, U[c], ex);
          } else {
            if constexpr (S == 6) {
              // T moved up as far as it goes, so that the degree above (|L| < 2^30,
              // in 2^-8 of T's unit) joins it below its own 53 leading bits
              const int sh = min(24, __clzll(x < 0 ? -x : x) - 2);
              x = (x << sh) + __float2ll_rn(L[c] * __int_as_float((127 + sh - 8) << 23));
              ex -= sh;
            }
            v = int_to_double(x, ex);
            if ((nan[g] >> j) & 1u) v = __longlong_as_double(0x7ff8000000000000LL);
          }
          if (epi.alpha != 1.0) v = epi.alpha == -1.0 ? -v : epi.alpha * v;
          double *p = o + (long long)c * epi.sn;
          if (epi.mode == 0) *p = v;
          else atomicAdd(p, v);
        }
      }
      __syncwarp();
    }
  }
  if (warp == 1 && lane == 0) mbar_wait(done, 0, status, kTcWaitDefault);
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols)
                 : "memory");
  }
}

// The width that wastes least: columns of all tiles, and as much as eight columns
// per tile for reading A again.
int emu_tile_width(long long n, int S) {
  const int w8[] = {16, 32, 48}, ws[] = {32, 80};
  int best = 0;
  long long cost = 0;
  for (int i = 0; i < (S == 8 ? 3 : 2); ++i) {
    const int w = S == 8 ? w8[i] : ws[i];
    const long long c = (n + w - 1) / w * (w + 8);
    if (!best || c <= cost) {
      cost = c;
      best = w;
    }
  }
  return best;
}

bool emu_encode_map(CUtensorMap *m, const void *base, const unsigned long long dims[4],
                    const unsigned long long strides[3], unsigned long long slice_bytes,
                    const unsigned box[3], int S, std::string *err, bool mn) {
  static const PFN_cuTensorMapEncodeTiled_v12000 encode = [] {
    void *fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) !=
            cudaSuccess || q != cudaDriverEntryPointSuccess)
      fn = nullptr;
    return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
  }();
  if (!encode) {
    *err = "cuTensorMapEncodeTiled is not available";
    return false;
  }
  cuuint64_t gd[5] = {dims[0], dims[1], dims[2], dims[3], (cuuint64_t)S};
  cuuint64_t gs[4] = {strides[0], strides[1], strides[2], slice_bytes};
  cuuint32_t bx[5] = {mn ? 64u : (cuuint32_t)kEmuKB, mn ? (cuuint32_t)kEmuKB : box[0], box[1], box[2], (cuuint32_t)S};
  cuuint32_t es[5] = {1, 1, 1, 1, 1};
  CUresult r = encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void *>(base), gd, gs, bx, es,
                      CU_TENSOR_MAP_INTERLEAVE_NONE, mn ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
                      CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    *err = "cuTensorMapEncodeTiled failed (" + std::to_string((int)r) + ")";
    return false;
  }
  return true;
}

template <int S, int N, bool AMN = false>
static cudaError_t launch_sn(const TcMaps &maps, const TcItem *items, const TcSeg *segs, int nitems,
                            const EmuEpi &epi, int *status, cudaStream_t st) {
  const int stage = (S == kEmuSlices ? kEmuStored : S) * (128 + epi.n) * kRowB;
  const int stages = std::max(2, std::min(6, (220 * 1024) / stage));
  const int smem = 1024 + stages * stage + 256;
  cudaError_t e = cudaFuncSetAttribute(emu_gemm_kernel<S, N, AMN>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  emu_gemm_kernel<S, N, AMN><<<std::min(nitems, 152), 320, smem, st>>>(maps, items, segs, nitems, stages, epi, status);
  return cudaGetLastError();
}

cudaError_t launch_emu_gemm(int S, const TcMaps &maps, const TcItem *items, const TcSeg *segs,
                            int nitems, const EmuEpi &epi, int *status, cudaStream_t st) {
  if (nitems <= 0) return cudaSuccess;
  switch (S * 1000 + epi.n + (epi.amn ? 100 : 0)) {
#define EMU_CASE(s, n) \
  case s * 1000 + n: return launch_sn<s, n>(maps, items, segs, nitems, epi, status, st)
#define EMU_CASE2(n)  \
  EMU_CASE(8, n);     \
  case 8100 + n: return launch_sn<8, n, true>(maps, items, segs, nitems, epi, status, st)
    EMU_CASE2(16);
    EMU_CASE2(32);
    EMU_CASE2(48);
    EMU_CASE(2, 32);
    EMU_CASE(2, 80);
    EMU_CASE(3, 32);
    EMU_CASE(3, 80);
    EMU_CASE(4, 32);
    EMU_CASE(4, 80);
    EMU_CASE(5, 32);
    EMU_CASE(5, 80);
    EMU_CASE(6, 32);
    EMU_CASE(6, 80);
#undef EMU_CASE
#undef EMU_CASE2
    default: return cudaErrorInvalidValue;
  }
}

// ---- scales ----
__global__ void __launch_bounds__(256) emu_absmax_kernel(const double *__restrict__ x, long long n,
                                                         EmuScale *scale) {
  const EmuScale inf = 0x7ffULL << 52;
  EmuScale m = 0;
  const long long step = (long long)gridDim.x * 256;
  long long i = (long long)blockIdx.x * 256 + threadIdx.x;
  for (; i + 3 * step < n; i += 4 * step) {
    EmuScale b[4];
#pragma unroll
    for (int q = 0; q < 4; ++q)
      b[q] = (EmuScale)__double_as_longlong(x[i + q * step]) & ~(1ULL << 63);
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (b[q] < inf && b[q] > m) m = b[q];
  }
  for (; i < n; i += step) {
    const EmuScale b = (EmuScale)__double_as_longlong(x[i]) & ~(1ULL << 63);
    if (b < inf && b > m) m = b;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const EmuScale b = __shfl_xor_sync(0xffffffffu, m, o);
    if (b > m) m = b;
  }
  __shared__ EmuScale red[8];
  if (threadIdx.x % 32 == 0) red[threadIdx.x / 32] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w)
      if (red[w] > m) m = red[w];
    if (m) atomicMax(scale, m);
  }
}

cudaError_t emu_absmax(const double *x, long long n, EmuScale *scale, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  const long long g = std::min<long long>((n + 2047) / 2048, 152LL * 8);
  emu_absmax_kernel<<<(int)std::max(1LL, g), 256, 0, st>>>(x, n, scale);
  return cudaGetLastError();
}

__global__ void emu_balance_kernel(EmuScale *a, const EmuScale *g, const EmuScale *t, EmuScale *u,
                                   int *status) {
  const int eg = scale_exp(*g), et = scale_exp(*t);
  const bool tu = *t != 0 && *u != 0;
  const int ea = tu ? max(scale_exp(*a), et + scale_exp(*u) - eg) : scale_exp(*a), eu = ea + eg - et;
  if (tu && (ea > 1024 || eu > 1024 || ea < -1022 || eu < -1022)) atomicOr(status, kStatusSpread);
  auto pack = [](int e) { return (EmuScale)min(2046, max(0, e + 1022)) << 52; };
  *a = pack(ea);
  *u = pack(eu);
}

cudaError_t emu_balance(EmuScale *a, const EmuScale *g, const EmuScale *t, EmuScale *u, int *status,
                        cudaStream_t st) {
  emu_balance_kernel<<<1, 1, 0, st>>>(a, g, t, u, status);
  return cudaGetLastError();
}

// ---- digits ----
// x over 2^(e - 63), rounded to nearest: an integer below 2^63 - 2^56 for a scale's e.
__device__ __forceinline__ long long to_fixed63(double x, int e) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  int ex = (int)((b >> 52) & 0x7ff);
  unsigned long long m = b & ((1ULL << 52) - 1);
  if (ex) m |= 1ULL << 52;
  else ex = 1;
  const int s = ex - 1012 - e;  // m 2^(ex - 1075) 2^(63 - e)
  unsigned long long q;
  if (s >= 0) q = m << min(s, 10);
  else if (s > -55) q = (m + (1ULL << (-s - 1))) >> -s;
  else q = 0;
  return (b >> 63) ? -(long long)q : (long long)q;
}

// Tiles of 32 rows x 64 K elements pass through shared memory, so that the loads
// run along whichever index is contiguous in the source; each thread then makes
// the digits of eight consecutive K elements of a row and writes 16 bytes of
// every slice.  The digits of the integer q are the bytes of
// q + 0x0080..80, minus 128 each (the top byte: q's own, in [-127, 127]); a byte
// becomes a bfloat16 through the FP32 number 2^23 + byte.  Bound by HBM: 8 bytes
// read and 18 written per element.
// MAXIMA: no digits, the rows' largest magnitudes instead.
template <bool MAXIMA>
__global__ void __launch_bounds__(256) emu_digits_kernel(const EmuView v, int Kp, long long slice,
                                                         int neg, EmuScale *scale, long long zs, int rs,
                                                         __nv_bfloat16 *__restrict__ out) {
  __shared__ double sm[32][65];
  __shared__ long long ro[32], ko[64];
  const int tid = threadIdx.x;
  const int tr = (v.R + 31) / 32, tk = (Kp + 63) / 64;
  const long long tiles = (long long)v.Z * tr * tk;
  const bool kfast = v.K2 > 1 ? v.sk2 == 1 : v.sk1 == 1;
  for (long long t = blockIdx.x; t < tiles; t += gridDim.x) {
    const int kt = (int)(t % tk);
    const long long t2 = t / tk;
    const int rt = (int)(t2 % tr), z = (int)(t2 / tr);
    const int r0 = rt * 32, k0 = kt * 64;
    __syncthreads();
    if (tid < 32) {
      const int r = r0 + tid;
      ro[tid] = r < v.R ? (long long)(r / v.R2) * v.sr1 + (long long)(r % v.R2) * v.sr2 : -1;
    } else if (tid < 96) {
      const int k = k0 + tid - 32;
      ko[tid - 32] = k < v.K ? (long long)(k / v.K2) * v.sk1 + (long long)(k % v.K2) * v.sk2 : -1;
    }
    __syncthreads();
    const double *src = v.x + (long long)(z / v.Z2) * v.sz1 + (long long)(z % v.Z2) * v.sz2;
    double x[8];
    int rr[8], kk[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int el = tid + 256 * q;
      if (kfast) {
        kk[q] = el % 64;
        rr[q] = el / 64;
      } else {
        rr[q] = el % 32;
        kk[q] = el / 32;
      }
      const long long a = ro[rr[q]], b = ko[kk[q]];
      x[q] = (a >= 0 && b >= 0) ? src[a + b] : 0.0;
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) sm[rr[q]][kk[q]] = x[q];
    __syncthreads();
    const int r = tid / 8, kg = (tid % 8) * 8;
    EmuScale *const rscale = scale + z * zs + (long long)(r0 + r) * rs;
    if constexpr (MAXIMA) {
      EmuScale m = 0;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const EmuScale b = (EmuScale)__double_as_longlong(sm[r][kg + j]) & ~(1ULL << 63);
        if (b < (0x7ffULL << 52) && b > m) m = b;
      }
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) {
        const EmuScale b = __shfl_xor_sync(0xffffffffu, m, o);
        if (b > m) m = b;
      }
      if (kg == 0 && m && r0 + r < v.R) atomicMax(rscale, m);
      continue;
    }
    if (r0 + r < v.R && k0 + kg < Kp) {
      const int e = scale_exp(*rscale);
      unsigned lo[8], hi[8], mag[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        double y = sm[r][kg + j];
        // |y| 2^-e in binary32 (20 bits of it), less c, in bfloat16
        const unsigned h = (unsigned)__double2hiint(y) & 0x7fffffffu;
        const int k = (int)(h >> 20) - 1023 - e;
        const float m = k < -100 ? 0.f : __uint_as_float(((unsigned)(127 + k) << 23) | ((h & 0xfffffu) << 3));
        mag[j] = __float_as_uint(m - kEmuRound) >> 16;
        if (m == kEmuRound) mag[j] = (127u - 40u) << 7;
        if ((h | (unsigned)__double2loint(y)) == 0) mag[j] = 0u;
        if (h >= 0x7ff00000u) {
          y = 0.0;
          mag[j] = 0x7fc0u;
        }
        long long q = to_fixed63(y, e);
        if (neg) q = -q;
        const unsigned long long w =
            ((unsigned long long)q + 0x0080808080808080ULL) ^ 0x8000000000000000ULL;
        lo[j] = (unsigned)w;
        hi[j] = (unsigned)(w >> 32);
      }
      uint4 *o = reinterpret_cast<uint4 *>(out + ((long long)z * v.R + r0 + r) * Kp + k0 + kg);
      const long long st = slice / 8;  // uint4 units
#pragma unroll
      for (int s = 0; s < 8; ++s) {
        unsigned p[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const unsigned wa = s < 4 ? hi[2 * j] : lo[2 * j], wb = s < 4 ? hi[2 * j + 1] : lo[2 * j + 1];
          const unsigned sel = 0x7440u | (unsigned)(3 - (s & 3));  // byte, 0, 0, 0x4B
          const float fa = __uint_as_float(__byte_perm(wa, 0x4B000000u, sel)) - 8388736.f;
          const float fb = __uint_as_float(__byte_perm(wb, 0x4B000000u, sel)) - 8388736.f;
          p[j] = __byte_perm(__float_as_uint(fa), __float_as_uint(fb), 0x7632);
        }
        o[s * st] = make_uint4(p[0], p[1], p[2], p[3]);
      }
      o[8 * st] = make_uint4(mag[0] | mag[1] << 16, mag[2] | mag[3] << 16, mag[4] | mag[5] << 16,
                             mag[6] | mag[7] << 16);
    }
  }
}

cudaError_t emu_digits(const EmuView &v, long long Kp, bool neg, const EmuScale *scale, long long zs,
                       int rs, __nv_bfloat16 *out, cudaStream_t st) {
  if (v.Z <= 0 || v.R <= 0 || Kp <= 0) return cudaSuccess;
  const long long tiles = (long long)v.Z * ((v.R + 31) / 32) * ((Kp + 63) / 64);
  const long long slice = (long long)v.Z * v.R * Kp;
  emu_digits_kernel<false><<<(int)std::min<long long>(tiles, 152LL * 32), 256, 0, st>>>(
      v, (int)Kp, slice, neg ? 1 : 0, const_cast<EmuScale *>(scale), zs, rs, out);
  return cudaGetLastError();
}

cudaError_t emu_row_maxima(const EmuView &v, EmuScale *scale, long long zs, int rs, cudaStream_t st) {
  if (v.Z <= 0 || v.R <= 0 || v.K <= 0) return cudaSuccess;
  const long long tiles = (long long)v.Z * ((v.R + 31) / 32) * ((v.K + 63) / 64);
  emu_digits_kernel<true><<<(int)std::min<long long>(tiles, 152LL * 32), 256, 0, st>>>(
      v, v.K, 0, 0, scale, zs, rs, nullptr);
  return cudaGetLastError();
}

}  // namespace mlcc3
