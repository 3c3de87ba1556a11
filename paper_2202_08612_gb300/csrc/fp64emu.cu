// FP64-accurate matrix products on the BF16 tensor cores by error-free
// splitting (the scheme of Ozaki, Ogita, Oishi and Rump): every row of A and of
// B is scaled by a power of two to below 1 in magnitude and written as s
// balanced base-256 digits, each an integer in [-128, 128] and so exact in
// bfloat16; emu_gemm_kernel multiplies the digit pairs (t, u) with t + u < s
// and sums them as integers.  The dropped terms lie below 2^-8s of the leading
// one, so s = 5 gives products to about 1e-12 relative (normwise), at
// s (s + 1) / 2 BF16 products per product.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <mutex>
#include <string>
#include <vector>

#include "kernels_emu.cuh"
#include "mlcc3.h"
#include "workpool.cuh"

namespace mlcc3 {

void set_last_error(const std::string &msg);

namespace {
constexpr int kMaxDev = 64;
std::mutex g_pool_mutex;
cudaMemPool_t g_pool[kMaxDev] = {};
}  // namespace

cudaError_t work_alloc(void **p, size_t bytes, cudaStream_t st) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDev) return cudaErrorInvalidDevice;
  cudaMemPool_t pool;
  {
    std::lock_guard<std::mutex> lock(g_pool_mutex);
    if (!g_pool[dev]) {
      cudaMemPoolProps props{};
      props.allocType = cudaMemAllocationTypePinned;
      props.location.type = cudaMemLocationTypeDevice;
      props.location.id = dev;
      if ((e = cudaMemPoolCreate(&g_pool[dev], &props)) != cudaSuccess) {
        g_pool[dev] = nullptr;
        return e;
      }
      uint64_t keep = kWorkKeep;
      cudaMemPoolSetAttribute(g_pool[dev], cudaMemPoolAttrReleaseThreshold, &keep);
    }
    pool = g_pool[dev];
  }
  return cudaMallocFromPoolAsync(p, bytes, pool, st);
}

void work_free(void *p, cudaStream_t st) {
  if (p) cudaFreeAsync(p, st);
}

void work_trim() {
  std::lock_guard<std::mutex> lock(g_pool_mutex);
  for (cudaMemPool_t pool : g_pool)
    if (pool) cudaMemPoolTrimTo(pool, 0);
}

// Row r of X (one block): its exponent e[r], |X[r][k]| < 2^e[r] (0 for a zero
// row), and its s digit slices: q = X[r][k] 2^(8s - 1 - e[r]) rounded to nearest
// even, |q| <= 2^(8s-1), as q = sum_t d_t 256^(s-1-t) with d_t in [-128, 128]
// (t = 0 the most significant, halves rounded to even); slice t is [rows][Kp] in
// bfloat16, zero for k >= K.  On the integer pipe: a form in FP64 arithmetic spent
// 1.5 ms on the 4096 x 4096 operands whose memory traffic takes 0.1 ms.  The row
// is read twice, the second time from the caches.  A row with an element that is
// not finite gives NaN products.
__global__ void __launch_bounds__(128) emu_slice_rows_kernel(const double *__restrict__ X, long long rows,
                                                             int K, long long ld, int Kp, int s,
                                                             int *__restrict__ e,
                                                             __nv_bfloat16 *__restrict__ slices) {
  const long long r = blockIdx.x;
  const double *x = X + r * ld;
  __shared__ unsigned long long red[4];
  unsigned long long m = 0;  // largest magnitude's bits: their order is the numbers'
  for (int k = threadIdx.x; k < K; k += 128) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x[k]) & ~(1ULL << 63);
    m = b > m ? b : m;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long b = __shfl_xor_sync(0xffffffffu, m, o);
    m = b > m ? b : m;
  }
  if (threadIdx.x % 32 == 0) red[threadIdx.x / 32] = m;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < 4; ++w) m = red[w] > m ? red[w] : m;
  int ex = 0;
  if (m != 0) {
    ex = (int)(m >> 52);
    if (ex == 0) ex = 12 - __clzll((long long)m);  // subnormal: 2^(ex - 1022) bounds it all the same
    ex -= 1022;
  }
  const bool bad = (m >> 52) == 0x7ff;
  if (threadIdx.x == 0) e[r] = bad ? 0 : ex;
  for (int k0 = threadIdx.x * 8; k0 < Kp; k0 += 128 * 8) {
    long long q[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const unsigned long long b =
          k0 + j < K && !bad ? (unsigned long long)__double_as_longlong(x[k0 + j]) : 0ULL;
      int eb = (int)((b >> 52) & 0x7ff);
      unsigned long long mm = b & ((1ULL << 52) - 1);
      if (eb) mm |= 1ULL << 52;
      else eb = 1;
      const int sh = 1075 - eb - (8 * s - 1 - ex);  // right shift of the significand
      unsigned long long v = 0;
      if (sh <= 0) v = mm << -sh;  // a subnormal row's significand may move left
      else if (sh < 55) v = (mm + ((1ULL << (sh - 1)) - 1) + ((mm >> sh) & 1)) >> sh;
      q[j] = (b >> 63) ? -(long long)v : (long long)v;
    }
    for (int t = s - 1; t >= 0; --t) {
      unsigned p[4];
#pragma unroll
      for (int j = 0; j < 8; j += 2) {
        float f[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int b = (int)(q[j + i] & 255);
          const long long h = q[j + i] >> 8;
          const int up = b + (int)(h & 1) > 128 ? 1 : 0;  // halves to even
          q[j + i] = h + up;
          f[i] = __int_as_float(0x4B400000 + b - 256 * up) - 12582912.f;
          if (t == 0 && bad) f[i] = __int_as_float(0x7fc00000);
        }
        p[j / 2] = __byte_perm(__float_as_uint(f[0]), __float_as_uint(f[1]), 0x7632);
      }
      *reinterpret_cast<uint4 *>(slices + ((long long)t * rows + r) * Kp + k0) = make_uint4(p[0], p[1], p[2], p[3]);
    }
  }
}

}  // namespace mlcc3

using namespace mlcc3;

extern "C" int mlcc3_release_workspace(void) {
  work_trim();
  return MLCC3_OK;
}

// C = A B^T (FP64 device arrays; A [M][K] rows lda apart, B [N][K] rows ldb
// apart, C [M][N] rows ldc apart) from `slices` digit slices of each operand.
// Takes its temporaries (digit slices, exponents, the tile list) from the work
// pool, runs on `stream` and returns when the product is in C.
extern "C" int mlcc3_fp64emu_gemm(const double *A, long long lda, const double *B, long long ldb,
                                  double *C, long long ldc, int M, int N, int K, int slices,
                                  void *stream) {
  if (!A || !B || !C || M <= 0 || N <= 0 || K <= 0 || lda < K || ldb < K || ldc < N ||
      slices < 2 || slices > 6) {
    set_last_error("mlcc3_fp64emu_gemm: bad arguments (slices must be 2..6)");
    return MLCC3_ERR_ARG;
  }
  for (const void *p : {static_cast<const void *>(A), static_cast<const void *>(B),
                        static_cast<const void *>(C)}) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess ||
        (a.type != cudaMemoryTypeDevice && a.type != cudaMemoryTypeManaged)) {
      cudaGetLastError();
      set_last_error("mlcc3_fp64emu_gemm: A, B and C must be device pointers");
      return MLCC3_ERR_ARG;
    }
  }
  const int s = slices;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int Kp = (K + kEmuKB - 1) / kEmuKB * kEmuKB;
  void *mem = nullptr;
  auto cleanup = [&] {
    work_free(mem, st);
    return cudaStreamSynchronize(st);
  };
  auto fail = [&](int code, const std::string &m) {
    cleanup();
    cudaGetLastError();
    set_last_error("mlcc3_fp64emu_gemm: " + m);
    return code;
  };
  // items: output tiles, their reductions cut where few tiles would leave SMs
  // idle (pieces of at least 512) or where they exceed an item's bound; the
  // pieces of one tile add into the zeroed C
  const int n = emu_tile_width(N, s), nk = Kp / kEmuKB;
  const long long tiles = (long long)((M + 127) / 128) * ((N + n - 1) / n);
  const int pieces = (int)std::max<long long>(
      (Kp + kEmuMaxK - 1) / kEmuMaxK,
      std::min<long long>((152 + tiles - 1) / tiles, std::max(1, nk * kEmuKB / 512)));
  const int per = (nk + pieces - 1) / pieces;
  std::vector<TcItem> items;
  std::vector<TcSeg> segs;
  for (int n0 = 0; n0 < N; n0 += n)
    for (int m0 = 0; m0 < M; m0 += 128)
      for (int k0 = 0; k0 < nk; k0 += per) {
        TcItem it{};
        it.seg_begin = (int)segs.size();
        it.seg_count = 1;
        it.r2_0 = m0;
        it.c0 = n0;
        TcSeg sg{};
        sg.amap = 0;
        sg.bmap = 1;
        sg.nk = std::min(per, nk - k0);
        sg.ac[0] = sg.bc[0] = kEmuKB * k0;
        sg.ac[1] = m0;
        sg.bc[1] = n0;
        it.chunks = sg.nk;
        segs.push_back(sg);
        items.push_back(it);
      }
  // one allocation: slices of A and B, exponents, tiles, status
  size_t total = 0;
  auto part = [&](size_t bytes) {
    const size_t at = total;
    total += (bytes + 255) / 256 * 256;
    return at;
  };
  const size_t oa = part(sizeof(__nv_bfloat16) * s * M * (size_t)Kp), ob = part(sizeof(__nv_bfloat16) * s * N * (size_t)Kp);
  const size_t oea = part(sizeof(int) * M), oeb = part(sizeof(int) * N);
  const size_t oi = part(sizeof(TcItem) * items.size()), os = part(sizeof(TcSeg) * segs.size()), ost = part(sizeof(int));
  if (work_alloc(&mem, total, st) != cudaSuccess) return fail(MLCC3_ERR_OOM, "workspace");
  char *base = static_cast<char *>(mem);
  __nv_bfloat16 *sa = reinterpret_cast<__nv_bfloat16 *>(base + oa), *sb = reinterpret_cast<__nv_bfloat16 *>(base + ob);
  int *ea = reinterpret_cast<int *>(base + oea), *eb = reinterpret_cast<int *>(base + oeb);
  int *status = reinterpret_cast<int *>(base + ost);
  cudaMemsetAsync(status, 0, sizeof(int), st);
  cudaMemcpyAsync(base + oi, items.data(), sizeof(TcItem) * items.size(), cudaMemcpyHostToDevice, st);
  cudaMemcpyAsync(base + os, segs.data(), sizeof(TcSeg) * segs.size(), cudaMemcpyHostToDevice, st);
  // C is cleared before the operands are sliced (beside the copies above; between kernels
  // it takes 6 us more), unless it may be one of them
  auto over = [&](const double *x, long long rows, long long ld) {
    return C < x + rows * ld && x < C + (long long)M * ldc;
  };
  const bool in_place = over(A, M, lda) || over(B, N, ldb);
  auto clear = [&] { cudaMemset2DAsync(C, sizeof(double) * ldc, 0, sizeof(double) * N, M, st); };
  if (pieces > 1 && !in_place) clear();
  emu_slice_rows_kernel<<<M, 128, 0, st>>>(A, M, K, lda, Kp, s, ea, sa);
  emu_slice_rows_kernel<<<N, 128, 0, st>>>(B, N, K, ldb, Kp, s, eb, sb);
  if (pieces > 1 && in_place) clear();
  if (cudaGetLastError() != cudaSuccess) return fail(MLCC3_ERR_CUDA, "slice kernels");
  TcMaps maps{};
  std::string err;
  auto enc = [&](int slot, const void *p, long long rows, unsigned box_rows) {
    const unsigned long long rb = (unsigned long long)Kp * 2;
    const unsigned long long dims[4] = {(unsigned long long)Kp, (unsigned long long)rows, 1, 1};
    const unsigned long long str[3] = {rb, rb * rows, rb * rows};
    const unsigned box[3] = {box_rows, 1, 1};
    return emu_encode_map(&maps.m[slot], p, dims, str, rb * rows, box, s, &err);
  };
  if (!enc(0, sa, M, 128) || !enc(1, sb, N, (unsigned)n)) return fail(MLCC3_ERR_CUDA, err);
  EmuEpi epi{};
  epi.out = C;
  epi.mode = pieces > 1 ? 1 : 0;
  epi.R2 = 128;
  epi.s2 = ldc;
  epi.sn = 1;
  epi.lim1 = 1;
  epi.lim2 = M;
  epi.nlim = N;
  epi.alpha = 1.0;
  epi.n = n;
  epi.ebias = -14;
  epi.ea = ea;
  epi.eb = eb;
  cudaError_t e = launch_emu_gemm(s, maps, reinterpret_cast<TcItem *>(base + oi), reinterpret_cast<TcSeg *>(base + os),
                                  (int)items.size(), epi, status, st);
  int hst = 0;
  if (e == cudaSuccess) e = cudaMemcpyAsync(&hst, status, sizeof(int), cudaMemcpyDeviceToHost, st);
  if (e != cudaSuccess) return fail(MLCC3_ERR_CUDA, cudaGetErrorString(e));
  if ((e = cleanup()) != cudaSuccess) {
    mem = nullptr;
    return fail(MLCC3_ERR_CUDA, cudaGetErrorString(e));
  }
  if (hst & kStatusTimeout) {
    set_last_error("mlcc3_fp64emu_gemm: a tensor-core pipeline wait timed out");
    return MLCC3_ERR_TIMEOUT;
  }
  return MLCC3_OK;
}
