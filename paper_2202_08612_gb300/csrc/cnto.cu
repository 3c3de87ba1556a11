// CNTO matrices (Sec. 2, Eqs. M and N): the occupied and virtual correlated
// natural transition orbitals of an excited state are the eigenvectors of
//   M_ij = sum_a R^a_i R^a_j + 1/2 sum_{abk} (1 + delta_{ai,bk} delta_ij) R^{ab}_{ik} R^{ab}_{jk}
//   N_ab = sum_i R^a_i R^b_i + 1/2 sum_{cij} (1 + delta_{ai,cj} delta_ab) R^{ac}_{ij} R^{bc}_{ij}
// Both are Gram matrices of views of the doubles (full storage
// R2[A][I][B][J] = R^{AB}_{IJ}) with a long reduction: M over (b, k) for every
// a, N over (i, c, j).  One FP64 kernel computes C[m][n] += alpha sum_k
// A[m][k] A[n][k] for a batch of strided views, the reduction split across
// blocks (partial sums added atomically), 64 x 64 output tiles staged through
// shared memory.  It runs where the digit slices (kernels_emu.cuh) with which the doubles'
// matrices run on the tensor cores find no room, or where an element of M or N is too
// small beside the largest amplitude for them (kStatusSpread); the
// singles and the diagonal term have a kernel of one thread per element.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstring>
#include <string>
#include <vector>

#include "kernels_emu.cuh"
#include "mlcc3.h"
#include "workpool.cuh"

namespace mlcc3 {
void set_last_error(const std::string &msg);
}

namespace {

constexpr int TM = 64, TK = 16;

struct GramView {
  const double *A;
  long long rows, K;     // C is rows x rows
  long long rs, ks;      // element strides of a row and of the reduction index
  long long batch, bs;   // batch count and stride (summed into the same C)
  long long kchunk;      // reduction elements per block (blockIdx.z)
};

// blockIdx.x: output tile (tm, tn) with tn >= tm (C symmetric: the mirror is
// written too), blockIdx.y: batch index, blockIdx.z: reduction chunk.
__global__ void __launch_bounds__(256) gram_kernel(GramView v, double alpha, double *C) {
  __shared__ double As[TK][TM + 1], Bs[TK][TM + 1];
  const long long nt = (v.rows + TM - 1) / TM;
  long long t = blockIdx.x, tm = 0;
  while (t >= nt - tm) {  // upper-triangular tile index -> (tm, tn)
    t -= nt - tm;
    ++tm;
  }
  const long long tn = tm + t;
  const double *A = v.A + (long long)blockIdx.y * v.bs;
  const long long k0 = (long long)blockIdx.z * v.kchunk;
  const long long k1 = min(v.K, k0 + v.kchunk);
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  double acc[4][4] = {};
  for (long long kb = k0; kb < k1; kb += TK) {
    for (int e = threadIdx.x; e < TK * TM; e += 256) {
      const int kk = e / TM, r = e % TM;
      const long long k = kb + kk;
      const long long ra = tm * TM + r, rb = tn * TM + r;
      As[kk][r] = (k < k1 && ra < v.rows) ? A[ra * v.rs + k * v.ks] : 0.0;
      Bs[kk][r] = (k < k1 && rb < v.rows) ? A[rb * v.rs + k * v.ks] : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < TK; ++kk) {
      double a[4], b[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        a[q] = As[kk][ty + 16 * q];
        b[q] = Bs[kk][tx + 16 * q];
      }
#pragma unroll
      for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[p][q] = fma(a[p], b[q], acc[p][q]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int p = 0; p < 4; ++p)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const long long m = tm * TM + ty + 16 * p, n = tn * TM + tx + 16 * q;
      if (m < v.rows && n < v.rows) {
        atomicAdd(C + m * v.rows + n, alpha * acc[p][q]);
        if (tm != tn) atomicAdd(C + n * v.rows + m, alpha * acc[p][q]);
      }
    }
}

// The singles' parts and the delta factor's diagonals (Eqs. M and N), which also set M and N:
// M_ij = sum_a R1_ai R1_aj + delta_ij 1/2 sum_a d_ai^2, N_ab = sum_i R1_ai R1_bi +
// delta_ab 1/2 sum_i d_ai^2 with d_ai = R^{aa}_{ii}.  A thread per element (64 x 64
// tiles of this size, mostly padding on the FP64 pipe, took 0.3 ms).
__global__ void cnto_singles_kernel(const double *R1, const double *R2, long long NO, long long NV,
                                    double *M, double *N) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const bool occ = e < NO * NO;
  const long long f = occ ? e : e - NO * NO, rows = occ ? NO : NV, K = occ ? NV : NO;
  if (f >= rows * rows) return;
  const long long p = f / rows, q = f % rows, rs = occ ? 1 : NO, ks = occ ? NO : 1;
  double s = 0.0, d2 = 0.0;
  for (long long k = 0; k < K; ++k) s = fma(R1[p * rs + k * ks], R1[q * rs + k * ks], s);
  if (p == q)
    for (long long k = 0; k < K; ++k) {
      const long long a = occ ? k : p, i = occ ? p : k;
      const double d = R2[((a * NO + i) * NV + a) * NO + i];
      d2 = fma(d, d, d2);
    }
  (occ ? M : N)[f] = fma(0.5, d2, s);
}

// X[i][j] += the copies' sum, for j >= i, and X[j][i] = X[i][j].
__global__ void fold_kernel(double *X, long long n, const double *copy, int copies) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n * n) return;
  const long long i = e / n, j = e % n;
  if (j < i) return;
  double s = 0.0;
  for (int c = 0; c < copies; ++c) s += copy[c * n * n + e];
  s += X[e];
  X[e] = s;
  X[j * n + i] = s;
}

// M_ij += 1/2 sum_a sum_K P[(a,i)][K] P[(a,j)][K] and N_ab += 1/2 sum_i sum_K P[(a,i)][K]
// P[(b,i)][K], P the doubles as an n x n matrix (n = N_O N_V), on the tensor cores.
// The digits of P's rows serve both: rows i of block a, or rows a (n_o rows apart)
// of block i, are two tensor maps over the same memory.  K runs in chunks whose
// digits take at most a gigabyte.  *status: the launches' status bits (with
// kStatusSpread M and N are left as they were).  39 / 263: 70.3 -> 3.6 ms, error 1.3e-15 -> 7e-17.
cudaError_t doubles_by_digits(long long NO, long long NV, const double *R2, double *M, double *N,
                              cudaStream_t st, int *hstatus, std::string *err) {
  using namespace mlcc3;
  const long long n = NO * NV;
  const long long most = std::max<long long>(kEmuKB, (((long long)1 << 30) - (64 << 20)) / (2 * kEmuStored * n) / kEmuKB * kEmuKB);
  const long long parts = (n + most - 1) / most, kc = ((n + parts - 1) / parts + kEmuKB - 1) / kEmuKB * kEmuKB;
  struct Gram {
    long long rows, blocks, row_stride, block_stride;  // strides in rows of P
    double *out;
    int copies;
  } g[2] = {{NO, NV, 1, NO, M, 1}, {NV, NO, NO, 1, N, 1}};
  std::vector<TcItem> items[2];
  std::vector<TcSeg> segs[2];
  // tiles on and above the diagonal, their reductions (all blocks' chunk after chunk)
  // cut into about eight items per SM of whole accumulation chains.  A thousand parts
  // added one by one to the same element would round more often than the FP64 kernel's
  // sums, so the p parts of a tile go to sqrt(p) copies, which one kernel adds up
  const int nk = (int)(kc / kEmuKB);
  int w[2];
  for (int q = 0; q < 2; ++q) {
    w[q] = emu_tile_width(g[q].rows, kEmuSlices);
    long long tiles = 0;
    for (long long m0 = 0; m0 < g[q].rows; m0 += 128) tiles += (g[q].rows + w[q] - 1) / w[q] - m0 / w[q];
    const long long all = g[q].blocks * nk, chain = kEmuChain;
    const long long per =
        std::min<long long>(kEmuMaxK / kEmuKB, std::max<long long>(1, all * tiles / (1216 * chain)) * chain);
    const long long np = (all + per - 1) / per;
    while (g[q].copies < 32 && g[q].copies * g[q].copies < np) ++g[q].copies;
    for (long long c0 = 0; c0 < all; c0 += per)
      for (long long m0 = 0; m0 < g[q].rows; m0 += 128)
        for (long long n0 = m0 / w[q] * w[q]; n0 < g[q].rows; n0 += w[q]) {
          TcItem it{};
          it.seg_begin = (int)segs[q].size();
          it.r2_0 = (int)m0;
          it.c0 = (int)n0;
          it.out_off = c0 / per % g[q].copies * g[q].rows * g[q].rows;
          for (long long c = c0; c < std::min(all, c0 + per);) {
            TcSeg sg{};
            sg.amap = 0;
            sg.bmap = 1;
            sg.nk = (int)std::min(nk - c % nk, std::min(all, c0 + per) - c);
            sg.ac[0] = sg.bc[0] = (int)(c % nk * kEmuKB);
            sg.ac[1] = (int)m0;
            sg.bc[1] = (int)n0;
            sg.ac[2] = sg.bc[2] = (int)(c / nk);
            segs[q].push_back(sg);
            it.seg_count += 1;
            it.chunks += sg.nk;
            c += sg.nk;
          }
          items[q].push_back(it);
        }
  }
  size_t total = 0;
  auto part = [&](size_t bytes) {
    const size_t at = total;
    total += (bytes + 255) / 256 * 256;
    return at;
  };
  const size_t od = part((size_t)2 * kEmuStored * n * kc), os = part(sizeof(EmuScale)), ost = os + sizeof(EmuScale);
  // scale, status (both zero) and the tile lists go over in one copy
  size_t oi[2], og[2];
  for (int q = 0; q < 2; ++q) {
    oi[q] = part(sizeof(TcItem) * items[q].size());
    og[q] = part(sizeof(TcSeg) * segs[q].size());
  }
  const size_t head_bytes = total - os;
  size_t oc[2];
  for (int q = 0; q < 2; ++q) oc[q] = part(sizeof(double) * g[q].copies * g[q].rows * g[q].rows);
  std::vector<char> head(head_bytes, 0);
  for (int q = 0; q < 2; ++q) {
    std::memcpy(head.data() + (oi[q] - os), items[q].data(), sizeof(TcItem) * items[q].size());
    std::memcpy(head.data() + (og[q] - os), segs[q].data(), sizeof(TcSeg) * segs[q].size());
  }
  void *mem = nullptr;
  cudaError_t e = work_alloc(&mem, total, st);
  if (e != cudaSuccess) return e;
  char *base = static_cast<char *>(mem);
  __nv_bfloat16 *dig = reinterpret_cast<__nv_bfloat16 *>(base + od);
  EmuScale *scale = reinterpret_cast<EmuScale *>(base + os);
  int *status = reinterpret_cast<int *>(base + ost), hst = 0;
  e = cudaMemcpyAsync(base + os, head.data(), head.size(), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(base + oc[0], 0, total - oc[0], st);
  if (e == cudaSuccess) e = emu_absmax(R2, n * n, scale, st);
  for (long long k0 = 0; k0 < n && e == cudaSuccess; k0 += kc) {
    // (a shorter last chunk is padded with zeros)
    const EmuView v{R2 + k0, 1, 1, (int)n, (int)n, (int)std::min(kc, n - k0), 1, 0, 0, 0, n, 1, 0};
    e = emu_digits(v, kc, false, scale, 0, 0, dig, st);
    for (int q = 0; q < 2 && e == cudaSuccess; ++q) {
      TcMaps maps{};
      const unsigned long long rb = (unsigned long long)kc * 2;
      const unsigned long long dims[4] = {(unsigned long long)kc, (unsigned long long)g[q].rows,
                                          (unsigned long long)g[q].blocks, 1};
      const unsigned long long str[3] = {rb * g[q].row_stride, rb * g[q].block_stride, rb * n};
      const unsigned ba[3] = {128, 1, 1}, bb[3] = {(unsigned)w[q], 1, 1};
      if (!emu_encode_map(&maps.m[0], dig, dims, str, rb * n, ba, kEmuStored, err) ||
          !emu_encode_map(&maps.m[1], dig, dims, str, rb * n, bb, kEmuStored, err)) {
        e = cudaErrorInvalidValue;
        break;
      }
      EmuEpi epi{};
      epi.out = reinterpret_cast<double *>(base + oc[q]);
      epi.mode = 1;
      epi.R2 = 1 << 30;
      epi.s2 = g[q].rows;
      epi.sn = 1;
      epi.lim1 = 1;
      epi.lim2 = epi.nlim = (int)g[q].rows;
      epi.alpha = 0.5;
      epi.n = w[q];
      epi.ebias = -14;
      epi.sa = epi.sb = scale;
      e = launch_emu_gemm(kEmuSlices, maps, reinterpret_cast<TcItem *>(base + oi[q]),
                          reinterpret_cast<TcSeg *>(base + og[q]), (int)items[q].size(), epi, status, st);
    }
  }
  // the sums are added where all of them hold (the host waits here anyway)
  if (e == cudaSuccess) e = cudaMemcpyAsync(&hst, status, sizeof(int), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  for (int q = 0; q < 2 && e == cudaSuccess && hst == 0; ++q) {
    fold_kernel<<<(unsigned)((g[q].rows * g[q].rows + 255) / 256), 256, 0, st>>>(
        g[q].out, g[q].rows, reinterpret_cast<double *>(base + oc[q]), g[q].copies);
    e = cudaGetLastError();
  }
  work_free(mem, st);
  const cudaError_t e2 = cudaStreamSynchronize(st);
  if (e == cudaSuccess) e = e2;
  *hstatus = hst;
  return e;
}

bool on_device(const void *p) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

cudaError_t gram(const GramView &v0, double alpha, double *C, cudaStream_t st) {
  GramView v = v0;
  const long long nt = (v.rows + TM - 1) / TM, tiles = nt * (nt + 1) / 2;
  // split the reduction until about 4 x 152 blocks run
  long long z = std::max(1LL, std::min((4LL * 152 + tiles * v.batch - 1) / (tiles * v.batch),
                                       (v.K + 1023) / 1024));
  z = std::min(z, 65535LL);
  v.kchunk = ((v.K + z - 1) / z + TK - 1) / TK * TK;
  z = (v.K + v.kchunk - 1) / v.kchunk;
  for (long long b0 = 0; b0 < v.batch; b0 += 65535) {
    GramView w = v;
    w.A = v.A + b0 * v.bs;
    w.batch = std::min(65535LL, v.batch - b0);
    gram_kernel<<<dim3((unsigned)tiles, (unsigned)w.batch, (unsigned)z), 256, 0, st>>>(w, alpha, C);
  }
  return cudaGetLastError();
}

}  // namespace

extern "C" int mlcc3_cnto_matrices(int64_t n_occ, int64_t n_vir, const double *R1,
                                   const double *R2, double *M, double *N, void *cuda_stream) {
  const long long NO = n_occ, NV = n_vir;
  if (NO < 1 || NV < 1 || !R1 || !R2 || !M || !N) {
    mlcc3::set_last_error("mlcc3_cnto_matrices: bad dimensions or null pointer");
    return MLCC3_ERR_ARG;
  }
  if (!on_device(R1) || !on_device(R2) || !on_device(M) || !on_device(N)) {
    mlcc3::set_last_error("mlcc3_cnto_matrices: every array must be a device pointer");
    return MLCC3_ERR_ARG;
  }
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  cnto_singles_kernel<<<(unsigned)((NO * NO + NV * NV + 255) / 256), 256, 0, st>>>(R1, R2, NO, NV, M, N);
  cudaError_t e = cudaGetLastError();
  // doubles: M_ij += 1/2 sum_a sum_{(b,k)} R2[a][i][(b,k)] R2[a][j][(b,k)]
  //          N_ab += 1/2 sum_{(i,c,j)} R2[a][(i,c,j)] R2[b][(i,c,j)]
  // (the singles' parts are symmetric, so mirroring the sums keeps them)
  std::string err;
  bool done = false;
  int status = 0;
  if (e == cudaSuccess && NO * NV < (1LL << 20)) {
    e = doubles_by_digits(NO, NV, R2, M, N, st, &status, &err);
    done = e == cudaSuccess && status == 0;
    if (e == cudaErrorMemoryAllocation) {  // no room for a workspace: the FP64 kernel needs none
      cudaGetLastError();
      e = cudaSuccess;
    }
  }
  if (status & mlcc3::kStatusTimeout) {
    mlcc3::set_last_error("mlcc3_cnto_matrices: a tensor-core pipeline wait timed out");
    return MLCC3_ERR_TIMEOUT;
  }
  if (e == cudaSuccess && !done)
    e = gram(GramView{R2, NO, NV * NO, NV * NO, 1, NV, NO * NV * NO, 0}, 0.5, M, st);
  if (e == cudaSuccess && !done)
    e = gram(GramView{R2, NV, NO * NV * NO, NO * NV * NO, 1, 1, 0, 0}, 0.5, N, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) {
    mlcc3::set_last_error(std::string("mlcc3_cnto_matrices: ") + (err.empty() ? cudaGetErrorString(e) : err));
    return MLCC3_ERR_CUDA;
  }
  return MLCC3_OK;
}
