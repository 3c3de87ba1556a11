// FP64-accurate contractions on the BF16 tensor cores: operands as balanced
// base-256 digit slices (exact in bfloat16), every digit pair of one K chunk
// multiplied in one pipeline stage, integer accumulation outside TMEM.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <string>

#include "kernels_tc.cuh"

namespace mlcc3 {

constexpr int kEmuKB = 32;      // K elements per pipeline stage (64-byte rows)
constexpr int kEmuSlices = 8;   // digit slices of the FP64 mode
constexpr int kEmuStored = 9;   // slices of an FP64 operand: its digits and its magnitudes
// K chunks of one TMEM accumulation chain of the FP64 mode: 192 products, whose sums
// FP32 holds exactly up to degree 4 (5 pairs of 2^14 each), and at any degree unless
// nearly all of their digits have the largest magnitude and one sign
constexpr int kEmuChain = 6;
constexpr int kEmuMaxK = 8192;  // longest reduction of one item (TcSeg chunks times kEmuKB)

// The device status bit of a product that the digits cannot hold to FP64 accuracy.  With
// |A|, |B| the powers of two above the largest elements that share the operands' scales (a
// row's, or the whole operand's), rounding an operand to
// 2^-63 of its own errs by up to 2^-64 (|A| sum |b_k| + |B| sum |a_k|) in an output, over the
// K with a_k b_k != 0, and the digit pairs left out by up to 2^-69.4 K |A| |B|.  The kernel
// measures, for every output, P - c (|A| sum |b_k| + |B| sum |a_k|) with P = sum |a_k| |b_k| and
// c = 2^-14, and sets the bit unless that is zero (as every product is) or at least
// 2^-22 K |A| |B|.  So an output errs by less than 2^-50 P + 2^-47.4 P, where FP64 sums of 64
// products (2^6 roundings of 2^-53) may err by 2^-47 P; and by about as much as FP64 sums
// where the errors have random signs (the pairs left out 2^-72 K^(1/2) |A| |B|, FP64's
// 2^-51.5 K^(1/2) |a| |b|).  Without the bit an operand spread over 10^6 lost ten digits of
// its small outputs.
constexpr int kStatusSpread = 4;
constexpr float kEmuRound = 0x1p-14f;  // c
constexpr float kEmuLeast = 0x1p-22f;

// A digit operand's scale: the binary64 pattern of the operand's largest finite
// magnitude (or of any number at least as large); |x| < (1 - 2^-7) 2^e with e its exponent,
// raised by one where the number's own leading bits are above that.
using EmuScale = unsigned long long;

// Epilogue: out[off + r1 s1 + r2 s2 + n sn] (op) alpha sum_k A[r][k] B[n][k].
// mode 0: store; 1: add (global reductions).  The rest as in TcEpi.
struct EmuEpi {
  double *out;
  int mode;
  int R2, linear;
  long long s1, s2, sn;
  int lim1, lim2, nlim;
  double alpha;
  int amn;          // as TcEpi::amn (S = 8)
  int n;            // columns of a tile (a multiple of 16, at most emu_max_cols)
  int ebias;        // power of two of the leading digit product: -14
  // scales of the operands: one, or (ra, rb) one per row of A and of B (r2_0 + row and the
  // column, from the item's ea and eb on); S < 8: one exponent per output row and column
  const EmuScale *sa, *sb;
  int ra, rb;
  const int *ea, *eb;
  long long wait;   // as TcEpi::wait
};

// Widest tile of an S-slice launch: S n FP32 columns fit in TMEM's 512 and
// n / 2 accumulators per epilogue thread in its registers.  S = 8: ten groups of n
// columns (degrees 0..8 and the magnitudes).
__host__ __device__ constexpr int emu_max_cols(int S) { return S >= 7 ? 48 : 80; }
int emu_tile_width(long long n, int S);

// Tensor map of a digit operand over (K, dims1, dims2, dims3, slice); strides in
// bytes for dims 1..3 and the slice.  mn: dims[0] are the rows, dims[1] is K, for
// boxes of 64 rows x kEmuKB.
bool emu_encode_map(CUtensorMap *m, const void *base, const unsigned long long dims[4],
                    const unsigned long long strides[3], unsigned long long slice_bytes,
                    const unsigned box[3], int S, std::string *err, bool mn = false);

cudaError_t launch_emu_gemm(int S, const TcMaps &maps, const TcItem *items, const TcSeg *segs,
                            int nitems, const EmuEpi &epi, int *status, cudaStream_t st);

// *scale = max(*scale, largest finite |x|)
cudaError_t emu_absmax(const double *x, long long n, EmuScale *scale, cudaStream_t st);
// Scales of the two products of Eq. R3 made equal: A G and t U accumulate in one
// chain, so e_A + e_G = e_t + e_U; e_A and e_U are raised where they have to be.  Scales
// beyond binary64's exponents set kStatusSpread.
cudaError_t emu_balance(EmuScale *a, const EmuScale *g, const EmuScale *t, EmuScale *u,
                        int *status, cudaStream_t st);

// Source of a digit operand: element (z, r, k) at z1 sz1 + z2 sz2 + r1 sr1 +
// r2 sr2 + k1 sk1 + k2 sk2 with z = z1 Z2 + z2 and so on.
struct EmuView {
  const double *x;
  int Z, Z2, R, R2, K, K2;
  long long sz1, sz2, sr1, sr2, sk1, sk2;
};
// The kEmuSlices digit slices of `v` at `scale` (negated if neg), K padded with zeros to
// Kp, and as slice kEmuSlices |x| 2^-e - c in bfloat16 (zero only for x = 0, NaN where x is
// not finite), whose products add up to what kStatusSpread asks for and c^2 K more:
// out[slice][z][r][Kp].  Scale of row (z, r): scale[z zs + r rs].
cudaError_t emu_digits(const EmuView &v, long long Kp, bool neg, const EmuScale *scale, long long zs,
                       int rs, __nv_bfloat16 *out, cudaStream_t st);
// Those scales: the largest finite magnitude of each row's elements (of all rows that
// share one), where it is larger than the one there.
cudaError_t emu_row_maxima(const EmuView &v, EmuScale *scale, long long zs, int rs, cudaStream_t st);

}  // namespace mlcc3
