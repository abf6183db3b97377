// FP64 GEMM on the BF16 tensor pipe by exact digit products (the error-free splitting of Ozaki, Ogita,
// Oishi and Rump, Numer. Algorithms 59, 95 (2012)).
//
// GB300 issues two FP64 multiply-adds per clock and SM (0.53e12/s on the chip, measured) but 1024 BF16
// ones through mma.sync, so a product that is spelled out in small integers is the faster FP64 product.
// Every row of op(A) and column of op(B) is scaled by its own power of two and rounded to a fixed-point
// number X of 56 bits, |X| <= 2^55; X is written in 8 balanced digits of base 128, each a BF16 integer
// in [-64, 64].  Digit products are at most 2^12, so 128 of them for up to eight digit pairs sum exactly
// in an FP32 accumulator (2^22 at most); the pairs (s, t) with s + t = g share one accumulator, g <= 8,
// and the pairs with s + t > 8 (below 2^-62 of the largest product) are left out.  Every 128 k the
// accumulators are read as integers (adding 1.5 * 2^23 leaves the integer in the mantissa) and summed
// in two 64-bit integers, which nothing rounds; one rounding to FP64 per K slice is the only one after
// the rounding of X.  What comes here instead of to the streaming kernels, with times, stands
// at dgemm in linalg.cu.
//
// The operands' rounding is relative to the largest entry of the row or column, so an output that collects only
// products far below (max of the row) (max of the column) has fewer correct digits than an FP64 sum: with
// S_ij = sum_k |A_ik| |B_kj|, sA_i = sum_k |A_ik| / 2^eA, sB_j likewise (2^e just above the largest entry), the
// error is at most 2^-56 (sA + sB) + 6 K 2^-63 in units of 2^(eA + eB), an FP64 sum's K 2^-53 S.  The products
// of the library's solvers are norms, overlaps and rotations of whole vectors, where only the former matters.
// With CHECK (bse_gemm) every output for which the bound is above half of an FP64 sum's is summed anew in FP64,
// and the result is an FP64 product entry by entry, whatever the grading of rows and columns: row_exponents
// also returns sA and sB, the kernel estimates S by one more product per tile and 16 k, of the first two digits'
// magnitudes rounded to BF16, and the outputs it finds weak are dealt to whole warps, or summed together when a tile
// has many.  Kernel time with CHECK (without): N T 80 x 216 x 6859 69 us (66), N N 80 x 2400 x 64 20.5 (19.5), T N
// 200 x 6859 x 128 111 (114); with every output weak 298, 53 and 417 (as tiled FP64 kernels 384, 69 and 391).
#include <algorithm>
#include <atomic>
#include <cstdint>
#include <type_traits>

#include <cuda_bf16.h>

#include "internal.cuh"

namespace bse {
namespace {

constexpr int kND = 8;              // digits
constexpr int kKC = 16;             // k per staged chunk
constexpr int kRawStride = kKC + 2;  // doubles per staged row (16-byte aligned, rows off the same banks)
constexpr int kDigStride = kKC + 8;  // bf16 per digit row: ldmatrix reads 8 rows without bank conflicts
// 16-row strips of A and B per CTA (with CHECK the sums of S take the place of the ninth)
template <bool CHECK>
constexpr int kMaxStrips = CHECK ? 8 : 9;
constexpr int kWarps = 16;
constexpr int kFlush = 8;           // chunks between reads of the FP32 accumulators (128 k)
constexpr int kBadExp = 1 << 28;    // row holds a non-finite value
constexpr int kMaxSlice = 1 << 19;  // longest K slice
constexpr int kFewWeak = 64;        // weak outputs of a tile that go to one warp each
constexpr int kStageK = 64;         // k at a time for more

// |x| < 2^e  ->  round(x 2^(55 - e))
__device__ __forceinline__ long long to_fixed(double x, int e) {
  const long long b = __double_as_longlong(x);
  const int E = (int)((b >> 52) & 0x7ff);
  unsigned long long m = (unsigned long long)b & 0xfffffffffffffull;
  if (E) m |= 1ull << 52;
  const int s = max(E, 1) - 1075 + (7 * kND - 1) - e;  // at most 2
  const int l = min(max(s, 0), 63), r = min(max(-s, 0), 63);  // (above 2: rows of denormals, or with infinities)
  m <<= l;
  m = (m + ((1ull << r) >> 1)) >> r;
  return b < 0 ? -(long long)m : (long long)m;
}
// sum over all digits of 64 * 128^j: makes every balanced digit a plain 7-bit field
__device__ __forceinline__ constexpr unsigned long long digit_bias() {
  unsigned long long c = 0;
  for (int j = 0; j < kND; ++j) c = c * 128 + 64;
  return c;
}

__device__ __forceinline__ unsigned smem_addr(const void *p) {
  return static_cast<unsigned>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void cp_async8(void *dst, const void *src, bool valid) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(smem_addr(dst)), "l"(src), "r"(valid ? 8 : 0)
               : "memory");
}
__device__ __forceinline__ void ldmatrix4(unsigned (&r)[4], unsigned addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}
__device__ __forceinline__ void mma16816(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Largest |x| of a row or of a slice of it, as the high word, with the low words or'ed; sums: also sum |x| from
// above, every term as its leading 21 bits below the largest so far, in units of 2^(its biased exponent - 1043) and
// rounded up (integers: the FP64 pipe would take longer than the loads)
struct RowPart {
  unsigned hi, lo;
  unsigned long long sum;
  __device__ __forceinline__ void raise(unsigned h) {
    const unsigned d = (h >> 20) - (hi >> 20);
    if (h > hi && d) sum = (d > 63 ? 0 : sum >> d) + 1;
    hi = max(hi, h);
  }
  // eight values; zeros count for next to nothing, denormals as if normal
  template <bool SUMS>
  __device__ __forceinline__ void take(const double (&x)[8]) {
    unsigned h[8], m = hi;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      h[i] = (unsigned)__double2hiint(x[i]) & 0x7fffffffu;
      lo |= (unsigned)__double2loint(x[i]);
      m = max(m, h[i]);
    }
    if (SUMS) {
      raise(m);
      unsigned t = 8;
#pragma unroll
      for (int i = 0; i < 8; ++i) t += ((h[i] & 0xfffffu) | 0x100000u) >> min((m >> 20) - (h[i] >> 20), 31u);
      sum += t;
    }
    hi = m;
  }
  __device__ __forceinline__ void add(RowPart o) {
    const unsigned h = max(hi, o.hi);
    raise(h);
    o.raise(h);
    lo |= o.lo;
    sum += o.sum;
  }
  // smallest e with |x| < 2^e (0 for a row of zeros, -1021 for denormals), and sum |x| / 2^e
  __device__ __forceinline__ void store(int *ex, float *rsum) const {
    const bool zero = (hi | lo) == 0;
    *ex = hi >= 0x7ff00000u ? kBadExp : zero ? 0 : max((int)(hi >> 20), 1) - 1022;
    if (rsum) *rsum = zero ? 0.f : fmaxf(0.5f, (float)sum * 0x1p-21f);
  }
};
// how the rows of an operand are read: contiguous ones by a CTA or a warp each, those across the memory 32 by a CTA
enum RowMode { kRowCta, kRowWarp, kRowAcross };
constexpr int kSliceRow = 8192;   // k per CTA when rows are cut: contiguous ones
constexpr int kSliceAcross = 512;  // and those across the memory

// Exponents of the rows of op(A) and the columns of op(B): the smallest e with |x| < 2^e over the row,
// kBadExp when a value is not finite; with CHECK also sum |x| / 2^e from above, 0 for a row of zeros.  Rows that
// are contiguous in k take one CTA each, eight short or many ones share one; rows that lie across the memory (k
// strides by ld) go 32 to a CTA, 8 k at a time, coalesced over the rows.  Few long rows are cut into sa (sb) slices of k,
// whose parts combine_rows adds: with one CTA per 32 columns, 64 x 40 x 120000 (N N) took 3.6 ms a call, 0.93 as a
// tiled FP64 product and 0.31 now, 8 x 64 x 6859 133 us, 115 and 54; as one CTA per row of one element 33 x 100000 x
// 1 (N T) 218 us, now 192.
template <bool CHECK>
__global__ void __launch_bounds__(256) row_exponents(int M, int N, int K, RowMode a_mode, const double *__restrict__ A,
                                                     int lda, RowMode b_mode, const double *__restrict__ B, int ldb,
                                                     int nblk_a, int sa, int sb, int *__restrict__ ex,
                                                     float *__restrict__ rsum, RowPart *__restrict__ parts) {
  __shared__ RowPart red[8][32];
  const bool isb = (int)blockIdx.x >= nblk_a;
  const int ns = isb ? sb : sa, idx = isb ? blockIdx.x - nblk_a : blockIdx.x;
  int blk = idx, slice = 0, kbeg = 0, kend = K;
  if (ns > 1) {
    blk = idx / ns;
    slice = idx - blk * ns;
    kbeg = (int)((long)K * slice / ns);
    kend = (int)((long)K * (slice + 1) / ns);
  }
  const RowMode mode = isb ? b_mode : a_mode;
  const double *X = isb ? B : A;
  const int ld = isb ? ldb : lda, rows = isb ? N : M, out = isb ? M : 0;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  RowPart p{0, 0, 0};
  // x[k stride] for k = k0, k0 + step, ... below kend, eight loads in flight
  auto scan = [&](const double *x, long stride, int k0, int step) {
    for (long k = k0; k < kend; k += 8 * step) {
      double v[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) v[i] = k + i * step < kend ? __ldg(&x[(k + i * step) * stride]) : 0.0;
      p.take<CHECK>(v);
    }
  };
  auto emit = [&](int row) {
    if (ns == 1) p.store(ex + out + row, CHECK ? rsum + out + row : nullptr);
    else parts[(isb && sa > 1 ? (long)M * sa : 0) + (long)row * ns + slice] = p;
  };
  auto over_warp = [&] {
    for (int w = 16; w > 0; w >>= 1) {
      RowPart o;
      o.hi = __shfl_xor_sync(0xffffffffu, p.hi, w);
      o.lo = __shfl_xor_sync(0xffffffffu, p.lo, w);
      o.sum = CHECK ? __shfl_xor_sync(0xffffffffu, p.sum, w) : 0;
      p.add(o);
    }
  };
  if (mode == kRowAcross) {
    const int row = blk * 32 + lane;
    if (row < rows) scan(X + row, ld, kbeg + warp, 8);
    red[warp][lane] = p;
    __syncthreads();
    if (warp == 0 && row < rows) {
      for (int w = 1; w < 8; ++w) p.add(red[w][lane]);
      emit(row);
    }
  } else if (mode == kRowWarp) {
    const int row = blk * 8 + warp;
    if (row >= rows) return;
    scan(X + (long)row * ld, 1, lane, 32);
    over_warp();
    if (lane == 0) emit(row);
  } else {
    scan(X + (long)blk * ld, 1, kbeg + threadIdx.x, 256);
    over_warp();
    if (lane == 0) red[0][warp] = p;
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int w = 1; w < 8; ++w) p.add(red[0][w]);
      emit(blk);
    }
  }
}

// the slices of the rows that were cut: one thread per row
__global__ void __launch_bounds__(256) combine_rows(int M, int N, int sa, int sb, const RowPart *__restrict__ parts,
                                                    int *__restrict__ ex, float *__restrict__ rsum) {
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i >= M + N) return;
  const int ns = i < M ? sa : sb, row = i < M ? i : i - M;
  if (ns == 1) return;
  parts += (i >= M && sa > 1 ? (long)M * sa : 0) + (long)row * ns;
  RowPart p = parts[0];
#pragma unroll 8
  for (int s = 1; s < ns; ++s) p.add(parts[s]);
  p.store(ex + i, rsum ? rsum + i : nullptr);
}

// Whether an output needs the FP64 sum: a row or column is not finite, or the bound above exceeds half of an FP64
// sum's.  S is overestimated by less than a tenth plus 2^-13 (sA + sB) (the digits left out), so an output that
// passes does meet it; the other half is for the roundings of up to K/64 slices, alpha and beta.
struct Bound {
  float c0, c1;  // S >= c0 + c1 (sA + sB)
  explicit Bound(int K) {
    const double per = 1.1 / (0.5 * K + 4.0);
    c0 = (float)(0.006 * K * per);
    c1 = (float)(0.125 * per + 1.25e-4);
  }
  __device__ __forceinline__ bool weak(int ea, int eb, float sa, float sb, float S) const {
    if (ea == kBadExp || eb == kBadExp) return true;
    return sa != 0.f && sb != 0.f && !(S >= c0 + c1 * (sa + sb));
  }
};
// sum_k a[k sa] b[k sb] by a warp, the result in every lane
__device__ __forceinline__ double warp_dot(const double *__restrict__ a, long sa, const double *__restrict__ b, long sb,
                                           int K) {
  double s = 0.0;
#pragma unroll 8
  for (int k = threadIdx.x & 31; k < K; k += 32) s = fma(__ldg(a + k * sa), __ldg(b + k * sb), s);
  for (int w = 16; w > 0; w >>= 1) s += __shfl_xor_sync(0xffffffffu, s, w);
  return s;
}

template <bool CHECK>
constexpr size_t digit_smem() {
  constexpr int rows = 16 * kMaxStrips<CHECK>;
  return (size_t)2 * rows * kRawStride * 8 + (size_t)2 * kND * rows * kDigStride * 2 +
         (size_t)kWarps * 32 * 8 * 16 + (CHECK ? (size_t)kWarps * 32 * 8 * 4 : 0) + rows * 12;
}

// One CTA: SM x SN warps (at most 16), each a 16 x 16 block of C over k in its K slice; the SM strips of
// A and SN strips of B (16 rows each) are staged as FP64 by cp.async, rewritten as digits by all threads
// and multiplied from the digit planes.  Two buffers of each: in every step the next chunk is rewritten
// and this one multiplied between the same two barriers, the even warps rewriting first and the odd ones
// multiplying first, so that rewriting (FP64 and integer pipes) and products (tensor pipe) overlap.
// 512 x 128 x 6859 takes 166 us; with the rewriting left out 136, with the products left out 115, and the
// tensor pipe alone (86 mma.sync of two clocks per warp and 16 k) would take 69: with four warps per
// scheduler and a barrier per 16 k, neither phase fills its pipe.  Strips past the end of C skip their
// products.
template <bool TA, bool TB, bool CHECK>
__global__ void __launch_bounds__(kWarps * 32, 1)
    digit_gemm_kernel(int M, int N, int K, int kslice, int SM, int SN, const double *__restrict__ A, int lda,
                      const double *__restrict__ B, int ldb, const int *__restrict__ ex,
                      const float *__restrict__ rsum, Bound bound, double alpha, double beta, double *__restrict__ C,
                      int ldc, double *__restrict__ part, float *__restrict__ part_s) {
  constexpr int kRows = 16 * kMaxStrips<CHECK>;
  extern __shared__ __align__(16) unsigned char smem[];
  double *raw = reinterpret_cast<double *>(smem);                                  // [2][rows][kRawStride]
  __nv_bfloat16 *dig = reinterpret_cast<__nv_bfloat16 *>(raw + 2 * kRows * kRawStride);  // [2][kND][rows][kDigStride]
  longlong2 *sums = reinterpret_cast<longlong2 *>(dig + (size_t)2 * kND * kRows * kDigStride);  // [8][512]
  float4 *mags = reinterpret_cast<float4 *>(sums + kWarps * 32 * 8);                       // [2][512] (CHECK): S
  double *rscale = reinterpret_cast<double *>(mags + (CHECK ? 2 * kWarps * 32 : 0));
  int *rexp = reinterpret_cast<int *>(rscale + kRows);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rows_a = 16 * SM, rows = 16 * (SM + SN);
  const int m0 = blockIdx.y * rows_a, n0 = blockIdx.x * 16 * SN;
  const int kbeg = blockIdx.z * kslice, kend = min(K, kbeg + kslice);
  __shared__ int tiny, nweak;
  if (tid == 0) tiny = nweak = 0;
  __syncthreads();
  for (int r = tid; r < rows; r += blockDim.x) {
    const bool a = r < rows_a;
    const int g = a ? m0 + r : n0 + r - rows_a;
    int e = 0;
    if (g < (a ? M : N)) e = ex[a ? g : M + g];
    rexp[r] = e = e == kBadExp ? 0 : e;
    // 2^(kBits - e), rows of very small numbers (where that could overflow) converted by to_fixed
    if (e > -900) rscale[r] = __longlong_as_double((long long)(1023 + 7 * kND - 1 - e) << 52);
    else atomicOr(&tiny, 1);
  }
  // 8-byte copies of 32-row groups of each operand, consecutive threads along its contiguous direction: a
  // thread keeps its k and its row within the group, so an address is one pointer plus a stride
  auto load_part = [&](const double *X, bool across, int ld, int x0, int rows_x, int n_x, int row_off, int k0, int buf) {
    const int r0 = across ? lane : tid / kKC, k = across ? warp : tid % kKC;
    const bool kok = k0 + k < kend;
    const double *src = X + (across ? (long)(k0 + k) * ld + x0 + r0 : (long)(x0 + r0) * ld + k0 + k);
    const long step = across ? 32 : 32L * ld;
    double *dst = raw + (buf * kRows + row_off + r0) * kRawStride + k;
    for (int r = r0; r < rows_x; r += 32) {
      const bool ok = kok && x0 + r < n_x;
      cp_async8(dst, ok ? src : X, ok);
      src += step;
      dst += 32 * kRawStride;
    }
  };
  auto load = [&](int k0, int buf) {
    load_part(A, TA, lda, m0, rows_a, M, 0, k0, buf);
    load_part(B, !TB, ldb, n0, rows - rows_a, N, rows_a, k0, buf);
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  const int wm = warp / SN, wn = warp - wm * SN;
  const bool active = wm < SM && m0 + 16 * wm < M && n0 + 16 * wn < N;
  const unsigned a_addr = smem_addr(dig + (16 * wm + (lane & 15)) * kDigStride + (lane >> 4) * 8);
  const unsigned b_addr =
      smem_addr(dig + (rows_a + 16 * wn + ((lane >> 4) << 3) + (lane & 7)) * kDigStride + ((lane >> 3) & 1) * 8);
  constexpr unsigned kPlane = kRows * kDigStride * 2;
  constexpr int NG = kND + 1;  // digit-pair groups s + t = 0 .. kND
  float acc[NG][2][4];
#pragma unroll
  for (int g = 0; g < NG; ++g)
#pragma unroll
    for (int t = 0; t < 2; ++t)
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[g][t][i] = 0.f;
#pragma unroll
  for (int o = 0; o < 8; ++o) sums[o * (kWarps * 32) + tid] = make_longlong2(0, 0);
  if constexpr (CHECK) mags[tid] = mags[kWarps * 32 + tid] = make_float4(0.f, 0.f, 0.f, 0.f);
  constexpr unsigned kBuffer = kND * kPlane;
  // FP64 -> digits, two k per thread and step
  auto rewrite = [&](int buf) {
    for (int i = tid; i < rows * (kKC / 2); i += kWarps * 32) {
      const int r = i / (kKC / 2), kp = i % (kKC / 2);
      const double2 x = *reinterpret_cast<const double2 *>(&raw[(buf * kRows + r) * kRawStride + 2 * kp]);
      unsigned long long y0, y1;
      if (!tiny) {
        // the scaling is exact and the conversion rounds to nearest: the FP64 pipe is free here
        const double sc = rscale[r];
        y0 = (unsigned long long)__double2ll_rn(x.x * sc) + digit_bias();
        y1 = (unsigned long long)__double2ll_rn(x.y * sc) + digit_bias();
      } else {
        y0 = (unsigned long long)to_fixed(x.x, rexp[r]) + digit_bias();
        y1 = (unsigned long long)to_fixed(x.y, rexp[r]) + digit_bias();
      }
      unsigned *d = reinterpret_cast<unsigned *>(dig + (size_t)buf * (kBuffer / 2) + r * kDigStride + 2 * kp);
#pragma unroll
      for (int s = 0; s < kND; ++s) {
        const int sh = 7 * (kND - 1 - s);
        // the leading field reaches 128; a 7-bit field u next to the BF16 bits of 128 reads 128 + u
        const unsigned msk = s == 0 ? 0xffu : 0x7fu;
        const unsigned hi = sh >= 16 ? (unsigned)(y1 >> (sh >= 16 ? sh - 16 : 0)) : (unsigned)(y1 << (sh < 16 ? 16 - sh : 0));
        const unsigned u = ((unsigned)(y0 >> sh) & msk) | 0x43004300u | (hi & (msk << 16));
        __nv_bfloat162 w = __hsub2(*reinterpret_cast<const __nv_bfloat162 *>(&u), __float2bfloat162_rn(192.f));
        d[s * (kPlane / 4)] = *reinterpret_cast<const unsigned *>(&w);
      }
    }
  };
  auto multiply = [&](int buf) {
    unsigned a[kND][4];
#pragma unroll
    for (int s = 0; s < kND; ++s) ldmatrix4(a[s], a_addr + buf * kBuffer + s * kPlane);
#pragma unroll
    for (int t = 0; t < kND; ++t) {
      unsigned b[4];
      ldmatrix4(b, b_addr + buf * kBuffer + t * kPlane);
#pragma unroll
      for (int s = 0; s < kND && s + t < NG; ++s) {
        mma16816(acc[s + t][0], a[s], b[0], b[1]);
        mma16816(acc[s + t][1], a[s], b[2], b[3]);
      }
    }
    if constexpr (CHECK) {
      // |x| as BF16 from the first two digits, in units of the leading one
      auto magnitude = [](unsigned (&r)[4], unsigned addr) {
        unsigned d[4];
        ldmatrix4(r, addr);
        ldmatrix4(d, addr + kPlane);
        const __nv_bfloat162 w = __float2bfloat162_rn(0.0078125f);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const __nv_bfloat162 x = __hfma2(*reinterpret_cast<const __nv_bfloat162 *>(&d[i]), w,
                                           *reinterpret_cast<const __nv_bfloat162 *>(&r[i]));
          r[i] = *reinterpret_cast<const unsigned *>(&x) & 0x7fff7fffu;
        }
      };
      unsigned am[4], bm[4];
      magnitude(am, a_addr + buf * kBuffer);
      magnitude(bm, b_addr + buf * kBuffer);
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        float4 &m = mags[t * (kWarps * 32) + tid];
        float d[4] = {m.x, m.y, m.z, m.w};
        mma16816(d, am, bm[2 * t], bm[2 * t + 1]);
        m = make_float4(d[0], d[1], d[2], d[3]);
      }
    }
  };
  const int nch = (kend - kbeg + kKC - 1) / kKC;
  load(kbeg, 0);
  if (nch > 1) load(kbeg + kKC, 1);
  if (nch > 1) asm volatile("cp.async.wait_group 1;" ::: "memory");
  else asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  rewrite(0);
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  int held = 0;
  for (int c = 0; c < nch; ++c) {
    // digits of chunk c and the FP64 rows of chunk c + 1 are in place, everything else is free
    if (c + 2 < nch) load(kbeg + (c + 2) * kKC, c & 1);
#pragma unroll 1
    for (int half = 0; half < 2; ++half) {
      if (half == (warp & 1)) {
        if (c + 1 < nch) rewrite((c + 1) & 1);
      } else if (active) {
        multiply(c & 1);
      }
    }
    if (active && (++held == kFlush || c + 1 == nch)) {
      held = 0;
#pragma unroll
      for (int t = 0; t < 2; ++t)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          int v[NG];
#pragma unroll
          for (int g = 0; g < NG; ++g) {
            v[g] = __float_as_int(acc[g][t][i] + 12582912.f) - 0x4B400000;
            acc[g][t][i] = 0.f;
          }
          longlong2 &s = sums[(t * 4 + i) * (kWarps * 32) + tid];
          longlong2 x = s;
          x.x += (((long long)v[0] * 128 + v[1]) * 128 + v[2]) * 128 + v[3];
          x.y += ((((long long)v[4] * 128 + v[5]) * 128 + v[6]) * 128 + v[7]) * 128 + v[8];
          s = x;
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
  }
  if constexpr (!CHECK)
    if (!active) return;
  if (part) part += (long)blockIdx.z * M * N;
  if (CHECK && part) part_s += (long)blockIdx.z * M * N;
  int *list = reinterpret_cast<int *>(raw);  // (CHECK) outputs of the tile to be summed in FP64
#pragma unroll
  for (int t = 0; t < 2; ++t)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (CHECK && !active) continue;
      const int m = m0 + 16 * wm + (lane >> 2) + (i >> 1) * 8;
      const int n = n0 + 16 * wn + t * 8 + (lane & 3) * 2 + (i & 1);
      if (m >= M || n >= N) continue;
      const int ea = ex[m], eb = ex[M + n];
      double v;
      if (!CHECK && (ea == kBadExp || eb == kBadExp)) {
        // infinities and NaN follow the plain FP64 sum
        v = 0.0;
        for (int k = kbeg; k < kend; ++k)
          v = fma(TA ? A[(long)k * lda + m] : A[(long)m * lda + k], TB ? B[(long)n * ldb + k] : B[(long)k * ldb + n], v);
      } else {
        // group g weighs 128^(14 - g) of 2^(ea + eb - 110)
        const longlong2 s = sums[(t * 4 + i) * (kWarps * 32) + tid];
        v = ldexp(fma((double)s.x, 34359738368.0, (double)s.y), ea + eb - 110 + 42);
      }
      float S = 0.f;
      if constexpr (CHECK) {
        const float4 q = mags[t * (kWarps * 32) + tid];
        S = (i == 0 ? q.x : i == 1 ? q.y : i == 2 ? q.z : q.w) * 0x1p-12f;  // leading digits weigh 2^-6
      }
      if (part) {
        part[(long)m * N + n] = v;
        if (CHECK) part_s[(long)m * N + n] = S;
      } else if (CHECK && bound.weak(ea, eb, rsum[m], rsum[M + n], S)) {
        list[atomicAdd(&nweak, 1)] = (m - m0) << 16 | (n - n0);
      } else {
        double *c = C + (long)m * ldc + n;
        *c = beta == 0.0 ? alpha * v : alpha * v + beta * (*c);
      }
    }
  if constexpr (CHECK) {
    if (part) return;
    __syncthreads();
    if (nweak > kFewWeak) {
      // rows and columns of the tile through shared memory, up to eight listed outputs per thread
      double *stage = raw + kWarps * 32 * 8 / 2;  // after the list: [rows][kStageK + 1]
      auto fill = [&](const double *X, bool across, int ld, int x0, int rows_x, int n_x, double *dst, int k0) {
        for (int e = tid; e < rows_x * kStageK; e += kWarps * 32) {
          const int r = across ? e % rows_x : e / kStageK, k = across ? e / rows_x : e % kStageK;
          const bool ok = x0 + r < n_x && k0 + k < K;
          dst[r * (kStageK + 1) + k] =
              ok ? __ldg(X + (across ? (long)(k0 + k) * ld + x0 + r : (long)(x0 + r) * ld + k0 + k)) : 0.0;
        }
      };
      double v[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] = 0.0;
      for (int k0 = 0; k0 < K; k0 += kStageK) {
        fill(A, TA, lda, m0, rows_a, M, stage, k0);
        fill(B, !TB, ldb, n0, rows - rows_a, N, stage + rows_a * (kStageK + 1), k0);
        __syncthreads();
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int q = tid + j * kWarps * 32;
          if (q < nweak) {
            const double *x = stage + (list[q] >> 16) * (kStageK + 1);
            const double *y = stage + (rows_a + (list[q] & 0xffff)) * (kStageK + 1);
#pragma unroll 8
            for (int k = 0; k < kStageK; ++k) v[j] = fma(x[k], y[k], v[j]);
          }
        }
        __syncthreads();
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int q = tid + j * kWarps * 32;
        if (q < nweak) {
          double *c = C + (long)(m0 + (list[q] >> 16)) * ldc + n0 + (list[q] & 0xffff);
          *c = beta == 0.0 ? alpha * v[j] : alpha * v[j] + beta * (*c);
        }
      }
      return;
    }
    for (int q = warp; q < nweak; q += kWarps) {
      const int m = m0 + (list[q] >> 16), n = n0 + (list[q] & 0xffff);
      const double v = warp_dot(TA ? A + m : A + (long)m * lda, TA ? lda : 1, TB ? B + (long)n * ldb : B + n,
                                TB ? 1 : ldb, K);
      if (lane == 0) {
        double *c = C + (long)m * ldc + n;
        *c = beta == 0.0 ? alpha * v : alpha * v + beta * (*c);
      }
    }
  }
}

// op(A) and op(B) of a CHECK launch as strided rows: element (m, k) at A[m am + k ak], (k, n) at B[n bn + k bk]
struct Operands {
  const double *A, *B;
  long am, ak, bn, bk;
  const int *ex;
  const float *rsum, *part_s;
  int K;
  Bound bound;
};

// C = alpha sum_z part[z] + beta C: 32 outputs per CTA, the slices dealt to eight warps and their sums added
// in order (as one thread per output, 44 x 216 outputs of 30 slices took 9 us, now 3).  CHECK: S is added
// likewise, and the weak outputs are dealt to the warps for an FP64 sum.
template <bool CHECK>
__global__ void __launch_bounds__(256) digit_reduce(int M, int N, int nsplit, const double *__restrict__ part,
                                                    double alpha, double beta, double *__restrict__ C, int ldc,
                                                    Operands op) {
  __shared__ double red[8][33];
  __shared__ float sred[CHECK ? 8 : 1][33];
  __shared__ unsigned todo;
  const long total = (long)M * N;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long i = blockIdx.x * 32L + lane;
  double s = 0;
  if (i < total)
#pragma unroll 4
    for (int z = warp; z < nsplit; z += 8) s += __ldg(&part[(long)z * total + i]);
  red[warp][lane] = s;
  float S = 0.f;
  if constexpr (CHECK) {
    if (i < total)
#pragma unroll 4
      for (int z = warp; z < nsplit; z += 8) S += __ldg(&op.part_s[(long)z * total + i]);
    sred[warp][lane] = S;
  }
  __syncthreads();
  if (warp == 0) {
    bool again = false;
    if (CHECK && i < total) {
      for (int w = 1; w < 8; ++w) S += sred[w][lane];
      const int m = (int)(i / N), n = M + (int)(i % N);
      again = op.bound.weak(op.ex[m], op.ex[n], op.rsum[m], op.rsum[n], S);
    }
    if (CHECK) {
      const unsigned all = __ballot_sync(0xffffffffu, again);
      if (lane == 0) todo = all;
    }
    if (i < total && !again) {
      for (int w = 1; w < 8; ++w) s += red[w][lane];
      double *c = C + (i / N) * ldc + (i % N);
      *c = beta == 0.0 ? alpha * s : alpha * s + beta * (*c);
    }
  }
  if constexpr (CHECK) {
    __syncthreads();
    int q = 0;
    for (unsigned left = todo; left; left &= left - 1, ++q) {
      if ((q & 7) != warp) continue;
      const long o = blockIdx.x * 32L + __ffs(left) - 1, m = o / N, n = o % N;
      const double v = warp_dot(op.A + m * op.am, op.ak, op.B + n * op.bn, op.bk, op.K);
      if (lane == 0) {
        double *c = C + m * ldc + n;
        *c = beta == 0.0 ? alpha * v : alpha * v + beta * (*c);
      }
    }
  }
}

// Strips per CTA and K slices: the fewest clocks by a model of one CTA per SM, a chunk of 16 k costing the
// larger of its rewriting (240 clocks per strip) and its products (172 per active warp) plus 500, a CTA 8000 more.
struct Shape {
  int sm, sn, kslice, nsplit;
};
Shape choose(int M, int N, int K, size_t part_cap, int strips) {
  static const int opts[][2] = {{4, 4}, {5, 3}, {3, 5}, {2, 7}, {7, 2}, {6, 2}, {2, 6}, {3, 3}, {2, 4}, {4, 2}, {2, 2},
                                {1, 8}, {8, 1}, {1, 7}, {7, 1}, {1, 4}, {4, 1}, {1, 1}};
  const int ms = (M + 15) / 16, ns = (N + 15) / 16;
  Shape best{4, 4, K, 1};
  double bc = 1e300;
  for (auto &o : opts) {
    const int sm = o[0], sn = o[1];
    if (sm > ms + 1 || sn > ns + 1 || sm + sn > strips) continue;
    if (sm + sn == 8 && std::max(sm, sn) == 7 && strips > 8) continue;  // in the place of 1 + 8
    const long tiles = (long)((ms + sm - 1) / sm) * ((ns + sn - 1) / sn);
    const double load = std::max(240.0 * (sm + sn), 172.0 * std::min(sm, ms) * std::min(sn, ns)) + 500.0;
    // a slice of at most kMaxSlice k keeps the 64-bit sums in range (2^50 per 128 k)
    const int mins = (K + kMaxSlice - 1) / kMaxSlice;
    const int maxs = (int)std::max(mins, std::min(K / 64, 128));
    for (int s = mins; s <= maxs; ++s) {
      if (s > mins && (size_t)s * M * N > part_cap) break;
      const int chunks = (K + kKC - 1) / kKC;
      const int per = (chunks + s - 1) / s;
      const int sr = (chunks + per - 1) / per;
      if (sr != s) continue;
      const double waves = (double)((tiles * s + 151) / 152);
      const double cost = waves * (per * load + 8000.0) + (s > 1 ? 4000.0 + 0.01 * s * M * N / 152.0 * 8 : 0.0);
      if (cost < bc) {
        bc = cost;
        best = {sm, sn, per * kKC, sr};
      }
    }
  }
  return best;
}

template <bool TA, bool TB, bool CHECK>
void go(dim3 grid, cudaStream_t s, int M, int N, int K, const Shape &h, const double *A, int lda, const double *B,
        int ldb, const int *ex, const float *rsum, double alpha, double beta, double *C, int ldc, double *part,
        float *part_s) {
  constexpr size_t smem = digit_smem<CHECK>();
  auto kernel = digit_gemm_kernel<TA, TB, CHECK>;
  // the limit is an attribute of the function on a device, the same at every launch: set once (a microsecond a call)
  static std::atomic<unsigned long long> set{0};
  int dev = 0;
  BSE_CUDA(cudaGetDevice(&dev));
  if (dev >= 64 || !(set.load() >> dev & 1)) {
    BSE_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    if (dev < 64) set.fetch_or(1ull << dev);
  }
  kernel<<<grid, kWarps * 32, smem, s>>>(M, N, K, h.kslice, h.sm, h.sn, A, lda, B, ldb, ex, rsum, Bound(K), alpha, beta,
                                         C, ldc, part, part_s);
  BSE_CHECK_LAUNCH();
}

template <bool CHECK>
void run(char ta, char tb, int M, int N, int K, double alpha, const double *A, int lda, const double *B, int ldb,
         double beta, double *C, int ldc, cudaStream_t s, DevBuf<double> &scratch, bool fixed, int split_pct) {
  // exponents (and the row sums of CHECK, at one float each) in doubles, ahead of the partial sums
  const size_t nex = CHECK ? (size_t)M + N : ((size_t)M + N + 1) / 2;
  const size_t cap = fixed ? (scratch.n > nex ? scratch.n - nex : 0) : (size_t)1 << 26;
  Shape h = choose(M, N, K, cap, kMaxStrips<CHECK>);
  if (split_pct != 100) {
    // the autotuner's variation of the number of K slices
    const int chunks = (K + kKC - 1) / kKC;
    int ns = std::max(1, std::min(chunks, h.nsplit * split_pct / 100));
    if (ns > 1) ns = (int)std::max<size_t>(1, std::min<size_t>(ns, cap / ((size_t)M * N)));
    ns = std::max(ns, (K + kMaxSlice - 1) / kMaxSlice);
    const int per = (chunks + ns - 1) / ns;
    h.kslice = per * kKC;
    h.nsplit = (chunks + per - 1) / per;
  }
  if ((M + 16 * h.sm - 1) / (16 * h.sm) > 65535) {
    // row tiles lie along y, which ends there (with 32 or 48 rows at two to three million): in two halves.
    // Numbering all tiles along x made m0 and n0 the results of a division and every product 8% slower.
    const int m = M / 2;
    run<CHECK>(ta, tb, m, N, K, alpha, A, lda, B, ldb, beta, C, ldc, s, scratch, fixed, split_pct);
    run<CHECK>(ta, tb, M - m, N, K, alpha, A + (ta == 'T' ? m : (long)m * lda), lda, B, ldb, beta,
                   C + (long)m * ldc, ldc, s, scratch, fixed, split_pct);
    return;
  }
  const long total = (long)M * N;
  const size_t npart = h.nsplit > 1 ? (size_t)h.nsplit * total : 0;
  // CTAs of the exponent pass, and slices of k where they would leave the chip empty; the slices' parts lie where
  // the partial sums come later
  const bool TA = ta == 'T', TB = tb == 'T';
  // (a warp per row of 600 entries: 4096 of them 20 -> 6 us)
  auto mode = [&](bool across, int rows) {
    return across ? kRowAcross : K <= 256 || (K <= 4096 && rows >= 1216) ? kRowWarp : kRowCta;
  };
  auto blocks = [](RowMode m, int rows) { return m == kRowAcross ? (rows + 31) / 32 : m == kRowWarp ? (rows + 7) / 8 : rows; };
  auto slices = [&](RowMode m, int nblk) {
    if (m == kRowWarp) return 1;
    return std::max(1, std::min(K / (m == kRowAcross ? kSliceAcross : kSliceRow), 1216 / nblk));
  };
  const RowMode am = mode(TA, M), bm = mode(!TB, N);
  const int ba = blocks(am, M), bb = blocks(bm, N);
  int sa = slices(am, ba), sb = slices(bm, bb);
  size_t nrow = ((sa > 1 ? (size_t)M * sa : 0) + (sb > 1 ? (size_t)N * sb : 0)) * sizeof(RowPart) / sizeof(double);
  if (fixed && nrow > cap) sa = sb = 1, nrow = 0;
  if (!fixed) scratch.alloc(nex + std::max(nrow, npart + (CHECK ? (npart + 1) / 2 : 0)));
  int *ex = reinterpret_cast<int *>(scratch.get());
  float *rsum = CHECK ? reinterpret_cast<float *>(ex + M + N) : nullptr;
  double *part = npart ? scratch.get() + nex : nullptr;
  float *part_s = CHECK && npart ? reinterpret_cast<float *>(part + npart) : nullptr;
  RowPart *parts = nrow ? reinterpret_cast<RowPart *>(scratch.get() + nex) : nullptr;
  row_exponents<CHECK><<<ba * sa + bb * sb, 256, 0, s>>>(M, N, K, am, A, lda, bm, B, ldb, ba * sa, sa, sb, ex, rsum,
                                                         parts);
  BSE_CHECK_LAUNCH();
  if (parts) {
    combine_rows<<<(M + N + 255) / 256, 256, 0, s>>>(M, N, sa, sb, parts, ex, rsum);
    BSE_CHECK_LAUNCH();
  }
  const dim3 grid((unsigned)((N + 16 * h.sn - 1) / (16 * h.sn)), (unsigned)((M + 16 * h.sm - 1) / (16 * h.sm)),
                  (unsigned)h.nsplit);
  auto launch = [&](auto a, auto b) {
    go<decltype(a)::value, decltype(b)::value, CHECK>(grid, s, M, N, K, h, A, lda, B, ldb, ex, rsum, alpha, beta, C,
                                                          ldc, part, part_s);
  };
  if (!TA && !TB) launch(std::false_type(), std::false_type());
  else if (!TA && TB) launch(std::false_type(), std::true_type());
  else if (TA && !TB) launch(std::true_type(), std::false_type());
  else launch(std::true_type(), std::true_type());
  if (part) {
    const Operands op{A, B, TA ? 1 : lda, TA ? lda : 1, TB ? ldb : 1, TB ? 1 : ldb, ex, rsum, part_s, K, Bound(K)};
    digit_reduce<CHECK><<<(unsigned)((total + 31) / 32), 256, 0, s>>>(M, N, h.nsplit, part, alpha, beta, C, ldc, op);
    BSE_CHECK_LAUNCH();
  }
}

}  // namespace

size_t digit_scratch(int M, int N, int K) {
  const size_t slices = ((size_t)K + kMaxSlice - 1) / kMaxSlice;
  return ((size_t)M + N + 1) / 2 + (slices > 1 ? slices * M * N : 0);
}

void splitk_sum(int M, int N, int nsplit, const double *part, double alpha, double beta, double *C, int ldc,
                cudaStream_t s) {
  digit_reduce<false><<<(unsigned)(((long)M * N + 31) / 32), 256, 0, s>>>(M, N, nsplit, part, alpha, beta, C, ldc,
                                                                             Operands{nullptr, nullptr, 0, 0, 0, 0, nullptr,
                                                                                      nullptr, nullptr, 0, Bound(0)});
  BSE_CHECK_LAUNCH();
}

void digit_gemm(char ta, char tb, int M, int N, int K, double alpha, const double *A, int lda,
                const double *B, int ldb, double beta, double *C, int ldc, cudaStream_t s, DevBuf<double> &scratch,
                bool fixed, int split_pct, bool entrywise) {
  if (entrywise) run<true>(ta, tb, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, s, scratch, fixed, split_pct);
  else run<false>(ta, tb, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, s, scratch, fixed, split_pct);
}

}  // namespace bse
