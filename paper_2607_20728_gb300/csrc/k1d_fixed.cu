// FP64 K1d contraction fused with the grid terms of the Liouville operator (Eq. 2),
//   Y_{b,v}(r) = V(r) a_{b,v}(r) + 2 v_H,b(r) phi_v(r) - sum_v' tau_{v'v}(r) a_{b,v'}(r),
// with the sum over v' in integers.  GB300 issues 2 FP64 multiply-adds per clock and SM but 32 of its
// 32 x 32 + 64 bit integer ones, so the contraction is bound by the FP64 pipe as FP64 (10.4 ms for one
// vector of the 63-well cell, N_occ = 128, 72^3) and by the tau stream as fixed point.
//
// tau is stored once per unordered pair as a 57-bit fixed-point number relative to the power of two
// above max_pairs |tau(r)| of its point r, as two signed limbs of 27 bits below: t = th 2^27 + tl,
// |th| <= 2^29, |tl| <= 2^26 (8 bytes, like the double it replaces).  a_v(r) is rounded the same way to
// 53 + s bits below max_v |a_v(r)|, so the three products th ah, th al + tl ah (tl al is a quarter of the last
// unit at most) are integers; s is a property of the point, as large as the 64-bit sums allow: with
// C = max_v sum_v' |tau_v'v|, |sum| <= C max|a|, and C is far below N_occ max|tau| where the diagonal dominates.
// The sums are rounded to 2^-(55 + s) of max|tau| max|a| as they are added to Y and to FP64 once at the end.
// Error over a point's orbitals (2-norm, emulated), s = 0 and all N_occ terms at the maximum assumed -> this ->
// an FP64 sum: 128 flat 1.6e-16 -> 0.3e-16 (3.6e-16), 128 with a dominant diagonal 6.3e-16 -> 2.1e-16 (3.8e-16),
// 200 likewise 13e-16 -> 2.6e-16 (3.9e-16), orbitals of very different size 3.3e-16 -> 0.6e-16 (3.0e-16).
//
// Every tau element is read from memory once: a CTA owns 32 points (one per lane) and walks the columns
// c of 8 orbitals; column c holds blocks of 16 rows x 8 orbitals below it (one of 8 rows when c is odd)
// and its own triangle, each one contiguous chunk of the tile-major tau that arrives by a 1D bulk copy
// into a ring of 32 KB stages.  Warps 0-3 accumulate Y_c += tau^T a_I in registers over the column
// ("role A", two orbitals each), warps 4-7 add tau a_c to the rows of Y_I chunk by chunk ("role B").
// Within a column no two warps write the same rows of Y; a named barrier separates columns.  One more warp
// is the producer and runs ahead over tile boundaries.  (Warp numbers for 8 consumer warps.)  Waits are
// bounded: a consumer whose wait runs out sets the device flag and the CTA's, every warp still passes the
// same barriers up to the next tile's first one, and all leave there; hold != 0 (self-test) makes them run out.
//
// Time of one launch, FP64 kernel before -> this one (tau at the measured copy rate): N_occ = 128, 72^3: one
// vector 10.41 -> 4.87 ms (3.64), two 20.28 -> 7.82; N_occ = 63, 72^3: 2.64 -> 1.38 (0.89), two 5.13 -> 2.63;
// N_occ = 48, 36^3: 240 -> 123 us (65), two 427 -> 187; N_occ = 16, 24^3: 22.7 -> 13.5 us.  One vector is
// held by shared-memory wavefronts and the stream, two by the integer pipe (half its peak) as well.
#include <algorithm>
#include <type_traits>

#include "internal.cuh"
#include "mbarrier.cuh"

namespace bse {
namespace {

constexpr int kR = 32;            // grid points per tile (one per lane)
constexpr int kC = 8;             // orbitals per column
constexpr int kRowsPer = 16;      // rows of a full chunk
constexpr int kStageElems = kRowsPer * kC * kR;
constexpr unsigned kStageBytes = kStageElems * 8;
constexpr size_t kSmemCap = 227 * 1024;
constexpr size_t kSmemHalf = 113 * 1024;  // two CTAs per SM
constexpr int kMaxStages = 6;
constexpr int kTauBits = 56;      // of tau below its point's power of two

template <int W>
__device__ __forceinline__ void consumers_sync() {
  asm volatile("bar.sync 1, %0;" ::"n"(W * 32) : "memory");
}

// position (in pairs) of the pair (v', v), v' <= v, inside one tile
__host__ __device__ inline long fixed_slot(int vp, int v, int nocc) {
  const int c = v / kC, jj = v % kC, c8 = c * kC;
  const int bj = nocc - c8 < kC ? nocc - c8 : kC;
  const long base = (long)c8 * (c8 + 1) / 2;
  if (vp >= c8) return base + (long)c8 * bj + jj * (jj + 1) / 2 + (vp - c8);
  const int I = vp / kRowsPer;
  if (I < c / 2) return base + (long)I * kRowsPer * bj + jj * kRowsPer + vp % kRowsPer;
  return base + (long)(c / 2) * kRowsPer * bj + jj * kC + (vp - (c8 - kC));
}

// |x| < 2^e -> round(x 2^(bits - e)); 0 <= bits <= 56
__device__ __forceinline__ long long to_fixed(double x, int e, int bits) {
  const long long b = __double_as_longlong(x);
  const int E = (int)((b >> 52) & 0x7ff);
  unsigned long long m = (unsigned long long)b & 0xfffffffffffffull;
  if (E) m |= 1ull << 52;
  const int s = max(E, 1) - 1075 + bits - e;
  const int l = min(max(s, 0), 10), r = min(max(-s, 0), 63);
  m = ((m << l) + ((1ull << r) >> 1)) >> r;
  return b < 0 ? -(long long)m : (long long)m;
}
// balanced limbs: x = hi 2^27 + lo, |lo| <= 2^26
__device__ __forceinline__ int2 limbs(long long x) {
  const long long h = (x + (1 << 26)) >> 27;
  return make_int2((int)h, (int)(x - (h << 27)));
}
// exponent of the smallest power of two above the value with the high word hi (|x| < 2^e)
__device__ __forceinline__ int exp_above(unsigned hi) { return max((int)(hi >> 20), 1) - 1022; }
// 2^e as a double, NaN when the high word of the maximum says infinity or NaN
__device__ __forceinline__ double scale_of(unsigned hi, int e) {
  return (hi >> 20) >= 0x7ff ? __longlong_as_double(0x7ff8000000000000ll) : ldexp(1.0, e);
}

struct Sums {
  long long hh, hl;
};
__device__ __forceinline__ void mac(Sums &s, int2 t, int2 a) {
  s.hh += (long long)t.x * a.x;
  s.hl += (long long)t.x * a.y;
  s.hl += (long long)t.y * a.x;
}
// in units of 2^54 of (tau unit) x (a unit)
__device__ __forceinline__ long long rounded(const Sums &s) { return s.hh + ((s.hl + (1ll << 26)) >> 27); }

// pairs (rows x orbitals) of chunk k of column c: full 16-row chunks, the 8-row one of an odd column,
// the triangle
__device__ __forceinline__ int chunk_pairs(int c, int k, int bj) {
  if (k < c / 2) return kRowsPer * bj;
  if ((c & 1) && k == c / 2) return kC * bj;
  return bj * (bj + 1) / 2;
}
__device__ __forceinline__ int chunks_of(int c) { return c / 2 + (c & 1) + 1; }

template <int NB, int W>
__global__ void __launch_bounds__(W * 32 + 32, 16 / W) k1d_fixed_kernel(
    const int2 *__restrict__ tau, const double2 *__restrict__ tscale, long npairs, long nr, int nocc, int nb_total,
    int b0, int stages, const double *__restrict__ phir, const double *__restrict__ vloc,
    const double *__restrict__ Pa, const double *__restrict__ Pvh, double *__restrict__ Py, int use_vloc, int use_k1e,
    int *__restrict__ err, int hold) {
  extern __shared__ __align__(128) unsigned char smem[];
  int2 *tau_s = reinterpret_cast<int2 *>(smem);                                     // [stages][128][32]
  int2 *a_s = tau_s + (size_t)stages * kStageElems;                                 // [NB][nocc][32]
  long long *y_s = reinterpret_cast<long long *>(a_s + (size_t)NB * nocc * kR);     // [NB][nocc][32]
  unsigned *top = reinterpret_cast<unsigned *>(y_s + (size_t)NB * nocc * kR);       // [NB][32]
  unsigned long long *full = reinterpret_cast<unsigned long long *>(top + NB * kR);
  constexpr int kRole = W / 2;    // warps per role
  constexpr int kOA = kC / kRole;  // role A: orbitals per warp
  unsigned long long *empty = full + kMaxStages;
  volatile int *fail = reinterpret_cast<volatile int *>(empty + kMaxStages);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ncol = (nocc + kC - 1) / kC;
  const long ntiles = (nr + kR - 1) / kR;
  if (tid == 0) {
    for (int st = 0; st < stages; ++st) {
      mbar_init(&full[st], 1);
      mbar_init(&empty[st], W);
    }
    *fail = 0;
    fence_async_shared();
  }
  if (tid < NB * kR) top[tid] = 0;
  __syncthreads();
  if (warp == W) {
    // ---- producer ----
    if (lane == 0 && !hold) {
      long g = 0;
      int st = 0;
      unsigned round = 0;  // completed trips around the ring
      bool ok = true;
      for (long t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
        const int2 *src = tau + (size_t)t * npairs * kR;
        for (int c = 0; c < ncol && ok; ++c) {
          const int bj = min(kC, nocc - c * kC);
          for (int k = 0; k < chunks_of(c); ++k, ++g) {
            if (round > 0 && !mbar_wait(&empty[st], (round - 1) & 1)) {
              atomicExch(err, 1);
              ok = false;
              break;
            }
            const int elems = chunk_pairs(c, k, bj) * kR;
            fence_async_shared();
            mbar_expect_tx(&full[st], elems * 8);
            bulk_load(tau_s + (size_t)st * kStageElems, src, elems * 8, &full[st]);
            src += elems;
            if (++st == stages) {
              st = 0;
              ++round;
            }
          }
        }
      }
      // copies in flight land (bounded) before the CTA can exit
      for (long q = (g > stages ? g - stages : 0); q < g; ++q)
        mbar_wait(&full[q % stages], (unsigned)((q / stages) & 1));
    }
    return;
  }
  // ---- consumers ----
  // real element (b, v) at point rr of a packed grid: f = b nocc + v
  auto at = [&](int b, int v, long rr) -> long {
    const long f = (long)(b0 + b) * nocc + v;
    return 2 * ((f >> 1) * nr + rr) + (f & 1);
  };
  const bool roleA = warp < kRole;
  const int wr = warp % kRole;
  // rows warp, warp + W, ... of a at this thread's point of tile t; the first kKeep of each vector stay in
  // registers from the last column of the tile before, so that their latency overlaps the tau stream
  // (one vector; two would spill)
  constexpr int kKeep = NB == 1 ? 8 : 0;
  double x[NB][kKeep > 0 ? kKeep : 1];
  auto row = [&](int b, int v, long rr) { return b0 + b < nb_total ? __ldg(&Pa[at(b, v, rr)]) : 0.0; };
  auto point = [&](long t) { return min(t * kR + lane, nr - 1); };
  // bits of a at the tile's point: with the rows for one vector and 16 warps (4.92 -> 4.82 ms at 128 orbitals), at
  // the top of the tile otherwise (with the rows 48 orbitals take 125 and 192 us, so 124 and 186)
  constexpr bool kAhead = NB == 1 && W == 16;
  double abits = 0;
  auto fetch = [&](long t) {
    const long rr = point(t);
    if (kAhead) abits = __ldg(&tscale[rr].y);
#pragma unroll
    for (int b = 0; b < NB; ++b)
#pragma unroll
      for (int i = 0; i < kKeep; ++i) x[b][i] = warp + W * i < nocc ? row(b, warp + W * i, rr) : 0.0;
  };
  int st = 0;
  unsigned phase = 0;
  bool ok = true;
  if (blockIdx.x < ntiles) fetch(blockIdx.x);
  for (long t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const bool live = t * kR + lane < nr;
    const long rr = point(t);
    if (!kAhead) abits = __ldg(&tscale[rr].y);
    // largest |a_v| of every point, then a as limbs
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      unsigned m = 0;
#pragma unroll
      for (int i = 0; i < kKeep; ++i) m = max(m, (unsigned)__double2hiint(x[b][i]) & 0x7fffffffu);
      for (int v = warp + W * kKeep; v < nocc; v += W) m = max(m, (unsigned)__double2hiint(row(b, v, rr)) & 0x7fffffffu);
      atomicMax(&top[b * kR + lane], m);
    }
    consumers_sync<W>();  // and the previous tile's epilogue is done
    if (*fail) break;     // a give-up recorded before the barrier: all leave together
    double ascale[NB];
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      const unsigned m = top[b * kR + lane];
      const int e = exp_above(m);
      ascale[b] = scale_of(m, e);
      auto put = [&](int v, double xv) {
        a_s[((size_t)b * nocc + v) * kR + lane] = limbs(to_fixed(xv, e, (int)abits));
        y_s[((size_t)b * nocc + v) * kR + lane] = 0;
      };
#pragma unroll
      for (int i = 0; i < kKeep; ++i)
        if (warp + W * i < nocc) put(warp + W * i, x[b][i]);
      for (int v = warp + W * kKeep; v < nocc; v += W) put(v, row(b, v, rr));
    }
    consumers_sync<W>();
    if (tid < NB * kR) top[tid] = 0;  // next written after the barriers of the columns
    for (int c = 0; c < ncol; ++c) {
      const int c8 = c * kC, bj = min(kC, nocc - c8);
      int ja[kOA];  // role A's orbitals (clamped)
      Sums sa[kOA][NB];
#pragma unroll
      for (int k = 0; k < kOA; ++k) ja[k] = min(kOA * wr + k, bj - 1);
#pragma unroll
      for (int k = 0; k < kOA; ++k)
#pragma unroll
        for (int b = 0; b < NB; ++b) sa[k][b] = {0, 0};
      if (c == ncol - 1 && t + gridDim.x < ntiles) fetch(t + gridDim.x);
      const int nch = chunks_of(c);
      for (int k = 0; k < nch; ++k) {
        if (ok) {
          if (*fail) {
            ok = false;
          } else if (!mbar_wait(&full[st], phase)) {
            ok = false;
            if (lane == 0) {
              atomicExch(err, 1);
              *fail = 1;
              __threadfence_block();
            }
          }
          ok = __all_sync(0xffffffffu, ok);
        }
        const int2 *T = tau_s + (size_t)st * kStageElems + lane;
        if (++st == stages) {
          st = 0;
          phase ^= 1;
        }
        if (!ok) continue;
        unsigned long long *done = &empty[st == 0 ? stages - 1 : st - 1];
        // Y rows row0 + RB wr .. += tau a_c over the bj orbitals of the column
        auto role_b = [&](auto width, int row0) {
          constexpr int R = decltype(width)::value, RB = R / kRole;
          Sums sb[RB][NB];
#pragma unroll
          for (int q = 0; q < RB; ++q)
#pragma unroll
            for (int b = 0; b < NB; ++b) sb[q][b] = {0, 0};
          auto one = [&](int jj) {
            int2 a[NB];
#pragma unroll
            for (int b = 0; b < NB; ++b) a[b] = a_s[((size_t)b * nocc + c8 + jj) * kR + lane];
#pragma unroll
            for (int q = 0; q < RB; ++q) {
              const int2 x = T[(jj * R + RB * wr + q) * kR];
#pragma unroll
              for (int b = 0; b < NB; ++b) mac(sb[q][b], x, a[b]);
            }
          };
          if (bj == kC) {
#pragma unroll
            for (int jj = 0; jj < kC; ++jj) one(jj);
          } else {
            for (int jj = 0; jj < bj; ++jj) one(jj);
          }
#pragma unroll
          for (int q = 0; q < RB; ++q)
#pragma unroll
            for (int b = 0; b < NB; ++b)
              y_s[((size_t)b * nocc + row0 + RB * wr + q) * kR + lane] += rounded(sb[q][b]);
        };
        auto role_a = [&](auto width, int row0) {
          constexpr int R = decltype(width)::value;
#pragma unroll
          for (int m = 0; m < R; ++m) {
            int2 x[kOA];
#pragma unroll
            for (int q = 0; q < kOA; ++q) x[q] = T[(ja[q] * R + m) * kR];
#pragma unroll
            for (int b = 0; b < NB; ++b) {
              const int2 a = a_s[((size_t)b * nocc + row0 + m) * kR + lane];
#pragma unroll
              for (int q = 0; q < kOA; ++q) mac(sa[q][b], x[q], a);
            }
          }
        };
        if (k < c / 2) {
          if (roleA) role_a(std::integral_constant<int, kRowsPer>(), k * kRowsPer);
          else role_b(std::integral_constant<int, kRowsPer>(), k * kRowsPer);
        } else if ((c & 1) && k == c / 2) {
          if (roleA) role_a(std::integral_constant<int, kC>(), c8 - kC);
          else role_b(std::integral_constant<int, kC>(), c8 - kC);
        } else if (roleA) {
          // the column's own triangle, packed with the smaller index first
          for (int m = 0; m < bj; ++m) {
            int2 x[kOA];
#pragma unroll
            for (int q = 0; q < kOA; ++q)
              x[q] = T[(m <= ja[q] ? ja[q] * (ja[q] + 1) / 2 + m : m * (m + 1) / 2 + ja[q]) * kR];
#pragma unroll
            for (int b = 0; b < NB; ++b) {
              const int2 a = a_s[((size_t)b * nocc + c8 + m) * kR + lane];
#pragma unroll
              for (int q = 0; q < kOA; ++q) mac(sa[q][b], x[q], a);
            }
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(done);
      }
      if (ok && roleA) {
#pragma unroll
        for (int k = 0; k < kOA; ++k)
          if (kOA * wr + k < bj)
#pragma unroll
            for (int b = 0; b < NB; ++b)
              y_s[((size_t)b * nocc + c8 + kOA * wr + k) * kR + lane] += rounded(sa[k][b]);
      }
      consumers_sync<W>();  // the rows of column c are complete up to here for role B of later columns
    }
    if (!ok || !live) continue;
    const double ts = tscale[rr].x, V = use_vloc ? vloc[rr] : 0.0;
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      if (b0 + b >= nb_total) break;
      const double s = -ts * ascale[b];
      const double vh2 = use_k1e ? 2.0 * Pvh[2 * ((long)((b0 + b) >> 1) * nr + rr) + ((b0 + b) & 1)] : 0.0;
#pragma unroll 4
      for (int v = warp; v < nocc; v += W) {
        const long o = at(b, v, rr);
        double y = s * (double)y_s[((size_t)b * nocc + v) * kR + lane];
        if (use_vloc) y = fma(V, __ldg(&Pa[o]), y);
        if (use_k1e) y = fma(vh2, __ldg(&phir[(long)v * nr + rr]), y);
        Py[o] = y;
        const long f = (long)(b0 + b) * nocc + v;
        if ((f & 1) == 0 && f == (long)nb_total * nocc - 1) Py[o + 1] = 0;  // unused partner
      }
    }
  }
}

size_t smem_bytes(int nb, int stages, int nocc) {
  return (size_t)stages * kStageBytes + (size_t)nb * nocc * kR * 16 + (size_t)nb * kR * 4 + 2 * kMaxStages * 8 + 16;
}
// Shape of a launch for nb vectors: two CTAs of 8 consumer warps per SM, each with its own ring of two
// stages or more, when they fit (the prologue and epilogue of one then overlap the stream of the other:
// N_occ = 48 one vector 172 -> 123 us, N_occ = 63 2.01 -> 1.38 ms), else one CTA of 16 (N_occ = 128: 4.9 ms,
// with 8 warps 6.1 ms).  stages 0: nb vectors do not fit at all.
struct Shape {
  int warps, stages;
};
Shape shape_for(int nb, int nocc) {
  for (int st = 3; st >= 2; --st)
    if (smem_bytes(nb, st, nocc) <= kSmemHalf) return {8, st};
  for (int st = kMaxStages; st >= 3; --st)
    if (smem_bytes(nb, st, nocc) <= kSmemCap) return {16, st};
  return {0, 0};
}

template <int NB, int W>
void launch(const Ctx &c, const K1dFixed &t, int stages, int nb, int b0, const double *phir, const double *vloc,
            const double2 *Pa, const double2 *Pvh, double2 *Py, bool use_vloc, bool use_k1e) {
  const size_t smem = smem_bytes(NB, stages, c.nocc);
  BSE_CUDA(cudaFuncSetAttribute(k1d_fixed_kernel<NB, W>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemCap));
  int dev = 0, nsm = 0;
  BSE_CUDA(cudaGetDevice(&dev));
  BSE_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  const unsigned grid = (unsigned)std::min<long>((c.nr + kR - 1) / kR, std::max(1, nsm) * (16 / W));
  k1d_fixed_kernel<NB, W><<<grid, W * 32 + 32, smem, c.stream>>>(
      t.tau, t.scale, t.npairs, c.nr, c.nocc, nb, b0, stages, phir, vloc, reinterpret_cast<const double *>(Pa),
      reinterpret_cast<const double *>(Pvh), reinterpret_cast<double *>(Py), use_vloc, use_k1e, t.err, t.hold);
  BSE_CHECK_LAUNCH();
}

// packed pair grids (list + p0 ..) -> tile-major doubles, and the largest high word of every point
__global__ void __launch_bounds__(256) tile_kernel(long nr, int np, int nocc, long npairs, const int2 *__restrict__ pairs,
                                                   const double2 *__restrict__ P, double *__restrict__ tau,
                                                   unsigned *__restrict__ top) {
  const long r = blockIdx.x * (long)blockDim.x + threadIdx.x;
  const long rpad = (nr + kR - 1) / kR * kR;
  if (r >= rpad) return;
  double *dst = tau + (r / kR) * npairs * kR + r % kR;
  unsigned m = 0;
  const int nq = (np + 1) / 2;
  for (int q = blockIdx.y; q < nq; q += gridDim.y) {
    const double2 x = r < nr ? P[(long)q * nr + r] : make_double2(0.0, 0.0);
    const int2 p0 = __ldg(&pairs[2 * q]);
    dst[fixed_slot(p0.x, p0.y, nocc) * kR] = x.x;
    m = max(m, (unsigned)__double2hiint(x.x) & 0x7fffffffu);
    if (2 * q + 1 < np) {
      const int2 p1 = __ldg(&pairs[2 * q + 1]);
      dst[fixed_slot(p1.x, p1.y, nocc) * kR] = x.y;
      m = max(m, (unsigned)__double2hiint(x.y) & 0x7fffffffu);
    }
  }
  if (r < nr) atomicMax(&top[r], m);
}

// Doubles -> limbs in place, relative to the power of two above the point's largest pair, and the point's scale:
// (unit of the sums for max|a| < 1, bits of a).  One CTA per tile; a warp takes whole columns v (sum over
// v' <= v in a register, the mirror terms by shared-memory integer atomics), in units of 2^36 rounded up.
//   th ah: C 2^36 2^(53 + s) / 2^54 <= 1.25 2^62;   th al + tl ah: C 2^36 / 2 + N_occ 2^(52 + s) < 2^63,
// the latter by s <= 4, 3 or 2 for up to 64, 128 or more orbitals; C <= N_occ (2^20 + 1), so s >= -1 up to 261.
// Bound by the read and write of tau (63-well cell 24.6 GB each).
__global__ void __launch_bounds__(256) fix_kernel(long nr, int nocc, long npairs, const unsigned *__restrict__ top,
                                                  double *__restrict__ tau, double2 *__restrict__ scale) {
  extern __shared__ unsigned csum[];  // [nocc][32]
  __shared__ unsigned cmax[kR];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long ntiles = (nr + kR - 1) / kR;
  const int smax = nocc <= 64 ? 4 : nocc <= 128 ? 3 : 2;
  for (long t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const long r = t * kR + lane;
    const bool live = r < nr;
    const unsigned hi = live ? top[r] : 0;
    const int e = exp_above(hi);
    double *tile = tau + (size_t)t * npairs * kR + lane;
    for (int v = warp; v < nocc; v += 8) csum[v * kR + lane] = 0;
    if (warp == 0) cmax[lane] = 0;
    __syncthreads();
    for (int v = warp; v < nocc; v += 8) {
      unsigned col = 0;
      for (int v0 = 0; v0 <= v; v0 += 8) {  // eight loads in flight
        double x[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) x[i] = v0 + i <= v && live ? tile[fixed_slot(v0 + i, v, nocc) * kR] : 0.0;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int vp = v0 + i;
          if (vp > v) break;
          const long long f = to_fixed(x[i], e, kTauBits);
          *reinterpret_cast<int2 *>(&tile[fixed_slot(vp, v, nocc) * kR]) = limbs(f);
          const unsigned m = (unsigned)((f < 0 ? -f : f) >> 36) + 1;
          col += m;
          if (vp != v) atomicAdd(&csum[vp * kR + lane], m);
        }
      }
      atomicAdd(&csum[v * kR + lane], col);
    }
    __syncthreads();
    unsigned c = 0;
    for (int v = warp; v < nocc; v += 8) c = max(c, csum[v * kR + lane]);
    atomicMax(&cmax[lane], c);
    __syncthreads();
    if (warp == 0 && live) {
      int s = smax;
      while (s > -1 && ((unsigned long long)cmax[lane] << (s + 1)) > (5ull << 26)) --s;  // C 2^s <= 1.25 2^27
      scale[r] = make_double2(scale_of(hi, e - kTauBits + 1 - s), 53 + s);
    }
    __syncthreads();
  }
}

}  // namespace

// From 16 orbitals on, as long as the limbs and sums of one vector fit beside the stages.  With 16 orbitals on
// 24^3 one vector takes 13.5 us (FP64 kernel 22.7); with 8 it would take 9.0 (12.2) and with 4 7.9 (7.1),
// which the read of the error flag after the call (about 8 us) outweighs.
bool k1d_fixed_supported(int nocc) { return nocc >= 16 && shape_for(1, nocc).stages > 0; }

size_t k1d_tiled_size(long npairs, long nr) { return (size_t)npairs * ((nr + kR - 1) / kR * kR); }

void k1d_fixed_tile(const Ctx &c, int np, const int2 *pairs, const double2 *P, double *tau, unsigned *top) {
  const long rpad = (c.nr + kR - 1) / kR * kR;
  const dim3 grid((unsigned)((rpad + 255) / 256), 8);
  tile_kernel<<<grid, 256, 0, c.stream>>>(c.nr, np, c.nocc, (long)c.nocc * (c.nocc + 1) / 2, pairs, P, tau, top);
  BSE_CHECK_LAUNCH();
}

void k1d_fixed_finish(const Ctx &c, double *tau, const unsigned *top, double2 *scale) {
  const long npairs = (long)c.nocc * (c.nocc + 1) / 2, ntiles = (c.nr + kR - 1) / kR;
  fix_kernel<<<(unsigned)std::min<long>(ntiles, 152L * 8), 256, (size_t)c.nocc * kR * 4, c.stream>>>(
      c.nr, c.nocc, npairs, top, tau, scale);
  BSE_CHECK_LAUNCH();
}

void k1d_fixed(const Ctx &c, const K1dFixed &t, int nb, const double *phir, const double *vloc, const double2 *Pa,
               const double2 *Pvh, double2 *Py, bool use_vloc, bool use_k1e) {
  auto go = [&](auto n, int b0) {
    constexpr int NB = decltype(n)::value;
    const Shape h = shape_for(NB, c.nocc);
    if (h.warps == 8) launch<NB, 8>(c, t, h.stages, nb, b0, phir, vloc, Pa, Pvh, Py, use_vloc, use_k1e);
    else launch<NB, 16>(c, t, h.stages, nb, b0, phir, vloc, Pa, Pvh, Py, use_vloc, use_k1e);
  };
  for (int b0 = 0; b0 < nb;) {
    if (nb - b0 >= 2 && shape_for(2, c.nocc).stages > 0) {
      go(std::integral_constant<int, 2>(), b0);
      b0 += 2;
    } else {
      go(std::integral_constant<int, 1>(), b0);
      b0 += 1;
    }
  }
}

}  // namespace bse
