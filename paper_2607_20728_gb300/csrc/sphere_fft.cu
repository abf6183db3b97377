// Sphere-pruned transforms between wave-function-sphere vectors and real-space grids.
//
// A function on the wave-function sphere |G|^2 <= Ecut occupies only the columns (n1, n2) of
// the grid whose disk the sphere projects onto, and within a z plane only the y lines of the
// n1 it reaches.  The transforms therefore run as two passes:
//   inverse (sphere -> grid):  z pass over the occupied columns, scattering the real-basis
//     coefficients of two functions (packed as re + i im, Gamma-point symmetry) straight into
//     shared memory; then one xy pass per z plane that places the column results, transforms
//     the occupied y lines and all x lines, and writes the plane once;
//   forward (grid -> sphere):  the mirror image, with the gather to real-basis coefficients
//     (and the diagonal D term of Eq. 2a when asked) fused into the z pass.
// Between the passes only the occupied columns travel through global memory ("column
// buffer", [q][z][column]).  The local-potential product H X = (-1/2 lap + V) X also has a
// fused form whose xy pass transforms, multiplies by V(r) and transforms back in shared
// memory, so the full grid never reaches global memory.
// Columns are ordered as mirror pairs (n1, n2), (-n1, -n2) followed by (0, 0); a z-pass CTA
// takes an even number of columns, so both +G and -G of every coefficient are in its shared
// memory.
#include <algorithm>
#include <map>
#include <mutex>
#include <type_traits>
#include <utility>
#include <vector>

#include "fft_codelets.cuh"
#include "fixed_fft.cuh"
#include "internal.cuh"

namespace bse {

namespace {
using namespace fftc;

constexpr double kRs2 = 0.70710678118654752440;  // 1/sqrt(2)
constexpr int kThreads = 256;
constexpr int kXYThreads = 512;  // the most threads of an FP32 plane pass
// and of a fixed-point one: 96 registers, and every 72-point line stage of 648 or 576 butterflies takes a single
// round (128 grids of 72^2, 512 threads: 512 and 691 us; 672: 502 and 669)
constexpr int kXYFixed = 672;
constexpr int kZMax = 288;      // largest CTA of the fixed-point z passes (two per SM with 112 registers)
constexpr size_t kSmemCap = 200 * 1024;

template <class C>
struct SphArgs {
  int N1, N2, N3, N3p, ncols_pad, CG, nxs;
  long nr;
  const int *colpos;  // [ncols_pad] j1 + N1 j2, -1 for padding
  const int *xs;      // [nxs] x indices with occupied y lines
  const int4 *ent;    // per group: (kk, slot_p N3p + j3_p, slot_m N3p + j3_m, 0)
  const int *ent_off; // [ngroups + 1]
  AxisArgs<C> ax[3];
};

struct StrideBase {
  int s;
  __device__ __forceinline__ int operator()(int t) const { return t * s; }
};
struct ListBase {
  const int *xs;
  __device__ __forceinline__ int operator()(int t) const { return __ldg(&xs[t]); }
};

// L lines of an axis in shared memory, ping-ponging between `in` and `out`; returns the buffer
// holding the result.  Consecutive threads take consecutive lines (of the z lines too: the sphere passes of 128
// orbitals on 72^3 45 / 28 us with consecutive butterflies of one line, 41 / 25 so).  SG is the sign of the
// exponent (+1 inverse, -1 forward), a compile-time constant so that the twiddle conjugation and the factors
// +-i of the codelets fold into additions.  The caller has synchronised the input; the result is synchronised
// on return.
template <class C, int SG, class Base>
__device__ C *lines_fft(C *in, C *out, int L, Base base, int es, const AxisArgs<C> &ax) {
  const typename RealOf<C>::T sg = (typename RealOf<C>::T)SG;
  const int N = ax.n;
  int Ns = 1;
  for (int s = 0; s < ax.nstage; ++s) {
    const int R = ax.radix[s];
    const int nb = N / R;
    const int work = L * nb;
    // e = threadIdx.x + k blockDim.x split as (j, t) = divmod(e, L), advanced without divisions
    int j = threadIdx.x / L, t = threadIdx.x - j * L;
    const int dj = blockDim.x / L, dt = blockDim.x - dj * L;
    for (int e = threadIdx.x; e < work; e += blockDim.x) {
      const int b0 = base(t);
      stage_bfly_any<C>(R, in + b0, out + b0, j, N, Ns, ax.tw, sg, es);
      t += dt;
      j += dj;
      if (t >= L) {
        t -= L;
        ++j;
      }
    }
    __syncthreads();
    C *tmp = in;
    in = out;
    out = tmp;
    Ns *= R;
  }
  return in;
}

// ---- z passes -------------------------------------------------------------------------------
// inverse: real-basis rows X[2q], X[2q+1] -> packed columns of group g -> z transform -> colbuf
template <class C>
__global__ void __launch_bounds__(kThreads) sph_z_inv(SphArgs<C> a, int nf, int npw, const double *__restrict__ X,
                                                      double scale, C *__restrict__ colbuf) {
  using T = typename RealOf<C>::T;
  extern __shared__ __align__(16) unsigned char sm_raw[];
  C *A = reinterpret_cast<C *>(sm_raw);
  C *B = A + (size_t)a.CG * a.N3p;
  const int g = blockIdx.x, q = blockIdx.y;
  const int nline = a.CG * a.N3p;
  for (int e = threadIdx.x; e < nline; e += blockDim.x) A[e] = mkc<C>(0, 0);
  __syncthreads();
  const double *f = X + (long)(2 * q) * npw;
  const bool hasg = (2 * q + 1) < nf;
  const double *h = X + (long)(2 * q + 1) * npw;
  const int e0 = a.ent_off[g], e1 = a.ent_off[g + 1];
  for (int e = e0 + threadIdx.x; e < e1; e += blockDim.x) {
    const int4 en = __ldg(&a.ent[e]);
    const int kk = en.x;
    if (kk == 0) {
      A[en.y] = mkc<C>((T)(f[0] * scale), (T)(hasg ? h[0] * scale : 0.0));
      continue;
    }
    const double r2 = kRs2 * scale;
    const double fc = f[2 * kk - 1] * r2, fs = f[2 * kk] * r2;
    const double gc = hasg ? h[2 * kk - 1] * r2 : 0.0, gs = hasg ? h[2 * kk] * r2 : 0.0;
    A[en.y] = mkc<C>((T)(fc - gs), (T)(fs + gc));  // c_f + i c_g at +G
    A[en.z] = mkc<C>((T)(fc + gs), (T)(gc - fs));  // conj(c_f) + i conj(c_g) at -G
  }
  __syncthreads();
  C *F = lines_fft<C, 1>(A, B, a.CG, StrideBase{a.N3p}, 1, a.ax[2]);
  C *dst = colbuf + (long)q * a.N3 * a.ncols_pad + (long)g * a.CG;
  for (int e = threadIdx.x; e < a.CG * a.N3; e += blockDim.x) {
    const int slot = e % a.CG, z = e / a.CG;
    dst[(long)z * a.ncols_pad + slot] = F[slot * a.N3p + z];
  }
}

// forward: colbuf -> z transform -> gather to real-basis rows (plus the D term when Xd is given)
template <class C>
__global__ void __launch_bounds__(kThreads) sph_z_fwd(SphArgs<C> a, int nf, int npw, const C *__restrict__ colbuf,
                                                      double *__restrict__ Y, double scale,
                                                      const double *__restrict__ Xd,
                                                      const double *__restrict__ kin,
                                                      const double *__restrict__ shift, int period,
                                                      double shift_const) {
  using T = typename RealOf<C>::T;
  extern __shared__ __align__(16) unsigned char sm_raw[];
  C *A = reinterpret_cast<C *>(sm_raw);
  C *B = A + (size_t)a.CG * a.N3p;
  const int g = blockIdx.x, q = blockIdx.y;
  const C *src = colbuf + (long)q * a.N3 * a.ncols_pad + (long)g * a.CG;
  for (int e = threadIdx.x; e < a.CG * a.N3; e += blockDim.x) {
    const int slot = e % a.CG, z = e / a.CG;
    A[slot * a.N3p + z] = src[(long)z * a.ncols_pad + slot];
  }
  __syncthreads();
  const C *F = lines_fft<C, -1>(A, B, a.CG, StrideBase{a.N3p}, 1, a.ax[2]);
  const int f0 = 2 * q, f1 = 2 * q + 1;
  const bool hasg = f1 < nf;
  const double sh0 = (shift ? shift[f0 % period] : 0.0) + shift_const;
  const double sh1 = (shift ? shift[f1 % period] : 0.0) + shift_const;
  const int e0 = a.ent_off[g], e1 = a.ent_off[g + 1];
  for (int e = e0 + threadIdx.x; e < e1; e += blockDim.x) {
    const int4 en = __ldg(&a.ent[e]);
    const int kk = en.x;
    double a0, a1 = 0.0, b0, b1 = 0.0;
    int i0, i1;
    if (kk == 0) {
      const C v = F[en.y];
      i0 = 0;
      i1 = -1;
      a0 = (double)v.x * scale;
      b0 = (double)v.y * scale;
    } else {
      const C Fp = F[en.y], Fm = F[en.z];
      const double s = kRs2 * scale;
      i0 = 2 * kk - 1;
      i1 = 2 * kk;
      a0 = ((double)Fp.x + (double)Fm.x) * s;
      a1 = ((double)Fp.y - (double)Fm.y) * s;
      b0 = ((double)Fp.y + (double)Fm.y) * s;
      b1 = ((double)Fm.x - (double)Fp.x) * s;
    }
    if (Xd) {
      a0 += (kin[i0] + sh0) * Xd[(long)f0 * npw + i0];
      if (i1 >= 0) a1 += (kin[i1] + sh0) * Xd[(long)f0 * npw + i1];
      if (hasg) {
        b0 += (kin[i0] + sh1) * Xd[(long)f1 * npw + i0];
        if (i1 >= 0) b1 += (kin[i1] + sh1) * Xd[(long)f1 * npw + i1];
      }
    }
    Y[(long)f0 * npw + i0] = a0;
    if (i1 >= 0) Y[(long)f0 * npw + i1] = a1;
    if (hasg) {
      Y[(long)f1 * npw + i0] = b0;
      if (i1 >= 0) Y[(long)f1 * npw + i1] = b1;
    }
  }
}

// A plane into its padded buffer, element e = y N1 + x to e + y, four loads in flight per thread (one at a time
// the pass waits for memory a dozen times over; with them orbitals of 72^3 to the grid and back 1.53 -> 1.49 ms).
template <class C, class Get>
__device__ void load_plane(C *dst, int np, int N1, int y, int x, int dy, int dx, Get get) {
  const int nt = blockDim.x;
  auto step = [&] {
    x += dx;
    y += dy;
    if (x >= N1) {
      x -= N1;
      ++y;
    }
  };
  int e = threadIdx.x;
  for (; e + 3 * nt < np; e += 4 * nt) {
    C u[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) u[i] = get(e + i * nt);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      dst[e + i * nt + y] = u[i];
      step();
    }
  }
  for (; e < np; e += nt) {
    dst[e + y] = get(e);
    step();
  }
}

// ---- xy passes (one CTA per plane z of grid q) ---------------------------------------------
// MODE 0: colbuf -> inverse y (occupied lines) and x -> grid plane
// MODE 1: grid plane -> forward x and y (occupied lines) -> colbuf
// MODE 2: colbuf -> inverse -> times V(r) -> forward -> colbuf (in place)
// MODE 3: as MODE 1 for the pair densities of src, multiplied as the plane is loaded (a pass of their own wrote
//   and read back every packed grid: 256 pairs on 40^3, FP32, 32 + 54 us against 58 now)
// The plane sits in shared memory with rows padded to N1 + 1 elements and consecutive threads on
// consecutive lines in both passes (x lines one padded row apart, y lines one x apart), so the
// strided butterfly loads and stores of every stage fall in distinct banks.
template <class C, int MODE>
__global__ void __launch_bounds__(kXYThreads) sph_xy(SphArgs<C> a, C *__restrict__ colbuf, C *__restrict__ P,
                                                     const typename RealOf<C>::T *__restrict__ vloc,
                                                     PairGrids<typename RealOf<C>::T> src) {
  using T = typename RealOf<C>::T;
  extern __shared__ __align__(16) unsigned char sm_raw[];
  const int N1 = a.N1, N1p = a.N1 + 1;
  const int np = N1 * a.N2, npp = N1p * a.N2;
  C *A = reinterpret_cast<C *>(sm_raw);
  C *B = A + npp;
  const int z = blockIdx.x, q = blockIdx.y;
  C *crow = colbuf + ((long)q * a.N3 + z) * a.ncols_pad;
  C *plane = P ? P + (long)q * a.nr + (long)z * np : nullptr;
  // the padded index of element e = y N1 + x of the plane is e + y; (y, x) stepped without divisions
  const int y0 = threadIdx.x / N1, x0 = threadIdx.x - y0 * N1;
  const int dy = blockDim.x / N1, dx = blockDim.x - dy * N1;
  auto for_plane = [&](auto body) {
    int y = y0, x = x0;
    for (int e = threadIdx.x; e < np; e += blockDim.x) {
      body(e, e + y);
      x += dx;
      y += dy;
      if (x >= N1) {
        x -= N1;
        ++y;
      }
    }
  };
  if (MODE == 3) src.select(q, (long)z * np, a.nr);
  C *F;
  if (MODE == 0 || MODE == 2) {
    // the y pass transforms the occupied lines only, so the buffer its result lands in must hold
    // zeros on the others: A with an even number of stages (B is then fully overwritten by the x
    // pass before it is read), B with an odd number
    const bool zero_b = (a.ax[1].nstage & 1) != 0;
    for (int e = threadIdx.x; e < npp; e += blockDim.x) {
      A[e] = mkc<C>(0, 0);
      if (zero_b) B[e] = mkc<C>(0, 0);
    }
    __syncthreads();
    for (int c0 = threadIdx.x; c0 < a.ncols_pad; c0 += 4 * blockDim.x) {
      C u[4];
      int pos[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int c = c0 + i * blockDim.x;
        pos[i] = c < a.ncols_pad ? __ldg(&a.colpos[c]) : -1;
        if (c < a.ncols_pad) u[i] = crow[c];
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (pos[i] >= 0) A[pos[i] + pos[i] / N1] = u[i];
    }
    __syncthreads();
    F = lines_fft<C, 1>(A, B, a.nxs, ListBase{a.xs}, N1p, a.ax[1]);
    C *O = F == A ? B : A;
    F = lines_fft<C, 1>(F, O, a.N2, StrideBase{N1p}, 1, a.ax[0]);
    if (MODE == 0) {
      for_plane([&](int e, int ep) { plane[e] = F[ep]; });
      return;
    }
    const T *v = vloc + (long)z * np;
    for_plane([&](int e, int ep) {
      const T w = v[e];
      const C u = F[ep];
      F[ep] = mkc<C>(u.x * w, u.y * w);
    });
    __syncthreads();
  } else {
    load_plane<C>(A, np, N1, y0, x0, dy, dx, [&](int e) { return src.template at<C, MODE>(plane, e); });
    __syncthreads();
    F = A;
  }
  C *O = F == A ? B : A;
  F = lines_fft<C, -1>(F, O, a.N2, StrideBase{N1p}, 1, a.ax[0]);
  O = F == A ? B : A;
  F = lines_fft<C, -1>(F, O, a.nxs, ListBase{a.xs}, N1p, a.ax[1]);
  for (int c = threadIdx.x; c < a.ncols_pad; c += blockDim.x) {
    const int pos = __ldg(&a.colpos[c]);
    crow[c] = pos >= 0 ? F[pos + pos / N1] : mkc<C>(0, 0);
  }
}

// ---- FP64 xy passes on 64-bit fixed point ---------------------------------------------------------
// The modes of sph_xy for FP64 data: columns and grids stay FP64 in memory, the lines are transformed as
// integers (fixed_fft.cuh).  As FP64 these passes were bound by the FP64 pipe (about 1840 operations per
// 72-point line at two per clock).  Scales, one power of two per plane and pass:
//   MODE 0, 2 (inverse): the sum of |re| + |im| over the plane's columns bounds both passes;
//   MODE 1 (forward): the largest such sum of an x line, then, from the result, of a y line (values are
//   shifted as the first stage of the y pass loads them);
//   MODE 2: the product with V(r) (fixed point below the plane's largest |V|), then as MODE 1.
// Each is an upper bound taken from the leading 21 bits.  Rounding is at 2^-61 of those sums: against extended
// precision (flat data, 24^3 to 72^3) the relative error of a transform is 1.0-2.1e-16, as FP64 3.1-4.1e-16.
// 64 packed grids of the 63-well cell (72^3, 4608 planes), FP64 pass -> this one: inverse 1490 -> 502 us,
// forward 1595 -> 669, H product 2710 -> 1017.  Bound by instruction issue (61 and 70 thousand warp
// instructions a plane, 46% and 42% of the issue slots used: few warps and a barrier per stage).  Measured
// and not kept: radices 8 3 3 for 72 (566 and 685 us), the plane in chunks of rows so that two CTAs share an
// SM (679 and 659).
struct FxArgs {
  int N1, N2, N3, ncols_pad, nxs;
  long nr;
  const int *colpos, *xs;
  fx::Axis ax[2];
};

// L lines in shared memory, consecutive threads on consecutive lines; `first` loads the inputs of the first
// stage (buffer, offset), later stages read the buffers; returns the buffer of the result
template <int SG, class Base, class First>
__device__ fx::C2 *lines_fx(fx::C2 *in, fx::C2 *out, int L, Base base, int es, const fx::Axis &ax, First first) {
  int Ns = 1;
  for (int s = 0; s < ax.nstage; ++s) {
    const int R = ax.radix[s];
    const int work = L * (ax.n / R);
    int j = threadIdx.x / L, t = threadIdx.x - j * L;
    const int dj = blockDim.x / L, dt = blockDim.x - dj * L;
    for (int e = threadIdx.x; e < work; e += blockDim.x) {
      const int b0 = base(t);
      if (s == 0) {
        fx::bfly_any<SG>(R, [&](int o) { return first(in[b0 + o]); }, out + b0, j, ax.n, Ns, ax.tw, es);
      } else {
        fx::bfly_any<SG>(R, [&](int o) { return in[b0 + o]; }, out + b0, j, ax.n, Ns, ax.tw, es);
      }
      t += dt;
      j += dj;
      if (t >= L) {
        t -= L;
        ++j;
      }
    }
    __syncthreads();
    fx::C2 *tmp = in;
    in = out;
    out = tmp;
    Ns *= R;
  }
  return in;
}

template <int MODE>
__global__ void __launch_bounds__(kXYFixed) sph_xy_fx(FxArgs a, double2 *__restrict__ colbuf,
                                                        double2 *__restrict__ P, const double *__restrict__ vloc,
                                                        PairGrids<double> src) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  __shared__ unsigned top, vtop, ltop[2];
  __shared__ int etop;
  __shared__ unsigned long long total;
  const int N1 = a.N1, N1p = a.N1 + 1;
  const int np = N1 * a.N2, npp = N1p * a.N2;
  fx::C2 *A = reinterpret_cast<fx::C2 *>(sm_raw), *B = A + npp;
  const int z = blockIdx.x, q = blockIdx.y;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
  double2 *crow = colbuf + ((long)q * a.N3 + z) * a.ncols_pad;
  double2 *plane = P ? P + (long)q * a.nr + (long)z * np : nullptr;
  const double *v = MODE == 2 ? vloc + (long)z * np : nullptr;
  if (threadIdx.x == 0) {
    top = vtop = ltop[0] = ltop[1] = 0;
    etop = -fx::kBadLine;
    total = 0;
  }
  const int y0 = threadIdx.x / N1, x0 = threadIdx.x - y0 * N1;
  const int dy = blockDim.x / N1, dx = blockDim.x - dy * N1;
  // e = y N1 + x over the plane, e + y its padded place
  auto for_plane = [&](auto body) {
    int y = y0, x = x0;
    for (int e = threadIdx.x; e < np; e += blockDim.x) {
      body(e, e + y);
      x += dx;
      y += dy;
      if (x >= N1) {
        x -= N1;
        ++y;
      }
    }
  };
  auto warp_max = [&](unsigned m, unsigned *dst) {
    m = __reduce_max_sync(0xffffffffu, m);
    if (lane == 0) atomicMax(dst, m);
  };
  // exponent of a bound of n units of 2^u
  auto above = [](unsigned long long n, int u) { return u + 64 - __clzll((long long)n); };
  const auto same = [](fx::C2 c) { return c; };
  fx::Unit unit{0, false};
  fx::C2 *F;
  if (MODE == 0 || MODE == 2) {
    // the y pass transforms the occupied lines only: the buffer of its result holds zeros on the others
    const bool zero_b = (a.ax[1].nstage & 1) != 0;
    for (int e = threadIdx.x; e < npp; e += blockDim.x) {
      A[e] = fx::C2{0, 0};
      if (zero_b) B[e] = fx::C2{0, 0};
    }
    __syncthreads();
    unsigned m = 0, mv = 0;
    for (int c = threadIdx.x; c < a.ncols_pad; c += blockDim.x)
      if (__ldg(&a.colpos[c]) >= 0) m = max(m, max(fx::high_abs(crow[c].x), fx::high_abs(crow[c].y)));
    warp_max(m, &top);
    if (MODE == 2) {
      for (int e = threadIdx.x; e < np; e += blockDim.x) mv = max(mv, fx::high_abs(__ldg(&v[e])));
      warp_max(mv, &vtop);
    }
    __syncthreads();
    const int E = (int)(top >> 20);
    unsigned long long sum = 0;
    for (int c = threadIdx.x; c < a.ncols_pad; c += blockDim.x)
      if (__ldg(&a.colpos[c]) >= 0) sum += fx::mag(crow[c].x, E) + fx::mag(crow[c].y, E);
    for (int w = 16; w > 0; w >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, w);
    if (lane == 0) atomicAdd(&total, sum);
    __syncthreads();
    const int e0 = above(total, E - 1043);
    unit.q = e0 - 61;
    unit.bad = E >= 0x7ff || (MODE == 2 && (vtop >> 20) >= 0x7ff);
    for (int c = threadIdx.x; c < a.ncols_pad; c += blockDim.x) {
      const int pos = __ldg(&a.colpos[c]);
      if (pos >= 0) {
        const double2 u = crow[c];
        A[pos + pos / N1] = fx::C2{fx::from_double(u.x, e0, 61), fx::from_double(u.y, e0, 61)};
      }
    }
    __syncthreads();
    F = lines_fx<1>(A, B, a.nxs, ListBase{a.xs}, N1p, a.ax[1], same);
    F = lines_fx<1>(F, F == A ? B : A, a.N2, StrideBase{N1p}, 1, a.ax[0], same);
    if (MODE == 0) {
      for_plane([&](int e, int ep) { plane[e] = make_double2(unit(F[ep].x), unit(F[ep].y)); });
      return;
    }
    const int ev = max((int)(vtop >> 20), 1) - 1022;  // |V| < 2^ev
    for_plane([&](int e, int ep) {
      const fx::W w = fx::split(fx::from_double(__ldg(&v[e]), ev, 62));
      F[ep] = fx::cscale(F[ep], w);
    });
    unit.q += ev;
    __syncthreads();
  } else {
    if (MODE == 3) src.select(q, (long)z * np, a.nr);
    load_plane<double2>(reinterpret_cast<double2 *>(A), np, N1, y0, x0, dy, dx,
                        [&](int e) { return src.template at<double2, MODE>(plane, e); });
    __syncthreads();
    F = A;
  }
  // forward: the largest sum of |re| + |im| over an x line, one warp per line
  for (int y = warp; y < a.N2; y += nwarp) {
    if (MODE & 1) {
      const double2 *row = reinterpret_cast<const double2 *>(F) + y * N1p;
      const int e = fx::line_exponent(N1, [&](int x) { return row[x]; });
      if (lane == 0) atomicMax(&etop, e);
    } else {
      unsigned s = 0;
      for (int x = lane; x < N1; x += 32) {
        const fx::C2 u = F[y * N1p + x];
        s += (unsigned)((unsigned long long)llabs(u.x) >> 40) + (unsigned)((unsigned long long)llabs(u.y) >> 40) + 2;
      }
      s = __reduce_add_sync(0xffffffffu, s);
      if (lane == 0) atomicMax(&ltop[0], s);
    }
  }
  __syncthreads();
  // values shifted as they are loaded: k > 0 right (rounded), k < 0 left
  auto shifted = [](fx::C2 c, int k) {
    if (k <= 0) return fx::C2{c.x << -k, c.y << -k};
    const long long h = 1ll << (k - 1);
    return fx::C2{(c.x + h) >> k, (c.y + h) >> k};
  };
  fx::C2 *O = F == A ? B : A;
  if (MODE & 1) {
    unit.bad = etop >= fx::kBadLine;
    const int e0 = unit.bad ? 0 : etop;
    unit.q = e0 - 61;
    F = lines_fx<-1>(F, O, a.N2, StrideBase{N1p}, 1, a.ax[0], [&](const fx::C2 &c) {
      return fx::C2{fx::from_double(__longlong_as_double(c.x), e0, 61), fx::from_double(__longlong_as_double(c.y), e0, 61)};
    });
  } else {
    const int k = max(above(ltop[0], 40) - 61, -30);
    unit.q += k;
    F = lines_fx<-1>(F, O, a.N2, StrideBase{N1p}, 1, a.ax[0], [&](const fx::C2 &c) { return shifted(c, k); });
  }
  for (int t = warp; t < a.nxs; t += nwarp) {
    const int x = __ldg(&a.xs[t]);
    unsigned s = 0;
    for (int y = lane; y < a.N2; y += 32) {
      const fx::C2 u = F[y * N1p + x];
      s += (unsigned)((unsigned long long)llabs(u.x) >> 40) + (unsigned)((unsigned long long)llabs(u.y) >> 40) + 2;
    }
    s = __reduce_add_sync(0xffffffffu, s);
    if (lane == 0) atomicMax(&ltop[1], s);
  }
  __syncthreads();
  const int k = max(above(ltop[1], 40) - 61, -30);
  unit.q += k;
  F = lines_fx<-1>(F, F == A ? B : A, a.nxs, ListBase{a.xs}, N1p, a.ax[1], [&](const fx::C2 &c) { return shifted(c, k); });
  for (int c = threadIdx.x; c < a.ncols_pad; c += blockDim.x) {
    const int pos = __ldg(&a.colpos[c]);
    const fx::C2 u = pos >= 0 ? F[pos + pos / N1] : fx::C2{0, 0};
    crow[c] = pos >= 0 ? make_double2(unit(u.x), unit(u.y)) : make_double2(0.0, 0.0);
  }
}

// ---- FP64 z passes on 64-bit fixed point ------------------------------------------------------------
// The z passes of FP64 data: CG columns of a group in shared memory as [slot][z], consecutive threads on
// consecutive columns, one power of two per CTA from the largest sum of |re| + |im| over a column.  As FP64
// (32 lines of 72 points per CTA) they were bound by the FP64 pipe like the plane passes.
struct FzArgs {
  int N1, N2, N3, N3p, ncols_pad, CG;
  const int *colpos;
  const int4 *ent;
  const int *ent_off;
  fx::Axis ax;
};

// FP64 columns in A (synchronised) -> transformed columns as integers of the unit set on return; B: scratch
template <int SG>
__device__ fx::C2 *z_lines(const FzArgs &a, double2 *Ad, fx::C2 *B, fx::Unit &unit) {
  __shared__ int ltop;
  if (threadIdx.x == 0) ltop = -fx::kBadLine;
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
  for (int l = warp; l < a.CG; l += nwarp) {
    const int e = fx::line_exponent(a.N3, [&](int z) { return Ad[l * a.N3p + z]; });
    if (lane == 0) atomicMax(&ltop, e);
  }
  __syncthreads();
  unit.bad = ltop >= fx::kBadLine;
  const int e0 = unit.bad ? 0 : ltop;
  unit.q = e0 - 61;
  return lines_fx<SG>(reinterpret_cast<fx::C2 *>(Ad), B, a.CG, StrideBase{a.N3p}, 1, a.ax, [&](const fx::C2 &c) {
    return fx::C2{fx::from_double(__longlong_as_double(c.x), e0, 61), fx::from_double(__longlong_as_double(c.y), e0, 61)};
  });
}

// A real factor and the same over sqrt(2), the latter in two parts: as one double, its rounding and that of
// 1 / sqrt(2) are the same for every element and were most of a fixed-point transform's error.  There and back
// with a product between (flat data, against extended precision): 36^3 2.8e-16 -> 1.1e-16, 45 40 54 3.5e-16 ->
// 1.1e-16, 72^3 2.9e-16 -> 1.4e-16; as FP64 2.4e-16, 3.2e-16 and 2.4e-16.  No difference in time.
struct PairScale {
  double all, hi, lo;
  explicit PairScale(long double scale) : all((double)scale) {
    const long double p = scale * 0.70710678118654752440084436210484903928L;
    hi = (double)p;
    lo = (double)(p - (long double)hi);
  }
  __device__ __forceinline__ double operator()(double x) const { return fma(x, hi, x * lo); }
};

__global__ void __launch_bounds__(kZMax, 2) sph_z_inv_fx(FzArgs a, int nf, int npw, const double *__restrict__ X,
                                                      PairScale scale, double2 *__restrict__ colbuf) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  double2 *A = reinterpret_cast<double2 *>(sm_raw);
  fx::C2 *B = reinterpret_cast<fx::C2 *>(A + (size_t)a.CG * a.N3p);
  const int g = blockIdx.x, q = blockIdx.y;
  for (int e = threadIdx.x; e < a.CG * a.N3p; e += blockDim.x) A[e] = make_double2(0, 0);
  __syncthreads();
  const double *f = X + (long)(2 * q) * npw;
  const bool hasg = (2 * q + 1) < nf;
  const double *h = X + (long)(2 * q + 1) * npw;
  const int e0 = a.ent_off[g], e1 = a.ent_off[g + 1];
  for (int e = e0 + threadIdx.x; e < e1; e += blockDim.x) {
    const int4 en = __ldg(&a.ent[e]);
    const int kk = en.x;
    if (kk == 0) {
      A[en.y] = make_double2(f[0] * scale.all, hasg ? h[0] * scale.all : 0.0);
      continue;
    }
    const double fc = scale(f[2 * kk - 1]), fs = scale(f[2 * kk]);
    const double gc = hasg ? scale(h[2 * kk - 1]) : 0.0, gs = hasg ? scale(h[2 * kk]) : 0.0;
    A[en.y] = make_double2(fc - gs, fs + gc);  // c_f + i c_g at +G
    A[en.z] = make_double2(fc + gs, gc - fs);  // conj(c_f) + i conj(c_g) at -G
  }
  __syncthreads();
  fx::Unit unit{0, false};
  const fx::C2 *F = z_lines<1>(a, A, B, unit);
  double2 *dst = colbuf + (long)q * a.N3 * a.ncols_pad + (long)g * a.CG;
  for (int e = threadIdx.x; e < a.CG * a.N3; e += blockDim.x) {
    const int slot = e % a.CG, z = e / a.CG;
    const fx::C2 u = F[slot * a.N3p + z];
    dst[(long)z * a.ncols_pad + slot] = make_double2(unit(u.x), unit(u.y));
  }
}

__global__ void __launch_bounds__(kZMax, 2) sph_z_fwd_fx(FzArgs a, int nf, int npw, const double2 *__restrict__ colbuf,
                                                      double *__restrict__ Y, PairScale scale,
                                                      const double *__restrict__ Xd, const double *__restrict__ kin,
                                                      const double *__restrict__ shift, int period,
                                                      double shift_const) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  double2 *A = reinterpret_cast<double2 *>(sm_raw);
  fx::C2 *B = reinterpret_cast<fx::C2 *>(A + (size_t)a.CG * a.N3p);
  const int g = blockIdx.x, q = blockIdx.y;
  const double2 *src = colbuf + (long)q * a.N3 * a.ncols_pad + (long)g * a.CG;
  for (int e = threadIdx.x; e < a.CG * a.N3; e += blockDim.x) {
    const int slot = e % a.CG, z = e / a.CG;
    A[slot * a.N3p + z] = src[(long)z * a.ncols_pad + slot];
  }
  fx::Unit unit{0, false};
  const fx::C2 *F = z_lines<-1>(a, A, B, unit);
  const int f0 = 2 * q, f1 = 2 * q + 1;
  const bool hasg = f1 < nf;
  const double sh0 = (shift ? shift[f0 % period] : 0.0) + shift_const;
  const double sh1 = (shift ? shift[f1 % period] : 0.0) + shift_const;
  const int e0 = a.ent_off[g], e1 = a.ent_off[g + 1];
  for (int e = e0 + threadIdx.x; e < e1; e += blockDim.x) {
    const int4 en = __ldg(&a.ent[e]);
    const int kk = en.x;
    double a0, a1 = 0.0, b0, b1 = 0.0;
    int i0, i1;
    if (kk == 0) {
      const fx::C2 v = F[en.y];
      i0 = 0;
      i1 = -1;
      a0 = unit(v.x) * scale.all;
      b0 = unit(v.y) * scale.all;
    } else {
      const fx::C2 Fp = F[en.y], Fm = F[en.z];
      i0 = 2 * kk - 1;
      i1 = 2 * kk;
      a0 = scale(unit(Fp.x + Fm.x));
      a1 = scale(unit(Fp.y - Fm.y));
      b0 = scale(unit(Fp.y + Fm.y));
      b1 = scale(unit(Fm.x - Fp.x));
    }
    if (Xd) {
      a0 += (kin[i0] + sh0) * Xd[(long)f0 * npw + i0];
      if (i1 >= 0) a1 += (kin[i1] + sh0) * Xd[(long)f0 * npw + i1];
      if (hasg) {
        b0 += (kin[i0] + sh1) * Xd[(long)f1 * npw + i0];
        if (i1 >= 0) b1 += (kin[i1] + sh1) * Xd[(long)f1 * npw + i1];
      }
    }
    Y[(long)f0 * npw + i0] = a0;
    if (i1 >= 0) Y[(long)f0 * npw + i1] = a1;
    if (hasg) {
      Y[(long)f1 * npw + i0] = b0;
      if (i1 >= 0) Y[(long)f1 * npw + i1] = b1;
    }
  }
}

// the pair pipelines' z passes (dsph_z_fwd, dsph_z_inv below) for FP64 data
__global__ void __launch_bounds__(kZMax, 2) dsph_z_fwd_fx(FzArgs a, int np, int npw, double2 *__restrict__ colbuf,
                                                       double *__restrict__ X, PairScale scale,
                                                       const double *__restrict__ vcg, double cscale) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  double2 *A = reinterpret_cast<double2 *>(sm_raw);
  fx::C2 *B = reinterpret_cast<fx::C2 *>(A + (size_t)a.CG * a.N3p);
  const int g = blockIdx.x, q = blockIdx.y;
  double2 *col = colbuf + (long)q * a.N3 * a.ncols_pad + (long)g * a.CG;
  for (int e = threadIdx.x; e < a.CG * a.N3; e += blockDim.x) {
    const int slot = e % a.CG, z = e / a.CG;
    A[slot * a.N3p + z] = col[(long)z * a.ncols_pad + slot];
  }
  fx::Unit unit{0, false};
  const fx::C2 *F = z_lines<-1>(a, A, B, unit);
  if (X) {
    const int f0 = 2 * q, f1 = 2 * q + 1;
    const bool hasg = f1 < np;
    for (int e = a.ent_off[g] + threadIdx.x; e < a.ent_off[g + 1]; e += blockDim.x) {
      const int4 en = __ldg(&a.ent[e]);
      const int kk = en.x;
      if (kk == 0) {
        const fx::C2 v = F[en.y];
        X[(long)f0 * npw] = unit(v.x) * scale.all;
        if (hasg) X[(long)f1 * npw] = unit(v.y) * scale.all;
        continue;
      }
      const fx::C2 Fp = F[en.y], Fm = F[en.z];
      X[(long)f0 * npw + 2 * kk - 1] = scale(unit(Fp.x + Fm.x));
      X[(long)f0 * npw + 2 * kk] = scale(unit(Fp.y - Fm.y));
      if (hasg) {
        X[(long)f1 * npw + 2 * kk - 1] = scale(unit(Fp.y + Fm.y));
        X[(long)f1 * npw + 2 * kk] = scale(unit(Fm.x - Fp.x));
      }
    }
  }
  const long np2 = (long)a.N1 * a.N2;
  for (int e = threadIdx.x; e < a.CG * a.N3; e += blockDim.x) {
    const int slot = e % a.CG, z = e / a.CG;
    const int pos = __ldg(&a.colpos[g * a.CG + slot]);
    const double w = pos >= 0 ? vcg[(long)z * np2 + pos] * cscale : 0.0;
    const fx::C2 v = F[slot * a.N3p + z];
    col[(long)z * a.ncols_pad + slot] = pos >= 0 ? make_double2(unit(v.x) * w, unit(v.y) * w) : make_double2(0.0, 0.0);
  }
}

__global__ void __launch_bounds__(kZMax, 2) dsph_z_inv_fx(FzArgs a, int np, int npw, const double *__restrict__ X,
                                                       PairScale scale, double2 *__restrict__ colbuf) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  double2 *A = reinterpret_cast<double2 *>(sm_raw);
  fx::C2 *B = reinterpret_cast<fx::C2 *>(A + (size_t)a.CG * a.N3p);
  const int g = blockIdx.x, q = blockIdx.y;
  double2 *col = colbuf + (long)q * a.N3 * a.ncols_pad + (long)g * a.CG;
  for (int e = threadIdx.x; e < a.CG * a.N3; e += blockDim.x) {
    const int slot = e % a.CG, z = e / a.CG;
    A[slot * a.N3p + z] = col[(long)z * a.ncols_pad + slot];
  }
  __syncthreads();
  if (X) {
    const double *f = X + (long)(2 * q) * npw;
    const bool hasg = (2 * q + 1) < np;
    const double *h = X + (long)(2 * q + 1) * npw;
    for (int e = a.ent_off[g] + threadIdx.x; e < a.ent_off[g + 1]; e += blockDim.x) {
      const int4 en = __ldg(&a.ent[e]);
      const int kk = en.x;
      double2 &tp = A[en.y];
      if (kk == 0) {
        tp = make_double2(tp.x + f[0] * scale.all, tp.y + (hasg ? h[0] * scale.all : 0.0));
        continue;
      }
      const double fc = scale(f[2 * kk - 1]), fs = scale(f[2 * kk]);
      const double gc = hasg ? scale(h[2 * kk - 1]) : 0.0, gs = hasg ? scale(h[2 * kk]) : 0.0;
      tp = make_double2(tp.x + (fc - gs), tp.y + (fs + gc));
      double2 &tm = A[en.z];
      tm = make_double2(tm.x + (fc + gs), tm.y + (gc - fs));
    }
    __syncthreads();
  }
  fx::Unit unit{0, false};
  const fx::C2 *F = z_lines<1>(a, A, B, unit);
  for (int e = threadIdx.x; e < a.CG * a.N3; e += blockDim.x) {
    const int slot = e % a.CG, z = e / a.CG;
    const fx::C2 u = F[slot * a.N3p + z];
    col[(long)z * a.ncols_pad + slot] = make_double2(unit(u.x), unit(u.y));
  }
}

// ---- pair pipelines on the density sphere (tau build, U vector; Eq. 2c and Eq. 3) ----------
// FP32, six CTAs per SM (a CTA only loads, transforms and stores, so it is their number that hides the memory
// behind them): 128 grids of 40^3, forward / inverse 28 / 23 us as the compiler left the registers, 25 / 22 now,
// 17 at the copy rate.  Sums in FP32 pairs instead of on the FP64 pipe and four loads in flight gave nothing.
// forward z pass: z lines of the occupied density columns, then the wave-function-sphere
// coefficients of the two packed pair densities into X (real basis, type R, times `scale`) for
// the PDEP projection, and every column element times v_c(G) * cscale (zero outside the density
// sphere) written back
template <class C, class R>
__global__ void __launch_bounds__(kThreads, 6) dsph_z_fwd(SphArgs<C> a, int np, int npw, C *__restrict__ colbuf,
                                                       R *__restrict__ X, double scale,
                                                       const R *__restrict__ vcg, R cscale) {
  using T = typename RealOf<C>::T;
  extern __shared__ __align__(16) unsigned char sm_raw[];
  C *A = reinterpret_cast<C *>(sm_raw);
  C *B = A + (size_t)a.CG * a.N3p;
  const int g = blockIdx.x, q = blockIdx.y;
  C *col = colbuf + (long)q * a.N3 * a.ncols_pad + (long)g * a.CG;
  for (int e = threadIdx.x; e < a.CG * a.N3; e += blockDim.x) {
    const int slot = e % a.CG, z = e / a.CG;
    A[slot * a.N3p + z] = col[(long)z * a.ncols_pad + slot];
  }
  __syncthreads();
  C *F = lines_fft<C, -1>(A, B, a.CG, StrideBase{a.N3p}, 1, a.ax[2]);
  if (X) {
    const int f0 = 2 * q, f1 = 2 * q + 1;
    const bool hasg = f1 < np;
    for (int e = a.ent_off[g] + threadIdx.x; e < a.ent_off[g + 1]; e += blockDim.x) {
      const int4 en = __ldg(&a.ent[e]);
      const int kk = en.x;
      if (kk == 0) {
        const C v = F[en.y];
        X[(long)f0 * npw] = (R)((double)v.x * scale);
        if (hasg) X[(long)f1 * npw] = (R)((double)v.y * scale);
        continue;
      }
      const C Fp = F[en.y], Fm = F[en.z];
      const double sc = kRs2 * scale;
      X[(long)f0 * npw + 2 * kk - 1] = (R)(((double)Fp.x + (double)Fm.x) * sc);
      X[(long)f0 * npw + 2 * kk] = (R)(((double)Fp.y - (double)Fm.y) * sc);
      if (hasg) {
        X[(long)f1 * npw + 2 * kk - 1] = (R)(((double)Fp.y + (double)Fm.y) * sc);
        X[(long)f1 * npw + 2 * kk] = (R)(((double)Fm.x - (double)Fp.x) * sc);
      }
    }
  }
  const long np2 = (long)a.N1 * a.N2;
  for (int e = threadIdx.x; e < a.CG * a.N3; e += blockDim.x) {
    const int slot = e % a.CG, z = e / a.CG;
    const int pos = __ldg(&a.colpos[g * a.CG + slot]);
    const T w = pos >= 0 ? (T)(vcg[(long)z * np2 + pos] * cscale) : (T)0;
    const C v = F[slot * a.N3p + z];
    col[(long)z * a.ncols_pad + slot] = mkc<C>(v.x * w, v.y * w);
  }
}

// inverse z pass: the PDEP back-projection X (real basis, type R, times `scale`) added at the
// wave-function-sphere coefficients of the two packed pairs, then z lines of the columns
template <class C, class R>
__global__ void __launch_bounds__(kThreads, 6) dsph_z_inv(SphArgs<C> a, int np, int npw, const R *__restrict__ X,
                                                       double scale, C *__restrict__ colbuf) {
  using T = typename RealOf<C>::T;
  extern __shared__ __align__(16) unsigned char sm_raw[];
  C *A = reinterpret_cast<C *>(sm_raw);
  C *B = A + (size_t)a.CG * a.N3p;
  const int g = blockIdx.x, q = blockIdx.y;
  C *col = colbuf + (long)q * a.N3 * a.ncols_pad + (long)g * a.CG;
  for (int e = threadIdx.x; e < a.CG * a.N3; e += blockDim.x) {
    const int slot = e % a.CG, z = e / a.CG;
    A[slot * a.N3p + z] = col[(long)z * a.ncols_pad + slot];
  }
  __syncthreads();
  if (X) {
    const R *f = X + (long)(2 * q) * npw;
    const bool hasg = (2 * q + 1) < np;
    const R *h = X + (long)(2 * q + 1) * npw;
    for (int e = a.ent_off[g] + threadIdx.x; e < a.ent_off[g + 1]; e += blockDim.x) {
      const int4 en = __ldg(&a.ent[e]);
      const int kk = en.x;
      if (kk == 0) {
        C &t = A[en.y];
        t = mkc<C>(t.x + (T)((double)f[0] * scale), t.y + (T)(hasg ? (double)h[0] * scale : 0.0));
        continue;
      }
      const double r2 = kRs2 * scale;
      const double fc = (double)f[2 * kk - 1] * r2, fs = (double)f[2 * kk] * r2;
      const double gc = hasg ? (double)h[2 * kk - 1] * r2 : 0.0, gs = hasg ? (double)h[2 * kk] * r2 : 0.0;
      C &tp = A[en.y];
      tp = mkc<C>(tp.x + (T)(fc - gs), tp.y + (T)(fs + gc));
      C &tm = A[en.z];
      tm = mkc<C>(tm.x + (T)(fc + gs), tm.y + (T)(gc - fs));
    }
  }
  __syncthreads();
  C *F = lines_fft<C, 1>(A, B, a.CG, StrideBase{a.N3p}, 1, a.ax[2]);
  for (int e = threadIdx.x; e < a.CG * a.N3; e += blockDim.x) {
    const int slot = e % a.CG, z = e / a.CG;
    col[(long)z * a.ncols_pad + slot] = F[slot * a.N3p + z];
  }
}

template <class C>
SphArgs<C> make_args(const Ctx &c, const SphereFFT &s) {
  SphArgs<C> a;
  a.N1 = c.N[0];
  a.N2 = c.N[1];
  a.N3 = c.N[2];
  a.N3p = c.N[2] + 1;
  a.ncols_pad = s.ncols_pad;
  a.CG = s.cg;
  a.nxs = s.nxs;
  a.nr = c.nr;
  a.colpos = s.colpos.get();
  a.xs = s.xs.get();
  a.ent = s.ent.get();
  a.ent_off = s.ent_off.get();
  for (int i = 0; i < 3; ++i) {
    const FFTAxis &x = c.fft.ax[i];
    a.ax[i].n = x.n;
    a.ax[i].nstage = x.nstage;
    for (int r = 0; r < 12; ++r) a.ax[i].radix[r] = x.radix[r];
    if constexpr (sizeof(C) == sizeof(double2)) a.ax[i].tw = reinterpret_cast<const C *>(x.tw);
    else a.ax[i].tw = reinterpret_cast<const C *>(x.tw32);
  }
  return a;
}

// one plane pass (MODE of sph_xy) over nq packed grids: FP64 in fixed point, FP32 as it is
template <class C, int MODE>
void launch_xy(Ctx &c, const SphereFFT &s, int nq, C *cb, C *P, const typename RealOf<C>::T *v,
               const PairGrids<typename RealOf<C>::T> &src = {});

template <class C>
size_t z_smem(const Ctx &c, const SphereFFT &s) { return (size_t)2 * s.cg * (c.N[2] + 1) * sizeof(C); }
template <class C>
size_t z_smem(const Ctx &c) { return z_smem<C>(c, c.sfft); }
template <class C>
size_t xy_smem(const Ctx &c) { return (size_t)2 * (c.N[0] + 1) * c.N[1] * sizeof(C); }

// dynamic shared-memory limits are per-device function attributes: set once per device
template <class C>
void set_attrs() {
  static std::mutex mu;
  static std::map<int, bool> done;
  int dev = 0;
  BSE_CUDA(cudaGetDevice(&dev));
  std::lock_guard<std::mutex> lock(mu);
  if (done[dev]) return;
  const int cap = (int)kSmemCap;
  if constexpr (sizeof(C) == sizeof(double2)) {
    BSE_CUDA(cudaFuncSetAttribute(sph_z_inv_fx, cudaFuncAttributeMaxDynamicSharedMemorySize, cap));
    BSE_CUDA(cudaFuncSetAttribute(sph_z_fwd_fx, cudaFuncAttributeMaxDynamicSharedMemorySize, cap));
    BSE_CUDA(cudaFuncSetAttribute(dsph_z_fwd_fx, cudaFuncAttributeMaxDynamicSharedMemorySize, cap));
    BSE_CUDA(cudaFuncSetAttribute(dsph_z_inv_fx, cudaFuncAttributeMaxDynamicSharedMemorySize, cap));
    BSE_CUDA(cudaFuncSetAttribute(sph_xy_fx<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, cap));
    BSE_CUDA(cudaFuncSetAttribute(sph_xy_fx<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, cap));
    BSE_CUDA(cudaFuncSetAttribute(sph_xy_fx<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, cap));
    BSE_CUDA(cudaFuncSetAttribute(sph_xy_fx<3>, cudaFuncAttributeMaxDynamicSharedMemorySize, cap));
  } else {
    using R = typename RealOf<C>::T;
    BSE_CUDA(cudaFuncSetAttribute(sph_z_inv<C>, cudaFuncAttributeMaxDynamicSharedMemorySize, cap));
    BSE_CUDA(cudaFuncSetAttribute(sph_z_fwd<C>, cudaFuncAttributeMaxDynamicSharedMemorySize, cap));
    BSE_CUDA(cudaFuncSetAttribute(dsph_z_fwd<C, R>, cudaFuncAttributeMaxDynamicSharedMemorySize, cap));
    BSE_CUDA(cudaFuncSetAttribute(dsph_z_inv<C, R>, cudaFuncAttributeMaxDynamicSharedMemorySize, cap));
    BSE_CUDA(cudaFuncSetAttribute(sph_xy<C, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, cap));
    BSE_CUDA(cudaFuncSetAttribute(sph_xy<C, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, cap));
    BSE_CUDA(cudaFuncSetAttribute(sph_xy<C, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, cap));
    BSE_CUDA(cudaFuncSetAttribute(sph_xy<C, 3>, cudaFuncAttributeMaxDynamicSharedMemorySize, cap));
  }
  done[dev] = true;
}

// Threads per plane-pass CTA: the autotuner's choice, else what an SM's registers hold (kXYSM, by type) over
// the planes that share an SM, which a plane's shared memory and the number of planes give.  More threads per
// plane only idle (a stage of 40^2 has 200 butterflies) and keep the other planes out; fewer leave the SM
// without warps.  256 functions on 128 grids, us, inverse / forward, with 512 FP32 or 256 (up to 54^2) and 672
// FP64 threads -> with this rule, and in brackets with 64 to 128 threads fewer or more:
//   FP32 36^2 74/73 -> 35/35, 40^2 85/86 -> 43/46, 48^2 171/193 -> 123/131 (121/159), 54^2 221/242 -> 172/197,
//        60^2 250/286 -> 216/256 (212/282, 241/240), 64^2 187/244 -> 162/234 (156/254, 183/218)
//   FP64 24^2 49/65 -> 35/51, 30^2 105/122 -> 83/102, 36^2 125/187 -> 110/172 (114/168), 40^2 146/209 -> 134/209
//        (139/233), 54^2 489/644 -> 450/558
constexpr int kXYSM32 = 1024, kXYSM64 = 768;
template <class C>
int xy_threads(const Ctx &c, int nq) {
  constexpr bool fixed = sizeof(C) == sizeof(double2);
  if (c.xy_threads > 0) return std::min(c.xy_threads, kXYThreads);
  const long fit = 227 * 1024 / (long)(xy_smem<C>(c) + 1024), share = ((long)c.N[2] * nq + 151) / 152;
  const int t = (fixed ? kXYSM64 : kXYSM32) / (int)std::max(1L, std::min(fit, share));
  return std::max(128, std::min(fixed ? kXYFixed : kXYThreads, (t + 32) / 64 * 64));
}

template <class C, int MODE>
void launch_xy(Ctx &c, const SphereFFT &s, int nq, C *cb, C *P, const typename RealOf<C>::T *v,
               const PairGrids<typename RealOf<C>::T> &src) {
  const dim3 grid(c.N[2], nq);
  if constexpr (sizeof(C) == sizeof(double2)) {
    FxArgs a;
    a.N1 = c.N[0];
    a.N2 = c.N[1];
    a.N3 = c.N[2];
    a.ncols_pad = s.ncols_pad;
    a.nxs = s.nxs;
    a.nr = c.nr;
    a.colpos = s.colpos.get();
    a.xs = s.xs.get();
    for (int i = 0; i < 2; ++i) {
      const FFTAxis &x = c.fft.ax[i];
      a.ax[i].n = x.n;
      a.ax[i].nstage = x.nstage;
      for (int r = 0; r < 12; ++r) a.ax[i].radix[r] = x.radix[r];
      a.ax[i].tw = x.twx;
    }
    sph_xy_fx<MODE><<<grid, xy_threads<C>(c, nq), xy_smem<C>(c), c.stream>>>(a, cb, P, v, src);
  } else {
    sph_xy<C, MODE><<<grid, xy_threads<C>(c, nq), xy_smem<C>(c), c.stream>>>(make_args<C>(c, s), cb, P, v, src);
  }
  BSE_CHECK_LAUNCH();
}

FzArgs fz_args(const Ctx &c, const SphereFFT &s) {
  FzArgs a;
  a.N1 = c.N[0];
  a.N2 = c.N[1];
  a.N3 = c.N[2];
  a.N3p = c.N[2] + 1;
  a.ncols_pad = s.ncols_pad;
  a.CG = s.cg;
  a.colpos = s.colpos.get();
  a.ent = s.ent.get();
  a.ent_off = s.ent_off.get();
  const FFTAxis &x = c.fft.ax[2];
  a.ax.n = x.n;
  a.ax.nstage = x.nstage;
  for (int r = 0; r < 12; ++r) a.ax.radix[r] = x.radix[r];
  a.ax.tw = x.twx;
  return a;
}
// threads of a fixed-point z pass: a stage of radix R takes N3/R rounds of one warp (32 columns), so the
// warp count (6 to 9) is the one with the fewest rounds over all stages per warp of occupancy
int z_threads(const Ctx &c) {
  const FFTAxis &x = c.fft.ax[2];
  int best = 8;
  double bc = 1e30;
  for (int w = 6; w <= kZMax / 32; ++w) {
    double rounds = 0;
    for (int s = 0; s < x.nstage; ++s) rounds += (x.n / x.radix[s] + w - 1) / w;
    const double cost = rounds * w;
    if (cost < bc - 1e-9) {
      bc = cost;
      best = w;
    }
  }
  return best * 32;
}

// the z passes of either precision: FP64 in fixed point, FP32 as it is
template <class C>
void launch_z_inv(Ctx &c, int nf, int nq, const double *X, long double scale, C *cb) {
  const dim3 grid(c.sfft.ngroups, nq);
  if constexpr (sizeof(C) == sizeof(double2))
    sph_z_inv_fx<<<grid, z_threads(c), z_smem<C>(c), c.stream>>>(fz_args(c, c.sfft), nf, c.npw, X, PairScale(scale), cb);
  else
    sph_z_inv<C><<<grid, kThreads, z_smem<C>(c), c.stream>>>(make_args<C>(c, c.sfft), nf, c.npw, X, (double)scale, cb);
  BSE_CHECK_LAUNCH();
}
template <class C>
void launch_z_fwd(Ctx &c, int nf, int nq, const C *cb, double *Y, long double scale, const double *Xd, const double *shift,
                  int period, double shift_const) {
  const dim3 grid(c.sfft.ngroups, nq);
  if constexpr (sizeof(C) == sizeof(double2))
    sph_z_fwd_fx<<<grid, z_threads(c), z_smem<C>(c), c.stream>>>(fz_args(c, c.sfft), nf, c.npw, cb, Y, PairScale(scale), Xd,
                                                               c.kin.get(), shift, period, shift_const);
  else
    sph_z_fwd<C><<<grid, kThreads, z_smem<C>(c), c.stream>>>(make_args<C>(c, c.sfft), nf, c.npw, cb, Y, (double)scale, Xd,
                                                             c.kin.get(), shift, period, shift_const);
  BSE_CHECK_LAUNCH();
}

template <class R>
CT<R> *colbuf_for(Ctx &c, int nq) {
  Grids<R> &g = c.grids<R>();
  g.colbuf.alloc((size_t)nq * c.N[2] * c.sfft.ncols_pad);
  return g.colbuf.get();
}

}  // namespace

// ---- plan ----------------------------------------------------------------------------------
namespace {
// Column tables of one sphere: the columns of `col_millers` ((n1, n2) pairs, closed under
// negation) as mirror pairs then (0, 0); the coefficient entries of the wave-function half
// sphere (miller_half) placed in that column layout.
void build_tables(Ctx &c, SphereFFT &s, const std::vector<std::pair<int, int>> &col_millers,
                  const std::vector<int> &miller_half) {
  s.ready = s.ok64 = s.ok32 = false;
  const int N1 = c.N[0], N2 = c.N[1], N3 = c.N[2];
  const int nh = (int)miller_half.size() / 3;  // entries kk = 0..nhalf (kk = 0 is G = 0)
  auto md = [](int v, int n) { return ((v % n) + n) % n; };
  std::map<std::pair<int, int>, int> col;
  std::vector<std::pair<int, int>> order;
  for (const auto &cm : col_millers) {
    const int n1 = cm.first, n2 = cm.second;
    const bool pos = n2 > 0 || (n2 == 0 && n1 > 0);
    if (!pos || col.count({n1, n2})) continue;
    col[{n1, n2}] = -1;
    order.push_back({n1, n2});
  }
  std::sort(order.begin(), order.end(), [](const std::pair<int, int> &x, const std::pair<int, int> &y) {
    return x.second != y.second ? x.second < y.second : x.first < y.first;
  });
  std::vector<std::pair<int, int>> cols;
  for (auto &p : order) {
    cols.push_back(p);
    cols.push_back({-p.first, -p.second});
  }
  cols.push_back({0, 0});
  col.clear();
  for (size_t i = 0; i < cols.size(); ++i) col[cols[i]] = (int)i;
  // columns per z-pass CTA: even, so that mirror pairs stay together; shared memory bounded
  // for FP64 lines
  int cg = 32;
  while (cg > 2 && (size_t)2 * cg * (N3 + 1) * sizeof(double2) > kSmemCap) cg -= 2;
  s.cg = cg;
  s.ncols = (int)cols.size();
  s.ngroups = (s.ncols + cg - 1) / cg;
  s.ncols_pad = s.ngroups * cg;
  std::vector<int> colpos(s.ncols_pad, -1);
  std::vector<int> xs_all;
  for (int i = 0; i < s.ncols; ++i) {
    const int j1 = md(cols[i].first, N1), j2 = md(cols[i].second, N2);
    colpos[i] = j1 + N1 * j2;
    xs_all.push_back(j1);
  }
  std::sort(xs_all.begin(), xs_all.end());
  xs_all.erase(std::unique(xs_all.begin(), xs_all.end()), xs_all.end());
  s.nxs = (int)xs_all.size();
  // entries grouped by the z-pass CTA that owns both of their columns
  std::vector<std::vector<int4>> per(s.ngroups);
  const int N3p = N3 + 1;
  for (int kk = 0; kk < nh; ++kk) {
    const int n1 = miller_half[3 * kk], n2 = miller_half[3 * kk + 1], n3 = miller_half[3 * kk + 2];
    const int cp = col.at({n1, n2}), cm = col.at({-n1, -n2});
    const int gp_ = cp / cg;
    BSE_REQUIRE(cm / cg == gp_, "internal: mirror columns split across z-pass groups");
    int4 e;
    e.x = kk;
    e.y = (cp % cg) * N3p + md(n3, N3);
    e.z = (cm % cg) * N3p + md(-n3, N3);
    e.w = 0;
    per[gp_].push_back(e);
  }
  std::vector<int4> ent;
  std::vector<int> off{0};
  for (auto &v : per) {
    ent.insert(ent.end(), v.begin(), v.end());
    off.push_back((int)ent.size());
  }
  s.colpos.alloc(colpos.size());
  s.xs.alloc(xs_all.size());
  s.ent.alloc(ent.size());
  s.ent_off.alloc(off.size());
  BSE_CUDA(cudaMemcpy(s.colpos.get(), colpos.data(), colpos.size() * sizeof(int), cudaMemcpyHostToDevice));
  BSE_CUDA(cudaMemcpy(s.xs.get(), xs_all.data(), xs_all.size() * sizeof(int), cudaMemcpyHostToDevice));
  BSE_CUDA(cudaMemcpy(s.ent.get(), ent.data(), ent.size() * sizeof(int4), cudaMemcpyHostToDevice));
  BSE_CUDA(cudaMemcpy(s.ent_off.get(), off.data(), off.size() * sizeof(int), cudaMemcpyHostToDevice));
  s.ok64 = z_smem<double2>(c, s) <= kSmemCap && xy_smem<double2>(c) <= kSmemCap;
  s.ok32 = z_smem<float2>(c, s) <= kSmemCap && xy_smem<float2>(c) <= kSmemCap;
  s.ready = true;
}
}  // namespace

void sphere_fft_init(Ctx &c, const std::vector<int> &miller_half, const std::vector<int> &dens_cols) {
  std::vector<std::pair<int, int>> wcols;
  for (size_t kk = 1; kk < miller_half.size() / 3; ++kk)
    for (int sgn : {1, -1}) wcols.push_back({sgn * miller_half[3 * kk], sgn * miller_half[3 * kk + 1]});
  build_tables(c, c.sfft, wcols, miller_half);
  std::vector<std::pair<int, int>> dcols;
  for (size_t i = 0; i + 1 < dens_cols.size(); i += 2) dcols.push_back({dens_cols[i], dens_cols[i + 1]});
  build_tables(c, c.dfft, dcols, miller_half);
}

template <class R>
bool dens_fft_ok(const Ctx &c) {
  return c.dfft.ready && (sizeof(R) == sizeof(double) ? c.dfft.ok64 : c.dfft.ok32) && !c.sfft.disabled;
}

// forward half of the pair pipeline: packed grids P, or the products of the grids that src names (P unused) ->
// density columns (Coulomb applied, scaled by cscale) and the wave-function-sphere coefficients X (times
// scale) for the PDEP part
template <class R>
void dens_forward(Ctx &c, int np, CT<R> *P, R *X, double scale, const R *vcg, R cscale, const PairGrids<R> &src) {
  using C = CT<R>;
  const int nq = (np + 1) / 2;
  set_attrs<C>();
  Grids<R> &g = c.grids<R>();
  g.colbuf_dens.alloc((size_t)nq * c.N[2] * c.dfft.ncols_pad);
  C *cb = g.colbuf_dens.get();
  if (src.list) launch_xy<C, 3>(c, c.dfft, nq, cb, nullptr, nullptr, src);
  else launch_xy<C, 1>(c, c.dfft, nq, cb, P, nullptr);
  const dim3 grid(c.dfft.ngroups, nq);
  if constexpr (std::is_same<R, double>::value)
    dsph_z_fwd_fx<<<grid, z_threads(c), z_smem<C>(c, c.dfft), c.stream>>>(fz_args(c, c.dfft), np, c.npw, cb, X,
                                                                        PairScale(scale), vcg, cscale);
  else
    dsph_z_fwd<C, R><<<grid, kThreads, z_smem<C>(c, c.dfft), c.stream>>>(make_args<C>(c, c.dfft), np, c.npw, cb, X,
                                                                         scale, vcg, cscale);
  BSE_CHECK_LAUNCH();
}

// inverse half: PDEP back-projection X (times scale) added in the columns, then to the grid P
template <class R>
void dens_inverse(Ctx &c, int np, const R *X, double scale, CT<R> *P) {
  using C = CT<R>;
  const int nq = (np + 1) / 2;
  set_attrs<C>();
  C *cb = c.grids<R>().colbuf_dens.get();
  const dim3 grid(c.dfft.ngroups, nq);
  if constexpr (std::is_same<R, double>::value)
    dsph_z_inv_fx<<<grid, z_threads(c), z_smem<C>(c, c.dfft), c.stream>>>(fz_args(c, c.dfft), np, c.npw, X,
                                                                        PairScale(scale), cb);
  else
    dsph_z_inv<C, R><<<grid, kThreads, z_smem<C>(c, c.dfft), c.stream>>>(make_args<C>(c, c.dfft), np, c.npw, X, scale,
                                                                         cb);
  BSE_CHECK_LAUNCH();
  launch_xy<C, 0>(c, c.dfft, nq, cb, P, nullptr);
}

template bool dens_fft_ok<double>(const Ctx &);
template bool dens_fft_ok<float>(const Ctx &);
template void dens_forward<double>(Ctx &, int, double2 *, double *, double, const double *, double,
                                   const PairGrids<double> &);
template void dens_forward<float>(Ctx &, int, float2 *, float *, double, const float *, float,
                                  const PairGrids<float> &);
template void dens_inverse<double>(Ctx &, int, const double *, double, double2 *);
template void dens_inverse<float>(Ctx &, int, const float *, double, float2 *);

template <class R>
bool sphere_fft_ok(const Ctx &c) {
  return c.sfft.ready && (sizeof(R) == sizeof(double) ? c.sfft.ok64 : c.sfft.ok32) && !c.sfft.disabled;
}

template <class R>
void sphere_to_grid(Ctx &c, int nf, const double *X, CT<R> *P, long double scale, CT<R> *colbuf) {
  using C = CT<R>;
  if (nf <= 0) return;
  const int nq = (nf + 1) / 2;
  set_attrs<C>();
  C *cb = colbuf ? colbuf : colbuf_for<R>(c, nq);
  launch_z_inv<C>(c, nf, nq, X, scale, cb);
  launch_xy<C, 0>(c, c.sfft, nq, cb, P, nullptr);
}

template <class R>
void grid_to_sphere(Ctx &c, int nf, CT<R> *P, double *Y, long double scale, const double *Xd, const double *shift,
                    int period, double shift_const, CT<R> *colbuf) {
  using C = CT<R>;
  if (nf <= 0) return;
  const int nq = (nf + 1) / 2;
  set_attrs<C>();
  C *cb = colbuf ? colbuf : colbuf_for<R>(c, nq);
  launch_xy<C, 1>(c, c.sfft, nq, cb, P, nullptr);
  launch_z_fwd<C>(c, nf, nq, cb, Y, scale, Xd, shift, period > 0 ? period : 1, shift_const);
}

template <class R>
void sphere_h(Ctx &c, int nf, const double *X, double *HX, const double *shift) {
  using C = CT<R>;
  if (nf <= 0) return;
  const int nq = (nf + 1) / 2;
  set_attrs<C>();
  C *cb = colbuf_for<R>(c, nq);
  const long double s_in = 1.0L / std::sqrt((long double)c.omega), s_out = std::sqrt((long double)c.omega) / c.nr;
  launch_z_inv<C>(c, nf, nq, X, s_in, cb);
  launch_xy<C, 2>(c, c.sfft, nq, cb, nullptr, c.grids<R>().vloc.get());
  launch_z_fwd<C>(c, nf, nq, cb, HX, s_out, X, shift, shift ? c.nocc : 1, 0.0);
}

template bool sphere_fft_ok<double>(const Ctx &);
template bool sphere_fft_ok<float>(const Ctx &);
template void sphere_to_grid<double>(Ctx &, int, const double *, double2 *, long double, double2 *);
template void sphere_to_grid<float>(Ctx &, int, const double *, float2 *, long double, float2 *);
template void grid_to_sphere<double>(Ctx &, int, double2 *, double *, long double, const double *, const double *, int,
                                     double, double2 *);
template void grid_to_sphere<float>(Ctx &, int, float2 *, double *, long double, const double *, const double *, int,
                                    double, float2 *);
template void sphere_h<double>(Ctx &, int, const double *, double *, const double *);
template void sphere_h<float>(Ctx &, int, const double *, double *, const double *);

}  // namespace bse
