// Radix-2/3/4/5/8/9 codelets on 64-bit fixed-point complex numbers, for FP64 transforms.
//
// GB300 issues two FP64 operations per clock and SM, 32 integer 32 x 32 + 64 bit multiply-adds and about 45
// 64-bit additions, so a butterfly on 64-bit integers takes a fifth to a tenth of the FP64 pipe's time.
// A block of lines shares one power of two; it is chosen so that the sum of |re| + |im| over any line (or
// over everything that one output can collect) is at most 2^61, which bounds every intermediate value of
// every stage below 2^62: each is a combination of inputs with weights of modulus at most one (sqrt 2
// inside the 8-point codelet).  Additions are exact; a product with a twiddle (62-bit fixed point, two
// 32-bit limbs) rounds at the last bit, 2^-61 of that sum.
#pragma once
#include <cuda_runtime.h>

namespace bse {
namespace fx {

struct __align__(16) C2 {
  long long x, y;
};

struct Axis {
  int n;
  int nstage;
  int radix[12];
  const int4 *tw;  // exp(-2 pi i k/n): cos (hi, lo), sin (hi, lo), hi 2^32 + lo = round(2^62 .), lo signed
};

// limbs of a constant round(2^62 w)
struct W {
  int h, l;
};
__host__ __device__ constexpr W limbs_of(long long w) {
  const int l = (int)(unsigned)(w & 0xffffffffll);
  return W{(int)((w - l) >> 32), l};
}
__device__ __forceinline__ W neg(W w) { return W{-w.h, -w.l}; }
// balanced limbs of a value, |lo| <= 2^31
__device__ __forceinline__ W split(long long v) {
  const int l = (int)v;
  return W{(int)(v >> 32) - (l >> 31), l};
}
// (t 2^64 + m 2^32) / 2^62, rounded
__device__ __forceinline__ long long join(long long t, long long m) { return (t << 2) + (m >> 30); }
constexpr long long kHalf = 1ll << 29;

__device__ __forceinline__ long long mul(W v, W w) {
  const long long m = (long long)v.l * w.h + ((long long)v.h * w.l + kHalf);
  return join((long long)v.h * w.h, m);
}
// a w + b z
__device__ __forceinline__ long long mul2(W a, W w, W b, W z) {
  long long m = (long long)a.h * w.l + kHalf;
  m += (long long)a.l * w.h;
  m += (long long)b.h * z.l;
  m += (long long)b.l * z.h;
  return join((long long)a.h * w.h + (long long)b.h * z.h, m);
}
// v (c + i s)
__device__ __forceinline__ C2 cmul(C2 v, W c, W s) {
  const W x = split(v.x), y = split(v.y);
  return C2{mul2(x, c, y, neg(s)), mul2(x, s, y, c)};
}
__device__ __forceinline__ C2 cscale(C2 v, W w) { return C2{mul(split(v.x), w), mul(split(v.y), w)}; }
__device__ __forceinline__ C2 operator+(C2 a, C2 b) { return C2{a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ C2 operator-(C2 a, C2 b) { return C2{a.x - b.x, a.y - b.y}; }
// a + SG i b
template <int SG>
__device__ __forceinline__ C2 add_i(C2 a, C2 b) {
  return SG > 0 ? C2{a.x - b.y, a.y + b.x} : C2{a.x + b.y, a.y - b.x};
}
__device__ __forceinline__ C2 half(C2 v) { return C2{(v.x + 1) >> 1, (v.y + 1) >> 1}; }

// small DFTs, SG = -1 forward (exp(-2 pi i jk/R)), +1 inverse
template <int SG>
__device__ __forceinline__ void dft3(C2 &v0, C2 &v1, C2 &v2) {
  constexpr W h = limbs_of(3993837246235628775ll);  // sqrt(3)/2
  const C2 t1 = v1 + v2, t2 = v0 - half(t1), t3 = cscale(v1 - v2, h);
  v0 = v0 + t1;
  v1 = add_i<SG>(t2, t3);
  v2 = add_i<-SG>(t2, t3);
}
template <int SG>
__device__ __forceinline__ void dft4(C2 &v0, C2 &v1, C2 &v2, C2 &v3) {
  const C2 t0 = v0 + v2, t1 = v0 - v2, t2 = v1 + v3, t3 = v1 - v3;
  v0 = t0 + t2;
  v2 = t0 - t2;
  v1 = add_i<SG>(t1, t3);
  v3 = add_i<-SG>(t1, t3);
}

template <int R, int SG>
struct Dft;
template <int SG>
struct Dft<2, SG> {
  static __device__ __forceinline__ void run(C2 *v) {
    const C2 a = v[0], b = v[1];
    v[0] = a + b;
    v[1] = a - b;
  }
};
template <int SG>
struct Dft<3, SG> {
  static __device__ __forceinline__ void run(C2 *v) { dft3<SG>(v[0], v[1], v[2]); }
};
template <int SG>
struct Dft<4, SG> {
  static __device__ __forceinline__ void run(C2 *v) { dft4<SG>(v[0], v[1], v[2], v[3]); }
};
template <int SG>
struct Dft<5, SG> {
  static __device__ __forceinline__ void run(C2 *v) {
    // cos and sin of 2 pi/5 and 4 pi/5
    constexpr W c1 = limbs_of(1425089352415399811ll), c2 = limbs_of(-3730932361629093763ll);
    constexpr W s1 = limbs_of(4385974038932618941ll), s2 = limbs_of(2710681029835013083ll);
    constexpr W n1 = limbs_of(-4385974038932618941ll);
    const C2 a = v[0], t1 = v[1] + v[4], t2 = v[2] + v[3], t3 = v[1] - v[4], t4 = v[2] - v[3];
    const W t1x = split(t1.x), t1y = split(t1.y), t2x = split(t2.x), t2y = split(t2.y);
    const W t3x = split(t3.x), t3y = split(t3.y), t4x = split(t4.x), t4y = split(t4.y);
    const C2 p = a + C2{mul2(t1x, c1, t2x, c2), mul2(t1y, c1, t2y, c2)};
    const C2 q = a + C2{mul2(t1x, c2, t2x, c1), mul2(t1y, c2, t2y, c1)};
    const C2 r = C2{mul2(t3x, s1, t4x, s2), mul2(t3y, s1, t4y, s2)};
    const C2 s = C2{mul2(t3x, s2, t4x, n1), mul2(t3y, s2, t4y, n1)};
    v[0] = a + (t1 + t2);
    v[1] = add_i<SG>(p, r);
    v[4] = add_i<-SG>(p, r);
    v[2] = add_i<SG>(q, s);
    v[3] = add_i<-SG>(q, s);
  }
};
// 8 points as 2 x 4: X[2p] from a_n = x_n + x_{n+4}, X[2p+1] from (x_n - x_{n+4}) w^n
template <int SG>
struct Dft<8, SG> {
  static __device__ __forceinline__ void run(C2 *v) {
    constexpr W h = limbs_of(3260954456333195553ll);  // 1/sqrt(2)
    C2 a[4], b[4];
#pragma unroll
    for (int n = 0; n < 4; ++n) {
      a[n] = v[n] + v[n + 4];
      b[n] = v[n] - v[n + 4];
    }
    b[1] = cscale(add_i<SG>(b[1], b[1]), h);                    // (1 + SG i)/sqrt 2
    b[2] = SG > 0 ? C2{-b[2].y, b[2].x} : C2{b[2].y, -b[2].x};  // SG i
    const C2 n3 = C2{-b[3].x, -b[3].y};
    b[3] = cscale(add_i<SG>(n3, b[3]), h);                      // (-1 + SG i)/sqrt 2
    dft4<SG>(a[0], a[1], a[2], a[3]);
    dft4<SG>(b[0], b[1], b[2], b[3]);
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      v[2 * p] = a[p];
      v[2 * p + 1] = b[p];
    }
  }
};
// 9 points as 3 x 3 with twiddles w^(b c), w = exp(SG 2 pi i/9)
template <int SG>
struct Dft<9, SG> {
  static __device__ __forceinline__ void run(C2 *v) {
    constexpr W c1 = limbs_of(3532756447825785444ll), s1 = limbs_of(SG * 2964334632409774423ll);
    constexpr W c2 = limbs_of(800810873071977681ll), s2 = limbs_of(SG * 4541624145405292212ll);
    constexpr W c4 = limbs_of(-4333567320897763126ll), s4 = limbs_of(SG * 1577289512995517789ll);
#pragma unroll
    for (int b = 0; b < 3; ++b) dft3<SG>(v[b], v[3 + b], v[6 + b]);  // v[3 c + b]
    v[4] = cmul(v[4], c1, s1);
    v[7] = cmul(v[7], c2, s2);
    v[5] = cmul(v[5], c2, s2);
    v[8] = cmul(v[8], c4, s4);
#pragma unroll
    for (int c = 0; c < 3; ++c) dft3<SG>(v[3 * c], v[3 * c + 1], v[3 * c + 2]);  // X[c + 3 d] at v[3 c + d]
    C2 t;
    t = v[1], v[1] = v[3], v[3] = t;
    t = v[2], v[2] = v[6], v[6] = t;
    t = v[5], v[5] = v[7], v[7] = t;
  }
};

// one radix-R Stockham butterfly: inputs load((j + r N/R) es), outputs dst[((j/Ns) Ns R + j%Ns + r Ns) es]
template <int R, int SG, class Load>
__device__ __forceinline__ void bfly(const Load &load, C2 *__restrict__ dst, int j, int N, int Ns,
                                     const int4 *__restrict__ tw, int es) {
  const int nb = N / R;
  C2 v[R];
#pragma unroll
  for (int r = 0; r < R; ++r) v[r] = load((j + r * nb) * es);
  int d0 = j * R;
  if (Ns > 1) {
    const int q = j / Ns, kk = j - q * Ns;
    const int step = kk * (N / (Ns * R));  // r * step < N for r < R
#pragma unroll
    for (int r = 1; r < R; ++r) {
      const int4 w = __ldg(&tw[r * step]);
      v[r] = cmul(v[r], W{w.x, w.y}, SG < 0 ? W{w.z, w.w} : W{-w.z, -w.w});
    }
    d0 = q * Ns * R + kk;
  }
  Dft<R, SG>::run(v);
#pragma unroll
  for (int r = 0; r < R; ++r) dst[(d0 + r * Ns) * es] = v[r];
}
template <int SG, class Load>
__device__ __forceinline__ void bfly_any(int R, const Load &load, C2 *__restrict__ dst, int j, int N, int Ns,
                                         const int4 *__restrict__ tw, int es) {
  switch (R) {
    case 8: bfly<8, SG>(load, dst, j, N, Ns, tw, es); break;
    case 9: bfly<9, SG>(load, dst, j, N, Ns, tw, es); break;
    case 4: bfly<4, SG>(load, dst, j, N, Ns, tw, es); break;
    case 2: bfly<2, SG>(load, dst, j, N, Ns, tw, es); break;
    case 3: bfly<3, SG>(load, dst, j, N, Ns, tw, es); break;
    default: bfly<5, SG>(load, dst, j, N, Ns, tw, es); break;
  }
}

// ---- conversions --------------------------------------------------------------------------------
__device__ __forceinline__ unsigned high_abs(double x) { return (unsigned)__double2hiint(x) & 0x7fffffffu; }
// an upper bound of |x| in units of 2^(E - 1043), E the biased exponent of the largest |x| (at most 2^21)
__device__ __forceinline__ unsigned mag(double x, int E) {
  const unsigned h = high_abs(x);
  const int sh = E - (int)(h >> 20);
  return (sh > 20 ? 0u : ((h & 0xfffffu) | 0x100000u) >> sh) + 1u;
}
// round(x 2^(bits - e)), |x| < 2^e
__device__ __forceinline__ long long from_double(double x, int e, int bits) {
  const long long b = __double_as_longlong(x);
  const int E = (int)((b >> 52) & 0x7ff);
  unsigned long long m = (unsigned long long)b & 0xfffffffffffffull;
  if (E) m |= 1ull << 52;
  const int s = max(E, 1) - 1075 + bits - e;
  const int l = min(max(s, 0), 10), r = min(max(-s, 0), 63);
  m = ((m << l) + ((1ull << r) >> 1)) >> r;
  return b < 0 ? -(long long)m : (long long)m;
}
// v 2^q with -1021 <= q <= 960 by integer arithmetic (the conversion instruction runs at the FP64 rate)
__device__ __forceinline__ double to_double(long long v, int q) {
  unsigned long long a = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
  const int z = __clzll((long long)a);
  a <<= z & 63;
  const unsigned long long m = (a >> 11) + ((a >> 10) & 1);
  unsigned long long bits = ((unsigned long long)(1085 - z + q) << 52) + m;
  bits |= (unsigned long long)v & 0x8000000000000000ull;
  return v == 0 ? 0.0 : __longlong_as_double((long long)bits);
}
// Bound of one line of n elements, by a whole warp: the smallest e (to one part in 2^20) with
// sum |re| + |im| < 2^e; kBadLine when an element is not finite
constexpr int kBadLine = 1 << 20;
template <class Get>
__device__ __forceinline__ int line_exponent(int n, const Get &get) {
  const int lane = threadIdx.x & 31;
  unsigned m = 0, s = 0;
  for (int i = lane; i < n; i += 32) {
    const double2 u = get(i);
    m = max(m, max(high_abs(u.x), high_abs(u.y)));
  }
  const int E = (int)(__reduce_max_sync(0xffffffffu, m) >> 20);
  for (int i = lane; i < n; i += 32) {
    const double2 u = get(i);
    s += mag(u.x, E) + mag(u.y, E);
  }
  s = __reduce_add_sync(0xffffffffu, s);
  return E >= 0x7ff ? kBadLine : E - 1043 + 32 - __clz(s);
}
// the unit 2^q of a block and whether it can be converted by to_double; bad: the block holds a NaN or infinity
struct Unit {
  int q;
  bool bad;
  __device__ __forceinline__ double operator()(long long v) const {
    if (bad) return __longlong_as_double(0x7ff8000000000000ll);
    return q >= -1021 && q <= 960 ? to_double(v, q) : ldexp((double)v, q);
  }
};

}  // namespace fx
}  // namespace bse
