// pft_tc64.cuh -- the FP64 convolutions of the separable march on the tensor cores
// (pft_tcgen05.cuh): tiles of 128 lines times the circulant matrix of the axis.
//
// Both factors carry FP64 accuracy as sums of small integers, every one exact in FP16, because
// GB300 does 2 FP64 multiply-adds a cycle and SM and 4096 FP16 ones on the tensor core.
//   X: line by line scaled to 2^54 / S with S the power of two above the line's largest value,
//      rounded to an integer and cut into six digits of 9 bits, X = sum_i X_i 2^(9 (5 - i)),
//      |X_0| <= 2^9, |X_i| <= 2^8: the rounding is 2^-55 of S, below an FP64 rounding of the
//      largest value.
//   K: kern 2^p = sum_j K_j 2^(-9 j), j = 0..6, |K_j| < 2^11 (K_0: sum |K_0| <= 2^13).  The
//      rounding of every K_j is chosen so that the sum of K_0 is 2^p and the sum of every other
//      K_j is zero: what the products left out below do to the mean of a line vanishes.
// Level l collects the products X_i K_j with i + j = l in one FP32 accumulator of the tensor
// core: integers, exact in any order of addition while their sums stay below 2^24.  Whatever the
// digits, that holds up to 64 points on levels 0 to 4, at 128 points on levels 0 to 2 and at 96,
// for kernels narrower than half the box, on 0 to 3.  Beyond it is not a bound: were every digit to
// line up with the kernel's signs, level 3 would reach 1.5 and level 5 2.2 times 2^24 (kernels of
// 0.02 to 400 grid cells), and an addition would round by two units, 2^-48 of S on level 3, 2^-57 on
// 4.  Digits without that order reach 0.3.  Level 5 holds X_0 K_6 too, K_6 stored 2^-9 smaller (an error of the kernel acts at
// every step, and its seventh digit keeps that below 1e-18 a step): fractions, rounded below 2^-60
// of S.  Levels 0 to 5 (22 products) are added up in 64-bit integers; the other products of
// level 6 are 2^-57 of S.  The sum is rounded once, to FP64.  Propagator slices against the FP64
// oracle: 2e-16 to 8e-16 relative (the FFT pair in FP64: the same or larger; the products with
// the Boltzmann factors set it).  128^3, Ns 100, phi against an extended-precision march: 2.3e-16, the
// FFT march 2.3e-15 (an FP64 reference whose diffusion factor is one rounded exponential is itself
// 1.6e-14 off).
//
// One CTA holds one tile: G warpgroups of 128 threads (thread = line) and one more warp that
// issues the products, level by level into a ring of NB accumulators, while the warpgroups
// read the levels before.  A line with an infinity or a NaN becomes NaN, as under the FFT.
//
// What bounds it: the chain of a tile's phases, which follow one another on 17 warps with one tile an
// SM; no pipe is full (ncu, real fields, y kernel / fused x kernel: integer pipe 37 / 32 %, tensor
// pipe 16 / 13 %, FP64 pipe 0 / 19 % at 64 points; 33 / 25, 28 / 21 and 0 / 15 % at 128, where the
// fused kernels also wait for their instructions).  A 64-point tile of 128 lines takes 15,000 cycles
// without and 37,000 with the Boltzmann products: 3,800 for the products of a convolution (2,800
// at the tensor core's rate), 4,400 for the digits, 4,200 for each conversion back, 8,200 for two
// FP64 multiplications by B, 2,000 each to load and to store.  The FFT pair needs about 26 FP64
// operations a point and convolution, 13 cycles an SM, this 1.8 to 4.  At 128 points the 17 warps'
// cap of 96 registers costs spills too (ptxas, bytes stored a thread: 648 in the fused z kernel, 628
// in x, 88 in y; complex fields 276, 236, 88; at most 120 at 96 points and 12 at 64).
// Measured, one field update with fields in and out, FFT pair -> this (ms): 32^3 real, Ns 64, 2.49 ->
// 1.33; 64^3 real, Ns 100, 6.59 -> 3.41, complex 12.26 -> 5.05; 128^3 real 50.9 -> 13.6, complex
// 104.3 -> 37.3.
// Tried: fields and factors in fixed point between the launches, one scale a slice (128^3 real 10.7
// ms, 64^3 complex 3.3): lines and factors far below the slice's largest lose digits there, and
// so does the block junction where the two blocks' largest factors lie apart (W- noise of 25, six
// steps, W+ shifted by 200: 1e-9 of a slice, 1e-4 of phi); left out.
// Tried: skipping the k steps where a digit of the kernel is zero (128 points: 26,000 -> 29,000
// cycles, the branches cost more than a quarter of the products); the smallest level first (saves
// two operations a point, but its eight products delay the first reading: 3,800 -> 5,100 cycles);
// a reading warpgroup's warp issuing the products (3,800 -> 4,700).
#pragma once
#include <type_traits>

#include "pft_tcgen05.cuh"

namespace pft {

constexpr int kTc64Head = 16;  // bytes of a table's header
// outputs a product computes: the axis, at 128 points half of it
constexpr int tc64_chunk(int n) { return n <= 96 ? n : 64; }
template <int N> struct Tc64Cfg {
  static constexpr int NS = 6;  // digits
  static constexpr int PPT = N <= 64 ? 16 : 32;
  static constexpr int G = N / PPT;
  static constexpr int WORK = 128 * G;
  static constexpr int THREADS = WORK + 32;
  static constexpr int CW = tc64_chunk(N);
  static constexpr int NCH = N / CW;
  static constexpr int CPW = CW / PPT;
  static constexpr int NB = N <= 64 ? 4 : 2;
  static constexpr int COLS_USED = NS * N / 2 + NB * CW;
  static constexpr int COLS = COLS_USED <= 128 ? 128 : (COLS_USED <= 256 ? 256 : 512);
  static constexpr int NSLOT = 2 * (N / 8) - 1;
  static constexpr int TAB = kTc64Head + (NS + 1) * NSLOT * 128;
  static_assert(N % PPT == 0 && N % CW == 0 && CW % PPT == 0 && COLS_USED <= 512, "whole chunks in tensor memory");
};
inline bool tc64_axis_ok(int n) { return n == 16 || n == 32 || n == 48 || n == 64 || n == 96 || n == 128; }
inline size_t tc64_table_bytes(int n) { return kTc64Head + (size_t)7 * (2 * (n / 8) - 1) * 128; }

// Host arithmetic of the table: the unevaluated sum of two doubles (Knuth's TwoSum, FMA product),
// the same on every host whatever its long double is.
struct Dd64 {
  double h, l;
};
inline Dd64 dd64_sum(double a, double b) {
  const double s = a + b, t = s - a;
  return {s, (a - (s - t)) + (b - t)};
}
inline Dd64 dd64_add(Dd64 a, Dd64 b) {
  const Dd64 s = dd64_sum(a.h, b.h);
  return dd64_sum(s.h, s.l + (a.l + b.l));
}
inline Dd64 dd64_mul(Dd64 a, Dd64 b) {
  const double p = a.h * b.h;
  return dd64_sum(p, fma(a.h, b.h, -p) + (a.h * b.l + a.l * b.h));
}
inline Dd64 dd64_from(long double x) {
  const double h = (double)x;
  return {h, (double)(x - (long double)h)};
}

// cos(2 pi j / n), j = 0 .. n-1, made once a length: long double is software on aarch64.
inline std::vector<Dd64> tc64_make_cosines(int n) {
  const int h = n / 2;
  std::vector<Dd64> cs((size_t)n);
  for (int j = 0; j <= n / 4; j++) {  // n is a multiple of 4; the other quarters by symmetry
    const Dd64 c = dd64_from(cosl(2.0L * 3.14159265358979323846264338327950288L * j / n));
    cs[j] = c;
    cs[h - j] = {-c.h, -c.l};
    cs[h + j] = {-c.h, -c.l};
    if (j) cs[n - j] = c;
  }
  return cs;
}
inline const std::vector<Dd64>& tc64_cosines(int n) {
  static const std::vector<Dd64> c16 = tc64_make_cosines(16), c32 = tc64_make_cosines(32), c48 = tc64_make_cosines(48),
                                 c64 = tc64_make_cosines(64), c96 = tc64_make_cosines(96), c128 = tc64_make_cosines(128);
  switch (n) {
    case 16: return c16;
    case 32: return c32;
    case 48: return c48;
    case 64: return c64;
    case 96: return c96;
    default: return c128;
  }
}

// The table of one axis: the header {int p}, then the blocks of K_0 .. K_6: block s
// of a digit holds kern[(8 (s - n/8 + 1) + r - e) mod n] at row r, element e.  d: the axis' factors exp(-k_a^2 ds) at k = 0 .. n/2.
inline void tc64_build_table(int n, const long double* d, unsigned char* dst) {
  const int h = n / 2;
  const std::vector<Dd64>& cs = tc64_cosines(n);
  auto mult = [&](int j) { return (j && j < n - j) ? 2 : 1; };
  // (k outside: the sums of the j are independent of one another, a chain of additions each)
  std::vector<Dd64> r((size_t)h + 1, Dd64{0.0, 0.0});
  for (int k = 0; k <= h; k++) {
    const Dd64 f = dd64_from(d[k] * (mult(k) / (long double)n));
    for (int j = 0, i = 0; j <= h; j++) {
      r[j] = dd64_add(r[j], dd64_mul(f, cs[(size_t)i]));
      i += k;
      if (i >= n) i -= n;
    }
  }
  double kmax = 0.0, ksum = 0.0;
  for (int j = 0; j <= h; j++) {
    kmax = std::max(kmax, fabs(r[j].h));
    ksum += mult(j) * fabs(r[j].h);
  }
  // |K_0| <= 2^11 - 2 (exact in FP16 after the correction of its sum), sum |K_0| <= 2^13
  int p = 13;
  while (p > 0 && (kmax * ldexp(1.0, p) > 2046.0 || ksum * ldexp(1.0, p) > 8192.0 + 1e-3)) p--;
  for (int j = 0; j <= h; j++) r[j] = {ldexp(r[j].h, p), ldexp(r[j].l, p)};
  memset(dst, 0, kTc64Head);
  memcpy(dst, &p, sizeof(p));
  const int nslot = 2 * (n / 8) - 1;
  std::vector<double> q((size_t)h + 1);
  std::vector<__half> q16((size_t)3 * n);  // the digit at distance j, over three periods
  __half* out = reinterpret_cast<__half*>(dst + kTc64Head);
  for (int sl = 0; sl < 7; sl++) {
    long long sum = 0;
    for (int j = 0; j <= h; j++) {
      q[j] = rint(r[j].h);
      sum += mult(j) * (long long)q[j];
    }
    long long off = (sl == 0 ? (1LL << p) : 0LL) - sum;  // to be added to the digits
    while (off != 0) {  // the value whose rounding went furthest the other way takes a unit
      const int dir = off > 0 ? 1 : -1;
      const bool odd = (off & 1) != 0;
      int b = -1;
      double best = -1e300;
      for (int j = 0; j <= h; j++) {
        if (odd != (mult(j) == 1)) continue;
        const double gain = dir * ((r[j].h - q[j]) + r[j].l);
        if (gain > best) {
          best = gain;
          b = j;
        }
      }
      q[b] += dir;
      off -= (long long)dir * mult(b);
    }
    for (int j = 0; j < n; j++) {
      const __half v = __float2half_rn((float)(q[j <= h ? j : n - j] * (sl == 6 ? 1.0 / 512.0 : 1.0)));
      q16[j] = q16[j + n] = q16[j + 2 * n] = v;
    }
    for (int b = 0; b < nslot; b++)
      for (int row = 0; row < 8; row++)
        for (int e = 0; e < 8; e++) *out++ = q16[(size_t)(n + 8 * (b - n / 8 + 1) + row - e)];
    for (int j = 0; j <= h; j++) {  // exact: the remainders of a rounding, times 2^9
      const Dd64 t = dd64_sum(r[j].h - q[j], r[j].l);
      r[j] = {t.h * 512.0, t.l * 512.0};
    }
  }
}

// z lines: staging rows of a warp, 16 bytes of padding a row
template <int N, int KIND> struct Tc64Z {
  static constexpr int PPT = Tc64Cfg<N>::PPT;
  static constexpr int PITCH = KIND ? 2 * PPT + 2 : PPT + 2;  // doubles
  static constexpr int ROWS = KIND ? 16 : 32;
  static constexpr int WARP_DOUBLES = ROWS * PITCH;
  static constexpr size_t BYTES = (size_t)(Tc64Cfg<N>::WORK / 32) * WARP_DOUBLES * sizeof(double);
};
template <int N, int KIND, int PW, int AX> constexpr size_t tc64_smem() {
  return tc_align(Tc64Cfg<N>::TAB) + Tc64Cfg<N>::WORK * sizeof(int) + 128 +
         (AX == 2 ? Tc64Z<N, KIND>::BYTES : (PW == 2 ? (size_t)N * 128 * sizeof(double) : 0));
}

// Tensor-core sums t as FP64, t 2^(eb - 1085) rounded to nearest, on the integer pipe (the FP64
// pipe converts 2 a cycle and SM): normalised by a shift, rounded by adding the bit below the last
// one kept (the carry runs into the exponent).  eb keeps the exponent in range.  A few at a time: a
// group with a value below 2^32 (2^-30 of the scale), whose upper word is empty, takes the FP64 pipe.
template <int K>
__device__ __forceinline__ void tc64_to_double(const long long (&t)[K], int eb, double (&y)[K]) {
  unsigned least = 0xffffffffu;
#pragma unroll
  for (int i = 0; i < K; i++) {
    const unsigned sg = (unsigned)((int)(t[i] >> 32) >> 31);
    // one's complement of a negative value: 1 less in the last of 62 bits
    const unsigned h = (unsigned)(t[i] >> 32) ^ sg, l = (unsigned)t[i] ^ sg;
    least = min(least, h);
    const int lz = __clz((int)h);
    const unsigned hn = __funnelshift_l(l, h, lz), ln = l << (lz & 31);
    const unsigned L = __funnelshift_r(ln, hn, 11);
    const unsigned H = (hn >> 11) + (unsigned)(eb - lz) * 0x100000u;
    const unsigned long long r = (((unsigned long long)H << 32) | L) + ((ln >> 10) & 1u);
    y[i] = __hiloint2double((int)((unsigned)(r >> 32) | (sg & 0x80000000u)), (int)(unsigned)r);
  }
  if (__any_sync(0xffffffffu, least == 0u)) {
    const double sc = __hiloint2double((eb - 62) << 20, 0);
#pragma unroll
    for (int i = 0; i < K; i++) y[i] = (double)t[i] * sc;
  }
}
// FP64 in the digits' form: X, the integer nearest x in units of 2^(eL - 1076) (eL the biased
// exponent of the line's largest value, at least 1), plus the digits' biases, above 8 bits of no
// meaning: digit i of X plus its bias is at bit 8 + 9 (5 - i).  The biases, 256 (512 for the leading
// digit), make all digits non-negative.  Ties go to even: values of a few bits below the unit meet
// them half of the time, and a fixed direction would shift every step's mean.  Lines down to
// the smallest subnormal keep their digits (0.3 to 1.4 % of a march for the two operations; a
// branch that lifts small lines cost 1 to 3 %).
constexpr unsigned long long kTc64Bias =
    256ull * (1ull + (1ull << 9) + (1ull << 18) + (1ull << 27) + (1ull << 36)) + (512ull << 45);
__device__ __forceinline__ unsigned long long tc64_digits(double x, int eL) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  // subnormals and zeros: no leading one, and the exponent of the smallest normal value
  const unsigned ha = hi & 0x7fffffffu;
  const int sh = eL + 2 - (int)(max(ha, 0x100000u) >> 20);  // 2 and more
  const unsigned mh = __funnelshift_l(lo, min(ha, (hi & 0xfffffu) | 0x100000u), 11), ml = lo << 11;  // leading bit 63
  const bool far = sh >= 32;
  const unsigned a = far ? mh : ml, b = far ? 0u : mh;
  const int s5 = far ? sh - 32 : sh;
  const unsigned wl = __funnelshift_rc(a, b, s5), wh = s5 >= 32 ? 0u : b >> s5;
  const unsigned sg = (unsigned)((int)hi >> 31);
  const unsigned long long v = (((unsigned long long)(wh ^ sg) << 32) | (wl ^ sg)) - (((unsigned long long)sg << 32) | sg);
  return v + ((kTc64Bias << 8) + 127ull) + (((unsigned)v >> 8) & 1u);
}

// Digit `dgt` (0 the leading one) of two biased integers as a pair of FP16: two bytes of each
// that hold it, shifted and masked, as the mantissa of 1024 + digit, then exactly minus
// (1024 + bias).
template <int dgt> __device__ __forceinline__ uint32_t tc64_digit_pair(unsigned lo0, unsigned hi0, unsigned lo1, unsigned hi1) {
  unsigned pk;
  if (dgt == 5) pk = __byte_perm(lo0, lo1, 0x6521);
  else if (dgt == 4) pk = __byte_perm(lo0, lo1, 0x7632) >> 1;
  else if (dgt == 3) pk = __byte_perm(__funnelshift_r(lo0, hi0, 26), __funnelshift_r(lo1, hi1, 26), 0x5410);
  else if (dgt == 2) pk = __byte_perm(hi0, hi1, 0x5410) >> 3;
  else if (dgt == 1) pk = __byte_perm(hi0, hi1, 0x6521) >> 4;
  else pk = __byte_perm(hi0, hi1, 0x7632) >> 5;
  const unsigned hb = dgt == 0 ? (pk & 0x07ff07ffu) + 0x64006400u : ((pk & 0x01ff01ffu) | 0x64006400u);
  const __half2 hv = __hsub2(*reinterpret_cast<const __half2*>(&hb),
                             __half2half2(__ushort_as_half(dgt == 0 ? 0x6600 : 0x6500)));
  return *reinterpret_cast<const uint32_t*>(&hv);
}

// The tile's lines, by the warpgroups that hold them (every thread but the issuing warp's).
template <int N, int KIND, int PW, int AX>
__device__ __forceinline__ void tc64_lines(const BatchStep& s, int nlines, int cin, int s_outer, int s_k, int* err,
                                           unsigned char* smraw, int tid, int warp, bool more) {
  using CF = Tc64Cfg<N>;
  constexpr int G = CF::G, PPT = CF::PPT, CW = CF::CW, NCH = CF::NCH, CPW = CF::CPW, NB = CF::NB, NS = CF::NS;
  constexpr uint32_t DCOL = NS * N / 2;  // first accumulator column
  constexpr int GS = 4;                  // points converted to FP64 at a time
  int* lexp = reinterpret_cast<int*>(smraw + tc_align(CF::TAB));
  uint64_t* full = reinterpret_cast<uint64_t*>(lexp + CF::WORK);
  uint64_t* empty = full + NCH * NB;
  uint64_t* done = empty + NB;
  uint32_t* tbase = reinterpret_cast<uint32_t*>(done + 1);
  const int lane = tid & 31;
  const int g = warp >> 2, m = tid & 127;
  const int col = blockIdx.x * 128 + m;
  const bool valid = col < nlines;
  const int colc = valid ? col : 0;
  double* F = reinterpret_cast<double*>(s.spec);
  const double* B = reinterpret_cast<const double*>(s.B);
  const double* Bn = reinterpret_cast<const double*>(s.Bnext);
  const bool same = (s.Bnext == s.B);
  int base, step;
  if (AX != 2) {
    base = (colc / cin) * s_outer + (colc % cin) + g * PPT * s_k;
    step = s_k;
  } else if (KIND == 0) {
    base = colc * N + g * PPT;
    step = 1;
  } else {
    base = (colc >> 1) * (2 * N) + 2 * g * PPT + (colc & 1);
    step = 2;
  }
  using ZS = Tc64Z<N, KIND>;
  double* area = reinterpret_cast<double*>(smraw + tc_align(CF::TAB) + CF::WORK * sizeof(int) + 128);
  double* zs = area + (AX == 2 ? warp * ZS::WARP_DOUBLES : 0);
  const int row0 = blockIdx.x * 128 + (m & ~31);
  double* zrow = KIND ? zs + (lane >> 1) * ZS::PITCH + (lane & 1) : zs + lane * ZS::PITCH;
  // rows of the warp into and out of shared memory in 16-byte pieces
  constexpr int CPR = KIND ? PPT : PPT / 2;
  auto zglob = [&](int r, int c2) -> long long {  // offset of piece c2 of row r
    return KIND ? ((long long)(row0 >> 1) + r) * (2 * N) + 2 * (g * PPT + c2)
                : (long long)(row0 + r) * N + g * PPT + 2 * c2;
  };
  auto zin = [&](const double* src) {
#pragma unroll 4
    for (int i = lane; i < ZS::ROWS * CPR; i += 32) {
      const int r = i / CPR, c2 = i % CPR;
      if (row0 + (KIND ? 2 * r : r) < nlines)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(zs + r * ZS::PITCH + 2 * c2)),
                     "l"(src + zglob(r, c2))
                     : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  auto zwait = [&]() {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncwarp();
  };
  auto zout = [&](double* dst) {
    __syncwarp();
#pragma unroll 4
    for (int i = lane; i < ZS::ROWS * CPR; i += 32) {
      const int r = i / CPR, c2 = i % CPR;
      if (row0 + (KIND ? 2 * r : r) < nlines)
        *reinterpret_cast<double2*>(dst + zglob(r, c2)) = *reinterpret_cast<const double2*>(zs + r * ZS::PITCH + 2 * c2);
    }
    __syncwarp();
  };
  auto zat = [&](int i) -> double& { return zrow[KIND ? 2 * i : i]; };
  auto mulB = [&](double x, double b) -> double {
    if constexpr (KIND == 0) {
      return x * b;
    } else {
      const double bo = __shfl_xor_sync(0xffffffffu, b, 1), xo = __shfl_xor_sync(0xffffffffu, x, 1);
      return (lane & 1) ? x * bo + xo * b : x * b - xo * bo;
    }
  };

  double v[PPT];
  if constexpr (AX == 2) {
    zin(PW == 1 ? reinterpret_cast<const double*>(s.in) : F);
    zwait();
#pragma unroll
    for (int i = 0; i < PPT; i++) v[i] = valid ? zat(i) : 0.0;
    if constexpr (PW == 1) {
      __syncwarp();
      zin(B);
      zwait();
#pragma unroll
      for (int i = 0; i < PPT; i++) v[i] = mulB(v[i], valid ? zat(i) : 0.0);
      __syncwarp();
    }
  } else {
    const double* fp = F + base;
#pragma unroll
    for (int i = 0; i < PPT; i++) {
      v[i] = *fp;
      fp += step;
    }
    if constexpr (PW == 2) {  // B_s of the tile, rows of 128 consecutive doubles
      for (int i = tid; i < N * 64; i += CF::WORK) {
        const int r = i >> 6, c2 = (i & 63) * 2;
        if ((int)blockIdx.x * 128 + c2 < nlines)
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(area + r * 128 + c2)),
                       "l"(B + (long long)r * s_k + blockIdx.x * 128 + c2)
                       : "memory");
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tm = __shfl_sync(0xffffffffu, *tbase, 0);
  const uint32_t tlane = tm + ((uint32_t)(warp & 3) << 21);
  const int p = *reinterpret_cast<const int*>(smraw);
  const int ch = g / CPW;       // this warpgroup's chunk
  // how often before: the chunk's barrier full[ch][l % NB] at its level l
  auto full_use = [](int turn, int l) -> unsigned {
    return (unsigned)(turn * ((NS - l % NB + NB - 1) / NB) + l / NB);
  };
  int ebase = 0;
  bool odd = false;
  double sc1 = 1.0, sc2 = 1.0;
  // conversions back to FP64 of values below 2^(eL - 1022): results near either end of the range
  // are scaled in two parts
  auto set_range = [&](int eL, bool bad) {
    odd = bad || eL < 300 || eL > 1900;
    const int eC = odd ? 1000 : eL;
    ebase = eC - 47 - p + 62;
    if (odd) {
      const int d = max(-2000, min(eL - 1000, 2000));
      sc1 = __hiloint2double((1023 + d / 2) << 20, 0);
      sc2 = bad ? __hiloint2double(0x7fffffff, -1) : __hiloint2double((1023 + d - d / 2) << 20, 0);
    }
  };

  // X into tensor memory
  auto split = [&](int turn) {
    unsigned mx = 0;
#pragma unroll
    for (int i = 0; i < PPT; i++) mx = max(mx, (unsigned)__double2hiint(v[i]) & 0x7fffffffu);
    lexp[g * 128 + m] = (int)(mx >> 20);
    if (turn) {  // every product of the convolution before has read X
      mbar_wait(done, 0, err, 1);
      tc_fence_after();
    }
    named_sync(2, CF::WORK);
    int eL = 0;
#pragma unroll
    for (int w = 0; w < G; w++) eL = max(eL, lexp[w * 128 + m]);
    const bool bad = eL == 0x7ff;  // an infinity or a NaN: the line becomes NaN
    eL = max(eL, 1);  // (subnormal lines: their unit is a subnormal's)
    set_range(eL, bad);
#pragma unroll
    for (int j = 0; j < PPT / 8; j++) {
      unsigned lo[8], hi[8];
#pragma unroll
      for (int i = 0; i < 8; i++) {
        const unsigned long long y = tc64_digits(v[8 * j + i], eL);
        lo[i] = (unsigned)y;
        hi[i] = (unsigned)(y >> 32);
      }
      auto put = [&](auto dg) {
        constexpr int dgt = decltype(dg)::value;
        uint32_t w[4];
#pragma unroll
        for (int i = 0; i < 4; i++) w[i] = tc64_digit_pair<dgt>(lo[2 * i], hi[2 * i], lo[2 * i + 1], hi[2 * i + 1]);
        // the two halves of each 16 points swapped
        tc_st4(tlane + (uint32_t)(dgt * (N / 2) + g * (PPT / 2) + 4 * (j ^ 1)), w);
      };
      put(std::integral_constant<int, 0>{});
      put(std::integral_constant<int, 1>{});
      put(std::integral_constant<int, 2>{});
      put(std::integral_constant<int, 3>{});
      put(std::integral_constant<int, 4>{});
      put(std::integral_constant<int, 5>{});
    }
    tc_wait_st();
    tc_fence_before();
    asm volatile("bar.arrive 1, %0;" ::"r"(CF::THREADS) : "memory");
  };

  const uint32_t dacc = tlane + DCOL + (uint32_t)((g % CPW) * PPT);
  long long acc[PPT];
  // the levels of this warpgroup's chunk, added up in units of 2^-39 of level 0's (level 0 first:
  // its products are the fewest, so that the reading starts early; a 64-bit multiply-add takes
  // the place of a sign extension and a 64-bit addition on the busier pipe)
  int one = 1;
  asm volatile("" : "+r"(one));
  auto collect = [&](int turn) {
#pragma unroll
    for (int l = 0; l < NS; l++) {
      const int b = l % NB;  // the accumulator of job ch NS + l of this turn
      mbar_wait(full + ch * NB + b, full_use(turn, l) & 1u, err, 1);
      tc_fence_after();
#pragma unroll
      for (int j = 0; j < PPT / 8; j++) {
        uint32_t r[8];
        tc_ld8(dacc + (uint32_t)(b * CW) + 8 * j, r);
        tc_wait_ld();
#pragma unroll
        for (int i = 0; i < 8; i++) {
          const float f = __uint_as_float(r[i]);
          const int d = __float2int_rn(l == 5 ? f * 0.015625f : f);
          long long& a = acc[8 * j + i];
          if (l == 0) a = (long long)((unsigned long long)(unsigned)(d * 128) << 32);
          else a += (long long)d * (l == 1 ? (1 << 30) : (l == 2 ? (1 << 21) : (l == 3 ? (1 << 12) : (l == 4 ? (1 << 3) : one))));
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0)
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(empty + b)) : "memory");
    }
  };
  // the convolution's values into v, unit 2^(eL + 1 - 1023) 2^-9 2^-p 2^-39
  auto finish = [&]() {
#pragma unroll
    for (int j = 0; j < PPT / GS; j++) {
      long long t[GS];
      double y[GS];
#pragma unroll
      for (int i = 0; i < GS; i++) t[i] = acc[GS * j + i];
      tc64_to_double(t, ebase, y);
#pragma unroll
      for (int i = 0; i < GS; i++) v[GS * j + i] = y[i];
    }
    if (odd) {
#pragma unroll 1
      for (int k = 0; k < PPT; k += 8) {
#pragma unroll
        for (int i = 0; i < PPT; i++)
          if (i / 8 == k / 8) v[i] = v[i] * sc1 * sc2;
      }
    }
  };

  split(0);
  if constexpr (PW == 2) {
    double* q = reinterpret_cast<double*>(s.out);
    if constexpr (AX == 2) {
      __syncwarp();
      zin(B);
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      named_sync(2, CF::WORK);  // every thread's pieces of the tile have landed
    }
    collect(0);
    if constexpr (AX == 2) zwait();
    const double* bt = area + (g * PPT) * 128 + m;
    double* qp = q + base;
    finish();
#pragma unroll
    for (int k = 0; k < PPT; k++) {
      double bk;
      if constexpr (AX == 2) bk = valid ? zat(k) : 0.0;
      else bk = bt[k * 128];
      const double x = mulB(v[k], bk);
      if constexpr (AX == 2) zat(k) = x;
      else if (valid) *qp = x;
      qp += step;
      v[k] = same ? mulB(x, bk) : x;
    }
    if constexpr (AX == 2) zout(q);
    if (more) {
      if (!same) {
        const double* bp = Bn + base;
#pragma unroll
        for (int k = 0; k < PPT; k++) {
          v[k] = mulB(v[k], valid ? *bp : 0.0);
          bp += step;
        }
      }
      split(1);
      collect(1);
    }
  } else {
    collect(0);
  }
  if (PW != 2 || more) {
    double* fo = F + base;
    finish();
#pragma unroll
    for (int k = 0; k < PPT; k++) {
      if constexpr (AX == 2) zat(k) = v[k];
      else if (valid) *fo = v[k];
      fo += step;
    }
    if constexpr (AX == 2) zout(F);
  }
  tc_fence_before();
  __syncthreads();
}

// AX 0, 1: lines along x or y; line c of the nlines starts at (c / cin) s_outer + c % cin doubles
// and its points lie s_k apart (complex fields: real and imaginary parts are lines of their own,
// in neighbouring threads).  AX 2: lines along z, nlines rows of N points (complex fields: two
// rows a pencil), staged in shared memory warp by warp.
// PW 0: the convolution; PW 1: x B_1 on q_0 = st.in, convolution; PW 2: convolution, x B_s,
// store q_s, then (if st.Bnext) x B_{s+1}, convolution.
template <int N, int KIND, int PW, int AX>
__global__ void __launch_bounds__(Tc64Cfg<N>::THREADS, 1)
kb_tc64_line(const BatchStep* __restrict__ st, int nlines, int cin, int s_outer, int s_k, int* err) {
  using CF = Tc64Cfg<N>;
  constexpr int G = CF::G, CW = CF::CW, NCH = CF::NCH, CPW = CF::CPW, NB = CF::NB, NS = CF::NS;
  constexpr uint32_t DCOL = NS * N / 2;  // first accumulator column
  const BatchStep& s = st[blockIdx.y];
  extern __shared__ __align__(16) unsigned char smraw[];
  int* lexp = reinterpret_cast<int*>(smraw + tc_align(CF::TAB));
  uint64_t* full = reinterpret_cast<uint64_t*>(lexp + CF::WORK);
  uint64_t* empty = full + NCH * NB;  // full: one set a chunk, so that its readers meet every phase
  uint64_t* done = empty + NB;
  uint32_t* tbase = reinterpret_cast<uint32_t*>(done + 1);
  static_assert(NCH == 1 || NS % NB == 0, "a chunk's levels use every accumulator equally often");
  const int tid = threadIdx.x;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // uniform
  const bool more = PW == 2 && s.Bnext != nullptr;

  // ---- table, barriers, tensor memory
  {
    const uint4* t4 = reinterpret_cast<const uint4*>(reinterpret_cast<const char*>(s.d[AX]) + tc_align(N * sizeof(double)));
    uint4* d4 = reinterpret_cast<uint4*>(smraw);
    for (int i = tid; i < CF::TAB / 16; i += CF::THREADS) d4[i] = t4[i];
  }
  if (tid == 0) {
#pragma unroll
    for (int i = 0; i < NCH * NB; i++) mbar_init(full + i, 1);
#pragma unroll
    for (int i = 0; i < NB; i++) mbar_init(empty + i, 4 * CPW);
    mbar_init(done, 1);
    mbar_init_fence();
  }
  if (warp == 4 * G) tc_alloc(tbase, CF::COLS);
  fence_proxy_async_smem();
  constexpr int NJ = NCH * NS;  // jobs a turn: (chunk, level) in order, job t in accumulator t % NB

  if (warp == 4 * G) {
    // ================================================= the issuing warp
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tm = __shfl_sync(0xffffffffu, *tbase, 0);
    const uint64_t k0 = tc_desc(smem_addr(smraw) + kTc64Head);
    for (int turn = 0; turn < (more ? 2 : 1); turn++) {
      named_sync(1, CF::THREADS);  // X is in tensor memory
      tc_fence_after();
      for (int ch = 0; ch < NCH; ch++) {
        for (int l = 0; l < NS; l++) {
          const int t = ch * NS + l, b = t % NB;
          if (t >= NB) {  // job t - NB has been read: it was use t / NB - 1 of this turn's
            mbar_wait(empty + b, (unsigned)(turn * ((NJ - b + NB - 1) / NB) + t / NB - 1) & 1u, err, 1);
            tc_fence_after();
          }
          __syncwarp();
          if (elect_one()) {
            const uint32_t d = tm + DCOL + (uint32_t)(b * CW);
            const int np = l + 1 + (l == NS - 1 ? 1 : 0);
            for (int i = 0; i < np; i++) {  // X_i K_{l-i}, and X_0 K_6 with the last level
              const int xi = i > l ? 0 : i, kj = i > l ? NS : l - i;
              const uint32_t a = tm + (uint32_t)(xi * (N / 2));
              const uint64_t kd = k0 + (uint64_t)((kj * CF::NSLOT + ch * (CW / 8)) * 8);
#pragma unroll
              for (int j = 0; j < N / 16; j++)
                tc_mma_f16_ts(d, a + 8 * j, kd + (N / 8 - 2 - 2 * j) * 8, tc_idesc(CW), (i > 0 || j > 0) ? 1u : 0u);
            }
            tc_commit(full + ch * NB + b);
            // only where the next turn's split waits for it: an arrival that nobody waits for could
            // come after the block has left its shared memory
            if (t == NJ - 1 && turn == 0 && more) tc_commit(done);
          }
          __syncwarp();
        }
      }
    }
    __syncthreads();  // every accumulator has been read
    tc_fence_after();
    tc_dealloc(tm, CF::COLS);
    return;
  }

  // =================================================== the lines' warpgroups
  tc64_lines<N, KIND, PW, AX>(s, nlines, cin, s_outer, s_k, err, smraw, tid, warp, more);
}

}  // namespace pft
