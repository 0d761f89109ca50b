// Shared-memory mixed-radix Stockham FFT for the longitude rings.
//
// The semi-naive SHT (App. C.1, last paragraph) starts with a DFT along every
// iso-latitude ring.  A ring of nlon = N points is transformed in shared memory by the
// Stockham autosort formulation: at the stage with radix R and span Ns, butterfly j
// (0 <= j < N/R) reads in[j + r N/R] (r < R), multiplies input r by W_N^{(j mod Ns) r N/(Ns R)},
// applies an R-point DFT and writes output r to out[(j div Ns) Ns R + (j mod Ns) + r Ns].
//
// Two fields travel together (C2; one field, C1, where a pair would not fit or would leave the
// chip short of work).  An element is the real parts of the two fields' values as
// one packed pair of FP32, then the imaginary parts.  Every butterfly and twiddle is packed
// arithmetic (add / mul / fma.rn.f32x2: two FP32 results an instruction, at half the rate of the
// scalar ones), every shared-memory access 16 bytes, and the index arithmetic serves both fields.
// What bounds these kernels is instruction issue (a scalar form of them used 54 % of the issue
// slots at 24 warps an SM, most of the rest waiting on barriers), so the packing takes away
// about half of what they wait for.
//
// Radices go up to 16 so that the rings of the usual grids take three stages
// (1440 = 15 * 8 * 12); a prime factor above 5 becomes a stage of its own with a generic
// butterfly (O(R) work per output, roots of unity from the plan's table), so any ring
// length has a plan.  The composite radices (6, 9, 10, 12, 15, 16) run as two
// register-resident levels of 2-, 3-, 4- and 5-point DFTs (Cooley-Tukey inside the
// butterfly) whose internal twiddles are compile-time constants.  The stage twiddles come
// from a per-stage table, r-major, so that consecutive lanes read consecutive entries: in shared
// memory for short rings, through L1 for long ones (every CTA reads the same N values).
#pragma once
#include <utility>

#include "shot_internal.cuh"

namespace shot {

// ---- packed pairs of FP32 (one value of each of two fields) ---------------------------
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pk2(float lo, float hi) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
// a constant twice, as integer arithmetic that the compiler folds into an immediate (the result of
// an asm statement would be hoisted out of a persistent kernel's loop over items and spilled)
__device__ __forceinline__ f32x2 kc2(float c) {
  return ((f32x2)__float_as_uint(c) << 32) | (f32x2)__float_as_uint(c);
}
__device__ __forceinline__ float2 unpk2(f32x2 a) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a));
  return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// the same on one FP32 value
__device__ __forceinline__ float add2(float a, float b) { return a + b; }
__device__ __forceinline__ float sub2(float a, float b) { return a - b; }
__device__ __forceinline__ float mul2(float a, float b) { return a * b; }
__device__ __forceinline__ float fma2(float a, float b, float c) { return fmaf(a, b, c); }
// one value for every field: a constant (kc) or a variable (dup)
template <class V> __device__ __forceinline__ V kc(float c);
template <> __device__ __forceinline__ float kc<float>(float c) { return c; }
template <> __device__ __forceinline__ f32x2 kc<f32x2>(float c) { return kc2(c); }
template <class V> __device__ __forceinline__ V dup(float x);
template <> __device__ __forceinline__ float dup<float>(float x) { return x; }
template <> __device__ __forceinline__ f32x2 dup<f32x2>(float x) { return pk2(x, x); }
// the value of field q, and the values of the fields of an element together
__device__ __forceinline__ float lane_of(float a, int) { return a; }
__device__ __forceinline__ float lane_of(f32x2 a, int q) {
  const float2 v = unpk2(a);
  return q ? v.y : v.x;
}
__device__ __forceinline__ float of_lanes(const float (&x)[1]) { return x[0]; }
__device__ __forceinline__ f32x2 of_lanes(const float (&x)[2]) { return pk2(x[0], x[1]); }

// One complex value of each of F fields: C2 two fields, C1 one.
template <class T>
struct __align__(2 * sizeof(T)) Cx {
  typedef T V;
  static constexpr int F = sizeof(T) / sizeof(float);
  V re, im;
};
using C2 = Cx<f32x2>;
using C1 = Cx<float>;
template <class V>
__device__ __forceinline__ Cx<V> cx(V re, V im) {
  Cx<V> r;
  r.re = re;
  r.im = im;
  return r;
}
template <class E> __device__ __forceinline__ E cadd(E a, E b) { return cx(add2(a.re, b.re), add2(a.im, b.im)); }
template <class E> __device__ __forceinline__ E csub(E a, E b) { return cx(sub2(a.re, b.re), sub2(a.im, b.im)); }
__device__ __forceinline__ f32x2 neg2(f32x2 a) { return a ^ 0x8000000080000000ull; }
__device__ __forceinline__ float neg2(float a) { return -a; }
// a * w (CONJ: a * conj w), the same w for every field
template <bool CONJ, class E>
__device__ __forceinline__ E cmul(E a, float2 w) {
  typedef typename E::V V;
  const V c = dup<V>(w.x), s = dup<V>(w.y), ns = dup<V>(-w.y);
  return CONJ ? cx(fma2(a.re, c, mul2(a.im, s)), fma2(a.im, c, mul2(a.re, ns)))
              : cx(fma2(a.re, c, mul2(a.im, ns)), fma2(a.re, s, mul2(a.im, c)));
}
// a -+ i b: a - i b (forward) or a + i b (inverse)
template <bool INV, class E>
__device__ __forceinline__ E add_mi(E a, E b) {
  return INV ? cx(sub2(a.re, b.im), add2(a.im, b.re)) : cx(add2(a.re, b.im), sub2(a.im, b.re));
}
// multiply by -i (forward) or +i (inverse)
template <bool INV, class E>
__device__ __forceinline__ E mul_mi(E a) {
  return INV ? cx(neg2(a.im), a.re) : cx(a.im, neg2(a.re));
}

// One row's piece of an element's spectra as it lies in memory, (re, im) of each field.
template <class E> struct Piece { typedef float4 T; };
template <> struct Piece<C1> { typedef float2 T; };
__device__ __forceinline__ C2 piece_value(float4 v) { return cx(pk2(v.x, v.z), pk2(v.y, v.w)); }
__device__ __forceinline__ C1 piece_value(float2 v) { return cx(v.x, v.y); }
__device__ __forceinline__ void store_piece(float* p, C2 v) {
  const float2 re = unpk2(v.re), im = unpk2(v.im);
  *reinterpret_cast<float4*>(p) = make_float4(re.x, im.x, re.y, im.y);
}
__device__ __forceinline__ void store_piece(float* p, C1 v) {
  *reinterpret_cast<float2*>(p) = make_float2(v.re, v.im);
}

// ---- compile-time roots of unity ----------------------------------------------------
// cos and sin of 2 pi j / R from their Taylor series; the angle is first reduced to
// [-pi, pi], where 40 terms are far below double rounding.  Only evaluated by the
// compiler (constexpr initialisers of the butterflies' internal twiddles).
__host__ __device__ constexpr double taylor_cos(double x) {
  double term = 1.0, sum = 1.0;
  for (int k = 1; k < 40; ++k) {
    term *= -x * x / ((2.0 * k - 1.0) * (2.0 * k));
    sum += term;
  }
  return sum;
}
__host__ __device__ constexpr double taylor_sin(double x) {
  double term = x, sum = x;
  for (int k = 1; k < 40; ++k) {
    term *= -x * x / ((2.0 * k) * (2.0 * k + 1.0));
    sum += term;
  }
  return sum;
}
__host__ __device__ constexpr double root_angle(int j, int R) {
  // 2 pi j / R with j reduced to (-R/2, R/2]
  int r = ((j % R) + R) % R;
  if (2 * r > R) r -= R;
  return 2.0 * 3.14159265358979323846 * r / R;
}

// a * W_R^J with W_R = exp(-2 pi i / R) (forward) or its conjugate (inverse)
template <int R, int J, bool INV, class E>
__device__ __forceinline__ E mul_root(E a) {
  typedef typename E::V V;
  constexpr int j = ((J % R) + R) % R;
  if constexpr (j == 0) {
    return a;
  } else if constexpr (2 * j == R) {
    return cx(neg2(a.re), neg2(a.im));
  } else if constexpr (4 * j == R) {
    return mul_mi<INV>(a);
  } else if constexpr (4 * j == 3 * R) {
    return mul_mi<!INV>(a);
  } else {
    constexpr float c = (float)taylor_cos(root_angle(j, R));
    constexpr float s = (float)taylor_sin(root_angle(j, R));
    constexpr float sy = INV ? s : -s;   // W^j = (c, -s) forward
    return cx(fma2(a.re, kc<V>(c), mul2(a.im, kc<V>(-sy))), fma2(a.re, kc<V>(sy), mul2(a.im, kc<V>(c))));
  }
}

// ---- prime-size butterflies (in place on v[0..R-1]) ---------------------------------
template <bool INV, class E>
__device__ __forceinline__ void bfly2(E* v) {
  const E a = v[0], b = v[1];
  v[0] = cadd(a, b);
  v[1] = csub(a, b);
}

template <bool INV, class E>
__device__ __forceinline__ void bfly4(E* v) {
  const E a = cadd(v[0], v[2]), b = csub(v[0], v[2]), c = cadd(v[1], v[3]), d = csub(v[1], v[3]);
  v[0] = cadd(a, c);
  v[2] = csub(a, c);
  v[1] = add_mi<INV>(b, d);
  v[3] = add_mi<!INV>(b, d);
}

template <bool INV, class E>
__device__ __forceinline__ void bfly8(E* v) {
  E e[4] = {v[0], v[2], v[4], v[6]};
  E o[4] = {v[1], v[3], v[5], v[7]};
  bfly4<INV>(e);
  bfly4<INV>(o);
  o[1] = mul_root<8, 1, INV>(o[1]);
  o[3] = mul_root<8, 3, INV>(o[3]);
  v[0] = cadd(e[0], o[0]);
  v[4] = csub(e[0], o[0]);
  v[1] = cadd(e[1], o[1]);
  v[5] = csub(e[1], o[1]);
  v[2] = add_mi<INV>(e[2], o[2]);
  v[6] = add_mi<!INV>(e[2], o[2]);
  v[3] = cadd(e[3], o[3]);
  v[7] = csub(e[3], o[3]);
}

template <bool INV, class E>
__device__ __forceinline__ void bfly3(E* v) {
  typedef typename E::V V;
  const V s = kc<V>(0.86602540378443865f);   // sin(2 pi / 3)
  const V h = kc<V>(-0.5f);
  const E t = cadd(v[1], v[2]);
  const E d = csub(v[1], v[2]);
  const E a = cx(fma2(h, t.re, v[0].re), fma2(h, t.im, v[0].im));
  const V ns = kc<V>(-0.86602540378443865f);
  v[0] = cadd(v[0], t);
  // a -+ i s d
  const E m = cx(fma2(s, d.im, a.re), fma2(ns, d.re, a.im));   // a - i s d
  const E p = cx(fma2(ns, d.im, a.re), fma2(s, d.re, a.im));   // a + i s d
  v[1] = INV ? p : m;
  v[2] = INV ? m : p;
}

template <bool INV, class E>
__device__ __forceinline__ void bfly5(E* v) {
  typedef typename E::V V;
  const V c1 = kc<V>(0.30901699437494742f);     // cos(2pi/5)
  const V k2 = kc<V>(-0.80901699437494742f);   // cos(4pi/5)
  const V s1 = kc<V>(0.95105651629515357f);     // sin(2pi/5)
  const V s2 = kc<V>(0.58778525229247313f);     // sin(4pi/5)
  const E t1 = cadd(v[1], v[4]), t2 = cadd(v[2], v[3]);
  const E d1 = csub(v[1], v[4]), d2 = csub(v[2], v[3]);
  const E x0 = v[0];
  const E a1 = cx(fma2(k2, t2.re, fma2(c1, t1.re, x0.re)), fma2(k2, t2.im, fma2(c1, t1.im, x0.im)));
  const E a2 = cx(fma2(c1, t2.re, fma2(k2, t1.re, x0.re)), fma2(c1, t2.im, fma2(k2, t1.im, x0.im)));
  const V ns1 = kc<V>(-0.95105651629515357f);
  const E b1 = cx(fma2(s1, d1.re, mul2(s2, d2.re)), fma2(s1, d1.im, mul2(s2, d2.im)));
  const E b2 = cx(fma2(s2, d1.re, mul2(ns1, d2.re)), fma2(s2, d1.im, mul2(ns1, d2.im)));
  v[0] = cadd(x0, cadd(t1, t2));
  v[1] = add_mi<INV>(a1, b1);
  v[4] = add_mi<!INV>(a1, b1);
  v[2] = add_mi<INV>(a2, b2);
  v[3] = add_mi<!INV>(a2, b2);
}

template <int R, bool INV, class E>
__device__ __forceinline__ void bfly_prime(E* v) {
  if constexpr (R == 2) bfly2<INV>(v);
  else if constexpr (R == 3) bfly3<INV>(v);
  else if constexpr (R == 4) bfly4<INV>(v);
  else if constexpr (R == 5) bfly5<INV>(v);
  else bfly8<INV>(v);
}

// R-point DFT of the registers v[O + S i], i < R
template <int R, int O, int S, bool INV, class E>
__device__ __forceinline__ void dft_at(E* v) {
  E t[R];
#pragma unroll
  for (int i = 0; i < R; ++i) t[i] = v[O + S * i];
  bfly_prime<R, INV>(t);
#pragma unroll
  for (int i = 0; i < R; ++i) v[O + S * i] = t[i];
}

// Composite R = R1 R2 with n = R2 n1 + n2, k = k1 + R1 k2:
//   X[k] = sum_{n2} W_R2^{n2 k2} W_R^{n2 k1} sum_{n1} W_R1^{n1 k1} x[R2 n1 + n2].
// After the call X[k1 + R1 k2] is in v[R2 k1 + k2].
template <int R1, int R2, bool INV, class E, int... I>
__device__ __forceinline__ void composite_level1(E* v, std::integer_sequence<int, I...>) {
  (dft_at<R1, I, R2, INV>(v), ...);
}
template <int R1, int R2, bool INV, class E, int... I>
__device__ __forceinline__ void composite_twiddle(E* v, std::integer_sequence<int, I...>) {
  // element I = R2 k1 + n2 takes W_R^{n2 k1}
  ((v[I] = mul_root<R1 * R2, (I % R2) * (I / R2), INV>(v[I])), ...);
}
template <int R1, int R2, bool INV, class E, int... I>
__device__ __forceinline__ void composite_level2(E* v, std::integer_sequence<int, I...>) {
  (dft_at<R2, R2 * I, 1, INV>(v), ...);
}

template <int R1, int R2, bool INV, class E>
__device__ __forceinline__ void bfly_composite(E* v) {
  composite_level1<R1, R2, INV>(v, std::make_integer_sequence<int, R2>{});
  composite_twiddle<R1, R2, INV>(v, std::make_integer_sequence<int, R1 * R2>{});
  composite_level2<R1, R2, INV>(v, std::make_integer_sequence<int, R1>{});
}

// Radix R butterfly and the register holding its output k.
template <int R>
struct Radix {
  static constexpr int R1 = 1, R2 = R;   // prime-size: output k in v[k]
};
template <> struct Radix<6> { static constexpr int R1 = 2, R2 = 3; };
template <> struct Radix<9> { static constexpr int R1 = 3, R2 = 3; };
template <> struct Radix<10> { static constexpr int R1 = 2, R2 = 5; };
template <> struct Radix<12> { static constexpr int R1 = 4, R2 = 3; };
template <> struct Radix<15> { static constexpr int R1 = 3, R2 = 5; };
template <> struct Radix<16> { static constexpr int R1 = 4, R2 = 4; };

template <int R, bool INV, class E>
__device__ __forceinline__ void butterfly(E* v) {
  if constexpr (Radix<R>::R1 == 1) bfly_prime<R, INV>(v);
  else bfly_composite<Radix<R>::R1, Radix<R>::R2, INV>(v);
}
template <int R>
__host__ __device__ constexpr int out_reg(int k) {
  return Radix<R>::R1 == 1 ? k : Radix<R>::R2 * (k % Radix<R>::R1) + k / Radix<R>::R1;
}

// Copies the plan's twiddle table into shared memory (asynchronous, 8 bytes an entry; the caller waits).
__device__ __forceinline__ void fft_copy_twiddles(float2* dst, const float2* __restrict__ tw, int len) {
  for (int k = threadIdx.x; k < len; k += blockDim.x)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(dst + k)),
                 "l"(tw + k)
                 : "memory");
}

// stride of consecutive sequences in the CTA's buffers
__host__ __device__ constexpr int seq_ld(int N) { return N + 1; }

// a / d for 0 <= a < 2^16 and 2 <= d < 2^16 with mul = ceil(2^32 / d) (exact: the
// error a (mul - 2^32/d) / 2^32 < 2^-16 never crosses an integer); mul == 0 means d == 1.
__device__ __forceinline__ int fast_div(int a, uint32_t mul) {
  return mul ? (int)__umulhi((uint32_t)a, mul) : a;
}

template <int R, bool INV, class E>
__device__ __forceinline__ void stockham_stage(const E* __restrict__ src, E* __restrict__ dst,
                                               const float2* __restrict__ tws, int N, int Ns, int nseq,
                                               uint32_t ns_mul, uint32_t nr_mul) {
  const int NR = N / R;
  const int ld = seq_ld(N);
  const int total = nseq * NR;
  for (int idx = threadIdx.x; idx < total; idx += blockDim.x) {
    const int q = fast_div(idx, nr_mul);
    const int j = idx - q * NR;
    const int jd = fast_div(j, ns_mul);
    const int k = j - jd * Ns;
    const E* s = src + q * ld + j;
    E v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = s[r * NR];
    if (Ns > 1) {   // the first stage's twiddles are all 1
#pragma unroll
      for (int r = 1; r < R; ++r) {
        v[r] = cmul<INV>(v[r], tws[(r - 1) * Ns + k]);
      }
    }
    butterfly<R, INV>(v);
    E* d = dst + q * ld + jd * Ns * R + k;
#pragma unroll
    for (int r = 0; r < R; ++r) d[r * Ns] = v[out_reg<R>(r)];
  }
}

// Stage with a radix that has no compiled butterfly (an odd prime above 5): a task computes outputs r
// and R - r of butterfly j together.  With v_t the stage-twiddled input t and W_R^{rt} = (c_t, s_t)
// from the plan's table, A = sum v_t c_t and B = sum v_t s_t give A +- i B: four packed FMAs a term for
// two outputs, where one output a task took twelve operations for two.  Tasks run r-major over the
// butterflies, so consecutive threads read consecutive inputs.  A solve of 101 rings of 211 longitudes, one field, 20
// iterations: 2.6 -> 1.8 ms (2.1 in the scalar form); 97 x 202, 8 fields 2.03 -> 1.60 (2.44).
template <bool INV, class E>
__device__ __noinline__ void stockham_stage_generic(const E* __restrict__ src, E* __restrict__ dst,
                                                    const float2* __restrict__ tws, const float2* __restrict__ roots,
                                                    int N, int R, int Ns, int nseq, uint32_t ns_mul,
                                                    uint32_t nr_mul) {
  const int NR = N / R, H = (R + 1) / 2;   // tasks r = 0 .. H - 1 of a butterfly
  const int ld = seq_ld(N);
  const int total = nseq * H * NR;
  for (int idx = threadIdx.x; idx < total; idx += blockDim.x) {
    const int qr = fast_div(idx, nr_mul);   // q H + r
    const int j = idx - qr * NR;
    const int q = qr / H, r = qr - q * H;
    const int jd = fast_div(j, ns_mul);
    const int k = j - jd * Ns;
    const E* s = src + q * ld + j;
    E A{}, B{};
    int e = 0;   // r t mod R
#pragma unroll 4
    for (int t = 0; t < R; ++t) {
      E v = s[t * NR];
      if (Ns > 1 && t > 0) v = cmul<INV>(v, tws[(t - 1) * Ns + k]);
      const float2 w = roots[e];
      const typename E::V c = dup<typename E::V>(w.x), sn = dup<typename E::V>(w.y);
      A = cx(fma2(v.re, c, A.re), fma2(v.im, c, A.im));
      B = cx(fma2(v.re, sn, B.re), fma2(v.im, sn, B.im));
      e += r;
      if (e >= R) e -= R;
    }
    E* d = dst + q * ld + jd * Ns * R + k;
    d[r * Ns] = add_mi<!INV>(A, B);   // A + i B (forward), A - i B (inverse)
    if (r) d[(R - r) * Ns] = add_mi<INV>(A, B);
  }
}

// Transforms nseq sequences of length plan.N stored at a[q * seq_ld(N) + k]; b is
// scratch of the same shape; tw holds the plan's stage twiddles (forward sign), in shared memory for
// the short rings, whose CTAs would wait a global-memory latency in every stage.  Returns
// the buffer holding the result.  All threads of the block must call it; it
// synchronises after every stage.
template <bool INV, class E>
__device__ E* fft_smem(E* a, E* b, const float2* tw, const FftPlan& pl, int nseq) {
  int Ns = 1;
#pragma unroll 1
  for (int s = 0; s < pl.nst; ++s) {
    const int R = pl.R[s];
    const float2* tws = tw + pl.tw_off[s];
    const uint32_t nsm = pl.ns_mul[s], nrm = pl.nr_mul[s];
    switch (R) {
      case 2: stockham_stage<2, INV>(a, b, tws, pl.N, Ns, nseq, nsm, nrm); break;
      case 3: stockham_stage<3, INV>(a, b, tws, pl.N, Ns, nseq, nsm, nrm); break;
      case 4: stockham_stage<4, INV>(a, b, tws, pl.N, Ns, nseq, nsm, nrm); break;
      case 5: stockham_stage<5, INV>(a, b, tws, pl.N, Ns, nseq, nsm, nrm); break;
      case 6: stockham_stage<6, INV>(a, b, tws, pl.N, Ns, nseq, nsm, nrm); break;
      case 8: stockham_stage<8, INV>(a, b, tws, pl.N, Ns, nseq, nsm, nrm); break;
      case 9: stockham_stage<9, INV>(a, b, tws, pl.N, Ns, nseq, nsm, nrm); break;
      case 10: stockham_stage<10, INV>(a, b, tws, pl.N, Ns, nseq, nsm, nrm); break;
      case 12: stockham_stage<12, INV>(a, b, tws, pl.N, Ns, nseq, nsm, nrm); break;
      case 15: stockham_stage<15, INV>(a, b, tws, pl.N, Ns, nseq, nsm, nrm); break;
      case 16: stockham_stage<16, INV>(a, b, tws, pl.N, Ns, nseq, nsm, nrm); break;
      default:
        stockham_stage_generic<INV>(a, b, tws, tw + pl.root_off[s], pl.N, R, Ns, nseq, nsm, nrm);
        break;
    }
    __syncthreads();
    E* t = a;
    a = b;
    b = t;
    Ns *= R;
  }
  return a;
}

// ---- plans fixed at compile time ---------------------------------------------------
// The same Stockham stages with N, the radices and the spans as template constants: the
// divisions by N/R and Ns become multiply-shifts and every load, twiddle and store offset an
// immediate.  CtPlan<0> is the runtime plan.
template <int N_, int R0_ = 1, int R1_ = 1, int R2_ = 1>
struct CtPlan {
  static constexpr int N = N_, R0 = R0_, R1 = R1_, R2 = R2_;
};
using RuntimePlan = CtPlan<0>;

template <int R, bool INV, int N, int NS, int TWOFF, class E>
__device__ __forceinline__ void stockham_stage_ct(const E* src, E* dst, const float2* __restrict__ tw, int nseq) {
  constexpr int NR = N / R, LD = seq_ld(N);
  const int total = nseq * NR;
  // opaque to the compiler, which would otherwise hoist a persistent kernel's index arithmetic and
  // twiddle loads out of its loop over items and spill them
  int idx = threadIdx.x;
  asm volatile("" : "+r"(idx));
  for (; idx < total; idx += blockDim.x) {
    const int q = idx / NR;
    const int j = idx - q * NR;
    const int jd = j / NS;
    const int k = j - jd * NS;
    const E* s = src + q * LD + j;
    E v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = s[r * NR];
    if constexpr (NS > 1) {
      const float2* tws = tw + TWOFF + k;
#pragma unroll
      for (int r = 1; r < R; ++r) v[r] = cmul<INV>(v[r], __ldg(tws + (r - 1) * NS));
    }
    butterfly<R, INV>(v);
    E* d = dst + q * LD + jd * NS * R + k;
#pragma unroll
    for (int r = 0; r < R; ++r) d[r * NS] = v[out_reg<R>(r)];
  }
  __syncthreads();
}

// three-stage compile-time plan; the twiddle table layout is the runtime plan's (stage s at
// sum over earlier stages s' >= 1 of (R_s' - 1) Ns_s')
template <bool INV, class PL, class E>
__device__ E* fft_smem_ct(E* a, E* b, const float2* tw, int nseq) {
  constexpr int N = PL::N, R0 = PL::R0, R1 = PL::R1, R2 = PL::R2;
  static_assert(R0 * R1 * R2 == N, "plan radices must multiply to N");
  stockham_stage_ct<R0, INV, N, 1, 0>(a, b, tw, nseq);
  stockham_stage_ct<R1, INV, N, R0, 0>(b, a, tw, nseq);
  stockham_stage_ct<R2, INV, N, R0 * R1, (R1 - 1) * R0>(a, b, tw, nseq);
  return b;
}

template <bool INV, class PL, class E>
__device__ __forceinline__ E* fft_smem_plan(E* a, E* b, const float2* tw, const FftPlan& pl,
                                                 int nseq) {
  if constexpr (PL::N == 0) return fft_smem<INV>(a, b, tw, pl, nseq);
  else return fft_smem_ct<INV, PL>(a, b, tw, nseq);
}

}  // namespace shot
