// Ring DFTs of the semi-naive SHT and the fused Sinkhorn epilogues.
//
// Forward (App. C.1, last paragraph; App. B quadrature): for a field f and ring j,
//   F_m(j) = sum_k f_jk e^{-i m phi_k},  m = 0..lmax.
// Rings j (north) and J = nlat-1-j (south) are transformed together as ONE complex
// sequence z = f_j + i f_J; F_N(m) = (Z(m) + conj Z(N-m))/2, F_S(m) = (Z(m) - conj Z(N-m))/(2i).
// Because Pbar_lm(-x) = (-1)^{l+m} Pbar_lm(x) and GL nodes are symmetric, the quadrature
// sum over j splits into an even part (l-m even) over S = a_j (F_N + F_S) and an odd part
// (l-m odd) over D = a_j (F_N - F_S) on the north half only.  The kernel writes S and D
// into the (m, parity) blocks X[2m+p][jh][2f + {re,im}].
//
// Inverse: the synthesis produces E_m(jh) (even degrees) and O_m(jh) (odd degrees); the
// north ring has G_N = E + O, the south ring G_S = E - O, and
//   (K v)(theta_j, phi_k) = Re G_0(j) + 2 Re sum_{m>=1} G_m(j) e^{i m phi_k}
// is evaluated for both rings by one inverse complex FFT of the Hermitian-extended
// spectrum Z(m) = G_N(m) + i G_S(m), Z(N-m) = conj G_N(m) + i conj G_S(m).
// The epilogue then applies Algorithm 1's pointwise step to K v (update, check or
// final objective) and reduces per-field partial sums (FP64) per ring pair.
#include "epilogue.cuh"

namespace shot {

namespace {

// A CTA of 192 threads takes one ring pair of F G fields, F = 2 (E = C2) or 1 (C1) fields an element
// (fft.cuh); in the pointwise parts each of its G groups of 192 / G threads (whole warps for G = 1, 2,
// 3, 6) takes one element's fields.  192 threads cover most butterflies of a long ring's stages in one step (96,
// 180 and 120 at 1440 longitudes), and three CTAs an SM leave 112 registers a thread, enough for
// the packed radix-16 butterfly without spills.
constexpr int kThreads = 192;
constexpr int kCtas = 3;

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(smem)),
               "l"(gmem)
               : "memory");
}
__device__ __forceinline__ void cp_async8(void* smem, const void* gmem) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(smem)),
               "l"(gmem)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// this thread's group of the CTA and its index in the group
template <int G, int NT>
struct Group {
  static constexpr int T = NT / G;
  int g, t;
  __device__ __forceinline__ Group() : g(G == 1 ? 0 : threadIdx.x / T), t(G == 1 ? threadIdx.x : threadIdx.x - g * T) {}
};

// Loads rings j (real parts) and J = nlat-1-j (imaginary parts; zero when J == j) of the CTA's
// fields into buf; the second field of an odd last pair is zero.  All rows of a batch of
// longitudes are in flight per thread.
template <int G, int NT, class E>
__device__ __forceinline__ void load_ring_pairs(const float* __restrict__ in, E* buf, int f0, int nf, int nlat, int N,
                                                int j, int J) {
  constexpr int F = E::F;
  const Group<G, NT> gr;
  const int fa = f0 + F * gr.g;
  if (fa >= nf) return;
  const bool second = fa + 1 < nf, two = J != j;   // (of a pair)
  const size_t fs = (size_t)nlat * N;
  const float* aj = in + (size_t)fa * fs + (size_t)j * N;
  const float* aJ = in + (size_t)fa * fs + (size_t)J * N;
  E* b = buf + gr.g * seq_ld(N);
  constexpr int kBatch = 4;
  for (int k0 = gr.t; k0 < N; k0 += kBatch * gr.T) {
    float4 v[kBatch];
#pragma unroll
    for (int i = 0; i < kBatch; ++i) {
      const int k = k0 + i * gr.T;
      v[i].x = k < N ? __ldg(aj + k) : 0.f;
      v[i].y = (k < N && second && F == 2) ? __ldg(aj + fs + k) : 0.f;
      v[i].z = (k < N && two) ? __ldg(aJ + k) : 0.f;
      v[i].w = (k < N && two && second && F == 2) ? __ldg(aJ + fs + k) : 0.f;
    }
#pragma unroll
    for (int i = 0; i < kBatch; ++i) {
      const int k = k0 + i * gr.T;
      if (k >= N) continue;
      if constexpr (F == 2) reinterpret_cast<float4*>(b)[k] = v[i];
      else b[k] = cx(v[i].x, v[i].z);
    }
  }
}

// Starts the gather of the ring pair's spectra of the CTA's fields, E_m and O_m for the orders up to
// mmax (the (2m+1) block of m = lmax is empty), into stg[blk][G] with asynchronous copies.  Row (blk,
// jh) holds the fields' (re, im) pairs contiguously; an even first field starts on a 16-byte
// boundary (ldc is a multiple of 4), and reading up to the next even field stays inside the row.
template <int G, int NT, class E>
__device__ __forceinline__ void issue_spectra(const float* __restrict__ Y, int ldc, int nh, int mmax, int lmax, int jh, int f0,
                                              int nf, typename Piece<E>::T* stg) {
  const int nblk = min(2 * mmax + 2, 2 * lmax + 1);
  const float* y = Y + (size_t)jh * ldc + 2 * f0;
  const size_t row = (size_t)nh * ldc;
  if constexpr (E::F == 1) {
    static_assert(G == 1, "one field a CTA");
    for (int blk = threadIdx.x; blk < nblk; blk += NT) cp_async8(stg + blk, y + blk * row);
  } else if (G == 1) {
    for (int blk = threadIdx.x; blk < nblk; blk += NT) cp_async16(stg + blk, y + blk * row);
  } else {   // consecutive threads read the pieces of a row
    for (int e = threadIdx.x; e < nblk * G; e += NT) {
      const int blk = e / G, c = e - blk * G;
      if (f0 + 2 * c < nf) cp_async16(stg + e, y + blk * row + 4 * c);
    }
  }
  cp_async_commit();
}

// Unfolds the staged spectra into the Hermitian-extended Z of each element:
// G_N = E + O, G_S = E - O, Z(m) = G_N + i G_S, Z(N-m) = conj G_N + i conj G_S; the band
// mmax < m < N - mmax is zero.
template <int G, int NT, class E>
__device__ __forceinline__ void unfold_spectra(const typename Piece<E>::T* stg, E* buf, int N, int mmax, int lmax) {
  const Group<G, NT> gr;
  E* z = buf + gr.g * seq_ld(N);
  for (int k = mmax + 1 + gr.t; k < N - mmax; k += gr.T) z[k] = E{};
  for (int m = gr.t; m <= mmax; m += gr.T) {
    const E e = piece_value(stg[2 * m * G + gr.g]);
    const E o = m < lmax ? piece_value(stg[(2 * m + 1) * G + gr.g]) : E{};
    const E GN = cadd(e, o), GS = csub(e, o);
    if (m == 0) {
      z[0] = cx(GN.re, GS.re);
    } else {
      z[m] = cx(sub2(GN.re, GS.im), add2(GN.im, GS.re));
      z[N - m] = cx(add2(GN.re, GS.im), sub2(GS.re, GN.im));
    }
  }
}

// Two-for-one unpack of the transformed ring pair (j north, J south) and the parity fold:
// F_N(m) = (Z(m) + conj Z(N-m))/2, F_S(m) = (Z(m) - conj Z(N-m))/(2i);
// S = a_j (F_N + F_S) -> block (m, even), D = a_j (F_N - F_S) -> block (m, odd), m <= mmax.
// The columns of an odd last field's missing partner (padding, inside ldc) take a pair's zeros.
template <int G, int NT, class E>
__device__ __forceinline__ void fold_store(const E* buf, int f0, int nf, int N, int mmax, int nh, int jh, float aj,
                                           const ProbState* __restrict__ ps, int scale_which, float* __restrict__ X,
                                           int ldc) {
  constexpr int F = E::F;
  typedef typename E::V V;
  const Group<G, NT> gr;
  const int fa = f0 + F * gr.g;
  if (fa >= nf) return;
  float sf[F];
#pragma unroll
  for (int q = 0; q < F; ++q) {
    sf[q] = 0.5f * aj;
    if (scale_which == 1 && fa + q < nf) sf[q] *= (float)ps[fa + q].beta;
  }
  const V sc = of_lanes(sf);
  const E* z = buf + gr.g * seq_ld(N);
  float* x = X + (size_t)jh * ldc + 2 * fa;
  const size_t row = (size_t)nh * ldc;
  for (int m = gr.t; m <= mmax; m += gr.T) {
    const E zm = z[m], zn = z[m ? N - m : 0];
    const V a = add2(zm.re, zn.re), b = sub2(zm.im, zn.im);   // 2 F_N
    const V c = add2(zm.im, zn.im), d = sub2(zm.re, zn.re);   // 2 F_S = (c, -d)
    store_piece(x + (size_t)(2 * m) * row, cx(mul2(sc, add2(a, c)), mul2(sc, sub2(b, d))));
    store_piece(x + (size_t)(2 * m + 1) * row, cx(mul2(sc, sub2(a, c)), mul2(sc, add2(b, d))));
  }
}

template <int G, int NT, int CTAS, class PL, class E>
__global__ void __launch_bounds__(NT, CTAS) k_dft_fwd(
    const float* __restrict__ in, int nf, int nlat, int nlon, int lmax, int nh,
    const float* __restrict__ a_ring, const ProbState* __restrict__ ps, int scale_which,
    float* __restrict__ X, int ldc, const __grid_constant__ FftPlan pl, const float2* tw, int tws,
    const int2* __restrict__ mlim, float* __restrict__ h, double t) {
  extern __shared__ __align__(16) uint8_t smem[];
  E* sm = reinterpret_cast<E*>(smem);
  if (blockIdx.y == gridDim.y - 1 && h) {   // the heat multipliers
    for (int l = blockIdx.x * blockDim.x + threadIdx.x; l <= lmax; l += gridDim.x * blockDim.x) h[l] = heat_mult(t, l);
    return;
  }
  E* b0 = sm;
  E* b1 = b0 + G * seq_ld(nlon);
  const int jh = blockIdx.y, f0 = blockIdx.x * E::F * G;
  if (tws) {   // twiddles beside the sequences
    fft_copy_twiddles(reinterpret_cast<float2*>(b1 + G * seq_ld(nlon)), tw, tws);
    tw = reinterpret_cast<const float2*>(b1 + G * seq_ld(nlon));
  }
  load_ring_pairs<G, NT>(in, b0, f0, nf, nlat, nlon, jh, nlat - 1 - jh);
  cp_async_wait_all();
  __syncthreads();
  const E* buf = fft_smem_plan<false, PL>(b0, b1, tw, pl, G);
  fold_store<G, NT>(buf, f0, nf, nlon, mlim ? mlim[jh].y : lmax, nh, jh, a_ring[jh], ps, scale_which, X, ldc);
}

template <int G, int NT, int CTAS, class PL, class E, bool LONG>
__global__ void __launch_bounds__(NT, CTAS) k_idft(
    const float* __restrict__ Y, int ldc, int nf, int nlat, int nlon, int lmax, int nh,
    const float* __restrict__ a_ring, const __grid_constant__ FftPlan pl, const float2* tw, int tws,
    EpiParams ep) {
  extern __shared__ __align__(16) uint8_t smem[];
  E* sm = reinterpret_cast<E*>(smem);
  constexpr int FG = E::F * G;
  __shared__ EpiRed<G, NT, E::F, LONG> red;
  __shared__ EpiField fi[FG];
  const int N = nlon, ld = seq_ld(N);
  E* buf = sm;
  E* b1 = buf + G * ld;
  const int jh = blockIdx.y, f0 = blockIdx.x * FG;
  const int j = jh, J = nlat - 1 - jh;
  const bool two = (J != j);   // false only for the equator ring of an odd grid
  if (tws) {   // twiddles beside the sequences
    fft_copy_twiddles(reinterpret_cast<float2*>(b1 + G * ld), tw, tws);
    tw = reinterpret_cast<const float2*>(b1 + G * ld);
  }
  typename Piece<E>::T* stg = reinterpret_cast<typename Piece<E>::T*>(b1);   // the spectra, before the transform needs b1
  const int2 ml = ep.mlim ? ep.mlim[jh] : make_int2(lmax, lmax);   // orders read, orders written
  issue_spectra<G, NT, E>(Y, ldc, nh, ml.x, lmax, jh, f0, nf, stg);
  const int nfg = min(FG, nf - f0);
  epi_fields_load<FG>(ep, f0, nfg, fi);
  const float aj = a_ring[j];
  cp_async_wait_all();
  __syncthreads();
  epi_prefetch_marginals<FG, true>(ep, fi, nfg, (size_t)j * N, (size_t)J * N, two, N, f0, (size_t)nlat * N);
  unfold_spectra<G, NT>(stg, buf, N, ml.x, lmax);
  __syncthreads();
  const E* z = fft_smem_plan<true, PL>(buf, b1, tw, pl, G);
  E* other = (z == buf) ? b1 : buf;   // input of the fused forward transform

  ring_pair_epilogue<G, NT, LONG>(z, other, ld, N, nf, f0, (size_t)nlat * N, (size_t)j * N, (size_t)J * N, two, aj,
                                  nh, jh, ep, red, fi);
  if ((ep.mode == EPI_UPDATE || ep.mode == EPI_SYM) && ep.xout) {
    // the new scaling of this ring pair is in `other`: transform it for the next half-step
    __syncthreads();
    const E* zf = fft_smem_plan<false, PL>(other, const_cast<E*>(z), tw, pl, G);
    fold_store<G, NT>(zf, f0, nf, N, ml.y, nh, jh, aj, nullptr, 0, ep.xout, ldc);
  }
}

// ---------------------------------------------------------------------------------
// Persistent form of k_idft for the solver's update half-steps (EPI_UPDATE with the fused
// forward transform of the new scaling) and its marginal checks (EPI_CHECK, no forward
// transform).  A CTA walks over items (ring pair jh, field group)
// item = blockIdx.x + i gridDim.x, consecutive items covering the field groups of one ring
// pair.  Right after it has unpacked one item's spectra it starts the cp.async gather of the
// next item's spectra rows into a staging area and asks L2 for the next item's marginal rows,
// so that neither the gather nor the update waits on DRAM (three CTAs per SM, ~69 KB each at
// 1440 longitudes and two fields).

// shared memory of k_idft_p (bytes): the two sequence buffers, then the spectra staging area
inline size_t idft_p_layout(int N, int lmax) {
  return (size_t)2 * seq_ld(N) * sizeof(C2) + (size_t)(2 * lmax + 1) * sizeof(float4);
}

template <class PL>
__global__ void __launch_bounds__(kThreads, kCtas) k_idft_p(
    const float* __restrict__ Y, int ldc, int nf, int nlat, int nlon, int lmax, int nh,
    const float* __restrict__ a_ring, const __grid_constant__ FftPlan pl, const float2* tw, EpiParams ep,
    int ngroups) {
  extern __shared__ __align__(16) C2 sm[];
  constexpr int G = 1, NT = kThreads, FG = 2 * G;
  __shared__ EpiRed<G, NT, 2, true> red;
  __shared__ EpiField fi[2][2];
  const int N = nlon, ld = seq_ld(N);
  C2* buf = sm;
  C2* b1 = buf + G * ld;
  float4* stg = reinterpret_cast<float4*>(b1 + G * ld);
  const int nitems = ngroups * nh;
  const size_t fs = (size_t)nlat * N;

  auto orders = [&](int j) { return ep.mlim ? ep.mlim[j] : make_int2(lmax, lmax); };   // read, written
  int item = blockIdx.x, slot = 0;
  int jh = item / ngroups, f0 = (item - jh * ngroups) * FG;
  if (item < nitems) {
    epi_fields_load<FG>(ep, f0, min(FG, nf - f0), fi[0]);
    issue_spectra<G, NT, C2>(Y, ldc, nh, orders(jh).x, lmax, jh, f0, nf, stg);
  }
  __syncthreads();
  if (item < nitems)
    epi_prefetch_marginals<FG>(ep, fi[0], min(FG, nf - f0), (size_t)jh * N, (size_t)(nlat - 1 - jh) * N,
                               nlat - 1 - jh != jh, N, f0, fs);
  while (item < nitems) {
    const int next = item + gridDim.x;
    const int jn = next / ngroups, fn = (next - jn * ngroups) * FG, nn = min(FG, nf - fn);
    const int j = jh, J = nlat - 1 - jh;
    const int2 ml = orders(jh);
    cp_async_wait_all();   // this item's spectra
    __syncthreads();
    unfold_spectra<G, NT>(stg, buf, N, ml.x, lmax);
    __syncthreads();
    if (next < nitems) {   // the staging area is free again: the next item's state and spectra
      epi_fields_load<FG>(ep, fn, nn, fi[slot ^ 1]);
      issue_spectra<G, NT, C2>(Y, ldc, nh, orders(jn).x, lmax, jn, fn, nf, stg);
    }
    const C2* z = fft_smem_plan<true, PL>(buf, b1, tw, pl, G);
    C2* other = (z == buf) ? b1 : buf;
    if (next < nitems)   // fi[slot ^ 1] is visible after the transform's barriers
      epi_prefetch_marginals<FG>(ep, fi[slot ^ 1], nn, (size_t)jn * N, (size_t)(nlat - 1 - jn) * N,
                                 nlat - 1 - jn != jn, N, fn, fs);
    const float aj = a_ring[j];
    // the persistent kernel runs updates and checks only: no final-objective branch
    ring_pair_epilogue<G, NT, true, false>(z, other, ld, N, nf, f0, fs, (size_t)j * N, (size_t)J * N, J != j, aj, nh,
                                           jh, ep, red, fi[slot]);
    if (ep.xout) {   // the update's new scaling: its spectra for the next half-step
      __syncthreads();
      const C2* zf = fft_smem_plan<false, PL>(other, const_cast<C2*>(z), tw, pl, G);
      fold_store<G, NT>(zf, f0, nf, N, ml.y, nh, jh, aj, nullptr, 0, ep.xout, ldc);
    }
    item = next;
    jh = jn;
    f0 = fn;
    slot ^= 1;
  }
  cp_async_wait_all();
}

// Pairs of fields a CTA takes: as few as fill the chip's resident CTAs once, for the work of one
// CTA is a chain of barriers whose length does not depend on G while 192 threads cover the
// butterflies; up to 1536 elements.  Over 64 to 384 rings of 128 to 768 longitudes and 8 to 72 fields (heat
// applications and solves), a limit of 768 elements is 8 % slower on average (up to 27 % at 200 rings), one of
// 3072 1 % (-8 to +11 %).
int pick_g(const Grid& g, int nf) {
  int G = 1;
  for (int c : {2, 3, 6}) {
    const long long items = (long long)g.nh * ((nf + 2 * G - 1) / (2 * G));
    if (items <= kCtas * g.num_sms || c * g.nlon > 1536 || 2 * G >= nf) break;
    G = c;
  }
  return G;
}

template <class E>
size_t idft_smem(int G, int N) { return (size_t)2 * G * seq_ld(N) * sizeof(E); }

// the runtime plan equals the compile-time one (same N and radices in the same order)
template <class PL>
bool plan_is(const FftPlan& p) {
  return p.N == PL::N && p.nst == 3 && p.R[0] == PL::R0 && p.R[1] == PL::R1 && p.R[2] == PL::R2;
}
// Plans compiled for the ring lengths of the 720- and 512-ring grids (one pair of fields a CTA).  Constant
// strides and divisions leave their kernels 80 registers without a spill that matters, so that four CTAs
// of 192 threads share an SM (kCtasCt; the shared memory allows it up to 1750 longitudes); the persistent
// form's staging area leaves room for three.  Heat applications, 24 fields, band limit 255, three -> four
// CTAs: 1440 longitudes 197 -> 187 us, 1024 145 -> 140.  Any other length runs the runtime plan, which these two
// would on 218 and 162 us (a solve of 24 problems, 20 iterations: 11.7 instead of 9.4 ms, 8.2 instead of 7.1).
using Plan1440 = CtPlan<1440, 15, 8, 12>;
using Plan1024 = CtPlan<1024, 4, 16, 16>;
constexpr int kCtasCt = 4;

// Entries of the twiddle table a CTA copies into shared memory: all for rings of up to 768
// longitudes (6 KB), where a CTA has few items and would wait for each stage's twiddles from L2 (32
// rings, one field: 9.4 us an update launch without the copy, 7.3 with it in the scalar form); none
// beyond, where many items read them through L1.
constexpr int kTwMax = 768;
int twiddles_in_smem(const Grid& g) { return g.nlon <= kTwMax ? fft_tw_len(g.plan) : 0; }

// Whether a CTA takes one field (C1, kThreads1 threads as one FFT butterfly needs half the registers)
// instead of a pair:
// - a single field, which leaves half of every pair idle.  A solve of one problem, 60 iterations, pairs -> one
//   field: 64 rings (TF32x3) 3.00 -> 2.85 ms, 256 rings 5.07 -> 4.77; a heat application on rings of 2000
//   longitudes 93 -> 84 us;
// - the solver's half-steps where one field each gives CTAs that are all resident at once, so that pairs
//   would halve the work in flight: five problems on 64 rings 2.99 -> 2.90 ms, three on 200 rings of 1000
//   longitudes (pairs in the persistent form) 1.51 -> 1.38.  Beyond it pairs are as fast or faster (eight
//   problems on 128 rings 3.52 against 3.53).  Not the plain transforms, whose CTAs have less to do (five
//   fields on 128 rings 25.9 -> 27.1 us a heat application), and not rings with a generic stage, whose pairs share
//   the roots' loads (eight problems on 97 x 202 4.12 -> 4.22 ms);
// - rings so long that one CTA of pairs fills an SM: three problems on rings of 4096 longitudes, 20 iterations
//   22.7 -> 15.2 ms (3000 longitudes, eight problems: 14.5 -> 16.4).
// Pairs stay on rings with a compiled plan (1024 longitudes, one field: 50 against 55 us) and on long rings
// with a generic radix above 16, whose roots come through L1 (4099 longitudes: 3.4 against 5.7 ms).
constexpr int kThreads1 = 256;
bool one_field(const Grid& g, int nf, bool solver) {
  const int generic = g.generic_radix;
  if (plan_is<Plan1440>(g.plan) || plan_is<Plan1024>(g.plan) || (generic > 16 && g.nlon > kTwMax)) return false;
  const bool fills_sm = 2 * (idft_smem<C2>(1, g.nlon) + 2048) > 228 * 1024;   // 2 KB: static and reserved
  return fills_sm || nf == 1 || (solver && generic == 1 && (long long)g.nh * nf <= kCtas * g.num_sms);
}

template <int G, class PL = RuntimePlan, int NT = kThreads, int CTAS = kCtas, class E = C2>
int launch_fwd_t(const Grid& g, const float* in, int nf, const ProbState* ps, int scale_which, float* X,
                 int ldc, cudaStream_t st, const int2* mlim, const double* heat_t) {
  const int tws = twiddles_in_smem(g);
  const size_t smem = idft_smem<E>(G, g.nlon) + tws * sizeof(float2);
  SHOT_CUDA(cudaFuncSetAttribute(k_dft_fwd<G, NT, CTAS, PL, E>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  // field groups of one ring pair run together
  dim3 grid((nf + E::F * G - 1) / (E::F * G), g.nh + (heat_t ? 1 : 0));
  ProfScope prof(PK_DFT, st);
  count_launch();
  k_dft_fwd<G, NT, CTAS, PL, E><<<grid, NT, smem, st>>>(in, nf, g.nlat, g.nlon, g.lmax, g.nh, g.a_d, ps, scale_which,
                                                       X, ldc, g.plan, g.tw_d, tws, mlim, heat_t ? g.h_d : nullptr,
                                                       heat_t ? *heat_t : 0.0);
  SHOT_CUDA(cudaGetLastError());
  return SHOT_OK;
}

template <int G, class PL = RuntimePlan, int NT = kThreads, int CTAS = kCtas, class E = C2, bool LONG = (PL::N > kTwMax)>
int launch_idft_t(const Grid& g, const float* Y, int ldc, int nf, const EpiParams& ep, cudaStream_t st) {
  const int tws = twiddles_in_smem(g);
  // two sequence buffers; the second first stages the spectra
  const size_t smem = idft_smem<E>(G, g.nlon) + tws * sizeof(float2);
  SHOT_CUDA(cudaFuncSetAttribute(k_idft<G, NT, CTAS, PL, E, LONG>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  dim3 grid((nf + E::F * G - 1) / (E::F * G), g.nh);   // field groups of one ring pair run together
  ProfScope prof(ep.mode == EPI_CHECK || ep.mode == EPI_FINAL ? PK_CHECK : PK_IDFT, st);
  count_launch();
  k_idft<G, NT, CTAS, PL, E, LONG><<<grid, NT, smem, st>>>(Y, ldc, nf, g.nlat, g.nlon, g.lmax, g.nh, g.a_d, g.plan,
                                                          g.tw_d, tws, ep);
  SHOT_CUDA(cudaGetLastError());
  return SHOT_OK;
}

template <class PL>
int launch_idft_p_t(const Grid& g, const float* Y, int ldc, int nf, const EpiParams& ep, cudaStream_t st) {
  const size_t smem = idft_p_layout(g.nlon, g.lmax);
  SHOT_CUDA(cudaFuncSetAttribute(k_idft_p<PL>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  const int ngroups = (nf + 1) / 2;
  const int nitems = ngroups * g.nh;
  const int grid = nitems < kCtas * g.num_sms ? nitems : kCtas * g.num_sms;
  ProfScope prof(ep.mode == EPI_CHECK || ep.mode == EPI_FINAL ? PK_CHECK : PK_IDFT, st);
  count_launch();
  k_idft_p<PL><<<grid, kThreads, smem, st>>>(Y, ldc, nf, g.nlat, g.nlon, g.lmax, g.nh, g.a_d, g.plan, g.tw_d, ep,
                                             ngroups);
  SHOT_CUDA(cudaGetLastError());
  return SHOT_OK;
}

}  // namespace

int dft_fields_per_cta(const Grid& g, int nf, bool solver) {
  if (g.quad == SHOT_QUAD_HEALPIX) return hp_fields_per_cta(g);
  return one_field(g, nf, solver) ? 1 : 2 * pick_g(g, nf);
}

int launch_dft_fwd(const Grid& g, const float* in, int nf, const ProbState* ps, int scale_which,
                   float* X, int ldc, cudaStream_t st, const int2* mlim, const double* heat_t) {
  if (g.quad == SHOT_QUAD_HEALPIX) {
    if (scale_which && scale_which != 1) {
      set_error("HEALPix ring transform: the per-field factor beta only");
      return SHOT_ERR_UNSUPPORTED;
    }
    return launch_hp_dft_fwd(g, in, nf, X, ldc, st, scale_which == 1 ? ps : nullptr, mlim, heat_t);
  }
  if (g.nlon > kFftCap) {
    set_error("nlon too large for the shared-memory ring FFT");
    return SHOT_ERR_UNSUPPORTED;
  }
  if (one_field(g, nf, false))
    return launch_fwd_t<1, RuntimePlan, kThreads1, kCtas, C1>(g, in, nf, ps, scale_which, X, ldc, st, mlim, heat_t);
  switch (pick_g(g, nf)) {
    case 6: return launch_fwd_t<6>(g, in, nf, ps, scale_which, X, ldc, st, mlim, heat_t);
    case 3: return launch_fwd_t<3>(g, in, nf, ps, scale_which, X, ldc, st, mlim, heat_t);
    case 2: return launch_fwd_t<2>(g, in, nf, ps, scale_which, X, ldc, st, mlim, heat_t);
    default:
      if (plan_is<Plan1440>(g.plan))
        return launch_fwd_t<1, Plan1440, kThreads, kCtasCt>(g, in, nf, ps, scale_which, X, ldc, st, mlim, heat_t);
      if (plan_is<Plan1024>(g.plan))
        return launch_fwd_t<1, Plan1024, kThreads, kCtasCt>(g, in, nf, ps, scale_which, X, ldc, st, mlim, heat_t);
      return launch_fwd_t<1>(g, in, nf, ps, scale_which, X, ldc, st, mlim, heat_t);
  }
}

// Whether launch_idft runs the persistent kernel for this epilogue: the solver's update half-steps
// and checks on rings of more than 768 longitudes (one pair of fields a CTA) whose buffers and staging
// area leave three CTAs on an SM.  Shorter rings take several pairs a CTA and have few items per
// CTA: one item a CTA was faster (256 rings, 48 fields: 59 against 80 us an update; four grids of 64
// to 180 rings, 72 fields each, in one solve: 19.7 against 20.9 ms).
static bool idft_is_persistent(const Grid& g, int nf, const EpiParams& ep) {
  return (((ep.mode == EPI_UPDATE || ep.mode == EPI_SYM) && ep.xout) || ep.mode == EPI_CHECK) &&
         !g.idft_nonpersistent && nf >= 2 && g.nlon > kTwMax && !one_field(g, nf, true) && pick_g(g, nf) == 1 &&
         idft_p_layout(g.nlon, g.lmax) <= 74 * 1024;
}

int launch_idft(const Grid& g, const float* Y, int ldc, int nf, const EpiParams& ep, cudaStream_t st) {
  if (g.quad == SHOT_QUAD_HEALPIX) return launch_hp_idft(g, Y, ldc, nf, ep, st);
  if (g.nlon > kFftCap) {
    set_error("nlon too large for the shared-memory ring FFT");
    return SHOT_ERR_UNSUPPORTED;
  }
  // the solver's update half-steps and marginal checks: persistent kernel with the next item's
  // inputs prefetched
  const int G = pick_g(g, nf);
  if (idft_is_persistent(g, nf, ep)) {
    if (plan_is<Plan1440>(g.plan)) return launch_idft_p_t<Plan1440>(g, Y, ldc, nf, ep, st);
    if (plan_is<Plan1024>(g.plan)) return launch_idft_p_t<Plan1024>(g, Y, ldc, nf, ep, st);
    return launch_idft_p_t<RuntimePlan>(g, Y, ldc, nf, ep, st);
  }
  if (one_field(g, nf, ep.mode != EPI_PLAIN))
    return launch_idft_t<1, RuntimePlan, kThreads1, kCtas, C1>(g, Y, ldc, nf, ep, st);
  switch (G) {
    case 6: return launch_idft_t<6>(g, Y, ldc, nf, ep, st);
    case 3: return launch_idft_t<3>(g, Y, ldc, nf, ep, st);
    case 2: return launch_idft_t<2>(g, Y, ldc, nf, ep, st);
    default:
      if (plan_is<Plan1440>(g.plan)) return launch_idft_t<1, Plan1440, kThreads, kCtasCt>(g, Y, ldc, nf, ep, st);
      if (plan_is<Plan1024>(g.plan)) return launch_idft_t<1, Plan1024, kThreads, kCtasCt>(g, Y, ldc, nf, ep, st);
      if (g.nlon > kTwMax) return launch_idft_t<1, RuntimePlan, kThreads, kCtas, C2, true>(g, Y, ldc, nf, ep, st);
      return launch_idft_t<1>(g, Y, ldc, nf, ep, st);
  }
}

}  // namespace shot
