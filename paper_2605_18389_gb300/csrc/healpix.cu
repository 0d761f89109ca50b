// HEALPix grids (App. C.1 "HEALPix"): ring geometry and the ring transforms.
//
// Rings i = 0 .. 4 nside - 2 run north to south; ring i has n_i pixels at longitudes
// phi0_i + 2 pi j / n_i (j = 0 .. n_i - 1) and every pixel the area 4 pi / N, N = 12 nside^2.
// Polar cap (k = i + 1 < nside): z = 1 - k^2/(3 nside^2), n = 4k, phi0 = pi/(4k);
// equatorial belt (nside <= k <= 2 nside): z = 4/3 - 2k/(3 nside), n = 4 nside,
// phi0 = pi (2 - s)/(4 nside), s = (k - nside + 1) mod 2; the south half mirrors the north
// (z -> -z, same n and phi0), so rings i and 4 nside - 2 - i form the same parity pairs as on
// the other grids and the Legendre stage is shared with them unchanged.
//
// A ring's length n_i is 4k, not always a product of 2, 3 and 5, and the band limit
// (3 nside - 1 by default) exceeds n_i / 2 on the polar rings.  The ring transforms run the
// shared-memory Stockham FFT of the rectangular grids (every length has a plan; prime factors
// above 5 are generic stages) with the aliasing made explicit:
//   forward  F_m = e^{-i m phi0} D_{m mod n},   D_k = sum_j f_j e^{-2 pi i k j / n}
//   inverse  f_j = sum_k Z_k e^{2 pi i k j / n},
//            Z_k = sum_{m = -lmax..lmax, m = k mod n} e^{i m phi0} G_m,   G_{-m} = conj G_m.
// Two rings (j north, J south) travel as one complex sequence and two fields as one packed
// element, as on the other grids; one field where two sequences of pairs exceed an SM's shared
// memory (from nside 1800 on).
#include <cmath>
#include <vector>

#include "epilogue.cuh"
#include "fft.cuh"

namespace shot {
namespace {

// One ring pair of one element's fields a CTA.  The chain of one CTA bounds these kernels (a solve's rings
// are short, and all CTAs of nside 64 and 8 fields are resident at once): 128 threads take most
// stages in one step, the generic stage of a prime factor p in p steps.
constexpr int kHpThreads = 128;
// longest ring of the grids whose CTAs copy their ring's twiddles into shared memory (a table has at
// most 2 n entries: n, and the roots of its generic stages)
constexpr int kHpTwMax = 1024;
// two sequences of the longest ring n and room for its twiddles
template <class E>
size_t hp_smem(int n) { return (size_t)2 * seq_ld(n) * sizeof(E) + (n <= kHpTwMax ? 2 * n * sizeof(float2) : 0); }
// what a block may have, less the kernels' own static shared memory (under 2 KB)
constexpr size_t kHpSmemMax = 225 * 1024;

// e^{i pi r / d} for an integer r reduced modulo 2d (exact argument reduction)
__device__ __forceinline__ float2 half_turns(int r, int d) {
  float s, c;
  sincospif((float)(r % (2 * d)) / (float)d, &s, &c);
  return make_float2(c, s);
}

// The ring's plan and, where tws says so, its twiddles into shared memory (asynchronously: the
// caller waits before the transform); returns where the twiddles are.
__device__ __forceinline__ const float2* load_plan(FftPlan* pl, const FftPlan* __restrict__ plans, int pi,
                                                   const float2* __restrict__ tw_all,
                                                   const int* __restrict__ tw_base, float2* sm, int tws) {
  const int* src = reinterpret_cast<const int*>(plans + pi);
  for (int i = threadIdx.x; i < (int)(sizeof(FftPlan) / sizeof(int)); i += blockDim.x)
    reinterpret_cast<int*>(pl)[i] = src[i];
  const int base = tw_base[pi];
  if (!tws) return tw_all + base;
  fft_copy_twiddles(sm, tw_all + base, tw_base[pi + 1] - base);
  return sm;
}

// from the transformed ring pair D: S = a (F_N + F_S), D = a (F_N - F_S) for m <= mmax into X
// (sc = a / 2 per field, with the field's factor), each order turned by e^{-i m phi0}
template <class E>
__device__ __forceinline__ void hp_fold_store(const E* D, int n, int2 phase, int f0, int mmax, int nh, int jh, typename E::V sc,
                                              float* __restrict__ X, int ldc) {
  typedef typename E::V V;
  float* x = X + (size_t)jh * ldc + 2 * f0;
  const size_t row = (size_t)nh * ldc;
  for (int m = threadIdx.x; m <= mmax; m += kHpThreads) {
    const int k = m % n;
    const E zm = D[k], zn = D[k ? n - k : 0];
    const float2 e = half_turns(m * phase.x, phase.y);
    // 2 F_N = z_k + conj z_{n-k}, 2 F_S = (z_k - conj z_{n-k}) / i, both times e^{-i m phi0}
    const E FN = cmul<true>(cx(add2(zm.re, zn.re), sub2(zm.im, zn.im)), e);
    const E FS = cmul<true>(cx(add2(zm.im, zn.im), sub2(zn.re, zm.re)), e);
    store_piece(x + (size_t)(2 * m) * row, cx(mul2(sc, add2(FN.re, FS.re)), mul2(sc, add2(FN.im, FS.im))));
    store_piece(x + (size_t)(2 * m + 1) * row, cx(mul2(sc, sub2(FN.re, FS.re)), mul2(sc, sub2(FN.im, FS.im))));
  }
}

template <class E>
__global__ void __launch_bounds__(kHpThreads, 4) k_hp_fwd(const float* __restrict__ in, int nf, size_t npix,
                                                       const int* __restrict__ rlen,
                                                       const long long* __restrict__ roff,
                                                       const int2* __restrict__ rphase, int nrings, int lmax, int nh,
                                                       float area, float* __restrict__ X, int ldc,
                                                       const int* __restrict__ rplan, const FftPlan* __restrict__ plans,
                                                       const float2* __restrict__ tw_all,
                                                       const int* __restrict__ tw_base, int tws,
                                                       const ProbState* __restrict__ ps,
                                                       const int2* __restrict__ mlim, float* __restrict__ h,
                                                       double t) {
  constexpr int F = E::F;
  extern __shared__ __align__(16) uint8_t smem[];
  __shared__ FftPlan pl;
  if (blockIdx.y == gridDim.y - 1 && h) {   // the heat multipliers
    for (int l = blockIdx.x * blockDim.x + threadIdx.x; l <= lmax; l += gridDim.x * blockDim.x) h[l] = heat_mult(t, l);
    return;
  }
  const int jh = blockIdx.y, f0 = blockIdx.x * F;
  const int j = jh, J = nrings - 1 - jh;
  const bool two = J != j;
  const int n = rlen[j], pi = rplan[j];
  E* zb = reinterpret_cast<E*>(smem);
  E* db = zb + seq_ld(n);
  const float2* tw = load_plan(&pl, plans, pi, tw_all, tw_base, reinterpret_cast<float2*>(db + seq_ld(n)), tws);
  const float* fj = in + (size_t)f0 * npix + roff[j];
  const float* fJ = in + (size_t)f0 * npix + roff[J];
  float sc[F];   // per-field factor (gradient sweeps)
#pragma unroll
  for (int q = 0; q < F; ++q) sc[q] = 0.5f * area * (ps && f0 + q < nf ? (float)ps[f0 + q].beta : 1.f);
  for (int k = threadIdx.x; k < n; k += kHpThreads) {
    float a[F], b[F];
#pragma unroll
    for (int q = 0; q < F; ++q) {
      a[q] = f0 + q < nf ? fj[q * npix + k] : 0.f;
      b[q] = two && f0 + q < nf ? fJ[q * npix + k] : 0.f;
    }
    zb[k] = cx(of_lanes(a), of_lanes(b));
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  const E* D = fft_smem<false>(zb, db, tw, pl, 1);
  hp_fold_store(D, n, rphase[j], f0, mlim ? mlim[jh].y : lmax, nh, jh, of_lanes(sc), X, ldc);
}

template <class E>
__global__ void __launch_bounds__(kHpThreads, 4) k_hp_idft(const float* __restrict__ Y, int ldc, int nf, size_t npix,
                                                        const int* __restrict__ rlen,
                                                        const long long* __restrict__ roff,
                                                        const int2* __restrict__ rphase, int nrings, int lmax,
                                                        int nh, float area, EpiParams ep,
                                                        const int* __restrict__ rplan,
                                                        const FftPlan* __restrict__ plans,
                                                        const float2* __restrict__ tw_all,
                                                        const int* __restrict__ tw_base, int tws, int nmax) {
  constexpr int F = E::F;
  typedef typename Piece<E>::T Pc;
  extern __shared__ __align__(16) uint8_t smem[];
  __shared__ FftPlan pl;
  __shared__ EpiRed<1, kHpThreads, F> red;
  __shared__ EpiField fi[F];
  const int jh = blockIdx.y, f0 = blockIdx.x * F;
  const int nfg = min(F, nf - f0);
  const int j = jh, J = nrings - 1 - jh;
  const bool two = (J != j);
  const int n = rlen[j], ld = seq_ld(n), pi = rplan[j];
  const size_t rj = (size_t)roff[j], rJ = (size_t)roff[J];
  const int2 phase = rphase[j];
  const int2 ml = ep.mlim ? ep.mlim[jh] : make_int2(lmax, lmax);   // orders read, orders written
  E* za = reinterpret_cast<E*>(smem);   // spectra Z; the buffers are of the longest ring's size
  E* zb = za + seq_ld(nmax);
  const float2* tw = load_plan(&pl, plans, pi, tw_all, tw_base, reinterpret_cast<float2*>(zb + seq_ld(nmax)), tws);
  epi_fields_load<F>(ep, f0, nfg, fi);
  // Z_k = A_k + B_{n-k}: A_r sums e^{i m phi0} (G_N + i G_S) over the orders m >= 0 of residue r
  // modulo n, B_r sums e^{-i m phi0} (conj G_N + i conj G_S) over the orders m >= 1; each spectra row is
  // read once, straight from global memory.  Where a thread would have 16 rows or more (the short rings
  // near the poles without a polar cut: plain synthesis, FP32 recurrence), S threads share a residue, four
  // rows in flight each (nside 64, one field, plain synthesis: 25.8 us with the rows gathered through shared
  // memory, 33.0 with one thread a residue, 23.0 so).  With the cut a residue of such a ring has a few orders.
  const int S = ml.x < 16 * n ? 1 : max(1, min(min(kHpThreads, nmax) / n, (ml.x + 4 * n) / (4 * n)));
  {
    const float* y = Y + (size_t)jh * ldc + 2 * f0;
    const size_t row = (size_t)nh * ldc;
    for (int i = threadIdx.x; i < S * n; i += kHpThreads) {
      E A{}, B{};
#pragma unroll 4
      for (int m = i; m <= ml.x; m += S * n) {
        const E e = piece_value(*reinterpret_cast<const Pc*>(y + (size_t)(2 * m) * row));
        const E o = m < lmax ? piece_value(*reinterpret_cast<const Pc*>(y + (size_t)(2 * m + 1) * row)) : E{};
        const E GN = cadd(e, o), GS = csub(e, o);
        const float2 w = half_turns(m * phase.x, phase.y);
        A = cadd(A, cmul<false>(cx(sub2(GN.re, GS.im), add2(GN.im, GS.re)), w));
        if (m > 0) B = cadd(B, cmul<true>(cx(add2(GN.re, GS.im), sub2(GS.re, GN.im)), w));
      }
      za[i] = A;   // part i / n of residue i % n
      zb[i] = B;
    }
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  epi_prefetch_marginals<F, true>(ep, fi, nfg, rj, rJ, two, n, f0, npix);
  for (int k = threadIdx.x; k < n; k += kHpThreads) {
    const int kb = k ? n - k : 0;
    E z = cadd(za[k], zb[kb]);
    for (int s = 1; s < S; ++s) z = cadd(z, cadd(za[s * n + k], zb[s * n + kb]));
    za[k] = z;
  }
  __syncthreads();
  E* z = fft_smem<true>(za, zb, tw, pl, 1);   // K v on the ring pair
  E* other = (z == za) ? zb : za;   // receives the new scaling
  ring_pair_epilogue<1, kHpThreads>(z, other, ld, n, nf, f0, npix, rj, rJ, two, area, nh, jh, ep, red, fi);
  if ((ep.mode == EPI_UPDATE || ep.mode == EPI_SYM) && ep.xout) {   // transform the new scaling
    __syncthreads();
    const E* D = fft_smem<false>(other, z, tw, pl, 1);
    hp_fold_store(D, n, phase, f0, ml.y, nh, jh, dup<typename E::V>(0.5f * area), ep.xout, ldc);
  }
}

template <class E>
int hp_fwd_t(const Grid& g, const float* in, int nf, float* X, int ldc, cudaStream_t st, const ProbState* ps,
             const int2* mlim, const double* heat_t) {
  const size_t smem = hp_smem<E>(g.nlon);
  SHOT_CUDA(cudaFuncSetAttribute(k_hp_fwd<E>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  ProfScope prof(PK_DFT, st);
  count_launch();
  k_hp_fwd<E><<<dim3((nf + E::F - 1) / E::F, g.nh + (heat_t ? 1 : 0)), kHpThreads, smem, st>>>(
      in, nf, g.npix, g.ring_len_d, g.ring_off_d, g.ring_phase_d, g.nlat, g.lmax, g.nh, (float)g.a_ring[0], X, ldc,
      g.ring_plan_d, g.hp_plan_d, g.hp_tw_d, g.hp_tw_base_d, g.nlon <= kHpTwMax, ps, mlim, heat_t ? g.h_d : nullptr,
      heat_t ? *heat_t : 0.0);
  SHOT_CUDA(cudaGetLastError());
  return SHOT_OK;
}

template <class E>
int hp_idft_t(const Grid& g, const float* Y, int ldc, int nf, const EpiParams& ep, cudaStream_t st) {
  const size_t smem = hp_smem<E>(g.nlon);
  SHOT_CUDA(cudaFuncSetAttribute(k_hp_idft<E>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  ProfScope prof(ep.mode == EPI_CHECK || ep.mode == EPI_FINAL ? PK_CHECK : PK_IDFT, st);
  count_launch();
  k_hp_idft<E><<<dim3((nf + E::F - 1) / E::F, g.nh), kHpThreads, smem, st>>>(
      Y, ldc, nf, g.npix, g.ring_len_d, g.ring_off_d, g.ring_phase_d, g.nlat, g.lmax, g.nh, (float)g.a_ring[0], ep,
      g.ring_plan_d, g.hp_plan_d, g.hp_tw_d, g.hp_tw_base_d, g.nlon <= kHpTwMax, g.nlon);
  SHOT_CUDA(cudaGetLastError());
  return SHOT_OK;
}

int hp_too_long() {
  set_error("nside too large for the shared-memory ring FFT");
  return SHOT_ERR_UNSUPPORTED;
}

}  // namespace

int hp_fields_per_cta(const Grid& g) { return hp_smem<C2>(g.nlon) <= kHpSmemMax ? 2 : 1; }

int launch_hp_dft_fwd(const Grid& g, const float* in, int nf, float* X, int ldc, cudaStream_t st,
                      const ProbState* ps, const int2* mlim, const double* heat_t) {
  if (hp_smem<C2>(g.nlon) <= kHpSmemMax) return hp_fwd_t<C2>(g, in, nf, X, ldc, st, ps, mlim, heat_t);
  if (hp_smem<C1>(g.nlon) <= kHpSmemMax) return hp_fwd_t<C1>(g, in, nf, X, ldc, st, ps, mlim, heat_t);
  return hp_too_long();
}

int launch_hp_idft(const Grid& g, const float* Y, int ldc, int nf, const EpiParams& ep, cudaStream_t st) {
  if (hp_smem<C2>(g.nlon) <= kHpSmemMax) return hp_idft_t<C2>(g, Y, ldc, nf, ep, st);
  if (hp_smem<C1>(g.nlon) <= kHpSmemMax) return hp_idft_t<C1>(g, Y, ldc, nf, ep, st);
  return hp_too_long();
}

// Ring geometry of a HEALPix grid of resolution nside (host, FP64), into the Grid: node
// z = cos(theta) per ring, ring lengths, offsets, longitude phases, per-pixel area.
void healpix_geometry(Grid& g, int nside) {
  const int nr = 4 * nside - 1;
  g.x.assign(nr, 0.0);
  g.ring_len.assign(nr, 0);
  g.ring_off.assign(nr + 1, 0);
  g.ring_phase.assign(nr, std::make_pair(0, 1));
  for (int i = 1; i <= nr; ++i) {
    const int k = i <= 2 * nside ? i : nr + 1 - i;   // mirrored into the north half
    double z;
    int n, pn, pd;
    if (k < nside) {
      z = 1.0 - (double)k * k / (3.0 * nside * nside);
      n = 4 * k;
      pn = 1;
      pd = 4 * k;   // phi0 = pi / (4k)
    } else {
      const int s = (k - nside + 1) % 2;
      z = 4.0 / 3.0 - 2.0 * k / (3.0 * nside);
      n = 4 * nside;
      pn = 2 - s;
      pd = 4 * nside;   // phi0 = pi (2 - s) / (4 nside)
    }
    g.x[i - 1] = (i <= 2 * nside) ? z : -z;
    g.ring_len[i - 1] = n;
    g.ring_phase[i - 1] = std::make_pair(pn, pd);
  }
  g.x[2 * nside - 1] = 0.0;   // the equator ring
  for (int i = 0; i < nr; ++i) g.ring_off[i + 1] = g.ring_off[i] + g.ring_len[i];
  g.npix = (size_t)g.ring_off[nr];
  const double area = 4.0 * M_PI / (double)g.npix;
  g.a_ring.assign(nr, area);
  g.w.resize(nr);
  for (int i = 0; i < nr; ++i) g.w[i] = area * g.ring_len[i] / (2.0 * M_PI);   // ring weight, sum 2
}

}  // namespace shot
