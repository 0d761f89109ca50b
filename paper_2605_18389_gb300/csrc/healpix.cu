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
// element, as on the other grids.
#include <cmath>
#include <vector>

#include "epilogue.cuh"
#include "fft.cuh"

namespace shot {
namespace {

// One ring pair of two fields a CTA.  The chain of one CTA bounds these kernels (a solve's rings
// are short, and all CTAs of nside 64 and 8 fields are resident at once): 128 threads take most
// stages in one step, the generic stage of a prime factor p in p steps.
constexpr int kHpThreads = 128;
// longest ring of the grids whose CTAs copy their ring's twiddles into shared memory (a table has at
// most 2 n entries: n, and the roots of its generic stages)
constexpr int kHpTwMax = 1024;
// two sequences of the longest ring n and room for its twiddles
size_t hp_smem(int n, int tws) { return (size_t)2 * seq_ld(n) * sizeof(C2) + (tws ? 2 * n * sizeof(float2) : 0); }

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
__device__ __forceinline__ void hp_fold_store(const C2* D, int n, int2 phase, int f0, int mmax, int nh, int jh, f32x2 sc,
                                              float* __restrict__ X, int ldc) {
  float* x = X + (size_t)jh * ldc + 2 * f0;
  const size_t row = (size_t)nh * ldc;
  for (int m = threadIdx.x; m <= mmax; m += kHpThreads) {
    const int k = m % n;
    const C2 zm = D[k], zn = D[k ? n - k : 0];
    const float2 e = half_turns(m * phase.x, phase.y);
    // 2 F_N = z_k + conj z_{n-k}, 2 F_S = (z_k - conj z_{n-k}) / i, both times e^{-i m phi0}
    const C2 FN = cmul<true>(c2(add2(zm.re, zn.re), sub2(zm.im, zn.im)), e);
    const C2 FS = cmul<true>(c2(add2(zm.im, zn.im), sub2(zn.re, zm.re)), e);
    const float2 Sr = unpk2(mul2(sc, add2(FN.re, FS.re))), Si = unpk2(mul2(sc, add2(FN.im, FS.im)));
    const float2 Dr = unpk2(mul2(sc, sub2(FN.re, FS.re))), Di = unpk2(mul2(sc, sub2(FN.im, FS.im)));
    *reinterpret_cast<float4*>(x + (size_t)(2 * m) * row) = make_float4(Sr.x, Si.x, Sr.y, Si.y);
    *reinterpret_cast<float4*>(x + (size_t)(2 * m + 1) * row) = make_float4(Dr.x, Di.x, Dr.y, Di.y);
  }
}

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
  extern __shared__ __align__(16) C2 sm[];
  __shared__ FftPlan pl;
  if (blockIdx.y == gridDim.y - 1 && h) {   // the heat multipliers
    for (int l = blockIdx.x * blockDim.x + threadIdx.x; l <= lmax; l += gridDim.x * blockDim.x) h[l] = heat_mult(t, l);
    return;
  }
  const int jh = blockIdx.y, f0 = blockIdx.x * 2;
  const int j = jh, J = nrings - 1 - jh;
  const bool second = f0 + 1 < nf, two = J != j;
  const int n = rlen[j], pi = rplan[j];
  C2* zb = sm;
  C2* db = zb + seq_ld(n);
  const float2* tw = load_plan(&pl, plans, pi, tw_all, tw_base, reinterpret_cast<float2*>(db + seq_ld(n)), tws);
  const float* fj = in + (size_t)f0 * npix + roff[j];
  const float* fJ = in + (size_t)f0 * npix + roff[J];
  for (int k = threadIdx.x; k < n; k += kHpThreads)
    reinterpret_cast<float4*>(zb)[k] =
        make_float4(fj[k], second ? fj[npix + k] : 0.f, two ? fJ[k] : 0.f, (two && second) ? fJ[npix + k] : 0.f);
  // per-field factor (gradient sweeps)
  const float s0 = 0.5f * area * (ps ? (float)ps[f0].beta : 1.f);
  const float s1 = 0.5f * area * (ps && second ? (float)ps[f0 + 1].beta : 1.f);
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  const C2* D = fft_smem<false>(zb, db, tw, pl, 1);
  hp_fold_store(D, n, rphase[j], f0, mlim ? mlim[jh].y : lmax, nh, jh, pk2(s0, s1), X, ldc);
}

__global__ void __launch_bounds__(kHpThreads, 4) k_hp_idft(const float* __restrict__ Y, int ldc, int nf, size_t npix,
                                                        const int* __restrict__ rlen,
                                                        const long long* __restrict__ roff,
                                                        const int2* __restrict__ rphase, int nrings, int lmax,
                                                        int nh, float area, EpiParams ep,
                                                        const int* __restrict__ rplan,
                                                        const FftPlan* __restrict__ plans,
                                                        const float2* __restrict__ tw_all,
                                                        const int* __restrict__ tw_base, int tws) {
  extern __shared__ __align__(16) C2 sm[];
  __shared__ FftPlan pl;
  __shared__ EpiRed<1, kHpThreads> red;
  __shared__ EpiField fi[2];
  const int jh = blockIdx.y, f0 = blockIdx.x * 2;
  const int nfg = min(2, nf - f0);
  const int j = jh, J = nrings - 1 - jh;
  const bool two = (J != j);
  const int n = rlen[j], ld = seq_ld(n), pi = rplan[j];
  const size_t rj = (size_t)roff[j], rJ = (size_t)roff[J];
  const int2 phase = rphase[j];
  const int2 ml = ep.mlim ? ep.mlim[jh] : make_int2(lmax, lmax);   // orders read, orders written
  C2* za = sm;          // spectra Z
  C2* zb = za + ld;
  const float2* tw = load_plan(&pl, plans, pi, tw_all, tw_base, reinterpret_cast<float2*>(zb + ld), tws);
  epi_fields_load<2>(ep, f0, nfg, fi);
  // Z_k = A_k + B_{n-k}: A_r sums e^{i m phi0} (G_N + i G_S) over the orders m >= 0 of residue r
  // modulo n, B_r sums e^{-i m phi0} (conj G_N + i conj G_S) over the orders m >= 1.  A thread owns
  // a residue, so every spectra row is read once, straight from global memory.
  {
    const float* y = Y + (size_t)jh * ldc + 2 * f0;
    const size_t row = (size_t)nh * ldc;
    for (int r = threadIdx.x; r < n; r += kHpThreads) {
      C2 A = c2(0ull, 0ull), B = A;
#pragma unroll 4
      for (int m = r; m <= ml.x; m += n) {
        const float4 e = *reinterpret_cast<const float4*>(y + (size_t)(2 * m) * row);
        const float4 o = m < lmax ? *reinterpret_cast<const float4*>(y + (size_t)(2 * m + 1) * row)
                                  : make_float4(0.f, 0.f, 0.f, 0.f);
        const C2 E = c2(pk2(e.x, e.z), pk2(e.y, e.w)), O = c2(pk2(o.x, o.z), pk2(o.y, o.w));
        const C2 GN = cadd(E, O), GS = csub(E, O);
        const float2 w = half_turns(m * phase.x, phase.y);
        A = cadd(A, cmul<false>(c2(sub2(GN.re, GS.im), add2(GN.im, GS.re)), w));
        if (m > 0) B = cadd(B, cmul<true>(c2(add2(GN.re, GS.im), sub2(GS.re, GN.im)), w));
      }
      za[r] = A;
      zb[r] = B;
    }
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  epi_prefetch_marginals<2, true>(ep, fi, nfg, rj, rJ, two, n, f0, npix);
  for (int k = threadIdx.x; k < n; k += kHpThreads) za[k] = cadd(za[k], zb[k ? n - k : 0]);
  __syncthreads();
  C2* z = fft_smem<true>(za, zb, tw, pl, 1);   // K v on the ring pair
  C2* other = (z == za) ? zb : za;   // receives the new scaling
  ring_pair_epilogue<1, kHpThreads>(z, other, ld, n, nf, f0, npix, rj, rJ, two, area, nh, jh, ep, red, fi);
  if ((ep.mode == EPI_UPDATE || ep.mode == EPI_SYM) && ep.xout) {   // transform the new scaling
    __syncthreads();
    const C2* D = fft_smem<false>(other, z, tw, pl, 1);
    hp_fold_store(D, n, phase, f0, ml.y, nh, jh, pk2(0.5f * area, 0.5f * area), ep.xout, ldc);
  }
}

}  // namespace

int launch_hp_dft_fwd(const Grid& g, const float* in, int nf, float* X, int ldc, cudaStream_t st,
                      const ProbState* ps, const int2* mlim, const double* heat_t) {
  const int tws = g.nlon <= kHpTwMax;
  const size_t smem = hp_smem(g.nlon, tws);
  SHOT_CUDA(cudaFuncSetAttribute(k_hp_fwd, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  ProfScope prof(PK_DFT, st);
  count_launch();
  k_hp_fwd<<<dim3((nf + 1) / 2, g.nh + (heat_t ? 1 : 0)), kHpThreads, smem, st>>>(
      in, nf, g.npix, g.ring_len_d, g.ring_off_d, g.ring_phase_d, g.nlat, g.lmax, g.nh, (float)g.a_ring[0], X, ldc,
      g.ring_plan_d, g.hp_plan_d, g.hp_tw_d, g.hp_tw_base_d, tws, ps, mlim, heat_t ? g.h_d : nullptr,
      heat_t ? *heat_t : 0.0);
  SHOT_CUDA(cudaGetLastError());
  return SHOT_OK;
}

int launch_hp_idft(const Grid& g, const float* Y, int ldc, int nf, const EpiParams& ep, cudaStream_t st) {
  const int tws = g.nlon <= kHpTwMax;
  const size_t smem = hp_smem(g.nlon, tws);
  SHOT_CUDA(cudaFuncSetAttribute(k_hp_idft, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  ProfScope prof(ep.mode == EPI_CHECK || ep.mode == EPI_FINAL ? PK_CHECK : PK_IDFT, st);
  count_launch();
  k_hp_idft<<<dim3((nf + 1) / 2, g.nh), kHpThreads, smem, st>>>(
      Y, ldc, nf, g.npix, g.ring_len_d, g.ring_off_d, g.ring_phase_d, g.nlat, g.lmax, g.nh, (float)g.a_ring[0], ep,
      g.ring_plan_d, g.hp_plan_d, g.hp_tw_d, g.hp_tw_base_d, tws);
  SHOT_CUDA(cudaGetLastError());
  return SHOT_OK;
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
