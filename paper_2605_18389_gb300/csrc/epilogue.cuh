// The Sinkhorn epilogue of the inverse ring transform, shared by the rectangular grids'
// FFT kernel and the HEALPix ring kernel.
//
// z holds K v on the ring pair of F G fields, F = 2 (C2) or 1 (C1) fields an element (real parts:
// ring j, imaginary parts: ring J; G sequences of N longitudes at stride ld); the epilogue applies
// Algorithm 1's pointwise step of the given mode and reduces the per-field partial sums of the
// pair into ep.part[f][jh][NPART]:
//   EPI_PLAIN   out = K v
//   EPI_UPDATE  u = r p / Kv (balanced) or (r p / Kv)^{tau/(tau+eps)} with the problem's FP32
//               buffer factor r (ProbState ru / rv); sums: sum u (gauge) or sum a p u^{-eps/tau}
//               (translation-invariant step) and sum u (unbalanced buffer level),
//               non-positive and non-finite counts; when ep.xout is set the new scaling is
//               also written into `other` (u_j + i u_J) for the forward transform that follows
//   EPI_CHECK   |u_true (K v_true) - p| sums for the marginal error (L2 or L1, App. C.3)
//   EPI_FINAL   u_true, v_true (or the potentials), the marginal error, m(pi) and the dual
//               objective (in FP64); m(pi) = sum a q when a balanced v-update has run (then
//               v (K u) = q node by node), else sum a u (K v)
//   EPI_SYM     self term (q = p): u = sqrt(u_old (p / Ku)^gamma) in place (ep.out holds u_old),
//               breakdown counts; with ep.xout the new u is also written into `other`
// Field f occupies out[f * fstride ...]; rings j and J start at rj and rJ within a field.
#pragma once
#include "fft.cuh"

namespace shot {

// Per-field state the epilogue needs, read into shared memory by epi_fields_load at the start
// of the kernel (while the spectra gather is in flight), so that the epilogue does not wait on
// the chain problem state -> marginal pointer -> marginal values.
struct EpiField {
  const float* marg;   // p (u-step) or q (v-step) of the field
  int live;            // EPI_FINAL: status >= 0; otherwise active
  int balanced;
  float gamma, et;
  float r;             // EPI_UPDATE: the buffer factor inside the ratio (ru or rv)
};

// Threads 0..FG-1 fill fi[q] for the CTA's fields f0 + q (q < nfg).
template <int FG>
__device__ __forceinline__ void epi_fields_load(const EpiParams& ep, int f0, int nfg, EpiField* fi) {
  const int q = threadIdx.x;
  if (q < FG && ep.mode != EPI_PLAIN) {
    if (q >= nfg) {
      fi[q] = EpiField{nullptr, 0, 1, 1.f, 0.f, 1.f};
      return;
    }
    const ProbState* P = ep.ps + f0 + q;
    EpiField e;
    e.marg = ep.marg[f0 + q];
    e.live = (ep.mode == EPI_FINAL) ? (P->status >= 0) : (P->active != 0);
    e.balanced = P->balanced;
    e.gamma = P->gamma;
    e.et = P->et;
    e.r = ep.which ? P->rv : P->ru;
    fi[q] = e;
  }
}

// After fi is visible to the block: asks L2 for the marginal rows j and J of the CTA's live
// fields (UPDATE and CHECK modes) and, for the check, the rows of the u buffer it reads (fields
// f0 + q at stride fstride in ep.other), one 128-byte line per thread, so that the epilogue's
// loads hit L2 instead of waiting on DRAM after the inverse transform.  TO_L1 (kernels with one
// item a CTA): a load of each line whose value is not used, so that they hit L1.
template <int FG, bool TO_L1 = false>
__device__ __forceinline__ void epi_prefetch_marginals(const EpiParams& ep, const EpiField* fi, int nfg, size_t rj,
                                                       size_t rJ, bool two, int N, int f0 = 0, size_t fstride = 0) {
  if (ep.mode != EPI_UPDATE && ep.mode != EPI_CHECK && ep.mode != EPI_SYM) return;
  const float* second = ep.mode == EPI_CHECK ? ep.other : (ep.mode == EPI_SYM ? ep.out : nullptr);
  const int nsrc = (second && fstride) ? 2 : 1;   // marginal (+ the u buffer the epilogue reads)
  const int lines = (N + 31) / 32 + 1;   // a row of N floats spans at most this many 128-byte lines
  const int per_field = 2 * nsrc * lines;
  for (int t = threadIdx.x; t < nfg * per_field; t += blockDim.x) {
    const int q = t / per_field, r = t - q * per_field;
    if (!fi[q].live) continue;
    const int src = r / (2 * lines), rr = r - src * 2 * lines;
    const int ring = rr / lines, l = rr - ring * lines;
    if (ring == 1 && !two) continue;
    const float* base = src ? second + (size_t)(f0 + q) * fstride : fi[q].marg;
    const float* row = base + (ring ? rJ : rj);
    const uintptr_t a0 = reinterpret_cast<uintptr_t>(row) & ~uintptr_t(127);
    const uintptr_t a = a0 + (uintptr_t)l * 128;
    if (a >= reinterpret_cast<uintptr_t>(row + N)) continue;
    if constexpr (TO_L1) {   // a word of the line that belongs to the row
      const uintptr_t w = a < reinterpret_cast<uintptr_t>(row) ? reinterpret_cast<uintptr_t>(row) : a;
      float x;
      asm volatile("ld.global.f32 %0, [%1];" : "=f"(x) : "l"(w));
    } else {
      asm volatile("prefetch.global.L2 [%0];" ::"l"(a));
    }
  }
}

// How the sums of a field on a ring pair are formed: FP32 terms, the two rings' terms added first, then
// a batch of longitudes, then a chain of batches (two alternating chains where a thread of a group of 32
// has many), then groups of 32 / P lanes, and FP64 from there on, with at least eight partial sums per
// field whatever number of threads share it.  No term passes more FP32 additions than with 256 threads
// and eight warps per field (4 + 2 ceil(N / 256): a chain of both rings' terms and five lane steps),
// which the short rings of G = 6 would otherwise exceed: 32 threads, 16 terms each.  The unbalanced
// update amplifies the rounding of its sum by tau / eps.  LONG (one pair of fields a CTA on rings of more
// than 768 longitudes): ceil(N / 192) + 5 additions are within that without batches and with whole-warp
// sums, and the shorter code keeps registers.  An update in the persistent kernel, plain chain -> batches ->
// LONG: 420 x 864, 12 problems 48.5 -> 51.8 -> 49.6 us; 720 x 1440, 24 problems, band limit 255 113.8 ->
// 117.3 -> 116.3.  Four grids of 64 to 180 rings, 40 iterations, against the plain chain: 18.47 -> 18.55 ms.
template <class V, bool TWO = false>
struct Chain {
  V a{}, b{};
  __device__ __forceinline__ void add(V x) {
    const V t = add2(TWO ? b : a, x);
    b = a;
    a = t;
  }
  __device__ __forceinline__ V value() const { return TWO ? add2(a, b) : a; }
};
struct CompInf {   // the error beside the sum (Knuth's two-sum); an infinite sum stays infinite
  float s = 0.f, c = 0.f;
  __device__ __forceinline__ void add(float x) {
    const float t = s + x, b = t - s;
    c += (s - (t - b)) + (x - b);
    s = t;
  }
  __device__ __forceinline__ double value() const { return fabsf(s) < INFINITY ? (double)s + (double)c : (double)s; }
};

// Partial sums of a CTA's warps: NT / G threads share an element's F fields, and each of their GW warps
// leaves P sums of 32 / P lanes.
template <int G, int NT, int F, bool LONG = false>
struct EpiRed {
  static constexpr int GW = NT / G / 32, P = LONG || GW >= 8 ? 1 : GW >= 4 ? 2 : GW >= 2 ? 4 : 8;
  static_assert(LONG || GW * P >= 8, "at least eight partial sums");
  float v[NT / 32][P][F * NPART];
  double d[NT / 32][F][2];   // EPI_FINAL: warp sums of m(pi) and the objective
};

// The update of one K v value in full generality: u, the terms (t0, t1) of its two sums and the
// breakdown counts.
__device__ __forceinline__ float epi_update_value(float pm, float kv, float rr, bool bal, float gam, float aj,
                                                  float& t0, float& t1, float (&bad)[2]) {
  const float ratio = __fdividef(pm, kv) * rr;   // MUFU reciprocal + multiply, <= 2 ulp
  const float u = bal ? ratio : exp2f(gam * __log2f(ratio));
  t0 = u;
  t1 = 0.f;
  if (!bal) {
    t0 = aj * u * kv * (1.f / rr);
    t1 = u;
  }
  // K v positive and finite, u finite (NaN fails each comparison); the failures are sorted into
  // non-positive (first in the status precedence) and non-finite
  if (!(kv > 0.f && kv < INFINITY && fabsf(u) < INFINITY)) {
    if (kv <= 0.f) bad[0] += 1.f;
    else bad[1] += 1.f;   // NaN or infinite K v, or u overflowed
  }
  return u;
}

// The update of a pair of live fields on a ring pair.  u = (r p/Kv)^gamma (hardware log2/exp2,
// ~2^-21 absolute in the exponent); the translation-invariant sum's p u^{-eps/tau} =
// p (r p/Kv)^{-eps/(tau+eps)} equals u (Kv) / r since gamma + eps/(tau+eps) = 1, so one power serves
// both (ratio = 0 gives u = 0 and adds nothing).
// An element whose four K v are normal and at most 2^125 takes the reciprocal directly (the value
// __fdividef gives there); any other goes through epi_update_value.  The check for a non-finite u is
// on the thread's sum: it is finite exactly if every u is (or the sum has overflowed, which stops
// the problem too).  The pointwise part is instruction issue: with a check and a scaled divide per
// value it took 38 of the update kernel's 79 million warp instructions (720 rings, 24 fields).
template <int GT, bool LONG>
__device__ __forceinline__ void epi_update_pair(const float4* zg, float4* og, int t, int N, const EpiField* fi,
                                                float* out, size_t fstride, size_t rj, int dJ, bool xout, float aj,
                                                float (&acc)[2][NPART]) {
  constexpr int kBatch = 2;   // (4 measured slower: registers)
  const float rr[2] = {fi[0].r, fi[1].r}, ri[2] = {1.f / rr[0], 1.f / rr[1]}, gam[2] = {fi[0].gamma, fi[1].gamma};
  const bool bal0 = fi[0].balanced, bal1 = fi[1].balanced;
  float bad[2][2] = {{0.f, 0.f}, {0.f, 0.f}};
  Chain<f32x2, (GT < 64)> s0, s1;
  const float* m00 = fi[0].marg + rj + t;   // ring j of the first field; ring J starts dJ further
  const float* m10 = fi[1].marg + rj + t;
  const float* m01 = m00 + dJ;
  const float* m11 = m10 + dJ;
  for (int k0 = t; k0 < N; k0 += kBatch * GT) {
    float4 pv[kBatch];   // (field 0, field 1) on ring j, then on ring J, as K v is stored
#pragma unroll
    for (int b = 0; b < kBatch; ++b) {
      if (k0 + b * GT < N)
        pv[b] = make_float4(__ldg(m00 + b * GT), __ldg(m10 + b * GT), __ldg(m01 + b * GT), __ldg(m11 + b * GT));
    }
    m00 += kBatch * GT;
    m10 += kBatch * GT;
    m01 += kBatch * GT;
    m11 += kBatch * GT;
    f32x2 x0 = 0, x1 = 0;
#pragma unroll
    for (int b = 0; b < kBatch; ++b) {
      const int k = k0 + b * GT;
      if (k >= N) break;
      const float4 z = zg[k];
      const uint32_t lo = 0x00800000u, span = 0x7e000000u - 0x00800000u;
      const uint32_t d = max(max(__float_as_uint(z.x) - lo, __float_as_uint(z.y) - lo),
                             max(__float_as_uint(z.z) - lo, __float_as_uint(z.w) - lo));
      float4 u, v0, v1;   // the new scaling and the terms of its sums
      if (d <= span) {
        auto one = [&](float pm, float kv, float r, float rinv, bool bal, float ga, float& t0, float& t1) {
          float rc;
          asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rc) : "f"(kv));
          const float ratio = pm * rc * r;
          const float w = bal ? ratio : exp2f(ga * __log2f(ratio));
          t0 = w;
          t1 = 0.f;
          if (!bal) {
            t0 = aj * w * kv * rinv;
            t1 = w;
          }
          return w;
        };
        u.x = one(pv[b].x, z.x, rr[0], ri[0], bal0, gam[0], v0.x, v1.x);
        u.y = one(pv[b].y, z.y, rr[1], ri[1], bal1, gam[1], v0.y, v1.y);
        u.z = one(pv[b].z, z.z, rr[0], ri[0], bal0, gam[0], v0.z, v1.z);
        u.w = one(pv[b].w, z.w, rr[1], ri[1], bal1, gam[1], v0.w, v1.w);
      } else {
        u.x = epi_update_value(pv[b].x, z.x, rr[0], bal0, gam[0], aj, v0.x, v1.x, bad[0]);
        u.y = epi_update_value(pv[b].y, z.y, rr[1], bal1, gam[1], aj, v0.y, v1.y, bad[1]);
        u.z = epi_update_value(pv[b].z, z.z, rr[0], bal0, gam[0], aj, v0.z, v1.z, bad[0]);
        u.w = epi_update_value(pv[b].w, z.w, rr[1], bal1, gam[1], aj, v0.w, v1.w, bad[1]);
      }
      const f32x2 y0 = add2(pk2(v0.x, v0.y), pk2(v0.z, v0.w));
      if constexpr (LONG) s0.add(y0);
      else x0 = add2(x0, y0);
      if (!(bal0 && bal1)) {
        const f32x2 y1 = add2(pk2(v1.x, v1.y), pk2(v1.z, v1.w));
        if constexpr (LONG) s1.add(y1);
        else x1 = add2(x1, y1);
      }
      if (out) {
        float* o = out + k;
        o[0] = u.x;
        o[fstride] = u.y;
        o[dJ] = u.z;
        o[fstride + dJ] = u.w;
      }
      if (xout) og[k] = u;
    }
    if constexpr (!LONG) {
      s0.add(x0);
      s1.add(x1);
    }
  }
  const float2 a0 = unpk2(s0.value()), a1 = unpk2(s1.value());
  acc[0][0] = a0.x;
  acc[1][0] = a0.y;
  acc[0][1] = a1.x;
  acc[1][1] = a1.y;
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    acc[q][2] = bad[q][0];
    acc[q][3] = bad[q][1];
    if (!(fabsf((q ? bal1 : bal0) ? acc[q][0] : acc[q][1]) < INFINITY) && acc[q][2] == 0.f) acc[q][3] += 1.f;
  }
}

// LONG: the sums' form for rings of more than 768 longitudes.  kFinal = false compiles the EPI_FINAL
// branch out (kernels never launched with it).
// The CTA's NT threads form G groups of NT / G (whole warps); group g takes the F fields from
// f0 + F g on, a thread longitude k of both rings of the pair, so that one set of sums per
// thread and one warp reduction serve a group whatever G is.
template <int G, int NT, bool LONG = false, bool kFinal = true, class E>
__device__ __forceinline__ void ring_pair_epilogue(const E* z, E* other, int ld, int N, int nf, int f0,
                                                   size_t fstride, size_t rj, size_t rJ, bool two, float aj,
                                                   int nh, int jh, const EpiParams& ep,
                                                   EpiRed<G, NT, E::F, LONG>& red, const EpiField* fi) {
  constexpr int GT = NT / G, GW = GT / 32, P = EpiRed<G, NT, E::F, LONG>::P, F = E::F;
  static_assert(NT % G == 0 && GT % 32 == 0, "a group is whole warps");
  constexpr int kBatchGen = 2;   // the general path of the update
  constexpr int kEpiBatch = 4;   // longitudes per thread whose marginal values are loaded together
  const int g = G == 1 ? 0 : threadIdx.x / GT, t = G == 1 ? threadIdx.x : threadIdx.x - g * GT;
  const int fa = f0 + F * g;                       // first field of the group
  const int nq = min(F, nf - fa);                  // fields of the group (<= 0: none)
  const E* zg = z + g * ld;
  E* og = other + g * ld;
  if (ep.mode == EPI_PLAIN) {
    float* o = ep.out + (size_t)fa * fstride;
    for (int k = t; k < N; k += GT) {
      const E zz = zg[k];
#pragma unroll
      for (int q = 0; q < F; ++q)
        if (q < nq) {
          o[q * fstride + rj + k] = lane_of(zz.re, q);
          if (two) o[q * fstride + rJ + k] = lane_of(zz.im, q);
        }
    }
    return;
  }
  // Per-element arithmetic is FP32, and the sums as described at Chain; the final pass, which runs
  // once a solve, compensates its threads' sums instead.
  float acc[F][NPART];
#pragma unroll
  for (int q = 0; q < F; ++q)
#pragma unroll
    for (int i = 0; i < NPART; ++i) acc[q][i] = 0.f;
  // EPI_FINAL: the dual objective and m(pi) reach the block's FP64 sums through per-thread
  // partials: the potentials' offsets eps la and eps lb cancel between the two marginals' terms
  // and, across the three problems, in the divergence, so the balanced objective is formed per
  // thread as la sum p + lb sum q + sum (p log u_buf + q log v_buf), with the sums of p and q
  // (and the masses) compensated (Kahan) in FP32 and the offsets applied in FP64; per element
  // the work stays FP32.  m(pi) enters S_dual times eps.
  if (ep.mode == EPI_UPDATE || ep.mode == EPI_SYM) {
    // the fields of an element in one pass: K v comes and the new scaling leaves in one piece
    const bool sym = ep.mode == EPI_SYM;
    const EpiField* f2 = fi + F * g;
    bool pair = false;   // a pair of live fields on two rings
    if constexpr (F == 2) {
      pair = !sym && two && nq > 1 && f2[0].live && f2[1].live;
      if (pair) {
        float* out = ep.skip_store ? nullptr : ep.out + (size_t)fa * fstride + rj;
        const int dJ = (int)(rJ - rj);   // a field has fewer than 2^31 nodes
        epi_update_pair<GT, LONG>(reinterpret_cast<const float4*>(zg), reinterpret_cast<float4*>(og), t, N, f2, out, fstride,
                            rj, dJ, ep.xout != nullptr, aj, acc);
      }
    }
    if (!pair) {
      float* outf[F];
      const float* mg[F];
      bool live[F], bal[F];
      float gam[F], rr[F], bad[F][2];
#pragma unroll
      for (int q = 0; q < F; ++q) {
        live[q] = q < nq && f2[q].live;
        bal[q] = f2[q].balanced;
        outf[q] = ep.out + (size_t)(fa + q) * fstride;
        mg[q] = f2[q].marg;
        gam[q] = f2[q].gamma;
        rr[q] = f2[q].r;
        bad[q][0] = bad[q][1] = 0.f;
      }
      Chain<typename E::V, (GT < 64)> s0, s1;
      for (int k0 = t; k0 < N && nq > 0; k0 += kBatchGen * GT) {
        // one field an element, the equator ring, an odd last field, frozen problems and self terms:
        // field by field; the marginal values (self term: and the old scaling's) of all this thread's
        // longitudes first, then the arithmetic; a frozen problem loads its stored scaling
        float pv[kBatchGen][F][2], uo[kBatchGen][F][2];
        typename E::V x0{}, x1{};
#pragma unroll
        for (int b = 0; b < kBatchGen; ++b) {
          const int k = k0 + b * GT;
#pragma unroll
          for (int q = 0; q < F; ++q) {
            const bool in = k < N && live[q], st = k < N && q < nq && (!live[q] || sym);
            pv[b][q][0] = in ? __ldg(mg[q] + rj + k) : 0.f;
            pv[b][q][1] = (in && two) ? __ldg(mg[q] + rJ + k) : 0.f;
            uo[b][q][0] = st ? outf[q][rj + k] : 0.f;
            uo[b][q][1] = (st && two) ? outf[q][rJ + k] : 0.f;
          }
        }
#pragma unroll
        for (int b = 0; b < kBatchGen; ++b) {
          const int k = k0 + b * GT;
          if (k >= N) break;
          const E zz = zg[k];
          float un[2][F], v0[F], v1[F];   // the new scaling on rings j and J, the terms of its sums
#pragma unroll
          for (int q = 0; q < F; ++q) {
            un[0][q] = uo[b][q][0];
            un[1][q] = uo[b][q][1];
            v0[q] = v1[q] = 0.f;
            if (!live[q]) continue;
#pragma unroll
            for (int r = 0; r < 2; ++r) {
              if (r == 1 && !two) { un[1][q] = 0.f; break; }
              const float kv = lane_of(r ? zz.im : zz.re, q);
              const float pm = pv[b][q][r];
              float u;
              if (sym) {
                const float ratio = __fdividef(pm, kv);
                const float x = bal[q] ? ratio : exp2f(gam[q] * __log2f(ratio));
                u = sqrtf(uo[b][q][r] * x);
                if (!(kv > 0.f && kv < INFINITY && fabsf(u) < INFINITY)) {
                  if (kv <= 0.f) bad[q][0] += 1.f;
                  else bad[q][1] += 1.f;
                }
              } else {
                float t0, t1;
                u = epi_update_value(pm, kv, rr[q], bal[q], gam[q], aj, t0, t1, bad[q]);
                v0[q] = r ? v0[q] + t0 : t0;
                v1[q] = r ? v1[q] + t1 : t1;
              }
              if (sym || !ep.skip_store) outf[q][(r ? rJ : rj) + k] = u;
              un[r][q] = u;
            }
          }
          if constexpr (LONG) {
            s0.add(of_lanes(v0));
            s1.add(of_lanes(v1));
          } else {
            x0 = add2(x0, of_lanes(v0));
            x1 = add2(x1, of_lanes(v1));
          }
          if (ep.xout) og[k] = cx(of_lanes(un[0]), of_lanes(un[1]));
        }
        if constexpr (!LONG) {
          s0.add(x0);
          s1.add(x1);
        }
      }
#pragma unroll
      for (int q = 0; q < F; ++q) {
        acc[q][0] = lane_of(s0.value(), q);
        acc[q][1] = lane_of(s1.value(), q);
        acc[q][2] = bad[q][0];
        acc[q][3] = bad[q][1];
      }
    }
  } else {
#pragma unroll
    for (int q = 0; q < F; ++q) {
      if (q >= nq) break;
      const int f = fa + q;
      const size_t fbase = (size_t)f * fstride;
      float* outf = ep.out + fbase;
      float* othf = ep.other ? ep.other + fbase : nullptr;
      const EpiField ef = fi[F * g + q];
      if (!ef.live) continue;
      if (ep.mode == EPI_CHECK) {
        const float* mg = ef.marg;
        const float cuv = ep.ps[f].cuv;
        Chain<float> e0, e1;
        for (int k0 = t; k0 < N; k0 += kEpiBatch * GT) {
          // the marginal and u values of all this thread's longitudes first, then the arithmetic
          float pv[kEpiBatch][2], uv[kEpiBatch][2];
#pragma unroll
          for (int b = 0; b < kEpiBatch; ++b) {
            const int k = k0 + b * GT;
            pv[b][0] = (k < N) ? __ldg(mg + rj + k) : 0.f;
            pv[b][1] = (k < N && two) ? __ldg(mg + rJ + k) : 0.f;
            uv[b][0] = (k < N) ? __ldg(othf + rj + k) : 0.f;
            uv[b][1] = (k < N && two) ? __ldg(othf + rJ + k) : 0.f;
          }
          float x0[kEpiBatch], x1[kEpiBatch];
#pragma unroll
          for (int b = 0; b < kEpiBatch; ++b) {
            const int k = k0 + b * GT;
            x0[b] = x1[b] = 0.f;
            if (k >= N) continue;
            const E zz = zg[k];
#pragma unroll
            for (int r = 0; r < 2; ++r) {
              if (r == 1 && !two) break;
              const float kv = lane_of(r ? zz.im : zz.re, q);
              const float pm = pv[b][r];
              const float d = fmaf(cuv * uv[b][r], kv, -pm);
              const float t0 = ep.norm_l1 ? aj * fabsf(d) : d * d, t1 = ep.norm_l1 ? aj * pm : pm * pm;
              x0[b] = r ? x0[b] + t0 : t0;
              x1[b] = r ? x1[b] + t1 : t1;
            }
          }
          static_assert(kEpiBatch == 4, "a batch's terms are added as a tree");
          e0.add((x0[0] + x0[1]) + (x0[2] + x0[3]));
          e1.add((x1[0] + x1[1]) + (x1[2] + x1[3]));
        }
        acc[q][0] = e0.value();
        acc[q][1] = e1.value();
      } else if constexpr (kFinal) {  // EPI_FINAL: z = K v_buf; ep.other = u buffer, ep.out = v buffer
        const ProbState* P = ep.ps + f;
        const float* pp = ep.marg[f];
        const float* qq = ep.marg2[f];
        const float cu = P->cu, cv = P->cv, cuv = P->cuv;
        // log u_true = la + log u_buf with la split into an FP32 head and a small remainder
        const float la_hi = (float)P->la, lb_hi = (float)P->lb;
        const float la_lo = (float)(P->la - (double)la_hi), lb_lo = (float)(P->lb - (double)lb_hi);
        const int bal = P->balanced;
        // balanced, after a v-update: v (K u) = q at every node, so m(pi) = sum a u (K v) =
        // sum a v (K u) = sum a q (K is self-adjoint in the area inner product)
        const bool mass_q = bal && !isnan(P->mass_v);
        const float epsf = (float)ep.eps, tauf = (float)P->tau, et = bal ? 0.f : (float)(ep.eps / P->tau);
        // balanced: A = sum p, B = sum q (compensated), C = sum p log u_buf + q log v_buf, D = sum
        // u (K v) (m(pi) before any v-update); unbalanced: A = sum u (K v), B = the objective's terms
        float A = 0.f, Ac = 0.f, B = 0.f, Bc = 0.f;
        CompInf C, D, e0, e1;
        auto kahan = [](float& s, float& c, float x) {
          const float y = x - c, t = s + y;
          c = (t - s) - y;
          s = t;
        };
        for (int k = t; k < N; k += GT) {
          const E zz = zg[k];
#pragma unroll
          for (int r = 0; r < 2; ++r) {
            if (r == 1 && !two) break;
            const float kv = lane_of(r ? zz.im : zz.re, q);
            const size_t o = (r ? rJ : rj) + k;
            const float pm = __ldg(pp + o), qm = __ldg(qq + o);
            const float ub = othf[o], vb = outf[o];
            const float lu = la_hi + (logf(ub) + la_lo), lv = lb_hi + (logf(vb) + lb_lo);
            if (ep.potentials) {
              othf[o] = epsf * lu;
              outf[o] = epsf * lv;
            } else {
              othf[o] = cu * ub;
              outf[o] = cv * vb;
            }
            const float ukv = cuv * ub * kv;   // u_true (K v_true)
            const float d = ukv - pm;
            e0.add(ep.norm_l1 ? aj * fabsf(d) : d * d);
            e1.add(ep.norm_l1 ? aj * pm : pm * pm);
            // phi = eps log u, psi = eps log v (App. C.2); terms with a zero marginal vanish.
            // Balanced: p (la + log u_buf) + q (lb + log v_buf), the offsets applied per thread
            // below; eps and a_j multiply the sums.
            if (bal) {
              kahan(A, Ac, pm);
              kahan(B, Bc, qm);
              C.add((pm > 0.f ? pm * logf(ub) : 0.f) + (qm > 0.f ? qm * logf(vb) : 0.f));
              D.add(ukv);
            } else {  // tau (1 - e^{-phi/tau}) = -tau expm1(-(eps/tau) log u), per node in FP32
              kahan(A, Ac, ukv);
              kahan(B, Bc, (pm > 0.f ? -tauf * expm1f(-et * lu) * pm : 0.f) +
                               (qm > 0.f ? -tauf * expm1f(-et * lv) * qm : 0.f));
            }
          }
        }
        acc[q][0] = (float)e0.value();
        acc[q][1] = (float)e1.value();
        // this thread's m(pi) and objective in FP64, then the warp's sums
        double vm, vo;
        if (bal) {
          vm = mass_q ? (double)B - (double)Bc : D.value();
          vo = P->la * ((double)A - (double)Ac) + P->lb * ((double)B - (double)Bc) + C.value();
        } else {
          vm = (double)A - (double)Ac;
          vo = (double)B - (double)Bc;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          vm += __shfl_xor_sync(0xffffffffu, vm, o);
          vo += __shfl_xor_sync(0xffffffffu, vo, o);
        }
        if ((threadIdx.x & 31) == 0) {
          red.d[threadIdx.x >> 5][q][0] = vm;
          red.d[threadIdx.x >> 5][q][1] = vo;
        }
      }
    }
  }
  // one block reduction, each group's warps for its own fields
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int q = 0; q < F; ++q)
#pragma unroll
    for (int i = 0; i < NPART; ++i) {
      float v = acc[q][i];
#pragma unroll
      for (int o = 16; o >= P; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane < P) red.v[wid][lane][q * NPART + i] = v;
    }
  __syncthreads();
  if constexpr (kFinal) {
    if (ep.mode == EPI_FINAL && threadIdx.x < 2 * F * G) {
      const int fq = threadIdx.x >> 1, i = threadIdx.x & 1;   // field of the CTA
      if (f0 + fq < nf && fi[fq].live) {
        double s = 0.0;
        for (int w = 0; w < GW; ++w) s += red.d[fq / F * GW + w][fq % F][i];
        // m(pi) sums a_j times the node values; the balanced objective's sums are of
        // p (la + log u_buf) + q (lb + log v_buf): times eps a_j
        const double sc = (i == 1 && fi[fq].balanced) ? ep.eps * (double)aj : (double)aj;
        ep.part[((size_t)(f0 + fq) * nh + jh) * NPART + 2 + i] = sc * s;
      }
    }
  }
  if constexpr (LONG) {
    if (threadIdx.x < F * G * NPART) {
      const int fq = threadIdx.x / NPART, i = threadIdx.x - fq * NPART;
      if (f0 + fq < nf && fi[fq].live && !(ep.mode == EPI_FINAL && i >= 2)) {
        double s = 0.0;
        for (int w = 0; w < GW; ++w) s += (double)red.v[fq / F * GW + w][0][fq % F * NPART + i];
        ep.part[((size_t)(f0 + fq) * nh + jh) * NPART + i] = s;
      }
    }
  } else {
    // four lanes a sum: the FP64 additions of one thread would be a chain that the CTA waits for
    constexpr int kSums = F * G * NPART;
    static_assert(4 * kSums <= NT && (4 * kSums < 32 || 4 * kSums % 32 == 0), "whole warps, or one");
    int tid = threadIdx.x;
    asm volatile("" : "+r"(tid));   // keeps a persistent kernel's loop from carrying the indices below
    if (tid < 4 * kSums) {
      const int x = tid >> 2, fq = x / NPART, i = x - fq * NPART;
      const int w0 = fq / F * GW, c = fq % F * NPART + i;
      double s = 0.0;
#pragma unroll
      for (int y = 0; y < (GW * P + 3) / 4; ++y) {
        const int e = 4 * y + (tid & 3);
        if (e < GW * P) s += (double)red.v[w0 + e / P][e % P][c];
      }
      constexpr unsigned kMask = 4 * kSums >= 32 ? 0xffffffffu : (1u << (4 * kSums % 32)) - 1;
      s += __shfl_xor_sync(kMask, s, 1);
      s += __shfl_xor_sync(kMask, s, 2);
      if ((tid & 3) == 0 && f0 + fq < nf && fi[fq].live && !(ep.mode == EPI_FINAL && i >= 2))
        ep.part[((size_t)(f0 + fq) * nh + jh) * NPART + i] = s;
    }
  }
}

}  // namespace shot
