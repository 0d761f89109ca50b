// Per-order Legendre contractions of the semi-naive SHT in FP32 (SIMT FFMA).
//
// Analysis (App. B, quadrature form; the area weights a_j are already folded into X by
// the ring DFT), for every block (m, p) and every column c = (field, re/im):
//   C[i][c] = h_{l} * sum_{jh < nh} Pbar_{l m}(x_jh) X[jh][c],   l = m + p + 2 i
// with h_l = exp(-t l(l+1)) (Sec. 3.2) or 1 for a plain transform.
// Synthesis, the transpose contraction over degrees:
//   Y[jh][c] = sum_i Pbar_{l m}(x_jh) C[i][c]
// Both are GEMMs with N = 2 * nfields columns.  The table is stored [i][jh] (jh
// contiguous): it is the K-contiguous A operand of the analysis and the M-contiguous A
// operand of the synthesis.  The tile lists are built at grid set-up so that large blocks are
// scheduled first.
#include "shot_internal.cuh"

namespace shot {

namespace {

// One CTA (two warps) computes a 64 x BN half of a tile of one block's product, BN = 8 TN; a warp
// owns 32 of the rows, a thread 8 rows x TN columns as TN/2 packed column pairs.  The terms arrive
// by cp.async in a ring of kSimtStages chunks of 16.
//
// What bounds it: FP32 FMA issue.  Packed FMAs (fma.rn.f32x2: two columns an instruction, at half
// the rate of a scalar FMA, so the same peak) leave every second issue slot to the shared-memory
// loads: 8 x 6 threads measured 67 TFLOP/s packed against 58 scalar in a loop without global
// loads, where the loads' words (14 a term for 48 FMAs) take the shared memory's bandwidth.
// Registers (96 a thread) hold 20 warps on an SM, so the warps must be busy ones: the blocks have
// 1 to lmax/2 rows, and with 64-row CTAs 8 % of the warps have no row (21 % with 128-row ones); a
// warp without rows skips its arithmetic, and a last chunk stops at its last term.  TMA chunks
// (64-byte rows) were slower than cp.async where the table streams (8 fields at 512 rings: 0.061
// against 0.047 ms).
//
// Measured, analysis / synthesis in ms, against a kernel of scalar FMAs on 128-row tiles with one
// chunk in flight: 720 rings, 24 fields 0.256 / 0.233 -> 0.230 / 0.186; 512 rings, 8 fields 0.087 /
// 0.068 -> 0.047 / 0.037 (16-column tiles instead of 32); 256 rings, 32 fields 0.047 / 0.030 ->
// 0.034 / 0.021.
constexpr int BM = 64, BK = 16, NT = 64, kSimtStages = 3;
constexpr int kAElems = BM * BK;

__device__ __forceinline__ void cp16(float* dst, const float* src, bool valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src), "r"(valid ? 16 : 0)
               : "memory");
}
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 dup2(float x) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ void fma2(f32x2& d, f32x2 a, f32x2 b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}

template <int TN, bool ANALYSIS>
__global__ void __launch_bounds__(NT, TN >= 6 ? 8 : 10) k_legendre_simt(
    const Tile* __restrict__ tiles, int ncolt, const float* __restrict__ tab, int ldt,
    const long long* __restrict__ row_off, const int* __restrict__ Mrows, int nh,
    const float* __restrict__ Bsrc, int ldc, int ncols, float* __restrict__ out,
    const float* __restrict__ h, int polar) {
  constexpr int BN = 8 * TN, NP = TN / 2;
  // [stage]: A (analysis: 64 rows of 16 terms, the 16-byte pieces of rows 2 i and 2 i + 1 permuted
  // by i so that the rows a warp reads together lie on different banks; synthesis: 16 terms of 64
  // nodes), B [term][BN]
  __shared__ __align__(16) float As[kSimtStages][kAElems];
  __shared__ __align__(16) float Bs[kSimtStages][BK * BN];

  const int half = blockIdx.x / ncolt;   // CTA = (128-row tile, half of it, column tile)
  const Tile tl = tiles[half >> 1];
  const int blk = tl.blk, r0 = tl.r0 + (half & 1) * BM;
  const int n0 = (blockIdx.x - half * ncolt) * BN;
  const int m = blk >> 1, p = blk & 1;
  const int M = Mrows[blk];
  const long long ro = row_off[blk];
  const int K = ANALYSIS ? nh : M;
  const int mvalid = ANALYSIS ? M : nh;   // rows of the output block
  if (r0 >= mvalid) return;
  const int ks = polar ? tl.k0[half & 1] : 0;   // first term of the sums

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int tn = lane & 7, tm = lane >> 3;
  // this thread's pieces of a chunk: A rows (analysis) tid/4 + 16 s, piece tid%4; A terms
  // (synthesis) tid/16 + 4 s, nodes 4 (tid%16); B term tid%16, columns 4 (tid/16) + 16 s
  const float* Ap = ANALYSIS ? tab + (ro + r0 + (tid >> 2)) * ldt + (tid & 3) * 4
                             : tab + (ro + (tid >> 4)) * ldt + r0 + (tid & 15) * 4;
  const bool a_in = ANALYSIS || r0 + (tid & 15) * 4 < ldt;
  const float* Bp = (ANALYSIS ? Bsrc + (size_t)blk * nh * ldc : Bsrc + ro * ldc) + (size_t)(tid & 15) * ldc + n0 +
                    (tid >> 4) * 4;
  const int a_dst = ANALYSIS ? (tid >> 2) * BK + (((tid & 3) ^ ((tid >> 3) & 3)) << 2) : tid * 4;
  const int b_dst = (tid & 15) * BN + (tid >> 4) * 4;
  auto load = [&](int kt, int st) {
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      if (ANALYSIS) {
        const bool ok = r0 + (tid >> 2) + 16 * s < M;
        cp16(&As[st][a_dst + 16 * s * BK], ok ? Ap + (size_t)(16 * s) * ldt + kt : tab, ok);
      } else {
        const bool ok = a_in && kt + (tid >> 4) + 4 * s < M;
        cp16(&As[st][a_dst + 4 * s * BM], ok ? Ap + (size_t)(kt + 4 * s) * ldt : tab, ok);
      }
    }
#pragma unroll
    for (int s = 0; s < BN / 16; ++s) {
      const bool ok = kt + (tid & 15) < K && n0 + (tid >> 4) * 4 + 16 * s < ncols;
      cp16(&Bs[st][b_dst + 16 * s], ok ? Bp + (size_t)kt * ldc + 16 * s : Bsrc, ok);
    }
  };

  const int wrow = warp * 32;
  const bool busy = r0 + wrow < mvalid;
  f32x2 acc[8][NP];
#pragma unroll
  for (int r = 0; r < 8; ++r)
#pragma unroll
    for (int c = 0; c < NP; ++c) acc[r][c] = 0;

#pragma unroll
  for (int t = 0; t < kSimtStages - 1; ++t) {
    if (ks + t * BK < K) load(ks + t * BK, t);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  int s = 0;
  for (int kt = ks; kt < K; kt += BK) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kSimtStages - 2) : "memory");
    __syncthreads();   // this chunk has landed for both warps, and the one before it has been read
    if (kt + (kSimtStages - 1) * BK < K) load(kt + (kSimtStages - 1) * BK, s == 0 ? kSimtStages - 1 : s - 1);
    asm volatile("cp.async.commit_group;" ::: "memory");
    if (busy) {
      const float* A = As[s];
      const float* B = Bs[s] + 2 * tn;
      // thread rows: analysis tm + 4 r (kT terms at once), synthesis 4 tm + {0..3} and
      // 16 + 4 tm + {0..3}
      constexpr int kT = 4;
      auto terms = [&](int k0, int nt) {
        float4 av[8];
        if (ANALYSIS) {
          const float* q = A + (wrow + tm) * BK;
          const int c0 = ((k0 >> 2) ^ (tm >> 1)) << 2, c1 = c0 ^ 8;
#pragma unroll
          for (int r = 0; r < 8; ++r) av[r] = *reinterpret_cast<const float4*>(q + 4 * r * BK + ((r & 1) ? c1 : c0));
        }
#pragma unroll
        for (int kk = 0; kk < kT; ++kk) {
          if (kk >= nt) break;
          float x[8];
          if (ANALYSIS) {
#pragma unroll
            for (int r = 0; r < 8; ++r) x[r] = kk == 0 ? av[r].x : kk == 1 ? av[r].y : kk == 2 ? av[r].z : av[r].w;
          } else {
            const float4 u = *reinterpret_cast<const float4*>(A + (k0 + kk) * BM + wrow + 4 * tm);
            const float4 v = *reinterpret_cast<const float4*>(A + (k0 + kk) * BM + wrow + 16 + 4 * tm);
            x[0] = u.x; x[1] = u.y; x[2] = u.z; x[3] = u.w;
            x[4] = v.x; x[5] = v.y; x[6] = v.z; x[7] = v.w;
          }
          f32x2 b[NP];
#pragma unroll
          for (int c = 0; c < NP; ++c) b[c] = *reinterpret_cast<const f32x2*>(B + (k0 + kk) * BN + 16 * c);
#pragma unroll
          for (int r = 0; r < 8; ++r) {
            const f32x2 xr = dup2(x[r]);
#pragma unroll
            for (int c = 0; c < NP; ++c) fma2(acc[r][c], xr, b[c]);
          }
        }
      };
      const int kend = min(BK, K - kt);
      int k0 = 0;
#pragma unroll 2
      for (; k0 + kT <= kend; k0 += kT) terms(k0, kT);
      if (k0 < kend) terms(k0, kend - k0);
    }
    if (++s == kSimtStages) s = 0;
  }
  if (!busy) return;

#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const int row = r0 + wrow + (ANALYSIS ? tm + 4 * r : 4 * tm + (r & 3) + 16 * (r >> 2));
    if (row >= mvalid) continue;
    float sc = 1.f;
    float* o;
    if (ANALYSIS) {
      if (h) sc = h[m + p + 2 * row];
      o = out + (size_t)(ro + row) * ldc;
    } else {
      o = out + ((size_t)blk * nh + row) * ldc;
    }
#pragma unroll
    for (int c = 0; c < NP; ++c) {
      const int col = n0 + 16 * c + 2 * tn;
      const float2 v = *reinterpret_cast<const float2*>(&acc[r][c]);
      if (col < ncols) *reinterpret_cast<float2*>(o + col) = make_float2(v.x * sc, v.y * sc);
    }
  }
}

template <int TN, bool ANALYSIS>
int launch_one(const Grid& g, int nf, const float* B, float* out, int ldc, const float* h, bool polar,
               cudaStream_t st) {
  const int ncols = 2 * nf, ncolt = (ncols + 8 * TN - 1) / (8 * TN);
  ProfScope prof(ANALYSIS ? PK_ANALYSIS : PK_SYNTHESIS, st);
  count_launch();
  k_legendre_simt<TN, ANALYSIS><<<2 * (ANALYSIS ? g.ntiles_ana : g.ntiles_syn) * ncolt, NT, 0, st>>>(
      ANALYSIS ? g.tiles_ana : g.tiles_syn, ncolt, g.tab, g.ldt, g.row_off_d, g.M_d, g.nh, B, ldc, ncols, out, h, polar);
  SHOT_CUDA(cudaGetLastError());
  return SHOT_OK;
}

template <int TN>
int launch_pair(const Grid& g, int nf, const float* X, float* C, float* Y, int ldc, bool ana, bool syn,
                const float* h, cudaStream_t st) {
  int rc = SHOT_OK;
  if (ana) rc = launch_one<TN, true>(g, nf, X, C, ldc, h, ana && syn, st);
  if (!rc && syn) rc = launch_one<TN, false>(g, nf, C, Y, ldc, nullptr, ana && syn, st);
  return rc;
}

int dispatch(const Grid& g, int nf, const float* X, float* C, float* Y, int ldc, bool ana, bool syn,
             const float* h, cudaStream_t st) {
  // the tile width: the tuned one, else the one that pads the columns least (the wider on a tie,
  // for more FMAs per shared-memory load and fewer passes over the table)
  int bn = (g.active.nf == nf) ? g.active.simt_bn : 0;
  if (bn == 0) {
    const int ncols = 2 * nf;
    auto padded = [&](int b) { return (ncols + b - 1) / b * b; };
    bn = 64;
    for (int b : {48, 32, 16})
      if (padded(b) < padded(bn)) bn = b;
    if (ncols > 64 && bn < 48) bn = padded(64) <= padded(48) ? 64 : 48;
  }
  switch (bn) {
    case 16: return launch_pair<2>(g, nf, X, C, Y, ldc, ana, syn, h, st);
    case 32: return launch_pair<4>(g, nf, X, C, Y, ldc, ana, syn, h, st);
    case 48: return launch_pair<6>(g, nf, X, C, Y, ldc, ana, syn, h, st);
    default: return launch_pair<8>(g, nf, X, C, Y, ldc, ana, syn, h, st);
  }
}

}  // namespace

int launch_legendre_simt(const Grid& g, int nf, const float* X, float* C, float* Y, int ldc, cudaStream_t st) {
  return dispatch(g, nf, X, C, Y, ldc, true, true, g.h_d, st);
}

int launch_analysis_simt(const Grid& g, int nf, const float* X, float* C, int ldc, bool apply_h,
                         cudaStream_t st) {
  return dispatch(g, nf, X, C, nullptr, ldc, true, false, apply_h ? g.h_d : nullptr, st);
}

int launch_synthesis_simt(const Grid& g, int nf, const float* C, float* Y, int ldc, cudaStream_t st) {
  return dispatch(g, nf, nullptr, const_cast<float*>(C), Y, ldc, false, true, nullptr, st);
}

}  // namespace shot
