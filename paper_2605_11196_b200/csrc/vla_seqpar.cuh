// Sequence-parallel VLA forward: the helper kernels around the chunk kernel.
//
// Section 3.4 writes the memory recurrence as a composition of per-token maps.  With the map
// acting on the right (S_t = S_{t-1} R_t + G_t, R_t = I - k_hat_t alpha_t^T, G_t = v_t alpha_t^T)
// a segment of tokens composes to S_end = S_start P + G with P = prod R_t and G the state the
// segment reaches from S = 0.  The penalty side needs no composition at all: A before token t
// is the inverse of M = lambda I + sum_{s<t} u_s u_s^T (Eq. "penalty"), a prefix SUM, so A at a
// segment start comes from a Gram matrix and one inversion.  A unit's sequence is therefore cut
// into P equal segments that are scanned at the same time:
//
//   1. gram     G_j = sum_{t in segment j} u_t u_t^T  (fp32 accuracy; sums in float pairs or fp64) and
//               the segment's sum of phi(k)
//   2. invert   A_start_j = (lambda I + sum_{i<j} G_i)^-1 in fp64 (Gauss-Jordan, no pivoting:
//               the matrix is symmetric positive definite), running key sum at the start;
//               with a carried-in A0, lambda I is replaced by A0^-1 (also formed in fp64)
//   3. scan     the pair kernel over units * P virtual units, three CTAs each: one carries A, one segment j from
//               S = 0 (readout o0_t, final state G_j), one its transfer scan from S = I with v = 0 (readout
//               w_t = P_t q_t / den_t, final state P_j)
//   4. combine  per unit, in order: S_start_{j+1} = S_start_j P_j + G_j
//   5. correct  o_t = o0_t + S_start_j w_t
//
// All of it is exact algebra; it costs about half more arithmetic than the plain scan (one A for both scans) and
// makes P times as many clusters, which is what a long sequence with few (batch, head) units needs.  16 units x 65536
// tokens at d = 64: 8.1 ms uncut, 2.72 in 16 segments (3.8 with both scans in one CTA of the FMA chunk kernel).
#pragma once

#include "vla_common.cuh"
#include "vla_mma.cuh"
#include "vla_seqpar_params.h"

namespace vla {


__device__ __forceinline__ float seqpar_phi(float x) { return x > 0.0f ? x + 1.0f : __expf(x); }

// ---- 1. Gram matrix and key sum of one slice of a segment.  Grid (units * P, kGramSplit): a
// segment's tokens are divided among kGramSplit CTAs of 256 threads, which add their results
// into the segment's (zeroed) matrix; the last segment of a unit needs neither and is skipped.
// Input rows: 8 lanes per token, 32 tokens per block, every load of a block in flight at once.

// The segments' tokens of one CTA: whole 32-token blocks except at the end
struct GramSlice { int unit, j, Ls, tlo, thi; };
__device__ __forceinline__ GramSlice gram_slice(const SeqParParams& p, int TB) {
  GramSlice s;
  s.unit = int(blockIdx.x) / p.P;
  s.j = int(blockIdx.x) % p.P;
  s.Ls = p.T / p.P;
  const int nblk = (s.Ls + TB - 1) / TB;
  s.tlo = int((long long)nblk * blockIdx.y / kGramSplit) * TB;
  s.thi = min(s.Ls, int((long long)nblk * (blockIdx.y + 1) / kGramSplit) * TB);
  return s;
}

// u = k_hat: unit rows, so the products run on warp-level tensor-core instructions in fp16.  The tensor core truncates when it
// adds, to one side, and over tens of thousands of tokens such a bias does not average out: with two rounded terms a factor
// (hi*hi + hi*lo + lo*hi) G's diagonal was 8e-8 short and A at a segment start up to four times as far off as with fp32
// products.  So a unit row, scaled to 2^9, is cut into a whole number H of at most ten bits and two fp16 terms M + L of the rest:
// every H H' and any sum of 32 of them (<= 2^23) is a whole number that fp32 holds, nothing is cut off, and the other products
// are 2^-10 of these or less.  Off from 64 bits in the 2-norm, 1024 to 8192 tokens a segment, every d: G 3e-8 to 9e-8 with two
// terms, 0.5e-8 to 5e-8 with fp32 FMAs, 0.1e-8 to 3e-8 so (what is left is the rounding of k_hat itself); A at a segment start,
// keys all alike, 2e-6 to 3.5e-5, 2e-6 to 9e-6, 3e-8 to 2e-7.  What bounded the FMA form was the fp64 addition of every 32-token
// partial sum (4096 of them at d = 64, at some 2 a clock and SM): here H H' is added in pairs of floats (the two-sum of
// Knuth, TAOCP 2, 4.2.2), and only a CTA's result goes to fp64.  A warp owns tiles of one 16-row strip; the next block's keys are
// fetched while this one is multiplied.  16 units x 65536 tokens, d = 64, bf16: 320 us with fp32 FMAs, 198 with two terms; the
// three products more cost the whole call 30 us (2.69 -> 2.72 ms), at d = 128 8 units x 32768 45 (2.49 -> 2.54).
template <int D>
struct GramUnitCfg {
  static constexpr int TB = 32;
  static constexpr uint32_t row = 6 * D + 16;   // H, M, L; an odd number of 16-byte pieces
  static constexpr uint32_t buf = TB * row, smem_bytes = 2 * buf;
};
template <int D, typename TIn>
__global__ void __launch_bounds__(256, D == 128 ? 1 : 2) seqpar_gram_unit_kernel(const SeqParParams p) {
  using Cfg = GramUnitCfg<D>;
  constexpr int TB = Cfg::TB, EPL = D / 8, F = EPL / 4;
  constexpr int NTW = D == 128 ? 8 : D == 64 ? 4 : 1;   // 16 x 8 tiles of a warp (d = 128: half the columns a CTA, blockIdx.z)
  constexpr int NG = NTW < 4 ? NTW : 4;                 // ... whose products are interleaved
  extern __shared__ __align__(128) unsigned char gram_smem[];
  const GramSlice sl = gram_slice(p, TB);
  if (sl.j == p.P - 1) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, tok = tid >> 3, pl = tid & 7;
  const bool ident = (p.flags & VLA_FLAG_IDENTITY_MAP) != 0;
  const int mt = D == 128 ? warp : D == 64 ? warp >> 1 : warp >> 2;
  const int nt0 = D == 128 ? 8 * int(blockIdx.z) : D == 64 ? 4 * (warp & 1) : warp & 3;
  const TIn* kk = static_cast<const TIn*>(p.k) + (size_t(sl.unit) * p.T + size_t(sl.j) * sl.Ls) * D;
  // ldmatrix addresses: the A operand's 16 columns of G, the B operand's eight (H and M; L of two tiles)
  const uint32_t lm = uint32_t((lane & 7) + (lane >> 4) * 8) * Cfg::row + ((lane >> 3) & 1) * 16 + mt * 32;
  const uint32_t lr = uint32_t((lane & 7) + ((lane >> 3) & 1) * 8) * Cfg::row + nt0 * 16;
  const uint32_t lk = lr + (lane >> 4) * (2 * D), ll = lr + (lane >> 4) * 16 + 4 * D;

  float2 hi[NTW][2], lo[NTW][2];
#pragma unroll
  for (int i = 0; i < NTW; ++i)
#pragma unroll
    for (int e = 0; e < 2; ++e) hi[i][e] = lo[i][e] = make_float2(0.f, 0.f);
  float zs[EPL] = {};
  float4 x[F];
  auto fetch = [&](int t0) {
    const int t = t0 + tok;
#pragma unroll
    for (int f = 0; f < F; ++f) x[f] = t < sl.thi ? load4(kk + size_t(t) * D, f * 8 + pl) : make_float4(0.f, 0.f, 0.f, 0.f);
  };
  if (sl.tlo < sl.thi) fetch(sl.tlo);
  const float2 m1 = make_float2(-1.0f, -1.0f);
  int ring = 0;
  for (int t0 = sl.tlo; t0 < sl.thi; t0 += TB, ring ^= 1) {
    const uint32_t base = smem_u32(gram_smem) + ring * Cfg::buf;
    {
      const bool act = t0 + tok < sl.thi;
      float ss = 0.0f;
#pragma unroll
      for (int f = 0; f < F; ++f) {
        if (act && !ident) x[f] = make_float4(seqpar_phi(x[f].x), seqpar_phi(x[f].y), seqpar_phi(x[f].z), seqpar_phi(x[f].w));
        zs[4 * f] += x[f].x; zs[4 * f + 1] += x[f].y; zs[4 * f + 2] += x[f].z; zs[4 * f + 3] += x[f].w;
        ss = fmaf(x[f].x, x[f].x, fmaf(x[f].y, x[f].y, fmaf(x[f].z, x[f].z, fmaf(x[f].w, x[f].w, ss))));
      }
#pragma unroll
      for (int off = 4; off >= 1; off >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, off);
      const float inv = 512.0f / fmaxf(sqrtf(ss), p.eps);
#pragma unroll
      for (int f = 0; f < F; ++f) {
        const float2 inv2 = make_float2(inv, inv), round = make_float2(12582912.0f, 12582912.0f);   // 1.5 * 2^23: to a whole number
        const float2 v[2] = {fmul2(make_float2(x[f].x, x[f].y), inv2), fmul2(make_float2(x[f].z, x[f].w), inv2)};
        uint32_t H[2], M[2], L[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const float2 h = ffma2(round, m1, fadd2(v[i], round)), r = ffma2(h, m1, v[i]);   // (both differences exact)
          asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(H[i]) : "f"(h.y), "f"(h.x));
          split_f16(r.x, r.y, M[i], L[i]);
        }
        const uint32_t at = base + uint32_t(tok) * Cfg::row + 8 * (f * 8 + pl);
        sts64(at, H[0], H[1]);
        sts64(at + 2 * D, M[0], M[1]);
        sts64(at + 4 * D, L[0], L[1]);
      }
    }
    __syncthreads();   // (two buffers: a warp that writes the next block's rows has passed this barrier after its last reads)
    fetch(t0 + TB);
#pragma unroll
    for (int n = 0; n < NTW; n += NG) {
      float y[NG][4], r[NG][4];   // H H', and the rest
#pragma unroll
      for (int i = 0; i < NG; ++i)
#pragma unroll
        for (int e = 0; e < 4; ++e) y[i][e] = r[i][e] = 0.f;
#pragma unroll
      for (int ks = 0; ks < 2; ++ks) {
        const uint32_t at = base + 16 * ks * Cfg::row;
        uint32_t aH[4], aM[4], aL[4], b[NG][4], bL[(NG + 1) / 2][4];
        ldsm_x4_t(aH, at + lm);
        ldsm_x4_t(aM, at + lm + 2 * D);
        ldsm_x4_t(aL, at + lm + 4 * D);
#pragma unroll
        for (int i = 0; i < NG; ++i) ldsm_x4_t(b[i], at + lk + 16 * (n + i));
#pragma unroll
        for (int i = 0; i < NG; i += 2) ldsm_x4_t(bL[i / 2], at + ll + 16 * (n + i));   // (d = 32: the second tile's is not used)
#pragma unroll
        for (int i = 0; i < NG; ++i) mma_f16(y[i], aH, b[i][0], b[i][1]);
#pragma unroll
        for (int i = 0; i < NG; ++i) mma_f16(r[i], aH, bL[i / 2][2 * (i & 1)], bL[i / 2][2 * (i & 1) + 1]);
#pragma unroll
        for (int i = 0; i < NG; ++i) mma_f16(r[i], aL, b[i][0], b[i][1]);
#pragma unroll
        for (int i = 0; i < NG; ++i) mma_f16(r[i], aM, b[i][2], b[i][3]);
#pragma unroll
        for (int i = 0; i < NG; ++i) mma_f16(r[i], aH, b[i][2], b[i][3]);
#pragma unroll
        for (int i = 0; i < NG; ++i) mma_f16(r[i], aM, b[i][0], b[i][1]);
      }
#pragma unroll
      for (int i = 0; i < NG; ++i)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          float2& h = hi[n + i][e];
          const float2 x2 = make_float2(y[i][2 * e], y[i][2 * e + 1]), sum = fadd2(h, x2), d = ffma2(h, m1, sum);
          const float2 err = fadd2(ffma2(ffma2(d, m1, sum), m1, h), ffma2(d, m1, x2));
          lo[n + i][e] = fadd2(lo[n + i][e], fadd2(err, make_float2(r[i][2 * e], r[i][2 * e + 1])));
          h = sum;
        }
    }
  }
  double* G = p.Gd + size_t(blockIdx.x) * D * D;
#pragma unroll
  for (int i = 0; i < NTW; ++i)
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      double* o = G + size_t(16 * mt + (lane >> 2) + 8 * e) * D + 8 * (nt0 + i) + 2 * (lane & 3);
      atomicAdd(o, (double(hi[i][e].x) + double(lo[i][e].x)) * (1.0 / 262144.0));
      atomicAdd(o + 1, (double(hi[i][e].y) + double(lo[i][e].y)) * (1.0 / 262144.0));
    }
  if (blockIdx.z == 0) {   // key sum: this thread's columns are (f * 8 + pl) * 4 + i; add over the 32 token slots
    __syncthreads();
    float* zpart = reinterpret_cast<float*>(gram_smem);
#pragma unroll
    for (int e = 0; e < EPL; ++e) zpart[tok * D + ((e / 4) * 8 + pl) * 4 + (e & 3)] = zs[e];
    __syncthreads();
    for (int c = tid; c < D; c += 256) {
      float s = 0.0f;
#pragma unroll
      for (int w = 0; w < TB; ++w) s += zpart[w * D + c];
      atomicAdd(&p.zsum[size_t(blockIdx.x) * D + c], s);
    }
  }
}

// An explicit u, of any norm: fp32 products (one scale per K step of fp16 products would not do for rows of different norms).
// Thread (ty, tx) of a 16 x 16 grid owns an R x R block of the D x D result, R = D / 16.
template <int D, typename TIn>
__global__ void __launch_bounds__(256) seqpar_gram_kernel(const SeqParParams p) {
  constexpr int R = D / 16;
  constexpr int TB = 32;          // tokens per shared-memory block (one fp32 partial sum)
  constexpr int EPL = D / 8;      // elements per lane of a token row (8 lanes per token)
  constexpr int LDU = D + 4;
  __shared__ __align__(16) float U[TB][LDU];
  __shared__ float zpart[TB][D];
  const int vu = blockIdx.x;
  const GramSlice sl = gram_slice(p, TB);
  const int unit = sl.unit, j = sl.j, Ls = sl.Ls, tlo = sl.tlo, thi = sl.thi;
  if (j == p.P - 1) return;
  const int tid = threadIdx.x;
  const int ty = tid >> 4, tx = tid & 15;
  const int tok = tid >> 3, pl = tid & 7;      // input stage: token of the block, lane of the token
  const bool ident = (p.flags & VLA_FLAG_IDENTITY_MAP) != 0;
  const TIn* kk = static_cast<const TIn*>(p.k) + (size_t(unit) * p.T + size_t(j) * Ls) * D;
  const TIn* uu = static_cast<const TIn*>(p.u) + (size_t(unit) * p.T + size_t(j) * Ls) * D;

  double accd[R][R];
#pragma unroll
  for (int a = 0; a < R; ++a)
#pragma unroll
    for (int b = 0; b < R; ++b) accd[a][b] = 0.0;
  float zs[EPL];
#pragma unroll
  for (int e = 0; e < EPL; ++e) zs[e] = 0.0f;

  for (int t0 = tlo; t0 < thi; t0 += TB) {
    // rows u_t of this block verbatim; the keys for their sum
    {
      const int t = t0 + tok;
      const bool act = t < thi;
#pragma unroll
      for (int f = 0; f < EPL / 4; ++f) {
        float4 k4 = make_float4(0.f, 0.f, 0.f, 0.f);
        if (act) k4 = load4(kk + size_t(t) * D, f * 8 + pl);
        if (act && !ident) {
          k4.x = seqpar_phi(k4.x); k4.y = seqpar_phi(k4.y);
          k4.z = seqpar_phi(k4.z); k4.w = seqpar_phi(k4.w);
        }
        zs[4 * f] += k4.x; zs[4 * f + 1] += k4.y; zs[4 * f + 2] += k4.z; zs[4 * f + 3] += k4.w;
        *reinterpret_cast<float4*>(&U[tok][(f * 8 + pl) * 4]) =
            act ? load4(uu + size_t(t) * D, f * 8 + pl) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
    __syncthreads();
    float acc[R][R];
#pragma unroll
    for (int a = 0; a < R; ++a)
#pragma unroll
      for (int b = 0; b < R; ++b) acc[a][b] = 0.0f;
#pragma unroll 4
    for (int tt = 0; tt < TB; ++tt) {
      float ra[R], cb[R];
#pragma unroll
      for (int a = 0; a < R; ++a) { ra[a] = U[tt][ty * R + a]; cb[a] = U[tt][tx * R + a]; }
#pragma unroll
      for (int a = 0; a < R; ++a)
#pragma unroll
        for (int b = 0; b < R; ++b) acc[a][b] = fmaf(ra[a], cb[b], acc[a][b]);
    }
#pragma unroll
    for (int a = 0; a < R; ++a)
#pragma unroll
      for (int b = 0; b < R; ++b) accd[a][b] += double(acc[a][b]);
    __syncthreads();
  }
  // the kGramSplit CTAs of a segment add into one matrix (zeroed by the host before the
  // launch): fp64 additions are scarce on this part, the inversion kernel should not repeat them
  double* G = p.Gd + size_t(vu) * D * D;
#pragma unroll
  for (int a = 0; a < R; ++a)
#pragma unroll
    for (int b = 0; b < R; ++b) atomicAdd(&G[(ty * R + a) * D + tx * R + b], accd[a][b]);
  // key sum: this thread's columns are (f * 8 + pl) * 4 + i; add over the 32 token slots
#pragma unroll
  for (int e = 0; e < EPL; ++e) zpart[tok][((e / 4) * 8 + pl) * 4 + (e & 3)] = zs[e];
  __syncthreads();
  for (int c = tid; c < D; c += 256) {
    float s = 0.0f;
#pragma unroll
    for (int w = 0; w < TB; ++w) s += zpart[w][c];
    atomicAdd(&p.zsum[size_t(vu) * D + c], s);
  }
}

// In-place Gauss-Jordan inversion of a symmetric positive definite D x D matrix held in
// registers by 256 threads (thread: row r, columns c0 .. c0 + EC - 1); no pivoting.  fp64
// arithmetic is scarce on this part: one FMA per element and pivot, the pivot's reciprocal
// folded into the column factor.
template <int D, int EC>
__device__ __forceinline__ void seqpar_gauss_jordan(double (&m)[EC], int r, int c0, double* rowraw,
                                                    double* colp) {
#pragma unroll 1
  for (int pv = 0; pv < D; ++pv) {
    if (r == pv) {
#pragma unroll
      for (int e = 0; e < EC; ++e) rowraw[c0 + e] = m[e];
    }
    if (pv >= c0 && pv < c0 + EC) {
      double x = 0.0;
#pragma unroll
      for (int e = 0; e < EC; ++e)
        if (c0 + e == pv) x = m[e];
      colp[r] = x;
    }
    __syncthreads();
    const double d = 1.0 / rowraw[pv];
    const double ncrd = -colp[r] * d;
    if (r == pv) {
#pragma unroll
      for (int e = 0; e < EC; ++e) m[e] = (c0 + e == pv) ? d : rowraw[c0 + e] * d;
    } else {
#pragma unroll
      for (int e = 0; e < EC; ++e) m[e] = (c0 + e == pv) ? ncrd : fma(ncrd, rowraw[c0 + e], m[e]);
    }
    __syncthreads();
  }
}

// ---- 2a. With a carried-in A0: M0 = A0^-1 per unit in fp64 (the penalty matrix the earlier
// tokens left behind).  One CTA of 256 threads per unit.
template <int D>
__global__ void __launch_bounds__(256) seqpar_m0_kernel(const SeqParParams p) {
  constexpr int EC = D * D / 256, TPR = D / EC;
  __shared__ double rowraw[D];
  __shared__ double colp[D];
  const int unit = blockIdx.x, tid = threadIdx.x;
  const int r = tid / TPR, c0 = (tid % TPR) * EC;
  double m[EC];
#pragma unroll
  for (int e = 0; e < EC; ++e) m[e] = double(p.A0[(size_t(unit) * D + r) * D + c0 + e]);
  seqpar_gauss_jordan<D, EC>(m, r, c0, rowraw, colp);
#pragma unroll
  for (int e = 0; e < EC; ++e) p.M0[(size_t(unit) * D + r) * D + c0 + e] = m[e];
}

// ---- 2. A at the start of segment j, and the running key sum there.  One CTA of 256
// threads per (unit, segment).  The matrix stays in registers: thread t owns D*D/256
// consecutive elements of one row; a pivot step exchanges only the pivot row and column
// through shared memory.
template <int D>
__global__ void __launch_bounds__(256) seqpar_invert_kernel(const SeqParParams p) {
  constexpr int EC = D * D / 256;     // elements per thread
  constexpr int TPR = D / EC;         // threads per row
  __shared__ double rowraw[D];        // pivot row before scaling
  __shared__ double colp[D];          // pivot column
  const int vu = blockIdx.x, unit = vu / p.P, j = vu % p.P;
  const int tid = threadIdx.x;
  const int r = tid / TPR, c0 = (tid % TPR) * EC;
  float* A = p.Astart + size_t(vu) * D * D;
  for (int c = tid; c < D; c += 256) {
    double s = p.z0 ? double(p.z0[size_t(unit) * D + c]) : 0.0;
    // the identity-map reading has no readout normaliser: the key sum is carried through
    if (!(p.flags & VLA_FLAG_IDENTITY_MAP))
      for (int i = 0; i < j; ++i) s += double(p.zsum[(size_t(unit) * p.P + i) * D + c]);
    p.zstart[size_t(vu) * D + c] = float(s);
  }
  if (j == 0) {
    const float dg = 1.0f / p.lambda;
#pragma unroll
    for (int e = 0; e < EC; ++e)
      A[r * D + c0 + e] = p.A0 ? p.A0[(size_t(unit) * D + r) * D + c0 + e] : ((c0 + e == r) ? dg : 0.0f);
    return;
  }
  // M = lambda I (or the carried-in A0^-1) + the Gram matrices of the earlier segments
  double m[EC];
#pragma unroll
  for (int e = 0; e < EC; ++e)
    m[e] = p.A0 ? p.M0[(size_t(unit) * D + r) * D + c0 + e] : ((c0 + e == r) ? double(p.lambda) : 0.0);
  for (int i = 0; i < j; ++i) {
    const double* G = p.Gd + (size_t(unit) * p.P + i) * D * D + r * D + c0;
#pragma unroll
    for (int e = 0; e < EC; ++e) m[e] += G[e];
  }
  seqpar_gauss_jordan<D, EC>(m, r, c0, rowraw, colp);
#pragma unroll
  for (int e = 0; e < EC; ++e) A[r * D + c0 + e] = float(m[e]);
}

// ---- 4. states at the segment starts, in order: S_start_{j+1} = S_start_j P_j + G_j.  The rows
// of S do not mix, so a unit is spread over D / 16 CTAs of 16 rows each: grid (units, D / 16),
// 256 threads (thread = one row of the block, D / 16 columns).  A chain of P steps, each bound by P_j's way from
// global memory: the next one is fetched into registers while a step computes (d = 32, 4 units x 16384 tokens in
// 64 segments: the whole call 271 -> 187 us).  The unit's first CTA also copies the last segment's A and key sum out.
template <int D>
__global__ void __launch_bounds__(256) seqpar_combine_kernel(const SeqParParams p, float* A_T, float* zT, const float* AT2,
                                                             const float* zT2) {
  extern __shared__ __align__(16) unsigned char seqpar_smem[];
  constexpr int LD = D + 4, R = D / 16, RB = 16, NF = D * D / 1024;
  float* Sc = reinterpret_cast<float*>(seqpar_smem);   // [RB][LD] current rows of S_start
  float* Pj = Sc + RB * LD;                            // [D][LD]
  const int unit = blockIdx.x, row0 = blockIdx.y * RB, tid = threadIdx.x;
  const int ty = tid >> 4, tx = tid & 15;
  const size_t N = size_t(p.units) * p.P;
  float s[R], g[R];
  float4 pre[NF];
  const size_t own = size_t(row0 + ty) * D + tx * R;   // this thread's entries of a D x D matrix
  auto fetch = [&](int j) {
    const size_t vu = size_t(unit) * p.P + j;
    const float4* Pg = reinterpret_cast<const float4*>(p.ST2 + (N + vu) * D * D);
#pragma unroll
    for (int i = 0; i < NF; ++i) pre[i] = Pg[i * 256 + tid];
#pragma unroll
    for (int b = 0; b < R; ++b) g[b] = p.ST2[vu * D * D + own + b];
  };
  fetch(0);
#pragma unroll
  for (int b = 0; b < R; ++b) s[b] = p.S0 ? p.S0[size_t(unit) * D * D + own + b] : 0.0f;
  for (int j = 0; j < p.P; ++j) {
    float* Ss = p.Sstart + (size_t(unit) * p.P + j) * D * D + own;
    float acc[R];
#pragma unroll
    for (int b = 0; b < R; ++b) {
      Ss[b] = s[b];
      Sc[ty * LD + tx * R + b] = s[b];
      acc[b] = g[b];
    }
#pragma unroll
    for (int i = 0; i < NF; ++i) {
      const int at = 4 * (i * 256 + tid);
      *reinterpret_cast<float4*>(&Pj[(at / D) * LD + at % D]) = pre[i];
    }
    __syncthreads();
    if (j + 1 < p.P) fetch(j + 1);
#pragma unroll 4
    for (int m = 0; m < D; ++m) {
      const float sa = Sc[ty * LD + m];
      float pr[R];
#pragma unroll
      for (int b = 0; b < R; b += 2) *reinterpret_cast<float2*>(pr + b) = *reinterpret_cast<const float2*>(&Pj[m * LD + tx * R + b]);
#pragma unroll
      for (int b = 0; b < R; ++b) acc[b] = fmaf(sa, pr[b], acc[b]);
    }
    __syncthreads();
#pragma unroll
    for (int b = 0; b < R; ++b) s[b] = acc[b];
  }
  const size_t last = size_t(unit) * p.P + p.P - 1;
#pragma unroll
  for (int b = 0; b < R; ++b) {
    if (p.S_T) p.S_T[size_t(unit) * D * D + own + b] = s[b];
    if (A_T) A_T[size_t(unit) * D * D + own + b] = AT2[last * D * D + own + b];
  }
  if (zT && row0 == 0 && tid < D) zT[size_t(unit) * D + tid] = zT2[last * D + tid];
}

// ---- 5. o_t += S_start_j w_t.  Grid (units * P, ceil(Ls / kCorrectTokens)), 8 warps; a warp takes 16 tokens at a
// time, all D rows of S_start_j.  fp32 operands as two tf32 terms, all four products (lanes
// take float4 pairs 2 c4, 2 c4 + 1 of every 32 columns, conflict-free at a row stride of D + 4); S_start_j is split once per CTA.
// Bound by memory (w once, o twice): the fp32-FMA form before it waited on its shared-memory operands (335 us of the
// 3.12 ms at d = 64, 16 units x 65536 tokens; the whole call is 2.96 ms now).
constexpr int kCorrectTokens = 512;

template <int D>
__global__ void __launch_bounds__(256, D == 128 ? 1 : 2) seqpar_correct_kernel(const SeqParParams p) {
  extern __shared__ __align__(16) unsigned char seqpar_smem[];
  constexpr int LD = D + 4, NT = D / 8;
  uint32_t* Sh = reinterpret_cast<uint32_t*>(seqpar_smem);   // [D][LD] upper terms
  uint32_t* Sl = Sh + D * LD;                                // [D][LD] remainders
  const int vu = blockIdx.x, j = vu % p.P;
  if (j == 0 && !p.S0) return;                 // S_start = 0: nothing to add
  const int Ls = p.T / p.P;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, c4 = lane & 3;
  const float4* Sg = reinterpret_cast<const float4*>(p.Sstart + size_t(vu) * D * D);
  for (int idx = tid; idx < D * D / 4; idx += 256) {
    const float4 x = Sg[idx];
    uint4 h, l;
    split_tf32(x.x, h.x, l.x); split_tf32(x.y, h.y, l.y); split_tf32(x.z, h.z, l.z); split_tf32(x.w, h.w, l.w);
    const int at = (idx / (D / 4)) * LD + (idx % (D / 4)) * 4;
    *reinterpret_cast<uint4*>(Sh + at) = h;
    *reinterpret_cast<uint4*>(Sl + at) = l;
  }
  __syncthreads();
  const int end = min(Ls, (int(blockIdx.y) + 1) * kCorrectTokens);
#pragma unroll 1
  for (int t0 = blockIdx.y * kCorrectTokens + warp * 16; t0 < end; t0 += 8 * 16) {
    float acc[NT][4];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[nt][e] = 0.0f;
#pragma unroll 1
    for (int c0 = 0; c0 < D; c0 += 32) {
      uint32_t ah[4][4], al[4][4];     // [8 columns]
      {
        float4 x[2][2];
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
          const int t = t0 + 8 * hf + g;
          const float4* w = reinterpret_cast<const float4*>(p.wn + (size_t(vu) * Ls + t) * D + c0) + 2 * c4;
#pragma unroll
          for (int k = 0; k < 2; ++k) x[hf][k] = t < end ? w[k] : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const float u0[4] = {x[0][k].x, x[0][k].y, x[1][k].x, x[1][k].y};
          const float u1[4] = {x[0][k].z, x[0][k].w, x[1][k].z, x[1][k].w};
          split_frag_tf32(u0, ah[2 * k], al[2 * k]);
          split_frag_tf32(u1, ah[2 * k + 1], al[2 * k + 1]);
        }
      }
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) {
        const int at = (8 * nt + g) * LD + c0 + 8 * c4;
        uint32_t bh[8], bl[8];
        *reinterpret_cast<uint4*>(bh) = *reinterpret_cast<const uint4*>(Sh + at);
        *reinterpret_cast<uint4*>(bh + 4) = *reinterpret_cast<const uint4*>(Sh + at + 4);
        *reinterpret_cast<uint4*>(bl) = *reinterpret_cast<const uint4*>(Sl + at);
        *reinterpret_cast<uint4*>(bl + 4) = *reinterpret_cast<const uint4*>(Sl + at + 4);
        {
          float y[4][4];
#pragma unroll
          for (int q = 0; q < 4; ++q) mma_tf32_zero(y[q], al[q], bl[2 * q], bl[2 * q + 1]);
#pragma unroll
          for (int q = 0; q < 4; ++q) mma_tf32(y[q], al[q], bh[2 * q], bh[2 * q + 1]);
#pragma unroll
          for (int q = 0; q < 4; ++q) mma_tf32(y[q], ah[q], bl[2 * q], bl[2 * q + 1]);
#pragma unroll
          for (int q = 0; q < 4; ++q) mma_tf32(y[q], ah[q], bh[2 * q], bh[2 * q + 1]);
#pragma unroll
          for (int e = 0; e < 4; ++e) acc[nt][e] += (y[0][e] + y[1][e]) + (y[2][e] + y[3][e]);
        }
      }
    }
#pragma unroll
    for (int hf = 0; hf < 2; ++hf) {
      const int t = t0 + 8 * hf + g;
      if (t >= end) continue;
      float2* o = reinterpret_cast<float2*>(p.out + (size_t(vu) * Ls + t) * D + 2 * c4);
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) {
        float2 x = o[4 * nt];
        x.x += acc[nt][2 * hf];
        x.y += acc[nt][2 * hf + 1];
        o[4 * nt] = x;
      }
    }
  }
}

}  // namespace vla
