// fwd_h_tile.cuh -- lifted-feature evaluation on the tensor cores with FP16
// operands split into high and low halves (ndg_forward, NDG_MODE_TC).
//
// Same quadratic-form evaluation as the TF32 kernels: for a tile with centre
// c the exponent of Eq. 1 is  s = phi(x~) . coef  with lifted features
// phi = [x~_i x~_j (j <= i), x~_i, 1] and per-(Gaussian, tile) coefficients
// coef = [A_ii | 2 A_ij, -2 A m~, m~^T A m~] * (-log2(e) / 2), A = M^T M.
// Here the operands are FP16 pairs v = hi + lo (11 + 11 significant bits,
// three products hi hi + hi lo + lo hi accumulated in FP32), which runs at
// twice the TF32 rate and halves the operand bytes.  FP16 has a narrow
// exponent range, so both sides are rescaled by powers of two (exact):
//   * per tile and dimension, x~_d is divided by h_d = 2^ceil(log2 half-extent),
//     so the features lie in [-1, 1];  the coefficients take the inverse
//     factors (h_i h_j for the quadratic terms, h_i for the linear ones);
//   * per candidate, a row whose largest coefficient exceeds 2^14 is divided
//     by 2^k; the epilogue multiplies the accumulator back by 2^k (the
//     stage carries a flag so that chunks without such rows skip it).
//
// CTA = one tile of up to 256 queries (two M = 128 row blocks sharing the
// candidate operand), 544 threads (96 registers), one CTA per SM.  What bounds
// the tile: at N = 6 the epilogue's chain of exponentials and colour sums, at
// N = 10 the MMAs (30 per chunk, at 70 cycles each against 48 alone, behind
// the shared-memory pipe).  What the layout answers to:
//   * the shared-memory pipe, shared by the MMAs' operand reads (a wavefront
//     per 128 bytes), the weight loads and the coefficient rows, was 68%
//     (N = 6) to 82% (N = 10) busy with Phi as a shared-memory operand.  Phi,
//     the same for all of a tile's chunks, is the A operand in tensor memory
//     (hi and lo; N = 10, 11 keep one block's lo in shared memory, N = 12 both),
//     and the chunks are of 96 candidates so that two double-buffered
//     accumulators and Phi share the 512 columns (an MMA of 96 columns costs
//     its share of one of 128);
//   * one builder warp per SM sub-partition issued an instruction every four
//     cycles and waited for its own record loads: eight builder warps (six at
//     N = 12), records by cp.async a group ahead, consecutive lanes copying
//     consecutive parts of a record;
//   * MUFU and FMA took turns inside an epilogue warp: the exponentials of 16
//     columns are issued with the sums of the 16 before.
// Measured, kernel alone: N = 6 256 x 256 frame (10,000 Gaussians) 235 -> 178
// us, N = 8 701 x 397 (60,000) 5.72 -> 4.20 ms, N = 10 480 x 272 (100,000)
// 6.79 -> 5.37 ms, N = 10 1080p (500,000) 491 -> 397 ms, N = 12 evaluation
// (10,000, 32,768 queries) 303 -> 233 us.  Four builders with 13 warps and
// eight rows per weight load measured 124 us where this takes 112 (N = 8,
// 5,000 Gaussians; 159 at first).
//   warps 0-7   builders: a warp turns its 32 candidates of a chunk into
//               coefficient rows (FP16 hi / lo, K-major no-swizzle layout)
//               and weight pair entries in one of CS shared-memory stages
//               and arrives on coef_full;
//   warps 8-15  epilogue: warps 8-11 serve row block 0, 12-15 row block 1;
//               warp w reads TMEM lanes 32 (w % 4) .. + 31 of its block with
//               the 16x256b load shape (a thread holds 4 rows x 2 columns of
//               every 8-column group, so each weight load serves four rows),
//               forms e = 2^s and accumulates w e; row sums are completed
//               with shuffles at the end;
//   warp 16     MMA issuer: one lane issues the MMAs of a row block of chunk i
//               once its stage is full and that block of accumulator buffer
//               i & 1 is free, commits them to acc_full and, after both
//               blocks, to coef_empty.
// Barrier operations are one per warp (an elected lane), and every wait is
// bounded: on a timeout the kernel records NDG_ERR_TIMEOUT, lets the issued
// MMAs finish (bounded), frees its tensor memory and returns.
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "common.cuh"
#include "internal.h"
#include "kernels.h"
#include "tcgen05.cuh"

namespace ndg {

// Warps of the forward's CTA: builders, epilogue, issuer.
constexpr int kFwdBuilders = 8;
constexpr int kFwdEpi0 = kFwdBuilders, kFwdIssuer = kFwdBuilders + 8;
constexpr int kFwdThreads = 32 * (kFwdIssuer + 1);

// Barriers and small shared state of one tile, sized for the largest shape
// (CS <= 4 coefficient stages, N <= 12).
struct FwdHSync {
  // accumulator barriers per (buffer, row block): index 2 b + h
  uint64_t coef_full[4], coef_empty[4], acc_full[4], acc_empty[4], drain;
  static constexpr int kBarriers = 17;
  uint32_t tmem_base;
  float sred[8 * 12 * 2];
  float sctr[12], sh[12];
  __align__(16) int sflag[4][4];  // per stage and 32-candidate group: a row was scaled
  int s_abort;
};

static_assert(sizeof(FwdHSync) <= 1536, "static shared memory");

template <int N>
struct FwdHShape {
  static constexpr int P = tri(N);
  static constexpr int F = P + N + 1;
  static constexpr int KP = (F + 15) / 16 * 16;  // K step of kind::f16 is 16
  static constexpr int NC = 96;                  // candidates per chunk (MMA N)
  static constexpr int GPC = NC / 32;            // builder groups (one warp's 32) per chunk
  static constexpr int R = rec_floats(N);
  static constexpr uint32_t SBO = (KP / 8) * 128;  // 8-row group stride (bytes)
  // tensor memory: four accumulators (buffer, row block) of NC columns, then
  // Phi as the MMAs' A operand, KP / 2 columns per row block and half: hi of
  // both blocks, and lo of as many (LO_TM) as the 512 columns hold: both for
  // N <= 9, one for N = 10, 11
  static constexpr uint32_t TM_PHI = 4u * NC;
  static constexpr int LO_TM = TM_PHI + 2 * KP <= 512 ? 2 : TM_PHI + KP + KP / 2 <= 512 ? 1 : 0;
  static_assert(TM_PHI + KP <= 512, "tensor memory");
  static constexpr uint32_t PHI_BYTES = (2 - LO_TM) * 128u * KP * 2;  // the other lo halves, in shared memory
  static constexpr uint32_t HALF_BYTES = 128u * KP * 2;  // one 128-row block of it
  static constexpr uint32_t B_BYTES = (uint32_t)NC * KP * 2;
  static constexpr uint32_t W_BYTES = (uint32_t)NC * 16;  // w0 w0' w1 w1' w2 w2' k k' per pair
  static constexpr uint32_t C_STAGE = 2 * B_BYTES + W_BYTES;
  // coefficient stages: as many as fit next to Phi (at most 4; 2 KB are left
  // for the static shared variables).  The builders run up to CS chunks ahead
  // of the epilogue, which frees a stage only at the end of its chunk.
  static constexpr uint32_t REC_STRIDE = (R / 4) | 1;  // float4s: odd, so that lanes' rows miss no bank
  static constexpr int BW = N <= 11 ? kFwdBuilders : 6;  // builder warps with room for their records
  static constexpr uint32_t REC_BYTES = (uint32_t)BW * 32 * REC_STRIDE * 16;  // a group of records per builder warp
  static constexpr uint32_t STAGE_ROOM = 227u * 1024u - 2048u - PHI_BYTES - REC_BYTES - 128u;
  static constexpr int CS = STAGE_ROOM / C_STAGE >= 4 ? 4 : (int)(STAGE_ROOM / C_STAGE);
  static constexpr uint32_t SMEM_USED = PHI_BYTES + CS * C_STAGE + REC_BYTES + 128;
  // more than half of the SM's shared memory: one CTA per SM
  static constexpr uint32_t SMEM = SMEM_USED > 116u * 1024u ? SMEM_USED : 116u * 1024u;
  static_assert(SMEM + 2048 <= 227u * 1024u, "shared memory");  // 2 KB: static variables
  static_assert(CS >= 2, "coefficient stages");
};

namespace {

// Splits (v0, v1) into FP16 high and low halves, packed as half2 words.
__device__ __forceinline__ void split_h2(float v0, float v1, uint32_t& hi, uint32_t& lo) {
  const __half2 h = __floats2half2_rn(v0, v1);
  const float2 hf = __half22float2(h);
  const __half2 l = __floats2half2_rn(v0 - hf.x, v1 - hf.y);
  hi = *reinterpret_cast<const uint32_t*>(&h);
  lo = *reinterpret_cast<const uint32_t*>(&l);
}

// Byte offset of element (row, k) of a K-major no-swizzle FP16 operand.
__device__ __forceinline__ uint32_t kmajor_off_h(int row, int k, uint32_t sbo) {
  return (uint32_t)(row >> 3) * sbo + (uint32_t)(k >> 3) * 128u + (uint32_t)(row & 7) * 16u +
         (uint32_t)(k & 7) * 2u;
}

constexpr float kNegHalfLog2eH = -0.72134752044448170368f;
constexpr float kRowMax = 16384.0f;  // coefficient rows are kept below 2^14 (FP16 max 65504)

}  // namespace

// The CTA's barriers and small shared state, and its dynamic shared memory
// (no rounding of its address: the alignment is declared, and every offset
// then is a constant).
static __shared__ FwdHSync s_fwd;
__device__ __forceinline__ FwdHSync& fwd_sync() { return s_fwd; }
__device__ __forceinline__ uint8_t* fwd_smem() {
  extern __shared__ __align__(1024) uint8_t dsm[];
  return dsm;
}

// Query tile t on the tensor cores, by the whole CTA.  The caller owns the
// tensor memory (all 512 columns, address in fwd_sync().tmem_base, visible
// after the tile's first block barrier).  Returns after a block barrier with
// every MMA of the tile complete, so that the caller may start another tile.
template <int N>
__device__ __forceinline__ void fwd_tile(const FwdArgs& a, long long t) {
  using S = FwdHShape<N>;
  constexpr int P = S::P, KP = S::KP, NC = S::NC, CS = S::CS, R = S::R, R4 = R / 4;
  static_assert(CS <= 4 && N <= 12, "FwdHSync sizes");
  FwdHSync& sy = fwd_sync();
  uint8_t* Alo = fwd_smem();  // Phi lo, where tensor memory does not hold it
  uint8_t* Cst = Alo + S::PHI_BYTES;  // CS stages of (Bhi, Blo, weights)
  uint8_t* Rec = Cst + CS * S::C_STAGE;  // 32 records per builder warp
  uint64_t* coef_full = sy.coef_full;
  uint64_t* coef_empty = sy.coef_empty;
  uint64_t* acc_full = sy.acc_full;
  uint64_t* acc_empty = sy.acc_empty;
  uint64_t& drain = sy.drain;
  float* sred = sy.sred;
  float* sctr = sy.sctr;
  float* sh = sy.sh;
  auto& sflag = sy.sflag;
  int& s_abort = sy.s_abort;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const long long qt = t * a.tile;
  const int nq = (int)(a.Q - qt < a.tile ? a.Q - qt : a.tile);
  const int nh = nq > 128 ? 2 : 1;  // row blocks with queries

  // ---- setup: barriers, tile centre and scales, Phi rows (epilogue warps)
  if (tid == 0) {
    for (int i = 0; i < 4; ++i) {
      mbar_init(&coef_full[i], S::GPC);
      mbar_init(&coef_empty[i], 1 + 4 * nh);  // issuer commit + the busy epilogue warps
    }
    for (int i = 0; i < 4; ++i) {
      mbar_init(&acc_full[i], 2);  // issuer commit and arrival
      mbar_init(&acc_empty[i], 4);
    }
    mbar_init(&drain, 1);
    s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  const int row = tid - 32 * kFwdEpi0;  // epilogue threads: Phi row
  const bool is_epi = warp >= kFwdEpi0 && warp < kFwdIssuer;
  const bool active_row = is_epi && row < nq;
  float xq[N];
#pragma unroll
  for (int d = 0; d < N; ++d) xq[d] = active_row ? a.x[(qt + row) * N + d] : 0.0f;
  if (is_epi) {
#pragma unroll
    for (int d = 0; d < N; ++d) {
      float lo = active_row ? xq[d] : INFINITY, hi = active_row ? xq[d] : -INFINITY;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
      }
      if (lane == 0) {
        sred[((warp - kFwdEpi0) * N + d) * 2] = lo;
        sred[((warp - kFwdEpi0) * N + d) * 2 + 1] = hi;
      }
    }
  }
  __syncthreads();
  if (tid < N) {
    float lo = INFINITY, hi = -INFINITY;
    for (int w = 0; w < 8; ++w) {
      lo = fminf(lo, sred[(w * N + tid) * 2]);
      hi = fmaxf(hi, sred[(w * N + tid) * 2 + 1]);
    }
    const float c = (lo <= hi) ? 0.5f * (lo + hi) : 0.0f;
    sctr[tid] = c;
    sh[tid] = (lo <= hi) ? pow2_ceil(fmaxf(hi - c, c - lo)) : 1.0f;
  }
  __syncthreads();
  if (is_epi) {
    float u[N];
#pragma unroll
    for (int d = 0; d < N; ++d) u[d] = active_row ? (xq[d] - sctr[d]) * (1.0f / sh[d]) : 0.0f;
    float phi[KP];
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
      for (int j = 0; j <= i; ++j) phi[tri(i) + j] = u[i] * u[j];
#pragma unroll
    for (int i = 0; i < N; ++i) phi[P + i] = u[i];
    phi[P + N] = active_row ? 1.0f : 0.0f;
#pragma unroll
    for (int k = P + N + 1; k < KP; ++k) phi[k] = 0.0f;
    // row `row` = lane 32 (warp % 4) + lane of its row block
    const uint32_t ph = sy.tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + S::TM_PHI +
                        (uint32_t)(((warp - kFwdEpi0) >> 2) * (KP / 2));
    fence_after_sync();
#pragma unroll
    for (int k = 0; k < KP; k += 8) {
      uint4 h, l;
      split_h2(phi[k], phi[k + 1], h.x, l.x);
      split_h2(phi[k + 2], phi[k + 3], h.y, l.y);
      split_h2(phi[k + 4], phi[k + 5], h.z, l.z);
      split_h2(phi[k + 6], phi[k + 7], h.w, l.w);
      tmem_st4(ph + (uint32_t)(k / 2), h);
      if (row < 128 * S::LO_TM) tmem_st4(ph + (uint32_t)(KP + k / 2), l);
      else *reinterpret_cast<uint4*>(Alo + kmajor_off_h(row - 128 * S::LO_TM, k, S::SBO)) = l;
    }
    tmem_wait_st();
  }
  fence_proxy_async();
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tmem = sy.tmem_base;
  const long long beg = a.offsets[t], end = a.offsets[t + 1];
  const int nchunks = (int)((end - beg + NC - 1) / NC);
  volatile int* abort_flag = &s_abort;
  auto fail = [&]() {
    atomicExch(&s_abort, 1);
    if (a.status) set_status(a.status, NDG_ERR_TIMEOUT);
  };

  if (warp < S::BW) {
    // ---- builders
    // warp w builds the 32-candidate groups w, w + BW, ...; group g is rows
    // 32 (g % GPC) .. + 31 of chunk g / GPC
    const int ngroups = nchunks * S::GPC;
    auto cand = [&](int gr) -> int {
      const long long c = beg + (long long)gr * 32 + lane;
      const int g = c < end ? a.ids[c] : -1;
      return ((unsigned)g < (unsigned)a.Ge) ? g : -1;
    };
    const int stride4 = a.rec_stride4 > 0 ? a.rec_stride4 : R4;
    // The records of a group come by asynchronous copies into the warp's 32
    // rows, issued as soon as the group before has been read into registers,
    // and arrive while that group is built.  Consecutive lanes copy
    // consecutive 16-byte parts of a record: one lane per record would take
    // 32 cache lines an instruction.
    float4* rows = reinterpret_cast<float4*>(Rec) + (size_t)warp * 32 * S::REC_STRIDE;
    auto fetch = [&](int g) {
#pragma unroll
      for (int k = 0; k < R4; ++k) {
        const int r = (k * 32 + lane) / R4, part = k * 32 + lane - r * R4;
        const int gr = __shfl_sync(0xffffffffu, g, r);
        if (gr >= 0)
          cp_async16(rows + r * S::REC_STRIDE + part,
                     reinterpret_cast<const float4*>(a.rec) + (size_t)gr * stride4 + part);
      }
    };
    int g_cur = cand(warp), g_next = cand(warp + S::BW);
    fetch(warp < ngroups ? g_cur : -1);
    for (int gr = warp; gr < ngroups; gr += S::BW) {
      const int i = gr / S::GPC, s = i % CS;
      const int j = (gr - i * S::GPC) * 32 + lane;
      bool ok = true;
      cp_async_wait_all();
      __syncwarp();
      // N >= 9: the record stays in its row and is read twice (in registers it
      // spilled, N = 12 evaluation 551 us against 233); smaller ones are read
      // into registers and the next group's copies start at once.
      constexpr bool STREAM = N >= 9;
      float4* mine = rows + lane * S::REC_STRIDE;
      if (g_cur < 0) {
#pragma unroll
        for (int k = 0; k < R4; ++k) mine[k] = make_float4(0.f, 0.f, 0.f, 0.f);
      }
      float buf[STREAM ? 4 : R];
      if constexpr (!STREAM) {
#pragma unroll
        for (int k = 0; k < R4; ++k) {
          const float4 r = mine[k];
          buf[4 * k] = r.x; buf[4 * k + 1] = r.y; buf[4 * k + 2] = r.z; buf[4 * k + 3] = r.w;
        }
        __syncwarp();  // every lane has its row: the next group's may land
        fetch(g_next);
        g_cur = g_next;
        g_next = cand(gr + 2 * S::BW);
      }
      if (ok && i >= CS) ok = warp_wait(&coef_empty[s], ((i / CS) - 1) & 1, abort_flag);
      if (!ok && lane == 0) fail();
      uint8_t* st = Cst + s * S::C_STAGE;
      bool scaled = false;
      if (ok) {
        float mt[N], tA[N], cst = 0.0f, mx = 0.0f;
        float cf[STREAM ? 8 : KP];
        float wc[3];
        // coefficient of the quadratic term (d, e), e <= d, from A_de
        auto quad_coef = [&](float av, int d, int e2) {
          const float kd = kNegHalfLog2eH * sh[d];
          return av * (d == e2 ? kd : 2.0f * kd) * sh[e2];
        };
        if constexpr (STREAM) {
#pragma unroll
          for (int k = P / 4; k < R4; ++k) {
            const float4 q = mine[k];
            const float qa[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              const int p = 4 * k + c - P;
              if (p >= 0 && p < N) mt[p] = qa[c] - sctr[p];
              if (p >= N && p < N + 3) wc[p - N] = qa[c];
            }
          }
#pragma unroll
          for (int d = 0; d < N; ++d) tA[d] = 0.0f;
          // A m~, every sum in the order of the products' second index, as below
#pragma unroll
          for (int k = 0; 4 * k < P; ++k) {
            const float4 q = mine[k];
            const float qa[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
            for (int c = 0; c < 4; ++c)
#pragma unroll
              for (int d = 0; d < N; ++d) {
                const int e2 = 4 * k + c - tri(d);
                if (e2 >= 0 && e2 <= d) {
                  tA[d] = fmaf(qa[c], mt[e2], tA[d]);
                  if (e2 < d) tA[e2] = fmaf(qa[c], mt[d], tA[e2]);
                  mx = fmaxf(mx, fabsf(quad_coef(qa[c], d, e2)));
                }
              }
          }
#pragma unroll
          for (int d = 0; d < N; ++d) cst = fmaf(mt[d], tA[d], cst);
#pragma unroll
          for (int d = 0; d < N; ++d) {
            tA[d] = (-2.0f * (kNegHalfLog2eH * sh[d])) * tA[d];
            mx = fmaxf(mx, fabsf(tA[d]));
          }
          cst *= kNegHalfLog2eH;
          mx = fmaxf(mx, fabsf(cst));
        } else {
#pragma unroll
          for (int d = 0; d < N; ++d) mt[d] = buf[P + d] - sctr[d];
#pragma unroll
          for (int d = 0; d < N; ++d) {
            float s2 = 0.0f;
#pragma unroll
            for (int k = 0; k < N; ++k) s2 = fmaf(buf[d >= k ? tri(d) + k : tri(k) + d], mt[k], s2);
            tA[d] = s2;
            cst = fmaf(mt[d], s2, cst);
          }
          // the coefficients, in the record's place (the scales are powers of
          // two, so their order does not change a bit): quadratic (d, e),
          // linear d, constant, zero padding
#pragma unroll
          for (int d = 0; d < N; ++d) {
#pragma unroll
            for (int e2 = 0; e2 <= d; ++e2) cf[tri(d) + e2] = quad_coef(buf[tri(d) + e2], d, e2);
            cf[P + d] = (-2.0f * (kNegHalfLog2eH * sh[d])) * tA[d];
          }
          cf[P + N] = kNegHalfLog2eH * cst;
#pragma unroll
          for (int k = P + N + 1; k < KP; ++k) cf[k] = 0.0f;
#pragma unroll
          for (int k = 0; k <= P + N; ++k) mx = fmaxf(mx, fabsf(cf[k]));
        }
        float back = 1.0f, down = 1.0f;
        if (mx > kRowMax) {  // divide the row by 2^e, e = exponent(mx) - 13
          int e = (int)((__float_as_uint(mx) >> 23) & 0xffu) - 127 - 13;
          e = e > 120 ? 120 : e;
          down = __uint_as_float((uint32_t)(127 - e) << 23);
          back = __uint_as_float((uint32_t)(127 + e) << 23);
          scaled = true;
          if constexpr (!STREAM) {
#pragma unroll
            for (int k = 0; k <= P + N; ++k) cf[k] *= down;
          }
        }
        if constexpr (STREAM) asm volatile("" ::: "memory");  // read the row again
#pragma unroll
        for (int kb = 0; kb < KP; kb += 8) {
          if constexpr (STREAM) {
#pragma unroll
            for (int q = 0; q < 8; ++q) cf[q] = 0.0f;
#pragma unroll
            for (int k = 0; k < 2; ++k) {
              if (kb + 4 * k >= P) continue;
              const float4 q = mine[kb / 4 + k];
              const float qa[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
              for (int c = 0; c < 4; ++c)
#pragma unroll
                for (int d = 0; d < N; ++d) {
                  const int e2 = kb + 4 * k + c - tri(d);
                  if (e2 >= 0 && e2 <= d) cf[4 * k + c] = quad_coef(qa[c], d, e2) * down;
                }
            }
#pragma unroll
            for (int d = 0; d < N; ++d)
              if (P + d >= kb && P + d < kb + 8) cf[P + d - kb] = tA[d] * down;
            if (P + N >= kb && P + N < kb + 8) cf[P + N - kb] = cst * down;
          }
          const float* c = STREAM ? cf : cf + kb;
          uint4 h, l;
          split_h2(c[0], c[1], h.x, l.x);
          split_h2(c[2], c[3], h.y, l.y);
          split_h2(c[4], c[5], h.z, l.z);
          split_h2(c[6], c[7], h.w, l.w);
          const uint32_t off = kmajor_off_h(j, kb, S::SBO);
          *reinterpret_cast<uint4*>(st + off) = h;
          *reinterpret_cast<uint4*>(st + S::B_BYTES + off) = l;
        }
        float* wd = reinterpret_cast<float*>(st + 2 * S::B_BYTES) + (j >> 1) * 8 + (j & 1);
#pragma unroll
        for (int c = 0; c < 3; ++c) wd[2 * c] = STREAM ? wc[c] : buf[STREAM ? 0 : P + N + c];
        wd[6] = back;
      }
      const bool any_scaled = __any_sync(0xffffffffu, scaled);
      if (lane == 0) sflag[s][gr - i * S::GPC] = any_scaled ? 1 : 0;
      fence_proxy_async();
      warp_arrive(&coef_full[s]);
      // a CTA that gives up stops every role at its next blocked wait
      if (!ok) break;
      if constexpr (STREAM) {
        __syncwarp();
        fetch(g_next);
        g_cur = g_next;
        g_next = cand(gr + 2 * S::BW);
      }
    }
    cp_async_wait_all();
  } else if (warp == kFwdIssuer) {
    // ---- MMA issuer
    if (elect_one()) {
      // descriptor bases (a descriptor for base + off is base + off / 16)
      const uint64_t dA0 = smem_desc(smem_u32(Alo), 128, S::SBO);
      const uint64_t dB0 = smem_desc(smem_u32(Cst), 128, S::SBO);
      constexpr uint64_t B_LO = S::B_BYTES >> 4;
      constexpr uint32_t IDESC = idesc_f16(NC);
      for (int i = 0; i < nchunks; ++i) {
        const int s = i % CS, b = i & 1;
        bool ok = lane_wait(&coef_full[s], (i / CS) & 1, abort_flag);
        const uint64_t dbh = dB0 + (uint64_t)((s * S::C_STAGE) >> 4);
        for (int h = 0; ok && h < nh; ++h) {
          // row block h of buffer b is free once its epilogue group has read chunk i - 2
          if (i >= 2) ok = lane_wait(&acc_empty[2 * b + h], ((i >> 1) - 1) & 1, abort_flag);
          if (!ok) break;
          fence_after_sync();
          const uint32_t d = tmem + (uint32_t)((2 * b + h) * NC);
          const uint32_t ah = tmem + S::TM_PHI + (uint32_t)(h * (KP / 2));
          const uint64_t dal = dA0 + (uint64_t)(((h - S::LO_TM) * (int)S::HALF_BYTES) >> 4);
#pragma unroll
          for (int ks = 0; ks < KP / 16; ++ks) {
            const uint64_t ko = (uint64_t)ks * 16u;  // two 16-byte core matrices per K step
            mma_f16_ts(d, ah + 8u * ks, dbh + ko, IDESC, ks > 0 ? 1u : 0u);
            mma_f16_ts(d, ah + 8u * ks, dbh + B_LO + ko, IDESC, 1u);
            if (h < S::LO_TM) mma_f16_ts(d, ah + KP + 8u * ks, dbh + ko, IDESC, 1u);
            else mma_f16(d, dal + ko, dbh + ko, IDESC, 1u);
          }
          mma_commit(&acc_full[2 * b + h]);
          mbar_arrive(&acc_full[2 * b + h]);  // after coef_full: hands the weights on to the epilogue
        }
        if (!ok) {
          fail();
          break;
        }
        mma_commit(&coef_empty[s]);
      }
    }
  } else if (is_epi) {
    // ---- epilogue (tcgen05.ld 16x256b: thread t holds lanes t/4 and t/4 + 8
    // of a 16-lane half at columns 2 (t % 4) + {0, 1} of every 8-column group).
    constexpr int NU = NC / 16;  // units of 16 columns
    const int quad = warp & 3, h = (warp - kFwdEpi0) >> 2;
    const int tq = lane & 3, tr = lane >> 2;
    // rows ri = hb * 2 + r8: 16-lane half hb, lane t/4 + 8 r8; .x / .y
    // accumulate the even / odd column of the thread's pairs
    float2 acc[4][3];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int c = 0; c < 3; ++c) acc[r][c] = make_float2(0.f, 0.f);
    const uint32_t lane_base = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(h * NC);
    // One chunk.  The exponentials of a unit are issued together with the
    // colour sums of the one before, so that MUFU and FMA work overlap inside
    // a warp; the next unit loads meanwhile.
    auto chunk = [&](int b, const float* wp, auto sc_tag) {
      constexpr bool SC = decltype(sc_tag)::value;
      uint32_t v[2][2][8];
      float4 w01[2][2];
      float2 w2[2][2], sc[2];
      auto load = [&](int u) {
#pragma unroll
        for (int hb = 0; hb < 2; ++hb)
          tmem_ld16x256_x2_nowait(
              lane_base + ((uint32_t)(hb * 16) << 16) + (uint32_t)(2 * b * NC + u * 16), v[u & 1][hb]);
      };
      auto exps = [&](int u, int k, int hb) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          float sv = __uint_as_float(v[u & 1][hb][4 * k + j]);
          if (SC) sv *= (j & 1) ? sc[k].y : sc[k].x;
          v[u & 1][hb][4 * k + j] = __float_as_uint(ex2_approx(sv));
        }
      };
      auto sums = [&](int u, int k, int hb) {
#pragma unroll
        for (int r8 = 0; r8 < 2; ++r8) {
          const float2 e = make_float2(__uint_as_float(v[u & 1][hb][4 * k + 2 * r8]),
                                       __uint_as_float(v[u & 1][hb][4 * k + 2 * r8 + 1]));
          const int ri = 2 * hb + r8;
          acc[ri][0] = __ffma2_rn(make_float2(w01[u & 1][k].x, w01[u & 1][k].y), e, acc[ri][0]);
          acc[ri][1] = __ffma2_rn(make_float2(w01[u & 1][k].z, w01[u & 1][k].w), e, acc[ri][1]);
          acc[ri][2] = __ffma2_rn(w2[u & 1][k], e, acc[ri][2]);
        }
      };
      load(0);
#pragma unroll
      for (int u = 0; u < NU; ++u) {
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const float* wk = wp + (8 * u + 4 * k) * 8;
          w01[u & 1][k] = *reinterpret_cast<const float4*>(wk);
          w2[u & 1][k] = *reinterpret_cast<const float2*>(wk + 4);
          if (SC) sc[k] = *reinterpret_cast<const float2*>(wk + 6);
        }
        tmem_wait_ld();
        tmem_reg_fence8(v[u & 1][0]);
        tmem_reg_fence8(v[u & 1][1]);
        if (u == NU - 1) {
          // this warp's reads of buffer b are complete
          fence_before_sync();
          warp_arrive(&acc_empty[2 * b + h]);
        }
#pragma unroll
        for (int k = 0; k < 2; ++k)
#pragma unroll
          for (int hb = 0; hb < 2; ++hb) {
            exps(u, k, hb);
            if (u > 0) sums(u - 1, k, hb);
          }
        if (u + 1 < NU) load(u + 1);
      }
#pragma unroll
      for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int hb = 0; hb < 2; ++hb) sums(NU - 1, k, hb);
    };
    for (int i = 0; h < nh && i < nchunks; ++i) {
      const int s = i % CS, b = i & 1;
      if (!warp_wait(&acc_full[2 * b + h], (i >> 1) & 1, abort_flag)) {
        if (lane == 0) fail();
        break;
      }
      fence_after_sync();
      const int4 fl = *reinterpret_cast<const int4*>(&sflag[s][0]);
      const bool scaled = (fl.x | fl.y | fl.z) != 0;
      // weight pair entries of this thread: p = 8 u + 4 k + tq
      const float* wp = reinterpret_cast<const float*>(Cst + s * S::C_STAGE + 2 * S::B_BYTES) + tq * 8;
      if (scaled) chunk(b, wp, BoolTag<true>{});
      else chunk(b, wp, BoolTag<false>{});
      warp_arrive(&coef_empty[s]);
    }
    // ---- row sums over the pair halves and the four threads sharing a lane
    // (shuffles); thread tq writes row ri = tq
    if (h < nh && !*abort_flag) {
#pragma unroll
      for (int ri = 0; ri < 4; ++ri) {
        float rs[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          float v = acc[ri][c].x + acc[ri][c].y;
          v += __shfl_xor_sync(0xffffffffu, v, 1);
          v += __shfl_xor_sync(0xffffffffu, v, 2);
          rs[c] = v;
        }
        const int qr = h * 128 + quad * 32 + (ri >> 1) * 16 + (ri & 1) * 8 + tr;
        if (ri == tq && qr < nq) {
#pragma unroll
          for (int c = 0; c < 3; ++c) a.y[(qt + qr) * 3 + c] = rs[c];
        }
      }
    }
  }
  // A barrier counts a warp each time a part of it arrives: the issuer's lane
  // and the other 31 come back together.
  __syncwarp();
  fence_before_sync();
  __syncthreads();
  if (warp == kFwdIssuer && elect_one()) {
    // every MMA this thread issued has completed once this commit arrives
    mma_commit(&drain);
    if (!mbar_wait_bounded(&drain, 0, kWaitLimit)) fail();
  }
  __syncwarp();
  fence_before_sync();
  __syncthreads();
  // a barrier must be invalidated before the next tile initialises it again
  // (without, the second tile of a CTA saw phases of the first)
  if (tid == 0)
    for (int i = 0; i < FwdHSync::kBarriers; ++i) mbar_inval(&sy.coef_full[0] + i);
  __syncthreads();
}

}  // namespace ndg
