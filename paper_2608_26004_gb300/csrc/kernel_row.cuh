// Streaming row kernel of the production programs (no per-row outputs,
// delta = a - b; greedy and stochastic mode, every gate) and the decision
// kernel that follows it.
//
// One cluster of C CTAs per row triple (a_k, b_k, t_k); CTA r takes vectors
// [r Wv, (r+1) Wv) of the three rows.  Pass 1 reads each logit once from HBM
// and leaves the row's normalisers (Eqs. 1-3) and, in greedy mode, its
// argmax; every warp pushes its record into every CTA of the cluster
// (distributed shared memory, st.async completing on the receiver's
// mbarrier).  With the normalisers a row knows whether it needs a second
// pass at all:
//   * the divergence D of Eq. 3 enters only gamma_eff = gamma exp(-D), and D
//     is bounded: 0 <= JSD <= ln 2, 0 <= KL (and D is known from the draft
//     token's own logits under the tuned-lambda gate, 0 without a gate).  A
//     row that passes its acceptance test at D = 0 passes at every D; one
//     that fails at the upper bound fails at every D; only between the two
//     does the row's decision depend on D.  (row_path)
//   * the residual max(0, q - p) is drawn from only where a row is rejected,
//     so a row that passes at D = 0 needs no masses, and the fused masses of
//     a bonus row are the warps' pass-1 sums.
// So pass 2 (the divergence and residual masses, re-read from the L2, where
// pass 1 just brought the row) runs for the rows whose decision depends on D
// and for rejected rows; the rest of the rows end after pass 1.  The results
// are those of running it for every row.
//
// What bounds it: HBM at B=64 (0.83 of the copy rate; 22 instructions per
// vocabulary entry on the benchmark's rows, about half of the issue slots);
// launch, ramp, exchange and decision where a batch is a wave or less.  Layout:
//   * no slice is held in shared memory.  Each warp owns a contiguous block
//     of the slice and reads it through a small ring in shared memory (kRing
//     steps of 32 consecutive 16-byte vectors per stream, filled with
//     cp.async).  The rows in flight at once (one per resident cluster; the
//     host picks C so that they stay within its L2 budget) sit inside the
//     129 MB L2, so a second pass finds them there.  With 48 KB of rings and
//     the cluster's records in shared memory, four 256-thread CTAs fit on an
//     SM (the register file is the limit);
//   * no CTA or cluster barrier between the passes but the one __syncthreads
//     after warp 0 has combined the records: a warp pushes its record as soon
//     as its block is done, and the exchange completes on each receiver's
//     mbarrier when the last record of the cluster lands;
//   * the block of a warp is one inverse-CDF group, whose mass the warp
//     reduces anyway (the decision kernel walks the group's vectors);
//   * one 16-byte vector per stream per step, unpacked pair by pair from the
//     raw words (bf16 -> fp32 is a shift or a mask), two fp32 lanes per
//     add/sub/mul/fma instruction;
//   * the JSD of Eq. 3 in one product per pair.  With p = softmax(a), q =
//     softmax(b) in log2 units, e = q/p = 2^d (d = log2 q - log2 p) and w = 1
//     + e, each entry contributes to 2 JSD (in bits)
//         p log2(2p/(p+q)) + q log2(2q/(p+q)) = p [w (1 - log2 w) + e d],
//     a sum of small non-negative terms with no cancellation at the end (a
//     block where e overflows is summed again term by term, row_jsd_wide);
//   * the residual max(0, q_f - p) and fused score (t + beta (a - b)) log2 e
//     are formed exactly as the decision kernel's draw forms them (res_pair), so
//     a group has residual mass only if an entry of it has.  The fused group
//     masses (bonus rows; a draft row without residual) are the warps' pass-1
//     sums and differ from the draw's by roundings (block_mass).
//
// EDGE: rows that do not start on a 16-byte boundary (V * element size not a
// multiple of 16, or an offset base), with a, b and t at the same offset.
// The row is cut at the 16-byte boundaries of memory: vector 0 starts `head`
// elements before the row and the last vector may end after it.  The whole
// vectors go through the rings as above; the at most VE - 1 elements of each
// partial vector are loaded one per lane by the warp that owns it, so no
// access leaves the row and the loops are the same.
//
// Waits: one cluster barrier at the start (every CTA's mbarrier is
// initialised before the first push), CTA barriers, its own cp.async groups,
// and the record exchange's mbarrier, bounded by %globaltimer: a wait that
// gives up, in any CTA of the cluster, reports ASYMSPEC_DATA_TIMEOUT for the
// row (late_end), and is waited for once more (bounded) before the CTA exits,
// so that a late push finds it alive.
#pragma once

#include "kernel_tma.cuh"

namespace asymspec_impl {

// A 16-byte vector of the slice, as raw words; pair(h) widens entries
// 2h, 2h + 1 to fp32.
template <typename T>
struct RawVec;
template <>
struct RawVec<__nv_bfloat16> {
  static constexpr int NP = 4;
  uint4 v;
  __device__ __forceinline__ f2 pair(int h) const {
    const unsigned w = h == 0 ? v.x : h == 1 ? v.y : h == 2 ? v.z : v.w;
    return pk(__uint_as_float(w << 16), __uint_as_float(w & 0xFFFF0000u));
  }
};
template <>
struct RawVec<float> {
  static constexpr int NP = 2;
  float4 v;
  __device__ __forceinline__ f2 pair(int h) const { return h == 0 ? pk(v.x, v.y) : pk(v.z, v.w); }
};
// A vector from global memory (read-only for the kernel's lifetime).
template <typename T>
__device__ __forceinline__ RawVec<T> raw_ldg(const T* p) {
  RawVec<T> r;
  r.v = __ldg(reinterpret_cast<const decltype(r.v)*>(p));
  return r;
}
__device__ __forceinline__ float elem_ldg(const float* p) { return __ldg(p); }
__device__ __forceinline__ float elem_ldg(const __nv_bfloat16* p) {
  return __uint_as_float(static_cast<unsigned>(__ldg(reinterpret_cast<const unsigned short*>(p)))
                         << 16);
}

// Constants of a row's pass 2 (log2 units): L2 = log2 e, bL2 = beta log2 e,
// nA2 = -LSE(a) log2 e, nS2 = -LSE(s) log2 e, cAB2 = (LSE(a) - LSE(b)) log2 e.
struct ResConst {
  f2 L2, nL2, bL2, nA2, nS2, cAB2, one2;
};

__device__ __forceinline__ ResConst res_const(float beta, float A2, float B2, float S2) {
  ResConst k;
  k.L2 = pk(kLog2e, kLog2e);
  k.nL2 = pk(-kLog2e, -kLog2e);
  const float bl = beta * kLog2e;
  k.bL2 = pk(bl, bl);
  k.nA2 = pk(-A2, -A2);
  k.nS2 = pk(-S2, -S2);
  const float c = A2 - B2;
  k.cAB2 = pk(c, c);
  k.one2 = pk(1.f, 1.f);
  return k;
}

// The masses of one pair of entries: p = softmax(a), the fused q_f =
// softmax(t + beta (a - b)) and the residual r = max(0, q_f - p); amb = a - b.
// The row kernel's pass 2 and the decision kernel's walk both use this.
__device__ __forceinline__ void res_pair(f2 a2, f2 b2, f2 t2, const ResConst& k, f2& amb, f2& p,
                                         f2& qf, f2& r) {
  amb = sub2(a2, b2);
  p = ex2_2(fma2(a2, k.L2, k.nA2));
  qf = ex2_2(fma2(t2, k.L2, fma2(k.bL2, amb, k.nS2)));
  r = relu2(sub2(qf, p));
}

// The JSD term of a pair (see the header): p [w (1 - log2 w) + e d] with
// d = log2 q - log2 p = -(a - b) log2 e + (LSE(a) - LSE(b)) log2 e.
__device__ __forceinline__ f2 jsd_pair(f2 amb, f2 p, const ResConst& k, f2 jacc) {
  const f2 d = fma2(amb, k.nL2, k.cAB2);
  const f2 e = ex2_2(d);
  const f2 w = add2(e, k.one2);
  const f2 x = sub2(k.one2, lg2_2(w));
  return fma2(p, fma2(w, x, mul2(e, d)), jacc);
}

// The KL term of a pair, subtracted: p d (the caller negates the sum).
__device__ __forceinline__ f2 kl_pair(f2 amb, f2 p, const ResConst& k, f2 jacc) {
  return fma2(p, fma2(amb, k.nL2, k.cAB2), jacc);
}

// ---------------------------------------------------------------- layout

constexpr int kRowThreads = 256;  // threads per CTA of the row kernel
constexpr int kRowMinBlocks = 4;  // CTAs per SM (64 registers a thread)
static_assert(kRowThreads / 32 <= kRowMaxWarps, "one record slot per warp");

// The block [b0, b1) of warp w in the slice of nv vectors that starts at the
// row's vector s0: equal parts.  LINES (the recording kernel's aligned rows):
// parts that start on the row's 128-byte lines, so that a step's 512 bytes lie in
// four lines and not five, but for blocks of almost the most vectors a draw
// takes, which are cut anywhere.  Recorded, greedy, V=128256 bf16: B=8, K=4 21.9 ->
// 20.1 us, B=64, K=7 145.9 -> 139.3; V=64000 fp32 B=64, K=7 108.6 -> 107.5 (the
// worst of 16: B=20, K=5 stochastic 39.6 -> 39.9).  (fuse_verify_row's blocks stay
// equal: lines took B=64, K=7 stochastic from 66.9 to 67.5.)
template <bool LINES>
__device__ __forceinline__ void row_block(int s0, int nv, int w, int& b0, int& b1) {
  constexpr int NW = kRowThreads / 32;
  const int part = row_block_vectors(nv, NW);
  if (LINES && part <= kWalkRounds * 32 - 8) {
    const int off = s0 & 7, bw = (row_block_vectors(nv + off, NW) + 7) & ~7;
    b0 = min(nv, max(0, w * bw - off));
    b1 = min(nv, max(0, (w + 1) * bw - off));
  } else {
    b0 = min(nv, w * part);
    b1 = min(nv, b0 + part);
  }
}

// A warp's pass-1 record: the references (whole numbers, in log2 units; EDGE:
// nats) and sums of 2^(x log2 e - ref) of a, b and the fused score (stochastic) or t
// (greedy); greedy: the largest fused score (t on an unfused bonus row) and
// the lowest vector of the row that holds it (INT_MAX: none; NaN: non-finite
// scores were seen).
struct __align__(16) W1 {
  float ref[3], s[3];
  float v;
  int vec;
};

// A stream's reference from one of its values: a whole number of log2 units,
// so that neither the exponents' reference nor a rescale between two
// references (a power of two) adds a rounding.
__device__ __forceinline__ float ref_of(float x) { return rintf(x * kLog2e); }

// 2^(x log2 e - ref_of(x)), the factor that takes a sum against x (nats) to
// one against its reference; 1 where fp32 does not resolve it (no finite sum
// has |x| that large but for logits of 10^6 and more).
__device__ __forceinline__ float ref_residual(float x, float ref) {
  return fabsf(ref) < 4194304.f ? ex2(fmaf(x, kLog2e, -ref)) : 1.f;
}

// ln(2^ref sum) with the exponents kept apart from the logarithm of the
// significand (ln 2 in two parts, the first of 12 bits, so that its product
// with the exponent is exact): ref + log2 sum is usually a small difference of
// larger numbers.
__device__ __forceinline__ float lse_of(float ref, float sum) {
  const bool normal = sum >= kMinNormal && sum <= 3.402823466e38f;  // else logf as it is
  const int bits = __float_as_int(sum);
  const float n = normal ? ref + static_cast<float>((bits >> 23) - 127) : ref;
  const float m = normal ? __int_as_float((bits & 0x007FFFFF) | 0x3F800000) : sum;
  constexpr double kLn2d = 0.69314718055994530942;
  constexpr double hi = 2839.0 / 4096.0;
  return fmaf(n, static_cast<float>(hi), fmaf(n, static_cast<float>(kLn2d - hi), logf(m)));
}

// EDGE rows and the cross-family step, which the generic kernel also took: a
// warp's sum s, against ref, restated against the warp's largest
// value M (nats), whose term is taken out as it went in and put back as exactly
// 1.  The first step's reference may lie far below an entry that holds most of
// a row, whose exponent then carries a rounding of up to 5e-7 and whose ex2 its
// own error.  RMS error of the LSEs against 64 bits, V = 16385 to 149173: 2.0e-7
// without, 7.1e-8 with it and 8.3e-8 in the generic kernel, which references each
// thread's maximum; B=32, K=4, V=100003 bf16 greedy 24.6 -> 25.4 us a step.
__device__ __forceinline__ void to_largest(float& s, float& ref, float M) {
  if (M > -INFINITY) {
    const float y = fmaf(M, kLog2e, -ref), rest = s - ex2(y);
    s = rest > 0.f ? fmaf(rest, ex2(-y), 1.f) : rest <= 0.f ? 1.f : NAN;
  }
  ref = M;
}

// Their records hold the references in nats, the others' in whole log2 units:
// the factor between two references, and the LSE.
template <bool NATS>
__device__ __forceinline__ float ref_factor(float d) {
  return ex2(NATS ? d * kLog2e : d);
}
template <bool NATS>
__device__ __forceinline__ float record_lse(float ref, float sum) {
  return NATS ? ref + logf(sum) : lse_of(ref, sum);
}

// The fused mass of a warp's block from its pass-1 sum: the group masses of a bonus
// row's draw, and of a draft row's where the whole residual is zero.  A block below
// 2^-100 has none: every entry of it, formed as the draw forms it (res_pair), may
// be flushed to zero (below 2^-126), and a draw at u = 0 would find no token.  (At
// most 2^12 entries a block and 2^7 blocks a row, so one that counts is kept, and
// has an entry that is not flushed.)
template <bool NATS>
__device__ __forceinline__ float block_mass(float ref, float sum, float S2) {
  const float m = sum > 0.f ? sum * ex2(NATS ? fmaf(ref, kLog2e, -S2) : ref - S2) : 0.f;
  return m >= 7.888609052210118e-31f ? m : 0.f;
}

// What pass 2 does for a row (row_path): nothing, the residual masses alone,
// or the divergence (and, in stochastic mode, the masses).
enum : int { kPathFull = 0, kPathAccept = 1, kPathReject = 2 };

// Shared state of the row kernel; the pass-1 records of every warp of the
// cluster follow it (recv(): C x kRowThreads / 32 records, the record of
// warp w of CTA r at r kRowThreads / 32 + w).
struct __align__(16) RowShared {
  float lse[4];             // the row's normalisers (a, b, t, s)
  unsigned long long xbar;  // completes when the cluster's records have landed
  int path;                 // kPath*
  int pad;
  __device__ W1* recv() { return reinterpret_cast<W1*>(this + 1); }
};
static_assert(sizeof(W1) == 32, "one warp record is two 16-byte words");
static_assert(sizeof(RowShared) % 16 == 0, "records after RowShared stay 16-byte aligned");

__host__ __device__ constexpr int row_shared_bytes(int C) {
  return static_cast<int>(sizeof(RowShared) + C * (kRowThreads / 32) * sizeof(W1));
}

// The cut of row `row` into 16-byte vectors: vector i holds elements
// [i VE - head, (i + 1) VE - head) of the row; base(x) is vector 0 of stream
// x.  Vectors [in0, in1) lie inside the row whole.
template <typename T, bool EDGE>
struct RowCut {
  static constexpr int VE = 16 / static_cast<int>(sizeof(T));
  long long off;  // element offset of vector 0 in the logit arrays (may precede the row)
  int head, nvec, in0, in1;
  __device__ __forceinline__ RowCut(const KParams& P, long long row) {
    off = row * P.V;
    head = 0;
    if constexpr (EDGE) {
      head = static_cast<int>((off + P.head0) & (VE - 1));
      off -= head;
    }
    nvec = (head + P.V + VE - 1) / VE;
    in0 = EDGE ? (head != 0) : 0;
    in1 = EDGE ? (head + P.V) / VE : nvec;
  }
  __device__ __forceinline__ const T* base(const void* p) const {
    return static_cast<const T*>(p) + off;
  }
};

// ---------------------------------------------------------------- the rings

// Each warp reads its block through a ring of kRing steps in shared memory:
// lane l copies its vector of the streams for a step into the step's slot
// with 16-byte cp.async (one commit group per step) and later reads back
// only what it copied itself, so no barrier is needed; kRing steps of every
// warp are in flight without holding registers.  AB, TT: the streams that a
// pass reads.
constexpr int kRing = 4;
constexpr int kRingBytes = (kRowThreads / 32) * kRing * 3 * 32 * 16;  // per CTA (48 KB)

__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

template <typename T>
struct Streams {
  const T *a, *b, *t;
};

// 16 bytes global -> shared, skipped (without a branch) unless `on`.
__device__ __forceinline__ void cp_async16_if(void* smem, const void* gmem, bool on) {
  asm volatile(
      "{ .reg .pred p; setp.ne.s32 p, %2, 0; @p cp.async.cg.shared.global [%0], [%1], 16; }" ::"r"(
          smem_u32(smem)),
      "l"(gmem), "r"(static_cast<int>(on))
      : "memory");
}

// The lane's vector at element offset o of the streams into ring slot `slot`.
template <typename T, bool AB, bool TT>
__device__ __forceinline__ void ring_issue(uint4* ring, int slot, const Streams<T>& g, size_t o,
                                           bool on) {
  uint4* d = ring + slot * 96 + (threadIdx.x & 31);
  if (AB) {
    cp_async16_if(d, g.a + o, on);
    cp_async16_if(d + 32, g.b + o, on);
  }
  if (TT) cp_async16_if(d + 64, g.t + o, on);
}
template <typename T, bool AB, bool TT>
__device__ __forceinline__ void ring_read(const uint4* ring, int slot, RawVec<T>& va,
                                          RawVec<T>& vb, RawVec<T>& vt) {
  using V = decltype(va.v);
  const V* d = reinterpret_cast<const V*>(ring + slot * 96 + (threadIdx.x & 31));
  if (AB) {
    va.v = d[0];
    vb.v = d[32];
  }
  if (TT) vt.v = d[64];
}
// The first kRing steps of a pass into the ring (one group each, empty past
// the block's end).  g: the lane's vector of step 0 (vector i0 of the slice)
// of each stream.
template <typename T, bool AB, bool TT>
__device__ __forceinline__ void ring_prologue(uint4* ring, const Streams<T>& g, int i0, int v1) {
  constexpr int VE = 16 / static_cast<int>(sizeof(T));
#pragma unroll
  for (int q = 0; q < kRing; ++q) {
    ring_issue<T, AB, TT>(ring, q, g, static_cast<size_t>(q) * 32 * VE, i0 + 32 * q < v1);
    cp_async_commit();
  }
}
// use(r, va, vb, vt, whole) for every step r of vectors [v0, v1) the lane has
// a vector in, after the prologue (whole: std::true_type where every lane of
// the warp has one).  kRing whole steps at a time with constant
// slots and no branch: step r + kRing goes into the slot step r was just used
// from (its values were consumed by instructions this thread has already
// issued, so the copy cannot overwrite unread data).  At most kRing steps
// remain after those, all of them already issued.
template <typename T, bool AB, bool TT, typename Use>
__device__ __forceinline__ void ring_steps(uint4* ring, const Streams<T>& g, int v0, int v1,
                                           Use&& use) {
  constexpr int VE = 16 / static_cast<int>(sizeof(T));
  const int i0 = v0 + static_cast<int>(threadIdx.x & 31);
  const int whole = (v1 - v0) / 32;
  RawVec<T> va, vb, vt;
  int r = 0;
  for (; r + kRing <= whole; r += kRing) {
#pragma unroll
    for (int u = 0; u < kRing; ++u) {
      cp_async_wait<kRing - 1>();
      ring_read<T, AB, TT>(ring, u, va, vb, vt);
      use(r + u, va, vb, vt, std::true_type{});
      ring_issue<T, AB, TT>(ring, u, g, static_cast<size_t>(r + u + kRing) * 32 * VE,
                            i0 + 32 * (r + u + kRing) < v1);
      cp_async_commit();
    }
  }
  cp_async_wait<0>();
#pragma unroll 1
  for (int u = 0; i0 + 32 * r < v1; ++r, ++u) {
    ring_read<T, AB, TT>(ring, u, va, vb, vt);
    use(r, va, vb, vt, std::false_type{});
  }
  __syncwarp();
}

// ---------------------------------------------------------------- pass 1

// The programs of pass 1: what a row's kind and the mode need.
enum : int {
  kStochDraft,    // LSE(a), LSE(b), LSE(s)
  kStochBonus,    // LSE(s)
  kGreedyDraft,   // LSE(a), LSE(b), LSE(t), argmax s
  kGreedyBonusT,  // argmax t (a and b are not read)
  kGreedyBonusS,  // argmax s (fused bonus)
};
__host__ __device__ constexpr bool prog_draft(int p) { return p == kStochDraft || p == kGreedyDraft; }
__host__ __device__ constexpr bool prog_ab(int p) { return p != kGreedyBonusT; }

// The elements of the row's partial vectors that a warp owns (EDGE): one per
// lane, the others kEdgeNone, which contributes nothing to any sum.  Lanes
// 0 .. VE - 1 take vector 0 (first), lanes 8 .. 8 + VE - 1 the last vector.
constexpr float kEdgeNone = -1e30f;
struct EdgeVals {
  bool own;           // the warp owns a partial vector
  bool head, tail;    // this lane holds an element of vector 0 / of the last vector
  int at;             // its index in the row (-1: none)
  float a, b, t;
};

// The edge elements of the warp whose block is vectors [b0, b1) of the slice
// that starts at vector s0; ab: a and b are wanted too.
template <typename T, bool EDGE>
__device__ __forceinline__ EdgeVals load_edges(const KParams& P, const RowCut<T, EDGE>& cut,
                                               unsigned row, int s0, int b0, int b1, bool ab) {
  constexpr int VE = 16 / static_cast<int>(sizeof(T));
  EdgeVals ed{false, false, false, -1, kEdgeNone, kEdgeNone, kEdgeNone};
  if constexpr (EDGE) {
    const int lane = static_cast<int>(threadIdx.x & 31);
    const bool h = cut.in0 > 0 && s0 == 0 && b0 == 0 && b1 > 0;
    const bool l = cut.in1 < cut.nvec && b1 > b0 && s0 + b1 == cut.nvec;
    ed.own = h || l;
    if (h && lane < VE && lane >= cut.head) {
      ed.head = true;
      ed.at = lane - cut.head;
    }
    const int el = cut.in1 * VE - cut.head + lane - 8;
    if (l && lane >= 8 && lane < 8 + VE && el < P.V) {
      ed.tail = true;
      ed.at = el;
    }
    if (ed.at >= 0) {
      const size_t o = static_cast<size_t>(row) * P.V + ed.at;
      ed.t = elem_ldg(static_cast<const T*>(P.t) + o);
      if (ab) {
        ed.a = elem_ldg(static_cast<const T*>(P.a) + o);
        ed.b = elem_ldg(static_cast<const T*>(P.b) + o);
      }
    }
  }
  return ed;
}

// The sum of a vector's pairs.
template <int NP>
__device__ __forceinline__ f2 vsum2(const f2 (&x)[NP]) {
  if constexpr (NP == 4) return add2(add2(x[0], x[1]), add2(x[2], x[3]));
  else return add2(x[0], x[1]);
}

// Larger of three with NaN winning (non-finite scores are flagged at the end).
__device__ __forceinline__ float max3_nan(float a, float b, float c) {
  float r;
  asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
template <int NP>
__device__ __forceinline__ float vmax_nan(const f2 (&x)[NP]) {
  if constexpr (NP == 4) {
    const float m = max3_nan(lo_of(x[0]), hi_of(x[0]), lo_of(x[1]));
    const float n = max3_nan(hi_of(x[1]), lo_of(x[2]), hi_of(x[2]));
    return max3_nan(max_nan(m, n), lo_of(x[3]), hi_of(x[3]));
  } else {
    return max_nan(max3_nan(lo_of(x[0]), hi_of(x[0]), lo_of(x[1])), hi_of(x[1]));
  }
}

// Pass 1 over vectors [v0, v1) of the slice (g: the lane's vector v0 + lane
// of each stream), read through the warp's ring (the caller issued
// the prologue), with one fixed reference per warp and stream: the largest
// of the first pairs of the lanes' first vectors.  vec0: the row's index of
// vector v0 + lane; lastvec: the row's last vector.  chk: a non-finite a or b
// makes the row a data error (it would make D non-finite); it is reported as
// a NaN sum of a.  Returns true when a lane's sum reached 2^100 or is not
// finite (the warp then redoes its block with running maxima).  Every lane
// ends with the warp's record.
template <typename T, int PROG, bool EDGE>
__device__ __forceinline__ bool row_pass1(uint4* ring, const Streams<T>& g, int v0, int v1,
                                          float beta, bool chk, const EdgeVals& ed, int vec0,
                                          int lastvec, W1& e) {
  constexpr int NP = RawVec<T>::NP;
  constexpr bool DRAFT = prog_draft(PROG), AB = prog_ab(PROG);
  constexpr bool STOCH = PROG == kStochDraft || PROG == kStochBonus;
  constexpr bool SUM3 = PROG == kStochDraft || PROG == kStochBonus || PROG == kGreedyDraft;
  constexpr bool ARG = !STOCH;
  const f2 L2 = pk(kLog2e, kLog2e);
  const float bl = beta * kLog2e;
  const f2 bL2 = pk(bl, bl), beta2 = pk(beta, beta);
  const int i0 = v0 + static_cast<int>(threadIdx.x & 31);
  float ra0 = -INFINITY, rb0 = -INFINITY, r30 = -INFINITY;
  cp_async_wait<kRing - 1>();  // step 0 (this lane's own copies)
  if (i0 < v1) {
    RawVec<T> va, vb, vt;
    ring_read<T, AB, true>(ring, 0, va, vb, vt);
    if (SUM3) {
      const f2 t2 = vt.pair(0);
      f2 x2 = t2;
      if (AB) {
        const f2 a2 = va.pair(0), b2 = vb.pair(0);
        ra0 = fmaxf(lo_of(a2), hi_of(a2));
        rb0 = fmaxf(lo_of(b2), hi_of(b2));
        if (STOCH) x2 = fma2(beta2, sub2(a2, b2), t2);
      }
      r30 = fmaxf(lo_of(x2), hi_of(x2));
    }
  }
  float se = 0.f;  // the edge element's fused score
  if (EDGE && ed.own) {
    se = AB ? fmaf(beta, ed.a - ed.b, ed.t) : ed.t;
    ra0 = fmaxf(ra0, ed.a);
    rb0 = fmaxf(rb0, ed.b);
    r30 = fmaxf(r30, STOCH ? se : ed.t);
  }
  if (DRAFT) {
    ra0 = warp_max(ra0);
    rb0 = warp_max(rb0);
  }
  if (SUM3) r30 = warp_max(r30);
  ra0 = ref_of(ra0);
  rb0 = ref_of(rb0);
  r30 = ref_of(r30);
  const float nA = -ra0, nB = -rb0, n3 = -r30;
  const f2 nA2 = pk(nA, nA), nB2 = pk(nB, nB), n32 = pk(n3, n3);
  f2 acc_a = 0ull, acc_b = 0ull, acc_3 = 0ull, fin = 0ull;
  float best = -INFINITY;
  float ma = -INFINITY, mb = -INFINITY, m3 = -INFINITY;  // EDGE: the largest values
  int rbest = -1;
  ring_steps<T, AB, true>(ring, g, v0, v1, [&](int r, const RawVec<T>& va, const RawVec<T>& vb,
                                               const RawVec<T>& vt, auto) {
    f2 sc[NP];  // the argmax's scores (EDGE, stochastic: the summed scores)
    f2 ea[NP], eb[NP], e3[NP], xa[NP], xb[NP], xt[NP];
#pragma unroll
    for (int h = 0; h < NP; ++h) {
      const f2 t2 = vt.pair(h);
      xt[h] = t2;
      if (AB) {
        const f2 a2 = va.pair(h), b2 = vb.pair(h);
        const f2 amb = sub2(a2, b2);
        xa[h] = a2;
        xb[h] = b2;
        if (DRAFT) {
          ea[h] = ex2_2(fma2(a2, L2, nA2));
          eb[h] = ex2_2(fma2(b2, L2, nB2));
          fin = fma2(amb, 0ull, fin);  // 0 x (non-finite) is NaN
        }
        if (STOCH && !EDGE) e3[h] = ex2_2(fma2(t2, L2, fma2(bL2, amb, n32)));
        if (ARG || EDGE) sc[h] = fma2(beta2, amb, t2);
        if (STOCH && EDGE) e3[h] = ex2_2(fma2(sc[h], L2, n32));
      } else {
        sc[h] = t2;
      }
      if (SUM3 && !STOCH) e3[h] = ex2_2(fma2(t2, L2, n32));
    }
    // a vector's terms are added among themselves first: one addition a step
    // in the running sums' chains of roundings
    if (DRAFT) {
      acc_a = add2(acc_a, vsum2(ea));
      acc_b = add2(acc_b, vsum2(eb));
    }
    if (SUM3) acc_3 = add2(acc_3, vsum2(e3));
    if (EDGE) {
      if (DRAFT) {
        ma = max_nan(ma, vmax_nan(xa));
        mb = max_nan(mb, vmax_nan(xb));
      }
      if (SUM3) m3 = max_nan(m3, STOCH ? vmax_nan(sc) : vmax_nan(xt));
    }
    if (ARG) {
      // strictly larger wins, so the lane's earliest vector keeps a tie
      const float c = vmax_nan(sc);
      rbest = c > best ? r : rbest;
      best = max_nan(best, c);
    }
  });
  if (EDGE && ed.own) {
    const float amb = ed.a - ed.b;
    if (DRAFT) {
      acc_a = add2(acc_a, pk(ex2(fmaf(ed.a, kLog2e, nA)), 0.f));
      acc_b = add2(acc_b, pk(ex2(fmaf(ed.b, kLog2e, nB)), 0.f));
      fin = fma2(pk(amb, 0.f), 0ull, fin);
    }
    const float x3 = STOCH ? se : ed.t;
    if (SUM3) acc_3 = add2(acc_3, pk(ex2(fmaf(x3, kLog2e, n3)), 0.f));
    ma = max_nan(ma, ed.a);
    mb = max_nan(mb, ed.b);
    m3 = max_nan(m3, x3);
  }
  bool ovf = false;
  e.ref[0] = ra0;
  e.ref[1] = rb0;
  e.ref[2] = r30;
  if (SUM3) {
    float sa = DRAFT ? hsum2(acc_a) : 0.f, sb = DRAFT ? hsum2(acc_b) : 0.f, s3 = hsum2(acc_3);
    ovf = !(s3 < kSumLimit) || (DRAFT && (!(sa < kSumLimit) || !(sb < kSumLimit)));
    if (DRAFT && chk) sa += hsum2(fin);  // 0, or NaN
    float z = 0.f;
    warp_sum4(sa, sb, s3, z);
    e.s[0] = sa;
    e.s[1] = sb;
    e.s[2] = s3;
    if (EDGE) {
      if (DRAFT) {
        to_largest(e.s[0], e.ref[0], warp_max(ma));
        to_largest(e.s[1], e.ref[1], warp_max(mb));
      }
      to_largest(e.s[2], e.ref[2], warp_max(m3));
    }
  } else {
    e.s[0] = e.s[1] = e.s[2] = 0.f;
  }
  e.v = 0.f;
  e.vec = 0;
  if (ARG) {
    int vec = rbest >= 0 ? vec0 + 32 * rbest : INT_MAX;
    if (EDGE && ed.own) {
      // vector 0 precedes every other, the last vector follows them
      if (ed.head && (se >= best || best != best) && se > -INFINITY) vec = 0;
      if (ed.tail && se > best) vec = lastvec;
      if (ed.head || ed.tail) best = max_nan(best, se);
    }
    const bool bad = !(best <= 3.402823466e38f);
    const float m = warp_max(best);
    const unsigned cand = best == m ? static_cast<unsigned>(vec) : static_cast<unsigned>(INT_MAX);
    e.vec = static_cast<int>(__reduce_min_sync(0xffffffffu, cand));
    e.v = __any_sync(0xffffffffu, bad) ? NAN : m;
  }
  return ovf;
}

// Fallback of row_pass1's sums (a sum reached 2^100, or non-finite data):
// each lane keeps a running maximum per stream over its vectors of the
// warp's block, rescaling its sum when the maximum rises; the lanes then
// merge.  The record's argmax stays as row_pass1 left it.  (Called out of
// line, so everything travels by value: a reference keeps the caller's record
// and pointers in local memory for every warp, 20 MB of stores a launch at
// B=64, K=7, V=128256 that reach HBM: stochastic 72.1 us a step against 66.4,
// greedy 64.2 against 59.8, B=256, K=4, V=151936 fp32 367 against 332.)
template <typename T, int PROG, bool EDGE>
__device__ __noinline__ W1 row_pass1_online(Streams<T> g, int v0, int v1, float beta, bool chk,
                                            EdgeVals ed, W1 e) {
  constexpr int NP = RawVec<T>::NP;
  constexpr int VE = 2 * NP;
  constexpr bool DRAFT = prog_draft(PROG);
  constexpr bool STOCH = PROG == kStochDraft || PROG == kStochBonus;
  float m[3] = {-INFINITY, -INFINITY, -INFINITY};  // running maxima of a, b, s or t (nats)
  float s[3] = {0.f, 0.f, 0.f};                    // sums of 2^((x - m) log2 e)
  float fin = 0.f;
  auto add = [&](int q, float v) {
    if (v > m[q]) {
      s[q] = s[q] * ex2((m[q] - v) * kLog2e);
      m[q] = v;
    }
    s[q] += ex2((v - m[q]) * kLog2e);
  };
  auto take = [&](float a, float b, float t) {
    if (DRAFT) {
      add(0, a);
      add(1, b);
      fin = fmaf(a - b, 0.f, fin);
    }
    add(2, STOCH ? fmaf(beta, a - b, t) : t);
  };
  const int lane = static_cast<int>(threadIdx.x & 31);
  for (int i = v0 + lane, q = 0; i < v1; i += 32, ++q) {
    const size_t o = static_cast<size_t>(q) * 32 * VE;
    const RawVec<T> va = raw_ldg(g.a + o), vb = raw_ldg(g.b + o), vt = raw_ldg(g.t + o);
#pragma unroll
    for (int h = 0; h < NP; ++h) {
      float a0, a1, b0, b1, t0, t1;
      upk(va.pair(h), a0, a1);
      upk(vb.pair(h), b0, b1);
      upk(vt.pair(h), t0, t1);
      take(a0, b0, t0);
      take(a1, b1, t1);
    }
  }
  if (EDGE && (ed.head || ed.tail)) take(ed.a, ed.b, ed.t);
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const float M = warp_max(m[q]);
    float sc = (s[q] == 0.f || m[q] == M) ? s[q] : s[q] * ex2((m[q] - M) * kLog2e);
    if (q == 0 && DRAFT && chk) sc += fin;  // 0, or NaN
    e.ref[q] = EDGE ? M : ref_of(M);
    e.s[q] = warp_sum(sc);
    if (!EDGE) e.s[q] *= ref_residual(M, e.ref[q]);
  }
  if (!DRAFT) {
    e.ref[0] = e.ref[1] = -INFINITY;
    e.s[0] = e.s[1] = 0.f;
  }
  return e;
}

// ---------------------------------------------------------------- pass 2

enum : int { kDivNone = 0, kDivJsd = 1, kDivKl = 2 };

// Pass 2 over the warp's block (from the L2, where pass 1 left it), through
// the warp's ring (the caller issued the prologue): the divergence terms
// (DIV) and the residual masses (RES).  Returns through jsum / msum the
// warp's sums (every lane ends with them): msum is the mass of the warp's
// inverse-CDF group.
template <typename T, int DIV, bool RES, bool EDGE>
__device__ __forceinline__ void row_pass2(uint4* ring, const Streams<T>& g, int v0, int v1,
                                          const ResConst& k, const EdgeVals& ed, float& jsum,
                                          float& msum) {
  constexpr int NP = RawVec<T>::NP;
  f2 jacc = 0ull, macc = 0ull;
  auto take = [&](f2 a2, f2 b2, f2 t2) {
    f2 amb, p;
    if (RES) {
      f2 qf, rr;
      res_pair(a2, b2, t2, k, amb, p, qf, rr);
      macc = add2(macc, rr);
    } else {
      amb = sub2(a2, b2);
      p = ex2_2(fma2(a2, k.L2, k.nA2));
    }
    if (DIV == kDivJsd) jacc = jsd_pair(amb, p, k, jacc);
    if (DIV == kDivKl) jacc = kl_pair(amb, p, k, jacc);
  };
  ring_steps<T, true, RES>(ring, g, v0, v1, [&](int, const RawVec<T>& va, const RawVec<T>& vb,
                                                const RawVec<T>& vt, auto) {
#pragma unroll
    for (int h = 0; h < NP; ++h) take(va.pair(h), vb.pair(h), RES ? vt.pair(h) : 0ull);
  });
  if (EDGE && ed.own) take(pk(ed.a, kEdgeNone), pk(ed.b, kEdgeNone), pk(ed.t, kEdgeNone));
  float j = hsum2(jacc), m = hsum2(macc), z0 = 0.f, z1 = 0.f;
  if (DIV == kDivKl) j = -j;
  warp_sum4(j, m, z0, z1);
  jsum = j;
  msum = m;
}

// The warp's JSD sum term by term, for a block where e = q/p overflowed
// (finite logits with b - a above about 88): p and q from their own
// exponents, an entry of no mass contributing nothing.  NaN where a or b is
// not finite.
template <typename T, bool EDGE>
__device__ __noinline__ float row_jsd_wide(Streams<T> g, int v0, int v1, float A2, float B2,
                                           EdgeVals ed) {
  constexpr int NP = RawVec<T>::NP;
  constexpr int VE = 2 * NP;
  float j = 0.f;
  auto take = [&](float a, float b) {
    const float la = fmaf(a, kLog2e, -A2), lb = fmaf(b, kLog2e, -B2);
    const float p = ex2(la), q = ex2(lb);
    const float lm = lg2(p + q) - 1.f;  // log2 of the mean
    if (p > 0.f) j += p * (la - lm);
    if (q > 0.f) j += q * (lb - lm);
    j = fmaf(a - b, 0.f, j);
  };
  const int lane = static_cast<int>(threadIdx.x & 31);
  for (int i = v0 + lane, q = 0; i < v1; i += 32, ++q) {
    const size_t o = static_cast<size_t>(q) * 32 * VE;
    const RawVec<T> va = raw_ldg(g.a + o), vb = raw_ldg(g.b + o);
#pragma unroll
    for (int h = 0; h < NP; ++h) {
      take(lo_of(va.pair(h)), lo_of(vb.pair(h)));
      take(hi_of(va.pair(h)), hi_of(vb.pair(h)));
    }
  }
  if (EDGE && (ed.head || ed.tail)) take(ed.a, ed.b);
  return warp_sum(j);
}

// ---------------------------------------------------------------- the kernel

// 16 bytes into CTA `rank`'s copy of the shared variable at `local`,
// completing 16 bytes of the transaction count of that CTA's copy of `bar`.
__device__ __forceinline__ void st_async16(const void* local, unsigned rank,
                                           unsigned long long* bar, float4 v) {
  unsigned ra, rb;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(smem_u32(local)), "r"(rank));
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(rb) : "r"(smem_u32(bar)), "r"(rank));
  asm volatile(
      "st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(ra),
      "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"(rb)
      : "memory");
}
__device__ __forceinline__ void cluster_wait() {
  asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
}
// Warp 0's wait for the records of the cluster; false: it gave up.
__device__ __forceinline__ bool wait_records(unsigned long long* bar, int rank) {
#ifdef ASYMSPEC_TEST_LATE_RANK  // a test build: the CTAs of one rank give up at once
  if (rank == ASYMSPEC_TEST_LATE_RANK) return false;
#endif
  return mbar_wait_cluster_bounded(bar, 0, kCopyTimeoutNs);
}
// The end of a CTA whose warp 0 gave up.  Its normalisers, and so its path and its
// masses, need not be the row's: it marks the row, whichever rank it has.  And no
// CTA exits while a push to it may be in flight (once the barrier has completed
// every push has landed): it waits once more, bounded, before it marks.
__device__ __forceinline__ void late_end(const KParams& P, unsigned row, unsigned long long* bar) {
  mbar_wait_cluster_bounded(bar, 0, kCopyTimeoutNs);
  if ((threadIdx.x & 31) == 0)
    atomicOr(&static_cast<RowStat*>(P.row_stat)[row].late, kBadTimeout);
}
// The start of a cluster: rank 0 clears the row's late word.  (Relaxed: a mark
// follows only after the waits of late_end.  A release here, or a mark that every
// CTA stores on every row, costs 64x7 bf16 V=128256 greedy 0.8 us of 59.5 and
// 1x4 0.3 of 5.1; this form nothing.)
__device__ __forceinline__ void cluster_start(const KParams& P, unsigned row, int rank) {
  if (rank == 0 && threadIdx.x == 0) static_cast<RowStat*>(P.row_stat)[row].late = 0u;
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
}
// Rank 0: the row's normalisers, argmaxes, error bits and path (not the late word).
__device__ __forceinline__ void store_stream_stat(const KParams& P, unsigned row,
                                                  const float (&lse)[4], int is, int it,
                                                  unsigned bad, int path) {
  float4* st = reinterpret_cast<float4*>(static_cast<RowStat*>(P.row_stat) + row);
  st[0] = make_float4(lse[0], lse[1], lse[2], lse[3]);
  st[1] = make_float4(__int_as_float(is), __int_as_float(it), __uint_as_float(bad),
                      __int_as_float(path));
}
// The row's pass-1 result from the n warp records of its cluster, by one
// warp: the largest reference of each stream, every record's sum restated
// against it, the sums added; the largest score and its lowest vector.
// Every lane ends with the same (bit-identical) result, and so does every
// CTA, whose records are the same.
template <bool NATS>
__device__ __forceinline__ void combine_records(const W1* rec, int n, float (&ref)[3],
                                                float (&sum)[3], float& v, int& vec) {
  const int lane = static_cast<int>(threadIdx.x & 31);
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    ref[q] = -INFINITY;
    sum[q] = 0.f;
  }
  v = -INFINITY;
  bool bad = false;
  for (int i = lane; i < n; i += 32) {
    const W1 r = rec[i];
#pragma unroll
    for (int q = 0; q < 3; ++q) ref[q] = fmaxf(ref[q], r.ref[q]);
    v = fmaxf(v, r.v);
    bad = bad || r.v != r.v;
  }
#pragma unroll
  for (int q = 0; q < 3; ++q) ref[q] = warp_max(ref[q]);
  v = warp_max(v);
  int lo = INT_MAX;
  for (int i = lane; i < n; i += 32) {
    const W1 r = rec[i];
#pragma unroll
    for (int q = 0; q < 3; ++q)
      sum[q] += (r.s[q] == 0.f || r.ref[q] == ref[q])
                    ? r.s[q]
                    : r.s[q] * ref_factor<NATS>(r.ref[q] - ref[q]);
    if (r.v == v) lo = min(lo, r.vec);
  }
  float z = 0.f;
  warp_sum4(sum[0], sum[1], sum[2], z);
  vec = static_cast<int>(__reduce_min_sync(0xffffffffu, static_cast<unsigned>(lo)));
  if (__any_sync(0xffffffffu, bad)) v = NAN;
}

// The row of this cluster: in memory order, but the bonus rows of the last
// elements (from KParams::tail_first on, about as many as the chip holds
// clusters; a grid of one wave has none) come last: they have no second pass,
// so the grid does not end on rows that have.  B=64, K=7, V=128256 bf16:
// stochastic 72.8 -> 71.4 us a step, greedy 65.5 -> 64.3.  (All bonus rows last
// cost fp32 rows of B=256 0.6 %, all rows k-major 1.4 %: the rows in flight lie
// on more pages.)
__device__ __forceinline__ void cluster_row(const KParams& P, unsigned& bi, unsigned& k) {
  asm("mov.u32 %0, %%clusterid.x;" : "=r"(k));
  asm("mov.u32 %0, %%clusterid.y;" : "=r"(bi));
  const unsigned first = static_cast<unsigned>(P.tail_first);
  if (bi < first) return;
  const unsigned K = static_cast<unsigned>(P.K);
  const unsigned l = (bi - first) * (K + 1u) + k;  // of the last elements' rows
  const unsigned drafts = (static_cast<unsigned>(P.B) - first) * K;
  if (l < drafts) {
    bi = first + l / K;
    k = l % K;
  } else {
    bi = first + l - drafts;
    k = K;
  }
}

// What a draft row's second pass has to find out, from its normalisers and
// its draft token's logits: nothing (the draft is accepted whatever D is),
// the residual masses alone (it is rejected whatever D is) or the divergence
// too.  Monotone in D: ln gamma - D is largest at D = 0 and smallest at the
// gate's upper bound, in fp32 as well; the stochastic test goes through
// expf, whose rounding the factors 1 +- 1e-6 cover.
template <bool STOCH>
__device__ __forceinline__ int row_path(const KParams& P, const float (&lse)[4], float da, float db,
                                        float dt, float u, float pd) {
  const bool jsd = P.divergence == ASYMSPEC_DIV_JSD, kl = P.divergence == ASYMSPEC_DIV_KL;
  const float lb = db - lse[1];
  float lo = P.ln_gamma, hi = P.ln_gamma;  // ln gamma_eff lies in [lo, hi]
  if (jsd) lo = P.ln_gamma - kLn2;
  if (kl) lo = -INFINITY;
  if (P.divergence == ASYMSPEC_DIV_LAMBDA) lo = hi = P.ln_gamma - P.lambda * ((da - lse[0]) - lb);
  if (!STOCH) {
    const float lr = (dt - lse[2]) - lb;
    if (lr > hi) return kPathAccept;
    return lr <= lo || !(jsd || kl) ? kPathReject : kPathFull;
  } else {
    const float qd = expf(fmaf(P.beta, da - db, dt) - lse[3]);
    const float slack = jsd || kl ? 1e-6f : 0.f;
    const float most = u * expf(hi) * pd, least = u * expf(lo) * pd;
    if (qd > most * (1.f + slack)) return kPathAccept;
    return (jsd && qd < least * (1.f - slack)) || !(jsd || kl) ? kPathReject : kPathFull;
  }
}

// Grid: C B (K+1) CTAs of kRowThreads threads in clusters of C, one cluster a
// row (cluster_row).  What it leaves for the
// decision kernel: rank 0's row statistics (the normalisers, the argmax, the
// row's path) and, for rows with a second pass and stochastic bonus rows,
// one record per warp of every CTA (KParams::pass2_rec, kRowMaxWarps records
// per CTA): the warp's divergence sum, the residual and fused masses of its
// block (its inverse-CDF group).  Dynamic shared memory: the fixed state and
// pushed records (row_shared_bytes(C)), then the warps' rings (kRingBytes) at
// KParams::sh_off.
template <typename T, bool STOCH, bool EDGE>
__global__ void __launch_bounds__(kRowThreads, kRowMinBlocks) fuse_verify_row(const KParams P) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  constexpr int NW = kRowThreads / 32;
  constexpr int VE = 16 / static_cast<int>(sizeof(T));
  extern __shared__ __align__(128) unsigned char smem_row[];
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = static_cast<int>(cluster.block_rank());
  const int tid = static_cast<int>(threadIdx.x);
  const int lane = tid & 31, warp = tid >> 5;
  const int C = P.C;
  unsigned ubi, uk;
  cluster_row(P, ubi, uk);
  const int k = static_cast<int>(uk), bi = static_cast<int>(ubi);
  const unsigned row32 = ubi * static_cast<unsigned>(P.K + 1) + uk;
  const RowCut<T, EDGE> cut(P, row32);
  const int Wv = P.W / VE, s0 = rank * Wv;  // the slice: vectors [s0, s0 + nv) of the row
  const int nv = max(0, min(Wv, cut.nvec - s0));
  int b0, b1;  // the warp's block of the slice
  row_block<false>(s0, nv, warp, b0, b1);
  // the block's whole vectors [v0, v1)
  const int v0 = EDGE ? max(b0, cut.in0 - s0) : b0;
  const int v1 = EDGE ? max(v0, min(b1, cut.in1 - s0)) : b1;
  const int i0 = v0 + lane;
  Streams<T> g;  // the lane's first vector
  {
    const size_t o = static_cast<size_t>(s0 + i0) * VE;
    g.a = cut.base(P.a) + o;
    g.b = cut.base(P.b) + o;
    g.t = cut.base(P.t) + o;
  }
  RowShared* sh = reinterpret_cast<RowShared*>(smem_row);
  uint4* ring = reinterpret_cast<uint4*>(smem_row + P.sh_off) + warp * (kRing * 96);
  const bool draft = k < P.K;
  const bool only_t = !STOCH && !draft && !P.fuse_bonus;  // Algorithm 1 emits argmax t
  const int nrec = C * NW;  // pass-1 records the cluster exchanges
  if (tid == 0) {
    mbar_init(&sh->xbar, 1);
    fence_mbar_init();
    mbar_arrive_expect_tx(&sh->xbar, static_cast<unsigned>(nrec * sizeof(W1)));
  }
  cluster_start(P, row32, rank);
  if (only_t) ring_prologue<T, false, true>(ring, g, i0, v1);
  else ring_prologue<T, true, true>(ring, g, i0, v1);
  const EdgeVals ed = load_edges<T, EDGE>(P, cut, row32, s0, b0, b1, !only_t);
  // every CTA's barrier is initialised before any push (the CTAs of a
  // cluster start together; this wait overlaps the first loads)
  cluster_wait();

  // ---- pass 1: the row normalisers, combined over the cluster
  // (a non-finite a or b makes D non-finite under a gate that sums it)
  const bool chk = P.divergence == ASYMSPEC_DIV_JSD || P.divergence == ASYMSPEC_DIV_KL;
  W1 e;
  auto pass1 = [&](auto prog) {
    constexpr int PROG = decltype(prog)::value;
    const bool ovf = row_pass1<T, PROG, EDGE>(ring, g, v0, v1, P.beta, chk, ed, s0 + i0,
                                              cut.nvec - 1, e);
    if (PROG != kGreedyBonusT && PROG != kGreedyBonusS && __any_sync(0xffffffffu, ovf)) {
      // an entry far above the warp's reference (or non-finite data): redo
      // the block with running maxima
      e = row_pass1_online<T, PROG, EDGE>(g, v0, v1, P.beta, chk, ed, e);
    }
  };
  if (STOCH) {
    if (draft) pass1(std::integral_constant<int, kStochDraft>{});
    else pass1(std::integral_constant<int, kStochBonus>{});
  } else {
    if (draft) pass1(std::integral_constant<int, kGreedyDraft>{});
    else if (only_t) pass1(std::integral_constant<int, kGreedyBonusT>{});
    else pass1(std::integral_constant<int, kGreedyBonusS>{});
  }
  cp_async_wait<0>();  // the pass's trailing (empty) groups; the ring is free
  if (lane < C) {
    // this warp's record into slot rank NW + warp of every CTA (lane j to CTA j)
    const float4* slot = reinterpret_cast<const float4*>(sh->recv() + rank * NW + warp);
    st_async16(slot, static_cast<unsigned>(lane), &sh->xbar,
               make_float4(e.ref[0], e.ref[1], e.ref[2], e.s[0]));
    st_async16(slot + 1, static_cast<unsigned>(lane), &sh->xbar,
               make_float4(e.s[1], e.s[2], e.v, __int_as_float(e.vec)));
  }
  bool got = true;
  if (warp == 0) {
    // the draft token's logits and scalars, loaded while the last records land
    float da = 0.f, db = 0.f, dt = 0.f, u = 0.f, pd = 1.f;
    bool tok_ok = false;
    if (draft) {
      const int d = __ldg(P.tokens + static_cast<size_t>(bi) * P.K + k);
      if (STOCH) {
        pd = __ldg(P.dprobs + static_cast<size_t>(bi) * P.K + k);
        u = __ldg(P.unif + row32);
      }
      tok_ok = d >= 0 && d < P.V;
      if (tok_ok) {
        const size_t o = static_cast<size_t>(row32) * P.V + d;
        da = elem_ldg(static_cast<const T*>(P.a) + o);
        db = elem_ldg(static_cast<const T*>(P.b) + o);
        dt = elem_ldg(static_cast<const T*>(P.t) + o);
      }
    }
    // every warp's record of the cluster is in this CTA once the barrier completes
    got = wait_records(&sh->xbar, rank);
    float ref[3], sum[3], v;
    int vec;
    combine_records<EDGE>(sh->recv(), nrec, ref, sum, v, vec);
    float lse[4];
    lse[0] = draft ? record_lse<EDGE>(ref[0], sum[0]) : NAN;
    lse[1] = draft ? record_lse<EDGE>(ref[1], sum[1]) : NAN;
    lse[2] = !STOCH && draft ? record_lse<EDGE>(ref[2], sum[2]) : NAN;
    lse[3] = STOCH ? record_lse<EDGE>(ref[2], sum[2]) : NAN;
    // (a token outside the vocabulary voids the element whatever the row does)
    const int path = draft && tok_ok ? row_path<STOCH>(P, lse, da, db, dt, u, pd) : kPathAccept;
    if (lane == 0) {
#pragma unroll
      for (int q = 0; q < 4; ++q) sh->lse[q] = lse[q];
      sh->path = path;
    }
    if (rank == 0) {
      // greedy: the element of the best vector, the lowest of the equal ones
      int idx = INT_MAX;
      if (!STOCH) {
        if (vec != INT_MAX) {
          const int el = vec * VE + lane - cut.head;
          bool eq = false;
          if (lane < VE && el >= 0 && el < P.V) {
            const size_t o = static_cast<size_t>(row32) * P.V + el;
            float x = elem_ldg(static_cast<const T*>(P.t) + o);
            if (!only_t)
              x = fmaf(P.beta, elem_ldg(static_cast<const T*>(P.a) + o) -
                                   elem_ldg(static_cast<const T*>(P.b) + o), x);
            eq = x == v;
          }
          const unsigned hit = __ballot_sync(0xffffffffu, eq);
          if (hit) idx = vec * VE + __ffs(hit) - 1 - cut.head;
        }
      }
      const unsigned bad = !STOCH && v != v ? (only_t ? kBadT : kBadS) : 0u;
      // the draft token's logits are read by the decision kernel itself
      if (lane == 0)
        store_stream_stat(P, row32, lse, only_t ? INT_MAX : idx, only_t ? idx : INT_MAX, bad, path);
    }
  }
  __syncthreads();

  // ---- pass 2: divergence terms and inverse-CDF masses, where the row needs them
  const int path = sh->path;
  const bool second = draft && path != kPathAccept && (STOCH || path == kPathFull);
  const float S2 = sh->lse[3] * kLog2e;
  float jsum = 0.f, msum = 0.f;
  if (second) {
    const float A2 = sh->lse[0] * kLog2e, B2 = sh->lse[1] * kLog2e;
    const ResConst kc = res_const(P.beta, A2, B2, S2);
    ring_prologue<T, true, STOCH>(ring, g, i0, v1);
    const bool jsd = P.divergence == ASYMSPEC_DIV_JSD;
    if (STOCH && path == kPathReject)
      row_pass2<T, kDivNone, STOCH, EDGE>(ring, g, v0, v1, kc, ed, jsum, msum);
    else if (jsd) row_pass2<T, kDivJsd, STOCH, EDGE>(ring, g, v0, v1, kc, ed, jsum, msum);
    else row_pass2<T, kDivKl, STOCH, EDGE>(ring, g, v0, v1, kc, ed, jsum, msum);
    cp_async_wait<0>();
    if (jsd && path == kPathFull && !(fabsf(jsum) <= 3.402823466e38f))
      jsum = row_jsd_wide<T, EDGE>(g, v0, v1, A2, B2, ed);
  }
  if (lane == 0 && (second || (STOCH && !draft))) {
    // this warp's record: its block is one inverse-CDF group of the row
    const float qf = STOCH ? block_mass<EDGE>(e.ref[2], e.s[2], S2) : 0.f;
    *reinterpret_cast<float4*>(
        P.pass2_rec + ((static_cast<size_t>(row32) * C + rank) * kRowMaxWarps + warp) * 8) =
        make_float4(jsum, msum, qf, 0.f);
  }
  if (warp == 0 && !got) late_end(P, row32, &sh->xbar);
}

// ---------------------------------------------------------------- row decisions

// One CTA per batch element.  Every warp decides rows k, k + 16, ... from
// their statistics (and, where the row's decision depends on D, its warps'
// divergence sums); Algorithm 1's scan then finds the row where the element
// stops, and in stochastic mode the whole CTA draws from that row alone: the
// group that holds the target (one lane per four groups, in the row's own
// warp), then the group's vectors, one per thread, in one trip to memory.
// (One warp per row walking its own group through shared memory, for every
// row, took 19 us cold and about 10 us of the step at B = 64, K = 7.)
constexpr int kDrawThreads = 512;  // a warp block holds at most this many vectors
constexpr int kDrawWarps = kDrawThreads / 32;
static_assert(kWalkRounds * 32 <= kDrawThreads, "one vector of a group per thread");

// What the decision of row (bi, k) needs from the kernel's inputs (not from
// the row kernel): the draft token, its three logits, the row's scalars.
// Loaded before griddepcontrol.wait, so that the loads overlap the row
// kernel's last CTAs.
struct RowInputs {
  int dtok;
  float ad, bd, td;
  RowScalars sc;
};

template <typename T, bool STOCH>
__device__ __forceinline__ RowInputs load_row_inputs(const KParams& P, int bi, int k) {
  RowInputs d;
  d.dtok = -1;
  d.ad = d.bd = d.td = 0.f;
  d.sc = STOCH ? load_row_scalars(P, bi, k) : RowScalars{0.f, 0.f, 0.f};
  if (k < P.K) {
    d.dtok = P.tokens[static_cast<size_t>(bi) * P.K + k];
    if (d.dtok >= 0 && d.dtok < P.V) {
      const size_t o = (static_cast<size_t>(bi) * (P.K + 1) + k) * P.V + d.dtok;
      d.ad = to_f32(static_cast<const T*>(P.a)[o]);
      d.bd = to_f32(static_cast<const T*>(P.b)[o]);
      d.td = to_f32(static_cast<const T*>(P.t)[o]);
    }
  }
  return d;
}

// Where a row's draw lies: the group (g = rank NW + warp; -1: the row has no
// mass), the target inside it, whether rounding left the target at or beyond
// the row's mass (the last positive entry is drawn), and which masses.
struct Draw {
  int g;
  float rem;
  int last, use_r;
};

// By one warp: the draw's group from the masses of the row's C x NW groups
// (lane l holds groups 4l .. 4l + 3, in index order); total: the row's mass.
__device__ __forceinline__ Draw select_group(const float (&Rm)[4], const float (&Qm)[4], bool bonus,
                                             float u_last, float& total) {
  const int lane = threadIdx.x & 31;
  const float Rl = (Rm[0] + Rm[1]) + (Rm[2] + Rm[3]), Ql = (Qm[0] + Qm[1]) + (Qm[2] + Qm[3]);
  const float R_all = warp_sum(Rl), Q_all = warp_sum(Ql);
  const bool r_ok = !bonus && R_all > 0.f;
  const float ml = r_ok ? Rl : Ql;
  total = r_ok ? R_all : Q_all;
  const float tau = u_last * total;
  Draw d{-1, 0.f, 0, r_ok ? 1 : 0};
  float incl = ml;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const float v = __shfl_up_sync(0xffffffffu, incl, off);
    if (lane >= off) incl += v;
  }
  const float excl = incl - ml;
  const unsigned hit = __ballot_sync(0xffffffffu, ml > 0.f && excl <= tau && tau < incl);
  const unsigned pos = __ballot_sync(0xffffffffu, ml > 0.f);
  if (!pos) return d;
  bool last = !hit;
  const int lc = hit ? __ffs(hit) - 1 : 31 - __clz(pos);
  // the group, inside lane lc's four
  int gsel = -1, glast = -1;
  float rem = 0.f;
  if (lane == lc) {
    float cum = excl;
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      const float m = r_ok ? Rm[h] : Qm[h];
      if (m > 0.f) glast = 4 * lane + h;
      if (!last && gsel < 0) {
        if (m > 0.f && cum + m > tau) {
          gsel = 4 * lane + h;
          rem = fmaxf(tau - cum, 0.f);
        } else {
          cum += m;
        }
      }
    }
    if (gsel < 0) {
      gsel = glast;
      last = true;
    }
  }
  d.g = __shfl_sync(0xffffffffu, gsel, lc);
  d.rem = __shfl_sync(0xffffffffu, rem, lc);
  d.last = __shfl_sync(0xffffffffu, last ? 1 : 0, lc);
  return d;
}

// A row's statistics and its warps' records, as decided from (one warp; one
// trip to the L2): the divergence sum (every lane) and the masses of groups
// 4 lane .. 4 lane + 3.  ng: the row's groups.
struct RowRecords {
  RowStat st;
  float j, R[4], Q[4];
};

__device__ __forceinline__ RowRecords load_records(const KParams& P, long long row, int ng) {
  RowRecords x;
  const int lane = threadIdx.x & 31;
  const float4* src = reinterpret_cast<const float4*>(static_cast<const RowStat*>(P.row_stat) + row);
  float4* dst = reinterpret_cast<float4*>(&x.st);
  dst[0] = __ldcg(src);
  dst[1] = __ldcg(src + 1);
  x.st.late = __ldcg(&static_cast<const RowStat*>(P.row_stat)[row].late);
  float j = 0.f;
#pragma unroll
  for (int h = 0; h < 4; ++h) {
    const int q = 4 * lane + h;
    x.R[h] = x.Q[h] = 0.f;
    if (q < ng) {  // record q: warp q % NW of CTA q / NW (ng = C NW)
      const float4 v = __ldcg(
          reinterpret_cast<const float4*>(P.pass2_rec + (static_cast<size_t>(row) * ng + q) * 8));
      j += v.x;
      x.R[h] = v.y;
      x.Q[h] = v.z;
    }
  }
  x.j = warp_sum(j);
  return x;
}

// The divergence from its sum: 2 JSD, or KL, in bits.
__device__ __forceinline__ float divergence_nats(const KParams& P, float j) {
  return P.divergence == ASYMSPEC_DIV_JSD ? 0.5f * kLn2 * j
         : P.divergence == ASYMSPEC_DIV_KL ? kLn2 * j
                                           : 0.f;
}

// The draw inside a group by the whole CTA (kDrawThreads threads), thread i
// holding the masses of the group's entries [2 NP i, 2 NP (i + 1)): the
// smallest entry whose cumulative mass exceeds the target; every thread
// returns it (-1: no mass).
template <int NP>
__device__ __forceinline__ int block_pick(const f2 (&m2)[NP], const Draw& dr) {
  __shared__ float wtot[kDrawWarps];
  __shared__ int wfirst[kDrawWarps], wlast[kDrawWarps], s_pick;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const float mv = vsum(m2);
  float vin = mv;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const float x = __shfl_up_sync(0xffffffffu, vin, off);
    if (lane >= off) vin += x;
  }
  if (lane == 31) wtot[warp] = vin;
  __syncthreads();
  float before = 0.f;
  for (int q = 0; q < warp; ++q) before += wtot[q];
  const unsigned over = __ballot_sync(0xffffffffu, !dr.last && mv > 0.f && before + vin > dr.rem);
  const unsigned pos = __ballot_sync(0xffffffffu, mv > 0.f);
  if (lane == 0) {
    wfirst[warp] = over ? __ffs(over) - 1 : -1;
    wlast[warp] = pos ? 31 - __clz(pos) : -1;
  }
  if (threadIdx.x == 0) s_pick = -1;
  __syncthreads();
  int first = -1, last = -1;
#pragma unroll
  for (int q = kDrawWarps - 1; q >= 0; --q) {
    if (wfirst[q] >= 0) first = 32 * q + wfirst[q];
    if (last < 0 && wlast[q] >= 0) last = 32 * q + wlast[q];
  }
  const int pick = first >= 0 ? first : last;  // the thread that holds the entry
  if (static_cast<int>(threadIdx.x) == pick) {
    const float rem = fmaxf(dr.rem - (before + (vin - mv)), 0.f);
    float cum = 0.f;
    int el = -1, lastel = -1;
#pragma unroll
    for (int h = 0; h < NP; ++h) {
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const float m = q == 0 ? lo_of(m2[h]) : hi_of(m2[h]);
        if (m > 0.f) lastel = 2 * h + q;
        cum += m;
        if (first >= 0 && el < 0 && cum > rem) el = 2 * h + q;
      }
    }
    if (el < 0) el = lastel;
    s_pick = pick * 2 * NP + el;
  }
  __syncthreads();
  return s_pick;
}

// The row's draw: the masses of the group's vectors, one per thread, formed
// exactly as the row kernel forms them; every thread returns the token (-1:
// no mass).
template <typename T, bool EDGE, bool LINES = false>
__device__ __forceinline__ int block_draw(const KParams& P, long long row, const Draw& dr, float A2,
                                          float S2) {
  constexpr int VE = 16 / static_cast<int>(sizeof(T));
  constexpr int NP = VE / 2;
  constexpr int NW = kRowThreads / 32;
  const RowCut<T, EDGE> cut(P, row);
  const int Wv = P.W / VE, rk = max(dr.g, 0) / NW, w = max(dr.g, 0) - rk * NW;
  const int s0 = rk * Wv, nv = max(0, min(Wv, cut.nvec - s0));
  int b0, b1;
  row_block<LINES>(s0, nv, w, b0, b1);
  const int g0 = s0 + b0, g1 = s0 + b1;
  const int i = g0 + static_cast<int>(threadIdx.x);  // this thread's vector of the row
  const ResConst kc = res_const(P.beta, A2, 0.f, S2);
  f2 m2[NP];
#pragma unroll
  for (int h = 0; h < NP; ++h) m2[h] = 0ull;
  if (dr.g >= 0 && i < g1) {
    const T *pa = cut.base(P.a), *pb = cut.base(P.b), *pt = cut.base(P.t);
    const size_t o = static_cast<size_t>(i) * VE;
    f2 xa[NP], xb[NP], xt[NP];
    if (!EDGE || (i >= cut.in0 && i < cut.in1)) {
      const RawVec<T> va = raw_ldg(pa + o), vb = raw_ldg(pb + o), vt = raw_ldg(pt + o);
#pragma unroll
      for (int h = 0; h < NP; ++h) {
        xa[h] = va.pair(h);
        xb[h] = vb.pair(h);
        xt[h] = vt.pair(h);
      }
    } else {
      const int el0 = i * VE - cut.head;
#pragma unroll
      for (int h = 0; h < NP; ++h) {
        float x[6];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const bool in = el0 + 2 * h + q >= 0 && el0 + 2 * h + q < P.V;
          const size_t oe = o + 2 * h + q;
          x[q] = in ? elem_ldg(pa + oe) : kEdgeNone;
          x[2 + q] = in ? elem_ldg(pb + oe) : kEdgeNone;
          x[4 + q] = in ? elem_ldg(pt + oe) : kEdgeNone;
        }
        xa[h] = pk(x[0], x[1]);
        xb[h] = pk(x[2], x[3]);
        xt[h] = pk(x[4], x[5]);
      }
    }
#pragma unroll
    for (int h = 0; h < NP; ++h) {
      f2 amb, p, qf, r;
      res_pair(xa[h], xb[h], xt[h], kc, amb, p, qf, r);
      m2[h] = dr.use_r ? r : qf;
    }
  }
  const int pick = block_pick(m2, dr);
  return pick < 0 ? -1 : g0 * VE + pick - cut.head;
}

// One batch element, by one CTA.  Rows: where the rows' inputs lie,
//   groups(P): warp records per row;  refused(P, bi): the whole call is a data
//   error (its outputs are written);  inputs(P, bi, k): load_row_inputs;
//   draw(P, row, dr, A2, S2): block_draw;  emit(P, bi, len, next): the
//   element's outputs (thread 0; next < 0 on a data error).
template <bool STOCH, typename Rows>
__device__ __forceinline__ void decide_element(const KParams& P, const Rows& rows) {
  __shared__ int4 srec[kDecideSmemRows];   // the element's records (accept, candidate, error bits)
  __shared__ Draw sdraw[kDecideSmemRows];  // where each row's draw lies
  __shared__ float slse[kDecideSmemRows][2];  // LSE(a), LSE(s) of each row
  __shared__ int s_len, s_err;
  const int bi = blockIdx.x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int K = P.K, K1 = K + 1;
  const bool in_smem = K1 <= kDecideSmemRows;
  // the kernel inputs of this warp's first row, loaded before the wait
  RowInputs pre{-1, 0.f, 0.f, 0.f, RowScalars{0.f, 0.f, 0.f}};
  if (warp < K1) pre = rows.inputs(P, bi, warp);
  // launched as a programmatic dependent of the row kernel: its CTAs may
  // start early; nothing of the workspace is read before that kernel is done
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (rows.refused(P, bi)) return;
  // Decides row k (one warp).  The group records are loaded with the row's
  // statistics (one trip) and used only where the row left some.
  auto decide = [&](int k, const RowInputs& din, Draw& dr, float (&lse_as)[2]) {
    const long long row = static_cast<long long>(bi) * K1 + k;
    const bool bonus = k == K;
    const RowRecords x = load_records(P, row, rows.groups(P));
    const RowStat& st = x.st;
    RowResult rr;
    rr.lse_a = bonus ? NAN : st.lse[0];
    rr.lse_b = bonus ? NAN : st.lse[1];
    rr.lse_t = st.lse[2];
    rr.lse_s = st.lse[3];
    rr.D = !bonus && st.path == kPathFull ? divergence_nats(P, x.j) : 0.f;
    rr.is = st.is;
    rr.it = st.it;
    rr.sample = 0;  // the stop row's draw follows the scan
    rr.mass = NAN;
    rr.bad = st.bad | st.late;
    rr.have_lse_t = !STOCH && !bonus;
    int4 rec = row_record<STOCH>(P, row, k, rr, din.dtok, din.ad, din.bd, din.td, din.sc, lane == 0);
    if (!bonus && st.path == kPathAccept) rec.x = 1;
    if (!bonus && st.path == kPathReject) rec.x = 0;
    lse_as[0] = st.lse[0];
    lse_as[1] = st.lse[3];
    if (STOCH && (bonus || rec.x == 0)) {
      float total;
      dr = select_group(x.R, x.Q, bonus, din.sc.u_last, total);
    }
    return rec;
  };
  for (int k = warp; k < K1; k += nw) {
    const RowInputs din = (k == warp) ? pre : rows.inputs(P, bi, k);
    Draw dr{-1, 0.f, 0, 0};
    float las[2];
    const int4 rec = decide(k, din, dr, las);
    if (lane == 0) {
      if (in_smem) {
        srec[k] = rec;
        sdraw[k] = dr;
        slse[k][0] = las[0];
        slse[k][1] = las[1];
      } else {
        P.recs[static_cast<size_t>(bi) * K1 + k] = rec;
      }
    }
  }
  __syncthreads();
  if (warp == 0) {
    // Algorithm 1: the first rejected draft, or K if none; any data error voids the element
    const int4* recs = P.recs + static_cast<size_t>(bi) * K1;
    bool any_err = false;
    int len = -1, next = -1;
    for (int base = 0; base < K1; base += 32) {
      const int j = base + lane;
      int4 v = make_int4(1, -1, 0, 0);
      if (j < K1) v = in_smem ? srec[j] : __ldcg(&recs[j]);
      any_err |= __any_sync(0xffffffffu, v.z != 0);
      if (len < 0) {
        const unsigned rej = __ballot_sync(0xffffffffu, j < K && v.x == 0);
        if (rej) len = base + __ffs(rej) - 1;
        else if (K < base + 32) len = K;
        if (len >= 0) next = __shfl_sync(0xffffffffu, v.y, len - base);
      }
    }
    if (STOCH && !in_smem && !any_err) {  // the stop row's group was not kept
      Draw dr{-1, 0.f, 0, 0};
      float las[2];
      decide(len, rows.inputs(P, bi, len), dr, las);
      if (lane == 0) {
        sdraw[0] = dr;
        slse[0][0] = las[0];
        slse[0][1] = las[1];
      }
    }
    if (lane == 0) {
      s_len = len;
      s_err = any_err;
      if (any_err) rows.emit(P, bi, -1, -1);
      else if (!STOCH) rows.emit(P, bi, len, next);
    }
  }
  if constexpr (STOCH) {
    __syncthreads();
    if (s_err) return;
    const int len = s_len, at = in_smem ? len : 0;
    const int tok = rows.draw(P, static_cast<long long>(bi) * K1 + len, sdraw[at],
                              slse[at][0] * kLog2e, slse[at][1] * kLog2e);
    if (threadIdx.x == 0) {
      // (no mass at all: non-finite data that the normalisers did not show)
      rows.emit(P, bi, tok < 0 ? -1 : len, tok);
      if (tok < 0 && P.err_word) atomicOr(P.err_word, ASYMSPEC_DATA_NONFINITE);
    }
  }
}

// Rows [B, K+1, V] of one vocabulary.
template <typename T, bool STOCH, bool EDGE>
struct PlainRows {
  __device__ __forceinline__ int groups(const KParams& P) const { return P.C * (kRowThreads / 32); }
  __device__ __forceinline__ bool refused(const KParams&, int) const { return false; }
  __device__ __forceinline__ RowInputs inputs(const KParams& P, int bi, int k) const {
    return load_row_inputs<T, STOCH>(P, bi, k);
  }
  __device__ __forceinline__ int draw(const KParams& P, long long row, const Draw& dr, float A2,
                                      float S2) const {
    return block_draw<T, EDGE>(P, row, dr, A2, S2);
  }
  __device__ __forceinline__ void emit(const KParams& P, int bi, int len, int next) const {
    P.out_len[bi] = len;
    P.out_next[bi] = next;
  }
};

template <typename T, bool STOCH, bool EDGE>
__global__ void __launch_bounds__(kDrawThreads) decide_blocks(const KParams P) {
  decide_element<STOCH>(P, PlainRows<T, STOCH, EDGE>{});
}

}  // namespace asymspec_impl
