// The augmented drafter's draw (Section 3.2, item 1; the drafting step of
// Algorithm 1): per position, greedy d = argmax a (lowest index on ties) or,
// sampling, the inverse CDF of softmax(a) at the position's uniform, plus
// the drafter's probability of its draw, softmax(a)[d].
//
// One cluster of C CTAs (1 <= C <= 8) per row: CTA c owns the vectors
// [c W, (c + 1) W) of the row (VE elements each; the last slice may be
// shorter or empty).  In a slice, vector v0 + r kDThreads + t is handled by
// thread t in round r, read through the thread's own slots of a ring in shared
// memory (cp.async, kDRing rounds in flight without holding registers).
// What bounds it: HBM in the middle, and about 7 us of starting a CTA, its
// reductions and the walk (512 rows of bf16 V=128256: 28.5 us, 19.7 at the
// copy rate; 29.7 with the next batch of rounds in registers instead of the
// ring, and one element at a time 80.6 us for V=100003, 28.9 now).
// EDGE: a row off the 16-byte boundaries is cut at them: vector 0 starts
// `head` elements before the row and the last may end after it; their
// elements inside the row are loaded one by one, the others stand as the
// type's lowest value, which adds no mass and is never drawn.
// Each CTA reads its slice once from HBM and pushes a summary (reference,
// mass relative to it, finiteness sum, argmax index) into every CTA of the
// cluster; after one cluster barrier every CTA combines the C summaries
// locally and identically, so no shared memory is read remotely.
//   greedy    per thread a running maximum, the lowest vector that holds it
//             and the sum of 2^((x - m) log2 e), rescaled when the maximum
//             moves.  Rank 0 writes d (the lowest index holding the row
//             maximum) and softmax(a)[d] = 1 / S.
//   sampling  one pass: every warp takes as its reference R_w (log2 units) the maximum of
//             its first round's vectors and stores the mass 2^(x log2 e
//             - R_w) of each group of 32 consecutive vectors (one warp in one
//             round) in shared memory.  If any group's mass reaches 2^100 (an
//             entry ~69 nats above its warp's reference) the CTA redoes the
//             slice against the slice maximum.  Combining: the row reference
//             R is the largest R_w; the CTA whose slice holds the target u S
//             (S in units of 2^R, R in log2 units) walks its groups, the 32 vectors of the
//             group (recomputed against R) and the elements of the vector.
//             If rounding leaves the target at or past a boundary with no
//             owner, the last entry of positive mass is taken.
// Finite logits of any size are taken.  What has a reference so far below zero that
// x log2 e has no room for a fraction, or overflows (masks of the type's lowest
// value), has no mass (greedy: thread_again); a row whose own reference lies there,
// or as far above, is worked again by wide_row.
// Non-finite data: every element also enters f = sum x 2^-40, finite
// exactly when all elements are (2^-40 keeps 2^20 fp32 maxima finite).  A
// row with a non-finite logit, or a uniform outside [0, 1), gets token -1
// and probability NaN.
#pragma once

#include "device_common.cuh"

namespace asymspec_impl {

constexpr int kDThreads = 256;
constexpr int kDWarps = kDThreads / 32;
constexpr int kDUnroll = 4;       // rounds used at a time
constexpr int kDRing = 8;         // rounds in flight
constexpr int kDRingBytes = kDRing * kDThreads * 16;
static_assert(kDRing == 2 * kDUnroll, "one batch in use, one behind it in flight");
constexpr int kDMaxCluster = 8;
constexpr float kDFinScale = 9.094947017729282e-13f;  // 2^-40
constexpr float kDGuard = 1.2676506002282294e30f;     // 2^100

struct DParams {
  const void* logits;  // [rows, V], row stride V
  const float* unif;   // [rows] (sampling)
  int32_t* tokens;     // [rows]
  float* probs;        // [rows]
  int rows, V;
  int W;               // vectors per CTA slice
  int head0;           // EDGE: elements from a 16-byte boundary to the logits
};

// A CTA's summary of its slice.
struct __align__(16) DSlice {
  float ref;  // greedy: the slice maximum; sampling: the largest warp reference
  float sum;  // sum of 2^((x - ref) log2 e) over the slice
  float fin;  // sum of x 2^-40 over the slice
  int idx;    // greedy: lowest element index holding the maximum (INT_MAX if none)
};

struct DShared {
  DSlice slot[kDMaxCluster];  // slot c: CTA c's summary (pushed by CTA c)
  float red[2 * kDWarps];
  int redi[kDWarps];
  float wref[kDWarps];    // sampling: the warps' references
  float wscale[kDWarps];  // sampling: 2^(R_w - R)
};

__device__ __forceinline__ float dwarp_max(float v) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, off));
  return v;
}

__device__ __forceinline__ float dwarp_sum(float v) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  return v;
}

__device__ __forceinline__ float dwarp_incl_scan(float v, int lane) {
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const float y = __shfl_up_sync(0xffffffffu, v, off);
    if (lane >= off) v += y;
  }
  return v;
}

// A vector of consecutive logits as loaded: 8 packed bf16 or 4 fp32.
template <typename T>
struct DRaw;
template <>
struct DRaw<__nv_bfloat16> {
  static constexpr int VE = 8;
  uint4 q;
};
template <>
struct DRaw<float> {
  static constexpr int VE = 4;
  float4 q;
};

// One row, cut into vectors: vector v holds elements [v VE - head, (v + 1) VE
// - head); vectors [in0, in1) lie inside the row whole.
template <typename T, bool EDGE>
struct DRow {
  static constexpr int VE = DRaw<T>::VE;
  const T* base;  // vector 0 (may precede the row)
  int V, head, nvec, in0, in1;
  __device__ __forceinline__ DRow(const DParams& P, int row) {
    const long long off = static_cast<long long>(row) * P.V;
    V = P.V;
    head = EDGE ? static_cast<int>((off + P.head0) & (VE - 1)) : 0;
    base = static_cast<const T*>(P.logits) + off - head;
    nvec = (head + V + VE - 1) / VE;
    in0 = EDGE ? (head != 0) : 0;
    in1 = EDGE ? (head + V) / VE : nvec;
  }
  __device__ __forceinline__ bool whole(int v) const { return !EDGE || (v >= in0 && v < in1); }
  __device__ __forceinline__ int element(int v, int e) const { return v * VE + e - head; }
  __device__ __forceinline__ bool inside(int v, int e) const {
    const int i = element(v, e);
    return !EDGE || (i >= 0 && i < V);
  }
};

// A partial vector: its elements inside the row, the others the type's lowest.
template <bool EDGE>
__device__ __noinline__ DRaw<__nv_bfloat16> dld_edge(DRow<__nv_bfloat16, EDGE> r, int v) {
  const unsigned short* p = reinterpret_cast<const unsigned short*>(r.base) + static_cast<long long>(v) * 8;
  unsigned w[4];
#pragma unroll
  for (int h = 0; h < 4; ++h) {
    const unsigned lo = r.inside(v, 2 * h) ? __ldg(p + 2 * h) : 0xFF7Fu;
    const unsigned hi = r.inside(v, 2 * h + 1) ? __ldg(p + 2 * h + 1) : 0xFF7Fu;
    w[h] = hi << 16 | lo;
  }
  return {make_uint4(w[0], w[1], w[2], w[3])};
}
template <bool EDGE>
__device__ __noinline__ DRaw<float> dld_edge(DRow<float, EDGE> r, int v) {
  const float* p = r.base + static_cast<long long>(v) * 4;
  float x[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) x[e] = r.inside(v, e) ? __ldg(p + e) : -3.402823466e38f;
  return {make_float4(x[0], x[1], x[2], x[3])};
}
// Vector v of the row.
template <typename T, bool EDGE>
__device__ __forceinline__ DRaw<T> dld(const DRow<T, EDGE>& r, int v) {
  if constexpr (EDGE) {
    if (!r.whole(v)) return dld_edge(r, v);
  }
  DRaw<T> x;
  x.q = __ldg(reinterpret_cast<const decltype(x.q)*>(r.base) + v);
  return x;
}

// The vector widened to fp32.
__device__ __forceinline__ void dwiden(const DRaw<__nv_bfloat16>& r, float (&x)[8]) {
  const unsigned w[4] = {r.q.x, r.q.y, r.q.z, r.q.w};
#pragma unroll
  for (int h = 0; h < 4; ++h) {
    x[2 * h] = __uint_as_float(w[h] << 16);
    x[2 * h + 1] = __uint_as_float(w[h] & 0xFFFF0000u);
  }
}
__device__ __forceinline__ void dwiden(const DRaw<float>& r, float (&x)[4]) {
  x[0] = r.q.x;
  x[1] = r.q.y;
  x[2] = r.q.z;
  x[3] = r.q.w;
}

// The thread's slots of the ring: slot q of round r = q (mod kDRing).  A
// thread reads back only what it copied itself, so no barrier is needed.
template <typename T, bool EDGE>
__device__ __forceinline__ void dring_issue(uint4* ring, const DRow<T, EDGE>& r, int v0, int v1,
                                            int round) {
#pragma unroll
  for (int u = 0; u < kDUnroll; ++u) {
    const int v = v0 + (round + u) * kDThreads + static_cast<int>(threadIdx.x);
    uint4* d = ring + ((round + u) % kDRing) * kDThreads + threadIdx.x;
    if (v < v1) {
      if (r.whole(v)) {
        cp_async16(d, r.base + static_cast<long long>(v) * DRaw<T>::VE);
      } else if constexpr (EDGE) {
        DRaw<T> x = dld_edge(r, v);
        *reinterpret_cast<decltype(x.q)*>(d) = x.q;
      }
    }
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}
// use(round, raw) for every batch of kDUnroll rounds of the slice, in order
// (raw[u] of a vector at or past v1 is undefined).
template <typename T, bool EDGE, typename Use>
__device__ __forceinline__ void dring_rounds(uint4* ring, const DRow<T, EDGE>& r, int v0, int v1,
                                             Use&& use) {
  const int rounds = (v1 - v0 + kDThreads - 1) / kDThreads;
  for (int q = 0; q < rounds; q += kDUnroll) {
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    DRaw<T> raw[kDUnroll];
#pragma unroll
    for (int u = 0; u < kDUnroll; ++u)
      raw[u].q = *reinterpret_cast<const decltype(raw[u].q)*>(
          ring + ((q + u) % kDRing) * kDThreads + threadIdx.x);
    use(q, raw);
    // the slots just used take the batch after the next (their values were
    // consumed by instructions this thread has already issued)
    dring_issue<T, EDGE>(ring, r, v0, v1, q + kDRing);
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
}
// The first kDRing rounds (two commit groups).
template <typename T, bool EDGE>
__device__ __forceinline__ void dring_start(uint4* ring, const DRow<T, EDGE>& r, int v0, int v1) {
  dring_issue<T, EDGE>(ring, r, v0, v1, 0);
  dring_issue<T, EDGE>(ring, r, v0, v1, kDUnroll);
}

// The finiteness sum f = sum x 2^-40: packed bf16 pairs for bf16 vectors
// (non-finite values propagate through bf16 arithmetic as through fp32), fp32
// pairs for fp32 vectors.
template <typename T>
struct DFin;
template <>
struct DFin<__nv_bfloat16> {
  unsigned acc = 0u;  // two bf16 partial sums
  __device__ __forceinline__ void add(const DRaw<__nv_bfloat16>& r) {
    const unsigned scale = 0x2B802B80u;  // 2^-40 in both halves
    const unsigned w[4] = {r.q.x, r.q.y, r.q.z, r.q.w};
#pragma unroll
    for (int h = 0; h < 4; ++h) asm("fma.rn.bf16x2 %0, %1, %2, %0;" : "+r"(acc) : "r"(w[h]), "r"(scale));
  }
  __device__ __forceinline__ float value() const {
    return __uint_as_float(acc << 16) + __uint_as_float(acc & 0xFFFF0000u);
  }
};
template <>
struct DFin<float> {
  f2 acc = 0ull;
  __device__ __forceinline__ void add(const DRaw<float>& r) {
    const f2 scale = pk(kDFinScale, kDFinScale);
    acc = fma2(pk(r.q.x, r.q.y), scale, acc);
    acc = fma2(pk(r.q.z, r.q.w), scale, acc);
  }
  __device__ __forceinline__ float value() const { return hsum2(acc); }
};
template <int VE>
__device__ __forceinline__ float dvmax(const float (&x)[VE]) {
  float m = x[0];
#pragma unroll
  for (int e = 1; e < VE; ++e) m = fmaxf(m, x[e]);
  return m;
}

// Sum of 2^(x log2 e + nm2) over a vector (nm2: minus its reference in log2
// units), in fp32 pairs.
template <int VE>
__device__ __forceinline__ float dmass(const float (&x)[VE], float nm2) {
  const f2 l2 = pk(kLog2e, kLog2e), n2 = pk(nm2, nm2);
  f2 acc = ex2_2(fma2(pk(x[0], x[1]), l2, n2));
#pragma unroll
  for (int h = 1; h < VE / 2; ++h) acc = add2(acc, ex2_2(fma2(pk(x[2 * h], x[2 * h + 1]), l2, n2)));
  return hsum2(acc);
}

// Warp sums of four per-lane values at once: lane l returns the sum over the
// warp of value q(l) = 2 (bit 4 of l) + (bit 3 of l), so lanes 0, 8, 16 and 24
// hold the sums of m0, m1, m2 and m3 (six shuffles instead of twenty).
__device__ __forceinline__ float dwarp_sum4(float m0, float m1, float m2, float m3, int lane) {
  const bool h16 = (lane & 16) != 0, h8 = (lane & 8) != 0;
  float a = h16 ? m2 : m0, b = h16 ? m3 : m1;
  a += __shfl_xor_sync(0xffffffffu, h16 ? m0 : m2, 16);
  b += __shfl_xor_sync(0xffffffffu, h16 ? m1 : m3, 16);
  float c = h8 ? b : a;
  c += __shfl_xor_sync(0xffffffffu, h8 ? a : b, 8);
  c += __shfl_xor_sync(0xffffffffu, c, 4);
  c += __shfl_xor_sync(0xffffffffu, c, 2);
  c += __shfl_xor_sync(0xffffffffu, c, 1);
  return c;
}

__device__ __forceinline__ bool dfinite(float f) { return fabsf(f) <= 3.402823466e38f; }

// 2^((ref - R) log2 e) times a mass; an empty mass stays 0 whatever ref is.
// LOG2: the references are in log2 units.
template <bool LOG2 = false>
__device__ __forceinline__ float drescale(float mass, float ref, float R) {
  return mass > 0.f ? mass * ex2(LOG2 ? ref - R : (ref - R) * kLog2e) : 0.f;
}

// Sampling's reference from one of its values: a whole number of log2 units,
// so that neither a reference nor a rescale between two rounds.  RMS relative
// error of the drawn token's probability against 64 bits, V = 32000 to 128256:
// 2.3e-7 bf16, 2.6e-7 fp32 (references in nats 3.8e-7 and 4.3e-7, at the same speed).
__device__ __forceinline__ float dref(float x) { return rintf(x * kLog2e); }
// References (log2 units) from here on are too large for their exponents: below
// it an exponent's rounding stays below 2^6, and a group's mass below kDGuard.
constexpr float kDWideRef = 536870912.f;  // 2^29

// ---------------------------------------------------------------- greedy slice

// The log2 units a greedy thread's masses are formed against: its maximum m times
// log2 e, rounded (a rescale takes the difference of two such, and greedy_mass takes
// the rounding out at the end: for m = 1e5 it is 2^-9 of a mass).
__device__ __forceinline__ float dlog2(float m) { return __fmul_rn(m, kLog2e); }
// A sum of masses against dlog2(m), restated against m.
__device__ __forceinline__ float greedy_mass(float s, float m) {
  return s * ex2(fmaf(-m, kLog2e, dlog2(m)));
}

// The thread's sum again, against its maximum m: it saw masks (or non-finite data)
// before its first ordinary vector, or nothing else.
template <typename T, bool EDGE>
__device__ __noinline__ float thread_again(DRow<T, EDGE> a, int v0, int v1, float m) {
  float s = 0.f;
  if (!(-m * kLog2e < kDWideRef)) return s;
  for (int v = v0 + static_cast<int>(threadIdx.x); v < v1; v += kDThreads) {
    float x[DRaw<T>::VE];
    dwiden(dld<T, EDGE>(a, v), x);
    s += dmass(x, -dlog2(m));
  }
  return greedy_mass(s, m);
}

template <typename T, bool EDGE>
__device__ __forceinline__ DSlice slice_greedy(const DRow<T, EDGE>& a, int v0, int v1, uint4* ring,
                                               DShared& sh) {
  constexpr int VE = DRaw<T>::VE;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float m = -INFINITY;
  float su[kDUnroll] = {};  // one sum per round of a batch: shorter chains of roundings
  DFin<T> fin;
  int bvec = INT_MAX;
  auto take = [&](const DRaw<T>& raw, int v, float& s) {
    float x[VE];
    dwiden(raw, x);
    const float vm = dvmax(x);
    if (vm > m) {  // strict: the lowest vector of this thread keeps the maximum
      const float f = ex2(__fsub_rn(dlog2(m), dlog2(vm)));
#pragma unroll
      for (int u = 0; u < kDUnroll; ++u) su[u] *= f;
      m = vm;
      bvec = v;
    }
    s += dmass(x, -dlog2(m));
    fin.add(raw);
  };
  dring_start<T, EDGE>(ring, a, v0, v1);
  dring_rounds<T, EDGE>(ring, a, v0, v1, [&](int r, const DRaw<T> (&raw)[kDUnroll]) {
#pragma unroll
    for (int u = 0; u < kDUnroll; ++u) {
      const int v = v0 + (r + u) * kDThreads + tid;
      if (v < v1) take(raw[u], v, su[u]);
    }
  });
  float s = greedy_mass((su[0] + su[1]) + (su[2] + su[3]), m);
  if (!dfinite(s)) s = thread_again<T, EDGE>(a, v0, v1, m);
  // the CTA maximum, the lowest vector holding it, the sum rescaled to it
  const float w = dwarp_max(m);
  if (lane == 0) sh.red[warp] = w;
  __syncthreads();
  const float M = dwarp_max(lane < kDWarps ? sh.red[lane] : -INFINITY);
  const int vsel = __reduce_min_sync(0xffffffffu, m == M ? bvec : INT_MAX);
  const float ws = dwarp_sum(drescale(s, m, M));
  const float wf = dwarp_sum(fin.value());
  __syncthreads();
  if (lane == 0) {
    sh.redi[warp] = vsel;
    sh.red[warp] = ws;
    sh.red[kDWarps + warp] = wf;
  }
  __syncthreads();
  DSlice out;
  out.ref = M;
  out.sum = dwarp_sum(lane < kDWarps ? sh.red[lane] : 0.f);
  out.fin = dwarp_sum(lane < kDWarps ? sh.red[kDWarps + lane] : 0.f);
  const int vi = __reduce_min_sync(0xffffffffu, lane < kDWarps ? sh.redi[lane] : INT_MAX);
  int idx = INT_MAX;
  if (warp == 0 && lane == 0 && vi < v1) {
    float x[VE];
    dwiden(dld<T, EDGE>(a, vi), x);
#pragma unroll
    for (int e = VE - 1; e >= 0; --e)
      if (x[e] == M && a.inside(vi, e)) idx = a.element(vi, e);
  }
  out.idx = __shfl_sync(0xffffffffu, idx, 0);
  return out;  // valid in warp 0
}

// -------------------------------------------------------------- sampling slice

// Group masses of the slice against the warp reference `ref`: gm[r kDWarps +
// warp] = the mass of vectors v0 + r kDThreads + warp 32 + [0, 32), summed
// kDUnroll rounds at a time, read through the ring (the caller started it).
// Adds the thread's share to tot (and, when FIN, its finiteness sum to fin);
// returns true if a group's mass reached kDGuard (or is not a number).
template <typename T, bool EDGE, bool FIN>
__device__ __forceinline__ bool slice_masses(const DRow<T, EDGE>& a, int v0, int v1, float ref,
                                             uint4* ring, float* gm, float& tot, DFin<T>& fin) {
  static_assert(kDUnroll == 4, "dwarp_sum4 sums four rounds");
  constexpr int VE = DRaw<T>::VE;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rounds = (v1 - v0 + kDThreads - 1) / kDThreads;
  const float nm2 = -ref;
  bool over = false;
  dring_rounds<T, EDGE>(ring, a, v0, v1, [&](int r, const DRaw<T> (&raw)[kDUnroll]) {
    float mv[kDUnroll];
#pragma unroll
    for (int u = 0; u < kDUnroll; ++u) {
      mv[u] = 0.f;
      if (v0 + (r + u) * kDThreads + tid < v1) {  // implies r + u < rounds
        float x[VE];
        dwiden(raw[u], x);
        mv[u] = dmass(x, nm2);
        if (FIN) fin.add(raw[u]);
      }
    }
    tot += (mv[0] + mv[1]) + (mv[2] + mv[3]);  // (a shorter chain of roundings)
    const float g = dwarp_sum4(mv[0], mv[1], mv[2], mv[3], lane);
    over |= !(g < kDGuard);
    const int q = lane >> 3;  // lanes 0, 8, 16, 24 hold rounds r .. r + 3
    if ((lane & 7) == 0 && r + q < rounds) gm[(r + q) * kDWarps + warp] = g;
  });
  return over;
}

template <typename T, bool EDGE>
__device__ __forceinline__ DSlice slice_sample(const DRow<T, EDGE>& a, int v0, int v1, uint4* ring,
                                               float* gm, DShared& sh) {
  constexpr int VE = DRaw<T>::VE;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // the warp reference: the maximum of the warp's first-round vectors (-inf
  // if none)
  dring_start<T, EDGE>(ring, a, v0, v1);
  asm volatile("cp.async.wait_group 1;" ::: "memory");
  float ref;
  {
    float r0 = -INFINITY;
    if (v0 + tid < v1) {
      DRaw<T> raw;
      raw.q = *reinterpret_cast<const decltype(raw.q)*>(ring + tid);
      float x[VE];
      dwiden(raw, x);
      r0 = dvmax(x);
    }
    ref = dref(dwarp_max(r0));
  }
  float tot = 0.f;
  DFin<T> fin;
  const bool over = slice_masses<T, EDGE, true>(a, v0, v1, ref, ring, gm, tot, fin);
  if (__syncthreads_or(over)) {
    // an entry far above its warp's reference: the exact slice maximum, then
    // every group again against it
    float m = -INFINITY;
    const int rounds = (v1 - v0 + kDThreads - 1) / kDThreads;
    for (int r = 0; r < rounds; ++r) {
      const int v = v0 + r * kDThreads + tid;
      if (v < v1) {
        float x[VE];
        dwiden(dld<T, EDGE>(a, v), x);
        m = fmaxf(m, dvmax(x));
      }
    }
    const float w = dwarp_max(m);
    if (lane == 0) sh.red[warp] = w;
    __syncthreads();
    ref = dref(dwarp_max(lane < kDWarps ? sh.red[lane] : -INFINITY));
    tot = 0.f;
    DFin<T> unused;
    dring_start<T, EDGE>(ring, a, v0, v1);
    // (a slice of nothing but masks: no mass)
    slice_masses<T, EDGE, false>(a, v0, v1, -ref < kDWideRef ? ref : INFINITY, ring, gm, tot, unused);
    __syncthreads();  // every warp has read sh.red
  }
  const float wt = dwarp_sum(tot), wf = dwarp_sum(fin.value());
  if (lane == 0) {
    sh.wref[warp] = ref;
    sh.red[warp] = wt;
    sh.red[kDWarps + warp] = wf;
  }
  __syncthreads();  // the group masses and the warp totals are in place
  DSlice out;
  const float rw = lane < kDWarps ? sh.wref[lane] : -INFINITY;
  out.ref = dwarp_max(rw);
  out.sum = dwarp_sum(lane < kDWarps ? drescale<true>(sh.red[lane], rw, out.ref) : 0.f);
  out.fin = dwarp_sum(lane < kDWarps ? sh.red[kDWarps + lane] : 0.f);
  out.idx = 0;
  return out;
}

// A whole row by one warp, masses against the row's maximum M formed as x - M
// first: rows without a logit within 3.7e8 of zero, and draws whose group turned
// out to hold nothing.  best: the greedy draw.
template <typename T, bool EDGE, bool STOCH>
__device__ __forceinline__ void wide_row(const DParams& P, const DRow<T, EDGE>& a, int row,
                                         int best) {
  const int lane = threadIdx.x & 31;
  auto logit = [&](int i) { return to_f32(a.base[a.head + i]); };
  float M = -INFINITY;
  for (int i = lane; i < a.V; i += 32) M = fmaxf(M, logit(i));
  M = dwarp_max(M);
  auto mass = [&](int i) { return ex2((logit(i) - M) * kLog2e); };
  const int seg = (a.V + 31) / 32, i0 = min(a.V, lane * seg), i1 = min(a.V, i0 + seg);
  float s = 0.f;
  for (int i = i0; i < i1; ++i) s += mass(i);
  const float incl = dwarp_incl_scan(s, lane), S = __shfl_sync(0xffffffffu, incl, 31);
  int tok = best;
  float m = 1.f;  // the maximum's
  if (STOCH) {
    const float tau = P.unif[row] * S;
    const unsigned over = __ballot_sync(0xffffffffu, s > 0.f && incl > tau);
    const unsigned pos = __ballot_sync(0xffffffffu, s > 0.f);
    if (lane != (over ? __ffs(over) - 1 : 31 - __clz(pos))) return;
    float cum = incl - s;
    for (int i = i0; i < i1; ++i) {
      const float q = mass(i);
      cum += q;
      if (q > 0.f) {  // the last entry of positive mass, unless one passes the target
        tok = i;
        m = q;
        if (cum > tau) break;
      }
    }
  } else if (lane != 0) {
    return;
  }
  P.tokens[row] = tok;
  P.probs[row] = m / S;
}

// Out of line, but for the greedy draw of bf16 rows (512 rows, V=128256: 24.6 us
// inline, 25.6 called; one fp32 row 2.92 and 2.84), and with the row cut again: a cut
// that the call needs costs 64 sampled rows 0.15 us of 6.9.
template <typename T, bool EDGE, bool STOCH>
__device__ __noinline__ void wide_call(const DParams& P, int row, int best) {
  wide_row<T, EDGE, STOCH>(P, DRow<T, EDGE>(P, row), row, best);
}

// The owner CTA's walk: the group, the vector and the element holding the
// target tau (in units of 2^R) inside the slice; `last` takes the last entry
// of positive mass instead.  Warp 0 only; lane `vc` writes the row's outputs.
// False: a draw at u = 0 fell to a group whose every mass, formed against R, is
// flushed to zero (below 2^-126), though its sum against its warp's reference is not.
template <typename T, bool EDGE>
__device__ __forceinline__ bool slice_walk(const DParams& P, const DRow<T, EDGE>& a, int v0, int v1,
                                           const float* gm, const DShared& sh, float R, float S,
                                           float tau, bool last, int row) {
  constexpr int VE = DRaw<T>::VE;
  const int lane = threadIdx.x & 31;
  const int ng = (v1 - v0 + kDThreads - 1) / kDThreads * kDWarps, gpl = (ng + 31) / 32;
  // lane l owns groups [l gpl, (l + 1) gpl)
  float pl = 0.f;
  for (int h = 0; h < gpl; ++h) {
    const int g = lane * gpl + h;
    if (g < ng) pl += gm[g] * sh.wscale[g & (kDWarps - 1)];
  }
  const float incl = dwarp_incl_scan(pl, lane), excl = incl - pl;
  const unsigned hit = __ballot_sync(0xffffffffu, !last && pl > 0.f && excl <= tau && tau < incl);
  const unsigned posl = __ballot_sync(0xffffffffu, pl > 0.f);
  if (!hit) last = true;
  const int lc = hit ? __ffs(hit) - 1 : (posl ? 31 - __clz(posl) : 0);
  int gsel = -1;
  float trem = 0.f;
  if (lane == lc) {
    float cum = excl;
    int glast = -1;
    for (int h = 0; h < gpl; ++h) {
      const int g = lane * gpl + h;
      if (g >= ng) break;
      const float gv = gm[g] * sh.wscale[g & (kDWarps - 1)];
      if (gv > 0.f) glast = g;
      if (!last && gsel < 0) {
        if (cum + gv > tau) {
          gsel = g;
          trem = tau - cum;
        } else {
          cum += gv;
        }
      }
    }
    if (gsel < 0) {
      gsel = glast;
      last = true;
    }
  }
  gsel = __shfl_sync(0xffffffffu, gsel, lc);
  trem = fmaxf(__shfl_sync(0xffffffffu, trem, lc), 0.f);
  last = __shfl_sync(0xffffffffu, last ? 1 : 0, lc) != 0;
  // the vector: lane l recomputes vector v0 + 32 gsel + l against R
  const float nm2 = -R;
  const int v = v0 + 32 * max(gsel, 0) + lane;
  float x[VE];
  float mv = 0.f;
  if (gsel >= 0 && v < v1) {
    dwiden(dld<T, EDGE>(a, v), x);
    mv = dmass(x, nm2);
  }
  const float vin = dwarp_incl_scan(mv, lane), vex = vin - mv;
  const unsigned vh = __ballot_sync(0xffffffffu, !last && mv > 0.f && vex <= trem && trem < vin);
  const unsigned posv = __ballot_sync(0xffffffffu, mv > 0.f);
  if (!posv) return false;
  if (!vh) last = true;
  const int vc = vh ? __ffs(vh) - 1 : 31 - __clz(posv);
  if (lane != vc) return true;
  // the element
  int tok = -1;
  float pr = NAN;
  if (v < v1) {
    const float te = fmaxf(trem - vex, 0.f);
    float cum = 0.f, qpick = 0.f, qlast = 0.f;
    int pick = -1, lastp = -1;
#pragma unroll
    for (int e = 0; e < VE; ++e) {
      const float q = ex2(fmaf(x[e], kLog2e, nm2));
      if (q > 0.f) {
        lastp = e;
        qlast = q;
      }
      cum += q;
      if (!last && pick < 0 && cum > te) {
        pick = e;
        qpick = q;
      }
    }
    if (pick < 0) {
      pick = lastp;
      qpick = qlast;
    }
    if (pick >= 0) {
      tok = a.element(v, pick);
      pr = qpick / S;
    }
  }
  P.tokens[row] = tok;
  P.probs[row] = pr;
  return true;
}

// ------------------------------------------------------------------- the kernel

// Grid: rows x C CTAs in clusters of C.  Shared memory: the ring, then
// (sampling) one float of group mass per warp and round of a slice.
template <typename T, bool EDGE, bool STOCH>
__global__ void __launch_bounds__(kDThreads) draft_kernel(const __grid_constant__ DParams P) {
  extern __shared__ __align__(16) unsigned char dsmem[];
  uint4* ring = reinterpret_cast<uint4*>(dsmem);
  float* gm = reinterpret_cast<float*>(dsmem + kDRingBytes);
  __shared__ DShared sh;
  cg::cluster_group cluster = cg::this_cluster();
  const int C = static_cast<int>(cluster.num_blocks());
  const int rank = static_cast<int>(cluster.block_rank());
  const int row = static_cast<int>(blockIdx.x) / C;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const DRow<T, EDGE> a(P, row);
  const int v0 = min(rank * P.W, a.nvec), v1 = min(v0 + P.W, a.nvec);

  const DSlice mine = STOCH ? slice_sample<T, EDGE>(a, v0, v1, ring, gm, sh)
                            : slice_greedy<T, EDGE>(a, v0, v1, ring, sh);
  if (warp == 0 && lane < C) *cluster.map_shared_rank(&sh.slot[rank], lane) = mine;
  cluster.sync();  // every CTA's summary is in every CTA; nothing remote after this
  if (warp != 0) return;

  const DSlice s = lane < C ? sh.slot[lane] : DSlice{-INFINITY, 0.f, 0.f, INT_MAX};
  const float R = dwarp_max(s.ref);
  const float mass = lane < C ? drescale<STOCH>(s.sum, s.ref, R) : 0.f;
  const float S = dwarp_sum(mass);
  const float F = dwarp_sum(s.fin);
  if constexpr (!STOCH) {
    const int idx = __reduce_min_sync(0xffffffffu, s.ref == R ? s.idx : INT_MAX);
    if (rank == 0 && lane == 0) {
      const bool ok = dfinite(F) && dfinite(R) && idx != INT_MAX;
      P.tokens[row] = ok ? idx : -1;
      P.probs[row] = ok ? 1.f / S : NAN;  // the maximum's own mass is 2^0
    }
    if (rank == 0 && !(fabsf(R) * kLog2e < kDWideRef) && dfinite(F)) {
      if constexpr (sizeof(T) == 2) wide_row<T, EDGE, STOCH>(P, a, row, idx);
      else wide_call<T, EDGE, STOCH>(P, row, idx);
    }
  } else {
    const float u = P.unif[row];
    if (!(dfinite(F) && u >= 0.f && u < 1.f)) {
      if (rank == 0 && lane == 0) {
        P.tokens[row] = -1;
        P.probs[row] = NAN;
      }
      return;
    }
    // the slice holding the target (the last with positive mass if none does)
    const float tau = u * S;
    const float incl = dwarp_incl_scan(mass, lane), excl = incl - mass;
    const unsigned hit = __ballot_sync(0xffffffffu, mass > 0.f && excl <= tau && tau < incl);
    const unsigned pos = __ballot_sync(0xffffffffu, mass > 0.f);
    const bool wide = !(fabsf(R) < kDWideRef);
    const int owner = wide ? 0 : hit ? __ffs(hit) - 1 : (pos ? 31 - __clz(pos) : 0);
    if (owner != rank) return;
    const float tloc = fmaxf(tau - __shfl_sync(0xffffffffu, excl, owner), 0.f);
    if (lane < kDWarps) sh.wscale[lane] = drescale<true>(1.f, sh.wref[lane], R);
    __syncwarp();
    if (wide || !slice_walk<T, EDGE>(P, a, v0, v1, gm, sh, R, S, tloc, hit == 0u, row))
      wide_call<T, EDGE, true>(P, row, -1);
  }
}

}  // namespace asymspec_impl
