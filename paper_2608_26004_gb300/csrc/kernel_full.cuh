// Streaming row kernel of the steps that record every row (row statistics,
// fused log-probabilities): fuse_verify_row's layout and exchange
// (kernel_row.cuh), with the full program for every row.
//
// Pass 1: LSE(a), LSE(b), LSE(t), LSE(s) and the argmaxes of s and t; pass 2
// (from the L2): the divergence of the gate, the residual masses in
// stochastic mode, the fused log-probabilities.  The staged kernel
// (kernel_tma.cuh) held whole slices, two CTAs an SM: 384 CTAs of B=8, K=5,
// V=151936 bf16 took two waves, 48 us a step; here three CTAs share an SM and
// the loads of the next steps overlap the arithmetic.  What bounds it: at B=24
// nothing alone (40 instructions per entry in greedy mode at 53 % of the issue
// slots, the transcendental unit at 38 %, DRAM active half of the time; the
// log-probabilities are 4 bytes written per entry against 6 read in bf16); a wave
// or less, as B=8, has the latencies of fuse_verify_row.
//
// decide_full, one CTA per row: the row's divergence and record; in
// stochastic mode every row's draw (the row tokens report it); the last row
// of an element runs Algorithm 1's scan (a counter that the row kernel clears).
#pragma once

#include "kernel_row.cuh"

namespace asymspec_impl {

constexpr int kFullMinBlocks = 3;  // CTAs per SM (85 registers a thread)

// A warp's pass-1 record: the references (whole numbers, in log2 units; EDGE: nats) and
// sums of 2^(x log2 e - ref) of a, b, t and s; the largest s and t and the lowest
// vectors that hold them (INT_MAX: none; NaN: non-finite values were seen).
struct __align__(16) WF {
  float ref[4], s[4];
  float vs;
  int is;
  float vt;
  int it;
};
static_assert(sizeof(WF) == 48, "one warp record is three 16-byte words");

__host__ __device__ constexpr int full_shared_bytes(int C) {
  return static_cast<int>(sizeof(RowShared) + C * (kRowThreads / 32) * sizeof(WF));
}

// The largest value of the warp and the lowest vector that holds it; NaN if
// any lane saw a value that is not finite (or larger than FLT_MAX).
__device__ __forceinline__ void warp_best(float& v, int& vec) {
  const bool bad = !(v <= 3.402823466e38f);
  const float m = warp_max(v);
  vec = static_cast<int>(
      __reduce_min_sync(0xffffffffu, static_cast<unsigned>(v == m ? vec : INT_MAX)));
  v = __any_sync(0xffffffffu, bad) ? NAN : m;
}

// Pass 1 over vectors [v0, v1) of the slice, as row_pass1.
template <typename T, bool EDGE>
__device__ __forceinline__ bool full_pass1(uint4* ring, const Streams<T>& g, int v0, int v1,
                                           float beta, const EdgeVals& ed, int vec0, int lastvec,
                                           WF& e) {
  constexpr int NP = RawVec<T>::NP;
  const f2 L2 = pk(kLog2e, kLog2e), beta2 = pk(beta, beta);
  const int i0 = v0 + static_cast<int>(threadIdx.x & 31);
  float ref[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
  cp_async_wait<kRing - 1>();  // step 0 (this lane's own copies)
  if (i0 < v1) {
    RawVec<T> va, vb, vt;
    ring_read<T, true, true>(ring, 0, va, vb, vt);
    const f2 x[4] = {va.pair(0), vb.pair(0), vt.pair(0),
                     fma2(beta2, sub2(va.pair(0), vb.pair(0)), vt.pair(0))};
#pragma unroll
    for (int q = 0; q < 4; ++q) ref[q] = fmaxf(lo_of(x[q]), hi_of(x[q]));
  }
  const float ev[4] = {ed.a, ed.b, ed.t, fmaf(beta, ed.a - ed.b, ed.t)};
  f2 n2[4], acc[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    if (EDGE && ed.own) ref[q] = fmaxf(ref[q], ev[q]);
    ref[q] = ref_of(warp_max(ref[q]));
    n2[q] = pk(-ref[q], -ref[q]);
    acc[q] = 0ull;
  }
  float bs = -INFINITY, bt = -INFINITY;
  float ma = -INFINITY, mb = -INFINITY;  // EDGE: the largest values
  int rs = -1, rt = -1;
  ring_steps<T, true, true>(ring, g, v0, v1, [&](int r, const RawVec<T>& va, const RawVec<T>& vb,
                                                 const RawVec<T>& vt, auto) {
    f2 sc[NP], tc[NP], e[4][NP], xa[NP], xb[NP];
#pragma unroll
    for (int h = 0; h < NP; ++h) {
      const f2 a2 = va.pair(h), b2 = vb.pair(h);
      xa[h] = a2;
      xb[h] = b2;
      tc[h] = vt.pair(h);
      sc[h] = fma2(beta2, sub2(a2, b2), tc[h]);
      e[0][h] = ex2_2(fma2(a2, L2, n2[0]));
      e[1][h] = ex2_2(fma2(b2, L2, n2[1]));
      e[2][h] = ex2_2(fma2(tc[h], L2, n2[2]));
      e[3][h] = ex2_2(fma2(sc[h], L2, n2[3]));
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[q] = add2(acc[q], vsum2(e[q]));
    if (EDGE) {
      ma = max_nan(ma, vmax_nan(xa));
      mb = max_nan(mb, vmax_nan(xb));
    }
    // strictly larger wins, so the lane's earliest vector keeps a tie
    const float cs = vmax_nan(sc), ct = vmax_nan(tc);
    rs = cs > bs ? r : rs;
    bs = max_nan(bs, cs);
    rt = ct > bt ? r : rt;
    bt = max_nan(bt, ct);
  });
  int vs = rs >= 0 ? vec0 + 32 * rs : INT_MAX, vt = rt >= 0 ? vec0 + 32 * rt : INT_MAX;
  if (EDGE && ed.own) {
    // vector 0 precedes every other, the last vector follows them
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[q] = add2(acc[q], pk(ex2(fmaf(ev[q], kLog2e, lo_of(n2[q]))), 0.f));
    if (ed.head && (ev[3] >= bs || bs != bs) && ev[3] > -INFINITY) vs = 0;
    if (ed.tail && ev[3] > bs) vs = lastvec;
    if (ed.head && (ev[2] >= bt || bt != bt) && ev[2] > -INFINITY) vt = 0;
    if (ed.tail && ev[2] > bt) vt = lastvec;
    ma = max_nan(ma, ev[0]);
    mb = max_nan(mb, ev[1]);
    if (ed.head || ed.tail) {
      bs = max_nan(bs, ev[3]);
      bt = max_nan(bt, ev[2]);
    }
  }
  bool ovf = false;
  float s[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    s[q] = hsum2(acc[q]);
    ovf = ovf || !(s[q] < kSumLimit);
  }
  warp_sum4(s[0], s[1], s[2], s[3]);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    e.ref[q] = ref[q];
    e.s[q] = s[q];
  }
  if (EDGE) {
    const float m[4] = {ma, mb, bt, bs};
#pragma unroll
    for (int q = 0; q < 4; ++q) to_largest(e.s[q], e.ref[q], warp_max(m[q]));
  }
  warp_best(bs, vs);
  warp_best(bt, vt);
  e.vs = bs;
  e.is = vs;
  e.vt = bt;
  e.it = vt;
  return ovf;
}

// Fallback of full_pass1's sums, as row_pass1_online.
template <typename T, bool EDGE>
__device__ __noinline__ WF full_pass1_online(Streams<T> g, int v0, int v1, float beta, EdgeVals ed,
                                             WF e) {
  constexpr int NP = RawVec<T>::NP;
  constexpr int VE = 2 * NP;
  float m[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY}, s[4] = {0.f, 0.f, 0.f, 0.f};
  auto take = [&](float a, float b, float t) {
    const float x[4] = {a, b, t, fmaf(beta, a - b, t)};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (x[q] > m[q]) {
        s[q] = s[q] * ex2((m[q] - x[q]) * kLog2e);
        m[q] = x[q];
      }
      s[q] += ex2((x[q] - m[q]) * kLog2e);
    }
  };
  const int lane = static_cast<int>(threadIdx.x & 31);
  for (int i = v0 + lane, q = 0; i < v1; i += 32, ++q) {
    const size_t o = static_cast<size_t>(q) * 32 * VE;
    const RawVec<T> va = raw_ldg(g.a + o), vb = raw_ldg(g.b + o), vt = raw_ldg(g.t + o);
#pragma unroll
    for (int h = 0; h < NP; ++h) {
      take(lo_of(va.pair(h)), lo_of(vb.pair(h)), lo_of(vt.pair(h)));
      take(hi_of(va.pair(h)), hi_of(vb.pair(h)), hi_of(vt.pair(h)));
    }
  }
  if (EDGE && (ed.head || ed.tail)) take(ed.a, ed.b, ed.t);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const float M = warp_max(m[q]);
    const float sc = (s[q] == 0.f || m[q] == M) ? s[q] : s[q] * ex2((m[q] - M) * kLog2e);
    e.ref[q] = EDGE ? M : ref_of(M);
    e.s[q] = warp_sum(sc);
    if (!EDGE) e.s[q] *= ref_residual(M, e.ref[q]);
  }
  return e;
}

// The row's pass-1 result from the cluster's warp records (combine_records,
// four streams and two argmaxes).
template <bool EDGE>
__device__ __forceinline__ void combine_full(const WF* rec, int n, float (&lse)[4], float& vs,
                                             int& is, float& vt, int& it) {
  const int lane = static_cast<int>(threadIdx.x & 31);
  float ref[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY}, sum[4] = {0.f, 0.f, 0.f, 0.f};
  vs = vt = -INFINITY;
  bool bad_s = false, bad_t = false;
  for (int i = lane; i < n; i += 32) {
#pragma unroll
    for (int q = 0; q < 4; ++q) ref[q] = fmaxf(ref[q], rec[i].ref[q]);
    vs = fmaxf(vs, rec[i].vs);
    vt = fmaxf(vt, rec[i].vt);
    bad_s = bad_s || rec[i].vs != rec[i].vs;
    bad_t = bad_t || rec[i].vt != rec[i].vt;
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) ref[q] = warp_max(ref[q]);
  vs = warp_max(vs);
  vt = warp_max(vt);
  is = it = INT_MAX;
  for (int i = lane; i < n; i += 32) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float s = rec[i].s[q], r = rec[i].ref[q];
      sum[q] += (s == 0.f || r == ref[q]) ? s : s * ref_factor<EDGE>(r - ref[q]);
    }
    if (rec[i].vs == vs) is = min(is, rec[i].is);
    if (rec[i].vt == vt) it = min(it, rec[i].it);
  }
  warp_sum4(sum[0], sum[1], sum[2], sum[3]);
#pragma unroll
  for (int q = 0; q < 4; ++q) lse[q] = record_lse<EDGE>(ref[q], sum[q]);
  is = static_cast<int>(__reduce_min_sync(0xffffffffu, static_cast<unsigned>(is)));
  it = static_cast<int>(__reduce_min_sync(0xffffffffu, static_cast<unsigned>(it)));
  if (__any_sync(0xffffffffu, bad_s)) vs = NAN;
  if (__any_sync(0xffffffffu, bad_t)) vt = NAN;
}

// The fused log-probabilities of a vector to out[0 .. 2 NP): with `vec` as
// 16-byte stores, a bf16 vector's two halves exchanged within lane pairs so
// that each store instruction fills whole 32-byte sectors (WHOLE: every lane
// of the warp has a vector).
template <int NP, bool WHOLE>
__device__ __forceinline__ void store_logprobs(float* out, const f2 (&x)[NP], bool vec) {
  if (!vec) {
#pragma unroll
    for (int h = 0; h < NP; ++h) {
      out[2 * h] = lo_of(x[h]);
      out[2 * h + 1] = hi_of(x[h]);
    }
    return;
  }
  auto f4 = [](f2 u, f2 v) { return make_float4(lo_of(u), hi_of(u), lo_of(v), hi_of(v)); };
  if constexpr (NP == 2) {
    __stcs(reinterpret_cast<float4*>(out), f4(x[0], x[1]));
  } else if constexpr (WHOLE) {
    const bool odd = (threadIdx.x & 1) != 0;
    const f2 y0 = __shfl_xor_sync(0xffffffffu, odd ? x[0] : x[2], 1);
    const f2 y1 = __shfl_xor_sync(0xffffffffu, odd ? x[1] : x[3], 1);
    // the even lane's vector, then the odd lane's, half by each lane
    float4* even = reinterpret_cast<float4*>(out - (odd ? 8 : 0)) + (odd ? 1 : 0);
    __stcs(even, odd ? f4(y0, y1) : f4(x[0], x[1]));
    __stcs(even + 2, odd ? f4(x[2], x[3]) : f4(y0, y1));
  } else {
    __stcs(reinterpret_cast<float4*>(out), f4(x[0], x[1]));
    __stcs(reinterpret_cast<float4*>(out) + 1, f4(x[2], x[3]));
  }
}

// Pass 2 over the warp's block: divergence terms (DIV), residual masses
// (RES), the fused log-probabilities to lp (NULL: none; the lane's vector of
// step 0; lpe: its edge element's).
template <typename T, int DIV, bool RES, bool EDGE>
__device__ __forceinline__ void full_pass2(uint4* ring, const Streams<T>& g, int v0, int v1,
                                           const ResConst& k, float beta, float lse_s,
                                           const EdgeVals& ed, float* lp, float* lpe, bool lpvec,
                                           float& jsum, float& msum) {
  constexpr int NP = RawVec<T>::NP;
  const f2 beta2 = pk(beta, beta), nl2 = pk(-lse_s, -lse_s);
  f2 jacc = 0ull, macc = 0ull;
  auto take = [&](f2 a2, f2 b2, f2 t2) {
    f2 amb, p;
    if (RES) {
      f2 qf, rr;
      res_pair(a2, b2, t2, k, amb, p, qf, rr);
      macc = add2(macc, rr);
    } else {
      amb = sub2(a2, b2);
      if (DIV != kDivNone) p = ex2_2(fma2(a2, k.L2, k.nA2));
    }
    if (DIV == kDivJsd) jacc = jsd_pair(amb, p, k, jacc);
    if (DIV == kDivKl) jacc = kl_pair(amb, p, k, jacc);
    return add2(fma2(beta2, amb, t2), nl2);
  };
  ring_steps<T, true, true>(ring, g, v0, v1, [&](int r, const RawVec<T>& va, const RawVec<T>& vb,
                                                 const RawVec<T>& vt, auto whole) {
    f2 l[NP];
#pragma unroll
    for (int h = 0; h < NP; ++h) l[h] = take(va.pair(h), vb.pair(h), vt.pair(h));
    if (lp)
      store_logprobs<NP, decltype(whole)::value>(lp + static_cast<size_t>(r) * 64 * NP, l, lpvec);
  });
  if (EDGE && ed.own) {
    const f2 l = take(pk(ed.a, kEdgeNone), pk(ed.b, kEdgeNone), pk(ed.t, kEdgeNone));
    if (lpe && ed.at >= 0) *lpe = lo_of(l);
  }
  float j = hsum2(jacc), m = hsum2(macc), z0 = 0.f, z1 = 0.f;
  if (DIV == kDivKl) j = -j;
  warp_sum4(j, m, z0, z1);
  jsum = j;
  msum = m;
}

// Grid and shared memory as fuse_verify_row (full_shared_bytes for the
// records).
template <typename T, bool STOCH, bool EDGE>
__global__ void __launch_bounds__(kRowThreads, kFullMinBlocks) fuse_verify_full(const KParams P) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  constexpr int NW = kRowThreads / 32;
  constexpr int VE = 16 / static_cast<int>(sizeof(T));
  extern __shared__ __align__(128) unsigned char smem_row[];
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = static_cast<int>(cluster.block_rank());
  const int tid = static_cast<int>(threadIdx.x);
  const int lane = tid & 31, warp = tid >> 5;
  const int C = P.C;
  unsigned bi, k;
  cluster_row(P, bi, k);
  // the counter of the element's decided rows (decide_full waits for this grid)
  if (k == 0 && rank == 0 && tid == 0) P.tickets[bi] = 0u;
  const unsigned row32 = bi * static_cast<unsigned>(P.K + 1) + k;
  const RowCut<T, EDGE> cut(P, row32);
  const int Wv = P.W / VE, s0 = rank * Wv;  // the slice: vectors [s0, s0 + nv) of the row
  const int nv = max(0, min(Wv, cut.nvec - s0));
  int b0, b1;  // the warp's block of the slice
  row_block<!EDGE>(s0, nv, warp, b0, b1);
  const int v0 = EDGE ? max(b0, cut.in0 - s0) : b0;
  const int v1 = EDGE ? max(v0, min(b1, cut.in1 - s0)) : b1;
  const int i0 = v0 + lane;
  const size_t o0 = static_cast<size_t>(s0 + i0) * VE;  // the lane's first vector
  const Streams<T> g{cut.base(P.a) + o0, cut.base(P.b) + o0, cut.base(P.t) + o0};
  RowShared* sh = reinterpret_cast<RowShared*>(smem_row);
  WF* recv = reinterpret_cast<WF*>(sh + 1);
  uint4* ring = reinterpret_cast<uint4*>(smem_row + P.sh_off) + warp * (kRing * 96);
  const int nrec = C * NW;
  if (tid == 0) {
    mbar_init(&sh->xbar, 1);
    fence_mbar_init();
    mbar_arrive_expect_tx(&sh->xbar, static_cast<unsigned>(nrec * sizeof(WF)));
  }
  cluster_start(P, row32, rank);
  ring_prologue<T, true, true>(ring, g, i0, v1);
  const EdgeVals ed = load_edges<T, EDGE>(P, cut, row32, s0, b0, b1, true);
  cluster_wait();  // every CTA's barrier is initialised before any push

  WF e;
  const bool ovf = full_pass1<T, EDGE>(ring, g, v0, v1, P.beta, ed, s0 + i0, cut.nvec - 1, e);
  if (__any_sync(0xffffffffu, ovf)) e = full_pass1_online<T, EDGE>(g, v0, v1, P.beta, ed, e);
  cp_async_wait<0>();
  // pass 2's first steps do not depend on the normalisers
  const bool jsd = P.divergence == ASYMSPEC_DIV_JSD, kl = P.divergence == ASYMSPEC_DIV_KL;
  const bool second = STOCH || jsd || kl || P.logprobs;
  if (second) ring_prologue<T, true, true>(ring, g, i0, v1);
  if (lane < C) {
    const float4* slot = reinterpret_cast<const float4*>(recv + rank * NW + warp);
    const unsigned to = static_cast<unsigned>(lane);
    st_async16(slot, to, &sh->xbar, make_float4(e.ref[0], e.ref[1], e.ref[2], e.ref[3]));
    st_async16(slot + 1, to, &sh->xbar, make_float4(e.s[0], e.s[1], e.s[2], e.s[3]));
    st_async16(slot + 2, to, &sh->xbar,
               make_float4(e.vs, __int_as_float(e.is), e.vt, __int_as_float(e.it)));
  }
  bool got = true;
  if (warp == 0) {
    got = wait_records(&sh->xbar, rank);
    float lse[4], vs, vt;
    int is, it;
    combine_full<EDGE>(recv, nrec, lse, vs, is, vt, it);
    if (lane == 0) {
#pragma unroll
      for (int q = 0; q < 4; ++q) sh->lse[q] = lse[q];
    }
    if (rank == 0) {
      // the element of each best vector, the lowest of the equal ones
      auto element = [&](int vec, float v, bool fused) {
        bool eq = false;
        const int el = vec == INT_MAX ? -1 : vec * VE + lane - cut.head;
        if (lane < VE && el >= 0 && el < P.V) {
          const size_t o = static_cast<size_t>(row32) * P.V + el;
          float x = elem_ldg(static_cast<const T*>(P.t) + o);
          if (fused)
            x = fmaf(P.beta, elem_ldg(static_cast<const T*>(P.a) + o) -
                                 elem_ldg(static_cast<const T*>(P.b) + o), x);
          eq = x == v;
        }
        const unsigned hit = __ballot_sync(0xffffffffu, eq);
        return hit ? vec * VE + __ffs(hit) - 1 - cut.head : INT_MAX;
      };
      const int es = element(is, vs, true), et = element(it, vt, false);
      const unsigned bad = (vs != vs ? kBadS : 0u) | (vt != vt ? kBadT : 0u);
      // the draft token's logits are read by the decision kernel itself
      if (lane == 0) store_stream_stat(P, row32, lse, es, et, bad, kPathFull);
    }
  }
  __syncthreads();

  const float lse_s = sh->lse[3], S2 = lse_s * kLog2e;
  float jsum = 0.f, msum = 0.f;
  if (second) {
    const float A2 = sh->lse[0] * kLog2e, B2 = sh->lse[1] * kLog2e;
    const ResConst kc = res_const(P.beta, A2, B2, S2);
    float *lp = nullptr, *lpe = nullptr;
    if (P.logprobs) {
      float* row0 = P.logprobs + static_cast<size_t>(row32) * P.V;
      lp = row0 + (static_cast<long long>(s0 + i0) * VE - cut.head);
      lpe = row0 + ed.at;
    }
    const bool lpvec = P.lp_vec != 0;
    if (jsd)
      full_pass2<T, kDivJsd, STOCH, EDGE>(ring, g, v0, v1, kc, P.beta, lse_s, ed, lp, lpe, lpvec,
                                          jsum, msum);
    else if (kl)
      full_pass2<T, kDivKl, STOCH, EDGE>(ring, g, v0, v1, kc, P.beta, lse_s, ed, lp, lpe, lpvec,
                                         jsum, msum);
    else
      full_pass2<T, kDivNone, STOCH, EDGE>(ring, g, v0, v1, kc, P.beta, lse_s, ed, lp, lpe, lpvec,
                                           jsum, msum);
    cp_async_wait<0>();
    if (jsd && !(fabsf(jsum) <= 3.402823466e38f))
      jsum = row_jsd_wide<T, EDGE>(g, v0, v1, A2, B2, ed);
  }
  if (lane == 0) {
    const float qf = STOCH ? block_mass<EDGE>(e.ref[3], e.s[3], S2) : 0.f;
    *reinterpret_cast<float4*>(
        P.pass2_rec + ((static_cast<size_t>(row32) * C + rank) * kRowMaxWarps + warp) * 8) =
        make_float4(jsum, msum, qf, 0.f);
  }
  if (warp == 0 && !got) late_end(P, row32, &sh->xbar);
}

// Grid: (K + 1, B).  One warp decides in greedy mode; in stochastic mode the
// CTA (kDrawThreads threads) draws the row's candidate.
template <typename T, bool STOCH, bool EDGE>
__global__ void __launch_bounds__(STOCH ? kDrawThreads : 32) decide_full(const KParams P) {
  const int k = static_cast<int>(blockIdx.x), bi = static_cast<int>(blockIdx.y);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, K1 = P.K + 1;
  const long long row = static_cast<long long>(bi) * K1 + k;
  const bool bonus = k == P.K;
  RowInputs din{-1, 0.f, 0.f, 0.f, RowScalars{0.f, 0.f, 0.f}};
  if (warp == 0) din = load_row_inputs<T, STOCH>(P, bi, k);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  __shared__ Draw sdraw;
  __shared__ float slse[2];
  RowResult rr;
  rr.sample = -1;
  rr.mass = NAN;
  if (warp == 0) {
    const RowRecords x = load_records(P, row, P.C * (kRowThreads / 32));
    rr.lse_a = x.st.lse[0];
    rr.lse_b = x.st.lse[1];
    rr.lse_t = x.st.lse[2];
    rr.lse_s = x.st.lse[3];
    rr.D = divergence_nats(P, x.j);
    rr.is = x.st.is;
    rr.it = x.st.it;
    rr.bad = x.st.bad | x.st.late;
    rr.have_lse_t = true;
    if (STOCH) {
      const Draw dr = select_group(x.R, x.Q, bonus, din.sc.u_last, rr.mass);
      if (lane == 0) {
        sdraw = dr;
        slse[0] = rr.lse_a;
        slse[1] = rr.lse_s;
      }
    }
  }
  if constexpr (STOCH) {
    __syncthreads();
    rr.sample = block_draw<T, EDGE, !EDGE>(P, row, sdraw, slse[0] * kLog2e, slse[1] * kLog2e);
  }
  if (warp == 0)
    finish_row_warp<STOCH>(P, row, bi, k, rr, din.dtok, din.ad, din.bd, din.td, din.sc);
}

}  // namespace asymspec_impl
