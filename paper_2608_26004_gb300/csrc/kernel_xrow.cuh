// The cross-family step on the drafter's and verifier's own rows: one kernel
// in the place of the gather and the row kernel that read its output.
//
// Materialising the restricted rows a', b', t' (kernel_xvocab.cuh) writes and
// reads back 3 S entries per row and keeps the chip waiting on two gathers
// that are each bound by latency: 182 of 273 us of a step at B=64, K=7,
// S=109568, V_d=151936, V_v=128256 bf16, which takes 187 us here.  One cluster
// of C CTAs takes a row, CTA r the pairs [r W, (r+1) W):
//   * t' in pair order is built in shared memory from the verifier's row and
//     the inverse map, both read in index order (a map_v in any order costs
//     shared-memory bank cycles, no DRAM sectors);
//   * a' and b' are read through map_d from global memory, lane l of a warp
//     taking pairs 2l, 2l + 1 of each 64: with an increasing map_d (the
//     paper's pairing) a load touches a few sectors, and any other map is read
//     correctly.
//   * the passes, the exchange and the paths are fuse_verify_row's, a warp's
//     block of pairs being its inverse-CDF group.
// The decision kernel commits the emitted pair as its verifier token.
//
// What bounds it: latency and the L1, not HBM (B=24, K=7 of those rows: DRAM
// active 26 % of the time, the L1 at 61 % of its peak; 46 % of the shared-memory
// wavefronts are bank conflicts, of the scattered 16-bit stores that build t'; a
// warp waits 4.6 issue slots per instruction on global loads, two of 16 bits per
// pair).  Tried: a and b in token order with wide loads and a word per eight
// tokens that says which are paired (pass 1 10 % slower: more instructions, and
// the unpaired tokens are worked too); C = 1 (215 us: the slice leaves the L1 no
// room to keep the sectors that neighbouring lanes share); 512-thread CTAs, two an
// SM (227 us, the same).
#pragma once

#include "kernel_row.cuh"
#include "kernel_xvocab.cuh"

namespace asymspec_impl {

struct XRowParams {
  const int32_t* map_d;
  const int32_t* map_v;
  const int* inv_v;         // the pair of each verifier token, -1 if none
  const unsigned* map_err;  // the map check's error word
  int32_t* out_index;       // [B] the emitted pair (-1 on a data error)
  int V_d, V_v;
  int t_vec;                // rows of t start on 16-byte boundaries
  int idx2;                 // map_d starts on an 8-byte boundary
};

constexpr int kXRowThreads = 1024;
constexpr int kXRowWarps = kXRowThreads / 32;
constexpr int kXVec = 8;  // pairs per unit of a warp's block, and per thread of a draw

__device__ __forceinline__ void l2_prefetch(const void* p, size_t bytes) {
  const uintptr_t a = (reinterpret_cast<uintptr_t>(p) + 15) & ~static_cast<uintptr_t>(15);
  const uintptr_t e = (reinterpret_cast<uintptr_t>(p) + bytes) & ~static_cast<uintptr_t>(15);
  if (e > a)
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(a),
                 "r"(static_cast<unsigned>(e - a))
                 : "memory");
}

// The slice of a restricted row: pairs [j0, j0 + n), t' in shared memory.
template <typename T>
struct XSlice {
  const T *a, *b;       // the drafter's rows
  const T* t;           // t' of pair j0 (shared memory)
  const int32_t* map_d;
  int j0;
  bool idx2;            // map_d starts on an 8-byte boundary
};

// use(j, a2, b2, t2) for pairs j, j + 1 of the warp's pairs [p0, p1), lane l
// taking pairs 2l, 2l + 1 of each 64, in increasing order; entries past p1
// have no mass (a = b = kEdgeNone, t = -inf, which no argmax takes).  The next
// step's map entries are loaded before this step's logits are used.  (Four
// consecutive pairs a lane: 2 % slower; one, with the next step's logits
// loaded ahead: 15 % slower, twice the sector requests and more instructions.)
template <typename T, bool AB, typename Use>
__device__ __forceinline__ void pair_steps(const XSlice<T>& x, int p0, int p1, Use&& use) {
  const int l2 = 2 * static_cast<int>(threadIdx.x & 31);
  auto index = [&](int base, int2 (&m)[4]) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int j = base + 64 * q + l2;
      m[q] = make_int2(0, 0);
      if (j + 1 < p1 && x.idx2) {
        m[q] = __ldg(reinterpret_cast<const int2*>(x.map_d + j));
      } else if (j < p1) {
        m[q].x = __ldg(x.map_d + j);
        if (j + 1 < p1) m[q].y = __ldg(x.map_d + j + 1);
      }
    }
  };
  auto at = [](const T* row, int i) {  // (32-bit offsets: a row is below 4 GB)
    return elem_ldg(reinterpret_cast<const T*>(
        reinterpret_cast<const char*>(row) +
        static_cast<unsigned>(i) * static_cast<unsigned>(sizeof(T))));
  };
  int2 m[4];
  if (AB) index(p0, m);
  auto step = [&](int base, auto whole) {
    constexpr bool WHOLE = decltype(whole)::value;
    float a[8], b[8];
    if (AB) {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        a[2 * q] = at(x.a, m[q].x);
        a[2 * q + 1] = at(x.a, m[q].y);
        b[2 * q] = at(x.b, m[q].x);
        b[2 * q + 1] = at(x.b, m[q].y);
      }
      if (WHOLE) index(base + 256, m);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int j = base + 64 * q + l2;
      if (WHOLE || j < p1) {
        const bool two = WHOLE || j + 1 < p1;
        const f2 t2 = first_pair(x.t + (j - x.j0));
        use(j, AB ? pk(a[2 * q], two ? a[2 * q + 1] : kEdgeNone) : 0ull,
            AB ? pk(b[2 * q], two ? b[2 * q + 1] : kEdgeNone) : 0ull,
            pk(lo_of(t2), two ? hi_of(t2) : -INFINITY));
      }
    }
  };
  int base = p0;
  for (; base + 256 <= p1; base += 256) step(base, std::true_type{});
  if (base < p1) step(base, std::false_type{});
}

// Pass 1 over the warp's pairs [p0, p1), as row_pass1 (e.vec: the pair that
// holds the best score).
template <typename T, int PROG>
__device__ __forceinline__ bool x_pass1(const XSlice<T>& x, int p0, int p1, float beta, bool chk,
                                        W1& e) {
  constexpr bool DRAFT = prog_draft(PROG), AB = prog_ab(PROG);
  constexpr bool STOCH = PROG == kStochDraft || PROG == kStochBonus;
  constexpr bool SUM3 = PROG == kStochDraft || PROG == kStochBonus || PROG == kGreedyDraft;
  constexpr bool ARG = !STOCH;
  const f2 L2 = pk(kLog2e, kLog2e);
  const f2 beta2 = pk(beta, beta);
  float ra0 = -INFINITY, rb0 = -INFINITY, r30 = -INFINITY;
  const int jf = p0 + static_cast<int>(threadIdx.x & 31);  // any pairs do as references
  if (SUM3 && jf < p1) {
    r30 = to_f32(x.t[jf - x.j0]);
    if (AB) {
      const int d = __ldg(x.map_d + jf);
      ra0 = elem_ldg(x.a + d);
      rb0 = elem_ldg(x.b + d);
      if (STOCH) r30 = fmaf(beta, ra0 - rb0, r30);
    }
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
  float ma = -INFINITY, mb = -INFINITY, m3 = -INFINITY;  // the largest values (to_largest)
  int jbest = INT_MAX;
  pair_steps<T, AB>(x, p0, p1, [&](int j, f2 a2, f2 b2, f2 t2) {
    f2 sc = t2;
    if (AB) {
      const f2 amb = sub2(a2, b2);
      if (DRAFT) {
        acc_a = add2(acc_a, ex2_2(fma2(a2, L2, nA2)));
        acc_b = add2(acc_b, ex2_2(fma2(b2, L2, nB2)));
        fin = fma2(amb, 0ull, fin);  // 0 x (non-finite) is NaN
        ma = max3_nan(ma, lo_of(a2), hi_of(a2));
        mb = max3_nan(mb, lo_of(b2), hi_of(b2));
      }
      sc = fma2(beta2, amb, t2);
    }
    if (SUM3) {
      const f2 x3 = STOCH ? sc : t2;
      acc_3 = add2(acc_3, ex2_2(fma2(x3, L2, n32)));
      m3 = max3_nan(m3, lo_of(x3), hi_of(x3));
    }
    if (ARG) {
      // strictly larger wins, so the lane's earliest pair keeps a tie
      jbest = lo_of(sc) > best ? j : jbest;
      best = max_nan(best, lo_of(sc));
      jbest = hi_of(sc) > best ? j + 1 : jbest;
      best = max_nan(best, hi_of(sc));
    }
  });
  bool ovf = false;
  e.ref[0] = ra0;
  e.ref[1] = rb0;
  e.ref[2] = r30;
  e.s[0] = e.s[1] = e.s[2] = 0.f;
  if (SUM3) {
    float sa = DRAFT ? hsum2(acc_a) : 0.f, sb = DRAFT ? hsum2(acc_b) : 0.f, s3 = hsum2(acc_3);
    ovf = !(s3 < kSumLimit) || (DRAFT && (!(sa < kSumLimit) || !(sb < kSumLimit)));
    if (DRAFT && chk) sa += hsum2(fin);  // 0, or NaN
    float z = 0.f;
    warp_sum4(sa, sb, s3, z);
    e.s[0] = sa;
    e.s[1] = sb;
    e.s[2] = s3;
    if (DRAFT) {
      to_largest(e.s[0], e.ref[0], warp_max(ma));
      to_largest(e.s[1], e.ref[1], warp_max(mb));
    }
    to_largest(e.s[2], e.ref[2], warp_max(m3));
  }
  e.v = 0.f;
  e.vec = 0;
  if (ARG) {
    const bool bad = !(best <= 3.402823466e38f);
    const float m = warp_max(best);
    const unsigned cand = static_cast<unsigned>(best == m ? jbest : INT_MAX);
    e.vec = static_cast<int>(__reduce_min_sync(0xffffffffu, cand));
    e.v = __any_sync(0xffffffffu, bad) ? NAN : m;
  }
  return ovf;
}

// Fallback of x_pass1's sums, as row_pass1_online.
template <typename T, int PROG>
__device__ __noinline__ W1 x_pass1_online(XSlice<T> x, int p0, int p1, float beta, bool chk, W1 e) {
  constexpr bool DRAFT = prog_draft(PROG);
  constexpr bool STOCH = PROG == kStochDraft || PROG == kStochBonus;
  float m[3] = {-INFINITY, -INFINITY, -INFINITY}, s[3] = {0.f, 0.f, 0.f}, fin = 0.f;
  auto add = [&](int q, float v) {
    if (v > m[q]) {
      s[q] = s[q] * ex2((m[q] - v) * kLog2e);
      m[q] = v;
    }
    s[q] += ex2((v - m[q]) * kLog2e);
  };
  for (int j = p0 + static_cast<int>(threadIdx.x & 31); j < p1; j += 32) {
    const int d = __ldg(x.map_d + j);
    const float a = elem_ldg(x.a + d), b = elem_ldg(x.b + d), t = to_f32(x.t[j - x.j0]);
    if (DRAFT) {
      add(0, a);
      add(1, b);
      fin = fmaf(a - b, 0.f, fin);
    }
    add(2, STOCH ? fmaf(beta, a - b, t) : t);
  }
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const float M = warp_max(m[q]);
    float sc = (s[q] == 0.f || m[q] == M) ? s[q] : s[q] * ex2((m[q] - M) * kLog2e);
    if (q == 0 && DRAFT && chk) sc += fin;  // 0, or NaN
    e.ref[q] = M;
    e.s[q] = warp_sum(sc);
  }
  if (!DRAFT) {
    e.ref[0] = e.ref[1] = -INFINITY;
    e.s[0] = e.s[1] = 0.f;
  }
  return e;
}

// Pass 2 over the warp's pairs, as row_pass2.
template <typename T, int DIV, bool RES>
__device__ __forceinline__ void x_pass2(const XSlice<T>& x, int p0, int p1, const ResConst& k,
                                        float& jsum, float& msum) {
  f2 jacc = 0ull, macc = 0ull;
  pair_steps<T, true>(x, p0, p1, [&](int, f2 a2, f2 b2, f2 t2) {
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
  });
  float j = hsum2(jacc), m = hsum2(macc), z0 = 0.f, z1 = 0.f;
  if (DIV == kDivKl) j = -j;
  warp_sum4(j, m, z0, z1);
  jsum = j;
  msum = m;
}

// The warp's JSD sum term by term, as row_jsd_wide.
template <typename T>
__device__ __noinline__ float x_jsd_wide(XSlice<T> x, int p0, int p1, float A2, float B2) {
  float j = 0.f;
  for (int i = p0 + static_cast<int>(threadIdx.x & 31); i < p1; i += 32) {
    const int d = __ldg(x.map_d + i);
    const float a = elem_ldg(x.a + d), b = elem_ldg(x.b + d);
    const float la = fmaf(a, kLog2e, -A2), lb = fmaf(b, kLog2e, -B2);
    const float p = ex2(la), q = ex2(lb);
    const float lm = lg2(p + q) - 1.f;  // log2 of the mean
    if (p > 0.f) j += p * (la - lm);
    if (q > 0.f) j += q * (lb - lm);
    j = fmaf(a - b, 0.f, j);
  }
  return warp_sum(j);
}

// t'_j = t[map_v[j]] for the slice's pairs, by the CTA: the verifier's row and
// the inverse map in index order, U vectors of each in flight per thread.  A
// map that passed the check gives every pair a distinct token, so every entry
// is written.  (The inverse map is read with __ldcg: the map check writes it
// while this kernel, its programmatic dependent, is already resident, and a
// read-only load (__ldg) is defined only for memory that nothing writes during
// the kernel.)
template <typename T>
__device__ __forceinline__ void build_t(const XRowParams& X, const T* src, T* out, int j0, int n) {
  constexpr int VE = 16 / static_cast<int>(sizeof(T));
  constexpr int U = 4, NT = kXRowThreads;
  const int tid = static_cast<int>(threadIdx.x);
  auto put = [&](int j, T v) {
    // (unsigned compare: unpaired tokens, -1, fall outside too)
    if (static_cast<unsigned>(j - j0) < static_cast<unsigned>(n)) out[j - j0] = v;
  };
  if (X.t_vec) {
    const int nvec = X.V_v / VE;  // exact: rows on 16-byte boundaries
    for (int i0 = tid; i0 < nvec; i0 += U * NT) {
      uint4 v[U];
      int4 jv[U][VE / 4];
#pragma unroll
      for (int q = 0; q < U; ++q) {
        const int i = i0 + q * NT;
        if (i < nvec) {
          v[q] = __ldg(reinterpret_cast<const uint4*>(src) + i);
#pragma unroll
          for (int h = 0; h < VE / 4; ++h)
            jv[q][h] = __ldcg(reinterpret_cast<const int4*>(X.inv_v) + i * (VE / 4) + h);
        }
      }
#pragma unroll
      for (int q = 0; q < U; ++q) {
        if (i0 + q * NT < nvec) {
#pragma unroll
          for (int h = 0; h < VE / 4; ++h) {
            put(jv[q][h].x, x_elem<T>(v[q], 4 * h));
            put(jv[q][h].y, x_elem<T>(v[q], 4 * h + 1));
            put(jv[q][h].z, x_elem<T>(v[q], 4 * h + 2));
            put(jv[q][h].w, x_elem<T>(v[q], 4 * h + 3));
          }
        }
      }
    }
  } else {
    for (int u0 = tid; u0 < X.V_v; u0 += 4 * U * NT) {
      T v[4 * U];
      int j[4 * U];
#pragma unroll
      for (int q = 0; q < 4 * U; ++q) {
        j[q] = -1;
        if (u0 + q * NT < X.V_v) {
          v[q] = src[u0 + q * NT];
          j[q] = __ldcg(X.inv_v + u0 + q * NT);
        }
      }
#pragma unroll
      for (int q = 0; q < 4 * U; ++q) put(j[q], v[q]);
    }
  }
}

// Shared memory: RowShared, the cluster's records, then t' of the slice at
// KParams::sh_off.
__host__ __device__ constexpr int xrow_shared_bytes(int C) {
  return static_cast<int>(sizeof(RowShared) + C * kXRowWarps * sizeof(W1));
}

// Grid: C B (K+1) CTAs of kXRowThreads threads in clusters of C, one CTA an SM.
// P.V = S; P.tokens holds pair indices.  Leaves what fuse_verify_row leaves, C
// kXRowWarps records a row.
template <typename T, bool STOCH>
__global__ void __launch_bounds__(kXRowThreads, 1) fuse_verify_xrow(const KParams P,
                                                                    const XRowParams X) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  constexpr int NW = kXRowWarps;
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
  const bool draft = k < P.K;
  const bool only_t = !STOCH && !draft && !P.fuse_bonus;  // Algorithm 1 emits argmax t
  const int j0 = rank * P.W, n = max(0, min(P.W, P.V - j0));
  RowShared* sh = reinterpret_cast<RowShared*>(smem_row);
  T* tsh = reinterpret_cast<T*>(smem_row + P.sh_off);
  const T* trow = static_cast<const T*>(P.t) + static_cast<size_t>(row32) * X.V_v;
  XSlice<T> x;
  x.a = static_cast<const T*>(P.a) + static_cast<size_t>(row32) * X.V_d;
  x.b = static_cast<const T*>(P.b) + static_cast<size_t>(row32) * X.V_d;
  x.t = tsh;
  x.map_d = X.map_d;
  x.j0 = j0;
  x.idx2 = X.idx2 != 0;
  if (tid == 0 && rank == 0 && !only_t) {
    l2_prefetch(x.a, static_cast<size_t>(X.V_d) * sizeof(T));
    l2_prefetch(x.b, static_cast<size_t>(X.V_d) * sizeof(T));
  }
  // a programmatic dependent of the map check
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (__ldcg(X.map_err)) return;  // every element is a data error (decide_xrow)
  const int nrec = C * NW;
  if (tid == 0) {
    mbar_init(&sh->xbar, 1);
    fence_mbar_init();
    mbar_arrive_expect_tx(&sh->xbar, static_cast<unsigned>(nrec * sizeof(W1)));
  }
  cluster_start(P, row32, rank);
  build_t<T>(X, trow, tsh, j0, n);
  __syncthreads();
  cluster_wait();  // every CTA's barrier is initialised before any push

  // ---- pass 1
  const int bw = row_block_vectors((n + kXVec - 1) / kXVec, NW);
  const int p0 = j0 + min(n, warp * bw * kXVec), p1 = j0 + min(n, (warp + 1) * bw * kXVec);
  const bool chk = P.divergence == ASYMSPEC_DIV_JSD || P.divergence == ASYMSPEC_DIV_KL;
  W1 e;
  auto pass1 = [&](auto prog) {
    constexpr int PROG = decltype(prog)::value;
    const bool ovf = x_pass1<T, PROG>(x, p0, p1, P.beta, chk, e);
    if (PROG != kGreedyBonusT && PROG != kGreedyBonusS && __any_sync(0xffffffffu, ovf))
      e = x_pass1_online<T, PROG>(x, p0, p1, P.beta, chk, e);
  };
  if (STOCH) {
    if (draft) pass1(std::integral_constant<int, kStochDraft>{});
    else pass1(std::integral_constant<int, kStochBonus>{});
  } else {
    if (draft) pass1(std::integral_constant<int, kGreedyDraft>{});
    else if (only_t) pass1(std::integral_constant<int, kGreedyBonusT>{});
    else pass1(std::integral_constant<int, kGreedyBonusS>{});
  }
  if (lane < C) {
    const float4* slot = reinterpret_cast<const float4*>(sh->recv() + rank * NW + warp);
    st_async16(slot, static_cast<unsigned>(lane), &sh->xbar,
               make_float4(e.ref[0], e.ref[1], e.ref[2], e.s[0]));
    st_async16(slot + 1, static_cast<unsigned>(lane), &sh->xbar,
               make_float4(e.s[1], e.s[2], e.v, __int_as_float(e.vec)));
  }
  bool got = true;
  if (warp == 0) {
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
        const int md = __ldg(X.map_d + d), mv = __ldg(X.map_v + d);
        da = elem_ldg(x.a + md);
        db = elem_ldg(x.b + md);
        dt = elem_ldg(trow + mv);
      }
    }
    got = wait_records(&sh->xbar, rank);
    float ref[3], sum[3], v;
    int vec;
    combine_records<true>(sh->recv(), nrec, ref, sum, v, vec);
    float lse[4];
    lse[0] = draft ? record_lse<true>(ref[0], sum[0]) : NAN;
    lse[1] = draft ? record_lse<true>(ref[1], sum[1]) : NAN;
    lse[2] = !STOCH && draft ? record_lse<true>(ref[2], sum[2]) : NAN;
    lse[3] = STOCH ? record_lse<true>(ref[2], sum[2]) : NAN;
    const int path = draft && tok_ok ? row_path<STOCH>(P, lse, da, db, dt, u, pd) : kPathAccept;
    if (lane == 0) {
#pragma unroll
      for (int q = 0; q < 4; ++q) sh->lse[q] = lse[q];
      sh->path = path;
    }
    if (rank == 0) {
      const unsigned bad = !STOCH && v != v ? (only_t ? kBadT : kBadS) : 0u;
      if (lane == 0)
        store_stream_stat(P, row32, lse, STOCH || only_t ? INT_MAX : vec,
                          !STOCH && only_t ? vec : INT_MAX, bad, path);
    }
  }
  __syncthreads();

  // ---- pass 2, where the row needs it
  const int path = sh->path;
  const bool second = draft && path != kPathAccept && (STOCH || path == kPathFull);
  const float S2 = sh->lse[3] * kLog2e;
  float jsum = 0.f, msum = 0.f;
  if (second) {
    const float A2 = sh->lse[0] * kLog2e, B2 = sh->lse[1] * kLog2e;
    const ResConst kc = res_const(P.beta, A2, B2, S2);
    const bool jsd = P.divergence == ASYMSPEC_DIV_JSD;
    if (STOCH && path == kPathReject) x_pass2<T, kDivNone, STOCH>(x, p0, p1, kc, jsum, msum);
    else if (jsd) x_pass2<T, kDivJsd, STOCH>(x, p0, p1, kc, jsum, msum);
    else x_pass2<T, kDivKl, STOCH>(x, p0, p1, kc, jsum, msum);
    if (jsd && path == kPathFull && !(fabsf(jsum) <= 3.402823466e38f))
      jsum = x_jsd_wide<T>(x, p0, p1, A2, B2);
  }
  if (lane == 0 && (second || (STOCH && !draft))) {
    const float qf = STOCH ? block_mass<true>(e.ref[2], e.s[2], S2) : 0.f;
    *reinterpret_cast<float4*>(
        P.pass2_rec + (static_cast<size_t>(row32) * nrec + rank * NW + warp) * 8) =
        make_float4(jsum, msum, qf, 0.f);
  }
  if (warp == 0 && !got) late_end(P, row32, &sh->xbar);
}

// The decisions over fuse_verify_xrow's rows; the emitted pair is committed as
// its verifier token.
template <typename T, bool STOCH>
struct PairRows {
  XRowParams X;
  __device__ __forceinline__ int groups(const KParams& P) const { return P.C * kXRowWarps; }
  __device__ __forceinline__ bool refused(const KParams& P, int bi) const {
    const unsigned err = __ldcg(X.map_err);
    if (err && threadIdx.x == 0) {
      emit(P, bi, -1, -1);
      if ((err & kMapOutside) && P.err_word) atomicOr(P.err_word, ASYMSPEC_DATA_NONFINITE);
    }
    return err != 0u;
  }
  __device__ __forceinline__ RowInputs inputs(const KParams& P, int bi, int k) const {
    RowInputs d;
    d.dtok = -1;
    d.ad = d.bd = d.td = 0.f;
    d.sc = STOCH ? load_row_scalars(P, bi, k) : RowScalars{0.f, 0.f, 0.f};
    if (k < P.K) {
      d.dtok = P.tokens[static_cast<size_t>(bi) * P.K + k];
      if (d.dtok >= 0 && d.dtok < P.V) {
        const size_t row = static_cast<size_t>(bi) * (P.K + 1) + k;
        // (an entry outside its vocabulary: the map check refuses the call)
        const int md = __ldg(X.map_d + d.dtok), mv = __ldg(X.map_v + d.dtok);
        if (static_cast<unsigned>(md) < static_cast<unsigned>(X.V_d) &&
            static_cast<unsigned>(mv) < static_cast<unsigned>(X.V_v)) {
          d.ad = elem_ldg(static_cast<const T*>(P.a) + row * X.V_d + md);
          d.bd = elem_ldg(static_cast<const T*>(P.b) + row * X.V_d + md);
          d.td = elem_ldg(static_cast<const T*>(P.t) + row * X.V_v + mv);
        }
      }
    }
    return d;
  }
  __device__ __forceinline__ int draw(const KParams& P, long long row, const Draw& dr, float A2,
                                      float S2) const {
    constexpr int NP = kXVec / 2;
    const int rk = max(dr.g, 0) / kXRowWarps, w = max(dr.g, 0) - rk * kXRowWarps;
    const int j0 = rk * P.W, n = max(0, min(P.W, P.V - j0));
    const int bw = row_block_vectors((n + kXVec - 1) / kXVec, kXRowWarps);
    const int p0 = j0 + min(n, w * bw * kXVec);
    const int p1 = dr.g >= 0 ? j0 + min(n, (w + 1) * bw * kXVec) : 0;
    const T* a = static_cast<const T*>(P.a) + static_cast<size_t>(row) * X.V_d;
    const T* b = static_cast<const T*>(P.b) + static_cast<size_t>(row) * X.V_d;
    const T* t = static_cast<const T*>(P.t) + static_cast<size_t>(row) * X.V_v;
    const ResConst kc = res_const(P.beta, A2, 0.f, S2);
    const int at = p0 + kXVec * static_cast<int>(threadIdx.x);
    int md[kXVec], mv[kXVec];
#pragma unroll
    for (int q = 0; q < kXVec; ++q) {
      const bool in = at + q < p1;
      md[q] = in ? __ldg(X.map_d + at + q) : -1;
      mv[q] = in ? __ldg(X.map_v + at + q) : -1;
    }
    f2 m2[NP];
#pragma unroll
    for (int h = 0; h < NP; ++h) {
      float xa[2], xb[2], xt[2];
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const bool in = md[2 * h + q] >= 0;
        xa[q] = in ? elem_ldg(a + md[2 * h + q]) : kEdgeNone;
        xb[q] = in ? elem_ldg(b + md[2 * h + q]) : kEdgeNone;
        xt[q] = in ? elem_ldg(t + mv[2 * h + q]) : kEdgeNone;
      }
      f2 amb, p, qf, r;
      res_pair(pk(xa[0], xa[1]), pk(xb[0], xb[1]), pk(xt[0], xt[1]), kc, amb, p, qf, r);
      m2[h] = dr.use_r ? r : qf;
    }
    const int pick = block_pick(m2, dr);
    return pick < 0 ? -1 : p0 + pick;
  }
  __device__ __forceinline__ void emit(const KParams& P, int bi, int len, int next) const {
    P.out_len[bi] = len;
    X.out_index[bi] = next;
    P.out_next[bi] = next < 0 ? -1 : __ldg(X.map_v + next);
  }
};

template <typename T, bool STOCH>
__global__ void __launch_bounds__(kDrawThreads) decide_xrow(const KParams P, const XRowParams X) {
  decide_element<STOCH>(P, PairRows<T, STOCH>{X});
}

}  // namespace asymspec_impl
