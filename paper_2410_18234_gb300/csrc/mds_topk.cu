// Top-k restricted verification: Section 5 runs every scheme on rows
// restricted to their k most probable tokens (k = 5 and 10, Tables 2 and 3),
// renormalised.  The restriction leaves a depth's laws on the union U of the
// rows' kept tokens, at most (1 + models) * k of them, so one pass over each
// visited row (the top-k selection) is the only full-vocabulary work and the
// scheme itself runs on U:
//   * single draft: Algorithm 1 with p_I the first valid branch's law;
//   * WIS: the pairwise stages (Remark 4) of the variant truncated LP
//     (appendix "Variant of Truncated LP"), Omega_1 the s largest keys
//     q - a b over the whole vocabulary (ties to the lower id): the positive
//     keys of U, then zero keys (tokens outside U and tokens of U with a zero
//     key) by increasing id, then negative keys;
//   * WIS with the sorted rule on Omega_2 (Section 4 Eq. heur, Eq. p_Ieq):
//     the same stages, a pair inside Omega_2 selecting the token earlier in
//     key order; its Omega_2 law needs each token's key-ordered suffix
//     masses, a sum over U;
//   * SpecTr: sequential rejection over the valid drafts.
// Tokens outside U carry zero mass in every law, so the inverse CDFs in
// token-id order (residual, bonus) run over U sorted by id.
//
// One CTA of 512 threads verifies one sequence.  Per depth: warp 0 plans the
// rows (the target row of the lowest valid branch, one draft row per model
// among the valid branches, read from its lowest valid branch; the single
// draft step reads only the first valid branch's).  For each row, the warps
// first take maxima of a share of the row; the k-th largest of them bounds
// the row's k-th logit from below.  Then every thread scans its share of the
// row and sets the tokens at or above that bound aside in shared memory,
// where counting ranks them.  Warp 0 then computes the kept entries'
// probabilities, the union, the scheme's decision and the walk.
#include "mds_device.cuh"
#include "mds_topk.h"

namespace mds {
namespace topk {
namespace {

using namespace mds::dev;

constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;
constexpr int kKMax = MDS_MAX_TOPK;
constexpr int kRowsMax = 1 + MDS_MAX_K;
constexpr int kEntMax = kRowsMax * kKMax;   // kept entries of one depth, and the largest |U|
constexpr unsigned FULL = 0xffffffffu;
constexpr int kPrefixUnits = 4;             // units per thread behind a row's first logit bound
constexpr int kFlight = 8;                  // 16-byte loads in flight per thread
constexpr int kCand = 1024;                 // tokens at or above the bound one row may set aside

static_assert(kWarps >= kKMax && kWarps <= 32, "kk warps bound a row's kk-th logit");
static_assert(kKMax <= 32, "a row's kept entries fit one warp");

struct Shared {
  unsigned wmax[kWarps];                  // order keys of the warps' largest logits
  __align__(16) unsigned ckey[kCand];     // tokens set aside: order key of the logit ...
  int cid[kCand];                         // ... and id
  int nc, cnt[kWarps];
  int id[kRowsMax][kKMax];                // each row's kept tokens, decreasing (logit, -id)
  float lg[kRowsMax][kKMax];              // their logits
  float pr[kRowsMax][kKMax];              // their renormalised probabilities
  int n[kRowsMax];                        // kept entries per row
  const char* rowp[kRowsMax];             // row pointers of the depth
  float rowc[kRowsMax];                   // log2(e) / T of each row
  int nrows;
  // the union U of the kept tokens by increasing id, each row's law on it
  int uid[kEntMax];
  float law[kRowsMax][kEntMax];
  float cur[kEntMax];                     // running law (stage output law, SpecTr target)
  float key[kEntMax];                     // stage keys q - a b
  float nxt[kEntMax];                     // the sorted rule's Omega_2 law, before it replaces cur
  unsigned char in1[kEntMax];             // U entry is in Omega_1 of the current stage
  short rank[kEntMax];                    // position in U of each kept entry
  unsigned char dup[kEntMax];             // entry repeats a token of an earlier entry
  int nU;
  __align__(16) unsigned kx[32];          // one word per lane, compared by all
  // the walk
  int X[MDS_MAX_K], vbr[MDS_MAX_K], vrow[MDS_MAX_K];
  int nv;
  unsigned valid;
  int done;
  // one stage: Omega_1 by increasing id, its values, the pair state
  int om[MDS_MAX_S];
  unsigned char om_in[MDS_MAX_S];         // the Omega_1 token is in U (index om_u)
  short om_u[MDS_MAX_S];
  float om_q[MDS_MAX_S], om_a[MDS_MAX_S], om_b[MDS_MAX_S], om_x[MDS_MAX_S];
  float RS[kMaxPairs], FL[kMaxPairs], FH[kMaxPairs];
  int Y;
  int bcast;                              // warp 0's broadcast word
  // bonus: the target row's kept entries by increasing id
  int bid[kKMax];
  float bw[kKMax];
};

// One row of the depth: units of 16 bytes from its start, whole and aligned
// (vec) or shifted together from aligned blocks.
template <int DT>
struct Row {
  const char* row;
  int V, nu;
  bool vec;
  __device__ __forceinline__ uint4 unit(int u) const {
    if (vec) return __ldcs(reinterpret_cast<const uint4*>(row) + u);
    return load_unit<DT>(row, row, row + (size_t)V * (16 / Elt<DT>::VE), u, V);
  }
};

// Every unit of the row, kFlight per thread in flight: fn(x, u).
template <int DT, class FN>
__device__ __forceinline__ void scan_row(const Row<DT>& w, int first, FN&& fn) {
  for (int u0 = first + (int)threadIdx.x; u0 < w.nu; u0 += kFlight * kThreads) {
    uint4 x[kFlight];
#pragma unroll
    for (int q = 0; q < kFlight; ++q)
      x[q] = u0 + q * kThreads < w.nu ? w.unit(u0 + q * kThreads) : Elt<DT>::neg_inf();
#pragma unroll
    for (int q = 0; q < kFlight; ++q) fn(x[q], u0 + q * kThreads);
  }
}

// The kk-th largest of the warps' maxima in S.wmax (0: fewer than kk warps
// saw a logit above -inf): kk distinct logits reach it.
__device__ __forceinline__ unsigned kth_warp_max(const Shared& S, int kk) {
  const int lane = threadIdx.x & 31;
  const unsigned k = lane < kWarps ? S.wmax[lane] : 0u;
  int above = 0;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) {
    const unsigned o = S.wmax[w];
    above += (o > k || (o == k && w < lane)) ? 1 : 0;
  }
  const unsigned who = __ballot_sync(FULL, lane < kWarps && above == kk - 1);
  return __shfl_sync(FULL, k, __ffs(who) - 1);
}
__device__ __forceinline__ void put_warp_max(Shared& S, float mx) {
  const unsigned k = __reduce_max_sync(FULL, mx > kNegInf ? ord_key(__fadd_rn(mx, 0.f)) : 0u);
  if ((threadIdx.x & 31) == 0) S.wmax[threadIdx.x >> 5] = k;
}

// Set aside unit u's logits whose order key is at least `lo`.
template <int DT>
__device__ __forceinline__ void offer(Shared& S, const uint4& x, int u, int V, unsigned lo, float lof) {
  using E = Elt<DT>;
  if (!(E::unit_max(x) >= lof)) return;
  float v[E::VE];
  E::unpack(x, v);
#pragma unroll
  for (int e = 0; e < E::VE; ++e) {
    const int id = u * E::VE + e;
    const unsigned k = ord_key(__fadd_rn(v[e], 0.f));
    if (v[e] == v[e] && k >= lo && id < V) {
      const int pos = atomicAdd(&S.nc, 1);
      if (pos < kCand) {
        S.ckey[pos] = k;
        S.cid[pos] = id;
      }
    }
  }
}

// The `need` lowest ids whose order key is exactly `key`, set aside too (in id
// order; all threads).
template <int DT>
__device__ void offer_equal(Shared& S, const Row<DT>& w, unsigned key, int need) {
  using E = Elt<DT>;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int u0 = 0; u0 < w.nu && need > 0; u0 += kThreads) {
    const int u = u0 + (int)threadIdx.x;
    float v[E::VE];
    E::unpack(u < w.nu ? w.unit(u) : E::neg_inf(), v);
    unsigned bits = 0u;
#pragma unroll
    for (int e = 0; e < E::VE; ++e)
      bits |= (u * E::VE + e < w.V && v[e] == v[e] && ord_key(__fadd_rn(v[e], 0.f)) == key) ? 1u << e : 0u;
    int incl = __popc(bits);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(FULL, incl, o);
      if (lane >= o) incl += t;
    }
    __syncthreads();   // the previous round's counts are read
    if (lane == 31) S.cnt[warp] = incl;
    __syncthreads();
    int before = incl - __popc(bits), total = 0;
    for (int q = 0; q < kWarps; ++q) {
      before += q < warp ? S.cnt[q] : 0;
      total += S.cnt[q];
    }
    for (; bits && before < need; bits &= bits - 1u, ++before) {
      const int pos = atomicAdd(&S.nc, 1);
      S.ckey[pos] = key;
      S.cid[pos] = u * E::VE + __ffs(bits) - 1;
    }
    need -= total;
  }
  __syncthreads();
}

// The row's top kk into S.id / S.lg / S.n[r] (all threads; ends synchronised):
// larger logit first, ties to the lower id.  A bound that kk distinct logits
// reach (the kk-th largest of the warps' maxima over the row's first units)
// lets the scan set aside some tens to a few hundred tokens, which are ranked
// by counting.  More than kCand of them, or no bound (few finite logits, ties,
// flat rows): the tokens above the bound from the whole row's maxima, and of
// those at it the lowest ids; should even those above be too many, the exact
// kk-th key by bisection.
// Bound by the row's stream: eight 16-byte loads in flight per thread, 512
// threads.  Against per-thread lists of 16 keys in registers with four loads
// in flight of 256 threads: B = 256, K = 8, V = 128256 WIS top-10 523 -> 428 us
// a call, smaller batches 1.6 to 2.6 times as fast.
template <int DT>
__device__ __noinline__ void select_row(const Params& p, Shared& S, int r, int kk) {
  using E = Elt<DT>;
  const int tid = threadIdx.x;
  const Row<DT> w{S.rowp[r], p.V, (p.V + E::VE - 1) / E::VE, p.vec != 0};
  if (tid == 0) S.nc = 0;
  {
    uint4 x[kPrefixUnits];
    float mx = kNegInf;
#pragma unroll
    for (int q = 0; q < kPrefixUnits; ++q) {
      x[q] = tid + q * kThreads < w.nu ? w.unit(tid + q * kThreads) : E::neg_inf();
      mx = fmaxf(mx, E::unit_max(x[q]));
    }
    put_warp_max(S, mx);
    __syncthreads();
    const unsigned lo = kth_warp_max(S, kk);
    if (lo) {
      const float lof = ord_val(lo);
#pragma unroll
      for (int q = 0; q < kPrefixUnits; ++q) offer<DT>(S, x[q], tid + q * kThreads, w.V, lo, lof);
      scan_row(w, kPrefixUnits * kThreads, [&](const uint4& y, int u) { offer<DT>(S, y, u, w.V, lo, lof); });
    }
    __syncthreads();
    if (!lo || S.nc > kCand) {
      // the whole row's maxima
      __syncthreads();
      if (tid == 0) S.nc = 0;
      mx = kNegInf;
      scan_row(w, 0, [&](const uint4& y, int) { mx = fmaxf(mx, E::unit_max(y)); });
      put_warp_max(S, mx);
      __syncthreads();
      constexpr unsigned kInf = 0x007fffffu;   // order key of -inf
      unsigned at = kth_warp_max(S, kk);
      if (!at) at = kInf;
      scan_row(w, 0, [&](const uint4& y, int u) { offer<DT>(S, y, u, w.V, at + 1u, ord_val(at)); });
      __syncthreads();
      if (S.nc > kCand) {
        // the largest key that kk logits reach, bit by bit
        unsigned t = 0u;
        for (int bit = 31; bit >= 0; --bit) {
          const unsigned cand = t | (1u << bit);
          unsigned c = 0u;
          scan_row(w, 0, [&](const uint4& y, int u) {
            float v[E::VE];
            E::unpack(y, v);
#pragma unroll
            for (int e = 0; e < E::VE; ++e)
              c += (u * E::VE + e < w.V && v[e] == v[e] && ord_key(__fadd_rn(v[e], 0.f)) >= cand) ? 1u : 0u;
          });
          c = __reduce_add_sync(FULL, c);
          __syncthreads();
          if ((tid & 31) == 0) S.cnt[tid >> 5] = (int)c;
          __syncthreads();
          int n = 0;
          for (int q = 0; q < kWarps; ++q) n += S.cnt[q];
          if (n >= kk) t = cand;
        }
        at = t;
        __syncthreads();
        if (tid == 0) S.nc = 0;
        __syncthreads();
        scan_row(w, 0, [&](const uint4& y, int u) { offer<DT>(S, y, u, w.V, at + 1u, ord_val(at)); });
        __syncthreads();
      }
      const int have = S.nc;
      if (have < kk) offer_equal(S, w, at, kk - have);
    }
  }
  // ranks by (key, id)
  const int n = S.nc;
  for (int i = n + tid; i < ((n + 3) & ~3); i += kThreads) S.ckey[i] = 0u;
  __syncthreads();
  for (int i = tid; i < n; i += kThreads) {
    const unsigned k = S.ckey[i];
    int rk = 0, eq = 0;
    for (int q = 0; q < n; q += 4) {
      const uint4 o = *reinterpret_cast<const uint4*>(S.ckey + q);
      rk += (o.x > k ? 1 : 0) + (o.y > k ? 1 : 0) + (o.z > k ? 1 : 0) + (o.w > k ? 1 : 0);
      eq += (o.x == k ? 1 : 0) + (o.y == k ? 1 : 0) + (o.z == k ? 1 : 0) + (o.w == k ? 1 : 0);
    }
    const int id = S.cid[i];
    if (eq > 1 && rk < kk)
      for (int q = 0; q < n; ++q) rk += (S.ckey[q] == k && S.cid[q] < id) ? 1 : 0;
    if (rk < kk) {
      S.id[r][rk] = id;
      S.lg[r][rk] = ord_val(k);
    }
  }
  if (tid == 0) S.n[r] = min(n, kk);
  __syncthreads();
}

// Warp 0: the depth's rows and valid branches (the tree walk's bookkeeping).
__device__ void plan(const Params& p, Shared& S, int b, int j, bool bonus) {
  const int lane = threadIdx.x & 31;
  const int K = p.K;
  const unsigned valid = S.valid;
  const bool v = lane < K && ((valid >> lane) & 1u);
  const int m = v ? (int)p.model_of[lane] : 64 + lane;
  const unsigned same = __match_any_sync(FULL, m);
  const bool first = v && (__ffs(same) - 1) == lane;   // lowest valid branch of its model
  const unsigned fm = __ballot_sync(FULL, first);
  const unsigned vm = __ballot_sync(FULL, v);
  const int myrow = first ? 1 + __popc(fm & ((1u << lane) - 1u)) : 0;
  const int row = __shfl_sync(FULL, myrow, __ffs(same) - 1);
  if (!bonus && v) {
    const int i = __popc(vm & ((1u << lane) - 1u));
    int x = p.tokens[((size_t)b * K + lane) * p.L + j];
    if (x < 0 || x >= p.V) {
      atomicOr(p.status, MDS_ST_BADTOKEN);
      x = 0;
    }
    S.X[i] = x;
    S.vbr[i] = lane;
    S.vrow[i] = row;
  }
  if (!bonus && first) {
    S.rowp[myrow] = p.drafts[lane] + (((size_t)b * p.L + j) * (size_t)p.V) * p.esize;
    float td = p.temps[(size_t)b * (1 + K) + 1 + lane];
    if (!(td > 0.f) || !(td < kPosInf)) {
      atomicOr(p.status, MDS_ST_BADTEMP);
      td = 1.f;
    }
    S.rowc[myrow] = __fdiv_rn(kLog2e, td);
  }
  if (lane == 0) {
    const int kstar = __ffs(valid) - 1;
    S.rowp[0] = p.target + ((((size_t)b * K + kstar) * (p.L + 1) + j) * (size_t)p.V) * p.esize;
    float tq = p.temps[(size_t)b * (1 + K)];
    if (!(tq > 0.f) || !(tq < kPosInf)) {
      atomicOr(p.status, MDS_ST_BADTEMP);
      tq = 1.f;
    }
    S.rowc[0] = __fdiv_rn(kLog2e, tq);
    // the single-draft step reads only the first valid branch's model row (row 1)
    S.nrows = bonus ? 1 : (p.scheme == MDS_SINGLE ? 2 : 1 + __popc(fm));
    S.nv = bonus ? 0 : __popc(vm);
  }
}

// Warp 0: the kept entries' probabilities, exp2((l - M) log2(e) / T) over
// their sum (M the row's largest kept logit).
__device__ void row_probs(const Params& p, Shared& S, int r) {
  const int lane = threadIdx.x & 31;
  const int n = S.n[r];
  const float M = S.lg[r][0], c = S.rowc[r];
  const float t = (lane < n) ? exp_term(S.lg[r][lane], M, c) : 0.f;
  const float Z = warp_sum(t);
  float pr;
  if (!(Z > 0.f) || !(Z < kPosInf)) {
    // no finite kept logit: the row's first kept token takes the mass
    if (lane == 0) atomicOr(p.status, MDS_ST_NONFINITE);
    pr = (lane == 0) ? 1.f : 0.f;
  } else {
    pr = __fmul_rn(t, __frcp_rn(Z));
  }
  if (lane < n) S.pr[r][lane] = pr;
  __syncwarp();
}

// Warp 0: U (the kept tokens of every row, by increasing id) and each row's
// law on it.
__device__ void build_union(Shared& S) {
  const int lane = threadIdx.x & 31;
  const int nr = S.nrows, ne = nr * kKMax;
  if (ne <= 32) {
    // two rows: one kept entry per lane, duplicates by a match, ranks by counting
    const int r = lane / kKMax, t = lane - r * kKMax;
    const bool have = r < nr && t < S.n[r < nr ? r : 0];
    const int id = have ? S.id[r][t] : 0x7fffffff;
    const unsigned same = __match_any_sync(FULL, id);
    const bool first = have && (same & ((1u << lane) - 1u)) == 0u;
    S.kx[lane] = first ? (unsigned)id : 0x7fffffffu;
    __syncwarp();
    int k = 0;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const uint4 o = reinterpret_cast<const uint4*>(S.kx)[c];
      k += (o.x < (unsigned)id ? 1 : 0) + (o.y < (unsigned)id ? 1 : 0) + (o.z < (unsigned)id ? 1 : 0) +
           (o.w < (unsigned)id ? 1 : 0);
    }
    const int nU = __popc(__ballot_sync(FULL, first));
    if (first) S.uid[k] = id;
    for (int q = 0; q < nr; ++q)
      if (lane < nU) S.law[q][lane] = 0.f;
    if (lane == 0) S.nU = nU;
    __syncwarp();
    if (have) S.law[r][k] = S.pr[r][t];
    __syncwarp();
    return;
  }
  for (int e = lane; e < ne; e += 32) {
    const int r = e / kKMax, t = e - r * kKMax;
    unsigned char d = 1;
    if (t < S.n[r]) {
      const int id = S.id[r][t];
      d = 0;
      for (int f = 0; f < e && !d; ++f) {
        const int rf = f / kKMax, tf = f - rf * kKMax;
        d = (tf < S.n[rf] && S.id[rf][tf] == id) ? 1 : 0;
      }
    }
    S.dup[e] = d;
  }
  __syncwarp();
  int cnt = 0;
  for (int e = lane; e < ne; e += 32) {
    const int r = e / kKMax, t = e - r * kKMax;
    if (t >= S.n[r]) continue;
    const int id = S.id[r][t];
    int k = 0;
    for (int f = 0; f < ne; ++f) {
      const int rf = f / kKMax, tf = f - rf * kKMax;
      k += (!S.dup[f] && tf < S.n[rf] && S.id[rf][tf] < id) ? 1 : 0;
    }
    S.rank[e] = (short)k;
    if (!S.dup[e]) {
      S.uid[k] = id;
      ++cnt;
    }
  }
  const int nU = __reduce_add_sync(FULL, cnt);
  for (int i = lane; i < nr * kEntMax; i += 32) {
    const int r = i / kEntMax, u = i - r * kEntMax;
    if (u < nU) S.law[r][u] = 0.f;
  }
  if (lane == 0) S.nU = nU;
  __syncwarp();
  for (int e = lane; e < ne; e += 32) {
    const int r = e / kKMax, t = e - r * kKMax;
    if (t < S.n[r]) S.law[r][S.rank[e]] = S.pr[r][t];
  }
  __syncwarp();
}

// Position of token x in U, or -1.
__device__ __forceinline__ int find_u(const Shared& S, int x) {
  int lo = 0, hi = S.nU;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (S.uid[mid] < x)
      lo = mid + 1;
    else
      hi = mid;
  }
  return (lo < S.nU && S.uid[lo] == x) ? lo : -1;
}
__device__ __forceinline__ float law_at(const Shared& S, const float* w, int x) {
  const int i = find_u(S, x);
  return i >= 0 ? w[i] : 0.f;
}

__device__ __forceinline__ bool better(float ka, int ia, float kb, int ib) {
  return ka > kb || (ka == kb && ia < ib);
}

// Warp 0: inverse CDF over n weights in U order (increasing token id): the
// first index whose running sum exceeds u * total, the last positive weight
// if rounding leaves none, -1 if the total is not positive.  Both passes sum
// in the same order, so the last running sum is the total.
template <class W>
__device__ int warp_cdf(int n, W w, float u01, float* total) {
  const int lane = threadIdx.x & 31;
  float carry = 0.f;
  for (int base = 0; base < n; base += 32) {
    float c = (base + lane < n) ? w(base + lane) : 0.f;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const float t = __shfl_up_sync(FULL, c, o);
      if (lane >= o) c = __fadd_rn(c, t);
    }
    carry = __fadd_rn(carry, __shfl_sync(FULL, c, 31));
  }
  *total = carry;
  if (!(carry > 0.f)) return -1;
  const float thr = __fmul_rn(u01, carry);
  carry = 0.f;
  int last = -1;
  for (int base = 0; base < n; base += 32) {
    const float x = (base + lane < n) ? w(base + lane) : 0.f;
    float c = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const float t = __shfl_up_sync(FULL, c, o);
      if (lane >= o) c = __fadd_rn(c, t);
    }
    const unsigned who = __ballot_sync(FULL, __fadd_rn(carry, c) > thr);
    if (who) return base + __ffs(who) - 1;
    const unsigned pos = __ballot_sync(FULL, x > 0.f);
    if (pos) last = base + 31 - __clz(pos);
    carry = __fadd_rn(carry, __shfl_sync(FULL, c, 31));
  }
  return last;
}

// Warp 0: the next Omega_1 entry among U's keys of one sign (sign > 0: key > 0,
// else key < 0) that comes after (lk, lid) in key order.  Returns its index in
// U or -1; *bk / *bid its key and id.
__device__ int next_key(const Shared& S, int sign, float lk, int lid, float* bk_out, int* bid_out) {
  float bk = kNegInf;
  int bid = 0x7fffffff, bi = -1;
  for (int i = threadIdx.x & 31; i < S.nU; i += 32) {
    const float k = S.key[i];
    if (sign > 0 ? !(k > 0.f) : !(k < 0.f)) continue;
    const int id = S.uid[i];
    if (!better(lk, lid, k, id)) continue;
    if (bi < 0 || better(k, id, bk, bid)) {
      bk = k;
      bid = id;
      bi = i;
    }
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    const float ok = __shfl_xor_sync(FULL, bk, o);
    const int oid = __shfl_xor_sync(FULL, bid, o);
    const int oi = __shfl_xor_sync(FULL, bi, o);
    if (oi >= 0 && (bi < 0 || better(ok, oid, bk, bid))) {
      bk = ok;
      bid = oid;
      bi = oi;
    }
  }
  *bk_out = bk;
  *bid_out = bid;
  return bi;
}

// Warp 0: one pairwise stage of the weighted scheme with input laws
// a = S.cur (the running law) and b = S.law[rb] against q = S.law[0]; ordered
// inputs (A, Btok) and selection uniform u.  Returns the stage's token and
// leaves its output law in S.cur.  With `sorted`, Omega_2 follows the sorted
// rule of the truncated LP (Section 4 Eq. heur and Eq. p_Ieq, the non-iid
// appendix): a pair inside Omega_2 selects the token earlier in key order, so
// p_I(k) = a_k b_k + b_k A_after(k) + a_k B_after(k) with the Omega_2 masses
// of the tokens after k; otherwise the variant's 1/2 rule.
__device__ int wis_stage(const Params& p, Shared& S, int A, int Btok, int rb, float u, bool sorted) {
  const int lane = threadIdx.x & 31;
  const int nU = S.nU;
  const float* q = S.law[0];
  const float* bl = S.law[rb];
  for (int i = lane; i < nU; i += 32) S.key[i] = __fadd_rn(__fmaf_rn(-S.cur[i], bl[i], q[i]), 0.f);
  __syncwarp();
  const int s = min(p.wis_s, p.V);
  // Omega_1 in key order: positive keys, zero keys by id, negative keys
  int taken = 0;
  for (int sign = 1; sign >= -1; sign -= 2) {
    if (sign < 0 && taken < s) {
      // zero keys by increasing id: tokens outside U and tokens of U whose key is 0
      if (lane == 0) {
        int c = 0, ptr = 0, t = taken;
        while (t < s && c < p.V) {
          while (ptr < nU && S.uid[ptr] < c) ++ptr;
          const bool inU = ptr < nU && S.uid[ptr] == c;
          if (!inU || S.key[ptr] == 0.f) {
            S.om[t] = c;
            S.om_in[t] = inU ? 1 : 0;
            S.om_u[t] = (short)(inU ? ptr : -1);
            ++t;
          }
          ++c;
        }
        S.bcast = t;
      }
      __syncwarp();
      taken = S.bcast;
      __syncwarp();
    }
    float lk = kPosInf;
    int lid = -1;
    while (taken < s) {
      float bk;
      int bid;
      const int bi = next_key(S, sign, lk, lid, &bk, &bid);
      if (bi < 0) break;
      if (lane == 0) {
        S.om[taken] = bid;
        S.om_in[taken] = 1;
        S.om_u[taken] = (short)bi;
      }
      lk = bk;
      lid = bid;
      ++taken;
    }
    __syncwarp();
  }
  if (lane == 0) {
    // Omega_1 by increasing id, with q, a, b at its tokens
    for (int x = 1; x < s; ++x)
      for (int y = x; y > 0 && S.om[y] < S.om[y - 1]; --y) {
        const int ti = S.om[y];
        S.om[y] = S.om[y - 1];
        S.om[y - 1] = ti;
        const unsigned char tc = S.om_in[y];
        S.om_in[y] = S.om_in[y - 1];
        S.om_in[y - 1] = tc;
        const short ts = S.om_u[y];
        S.om_u[y] = S.om_u[y - 1];
        S.om_u[y - 1] = ts;
      }
    for (int t = 0; t < MDS_MAX_S; ++t) {
      const bool in = t < s && S.om_in[t];
      const int i = in ? S.om_u[t] : 0;
      if (t >= s) S.om[t] = 0x7fffffff;
      S.om_q[t] = in ? q[i] : 0.f;
      S.om_a[t] = in ? S.cur[i] : 0.f;
      S.om_b[t] = in ? bl[i] : 0.f;
    }
  }
  __syncwarp();
  // Omega_2 masses of the two input laws
  float sa = 0.f, sb = 0.f;
  for (int i = lane; i < nU; i += 32) {
    bool in1 = false;
    for (int t = 0; t < s; ++t) in1 |= (S.om_in[t] && S.om_u[t] == i);
    S.in1[i] = in1 ? 1 : 0;
    if (!in1) {
      sa = __fadd_rn(sa, S.cur[i]);
      sb = __fadd_rn(sb, bl[i]);
    }
  }
  const float A2 = warp_sum(sa), B2 = warp_sum(sb);
  __syncwarp();
  if (sorted) {
    // Omega_2 values of the sorted rule (tokens outside U carry no mass)
    for (int i = lane; i < nU; i += 32) {
      if (S.in1[i]) continue;
      const float ki = S.key[i];
      const int idi = S.uid[i];
      float aa = 0.f, ba = 0.f;
      for (int j = 0; j < nU; ++j)
        if (!S.in1[j] && better(ki, idi, S.key[j], S.uid[j])) {
          aa = __fadd_rn(aa, S.cur[j]);
          ba = __fadd_rn(ba, bl[j]);
        }
      const float ai = S.cur[i], bi = bl[i];
      S.nxt[i] = __fadd_rn(__fadd_rn(__fmul_rn(ai, bi), __fmul_rn(bi, aa)), __fmul_rn(ai, ba));
    }
    __syncwarp();
  }
  int y = 0;
  if (s <= 5) {
    float x;
    bool capped;
    y = stage_solve5(A2, B2, A, Btok, u, S.om, S.om_q, S.om_a, S.om_b, x, &capped);
    if (capped && lane == 0) atomicOr(p.status, MDS_ST_LP_CAP);
    if (lane < 5) S.om_x[lane] = x;
  }
  if (lane == 0) {
    if (s > 5) {
      bool capped = false;
      y = stage_solve<MDS_MAX_S>(s, A2, B2, A, Btok, u, S.om, S.om_q, S.om_a, S.om_b, S.om_x, &capped, S.RS, S.FL,
                                 S.FH);
      if (capped) atomicOr(p.status, MDS_ST_LP_CAP);
    }
    if (sorted && A != Btok) {
      // both inputs in Omega_2: the one earlier in key order (a token outside U has key 0)
      bool ia = false, ib = false;
      for (int t = 0; t < s; ++t) {
        ia |= (S.om[t] == A);
        ib |= (S.om[t] == Btok);
      }
      if (!ia && !ib) {
        const int ua = find_u(S, A), ub = find_u(S, Btok);
        const float ka = ua >= 0 ? S.key[ua] : 0.f, kb = ub >= 0 ? S.key[ub] : 0.f;
        y = better(ka, A, kb, Btok) ? A : Btok;
      }
    }
    S.Y = y;
  }
  __syncwarp();
  // the stage's output law: p_I on Omega_1 from the LP; on Omega_2 the sorted
  // rule's values or (a B2 + b A2) / 2
  for (int i = lane; i < nU; i += 32) {
    int pos = -1;
    for (int t = 0; t < s; ++t)
      if (S.om_in[t] && S.om_u[t] == i) pos = t;
    S.cur[i] = (pos >= 0) ? S.om_x[pos]
               : sorted   ? S.nxt[i]
                          : __fmul_rn(0.5f, __fadd_rn(__fmul_rn(S.cur[i], B2), __fmul_rn(bl[i], A2)));
  }
  y = S.Y;
  __syncwarp();
  return y;
}

// Warp 0: the pairwise stages of the weighted scheme with the 1/2 rule, one
// entry of U per lane (nU <= 32, s <= 5), the state in registers; *Yo the
// stages' token so far.  Returns the first stage with fewer than s positive
// keys (Omega_1 then takes zero keys, tokens outside U among them), nv if
// none; the law so far is in S.cur.  Same arithmetic as wis_stage (B = 256,
// K = 8, V = 128256 top-10 428 us a call with it alone, 321 with this).
__device__ int wis_stages_small(const Params& p, Shared& S, float ul, int* Yo) {
  const int lane = threadIdx.x & 31;
  const int nU = S.nU, nv = S.nv, s = min(p.wis_s, p.V);
  const bool have = lane < nU;
  const int id = have ? S.uid[lane] : -1;
  const float q = have ? S.law[0][lane] : 0.f;
  float a = have ? S.law[S.vrow[0]][lane] : 0.f;
  int A = S.X[0], m = 1;
#pragma unroll 1
  for (; m < nv; ++m) {
    const int Btok = S.X[m];
    const float u = __shfl_sync(FULL, ul, m - 1);
    const float bq = have ? S.law[S.vrow[m]][lane] : 0.f;
    const float key = __fadd_rn(__fmaf_rn(-a, bq, q), 0.f);
    const bool pos = have && key > 0.f;
    const unsigned kk = pos ? ord_key(key) : 0u;
    if (__popc(__ballot_sync(FULL, pos)) < s) break;
    S.kx[lane] = kk;
    __syncwarp();
    // Omega_1: the entries with fewer than s larger keys; where the last of
    // them tie, the smaller token ids (the lower lanes)
    int above = 0;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const uint4 o = reinterpret_cast<const uint4*>(S.kx)[c];
      above += (o.x > kk ? 1 : 0) + (o.y > kk ? 1 : 0) + (o.z > kk ? 1 : 0) + (o.w > kk ? 1 : 0);
    }
    unsigned selm = __ballot_sync(FULL, pos && above < s);
    if (__popc(selm) > s) {
      const int last = (int)__reduce_max_sync(FULL, (selm >> lane & 1u) ? (unsigned)above : 0u);
      const unsigned tie = __ballot_sync(FULL, pos && above == last);
      selm = __ballot_sync(FULL, (selm >> lane & 1u) &&
                                     (above < last || __popc(tie & ((1u << lane) - 1u)) < s - last));
    }
    const bool sel = (selm >> lane) & 1u;
    float ra = (have && !sel) ? a : 0.f, rb = (have && !sel) ? bq : 0.f;
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      ra = __fadd_rn(ra, __shfl_xor_sync(FULL, ra, o));
      rb = __fadd_rn(rb, __shfl_xor_sync(FULL, rb, o));
    }
    const int rk = __popc(selm & ((1u << lane) - 1u));
    if (lane >= s && lane < MDS_MAX_S) {
      S.om[lane] = 0x7fffffff;
      S.om_q[lane] = 0.f;
      S.om_a[lane] = 0.f;
      S.om_b[lane] = 0.f;
    }
    if (sel) {
      S.om[rk] = id;
      S.om_q[rk] = q;
      S.om_a[rk] = a;
      S.om_b[rk] = bq;
    }
    __syncwarp();
    float x;
    bool capped;
    A = stage_solve5(ra, rb, A, Btok, u, S.om, S.om_q, S.om_a, S.om_b, x, &capped);
    if (capped && lane == 0) atomicOr(p.status, MDS_ST_LP_CAP);
    const float xr = __shfl_sync(FULL, x, rk & 31);
    a = sel ? xr : __fmul_rn(0.5f, __fadd_rn(__fmul_rn(a, rb), __fmul_rn(bq, ra)));
    __syncwarp();   // the tables are read before the next stage writes them
  }
  if (have) S.cur[lane] = a;
  __syncwarp();
  *Yo = A;
  return m;
}

// Warp 0: Algorithm 1 on the intermediate token Y with law p_I = a (on U):
// accept with probability min(1, q(Y) / p_I(Y)), otherwise draw from the
// residual max(0, q - p_I) in token-id order.  *R: the residual mass after a
// rejection (and with acc_prob always), else 0.
__device__ int accept_resid(const Params& p, Shared& S, int b, int j, int Y, const float* a, float* R, float* qY,
                            float* pIY) {
  const int lane = threadIdx.x & 31;
  const float* q = S.law[0];
  const float qy = law_at(S, q, Y), py = law_at(S, a, Y);
  const float ratio = py > 0.f ? __fdiv_rn(qy, py) : kPosInf;
  const bool acc = draw_uniform(p.seed, b, j, kDrawAccept) < fminf(1.f, ratio);
  *qY = qy;
  *pIY = py;
  *R = 0.f;
  if (acc && !p.acc_prob) return Y;
  const float ures = acc ? 0.f : draw_uniform(p.seed, b, j, kDrawResidual);
  float tot;
  int z = warp_cdf(S.nU, [&](int i) { return fmaxf(0.f, __fsub_rn(q[i], a[i])); }, ures, &tot);
  *R = tot;
  if (acc) return Y;
  if (z < 0) {
    // only by rounding: sample q
    if (lane == 0) atomicOr(p.status, MDS_ST_ZERO_RESID);
    float t;
    z = warp_cdf(S.nU, [&](int i) { return q[i]; }, ures, &t);
  }
  return z >= 0 ? S.uid[z] : (S.nU > 0 ? S.uid[0] : 0);
}

// Warp 0: sequential rejection over the valid drafts (the SpecTr baseline):
// round i accepts X_i with probability min(1, q_i(X_i) / p_i(X_i)); on
// rejection q_{i+1} = max(0, q_i - p_i) / R_i.  If every round rejects, Z is
// drawn from the last target.  *R: prod_i R_i (0 after an acceptance unless
// acc_prob, which computes the later rounds too).
__device__ int spectr(const Params& p, Shared& S, int b, int j, float* R, float* qY, float* pIY) {
  const int lane = threadIdx.x & 31;
  const int nU = S.nU, nv = S.nv;
  for (int i = lane; i < nU; i += 32) S.cur[i] = S.law[0][i];
  __syncwarp();
  float prodR = 1.f;
  int zacc = -1;
  for (int i = 0; i < nv; ++i) {
    const float* pl = S.law[S.vrow[i]];
    if (zacc < 0) {
      const int x = S.X[i];
      const float qi = law_at(S, S.cur, x), pv = law_at(S, pl, x);
      const float ratio = pv > 0.f ? __fdiv_rn(qi, pv) : kPosInf;
      if (i == 0) {
        *qY = qi;
        *pIY = pv;
      }
      if (draw_uniform(p.seed, b, j, kDrawAccept + i) < fminf(1.f, ratio)) {
        zacc = x;
        if (!p.acc_prob) {
          *R = 0.f;
          return zacc;
        }
      }
    }
    float part = 0.f;
    for (int t = lane; t < nU; t += 32) part = __fadd_rn(part, fmaxf(0.f, __fsub_rn(S.cur[t], pl[t])));
    const float Ri = warp_sum(part);
    prodR = __fmul_rn(prodR, Ri);
    if (Ri > 0.f) {
      const float inv = __frcp_rn(Ri);
      for (int t = lane; t < nU; t += 32) S.cur[t] = __fmul_rn(fmaxf(0.f, __fsub_rn(S.cur[t], pl[t])), inv);
    }
    __syncwarp();
  }
  *R = prodR;
  if (zacc >= 0) return zacc;
  float tot;
  int z = warp_cdf(nU, [&](int t) { return S.cur[t]; }, draw_uniform(p.seed, b, j, kDrawResidual), &tot);
  if (z < 0) {
    if (lane == 0) atomicOr(p.status, MDS_ST_ZERO_RESID);
    z = warp_cdf(nU, [&](int t) { return S.law[0][t]; }, draw_uniform(p.seed, b, j, kDrawResidual), &tot);
  }
  return z >= 0 ? S.uid[z] : (S.nU > 0 ? S.uid[0] : 0);
}

// Warp 0: one depth below L: the rows' laws on U, the scheme's token, the walk.
__device__ __noinline__ void decide(const Params& p, Shared& S, int b, int j) {
  const int lane = threadIdx.x & 31;
  for (int r = 0; r < S.nrows; ++r) row_probs(p, S, r);
  build_union(S);
  const int nv = S.nv;
  int Z, Yd;
  float R = 0.f, qY = 0.f, pIY = 0.f;
  if (p.scheme == MDS_SPECTR) {
    Z = spectr(p, S, b, j, &R, &qY, &pIY);
    Yd = S.X[0];
  } else {
    int Y = S.X[0];
    const float* a = S.law[S.vrow[0]];
    if ((p.scheme == MDS_WIS || p.scheme == MDS_WISSORT) && nv > 1) {
      // every stage's selection uniform at once (lane m - 1 draws stage m's)
      const float ul = (lane + 1 < nv) ? draw_uniform(p.seed, b, j, kDrawSelect + lane) : 0.f;
      const bool sorted = p.scheme == MDS_WISSORT;
      int m = 1;
      if (!sorted && S.nU <= 32 && p.wis_s <= 5) {
        m = wis_stages_small(p, S, ul, &Y);
      } else {
        for (int i = lane; i < S.nU; i += 32) S.cur[i] = a[i];
        __syncwarp();
      }
      for (; m < nv; ++m)
        Y = wis_stage(p, S, Y, S.X[m], S.vrow[m], __shfl_sync(FULL, ul, m - 1), sorted);
      a = S.cur;
    }
    Z = accept_resid(p, S, b, j, Y, a, &R, &qY, &pIY);
    Yd = Y;
  }
  if (lane == 0) {
    p.out_tokens[(size_t)b * (p.L + 1) + j] = Z;
    if (p.out_diag) {
      float* dg = p.out_diag + ((size_t)b * (p.L + 1) + j) * 4;
      dg[0] = qY;
      dg[1] = pIY;
      dg[2] = R;
      dg[3] = (float)Yd;
    }
    unsigned nvm = 0u;
    for (int i = 0; i < nv; ++i)
      if (S.X[i] == Z) nvm |= 1u << S.vbr[i];
    S.valid = nvm;
    if (!nvm) {
      p.out_accept[b] = j;
      S.done = 1;
    }
  }
  __syncwarp();
}

// Warp 0: every draft accepted: the bonus token from the restricted target
// row at depth L, by inverse CDF in token-id order.
__device__ __noinline__ void bonus_step(const Params& p, Shared& S, int b) {
  const int lane = threadIdx.x & 31;
  row_probs(p, S, 0);
  const int n = S.n[0];
  if (lane < n) {
    const int id = S.id[0][lane];
    int k = 0;
    for (int f = 0; f < n; ++f) k += (S.id[0][f] < id) ? 1 : 0;
    S.bid[k] = id;
    S.bw[k] = S.pr[0][lane];
  }
  __syncwarp();
  float Q;
  const int z = warp_cdf(n, [&](int i) { return S.bw[i]; }, draw_uniform(p.seed, b, p.L, kDrawBonus), &Q);
  if (lane == 0) {
    p.out_tokens[(size_t)b * (p.L + 1) + p.L] = z >= 0 ? S.bid[z] : (n > 0 ? S.bid[0] : 0);
    if (p.out_diag) {
      float* dg = p.out_diag + ((size_t)b * (p.L + 1) + p.L) * 4;
      dg[0] = 0.f;
      dg[1] = 0.f;
      dg[2] = Q;
      dg[3] = -1.f;
    }
    p.out_accept[b] = p.L;
    S.done = 1;
  }
  __syncwarp();
}

template <int DT>
__global__ void __launch_bounds__(kThreads, 2) topk_kernel(const Params p) {
  __shared__ Shared S;
  const int b = blockIdx.x;
  const int tid = threadIdx.x, warp = tid >> 5;
  const int kk = min(p.top_k, p.V);
  for (int j = tid; j <= p.L; j += kThreads) p.out_tokens[(size_t)b * (p.L + 1) + j] = -1;
  if (tid == 0) {
    S.valid = (p.K >= 32) ? FULL : ((1u << p.K) - 1u);
    S.done = 0;
  }
  __syncthreads();
  for (int j = 0; j <= p.L; ++j) {
    const bool bonus = (j == p.L);
    if (warp == 0) plan(p, S, b, j, bonus);
    __syncthreads();
    const int nr = S.nrows;
    for (int r = 0; r < nr; ++r) select_row<DT>(p, S, r, kk);
    if (warp == 0) {
      if (bonus)
        bonus_step(p, S, b);
      else
        decide(p, S, b, j);
    }
    __syncthreads();
    if (S.done) break;
  }
}

template <int DT>
cudaError_t launch_dt(const Params& p, cudaStream_t stream) {
  topk_kernel<DT><<<p.B, kThreads, 0, stream>>>(p);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch(const Params& p, cudaStream_t stream) {
  if (p.B <= 0) return cudaSuccess;
  return p.dtype == MDS_F32 ? launch_dt<MDS_F32>(p, stream) : launch_dt<MDS_BF16>(p, stream);
}

int verify(const mds_config& c, int scheme, const int8_t* model_of, bool vec, const void* target_logits,
           const void* const* draft_logits, const int32_t* draft_tokens, const float* temperatures,
           int32_t* out_tokens, int32_t* out_accept_len, float* out_diag, int B, uint64_t seed, unsigned* status,
           cudaStream_t stream) {
  if (!serves(scheme)) return MDS_EUNSUP;
  Params p{};
  p.target = static_cast<const char*>(target_logits);
  for (int k = 0; k < c.K; ++k) {
    p.drafts[k] = static_cast<const char*>(draft_logits[k]);
    p.model_of[k] = model_of[k];
  }
  p.tokens = draft_tokens;
  p.temps = temperatures;
  p.out_tokens = out_tokens;
  p.out_accept = out_accept_len;
  p.out_diag = out_diag;
  p.status = status;
  p.seed = seed;
  p.B = B;
  p.K = c.K;
  p.L = c.L;
  p.V = c.V;
  p.dtype = c.dtype;
  p.esize = c.dtype == MDS_F32 ? 4 : 2;
  p.top_k = c.top_k;
  p.wis_s = c.wis_s;
  p.scheme = scheme;
  p.acc_prob = c.acc_prob;
  p.vec = vec ? 1 : 0;
  const cudaError_t e = launch(p, stream);
  return e == cudaSuccess ? MDS_OK : record_cuda_error(e, "top-k kernel launch");
}

}  // namespace topk
}  // namespace mds
