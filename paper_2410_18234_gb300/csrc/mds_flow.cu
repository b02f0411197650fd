// Slice-dataflow engine for batched multi-draft speculative verification on
// GB300 (sm_103a): schemes single, weighted importance sampling (WIS) and the
// truncated alphabet (WIS0).
//
// Every row the walk visits (the target row and one row per distinct draft
// model at a depth, the target row at the bonus depth) is cut into slices of
// T tokens.  One pass of one sequence is ns slice tasks over the same rows.
// The grid is persistent (every CTA of the launch resident): in each CTA one
// scheduler warp takes task numbers from a global counter, waits for the
// task's publication in a ring in global memory, reads the sequence's pass
// descriptor and bulk-copies the task's slice of every row of the pass into
// one of two shared-memory buffers (cp.async.bulk, mbarrier completion).  The
// eight compute warps reduce the slice to a record in global memory:
//   stats    row maxima and exp sums (2^fma(l, c, -round(m c)) against the
//            slice maximum m) and, for the weighted schemes, the slice's
//            largest target logits (the candidate list) with every row's logit
//            there; the sums leave the list out, so every later mass is a sum
//            of positive terms;
//   resid    the residual mass sum max(0, q - p_I) of Algorithm 1;
//   replace  the target mass outside Omega_0 (truncated alphabet);
//   full     a full-vocabulary stage of the weighted scheme: the slice's top-s
//            keys q - a b with a and b, and the Omega_2 masses of the rest;
//   bonus    the target row's maximum, sum and run sums at depth L.
// The compute warps work on their own shares of a slice (one block barrier
// where a list is wanted: its bound comes from all of them) and leave partial
// results in a record slot in shared memory; a
// publishing warp merges them, stores the record and counts the pass's
// slices.  The one that counts a pass's last slice posts a decision request.
// A decision warp combines the records in slice order, runs the importance
// step (the WIS stages on the merged candidate list, Omega_1 by
// the keys q - a b, the stage LP, Remark 4's pairwise stages), Algorithm 1's
// accept test, and the inverse-CDF search of a residual draw (slice by the
// records, token by one re-read of that slice), then advances the walk and
// publishes the sequence's next pass.  Decisions depend only on the data and
// the Philox draws, never on which CTA takes a task, so results are
// bit-reproducible.  Every wait is bounded in time; a wait that gives up sets
// MDS_ST_TIMEOUT and an abort flag on which every CTA leaves, after waiting
// for its own copies in flight.
#include <cstdlib>
#include <cuda_bf16.h>

#include "mds_device.cuh"
#include "mds_flow.h"

namespace mds {
namespace flow {
namespace {

using namespace mds::dev;

constexpr int kCW = 8;                 // compute warps
constexpr int kCT = kCW * 32;          // compute threads
constexpr int kBlock = kCT + 64;       // + the scheduler warp and the publishing warp
constexpr int kNBuf = 2;               // slice buffers per CTA
// Task descriptors: a buffer is released before its task is done, so task k's
// descriptor lives on until task k + 3 is issued, which waits for every warp
// to release task k + 1's buffer, so to have done task k.
constexpr int kNDesc = kNBuf + 1;
constexpr int kSlots = 3;              // records between the compute warps and the publishing warp
constexpr int kFastUnits = kBufBytes / 16;   // units of all rows one slice holds
constexpr int kWarpCand = 32;          // tokens one warp may set aside in a slice
constexpr int kSlotCand = kCW * kWarpCand;
constexpr int kMaxRuns = kFastUnits / 32;    // runs of 32 units of a slice
constexpr int kCtasPerSm = 2;          // resident CTAs per SM (the launch bound)
constexpr int kCandCap = 512;          // candidate tokens one slice may set aside
constexpr int kListMax = 64;           // candidate list length at most
constexpr int kSliceListMax = 32;      // a slice's list found warp by warp, at most
constexpr int kRankMax = 64;           // tokens the publishing warp ranks by counting
constexpr int kGroups = 8;             // groups of a warp's lanes with a maximum each
constexpr int kHdr = 2 * kMaxRows + 2; // record: (max, sum) per row, tau, list length
constexpr int kTopF = 8;               // per-thread candidates of a full stage (>= MDS_MAX_S)
constexpr int kMaxEntries = 512;       // slices x slice list length, at most
constexpr int kDecStage = 8192;        // bytes of a pass's slice records ([ns][rec_floats]) at most
constexpr unsigned long long kWaitNs = 2000000000ull;   // 2 s bound on every wait
constexpr unsigned FULLM = 0xffffffffu;
static_assert(kHdr % 4 == 0, "record header keeps 16-byte alignment");
static_assert(kTopF >= MDS_MAX_S, "full-stage candidates");

enum : int { kNone = 0, kStats = 1, kResid = 2, kBonus = 3, kFull = 4, kReplace = 5 };

// A decision request: sequence (16 bits), depth (7), whether the pass is the
// sequence's first (its descriptor is not in memory yet).
__host__ __device__ constexpr unsigned dec_payload(int b, int j, bool first) {
  return ((unsigned)b << 8) | ((unsigned)j << 1) | (first ? 1u : 0u);
}
static_assert(MDS_MAX_L < 127, "decision request fields");

// Phase-timer slots (SM cycles summed over CTAs, or counts).
enum : int {
  kPhKernel = 0,        // time in the kernel (per CTA, summed)
  kPhWaitFull,          // compute warps waiting for a loaded slice
  kPhTaskList,          // stats tasks with the candidate list
  kPhTaskStats,         // stats tasks without it (and the bonus row)
  kPhTaskResid,         // residual and replace tasks
  kPhTaskFull,          // full-vocabulary stage tasks
  kPhDecStats,          // stats decisions (all of it)
  kPhDecCombine,        //   of which: combining records and the list merge
  kPhDecStages,         //   of which: the WIS stages on the list
  kPhDecResid,          // residual and replace decisions (with the search)
  kPhDecFull,           // full-stage decisions
  kPhDecBonus,          // bonus decisions
  kPhPush,              // publishing the next pass
  kPhSchedPoll,         // scheduler waiting for a published task
  kPhSchedEmpty,        // scheduler waiting for a free buffer
  kPhDecPoll,           // decision warps waiting for a request
  kPhDecPlan,           // decisions: planning a pass (rows, tokens, cached logits)
  kPhDecLoad,           // decisions: staging the state, inputs and records
  kPhDecSelect,         // decisions: WIS stage selection and masses (list)
  kPhDecAccept,         // decisions: the accept step (with its push or walk)
  kPhDecWalk,           // decisions: the walk to the next depth
  kPhListA,             // list tasks: maxima and the candidate threshold
  kPhListB,             // list tasks: the sums and the candidates
  kPhListC,             // list tasks: ranking and the record
  kPhPublish,           // a task's record publication (fence, pass counter)
  kPhCombine,           // (unused)
  kPhLp,                // the stage LPs
  kPhLpCalls,           // count: stage LPs
  kPhTasks,             // count: slice tasks
  kPhDecisions,         // count: decisions
  kPhaseN
};

// ------------------------------------------------------------------ state

struct FRow {
  const char* ptr;     // row start (token 0)
  float c;             // log2(e) / temperature
  float M, invZ;       // row maximum and inverse normaliser (after the stats decision)
  float gamma;         // WIS: coefficient of this draft row in the generic law
};
struct __align__(16) FPass {   // what the slice tasks of a pass read
  int kind, j, nrows, nstream;
  int list, rb, nspec, all0;
  float cut;
  int pad0, pad1, pad2;
  FRow row[kMaxRows];          // target, then one row per distinct draft model of the valid branches
  int spec_id[kMaxSpecial];    // WIS: tokens with an explicit law value (every Omega_1 so far)
  float spec_val[kMaxSpecial];
  int pad3[2];
};
static_assert(sizeof(FPass) % 16 == 0, "pass descriptor copies in 16-byte chunks");
struct __align__(16) FWalk {   // decision state of a sequence between passes
  unsigned valid;              // valid branches at the current depth
  int stage, A;                // WIS full stages: next stage, current stage input
  int Y;                       // intermediate token
  float qY, pIY;
  int acc;                     // accept test passed
  float ures;                  // uniform of the pending inverse-CDF draw
  float R;                     // residual mass (diagnostics)
  int Yp;                      // WIS0: output of the inner step on Omega_0 (-1: none)
  int Ydiag;
  int zres;                    // the pending draw is the zero-residual fallback (sample q)
  int pad[4];
};
static_assert(sizeof(FWalk) % 16 == 0, "walk state copies in 16-byte chunks");
struct __align__(16) FSeq {
  FPass P;
  FWalk W;
};

struct __align__(16) FDesc {
  FPass P;
  int b, slice, end, exit;     // the sequence, the next slice and the end of its group
  int first, pad[3];           // the group's first slice
};
static_assert(sizeof(FDesc) % 16 == 0, "descriptor moves in 16-byte chunks");

struct Cand {  // full-stage candidate: larger key first, then smaller token id
  float key;
  int id;
  float a, b;
};
#define CAND_NONE Cand{kNegInf, 0x7fffffff, 0.f, 0.f}
__device__ __forceinline__ bool better(float ka, int ia, float kb, int ib) {
  return ka > kb || (ka == kb && ia < ib);
}

// The uniforms of one depth, drawn together by the lanes of a decision warp.
enum : int { kDrSelect = 0, kDrAccept = 16, kDrResidual, kDrBonus, kDrKeep, kDrOutside, kDrawsN };
__device__ __forceinline__ int draw_id(int i) {
  return i < 16 ? kDrawSelect + i
                : (i == kDrAccept ? kDrawAccept
                                  : (i == kDrResidual ? kDrawResidual
                                                      : (i == kDrBonus ? kDrawBonus
                                                                       : (i == kDrKeep ? kDrawKeep : kDrawOutside))));
}

struct DState {                // the decision's working state (shared memory)
  FPass P;
  FWalk W;
  int nv;
  int vbr[MDS_MAX_K], X[MDS_MAX_K], vrow[MDS_MAX_K];
  float xl[MDS_MAX_K][kMaxRows];   // every row's logit at each valid draft token (X[k])
  int xl_ok;
  // candidate list (token-id order)
  int n, cand_all;
  float cand_q, cand_tau;
  int cm_id[kListMax];
  float cm_l0[kListMax];
  float cm_e[kListRowsMax][kListMax];
  float pc[kListRowsMax];
  // stage
  __align__(16) unsigned kx[32];   // the list's keys of a stage
  int om[MDS_MAX_S];
  float om_q[MDS_MAX_S], om_a[MDS_MAX_S], om_b[MDS_MAX_S], om_x[MDS_MAX_S];
  int Y;
  Cand fin[kTopF];
  float lp_rs[kMaxPairs], lp_fl[kMaxPairs], lp_fh[kMaxPairs];   // LP pair state in shared memory
  // search
  int tok;
  // truncated alphabet
  int k_lane[MDS_MAX_K], k_row[MDS_MAX_K];
  int o0_n, o0_all;
  // inputs of the sequence staged by the decision: draft tokens at the
  // depth (tk0) and the next depth (tk1), temperatures (target, drafts)
  int tk0[MDS_MAX_K], tk1[MDS_MAX_K];
  float tmp[MDS_MAX_K + 1];
  float dr[kDrawsN];           // the depth's uniforms, by kDr*
  int xl_wait;                 // the row logits at the draft tokens are still in flight
  float o0_cut, o0_pa;
};
static_assert(offsetof(DState, W) == offsetof(DState, P) + sizeof(FPass) && offsetof(FSeq, W) == sizeof(FPass),
              "a sequence's state copies into the decision state in one piece");

// What the compute warps hand the publishing warp of one slice.
enum : int { kSlotDone = 0,   // the record is in global memory already
             kSlotSums, kSlotList, kSlotBonus, kSlotRuns, kSlotExit };
struct __align__(16) Slot {
  int mode, b, slice, kind, j, R, nrun;
  int count;                   // slices to count with this one: its group's, at the group's end (else 0)
  float c[kListRowsMax];
  int nc[kCW];                 // per warp: tokens set aside
  float tau[kCW];              // per warp: largest target logit not set aside
  float m[kCW][kListRowsMax], s[kCW][kListRowsMax];
  float run[kMaxRuns];
  __align__(16) unsigned sel[kRankMax];    // the tokens ranked for the list: keys ...
  unsigned short at[kRankMax];             // ... and entries
  __align__(16) unsigned key[kSlotCand];   // tokens set aside, warp by warp: rank key (see cand_key),
  unsigned short loc[kSlotCand];           // place in the slice,
  float l[kListRowsMax][kSlotCand];        // every row's logit
};
static_assert(kListRowsMax * kSlotCand >= 2 * kCandCap, "the block-wise list's arrays lie over two slots' logits");

struct FShared {
  uint64_t full[kNBuf], empty[kNBuf], done[kSlots], free[kSlots];
  FDesc desc[kNDesc];
  FDesc pend;                  // the scheduler's next task, resolved ahead
  float red[kCW * 2 * kMaxRows];
  float wth[kCW];
  unsigned gmax[kCW * kGroups];   // order keys of the lane groups' largest target logits
  int ncand, issued, consumed;
  float addtau;
  float add[kMaxRows];
  uint32_t bitmap[64];         // one bit per 16-byte unit of a slice holding a special token
  Cand wcand[kCW * kTopF];
  Cand blk[kTopF];
  int flag_ok[2];
#ifdef MDS_PHASE_TIMERS
  unsigned long long tm[kPhaseN];
#endif
};

// ------------------------------------------------------------------ memory helpers

__device__ __forceinline__ unsigned long long ld_acquire(const unsigned long long* a) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.u64 %0, [%1];" : "=l"(v) : "l"(a) : "memory");
  return v;
}
__device__ __forceinline__ void st_release(unsigned long long* a, unsigned long long v) {
  asm volatile("st.release.gpu.u64 [%0], %1;" ::"l"(a), "l"(v) : "memory");
}
__device__ __forceinline__ unsigned ld_relaxed(const unsigned* a) {
  unsigned v;
  asm volatile("ld.relaxed.gpu.u32 %0, [%1];" : "=r"(v) : "l"(a) : "memory");
  return v;
}
__device__ __forceinline__ unsigned atom_add_acq_rel(unsigned* a, unsigned v) {
  unsigned old;
  asm volatile("atom.add.acq_rel.gpu.u32 %0, [%1], %2;" : "=r"(old) : "l"(a), "r"(v) : "memory");
  return old;
}
__device__ __forceinline__ unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Ring words: launch, lap over the ring, payload of 24 bits (tasks: sequence
// << 8 | group of slices; decisions: dec_payload).
constexpr unsigned long long kRingPay = 0xffffffull;
__device__ __forceinline__ unsigned long long ring_word(unsigned epoch, unsigned lap, unsigned pay) {
  return ((unsigned long long)(epoch & 0x3fffffffu) << 34) | ((unsigned long long)((lap + 1u) & 0x3ffu) << 24) | pay;
}
__device__ __forceinline__ void st_relaxed(unsigned long long* a, unsigned long long v) {
  asm volatile("st.relaxed.gpu.u64 [%0], %1;" ::"l"(a), "l"(v) : "memory");
}
__device__ __forceinline__ void cbar() { asm volatile("bar.sync 1, %0;" ::"n"(kCT) : "memory"); }

// 16-byte chunk copies of state between global (L2, coherent) and shared memory.
__device__ __forceinline__ void copy_in(void* dst, const void* src, int bytes, int t, int nt) {
  const int4* s = reinterpret_cast<const int4*>(src);
  int4* d = reinterpret_cast<int4*>(dst);
  for (int i = t; i < bytes / 16; i += nt) d[i] = __ldcg(s + i);
}
__device__ __forceinline__ void copy_out(void* dst, const void* src, int bytes, int t, int nt) {
  const int4* s = reinterpret_cast<const int4*>(src);
  int4* d = reinterpret_cast<int4*>(dst);
  for (int i = t; i < bytes / 16; i += nt) __stcg(d + i, s[i]);
}

// Asynchronous copies global -> shared (the issuing thread's own copies
// complete at cpa_wait): 16 bytes through L2 only (data other SMs write
// during the launch), 4 bytes cached (inputs only).
__device__ __forceinline__ void cpa16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cpa4(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cpa_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// ------------------------------------------------------------------ phase timers
// Built with -DMDS_PHASE_TIMERS, every CTA accumulates SM cycles per phase
// (thread 0 of the compute warps, lane 0 of the scheduler warp) and adds them
// to g_phase when it leaves; mds_phase_timers() reads and clears them.
// Without it the macros vanish.
#ifdef MDS_PHASE_TIMERS
__device__ unsigned long long g_phase[kPhaseN];
#define PT_T0(v) const long long v = clock64()
#define PT_ADD(i, v)                                             \
  do {                                                           \
    if ((threadIdx.x & 0xff) == 0) S.tm[i] += (unsigned long long)(clock64() - (v)); \
  } while (0)
#define PT_CNT(i)                                 \
  do {                                            \
    if ((threadIdx.x & 0xff) == 0) S.tm[i] += 1ull; \
  } while (0)
#define PT_ADDW(i, v)                                                               \
  do {                                                                              \
    if ((threadIdx.x & 31) == 0) atomicAdd(&S.tm[i], (unsigned long long)(clock64() - (v))); \
  } while (0)
#define PT_CNTW(i)                                         \
  do {                                                     \
    if ((threadIdx.x & 31) == 0) atomicAdd(&S.tm[i], 1ull); \
  } while (0)
#else
#define PT_T0(v)
#define PT_ADD(i, v)
#define PT_CNT(i)
#define PT_ADDW(i, v)
#define PT_CNTW(i)
#endif

// ------------------------------------------------------------------ slice loading (plain loads)
// Rows [0, R) of the slice [tok0, tok0 + n) into shared memory, every
// thread its own units (u = thread, thread + 256, ...): used where bulk
// copies are not (mapped host memory, rows not 16-byte aligned).
template <int DT>
__device__ __noinline__ void load_rows(const FPass& P, int R, char* b, int tok0, int n, int T, int V) {
  constexpr int VE = Elt<DT>::VE, es = 16 / VE;
  const int U = (n + VE - 1) / VE;
  for (int r = 0; r < R; ++r) {
    const char* first = P.row[r].ptr;
    const char* src = first + (size_t)tok0 * es;
    const char* end = first + (size_t)V * es;
    char* dst = b + (size_t)r * T * es;
#pragma unroll 4
    for (int u = threadIdx.x; u < U; u += kCT)
      *reinterpret_cast<uint4*>(dst + 16 * (size_t)u) = load_unit<DT>(src, first, end, u, n);
  }
}

// ------------------------------------------------------------------ tokens set aside
// Their numbers in a slot, warp by warp.
struct Numbers {
  int first[kCW + 1];   // each warp's first token
  __device__ __forceinline__ explicit Numbers(const Slot& T) {
    first[0] = 0;
#pragma unroll
    for (int w = 0; w < kCW; ++w) first[w + 1] = first[w] + T.nc[w];
  }
  __device__ __forceinline__ int entry(int j) const {   // slot entry of token j < first[kCW]
    int at = j;
#pragma unroll
    for (int w = 1; w < kCW; ++w) at = j >= first[w] ? w * kWarpCand + j - first[w] : at;
    return at;
  }
};
// The first LN of n > LN tokens: those with a larger key than x, or x itself
// and a place of at most y (equal 32-bit logits; 16-bit keys are distinct).
// Warp-wide; out of line, few slices need it.
template <int DT>
__device__ __noinline__ uint2 list_cut(const Slot& T, int n, int LN) {
  const int lane = threadIdx.x & 31;
  const Numbers num(T);
  auto count = [&](auto&& in) {
    unsigned k = 0u;
#pragma unroll 1
    for (int j = lane; j < n; j += 32) k += in(num.entry(j)) ? 1u : 0u;
    return (int)__reduce_add_sync(FULLM, k);
  };
  unsigned thr = 0u, last = 0xffffu;
  int have = n;
#pragma unroll 1
  for (int bit = 31; bit >= 0; --bit) {
    if (have == LN) break;
    const unsigned c = thr | (1u << bit);
    const int k = count([&](int i) { return T.key[i] >= c; });
    if (k >= LN) {
      thr = c;
      have = k;
    }
  }
  if (DT != MDS_BF16 && have > LN) {
    const int need = LN - count([&](int i) { return T.key[i] > thr; });
    last = 0u;
#pragma unroll 1
    for (int bit = 15; bit >= 0; --bit) {
      const unsigned c = last | ((1u << bit) - 1u);
      if (count([&](int i) { return T.key[i] == thr && T.loc[i] <= c; }) < need) last |= 1u << bit;
    }
  }
  return make_uint2(thr, last);
}

// ------------------------------------------------------------------ the engine

template <int DT>
struct Eng {
  using E = Elt<DT>;
  static constexpr int VE = E::VE;

  const Params& p;
  FShared& S;
  char* bufs;     // kNBuf x kBufBytes
  Slot* slots;    // kSlots records on their way to the publishing warp
  int* cid;       // candidate ids
  float* cl;      // candidate target logits
  int* crank;     // candidate ranks
  int* cord;      // candidates ranked past the list, in rank order

  __device__ __forceinline__ bool aborted() const { return ld_relaxed(&p.ctl[kCtlAbort]) != 0u; }
  __device__ __forceinline__ void set_abort(unsigned bits) const {
    atomicOr(p.status, bits);
    atomicExch(&p.ctl[kCtlAbort], 1u);
  }
  __device__ __forceinline__ char* buf(int bi) const { return bufs + (size_t)bi * kBufBytes; }
  __device__ __forceinline__ const char* srow(const char* b, int r) const { return b + (size_t)r * p.T * p.esize; }
  __device__ __forceinline__ uint4 raw(const char* b, int r, int u) const {
    return *reinterpret_cast<const uint4*>(srow(b, r) + 16 * u);
  }
  // This warp has read its part of a buffer (the wait for the loads' values is
  // the reads' own).
  __device__ __forceinline__ void release(int bi) const {
    __syncwarp();
    if ((threadIdx.x & 31) == 0) mbar_arrive(&S.empty[bi]);
  }
  // Explicit value of a special token of the current law, else fallback.
  __device__ __forceinline__ float spec_lookup(const FPass& P, int tok, float fallback) const {
    for (int i = 0; i < P.nspec; ++i)
      if (P.spec_id[i] == tok) return P.spec_val[i];
    return fallback;
  }

  // -------------------------------------------------------------- scheduler warp
  __device__ bool wait_mbar(uint64_t* bar, uint32_t parity) const {
    if (mbar_try_wait(bar, parity)) return true;
    const unsigned long long t0 = now_ns();
    for (int it = 0;; ++it) {
      if (mbar_try_wait(bar, parity)) return true;
      if ((it & 63) == 63 && now_ns() - t0 > kWaitNs) return false;
    }
  }

  // Warp-parallel plan of a sequence's depth-0 pass (every branch valid):
  // lane k < K takes branch k, and a draft model's row is that of its first
  // branch (the same rows, in the same order, as Dec::plan_warp).
  __device__ void plan_depth0_warp(int b, FPass& P) const {
    const int lane = threadIdx.x & 31;
    const int K = p.K;
    const int m = (lane < K) ? (int)p.model_of[lane] : 64 + lane;
    const unsigned same = __match_any_sync(FULLM, m);
    const bool first = lane < K && (__ffs(same) - 1) == lane;
    const unsigned fm = __ballot_sync(FULLM, first);
    const int nr = 1 + __popc(fm);
    if (first) {
      const int r = 1 + __popc(fm & ((1u << lane) - 1u));
      P.row[r].ptr = p.drafts[lane] + ((size_t)b * p.L * (size_t)p.V) * p.esize;
      float td = p.temps[(size_t)b * (1 + K) + 1 + lane];
      if (!(td > 0.f) || !(td < kPosInf)) {
        atomicOr(p.status, MDS_ST_BADTEMP);
        td = 1.f;
      }
      P.row[r].c = __fdiv_rn(kLog2e, td);
      P.row[r].M = 0.f;
      P.row[r].invZ = 0.f;
      P.row[r].gamma = 0.f;
    }
    if (lane == 0) {
      P.row[0].ptr = p.target + ((size_t)b * K * (p.L + 1) * (size_t)p.V) * p.esize;
      float tq = p.temps[(size_t)b * (1 + K)];
      if (!(tq > 0.f) || !(tq < kPosInf)) {
        atomicOr(p.status, MDS_ST_BADTEMP);
        tq = 1.f;
      }
      P.row[0].c = __fdiv_rn(kLog2e, tq);
      P.row[0].M = 0.f;
      P.row[0].invZ = 0.f;
      P.row[0].gamma = 0.f;
      P.nrows = nr;
      P.j = 0;
      P.nspec = 0;
      P.rb = 0;
      P.cut = 0.f;
      P.all0 = 0;
      P.kind = kStats;
      if (p.scheme == MDS_WIS0) {
        P.nstream = 1;
        P.list = 1;
      } else if (p.scheme == MDS_WIS) {
        P.nstream = nr;
        P.list = (K > 1 && nr <= kListRowsMax && p.ln > 0) ? 1 : 0;
      } else {
        P.nstream = min(2, nr);
        P.list = 0;
      }
    }
  }

  // Claim the next task number and resolve it into Pd: the sequence, its
  // slices and the sequence's pass descriptor (depth-0 tasks are implicit:
  // task t < B * ng0 is group t % ng0 of sequence t / ng0).  Returns 0 when no
  // work is left (every sequence finished, or an abort).  The number was
  // claimed one task ahead (tn, lane 0), so that its round trip is over; the
  // next one is claimed here.  Warp-wide.
  __device__ int resolve(FDesc& Pd, unsigned& tn) {
    const int lane = threadIdx.x & 31;
    const unsigned N0 = (unsigned)p.B * (unsigned)p.ng0;
    int have = 0, b = 0, g = 0;
    if (lane == 0) {
      // the slot's word holds all of a task, and an acquire load orders the
      // store that gives the slot back
      const unsigned t = tn;
      tn = atomicAdd(&p.ctl[kCtlHead], 1u);
      const bool ab = aborted();
      const unsigned slot = t % (unsigned)p.ring_cap;
      const unsigned long long want = ring_word(p.epoch, t / (unsigned)p.ring_cap, 0u);
      if (t < N0) {
        b = (int)(t / (unsigned)p.ng0);
        g = (int)(t % (unsigned)p.ng0);
        st_relaxed(&p.ring_rtag[slot], want);
        have = ab ? 0 : 1;
      } else if (!ab) {
        const unsigned long long t0 = now_ns();
        PT_T0(t_poll);
        for (int it = 0;; ++it) {
          const unsigned long long w = ld_acquire(&p.ring_tag[slot]);
          if ((w & ~kRingPay) == want) {
            b = (int)((w >> 8) & 0xffffu);
            g = (int)(w & 0xffu);
            st_relaxed(&p.ring_rtag[slot], want);
            have = 2;
            break;
          }
          if ((it & 3) == 3 && (ld_relaxed(&p.ctl[kCtlDone]) >= (unsigned)p.B || aborted())) break;
          if ((it & 15) == 15 && now_ns() - t0 > kWaitNs) {
            set_abort(MDS_ST_TIMEOUT);
            break;
          }
          __nanosleep(it < 16 ? 32 : 128);
        }
        PT_ADD(kPhSchedPoll, t_poll);
      }
    }
    have = __shfl_sync(FULLM, have, 0);
    b = __shfl_sync(FULLM, b, 0);
    g = __shfl_sync(FULLM, g, 0);
    if (have == 1)
      plan_depth0_warp(b, Pd.P);
    else if (have == 2)
      copy_in(&Pd.P, &reinterpret_cast<const FSeq*>(p.seq)[b].P, (int)sizeof(FPass), lane, 32);
    if (lane == 0) {
      Pd.b = b;
      const int group = have == 1 ? p.group0 : p.group;
      Pd.slice = Pd.first = g * group;
      Pd.end = min(p.ns, (g + 1) * group);
      Pd.exit = have ? 0 : 1;
    }
    __syncwarp();
    return have != 0;
  }

  // The scheduler warp: the next task is resolved ahead (while the compute
  // warps work on the other buffer), so that a freed buffer only waits for
  // the descriptor move and the bulk copies.
  __device__ void scheduler() {
    const int lane = threadIdx.x & 31;
    unsigned tn = lane == 0 ? atomicAdd(&p.ctl[kCtlHead], 1u) : 0u;
    int have = resolve(S.pend, tn);
    for (int k = 0;; ++k) {
      const int bi = k % kNBuf;
      FDesc& D = S.desc[k % kNDesc];
      // the compute warps released this buffer (lane 0 waits; bounded)
      int ok = 1;
      PT_T0(t_empty);
      if (lane == 0 && k >= kNBuf) ok = wait_mbar(&S.empty[bi], ((k / kNBuf) - 1) & 1) ? 1 : 0;
      PT_ADD(kPhSchedEmpty, t_empty);
      ok = __shfl_sync(FULLM, ok, 0);
      if (!ok) {
        // the compute warps still hold the buffer: leave it untouched
        if (lane == 0) set_abort(MDS_ST_TIMEOUT);
        return;
      }
      {
        const int4* src = reinterpret_cast<const int4*>(&S.pend);
        int4* dst = reinterpret_cast<int4*>(&D);
        for (int i = lane; i < (int)(sizeof(FDesc) / 16); i += 32) dst[i] = src[i];
      }
      __syncwarp();
      int more = 0;
      if (lane == 0) {
        if (have && p.bulk) {
          const int s = D.slice;
          const int tok0 = s * p.T;
          const int n = min(p.T, p.V - tok0);
          const uint32_t bytes = (uint32_t)n * (uint32_t)p.esize;
          mbar_expect_tx(&S.full[bi], bytes * (uint32_t)D.P.nstream);
          for (int r = 0; r < D.P.nstream; ++r)
            bulk_copy(buf(bi) + (size_t)r * p.T * p.esize, D.P.row[r].ptr + (size_t)tok0 * p.esize, bytes, &S.full[bi]);
        } else {
          mbar_arrive(&S.full[bi]);
        }
        S.issued = k + 1;
        S.pend.slice += 1;
        more = S.pend.slice < S.pend.end ? 1 : 0;
      }
      more = __shfl_sync(FULLM, more, 0);
      __syncwarp();
      if (!have) return;
      if (!more) have = resolve(S.pend, tn);
    }
  }

  // Rows [0, R) of a slice by plain loads, every thread its own units.
  __device__ __forceinline__ void load_own(const FPass& P, int R, char* b, int tok0, int n) const {
    load_rows<DT>(P, R, b, tok0, n, p.T, p.V);
  }
  // The same for readers of other threads' units.
  __device__ void load_plain(const FPass& P, int R, char* b, int tok0, int n) const {
    load_own(P, R, b, tok0, n);
    cbar();
  }

  // One bit per 16-byte unit of the slice that holds a special token.
  __device__ void build_bitmap(const FPass& P, int tok0, int n) const {
    const int words = ((n + VE - 1) / VE + 31) / 32;
    for (int i = threadIdx.x; i < words; i += kCT) S.bitmap[i] = 0u;
    cbar();
    for (int i = threadIdx.x; i < P.nspec; i += kCT) {
      const int loc = P.spec_id[i] - tok0;
      if (loc >= 0 && loc < n) atomicOr(&S.bitmap[(loc / VE) >> 5], 1u << ((loc / VE) & 31));
    }
    cbar();
  }

  // -------------------------------------------------------------- block reductions (fixed order)
  // Sum over the compute threads: warp trees, then warps in order.  Every
  // compute thread gets the result.
  __device__ float block_sum(float v, float* scratch) const {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    v = warp_sum(v);
    cbar();
    if (lane == 0) scratch[warp] = v;
    cbar();
    float t = 0.f;
#pragma unroll
    for (int w = 0; w < kCW; ++w) t = __fadd_rn(t, scratch[w]);
    return t;
  }
  __device__ float block_max(float v, float* scratch) const {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    v = warp_max(v);
    cbar();
    if (lane == 0) scratch[warp] = v;
    cbar();
    float t = kNegInf;
#pragma unroll
    for (int w = 0; w < kCW; ++w) t = fmaxf(t, scratch[w]);
    return t;
  }

  // -------------------------------------------------------------- statistics of a slice, warp by warp
  // R rows (compile time) of a slice of at most 2048 / R units a row.  Every
  // thread keeps its units (u = thread, thread + 256, ...: the warps
  // interleave in chunks of 32 units) in registers and every warp works on
  // its own share, with its own exponent references:
  // the row maxima (packed), then the sums of 2^(l c - m c).  With LIST the
  // warp first sets aside the tokens whose target logit reaches a bound, the
  // p.kth-th largest of the maxima of the slice's 64 groups of four lanes (one
  // block barrier), and leaves them out of its sums.  p.kth is the slice's
  // list length and the maxima are distinct tokens, so none of the slice's
  // p.kth largest is missed; on independent logits 8.5 tokens a slice are set
  // aside for p.kth = 8, 18 for 16 and 44 for 32.  More than kWarpCand of them
  // in one warp (large logits next to each other): the same bound of the
  // warp's 64 half lanes (every lane's largest at the even and at the odd
  // places of its units); then the ties at the bound stay out, or, should that
  // not do, the bound rises to the lowest that leaves at most that many.
  // With RUNS (the bonus row) the chunks' sums are kept too.  The publishing
  // warp merges the eight warps' results.
  //
  // Against one pass by the whole block with five barriers and the publication
  // in it (GB300, a 32 KB slice of two rows): with a list 17k -> 4k SM cycles,
  // without 8k -> 2.7k; the publishing warp takes 4.5k beside it, and a CTA
  // turns a slice over about every 5.5k.
  template <int R, bool LIST, bool RUNS>
  __device__ __forceinline__ void stats_fast(const FPass& P, int bi, int tok0, int n, Slot& T) {
    char* b = buf(bi);
    constexpr int NU = (kFastUnits / R + kCT - 1) / kCT;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int U = (n + VE - 1) / VE;
    if (!p.bulk) load_own(P, R, b, tok0, n);
    uint4 x[R][NU];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int i = 0; i < NU; ++i) {
        const int u = i * kCT + tid;
        x[r][i] = (u < U) ? raw(b, r, u) : E::neg_inf();
      }
    float m[R];
    unsigned h0 = 0u, h1 = 0u;   // order keys of this lane's largest target logits at the units' even and odd places
#pragma unroll
    for (int r = 0; r < R; ++r) {
      uint4 mx = x[r][0];
#pragma unroll
      for (int i = 1; i < NU; ++i) mx = E::max4(mx, x[r][i]);
      const float2 lm = E::unit_max2(mx);
      if (LIST && r == 0) {
        h0 = lane_key(lm.x);
        h1 = lane_key(lm.y);
      }
      const unsigned km = __reduce_max_sync(FULLM, lane_key(fmaxf(lm.x, lm.y)));
      m[r] = km ? ord_val(km) : kNegInf;
    }
    if constexpr (LIST) {
      // 16-bit logits differ in the upper half of their keys only
      constexpr int kLow = DT == MDS_BF16 ? 16 : 0;
      // the largest key that p.kth of the lanes' pairs reach (0: fewer have a logit)
      auto kth_key = [&](unsigned k0, unsigned k1) {
        const unsigned hi = __reduce_max_sync(FULLM, max(k0, k1)), lo = __reduce_min_sync(FULLM, min(k0, k1));
        int bit = 31 - __clz(hi ^ lo);   // the keys share the bits above this one (-1: equal)
        unsigned t = bit < 31 ? hi & (FULLM << max(bit + 1, kLow)) : 0u;
#pragma unroll 1
        for (; bit >= kLow; --bit) {
          const unsigned c = t | (1u << bit);
          if (__popc(__ballot_sync(FULLM, k0 >= c)) + __popc(__ballot_sync(FULLM, k1 >= c)) >= p.kth) t = c;
        }
        return t;
      };
      {
        static_assert(kGroups == 8 && kCW * kGroups == 64, "four lanes a group, two groups a lane");
        unsigned g = max(h0, h1);
        g = max(g, __shfl_xor_sync(FULLM, g, 1));
        g = max(g, __shfl_xor_sync(FULLM, g, 2));
        if ((lane & 3) == 0) S.gmax[warp * kGroups + (lane >> 2)] = g;
      }
      cbar();   // the next slice's first barrier comes after this slice's reads
      unsigned th = kth_key(S.gmax[lane], S.gmax[lane + 32]);
      unsigned long long bits = 0ull;   // this lane's tokens that reach th, VE to a unit
      auto mark = [&](float theta) {
        unsigned um = 0u;   // units that hold one
#pragma unroll
        for (int i = 0; i < NU; ++i) um |= E::unit_max(x[0][i]) >= theta ? 1u << i : 0u;
        bits = 0ull;
        for (; um; um &= um - 1u) {
          const int i = __ffs(um) - 1;
          float v[VE];
          E::unpack(i * kCT + tid < U ? raw(b, 0, i * kCT + tid) : E::neg_inf(), v);
          unsigned bb = 0u;
#pragma unroll
          for (int e = 0; e < VE; ++e) bb |= (v[e] >= theta && v[e] > kNegInf) ? 1u << e : 0u;
          bits |= (unsigned long long)bb << (i * VE);
        }
        return (int)__reduce_add_sync(FULLM, (unsigned)__popcll(bits));
      };
      int tot = mark(th ? ord_val(th) : kNegInf);
      if (tot > kWarpCand) {
        // large logits next to each other: the bound of this warp's half lanes
        const unsigned own = kth_key(h0, h1);
        if (own > th) {
          th = own;
          tot = mark(ord_val(th));
        }
        // ties at the bound (flat rows, rows masked with a finite value) stay out
        if (tot > kWarpCand && th) tot = mark(ord_val(th + (1u << kLow)));
      }
      if (tot > kWarpCand) {
        // the largest key that more than kWarpCand tokens reach, and one up
        th = 0u;
#pragma unroll 1
        for (int bit = 31; bit >= kLow; --bit) {
          const unsigned cand = th | (1u << bit);
          unsigned c = 0u;
#pragma unroll 1
          for (int u = tid; u < U; u += kCT) {
            float v[VE];
            E::unpack(raw(b, 0, u), v);
#pragma unroll
            for (int e = 0; e < VE; ++e) c += (v[e] == v[e] && ord_key(__fadd_rn(v[e], 0.f)) >= cand) ? 1u : 0u;
          }
          if (__reduce_add_sync(FULLM, c) > (unsigned)kWarpCand) th = cand;
        }
        tot = mark(ord_val(th + (1u << kLow)));
      }
      if (lane == 0) T.nc[warp] = tot;
      // set aside: into the slot (lanes in order), and out of the slice (-inf
      // in every row; this thread's own units, read back into its registers)
      if (tot) {
        const int cnt = __popcll(bits);
        int pos = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int t = __shfl_up_sync(FULLM, pos, o);
          if (lane >= o) pos += t;
        }
        pos += warp * kWarpCand - cnt;
        for (unsigned long long q = bits; q; q &= q - 1ull) {
          const int at = __ffsll((long long)q) - 1;
          const int loc = ((at / VE) * kCT + tid) * VE + at % VE;
          T.loc[pos] = (unsigned short)loc;
#pragma unroll
          for (int rr = 0; rr < R; ++rr) {
            char* row = b + (size_t)rr * p.T * p.esize;
            T.l[rr][pos] = E::at(row, loc);
            E::clear(row, loc);
          }
          T.key[pos] = cand_key(T.l[0][pos], loc);
          ++pos;
        }
        asm volatile("" ::: "memory");
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
          for (int i = 0; i < NU; ++i)
            if ((unsigned)(bits >> (i * VE)) & ((1u << VE) - 1u)) x[r][i] = raw(b, r, i * kCT + tid);
      }
      fence_proxy_async();   // these stores before the next bulk copy into the buffer
    }
    // the slice is in registers: the buffer can be filled again (released at
    // the task's end, a 32 KB slice's loads waited 1.5 to 3 us for it)
    release(bi);
    if constexpr (LIST) {
      float tm = kNegInf;
#pragma unroll
      for (int i = 0; i < NU; ++i) tm = fmaxf(tm, E::unit_max(x[0][i]));
      const unsigned tk = __reduce_max_sync(FULLM, (tm > kNegInf) ? ord_key(tm) : 0u);
      if (lane == 0) T.tau[warp] = tk ? ord_val(tk) : kNegInf;
    }
    float s[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const float c = P.row[r].c;
      m[r] = sum_ref(m[r], c);
      const float mc = ref_exp(m[r], c);
      float acc = 0.f;
#pragma unroll
      for (int i = 0; i < NU; ++i) {
        if (i * kCT + warp * 32 >= U) break;   // warp-uniform
        float v[VE];
        E::unpack(x[r][i], v);
#pragma unroll
        for (int e = 0; e < VE; ++e) v[e] = ex2(__fmaf_rn(v[e], c, -mc));
        float t;
        if constexpr (VE == 8)
          t = __fadd_rn(__fadd_rn(__fadd_rn(v[0], v[1]), __fadd_rn(v[2], v[3])),
                        __fadd_rn(__fadd_rn(v[4], v[5]), __fadd_rn(v[6], v[7])));
        else
          t = __fadd_rn(__fadd_rn(v[0], v[1]), __fadd_rn(v[2], v[3]));
        if constexpr (RUNS) {
          const float w = warp_sum(t);
          if (lane == 0) T.run[i * kCW + warp] = w;
          acc = __fadd_rn(acc, w);
        } else {
          acc = __fadd_rn(acc, t);
        }
      }
      s[r] = acc;
    }
    if constexpr (!RUNS) {
#pragma unroll
      for (int r = 0; r < R; ++r) s[r] = warp_sum(s[r]);
    }
    if (lane == 0) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        T.m[warp][r] = m[r];
        T.s[warp][r] = s[r];
      }
    }
  }

  // -------------------------------------------------------------- stats task
  // Slices too small for the warp-wise path (fewer units than threads): R rows
  // (compile time, at most kListRowsMax) with the candidate list, by the whole
  // block in two passes over the slice in shared memory.  Pass A: every
  // row's maximum (the slice's exponent reference) and the candidate
  // threshold theta: the smallest of the warps' largest target logits, so
  // that at least one token per warp is >= theta (theta = -inf for a slice
  // of at most kCandCap tokens: every token is a candidate).  Pass B: every
  // row's sum of 2^(l c - m c) over the tokens that are not candidates (the
  // candidates, target logit > theta, are set aside with every row's logit).
  // Then the candidates are ranked (larger target logit first, ties to the
  // smaller id): the first LN form the slice's list, the others rejoin the
  // sums in rank order.  tau = the largest target logit outside the list.
  // Should more than kCandCap tokens pass theta, theta is raised to the
  // kCandCap-th largest target logit (bisection) and pass B repeated.
  // Record: (max, sum) per row, tau, list length, then the list: ids, then
  // each row's logits.
  template <int R>
  __device__ void stats_small(const FPass& P, const char* b, int tok0, int n, float* rec) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int U = (n + VE - 1) / VE;
    const int LN = p.lns;   // this slice's list length
    float c[R];
#pragma unroll
    for (int r = 0; r < R; ++r) c[r] = P.row[r].c;
    // pass A: maxima
    PT_T0(t_a);
    float tmax = kNegInf;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      float mx = kNegInf;
      for (int u = tid; u < U; u += kCT) mx = fmaxf(mx, E::unit_max(raw(b, r, u)));
      if (r == 0) tmax = mx;
      mx = warp_max(mx);
      if (lane == 0) S.red[warp * kMaxRows + r] = mx;
    }
    {
      // this warp's k-th largest thread maximum (distinct tokens), k = LN / kCW
      // rounded up: every warp then holds k tokens >= its value
      const int k = (LN + kCW - 1) / kCW;
      unsigned key = (tmax > kNegInf) ? ord_key(__fadd_rn(tmax, 0.f)) : 0u;
      unsigned km = 0u;
      for (int t = 0; t < k; ++t) {
        km = __reduce_max_sync(FULLM, key);
        if (!km) break;
        const unsigned who = __ballot_sync(FULLM, key == km);
        if (lane == __ffs(who) - 1) key = 0u;
      }
      if (lane == 0) S.wth[warp] = km ? ord_val(km) : kNegInf;
    }
    cbar();
    float m[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      float t = kNegInf;
#pragma unroll
      for (int w = 0; w < kCW; ++w) t = fmaxf(t, S.red[w * kMaxRows + r]);
      m[r] = sum_ref(t, c[r]);
    }
    // theta: the smallest of the warps' k-th largest thread maxima (warps
    // with fewer than k tokens left out), so at least LN tokens are >= theta
    // when every warp takes part; -inf (every token a candidate) for a slice
    // of at most kCandCap tokens
    float theta = kNegInf;
    {
      if (n > kCandCap) {
        theta = kPosInf;
#pragma unroll
        for (int w = 0; w < kCW; ++w) {
          const float wm = S.wth[w];
          if (wm > kNegInf) theta = fminf(theta, wm);
        }
        if (theta == kPosInf) theta = kNegInf;
      }
    }
    PT_ADD(kPhListA, t_a);
    PT_T0(t_b);
    float sm[R], tau;
    int nc = 0;
    for (int attempt = 0; attempt < 2; ++attempt) {
#pragma unroll
      for (int r = 0; r < R; ++r) sm[r] = 0.f;
      tau = kNegInf;
      for (int u = tid; u < U; u += kCT) {
        const uint4 x0 = raw(b, 0, u);
        float v0[VE];
        E::unpack(x0, v0);
        uint32_t cm = 0u;
        {
          const float um = E::unit_max(x0);
          if (um > theta) {
#pragma unroll
            for (int e = 0; e < VE; ++e) {
              if (v0[e] > theta)
                cm |= 1u << e;
              else
                tau = fmaxf(tau, v0[e]);
            }
            const int cnt = __popc(cm);
            const int pos = atomicAdd(&S.ncand, cnt);
            int q = pos;
#pragma unroll
            for (int e = 0; e < VE; ++e)
              if (cm >> e & 1u) {
                if (q < kCandCap) {
                  cid[q] = tok0 + u * VE + e;
                  cl[q] = v0[e];
                }
                ++q;
              }
          } else {
            tau = fmaxf(tau, um);
          }
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
          float v[VE];
          if (r == 0) {
#pragma unroll
            for (int e = 0; e < VE; ++e) v[e] = v0[e];
          } else {
            E::unpack(raw(b, r, u), v);
          }
          const float mc = ref_exp(m[r], c[r]);
          if (!cm) {
#pragma unroll
            for (int e = 0; e < VE; ++e) sm[r] = __fadd_rn(sm[r], ex2(__fmaf_rn(v[e], c[r], -mc)));
          } else {
#pragma unroll
            for (int e = 0; e < VE; ++e) {
              const float t = ex2(__fmaf_rn(v[e], c[r], -mc));
              sm[r] = __fadd_rn(sm[r], (cm >> e & 1u) ? 0.f : t);
            }
          }
        }
      }
      cbar();
      nc = S.ncand;
      if (nc <= kCandCap) break;
      // more than kCandCap tokens above theta: raise it to the kCandCap-th
      // largest target logit (bisection on order-preserving keys over every
      // bit: keys of negative logits use the low bits too) and repeat
      unsigned t = 0u;
      for (int bit = 31; bit >= 0; --bit) {
        const unsigned cand = t | (1u << bit);
        int cnt = 0;
        for (int u = tid; u < U; u += kCT) {
          float v[VE];
          E::unpack(raw(b, 0, u), v);
#pragma unroll
          for (int e = 0; e < VE; ++e) cnt += (v[e] == v[e] && ord_key(__fadd_rn(v[e], 0.f)) >= cand) ? 1 : 0;
        }
        cnt = __reduce_add_sync(FULLM, cnt);
        cbar();
        if (lane == 0) S.red[warp] = __int_as_float(cnt);
        cbar();
        int tot = 0;
#pragma unroll
        for (int w = 0; w < kCW; ++w) tot += __float_as_int(S.red[w]);
        if (tot >= kCandCap) t = cand;
      }
      theta = fmaxf(theta, ord_val(t));
      cbar();
      if (tid == 0) S.ncand = 0;
      cbar();
    }
    nc = min(nc, kCandCap);   // the bisection leaves fewer than kCandCap; never read past the arrays
    PT_ADD(kPhListB, t_b);
    PT_T0(t_c);
    // block sums of the rows (fixed order)
    float tot[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const float v = warp_sum(sm[r]);
      if (lane == 0) S.red[warp * kMaxRows + r] = v;
    }
    {
      tau = warp_max(tau);
      if (lane == 0) S.wth[warp] = tau;
    }
    cbar();
#pragma unroll
    for (int r = 0; r < R; ++r) {
      float t = 0.f;
#pragma unroll
      for (int w = 0; w < kCW; ++w) t = __fadd_rn(t, S.red[w * kMaxRows + r]);
      tot[r] = t;
    }
    {
      tau = kNegInf;
#pragma unroll
      for (int w = 0; w < kCW; ++w) tau = fmaxf(tau, S.wth[w]);
      // ranks; the first LN go to the record, the rest back to the sums
      for (int i = tid; i < nc; i += kCT) {
        const float li = cl[i];
        const int ii = cid[i];
        int rk = 0;
        for (int q = 0; q < nc; ++q) rk += better(cl[q], cid[q], li, ii) ? 1 : 0;
        crank[i] = rk;
        if (rk >= LN) cord[rk - LN] = i;
      }
      cbar();
      int* rid = reinterpret_cast<int*>(rec + kHdr);
      for (int i = tid; i < nc; i += kCT) {
        const int rk = crank[i];
        if (rk < LN) {
          const int id = cid[i];
          __stcg(rid + rk, id);
          __stcg(rec + kHdr + LN + rk, cl[i]);
#pragma unroll
          for (int r = 1; r < R; ++r) {
            float v[VE];
            const int loc = id - tok0;
            E::unpack(raw(b, r, loc / VE), v);
            float l = v[0];
#pragma unroll
            for (int e = 1; e < VE; ++e)
              if (e == loc % VE) l = v[e];
            __stcg(rec + kHdr + LN * (1 + r) + rk, l);
          }
        }
      }
      const int nd = nc - LN;
      if (nd > 0) {
        if (warp == 0) {
          float add[R];
#pragma unroll
          for (int r = 0; r < R; ++r) add[r] = 0.f;
          float at = kNegInf;
          for (int t = lane; t < nd; t += 32) {
            const int i = cord[t];
            const int loc = cid[i] - tok0;
            at = fmaxf(at, cl[i]);
#pragma unroll
            for (int r = 0; r < R; ++r) {
              float v[VE];
              E::unpack(raw(b, r, loc / VE), v);
              float l = v[0];
#pragma unroll
              for (int e = 1; e < VE; ++e)
                if (e == loc % VE) l = v[e];
              if (m[r] > kNegInf) add[r] = __fadd_rn(add[r], exp_term(l, m[r], c[r]));
            }
          }
#pragma unroll
          for (int r = 0; r < R; ++r) add[r] = warp_sum(add[r]);
          at = warp_max(at);
          if (lane == 0) {
#pragma unroll
            for (int r = 0; r < R; ++r) S.add[r] = add[r];
            S.addtau = at;
          }
        }
        cbar();
#pragma unroll
        for (int r = 0; r < R; ++r) tot[r] = __fadd_rn(tot[r], S.add[r]);
        tau = fmaxf(tau, S.addtau);
      }
    }
    if (tid == 0) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        __stcg(rec + 2 * r, m[r]);
        __stcg(rec + 2 * r + 1, tot[r]);
      }
      __stcg(rec + 2 * kMaxRows, tau);
      __stcg(reinterpret_cast<int*>(rec) + 2 * kMaxRows + 1, min(nc, LN));
      S.ncand = 0;   // for the next slice (every reader is past the barriers above)
    }
    PT_ADD(kPhListC, t_c);
  }

  // Stats of any number of rows, one row at a time, no candidate list.
  __device__ void stats_rows(const FPass& P, const char* b, int n, float* rec) {
    const int tid = threadIdx.x;
    const int U = (n + VE - 1) / VE;
    for (int r = 0; r < P.nstream; ++r) {
      float mx = kNegInf;
      for (int u = tid; u < U; u += kCT) mx = fmaxf(mx, E::unit_max(raw(b, r, u)));
      const float c = P.row[r].c;
      mx = sum_ref(block_max(mx, S.red), c);
      float sm = 0.f;
      const float mc = ref_exp(mx, c);
      for (int u = tid; u < U; u += kCT) {
        float v[VE];
        E::unpack(raw(b, r, u), v);
#pragma unroll
        for (int e = 0; e < VE; ++e) sm = __fadd_rn(sm, ex2(__fmaf_rn(v[e], c, -mc)));
      }
      sm = block_sum(sm, S.red + kCW);
      if (tid == 0) {
        __stcg(rec + 2 * r, mx);
        __stcg(rec + 2 * r + 1, sm);
      }
    }
  }

  // -------------------------------------------------------------- weights of the inverse-CDF draws
  // Residual max(0, q - p_I), p_I = sum_r gamma_r p_r with the special
  // tokens' explicit values, of one unit.
  __device__ __forceinline__ void weights(const FPass& P, const char* b, int u, int tok0, float* w) const {
    float v0[VE], a[VE];
    E::unpack(raw(b, 0, u), v0);
#pragma unroll
    for (int e = 0; e < VE; ++e) a[e] = 0.f;
    for (int r = 1; r < P.nstream; ++r) {
      const float g = P.row[r].gamma;
      if (g == 0.f) continue;
      float v[VE];
      E::unpack(raw(b, r, u), v);
      const float M = P.row[r].M, c = P.row[r].c, iz = P.row[r].invZ;
#pragma unroll
      for (int e = 0; e < VE; ++e) a[e] = __fmaf_rn(g, prob_of(v[e], M, c, iz), a[e]);
    }
    if (P.nspec > 0 && ((S.bitmap[u >> 5] >> (u & 31)) & 1u)) {
#pragma unroll
      for (int e = 0; e < VE; ++e) a[e] = spec_lookup(P, tok0 + u * VE + e, a[e]);
    }
    const float M0 = P.row[0].M, c0 = P.row[0].c, iz0 = P.row[0].invZ;
#pragma unroll
    for (int e = 0; e < VE; ++e) w[e] = fmaxf(0.f, __fsub_rn(prob_of(v0[e], M0, c0, iz0), a[e]));
  }

  // The masses of the slice's runs of 32 units, the runs the decision's
  // search walks, one warp a run (runs warp, warp + 8, ...): a unit's mass
  // adds its tokens in order, a run's its units by a butterfly.  Up to four
  // rows a thread's units are kept in registers (the buffer is released at
  // once) with the rows' constants.
  template <int R>
  __device__ __forceinline__ void resid_fast(const FPass& P, int bi, int tok0, int n, Slot& T) {
    constexpr int NU = (kFastUnits / R + kCT - 1) / kCT;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int U = (n + VE - 1) / VE;
    char* b = buf(bi);
    uint4 x[R][NU];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int i = 0; i < NU; ++i) {
        const int u = i * kCT + tid;
        x[r][i] = (u < U) ? raw(b, r, u) : E::neg_inf();
      }
    release(bi);
    if (P.kind == kResid && P.nspec > 0) build_bitmap(P, tok0, n);
    float mc[R], c[R], iz[R], gm[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      c[r] = P.row[r].c;
      mc[r] = __fmul_rn(P.row[r].M, c[r]);
      iz[r] = P.row[r].invZ;
      gm[r] = r ? P.row[r].gamma : 1.f;
    }
    const bool resid = P.kind == kResid, special = resid && P.nspec > 0;
    const bool none = P.kind == kReplace && P.all0;
    const float cut = P.kind == kReplace ? P.cut : kPosInf;
#pragma unroll
    for (int i = 0; i < NU; ++i) {
      if (i * kCT + warp * 32 >= U) break;   // warp-uniform
      const int u = i * kCT + tid;
      float q[VE], us = 0.f;
      E::unpack(x[0][i], q);
      if constexpr (R == 1) {
        // the target mass outside Omega_0 (kReplace)
#pragma unroll
        for (int e = 0; e < VE; ++e) {
          const float pq = __fmul_rn(ex2(__fmaf_rn(q[e], c[0], -mc[0])), iz[0]);
          us = __fadd_rn(us, (none || q[e] > cut) ? 0.f : pq);
        }
      } else {
        float a[VE];
#pragma unroll
        for (int e = 0; e < VE; ++e) a[e] = 0.f;
#pragma unroll
        for (int r = 1; r < R; ++r) {
          if (gm[r] == 0.f) continue;
          float v[VE];
          E::unpack(x[r][i], v);
#pragma unroll
          for (int e = 0; e < VE; ++e)
            a[e] = __fmaf_rn(gm[r], __fmul_rn(ex2(__fmaf_rn(v[e], c[r], -mc[r])), iz[r]), a[e]);
        }
        if (special && ((S.bitmap[u >> 5] >> (u & 31)) & 1u)) {
#pragma unroll
          for (int e = 0; e < VE; ++e) a[e] = spec_lookup(P, tok0 + u * VE + e, a[e]);
        }
#pragma unroll
        for (int e = 0; e < VE; ++e)
          us = __fadd_rn(us, fmaxf(0.f, __fsub_rn(__fmul_rn(ex2(__fmaf_rn(q[e], c[0], -mc[0])), iz[0]), a[e])));
      }
      us = warp_sum(us);
      if (lane == 0) T.run[i * kCW + warp] = us;
    }
  }
  // More rows than that.
  __device__ void resid_task(const FPass& P, const char* b, int tok0, int n, Slot& T) {
    if (P.kind == kResid && P.nspec > 0) build_bitmap(P, tok0, n);
    const int U = (n + VE - 1) / VE;
    const int tid = threadIdx.x, lane = tid & 31;
    for (int u = tid; u - lane < U; u += kCT) {
      float us = 0.f;
      if (u < U) {
        float w[VE];
        weights(P, b, u, tok0, w);
#pragma unroll
        for (int e = 0; e < VE; ++e) us = __fadd_rn(us, w[e]);
      }
      us = warp_sum(us);
      if (lane == 0) T.run[u >> 5] = us;
    }
  }

  // -------------------------------------------------------------- full-vocabulary stage task
  __device__ __forceinline__ static void cand_insert(Cand (&top)[kTopF], const Cand& c, float& ra, float& rb) {
    if (better(c.key, c.id, top[kTopF - 1].key, top[kTopF - 1].id)) {
      ra = __fadd_rn(ra, top[kTopF - 1].a);
      rb = __fadd_rn(rb, top[kTopF - 1].b);
      top[kTopF - 1] = c;
#pragma unroll
      for (int t = kTopF - 1; t > 0; --t) {
        if (better(top[t].key, top[t].id, top[t - 1].key, top[t - 1].id)) {
          const Cand x = top[t];
          top[t] = top[t - 1];
          top[t - 1] = x;
        }
      }
    } else {
      ra = __fadd_rn(ra, c.a);
      rb = __fadd_rn(rb, c.b);
    }
  }

  // Warp-wide merge of per-lane sorted lists (best first): lane 0 writes the
  // warp's best `rounds` entries to out[0..rounds) and CAND_NONE after them;
  // every entry not popped adds its a and b (fixed order) to rest_a / rest_b.
  __device__ static void warp_merge(Cand (&top)[kTopF], Cand* out, int rounds, float& rest_a, float& rest_b) {
    const int lane = threadIdx.x & 31;
#pragma unroll 1
    for (int t = 0; t < kTopF; ++t) {
      if (t >= rounds) {
        if (lane == 0) out[t] = CAND_NONE;
        continue;
      }
      float bk = top[0].key;
      int bid = top[0].id;
#pragma unroll
      for (int o = 16; o; o >>= 1) {
        const float ok = __shfl_xor_sync(FULLM, bk, o);
        const int oid = __shfl_xor_sync(FULLM, bid, o);
        if (better(ok, oid, bk, bid)) {
          bk = ok;
          bid = oid;
        }
      }
      const bool mine = (top[0].id == bid && top[0].key == bk && bid != 0x7fffffff);
      const unsigned who = __ballot_sync(FULLM, mine);
      const int src = who ? __ffs(who) - 1 : 0;
      const float wa = __shfl_sync(FULLM, top[0].a, src);
      const float wb = __shfl_sync(FULLM, top[0].b, src);
      if (mine) {
#pragma unroll
        for (int i = 0; i < kTopF - 1; ++i) top[i] = top[i + 1];
        top[kTopF - 1] = CAND_NONE;
      }
      if (lane == 0) out[t] = who ? Cand{bk, bid, wa, wb} : CAND_NONE;
    }
    float ra = 0.f, rb = 0.f;
#pragma unroll
    for (int i = 0; i < kTopF; ++i) {
      ra = __fadd_rn(ra, top[i].a);
      rb = __fadd_rn(rb, top[i].b);
    }
    rest_a = warp_sum(ra);
    rest_b = warp_sum(rb);
  }

  // Record: [0] a-mass and [1] b-mass of the slice outside its top s, [4..)
  // the top s (key, id, a, b) as four arrays of kTopF.
  __device__ void full_task(const FPass& P, const char* b, int tok0, int n, float* rec) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int s = min(p.wis_s, p.V);
    const int rb = P.rb;
    if (P.nspec > 0) build_bitmap(P, tok0, n);
    Cand top[kTopF];
#pragma unroll
    for (int t = 0; t < kTopF; ++t) top[t] = CAND_NONE;
    float suma = 0.f, sumb = 0.f;
    const int U = (n + VE - 1) / VE;
    const float M0 = P.row[0].M, c0 = P.row[0].c, iz0 = P.row[0].invZ;
    for (int u = tid; u < U; u += kCT) {
      float v0[VE], a[VE], bb[VE];
      E::unpack(raw(b, 0, u), v0);
#pragma unroll
      for (int e = 0; e < VE; ++e) {
        a[e] = 0.f;
        bb[e] = 0.f;
      }
      for (int r = 1; r < P.nstream; ++r) {
        const float g = P.row[r].gamma;
        if (g == 0.f && r != rb) continue;
        float v[VE];
        E::unpack(raw(b, r, u), v);
        const float M = P.row[r].M, c = P.row[r].c, iz = P.row[r].invZ;
#pragma unroll
        for (int e = 0; e < VE; ++e) {
          const float pr = prob_of(v[e], M, c, iz);
          if (g != 0.f) a[e] = __fmaf_rn(g, pr, a[e]);
          if (r == rb) bb[e] = pr;
        }
      }
      if (P.nspec > 0 && ((S.bitmap[u >> 5] >> (u & 31)) & 1u)) {
#pragma unroll
        for (int e = 0; e < VE; ++e) a[e] = spec_lookup(P, tok0 + u * VE + e, a[e]);
      }
#pragma unroll
      for (int e = 0; e < VE; ++e) {
        if (u * VE + e >= n) break;
        const float q = prob_of(v0[e], M0, c0, iz0);
        cand_insert(top, Cand{__fmaf_rn(-a[e], bb[e], q), tok0 + u * VE + e, a[e], bb[e]}, suma, sumb);
      }
    }
    {
      float ra, rbs;
      warp_merge(top, S.wcand + warp * kTopF, s, ra, rbs);
      suma = warp_sum(suma);
      sumb = warp_sum(sumb);
      if (lane == 0) {
        S.red[warp * 2] = __fadd_rn(suma, ra);
        S.red[warp * 2 + 1] = __fadd_rn(sumb, rbs);
      }
    }
    cbar();
    if (warp == 0) {
#pragma unroll
      for (int t = 0; t < kTopF; ++t) top[t] = (lane < kCW) ? S.wcand[lane * kTopF + t] : CAND_NONE;
      float ra, rbs;
      warp_merge(top, S.blk, s, ra, rbs);
      __syncwarp();
      if (lane == 0) {
        float sa = ra, sb = rbs;
        for (int w = 0; w < kCW; ++w) {
          sa = __fadd_rn(sa, S.red[w * 2]);
          sb = __fadd_rn(sb, S.red[w * 2 + 1]);
        }
        __stcg(rec + 0, sa);
        __stcg(rec + 1, sb);
      }
      if (lane < kTopF) {
        __stcg(rec + 4 + lane, S.blk[lane].key);
        __stcg(reinterpret_cast<int*>(rec) + 4 + kTopF + lane, S.blk[lane].id);
        __stcg(rec + 4 + 2 * kTopF + lane, S.blk[lane].a);
        __stcg(rec + 4 + 3 * kTopF + lane, S.blk[lane].b);
      }
    }
  }

  // -------------------------------------------------------------- the publishing warp
  // Merges the compute warps' results of one slice into its record and counts
  // the pass's slices; the warp that counts a pass's last slice posts the
  // decision request.  The compute warps are meanwhile on later slices: the
  // record's stores, the fence and the counter's round trip (about 3 us) cost
  // them nothing.  A group of slices is counted once, at its end.
  //
  // Rows: the slice maximum and the warps' sums moved to it, warps in order.
  __device__ void merge_rows(const Slot& T, float (&m)[kListRowsMax], float (&s)[kListRowsMax]) const {
    const int lane = threadIdx.x & 31;
    const int w = lane & 7;
#pragma unroll
    for (int r = 0; r < kListRowsMax; ++r) {
      m[r] = kNegInf;
      s[r] = 0.f;
      if (r >= T.R) continue;
      const float mw = T.m[w][r], sw = T.s[w][r];
      float mm = mw;
#pragma unroll
      for (int o = 4; o; o >>= 1) mm = fmaxf(mm, __shfl_xor_sync(FULLM, mm, o));
      float v = moved_sum(sw, mw, mm, T.c[r]);
#pragma unroll
      for (int o = 4; o; o >>= 1) v = __fadd_rn(v, __shfl_xor_sync(FULLM, v, o));
      m[r] = mm;
      s[r] = v;
    }
  }
  // Order key of a lane's largest logit, 0 for none.
  __device__ __forceinline__ static unsigned lane_key(float m) {
    return m > kNegInf ? ord_key(__fadd_rn(m, 0.f)) : 0u;
  }
  // Rank key of a token set aside: larger first.  A 16-bit logit's key needs
  // 16 bits, so the place in the slice (below 65536, smaller first) fits
  // beside it and the keys are distinct; 32-bit logits tie by place apart.
  __device__ __forceinline__ static unsigned cand_key(float l, int loc) {
    const unsigned k = ord_key(__fadd_rn(l, 0.f));
    return DT == MDS_BF16 ? ((k & 0xffff0000u) | (0xffffu - (unsigned)loc)) : k;
  }

  // The slice's list: the first LN of the tokens set aside, by target logit
  // (ties: smaller id), with every row's logit; the others rejoin the sums,
  // tau covers them and every token not set aside.  The tokens are numbered
  // warp by warp; more than kRankMax of them are first cut to LN by their keys.
  __device__ void merge_list(Slot& T, float* rec, const float (&m)[kListRowsMax], float (&s)[kListRowsMax]) const {
    const int lane = threadIdx.x & 31;
    const int LN = p.lns;
    float tau = (lane < kCW) ? T.tau[lane] : kNegInf;
    const Numbers num(T);
    auto entry = [&](int j) { return num.entry(j); };
    float add[kListRowsMax];
#pragma unroll
    for (int r = 0; r < kListRowsMax; ++r) add[r] = 0.f;
    auto rejoin = [&](int i) {
      tau = fmaxf(tau, T.l[0][i]);
#pragma unroll
      for (int r = 0; r < kListRowsMax; ++r)
        if (r < T.R && m[r] > kNegInf) add[r] = __fadd_rn(add[r], exp_term(T.l[r][i], m[r], T.c[r]));
    };
    int n = num.first[kCW];
    if (n <= kRankMax) {
#pragma unroll
      for (int h = 0; h < kRankMax / 32; ++h) {
        const int j = lane + 32 * h;
        const int i = j < n ? entry(j) : 0;
        T.sel[j] = j < n ? T.key[i] : 0u;
        T.at[j] = (unsigned short)i;
      }
    } else {
      const uint2 cut = list_cut<DT>(T, n, LN);
      const unsigned thr = cut.x, last = cut.y;
      int base = 0;
#pragma unroll 1
      for (int j0 = 0; j0 < n; j0 += 32) {
        const int j = j0 + lane, i = j < n ? entry(j) : 0;
        const unsigned key = j < n ? T.key[i] : 0u;
        const bool take = j < n && (key > thr || (key == thr && T.loc[i] <= last));
        const unsigned mk = __ballot_sync(FULLM, take);
        if (take) {
          const int at = base + __popc(mk & ((1u << lane) - 1u));
          T.sel[at] = key;
          T.at[at] = (unsigned short)i;
        } else if (j < n) {
          rejoin(i);
        }
        base += __popc(mk);
      }
      n = base;   // LN
      T.sel[n + lane] = 0u;
    }
    __syncwarp();
    int* rid = reinterpret_cast<int*>(rec + kHdr);
#pragma unroll 1
    for (int j = lane; j < n; j += 32) {
      const unsigned kj = T.sel[j];
      const int i = T.at[j], place = T.loc[i];
      int rk = 0;
#pragma unroll 4
      for (int q = 0; q < n; q += 4) {
        const uint4 o = *reinterpret_cast<const uint4*>(T.sel + q);
        rk += (o.x > kj ? 1 : 0) + (o.y > kj ? 1 : 0) + (o.z > kj ? 1 : 0) + (o.w > kj ? 1 : 0);
      }
      if constexpr (DT != MDS_BF16)
        for (int q = 0; q < n; ++q) rk += (T.sel[q] == kj && T.loc[T.at[q]] < place) ? 1 : 0;
      if (rk < LN) {
        __stcg(rid + rk, T.slice * p.T + place);
#pragma unroll
        for (int r = 0; r < kListRowsMax; ++r)
          if (r < T.R) __stcg(rec + kHdr + LN * (1 + r) + rk, T.l[r][i]);
      } else {
        rejoin(i);
      }
    }
    __syncwarp();
    tau = warp_max(tau);
#pragma unroll
    for (int r = 0; r < kListRowsMax; ++r)
      if (r < T.R) s[r] = __fadd_rn(s[r], warp_sum(add[r]));
    if (lane == 0) {
      __stcg(rec + 2 * kMaxRows, tau);
      __stcg(reinterpret_cast<int*>(rec) + 2 * kMaxRows + 1, min(n, LN));
    }
  }

  __device__ void publisher() {
    const int lane = threadIdx.x & 31;
    for (int k = 0;; ++k) {
      Slot& T = slots[k % kSlots];
      if (!__all_sync(FULLM, wait_mbar(&S.done[k % kSlots], (k / kSlots) & 1))) {
        if (lane == 0) set_abort(MDS_ST_TIMEOUT);
        return;
      }
      const int mode = T.mode;
      if (mode == kSlotExit) return;
      const int b = T.b, s = T.slice;
      float* rec = p.rec + ((size_t)b * p.ns + s) * p.rec_floats;
      PT_T0(t_pub);
      if (mode == kSlotSums || mode == kSlotList || mode == kSlotBonus) {
        float m[kListRowsMax], sm[kListRowsMax];
        merge_rows(T, m, sm);
        if (mode == kSlotList) merge_list(T, rec, m, sm);
        if (mode == kSlotBonus) {
          // the chunks' sums, each against its warp's reference, moved to the slice's
          for (int q = lane; q < T.nrun; q += 32) {
            const float mw = T.m[q & (kCW - 1)][0];
            __stcg(rec + 4 + q, moved_sum(T.run[q], mw, m[0], T.c[0]));
          }
        }
        if (lane == 0) {
#pragma unroll
          for (int r = 0; r < kListRowsMax; ++r)
            if (r < T.R) {
              __stcg(rec + 2 * r, m[r]);
              __stcg(rec + 2 * r + 1, sm[r]);
            }
        }
      } else if (mode == kSlotRuns) {
        // run masses, and the slice's: the runs in chunks of 32
        float tot = 0.f;
        for (int q0 = 0; q0 < T.nrun; q0 += 32) {
          const int q = q0 + lane;
          const float v = q < T.nrun ? T.run[q] : 0.f;
          if (q < T.nrun) __stcg(rec + 4 + q, v);
          tot = __fadd_rn(tot, warp_sum(v));
        }
        if (lane == 0) __stcg(rec, tot);
      }
      const int kind = T.kind, j = T.j;
      if (kind == kStats && j == 0 && s == 0) {
        // the sequence's outputs start as -1 (the decisions overwrite them)
        for (int q = lane; q <= p.L; q += 32) __stcg(p.out_tokens + (size_t)b * (p.L + 1) + q, -1);
        if (lane == 0) __stcg(p.out_accept + b, -1);
      }
      __syncwarp();
      const int count = T.count;
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(&S.free[k % kSlots]);
        // the group's records before the count (release; the last one also acquires the others')
        if (count && atom_add_acq_rel(&p.cnt[b], (unsigned)count) == (unsigned)(p.ns - count))
          post_decision(dec_payload(b, j, kind == kStats && j == 0));
      }
      PT_ADDW(kPhPublish, t_pub);
      __syncwarp();
    }
  }

  // -------------------------------------------------------------- compute warps
  // The pass of a sequence is complete: publish a decision request (one
  // thread, after acquiring every slice's record through the pass counter;
  // the release of the request's tag passes them on to the decision warp).
  __device__ void post_decision(unsigned pay) const {
    const unsigned t = atomicAdd(&p.ctl[kCtlDecTail], 1u);
    const unsigned slot = t % (unsigned)p.dec_cap, lap = t / (unsigned)p.dec_cap;
    if (lap) {
      const unsigned long long prev = ring_word(p.epoch, lap - 1u, 0u);
      const unsigned long long t0 = now_ns();
      for (int it = 0; ld_acquire(&p.dec_rtag[slot]) != prev; ++it) {
        if (aborted()) break;
        if ((it & 15) == 15 && now_ns() - t0 > kWaitNs) {
          set_abort(MDS_ST_TIMEOUT);
          break;
        }
        __nanosleep(64);
      }
    }
    st_release(&p.dec_tag[slot], ring_word(p.epoch, lap, pay));
  }

  // One slice: this warp's part of the results into T, or (slices too small
  // for the warp-wise paths, more rows than they take, full stages) the whole
  // record into global memory.  Thread 0 fills T's description.
  __device__ void process(int bi, const FDesc& Dd, Slot& T) {
    char* b = buf(bi);
    const int s = Dd.slice, seqb = Dd.b;
    const int tok0 = s * p.T, n = min(p.T, p.V - tok0);
    const FPass& P = Dd.P;
    float* rec = p.rec + ((size_t)seqb * p.ns + s) * p.rec_floats;
    PT_T0(t_task);
    PT_CNT(kPhTasks);
    int mode = kSlotDone;
    const int U = (n + VE - 1) / VE;
    switch (P.kind) {
      case kBonus:
        mode = kSlotBonus;
        stats_fast<1, false, true>(P, bi, tok0, n, T);
        break;
      case kStats:
        if (P.list && p.fast_list) {
          mode = kSlotList;
          switch (P.nstream) {
            case 1: stats_fast<1, true, false>(P, bi, tok0, n, T); break;
            case 2: stats_fast<2, true, false>(P, bi, tok0, n, T); break;
            case 3: stats_fast<3, true, false>(P, bi, tok0, n, T); break;
            default: stats_fast<4, true, false>(P, bi, tok0, n, T); break;
          }
        } else if (P.list) {
          if (!p.bulk) load_plain(P, P.nstream, b, tok0, n);
          switch (P.nstream) {
            case 1: stats_small<1>(P, b, tok0, n, rec); break;
            case 2: stats_small<2>(P, b, tok0, n, rec); break;
            case 3: stats_small<3>(P, b, tok0, n, rec); break;
            default: stats_small<4>(P, b, tok0, n, rec); break;
          }
          release(bi);
        } else {
          switch (P.nstream) {
            case 1:
              mode = kSlotSums;
              stats_fast<1, false, false>(P, bi, tok0, n, T);
              break;
            case 2:
              mode = kSlotSums;
              stats_fast<2, false, false>(P, bi, tok0, n, T);
              break;
            default:
              if (!p.bulk) load_plain(P, P.nstream, b, tok0, n);
              stats_rows(P, b, n, rec);
              release(bi);
              break;
          }
        }
        break;
      case kResid:
      case kReplace:
        mode = kSlotRuns;
        if (!p.bulk) load_own(P, P.nstream, b, tok0, n);
        switch (P.nstream) {
          case 1: resid_fast<1>(P, bi, tok0, n, T); break;
          case 2: resid_fast<2>(P, bi, tok0, n, T); break;
          case 3: resid_fast<3>(P, bi, tok0, n, T); break;
          case 4: resid_fast<4>(P, bi, tok0, n, T); break;
          default:
            resid_task(P, b, tok0, n, T);
            release(bi);
            break;
        }
        break;
      case kFull:
        if (!p.bulk) load_plain(P, P.nstream, b, tok0, n);
        full_task(P, b, tok0, n, rec);
        release(bi);
        break;
      default: release(bi); break;
    }
    PT_ADD(P.kind == kStats ? (P.list ? kPhTaskList : kPhTaskStats)
                            : (P.kind == kBonus ? kPhTaskStats : (P.kind == kFull ? kPhTaskFull : kPhTaskResid)),
           t_task);
    if (threadIdx.x == 0) {
      T.mode = mode;
      T.b = seqb;
      T.slice = s;
      T.kind = P.kind;
      T.j = P.j;
      T.R = P.nstream;
      T.nrun = (U + 31) / 32;
      T.count = (s + 1 == Dd.end) ? s + 1 - Dd.first : 0;
    }
    if (threadIdx.x < kListRowsMax) T.c[threadIdx.x] = P.row[threadIdx.x].c;
  }

  __device__ void compute() {
    const int lane = threadIdx.x & 31;
    for (int k = 0;; ++k) {
      const int bi = k % kNBuf, sl = k % kSlots;
      // thread 0 waits for the slice and for a free record slot (bounded);
      // the others then see the completed phases
      PT_T0(t_wait);
      if (threadIdx.x == 0) {
        bool ok = wait_mbar(&S.full[bi], (k / kNBuf) & 1);
        if (ok) S.consumed = k + 1;
        if (ok && k >= kSlots) ok = wait_mbar(&S.free[sl], ((k / kSlots) - 1) & 1);
        if (!ok) set_abort(MDS_ST_TIMEOUT);
        S.flag_ok[k & 1] = ok ? 1 : 0;
      }
      cbar();
      PT_ADD(kPhWaitFull, t_wait);
      if (!S.flag_ok[k & 1]) return;   // the publishing warp's own wait runs out
      while (!mbar_try_wait(&S.full[bi], (k / kNBuf) & 1)) {
      }
      const FDesc& Dd = S.desc[k % kNDesc];
      if (Dd.exit) {
        if (threadIdx.x == 0) slots[sl].mode = kSlotExit;
        __syncwarp();
        if (lane == 0) mbar_arrive(&S.done[sl]);
        return;
      }
      process(bi, Dd, slots[sl]);
      // this warp is done with its part of the record
      __syncwarp();
      if (lane == 0) mbar_arrive(&S.done[sl]);
    }
  }

};

// ================================================================== decisions
// One decision warp (on a decision SM) runs one sequence's decision at a
// time: the records of the pass just completed, the importance step, the
// accept test and the inverse-CDF search, then the sequence's next pass.
// Single-warp code throughout (lane 0 for the serial steps); its state and
// scratch are this warp's own shared memory.

constexpr int kDecScratch = kDecStage + 2 * kMaxSlices * 4 + 64 * 4;   // + slice masses, maxima, bitmap

// Each kind of decision out of line (its own register allocation); each
// rebuilds the warp's view of its shared state.
template <int DT> __device__ __noinline__ void dec_stats_nl(int b, int j);
template <int DT> __device__ __noinline__ void dec_resid_nl(int b);
template <int DT> __device__ __noinline__ void dec_replace_nl(int b);
template <int DT> __device__ __noinline__ void dec_full_nl(int b);
template <int DT> __device__ __noinline__ void dec_bonus_nl(int b);
template <int DT> __device__ __noinline__ void dec_wis0_nl(int b);
template <int DT> __device__ __noinline__ void dec_accept_nl(int b);
__device__ __noinline__ int lp_solve8(int s, float A2, float B2, int A, int Btok, float u);

template <int DT>
struct Dec {
  using E = Elt<DT>;
  static constexpr int VE = E::VE;

  const Params& p;
  FShared& S;      // the CTA's shared state (phase timers)
  DState& D;       // this warp's decision state
  char* scr;       // this warp's scratch: staged records
  float* Rs;       // slice masses of a search [kMaxSlices]
  float* Hm;       // slice maxima of the bonus draw [kMaxSlices]
  uint32_t* bm;    // special-token bits of a re-read slice [64]
  int lane;

  __device__ __forceinline__ bool aborted() const { return ld_relaxed(&p.ctl[kCtlAbort]) != 0u; }
  __device__ __forceinline__ void set_abort(unsigned bits) const {
    atomicOr(p.status, bits);
    atomicExch(&p.ctl[kCtlAbort], 1u);
  }

  // -------------------------------------------------------------- point values
  __device__ __forceinline__ float logit_at(const FPass& P, int r, int x) const {
    if (D.xl_ok)
      for (int k = 0; k < D.nv; ++k)
        if (D.X[k] == x) return D.xl[k][r];
    return E::global(P.row[r].ptr, x);
  }
  __device__ __forceinline__ float prob_row(const FPass& P, int r, int x) const {
    return prob_of(logit_at(P, r, x), P.row[r].M, P.row[r].c, P.row[r].invZ);
  }
  __device__ __forceinline__ float spec_lookup(const FPass& P, int tok, float fallback) const {
    for (int i = 0; i < P.nspec; ++i)
      if (P.spec_id[i] == tok) return P.spec_val[i];
    return fallback;
  }
  // Point value of the current law p_I (WIS): explicit value of a special
  // token, else sum_r gamma_r p_r(x) in row order.
  __device__ float law_at(const FPass& P, int x) const {
    float a = 0.f;
    for (int r = 1; r < P.nrows; ++r)
      if (P.row[r].gamma != 0.f) a = __fmaf_rn(P.row[r].gamma, prob_row(P, r, x), a);
    return spec_lookup(P, x, a);
  }

  // -------------------------------------------------------------- planning
  // Rows of depth j for the valid branches (the lowest valid branch's target
  // row, then one row per distinct draft model in branch order), one lane per
  // branch; the valid branches, their tokens (tk: the staged tokens of depth
  // j) and rows; with want_xl, every row's logit at each draft token, by
  // asynchronous copies that xl_sync completes.
  __device__ void plan_warp(int b, int j, unsigned valid, bool bonus, bool set_pass, bool want_xl, const int* tk) {
    FPass& P = D.P;
    const int K = p.K;
    const bool v = !bonus && lane < K && ((valid >> lane) & 1u);
    const int m = v ? (int)p.model_of[lane] : 64 + lane;
    const unsigned same = __match_any_sync(FULLM, m);
    const bool first = v && (__ffs(same) - 1) == lane;
    const unsigned fm = __ballot_sync(FULLM, first);
    const unsigned vm = __ballot_sync(FULLM, v);
    const int nr = 1 + __popc(fm);
    const int myrow = first ? 1 + __popc(fm & ((1u << lane) - 1u)) : 0;
    const int row = __shfl_sync(FULLM, myrow, __ffs(same) - 1);
    if (v) {
      const int i = __popc(vm & ((1u << lane) - 1u));
      int x = tk[lane];
      if (x < 0 || x >= p.V) {
        atomicOr(p.status, MDS_ST_BADTOKEN);
        x = 0;
      }
      D.vbr[i] = lane;
      D.X[i] = x;
      D.vrow[i] = row;
    }
    if (set_pass && first) {
      P.row[myrow].ptr = p.drafts[lane] + (((size_t)b * p.L + j) * (size_t)p.V) * p.esize;
      float td = D.tmp[1 + lane];
      if (!(td > 0.f) || !(td < kPosInf)) {
        atomicOr(p.status, MDS_ST_BADTEMP);
        td = 1.f;
      }
      P.row[myrow].c = __fdiv_rn(kLog2e, td);
      P.row[myrow].M = 0.f;
      P.row[myrow].invZ = 0.f;
      P.row[myrow].gamma = 0.f;
    }
    if (lane == 0) {
      D.nv = __popc(vm);
      if (set_pass) {
        const int kstar = __ffs(valid) - 1;
        P.row[0].ptr = p.target + ((((size_t)b * K + kstar) * (p.L + 1) + j) * (size_t)p.V) * p.esize;
        float tq = D.tmp[0];
        if (!(tq > 0.f) || !(tq < kPosInf)) {
          atomicOr(p.status, MDS_ST_BADTEMP);
          tq = 1.f;
        }
        P.row[0].c = __fdiv_rn(kLog2e, tq);
        P.row[0].M = 0.f;
        P.row[0].invZ = 0.f;
        P.row[0].gamma = 0.f;
        P.nrows = nr;
        P.j = j;
        P.nspec = 0;
        P.rb = 0;
        P.cut = 0.f;
        P.all0 = 0;
        if (bonus) {
          P.kind = kBonus;
          P.nstream = 1;
          P.list = 0;
        } else {
          P.kind = kStats;
          if (p.scheme == MDS_WIS0) {
            P.nstream = 1;
            P.list = 1;
          } else if (p.scheme == MDS_WIS) {
            P.nstream = nr;
            P.list = (__popc(vm) > 1 && nr <= kListRowsMax && p.ln > 0) ? 1 : 0;
          } else {
            P.nstream = min(2, nr);
            P.list = 0;
          }
        }
      }
    }
    if (lane == 0) {
      D.xl_ok = 0;
      D.xl_wait = 0;
    }
    __syncwarp();
    if (want_xl && !bonus) {
      const int nv = D.nv, nrow = P.nrows;
      for (int i = lane; i < nv * nrow; i += 32) {
        const int k = i / nrow, r = i - k * nrow;
        const char* at = P.row[r].ptr + (size_t)D.X[k] * p.esize;
        if (p.bulk)
          cpa4(&D.xl[k][r], reinterpret_cast<const char*>(reinterpret_cast<uintptr_t>(at) & ~uintptr_t(3)));
        else
          D.xl[k][r] = E::global(P.row[r].ptr, D.X[k]);
      }
      if (lane == 0) D.xl_wait = 1;
      __syncwarp();
    }
  }

  // Complete plan_warp's copies of the row logits at the draft tokens (the
  // 4-byte word holding a 16-bit logit is copied, its half taken here).
  // Warp-wide; afterwards logit_at answers those points from the cache.
  __device__ void xl_sync() {
    if (!D.xl_wait) return;
    cpa_wait();
    __syncwarp();
    if (p.bulk) {
      const int nv = D.nv, nrow = D.P.nrows;
      for (int i = lane; i < nv * nrow; i += 32) {
        const int k = i / nrow, r = i - k * nrow;
        if constexpr (DT == MDS_BF16) {
          const uint32_t w = __float_as_uint(D.xl[k][r]);
          const uintptr_t at = reinterpret_cast<uintptr_t>(D.P.row[r].ptr) + (uintptr_t)D.X[k] * 2u;
          D.xl[k][r] = __uint_as_float((at & 2u) ? (w & 0xffff0000u) : (w << 16));
        }
      }
    }
    __syncwarp();
    if (lane == 0) {
      D.xl_wait = 0;
      D.xl_ok = 1;
    }
    __syncwarp();
  }

  // -------------------------------------------------------------- publishing
  __device__ void push(int b, int kind) {
    PT_T0(t_push);
    unsigned base = 0u;
    if (lane == 0) {
      // ring numbers first: their round trip runs beside the state's stores
      base = (unsigned)p.B * (unsigned)p.ng0 + atomicAdd(&p.ctl[kCtlTail], (unsigned)p.ng);
      D.P.kind = kind;
    }
    __syncwarp();
    FSeq* g = &reinterpret_cast<FSeq*>(p.seq)[b];
    copy_out(&g->P, &D.P, (int)sizeof(FPass), lane, 32);
    copy_out(&g->W, &D.W, (int)sizeof(FWalk), lane, 32);
    if (lane == 0) __stcg(p.cnt + b, 0u);
    base = __shfl_sync(FULLM, base, 0);
    for (int i0 = 0; i0 < p.ng; i0 += 32) {
      const int i = i0 + lane;
      const unsigned t = base + (unsigned)i;
      const unsigned slot = t % (unsigned)p.ring_cap, lap = t / (unsigned)p.ring_cap;
      if (i < p.ng && lap) {
        // the slot's previous task must have been taken
        const unsigned long long prev = ring_word(p.epoch, lap - 1u, 0u);
        const unsigned long long t0 = now_ns();
        for (int it = 0; ld_acquire(&p.ring_rtag[slot]) != prev; ++it) {
          if (aborted()) break;
          if ((it & 15) == 15 && now_ns() - t0 > kWaitNs) {
            set_abort(MDS_ST_TIMEOUT);
            break;
          }
          __nanosleep(64);
        }
      }
      // every lane's state stores (joined by the warp barrier) before any publication
      __syncwarp();
      __threadfence();
      if (i < p.ng) st_relaxed(&p.ring_tag[slot], ring_word(p.epoch, lap, ((unsigned)b << 8) | (unsigned)i));
    }
    __syncwarp();
    PT_ADDW(kPhPush, t_push);
  }

  __device__ void finish(int b, int acc_len) {
    if (lane == 0) {
      __stcg(p.out_accept + b, acc_len);
      __stcg(p.cnt + b, 0u);
      __threadfence();
      atomicAdd(&p.ctl[kCtlDone], 1u);
    }
    __syncwarp();
  }

  // Z decided at the current depth: outputs, then the next depth's pass,
  // the bonus pass, or the end of the sequence.
  __device__ void walk(int b, int Z, float R, float qY, float pIY, int Ydiag) {
    const int j = D.P.j;
    PT_T0(t_walk);
    __syncwarp();
    int next = kNone;
    if (lane == 0) {
      __stcg(p.out_tokens + (size_t)b * (p.L + 1) + j, Z);
      if (p.out_diag) {
        float* dg = p.out_diag + ((size_t)b * (p.L + 1) + j) * 4;
        __stcg(dg + 0, qY);
        __stcg(dg + 1, pIY);
        __stcg(dg + 2, R);
        __stcg(dg + 3, (float)Ydiag);
      }
      unsigned nv = 0u;
      for (int i = 0; i < D.nv; ++i)
        if (D.X[i] == Z) nv |= 1u << D.vbr[i];
      D.W.valid = nv;
      next = nv ? ((j + 1 == p.L) ? kBonus : kStats) : kNone;
      if (nv) {
        D.W.stage = 0;
        D.W.zres = 0;
      }
    }
    next = __shfl_sync(FULLM, next, 0);
    __syncwarp();
    // the next depth's pass, planned from the staged tokens of depth j + 1
    if (next != kNone) plan_warp(b, j + 1, D.W.valid, next == kBonus, true, false, D.tk1);
    if (next == kNone)
      finish(b, j);
    else
      push(b, next);
    PT_ADDW(kPhDecWalk, t_walk);
  }

  // -------------------------------------------------------------- stats decision
  // The records of a stats pass into the scratch: per row the slice maxima
  // and sums, and with lists each slice's tau, list length and entries.
  __device__ void finish_row(int r, float Z) {
    if (!(Z > 0.f) || !(Z < kPosInf) || Z != Z) {
      atomicOr(p.status, MDS_ST_NONFINITE);
      Z = 1.f;
    }
    D.P.row[r].invZ = __frcp_rn(Z);
  }

  // Test export: the statistics of the depth's rows (M, 1/Z, c, source:
  // the target row's branch, or 100 + the branch whose draft row it is).
  __device__ void debug_rows(int b, int j, int R) const {
    for (int r = lane; r < R && r < MDS_DEBUG_ROWS; r += 32) {
      int src = __ffs(D.W.valid) - 1;
      if (r > 0) {
        src = -1;
        for (int i = 0; i < D.nv; ++i)
          if (D.vrow[i] == r) {
            src = 100 + D.vbr[i];
            break;
          }
      }
      float* o = p.dbg_rows + (((size_t)b * (p.L + 1) + j) * MDS_DEBUG_ROWS + r) * 4;
      o[0] = D.P.row[r].M;
      o[1] = D.P.row[r].invZ;
      o[2] = D.P.row[r].c;
      o[3] = (float)src;
    }
    __syncwarp();
  }

  // Combine the slice records of a stats pass (staged in scr): every row's M
  // and 1/Z and, with candidate lists, the sequence's list (the first LF of
  // the slices' entries by target logit, then slice, then position; in
  // token-id order), its complement masses and tau.  Sums over slices and entries run in fixed orders.
  __device__ void combine(int R, bool list) {
    const int ns = p.ns, rf = p.rec_floats;
    const float* sr = reinterpret_cast<const float*>(scr);
    for (int r = 0; r < R; ++r) {
      float M = kNegInf;
      for (int sl = lane; sl < ns; sl += 32) M = fmaxf(M, sr[sl * rf + 2 * r]);
      M = warp_max(M);
      if (!(M > kNegInf) || M != M) {
        if (lane == 0) atomicOr(p.status, MDS_ST_NONFINITE);
        M = 0.f;
      }
      const float c = D.P.row[r].c;
      float z = 0.f;
      for (int sl = lane; sl < ns; sl += 32) {
        z = __fadd_rn(z, moved_sum_near(sr[sl * rf + 2 * r + 1], sr[sl * rf + 2 * r], M, c));
      }
      z = warp_sum(z);
      if (lane == 0) {
        D.P.row[r].M = M;
        if (list)
          D.pc[r] = z;   // of the slices; the entries not taken join below
        else
          finish_row(r, z);
      }
    }
    __syncwarp();
    if (!list) return;
    if (ns * p.lns <= 128)
      combine_list<4>(R);
    else
      combine_list<kMaxEntries / 32>(R);
  }

  // The list part of combine, NT entries per lane at most (the small one
  // serves all but the shortest rows and the smallest batches; unrolled code
  // that one warp runs once costs its instruction fetches).
  template <int NT>
  __device__ __forceinline__ void combine_list(int R) {
    const int ns = p.ns, rf = p.rec_floats;
    const float* sr = reinterpret_cast<const float*>(scr);
    // the entries' order keys, entry lane + 32 t (0: none); 16-bit logits
    // differ in the key's upper half only
    constexpr int kBits = DT == MDS_BF16 ? 16 : 32;
    const int LN = p.lns, LF = p.ln;
    unsigned key[NT];
    unsigned cnt = 0u;
#pragma unroll
    for (int t = 0; t < NT; ++t) {
      key[t] = 0u;
      const int i = lane + 32 * t, sl = (int)__umulhi((unsigned)i, p.lns_rcp), q = i - sl * LN;
      if (sl < ns && q < __float_as_int(sr[sl * rf + 2 * kMaxRows + 1]))
        key[t] = ord_key(__fadd_rn(sr[sl * rf + kHdr + LN + q], 0.f)) >> (32 - kBits);
      cnt += key[t] ? 1u : 0u;
    }
    const int nv = (int)__reduce_add_sync(FULLM, cnt);
    // the largest key that at least LF entries reach
    unsigned thr = 0u;
    int ties = 0;
    if (nv > LF) {
#pragma unroll 1
      for (int bit = kBits - 1; bit >= 0; --bit) {
        const unsigned cand = thr | (1u << bit);
        unsigned c = 0u;
#pragma unroll
        for (int t = 0; t < NT; ++t)
          c += key[t] >= cand ? 1u : 0u;
        if ((int)__reduce_add_sync(FULLM, c) >= LF) thr = cand;
      }
      unsigned c = 0u;
#pragma unroll
      for (int t = 0; t < NT; ++t)
        c += key[t] > thr ? 1u : 0u;
      ties = LF - (int)__reduce_add_sync(FULLM, c);
    }
    const unsigned lt = (1u << lane) - 1u;
    int base = 0, tbase = 0;
    float tau = kNegInf, add[kListRowsMax], in[kListRowsMax];
#pragma unroll
    for (int r = 0; r < kListRowsMax; ++r) add[r] = in[r] = 0.f;
    for (int sl = lane; sl < ns; sl += 32) tau = fmaxf(tau, sr[sl * rf + 2 * kMaxRows]);
#pragma unroll
    for (int t = 0; t < NT; ++t) {
      const int i = lane + 32 * t, sl = (int)__umulhi((unsigned)i, p.lns_rcp), q = i - sl * LN;
      const unsigned tm = __ballot_sync(FULLM, key[t] == thr && thr);
      const bool take = key[t] > thr || (thr && key[t] == thr && tbase + __popc(tm & lt) < ties);
      const unsigned mk = __ballot_sync(FULLM, take);
      const int pos = base + __popc(mk & lt);
      base += __popc(mk);
      tbase += __popc(tm);
      if (key[t]) {
        const float* e = sr + sl * rf + kHdr + q;
        if (take) {
          D.cm_id[pos] = __float_as_int(e[0]);
          D.cm_l0[pos] = e[LN];
        } else {
          tau = fmaxf(tau, e[LN]);
        }
#pragma unroll
        for (int r = 0; r < kListRowsMax; ++r)
          if (r < R) {
            const float v = exp_term(e[(1 + r) * LN], D.P.row[r].M, D.P.row[r].c);
            if (take) {
              D.cm_e[r][pos] = v;
              in[r] = __fadd_rn(in[r], v);
            } else {
              add[r] = __fadd_rn(add[r], v);
            }
          }
      }
    }
    const int n = base;
    tau = warp_max(tau);
#pragma unroll
    for (int r = 0; r < kListRowsMax; ++r) {
      if (r >= R) break;
      const float a = warp_sum(add[r]), z = warp_sum(in[r]);
      if (lane == 0) {
        const float pc = __fadd_rn(D.pc[r], a);
        D.pc[r] = pc;
        finish_row(r, __fadd_rn(pc, z));
      }
    }
    if (lane == 0) {
      D.n = n;
      D.cand_tau = tau;
      D.cand_all = (n == p.V) ? 1 : 0;
      D.cand_q = (tau > kNegInf) ? exp_term(tau, D.P.row[0].M, D.P.row[0].c) : 0.f;
    }
    __syncwarp();
    // token-id order: the lanes of a stage then break ties and order Omega_1
    // by their number
    int id[2], at[2] = {0, 0};
    float l0[2], e[2][kListRowsMax];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int i = lane + 32 * h;
      id[h] = i < n ? D.cm_id[i] : 0;
      l0[h] = i < n ? D.cm_l0[i] : 0.f;
#pragma unroll
      for (int r = 0; r < kListRowsMax; ++r) e[h][r] = (r < R && i < n) ? D.cm_e[r][i] : 0.f;
    }
    for (int u = 0; u < n; ++u) {
      const int iu = D.cm_id[u];
#pragma unroll
      for (int h = 0; h < 2; ++h) at[h] += iu < id[h] ? 1 : 0;
    }
    __syncwarp();
#pragma unroll
    for (int h = 0; h < 2; ++h)
      if (lane + 32 * h < n) {
        D.cm_id[at[h]] = id[h];
        D.cm_l0[at[h]] = l0[h];
#pragma unroll
        for (int r = 0; r < kListRowsMax; ++r)
          if (r < R) D.cm_e[r][at[h]] = e[h][r];
      }
    __syncwarp();
  }

  // -------------------------------------------------------------- WIS stages on the candidate list
  // The pairwise stages (Remark 4) with one list entry per lane, its state in
  // registers throughout: the target probability, the rows' probabilities,
  // the law's explicit value where a stage has set one.  Returns the first
  // stage the list could not certify (fewer than s entries, or the s-th key
  // not above every key outside the list, each of which is <= its q <=
  // q(tau)), nv if none; *Ao the stages' token so far.  The law is left in
  // the pass (gamma, the special tokens' table).  A stage takes 5k SM cycles
  // alone (the same through shared memory with the LP on one lane: 9k; 12.7k
  // with eight decision warps an SM, 7.8k now).
  __device__ int wis_stages_list(int b, int j, int* Ao) {
    const int n = D.n, nv = D.nv, R = D.P.nrows;
    const int s = min(p.wis_s, p.V);
    const bool have = lane < n;
    const int id = have ? D.cm_id[lane] : 0x7fffffff;
    const float q = have ? __fmul_rn(D.cm_e[0][lane], D.P.row[0].invZ) : 0.f;
    const float qout = __fmul_rn(__fmul_rn(D.cand_q, D.P.row[0].invZ), 1.0001f);
    float pr[kListRowsMax], pz[kListRowsMax], gm[kListRowsMax];   // rows 1.. : here, outside the list, coefficient
#pragma unroll
    for (int r = 1; r < kListRowsMax; ++r) {
      const float iz = r < R ? D.P.row[r].invZ : 0.f;
      pr[r] = (r < R && have) ? __fmul_rn(D.cm_e[r][lane], iz) : 0.f;
      pz[r] = r < R ? __fmul_rn(D.pc[r], iz) : 0.f;
      gm[r] = r == D.vrow[0] ? 1.f : 0.f;
    }
    bool sp = false;
    float as = 0.f;
    int A = D.X[0], m = 1;
#pragma unroll 1
    for (; m < nv; ++m) {
      PT_T0(t_sel);
      const float u = D.dr[kDrSelect + m - 1];
      const int rb = D.vrow[m], Btok = D.X[m];
      float a = 0.f, bq = 0.f, sa = 0.f, sb = 0.f;
#pragma unroll
      for (int r = 1; r < kListRowsMax; ++r) {
        if (r >= R) break;
        a = __fmaf_rn(gm[r], pr[r], a);
        sa = __fmaf_rn(gm[r], pz[r], sa);
        if (r == rb) {
          bq = pr[r];
          sb = pz[r];
        }
      }
      if (sp) a = as;
      const float key = __fadd_rn(__fmaf_rn(-a, bq, q), 0.f);   // -0 -> +0: keys compare as floats
      // Omega_1: the entries with fewer than s larger keys; where the last of
      // them tie, the smaller token ids (the lower lanes)
      const unsigned kk = have ? ord_key(key) : 0u;
      D.kx[lane] = kk;
      __syncwarp();
      int above = 0;
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const uint4 o = reinterpret_cast<const uint4*>(D.kx)[c];
        above += (o.x > kk ? 1 : 0) + (o.y > kk ? 1 : 0) + (o.z > kk ? 1 : 0) + (o.w > kk ? 1 : 0);
      }
      uint32_t selm = __ballot_sync(FULLM, have && above < s);
      if (__popc(selm) > s) {
        const int last = (int)__reduce_max_sync(FULLM, (selm >> lane & 1u) ? (unsigned)above : 0u);
        const uint32_t tie = __ballot_sync(FULLM, have && above == last);
        selm = __ballot_sync(FULLM, (selm >> lane & 1u) &&
                                        (above < last || __popc(tie & ((1u << lane) - 1u)) < s - last));
      }
      const unsigned kth = __reduce_min_sync(FULLM, (selm >> lane & 1u) ? kk : FULLM);
      if (__popc(selm) != s || !(D.cand_all || ord_val(kth) > qout)) break;
      const bool sel = (selm >> lane) & 1u;
      // Omega_2 masses: complement (generic law) + list entries outside Omega_1
      float ra = (have && !sel) ? a : 0.f, rbm = (have && !sel) ? bq : 0.f;
#pragma unroll
      for (int o = 16; o; o >>= 1) {
        ra = __fadd_rn(ra, __shfl_xor_sync(FULLM, ra, o));
        rbm = __fadd_rn(rbm, __shfl_xor_sync(FULLM, rbm, o));
      }
      const float A2 = __fadd_rn(sa, ra), B2 = __fadd_rn(sb, rbm);
      const int rk = __popc(selm & ((1u << lane) - 1u));   // position in Omega_1 by token id
      if (lane >= s && lane < MDS_MAX_S) {
        D.om[lane] = -1;
        D.om_q[lane] = 0.f;
        D.om_a[lane] = 0.f;
        D.om_b[lane] = 0.f;
      }
      if (sel) {
        D.om[rk] = id;
        D.om_q[rk] = q;
        D.om_a[rk] = a;
        D.om_b[rk] = bq;
      }
      __syncwarp();
      PT_ADDW(kPhDecSelect, t_sel);
      PT_T0(t_lp);
      float xr = 0.f;
      if (s <= 5) {
        float x;
        bool capped;
        A = stage_solve5(A2, B2, A, Btok, u, D.om, D.om_q, D.om_a, D.om_b, x, &capped);
        if (capped && lane == 0) atomicOr(p.status, MDS_ST_LP_CAP);
        xr = __shfl_sync(FULLM, x, rk & 31);
      } else {
        if (lane == 0) D.Y = lp_solve8(s, A2, B2, A, Btok, u);
        __syncwarp();
        A = D.Y;
        xr = D.om_x[rk & (MDS_MAX_S - 1)];
      }
      PT_ADDW(kPhLp, t_lp);
      PT_CNTW(kPhLpCalls);
      if (sel) {
        as = xr;
        sp = true;
      } else if (sp) {
        as = __fmul_rn(0.5f, __fadd_rn(__fmul_rn(a, B2), __fmul_rn(bq, A2)));
      }
      // generic law: gamma <- (B2/2) gamma + (A2/2) e_rb
      const float hB = __fmul_rn(0.5f, B2), hA = __fmul_rn(0.5f, A2);
#pragma unroll
      for (int r = 1; r < kListRowsMax; ++r) {
        gm[r] = __fmul_rn(hB, gm[r]);
        if (r == rb) gm[r] = __fadd_rn(gm[r], hA);
      }
      __syncwarp();   // the tables are read before the next stage writes them
    }
    // the law into the pass: coefficients and the special tokens' table
    const uint32_t spm = __ballot_sync(FULLM, sp);
    if (sp) {
      const int k = __popc(spm & ((1u << lane) - 1u));
      D.P.spec_id[k] = id;
      D.P.spec_val[k] = as;
    }
    if (lane == 0) {
      D.P.nspec = __popc(spm);
#pragma unroll
      for (int r = 1; r < kListRowsMax; ++r)
        if (r < R) D.P.row[r].gamma = gm[r];
    }
    __syncwarp();
    *Ao = A;
    return m;
  }

  // The stage LP on the tables om, om_q, om_a, om_b (warp-wide): p_I on
  // Omega_1 to om_x, the stage's token returned.
  __device__ int solve(int s, float A2, float B2, int A, int Btok, float u) {
    PT_T0(t_lp);
    int y;
    if (s <= 5) {
      float x;
      bool capped;
      y = stage_solve5(A2, B2, A, Btok, u, D.om, D.om_q, D.om_a, D.om_b, x, &capped);
      if (capped && lane == 0) atomicOr(p.status, MDS_ST_LP_CAP);
      if (lane < 5) D.om_x[lane] = x;
    } else {
      if (lane == 0) D.Y = lp_solve8(s, A2, B2, A, Btok, u);
      __syncwarp();
      y = D.Y;
    }
    __syncwarp();
    PT_ADDW(kPhLp, t_lp);
    PT_CNTW(kPhLpCalls);
    return y;
  }

  // Generic law after a stage: gamma <- (B2/2) gamma + (A2/2) e_rb.  One thread.
  __device__ void gamma_update(int rb, float A2, float B2) {
    const float hB = __fmul_rn(0.5f, B2), hA = __fmul_rn(0.5f, A2);
    for (int r = 1; r < D.P.nrows; ++r) D.P.row[r].gamma = __fmul_rn(hB, D.P.row[r].gamma);
    D.P.row[rb].gamma = __fadd_rn(D.P.row[rb].gamma, hA);
  }

  // -------------------------------------------------------------- decisions per pass kind
  __device__ void accept_step(int b) {
    PT_T0(t_acc);
    int walk_now = 0;
    if (lane == 0) {
      const float u = D.dr[kDrAccept];
      const float ratio = D.W.pIY > 0.f ? __fdiv_rn(D.W.qY, D.W.pIY) : kPosInf;
      const bool acc = u < fminf(1.f, ratio);
      D.W.acc = acc ? 1 : 0;
      D.W.Ydiag = D.W.Y;
      walk_now = (acc && !p.acc_prob) ? 1 : 0;
      if (!walk_now) {
        D.W.ures = acc ? 0.f : D.dr[kDrResidual];
        if (p.scheme == MDS_SINGLE || D.nv == 1 || p.scheme != MDS_WIS) {
          // residual against one draft law: rows 0 and the first valid branch's
          for (int r = 0; r < D.P.nrows; ++r) D.P.row[r].gamma = 0.f;
          D.P.row[D.vrow[0]].gamma = 1.f;
          D.P.nspec = 0;
          D.P.nstream = max(2, D.vrow[0] + 1);
        } else {
          D.P.nstream = D.P.nrows;
        }
      }
    }
    walk_now = __shfl_sync(FULLM, walk_now, 0);
    __syncwarp();
    if (walk_now)
      walk(b, D.W.Y, 0.f, D.W.qY, D.W.pIY, D.W.Y);
    else
      push(b, kResid);
    PT_ADDW(kPhDecAccept, t_acc);
  }

  __device__ void decide_stats(int b, int j) {
    if (j == 0 && lane == 0) {
      D.W = FWalk{};
      D.W.valid = (p.K >= 32) ? FULLM : ((1u << p.K) - 1u);
      D.W.Yp = -1;
    }
    __syncwarp();
    PT_T0(t_plan);
    plan_warp(b, j, D.W.valid, false, true, true, D.tk0);
    PT_ADDW(kPhDecPlan, t_plan);
    PT_T0(t_comb);
    const int R = D.P.nstream;   // the planned pass is the completed one
    const bool list = D.P.list != 0;
    combine(R, list);
    if (p.dbg_rows) debug_rows(b, j, R);
    xl_sync();
    PT_ADDW(kPhDecCombine, t_comb);
    if (p.scheme == MDS_WIS0) {
      dec_wis0_nl<DT>(b);
      return;
    }
    if (p.scheme == MDS_SINGLE || D.nv == 1) {
      if (lane == 0) {
        const int Y = D.X[0];
        D.W.Y = Y;
        D.W.qY = prob_row(D.P, 0, Y);
        D.W.pIY = prob_row(D.P, D.vrow[0], Y);
      }
      __syncwarp();
      dec_accept_nl<DT>(b);
      return;
    }
    // WIS: the pairwise stages (Remark 4) on the candidate list while it
    // certifies Omega_1; from the first stage it cannot, full-vocabulary passes
    PT_T0(t_stg);
    if (lane == 0) {
      for (int r = 0; r < D.P.nrows; ++r) D.P.row[r].gamma = 0.f;
      D.P.row[D.vrow[0]].gamma = 1.f;
      D.P.nspec = 0;
    }
    __syncwarp();
    int A = D.X[0];
    int m = 1;
    if (list) m = wis_stages_list(b, j, &A);
    if (lane == 0) {
      D.W.stage = m;
      D.W.A = A;
      if (m < D.nv) {
        D.P.rb = D.vrow[m];
        D.P.nstream = D.P.nrows;
      } else {
        D.W.Y = A;
        D.W.qY = prob_row(D.P, 0, A);
        D.W.pIY = law_at(D.P, A);
      }
    }
    __syncwarp();
    PT_ADDW(kPhDecStages, t_stg);
    if (m < D.nv) {
      push(b, kFull);
      return;
    }
    dec_accept_nl<DT>(b);
  }

  // One full-vocabulary stage's decision: Omega_1 = the top s of the slices'
  // top s (s rounds of a warp argmax), the Omega_2 masses (the slices' rests
  // plus their entries not taken), the LP, the selection and the law update.
  __device__ void decide_full(int b) {
    const int j = D.P.j, ns = p.ns;
    plan_warp(b, j, D.W.valid, false, false, false, D.tk0);
    const int m = D.W.stage;
    const int A = D.W.A, Btok = D.X[m], rb = D.vrow[m];
    const float u = D.dr[kDrSelect + m - 1];
    const int s = min(p.wis_s, p.V);
    const float* recb = p.rec + (size_t)b * ns * p.rec_floats;
    for (int r = 0; r < s; ++r) {
      float bk = kNegInf;
      int bid = 0x7fffffff, bi = -1;
      for (int i = lane; i < ns * kTopF; i += 32) {
        const int sl = i / kTopF, t = i - sl * kTopF;
        if (t >= s) continue;
        const float* rc = recb + (size_t)sl * p.rec_floats;
        const int id = __ldcg(reinterpret_cast<const int*>(rc) + 4 + kTopF + t);
        bool taken = false;
        for (int q = 0; q < r; ++q) taken |= (D.fin[q].id == id);
        if (taken) continue;
        const float key = __ldcg(rc + 4 + t);
        if (id != 0x7fffffff && better(key, id, bk, bid)) {
          bk = key;
          bid = id;
          bi = i;
        }
      }
#pragma unroll
      for (int o = 16; o; o >>= 1) {
        const float ok = __shfl_xor_sync(FULLM, bk, o);
        const int oid = __shfl_xor_sync(FULLM, bid, o);
        const int oi = __shfl_xor_sync(FULLM, bi, o);
        if (better(ok, oid, bk, bid)) {
          bk = ok;
          bid = oid;
          bi = oi;
        }
      }
      if (lane == 0) {
        Cand c = CAND_NONE;
        if (bi >= 0) {
          const float* rc = recb + (size_t)(bi / kTopF) * p.rec_floats;
          const int t = bi % kTopF;
          c = Cand{bk, bid, __ldcg(rc + 4 + 2 * kTopF + t), __ldcg(rc + 4 + 3 * kTopF + t)};
        }
        D.fin[r] = c;
      }
      __syncwarp();
    }
    // Omega_2 masses: the slices' rests plus their top-s entries not taken
    float sa = 0.f, sb = 0.f;
    for (int i = lane; i < ns * kTopF; i += 32) {
      const int sl = i / kTopF, t = i - sl * kTopF;
      const float* rc = recb + (size_t)sl * p.rec_floats;
      if (t == 0) {
        sa = __fadd_rn(sa, __ldcg(rc + 0));
        sb = __fadd_rn(sb, __ldcg(rc + 1));
      }
      if (t >= s) continue;
      const int id = __ldcg(reinterpret_cast<const int*>(rc) + 4 + kTopF + t);
      if (id == 0x7fffffff) continue;
      bool taken = false;
      for (int q = 0; q < s; ++q) taken |= (D.fin[q].id == id);
      if (taken) continue;
      sa = __fadd_rn(sa, __ldcg(rc + 4 + 2 * kTopF + t));
      sb = __fadd_rn(sb, __ldcg(rc + 4 + 3 * kTopF + t));
    }
    const float ra = warp_sum(sa), rbs = warp_sum(sb);
    if (lane < s) {
      int id = D.fin[lane].id;
      if (id < 0 || id >= p.V) id = 0;   // only with non-finite keys (status already set)
      D.fin[lane].id = id;
      D.om_q[lane] = prob_row(D.P, 0, id);
    }
    __syncwarp();
    if (lane == 0) {
      // Omega_1 by token id; q follows its token
      int om[MDS_MAX_S];
      float ak[MDS_MAX_S], bk[MDS_MAX_S], qk[MDS_MAX_S];
      for (int t = 0; t < MDS_MAX_S; ++t) {
        om[t] = (t < s) ? D.fin[t].id : 0x7fffffff;
        ak[t] = (t < s) ? D.fin[t].a : 0.f;
        bk[t] = (t < s) ? D.fin[t].b : 0.f;
        qk[t] = (t < s) ? D.om_q[t] : 0.f;
      }
      for (int x = 1; x < MDS_MAX_S; ++x)   // insertion sort by id (at most 8 entries)
        for (int y = x; y > 0 && om[y] < om[y - 1]; --y) {
          const int ti = om[y];
          om[y] = om[y - 1];
          om[y - 1] = ti;
          float tf = ak[y];
          ak[y] = ak[y - 1];
          ak[y - 1] = tf;
          tf = bk[y];
          bk[y] = bk[y - 1];
          bk[y - 1] = tf;
          tf = qk[y];
          qk[y] = qk[y - 1];
          qk[y - 1] = tf;
        }
      for (int t = 0; t < MDS_MAX_S; ++t) {
        D.om[t] = (t < s) ? om[t] : -1;
        D.om_a[t] = ak[t];
        D.om_b[t] = bk[t];
        D.om_q[t] = qk[t];
      }
    }
    __syncwarp();
    const float A2 = ra, B2 = rbs;
    const int Y = solve(s, A2, B2, A, Btok, u);
    // law update: special tokens outside Omega_1, gamma, Omega_1 values
    for (int i = lane; i < D.P.nspec; i += 32) {
      const int tokn = D.P.spec_id[i];
      bool in1 = false;
      for (int t = 0; t < s; ++t) in1 |= (D.om[t] == tokn);
      if (!in1)
        D.P.spec_val[i] =
            __fmul_rn(0.5f, __fadd_rn(__fmul_rn(D.P.spec_val[i], B2), __fmul_rn(prob_row(D.P, rb, tokn), A2)));
    }
    __syncwarp();
    if (lane == 0) {
      gamma_update(rb, A2, B2);
      for (int t = 0; t < s; ++t) {
        int i = 0;
        while (i < D.P.nspec && D.P.spec_id[i] != D.om[t]) ++i;
        if (i == D.P.nspec && D.P.nspec < kMaxSpecial) {
          D.P.spec_id[i] = D.om[t];
          ++D.P.nspec;
        }
        if (i < kMaxSpecial) D.P.spec_val[i] = D.om_x[t];
      }
      D.W.A = Y;
      D.W.stage = m + 1;
      if (m + 1 < D.nv) D.P.rb = D.vrow[m + 1];
    }
    __syncwarp();
    if (m + 1 < D.nv) {
      push(b, kFull);
      return;
    }
    if (lane == 0) {
      D.W.Y = Y;
      D.W.qY = prob_row(D.P, 0, Y);
      D.W.pIY = law_at(D.P, Y);
    }
    __syncwarp();
    dec_accept_nl<DT>(b);
  }

  // -------------------------------------------------------------- inverse-CDF search
  // Weights of unit u (tokens tok0 + u*VE + e) of a re-read slice, read from
  // global memory: the residual max(0, q - p_I) (kResid), the target mass
  // outside Omega_0 (kReplace) or the target mass (kBonus); tokens past the
  // slice weigh 0.
  __device__ void weights_g(const FPass& P, int u, int tok0, int n, float* w) const {
    auto load = [&](int r, float* v) {
      const char* row = P.row[r].ptr;
      const int t0 = tok0 + u * VE;
      if (p.aligned && u * VE + VE <= n) {
        E::unit_global(row + (size_t)t0 * p.esize, v);
      } else {
#pragma unroll
        for (int e = 0; e < VE; ++e) v[e] = (u * VE + e < n) ? E::global(row, t0 + e) : kNegInf;
      }
    };
    float v0[VE];
    load(0, v0);
    const float M0 = P.row[0].M, c0 = P.row[0].c, iz0 = P.row[0].invZ;
    if (P.kind == kResid) {
      float a[VE];
#pragma unroll
      for (int e = 0; e < VE; ++e) a[e] = 0.f;
      for (int r = 1; r < P.nstream; ++r) {
        const float g = P.row[r].gamma;
        if (g == 0.f) continue;
        float v[VE];
        load(r, v);
        const float M = P.row[r].M, c = P.row[r].c, iz = P.row[r].invZ;
#pragma unroll
        for (int e = 0; e < VE; ++e) a[e] = __fmaf_rn(g, prob_of(v[e], M, c, iz), a[e]);
      }
      if (P.nspec > 0 && ((bm[u >> 5] >> (u & 31)) & 1u)) {
#pragma unroll
        for (int e = 0; e < VE; ++e) a[e] = spec_lookup(P, tok0 + u * VE + e, a[e]);
      }
#pragma unroll
      for (int e = 0; e < VE; ++e) w[e] = fmaxf(0.f, __fsub_rn(prob_of(v0[e], M0, c0, iz0), a[e]));
    } else if (P.kind == kReplace) {
#pragma unroll
      for (int e = 0; e < VE; ++e) w[e] = (P.all0 || v0[e] > P.cut) ? 0.f : prob_of(v0[e], M0, c0, iz0);
    } else {
#pragma unroll
      for (int e = 0; e < VE; ++e) w[e] = prob_of(v0[e], M0, c0, iz0);
    }
  }

  // Inclusive warp scan (fixed order) of v over the lanes.
  __device__ __forceinline__ static float scan_incl(float v, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const float t = __shfl_up_sync(FULLM, v, o);
      if (lane >= o) v = __fadd_rn(v, t);
    }
    return v;
  }

  // The smallest token whose running mass exceeds T, else the last token
  // with positive weight.  Four levels in token order, each a warp scan:
  // the slices (masses Rs[0..ns)), the slice's runs of 32 units (masses from
  // its staged record, two per lane; the bonus row's against the slice's own
  // maximum), the owning run's units (re-read, one per lane), the owning
  // unit's tokens (in that lane's registers).
  __device__ int search(FPass& P, float T, bool bonus) {
    // level 0: slices
    int s = -1, slast = -1;
    float base = 0.f, blast = 0.f;
    {
      float run = 0.f;
      for (int c = 0; c < p.ns && s < 0; c += 32) {
        const int q = c + lane;
        const float v = q < p.ns ? Rs[q] : 0.f;
        const float incl = scan_incl(v, lane);
        const float ex = __fadd_rn(run, __fsub_rn(incl, v));
        const unsigned h = __ballot_sync(FULLM, __fadd_rn(run, incl) > T && v > 0.f);
        const unsigned pz = __ballot_sync(FULLM, v > 0.f);
        if (h) {
          const int l = __ffs(h) - 1;
          s = c + l;
          base = __shfl_sync(FULLM, ex, l);
        } else if (pz) {
          const int l = 31 - __clz(pz);
          slast = c + l;
          blast = __shfl_sync(FULLM, ex, l);
        }
        run = __shfl_sync(FULLM, __fadd_rn(run, incl), 31);
      }
      if (s < 0) {
        s = max(slast, 0);
        base = blast;
      }
    }
    const int tok0 = s * p.T, n = min(p.T, p.V - tok0);
    const int U = (n + VE - 1) / VE;
    if (P.kind == kResid && P.nspec > 0) {
      for (int i = lane; i < 64; i += 32) bm[i] = 0u;
      __syncwarp();
      for (int i = lane; i < P.nspec; i += 32) {
        const int loc = P.spec_id[i] - tok0;
        if (loc >= 0 && loc < n) atomicOr(&bm[(loc / VE) >> 5], 1u << ((loc / VE) & 31));
      }
      __syncwarp();
    }
    // level 1: runs lane and 32 + lane
    const int nrun = (U + 31) / 32;
    const float* rr = reinterpret_cast<const float*>(scr) + s * p.rec_floats + 4;
    const float sc = bonus ? __fmul_rn(ref_shift(Hm[s], P.row[0].M, P.row[0].c), P.row[0].invZ) : 1.f;
    const float r0 = lane < nrun ? __fmul_rn(rr[lane], sc) : 0.f;
    const float r1 = lane + 32 < nrun ? __fmul_rn(rr[lane + 32], sc) : 0.f;
    const float i0 = scan_incl(r0, lane);
    const float i1 = __fadd_rn(__shfl_sync(FULLM, i0, 31), scan_incl(r1, lane));
    const unsigned h0 = __ballot_sync(FULLM, __fadd_rn(base, i0) > T && r0 > 0.f);
    const unsigned h1 = __ballot_sync(FULLM, __fadd_rn(base, i1) > T && r1 > 0.f);
    const unsigned z0 = __ballot_sync(FULLM, r0 > 0.f), z1 = __ballot_sync(FULLM, r1 > 0.f);
    if (!(z0 | z1)) return tok0;   // no mass in the slice (only by rounding)
    const int own = h0 ? __ffs(h0) - 1 : (h1 ? 31 + __ffs(h1) : (z1 ? 63 - __clz(z1) : 31 - __clz(z0)));
    const float run = __fadd_rn(base, own < 32 ? __shfl_sync(FULLM, __fsub_rn(i0, r0), own & 31)
                                               : __shfl_sync(FULLM, __fsub_rn(i1, r1), own & 31));
    // level 2: the run's units, one per lane; level 3 in the owning lane
    const int u = own * 32 + lane;
    float w[VE], us = 0.f;
#pragma unroll
    for (int e = 0; e < VE; ++e) w[e] = 0.f;
    if (u < U) {
      weights_g(P, u, tok0, n, w);
#pragma unroll
      for (int e = 0; e < VE; ++e) us = __fadd_rn(us, w[e]);
    }
    const float ui = scan_incl(us, lane);
    const unsigned h2 = __ballot_sync(FULLM, __fadd_rn(run, ui) > T && us > 0.f);
    const unsigned z2 = __ballot_sync(FULLM, us > 0.f);
    const int l2 = h2 ? __ffs(h2) - 1 : (z2 ? 31 - __clz(z2) : 0);
    int tok = 0;
    if (lane == l2) {
      float acc = __fadd_rn(run, __fsub_rn(ui, us));
      int hit = -1, last = -1;
#pragma unroll
      for (int e = 0; e < VE; ++e) {
        if (w[e] > 0.f) last = e;
        acc = __fadd_rn(acc, w[e]);
        if (hit < 0 && acc > T && w[e] > 0.f) hit = e;
      }
      if (hit < 0) hit = last < 0 ? 0 : last;
      tok = min(tok0 + u * VE + hit, p.V - 1);
    }
    return __shfl_sync(FULLM, tok, l2);
  }

  // Slice masses of the pass just completed (Rs) and their total.
  __device__ float slice_masses(int b) {
    const float* rec = reinterpret_cast<const float*>(scr);
    float R = 0.f;
    for (int q = lane; q < p.ns; q += 32) {
      Rs[q] = rec[q * p.rec_floats];
      R = __fadd_rn(R, Rs[q]);
    }
    __syncwarp();
    return warp_sum(R);
  }

  __device__ void decide_resid(int b) {
    plan_warp(b, D.P.j, D.W.valid, false, false, false, D.tk0);
    const float R = slice_masses(b);
    int Z = D.W.Y;
    if (!D.W.acc) {
      if (R > 0.f) {
        Z = search(D.P, __fmul_rn(D.W.ures, R), false);
      } else {
        // zero residual mass (only by rounding): sample the target row
        if (lane == 0) {
          atomicOr(p.status, MDS_ST_ZERO_RESID);
          D.W.zres = 1;
          D.W.R = R;
          D.P.cut = kPosInf;
          D.P.all0 = 0;
          D.P.nstream = 1;
        }
        __syncwarp();
        push(b, kReplace);
        return;
      }
    }
    walk(b, Z, R, D.W.qY, D.W.pIY, D.W.Ydiag);
  }

  __device__ void decide_replace(int b) {
    plan_warp(b, D.P.j, D.W.valid, false, false, false, D.tk0);
    const float R = slice_masses(b);
    int Z;
    if (R > 0.f) {
      Z = search(D.P, __fmul_rn(D.W.ures, R), false);
    } else if (!D.W.zres && D.W.Yp >= 0) {
      Z = D.W.Yp;   // no target mass outside Omega_0
    } else if (!D.W.zres) {
      if (lane == 0) {
        atomicOr(p.status, MDS_ST_ZERO_RESID);
        D.W.zres = 1;
        D.P.cut = kPosInf;
        D.P.all0 = 0;
      }
      __syncwarp();
      push(b, kReplace);
      return;
    } else {
      if (lane == 0) atomicOr(p.status, MDS_ST_NONFINITE);
      Z = 0;
    }
    const float Rd = (p.scheme == MDS_WIS0) ? D.W.R : (D.W.zres ? D.W.R : R);
    walk(b, Z, Rd, D.W.qY, D.W.pIY, D.W.Ydiag);
  }

  __device__ void decide_bonus(int b) {
    const float* rec = reinterpret_cast<const float*>(scr);
    float M = kNegInf;
    for (int q = lane; q < p.ns; q += 32) {
      Hm[q] = rec[q * p.rec_floats];
      Rs[q] = rec[q * p.rec_floats + 1];
      M = fmaxf(M, Hm[q]);
    }
    M = warp_max(M);
    if (!(M > kNegInf) || M != M) {
      if (lane == 0) atomicOr(p.status, MDS_ST_NONFINITE);
      M = 0.f;
    }
    const float c = D.P.row[0].c;
    float Zs = 0.f;
    for (int q = lane; q < p.ns; q += 32) Zs = __fadd_rn(Zs, moved_sum(Rs[q], Hm[q], M, c));
    Zs = warp_sum(Zs);
    if (lane == 0) {
      D.P.row[0].M = M;
      finish_row(0, Zs);
    }
    __syncwarp();
    if (p.dbg_rows && lane == 0) {
      float* o = p.dbg_rows + (((size_t)b * (p.L + 1) + p.L) * MDS_DEBUG_ROWS) * 4;
      o[0] = D.P.row[0].M;
      o[1] = D.P.row[0].invZ;
      o[2] = D.P.row[0].c;
      o[3] = (float)(__ffs(D.W.valid) - 1);
    }
    const float iz = D.P.row[0].invZ;
    float Q = 0.f;
    for (int q = lane; q < p.ns; q += 32) {
      Rs[q] = (Hm[q] > kNegInf) ? __fmul_rn(__fmul_rn(Rs[q], ref_shift(Hm[q], M, c)), iz) : 0.f;
      Q = __fadd_rn(Q, Rs[q]);
    }
    __syncwarp();
    Q = warp_sum(Q);
    const int Z = search(D.P, __fmul_rn(D.dr[kDrBonus], Q), true);
    if (lane == 0) {
      __stcg(p.out_tokens + (size_t)b * (p.L + 1) + p.L, Z);
      if (p.out_diag) {
        float* dg = p.out_diag + ((size_t)b * (p.L + 1) + p.L) * 4;
        __stcg(dg + 0, 0.f);
        __stcg(dg + 1, 0.f);
        __stcg(dg + 2, Q);
        __stcg(dg + 3, -1.f);
      }
    }
    finish(b, p.L);
  }
  // -------------------------------------------------------------- truncated alphabet
  // Inverse CDF over the list entries in token order, two per lane (entry
  // lane and 32 + lane; weights w0, w1): the first entry whose running sum
  // exceeds u01 * total, else the last with positive weight; -1 when the
  // total is 0.  Sums: a warp scan of each half, the halves in order.
  __device__ __forceinline__ int lane_cdf2(float w0, float w1, float u01, float* total) const {
    float c0 = w0, c1 = w1;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const float t0 = __shfl_up_sync(FULLM, c0, o);
      const float t1 = __shfl_up_sync(FULLM, c1, o);
      if (lane >= o) {
        c0 = __fadd_rn(c0, t0);
        c1 = __fadd_rn(c1, t1);
      }
    }
    const float h0 = __shfl_sync(FULLM, c0, 31);
    c1 = __fadd_rn(h0, c1);
    const float tot = __shfl_sync(FULLM, c1, 31);
    *total = tot;
    if (!(tot > 0.f)) return -1;
    const float T = __fmul_rn(u01, tot);
    const unsigned who0 = __ballot_sync(FULLM, c0 > T);
    if (who0) return __ffs(who0) - 1;
    const unsigned who1 = __ballot_sync(FULLM, c1 > T);
    if (who1) return 32 + __ffs(who1) - 1;
    const unsigned p1 = __ballot_sync(FULLM, w1 > 0.f);
    if (p1) return 32 + 31 - __clz(p1);
    return 31 - __clz(__ballot_sync(FULLM, w0 > 0.f));
  }

  // One depth of the truncated-alphabet scheme (Section 4, read with the
  // non-iid appendix's remark on keeping only the inputs in Omega_0).
  // Omega_0 = the target tokens above the (M+1)-th largest target logit, read
  // off the candidate list (exact when the list's (M+1)-th entry is >= tau,
  // the list holds the whole vocabulary, or every token outside it is -inf;
  // otherwise the tokens above tau, with MDS_ST_OMEGA0).  The warp runs the
  // WIS stages on Omega_0 against q~ = q / p_a with the kept inputs' draft
  // laws restricted to Omega_0 and renormalised (point loads of the draft
  // logits there), then Algorithm 1 against q~.  Y' is kept with probability
  // p_a, else a replace pass draws from the tokens outside Omega_0 by q.
  // The list (token-id order, up to 64 entries) sits two entries per lane:
  // entry lane (half 0) and 32 + lane (half 1).
  __device__ void wis0_decide(int b) {
    {
      const int n = D.n;
      bool have[2], in0[2];
      int id[2], rk[2] = {0, 0};
      float l[2], q[2], qt[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int e = lane + 32 * h;
        have[h] = e < n;
        id[h] = have[h] ? D.cm_id[e] : 0;
        l[h] = have[h] ? D.cm_l0[e] : kNegInf;
      }
      // rank in the list by (larger logit, then lower id)
      for (int t = 0; t < n; ++t) {
        const float lt = D.cm_l0[t];
        const int it = D.cm_id[t];
#pragma unroll
        for (int h = 0; h < 2; ++h) rk[h] += better(lt, it, l[h], id[h]) ? 1 : 0;
      }
      const int M = p.omega0;
      const bool all0 = M >= p.V;
      float cut = kNegInf;
      bool cert;
      if (all0) {
        cert = D.cand_all != 0;
      } else {
        const unsigned w0 = __ballot_sync(FULLM, have[0] && rk[0] == M);
        const unsigned w1 = __ballot_sync(FULLM, have[1] && rk[1] == M);
        const bool found = (w0 | w1) != 0u;
        if (w0)
          cut = __shfl_sync(FULLM, l[0], __ffs(w0) - 1);
        else if (w1)
          cut = __shfl_sync(FULLM, l[1], __ffs(w1) - 1);
        const float tau = D.cand_tau;
        cert = D.cand_all || (found ? cut >= tau : !(tau > kNegInf));
        if (!cert) cut = fmaxf(cut, tau);
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        in0[h] = have[h] && (all0 || l[h] > cut);
        q[h] = in0[h] ? prob_of(l[h], D.P.row[0].M, D.P.row[0].c, D.P.row[0].invZ) : 0.f;
      }
      const int n0 = __popc(__ballot_sync(FULLM, in0[0])) + __popc(__ballot_sync(FULLM, in0[1]));
      const float pa = warp_sum(__fadd_rn(q[0], q[1]));
#pragma unroll
      for (int h = 0; h < 2; ++h) qt[h] = (in0[h] && pa > 0.f) ? __fdiv_rn(q[h], pa) : 0.f;
      // draft laws restricted to Omega_0 (exponents against their own maximum
      // there; the rows' full normalisers cancel), per row and entry, in the
      // warp's scratch (the staged records are spent)
      float* ew = reinterpret_cast<float*>(scr);   // [nrows][64]
      for (int r = 1; r < D.P.nrows; ++r) {
        float lr[2], e[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) lr[h] = in0[h] ? E::global(D.P.row[r].ptr, id[h]) : kNegInf;
        const float cr = D.P.row[r].c;
        const float ref = sum_ref(warp_max(fmaxf(lr[0], lr[1])), cr);
#pragma unroll
        for (int h = 0; h < 2; ++h) e[h] = (in0[h] && ref > kNegInf) ? exp_term(lr[h], ref, cr) : 0.f;
        const float Pm = warp_sum(__fadd_rn(e[0], e[1]));
        if (lane == 0 && Pm != Pm) atomicOr(p.status, MDS_ST_NONFINITE);
#pragma unroll
        for (int h = 0; h < 2; ++h) ew[r * 64 + lane + 32 * h] = (Pm > 0.f) ? __fdiv_rn(e[h], Pm) : 0.f;
      }
      __syncwarp();
      // kept inputs: valid branches (branch order) whose token lies in Omega_0
      int nk = 0;
      for (int i = 0; i < D.nv; ++i) {
        const unsigned w0 = __ballot_sync(FULLM, in0[0] && id[0] == D.X[i]);
        const unsigned w1 = __ballot_sync(FULLM, in0[1] && id[1] == D.X[i]);
        if (!(w0 | w1)) continue;
        const int ei = w0 ? __ffs(w0) - 1 : 32 + __ffs(w1) - 1;
        if (!(ew[D.vrow[i] * 64 + ei] > 0.f)) continue;   // impossible draw: dropped
        if (lane == 0) {
          D.k_lane[nk] = ei;
          D.k_row[nk] = D.vrow[i];
        }
        ++nk;
      }
      __syncwarp();
      int yl = -1, Yl = -1;
      float qY = 0.f, pIY = 0.f, R = 0.f;
      if (n0 > 0 && nk == 0) {
        float t;
        yl = lane_cdf2(qt[0], qt[1], D.dr[kDrResidual], &t);
      } else if (n0 > 0) {
        float a[2];
        {
          const float* w = ew + D.k_row[0] * 64;
          a[0] = w[lane];
          a[1] = w[lane + 32];
        }
        int A = D.k_lane[0];
        const int s = min(p.wis_s, n0);
        const unsigned lt = (1u << lane) - 1u;
        for (int m = 1; m < nk; ++m) {
          const int Bl = D.k_lane[m];
          const float* wb = ew + D.k_row[m] * 64;
          const float bb[2] = {wb[lane], wb[lane + 32]};
          const float u = D.dr[kDrSelect + m - 1];
          unsigned kk[2];
#pragma unroll
          for (int h = 0; h < 2; ++h) kk[h] = in0[h] ? ord_key(__fadd_rn(__fmaf_rn(-a[h], bb[h], qt[h]), 0.f)) : 0u;
          // Omega_1: s rounds of the largest key, ties to the smaller id
          // (the lower entry)
          uint32_t sel0 = 0u, sel1 = 0u;
          for (int t = 0; t < s; ++t) {
            const unsigned km = __reduce_max_sync(FULLM, max(kk[0], kk[1]));
            if (!km) break;
            const uint32_t w0 = __ballot_sync(FULLM, kk[0] == km);
            if (w0) {
              const int wl = __ffs(w0) - 1;
              sel0 |= 1u << wl;
              if (lane == wl) kk[0] = 0u;
            } else {
              const int wl = __ffs(__ballot_sync(FULLM, kk[1] == km)) - 1;
              sel1 |= 1u << wl;
              if (lane == wl) kk[1] = 0u;
            }
          }
          const bool sl[2] = {((sel0 >> lane) & 1u) != 0u, ((sel1 >> lane) & 1u) != 0u};
          const int sn = __popc(sel0) + __popc(sel1);
          const float A2 = warp_sum(__fadd_rn((in0[0] && !sl[0]) ? a[0] : 0.f, (in0[1] && !sl[1]) ? a[1] : 0.f));
          const float B2 = warp_sum(__fadd_rn((in0[0] && !sl[0]) ? bb[0] : 0.f, (in0[1] && !sl[1]) ? bb[1] : 0.f));
          const int rk1[2] = {__popc(sel0 & lt), __popc(sel0) + __popc(sel1 & lt)};
          if (lane >= sn && lane < MDS_MAX_S) {
            D.om[lane] = -1;
            D.om_q[lane] = 0.f;
            D.om_a[lane] = 0.f;
            D.om_b[lane] = 0.f;
          }
#pragma unroll
          for (int h = 0; h < 2; ++h)
            if (sl[h]) {
              D.om[rk1[h]] = id[h];
              D.om_q[rk1[h]] = qt[h];
              D.om_a[rk1[h]] = a[h];
              D.om_b[rk1[h]] = bb[h];
            }
          __syncwarp();
          const int Yt = solve(sn, A2, B2, D.cm_id[A], D.cm_id[Bl], u);
          const unsigned y0 = __ballot_sync(FULLM, in0[0] && id[0] == Yt);
          const unsigned y1 = __ballot_sync(FULLM, in0[1] && id[1] == Yt);
          A = y0 ? __ffs(y0) - 1 : (y1 ? 32 + __ffs(y1) - 1 : 0);
#pragma unroll
          for (int h = 0; h < 2; ++h)
            a[h] = sl[h] ? D.om_x[rk1[h]]
                         : (in0[h] ? __fmul_rn(0.5f, __fadd_rn(__fmul_rn(a[h], B2), __fmul_rn(bb[h], A2))) : 0.f);
          __syncwarp();
        }
        Yl = A;
        const int Ah = A >> 5, Alane = A & 31;
        qY = __shfl_sync(FULLM, Ah ? qt[1] : qt[0], Alane);
        pIY = __shfl_sync(FULLM, Ah ? a[1] : a[0], Alane);
        const float ratio = pIY > 0.f ? __fdiv_rn(qY, pIY) : kPosInf;
        if (D.dr[kDrAccept] < fminf(1.f, ratio)) {
          yl = A;
        } else {
          const float ures = D.dr[kDrResidual];
          yl = lane_cdf2(in0[0] ? fmaxf(0.f, __fsub_rn(qt[0], a[0])) : 0.f,
                         in0[1] ? fmaxf(0.f, __fsub_rn(qt[1], a[1])) : 0.f, ures, &R);
          if (yl < 0) {   // only by rounding: sample q~
            if (lane == 0) atomicOr(p.status, MDS_ST_ZERO_RESID);
            float t;
            yl = lane_cdf2(qt[0], qt[1], ures, &t);
          }
        }
      }
      if (lane == 0) {
        if (!cert) atomicOr(p.status, MDS_ST_OMEGA0);
        D.o0_n = n0;
        D.o0_all = (all0 && D.cand_all) ? 1 : 0;
        D.o0_cut = cut;
        D.o0_pa = pa;
        D.W.R = R;
        D.W.Yp = (yl >= 0) ? D.cm_id[yl] : -1;
        D.W.Ydiag = (Yl >= 0) ? D.cm_id[Yl] : -1;
        D.W.qY = qY;
        D.W.pIY = pIY;
        D.W.zres = 0;
        const bool keep = D.o0_n > 0 && (D.o0_all || D.dr[kDrKeep] < D.o0_pa);
        D.tok = keep ? 1 : 0;
        if (!keep) {
          D.W.ures = D.dr[kDrOutside];
          D.P.cut = cut;
          D.P.all0 = D.o0_all;
          D.P.nstream = 1;
        }
      }
    }
    __syncwarp();
    if (D.tok)
      walk(b, D.W.Yp, D.W.R, D.W.qY, D.W.pIY, D.W.Ydiag);
    else
      push(b, kReplace);
  }

  // -------------------------------------------------------------- one decision
  // Request fields: the sequence, the depth of the pass that just completed
  // and whether it is the sequence's first.
  __device__ void decide(int b, int j, bool first) {
    // One round of asynchronous copies: the sequence's state (a depth-0
    // stats pass has none yet), its draft tokens at depths j and j + 1, its
    // temperatures and the slice records of the pass.
    const int K = p.K, L = p.L;
    PT_T0(t_load);
    if (!first) {
      const int4* src = reinterpret_cast<const int4*>(reinterpret_cast<const FSeq*>(p.seq) + b);
      int4* dst = reinterpret_cast<int4*>(&D.P);
      for (int i = lane; i < (int)(sizeof(FSeq) / 16); i += 32) cpa16(dst + i, src + i);
    }
    if (lane < K) {
      const int32_t* tk = p.tokens + ((size_t)b * K + lane) * L;
      cpa4(&D.tk0[lane], tk + j);
      if (j + 1 < L) cpa4(&D.tk1[lane], tk + j + 1);
    }
    if (lane <= K) cpa4(&D.tmp[lane], p.temps + (size_t)b * (1 + K) + lane);
    {
      const float* recb = p.rec + (size_t)b * p.ns * p.rec_floats;
      const int n16 = p.ns * p.rec_floats / 4;
      for (int i = lane; i < n16; i += 32) cpa16(scr + 16 * i, recb + 4 * i);
    }
    if (lane < kDrawsN) D.dr[lane] = draw_uniform(p.seed, b, j, draw_id(lane));   // beside the copies
    cpa_wait();
    __syncwarp();
    if (lane == 0) {
      D.xl_ok = 0;
      D.xl_wait = 0;
    }
    __syncwarp();
    PT_ADDW(kPhDecLoad, t_load);
    PT_T0(t_dec);
    PT_CNTW(kPhDecisions);
    const int kind = first ? kStats : D.P.kind;
    switch (kind) {
      case kStats: dec_stats_nl<DT>(b, j); break;
      case kResid: dec_resid_nl<DT>(b); break;
      case kReplace: dec_replace_nl<DT>(b); break;
      case kFull: dec_full_nl<DT>(b); break;
      case kBonus: dec_bonus_nl<DT>(b); break;
      default: break;
    }
    __syncwarp();
    PT_ADDW(kind == kStats ? kPhDecStats
                           : (kind == kFull ? kPhDecFull : (kind == kBonus ? kPhDecBonus : kPhDecResid)),
            t_dec);
  }

  // The decision warp's loop: take request numbers from the decision ring,
  // wait for each request's publication, decide.  Leaves when every sequence
  // is finished (or on an abort).
  __device__ __forceinline__ void loop() {
    for (;;) {
      int have = 0;
      unsigned pay = 0u;
      if (lane == 0 && !aborted()) {
        const unsigned t = atomicAdd(&p.ctl[kCtlDecHead], 1u);
        const unsigned slot = t % (unsigned)p.dec_cap;
        const unsigned long long want = ring_word(p.epoch, t / (unsigned)p.dec_cap, 0u);
        const unsigned long long t0 = now_ns();
        PT_T0(t_poll);
        for (int it = 0;; ++it) {
          const unsigned long long w = ld_acquire(&p.dec_tag[slot]);
          if ((w & ~kRingPay) == want) {
            pay = (unsigned)(w & kRingPay);
            st_relaxed(&p.dec_rtag[slot], want);
            have = 1;
            break;
          }
          if ((it & 3) == 3 && (ld_relaxed(&p.ctl[kCtlDone]) >= (unsigned)p.B || aborted())) break;
          if ((it & 15) == 15 && now_ns() - t0 > kWaitNs) {
            set_abort(MDS_ST_TIMEOUT);
            break;
          }
          __nanosleep(it < 16 ? 32 : 128);
        }
        PT_ADDW(kPhDecPoll, t_poll);
      }
      have = __shfl_sync(FULLM, have, 0);
      pay = __shfl_sync(FULLM, pay, 0);
      if (!have) return;
      decide((int)(pay >> 8), (int)((pay >> 1) & 127u), (pay & 1u) != 0u);
    }
  }
};


// Shared memory of a CTA, at file scope so that the decision code (out of
// line) addresses it as shared memory: the dynamic buffers, the CTA state and,
// in decision CTAs, a copy of the launch parameters.
extern __shared__ __align__(128) char g_dsm[];
__shared__ FShared g_S;
__shared__ Params g_dp;

constexpr int kDStateBytes = (int)((sizeof(DState) + 127) / 128 * 128);
constexpr int kDecPerWarp = kDStateBytes + (kDecScratch + 127) / 128 * 128;
constexpr int kSlotOff = kNBuf * kBufBytes;
constexpr int kDynBytes = kSlotOff + kSlots * (int)sizeof(Slot);
constexpr int kDecWarps = 4;   // decision warps per decision CTA
static_assert(kDecWarps * kDecPerWarp <= kDynBytes && kDecWarps <= kBlock / 32, "decision warps' shared memory");

// The calling warp's decision view: its state and scratch in the CTA's
// dynamic shared memory, the parameters from the CTA's shared copy.
template <int DT>
__device__ __forceinline__ Dec<DT> dec_view() {
  char* base = g_dsm + (size_t)(threadIdx.x >> 5) * kDecPerWarp;
  char* scr = base + kDStateBytes;
  float* rs = reinterpret_cast<float*>(scr + kDecStage);
  return Dec<DT>{g_dp, g_S, *reinterpret_cast<DState*>(base), scr, rs, rs + kMaxSlices,
                 reinterpret_cast<uint32_t*>(rs + 2 * kMaxSlices), (int)(threadIdx.x & 31)};
}
template <int DT> __device__ __noinline__ void dec_stats_nl(int b, int j) { dec_view<DT>().decide_stats(b, j); }
template <int DT> __device__ __noinline__ void dec_resid_nl(int b) { dec_view<DT>().decide_resid(b); }
template <int DT> __device__ __noinline__ void dec_replace_nl(int b) { dec_view<DT>().decide_replace(b); }
template <int DT> __device__ __noinline__ void dec_full_nl(int b) { dec_view<DT>().decide_full(b); }
template <int DT> __device__ __noinline__ void dec_bonus_nl(int b) { dec_view<DT>().decide_bonus(b); }
template <int DT> __device__ __noinline__ void dec_wis0_nl(int b) { dec_view<DT>().wis0_decide(b); }
template <int DT> __device__ __noinline__ void dec_accept_nl(int b) { dec_view<DT>().accept_step(b); }

// The stage LP for s > 5 of the calling warp's decision (one lane), on its
// Omega_1 tables: pair state in shared memory.
__device__ __noinline__ int lp_solve8(int s, float A2, float B2, int A, int Btok, float u) {
  DState& D = *reinterpret_cast<DState*>(g_dsm + (size_t)(threadIdx.x >> 5) * kDecPerWarp);
  bool capped = false;
  const int y = stage_solve<MDS_MAX_S>(s, A2, B2, A, Btok, u, D.om, D.om_q, D.om_a, D.om_b, D.om_x, &capped,
                                       D.lp_rs, D.lp_fl, D.lp_fh);
  if (capped) atomicOr(g_dp.status, MDS_ST_LP_CAP);
  return y;
}

// A decision warp's loop, out of line with the whole register budget.
template <int DT>
__device__ __noinline__ void decision_warp() { dec_view<DT>().loop(); }

template <int DT>
__global__ void __launch_bounds__(kBlock, kCtasPerSm) flow_kernel(const __grid_constant__ Params p) {
  char* dsm = g_dsm;
  FShared& S = g_S;
  Eng<DT> e{p, S};
  e.bufs = dsm;
  e.slots = reinterpret_cast<Slot*>(dsm + kSlotOff);
  // the block-wise list's arrays: a launch that uses them hands no lists over
  e.cid = reinterpret_cast<int*>(&e.slots[0].l[0][0]);
  e.cl = reinterpret_cast<float*>(e.cid + kCandCap);
  e.crank = reinterpret_cast<int*>(&e.slots[1].l[0][0]);
  e.cord = e.crank + kCandCap;
  if (threadIdx.x == 0) {
    for (int i = 0; i < kNBuf; ++i) {
      mbar_init(&S.full[i], 1);
      mbar_init(&S.empty[i], kCW);
    }
    for (int i = 0; i < kSlots; ++i) {
      mbar_init(&S.done[i], kCW);
      mbar_init(&S.free[i], 1);
    }
    S.issued = 0;
    S.consumed = 0;
    S.ncand = 0;
#ifdef MDS_PHASE_TIMERS
    for (int i = 0; i < kPhaseN; ++i) S.tm[i] = 0ull;
#endif
    mbar_init_fence();
  }
  // Roles: the CTAs on the first dec_sms SMs run decisions (kDecWarps
  // decision warps each, the rest of their warps idle), every other CTA
  // streams slices (eight compute warps, a scheduler warp, a publishing warp).
  // Decisions are serial code of single warps, bound by latencies and
  // instruction fetches: on their own SMs they share neither issue slots nor
  // the instruction caches with the stream (B = 256, K = 8, V = 128256 WIS: a
  // decision warp in every CTA instead took 1.2 times as long).
  __shared__ int role;
  if (threadIdx.x == 0) {
    unsigned smid;
    asm volatile("mov.u32 %0, %%smid;" : "=r"(smid));
    role = (smid < (unsigned)p.dec_sms) ? 1 : 0;
  }
  __syncthreads();
  PT_T0(t_kernel);
  if (role) {
    // the parameters into shared memory, where the decision code reads them
    static_assert(sizeof(Params) % 4 == 0, "parameter copy in words");
    for (int i = threadIdx.x; i < (int)(sizeof(Params) / 4); i += kBlock)
      reinterpret_cast<int*>(&g_dp)[i] = reinterpret_cast<const int*>(&p)[i];
    __syncthreads();
    const int w = threadIdx.x >> 5;
    if (w < kDecWarps) decision_warp<DT>();
  } else if (threadIdx.x >= kCT + 32) {
    e.publisher();
  } else if (threadIdx.x >= kCT) {
    e.scheduler();
  } else {
    e.compute();
  }
  __syncthreads();
  // copies issued but never consumed (only after an abort): wait for them
  if (threadIdx.x == kCT) {
    for (int k = S.consumed; k < S.issued; ++k) (void)e.wait_mbar(&S.full[k % kNBuf], (k / kNBuf) & 1);
  }
  __syncthreads();
#ifdef MDS_PHASE_TIMERS
  if (threadIdx.x == 0) S.tm[kPhKernel] += (unsigned long long)(clock64() - t_kernel);
  __syncthreads();
  if (threadIdx.x < kPhaseN) atomicAdd(&g_phase[threadIdx.x], S.tm[threadIdx.x]);
#endif
  if (threadIdx.x == 0) {
    __threadfence();
    const unsigned out = atomicAdd(&p.ctl[kCtlExit], 1u);
    if (out == gridDim.x - 1) {
      // every CTA has left: reset for the next launch
      if (ld_relaxed(&p.ctl[kCtlAbort]))
        for (int b = 0; b < p.B; ++b) p.cnt[b] = 0u;
      p.ctl[kCtlHead] = 0u;
      p.ctl[kCtlTail] = 0u;
      p.ctl[kCtlDecHead] = 0u;
      p.ctl[kCtlDecTail] = 0u;
      p.ctl[kCtlDone] = 0u;
      p.ctl[kCtlAbort] = 0u;
      __threadfence();
      p.ctl[kCtlExit] = 0u;
    }
  }
}

size_t dyn_smem() { return (size_t)kDynBytes; }

}  // namespace

size_t seq_bytes() { return sizeof(FSeq); }

namespace {
size_t up256(size_t x) { return (x + 255) / 256 * 256; }
struct Layout {
  size_t ctl, tag, dtag, cnt, seq, rec;
  size_t cap, dcap;
};
Layout layout(const Params& p, int nseq, int grid) {
  Layout L;
  L.cap = (size_t)nseq * p.ng + (size_t)grid + 64;   // every sequence's tasks of one pass, plus the claims
  L.dcap = (size_t)nseq + (size_t)grid * kDecWarps + 64;   // one request per sequence, plus the claims
  L.ctl = kCtlWords * 4;
  L.tag = up256(L.cap * 8);
  L.dtag = up256(L.dcap * 8);
  L.cnt = up256((size_t)nseq * 4);
  L.seq = up256((size_t)nseq * sizeof(FSeq));
  L.rec = up256((size_t)nseq * p.ns * p.rec_floats * 4);
  return L;
}
}  // namespace

size_t workspace_bytes(const Params& p, int nseq, int grid) {
  const Layout L = layout(p, nseq, grid);
  return L.ctl + 2 * L.tag + 2 * L.dtag + L.cnt + L.seq + L.rec;
}

size_t clear_bytes(const Params& p, int nseq, int grid) {
  const Layout L = layout(p, nseq, grid);
  return L.ctl + 2 * L.tag + 2 * L.dtag + L.cnt;
}

void carve_workspace(Params& p, char* w, int nseq, int grid) {
  const Layout L = layout(p, nseq, grid);
  p.ctl = reinterpret_cast<unsigned*>(w);
  w += L.ctl;
  p.ring_tag = reinterpret_cast<unsigned long long*>(w);
  w += L.tag;
  p.ring_rtag = reinterpret_cast<unsigned long long*>(w);
  w += L.tag;
  p.dec_tag = reinterpret_cast<unsigned long long*>(w);
  w += L.dtag;
  p.dec_rtag = reinterpret_cast<unsigned long long*>(w);
  w += L.dtag;
  p.cnt = reinterpret_cast<unsigned*>(w);
  w += L.cnt;
  p.seq = w;
  w += L.seq;
  p.rec = reinterpret_cast<float*>(w);
  p.ring_cap = (int)L.cap;
  p.dec_cap = (int)L.dcap;
}

// SMs whose CTAs run the decisions, at least one and never all of them: a
// twentieth of the grid's SMs for single, whose decisions are short, a tenth
// for WIS, a seventh for WIS0, which streams one row only per decision.  By
// scheme alone, set at B = 256, K = 8, V = 128256 and B = 1024, V = 151936
// (us a call on 152 SMs): single 4 SMs 655, 8 439, 12 451, 18 466; WIS 8 272,
// 12 226, 15 219, 22 222; WIS0 12 197, 15 181, 18 161, 22 162.  Batches of 64 to
// 300 at V = 50272 to 151936 move by 2% from 8 SMs on.  Many sequences of short
// rows want more: B = 1024, V = 32000 WIS 15 SMs 341, 28 229, WIS0 22 221, 28
// 193.  The environment variable MDS_DEC_SMS overrides the count (read once
// per process), for tuning.
int decision_sms(int grid, int scheme) {
  static const int env = [] {
    const char* e = getenv("MDS_DEC_SMS");
    return e ? atoi(e) : 0;
  }();
  const int sms = grid / kCtasPerSm;
  int d = env > 0 ? env : (scheme == MDS_SINGLE ? (sms + 10) / 20 : (scheme == MDS_WIS0 ? (sms + 3) / 7 : (sms + 5) / 10));
  if (d < 1) d = 1;
  if (d > sms - 1) d = sms - 1;
  return d;
}

bool plan_geometry(Params& p, int grid) {
  const int es = p.esize;
  int nstream;
  int list = 0;
  if (p.scheme == MDS_WIS0) {
    nstream = 1;
    list = 1;
  } else if (p.scheme == MDS_WIS) {
    nstream = 1 + p.n_models;
    list = (p.K > 1 && nstream <= kListRowsMax) ? 1 : 0;
  } else if (p.scheme == MDS_SINGLE) {
    nstream = 2;
  } else {
    return false;
  }
  if (nstream > kMaxRows) return false;
  int Tmax = kBufBytes / (nstream * es);   // the slice buffer's bound
  Tmax = (Tmax / kSliceQuantum) * kSliceQuantum;
  if (Tmax < kSliceQuantum) return false;
  const int cap = list ? kMaxSlicesList : kMaxSlices;
  int ns = (p.V + Tmax - 1) / Tmax;
  if (ns > cap) return false;
  // enough tasks for the grid: at least two per CTA at depth 0 where the
  // vocabulary allows
  const long want = (2L * grid + p.B - 1) / p.B;
  if (ns < want) {
    const int nsw = (int)(want < cap ? want : cap);
    int T = (p.V + nsw - 1) / nsw;
    T = ((T + kSliceQuantum - 1) / kSliceQuantum) * kSliceQuantum;
    // a unit for every thread at least: shorter slices cost their fixed work
    // (record, count, combine) and use fewer lanes
    if (T < kCT * (16 / es)) T = kCT * (16 / es);
    if (T > Tmax) T = Tmax;
    ns = (p.V + T - 1) / T;
  }
  p.ln = list ? ((p.scheme == MDS_WIS0 && p.omega0 >= 32) ? 64 : 32) : 0;
  if (p.ln > kListMax) return false;
  const int lrows = list ? nstream : 0;
  // a decision stages a pass's records ([ns][rec_floats]) in its warp's
  // staging area: fewer, longer slices where they would not fit
  const int ns_min = (p.V + Tmax - 1) / Tmax;
  for (;; --ns) {
    if (ns < ns_min) return false;
    int T = (p.V + ns - 1) / ns;
    T = ((T + kSliceQuantum - 1) / kSliceQuantum) * kSliceQuantum;
    if (T > Tmax) return false;
    ns = (p.V + T - 1) / T;
    p.T = T;
    p.ns = ns;
    // a slice's list: enough that the slices' lists together hold the
    // sequence's list whenever its tokens are spread over the slices (a
    // slice holding more of them only shortens the certified list)
    if (list) {
      const int base = (p.scheme == MDS_WIS0) ? 16 : 8;
      // twice a slice's even share (the long list of a small batch: four times)
      const int share = (p.ln > 32 && (long)p.B * ns <= 2L * grid) ? 4 : 2;
      int lns = (share * p.ln + ns - 1) / ns;
      lns = (lns + 7) / 8 * 8;
      p.lns = lns < base ? base : (lns > p.ln ? p.ln : lns);
      p.lns_rcp = (unsigned)((0x100000000ull + (unsigned)p.lns - 1u) / (unsigned)p.lns);
    } else {
      p.lns = 0;
    }
    int rf = kHdr + p.lns * (1 + lrows);
    if (rf < 4 + 4 * kTopF) rf = 4 + 4 * kTopF;
    const int runs = (T * es / 16 + 31) / 32;
    if (rf < 4 + runs) rf = 4 + runs;
    p.rec_floats = (rf + 3) & ~3;
      if ((size_t)ns * p.rec_floats * 4 <= (size_t)kDecStage && ns * p.lns <= kMaxEntries) break;
  }
  // Warp-wise candidate lists where every thread has a unit and the slice's
  // list is short.  Each warp's bound is one that as many of its tokens reach
  // as the slice's list holds, so the list is the slice's largest tokens
  // wherever they lie (up to ties at the bound).
  p.fast_list = (list && p.T * es / 16 >= kCT && p.lns <= kSliceListMax) ? 1 : 0;
  p.kth = p.lns;
  p.group = p.group0 = 1;
  p.ng = p.ng0 = p.ns;
  p.dec_sms = decision_sms(grid, p.scheme);
  return p.dec_sms > 0;
}

// Slices per task: the scheduler's round trips for one task (claim, ring
// word, descriptor: about 2 us) are shared by a group of slices where there
// are many tasks per CTA; one slice a task where a pass's slices should
// spread over the GPU.  By the call's own batch: by the context's largest, a
// small call's slices went to a few CTAs one after the other.  Later passes
// and depth 0, us a call at 64, 19, 13, 13 and 3 slices a CTA: single B = 1024,
// V = 151936 1/1 491, 1/4 480, 2/4 436, 4/4 439; B = 300 1/1 164, 1/4 155, 2/4
// 158, 4/8 164; WIS B = 256, V = 128256 1/1 214, 1/4 218, 2/4 225, 4/4 235; two
// models B = 128, V = 50272 1/1 150, 1/4 156, 2/4 162, 4/4 178; B = 64,
// V = 128256 1/1 146, 1/2 144, 2/2 154, 4/4 166.
void plan_tasks(Params& p, int grid, int B) {
  const long per_cta = (long)B * p.ns / grid;
  p.group = per_cta >= 32 ? 4 : (per_cta >= 16 ? 2 : 1);
  p.group0 = per_cta >= 8 ? 4 : (per_cta >= 4 ? 2 : 1);   // depth 0: every sequence's slices at once
  p.ng = (p.ns + p.group - 1) / p.group;
  p.ng0 = (p.ns + p.group0 - 1) / p.group0;
  p.B = B;
}

// Every token's probability under given row statistics, by prob_of.
template <int DT>
__global__ void probs_kernel(const char* row, int V, float M, float invZ, float c, float* out) {
  for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < V; x += gridDim.x * blockDim.x)
    out[x] = prob_of(Elt<DT>::global(row, x), M, c, invZ);
}

cudaError_t launch_probs(const void* row, int dtype, int V, float M, float invZ, float c, float* out,
                         cudaStream_t stream) {
  const int blocks = (V + 255) / 256 < 1024 ? (V + 255) / 256 : 1024;
  if (dtype == MDS_BF16)
    probs_kernel<MDS_BF16><<<blocks, 256, 0, stream>>>(static_cast<const char*>(row), V, M, invZ, c, out);
  else
    probs_kernel<MDS_F32><<<blocks, 256, 0, stream>>>(static_cast<const char*>(row), V, M, invZ, c, out);
  return cudaGetLastError();
}

int grid_size(int device) {
  int sms = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess) return 0;
  int per = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, flow_kernel<MDS_BF16>, kBlock, dyn_smem()) != cudaSuccess)
    return 0;
  int per32 = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per32, flow_kernel<MDS_F32>, kBlock, dyn_smem()) != cudaSuccess)
    return 0;
  if (per32 < per) per = per32;
  return per * sms;
}

cudaError_t configure(int) {
  // both logit types: the grid size is taken over both
  cudaError_t e = cudaFuncSetAttribute((const void*)flow_kernel<MDS_F32>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)dyn_smem());
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute((const void*)flow_kernel<MDS_BF16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)dyn_smem());
  return e;
}

int read_phase_timers(unsigned long long* out, int n) {
#ifdef MDS_PHASE_TIMERS
  unsigned long long h[kPhaseN];
  if (cudaDeviceSynchronize() != cudaSuccess) return -1;
  if (cudaMemcpyFromSymbol(h, g_phase, sizeof(h)) != cudaSuccess) return -1;
  const unsigned long long z[kPhaseN] = {};
  if (cudaMemcpyToSymbol(g_phase, z, sizeof(z)) != cudaSuccess) return -1;
  const int m = n < kPhaseN ? n : kPhaseN;
  for (int i = 0; i < m; ++i) out[i] = h[i];
  return kPhaseN;
#else
  (void)out;
  (void)n;
  return -2;
#endif
}

cudaError_t launch(const Params& p, int grid, cudaStream_t stream) {
  const size_t smem = dyn_smem();
  if (p.dtype == MDS_F32) {
    flow_kernel<MDS_F32><<<grid, kBlock, smem, stream>>>(p);
  } else {
    flow_kernel<MDS_BF16><<<grid, kBlock, smem, stream>>>(p);
  }
  return cudaGetLastError();
}

}  // namespace flow
}  // namespace mds
