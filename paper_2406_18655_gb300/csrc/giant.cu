// One giant shot decoded by the whole GPU: BP (Sec. 4.3) with one thread per check and per
// variable, every iteration in one cooperative launch (grid barriers between the check and
// variable halves), then P-LSD (App. B, Alg. 2): every invalid cluster grows in parallel, clusters
// merge through a lock-free union-find, and each cluster keeps its own on-the-fly
// elimination (Sec. 4.2) in a block of a device arena.
//
// Results are those of the batch decoder (and of the oracle) on the same shot: growth is
// synchronous, ties are broken by the (LLR, index) key, and a cluster's pivot columns do not
// depend on how its elimination rows are numbered.
//
// Cluster state.  Clusters are named by seed ordinal (flipped detectors in the order the
// seeding kernel meets them; the labels do not affect any result).  A cluster root r owns a
// block of cap[r] slots (a multiple of 32; W = cap/32 words per row):
//   R[cap][W]   reduced pivot rows over the cluster's slots (row p exists iff pcol[p] >= 0)
//   T[cap][W]   the combination of pivot columns giving each row
//   pcol[cap]   pivot column of a slot (-1 none), det[cap] detector of a slot
//   sred[W]     the cluster's syndrome reduced by the pivots (zero iff valid, Def. 4.2)
//   xsol[W]     the pivot columns whose sum gives the cleared part of the syndrome
// A detector's slot in its cluster is lslot[d].  When clusters merge, the absorbed blocks
// are copied into the root's (new) block at an offset, rows shifted by that many bits: the
// row supports are disjoint, so the merged rows stay reduced.
//
// All in one cooperative launch, a grid barrier after each phase.  Per growth step:
//   find      every candidate fault offers its key to the growing clusters next to it
//   union     each invalid cluster takes its best candidate; collisions unite clusters
//   plan      union-find paths compressed to one hop; slot offsets of absorbed clusters and of
//             newly claimed detectors, per root
//   relocate  a root that merged or outgrew its block moves to a new, larger block
//   absorb    absorbed blocks copied (shifted) into their root's block; new detectors get slots,
//             and faults next to them become candidates
//   add       each changed root adds its new columns in key order (on-the-fly elimination);
//             the invalid ones are the next step's
#include <algorithm>
#include <climits>
#include <cstdint>
#include <cstring>
#include <new>
#include <utility>
#include <vector>

#include "bp_shot.cuh"
#include "lsd_internal.cuh"

using namespace lsdgb;

namespace {

constexpr unsigned kFullMask = 0xffffffffu;
constexpr unsigned long long kNoKey = ~0ull;
constexpr int kWcMax = 8;                     // reduction words per lane
constexpr int kMaxSlots = 32 * 32 * kWcMax;   // 8192 detectors per cluster
constexpr int kLsdBlock = 1024;               // threads of a block of the persistent P-LSD
constexpr int kTailClusters = 64;             // invalid clusters that one block goes on with
// bound of its barrier waits, from the last sign of progress on: a phase may hold thousands of
// eliminations in one large cluster, and block 0 goes through the last steps alone
constexpr long long kLsdLimitNs = 30000000000LL;
constexpr int kUfLimit = 1 << 20;             // bound on union-find retries and path length
// a minimum over an empty set (a check of degree 1): 2^100, as in the batch kernels
constexpr float kEmptyMinF = 1267650600228229401496703205376.0f;

struct GCtr {
  // whole call
  int ns, nfront, unsolvable, overflow, uf_fail, too_big, ndep, dep_top;
  int bp_stop, bp_unsat[2], bp_iters, bp_conv, bp_fail;
  unsigned bar_arrive;  // grid barrier of the persistent launches
  int progress;         // P-LSD: changes while blocks that the others wait for get on
  int nu, kappa, steps, stuck;
  int ninv[2];
  // reset every step
  int nmerged, nchg, nnew, nclaim, bucket_top, pad;
  unsigned long long arena_top;  // words
};

struct GD {
  int m, n;
  const int *chk_ptr, *chk_var, *var_ptr, *var_chk;
  const float* prior;
  // BP: position-major (ELL) tables padded with -1: ell_col[k * m + i] = column of the k-th
  // edge of check i; ell_pos[k * n + j] = position (k' * m + i) of the k-th edge of column j
  // in ascending row order.  Messages r[dc * m] live at those positions.
  int dc, dv;
  const int *ell_col, *ell_pos;
  float *r, *lam;
  // per detector / per fault
  int *dlab, *lslot, *fst, *front;
  // per seed ordinal (at most m)
  int *parent, *inv0, *inv1, *mlist, *chg, *cap, *nsl, *ncol, *grow, *mark, *extra,
      *newslots, *aoff, *newcnt, *boff;
  unsigned long long *best, *blk;
  // per step lists (at most m entries each)
  int *nc_g, *nc_r, *nc_rank, *bucket, *cl_d, *cl_r, *cl_rel;
  unsigned long long* nc_key;
  unsigned* arena;
  unsigned long long arena_words;
  GCtr* ctr;
  // LSD-mu (App. D): growth steps, reprocessing (-1 OSD-E, w >= 0 OSD-CS-w), cost weights;
  // dependent columns met by the elimination [n] and their per-root buckets
  int order, osd_cs;
  const long long* wfix;
  int *dep_f, *dep_rank, *dep_bucket, *depcnt, *depoff;
};

__host__ __device__ inline size_t blk_words(int C) {
  const int W = C >> 5;
  return 2 * (size_t)C * W + 2 * (size_t)C + 2 * (size_t)W;
}

struct Blk {
  unsigned* b;
  int C, W;
  __device__ unsigned* R(int p) const { return b + (size_t)p * W; }
  __device__ unsigned* T(int p) const { return b + (size_t)C * W + (size_t)p * W; }
  __device__ int* pcol() const { return reinterpret_cast<int*>(b + 2 * (size_t)C * W); }
  __device__ int* det() const { return pcol() + C; }
  __device__ unsigned* sred() const { return reinterpret_cast<unsigned*>(det() + C); }
  __device__ unsigned* xsol() const { return sred() + W; }
};

__device__ __forceinline__ Blk blk_at(const GD& g, unsigned long long off, int C) {
  Blk B;
  B.b = g.arena + off;
  B.C = C;
  B.W = C >> 5;
  return B;
}

__device__ __forceinline__ Blk blk_of(const GD& g, int r) {
  return blk_at(g, g.blk[r], g.cap[r]);
}

__device__ long long arena_alloc(const GD& g, size_t words) {
  const unsigned long long off = atomicAdd(&g.ctr->arena_top, (unsigned long long)words);
  if (off + words > g.arena_words) {
    atomicOr(&g.ctr->overflow, 1);
    return -1;
  }
  return (long long)off;
}

// Next place of a counter for each of the warp's active lanes, one atomic for all of them.
__device__ __forceinline__ int take_place(int* ctr) {
  const unsigned act = __activemask();
  const int lane = threadIdx.x & 31, lead = __ffs(act) - 1;
  int base = 0;
  if (lane == lead) base = atomicAdd(ctr, __popc(act));
  return __shfl_sync(act, base, lead) + __popc(act & ((1u << lane) - 1u));
}

__device__ __forceinline__ unsigned long long llr_key(float x, int j) {
  x = __fadd_rn(x, 0.0f);  // -0 -> +0
  unsigned u = __float_as_uint(x);
  u = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
  return ((unsigned long long)u << 32) | (unsigned)j;
}

__device__ __forceinline__ long long gtid() {
  return (long long)blockIdx.x * blockDim.x + threadIdx.x;
}
__device__ __forceinline__ long long gstride() { return (long long)gridDim.x * blockDim.x; }
__device__ __forceinline__ long long gwarp() { return gtid() >> 5; }
__device__ __forceinline__ long long gwarps() { return gstride() >> 5; }

// ---------------------------------------------------------------------------------------
// BP over one shot (flooding min-sum, every operation rounded to float in the order of the
// batch kernels and of the oracle's FP32 mirror)
// ---------------------------------------------------------------------------------------

__global__ void __launch_bounds__(256) gbp_init(GD g) {
  const long long slots = (long long)g.dc * g.m;
  for (long long k = gtid(); k < slots; k += gstride()) g.r[k] = 0.0f;
  for (long long j = gtid(); j < g.n; j += gstride()) g.lam[j] = g.prior[j];
}

// Iteration t (t >= 1): q = Lam - r on every edge of a check, then the scaled min-sum
// message.  For t >= 2 its return value (a check is unsatisfied) also tests the hard decision
// [Lam < 0] of iteration t-1 against s (Sec. 4.3's early exit; sign bits stand for "< 0": no
// Lam is -0): ored into bp_unsat[t & 1], once per block; the variable half of iteration t
// stops the shot, keeping Lam of iteration t-1, when it passed.
// A warp reads 32 consecutive checks' k-th edges: the column indices and messages are
// contiguous, Lam is gathered.
template <int DCMAX>
__device__ __forceinline__ bool check_phase(const GD& g, const uint8_t* __restrict__ s,
                                            float alpha) {
  bool bad = false;
  for (long long i = gtid(); i < g.m; i += gstride()) {
    unsigned hp = s[i] ? 0x80000000u : 0u;  // bit 31: syndrome ^ signs of Lam
    unsigned sx = 0u;                        // bit 31: signs of q
    float m1 = kEmptyMinF, m2 = kEmptyMinF;
    int am = -1, deg = 0;
    unsigned qb[DCMAX];
#pragma unroll
    for (int k = 0; k < DCMAX; ++k) {
      qb[k] = 0u;
      const int j = k < g.dc ? g.ell_col[(long long)k * g.m + i] : -1;
      if (j < 0) continue;
      const float L = __ldcg(&g.lam[j]);  // L2: written by other blocks
      hp ^= __float_as_uint(L);
      const float q = __fsub_rn(L, __ldcg(&g.r[(long long)k * g.m + i]));
      qb[k] = __float_as_uint(q);
      sx ^= qb[k];
      const float a = fabsf(q);
      if (a < m1) {
        m2 = m1;
        m1 = a;
        am = k;
      } else if (a < m2) {
        m2 = a;
      }
      deg = k + 1;
    }
    bad |= (hp >> 31) != 0u;
    const unsigned par = (s[i] ? 0x80000000u : 0u) ^ sx;
    const float mag1 = __fmul_rn(alpha, m1), mag2 = __fmul_rn(alpha, m2);
#pragma unroll
    for (int k = 0; k < DCMAX; ++k) {
      if (k >= deg) continue;
      const float mag = k == am ? mag2 : mag1;
      g.r[(long long)k * g.m + i] =
          __uint_as_float(__float_as_uint(mag) | ((par ^ qb[k]) & 0x80000000u));
    }
  }
  return bad;
}

template <int DCMAX>
__global__ void __launch_bounds__(256) gbp_check(GD g, const uint8_t* __restrict__ s,
                                                  float alpha, int t) {
  if (*(volatile int*)&g.ctr->bp_stop) return;
  const bool bad = check_phase<DCMAX>(g, s, alpha);
  if (__syncthreads_or(t >= 2 && bad) && threadIdx.x == 0) atomicOr(&g.ctr->bp_unsat[t & 1], 1);
}

// Lam of iteration t: prior plus the incoming messages in ascending check order.
__device__ __forceinline__ void var_phase(const GD& g) {
  for (long long j = gtid(); j < g.n; j += gstride()) {
    float L = g.prior[j];
    for (int k = 0; k < g.dv; ++k) {
      const int p = g.ell_pos[(long long)k * g.n + j];
      if (p < 0) break;
      L = __fadd_rn(L, __ldcg(&g.r[p]));
    }
    g.lam[j] = L;
  }
}

// Iteration t's decision before its variable half: stop (true) when iteration t-1
// satisfied the syndrome (unsat: its test's result), keeping its posteriors; else clear the
// next test's slot.
__device__ __forceinline__ bool bp_converged_before(const GD& g, int t, int unsat) {
  if (t >= 2 && unsat == 0) {
    if (gtid() == 0) {
      g.ctr->bp_conv = 1;
      g.ctr->bp_iters = t - 1;
      g.ctr->bp_stop = 1;
    }
    return true;
  }
  if (gtid() == 0) {
    g.ctr->bp_unsat[(t + 1) & 1] = 0;
    g.ctr->bp_iters = t;
  }
  return false;
}

__global__ void __launch_bounds__(256) gbp_var(GD g, int t) {
  if (*(volatile int*)&g.ctr->bp_stop) return;
  if (bp_converged_before(g, t, *(volatile int*)&g.ctr->bp_unsat[t & 1])) return;
  var_phase(g);
}

// The test after the last iteration T (slot (T+1) & 1, cleared by iteration T).
__device__ __forceinline__ bool syn_phase(const GD& g, const uint8_t* __restrict__ s) {
  bool bad = false;
  for (long long i = gtid(); i < g.m; i += gstride()) {
    unsigned hp = s[i] ? 0x80000000u : 0u;
    for (int k = 0; k < g.dc; ++k) {
      const int j = g.ell_col[(long long)k * g.m + i];
      if (j < 0) break;
      hp ^= __float_as_uint(__ldcg(&g.lam[j]));
    }
    bad |= (hp >> 31) != 0u;
  }
  return bad;
}

__global__ void __launch_bounds__(256) gbp_syn(GD g, const uint8_t* __restrict__ s, int slot) {
  if (*(volatile int*)&g.ctr->bp_stop) return;
  const bool bad = syn_phase(g, s);
  if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(&g.ctr->bp_unsat[slot], 1);
}

// Grid-wide barrier of the persistent launches (all blocks co-resident: cooperative launch).
// The arrival counter only grows; barrier b waits for b * gridDim.x arrivals.  Before arriving
// the block ors `bad` over its threads into *flag; the return value is *flag after the barrier,
// or -1: the wait is bounded by limit_ns of the global timer since its start or the last change
// of `progress` that it saw, past it the block flags bp_fail and every block leaves at its next
// barrier, the host reporting LSD_ERR_TIMEOUT.  Only one thread of a block reads the flags.  `arrive` false (the timeout test only) withholds this
// block's arrival.
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ int grid_barrier(const GD& g, unsigned target, long long limit_ns,
                                            int* flag, bool bad, bool arrive = true) {
  __shared__ int s_flag;
  const int any = __syncthreads_or(bad);
  if (threadIdx.x == 0) {
    if (any) atomicOr(flag, 1);
    __threadfence();
    if (arrive) atomicAdd(&g.ctr->bar_arrive, 1u);
    bool ok = true;
    unsigned long long t0 = 0;
    int seen = 0;
    for (unsigned spin = 1; *(volatile unsigned*)&g.ctr->bar_arrive < target; ++spin) {
      if (spin & 63u) continue;  // the clock and the flags are looked at now and then
      const unsigned long long now = global_ns();
      const int got_to = *(volatile int*)&g.ctr->progress;
      if (t0 == 0 || got_to != seen) t0 = now;
      seen = got_to;
      if ((long long)(now - t0) > limit_ns) atomicOr(&g.ctr->bp_fail, 1);
      if (*(volatile int*)&g.ctr->bp_fail) {
        ok = false;
        break;
      }
    }
    __threadfence();
    s_flag = ok ? *(volatile int*)flag : -1;
  }
  __syncthreads();
  const int f = s_flag;
  __syncthreads();
  return f;
}

// Frame of the persistent launches: check half, barrier, decision, variable half, barrier, for
// all T iterations, then the last test.  hold != 0 (the timeout test only): block 0 withholds
// its first arrival.
template <class Check, class Var, class Syn>
__device__ __forceinline__ void bp_persistent(const GD& g, int T, long long limit_ns, int hold,
                                              Check&& check, Var&& var, Syn&& syn) {
  unsigned target = 0;
  const unsigned nb = gridDim.x;
  for (int t = 1; t <= T; ++t) {
    const bool bad = check(t);
    target += nb;
    const int unsat = grid_barrier(g, target, limit_ns, &g.ctr->bp_unsat[t & 1], t >= 2 && bad,
                                   !(hold && t == 1 && blockIdx.x == 0));
    if (unsat < 0) return;
    if (bp_converged_before(g, t, unsat)) return;
    var();
    target += nb;
    if (grid_barrier(g, target, limit_ns, &g.ctr->bp_unsat[t & 1], false) < 0) return;
  }
  const bool bad = syn();
  target += nb;
  const int unsat = grid_barrier(g, target, limit_ns, &g.ctr->bp_unsat[(T + 1) & 1], bad);
  if (unsat >= 0 && gtid() == 0) {
    g.ctr->bp_conv = unsat == 0;
    g.ctr->bp_stop = 1;
  }
}

// Any graph: tables and messages through L2.
template <int DCMAX>
__global__ void __launch_bounds__(256) gbp_persistent(GD g, const uint8_t* __restrict__ s,
                                                       float alpha, int T, long long limit_ns,
                                                       int hold, int, int) {
  bp_persistent(
      g, T, limit_ns, hold, [&](int) { return check_phase<DCMAX>(g, s, alpha); },
      [&] { var_phase(g); }, [&] { return syn_phase(g, s); });
}

// Graphs whose tables fit the SMs' shared memory (640 000 faults, 307 200 detectors of column
// weight 3 to 4: 217 KB of each): one block per SM, thread t owns the checks and variables
// (c gridDim + block) blockDim + t; their tables, priors and messages stay on chip, so an
// iteration moves the gathered posteriors and messages and the stored ones, half of what
// gbp_persistent moves, and each half waits for one L2 access instead of two in a row.
// Measured per iteration at 640 000 faults: gbp_persistent 24.6 us, this kernel 10.4 (15.0 with
// the gathers past the L1: half of them are of single words, and 1024 consecutive checks or
// variables share their sectors); 160 000 faults, 10.3 -> 4.5 us.  Of that, one arrival and one
// flag update per block instead of 1216 blocks' and every warp's, and a poll without sleep.
// The gathers are plain loads: the barrier's fences on both sides make other blocks' stores
// visible to them (and drop stale L1 lines).
// Same values as gbp_persistent (the check update is that of the batch kernels, bp_shot.cuh).
constexpr int kResDc = 8, kResDv = 4, kResC = 2, kResV = 6;
__global__ void __launch_bounds__(1024) gbp_resident(GD g, const uint8_t* __restrict__ s, float alpha,
                                                      int T, long long limit_ns, int hold, int cpt,
                                                      int vpt) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int NT = blockDim.x, tid = threadIdx.x;
  int* const col = reinterpret_cast<int*>(smem);                  // [cpt][dc][NT], -1 past a row
  float* const msg = reinterpret_cast<float*>(col + cpt * g.dc * NT);
  int* const pos = reinterpret_cast<int*>(msg + cpt * g.dc * NT);  // [vpt][dv][NT], -1 past a column
  float* const pri = reinterpret_cast<float*>(pos + vpt * g.dv * NT);
  const int i0 = blockIdx.x * NT + tid, step = gridDim.x * NT;
  unsigned sbits = 0;
  for (int c = 0; c < cpt; ++c) {
    const int i = i0 + c * step;
    if (i < g.m && s[i]) sbits |= 1u << c;
    for (int k = 0; k < g.dc; ++k) {
      col[(c * g.dc + k) * NT + tid] = i < g.m ? g.ell_col[(long long)k * g.m + i] : -1;
      msg[(c * g.dc + k) * NT + tid] = 0.f;
    }
  }
  for (int v = 0; v < vpt; ++v) {
    const int j = i0 + v * step;
    for (int k = 0; k < g.dv; ++k)
      pos[(v * g.dv + k) * NT + tid] = j < g.n ? g.ell_pos[(long long)k * g.n + j] : -1;
    pri[v * NT + tid] = j < g.n ? g.prior[j] : 0.f;
  }
  const float kInf = __uint_as_float(0x7f800000u);
  // the gathers of every check (variable) are asked for before any is used
  auto check = [&](int t) {
    const float* const lam = t == 1 ? g.prior : g.lam;
    float q[kResC][kResDc];
#pragma unroll
    for (int c = 0; c < kResC; ++c)
#pragma unroll
      for (int k = 0; k < kResDc; ++k) {
        const int j = c < cpt && k < g.dc ? col[(c * g.dc + k) * NT + tid] : -1;
        q[c][k] = j >= 0 ? lam[j] : kInf;  // +inf changes no minimum, sign or parity
      }
    bool bad = false;
#pragma unroll
    for (int c = 0; c < kResC; ++c) {
      const uint32_t sbit = (sbits >> c) << 31;
      uint32_t hp = sbit;
      float x[kResDc];
#pragma unroll
      for (int k = 0; k < kResDc; ++k) {
        hp ^= __float_as_uint(q[c][k]);
        if (c < cpt && k < g.dc) q[c][k] = __fsub_rn(q[c][k], msg[(c * g.dc + k) * NT + tid]);
      }
      bad |= (hp >> 31) != 0u;
      excluded_min<kResDc>(q[c], x);
      const float salpha = __uint_as_float(__float_as_uint(alpha) ^ sbit);
      const int i = i0 + c * step;
#pragma unroll
      for (int k = 0; k < kResDc; ++k) {
        if (c < cpt && k < g.dc && i < g.m) {
          const float y = __fmul_rn(x[k], salpha);
          msg[(c * g.dc + k) * NT + tid] = y;
          g.r[(long long)k * g.m + i] = y;  // (a place past the row's end is read by nobody)
        }
      }
    }
    return bad;
  };
  auto var = [&] {
    float in[kResV][kResDv];
#pragma unroll
    for (int v = 0; v < kResV; ++v)
#pragma unroll
      for (int k = 0; k < kResDv; ++k) {
        const int p = v < vpt && k < g.dv ? pos[(v * g.dv + k) * NT + tid] : -1;
        in[v][k] = p >= 0 ? g.r[p] : 0.f;  // + 0 leaves the sum as it is (never -0)
      }
#pragma unroll
    for (int v = 0; v < kResV; ++v) {
      const int j = i0 + v * step;
      if (v < vpt && j < g.n) {
        float L = pri[v * NT + tid];
#pragma unroll
        for (int k = 0; k < kResDv; ++k) L = __fadd_rn(L, in[v][k]);
        g.lam[j] = L;
      }
    }
  };
  bp_persistent(g, T, limit_ns, hold, check, var, [&] { return syn_phase(g, s); });
}

__global__ void gbp_final(GD g, int slot) {
  if (g.ctr->bp_stop) return;
  g.ctr->bp_conv = g.ctr->bp_unsat[slot] == 0;
  g.ctr->bp_stop = 1;
}

__global__ void __launch_bounds__(256) gcopy_hard(GD g, uint8_t* __restrict__ corr) {
  for (long long j = gtid(); j < g.n; j += gstride()) corr[j] = g.lam[j] < 0.0f ? 1 : 0;
}

// ---------------------------------------------------------------------------------------
// P-LSD
// ---------------------------------------------------------------------------------------

// The threads that share a phase: the grid's, or one block's.
struct Span {
  long long tid, n;
};
__device__ __forceinline__ Span grid_span() { return {gtid(), gstride()}; }

__device__ int gfind(const GD& g, int x) {
  const volatile int* par = g.parent;
  for (int it = 0; it < kUfLimit; ++it) {
    const int p = par[x];
    if (p == x) return x;
    x = p;
  }
  atomicOr(&g.ctr->uf_fail, 1);
  return x;
}

// Links the larger root under the smaller; the absorbed root is listed once in mlist.
__device__ void gunite(const GD& g, int a, int b) {
  for (int it = 0; it < kUfLimit; ++it) {
    a = gfind(g, a);
    b = gfind(g, b);
    if (a == b) return;
    if (a < b) {
      const int t = a;
      a = b;
      b = t;
    }
    if (atomicCAS(g.parent + a, a, b) == a) {
      const int k = take_place(&g.ctr->nmerged);
      g.mlist[k] = a;
      return;
    }
  }
  atomicOr(&g.ctr->uf_fail, 1);
}

__device__ __forceinline__ void add_candidate(const GD& g, int f) {
  if (atomicCAS(&g.fst[f], -2, -1) == -2) g.front[take_place(&g.ctr->nfront)] = f;
}

__device__ __forceinline__ void glsd_reset(const GD& g, const Span& S, uint8_t* corr) {
  for (long long d = S.tid; d < g.m; d += S.n) g.dlab[d] = -1;
  for (long long j = S.tid; j < g.n; j += S.n) g.fst[j] = -2;
  for (long long j = S.tid; j < g.n; j += S.n) corr[j] = 0;
}

// One cluster per flipped detector (Alg. 2's initialization), each in a 32-slot block: seed `ord`
// takes the ord-th block of the arena.  The seeds' candidates are dealt to the lanes by (seed,
// edge) and collected per block: an atomic on one counter per warp took as long as the rest.
__device__ __forceinline__ void glsd_seed(const GD& g, const Span& S, const uint8_t* __restrict__ s) {
  constexpr int C = 32;
  constexpr int words = 2 * C + 2 * C + 2;  // blk_words(C)
  constexpr int kFound = 2048;
  __shared__ int s_found[kFound], s_det[32][32], s_cnt[32], s_nfound, s_base;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int dc = g.dc;
  for (long long b0 = S.tid - threadIdx.x; b0 < g.m; b0 += S.n) {
    const long long d = b0 + threadIdx.x;
    const bool seed = d < g.m && s[d] != 0;
    const unsigned sb = __ballot_sync(kFullMask, seed);
    const int cnt = __popc(sb), rank = __popc(sb & ((1u << lane) - 1u));
    if (seed) s_det[warp][rank] = (int)d;
    if (lane == 0) s_cnt[warp] = cnt;
    if (threadIdx.x == 0) s_nfound = 0;
    __syncthreads();
    // ordinals: the warps' counts summed by warp 0, one atomic for the block
    if (warp == 0) {
      const int mine = lane < (int)(blockDim.x >> 5) ? s_cnt[lane] : 0;
      int pre = mine;
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(kFullMask, pre, o);
        if (lane >= o) pre += v;
      }
      int base = 0;
      if (lane == 31 && pre) {
        base = atomicAdd(&g.ctr->ns, pre);
        atomicAdd(&g.ctr->ninv[0], pre);
        atomicAdd(&g.ctr->arena_top, (unsigned long long)words * pre);
      }
      base = __shfl_sync(kFullMask, base, 31);
      s_cnt[lane] = base + pre - mine;
    }
    __syncthreads();
    const int ord0 = s_cnt[warp];
    const unsigned long long off0 = (unsigned long long)ord0 * words;
    const bool fits = off0 + (unsigned long long)words * cnt <= g.arena_words;
    if (cnt && !fits && lane == 0) atomicOr(&g.ctr->overflow, 1);
    if (seed) {
      const int ord = ord0 + rank;
      g.dlab[d] = ord;
      g.lslot[d] = 0;
      g.parent[ord] = ord;
      g.inv0[ord] = ord;
    }
    if (fits) {
      for (int w = lane; w < words * cnt; w += 32) {
        const int q = w % words;  // pcol = -1, det[0] the seed, sred[0] = 1
        g.arena[off0 + w] = (unsigned)(q - 2 * C) < (unsigned)C ? 0xffffffffu
                            : q == 3 * C ? (unsigned)s_det[warp][w / words] : q == 4 * C ? 1u : 0u;
      }
      if (seed) {
        const int ord = ord0 + rank;
        g.blk[ord] = off0 + (unsigned long long)rank * words;
        g.cap[ord] = C;
        g.nsl[ord] = 1;
        g.ncol[ord] = 0;
        g.grow[ord] = 1;
        g.best[ord] = kNoKey;
        g.mark[ord] = 0;
        g.extra[ord] = 0;
        g.newslots[ord] = 0;
        g.newcnt[ord] = 0;
        g.depcnt[ord] = 0;
      }
      for (int i = lane; i < cnt * dc; i += 32) {
        const int ds = s_det[warp][i / dc];
        const int e = g.chk_ptr[ds] + i % dc;
        if (e >= g.chk_ptr[ds + 1]) continue;
        const int f = g.chk_var[e];
        if (atomicCAS(&g.fst[f], -2, -1) != -2) continue;
        const int k = atomicAdd(&s_nfound, 1);
        if (k < kFound) s_found[k] = f;
        else g.front[atomicAdd(&g.ctr->nfront, 1)] = f;
      }
    }
    __syncthreads();
    const int nf = min(s_nfound, kFound);
    if (threadIdx.x == 0 && nf) s_base = atomicAdd(&g.ctr->nfront, nf);
    __syncthreads();
    for (int k = threadIdx.x; k < nf; k += blockDim.x) g.front[s_base + k] = s_found[k];
    __syncthreads();
  }
}

// find_candidate: every live candidate offers its key to the growing roots next to it.  The
// step's counters are cleared here (nothing in this phase reads them).
__device__ __forceinline__ void glsd_find(const GD& g, const Span& S, const float* __restrict__ llr, int par) {
  if (S.tid == 0) {
    g.ctr->nmerged = g.ctr->nchg = g.ctr->nnew = g.ctr->nclaim = g.ctr->bucket_top = 0;
    g.ctr->ninv[par ^ 1] = 0;
  }
  const int nf = g.ctr->nfront;
  for (long long i = S.tid; i < nf; i += S.n) {
    const int f = g.front[i];
    if (g.fst[f] != -1) continue;
    const unsigned long long key = llr_key(llr[f], f);
    for (int q = g.var_ptr[f]; q < g.var_ptr[f + 1]; ++q) {
      const int c = g.dlab[g.var_chk[q]];
      if (c < 0) continue;
      const int R = g.parent[c];
      if (g.grow[R]) atomicMin(&g.best[R], key);
    }
  }
}

// The same from the side of a few growing roots: warps share the 32-slot chunks of each.
__device__ __forceinline__ void glsd_find_roots(const GD& g, const Span& S,
                                                const float* __restrict__ llr, int par) {
  if (S.tid == 0) {
    g.ctr->nmerged = g.ctr->nchg = g.ctr->nnew = g.ctr->nclaim = g.ctr->bucket_top = 0;
    g.ctr->ninv[par ^ 1] = 0;
  }
  const int cnt = g.ctr->ninv[par];
  const int* inv = par ? g.inv1 : g.inv0;
  const int lane = threadIdx.x & 31;
  const long long warp = S.tid >> 5, warps = S.n >> 5;
  for (int t0 = 0; t0 < cnt; t0 += 32) {
    const int mine = t0 + lane < cnt ? inv[t0 + lane] : 0;
    const int nmine = t0 + lane < cnt ? g.nsl[mine] : 0;
    for (int i = 0; i < min(32, cnt - t0); ++i) {
      const int n = __shfl_sync(kFullMask, nmine, i);
      const long long c0 = (warp + warps - i % warps) % warps;
      if (c0 * 32 >= n) continue;
      const int r = __shfl_sync(kFullMask, mine, i);
      const Blk D = blk_of(g, r);
      unsigned long long best = kNoKey;
      for (long long c = c0; c * 32 < n; c += warps) {
        const long long sl = c * 32 + lane;
        if (sl >= n) continue;
        const int d = D.det()[sl];
        for (int e = g.chk_ptr[d]; e < g.chk_ptr[d + 1]; ++e) {
          const int f = g.chk_var[e];
          if (g.fst[f] == -1) best = min(best, llr_key(llr[f], f));
        }
      }
      for (int off = 16; off > 0; off >>= 1)
        best = min(best, __shfl_xor_sync(kFullMask, best, off));
      if (lane == 0 && best != kNoKey) atomicMin(&g.best[r], best);
    }
  }
}

// parallel_union: each invalid cluster takes its pick; collisions unite.
__device__ __forceinline__ void glsd_union(const GD& g, const Span& S, int par, int strict) {
  const int cnt = g.ctr->ninv[par];
  const int* inv = par ? g.inv1 : g.inv0;
  const int per = 1 + g.dv;  // a thread per pick and per detector next to it
  for (long long t = S.tid; t < (long long)cnt * per; t += S.n) {
    const int r = inv[t / per], i = (int)(t % per);
    const unsigned long long key = g.best[r];
    if (key == kNoKey) {
      if (strict && i == 0) atomicOr(&g.ctr->unsolvable, 1);  // LSD-mu: a full cluster just stops
      continue;
    }
    const int f = (int)(key & 0xffffffffu);
    if (i == 0) {
      const int old = atomicCAS(&g.fst[f], -1, r);
      if (old == -1) {
        const int k = take_place(&g.ctr->nnew);
        g.nc_g[k] = f;
        g.nc_r[k] = r;
        g.nc_key[k] = key;
      } else {
        gunite(g, r, old);
      }
      continue;
    }
    const int q = g.var_ptr[f] + i - 1;
    if (q >= g.var_ptr[f + 1]) continue;
    const int d = g.var_chk[q];
    const int o = atomicCAS(&g.dlab[d], -1, r);
    if (o == -1) {
      const int k = take_place(&g.ctr->nclaim);
      g.cl_d[k] = d;
      g.cl_r[k] = r;
    } else if (o != r) {
      gunite(g, r, o);
    }
  }
}

__device__ __forceinline__ void mark_changed(const GD& g, int R) {
  if (atomicCAS(&g.mark[R], 0, 1) == 0) g.chg[take_place(&g.ctr->nchg)] = R;
}

// Offsets inside each root's grown block: absorbed clusters, then new detectors; ranks of
// the new columns.  The labels used below are left one hop from their root, with `flat` all
// labels (a step without a union leaves them so).
__device__ __forceinline__ void glsd_plan(const GD& g, const Span& S, bool flat) {
  const int nm = g.ctr->nmerged, nc = g.ctr->nclaim, nn = g.ctr->nnew;
  const int ns = flat && nm > 0 ? g.ctr->ns : 0;
  for (long long x = S.tid; x < ns; x += S.n) g.parent[x] = gfind(g, (int)x);
  for (long long t = S.tid; t < (long long)nm + nc + nn; t += S.n) {
    const int k = (int)(t < nm ? t : t < nm + nc ? t - nm : t - nm - nc);
    const int A = t < nm ? g.mlist[k] : t < nm + nc ? g.cl_r[k] : g.nc_r[k];
    const int R = gfind(g, A);
    g.parent[A] = R;
    if (t < nm)
      g.aoff[A] = atomicAdd(&g.extra[R], g.nsl[A]);
    else if (t < nm + nc)
      g.cl_rel[k] = atomicAdd(&g.newslots[R], 1);
    else
      g.nc_rank[k] = atomicAdd(&g.newcnt[R], 1);
    mark_changed(g, R);
  }
}

// A root that merged or outgrew its block moves to a new zeroed block (its own slots copied
// at the same positions); every changed root reserves room for its new columns' list.
__device__ __forceinline__ void glsd_relocate(const GD& g, const Span& S) {
  const int lane = threadIdx.x & 31;
  const int nchg = g.ctr->nchg;
  for (long long t = (S.tid >> 5); t < nchg; t += (S.n >> 5)) {
    const int R = g.chg[t];
    const int base = g.nsl[R];
    const int need = base + g.extra[R] + g.newslots[R];
    if (lane == 0) g.boff[R] = atomicAdd(&g.ctr->bucket_top, g.newcnt[R]);
    if (need > kMaxSlots) {
      if (lane == 0) atomicOr(&g.ctr->too_big, 1);
      continue;
    }
    const Blk O = blk_of(g, R);
    if (g.extra[R] == 0 && need <= O.C) {
      for (int p = base + lane; p < need; p += 32) O.pcol()[p] = -1;
      continue;
    }
    const int want = need + need / 2;
    const int C = max(O.C, min(kMaxSlots, max(32, (want + 31) & ~31)));  // never shrinks
    const size_t words = blk_words(C);
    long long off = 0;
    if (lane == 0) off = arena_alloc(g, words);
    off = __shfl_sync(kFullMask, off, 0);
    if (off < 0) continue;
    const Blk N = blk_at(g, (unsigned long long)off, C);
    for (size_t w = lane; w < words; w += 32) N.b[w] = 0u;
    __syncwarp();
    for (int p = lane; p < C; p += 32) N.pcol()[p] = p < base ? O.pcol()[p] : -1;
    for (int p = lane; p < base; p += 32) N.det()[p] = O.det()[p];
    for (int w = lane; w < O.W; w += 32) {
      N.sred()[w] = O.sred()[w];
      N.xsol()[w] = O.xsol()[w];
    }
    for (int p = 0; p < base; ++p) {
      if (O.pcol()[p] < 0) continue;
      for (int w = lane; w < O.W; w += 32) {
        N.R(p)[w] = O.R(p)[w];
        N.T(p)[w] = O.T(p)[w];
      }
    }
    __syncwarp();
    if (lane == 0) {
      g.blk[R] = (unsigned long long)off;
      g.cap[R] = C;
    }
  }
}

// Word w of a bit vector `src` (sw words) shifted up by `sh` bits.
__device__ __forceinline__ unsigned shifted_word(const unsigned* src, int sw, int sh, int w) {
  const int q = sh >> 5, b = sh & 31;
  const int i = w - q;
  unsigned v = (i >= 0 && i < sw) ? src[i] << b : 0u;
  if (b && i - 1 >= 0 && i - 1 < sw) v |= src[i - 1] >> (32 - b);
  return v;
}

// The same for a cluster of at most 32 slots by one thread (into a fresh block: zero words are
// left out).
__device__ __forceinline__ void or_shifted(unsigned* dst, unsigned v, int o) {
  const int q = o >> 5, b = o & 31;
  if (v << b) atomicOr(&dst[q], v << b);
  if (b && (v >> (32 - b))) atomicOr(&dst[q + 1], v >> (32 - b));
}
__device__ __forceinline__ void absorb_small(const GD& g, const Blk& A, const Blk& D, int o, int nA) {
  or_shifted(D.sred(), A.sred()[0], o);
  or_shifted(D.xsol(), A.xsol()[0], o);
  for (int p = 0; p < nA; ++p) {
    const int c = A.pcol()[p], d = A.det()[p];
    D.pcol()[o + p] = c;
    D.det()[o + p] = d;
    g.lslot[d] = o + p;
    if (c < 0) continue;
    or_shifted(D.R(o + p), A.R(p)[0], o);
    or_shifted(D.T(o + p), A.T(p)[0], o);
  }
}

// Absorbed clusters copied into their root's block at their offset (rows shifted): a warp per
// cluster; where there are more of them than warps (the first step: single seeds) a warp takes
// `per`, a lane each, and the ones of more than 8 slots together.
__device__ __forceinline__ void glsd_absorb(const GD& g, const Span& S) {
  const int lane = threadIdx.x & 31;
  const int nm = g.ctr->nmerged;
  if (g.ctr->too_big || g.ctr->overflow) return;
  const long long warps = S.n >> 5;
  const int per = (int)min(32LL, (nm + warps - 1) / warps);
  for (long long t0 = (S.tid >> 5) * per; t0 < nm; t0 += warps * per) {
    const bool have = lane < per && t0 + lane < nm;
    const int mine = have ? g.mlist[t0 + lane] : 0;
    const int mroot = have ? g.parent[mine] : 0;
    const int mn = have ? g.nsl[mine] : 0;
    const int mo = have ? g.nsl[mroot] + g.aoff[mine] : 0;
    const bool small = have && per > 1 && mn <= 8;
    if (small) absorb_small(g, blk_of(g, mine), blk_of(g, mroot), mo, mn);
    if (have) {
      const int nc = g.ncol[mine];
      if (nc) atomicAdd(&g.ncol[mroot], nc);
    }
    __syncwarp();
    for (unsigned left = __ballot_sync(kFullMask, have && !small); left; left &= left - 1) {
      const int src = __ffs(left) - 1;
      const Blk A = blk_of(g, __shfl_sync(kFullMask, mine, src));
      const Blk D = blk_of(g, __shfl_sync(kFullMask, mroot, src));
      const int o = __shfl_sync(kFullMask, mo, src), nA = __shfl_sync(kFullMask, mn, src);
      for (int p = lane; p < nA; p += 32) {
        D.pcol()[o + p] = A.pcol()[p];
        const int d = A.det()[p];
        D.det()[o + p] = d;
        g.lslot[d] = o + p;
      }
      const int w0 = o >> 5, w1 = min(D.W, ((o + nA + 31) >> 5) + 1);
      for (int w = w0 + lane; w < w1; w += 32) {
        const unsigned a = shifted_word(A.sred(), A.W, o, w);
        const unsigned b = shifted_word(A.xsol(), A.W, o, w);
        if (a) atomicOr(&D.sred()[w], a);
        if (b) atomicOr(&D.xsol()[w], b);
      }
      for (int p = 0; p < nA; ++p) {
        if (A.pcol()[p] < 0) continue;
        for (int w = w0 + lane; w < w1; w += 32) {
          D.R(o + p)[w] = shifted_word(A.R(p), A.W, o, w);
          D.T(o + p)[w] = shifted_word(A.T(p), A.W, o, w);
        }
      }
    }
  }
}

// New detectors take their slots; faults next to them become candidates (Def. 4.3); the new
// columns are placed in their root's list.
__device__ __forceinline__ void glsd_claim(const GD& g, const Span& S) {
  const int nc = g.ctr->nclaim, nn = g.ctr->nnew;
  if (g.ctr->too_big || g.ctr->overflow) return;
  const int dc = g.dc;  // a thread per new detector and edge
  for (long long t = S.tid; t < (long long)nc * dc + nn; t += S.n) {
    if (t < (long long)nc * dc) {
      const int k = (int)(t / dc), i = (int)(t % dc);
      const int d = g.cl_d[k];
      if (i == 0) {
        const int R = g.parent[g.cl_r[k]];
        const int slot = g.nsl[R] + g.extra[R] + g.cl_rel[k];
        blk_of(g, R).det()[slot] = d;
        g.lslot[d] = slot;
      }
      const int e = g.chk_ptr[d] + i;
      if (e < g.chk_ptr[d + 1]) add_candidate(g, g.chk_var[e]);
    } else {
      const int k = (int)(t - (long long)nc * dc);
      const int R = g.parent[g.nc_r[k]];
      g.bucket[g.boff[R] + g.nc_rank[k]] = k;
    }
  }
}

// Adds fault f to the elimination of block D (nslots slots in use), as the batch kernels do; WC: words
// per lane (one holds 1024 slots, which few clusters outgrow).
template <int WC>
__device__ __forceinline__ void gadd_column(const GD& g, const Blk& D, int nslots, int f, int lane) {
  const int wc = (nslots + 31) >> 5;
  unsigned bw[WC], tw[WC];
#pragma unroll
  for (int c = 0; c < WC; ++c) bw[c] = tw[c] = 0u;
  for (int q = g.var_ptr[f]; q < g.var_ptr[f + 1]; ++q) {
    const int sl = g.lslot[g.var_chk[q]];
    const bool piv = D.pcol()[sl] >= 0;
#pragma unroll
    for (int c = 0; c < WC; ++c) {
      const int w = c * 32 + lane;
      if (w < wc) {
        if ((sl >> 5) == w) bw[c] ^= 1u << (sl & 31);
        if (piv) {
          bw[c] ^= D.R(sl)[w];
          tw[c] ^= D.T(sl)[w];
        }
      }
    }
  }
  int p = -1;
#pragma unroll
  for (int c = 0; c < WC; ++c) {
    const unsigned nz = __ballot_sync(kFullMask, bw[c] != 0u);
    if (p < 0 && nz) {
      const int wl = __ffs(nz) - 1;
      const unsigned word = __shfl_sync(kFullMask, bw[c], wl);
      p = (c * 32 + wl) * 32 + __ffs(word) - 1;
    }
  }
  if (p < 0) {  // dependent column: the span does not change; LSD-mu lists it
    if (g.order > 0 && lane == 0) g.dep_f[atomicAdd(&g.ctr->ndep, 1)] = f;
    return;
  }
  const int pw = p >> 5;
  const unsigned pb = 1u << (p & 31);
#pragma unroll
  for (int c = 0; c < WC; ++c)
    if (c * 32 + lane == pw) tw[c] ^= pb;
  const bool sflag = (D.sred()[pw] & pb) != 0u;
  __syncwarp();
#pragma unroll
  for (int c = 0; c < WC; ++c) {
    const int w = c * 32 + lane;
    if (w < wc) {
      D.R(p)[w] = bw[c];
      D.T(p)[w] = tw[c];
    }
  }
  if (lane == 0) D.pcol()[p] = f;
  __syncwarp();
  for (int d0 = 0; d0 < nslots; d0 += 32) {
    const int d = d0 + lane;
    const bool hit = d < nslots && d != p && D.pcol()[d] >= 0 && (D.R(d)[pw] & pb) != 0u;
    unsigned bal = __ballot_sync(kFullMask, hit);
    while (bal) {
      const int dd = d0 + __ffs(bal) - 1;
      bal &= bal - 1;
#pragma unroll
      for (int c = 0; c < WC; ++c) {
        const int w = c * 32 + lane;
        if (w < wc) {
          D.R(dd)[w] ^= bw[c];
          D.T(dd)[w] ^= tw[c];
        }
      }
    }
    __syncwarp();
  }
  if (sflag) {
#pragma unroll
    for (int c = 0; c < WC; ++c) {
      const int w = c * 32 + lane;
      if (w < wc) {
        D.sred()[w] ^= bw[c];
        D.xsol()[w] ^= tw[c];
      }
    }
  }
  __syncwarp();
}

// The same by one thread, for a cluster of at most 32 slots: a row is one word.
__device__ __forceinline__ void gadd_column_small(const GD& g, const Blk& D, int nslots, int f) {
  unsigned bw = 0u, tw = 0u;
  for (int q = g.var_ptr[f]; q < g.var_ptr[f + 1]; ++q) {
    const int sl = g.lslot[g.var_chk[q]];
    bw ^= 1u << sl;
    if (D.pcol()[sl] >= 0) {
      bw ^= D.R(sl)[0];
      tw ^= D.T(sl)[0];
    }
  }
  if (bw == 0u) {
    if (g.order > 0) g.dep_f[atomicAdd(&g.ctr->ndep, 1)] = f;
    return;
  }
  const int p = __ffs(bw) - 1;
  const unsigned pb = 1u << p;
  tw ^= pb;
  D.R(p)[0] = bw;
  D.T(p)[0] = tw;
  D.pcol()[p] = f;
  for (int d = 0; d < nslots; ++d) {
    if (d == p || D.pcol()[d] < 0) continue;
    const unsigned r = D.R(d)[0];
    if (r & pb) {
      D.R(d)[0] = r ^ bw;
      D.T(d)[0] ^= tw;
    }
  }
  if (D.sred()[0] & pb) {
    D.sred()[0] ^= bw;
    D.xsol()[0] ^= tw;
  }
}

// After the columns of root R: its sizes, and (collect) whether it grows in the next step.
__device__ __forceinline__ void added(const GD& g, int R, int nslots, int cnt, bool invalid,
                                      int par_next, bool collect) {
  g.ncol[R] += cnt;
  g.nsl[R] = nslots;
  g.extra[R] = 0;
  g.newslots[R] = 0;
  g.newcnt[R] = 0;
  g.mark[R] = 0;
  if (!collect) return;
  g.grow[R] = invalid ? 1 : 0;
  if (invalid) {
    g.best[R] = kNoKey;
    (par_next ? g.inv1 : g.inv0)[atomicAdd(&g.ctr->ninv[par_next], 1)] = R;
  }
}

// on_the_fly_elimination of every changed root: its new columns in key order, then its
// validity; collect: the invalid ones are the next step's (an invalid root always changes: it
// takes a fault, or unites with the cluster that took it, or the shot is unsolvable).  A warp
// per root; where there are more roots than warps (the first steps: clusters of a few slots) a
// warp takes `per` of them, a lane each, and works on the larger ones together.
__device__ __forceinline__ void glsd_add(const GD& g, const Span& S, int par_next, bool collect) {
  const int lane = threadIdx.x & 31;
  const int nchg = g.ctr->nchg;
  if (g.ctr->too_big || g.ctr->overflow) return;
  const long long warps = S.n >> 5;
  const int per = (int)min(32LL, (nchg + warps - 1) / warps);
  for (long long t0 = (S.tid >> 5) * per; t0 < nchg; t0 += warps * per) {
    const bool have = lane < per && t0 + lane < nchg;
    const int mine = have ? g.chg[t0 + lane] : 0;
    const int mslots = have ? g.nsl[mine] + g.extra[mine] + g.newslots[mine] : 0;
    const bool small = have && per > 1 && mslots <= 32;
    if (small) {
      const Blk D = blk_of(g, mine);
      const int cnt = g.newcnt[mine];
      const int* bk = g.bucket + g.boff[mine];
      unsigned long long last = 0;
      for (int it = 0; it < cnt; ++it) {
        unsigned long long best = kNoKey;
        int bi = -1;
        for (int u = 0; u < cnt; ++u) {
          const int k = bk[u];
          const unsigned long long key = g.nc_key[k];
          if ((it == 0 || key > last) && key < best) {
            best = key;
            bi = k;
          }
        }
        last = best;
        gadd_column_small(g, D, mslots, g.nc_g[bi]);
      }
      added(g, mine, mslots, cnt, D.sred()[0] != 0u, par_next, collect);
    }
    __syncwarp();
    for (unsigned left = __ballot_sync(kFullMask, have && !small); left; left &= left - 1) {
      const int R = __shfl_sync(kFullMask, mine, __ffs(left) - 1);
      const int nslots = __shfl_sync(kFullMask, mslots, __ffs(left) - 1);
      const Blk D = blk_of(g, R);
      const int cnt = g.newcnt[R];
      const int* bk = g.bucket + g.boff[R];
      unsigned long long last = 0;
      for (int it = 0; it < cnt; ++it) {
        unsigned long long best = kNoKey;
        int bi = -1;
        for (int u = lane; u < cnt; u += 32) {
          const int k = bk[u];
          const unsigned long long key = g.nc_key[k];
          if ((it == 0 || key > last) && key < best) {
            best = key;
            bi = k;
          }
        }
        for (int off = 16; off > 0; off >>= 1) {
          const unsigned long long ob = __shfl_xor_sync(kFullMask, best, off);
          const int oi = __shfl_xor_sync(kFullMask, bi, off);
          if (ob < best) {
            best = ob;
            bi = oi;
          }
        }
        last = best;
        if (nslots <= 1024) {
          gadd_column<1>(g, D, nslots, g.nc_g[bi], lane);
        } else {  // (milliseconds each in the largest clusters)
          if (lane == 0) atomicAdd(&g.ctr->progress, 1);
          gadd_column<kWcMax>(g, D, nslots, g.nc_g[bi], lane);
        }
      }
      bool any = false;
      for (int w = lane; w < ((nslots + 31) >> 5); w += 32) any |= D.sred()[w] != 0u;
      any = __any_sync(kFullMask, any);
      if (lane == 0) added(g, R, nslots, cnt, any, par_next, collect);
      __syncwarp();
    }
  }
}

// LSD-mu: every root grows (App. D's extra steps).
__global__ void __launch_bounds__(256) glsd_collect_all(GD g, int par) {
  const int ns = g.ctr->ns;
  int* inv = par ? g.inv1 : g.inv0;
  for (long long x = gtid(); x < ns; x += gstride()) {
    const bool root = g.parent[x] == x;
    g.grow[x] = root ? 1 : 0;
    if (root) {
      g.best[x] = kNoKey;
      inv[atomicAdd(&g.ctr->ninv[par], 1)] = (int)x;
    }
  }
}

// Dependent columns grouped by final root: rank in the root's bucket, bucket offsets, placement.
__global__ void __launch_bounds__(256) glsd_dep_rank(GD g) {
  const int nd = g.ctr->ndep;
  for (long long k = gtid(); k < nd; k += gstride())
    g.dep_rank[k] = atomicAdd(&g.depcnt[g.parent[g.fst[g.dep_f[k]]]], 1);
}

__global__ void __launch_bounds__(256) glsd_dep_offsets(GD g) {
  const int ns = g.ctr->ns;
  for (long long x = gtid(); x < ns; x += gstride())
    if (g.parent[x] == x && g.depcnt[x] > 0) g.depoff[x] = atomicAdd(&g.ctr->dep_top, g.depcnt[x]);
}

__global__ void __launch_bounds__(256) glsd_dep_place(GD g) {
  const int nd = g.ctr->ndep;
  for (long long k = gtid(); k < nd; k += gstride()) {
    const int R = g.parent[g.fst[g.dep_f[k]]];
    g.dep_bucket[g.depoff[R] + g.dep_rank[k]] = g.dep_f[k];
  }
}

// Cost of root block D's local solution (xsol) with the dependent columns i1, i2 of the
// sorted list flipped (-1 none): tw vectors at tw + i * wc.
__device__ long long gpattern_cost(const GD& g, const Blk& D, int wc, const unsigned* tw,
                                   const int* cols, int i1, int i2) {
  long long cost = 0;
  for (int w = 0; w < wc; ++w) {
    unsigned v = D.xsol()[w];
    if (i1 >= 0) v ^= tw[(size_t)i1 * wc + w];
    if (i2 >= 0) v ^= tw[(size_t)i2 * wc + w];
    while (v) {
      const int b = __ffs(v) - 1;
      v &= v - 1;
      cost += g.wfix[D.pcol()[w * 32 + b]];
    }
  }
  if (i1 >= 0) cost += g.wfix[cols[i1]];
  if (i2 >= 0) cost += g.wfix[cols[i2]];
  return cost;
}

// LSD-mu reprocessing of every root with dependent columns (App. D), as the batch kernels:
// OSD-E over the first min(mu, #dependent) in key order (ties to the smaller pattern), or
// the combination sweep OSD-CS-w (no flip, every single, every pair among the first w; ties
// to the earlier pattern).  A dependent column's representation tw over the pivots is
// recomputed from the root's final rows (the pivots only grow, so it is the same unique
// combination).  Chosen dependent columns go straight to the correction; xsol takes their tw.
__global__ void __launch_bounds__(256) glsd_reprocess(GD g, const float* __restrict__ llr,
                                                       uint8_t* __restrict__ corr) {
  const int lane = threadIdx.x & 31;
  const int ns = g.ctr->ns;
  for (long long x = gwarp(); x < ns; x += gwarps()) {
    if (g.parent[x] != x) continue;
    const int cnt = g.depcnt[x];
    if (cnt == 0) continue;
    const Blk D = blk_of(g, (int)x);
    const int wc = (g.nsl[x] + 31) >> 5;
    const int* bk = g.dep_bucket + g.depoff[x];
    long long off = 0;
    if (lane == 0) off = arena_alloc(g, 1 + 2 * (size_t)cnt + (size_t)cnt * (1 + wc));
    off = __shfl_sync(kFullMask, off, 0);
    if (off < 0) continue;
    off += off & 1;  // 8-byte alignment of the keys
    unsigned long long* keys = reinterpret_cast<unsigned long long*>(g.arena + off);  // [cnt]
    int* cols = reinterpret_cast<int*>(g.arena + off + 2 * (size_t)cnt);            // [cnt]
    unsigned* tw = g.arena + off + 3 * (size_t)cnt;                                  // [cnt][wc]
    // sort the bucket by (LLR, index) key: rank of each entry among the bucket
    for (int u = lane; u < cnt; u += 32) {
      const int f = bk[u];
      const unsigned long long ku = llr_key(llr[f], f);
      int pos = 0;
      for (int v = 0; v < cnt; ++v) {
        const int fv = bk[v];
        pos += llr_key(llr[fv], fv) < ku ? 1 : 0;
      }
      cols[pos] = f;
      keys[pos] = ku;
    }
    __syncwarp();
    // representations over the pivots
    for (int i = 0; i < cnt; ++i) {
      const int f = cols[i];
      for (int w = lane; w < wc; w += 32) {
        unsigned t = 0u;
        for (int q = g.var_ptr[f]; q < g.var_ptr[f + 1]; ++q) {
          const int sl = g.lslot[g.var_chk[q]];
          if (D.pcol()[sl] >= 0) t ^= D.T(sl)[w];
        }
        tw[(size_t)i * wc + w] = t;
      }
    }
    __syncwarp();
    long long bc = LLONG_MAX;
    int b1 = -1, b2 = -1;
    if (g.osd_cs < 0) {
      const int nt = min(g.order, cnt);
      int bt = 0;
      for (int t = lane; t < (1 << nt); t += 32) {
        long long cost = 0;
        for (int w = 0; w < wc; ++w) {
          unsigned v = D.xsol()[w];
          for (int k = 0; k < nt; ++k)
            if ((t >> k) & 1) v ^= tw[(size_t)k * wc + w];
          while (v) {
            const int b = __ffs(v) - 1;
            v &= v - 1;
            cost += g.wfix[D.pcol()[w * 32 + b]];
          }
        }
        for (int k = 0; k < nt; ++k)
          if ((t >> k) & 1) cost += g.wfix[cols[k]];
        if (cost < bc) {
          bc = cost;
          bt = t;
        }
      }
      for (int o = 16; o > 0; o >>= 1) {
        const long long oc = __shfl_xor_sync(kFullMask, bc, o);
        const int ot = __shfl_xor_sync(kFullMask, bt, o);
        if (oc < bc || (oc == bc && ot < bt)) {
          bc = oc;
          bt = ot;
        }
      }
      if (bt == 0) continue;
      for (int w = lane; w < wc; w += 32) {
        unsigned delta = 0u;
        for (int k = 0; k < nt; ++k)
          if ((bt >> k) & 1) delta ^= tw[(size_t)k * wc + w];
        D.xsol()[w] ^= delta;
      }
      for (int k = lane; k < nt; k += 32)
        if ((bt >> k) & 1) corr[cols[k]] = 1;
      __syncwarp();
      continue;
    }
    // combination sweep
    const int wp = min(g.osd_cs, cnt);
    int bcls = 3;
    unsigned long long bkey = 0;
    auto consider = [&](long long c, int cls, unsigned long long key, int i1, int i2) {
      if (c < bc || (c == bc && (cls < bcls || (cls == bcls && key < bkey)))) {
        bc = c;
        bcls = cls;
        bkey = key;
        b1 = i1;
        b2 = i2;
      }
    };
    if (lane == 0) consider(gpattern_cost(g, D, wc, tw, cols, -1, -1), 0, 0, -1, -1);
    for (int i = lane; i < cnt; i += 32)
      consider(gpattern_cost(g, D, wc, tw, cols, i, -1), 1, keys[i], i, -1);
    const int npairs = wp * (wp - 1) / 2;
    for (int t = lane; t < npairs; t += 32) {
      int i = 0, rem = t;
      while (rem >= wp - 1 - i) {
        rem -= wp - 1 - i;
        ++i;
      }
      const int j = i + 1 + rem;
      consider(gpattern_cost(g, D, wc, tw, cols, i, j), 2, (unsigned long long)(i * 16 + j), i, j);
    }
    for (int o = 16; o > 0; o >>= 1) {
      const long long oc = __shfl_xor_sync(kFullMask, bc, o);
      const int ocls = __shfl_xor_sync(kFullMask, bcls, o);
      const unsigned long long okey = __shfl_xor_sync(kFullMask, bkey, o);
      const int o1 = __shfl_xor_sync(kFullMask, b1, o);
      const int o2 = __shfl_xor_sync(kFullMask, b2, o);
      consider(oc, ocls, okey, o1, o2);
    }
    if (b1 < 0) continue;
    for (int w = lane; w < wc; w += 32) {
      unsigned delta = tw[(size_t)b1 * wc + w];
      if (b2 >= 0) delta ^= tw[(size_t)b2 * wc + w];
      D.xsol()[w] ^= delta;
    }
    if (lane == 0) {
      corr[cols[b1]] = 1;
      if (b2 >= 0) corr[cols[b2]] = 1;
    }
    __syncwarp();
  }
}

// Local solutions (Eq. 2): the pivot columns in each root's xsol; nu and kappa.
__device__ __forceinline__ void glsd_solve(const GD& g, const Span& S, uint8_t* __restrict__ corr, bool write) {
  const int lane = threadIdx.x & 31;
  const int ns = g.ctr->ns;
  for (long long x0 = (S.tid >> 5) * 32; x0 < ns; x0 += S.n) {
    const long long x = x0 + lane;
    const bool root = x < ns && g.parent[x] == x;
    const int nu = __popc(__ballot_sync(kFullMask, root));
    const int kappa = __reduce_max_sync(kFullMask, root ? g.ncol[x] : 0);
    if (lane == 0 && nu) {
      atomicAdd(&g.ctr->nu, nu);
      atomicMax(&g.ctr->kappa, kappa);
    }
  }
  if (!write) return;
  for (long long x = (S.tid >> 5); x < ns; x += (S.n >> 5)) {
    if (g.parent[x] != x) continue;
    const Blk D = blk_of(g, (int)x);
    const int nx = g.nsl[x];
    for (int p = lane; p < nx; p += 32) {
      const int c = D.pcol()[p];
      if (c >= 0 && ((D.xsol()[p >> 5] >> (p & 31)) & 1u)) corr[c] = 1;
    }
  }
}

// One phase per launch: LSD-mu's growth steps (every cluster grows, none is collected).
enum Phase { kFind, kUnion, kPlan, kRelocate, kAbsorb, kAdd, kSolve };
struct PhaseArgs {
  const float* llr;
  const uint8_t* s;
  uint8_t* corr;
};

template <int P>
__global__ void __launch_bounds__(256) glsd_phase(GD g, PhaseArgs a) {
  const Span S = grid_span();
  if constexpr (P == kFind) glsd_find(g, S, a.llr, 0);
  if constexpr (P == kUnion) glsd_union(g, S, 0, 0);
  if constexpr (P == kPlan) glsd_plan(g, S, true);
  if constexpr (P == kRelocate) glsd_relocate(g, S);
  if constexpr (P == kAbsorb) {
    glsd_absorb(g, S);
    glsd_claim(g, S);
  }
  if constexpr (P == kAdd) glsd_add(g, S, 1, false);
  if constexpr (P == kSolve) glsd_solve(g, S, a.corr, true);
}

// P-LSD in one cooperative launch, a grid barrier between the phases: every block reads the
// step's verdict from counters that do not change before the next barrier, so all leave the
// loop together.  Bound by the latency of dependent loads and atomics: a thread or a warp per
// item of a phase, and a barrier of about 2.5 us.  Most steps are the growth of a last few
// clusters: from kTailClusters invalid ones on (their number never grows) block 0 goes on alone,
// with barriers of its own and its L1 kept from phase to phase, and looks for candidates from the
// clusters' side; the others wait at the last grid barrier, whose bound starts again at every step
// of block 0, which leaves in turn when they have given up.  640 000 faults at p = 0.03: 22 steps
// 2.02 -> 0.65 ms, 3 steps 0.56 -> 0.29 (before: nine launches and a look by the host per step,
// 79 us; all steps on the grid: 1.25 ms and 0.39; seeds counted by warp and single seeds absorbed
// by a warp each: 0.71 and 0.36).  kTailClusters 16: the same; 256: 0.07 ms longer.
__global__ void __launch_bounds__(kLsdBlock) glsd_persistent(GD g, PhaseArgs a, long long limit_ns, int hold) {
  unsigned target = 0;
  bool alone = false;
  Span S = grid_span();
  auto grid_sync = [&] {
    target += gridDim.x;
    // hold (the timeout test only): block 0 withholds its first arrival
    const bool arrive = !(hold && target == gridDim.x && blockIdx.x == 0);
    return grid_barrier(g, target, limit_ns, &g.ctr->unsolvable, false, arrive) >= 0;
  };
  auto sync = [&] {
    if (!alone) return grid_sync();
    __syncthreads();
    return true;
  };
  glsd_reset(g, S, a.corr);
  if (!sync()) return;
  glsd_seed(g, S, a.s);
  if (!sync()) return;
  int par = 0, steps = 0;
  const auto failed = [&] { return (g.ctr->overflow | g.ctr->uf_fail | g.ctr->too_big) != 0; };
  while (!failed() && !g.ctr->unsolvable && g.ctr->ninv[par] != 0 && steps <= g.n) {
    if (!alone && g.ctr->ninv[par] <= kTailClusters) {
      alone = true;
      if (blockIdx.x != 0) break;
      S = {(long long)threadIdx.x, (long long)blockDim.x};
    }
    if (alone)
      glsd_find_roots(g, S, a.llr, par);
    else
      glsd_find(g, S, a.llr, par);
    if (!sync()) return;
    glsd_union(g, S, par, 1);
    if (!sync()) return;
    glsd_plan(g, S, !alone);
    if (!sync()) return;
    glsd_relocate(g, S);
    if (!sync()) return;
    glsd_absorb(g, S);
    glsd_claim(g, S);
    if (!sync()) return;
    int given_up = 0;  // (asked for before the phase, so that its reply does not add to the step)
    if (alone && threadIdx.x == 0) {
      atomicAdd(&g.ctr->progress, 1);
      given_up = *(volatile int*)&g.ctr->bp_fail;
    }
    glsd_add(g, S, par ^ 1, true);
    if (alone ? __syncthreads_or(given_up) != 0 : !grid_sync()) return;
    // a step in which some invalid cluster found no candidate does not count (Alg. 1)
    if (g.ctr->unsolvable) break;
    ++steps;
    par ^= 1;
  }
  if (gtid() == 0) {
    g.ctr->steps = steps;
    g.ctr->stuck = g.ctr->unsolvable || (!failed() && g.ctr->ninv[par] != 0);
  }
  if (!grid_sync()) return;
  S = grid_span();
  const bool stuck = g.ctr->stuck != 0;
  if (stuck || (g.order == 0 && !failed())) glsd_solve(g, S, a.corr, !stuck);
  if (g.order > 0)  // LSD-mu's steps look labels up in one hop
    for (long long x = S.tid; x < g.ctr->ns; x += S.n) g.parent[x] = gfind(g, (int)x);
}

}  // namespace

struct lsd_giant {
  int m = 0, n = 0;
  long long E = 0;
  int bp_iters = 0;
  float alpha = 0.625f;
  cudaStream_t st = nullptr;
  int sms = 0;
  GD g{};
  GCtr* h_ctr = nullptr;  // pinned
  std::vector<void*> allocs;
  size_t bytes = 0;
  cudaEvent_t ev[3] = {nullptr, nullptr, nullptr};
  int64_t launches = 0;
  int coop_grid = 0;  // blocks of the persistent BP launch (0: launch per half-iteration)
  const void* coop_fn = nullptr;
  int coop_block = 256, coop_cpt = 0, coop_vpt = 0;  // cpt > 0: gbp_resident
  size_t coop_smem = 0;
  int lsd_grid = 1;  // blocks of glsd_persistent (1: no cooperative launch needed)
  long long bar_limit_ns = 1000000000LL;  // bound of a grid-barrier wait
  int hold_barrier = 0;                   // timeout test: block 0 withholds an arrival
  long long lsd_limit_ns = kLsdLimitNs;   // the same of P-LSD's launch
  int lsd_hold = 0;
};

namespace {

int gfail(cudaError_t e) {
  record_cuda_error(e);
  return e == cudaErrorMemoryAllocation ? LSD_ERR_OOM : LSD_ERR_CUDA;
}

template <class T>
int galloc(lsd_giant* G, T** p, size_t count) {
  const size_t bytes = std::max<size_t>(count * sizeof(T), 16);
  cudaError_t e = cudaMalloc(reinterpret_cast<void**>(p), bytes);
  if (e != cudaSuccess) {
    *p = nullptr;
    return gfail(e);
  }
  G->allocs.push_back(*p);
  G->bytes += bytes;
  return LSD_OK;
}

int grid_threads(const lsd_giant* G) { return G->sms * 8; }

int read_ctr(lsd_giant* G) {
  cudaError_t e = cudaMemcpyAsync(G->h_ctr, G->g.ctr, sizeof(GCtr), cudaMemcpyDeviceToHost,
                                  G->st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(G->st);
  return e == cudaSuccess ? LSD_OK : gfail(e);
}

int check_launch(lsd_giant* G) {
  G->launches++;
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? LSD_OK : gfail(e);
}

template <int P>
int run_phase(lsd_giant* G, const PhaseArgs& a) {
  glsd_phase<P><<<grid_threads(G), 256, 0, G->st>>>(G->g, a);
  return check_launch(G);
}

int step_error(const GCtr& h) {
  if (h.overflow) return LSD_ERR_ADMISSION;
  if (h.uf_fail) return LSD_ERR_TIMEOUT;
  if (h.too_big) return LSD_ERR_UNSUPPORTED;
  return LSD_OK;
}

// P-LSD of the shot; writes corr (zero unless solved) and the info fields.
int run_plsd(lsd_giant* G, const float* llr, const uint8_t* s, uint8_t* corr,
             lsd_giant_info* info) {
  const GD& g = G->g;
  const int grid = grid_threads(G);
  const GCtr& h = *G->h_ctr;
  PhaseArgs a{llr, s, corr};
  int rc;
  cudaError_t e = cudaMemsetAsync(g.ctr, 0, sizeof(GCtr), G->st);
  if (e != cudaSuccess) return gfail(e);
  void* args[] = {(void*)&g, (void*)&a, (void*)&G->lsd_limit_ns, (void*)&G->lsd_hold};
  const void* fn = (const void*)glsd_persistent;
  e = G->lsd_grid > 1 ? cudaLaunchCooperativeKernel(fn, G->lsd_grid, kLsdBlock, args, 0, G->st)
                      : cudaLaunchKernel(fn, 1, kLsdBlock, args, 0, G->st);
  G->launches++;
  if (e != cudaSuccess) return gfail(e);
  if ((rc = read_ctr(G))) return rc;
  if (h.bp_fail) return LSD_ERR_TIMEOUT;
  const bool unsolvable = h.stuck != 0;
  if (!unsolvable && (rc = step_error(h))) return rc;
  // ---- LSD-mu: mu more steps in which every cluster grows, then local reprocessing ----
  if (!unsolvable && g.order > 0) {
    for (int k = 0; k < g.order; ++k) {
      e = cudaMemsetAsync(g.ctr->ninv, 0, sizeof(g.ctr->ninv), G->st);
      if (e != cudaSuccess) return gfail(e);
      glsd_collect_all<<<grid, 256, 0, G->st>>>(g, 0);
      if ((rc = check_launch(G))) return rc;
      if ((rc = run_phase<kFind>(G, a)) || (rc = run_phase<kUnion>(G, a)) ||
          (rc = run_phase<kPlan>(G, a)) || (rc = run_phase<kRelocate>(G, a)) ||
          (rc = run_phase<kAbsorb>(G, a)) || (rc = run_phase<kAdd>(G, a)) ||
          (rc = read_ctr(G)) || (rc = step_error(h)))
        return rc;
      if (h.nnew == 0 && h.nclaim == 0 && h.nmerged == 0) break;  // nothing could grow
    }
    glsd_dep_rank<<<grid, 256, 0, G->st>>>(g);
    if ((rc = check_launch(G))) return rc;
    glsd_dep_offsets<<<grid, 256, 0, G->st>>>(g);
    if ((rc = check_launch(G))) return rc;
    glsd_dep_place<<<grid, 256, 0, G->st>>>(g);
    if ((rc = check_launch(G))) return rc;
    glsd_reprocess<<<grid, 256, 0, G->st>>>(g, llr, corr);
    if ((rc = check_launch(G)) || (rc = run_phase<kSolve>(G, a)) || (rc = read_ctr(G))) return rc;
  }
  if (h.overflow) return LSD_ERR_ADMISSION;
  if (info) {
    info->status = unsolvable ? LSD_SHOT_UNSOLVABLE : LSD_SHOT_OK_LSD;
    info->nu = h.nu;
    info->kappa = h.kappa;
    info->steps = h.steps;
    info->arena_bytes_used = (int64_t)h.arena_top * 4;
  }
  return LSD_OK;
}

}  // namespace

extern "C" {

int lsd_giant_create(lsd_giant** out, int32_t m, int32_t n, int64_t nnz, const int32_t* rows,
                     const int32_t* cols, const float* channel_probs, int32_t bp_iters,
                     int32_t lsd_order, size_t arena_bytes, const lsd_options* opt) {
  if (!out) return LSD_ERR_INVALID_ARG;
  *out = nullptr;
  if (m < 1 || n < 1 || nnz < 1 || nnz >= INT32_MAX || !rows || !cols || !channel_probs ||
      bp_iters < 0)
    return LSD_ERR_INVALID_ARG;
  lsd_options o{};
  if (opt) o = *opt;
  if (o.ms_scaling < 0.f || lsd_order < 0 || o.osd_method < 0 || o.osd_method > 1 ||
      o.osd_cs_order < 0 || o.osd_cs_order > kMaxCsOrder ||
      (o.osd_method == 0 && o.osd_cs_order != 0) ||
      lsd_order > (o.osd_method == 1 ? kMaxCsGrowth : kMaxOrder))
    return LSD_ERR_INVALID_ARG;
  for (int j = 0; j < n; ++j)
    if (!(channel_probs[j] > 0.f && channel_probs[j] < 1.f)) return LSD_ERR_INVALID_ARG;
  std::vector<std::pair<int, int>> e((size_t)nnz);
  for (int64_t k = 0; k < nnz; ++k) {
    if (rows[k] < 0 || rows[k] >= m || cols[k] < 0 || cols[k] >= n) return LSD_ERR_INVALID_ARG;
    e[(size_t)k] = {rows[k], cols[k]};
  }
  std::sort(e.begin(), e.end());
  for (size_t k = 1; k < e.size(); ++k)
    if (e[k] == e[k - 1]) return LSD_ERR_INVALID_ARG;
  const int E = (int)e.size();
  std::vector<int> chk_ptr(m + 1, 0), var_ptr(n + 1, 0), chk_var(E), var_edge(E), var_chk(E);
  for (auto& p : e) {
    chk_ptr[p.first + 1]++;
    var_ptr[p.second + 1]++;
  }
  for (int i = 0; i < m; ++i) chk_ptr[i + 1] += chk_ptr[i];
  for (int j = 0; j < n; ++j) var_ptr[j + 1] += var_ptr[j];
  std::vector<int> fill(var_ptr.begin(), var_ptr.end() - 1);
  for (int k = 0; k < E; ++k) {  // ascending (row, column): each column's list ascends in row
    chk_var[k] = e[k].second;
    const int slot = fill[e[k].second]++;
    var_edge[slot] = k;
    var_chk[slot] = e[k].first;
  }
  int dc = 0, dv = 0;
  for (int i = 0; i < m; ++i) dc = std::max(dc, chk_ptr[i + 1] - chk_ptr[i]);
  for (int j = 0; j < n; ++j) dv = std::max(dv, var_ptr[j + 1] - var_ptr[j]);
  if (dc > 32) return LSD_ERR_UNSUPPORTED;  // check degree of the BP kernel
  std::vector<int> ell_col((size_t)dc * m, -1), ell_pos((size_t)dv * n, -1);
  for (int i = 0; i < m; ++i)
    for (int k = chk_ptr[i]; k < chk_ptr[i + 1]; ++k)
      ell_col[(size_t)(k - chk_ptr[i]) * m + i] = chk_var[k];
  for (int j = 0; j < n; ++j)
    for (int a = var_ptr[j]; a < var_ptr[j + 1]; ++a) {
      const int k = var_edge[a], i = var_chk[a];
      ell_pos[(size_t)(a - var_ptr[j]) * n + j] = (k - chk_ptr[i]) * m + i;
    }
  if ((size_t)dc * m >= (size_t)INT32_MAX) return LSD_ERR_UNSUPPORTED;

  lsd_giant* G = new (std::nothrow) lsd_giant();
  if (!G) return LSD_ERR_OOM;
  G->m = m;
  G->n = n;
  G->E = E;
  G->bp_iters = bp_iters;
  G->alpha = o.ms_scaling > 0.f ? o.ms_scaling : 0.625f;
  G->st = static_cast<cudaStream_t>(o.stream);
  GD& g = G->g;
  g.m = m;
  g.n = n;
  const size_t words = arena_bytes ? arena_bytes / 4 : ((size_t)64 << 20);  // 256 MiB
  int rc = LSD_OK;
  int *d_chk_ptr = nullptr, *d_chk_var = nullptr, *d_var_ptr = nullptr, *d_var_chk = nullptr;
  float *d_prior = nullptr, *d_probs = nullptr;
  long long* d_wfix = nullptr;
  auto A = [&](auto** p, size_t count) {
    if (rc == LSD_OK) rc = galloc(G, p, count);
  };
  A(&d_chk_ptr, m + 1);
  A(&d_chk_var, E);
  A(&d_var_ptr, n + 1);
  A(&d_var_chk, E);
  A(&d_prior, n);
  A(&d_probs, n);
  A(&d_wfix, n);
  int *d_ell_col = nullptr, *d_ell_pos = nullptr;
  A(&d_ell_col, (size_t)dc * m);
  A(&d_ell_pos, (size_t)dv * n);
  A(&g.r, (size_t)dc * m);
  A(&g.lam, n);
  A(&g.dlab, m);
  A(&g.lslot, m);
  A(&g.fst, n);
  A(&g.front, n);
  for (int** p : {&g.parent, &g.inv0, &g.inv1, &g.mlist, &g.chg, &g.cap, &g.nsl, &g.ncol,
                  &g.grow, &g.mark, &g.extra, &g.newslots, &g.aoff, &g.newcnt,
                  &g.boff, &g.nc_g, &g.nc_r, &g.nc_rank, &g.bucket, &g.cl_d, &g.cl_r,
                  &g.cl_rel})
    A(p, m);
  A(&g.best, m);
  A(&g.blk, m);
  A(&g.nc_key, m);
  A(&g.dep_f, n);
  A(&g.dep_rank, n);
  A(&g.dep_bucket, n);
  A(&g.depcnt, m);
  A(&g.depoff, m);
  A(&g.arena, words);
  A(&g.ctr, 1);
  g.arena_words = words;
  if (rc == LSD_OK) {
    cudaError_t err = cudaMallocHost(reinterpret_cast<void**>(&G->h_ctr), sizeof(GCtr));
    if (err != cudaSuccess) rc = gfail(err);
  }
  if (rc == LSD_OK) {
    cudaError_t err = cudaMemcpyAsync(d_chk_ptr, chk_ptr.data(), (m + 1) * sizeof(int),
                                      cudaMemcpyHostToDevice, G->st);
    if (err == cudaSuccess)
      err = cudaMemcpyAsync(d_chk_var, chk_var.data(), (size_t)E * sizeof(int),
                            cudaMemcpyHostToDevice, G->st);
    if (err == cudaSuccess)
      err = cudaMemcpyAsync(d_var_ptr, var_ptr.data(), (n + 1) * sizeof(int),
                            cudaMemcpyHostToDevice, G->st);
    if (err == cudaSuccess)
      err = cudaMemcpyAsync(d_var_chk, var_chk.data(), (size_t)E * sizeof(int),
                            cudaMemcpyHostToDevice, G->st);
    if (err == cudaSuccess)
      err = cudaMemcpyAsync(d_ell_col, ell_col.data(), ell_col.size() * sizeof(int),
                            cudaMemcpyHostToDevice, G->st);
    if (err == cudaSuccess)
      err = cudaMemcpyAsync(d_ell_pos, ell_pos.data(), ell_pos.size() * sizeof(int),
                            cudaMemcpyHostToDevice, G->st);
    if (err == cudaSuccess)
      err = cudaMemcpyAsync(d_probs, channel_probs, (size_t)n * sizeof(float),
                            cudaMemcpyHostToDevice, G->st);
    if (err == cudaSuccess) err = launch_priors(d_probs, d_prior, d_wfix, n, G->st);
    if (err == cudaSuccess) err = cudaStreamSynchronize(G->st);
    if (err != cudaSuccess) rc = gfail(err);
  }
  if (rc == LSD_OK) {
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err == cudaSuccess)
      err = cudaDeviceGetAttribute(&G->sms, cudaDevAttrMultiProcessorCount, dev);
    for (int k = 0; k < 3 && err == cudaSuccess; ++k) err = cudaEventCreate(&G->ev[k]);
    // the persistent BP launch: every block must be resident at once (cooperative launch)
    int coop = 0, per_sm = 0;
    if (err == cudaSuccess) err = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    const void* fn = dc <= 8    ? (const void*)gbp_persistent<8>
                     : dc <= 16 ? (const void*)gbp_persistent<16>
                                : (const void*)gbp_persistent<32>;
    if (err == cudaSuccess && coop)
      err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, 256, 0);
    if (err == cudaSuccess && coop && per_sm > 0) {
      const long long need = (std::max<long long>(m, n) + 255) / 256;
      G->coop_grid = (int)std::min<long long>(need, (long long)per_sm * G->sms);
      G->coop_fn = fn;
      // tables on chip when they fit: a block per SM, as many threads as give each about two
      // variables (at most 1024)
      int max_smem = 0;
      err = cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
      const int block = (int)std::min<long long>(1024, (n / (2LL * G->sms) + 128) / 128 * 128);
      const long long cap = (long long)block * G->sms;
      const long long cpt = (m + cap - 1) / cap, vpt = (n + cap - 1) / cap;
      if (err == cudaSuccess && dc >= 1 && dc <= kResDc && dv <= kResDv && cpt <= kResC && vpt <= kResV) {
        const size_t smem = (size_t)block * 4 * (2 * cpt * dc + vpt * (dv + 1));
        int res_per_sm = 0;
        const void* res = (const void*)gbp_resident;
        if (smem + 1024 <= (size_t)max_smem &&
            allow_max_dynamic_smem(res, max_smem) == cudaSuccess &&
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&res_per_sm, res, block, smem) == cudaSuccess &&
            res_per_sm > 0) {
          G->coop_fn = res;
          G->coop_grid = (int)std::min<long long>(G->sms, (std::max<long long>(m, n) + block - 1) / block);
          G->coop_block = block;
          G->coop_cpt = (int)((m + (long long)block * G->coop_grid - 1) / ((long long)block * G->coop_grid));
          G->coop_vpt = (int)((n + (long long)block * G->coop_grid - 1) / ((long long)block * G->coop_grid));
          G->coop_smem = smem;
        }
        cudaGetLastError();
      }
    }
    // persistent P-LSD: a block per SM, and no more than give every cluster there can be a warp
    if (err == cudaSuccess && coop)
      err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, (const void*)glsd_persistent,
                                                          kLsdBlock, 0);
    if (err == cudaSuccess && coop && per_sm > 0)
      G->lsd_grid = std::min(G->sms, (m + kLsdBlock / 32 - 1) / (kLsdBlock / 32));
    if (err != cudaSuccess) rc = gfail(err);
  }
  g.dc = dc;
  g.dv = dv;
  g.order = lsd_order;
  g.osd_cs = o.osd_method == 1 ? o.osd_cs_order : -1;
  g.wfix = d_wfix;
  g.ell_col = d_ell_col;
  g.ell_pos = d_ell_pos;
  g.chk_ptr = d_chk_ptr;
  g.chk_var = d_chk_var;
  g.var_ptr = d_var_ptr;
  g.var_chk = d_var_chk;
  g.prior = d_prior;
  if (rc != LSD_OK) {
    lsd_giant_destroy(G);
    return rc;
  }
  *out = G;
  return LSD_OK;
}

int lsd_giant_postprocess(lsd_giant* G, const float* llr, const uint8_t* syndrome,
                          uint8_t* correction, lsd_giant_info* info) {
  if (!G || !llr || !syndrome || !correction) return LSD_ERR_INVALID_ARG;
  if (info) std::memset(info, 0, sizeof(*info));
  cudaEventRecord(G->ev[1], G->st);
  const int rc = run_plsd(G, llr, syndrome, correction, info);
  if (rc) return rc;
  cudaEventRecord(G->ev[2], G->st);
  cudaError_t e = cudaEventSynchronize(G->ev[2]);
  if (e != cudaSuccess) return gfail(e);
  if (info) cudaEventElapsedTime(&info->ms_lsd, G->ev[1], G->ev[2]);
  return LSD_OK;
}

int lsd_giant_decode(lsd_giant* G, const uint8_t* syndrome, uint8_t* correction,
                     float* posteriors, lsd_giant_info* info) {
  if (!G || !syndrome || !correction) return LSD_ERR_INVALID_ARG;
  if (info) std::memset(info, 0, sizeof(*info));
  const GD& g = G->g;
  const int grid = grid_threads(G);
  int rc;
  cudaEventRecord(G->ev[0], G->st);
  cudaError_t e = cudaMemsetAsync(g.ctr, 0, sizeof(GCtr), G->st);
  if (e != cudaSuccess) return gfail(e);
  if (G->coop_cpt == 0 || G->bp_iters == 0) {  // (gbp_resident starts from the priors itself)
    gbp_init<<<grid, 256, 0, G->st>>>(g);
    if ((rc = check_launch(G))) return rc;
  }
  // iterations in chunks of 2, 4, 8, ... with a look at the stop flag after each, so that a
  // shot that converges early is not followed by the remaining iterations' launches
  bool stopped = false;
  if (G->bp_iters > 0 && G->coop_grid > 0) {
    // one persistent launch for every iteration (grid barriers between the halves)
    const uint8_t* sp = syndrome;
    float alpha = G->alpha;
    int T = G->bp_iters;
    long long limit = G->bar_limit_ns;
    int hold = G->hold_barrier;
    void* args[] = {(void*)&g,     (void*)&sp,   (void*)&alpha,        (void*)&T,
                    (void*)&limit, (void*)&hold, (void*)&G->coop_cpt, (void*)&G->coop_vpt};
    e = cudaLaunchCooperativeKernel(G->coop_fn, G->coop_grid, G->coop_block, args, G->coop_smem, G->st);
    G->launches++;
    if (e != cudaSuccess) return gfail(e);
    stopped = true;
  }
  for (int t = 1, chunk = 2; t <= G->bp_iters && !stopped; chunk *= 2) {
    const int t1 = std::min(G->bp_iters, t + chunk - 1);
    for (; t <= t1; ++t) {
      if (g.dc <= 8)
        gbp_check<8><<<grid, 256, 0, G->st>>>(g, syndrome, G->alpha, t);
      else if (g.dc <= 16)
        gbp_check<16><<<grid, 256, 0, G->st>>>(g, syndrome, G->alpha, t);
      else
        gbp_check<32><<<grid, 256, 0, G->st>>>(g, syndrome, G->alpha, t);
      if ((rc = check_launch(G))) return rc;
      gbp_var<<<grid, 256, 0, G->st>>>(g, t);
      if ((rc = check_launch(G))) return rc;
    }
    if ((rc = read_ctr(G))) return rc;
    stopped = G->h_ctr->bp_stop != 0;
  }
  if (G->bp_iters > 0 && !stopped) {
    const int slot = (G->bp_iters + 1) & 1;
    gbp_syn<<<grid, 256, 0, G->st>>>(g, syndrome, slot);
    if ((rc = check_launch(G))) return rc;
    gbp_final<<<1, 1, 0, G->st>>>(g, slot);
    if ((rc = check_launch(G))) return rc;
  }
  if (posteriors) {
    e = cudaMemcpyAsync(posteriors, g.lam, (size_t)G->n * sizeof(float),
                        cudaMemcpyDeviceToDevice, G->st);
    if (e != cudaSuccess) return gfail(e);
  }
  cudaEventRecord(G->ev[1], G->st);
  if ((rc = read_ctr(G))) return rc;
  if (G->h_ctr->bp_fail) return LSD_ERR_TIMEOUT;
  const int conv = G->h_ctr->bp_conv, iters = G->h_ctr->bp_iters;
  if (conv) {
    gcopy_hard<<<grid, 256, 0, G->st>>>(g, correction);
    if ((rc = check_launch(G))) return rc;
    if (info) info->status = LSD_SHOT_OK_BP;
  } else {
    rc = run_plsd(G, g.lam, syndrome, correction, info);
    if (rc) return rc;
  }
  cudaEventRecord(G->ev[2], G->st);
  e = cudaEventSynchronize(G->ev[2]);
  if (e != cudaSuccess) return gfail(e);
  if (info) {
    info->bp_iterations = iters;
    cudaEventElapsedTime(&info->ms_bp, G->ev[0], G->ev[1]);
    cudaEventElapsedTime(&info->ms_lsd, G->ev[1], G->ev[2]);
  }
  return LSD_OK;
}

int lsd_giant_test_hold_barrier(lsd_giant* G, int32_t hold, int64_t limit_ns) {
  if (!G || limit_ns < 0) return LSD_ERR_INVALID_ARG;
  if (!G->coop_grid) return LSD_ERR_UNSUPPORTED;
  G->hold_barrier = hold ? 1 : 0;
  G->bar_limit_ns = hold ? (long long)limit_ns : 1000000000LL;
  return LSD_OK;
}

int lsd_giant_test_lsd_bound(lsd_giant* G, int32_t hold, int64_t limit_ns) {
  if (!G || limit_ns < 0) return LSD_ERR_INVALID_ARG;
  G->lsd_hold = hold ? 1 : 0;
  G->lsd_limit_ns = limit_ns ? (long long)limit_ns : kLsdLimitNs;
  return LSD_OK;
}

int lsd_giant_kernel_launches(const lsd_giant* G, int64_t* count) {
  if (!G || !count) return LSD_ERR_INVALID_ARG;
  *count = G->launches;
  return LSD_OK;
}

int lsd_giant_destroy(lsd_giant* G) {
  if (!G) return LSD_OK;
  cudaStreamSynchronize(G->st);
  for (void* p : G->allocs) cudaFree(p);
  if (G->h_ctr) cudaFreeHost(G->h_ctr);
  for (auto& ev : G->ev)
    if (ev) cudaEventDestroy(ev);
  delete G;
  return LSD_OK;
}

}  // extern "C"
