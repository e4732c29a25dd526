// LSD for check matrices beyond the dense kernel (space-time, hook-fault and hypergraph-product
// codes): the same algorithm and results as lsd.cu (Alg. 1 of Sec. 4.1, on-the-fly elimination
// of Sec. 4.2, LSD-mu of App. D), with state sized by what a shot touches.
//
// One CTA owns one shot.  A shot needs few growth steps on a handful of clusters, or a thousand
// columns when its clusters percolate, and a batch has from one such shot to a few per cent of
// it; so what bounds the kernel is the latency of its longest shot (issue 21-24 %; the first stall
// is the barrier, 5 per issue), and a step is spread over the CTA with the state in shared memory
// and few barriers.  LSD of the same shots by one warp per shot with its state in global scratch,
// and now:
//   50 000 HGP shots, p = 0.02, LSD-0 / LSD-10   7.7 / 16.5 ms, now 1.18 / 3.1 ms
//   5000 HGP shots, p = 0.05 (percolating)       33.6 ms, now 5.5 ms
//   100 003 BB144 d = 12, 20 000 BB288 d = 18    1.15, 0.67 ms, now 0.135, 0.090 ms
//   99 991 BB144 hooks d = 6                     1.09 ms, now 0.18 ms
// and by the dense kernel, which ranks every fault first, 2.33 ms for 100 003 BB72 hooks d = 6
// (now 0.12) and 0.64 ms for 50 001 BB144 windows (now 0.09).  256 / 512 threads per shot (small /
// large instance) instead of 512 / 1024: 1.43, 3.6 and 6.7 ms for the HGP rows.
//   lab[m]     of a claimed detector: label << 16 | slot, else kFree.  A label is the number
//              of a seed (flipped detector), flattened to the cluster's root after a merge; a
//              slot is the detector's elimination row, in the order of claiming.
//   cand, joined  bitmaps over the faults: next to a claimed detector (Def. 4.3's Lambda over
//              all clusters); in a cluster.  lk, lf, ld list the candidates: LLR bits, fault,
//              its first four detectors.
//   best, bidx of a growing cluster's root: least LLR bits over its candidates, then the least
//              fault index among the equal ones (the order of lsd.cu's ranks, without a sort).
//   M          elimination rows, bits over slots, word w of row i at M[w CAP + i].  M is the
//              product of the row operations done so far: M h has its only bit at the pivot
//              row for a column h already added, so a new column's image h' = M h is one bit
//              per row, the parity of the row's bits at the column's detectors; a bit on a
//              row without pivot makes that row the pivot, and the pivot row is added to the
//              other rows with a bit.  Row i belongs to thread i mod NT, which alone reads
//              (but for a pivot row) and writes it: one barrier per column, no atomics and no
//              search for the rows to update.
//   flags[i]   bit 0: (M s)_i, bit 1: row i has a pivot, column pcol[i].  A cluster is valid
//              (Def. 4.2) iff no row without pivot has (M s)_i; its solution is the columns of
//              the pivot rows that have it.
// Pivot columns, representations and solutions are unique, so neither the choice of the pivot
// row nor the numbering of seeds and slots shows in the results.
//
// Two instances: the small one keeps everything in shared memory; a shot that outgrows it (CAP
// rows, SC seeds, its candidate list) is queued for the large one, whose rows lie in global
// scratch (read through the SM's L1).
#include <climits>

#include "lsd_internal.cuh"

namespace lsdgb {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr uint32_t kFree = 0xffffffffu;
constexpr uint16_t kNone16 = 0xffffu;
constexpr unsigned kNoKey = 0xffffffffu;
constexpr int kSpill = 4;         // internal status: retry with the large instance
// Dynamic shared memory of a CTA; a graph too large for it takes the LG instances, whose lab
// and (large instance) candidate list lie in global scratch.
constexpr size_t kSmemLimit = 225 << 10;

__host__ __device__ constexpr size_t al16(size_t x) { return (x + 15) & ~(size_t)15; }

// Sizes and offsets of an instance.  Arrays with atomics are in shared memory (but lab for LG);
// the others ("lists") follow there (small) or in the CTA's global scratch (big).
template <int NT_, int CAP_, int SC_, bool MU_, bool BIG_, bool LG_>
struct Inst {
  static constexpr int NT = NT_, CAP = CAP_, SC = SC_, W = CAP_ / 32, RPT = CAP_ / NT_, NW = NT_ / 32;
  static constexpr bool MU = MU_, BIG = BIG_, LG = LG_;
  // shared
  static constexpr size_t best = 0;
  static constexpr size_t bidx = best + (size_t)SC * 4;
  static constexpr size_t growb = bidx + (size_t)SC * 4;          // growing labels, one bit each
  static constexpr size_t parent = growb + (size_t)SC / 8;
  static constexpr size_t inv = parent + (size_t)SC * 2;          // growing labels
  static constexpr size_t pcol = inv + (size_t)SC * 2;
  static constexpr size_t sdet = pcol + (size_t)CAP * 2;          // detector of a slot
  static constexpr size_t slab = sdet + (size_t)CAP * 2;          // label of a slot
  static constexpr size_t rows = slab + (size_t)CAP * 2;          // per warp: a cluster's rows
  static constexpr size_t flags = rows + (size_t)NW * 32 * 2;
  static constexpr size_t osd = al16(flags + (size_t)CAP);        // per warp: cluster's x, U words
  static constexpr size_t fixed = al16(osd + (MU ? (size_t)NW * 2 * W * 4 : 0));
  // lists
  static constexpr size_t newk = 0;                               // new columns of a step
  static constexpr size_t ssl = newk + (size_t)SC * 8;            // slots of new columns
  static constexpr size_t sg = ssl + (size_t)SC * 8;              // their faults, in key order
  static constexpr size_t sroot = sg + (size_t)SC * 2;            // their clusters
  static constexpr size_t dpf = sroot + (size_t)SC * 2;           // faults of dependent columns
  static constexpr size_t ext = dpf + (MU ? (size_t)CAP * 2 : 0);
  static constexpr size_t dpr = ext + (MU ? (size_t)CAP * 2 : 0);      // their clusters
  static constexpr size_t dpk = dpr + (MU ? (size_t)CAP * 2 : 0);      // their LLR bits
  static constexpr size_t M = al16(dpk + (MU ? (size_t)CAP * 4 : 0));
  // Rows of M and bits of the dependent columns' images (npN, after M): a shot has at most as
  // many slots as the graph has detectors.
  static __host__ __device__ int row_stride(int m) {
    const int r = (m + 31) & ~31;
    return BIG && r < CAP ? r : CAP;
  }
  static __host__ __device__ size_t list_bytes(int m) {
    const size_t r = (size_t)row_stride(m);
    return al16(M + r * (r / 32) * 4 + (MU ? (size_t)CAP * (r / 32) * 4 : 0));
  }
  // Candidate list entries.  A shot that lists half of a large code's faults has percolated
  // and goes to the large instance.
  static __host__ __device__ int lcap(int n) {
    if (BIG) return n;
    const int half = n / 2 > 1536 ? n / 2 : 1536;
    const int cap = half < 2816 ? half : 2816;
    return cap < n ? cap : n;
  }
};

// Candidate list of `cap` entries: detectors, LLR bits, faults.
__host__ __device__ inline size_t cand_bytes(size_t cap) {
  return al16(cap * 8) + al16(cap * 4) + al16(cap * 2);
}

// No shot can outgrow the small instance I: the large one is not launched.
template <class I>
bool always_fits(int m, int n) {
  return m <= I::CAP && m <= I::SC && n <= I::lcap(n) && (!I::MU || n <= I::CAP);
}

template <class I>
size_t smem_bytes(int m, int n) {
  return I::fixed + (I::LG ? 0 : al16((size_t)m * 4)) + 2 * al16((size_t)(n + 31) / 32 * 4) +
         (I::BIG ? 0 : I::list_bytes(m)) + (I::BIG && I::LG ? 0 : cand_bytes((size_t)I::lcap(n)));
}
// Global scratch bytes of a CTA.
template <class I>
size_t scratch_bytes(int m, int n) {
  return (I::LG ? al16((size_t)m * 4) : 0) + (I::BIG ? I::list_bytes(m) : 0) +
         (I::BIG && I::LG ? cand_bytes((size_t)n) : 0);
}

struct SGraph {
  const int32_t* chk_ptr;
  const int32_t* var_ptr;
  const uint16_t* var_chk;
  const uint16_t* chk_pad;  // [m][max_row_deg], 0xffff past the row's end
  const uint2* var_pad;     // [n] the first four detectors, 0xffff past the column's end
  int max_col_deg, max_row_deg;
};

// Shared scalars.  nsl, nf and np go on counting past the arrays' ends: a shot has outgrown the
// instance when one of them has, which is looked at after a barrier that no writer of that
// counter passes before the next one, so that all threads see the same.
struct Scal {
  int ns, nsl, nf;   // seeds, slots, candidates so far
  int n_new, merged; // columns and merges of the step
  int ng, ncr;       // growing clusters; clusters with new columns
  int np, ext;       // dependent columns for LSD-mu; those in the solution
  int piv[3];
  unsigned item;
  uint2 ssl;         // the single cluster's new column: slots of its detectors,
  uint2 mlab;        // labels of the clusters it absorbs there,
  unsigned fresh;    // and which of them are newly claimed
  unsigned red[2][32];
};

template <class I>
struct Shot {
  unsigned char* sm;
  unsigned char* li;
  uint32_t* lab;
  uint32_t* cand;
  uint32_t* joined;
  uint2* ld;
  uint32_t* lk;
  uint16_t* lf;
  int lcap;
  int rs;               // row stride of M (large instance; constant for the small one)
  Scal* sc;
  __device__ __forceinline__ int stride() const { return I::BIG ? rs : I::CAP; }
  __device__ __forceinline__ int words() const { return stride() >> 5; }
  template <class T>
  __device__ __forceinline__ T* s(size_t off) const { return reinterpret_cast<T*>(sm + off); }
  template <class T>
  __device__ __forceinline__ T* l(size_t off) const { return reinterpret_cast<T*>(li + off); }
  __device__ __forceinline__ uint32_t* best() const { return s<uint32_t>(I::best); }
  __device__ __forceinline__ uint32_t* bidx() const { return s<uint32_t>(I::bidx); }
  __device__ __forceinline__ uint32_t* growb() const { return s<uint32_t>(I::growb); }
  __device__ __forceinline__ uint16_t* parent() const { return s<uint16_t>(I::parent); }
  __device__ __forceinline__ uint16_t* inv() const { return s<uint16_t>(I::inv); }
  __device__ __forceinline__ uint16_t* pcol() const { return s<uint16_t>(I::pcol); }
  __device__ __forceinline__ uint16_t* sdet() const { return s<uint16_t>(I::sdet); }
  __device__ __forceinline__ uint16_t* slab() const { return s<uint16_t>(I::slab); }
  __device__ __forceinline__ unsigned char* flags() const { return s<unsigned char>(I::flags); }
  __device__ __forceinline__ unsigned long long* newk() const { return l<unsigned long long>(I::newk); }
  __device__ __forceinline__ uint32_t* M() const { return l<uint32_t>(I::M); }
  __device__ __forceinline__ uint32_t* npN() const { return M() + (size_t)stride() * words(); }
  __device__ __forceinline__ uint16_t* ssl() const { return l<uint16_t>(I::ssl); }
  __device__ __forceinline__ uint16_t* sg() const { return l<uint16_t>(I::sg); }
  __device__ __forceinline__ uint16_t* sroot() const { return l<uint16_t>(I::sroot); }
  __device__ __forceinline__ uint16_t* dpf() const { return l<uint16_t>(I::dpf); }
  __device__ __forceinline__ uint16_t* ext() const { return l<uint16_t>(I::ext); }
  __device__ __forceinline__ uint16_t* dpr() const { return l<uint16_t>(I::dpr); }
  __device__ __forceinline__ uint32_t* dpk() const { return l<uint32_t>(I::dpk); }
};

// Order-preserving bits of an LLR (-0.0 folded into +0.0).
__device__ __forceinline__ unsigned llr_bits(float x) {
  x = __fadd_rn(x, 0.0f);
  const unsigned u = __float_as_uint(x);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ __forceinline__ int uf_find(const volatile uint16_t* parent, int x) {
  int p = parent[x];
  while (p != x) {
    x = p;
    p = parent[x];
  }
  return x;
}

template <class I>
__device__ __forceinline__ void uf_unite(const Shot<I>& S, int a, int b) {
  const volatile uint16_t* vp = S.parent();
#pragma unroll 1
  for (;;) {
    a = uf_find(vp, a);
    b = uf_find(vp, b);
    if (a == b) return;
    if (a < b) {
      const int t = a;
      a = b;
      b = t;
    }
    if (atomicCAS(reinterpret_cast<unsigned short*>(S.parent()) + a, (unsigned short)a,
                  (unsigned short)b) == (unsigned short)a) {
      S.sc->merged = 1;
      return;
    }
  }
}

// Claims detector d for the cluster of label r.
template <class I>
__device__ __forceinline__ void claim(const Shot<I>& S, int d, int r) {
  const uint32_t o = atomicCAS(&S.lab[d], kFree, ((uint32_t)r << 16) | 0xffffu);
  if (o == kFree) {
    const int sl = atomicAdd(&S.sc->nsl, 1);
    if (sl >= I::CAP) return;
    S.lab[d] = ((uint32_t)r << 16) | (uint32_t)sl;
    S.sdet()[sl] = (uint16_t)d;
    S.slab()[sl] = (uint16_t)r;
    S.flags()[sl] = 0;
  } else if ((int)(o >> 16) != r) {
    uf_unite(S, r, (int)(o >> 16));
  }
}

// The i-th of the four packed 16-bit values.
__device__ __forceinline__ uint32_t half4(uint2 v, int i) {
  return ((i & 2 ? v.y : v.x) >> (16 * (i & 1))) & 0xffffu;
}

// Calls fn(d) for every detector of fault f, the first four of which are v.
template <class F>
__device__ __forceinline__ void each_det(const SGraph& G, uint2 v, int f, F&& fn) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint32_t d = half4(v, i);
    if (d != kNone16) fn((int)d);
  }
  if (G.max_col_deg > 4) {
    const int v1 = G.var_ptr[f + 1];
#pragma unroll 1
    for (int q = G.var_ptr[f] + 4; q < v1; ++q) fn((int)G.var_chk[q]);
  }
}

// The thread's rows among the slots from..to become unit rows; its older rows get zeros in the
// words that the new slots opened.
template <class I>
__device__ __forceinline__ void open_rows(const Shot<I>& S, int from, int to, int tid) {
  const int w0 = (from + 31) >> 5, w1 = (to + 31) >> 5;
#pragma unroll 1
  for (int i = tid; i < to; i += I::NT)
#pragma unroll 1
    for (int w = i < from ? w0 : 0; w < w1; ++w)
      S.M()[(size_t)w * S.stride() + i] = (i >> 5) == w && i >= from ? 1u << (i & 31) : 0u;
}

// Fault f is next to a newly claimed detector: lists it if it is not listed; returns its entry
// (key and detectors in k, v) or -1.
template <class I>
__device__ __forceinline__ int list_candidate(const SGraph& G, const Shot<I>& S, const float* llr,
                                              int f, unsigned& k, uint2& v) {
  const uint32_t b = 1u << (f & 31);
  if ((atomicOr(&S.cand[f >> 5], b) & b) != 0) return -1;
  const int q = atomicAdd(&S.sc->nf, 1);
  if (q >= S.lcap) return -1;
  v = G.var_pad[f];
  k = llr_bits(llr[f]);
  S.lf[q] = (uint16_t)f;
  S.ld[q] = v;
  S.lk[q] = k;
  return q;
}

// Rows and candidates of the slots from..to.
template <class I>
__device__ __forceinline__ void open_slots(const SGraph& G, const Shot<I>& S, const float* llr,
                                           int from, int to, int tid) {
  open_rows(S, from, to, tid);
  const int D = G.max_row_deg;
#pragma unroll 1
  for (int x = tid; x < (to - from) * D; x += I::NT) {
    const int f = G.chk_pad[(size_t)S.sdet()[from + x / D] * D + x % D];
    unsigned k;
    uint2 v;
    if (f != kNone16) list_candidate(G, S, llr, f, k, v);
  }
}

// Image of a column under M on the thread's rows i = tid + NT j < nsl: bit j of the result; pc
// = one of those with a bit and no pivot (or unchanged).  sl: slots of its first four detectors.
template <class I>
__device__ __forceinline__ uint32_t column_image(const SGraph& G, const Shot<I>& S, uint2 sl, int g,
                                                 int nsl, int tid, int& pc) {
  constexpr int NT = I::NT, CAP = I::CAP;
  uint32_t hit = 0;
#pragma unroll
  for (int j = 0; j < I::RPT; ++j) {
    const int i = tid + NT * j;
    if (i < nsl) {
      uint32_t x = 0;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const uint32_t s = half4(sl, q);
        if (s != kNone16) x ^= S.M()[(size_t)(s >> 5) * S.stride() + i] >> (s & 31);
      }
      hit |= (x & 1u) << j;
    }
  }
  if (G.max_col_deg > 4) {
    const int v1 = G.var_ptr[g + 1];
#pragma unroll 1
    for (int q = G.var_ptr[g] + 4; q < v1; ++q) {
      const uint32_t s = S.lab[G.var_chk[q]] & 0xffffu;
#pragma unroll 1
      for (int j = 0; tid + NT * j < nsl; ++j)
        hit ^= ((S.M()[(size_t)(s >> 5) * S.stride() + tid + NT * j] >> (s & 31)) & 1u) << j;
    }
  }
#pragma unroll 1
  for (uint32_t h = hit; h; h &= h - 1) {
    const int i = tid + NT * (__ffs(h) - 1);
    if (!(S.flags()[i] & 2)) pc = i;
  }
  return hit;
}

// Makes p the pivot row of column g (hit: the column's image on the thread's rows) and adds it
// to the other rows with a bit.
template <class I>
__device__ __forceinline__ void pivot_update(const Shot<I>& S, int p, int g, uint32_t hit, int nsl,
                                             int tid) {
  constexpr int NT = I::NT, CAP = I::CAP;
  const int lane = tid & 31, wc = (nsl + 31) >> 5;
  if (p % NT == tid) {
    hit &= ~(1u << (p / NT));
    S.flags()[p] |= 2;
    S.pcol()[p] = (uint16_t)g;
  }
  const bool sp = S.flags()[p] & 1;
  if (!__any_sync(kFull, hit != 0)) return;
#pragma unroll 1
  for (int c0 = 0; c0 < wc; c0 += 32) {
    const uint32_t v = c0 + lane < wc ? S.M()[(size_t)(c0 + lane) * S.stride() + p] : 0u;
    unsigned nz = __ballot_sync(kFull, v != 0);
    while (nz) {
      const int w = __ffs(nz) - 1;
      nz &= nz - 1;
      const uint32_t pv = __shfl_sync(kFull, v, w);
      uint32_t* const row = S.M() + (size_t)(c0 + w) * S.stride() + tid;
#pragma unroll
      for (int j = 0; j < I::RPT; ++j)
        if ((hit >> j) & 1u) row[NT * j] ^= pv;
    }
  }
  if (sp)
#pragma unroll 1
    for (uint32_t h = hit; h; h &= h - 1) S.flags()[tid + NT * (__ffs(h) - 1)] ^= 1;
}

// Keeps a dependent column for LSD-mu: its image is its combination of pivot rows.  np counts
// the ones without room too (the same in every thread; the caller compares it with CAP).
template <class I>
__device__ __forceinline__ void keep_dependent(const Shot<I>& S, int& np, int g, uint32_t hit, int tid) {
  if constexpr (I::MU) {
    if (np++ >= I::CAP) return;
    const int at = np - 1;
#pragma unroll
    for (int j = 0; j < I::RPT; ++j) {
      const unsigned b = __ballot_sync(kFull, (hit >> j) & 1u);
      const int w = I::NW * j + (tid >> 5);
      if ((tid & 31) == 0 && w < S.words()) S.npN()[(size_t)at * S.words() + w] = b;
    }
    if (tid == 0) S.dpf()[at] = (uint16_t)g;
  }
}

// Columns of the clusters with at most 32 rows, a warp per cluster.  Larger clusters keep
// their bit in growb.
template <class I>
__device__ void add_columns_by_warp(const Shot<I>& S, int n_new, int nsl, int tid) {
  constexpr int CAP = I::CAP;
  const int lane = tid & 31, warp = tid >> 5;
  const int ncr = S.sc->ncr, wc = (nsl + 31) >> 5;
  uint16_t* const rows = S.template s<uint16_t>(I::rows) + warp * 32;
  uint32_t* const M = S.M();
#pragma unroll 1
  for (int c = warp; c < ncr; c += I::NW) {
    const int r = S.inv()[c];
    int cnt = 0;
#pragma unroll 1
    for (int b0 = 0; b0 < nsl; b0 += 32) {
      const bool in = b0 + lane < nsl && S.slab()[b0 + lane] == r;
      const unsigned b = __ballot_sync(kFull, in);
      const int at = cnt + __popc(b & ((1u << lane) - 1u));
      if (in && at < 32) rows[at] = (uint16_t)(b0 + lane);
      cnt += __popc(b);
    }
    if (cnt > 32) continue;
    __syncwarp();
    const bool mine = lane < cnt;
    const int i = mine ? rows[lane] : 0;
#pragma unroll 1
    for (int t0 = 0; t0 < n_new; t0 += 32) {
      unsigned todo = __ballot_sync(kFull, t0 + lane < n_new && S.sroot()[t0 + lane] == r);
      while (todo) {
        const int t = t0 + __ffs(todo) - 1;
        todo &= todo - 1;
        const uint2 sl = reinterpret_cast<const uint2*>(S.ssl())[t];
        const int g = S.sg()[t];
        uint32_t x = 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const uint32_t s = half4(sl, q);
          if (mine && s != kNone16) x ^= M[(size_t)(s >> 5) * S.stride() + i] >> (s & 31);
        }
        bool hit = (x & 1u) != 0;
        const unsigned nb = __ballot_sync(kFull, hit && !(S.flags()[i] & 2));
        if (nb == 0) {
          if constexpr (I::MU) {
            int k = 0;
            if (lane == 0) k = atomicAdd(&S.sc->np, 1);
            k = __shfl_sync(kFull, k, 0);
            if (k >= CAP) continue;
            uint32_t* const row = S.npN() + (size_t)k * S.words();
#pragma unroll 1
            for (int w = lane; w < S.words(); w += 32) row[w] = 0u;
            __syncwarp();
            if (hit) atomicOr(row + (i >> 5), 1u << (i & 31));
            if (lane == 0) S.dpf()[k] = (uint16_t)g;
          }
          continue;
        }
        const int pl = __ffs(nb) - 1;
        const int p = __shfl_sync(kFull, i, pl);
        const bool sp = S.flags()[p] & 1;
        __syncwarp();
        if (lane == pl) {
          hit = false;
          S.flags()[p] |= 2;
          S.pcol()[p] = (uint16_t)g;
        }
        if (__any_sync(kFull, hit)) {
#pragma unroll 1
          for (int c0 = 0; c0 < wc; c0 += 32) {
            const uint32_t v = c0 + lane < wc ? M[(size_t)(c0 + lane) * S.stride() + p] : 0u;
            unsigned nz = __ballot_sync(kFull, v != 0);
            while (nz) {
              const int w = __ffs(nz) - 1;
              nz &= nz - 1;
              const uint32_t pv = __shfl_sync(kFull, v, w);
              if (hit) M[(size_t)(c0 + w) * S.stride() + i] ^= pv;
            }
          }
          if (sp && hit) S.flags()[i] ^= 1;
        }
        __syncwarp();
      }
    }
    if (lane == 0) atomicAnd(&S.growb()[r >> 5], ~(1u << (r & 31)));
    __syncwarp();
  }
}

// Adds the n_new columns of a step, in key order within each cluster, to the eliminations.
template <class I>
__device__ __forceinline__ void add_columns(const SGraph& G, const Shot<I>& S, int n_new, int nsl,
                                            int tid) {
  const bool by_warp = n_new > 1 && G.max_col_deg <= 4;
  if (by_warp) {
    add_columns_by_warp(S, n_new, nsl, tid);
    __syncthreads();
  }
  int np = S.sc->np, done = 0;
#pragma unroll 1
  for (int t = 0; t < n_new; ++t) {
    if (by_warp) {
      const int r = S.sroot()[t];
      if (!((S.growb()[r >> 5] >> (r & 31)) & 1u)) continue;
    }
    const int g = S.sg()[t];
    int pc = -1;
    const uint32_t hit = column_image(G, S, reinterpret_cast<const uint2*>(S.ssl())[t], g, nsl, tid, pc);
    // any row with a bit and no pivot will do: one of the stores stands
    if (pc >= 0) S.sc->piv[done % 3] = pc;
    if (tid == 0) S.sc->piv[(done + 1) % 3] = -1;
    __syncthreads();
    const int p = S.sc->piv[done % 3];
    ++done;
    if (p < 0) keep_dependent(S, np, g, hit, tid);
    else pivot_update(S, p, g, hit, nsl, tid);
  }
  __syncthreads();
  if (by_warp)
#pragma unroll 1
    for (int c = tid; c < S.sc->ncr; c += I::NT) {
      const int r = S.inv()[c];
      atomicAnd(&S.growb()[r >> 5], ~(1u << (r & 31)));
    }
  if (tid == 0) S.sc->np = np;
  __syncthreads();
}

// Lists the labels of the invalid clusters (only_invalid) or of all clusters in inv.
template <class I>
__device__ __forceinline__ int collect(const Shot<I>& S, int nsl, bool only_invalid, int tid) {
  if (only_invalid) {
#pragma unroll 1
    for (int i = tid; i < nsl; i += I::NT) {
      if ((S.flags()[i] & 3) != 1) continue;
      const int r = S.slab()[i];
      const uint32_t b = 1u << (r & 31);
      if (!(atomicOr(&S.growb()[r >> 5], b) & b)) S.inv()[atomicAdd(&S.sc->ng, 1)] = (uint16_t)r;
    }
  } else {
    const int ns = S.sc->ns;
#pragma unroll 1
    for (int r = tid; r < ns; r += I::NT) {
      if (S.parent()[r] != r) continue;
      atomicOr(&S.growb()[r >> 5], 1u << (r & 31));
      S.inv()[atomicAdd(&S.sc->ng, 1)] = (uint16_t)r;
    }
  }
  __syncthreads();
  return S.sc->ng;
}

// One synchronous growth step of the k clusters listed in inv (marked in growb).  On return the
// list is empty.  0: grown, 1: strict and a cluster had no candidate, 2: none grew, 3: no room.
template <class I>
__device__ int sparse_step(const SGraph& G, const Shot<I>& S, const float* llr, int k, bool strict,
                           int tid) {
  constexpr int NT = I::NT;
  Scal& sc = *S.sc;
  const int nf = sc.nf, nsl0 = sc.nsl;
  // ---- find_candidate: the least LLR bits of every growing cluster, then the least fault
  // that has them ----
#pragma unroll 1
  for (int t = tid; t < k; t += NT) {
    const int r = S.inv()[t];
    S.best()[r] = kNoKey;
    S.bidx()[r] = kNoKey;
  }
  __syncthreads();
#pragma unroll 1
  for (int pass = 0; pass < 2; ++pass) {
#pragma unroll 1
    for (int x = tid; x < nf; x += NT) {
      const int f = S.lf[x];
      if ((S.joined[f >> 5] >> (f & 31)) & 1u) continue;
      const unsigned key = S.lk[x];
      each_det(G, S.ld[x], f, [&](int d) {
        const uint32_t y = S.lab[d];
        if (y == kFree) return;
        const int r = (int)(y >> 16);
        if (!((S.growb()[r >> 5] >> (r & 31)) & 1u)) return;
        if (pass == 0) {
          if (key < S.best()[r]) atomicMin(&S.best()[r], key);
        } else if (key == S.best()[r]) {
          atomicMin(&S.bidx()[r], (unsigned)f);
        }
      });
    }
    __syncthreads();
  }
  bool some = false, none = false;
#pragma unroll 1
  for (int t = tid; t < k; t += NT) {
    const bool has = S.bidx()[S.inv()[t]] != kNoKey;
    some |= has;
    none |= !has;
  }
  none = __syncthreads_or(none);
  some = __syncthreads_or(some);
  const bool stop = (strict && none) || !some;
  // ---- every pick joins its cluster and claims its detectors; clusters that meet merge ----
#pragma unroll 1
  for (int t = tid; t < k; t += NT) {
    const int r = S.inv()[t];
    atomicAnd(&S.growb()[r >> 5], ~(1u << (r & 31)));
    const unsigned f = S.bidx()[r];
    if (stop || f == kNoKey) continue;
    const uint32_t b = 1u << (f & 31);
    // (a fault picked twice joins once; its pickers meet at its detectors)
    if (!(atomicOr(&S.joined[f >> 5], b) & b))
      S.newk()[atomicAdd(&sc.n_new, 1)] = ((unsigned long long)S.best()[r] << 32) | f;
    each_det(G, G.var_pad[f], (int)f, [&](int d) { claim(S, d, r); });
  }
  if (tid == 0) {
    sc.ng = sc.ncr = 0;
    sc.piv[0] = -1;
  }
  __syncthreads();
  if (stop) return strict && none ? 1 : 2;
  const int nsl = sc.nsl, n_new = sc.n_new;
  if (nsl > I::CAP) return 3;
  // ---- labels to roots after a merge ----
  if (sc.merged) {
    const int ns = sc.ns;
#pragma unroll 1
    for (int x = tid; x < ns; x += NT) S.parent()[x] = (uint16_t)uf_find(S.parent(), x);
    __syncthreads();
#pragma unroll 1
    for (int i = tid; i < nsl; i += NT) {
      const int r = S.parent()[S.slab()[i]];
      S.slab()[i] = (uint16_t)r;
      S.lab[S.sdet()[i]] = ((uint32_t)r << 16) | (uint32_t)i;
    }
    __syncthreads();
  }
  open_slots(G, S, llr, nsl0, nsl, tid);
  // ---- the new columns in key order, with their clusters and the slots of their detectors ----
#pragma unroll 1
  for (int t = tid; t < n_new; t += NT) {
    const unsigned long long kt = S.newk()[t];
    int pos = 0;
#pragma unroll 1
    for (int u = 0; u < n_new; ++u) pos += S.newk()[u] < kt ? 1 : 0;
    const int g = (int)(kt & 0xffffffffu);
    S.sg()[pos] = (uint16_t)g;
    const uint2 v = G.var_pad[g];
    uint32_t sl[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const uint32_t d = half4(v, q);
      sl[q] = d != kNone16 ? S.lab[d] & 0xffffu : kNone16;
    }
    reinterpret_cast<uint2*>(S.ssl())[pos] = make_uint2(sl[0] | sl[1] << 16, sl[2] | sl[3] << 16);
    if (n_new > 1) {
      const int r = S.slab()[sl[0]];
      const uint32_t b = 1u << (r & 31);
      S.sroot()[pos] = (uint16_t)r;
      if (!(atomicOr(&S.growb()[r >> 5], b) & b)) S.inv()[atomicAdd(&sc.ncr, 1)] = (uint16_t)r;
    }
  }
  __syncthreads();
  if (sc.nf > S.lcap) return 3;
  if (tid == 0) sc.n_new = sc.merged = 0;
  add_columns(G, S, n_new, nsl, tid);
  if (I::MU && sc.np > I::CAP) return 3;
  if (n_new > 1 && G.max_col_deg > 4) {  // (the marks of the clusters with columns, unused there)
#pragma unroll 1
    for (int c = tid; c < sc.ncr; c += NT) {
      const int r = S.inv()[c];
      atomicAnd(&S.growb()[r >> 5], ~(1u << (r & 31)));
    }
    __syncthreads();
  }
  return 0;
}

// Growth of the only invalid cluster (label r) until it is valid: the step of sparse_step with
// three barriers.  While the new column is eliminated the candidates of the next step are
// searched, so the next pick is known when the validity is.  No other cluster grows, so the
// absorbed clusters are relabelled at once and r stays the root.  Steps taken are added to
// `steps`; returns as sparse_step (0: valid).  Needs columns of at most four detectors.
// Every thread has to leave at the same barrier, so room is judged by counters that nobody
// writes between the barrier after which they are read and the next one (nsl, nf), or that
// every thread counts for itself (np).
template <class I>
__device__ int grow_single(const SGraph& G, const Shot<I>& S, const float* llr, uint32_t r, int n,
                           int& steps, int tid) {
  constexpr int NT = I::NT;
  Scal& sc = *S.sc;
  const int lane = tid & 31, warp = tid >> 5;
  int nf = sc.nf, nsl = sc.nsl, np = sc.np;
  const int D = G.max_row_deg;
  unsigned bk, bx;  // the thread's best entry: LLR bits, then fault << 16 | entry
  auto scan = [&] {
#pragma unroll 1
    for (int x = tid; x < nf; x += NT) {
      const unsigned key = S.lk[x];
      if (key > bk) continue;
      const unsigned fx = ((unsigned)S.lf[x] << 16) | (unsigned)x;
      if (key == bk && fx > bx) continue;
      const int f = (int)(fx >> 16);
      if ((S.joined[f >> 5] >> (f & 31)) & 1u) continue;
      const uint2 v = S.ld[x];
      bool mine = false;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const uint32_t d = half4(v, i);
        if (d != kNone16) mine |= (S.lab[d] >> 16) == r;
      }
      if (mine) {
        bk = key;
        bx = fx;
      }
    }
  };
  auto publish = [&] {
    const unsigned wk = __reduce_min_sync(kFull, bk);
    const unsigned wx = __reduce_min_sync(kFull, bk == wk ? bx : kNoKey);
    if (lane == 0) {
      sc.red[0][warp] = wk;
      sc.red[1][warp] = wx;
    }
  };
  auto fetch = [&] {
    const unsigned k0 = lane < I::NW ? sc.red[0][lane] : kNoKey;
    const unsigned x0 = lane < I::NW ? sc.red[1][lane] : kNoKey;
    bk = __reduce_min_sync(kFull, k0);
    bx = __reduce_min_sync(kFull, k0 == bk ? x0 : kNoKey);
  };
  bk = bx = kNoKey;
  scan();
  publish();
  if (tid == 0) sc.piv[0] = -1;
  __syncthreads();
  fetch();
  if (tid == 0) {  // (after the barrier: the caller's threads read ng after the one before it)
    S.growb()[r >> 5] = 0u;
    sc.ng = sc.merged = 0;
  }
#pragma unroll 1
  for (int it = 0;; ++it) {
    if (bx == kNoKey) return 1;
    if (steps > n) return 1;  // each step adds a column: cannot be reached
    const int g = (int)(bx >> 16);
    const uint2 dets = S.ld[bx & 0xffffu];
    // ---- the pick joins and claims its detectors: one lane each ----
    if (warp == 0) {
      const uint32_t d = half4(dets, lane & 3);
      const bool on = lane < 4 && d != kNone16;
      const uint32_t y = on ? S.lab[d] : 0u;
      const bool free = on && y == kFree;
      const unsigned fb = __ballot_sync(kFull, free);
      const int sl = free ? nsl + __popc(fb & ((1u << lane) - 1u)) : (int)(y & 0xffffu);
      const uint32_t other = on && !free && (y >> 16) != r ? y >> 16 : kNone16;
      if (free && sl < I::CAP) {
        S.lab[d] = (r << 16) | (uint32_t)sl;
        S.sdet()[sl] = (uint16_t)d;
        S.slab()[sl] = (uint16_t)r;
        S.flags()[sl] = 0;
      }
      if (other != kNone16) S.parent()[other] = (uint16_t)r;
      if (lane < 4) {
        reinterpret_cast<uint16_t*>(&sc.ssl)[lane] = on ? (uint16_t)sl : kNone16;
        reinterpret_cast<uint16_t*>(&sc.mlab)[lane] = (uint16_t)other;
      }
      if (lane == 0) {
        S.joined[g >> 5] |= 1u << (g & 31);
        sc.fresh = fb;
        sc.nsl = nsl + __popc(fb);
      }
    }
    // the faults next to those detectors, asked for now and used if the detector is new: thread
    // (detector q, edge e) from warp 1 on
    static_assert(NT - 32 >= 4 * kMaxRowDeg, "a thread for every edge of four detectors");
    const int q0 = (tid - 32) / D;
    int near = kNone16;
    if (tid >= 32 && q0 < 4) {
      const uint32_t d = half4(dets, q0);
      if (d != kNone16) near = G.chk_pad[(size_t)d * D + (tid - 32) % D];
    }
    __syncthreads();
    const int nsl0 = nsl;
    nsl = sc.nsl;
    if (nsl > I::CAP) return 3;
    const uint2 sl = sc.ssl, ml = sc.mlab;
    const unsigned fresh = sc.fresh;
    if ((ml.x & ml.y) != kFull) {
      // ---- absorbed clusters take the label r ----
      const uint32_t m0 = ml.x & 0xffffu, m1 = ml.x >> 16, m2 = ml.y & 0xffffu, m3 = ml.y >> 16;
#pragma unroll 1
      for (int i = tid; i < nsl0; i += NT) {
        const uint32_t y = S.slab()[i];
        if (y == m0 || y == m1 || y == m2 || y == m3) {
          S.slab()[i] = (uint16_t)r;
          S.lab[S.sdet()[i]] = (r << 16) | (uint32_t)i;
        }
      }
      __syncthreads();
    }
    bk = bx = kNoKey;
    // ---- new candidates; a fault listed here is a candidate of the cluster ----
    auto admit = [&](int f) {
      unsigned key;
      uint2 v;
      const int x = list_candidate(G, S, llr, f, key, v);
      const unsigned fx = ((unsigned)f << 16) | (unsigned)x;
      if (x >= 0 && (key < bk || (key == bk && fx < bx))) {
        bk = key;
        bx = fx;
      }
    };
    if (near != kNone16 && ((fresh >> q0) & 1u)) admit(near);
    // ---- the column's image; meanwhile the search for the next pick ----
    open_rows(S, nsl0, nsl, tid);
    int pc = -1;
    const uint32_t hit = column_image(G, S, sl, g, nsl, tid, pc);
    if (pc >= 0) sc.piv[it % 3] = pc;
    if (tid == 0) sc.piv[(it + 1) % 3] = -1;
    scan();
    publish();
    __syncthreads();
    const int p = sc.piv[it % 3];
    nf = sc.nf;
    if (nf > S.lcap) return 3;
    fetch();
    if (p < 0) keep_dependent(S, np, g, hit, tid);
    else pivot_update(S, p, g, hit, nsl, tid);
    if (I::MU && np > I::CAP) return 3;
    bool bad = false;
#pragma unroll 1
    for (int i = tid; i < nsl; i += NT) bad |= (S.flags()[i] & 3) == 1;
    ++steps;
    if (!__syncthreads_or(bad)) break;
  }
  if (tid == 0) sc.np = np;
  __syncthreads();
  return 0;
}

// ---- LSD-mu reprocessing, one warp per cluster ----

// Order key of the dependent column of index u.
template <class I>
__device__ __forceinline__ unsigned long long dep_key(const Shot<I>& S, int u) {
  return ((unsigned long long)S.dpk()[u] << 32) | S.dpf()[u];
}

// The first `want` dependent columns of cluster r in key order; lane j returns the j-th (or
// -1), count = how many there are.
template <class I>
__device__ int first_dependent(const Shot<I>& S, int r, int np, int want, int lane, int& count) {
  int mine = -1;
  unsigned long long last = 0;
  int nt = 0;
#pragma unroll 1
  for (int it = 0; it < want; ++it) {
    unsigned long long bk = ~0ull;
    int bi = -1;
#pragma unroll 1
    for (int u = lane; u < np; u += 32) {
      if (S.dpr()[u] != r) continue;
      const unsigned long long ku = dep_key(S, u);
      if ((it > 0 && ku <= last) || ku >= bk) continue;
      bk = ku;
      bi = u;
    }
#pragma unroll 1
    for (int off = 16; off > 0; off >>= 1) {
      const unsigned long long ok = __shfl_xor_sync(kFull, bk, off);
      const int oi = __shfl_xor_sync(kFull, bi, off);
      if (ok < bk) {
        bk = ok;
        bi = oi;
      }
    }
    if (bi < 0) break;
    if (lane == nt) mine = bi;
    ++nt;
    last = bk;
  }
  count = nt;
  return mine;
}

// Words of the local solution of every row (bit = the row's pivot column is in it).
template <class I>
__device__ void solution_words(const Shot<I>& S, uint32_t* xw, int nsl, int lane) {
#pragma unroll 1
  for (int c = 0; 32 * c < nsl; ++c) {
    const int i = 32 * c + lane;
    const unsigned b = __ballot_sync(kFull, i < nsl && (S.flags()[i] & 3) == 3);
    if (lane == 0) xw[c] = b;
  }
  __syncwarp();
}

// Exhaustive OSD over the first min(mu, #dependent) dependent columns of cluster r (App. D);
// cost = sum of 2^-32 fixed-point channel weights, ties to the smaller pattern.  Rows that no
// selected column touches cost every pattern the same and are left out.
template <class I>
__device__ void osd_e(const LSDArgs& a, const Shot<I>& S, int r, int np, int nsl, uint32_t* xw,
                      uint32_t* uw, int lane) {
  const long long* wfix = a.g.wfix;
  const int wc = (nsl + 31) >> 5;
  int nt;
  const int mine = first_dependent(S, r, np, a.order, lane, nt);
  if (nt == 0) return;
  solution_words(S, xw, nsl, lane);
#pragma unroll 1
  for (int w0 = 0; w0 < wc; w0 += 32) {  // rows that some selected column touches
    const int w = w0 + lane;
    uint32_t rows = 0;
#pragma unroll 1
    for (int j = 0; j < nt; ++j) {
      const int u = __shfl_sync(kFull, mine, j);
      if (w < wc) rows |= S.npN()[(size_t)u * S.words() + w];
    }
    if (w < wc) uw[w] = rows;
  }
  __syncwarp();
  const long long wmine = lane < nt ? wfix[S.dpf()[mine]] : 0;
  long long bcost = LLONG_MAX;
  int bt = 0;
#pragma unroll 1
  for (int t0 = 0; t0 < (1 << nt); t0 += 32) {
    const int t = t0 + lane;
    long long cost = 0;
#pragma unroll 1
    for (int w = 0; w < wc; ++w) {
      uint32_t rows = uw[w];
      if (rows == 0) continue;
      const uint32_t nw = lane < nt ? S.npN()[(size_t)mine * S.words() + w] : 0u;
      const uint32_t x = xw[w];
      while (rows) {
        const int b = __ffs(rows) - 1;
        rows &= rows - 1;
        const unsigned pm = __ballot_sync(kFull, (nw >> b) & 1u);
        if (((x >> b) ^ __popc(pm & (unsigned)t)) & 1u) cost += wfix[S.pcol()[32 * w + b]];
      }
    }
#pragma unroll 1
    for (int j = 0; j < nt; ++j) {
      const long long wj = __shfl_sync(kFull, wmine, j);
      if ((t >> j) & 1) cost += wj;
    }
    if (t < (1 << nt) && cost < bcost) {
      bcost = cost;
      bt = t;
    }
  }
#pragma unroll 1
  for (int off = 16; off > 0; off >>= 1) {
    const long long oc = __shfl_xor_sync(kFull, bcost, off);
    const int ot = __shfl_xor_sync(kFull, bt, off);
    if (oc < bcost || (oc == bcost && ot < bt)) {
      bcost = oc;
      bt = ot;
    }
  }
#pragma unroll 1
  for (int j = 0; j < nt; ++j) {
    if (!((bt >> j) & 1)) continue;
    const int u = __shfl_sync(kFull, mine, j);
#pragma unroll 1
    for (int w = 0; w < wc; ++w)
      if ((S.npN()[(size_t)u * S.words() + w] >> lane) & 1u) S.flags()[32 * w + lane] ^= 1;
    if (lane == 0) S.ext()[atomicAdd(&S.sc->ext, 1)] = S.dpf()[u];
  }
}

// Cost of the cluster's solution with dependent columns u1 and u2 (-1 = none) flipped, less the
// unflipped solution's.
template <class I>
__device__ __forceinline__ long long pattern_delta(const LSDArgs& a, const Shot<I>& S,
                                                   const uint32_t* xw, int wc, int u1, int u2) {
  const long long* wfix = a.g.wfix;
  long long cost = wfix[S.dpf()[u1]];
  if (u2 >= 0) cost += wfix[S.dpf()[u2]];
#pragma unroll 1
  for (int w = 0; w < wc; ++w) {
    uint32_t rows = S.npN()[(size_t)u1 * S.words() + w];
    if (u2 >= 0) rows ^= S.npN()[(size_t)u2 * S.words() + w];
    const uint32_t x = xw[w];
    while (rows) {
      const int b = __ffs(rows) - 1;
      rows &= rows - 1;
      const long long c = wfix[S.pcol()[32 * w + b]];
      cost += (x >> b) & 1u ? -c : c;
    }
  }
  return cost;
}

// Combination sweep OSD-CS-w of cluster r (App. D), as osd_cs in lsd.cu: no flip, every single
// dependent column, every pair among the first w in key order; ranked by (cost, class, key)
// with class 0 = no flip, 1 = single (key = the column's order key), 2 = pair (key = 16 i + j).
template <class I>
__device__ void osd_cs(const LSDArgs& a, const Shot<I>& S, int r, int np, int nsl, uint32_t* xw,
                       int lane) {
  const int wc = (nsl + 31) >> 5;
  int nt;
  const int sel = first_dependent(S, r, np, a.osd_cs, lane, nt);
  solution_words(S, xw, nsl, lane);
  long long bc = LLONG_MAX;
  int bcls = 3, b1 = -1, b2 = -1;
  unsigned long long bkey = 0;
  auto consider = [&](long long c, int cls, unsigned long long key, int u1, int u2) {
    if (c < bc || (c == bc && (cls < bcls || (cls == bcls && key < bkey)))) {
      bc = c;
      bcls = cls;
      bkey = key;
      b1 = u1;
      b2 = u2;
    }
  };
  if (lane == 0) consider(0, 0, 0, -1, -1);
#pragma unroll 1
  for (int u = lane; u < np; u += 32) {
    if (S.dpr()[u] != r) continue;
    consider(pattern_delta(a, S, xw, wc, u, -1), 1, dep_key(S, u), u, -1);
  }
  const int npairs = nt * (nt - 1) / 2;
#pragma unroll 1
  for (int t0 = 0; t0 < npairs; t0 += 32) {
    const int t = t0 + lane;
    int i = 0, rem = t < npairs ? t : 0;
    while (rem >= nt - 1 - i) {
      rem -= nt - 1 - i;
      ++i;
    }
    const int j = i + 1 + rem;
    const int u1 = __shfl_sync(kFull, sel, i), u2 = __shfl_sync(kFull, sel, j);
    if (t < npairs)
      consider(pattern_delta(a, S, xw, wc, u1, u2), 2, (unsigned long long)(i * 16 + j), u1, u2);
  }
#pragma unroll 1
  for (int off = 16; off > 0; off >>= 1) {
    const long long oc = __shfl_xor_sync(kFull, bc, off);
    const int ocls = __shfl_xor_sync(kFull, bcls, off);
    const unsigned long long okey = __shfl_xor_sync(kFull, bkey, off);
    const int o1 = __shfl_xor_sync(kFull, b1, off);
    const int o2 = __shfl_xor_sync(kFull, b2, off);
    consider(oc, ocls, okey, o1, o2);
  }
  if (b1 < 0) return;  // no flip: OSD-0's local solution stands
#pragma unroll 1
  for (int w = 0; w < wc; ++w) {
    uint32_t delta = S.npN()[(size_t)b1 * S.words() + w];
    if (b2 >= 0) delta ^= S.npN()[(size_t)b2 * S.words() + w];
    if ((delta >> lane) & 1u) S.flags()[32 * w + lane] ^= 1;
  }
  if (lane == 0) {
    S.ext()[atomicAdd(&S.sc->ext, 1)] = S.dpf()[b1];
    if (b2 >= 0) S.ext()[atomicAdd(&S.sc->ext, 1)] = S.dpf()[b2];
  }
}

// Work items come from a.queue / a.count as in lsd.cu.  Shots that outgrow the instance are
// appended to spill[] (counted in ctr->spill_count) when spill != nullptr, else reported
// unsolvable.  The large instance (items != nullptr) takes those.
template <class I>
__global__ void __launch_bounds__(I::NT, I::BIG ? 1 : 2)
lsd_sparse_kernel(LSDArgs a, unsigned char* scratch, size_t stride, int* spill, const int* items) {
  constexpr int NT = I::NT;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ Scal sc;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int m = a.g.m, n = a.g.n;
  const int wn = (n + 31) / 32;
  Shot<I> S;
  S.sc = &sc;
  S.sm = smem;
  {
    unsigned char* sp = smem + I::fixed;
    unsigned char* gp = scratch + (size_t)blockIdx.x * stride;
    auto take = [](unsigned char*& p, size_t bytes) {
      unsigned char* q = p;
      p += al16(bytes);
      return q;
    };
    S.cand = reinterpret_cast<uint32_t*>(take(sp, (size_t)wn * 4));
    S.joined = reinterpret_cast<uint32_t*>(take(sp, (size_t)wn * 4));
    if constexpr (I::LG) S.lab = reinterpret_cast<uint32_t*>(take(gp, (size_t)m * 4));
    else S.lab = reinterpret_cast<uint32_t*>(take(sp, (size_t)m * 4));
    S.li = I::BIG ? take(gp, I::list_bytes(m)) : take(sp, I::list_bytes(m));
    S.rs = I::row_stride(m);
    S.lcap = I::lcap(n);
    auto list = [&](unsigned char*& p) {
      S.ld = reinterpret_cast<uint2*>(take(p, (size_t)S.lcap * 8));
      S.lk = reinterpret_cast<uint32_t*>(take(p, (size_t)S.lcap * 4));
      S.lf = reinterpret_cast<uint16_t*>(take(p, (size_t)S.lcap * 2));
    };
    if constexpr (I::BIG && I::LG) list(gp);
    else list(sp);
  }
  const SGraph G{a.g.chk_ptr, a.g.var_ptr, a.g.var_chk, a.g.chk_pad,
                 reinterpret_cast<const uint2*>(a.g.var_pad), a.g.max_col_deg, a.g.max_row_deg};
  unsigned long long* const next = I::BIG ? &a.ctr->spill_next : &a.ctr->lsd_next;
  const unsigned count = (unsigned)(items               ? a.ctr->spill_count
                                    : a.count_from_ctr ? a.ctr->lsd_count
                                                       : (unsigned long long)a.count);
  unsigned long long steps_acc = 0, unsolv = 0;
  int kappa_max = 0, nu_max = 0;
  // the first item of a CTA is its block index, the others come from the counter
#pragma unroll 1
  for (unsigned item = blockIdx.x; item < count;) {
    const long long qi = items ? (long long)items[item] : (long long)item;
    const long long shot = a.queue ? (long long)a.queue[qi] : qi;
    const float* llr = a.llr + (a.llr_by_item ? qi : shot) * n;
    // the shot's correction: bytes, or packed words (set bits with atomicOr: threads share words)
    uint8_t* co = a.packed ? nullptr : a.corrections + shot * n;
    uint32_t* cw = a.packed ? reinterpret_cast<uint32_t*>(a.corrections) + shot * packed_words(n)
                            : nullptr;

    // ---- init: one cluster per flipped detector ----
#pragma unroll 1
    for (int d = tid; d < (m + 3) / 4; d += NT)
      reinterpret_cast<uint4*>(S.lab)[d] = make_uint4(kFree, kFree, kFree, kFree);
#pragma unroll 1
    for (int w = tid; w < wn; w += NT) S.cand[w] = S.joined[w] = 0u;
#pragma unroll 1
    for (int w = tid; w < I::SC / 32; w += NT) S.growb()[w] = 0u;
    if (tid == 0) {
      sc.ns = sc.nf = sc.n_new = sc.merged = sc.ng = sc.np = sc.ext = 0;
      sc.item = gridDim.x + (unsigned)atomicAdd(next, 1ULL);
    }
    __syncthreads();
    const unsigned next_item = sc.item;
    auto seed = [&](int d) {
      const int k = atomicAdd(&sc.ns, 1);
      if (k < I::SC && k < I::CAP) {
        S.lab[d] = ((uint32_t)k << 16) | (uint32_t)k;
        S.sdet()[k] = (uint16_t)d;
        S.slab()[k] = (uint16_t)k;
        S.parent()[k] = (uint16_t)k;
        S.flags()[k] = 1;
        S.inv()[k] = (uint16_t)k;
        atomicOr(&S.growb()[k >> 5], 1u << (k & 31));
      }
    };
    const uint8_t* sp = a.syndromes + shot * m;
    if (!a.packed && (m & 3) == 0 && (reinterpret_cast<uintptr_t>(sp) & 3) == 0) {
#pragma unroll 1
      for (int q = tid; q < m / 4; q += NT) {  // four detectors a load
        const uint32_t v = reinterpret_cast<const uint32_t*>(sp)[q];
        if (v == 0) continue;
#pragma unroll 1
        for (int b = 0; b < 4; ++b)
          if ((v >> (8 * b)) & 0xffu) seed(4 * q + b);
      }
    } else {
#pragma unroll 1
      for (int d = tid; d < m; d += NT)
        if (syn_bit(a.syndromes, a.packed, shot, m, d)) seed(d);
    }
    __syncthreads();
    const int ns = sc.ns;
    int status = LSD_SHOT_OK_LSD, steps = 0;
    if (ns > I::SC || ns > I::CAP) {
      status = kSpill;
    } else {
      if (tid == 0) sc.nsl = ns;
      open_slots(G, S, llr, 0, ns, tid);
      __syncthreads();
      if (sc.nf > S.lcap) status = kSpill;
    }

    // ---- LSD-0: grow every invalid cluster until all are valid ----
    int k = status == LSD_SHOT_OK_LSD ? ns : 0;
    while (k > 0) {
      if (steps > n) {  // each step adds a column: cannot be reached
        status = LSD_SHOT_UNSOLVABLE;
        break;
      }
      const bool single = k == 1 && G.max_col_deg <= 4;
      const int rc = single ? grow_single(G, S, llr, S.inv()[0], n, steps, tid)
                            : sparse_step(G, S, llr, k, true, tid);
      if (rc) {
        status = rc == 1 ? LSD_SHOT_UNSOLVABLE : kSpill;
        break;
      }
      if (single) break;
      ++steps;
      k = collect(S, sc.nsl, true, tid);
    }
    // ---- LSD-mu: mu more steps for every cluster, then the local reprocessing ----
    if constexpr (I::MU) {
#pragma unroll 1
      for (int e = 0; e < a.order && status == LSD_SHOT_OK_LSD; ++e) {
        k = collect(S, sc.nsl, false, tid);
        if (k == 0) break;
        const int rc = sparse_step(G, S, llr, k, false, tid);
        if (rc == 3) status = kSpill;
        if (rc == 2) break;
      }
      __syncthreads();
      const int np = sc.np;
      if (status == LSD_SHOT_OK_LSD)
#pragma unroll 1
        for (int u = tid; u < np; u += NT) {
          const int f = S.dpf()[u];
          S.dpr()[u] = (uint16_t)(S.lab[half4(G.var_pad[f], 0)] >> 16);
          S.dpk()[u] = llr_bits(llr[f]);
        }
      __syncthreads();
      if (status == LSD_SHOT_OK_LSD && np > 0) {
        uint32_t* xw = S.template s<uint32_t>(I::osd) + (size_t)warp * 2 * I::W;
        const int nsl = sc.nsl;
#pragma unroll 1
        for (int r = warp; r < ns; r += NT / 32) {
          if (S.parent()[r] != r) continue;
          if (a.osd_cs >= 0) osd_cs(a, S, r, np, nsl, xw, lane);
          else osd_e(a, S, r, np, nsl, xw, xw + I::W, lane);
          __syncwarp();
        }
      }
    }
    __syncthreads();

    // ---- the correction row, cleared; a shot without room goes to the large instance ----
    if (status != kSpill || !spill) {
      if (cw) {
#pragma unroll 1
        for (int w = tid; w < packed_words(n); w += NT) cw[w] = 0u;
      } else if ((n & 3) == 0 && (reinterpret_cast<uintptr_t>(co) & 3) == 0) {
#pragma unroll 1
        for (int j = tid; j < n / 4; j += NT) reinterpret_cast<uint32_t*>(co)[j] = 0u;
      } else {
#pragma unroll 1
        for (int j = tid; j < n; j += NT) co[j] = 0;
      }
    }
    if (status == kSpill) {
      if (tid == 0) {
        if (spill) spill[atomicAdd(&a.ctr->spill_count, 1ULL)] = (int)qi;
        else if (a.status) a.status[shot] = LSD_SHOT_UNSOLVABLE;
      }
      if (!spill) unsolv += 1;
      __syncthreads();
      item = next_item;
      continue;
    }
    // ---- statistics: nu clusters, kappa = largest cluster in columns ----
#pragma unroll 1
    for (int r = tid; r < ns; r += NT) S.best()[r] = 0u;
    if (tid == 0) sc.red[0][0] = sc.red[1][0] = 0u;
    __syncthreads();
    const int nf = sc.nf, nsl = sc.nsl;
#pragma unroll 1
    for (int x = tid; x < nf; x += NT) {
      const int f = S.lf[x];
      if ((S.joined[f >> 5] >> (f & 31)) & 1u)
        atomicAdd(&S.best()[S.lab[half4(S.ld[x], 0)] >> 16], 1u);
    }
    // ---- global decoding: union of the local solutions (Eq. 2) ----
    if (status == LSD_SHOT_OK_LSD) {
      auto set = [&](int j) {
        if (cw) atomicOr(cw + (j >> 5), 1u << (j & 31));
        else co[j] = 1;
      };
#pragma unroll 1
      for (int i = tid; i < nsl; i += NT)
        if ((S.flags()[i] & 3) == 3) set(S.pcol()[i]);
      if constexpr (I::MU) {
        const int ne = sc.ext;
#pragma unroll 1
        for (int t = tid; t < ne; t += NT) set(S.ext()[t]);
      }
    }
    __syncthreads();
    unsigned nu = 0, kappa = 0;
#pragma unroll 1
    for (int r = tid; r < ns; r += NT)
      if (S.parent()[r] == r) {
        ++nu;
        kappa = max(kappa, S.best()[r]);
      }
    nu = __reduce_add_sync(kFull, nu);
    kappa = __reduce_max_sync(kFull, kappa);
    if (lane == 0) {
      atomicAdd(&sc.red[0][0], nu);
      atomicMax(&sc.red[1][0], kappa);
    }
    __syncthreads();
    if (tid == 0) {
      nu = sc.red[0][0];
      kappa = sc.red[1][0];
      if (a.status) a.status[shot] = (uint8_t)status;
      if (a.shot_info) {
        a.shot_info[3 * shot] = (int)nu;
        a.shot_info[3 * shot + 1] = (int)kappa;
        a.shot_info[3 * shot + 2] = steps;
      }
      steps_acc += steps;
      unsolv += status == LSD_SHOT_UNSOLVABLE ? 1 : 0;
      kappa_max = max(kappa_max, (int)kappa);
      nu_max = max(nu_max, (int)nu);
    }
    item = next_item;
  }
  if (tid == 0) {
    if (steps_acc) atomicAdd(&a.ctr->lsd_steps, steps_acc);
    if (unsolv) atomicAdd(&a.ctr->unsolvable, unsolv);
    if (kappa_max) atomicMax(&a.ctr->kappa_max, kappa_max);
    if (nu_max) atomicMax(&a.ctr->nu_max, nu_max);
  }
}

template <bool MU, bool LG>
using Small = Inst<512, 512, 512, MU, false, LG>;
template <bool MU, bool LG>
using Big = Inst<1024, 4096, 4096, MU, true, LG>;

// Calls fn with the instance for an m x n matrix.
template <template <bool, bool> class T, bool MU, class F>
auto pick_instance(int m, int n, F&& fn) {
  if (smem_bytes<T<MU, false>>(m, n) > kSmemLimit) return fn(T<MU, true>());
  return fn(T<MU, false>());
}
template <class F>
auto with_instance(bool big, bool mu, int m, int n, F&& fn) {
  if (big) return mu ? pick_instance<Big, true>(m, n, fn) : pick_instance<Big, false>(m, n, fn);
  return mu ? pick_instance<Small, true>(m, n, fn) : pick_instance<Small, false>(m, n, fn);
}

}  // namespace

// Global scratch bytes per CTA.
size_t sparse_scratch_bytes(int m, int n, bool big, bool mu) {
  return with_instance(big, mu, m, n, [&](auto inst) { return scratch_bytes<decltype(inst)>(m, n); });
}

cudaError_t sparse_config(const DevGraph& g, int order, int* grid_small, int* grid_big) {
  int dev = 0, sms = 0, max_smem = 0;
  cudaError_t err = cudaGetDevice(&dev);
  if (err != cudaSuccess) return err;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  *grid_big = 0;
  for (const bool big : {false, true}) {
    if (big && with_instance(false, order > 0, g.m, g.n,
                             [&](auto inst) { return always_fits<decltype(inst)>(g.m, g.n); }))
      break;
    err = with_instance(big, order > 0, g.m, g.n, [&](auto inst) {
      using I = decltype(inst);
      const void* fn = (const void*)lsd_sparse_kernel<I>;
      cudaError_t e = allow_max_dynamic_smem(fn, max_smem);
      if (e != cudaSuccess) return e;
      int per_sm = 0;
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, I::NT, smem_bytes<I>(g.m, g.n));
      if (e != cudaSuccess) return e;
      if (per_sm < 1) return cudaErrorInvalidValue;
      *(big ? grid_big : grid_small) = per_sm * sms;
      return cudaSuccess;
    });
    if (err != cudaSuccess) return err;
  }
  return cudaSuccess;
}

cudaError_t launch_sparse(const LSDArgs& a, bool big, int grid, unsigned char* scratch, size_t stride,
                          int* spill, const int* items, cudaStream_t st) {
  return with_instance(big, a.order > 0, a.g.m, a.g.n, [&](auto inst) {
    using I = decltype(inst);
    lsd_sparse_kernel<I><<<grid, I::NT, smem_bytes<I>(a.g.m, a.g.n), st>>>(a, scratch, stride, spill, items);
    return cudaGetLastError();
  });
}

}  // namespace lsdgb
