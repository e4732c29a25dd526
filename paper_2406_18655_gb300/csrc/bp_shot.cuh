// Min-sum BP of one shot by a group of G lanes (G | 32) whose graph tables and messages sit
// in registers: lane l owns checks l, l + G, ... and variables l, l + G, ....  Used by
// bp_reg_kernel.  Same results as bp_kernel<G, 0> (the flooding min-sum of Sec. 4.3), bit for
// bit: every float operation that rounds is the same, in the same order.
#pragma once

#include "lsd_internal.cuh"

namespace lsdgb {

constexpr float kBig = 0x1p100f;  // minimum over an empty set (a degree-1 check)

// min(|a|, |b|) carrying the product of the signs: one instruction for what the scalar rule
// does with two absolute values, a minimum and a sign exclusive-or.  The BP values are never
// NaN (priors finite, messages at most alpha 2^100).
__device__ __forceinline__ float xorsign_min(float a, float b) {
  float d;
  asm("min.xorsign.abs.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
  return d;
}

// out[k] = min over the other entries of |q| (at most kBig), signed with the product of their
// signs: the check update before its scaling.  Prefix and suffix minima: 3 DC - 4 instructions
// of the ALU pipe, which bounds these kernels, against about 6 DC for tracking the two
// smallest magnitudes, comparing every edge with them and moving signs with logic.
// A minimum does not depend on the order it is taken in, so the result is the same bits.
template <int DC>
__device__ __forceinline__ void excluded_min(const float (&q)[DC], float (&out)[DC]) {
  static_assert(DC >= 2, "a check of a register shape has at least two edges");
  float p[DC];
  p[0] = xorsign_min(q[0], kBig);
#pragma unroll
  for (int k = 1; k < DC - 1; ++k) p[k] = xorsign_min(p[k - 1], q[k]);
  float s = xorsign_min(q[DC - 1], kBig);
  out[DC - 1] = p[DC - 2];
#pragma unroll
  for (int k = DC - 2; k > 0; --k) {
    out[k] = xorsign_min(p[k - 1], s);
    s = xorsign_min(s, q[k]);
  }
  out[0] = s;
}

namespace bpreg {

// Shared memory of a group: messages r, one word per (check slot c, edge k, lane), so that
// the lanes of a store or of a gather over consecutive checks hit consecutive banks, then
// Lam[VPL G].  Groups of less than a warp start half a row of banks apart.
template <int G, int CPL, int DC, int VPL>
struct Layout {
  static constexpr int kR = CPL * DC * G;
  static constexpr int kWords = kR + VPL * G;
  static constexpr int kPad = (G - kWords % 32 + 32) % 32;  // group g starts at bank g G mod 32
  static constexpr int kBytes = (kWords + kPad) * 4;
};

// Byte offsets from the start of the CTA's dynamic shared memory, two per register: the
// posterior of each edge of the lane's checks, the message of each edge of its variables.
// (An offset is one instruction away and a load adds nothing to it.)
template <int CPL, int DC, int VPL, int DV>
struct Tables {
  uint32_t cv[CPL][(DC + 1) / 2];
  uint32_t ve[VPL][(DV + 1) / 2];
  float prior[VPL];
};

template <int G, int CPL, int DC, int VPL, int DV>
__device__ __forceinline__ void load_tables(const DevGraph& g, int lane, int base,
                                            Tables<CPL, DC, VPL, DV>& T) {
  using Y = Layout<G, CPL, DC, VPL>;
  static_assert(Y::kBytes * (256 / G) <= 65536, "offsets are 16 bits");
  const uint32_t lam0 = (uint32_t)(base + 4 * Y::kR);
#pragma unroll
  for (int c = 0; c < CPL; ++c) {
    const int i = lane + G * c;
#pragma unroll
    for (int k = 0; k < (DC + 1) / 2; ++k) T.cv[c][k] = 0;
#pragma unroll
    for (int k = 0; k < DC; ++k) {
      // a lane without this check reads one posterior DC times (DC is even: parity 0)
      const uint32_t j = i < g.m ? g.chk_var[i * DC + k] : 0;
      T.cv[c][k >> 1] |= (lam0 + 4 * j) << (16 * (k & 1));
    }
  }
#pragma unroll
  for (int v = 0; v < VPL; ++v) {
    const int j = lane + G * v;
    T.prior[v] = j < g.n ? g.prior[j] : 0.f;
#pragma unroll
    for (int k = 0; k < (DV + 1) / 2; ++k) T.ve[v][k] = 0;
#pragma unroll
    for (int k = 0; k < DV; ++k) {
      const int e = j < g.n ? (int)g.var_edge[j * DV + k] : 0;
      const int i = e / DC, slot = ((i / G) * DC + (e - i * DC)) * G + i % G;
      T.ve[v][k >> 1] |= (uint32_t)(base + 4 * slot) << (16 * (k & 1));
    }
  }
}

__device__ __forceinline__ float at(const unsigned char* smem, uint32_t pair, int half) {
  const uint32_t off = half ? pair >> 16 : pair & 0xffffu;
  return *reinterpret_cast<const float*>(smem + off);
}

// Syndrome bits of the lane's checks (bit c = check lane + G c).
template <int G, int CPL, bool PK>
__device__ __forceinline__ unsigned load_syndrome(const BPArgs& a, unsigned shot, int lane) {
  const int m = a.g.m;
  unsigned bits = 0;
#pragma unroll
  for (int c = 0; c < CPL; ++c) {
    const int i = lane + G * c;
    if (i < m) {
      if constexpr (PK) {  // bit-packed syndromes (lsd_decode_batch_packed)
        const uint32_t* w = reinterpret_cast<const uint32_t*>(a.syndromes) + (size_t)shot * packed_words(m);
        if ((w[i >> 5] >> (i & 31)) & 1u) bits |= 1u << c;
      } else {
        if (a.syndromes[(size_t)shot * m + i]) bits |= 1u << c;
      }
    }
  }
  return bits;
}

// BP on a shot from the channel priors, given the syndrome bits of the lane's checks; returns
// the iterations run and sets conv (the hard decision of the final Lam satisfies the
// syndrome).  Lam holds the posteriors on return.  Lanes without a check or variable in a slot
// compute it all the same, on words of their own that nothing reads: no predicate on the way.
template <int G, int CPL, int DC, int VPL, int DV>
__device__ __forceinline__ int shot_bp(const BPArgs& a, const Tables<CPL, DC, VPL, DV>& T,
                                       unsigned sbits, unsigned char* smem, float* r, float* Lam,
                                       int lane, unsigned gmask, bool& conv) {
  static_assert(DC % 2 == 0, "an idle check slot must have even parity");
  float msg[CPL][DC];  // the lane's messages of the last check phase
#pragma unroll
  for (int c = 0; c < CPL; ++c)
#pragma unroll
    for (int k = 0; k < DC; ++k) msg[c][k] = 0.f;
#pragma unroll
  for (int v = 0; v < VPL; ++v) Lam[lane + G * v] = T.prior[v];
  __syncwarp(gmask);

  int t = 0;
  conv = false;
  for (;;) {
    // ---- check phase: the parity of [Lam^(t) < 0] first (a converged shot needs no messages),
    // then the messages r^(t+1); q takes the messages' place in between.  Sign bits stand for
    // the comparisons "< 0": the priors are finite and never -0 (0 < p < 1), so no Lam and no
    // q = Lam - r is -0 or NaN.
    uint32_t unsat = 0;  // bit 31: syndrome ^ signs of Lam, over the lane's checks
#pragma unroll
    for (int c = 0; c < CPL; ++c) {
      uint32_t hp = (sbits >> c) << 31;
#pragma unroll
      for (int k = 0; k < DC; ++k) {
        const float L = at(smem, T.cv[c][k >> 1], k & 1);
        hp ^= __float_as_uint(L);
        msg[c][k] = __fsub_rn(L, msg[c][k]);
      }
      unsat |= hp;
    }
    if (t > 0) {
      conv = !__any_sync(gmask, (unsat >> 31) != 0);
      if (conv && a.early_exit) break;
    }
    if (t >= a.iters) break;
#pragma unroll
    for (int c = 0; c < CPL; ++c) {
      float x[DC];
      excluded_min<DC>(msg[c], x);
      const float salpha = __uint_as_float(__float_as_uint(a.alpha) ^ ((sbits >> c) << 31));
#pragma unroll
      for (int k = 0; k < DC; ++k) {
        msg[c][k] = __fmul_rn(x[k], salpha);
        r[(c * DC + k) * G + lane] = msg[c][k];
      }
    }
    __syncwarp(gmask);
    // ---- variable phase: Lam^(t+1) ----
#pragma unroll
    for (int v = 0; v < VPL; ++v) {
      float L = T.prior[v];
#pragma unroll
      for (int k = 0; k < DV; ++k) L = __fadd_rn(L, at(smem, T.ve[v][k >> 1], k & 1));
      Lam[lane + G * v] = L;
    }
    __syncwarp(gmask);
    ++t;
  }
  return t;
}

}  // namespace bpreg
}  // namespace lsdgb
