// Adaptive parallel tempering with isoenergetic cluster moves (Algorithm S2)
// as one persistent CTA per problem: checkerboard p-bit sweeps of every
// replica, replica energies, best-energy tracking, Houdayer cluster moves
// and replica exchange all run on chip between kernel launches.  The same
// kernel also drives the chains of the adaptive-ladder preprocessing
// (energy sums over a tail window) and of the pilot runs (energy
// histograms).
//
// Layout.  Replicas ("buffers") of one problem are packed eight to a 32-bit
// word, one spin per nibble (bit 0 = +1): group g holds buffers 8g..8g+7.
// Sites are split by checkerboard colour c = (x+y+z)&1 and indexed inside a
// colour by j = lin >> 1.  Between launches global memory holds a word per
// (g, c, j), group by group; a CTA keeps up to four groups of a site side by
// side (a quad, the array S at Ctl), so that they move as one vector access.
// All replicas of a problem share the couplings, hence one word gives the
// nibble-packed satisfied-bond counts of eight replicas with six multiply-adds,
// and one Philox4x32-10 call gives their eight 16-bit uniforms.
//
// Replica slots are fixed: temperature r with ICM label a lives in buffer
// a*Tp + r (Tp = 8 ceil(T/8)), so the two labels of temperature r sit in the
// same nibble of groups h and h + G/2.  An accepted swap exchanges the two
// replicas' states (Algorithm S2) with SWAR nibble swaps, and the overlap of
// eight ICM pairs is one XOR of two words, which makes the cluster growth a
// nibble-parallel flood fill over all pairs at once.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "apt_dev.h"
#include "device.cuh"
#include "internal.h"

// Optional per-phase cycle counters of CTAs 0 and 1 (the two ranks of the
// first problem when problems split; build with -DPC_APT_PROFILE=1; read the
// 2 x 16 counters with pc_apt_profile_read).  Off by default.
#ifndef PC_APT_PROFILE
#define PC_APT_PROFILE 0
#endif
// Rounds of spreading inside a block per flood-fill pass (build-time knob).
#ifndef PC_APT_FILL_ROUNDS
#define PC_APT_FILL_ROUNDS 1
#endif
#if PC_APT_PROFILE
__device__ unsigned long long g_apt_prof[32];
#define PROF_MARK(slot, t0)                                                     \
  do {                                                                          \
    if (blockIdx.x < 2 && threadIdx.x == 0) {                                   \
      const long long t1_ = clock64();                                          \
      atomicAdd(&g_apt_prof[16 * blockIdx.x + (slot)], (unsigned long long)(t1_ - (t0))); \
      (t0) = t1_;                                                               \
    }                                                                           \
  } while (0)
#else
#define PROF_MARK(slot, t0) do { } while (0)
#endif

namespace {
using namespace pcdev;
using pc::AptArgs;
using pc::AptProbDev;

// The first two rounds of philox(c0, c1, c2, c3) taken apart, for draws that
// pair many (c0, c3) with many (c1, c2).  Round 1 turns c0 and c2 into
// products that do not meet before round 2, whose product of the c2 lane
// depends on (c0, c3) alone and whose product of the c0 lane depends on
// (c1, c2) alone: a site's part is shared by its replica groups, a group's
// part by the sites, and a draw starts at round 3 after two XORs (saves 4 of
// 20 wide products, the half-rate instructions, and 2 of 20 XORs).
struct PhiloxA { uint32_t lo0, b_lo, b_hi; };   // of (c0, c3)
struct PhiloxB { uint32_t x0, x2, lo; };        // of (c1, c2), round-2 keys folded in

__device__ __forceinline__ PhiloxA philox_a(uint32_t c0, uint32_t c3, uint32_t k1) {
  PhiloxA p;
  p.lo0 = 0xD2511F53u * c0;
  const uint32_t n2 = __umulhi(0xD2511F53u, c0) ^ c3 ^ k1;
  p.b_lo = 0xCD9E8D57u * n2;
  p.b_hi = __umulhi(0xCD9E8D57u, n2);
  return p;
}
__device__ __forceinline__ PhiloxB philox_b(uint32_t c1, uint32_t c2, uint32_t k0, uint32_t k1) {
  PhiloxB p;
  const uint32_t n0 = __umulhi(0xCD9E8D57u, c2) ^ c1 ^ k0;
  p.x0 = (0xCD9E8D57u * c2) ^ (k0 + 0x9E3779B9u);
  p.x2 = __umulhi(0xD2511F53u, n0) ^ (k1 + 0xBB67AE85u);
  p.lo = 0xD2511F53u * n0;
  return p;
}
__device__ __forceinline__ uint4 philox_ab(const PhiloxA &a, const PhiloxB &b, uint32_t k0, uint32_t k1) {
  uint32_t c0 = a.b_hi ^ b.x0, c1 = a.b_lo, c2 = b.x2 ^ a.lo0, c3 = b.lo;
  k0 += 2u * 0x9E3779B9u;
  k1 += 2u * 0xBB67AE85u;
#pragma unroll
  for (int r = 2; r < 10; ++r) {
    const uint32_t lo0 = 0xD2511F53u * c0, hi0 = __umulhi(0xD2511F53u, c0);
    const uint32_t lo1 = 0xCD9E8D57u * c2, hi1 = __umulhi(0xCD9E8D57u, c2);
    c0 = hi1 ^ c1 ^ k0;
    c2 = hi0 ^ c3 ^ k1;
    c1 = lo1;
    c3 = lo0;
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
  return make_uint4(c0, c1, c2, c3);
}

// The 16-bit word at a shared-window address.
__device__ __forceinline__ uint32_t lds_u16(uint32_t addr) {
  uint32_t v;
  asm("ld.shared.u16 %0, [%1];" : "=r"(v) : "r"(addr));
  return v;
}

// Everything a phase of the kernel needs to know about its CTA, at the start
// of dynamic shared memory.  The phases are functions of their own that read
// it from there: each gets its own register allocation, and nothing but the
// loop counters lives in registers across them (as one inlined kernel the
// phases shared the 128-register limit and every edit of one moved the code
// of the others).  Both CTAs of a split problem have it at the same address.
struct __align__(16) Ctl {
  int Lx, Ly, Lz, N, H, hx;
  uint32_t mhx, mLy, mLy2;
  int T, Tp, A, B, Bc, Gc, g0;
  // this CTA holds, for every label, the temperature groups [g0, g0 + Gu) of
  // the Glp groups per label (APT; ladder / pilot: A = 1, groups g0 ..);
  // split problems run as a cluster of two CTAs, rank 0 holding the hotter
  // (lower-beta, first) half.  parts: thread chunks per quad, where there are
  // more chunks than quads (PARTS kernels): chunk q sweeps part q % parts of
  // quad q / parts
  int Gu, Glp, parts, rank;
  int nbonds;        // bonds present (3N with periodic axes)
  int nreal;         // spins present (N without vacancies)
  uint32_t open;     // bit a: axis a open; bit 3: vacancies
  uint32_t ent;
  // replica groups in quads: quad q holds groups [q gq, (q + 1) gq), W = 1 << lw
  // words apart; the threads in nch chunks of tpc, chunk q sweeping quads q, q + nch, ..
  int nq, gq, lw, nch, tpc;
  uint32_t k0, k1, tag_main, tag_ref;
  int joint, icm_big;
  int swt_len;       // entries of each pair's swap table in shared memory
  int oThr, oThh, oHist, oS, oV, oJn, oPos, oStage, oSwt;   // word offsets of the arrays below
  const uint32_t *swapidx, *swaptab;   // the problem's swap tables in global memory
  int8_t *best_spins;                  // where this CTA's best state goes
  int64_t m64[4];      // best E, best sweep, hit sweep, target
  int64_t sum1[64], sum2[64];   // ladder sums
  int32_t m32[8];      // best buffer, flag, icm counters x3, any-swap flag, -, local best buffer
  int32_t E[64], Eacc[64], temp_of[64];
  int32_t satt[128], sacc[128];   // swap attempts / accepts of this launch
  uint32_t ikx[64];    // per pair: Philox word 0
  int32_t ibit[64];    // per pair: replica choice bit; [32 ..]: 4-label matching per temperature
  int32_t inm[32];     // per pair: mismatch count
  int32_t isz[32];     // per pair: cluster size
  uint32_t imask[24];  // [3][8] per group: cluster-flip masks, whole flips
  uint32_t swm[24];    // [8] per group: in-group swap nibble mask; [8] cross-group flags;
                       // [6] ICM matching nibble masks (4 labels)
  int32_t gmap[8];     // global group of each local group
  int32_t xch[24];     // split problems: [2][4] boundary energies by attempt parity;
                       // [8] accepted boundary labels; [12..17] the peer's best at launch
                       // end; [18..21] boundary draws
};
// Arrays after Ctl:
//   thr  [64][16]    p-bit thresholds of each buffer, entry I + 6
//   thh  [64][16]    their top halves, 16-bit, each group's 256 bytes on a 256-byte boundary
//   hist [T][n_bins] pilot histogram
//   stage [2][4][64] peer boundary spins by attempt parity, one bit per site (split)
//   swt  [T-1][swt_len] first entries (|dE| = 0, 2, ..) of each pair's swap table; larger |dE| read
//                    the table in global memory, two dependent loads on the deciding warp's path
//   S    [nq][2][H][W]  spin words: group q gq + u, colour c, site j at ((2 q + c) H + j) W + u, so
//                    the words of a site's groups move as one vector access
//   V    ICM cluster bits and overlap bits, block-major (below), transposed overlaps
//        [N/32][33], root masks
//   pos  [2][H] 16-bit: a site's place in the block-major arrays
//   jn   [2][H]      coupling signs (bits 0-5), missing bonds (8-13), vacancy (15) and, from bit
//                    16, the site's place: x odd in its row pair, wraps of +x -x +y -y +z -z

// The cluster and overlap words of ICM are kept by 2 x 2 x 2 block: site
// i = dx + 2 dy + 4 dz of block b at i kBlk + b (at most 512 blocks).  The
// constant stride makes every access of the flood fill a block index plus an
// immediate, and block kBlk - 1 of the cluster words stays 0, so that an
// absent outside neighbour (open axis) needs no mask.
constexpr int kBlk = 513;
constexpr int kFillRounds = PC_APT_FILL_ROUNDS;
constexpr int kXtStride = 33;   // a lane per chunk or a lane per pair: no bank conflict either way
// words from V on: V, X, the transposed X (or the cluster labels), root masks
__host__ __device__ inline int icm_words(int N) {
  const int nchunk = (N + 31) >> 5;
  return 16 * kBlk + kXtStride * nchunk + nchunk;
}

extern __shared__ __align__(16) uint32_t smem_words[];
__device__ __forceinline__ uint32_t *dyn_smem() { return smem_words; }
__device__ __forceinline__ Ctl &ctl() { return *reinterpret_cast<Ctl *>(dyn_smem()); }

// Groups per quad and words per quad and site: as few quads of at most four
// groups as hold Gc, evenly filled (8 -> 4 + 4, 6 -> 3 + 3).  A thread's four
// groups share the site's neighbours and couplings and one 16-byte access
// per neighbour.
__host__ __device__ inline int quads_of(int Gc) { return (Gc + 3) >> 2; }
__host__ __device__ inline int quad_groups(int Gc) { return (Gc + quads_of(Gc) - 1) / quads_of(Gc); }
__host__ __device__ inline int quad_shift(int Gc) { const int g = quad_groups(Gc); return g > 2 ? 2 : g - 1; }
// spin words per site of a CTA with Gc groups
__host__ __device__ inline int site_words(int Gc) { return quads_of(Gc) << quad_shift(Gc); }

// First word of local group g in S, and the word of canonical site kk = c H + j.
__device__ __forceinline__ int group_off(const Ctl &k, int g) {
  const int q = g / k.gq;
  return ((2 * k.H * q) << k.lw) + (g - q * k.gq);
}
__device__ __forceinline__ uint32_t &spin_word(const Ctl &k, uint32_t *S, int g, int kk) {
  return S[group_off(k, g) + (kk << k.lw)];
}

// Label of local group g (at most four labels of Gu groups each).
__device__ __forceinline__ int label_of(const Ctl &k, int g) {
  return (g >= k.Gu ? 1 : 0) + (g >= 2 * k.Gu ? 1 : 0) + (g >= 3 * k.Gu ? 1 : 0);
}

// Neighbours (other colour, colour-local index) of site (c, j) with packed
// word jb, in the direction order +x, -x, +y, -y, +z, -z; periodic wraps.
__device__ __forceinline__ void neighbours(const Ctl &k, int j, uint32_t jb, int (&n)[6]) {
  const int hx = k.hx, sy = hx, sz = hx * k.Ly, wy = sz - sy, wz = sz * (k.Lz - 1);
  n[0] = j + ((jb & (1u << 16)) ? ((jb & (1u << 17)) ? 1 - hx : 1) : 0);
  n[1] = j + ((jb & (1u << 16)) ? 0 : ((jb & (1u << 18)) ? hx - 1 : -1));
  n[2] = j + ((jb & (1u << 19)) ? -wy : sy);
  n[3] = j + ((jb & (1u << 20)) ? wy : -sy);
  n[4] = j + ((jb & (1u << 21)) ? -wz : sz);
  n[5] = j + ((jb & (1u << 22)) ? wz : -sz);
}

// The place bits (16 ..) of site (c, j).
__device__ __forceinline__ uint32_t place_bits(const Ctl &k, int c, int j) {
  const int row = (int)fdiv((uint32_t)j, k.mhx);   // j / hx
  const int jx = j - row * k.hx;
  const int z = (int)fdiv((uint32_t)row, k.mLy);   // row / Ly
  const int y = row - z * k.Ly;
  const uint32_t p = (uint32_t)((y + z + c) & 1);  // x = 2 jx + p
  return (p << 16) | (jx + 1 == k.hx ? 1u << 17 : 0u) | (jx == 0 ? 1u << 18 : 0u) |
         (y + 1 == k.Ly ? 1u << 19 : 0u) | (y == 0 ? 1u << 20 : 0u) | (z + 1 == k.Lz ? 1u << 21 : 0u) |
         (z == 0 ? 1u << 22 : 0u);
}

// lin = x + Lx (y + Ly z) of site (c, j).
__device__ __forceinline__ int lin_of(const Ctl &k, int c, int j) {
  const int row = (int)fdiv((uint32_t)j, k.mhx);
  const int jx = j - row * k.hx;
  const int z = (int)fdiv((uint32_t)row, k.mLy);
  const int y = row - z * k.Ly;
  return 2 * jx + ((y + z + c) & 1) + k.Lx * row;
}

// The first NG of the W words of a (quad, site), which start on a W-word
// boundary.
template <int NG>
__device__ __forceinline__ void load_vec(const uint32_t *p, uint32_t (&v)[NG]) {
  if constexpr (NG >= 3) {
    const uint4 t = *reinterpret_cast<const uint4 *>(p);
    v[0] = t.x; v[1] = t.y; v[2] = t.z;
    if constexpr (NG == 4) v[3] = t.w;
  } else if constexpr (NG == 2) {
    const uint2 t = *reinterpret_cast<const uint2 *>(p);
    v[0] = t.x; v[1] = t.y;
  } else {
    v[0] = *p;
  }
}
template <int NG>
__device__ __forceinline__ void store_vec(uint32_t *p, const uint32_t (&v)[NG]) {
  if constexpr (NG >= 3) {
    *reinterpret_cast<uint4 *>(p) = make_uint4(v[0], v[1], v[2], NG == 4 ? v[NG - 1] : 0u);
  } else if constexpr (NG == 2) {
    *reinterpret_cast<uint2 *>(p) = make_uint2(v[0], v[1]);
  } else {
    *p = v[0];
  }
}

// Eq. neuron for the 8 nibbles of one word.  SCALE 2: C holds per nibble
// the satisfied count of a site with all six bonds, whose entry is 2C;
// SCALE 1: C holds the threshold index I + 6.  thh holds the thresholds' top
// halves t as 16-bit entries [buffer][16], each group's 256 bytes starting
// on a 256-byte boundary of shared memory (tb, a shared-window address), so
// the entry of nibble i sits at tb | (32 i + 2 SCALE c_i), at most 248: the
// offsets of 4 nibbles are formed in one word and each address is one byte
// permute of that word with tb.  The sign of d = v - t for the main half v is
// the decision, and the top 4 bits of each d are shifted into w so that bit 3
// of nibble i carries half i's sign.  A zero product of the differences
// (mod 2^32) flags a possible tie, which refine8_grp settles exactly (a
// product that only wraps to 0 costs a needless refine).
template <int SCALE>
__device__ __forceinline__ uint32_t decide8_grp(const uint4 &x, uint32_t C, uint32_t tb, bool &tie) {
  // byte k of Dlo: offset of nibble 2k (64 k + 2 SCALE c); of Dhi: nibble 2k+1
  const uint32_t Dlo = (C & 0x0F0F0F0Fu) * (2u * SCALE) + 0xC0804000u;
  const uint32_t Dhi = ((C >> 4) & 0x0F0F0F0Fu) * (2u * SCALE) + 0xE0A06020u;
  uint32_t w = 0, tp = 1u;
#pragma unroll
  for (int i = 7; i >= 0; --i) {
    // byte 0 from the offsets, bytes 1-3 from tb
    const uint32_t th = lds_u16(__byte_perm((i & 1) ? Dhi : Dlo, tb, 0x7650u + (uint32_t)(i >> 1)));
    const uint32_t d = half_lo(x, i) - th;
    w = __funnelshift_l(d, w, 4);
    tp *= d;
  }
  tie |= (tp == 0u);
  return (w >> 3) & 0x11111111u;
}

// Threshold of nibble i (thr points at the group's 128 entries: 8 buffers x
// 16, entry I + 6 for I = -6..6).  SCALE 1: C holds I + 6 per nibble;
// SCALE 2: C holds the satisfied count, whose entry is 2C.
template <int SCALE>
__device__ __noinline__ uint32_t refine8_grp(uint32_t w, uint4 x, uint4 y, uint32_t C, const uint32_t *thr) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const uint32_t t = thr[16 * i + SCALE * ((C >> (4 * i)) & 0xFu)];
    const uint32_t v = half_hi(x, i);
    if (v == (t & 0xFFFF0000u)) {
      const uint32_t u = v | half_lo(y, i);
      w = (u < t) ? (w | (1u << (4 * i))) : (w & ~(1u << (4 * i)));
    }
  }
  return w;
}

// Satisfied-bond counts of NG groups in byte lanes: e8[u][0] byte k counts
// nibble 2k, e8[u][1] byte k nibble 2k + 1.  A site adds at most 6 to a
// lane, so a thread reduces them after at most kFlushSites sites.
constexpr int kFlushSites = 32;

// The NG groups of quad `quad` from its group u0 on at site (c, j), whose words
// start at Sq: the neighbour vectors are loaded first, then the NG decisions
// run as one branch-free block whose Philox chains are independent, ties
// (about 2^-13 per word) are settled after it, and the store comes last.  The
// field of 8 spins is
// C = n_neg 0x11111111 + sum_d eps_d W_d with eps_d = +1 (J > 0), -1 (J < 0)
// or 0 (absent bond): per nibble the count of satisfied present bonds
// (W ^ 1 for a negative bond is 1 - W), exact mod 2^32 because every final
// nibble lies in 0..6.
template <int NG, int W, bool UPDATE, bool ENERGY, bool OPEN>
__device__ __forceinline__ void quad_site(const Ctl &k, uint32_t *Sq, const uint32_t *jn, uint32_t tb0, int c, int j,
                                          int quad, int u0, uint32_t sweep, const PhiloxB (&pb)[NG],
                                          uint32_t (&e8)[NG][2]) {
  const int H = k.H;
  const uint32_t *Wo = Sq + (1 - c) * H * W;
  uint32_t *Wc = Sq + (c * H + j) * W;
  const uint32_t jb = jn[c * H + j];
  int n[6];
  neighbours(k, j, jb, n);
  const uint32_t miss = OPEN ? (jb >> 8) & 0x3Fu : 0u;
  const uint32_t K = OPEN ? (uint32_t)__popc(miss) * 0x11111111u : 0u;
  uint32_t C[NG], w[NG];
#pragma unroll
  for (int u = 0; u < NG; ++u) C[u] = (uint32_t)__popc(jb & 0x3Fu & ~miss) * 0x11111111u;
#pragma unroll
  for (int d = 0; d < 6; ++d) {
    uint32_t e = 1u - 2u * ((jb >> d) & 1u), nv[NG];
    if (OPEN && ((miss >> d) & 1u)) e = 0u;
    load_vec<NG>(Wo + n[d] * W, nv);
#pragma unroll
    for (int u = 0; u < NG; ++u) C[u] += e * nv[u];
  }
  if (UPDATE) {
    const PhiloxA pa = philox_a((uint32_t)j, (k.ent << 8) | k.tag_main, k.k1);
    uint32_t tmask = 0u;
#pragma unroll
    for (int u = 0; u < NG; ++u) {
      const uint4 x = philox_ab(pa, pb[u], k.k0, k.k1);
      // threshold index I + 6 = 2C + k per nibble when bonds are absent
      bool tie = false;
      w[u] = decide8_grp<OPEN ? 1 : 2>(x, OPEN ? 2u * C[u] + K : C[u], tb0 + 256u * (uint32_t)u, tie);
      tmask |= tie ? (1u << u) : 0u;
    }
    if (tmask) {
      const uint32_t *thr = dyn_smem() + k.oThr;
#pragma unroll
      for (int u = 0; u < NG; ++u) {
        if (!((tmask >> u) & 1u)) continue;
        const int g = quad * k.gq + u0 + u;
        const uint32_t c2 = ((uint32_t)c << 16) | (uint32_t)k.gmap[g];
        const uint4 x = philox((uint32_t)j, sweep, c2, (k.ent << 8) | k.tag_main, k.k0, k.k1);
        const uint4 y = philox((uint32_t)j, sweep, c2, (k.ent << 8) | k.tag_ref, k.k0, k.k1);
        w[u] = refine8_grp<OPEN ? 1 : 2>(w[u], x, y, OPEN ? 2u * C[u] + K : C[u], thr + 128 * g);
      }
    }
    store_vec<NG>(Wc, w);
  } else {
    load_vec<NG>(Wc, w);
  }
  if (ENERGY) {
#pragma unroll
    for (int u = 0; u < NG; ++u) {
      const uint32_t full = w[u] * 0xFu;    // nibble of all ones where the spin is +1
      const uint32_t sat = (C[u] & full) | ((0x66666666u - K - C[u]) & ~full);
      e8[u][0] += sat & 0x0F0F0F0Fu;
      e8[u][1] += (sat >> 4) & 0x0F0F0F0Fu;
    }
  }
}

// Colour c of NG groups of one quad, from its group u0 on: sites lt, lt + tpc,
// .. in blocks of at most kFlushSites per thread, so that the byte lanes of the
// energy counts cannot overflow.  Whole warps call it (the warp reductions).
// The counts leave a warp through one warp-wide add per packed word (two 16-bit
// lanes, at most 32 x 192 each) and one atomic per buffer, all buffers' lanes
// at once.
template <int NG, int W, bool UPDATE, bool ENERGY, bool OPEN>
__device__ __forceinline__ void quad_sites(Ctl &k, int c, uint32_t sweep, int quad, int lt, int tpc, int u0 = 0) {
  const int H = k.H;
  uint32_t *Sq = dyn_smem() + k.oS + 2 * quad * H * W + u0;
  const uint32_t *jn = dyn_smem() + k.oJn;
  const uint32_t tb0 = (uint32_t)__cvta_generic_to_shared(dyn_smem() + k.oThh) + 256u * (uint32_t)(quad * k.gq + u0);
  PhiloxB pb[NG];
  if (UPDATE) {
#pragma unroll
    for (int u = 0; u < NG; ++u)
      pb[u] = philox_b(sweep, ((uint32_t)c << 16) | (uint32_t)k.gmap[quad * k.gq + u0 + u], k.k0, k.k1);
  }
  for (int b0 = 0; b0 < H; b0 += ENERGY ? kFlushSites * tpc : H) {
    const int b1 = ENERGY ? min(H, b0 + kFlushSites * tpc) : H;
    uint32_t e8[NG][2];
#pragma unroll
    for (int u = 0; u < NG; ++u) e8[u][0] = e8[u][1] = 0u;
    for (int j = b0 + lt; j < b1; j += tpc)
      quad_site<NG, W, UPDATE, ENERGY, OPEN>(k, Sq, jn, tb0, c, j, quad, u0, sweep, pb, e8);
    if (ENERGY) {
      const int lane = threadIdx.x & 31;
      uint32_t mine = 0u;
#pragma unroll
      for (int u = 0; u < NG; ++u)
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          // low 16 bits: nibble m, high 16 bits: nibble m + 4
          const uint32_t v = __reduce_add_sync(0xFFFFFFFFu, (e8[u][m & 1] >> (8 * (m >> 1))) & 0x00FF00FFu);
          if ((lane >> 3) == u && (lane & 3) == m) mine = v;
        }
      if (lane < 8 * NG)
        atomicAdd(&k.Eacc[8 * (quad * k.gq + u0) + lane], (int)((lane & 4) ? mine >> 16 : mine & 0xFFFFu));
    }
  }
}

template <bool UPDATE, bool ENERGY, bool OPEN>
__device__ __forceinline__ void colour_phase_t(Ctl &k, int c, uint32_t sweep) {
  const int q = (int)threadIdx.x >= k.tpc ? 1 : 0, lt = (int)threadIdx.x - q * k.tpc;   // nch is 1 or 2: at most two quads
  for (int quad = q; quad < k.nq; quad += k.nch) {
    switch (k.gq) {
      case 4: quad_sites<4, 4, UPDATE, ENERGY, OPEN>(k, c, sweep, quad, lt, k.tpc); break;
      case 3: quad_sites<3, 4, UPDATE, ENERGY, OPEN>(k, c, sweep, quad, lt, k.tpc); break;
      case 2: quad_sites<2, 2, UPDATE, ENERGY, OPEN>(k, c, sweep, quad, lt, k.tpc); break;
      default: quad_sites<1, 1, UPDATE, ENERGY, OPEN>(k, c, sweep, quad, lt, k.tpc); break;
    }
  }
}

// The same with more chunks than quads (a launch shape asked for by nch):
// each of the `parts` chunks of a quad sweeps an even share of its groups,
// two or one.
template <bool UPDATE, bool ENERGY, bool OPEN>
__device__ __forceinline__ void colour_parts_t(Ctl &k, int c, uint32_t sweep) {
  const int q = (int)threadIdx.x / k.tpc, lt = (int)threadIdx.x - q * k.tpc;
  const int quad = q / k.parts, per = (k.gq + k.parts - 1) / k.parts, u0 = (q - quad * k.parts) * per;
  const int ng = min(per, k.gq - u0);
  if (ng < 1 || quad * k.gq + u0 >= k.Gc) return;   // three groups in four parts, or no group there
  if (ng == 2)
    quad_sites<2, 4, UPDATE, ENERGY, OPEN>(k, c, sweep, quad, lt, k.tpc, u0);
  else if (k.lw == 2)
    quad_sites<1, 4, UPDATE, ENERGY, OPEN>(k, c, sweep, quad, lt, k.tpc, u0);
  else
    quad_sites<1, 2, UPDATE, ENERGY, OPEN>(k, c, sweep, quad, lt, k.tpc, u0);
}
template <bool UPDATE, bool ENERGY>
__device__ __noinline__ void colour_parts(int c, uint32_t sweep) {
  Ctl &k = ctl();
  if (k.open)
    colour_parts_t<UPDATE, ENERGY, true>(k, c, sweep);
  else
    colour_parts_t<UPDATE, ENERGY, false>(k, c, sweep);
}

// One colour phase of a sweep over the CTA's groups.  UPDATE: Eq. synapse +
// Eq. neuron for every site of colour c.  ENERGY: accumulate, per buffer,
// the satisfied bonds of the colour-c sites (every bond has exactly one
// colour-1 endpoint, so the colour-1 pass gives E = nbonds - 2 * satisfied).
// A site missing k of its six bonds (open boundaries) counts its satisfied
// present bonds C, so I = 2C - (6 - k); the threshold row is indexed by
// I + 6 = 2C + k.  Periodic problems take the path without absent bonds.
template <bool UPDATE, bool ENERGY>
__device__ __noinline__ void colour_phase(int c, uint32_t sweep) {
  Ctl &k = ctl();
  if (k.open)
    colour_phase_t<UPDATE, ENERGY, true>(k, c, sweep);
  else
    colour_phase_t<UPDATE, ENERGY, false>(k, c, sweep);
}

// PARTS: the CTAs of this kernel may have more chunks than quads.  The choice
// is the kernel's, because a test per phase costs every launch that has no use
// for it (one function for both forms: adaptive ladders of 64 x L = 12 189.8 ->
// 194.7 ms, of 20 x L = 6 5.13 -> 5.37 ms).
template <bool UPDATE, bool ENERGY, bool PARTS>
__device__ __forceinline__ void colour(int c, uint32_t sweep) {
  if (PARTS && ctl().parts > 1)
    colour_parts<UPDATE, ENERGY>(c, sweep);
  else
    colour_phase<UPDATE, ENERGY>(c, sweep);
}

// Energies of label 0 only (two labels): its groups lead quad 0, all threads
// share the sites.
template <bool OPEN>
__device__ __forceinline__ void label0_energies_t(Ctl &k) {
  const int lt = (int)threadIdx.x, tpc = (int)blockDim.x;
  switch (k.Gu) {
    case 4: quad_sites<4, 4, false, true, OPEN>(k, 1, 0u, 0, lt, tpc); break;
    case 3: quad_sites<3, 4, false, true, OPEN>(k, 1, 0u, 0, lt, tpc); break;
    case 2: quad_sites<2, 4, false, true, OPEN>(k, 1, 0u, 0, lt, tpc); break;
    default: quad_sites<1, 2, false, true, OPEN>(k, 1, 0u, 0, lt, tpc); break;
  }
}
__device__ __noinline__ void label0_energies() {
  Ctl &k = ctl();
  if (k.open)
    label0_energies_t<true>(k);
  else
    label0_energies_t<false>(k);
}

// Warp 0, after the barrier that ends an energy pass: E_b = nbonds - 2
// (satisfied bonds), the accumulators back to 0 (half: label 0 was counted
// alone after a cluster move, which keeps each pair's E_a + E_b, so label 1
// follows), then the minimum-energy selection (Algorithm S2 output): strict
// improvement, lowest slot index (r * A + a) on ties.  The two CTAs of a
// split problem track their own candidates (rank 1 into a scratch state) and
// combine them at the end of the launch: the global best is the lower
// energy, found at the earlier sweep, rank 0 (the lower slots) on ties, and
// the target is first hit at the earlier of the two hits.  m32[1] tells the
// CTA that the state of buffer m32[7] is to be kept (copy_best).
__device__ __noinline__ void measure(int half, int64_t sweeps) {
  Ctl &k = ctl();
  const int lane = threadIdx.x, n = half ? 8 * k.Gu : 8 * k.Gc;
  for (int b = lane; b < n; b += 32) {
    const int e0 = k.nbonds - 2 * k.Eacc[b];
    if (half) k.E[b + n] += k.E[b] - e0;
    k.E[b] = e0;
    k.Eacc[b] = 0;
  }
  __syncwarp();
  // one warp minimum of the key (E + 2^18) 2^8 + slot (|E| <= 3N < 2^18, slot < 2^8)
  uint32_t key = 0xFFFFFFFFu;
  int bestb = 0;
  for (int b = lane; b < 8 * k.Gc; b += 32) {
    const int lg = b >> 3, lab = label_of(k, lg), r = 8 * (k.g0 + lg - lab * k.Gu) + (b & 7);
    if (r >= k.T) continue;
    const uint32_t kb = ((uint32_t)(k.E[b] + (1 << 18)) << 8) | (uint32_t)(r * k.A + lab);
    if (kb < key) {
      key = kb;
      bestb = b;
    }
  }
  const uint32_t mn = __reduce_min_sync(0xFFFFFFFFu, key);
  // the lane holding the minimum (keys are distinct), or lane 0 if no buffer holds a temperature
  if (mn != 0xFFFFFFFFu ? key == mn : lane == 0) {
    const int bestE = mn != 0xFFFFFFFFu ? (int)(mn >> 8) - (1 << 18) : 0x7FFFFFFF;
    int flag = 0;
    if ((int64_t)bestE < k.m64[0]) {
      k.m64[0] = bestE;
      k.m64[1] = sweeps;
      k.m32[0] = 8 * k.gmap[bestb >> 3] + (bestb & 7);
      k.m32[7] = bestb;
      flag = 1;
    }
    if (k.m64[2] < 0 && k.m64[0] <= k.m64[3]) k.m64[2] = sweeps;
    k.m32[1] = flag;
  }
  __syncwarp();
}

// The state of a new best replica, in lin order.
__device__ __noinline__ void copy_best() {
  Ctl &k = ctl();
  uint32_t *S = dyn_smem() + k.oS;
  const int b = k.m32[7], g = b >> 3, i = b & 7;
  int8_t *dst = k.best_spins;
  for (int kk = threadIdx.x; kk < k.N; kk += blockDim.x) {
    const int c = kk >= k.H ? 1 : 0, j = kk - c * k.H;
    dst[lin_of(k, c, j)] = ((spin_word(k, S, g, kk) >> (4 * i)) & 1u) ? 1 : -1;
  }
}

// 32 x 32 bit-matrix transpose across a warp: lane l holds row l on entry
// (bit c = element (l, c)) and column l on exit (bit r = element (r, l)).
// Five butterfly stages exchange the off-diagonal blocks of size 16..1.
__device__ __forceinline__ uint32_t warp_transpose32(uint32_t x) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int j = 16; j >= 1; j >>= 1) {
    const uint32_t m = j == 16 ? 0x0000FFFFu : j == 8 ? 0x00FF00FFu : j == 4 ? 0x0F0F0F0Fu
                                                     : j == 2 ? 0x33333333u : 0x55555555u;
    const uint32_t y = __shfl_xor_sync(0xFFFFFFFFu, x, j);
    x = (lane & j) ? ((x & ~m) | ((y & ~m) >> j)) : ((x & m) | ((y & m) << j));
  }
  return x;
}

// Pair p of temperature r = r0 + 8h + i owns bit 4i + b, b = h P + p < 4, of
// the per-site overlap and cluster words (A labels form P = A/2 pairs): eight
// pairs' nibble bits enter with one shift and leave with one.  Temperature
// of pair bit pb, or T and more where the bit has no pair.
__device__ __forceinline__ int pair_temp(const Ctl &k, int pb) {
  const int P = k.A >> 1, b = pb & 3;
  return b < k.Gu * P ? 8 * (k.g0 + (b >> (P - 1))) + (pb >> 2) : k.T;
}

// Place of canonical site kk = c H + j in the block-major arrays.
__device__ __forceinline__ int block_pos(const Ctl &k, int kk) {
  const int c = kk >= k.H ? 1 : 0, j = kk - c * k.H;
  const int row = (int)fdiv((uint32_t)j, k.mhx);   // j / hx
  const int bx = j - row * k.hx;
  const int z = (int)fdiv((uint32_t)row, k.mLy);   // row / Ly
  const int y = row - z * k.Ly;
  const int i = ((y + z + c) & 1) + 2 * (y & 1) + 4 * (z & 1);
  return i * kBlk + bx + k.hx * ((y >> 1) + (k.Ly >> 1) * (z >> 1));
}

// Union-find over 32-bit parent words in shared memory, every parent no
// larger than its child, so a root is the smallest index of its set.  A
// failed atomicMin means the word decreased meanwhile, which bounds the
// retries; the cap only guards the loop.
__device__ __forceinline__ uint32_t uf_find(volatile uint32_t *L, uint32_t x) {
  uint32_t p = L[x];
  for (int it = 0; p != x && it < 8192; ++it) {
    x = p;
    p = L[x];
  }
  return x;
}

__device__ __forceinline__ void uf_union(uint32_t *L, uint32_t a, uint32_t b) {
  volatile uint32_t *Lv = L;
  for (int it = 0; it < 1 << 16; ++it) {
    a = uf_find(Lv, a);
    b = uf_find(Lv, b);
    if (a == b) return;
    if (a < b) {
      const uint32_t t = a;
      a = b;
      b = t;
    }
    const uint32_t old = atomicMin(&L[a], b);   // link the larger root under the smaller
    if (old == a) return;
    a = old;
  }
}

// Seeds of the cluster-seed rule ("randomly pick one cluster" read as a
// uniform choice among the mismatch clusters): for each pair in turn, a
// union-find over the lattice bonds between its mismatch sites labels the
// clusters by their first site in canonical order (c*H + j); with n
// clusters, the k-th root, k = floor(x0 n / 2^32), seeds the pair's flood
// fill.  The labels use the transposed-overlap words, which this rule does
// not need; R holds one root bit per site.
__device__ __forceinline__ void icm_cluster_seeds(Ctl &k) {
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5;
  const int N = k.N, H = k.H, nchunk = (N + 31) >> 5;
  uint32_t *V = dyn_smem() + k.oV, *X = V + 8 * kBlk, *Lb = V + 16 * kBlk, *R = Lb + kXtStride * nchunk;
  const uint32_t *jn = dyn_smem() + k.oJn;
  const uint16_t *pos = reinterpret_cast<const uint16_t *>(dyn_smem() + k.oPos);
  volatile uint32_t *Lv = Lb;
  for (int pb = 0; pb < 32; ++pb) {
    if (pair_temp(k, pb) >= k.T || k.inm[pb] == 0) continue;
    for (int kk = tid; kk < N; kk += nt) Lb[kk] = ((X[pos[kk]] >> pb) & 1u) ? (uint32_t)kk : 0xFFFFFFFFu;
    __syncthreads();
    // every bond has one colour-0 end: unite each colour-0 mismatch site
    // with its mismatched neighbours over the bonds present
    for (int j = tid; j < H; j += nt) {
      if (!((X[pos[j]] >> pb) & 1u)) continue;
      int nb[6];
      neighbours(k, j, jn[j], nb);
      const uint32_t miss = (jn[j] >> 8) & 0x3Fu;
#pragma unroll
      for (int d = 0; d < 6; ++d) {
        const int kk2 = H + nb[d];
        if (((miss >> d) & 1u) == 0u && ((X[pos[kk2]] >> pb) & 1u)) uf_union(Lb, (uint32_t)j, (uint32_t)kk2);
      }
    }
    __syncthreads();
    for (int ch = warp; ch < nchunk; ch += (nt >> 5)) {
      const int kk = ch * 32 + lane;
      const bool root = kk < N && ((X[pos[kk]] >> pb) & 1u) && uf_find(Lv, (uint32_t)kk) == (uint32_t)kk;
      const uint32_t m = __ballot_sync(0xFFFFFFFFu, root);
      if (lane == 0) R[ch] = m;
    }
    __syncthreads();
    if (warp == 0) {
      int tot = 0;
      for (int ch = lane; ch < nchunk; ch += 32) tot += __popc(R[ch]);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(0xFFFFFFFFu, tot, o);
      const int kth = (int)(((uint64_t)k.ikx[pb] * (uint64_t)tot) >> 32);
      int base = 0;
      for (int ch0 = 0; ch0 < nchunk; ch0 += 32) {
        const int ch = ch0 + lane;
        uint32_t w = ch < nchunk ? R[ch] : 0u;
        const int cn = __popc(w);
        int inc = cn;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
          if (lane >= o) inc += y;
        }
        const int ex = base + inc - cn;
        const bool hit = kth >= ex && kth < ex + cn;
        if (hit) {
          int q = kth - ex, at = 0;
#pragma unroll
          for (int h = 16; h >= 1; h >>= 1) {
            const int cl = __popc(w & ((1u << h) - 1u));
            if (q >= cl) {
              q -= cl;
              w >>= h;
              at += h;
            }
          }
          V[pos[ch * 32 + at]] |= 1u << pb;
        }
        if (__any_sync(0xFFFFFFFFu, hit)) break;
        base += __shfl_sync(0xFFFFFFFFu, inc, 31);
      }
    }
    __syncthreads();
  }
}

// Overlap bits of one site: the XOR of the two labels' words of each pair,
// pair bit 4i + h A/2 + p for nibble i of group h.  p points at the
// site's words of quad 0, p1 at those of quad 1.
template <int A, int GL>
__device__ __forceinline__ uint32_t site_overlap(const Ctl &k, const uint32_t *p, const uint32_t *p1) {
  uint32_t xb = 0;
  if constexpr (A == 2) {
    constexpr int NW = GL <= 2 ? 2 * GL : GL;   // one quad holds both labels, or each label its own
    uint32_t w[NW], w1[GL];
    load_vec<NW>(p, w);
    if constexpr (GL > 2) load_vec<GL>(p1, w1);
#pragma unroll
    for (int h = 0; h < GL; ++h) xb |= (w[h] ^ (GL > 2 ? w1[h] : w[NW - GL + h])) << h;
  } else {
    // the two labels of pair p depend on each temperature's matching:
    // select nibbles by the matching masks
    uint32_t w[4 * GL];
    {
      uint32_t t[4];
      load_vec<4>(p, t);
#pragma unroll
      for (int i = 0; i < 4; ++i) w[i] = t[i];
      if constexpr (GL == 2) {
        load_vec<4>(p1, t);
#pragma unroll
        for (int i = 0; i < 4; ++i) w[4 * GL - 4 + i] = t[i];
      }
    }
#pragma unroll
    for (int h = 0; h < GL; ++h) {
      const uint32_t w0 = w[h], wa = w[GL + h], wb = w[2 * GL + h], wc = w[3 * GL + h];
      const uint32_t m0 = k.swm[16 + 3 * h], m1 = k.swm[17 + 3 * h], m2 = k.swm[18 + 3 * h];
      const uint32_t x0 = ((w0 ^ wa) & m0) | ((w0 ^ wb) & m1) | ((w0 ^ wc) & m2);
      const uint32_t x1 = ((wb ^ wc) & m0) | ((wa ^ wc) & m1) | ((wa ^ wb) & m2);
      xb |= (x0 << (2 * h)) | (x1 << (2 * h + 1));
    }
  }
  return xb;
}

// The cluster moves of one site: cluster bits v, flip masks imask.
template <int A, int GL>
__device__ __forceinline__ void site_flip(const Ctl &k, uint32_t *p, uint32_t *p1, uint32_t v, const uint32_t (&fm)[4 * GL]) {
  if constexpr (A == 2) {
    constexpr int NW = GL <= 2 ? 2 * GL : GL;
    uint32_t w[NW], w1[GL];
    load_vec<NW>(p, w);
    if constexpr (GL > 2) load_vec<GL>(p1, w1);
#pragma unroll
    for (int h = 0; h < GL; ++h) {
      const uint32_t vv = v >> h;   // the masks keep every fourth bit
      w[h] ^= (vv & fm[4 * h]) | fm[4 * h + 1];
      (GL > 2 ? w1[h] : w[NW - GL + h]) ^= (vv & fm[4 * h + 2]) | fm[4 * h + 3];
    }
    store_vec<NW>(p, w);
    if constexpr (GL > 2) store_vec<GL>(p1, w1);
  } else {
#pragma unroll
    for (int q = 0; q < GL; ++q) {
      uint32_t *pq = q ? p1 : p, w[4];
      load_vec<4>(pq, w);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int g = 4 * q + u, h = g % GL;   // g = label GL + h
        const uint32_t n0 = v >> (2 * h), n1 = v >> (2 * h + 1);
        w[u] ^= k.imask[16 + g] | (n0 & k.imask[2 * g]) | (n1 & k.imask[2 * g + 1]);
      }
      store_vec<4>(pq, w);
    }
  }
}

// (A) overlaps.  Warp w takes chunks of 32 sites in canonical order; the
// transpose of the chunk's X words gives lane r the chunk's mismatch
// bitmask of pair r, kept in Xt[chunk][r].
template <int A, int GL>
__device__ __forceinline__ void icm_overlaps(Ctl &k) {
  constexpr int W = A * GL == 2 ? 2 : 4;   // words per site and quad
  const int N = k.N, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5, nchunk = (N + 31) >> 5;
  const uint32_t *S = dyn_smem() + k.oS, *jn = dyn_smem() + k.oJn;
  uint32_t *V = dyn_smem() + k.oV, *X = V + 8 * kBlk, *Xt = V + 16 * kBlk;
  const uint16_t *pos = reinterpret_cast<const uint16_t *>(dyn_smem() + k.oPos);
  uint32_t nmis = 0;             // lane r: mismatches of pair r in this warp's chunks
#pragma unroll 2
  for (int ch = warp; ch < nchunk; ch += nw) {
    const int kk = ch * 32 + lane;
    uint32_t xb = 0;
    if (kk < N) {
      xb = site_overlap<A, GL>(k, S + kk * W, S + (N + kk) * W);
      if (jn[kk] & 0x8000u) xb = 0;   // a vacancy has no overlap: never a seed or member
      const int q = pos[kk];
      X[q] = xb;
      V[q] = 0u;
    }
    const uint32_t col = warp_transpose32(xb);
    Xt[ch * kXtStride + lane] = col;
    nmis += __popc(col);
  }
  if (nmis) atomicAdd(&k.inm[lane], (int)nmis);
}

// (E) flips, the masks read once into registers.
template <int A, int GL>
__device__ __forceinline__ void icm_flips(Ctl &k) {
  constexpr int W = A * GL == 2 ? 2 : 4;   // words per site and quad
  const int N = k.N;
  uint32_t *S = dyn_smem() + k.oS;
  const uint32_t *V = dyn_smem() + k.oV;
  const uint16_t *pos = reinterpret_cast<const uint16_t *>(dyn_smem() + k.oPos);
  uint32_t fm[4 * GL];
  if constexpr (A == 2) {
#pragma unroll
    for (int h = 0; h < GL; ++h) {
      fm[4 * h] = k.imask[h];
      fm[4 * h + 1] = k.imask[16 + h];
      fm[4 * h + 2] = k.imask[GL + h];
      fm[4 * h + 3] = k.imask[16 + GL + h];
    }
  }
  for (int kk = threadIdx.x; kk < N; kk += blockDim.x)
    site_flip<A, GL>(k, S + kk * W, S + (N + kk) * W, V[pos[kk]], fm);
}

// ICMop of Algorithm S2 for every temperature at once.  With A labels per
// temperature (2 or 4) the labels of temperature r = 8h + i sit in nibble i
// of groups l Gu + h, and pair p of the temperature's random matching owns bit
// 4i + h A/2 + p of the per-site overlap word X.  The seed of a pair is the
// k-th site (canonical order c*H + j) with its bit set, k = floor(x0 n_minus /
// 2^32); its cluster grows by a flood fill V <- V | (X & OR_nbr V) until no
// cluster changes.  Clusters larger than half of the spins present flip one
// whole replica (x1 bit 0: the pair's first or second label), smaller ones
// flip in both replicas.  The caller recounts the energies.
template <bool CSEED>
__device__ __noinline__ void icm_all(uint32_t t) {
  Ctl &k = ctl();
#if PC_APT_PROFILE
  long long pt = clock64();
#endif
  const int tid = threadIdx.x, nt = blockDim.x;
  const int N = k.N, H = k.H;
  // label l's groups are l*Gl .. l*Gl + Gl - 1; A is 2 or 4
  const int A = k.A, P = A >> 1, Gl = k.Gu;
  const int r0 = 8 * k.g0;   // first temperature held here
  uint32_t *V = dyn_smem() + k.oV;   // cluster bits (one bit per pair), block-major
  uint32_t *X = V + 8 * kBlk;        // overlap bits, block-major
  uint32_t *Xt = V + 16 * kBlk;      // [nchunk][kXtStride]
  const uint16_t *pos = reinterpret_cast<const uint16_t *>(dyn_smem() + k.oPos);
  int *match = k.ibit + 32;          // [32] matching of the labels of each temperature
  // the draws, on warp 1 (warp 0 may still be measuring)
  if (tid >= 32 && tid < 64) {
    const int pb = tid - 32, p = pb & (P - 1), r = pair_temp(k, pb);   // b = h P + p, P is 1 or 2
    if (r < k.T) {
      const uint4 x = philox((uint32_t)r, t, (uint32_t)p, (k.ent << 8) | TAG_ICM, k.k0, k.k1);
      k.ikx[pb] = x.x;
      k.ibit[pb] = (int)(x.y & 1u);
      // Algorithm S2 "randomly partition ICM replicas into pairs": with four
      // labels, one of the three perfect matchings, floor(3 x2 / 2^32) of
      // pair 0's draw; two labels always pair (0, 1)
      if (p == 0) match[r] = A == 4 ? (int)(((uint64_t)x.z * 3u) >> 32) : 0;
    }
  }
  if (tid >= 32 && tid < 64) {
    k.isz[tid - 32] = 0;
    k.inm[tid - 32] = 0;
  }
  __syncthreads();
  if (k.m32[1]) copy_best();
  if (A == 4) {
    if (tid < 3 * Gl) {
      // nibble masks of the temperatures of group h that use matching m
      const int h = tid / 3, m = tid - 3 * h;
      uint32_t mk = 0;
      for (int i = 0; i < 8; ++i) {
        const int r = r0 + 8 * h + i;
        if (r < k.T && match[r] == m) mk |= 0xFu << (4 * i);
      }
      k.swm[16 + tid] = mk;
    }
    __syncthreads();
  }
  const int lane = tid & 31, warp = tid >> 5, nw = nt >> 5, nchunk = (N + 31) >> 5;
  if (A == 2) {
    switch (Gl) {
      case 4: icm_overlaps<2, 4>(k); break;
      case 3: icm_overlaps<2, 3>(k); break;
      case 2: icm_overlaps<2, 2>(k); break;
      default: icm_overlaps<2, 1>(k); break;
    }
  } else if (Gl == 2) {
    icm_overlaps<4, 2>(k);
  } else {
    icm_overlaps<4, 1>(k);
  }
  __syncthreads();
  PROF_MARK(4, pt);
  // seeds: warp w finds the k-th mismatch of pairs w, w + nw, ...: chunk
  // counts by popcount, a warp scan over chunks, then the set bit inside
  // the chunk (the cluster-seed rule finds the k-th cluster instead)
  if (CSEED) icm_cluster_seeds(k);
  if (!CSEED && nchunk <= 8 && warp == 0) {
    // few chunks: a lane per pair walks them
    const int r = lane, nm = pair_temp(k, r) < k.T ? k.inm[r] : 0;
    int q = (int)(((uint64_t)k.ikx[r] * (uint64_t)nm) >> 32);
    bool find = nm > 0;
    for (int ch = 0; ch < nchunk && find; ++ch) {
      uint32_t w = Xt[ch * kXtStride + r];
      const int cn = __popc(w);
      if (q < cn) {
        int at = 0;
#pragma unroll
        for (int h = 16; h >= 1; h >>= 1) {
          const int cl = __popc(w & ((1u << h) - 1u));
          if (q >= cl) {
            q -= cl;
            w >>= h;
            at += h;
          }
        }
        atomicOr(&V[pos[ch * 32 + at]], 1u << r);
        find = false;
      }
      q -= cn;
    }
  }
  const int nb = Gl * P;   // pairs per nibble, 1 .. 4
  for (int v = warp; v < 8 * nb && !CSEED && nchunk > 8; v += nw) {
    const int vi = nb == 4 ? v >> 2 : nb == 3 ? (v * 43) >> 7 : v >> (nb - 1);   // v / nb, v < 32
    const int r = 4 * vi + v - nb * vi;                                           // pair bit
    if (pair_temp(k, r) >= k.T) continue;
    const int nm = k.inm[r];
    if (nm == 0) continue;
    int kth = (int)(((uint64_t)k.ikx[r] * (uint64_t)nm) >> 32);
    // lane l takes chunks [l cl, (l + 1) cl): its count, one scan over the
    // lanes, and the lane that holds the kth mismatch walks its chunks
    const int cl = (nchunk + 31) >> 5, c0 = lane * cl, c1 = min(nchunk, c0 + cl);
    int cn = 0;
#pragma unroll 4
    for (int ch = c0; ch < c1; ++ch) cn += __popc(Xt[ch * kXtStride + r]);
    int inc = cn;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
      if (lane >= o) inc += y;
    }
    kth -= inc - cn;
    if (kth >= 0 && kth < cn) {
      for (int ch = c0; ch < c1; ++ch) {
        uint32_t w = Xt[ch * kXtStride + r];
        const int n1 = __popc(w);
        if (kth < n1) {
          // set bit number kth of w: binary search on popcounts of the low
          // half of the remaining window
          int at = 0;
#pragma unroll
          for (int h = 16; h >= 1; h >>= 1) {
            const int lo = __popc(w & ((1u << h) - 1u));
            if (kth >= lo) {
              kth -= lo;
              w >>= h;
              at += h;
            }
          }
          atomicOr(&V[pos[ch * 32 + at]], 1u << r);
          break;
        }
        kth -= n1;
      }
    }
  }
  __syncthreads();
  PROF_MARK(5, pt);
  // (B) flood fill.  The cluster is the least fixed point of the monotone
  // update V <- V | (X & OR_nbr V).  A thread owns 2x2x2 blocks of sites: per
  // pass it reads the 24 outside neighbours of a block (each the opposite
  // site's word of an adjacent block), then spreads inside the cube axis by
  // axis, kFillRounds times.  Each site word has one writer, so passes run
  // without inner barriers (a stale neighbour read only delays growth), and a
  // pass with no change anywhere, started after a barrier, proves the fixed
  // point: it ORs in every neighbour of every site.  A pass is a chain of
  // dependent loads and logic on few warps (216 blocks at L = 12), so what
  // counts is its length: 64 x L = 12, 14 passes, 15.1k cycles with 24
  // computed addresses and masks and three rounds of all six directions,
  // 10.5k so (two rounds per pass 11.0k, three 11.6k: fewer passes do not
  // pay for longer ones).
  {
    const int hx = k.hx, hy = k.Ly >> 1, hz = k.Lz >> 1, nblk = N >> 3;
    constexpr int kZero = kBlk - 1;   // the block of zeros
    // indices of the six adjacent blocks, -x +x -y +y -z +z; an open axis has
    // no bond across its ends
    auto adjacent = [&](int blk, int (&nb)[6]) {
      const int rest = (int)fdiv((uint32_t)blk, k.mhx);           // blk / hx
      const int bx = blk - rest * hx;
      const int bz = (int)fdiv((uint32_t)rest, k.mLy2);           // rest / (Ly/2)
      const int by = rest - bz * hy;
      const int sy = hx, sz = hx * hy;
      nb[0] = bx > 0 ? blk - 1 : ((k.open & 1u) ? kZero : blk + hx - 1);
      nb[1] = bx + 1 < hx ? blk + 1 : ((k.open & 1u) ? kZero : blk - (hx - 1));
      nb[2] = by > 0 ? blk - sy : ((k.open & 2u) ? kZero : blk + sz - sy);
      nb[3] = by + 1 < hy ? blk + sy : ((k.open & 2u) ? kZero : blk - (sz - sy));
      nb[4] = bz > 0 ? blk - sz : ((k.open & 4u) ? kZero : blk + sz * (hz - 1));
      nb[5] = bz + 1 < hz ? blk + sz : ((k.open & 4u) ? kZero : blk - sz * (hz - 1));
    };
    // one relaxation of a block; writes its words if any changed
    auto relax = [&](int blk, const int (&nb)[6], const uint32_t (&x)[8], uint32_t (&v)[8]) {
      uint32_t nv[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const uint32_t ox = V[(i ^ 1) * kBlk + nb[i & 1]];
        const uint32_t oy = V[(i ^ 2) * kBlk + nb[2 + ((i >> 1) & 1)]];
        const uint32_t oz = V[(i ^ 4) * kBlk + nb[4 + (i >> 2)]];
        nv[i] = v[i] | (x[i] & (ox | oy | oz));
      }
#pragma unroll
      for (int round = 0; round < kFillRounds; ++round) {
#pragma unroll
        for (int ax = 1; ax <= 4; ax <<= 1) {
#pragma unroll
          for (int i = 0; i < 8; ++i)
            if (!(i & ax)) {
              const uint32_t a0 = nv[i], a1 = nv[i ^ ax];
              nv[i] = a0 | (x[i] & a1);
              nv[i ^ ax] = a1 | (x[i ^ ax] & a0);
            }
        }
      }
      uint32_t d = 0;
#pragma unroll
      for (int i = 0; i < 8; ++i) d |= nv[i] ^ v[i];
      if (d) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          V[i * kBlk + blk] = nv[i];
          v[i] = nv[i];
        }
      }
      return d != 0u;
    };
    if (nblk <= 32) {
      // small lattices: one warp, passes end with a vote instead of a barrier
      if (warp == 0) {
        int nb[6];
        uint32_t v[8], x[8];
        if (lane < nblk) adjacent(lane, nb);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          v[i] = lane < nblk ? V[i * kBlk + lane] : 0u;
          x[i] = lane < nblk ? X[i * kBlk + lane] : 0u;
        }
        for (int it = 0; it < N; ++it) {
          const bool changed = lane < nblk && relax(lane, nb, x, v);
          __syncwarp();
          if (!__any_sync(0xFFFFFFFFu, changed)) break;
        }
      }
      __syncthreads();
    } else if (nblk <= nt) {
      // one block per thread: its neighbours, cluster and overlap words stay
      // in registers across passes (the thread is their only writer)
      int nb[6];
      uint32_t v[8], x[8];
      bool open = false;
      if (tid < nblk) {
        adjacent(tid, nb);
        uint32_t o = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          v[i] = V[i * kBlk + tid];
          x[i] = X[i * kBlk + tid];
          o |= x[i] & ~v[i];
        }
        open = o != 0;
      }
      for (int it = 0; it < N; ++it) {
        int changed = 0;
        if (open) {
          changed = relax(tid, nb, x, v);
          uint32_t o = 0;
#pragma unroll
          for (int i = 0; i < 8; ++i) o |= x[i] & ~v[i];
          open = o != 0;
        }
        if (!__syncthreads_or(changed)) {
#if PC_APT_PROFILE
          if (blockIdx.x < 2 && tid == 0) atomicAdd(&g_apt_prof[16 * blockIdx.x + 11], (unsigned long long)(it + 1));
#endif
          break;
        }
      }
    } else {
      for (int it = 0; it < N; ++it) {
        int changed = 0;
        for (int blk = tid; blk < nblk; blk += nt) {
          uint32_t x[8], v[8];
          uint32_t open = 0;
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            x[i] = X[i * kBlk + blk];
            v[i] = V[i * kBlk + blk];
            open |= x[i] & ~v[i];
          }
          if (open) {
            int nb[6];
            adjacent(blk, nb);
            changed |= relax(blk, nb, x, v);
          }
        }
        if (!__syncthreads_or(changed)) break;
      }
    }
  }
  PROF_MARK(6, pt);
  // (C) cluster sizes.  A lane adds the eight words of its block into four
  // bit planes (counts 0 .. 8 of every pair); the transposes of a warp's
  // planes give lane r pair r's counts over 32 blocks.
  {
    const int nblk = N >> 3;
    uint32_t sz = 0;
    for (int b0 = 32 * warp; b0 < nblk; b0 += nt) {
      const int b = b0 + lane;
      uint32_t w[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) w[i] = b < nblk ? V[i * kBlk + b] : 0u;
      auto add3 = [](uint32_t x, uint32_t y, uint32_t z, uint32_t &cy) {
        cy = (x & y) | (x & z) | (y & z);
        return x ^ y ^ z;
      };
      uint32_t c0, c1, c2, c3, c4, c5;
      const uint32_t s0 = add3(w[0], w[1], w[2], c0), s1 = add3(w[3], w[4], w[5], c1);
      const uint32_t s2 = add3(s0, s1, w[6], c2), p0 = s2 ^ w[7];
      c3 = s2 & w[7];
      const uint32_t t = add3(c0, c1, c2, c4), p1 = t ^ c3;
      c5 = t & c3;
      sz += (uint32_t)__popc(warp_transpose32(p0)) + 2u * (uint32_t)__popc(warp_transpose32(p1)) +
            4u * (uint32_t)__popc(warp_transpose32(c4 ^ c5)) + 8u * (uint32_t)__popc(warp_transpose32(c4 & c5));
    }
    if (sz) atomicAdd(&k.isz[lane], (int)sz);
  }
  __syncthreads();
  // (D) decisions, warp 0, a lane per pair.  imask[(g P + p)] (g = l Gl + h):
  // nibbles of label l's group h flipped by pair p's cluster; imask[16 + g]:
  // whole-replica flips.  The lanes' bits reach the masks as ballots: pair
  // bits h P + p, h P + p + 4, .. are the nibbles of group h.
  if (warp == 0) {
    const int pb = lane, p = pb & (P - 1), r = pair_temp(k, pb);
    const bool valid = r < k.T;
    const int m = valid ? match[r] : 0;
    const int la = p == 0 ? 0 : (m == 0 ? 2 : 1);
    const int lb = p == 0 ? m + 1 : (m == 2 ? 2 : 3);
    const bool none = valid && k.inm[pb] == 0;
    const bool big = valid && !none && k.icm_big && 2 * k.isz[pb] > k.nreal;   // more than half of the spins present
    const bool small = valid && !none && !big;
    const int whole = big ? (k.ibit[pb] ? lb : la) : -1;   // the replica that flips whole
    const uint32_t mn = __ballot_sync(0xFFFFFFFFu, none), ms = __ballot_sync(0xFFFFFFFFu, small),
                   mb = __ballot_sync(0xFFFFFFFFu, big);
    for (int l = 0; l < A; ++l) {
      const uint32_t fl = __ballot_sync(0xFFFFFFFFu, small && (la == l || lb == l));
      const uint32_t wh = __ballot_sync(0xFFFFFFFFu, whole == l);
      if (lane < Gl * P) k.imask[l * Gl * P + lane] = (fl >> lane) & 0x11111111u;
      if (lane < Gl) {
        uint32_t w = 0u;
        for (int q = 0; q < P; ++q) w |= (wh >> (lane * P + q)) & 0x11111111u;
        k.imask[16 + l * Gl + lane] = w;
      }
    }
    if (lane == 0) {
      k.m32[2] += __popc(mn);
      k.m32[3] += __popc(ms);
      k.m32[4] += __popc(mb);
    }
  }
  __syncthreads();
  PROF_MARK(7, pt);
  if (A == 2) {
    switch (Gl) {
      case 4: icm_flips<2, 4>(k); break;
      case 3: icm_flips<2, 3>(k); break;
      case 2: icm_flips<2, 2>(k); break;
      default: icm_flips<2, 1>(k); break;
    }
  } else if (Gl == 2) {
    icm_flips<4, 2>(k);
  } else {
    icm_flips<4, 1>(k);
  }
  __syncthreads();
  PROF_MARK(8, pt);
}


// Applies the swap masks of the last attempt (Ctl::swm) to the words of
// colour c.  The groups that exchange nibbles with one another belong to one
// label, hence to one quad.  A split problem's boundary swap (bmask:
// accepted labels) also writes the peer CTA's spins, pushed into `stage`,
// into this CTA's boundary nibble.
template <int GQ>
__device__ __forceinline__ void swap_quads(Ctl &k, int c, uint32_t bmask, const uint32_t *stage) {
  constexpr int W = GQ == 3 ? 4 : GQ;
  const int H = k.H;
  // rank 0 receives into nibble 7 of each label's last group, rank 1 into
  // nibble 0 of each label's first group
  const int bsh = k.rank == 0 ? 28 : 0, bgoff = k.rank == 0 ? k.Gu - 1 : 0;
  for (int quad = 0; quad < k.nq; ++quad) {
    // in-group nibble masks, pairs (u, u + 1) whose nibbles 7 and 0 exchange,
    // and the labels whose boundary group lies in this quad
    uint32_t m[GQ], cross = 0, any = 0, bl[GQ];
#pragma unroll
    for (int u = 0; u < GQ; ++u) {
      const int g = quad * GQ + u;
      m[u] = g < k.Gc ? k.swm[g] : 0u;
      any |= m[u];
      if (u + 1 < GQ && g + 1 < k.Gc && k.swm[8 + g]) cross |= 1u << u;
      bl[u] = 0u;
      if (bmask && g < k.Gc) {
        const int l = label_of(k, g);
        if (g - l * k.Gu == bgoff && ((bmask >> l) & 1u)) bl[u] = (uint32_t)(64 * l) + 1u;   // 1 + its stage row
        any |= bl[u];
      }
    }
    if (!(any | cross)) continue;
    uint32_t *Sq = dyn_smem() + k.oS + (2 * quad + c) * H * W;
    for (int j = threadIdx.x; j < H; j += blockDim.x) {
      uint32_t w[GQ];
      load_vec<GQ>(Sq + j * W, w);
#pragma unroll
      for (int u = 0; u < GQ; ++u) {
        const uint32_t d = (w[u] ^ (w[u] >> 4)) & m[u];
        w[u] ^= d | (d << 4);
      }
#pragma unroll
      for (int u = 0; u + 1 < GQ; ++u)
        if ((cross >> u) & 1u) {
          const uint32_t d = ((w[u] >> 28) ^ w[u + 1]) & 1u;
          w[u] ^= d << 28;
          w[u + 1] ^= d;
        }
#pragma unroll
      for (int u = 0; u < GQ; ++u)
        if (bl[u]) {
          const uint32_t bit = (stage[bl[u] - 1u + (uint32_t)(j >> 5)] >> (j & 31)) & 1u;
          w[u] = (w[u] & ~(1u << bsh)) | (bit << bsh);
        }
      store_vec<GQ>(Sq + j * W, w);
    }
  }
}
__device__ __noinline__ void swap_words(int c, uint32_t bmask, int par) {
  Ctl &k = ctl();
  const uint32_t *stage = dyn_smem() + k.oStage + 256 * par;
  switch (k.gq) {
    case 4: swap_quads<4>(k, c, bmask, stage); break;
    case 3: swap_quads<3>(k, c, bmask, stage); break;
    case 2: swap_quads<2>(k, c, bmask, stage); break;
    default: swap_quads<1>(k, c, bmask, stage); break;
  }
}

// Split problems: writes this CTA's boundary spins of colour c, every
// label, one bit per site, into the peer CTA's stage[par] (distributed
// shared memory).  Rank 0 sends the last (coldest) temperature of its half
// (nibble 7 of each label's last group), rank 1 the first (hottest) of its
// half (nibble 0 of each label's first group).
__device__ __noinline__ void push_boundary(int c, int par, int w0) {
  namespace cg = cooperative_groups;
  Ctl &k = ctl();
  const int H = k.H;
  uint32_t *S = dyn_smem() + k.oS;
  uint32_t *pstage = cg::this_cluster().map_shared_rank(dyn_smem() + k.oStage, k.rank ^ 1) + 256 * par;
  const int sh_own = k.rank == 0 ? 28 : 0, goff = k.rank == 0 ? k.Gu - 1 : 0;
  // warps w0 .. take part
  const int lane = threadIdx.x & 31, nw = (blockDim.x >> 5) - w0;
  for (int base = ((int)(threadIdx.x >> 5) - w0) * 32; base < H; base += nw * 32) {
    const int e = base + lane;
    for (int l = 0; l < k.A; ++l) {
      uint32_t bit = 0;
      if (e < H) bit = (spin_word(k, S, l * k.Gu + goff, c * H + e) >> sh_own) & 1u;
      const uint32_t word = __ballot_sync(0xFFFFFFFFu, bit);
      if (lane == 0) pstage[64 * l + (base >> 5)] = word;
    }
  }
}
// Replica exchange of attempt t (Sec. "Comparison with Adaptive Parallel
// Tempering"; Methods): even t pairs (0,1),(2,3)..., odd t (1,2),(3,4)...;
// each label decides on its own; p_swap = min(1, exp(dbeta dE)).  Accepted
// pairs exchange their p-bit states (SWAR nibble swaps over all sites) and
// energies.  A split problem pushes its boundary spins and energies to the
// peer CTA before one cluster barrier; both CTAs then decide the boundary
// pair from the same energies and random word, and take the peer's spins
// for the accepted labels.  Buffers alternate with the attempt's parity, so
// one barrier per attempt orders every exchange.
template <bool SPLIT>
__device__ __noinline__ void swap_step(uint32_t t) {
  Ctl &k = ctl();
#if PC_APT_PROFILE
  long long pt = clock64();
#endif
  const int A = k.A, lA2 = A >> 1, q = (int)(t & 1u);   // A = 1 << lA2 (1, 2 or 4)
  const int r0 = 8 * k.g0, r1 = min(8 * (k.g0 + k.Gu), k.T);   // temperatures held here
  // local buffer of (label l, temperature r): l * 8 Gu + r - r0
  const int lb = 8 * k.Gu;
  auto swap_table = [&](int r, int dE) {
    const int kk = (-dE) >> 1;
    if (kk < k.swt_len) return dyn_smem()[k.oSwt + r * k.swt_len + kk];   // staged at launch
    const uint32_t off = k.swapidx[2 * r], len = k.swapidx[2 * r + 1];
    return ((uint32_t)kk < len) ? k.swaptab[off + kk] : 0u;
  };
  const int par = (int)(t & 1u);
  const int warp = threadIdx.x >> 5;
  if (SPLIT) {
    // energies of this side of the boundary pair, and its colour-1 spins
    // (warps 1 ..; warp 0 starts on the decisions meanwhile)
    const int rb_own = k.rank == 0 ? r1 - 1 : r0;
    int *pe = cooperative_groups::this_cluster().map_shared_rank(k.xch, k.rank ^ 1) + 4 * par;
    if (threadIdx.x < A) pe[threadIdx.x] = k.E[threadIdx.x * lb + rb_own - r0];
    if (warp >= 1) push_boundary(1, par, 1);
    // the boundary pair's draws do not depend on the energies: warp 1 takes
    // them now, before the cluster barrier
    const int rb = k.rank == 0 ? r1 : r0;
    const int lane1 = threadIdx.x - 32;
    if (warp == 1 && lane1 < A && rb < k.T && ((rb - 1) & 1) == q)
      k.xch[18 + lane1] =
          (int)philox((uint32_t)(rb - 1), t, (uint32_t)lane1, (k.ent << 8) | TAG_SWAP, k.k0, k.k1).x;
  }
  PROF_MARK(12, pt);
  if (threadIdx.x < 32) {
    const int lane = threadIdx.x;
    if (lane < 16) k.swm[lane] = 0;
    __syncwarp();
    const int first = r0 + q;                          // r0 is even
    const int np = r1 - 1 > first ? (r1 - first) / 2 : 0;   // pairs (r, r + 1), r + 1 < r1
    int any = 0;
    // joint mode (Algorithm S2 read literally): lane idx decides pair idx
    // for all labels at once, with the summed energy difference
    const int nd = k.joint ? np : np * A;
    for (int idx = lane; idx < nd; idx += 32) {
      const int r = first + 2 * (k.joint ? idx : idx >> lA2), al = k.joint ? 0 : idx & (A - 1);
      // the draw first: it does not depend on the energies
      const uint32_t x0 = philox((uint32_t)r, t, (uint32_t)al, (k.ent << 8) | TAG_SWAP, k.k0, k.k1).x;
      const int bA = al * lb + r - r0, bB = bA + 1;
      int dE = k.E[bB] - k.E[bA];
      if (k.joint)
        for (int l = 1; l < A; ++l) dE += k.E[l * lb + r - r0 + 1] - k.E[l * lb + r - r0];
      const bool acc = dE >= 0 || x0 < swap_table(r, dE);
      for (int l = al; l < (k.joint ? A : al + 1); ++l) {
        const int lA = l * lb + r - r0, lB = lA + 1;
        k.satt[r * A + l] += 1;
        if (acc) {
          k.sacc[r * A + l] += 1;
          const int eA = k.E[lA];
          k.E[lA] = k.E[lB];
          k.E[lB] = eA;
          if ((lA & 7) != 7) atomicOr(&k.swm[lA >> 3], 1u << (4 * (lA & 7)));
          else k.swm[8 + (lA >> 3)] = 1u;
          any = 1;
        }
      }
    }
    any = __any_sync(0xFFFFFFFFu, any);
    if (lane == 0) k.m32[5] = any;
  }
  PROF_MARK(13, pt);
  uint32_t bmask = 0;
  if (SPLIT) {
    cooperative_groups::this_cluster().sync();   // the peer's energies and spins have landed
    // the pair (rb - 1, rb) across the two CTAs, if this attempt's parity
    const int rb = k.rank == 0 ? r1 : r0;
    if (threadIdx.x < 32) {
      // a lane per label
      const int l = threadIdx.x, rb_own = k.rank == 0 ? r1 - 1 : r0;
      const bool on = l < A && rb < k.T && ((rb - 1) & 1) == q;
      int e_lo = 0, e_hi = 0;               // energies at rb - 1 (rank 0's) and rb (rank 1's)
      if (on) {
        const int own = k.E[l * lb + rb_own - r0], peer = k.xch[4 * par + l];
        e_lo = k.rank == 0 ? own : peer;
        e_hi = k.rank == 0 ? peer : own;
      }
      const int sum = (int)__reduce_add_sync(0xFFFFFFFFu, (unsigned)(e_hi - e_lo));
      bool acc = false;
      if (on) {
        const int dE = k.joint ? sum : e_hi - e_lo;
        // the draw taken by warp 1 before the barrier
        acc = dE >= 0 || (uint32_t)k.xch[18 + (k.joint ? 0 : l)] < swap_table(rb - 1, dE);
        if (k.rank == 0) {   // counted once, by rank 0
          k.satt[(rb - 1) * A + l] += 1;
          if (acc) k.sacc[(rb - 1) * A + l] += 1;
        }
        if (acc) k.E[l * lb + rb_own - r0] = k.rank == 0 ? e_hi : e_lo;
      }
      const uint32_t accm = __ballot_sync(0xFFFFFFFFu, acc);
      if (l == 0) k.xch[8] = (int)accm;
    }
    __syncthreads();
    bmask = (uint32_t)k.xch[8];
  } else {
    __syncthreads();
  }
  PROF_MARK(14, pt);
  // the measurement before this step may have found a new best state; its
  // words have not moved yet
  if (k.m32[1]) {
    copy_best();
    __syncthreads();
  }
  if (!k.m32[5] && !bmask) return;
  // colour 0 is rewritten by the next sweep without being read (a Gibbs
  // update depends on the neighbours only), so only colour 1 moves now; the
  // kernel applies the last attempt's swaps to colour 0 before it stores
  swap_words(1, bmask, par);
  PROF_MARK(15, pt);
}

// MODE (pc::APT_MODE_*), SPLIT (a cluster of two CTAs per problem), CSEED (the
// cluster-seed rule) and PARTS (thread chunks below a quad) are template
// arguments, so that each kernel carries only its own code (the launcher picks
// the instantiation from the arguments).
template <int MODE, bool SPLIT, bool CSEED, bool PARTS>
__global__ void __launch_bounds__(512) apt_kernel(const __grid_constant__ AptArgs a) {
  uint32_t *const smem = dyn_smem();
  Ctl &k = ctl();
  const int cta = blockIdx.x;
  const int p = a.cta_prob[cta];
  const AptProbDev &P = a.prob[p];
  const int N = P.N, H = N >> 1;
  const int64_t s0 = a.ctr[0], t0 = a.ctr[1];
  const bool icm = MODE == pc::APT_MODE_APT && a.icm;
  const int rank = SPLIT ? (int)cooperative_groups::this_cluster().block_rank() : 0;
  if (threadIdx.x == 0) {
    k.Lx = P.Lx;
    k.Ly = P.Ly;
    k.Lz = P.Lz;
    k.N = N;
    k.H = H;
    k.hx = P.Lx >> 1;
    k.mhx = P.mhx;
    k.mLy = P.mLy;
    k.mLy2 = P.mLy2;
    k.nbonds = P.nbonds;
    k.nreal = P.nreal;
    k.open = P.open;
    k.T = P.T;
    k.Tp = P.Tp;
    k.A = P.A;
    k.B = P.B;
    k.ent = P.ent;
    k.g0 = a.cta_g0[cta];
    k.Gc = a.cta_gc[cta];
    k.Bc = min(8 * k.Gc, P.B - 8 * k.g0);
    k.rank = rank;
    if (MODE == pc::APT_MODE_APT || MODE == pc::APT_MODE_ENERGY) {
      k.Gu = k.Gc / k.A;   // A is 1, 2 or 4
      k.Glp = k.Tp >> 3;
    } else {
      k.Gu = k.Gc;
      k.Glp = (k.B + 7) >> 3;
    }
    k.nq = quads_of(k.Gc);
    k.gq = quad_groups(k.Gc);
    k.lw = quad_shift(k.Gc);
    k.nch = PARTS ? a.cta_nch[cta] : min(a.cta_nch[cta], k.nq);
    k.tpc = blockDim.x / k.nch;
    k.parts = max(1, k.nch / k.nq);
    k.k0 = a.k0;
    k.k1 = a.k1;
    k.tag_main = a.tag_main;
    k.tag_ref = a.tag_ref;
    k.joint = a.joint_swap;
    k.icm_big = a.icm_big;
    k.swt_len = MODE == pc::APT_MODE_APT ? a.swt_len : 0;
    k.swapidx = a.swapidx + P.swapidx_off;
    k.swaptab = a.swaptab;
    k.best_spins = (rank ? a.best_spins2 : a.best_spins) + P.best_off;
    // carve shared memory; both CTAs of a split problem alike (for the
    // larger of the two parts), so that distributed-shared-memory addresses
    // correspond
    const int Gm = SPLIT ? k.A * max(k.Gu, k.Glp - k.Gu) : k.Gc, Gp = quads_of(Gm) * quad_groups(Gm);
    int o = (int)(sizeof(Ctl) / 4);
    k.oThr = o;    o += 128 * Gp;
    // each group's block of thh starts on a 256-byte boundary of the shared window
    o += (int)((256u - (((uint32_t)__cvta_generic_to_shared(smem) + 4u * (uint32_t)o) & 255u)) & 255u) >> 2;
    k.oThh = o;    o += 64 * Gp;
    k.oHist = o;   o += MODE == pc::APT_MODE_PILOT ? (P.T * a.n_bins + 3) & ~3 : 0;
    k.oStage = o;  o += SPLIT ? 512 : 0;
    k.oSwt = o;    o += (max(P.T - 1, 0) * k.swt_len + 3) & ~3;
    k.oS = o;      o += site_words(Gm) * N;
    k.oV = o;      o += icm ? icm_words(N) : 0;
    k.oJn = o;     o += N;
    k.oPos = o;
    k.m64[0] = a.best_E[p];
    k.m64[1] = a.best_sweep[p];
    k.m64[2] = a.hit_sweep[p];
    k.m64[3] = a.target[p];
    k.m32[0] = a.best_buf[p];
    for (int i = 1; i < 8; ++i) k.m32[i] = 0;
    // local group u is global group gmap[u]
    for (int g = 0; g < 8; ++g) k.gmap[g] = (g / max(k.Gu, 1)) * k.Glp + k.g0 + g % max(k.Gu, 1);
  }
  __syncthreads();
  // load state
  {
    uint32_t *S = smem + k.oS, *jn = smem + k.oJn, *thr = smem + k.oThr;
    uint16_t *thh = reinterpret_cast<uint16_t *>(smem + k.oThh);
    for (int i = threadIdx.x; i < k.Gc * N; i += blockDim.x) {
      const int g = i / N, kk = i - g * N;
      spin_word(k, S, g, kk) = a.spins[P.spin_off + (size_t)k.gmap[g] * N + kk];
    }
    for (int i = threadIdx.x; i < N; i += blockDim.x) {
      const int c = i >= H ? 1 : 0;
      jn[i] = (uint32_t)a.jneg[P.jneg_off + i] | place_bits(k, c, i - c * H);
      if (icm) reinterpret_cast<uint16_t *>(smem + k.oPos)[i] = (uint16_t)block_pos(k, i);
    }
    if (icm && threadIdx.x < 8) smem[k.oV + threadIdx.x * kBlk + kBlk - 1] = 0u;
    for (int b = threadIdx.x; b < 64; b += blockDim.x) {
      k.Eacc[b] = 0;
      if (b >= 8 * k.Gc) continue;
      const int gb = 8 * k.gmap[b >> 3] + (b & 7);
      const int tb = (b < k.Bc) ? a.temp_of[P.buf_off + gb] : 0;
      k.temp_of[b] = tb;
      k.E[b] = (b < k.Bc) ? a.E[P.buf_off + gb] : 0;
      k.sum1[b] = 0;
      k.sum2[b] = 0;
      for (int e = 0; e < 16; ++e) {
        const uint32_t th = a.pbit[P.pbit_off + 16 * tb + e];
        thr[16 * b + e] = th;
        thh[16 * b + e] = (uint16_t)(th >> 16);
      }
    }
    for (int i = threadIdx.x; i < 128; i += blockDim.x) {
      k.satt[i] = 0;
      k.sacc[i] = 0;
    }
    if (threadIdx.x < 24) k.xch[threadIdx.x] = 0;
    for (int i = threadIdx.x; i < (k.T - 1) * k.swt_len; i += blockDim.x) {
      const int r = i / k.swt_len, kk = i - r * k.swt_len;
      const uint32_t off = k.swapidx[2 * r], len = k.swapidx[2 * r + 1];
      smem[k.oSwt + i] = ((uint32_t)kk < len) ? a.swaptab[off + kk] : 0u;
    }
    if (MODE == pc::APT_MODE_PILOT)
      for (int i = threadIdx.x; i < k.T * a.n_bins; i += blockDim.x) smem[k.oHist + i] = 0u;
  }
  // a split problem's first swap step writes the peer's exchange words and
  // stage: only once the peer runs and has set them up
  if (SPLIT && MODE == pc::APT_MODE_APT)
    cooperative_groups::this_cluster().sync();
  else
    __syncthreads();

  if (MODE == pc::APT_MODE_ENERGY) {
    colour<false, true, PARTS>(1, 0u);
    __syncthreads();
    for (int b = threadIdx.x; b < 8 * k.Gc; b += blockDim.x) k.E[b] = k.nbonds - 2 * k.Eacc[b];
    __syncthreads();
  } else if (MODE == pc::APT_MODE_APT) {
#if PC_APT_PROFILE
    long long pt = clock64();
#endif
    const int spp = a.spp;
    for (int it = 0; it < a.n_iter; ++it) {
      const uint32_t t = (uint32_t)(t0 + it);
      const uint32_t sf = (uint32_t)(s0 + (int64_t)it * spp);
      for (int qq = 0; qq < spp; ++qq) {
        colour<true, false, PARTS>(0, sf + (uint32_t)qq);
        __syncthreads();
        PROF_MARK(0, pt);
        // energies are read only after the attempt's last sweep
        if (qq + 1 < spp)
          colour<true, false, PARTS>(1, sf + (uint32_t)qq);
        else
          colour<true, true, PARTS>(1, sf + (uint32_t)qq);
        __syncthreads();
        PROF_MARK(1, pt);
      }
      const int64_t sweeps = s0 + (int64_t)(it + 1) * spp;
      // warp 0 measures while the others go on to the next barrier
      if (threadIdx.x < 32) measure(0, sweeps);
      if (icm) {
        icm_all<CSEED>(t);
#if PC_APT_PROFILE
        pt = clock64();
#endif
        if (k.A == 2)
          label0_energies();
        else
          colour<false, true, PARTS>(1, 0u);   // the pairs change with the temperature
        __syncthreads();
        PROF_MARK(9, pt);
        if (threadIdx.x < 32) {
          // a flag of the first measurement stands until the copy is made there
          measure(k.A == 2, sweeps);
        }
      }
      swap_step<SPLIT>(t);
      __syncthreads();
      PROF_MARK(3, pt);
    }
  } else {
    // ladder and pilot chains: energies from window_from on only
    for (int it = 0; it < a.n_iter; ++it) {
      const uint32_t s = (uint32_t)(s0 + it);
      colour<true, false, PARTS>(0, s);
      __syncthreads();
      const bool count = MODE == pc::APT_MODE_LADDER ? (int64_t)it >= a.window_from : (int64_t)s >= a.window_from;
      if (!count) {
        colour<true, false, PARTS>(1, s);
        __syncthreads();
        continue;
      }
      colour<true, true, PARTS>(1, s);
      __syncthreads();
      // the next energy pass is two barriers away
      for (int b = threadIdx.x; b < 8 * k.Gc; b += blockDim.x) {
        const int64_t e = k.nbonds - 2 * k.Eacc[b];
        k.Eacc[b] = 0;
        k.E[b] = (int32_t)e;
        if (b >= k.Bc) continue;
        if (MODE == pc::APT_MODE_LADDER) {
          k.sum1[b] += e;
          k.sum2[b] += e * e;
        } else {
          const int64_t span = 3 * (int64_t)N;
          const int64_t num = (e + span) * a.n_bins;
          int64_t bin = num < 0 ? 0 : num / span;
          if (bin > a.n_bins - 1) bin = a.n_bins - 1;
          atomicAdd(reinterpret_cast<int *>(smem + k.oHist) + k.temp_of[b] * a.n_bins + (int)bin, 1);
        }
      }
    }
  }

  // every thread's last histogram / sum update lands before the write-back,
  // and colour 0 takes the last attempt's swaps
  __syncthreads();
  if (MODE == pc::APT_MODE_APT && a.n_iter > 0) {
    const int lpar = (int)((t0 + a.n_iter - 1) & 1);   // parity of the last attempt
    uint32_t bmask = 0;
    if (SPLIT) {
      // colour-0 spins of the last boundary swap, and this rank's best
      // candidate, to the peer (the other parity's buffers are free)
      push_boundary(0, lpar ^ 1, 0);
      if (threadIdx.x == 0) {
        int *px = cooperative_groups::this_cluster().map_shared_rank(k.xch, k.rank ^ 1);
        px[12] = (int)k.m64[0];
        px[13] = k.m32[0];
        px[14] = (int)(uint32_t)((uint64_t)k.m64[1] & 0xFFFFFFFFu);
        px[15] = (int)(uint32_t)((uint64_t)k.m64[1] >> 32);
        px[16] = (int)(uint32_t)((uint64_t)k.m64[2] & 0xFFFFFFFFu);
        px[17] = (int)(uint32_t)((uint64_t)k.m64[2] >> 32);
      }
      cooperative_groups::this_cluster().sync();   // last access to the peer's memory
      if (threadIdx.x == 0) {
        const int64_t pE = k.xch[12];
        const int64_t psw = (int64_t)(((uint64_t)(uint32_t)k.xch[15] << 32) | (uint32_t)k.xch[14]);
        const int64_t phit = (int64_t)(((uint64_t)(uint32_t)k.xch[17] << 32) | (uint32_t)k.xch[16]);
        // rank 0's candidate against rank 1's: lower energy, earlier sweep,
        // then rank 0 (its slots are the lower ones)
        const int64_t E0 = k.rank == 0 ? k.m64[0] : pE, E1 = k.rank == 0 ? pE : k.m64[0];
        const int64_t S0 = k.rank == 0 ? k.m64[1] : psw, S1 = k.rank == 0 ? psw : k.m64[1];
        const bool win1 = E1 < E0 || (E1 == E0 && S1 < S0);
        int copy = 0;
        if (k.rank == 0 && win1) {
          k.m64[0] = pE;
          k.m64[1] = psw;
          k.m32[0] = k.xch[13];
        }
        if (k.rank == 1) copy = win1 && k.m64[0] == E1 && k.m64[1] == S1 && k.m64[1] >= s0;
        const int64_t h = k.m64[2];
        k.m64[2] = h < 0 ? phit : (phit < 0 ? h : min(h, phit));
        k.m32[1] = copy;
      }
      __syncthreads();
      bmask = (uint32_t)k.xch[8];
      if (k.m32[1]) {   // rank 1 found the problem's best: it moves its state
        for (int i = threadIdx.x; i < N; i += blockDim.x)
          a.best_spins[P.best_off + i] = a.best_spins2[P.best_off + i];
      }
    }
    if (k.m32[5] || bmask) {
      swap_words(0, bmask, lpar ^ 1);
      __syncthreads();
    }
  }
  // store state
  {
    uint32_t *S = smem + k.oS;
    for (int i = threadIdx.x; i < k.Gc * N; i += blockDim.x) {
      const int g = i / N, kk = i - g * N;
      a.spins[P.spin_off + (size_t)k.gmap[g] * N + kk] = spin_word(k, S, g, kk);
    }
  }
  for (int b = threadIdx.x; b < k.Bc; b += blockDim.x) {
    const int gb = 8 * k.gmap[b >> 3] + (b & 7);
    a.E[P.buf_off + gb] = k.E[b];
    if (MODE == pc::APT_MODE_LADDER) {
      a.sum1[P.buf_off + gb] = k.sum1[b];
      a.sum2[P.buf_off + gb] = k.sum2[b];
    }
  }
  if (MODE == pc::APT_MODE_PILOT)
    for (int i = threadIdx.x; i < k.T * a.n_bins; i += blockDim.x)
      atomicAdd(reinterpret_cast<unsigned long long *>(&a.hist[P.hist_off + i]), (unsigned long long)smem[k.oHist + i]);
  if (MODE == pc::APT_MODE_APT) {
    // statistics: both CTAs of a split problem add theirs
    unsigned long long *st = reinterpret_cast<unsigned long long *>(a.stats + P.stat_off);
    const int npair = (k.T - 1) * k.A;
    for (int i = threadIdx.x; i < npair; i += blockDim.x) {
      if (k.satt[i]) atomicAdd(st + i, (unsigned long long)k.satt[i]);
      if (k.sacc[i]) atomicAdd(st + npair + i, (unsigned long long)k.sacc[i]);
    }
    if (threadIdx.x < 3 && k.m32[2 + threadIdx.x])
      atomicAdd(st + 2 * npair + threadIdx.x, (unsigned long long)k.m32[2 + threadIdx.x]);
    if (threadIdx.x == 0 && k.rank == 0) {
      a.best_E[p] = k.m64[0];
      a.best_sweep[p] = k.m64[1];
      a.hit_sweep[p] = k.m64[2];
      a.best_buf[p] = k.m32[0];
    }
  }
}

__global__ void apt_advance_kernel(int64_t *ctr, int64_t sweeps, int64_t swaps) {
  ctr[0] += sweeps;
  ctr[1] += swaps;
}

// Random initial state of every replica: +1 iff the init half-word < 2^15.
__global__ void apt_init_kernel(const AptArgs a, int n_prob) {
  const int p = blockIdx.y;
  if (p >= n_prob) return;
  const AptProbDev &P = a.prob[p];
  const int N = P.N, H = N >> 1;
  const int G = (P.B + 7) >> 3;
  for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < G * N; idx += gridDim.x * blockDim.x) {
    const int g = idx / N, rem = idx - g * N, c = rem / H, j = rem - c * H;
    const uint4 x = philox((uint32_t)j, 0u, ((uint32_t)c << 16) | (uint32_t)g,
                           (P.ent << 8) | a.tag_init, a.k0, a.k1);
    uint32_t w = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) w |= (half_lo(x, i) < 0x8000u) ? (1u << (4 * i)) : 0u;
    a.spins[P.spin_off + idx] = w;
  }
}

}  // namespace

namespace pc {

size_t apt_smem_bytes(int N, int Gc, int mode, int icm, int T, int n_bins, int swt_len) {
  const int Gp = quads_of(Gc) * quad_groups(Gc);
  size_t words = sizeof(Ctl) / 4 + 192 * (size_t)Gp + 64 + 512;   // thr, thh and its alignment, stage
  if (mode == APT_MODE_PILOT) words += ((size_t)T * n_bins + 3) & ~(size_t)3;
  if (mode == APT_MODE_APT) words += ((size_t)(T > 1 ? T - 1 : 0) * swt_len + 3) & ~(size_t)3;   // staged swap tables
  words += (size_t)site_words(Gc) * N;
  if (mode == APT_MODE_APT && icm) words += (size_t)icm_words(N) + (size_t)(N + 1) / 2;   // and the sites' places
  return (words + (size_t)N) * 4;
}

template <int MODE, bool CSEED, bool PARTS>
int apt_launch_mode(const AptArgs &a, int n_cta, int tpb, size_t smem, cudaStream_t st) {
  if (!a.split) {
    apt_kernel<MODE, false, CSEED, PARTS><<<n_cta, tpb, smem, st>>>(a);
  } else {
    // split problems: consecutive CTA pairs form one cluster
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)n_cta);
    cfg.blockDim = dim3((unsigned)tpb);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (a.prio) {   // a mixed placement starts its clusters (the largest problems) first
      attr[1].id = cudaLaunchAttributePriority;
      attr[1].val.priority = a.prio;
      cfg.numAttrs = 2;
    }
    PC_CUDA_TRY(cudaLaunchKernelEx(&cfg, apt_kernel<MODE, true, CSEED, PARTS>, a));
  }
  PC_CUDA_TRY(cudaGetLastError());
  return PC_OK;
}

int apt_launch(const AptArgs &a, int n_cta, int tpb, size_t smem, cudaStream_t st) {
  if (n_cta <= 0) return PC_OK;
  // raise the dynamic shared-memory limit of every mode's kernel once per
  // device (never inside a stream capture: the first launch on a device
  // happens at load time)
  static size_t set_for[64] = {0};
  int dev = 0;
  PC_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return fail(PC_EINVAL, "device index out of range");
  if (smem > set_for[dev]) {
    const void *const kernels[] = {
        (const void *)apt_kernel<pc::APT_MODE_APT, false, false, false>, (const void *)apt_kernel<pc::APT_MODE_APT, true, false, false>,
        (const void *)apt_kernel<pc::APT_MODE_APT, false, true, false>,  (const void *)apt_kernel<pc::APT_MODE_APT, true, true, false>,
        (const void *)apt_kernel<pc::APT_MODE_APT, false, false, true>,  (const void *)apt_kernel<pc::APT_MODE_APT, true, false, true>,
        (const void *)apt_kernel<pc::APT_MODE_APT, false, true, true>,   (const void *)apt_kernel<pc::APT_MODE_APT, true, true, true>,
        (const void *)apt_kernel<pc::APT_MODE_LADDER, false, false, false>, (const void *)apt_kernel<pc::APT_MODE_LADDER, true, false, false>,
        (const void *)apt_kernel<pc::APT_MODE_PILOT, false, false, false>,  (const void *)apt_kernel<pc::APT_MODE_PILOT, true, false, false>,
        (const void *)apt_kernel<pc::APT_MODE_ENERGY, false, false, false>, (const void *)apt_kernel<pc::APT_MODE_ENERGY, true, false, false>};
    for (const void *k : kernels)
      PC_CUDA_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    set_for[dev] = smem;
  }
  switch (a.mode) {
    case pc::APT_MODE_APT:
      // the cluster-seed ICM rule and chunks below a quad have instantiations
      // of their own, so the default's code is compiled without them
      if (a.parts)
        return a.icm_seed ? apt_launch_mode<pc::APT_MODE_APT, true, true>(a, n_cta, tpb, smem, st)
                          : apt_launch_mode<pc::APT_MODE_APT, false, true>(a, n_cta, tpb, smem, st);
      return a.icm_seed ? apt_launch_mode<pc::APT_MODE_APT, true, false>(a, n_cta, tpb, smem, st)
                        : apt_launch_mode<pc::APT_MODE_APT, false, false>(a, n_cta, tpb, smem, st);
    case pc::APT_MODE_LADDER: return apt_launch_mode<pc::APT_MODE_LADDER, false, false>(a, n_cta, tpb, smem, st);
    case pc::APT_MODE_PILOT: return apt_launch_mode<pc::APT_MODE_PILOT, false, false>(a, n_cta, tpb, smem, st);
    case pc::APT_MODE_ENERGY: return apt_launch_mode<pc::APT_MODE_ENERGY, false, false>(a, n_cta, tpb, smem, st);
    default: return fail(PC_EINVAL, "unknown kernel mode");
  }
}

#if PC_APT_PROFILE
extern "C" int pc_apt_profile_read(unsigned long long *out, int reset) {
  PC_CUDA_TRY(cudaMemcpyFromSymbol(out, g_apt_prof, sizeof(unsigned long long) * 32));
  if (reset) {
    unsigned long long z[32] = {0};
    PC_CUDA_TRY(cudaMemcpyToSymbol(g_apt_prof, z, sizeof(z)));
  }
  return PC_OK;
}
#endif

int apt_advance_launch(int64_t *ctr, int64_t sweeps, int64_t swaps, cudaStream_t st) {
  apt_advance_kernel<<<1, 1, 0, st>>>(ctr, sweeps, swaps);
  PC_CUDA_TRY(cudaGetLastError());
  return PC_OK;
}

int apt_init_launch(const AptArgs &a, int n_prob, int max_words, cudaStream_t st) {
  if (n_prob <= 0) return PC_OK;
  const int tpb = 256;
  int bx = (max_words + tpb - 1) / tpb;
  if (bx > 64) bx = 64;
  if (bx < 1) bx = 1;
  dim3 grid((unsigned)bx, (unsigned)n_prob);
  apt_init_kernel<<<grid, tpb, 0, st>>>(a, n_prob);
  PC_CUDA_TRY(cudaGetLastError());
  return PC_OK;
}

}  // namespace pc
