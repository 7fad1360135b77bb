// Discrete-time simulated quantum annealing (Suzuki-Trotter mapping, Eq. S.3;
// Algorithm S1) as one persistent CTA per independent run.
//
// Layout.  A run is the (d+1)-dimensional lattice of P slices of the 3D
// lattice.  Its 4D checkerboard colour is c = (x + y + z + k) & 1, so at a
// 3D site s of parity q the slices of colour c are k = 2m + (c ^ q).  Eight
// consecutive m of one (colour, site) share a 32-bit word, one spin per
// nibble (bit 0 = spin +1), block b = m >> 3.  Shared memory holds
// W[c][s][b] for the whole run (N * P / 2 bytes; the NB words of a site are
// contiguous, so they move as one vector access).  With this packing
//  - the six spatial neighbours of a word are the words of the other colour
//    at the neighbouring sites with the SAME block: nibble-aligned, and the
//    coupling J (common to all slices) is one mask per direction;
//  - the two imaginary-time neighbours are the other colour's word at the
//    same site and that word shifted by one nibble (carry from block b +- 1).
// So one word yields 8 nibble-packed satisfied-bond counts (0..6) and 8
// time-neighbour counts (0..2) with a handful of 32-bit ops, and one
// Philox4x32-10 call supplies the 8 16-bit uniforms.
#include <cuda_runtime.h>

#include <mutex>

#include "device.cuh"
#include "internal.h"

// Threads per CTA of the anneal kernel (build-time knob).
#ifndef PC_SQA_TPB
#define PC_SQA_TPB 512
#endif

namespace {
using namespace pcdev;

// Site coordinates of a 3D site index.
struct Site {
  int s, x, y, z, q;
  uint32_t jb;
};

__device__ __forceinline__ Site site_of(const pc::SqaArgs &a, int s, const uint16_t *jn) {
  Site t;
  t.s = s;
  const int r = (int)fdiv((uint32_t)s, a.mLx);   // s / Lx
  t.x = s - r * a.Lx;
  t.z = (int)fdiv((uint32_t)r, a.mLy);           // r / Ly
  t.y = r - t.z * a.Ly;
  t.q = (t.x + t.y + t.z) & 1;
  t.jb = jn[s];
  return t;
}

// Neighbour of site t along direction d (0:+x 1:-x 2:+y 3:-y 4:+z 5:-z),
// periodic boundaries.
__device__ __forceinline__ int neighbour(const pc::SqaArgs &a, const Site &t, int d) {
  const int LxLy = a.Lx * a.Ly;
  switch (d) {
    case 0: return (t.x + 1 == a.Lx) ? t.s - (a.Lx - 1) : t.s + 1;
    case 1: return (t.x == 0) ? t.s + (a.Lx - 1) : t.s - 1;
    case 2: return (t.y + 1 == a.Ly) ? t.s - (a.Ly - 1) * a.Lx : t.s + a.Lx;
    case 3: return (t.y == 0) ? t.s + (a.Ly - 1) * a.Lx : t.s - a.Lx;
    case 4: return (t.z + 1 == a.Lz) ? t.s - (a.Lz - 1) * LxLy : t.s + LxLy;
    default: return (t.z == 0) ? t.s + (a.Lz - 1) * LxLy : t.s - LxLy;
  }
}

// Nibble-packed counts, per block, of satisfied terms J_d s_nbr = +1 over
// the spatial bonds present (Eq. synapse with I = 2C - deg).  XOR with the
// all-nibbles mask turns a neighbour spin into J_d s_nbr for J_d = -1.
template <int NB>
__device__ __forceinline__ void spatial_counts(const pc::SqaArgs &a, const uint32_t *Wo,
                                               const Site &t, uint32_t (&C)[NB]) {
#pragma unroll
  for (int b = 0; b < NB; ++b) C[b] = 0;
#pragma unroll
  for (int d = 0; d < 6; ++d) {
    if ((t.jb >> (8 + d)) & 1u) continue;   // absent bond (open axis)
    const int n = neighbour(a, t, d);
    const uint32_t m = nib_mask((t.jb >> d) & 1u);
#pragma unroll
    for (int b = 0; b < NB; ++b) C[b] += Wo[(size_t)n * NB + b] ^ m;
  }
}

// Per-site constants of the sweep: neighbour indices and the coupling
// signs.  With s_nbr in {0,1} per nibble, J s_nbr "satisfied" is s_nbr for
// J = +1 and 1 - s_nbr for J = -1, so the packed count of satisfied terms is
// C = K + sum_d eps_d W_d with eps_d = +-1 and K = 0x11111111 * #(J = -1):
// six multiply-adds per word.
struct SiteK {
  int nb[6];
  int eps[6];        // +-1, 0 for an absent bond
  uint32_t K;
  uint32_t kb;       // absent bonds k: 4k in every byte (threshold index I + 6 = 2C + k)
  int q;
};

// The same in 20 bytes per site of shared memory, for lattices with more
// sites than threads: v = the neighbours as 16-bit pairs and eps_0 .. eps_3
// as bytes, u = eps_4, eps_5, #(J = -1) + 128 q, 4k.
struct SitePack {
  uint4 v;
  uint32_t u;
};

__device__ __forceinline__ SitePack site_pack(const pc::SqaArgs &a, int s, const uint16_t *jn) {
  const Site t = site_of(a, s, jn);
  uint32_t nb[6], eps[6], nneg = 0, nmiss = 0;
#pragma unroll
  for (int d = 0; d < 6; ++d) {
    nb[d] = (uint32_t)neighbour(a, t, d);
    const uint32_t neg = (t.jb >> d) & 1u, miss = (t.jb >> (8 + d)) & 1u;
    eps[d] = miss ? 0u : (neg ? 0xFFu : 1u);
    nneg += miss ? 0u : neg;
    nmiss += miss;
  }
  SitePack k;
  k.v = make_uint4(nb[0] | (nb[1] << 16), nb[2] | (nb[3] << 16), nb[4] | (nb[5] << 16),
                   eps[0] | (eps[1] << 8) | (eps[2] << 16) | (eps[3] << 24));
  k.u = eps[4] | (eps[5] << 8) | ((nneg + 128u * (uint32_t)t.q) << 16) | (nmiss << 26);
  return k;
}

// Byte B of x as a signed value (prmt's sign mode spreads its top bit over
// the upper bytes).
template <int B>
__device__ __forceinline__ int signed_byte(uint32_t x) {
  uint32_t r;
  asm("prmt.b32 %0, %1, 0, %2;" : "=r"(r) : "r"(x), "n"(0x8880 + 0x1111 * B));
  return (int)r;
}

__device__ __forceinline__ SiteK site_unpack(const SitePack &p) {
  SiteK k;
  k.nb[0] = (int)(p.v.x & 0xFFFFu); k.nb[1] = (int)(p.v.x >> 16);
  k.nb[2] = (int)(p.v.y & 0xFFFFu); k.nb[3] = (int)(p.v.y >> 16);
  k.nb[4] = (int)(p.v.z & 0xFFFFu); k.nb[5] = (int)(p.v.z >> 16);
  k.eps[0] = signed_byte<0>(p.v.w); k.eps[1] = signed_byte<1>(p.v.w);
  k.eps[2] = signed_byte<2>(p.v.w); k.eps[3] = signed_byte<3>(p.v.w);
  k.eps[4] = signed_byte<0>(p.u);   k.eps[5] = signed_byte<1>(p.u);
  k.K = 0x11111111u * ((p.u >> 16) & 7u);
  k.kb = __byte_perm(p.u, 0u, 0x3333u);
  k.q = (int)((p.u >> 23) & 1u);
  return k;
}

// Threshold rows of two sweeps (the current one and the next, which arrives
// by asynchronous copy meanwhile), entry I + 6 + kRowStep m for in-slice field
// I = -6..6 and time count m = 0..2: 23 words per step of m put the 21 entries
// of a lattice without absent bonds (even I) into 21 banks.  Each row starts
// on a 256-byte boundary of the shared window, so that a byte of a packed
// offset word and the row's address make an entry's address in one byte
// permute.  The copy replaces a load, a wait and two stores by two warps at
// the start of each sweep (512 spins, 64 slices: 52.6 -> 51.9 ms with the
// kernels by HOIST).
constexpr uint32_t kRowStep = 23;
__shared__ __align__(256) uint32_t s_Tf[2][64];

__device__ __forceinline__ uint32_t entry_addr(uint32_t Dlo, uint32_t Dhi, uint32_t tb, int i) {
  return __byte_perm((i & 1) ? Dhi : Dlo, tb, 0x7650u + (uint32_t)(i >> 1));
}

// Eq. neuron for the 8 nibbles of one word.  Byte k of Dlo / Dhi is the
// byte offset of the threshold of nibble 2k / 2k+1 in the row at tb.  The
// main half v decides against the top half t of the threshold: d = v - t is
// negative iff v < t, and d = 0 is a tie, which the main half cannot decide.
__device__ __forceinline__ uint32_t decide_word(const uint4 &x, uint32_t Dlo, uint32_t Dhi, uint32_t tb, bool &tie) {
  uint32_t w = 0;
  uint32_t tp = 1u;   // product of the differences (mod 2^32): 0 when some half equals its threshold
#pragma unroll
  for (int i = 7; i >= 0; --i) {
    uint32_t th;
    asm("ld.shared.u16 %0, [%1+2];" : "=r"(th) : "r"(entry_addr(Dlo, Dhi, tb, i)));
    const uint32_t d = half_lo(x, i) - th;   // both below 2^16: bit 31 set iff v < th
    // the top 4 bits of d enter w as its new nibble 0, so after the loop
    // bit 3 of nibble i is the sign of half i's difference
    w = __funnelshift_l(d, w, 4);
    tp *= d;
  }
  // a zero product flags a tie; a product that merely wraps to 0 only sends
  // the word through settle_ties, which rechecks every half exactly
  tie |= (tp == 0);
  return (w >> 3) & 0x11111111u;
}

__device__ __noinline__ uint32_t settle_ties(uint32_t w, uint4 x, uint4 y, uint32_t Dlo, uint32_t Dhi, uint32_t tb) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    uint32_t t;
    asm("ld.shared.u32 %0, [%1];" : "=r"(t) : "r"(entry_addr(Dlo, Dhi, tb, i)));
    const uint32_t v = half_hi(x, i);
    if (v == (t & 0xFFFF0000u)) {
      const uint32_t u = v | half_lo(y, i);
      w = (u < t) ? (w | (1u << (4 * i))) : (w & ~(1u << (4 * i)));
    }
  }
  return w;
}

// Starts the asynchronous copy of a threshold row into shared memory.
__device__ __forceinline__ void fetch_row(const uint32_t *row, uint32_t *dst) {
  for (uint32_t e = threadIdx.x; e < 39u; e += blockDim.x) {   // small runs have fewer threads than entries
    const uint32_t d = e + (kRowStep - 13u) * ((e >= 13u ? 1u : 0u) + (e >= 26u ? 1u : 0u));
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst + d)),
                 "l"(row + e) : "memory");
  }
}
__device__ __forceinline__ void rows_landed() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// NB consecutive words as one vector access (NB = 1, 2, 4, 8; else scalar).
template <int NB>
__device__ __forceinline__ void load_words(const uint32_t *p, uint32_t (&v)[NB]) {
  if constexpr (NB % 4 == 0) {
#pragma unroll
    for (int q = 0; q < NB; q += 4) {
      const uint4 t = *reinterpret_cast<const uint4 *>(p + q);
      v[q] = t.x; v[q + 1] = t.y; v[q + 2] = t.z; v[q + 3] = t.w;
    }
  } else if constexpr (NB % 2 == 0) {
#pragma unroll
    for (int q = 0; q < NB; q += 2) {
      const uint2 t = *reinterpret_cast<const uint2 *>(p + q);
      v[q] = t.x; v[q + 1] = t.y;
    }
  } else {
#pragma unroll
    for (int q = 0; q < NB; ++q) v[q] = p[q];
  }
}
template <int NB>
__device__ __forceinline__ void store_words(uint32_t *p, const uint32_t (&v)[NB]) {
  if constexpr (NB % 4 == 0) {
#pragma unroll
    for (int q = 0; q < NB; q += 4)
      *reinterpret_cast<uint4 *>(p + q) = make_uint4(v[q], v[q + 1], v[q + 2], v[q + 3]);
  } else if constexpr (NB % 2 == 0) {
#pragma unroll
    for (int q = 0; q < NB; q += 2) *reinterpret_cast<uint2 *>(p + q) = make_uint2(v[q], v[q + 1]);
  } else {
#pragma unroll
    for (int q = 0; q < NB; ++q) p[q] = v[q];
  }
}

// Words b0 .. b0 + WT - 1 of one (site, colour) in one sweep.
template <int NB, int WT>
__device__ __forceinline__ void update_site(const pc::SqaArgs &a, const uint32_t *Wo, uint32_t *Wc, int s, int b0,
                                            const SiteK &k, int c, uint32_t sw, uint32_t tb, uint32_t ent) {
  const int e = c ^ k.q;   // slice parity of this word's nibbles
  const uint32_t c2 = ((uint32_t)c << 16) | (uint32_t)b0;
  uint32_t O[WT], C[WT], w[WT];
  load_words<WT>(Wo + s * NB + b0, O);
  // time neighbours k-1, k+1 of word b: the other colour's word and that
  // word shifted by one nibble (funnel shift through the adjacent block, of
  // which the parity needs the next (e = 1) or the previous one)
  uint32_t M[WT];
  {
    const int bx = e ? (b0 + WT == NB ? 0 : b0 + WT) : (b0 == 0 ? NB - 1 : b0 - 1);
    const uint32_t X = WT == NB ? (e ? O[0] : O[WT - 1]) : Wo[s * NB + bx];
    uint32_t lo = e ? O[0] : X;
    const uint32_t sh = e ? 4u : 28u;
#pragma unroll
    for (int i = 0; i < WT; ++i) {
      const uint32_t hi = e ? (i + 1 == WT ? X : O[i + 1 == WT ? i : i + 1]) : O[i];
      M[i] = O[i] + __funnelshift_r(lo, hi, sh);
      lo = hi;
    }
  }
#pragma unroll
  for (int b = 0; b < WT; ++b) C[b] = k.K;
#pragma unroll
  for (int d = 0; d < 6; ++d) {
    uint32_t Nw[WT];
    load_words<WT>(Wo + k.nb[d] * NB + b0, Nw);
#pragma unroll
    for (int b = 0; b < WT; ++b) C[b] += (uint32_t)k.eps[d] * Nw[b];
  }
  // byte offsets 4 (2C + k + 23 m): at most 232
  auto offsets = [&](int b, uint32_t &Dlo, uint32_t &Dhi) {
    const uint32_t m = M[b];
    Dlo = ((C[b] & 0x0F0F0F0Fu) << 3) + (m & 0x0F0F0F0Fu) * (4u * kRowStep) + k.kb;
    Dhi = (((C[b] >> 4) & 0x0F0F0F0Fu) << 3) + ((m >> 4) & 0x0F0F0F0Fu) * (4u * kRowStep) + k.kb;
  };
  const uint32_t c3 = (ent << 8) | TAG_SQA_SWEEP;
  auto settle = [&](int b, uint32_t Dlo, uint32_t Dhi) {
    const uint4 x = philox((uint32_t)s, sw, c2 + (uint32_t)b, c3, a.k0, a.k1);
    const uint4 y = philox((uint32_t)s, sw, c2 + (uint32_t)b, (ent << 8) | TAG_SQA_REFINE, a.k0, a.k1);
    w[b] = settle_ties(w[b], x, y, Dlo, Dhi, tb);
  };
  // up to 4 words, the decisions form one branch-free block and ties
  // (probability 2^-16 per spin) are settled after it; with more words the
  // register budget settles each word's ties at once
  uint32_t tmask = 0u;
#pragma unroll
  for (int b = 0; b < WT; ++b) {
    uint32_t Dlo, Dhi;
    offsets(b, Dlo, Dhi);
    const uint4 x = philox((uint32_t)s, sw, c2 + (uint32_t)b, c3, a.k0, a.k1);
    bool tie = false;
    w[b] = decide_word(x, Dlo, Dhi, tb, tie);
    if constexpr (WT <= 4) {
      tmask |= tie ? (1u << b) : 0u;
    } else if (tie) {
      settle(b, Dlo, Dhi);
    }
  }
  if (WT <= 4 && tmask) {
#pragma unroll
    for (int b = 0; b < WT; ++b) {
      if (!((tmask >> b) & 1u)) continue;
      uint32_t Dlo, Dhi;
      offsets(b, Dlo, Dhi);
      settle(b, Dlo, Dhi);
    }
  }
  store_words<WT>(Wc + s * NB + b0, w);
}

__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Bounded wait until *flag >= want (acquire); false after limit_ns.
__device__ __forceinline__ bool wait_at_least(const int *flag, int want, uint64_t limit_ns) {
  const uint64_t t0 = global_ns();
  for (;;) {
    int v;
    asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(flag) : "memory");
    if (v >= want) return true;
    if (global_ns() - t0 > limit_ns) return false;
    __nanosleep(256);
  }
}

// Anneal of sweeps [s0, s1) of one run.  s0 == 0 draws the random initial
// state, otherwise the state comes from the run's slot in global memory;
// s1 == S computes the final slice energies, otherwise the state goes back.
template <int NB, int WT, bool HOIST>
__device__ __forceinline__ void anneal_span(const pc::SqaArgs &a, uint32_t *W, int32_t *Eacc,
                                            const uint16_t *jn, const uint4 *sv, const uint32_t *su, const SiteK &kh,
                                            int run, int s0, int s1) {
  constexpr int parts = NB / WT;   // threads per site
  const int N = a.N, P = a.P;
  const uint32_t ent = a.run0 + (uint32_t)run;
  const int tid = threadIdx.x, nt = blockDim.x;
  uint32_t *gstate = a.state ? a.state + (size_t)run * 2 * NB * N : nullptr;
  if (s0 == 0) {
    // Algorithm S1: all spins of all slices start random (+1 iff half < 2^15)
    for (int idx = tid; idx < 2 * NB * N; idx += nt) {
      const int b = idx % NB, cs = idx / NB, s = cs % N, c = cs / N;   // W[c][s][b]
      const uint4 x = philox((uint32_t)s, 0u, ((uint32_t)c << 16) | (uint32_t)b,
                             (ent << 8) | TAG_SQA_INIT, a.k0, a.k1);
      uint32_t w = 0;
#pragma unroll
      for (int i = 0; i < 8; ++i) w |= (half_lo(x, i) < 0x8000u) ? (1u << (4 * i)) : 0u;
      W[idx] = w;
    }
  } else {
    for (int idx = tid; idx < 2 * NB * N; idx += nt) W[idx] = __ldcg(gstate + idx);
  }
  if (s0 < a.S) fetch_row(a.table + (size_t)s0 * pc::kSqaTab, s_Tf[s0 & 1]);
  rows_landed();
  const int sh = tid / parts, bh = (tid - sh * parts) * WT;   // the thread's site and first word, one item per thread
  __syncthreads();

  for (int sw = s0; sw < s1; ++sw) {
    // the transverse coupling of this sweep lives in its threshold row; the
    // next sweep's row lands in the other buffer meanwhile
    if (sw + 1 < a.S) fetch_row(a.table + (size_t)(sw + 1) * pc::kSqaTab, s_Tf[(sw + 1) & 1]);
    const uint32_t tb = (uint32_t)__cvta_generic_to_shared(s_Tf[sw & 1]);
#pragma unroll 1
    for (int c = 0; c < 2; ++c) {
      const uint32_t *Wo = W + (1 - c) * NB * N;
      uint32_t *Wc = W + c * NB * N;
      if constexpr (HOIST) {
        if (sh < N) update_site<NB, WT>(a, Wo, Wc, sh, bh, kh, c, (uint32_t)sw, tb, ent);
      } else {
        for (int it = tid; it < N * parts; it += nt) {
          const int s = it / parts, b0 = (it - s * parts) * WT;
          update_site<NB, WT>(a, Wo, Wc, s, b0, site_unpack(SitePack{sv[s], su[s]}), c, (uint32_t)sw, tb, ent);
        }
      }
      if (c) rows_landed();
      __syncthreads();
    }
  }

  if (s1 < a.S) {
    for (int idx = tid; idx < 2 * NB * N; idx += nt) __stcg(gstate + idx, W[idx]);
    return;
  }
  // Algorithm S1: classical energy of every slice (full J, no J_perp).  Each
  // bond has one endpoint with 3D parity 1, so E_k = nbonds - 2 sum_{q(s)=1} sat.
  for (int k = tid; k < P; k += nt) Eacc[k] = 0;
  __syncthreads();
  for (int c = 0; c < 2; ++c) {
    const uint32_t *Wo = W + (1 - c) * NB * N;
    const uint32_t *Wc = W + c * NB * N;
    for (int s = tid; s < N; s += nt) {
      const Site t = site_of(a, s, jn);
      if (!t.q) continue;
      const int e = c ^ 1;
      uint32_t C[NB];
      spatial_counts<NB>(a, Wo, t, C);
      const int deg = 6 - __popc((t.jb >> 8) & 0x3Fu);
      for (int b = 0; b < NB; ++b) {
        const uint32_t w = Wc[(size_t)s * NB + b];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int ci = (C[b] >> (4 * i)) & 0xF;
          const int sat = ((w >> (4 * i)) & 1u) ? ci : deg - ci;
          atomicAdd(&Eacc[2 * (8 * b + i) + e], sat);
        }
      }
    }
  }
  __syncthreads();
  for (int k = tid; k < P; k += nt) {
    Eacc[k] = a.nbonds - 2 * Eacc[k];
    a.E[(size_t)run * P + k] = Eacc[k];
  }
  __syncthreads();
  if (a.best && tid == 0) {
    int kb = 0;
    for (int k = 1; k < P; ++k)
      if (Eacc[k] < Eacc[kb]) kb = k;
    a.best[2 * run] = Eacc[kb];
    a.best[2 * run + 1] = kb;
  }
  if (a.corr) {
    // replica-direction correlation (Fig. S17): sum over sites of
    // s(s,0) s(s,k) = 2 #agree - N.  Slice k of site s is nibble (k>>1)&7 of
    // word W[(k&1) ^ q(s)][s][k>>4].  Eacc is reused once the best slice
    // has been read from it.
    __syncthreads();
    for (int k = tid; k < P; k += nt) Eacc[k] = 0;
    __syncthreads();
    for (int s = tid; s < N; s += nt) {
      const int r = (int)fdiv((uint32_t)s, a.mLx), x = s - r * a.Lx;
      const int z = (int)fdiv((uint32_t)r, a.mLy), y = r - z * a.Ly;
      const int q = (x + y + z) & 1;
      const uint32_t s0 = W[(size_t)q * NB * N + (size_t)s * NB] & 1u;   // slice 0
      const uint32_t flip = s0 ? 0u : 0x11111111u;
      for (int c = 0; c < 2; ++c)
        for (int b = 0; b < NB; ++b) {
          const uint32_t agree = (W[(size_t)c * NB * N + (size_t)s * NB + b] ^ flip) & 0x11111111u;
#pragma unroll
          for (int i = 0; i < 8; ++i)
            if ((agree >> (4 * i)) & 1u) atomicAdd(&Eacc[2 * (8 * b + i) + (c ^ q)], 1);
        }
    }
    __syncthreads();
    for (int k = tid; k < P; k += nt) a.corr[(size_t)run * P + k] = 2 * Eacc[k] - N;
    __syncthreads();
  }
  if (a.spins) {
    for (int idx = tid; idx < 2 * NB * N; idx += nt) {
      const int b = idx % NB, cs = idx / NB, s = cs % N, c = cs / N;   // W[c][s][b]
      const int r = (int)fdiv((uint32_t)s, a.mLx), x = s - r * a.Lx;
      const int z = (int)fdiv((uint32_t)r, a.mLy), y = r - z * a.Ly;
      const int e = c ^ ((x + y + z) & 1);
      const uint32_t w = W[idx];
      for (int i = 0; i < 8; ++i) {
        const int k = 2 * (8 * b + i) + e;
        a.spins[((size_t)run * P + k) * N + s] = ((w >> (4 * i)) & 1u) ? 1 : -1;
      }
    }
  }
  __syncthreads();
}

// PERSIST = false: one CTA per run, the whole schedule.  PERSIST = true: a
// persistent grid pulls (chunk, run) items in chunk-major order from a
// queue; chunk k of a run waits (bounded) until chunk k-1 of that run has
// stored its state.  Time-slicing the runs keeps every SM busy when the
// number of runs is not a multiple of the number of SMs.
template <int NB, int WT, bool HOIST, bool PERSIST>
__global__ void __launch_bounds__(PC_SQA_TPB, 1) sqa_kernel(const pc::SqaArgs a) {
  extern __shared__ __align__(16) uint32_t smem[];
  __shared__ int s_item;
  const int N = a.N, P = a.P;
  uint32_t *W = smem;                                       // [2][NB][N]
  const int tid = threadIdx.x, nt = blockDim.x;
  const int np = HOIST ? 0 : N;
  uint4 *sv = reinterpret_cast<uint4 *>(W + 2 * NB * N);    // [np] SitePack::v (2 NB N words: a multiple of 4)
  uint32_t *su = reinterpret_cast<uint32_t *>(sv + np);     // [np] SitePack::u
  int32_t *Eacc = reinterpret_cast<int32_t *>(su + np);     // [P]
  uint16_t *jn = reinterpret_cast<uint16_t *>(Eacc + P);    // [N]
  for (int i = tid; i < N; i += nt) {
    jn[i] = a.jneg[i];
    if constexpr (!HOIST) {
      const SitePack k = site_pack(a, i, jn);
      sv[i] = k.v;
      su[i] = k.u;
    }
  }
  __syncthreads();
  SiteK kh;
  if (HOIST && tid / (NB / WT) < N) kh = site_unpack(site_pack(a, tid / (NB / WT), jn));
  if constexpr (!PERSIST) {
    anneal_span<NB, WT, HOIST>(a, W, Eacc, jn, sv, su, kh, blockIdx.x, 0, a.S);
  } else {
    for (;;) {
      if (tid == 0) s_item = atomicAdd(a.queue, 1) + a.first_item;
      __syncthreads();
      const int item = s_item;
      __syncthreads();
      if (item >= a.n_items) break;
      const int chunk = item / a.R, run = item - chunk * a.R;
      const int s0 = chunk * a.K, s1 = min(a.S, s0 + a.K);
      if (chunk > 0) {
        if (tid == 0 && !wait_at_least(a.done + run, chunk, a.wait_ns)) atomicExch(a.err, 1);
        __syncthreads();
      }
      anneal_span<NB, WT, HOIST>(a, W, Eacc, jn, sv, su, kh, run, s0, s1);
      __syncthreads();
      if (tid == 0) {
        __threadfence();
        asm volatile("st.release.gpu.global.b32 [%0], %1;" ::"l"(a.done + run), "r"(chunk + 1) : "memory");
      }
    }
  }
}

__global__ void philox_kernel(const uint32_t *ctr, uint32_t *out, int64_t n, uint32_t k0,
                              uint32_t k1) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const uint4 x = philox(ctr[4 * i], ctr[4 * i + 1], ctr[4 * i + 2], ctr[4 * i + 3], k0, k1);
  out[4 * i] = x.x;
  out[4 * i + 1] = x.y;
  out[4 * i + 2] = x.z;
  out[4 * i + 3] = x.w;
}

// Words of a site that a thread updates: all of them up to 5 (and 7), else a
// half, which fits the registers as one block of decisions (128 slices, 512
// spins, 128 runs, 1000 sweeps: 8 words per thread 7.19 ms, 4 6.41 ms, 2
// 7.15 ms; 96 slices, 630 spins open: 6 words 3.67 ms, 3 3.44 ms, 2 3.52 ms).
// Twice the threads with half the words and registers (1024 x 64) ran slower
// everywhere (64 slices, 512 spins: 64.3 against 52.6 ms).
constexpr int words_per_thread(int NB) { return NB == 8 ? 4 : NB == 6 ? 3 : NB; }

template <int NB, bool HOIST>
int launch_h(const pc::SqaArgs &a, int R, int tpb, cudaStream_t st) {
  constexpr int WT = words_per_thread(NB);
  // the packed site constants only where a thread has more than one item
  const size_t smem = pc::sqa_smem_bytes(a.N, a.P) - (HOIST ? 20 * (size_t)a.N : 0);
  if (!a.state) {
    PC_CUDA_TRY(cudaFuncSetAttribute(sqa_kernel<NB, WT, HOIST, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)smem));
    sqa_kernel<NB, WT, HOIST, false><<<R, tpb, smem, st>>>(a);
  } else {
    PC_CUDA_TRY(cudaFuncSetAttribute(sqa_kernel<NB, WT, HOIST, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)smem));
    int dev = 0, sms = 0, per_sm = 0;
    PC_CUDA_TRY(cudaGetDevice(&dev));
    PC_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    PC_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, sqa_kernel<NB, WT, HOIST, true>, tpb, smem));
    if (per_sm < 1) per_sm = 1;
    sqa_kernel<NB, WT, HOIST, true><<<pc::sqa_grid(sms * per_sm, R, a.n_items), tpb, smem, st>>>(a);
  }
  PC_CUDA_TRY(cudaGetLastError());
  return PC_OK;
}

// HOIST: one item (a thread's words of one site) per thread, whose constants
// stay in registers across the sweeps; else the threads loop over the items
// and unpack the constants from shared memory (about 20 instructions; computed
// anew from the site's coordinates they were about 60 per site and colour, and
// with one kernel for both forms the registers were allotted for both).  64
// slices: 15 x 15 x 12 open, 132 runs, 1000 sweeps 19.8 -> 17.0 ms, 12^3 6.57
// -> 5.19 ms and 16^3 8.45 -> 4.57 ms (64 and 16 runs, 500 and 200 sweeps).
template <int NB>
int launch_nb(const pc::SqaArgs &a, int R, cudaStream_t st) {
  const int items = a.N * (NB / words_per_thread(NB));
  if (items <= PC_SQA_TPB) return launch_h<NB, true>(a, R, ((items + 31) / 32) * 32, st);
  return launch_h<NB, false>(a, R, PC_SQA_TPB, st);
}

}  // namespace

namespace pc {

size_t sqa_smem_bytes(int N, int P) {
  const int NB = P / 16;
  return (size_t)2 * NB * N * 4 + (size_t)P * 4 + (size_t)N * 2 + (size_t)N * 20;
}

// At most one CTA per run: the queue is in chunk-major order, so a CTA beyond
// the runs would start on a later chunk of a run still in progress, polling
// beside the CTAs that work (64 spins, 200 runs of 16 slices on 152 SMs: 11.5
// -> 10.1 ms; 304 runs of 64 slices 5.0 -> 3.7 ms) and, with several chunks between, waiting for all of them within one
// wait's limit.
int sqa_grid(int resident, int R, int n_items) {
  int grid = resident < R ? resident : R;
  return grid < n_items ? grid : n_items;
}

int sqa_launch(const SqaArgs &a, int R, cudaStream_t st) {
  switch (a.NB) {
    case 1: return launch_nb<1>(a, R, st);
    case 2: return launch_nb<2>(a, R, st);
    case 3: return launch_nb<3>(a, R, st);
    case 4: return launch_nb<4>(a, R, st);
    case 5: return launch_nb<5>(a, R, st);
    case 6: return launch_nb<6>(a, R, st);
    case 7: return launch_nb<7>(a, R, st);
    case 8: return launch_nb<8>(a, R, st);
    default: return fail(PC_EINVAL, "P must be 16 * k with 1 <= k <= 8");
  }
}

int philox_launch(const uint32_t *ctr, uint32_t *out, int64_t n, uint32_t k0, uint32_t k1,
                  cudaStream_t st) {
  if (n <= 0) return PC_OK;
  const int tpb = 256;
  philox_kernel<<<(unsigned)((n + tpb - 1) / tpb), tpb, 0, st>>>(ctr, out, n, k0, k1);
  PC_CUDA_TRY(cudaGetLastError());
  return PC_OK;
}

}  // namespace pc

// ---------------------------------------------------------------------------
// DT-SQA entry point that allocates nothing.
//
// Some callers cannot call cudaMalloc: code running under a memory manager
// that owns every device allocation (a framework's caching allocator or a
// fixed arena), or code that must not allocate on a latency-critical path.
// pc_sqa_anneal_noalloc runs the same anneal kernel as pc_sqa_run_dev but
// keeps its scratch (the packed couplings and the per-sweep threshold
// tables) in the file-scope device array below instead of in
// library-allocated buffers.  Every GPU that loads this library keeps this
// array (about 1.57 MiB) until the process exits.
namespace {

constexpr int kNoallocMaxSweeps = 10240;
constexpr int kNoallocJnegBytes = 8192;   // N <= 4096 sites, 16-bit coupling words
constexpr size_t kNoallocTableBytes = (size_t)kNoallocMaxSweeps * pc::kSqaTab * 4;
constexpr size_t kNoallocBytes = kNoallocJnegBytes + kNoallocTableBytes;

static __device__ __align__(256) unsigned char g_sqa_noalloc_scratch[kNoallocBytes];

// Host data reaches the scratch array as kernel parameters, which the
// launch copies by value: no host buffer has to outlive the call and no
// pageable copy is issued.  One chunk carries 12 KiB (a host stack buffer).
constexpr int kStageWords = 3072;
struct StageChunk {
  uint32_t off;                 // destination offset in 32-bit words
  uint32_t n;                   // words carried (<= kStageWords)
  uint32_t w[kStageWords];
};

__global__ void noalloc_stage_kernel(uint32_t *dst, const __grid_constant__ StageChunk c) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < c.n; i += gridDim.x * blockDim.x)
    dst[c.off + i] = c.w[i];
}

int stage_words(uint32_t *dst, StageChunk &c, cudaStream_t st) {
  if (c.n == 0) return PC_OK;
  noalloc_stage_kernel<<<8, 512, 0, st>>>(dst, c);
  PC_CUDA_TRY(cudaGetLastError());
  return PC_OK;
}

// Device address of the scratch array, looked up once per device (with that
// device current) under a lock, so that host threads making their first
// calls at the same time do not race.  The symbol's name is a host-side
// stand-in, never a device address, so only this pointer is handed to
// kernels.
constexpr int kMaxDevices = 64;
std::mutex g_scratch_lock;
unsigned char *g_scratch_ptr[kMaxDevices] = {nullptr};

int noalloc_scratch(int device, unsigned char **out) {
  if (device < 0 || device >= kMaxDevices) return pc::fail(PC_EINVAL, "device index out of range");
  std::lock_guard<std::mutex> lock(g_scratch_lock);
  if (!g_scratch_ptr[device]) {
    void *p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_sqa_noalloc_scratch);
    if (e != cudaSuccess)
      return pc::fail(PC_ECUDA, std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e));
    g_scratch_ptr[device] = static_cast<unsigned char *>(p);
  }
  *out = g_scratch_ptr[device];
  return PC_OK;
}

}  // namespace

extern "C" int pc_sqa_anneal_noalloc(int device, void *stream, uint64_t seed, const int32_t *dims,
                                     const int8_t *J, int P, double T, int n_sweeps,
                                     const double *gamma, int R, uint32_t run0, int32_t *E_dev,
                                     int32_t *best_dev) try {
  using namespace pc;
  if (!dims || !J || (n_sweeps > 0 && !gamma) || (R > 0 && !E_dev))
    return fail(PC_EINVAL, "NULL argument");
  Lattice lat;
  int rc = check_lattice(dims, J, &lat);
  if (rc) return rc;
  if (P < 16 || P % 16 || P > 128) return fail(PC_EINVAL, "P must be a multiple of 16 in [16, 128]");
  if ((int64_t)lat.N * P > 262144) return fail(PC_EINVAL, "N * P must be <= 262144");
  if (!(T > 0.0) || n_sweeps < 0) return fail(PC_EINVAL, "T must be > 0 and n_sweeps >= 0");
  if (n_sweeps > kNoallocMaxSweeps)
    return fail(PC_EINVAL, "pc_sqa_anneal_noalloc: n_sweeps exceeds the scratch limit of 10240");
  if (R < 0 || (uint64_t)run0 + (uint64_t)R > (1ull << 24))
    return fail(PC_EINVAL, "R must be >= 0 and run ids < 2^24");
  for (int s = 0; s < n_sweeps; ++s)
    if (!(gamma[s] > 0.0)) return fail(PC_EINVAL, "every Gamma must be > 0");
  PC_CUDA_TRY(cudaSetDevice(device));
  unsigned char *scratch = nullptr;
  if ((rc = noalloc_scratch(device, &scratch))) return rc;
  if (R == 0) return PC_OK;
  cudaStream_t st = (cudaStream_t)stream;
  uint32_t *words = reinterpret_cast<uint32_t *>(scratch);
  StageChunk chunk_buf;
  StageChunk *chunk = &chunk_buf;

  // couplings: one 16-bit word per site (periodic: no absent bonds), two
  // per staged 32-bit word (N is even)
  {
    const int Lx = lat.L[0], Ly = lat.L[1], Lz = lat.L[2];
    uint16_t *jn = reinterpret_cast<uint16_t *>(chunk->w);
    for (int s = 0; s < lat.N; ++s) {
      const int x = s % Lx, y = (s / Lx) % Ly, z = s / (Lx * Ly);
      const int xm = (x + Lx - 1) % Lx + Lx * (y + Ly * z);
      const int ym = x + Lx * ((y + Ly - 1) % Ly + Ly * z);
      const int zm = x + Lx * (y + Ly * ((z + Lz - 1) % Lz));
      const int8_t j6[6] = {J[3 * s], J[3 * xm], J[3 * s + 1], J[3 * ym + 1], J[3 * s + 2],
                            J[3 * zm + 2]};
      uint16_t m = 0;
      for (int d = 0; d < 6; ++d)
        if (j6[d] < 0) m |= (uint16_t)(1u << d);
      jn[s] = m;
    }
    chunk->off = 0;
    chunk->n = (uint32_t)lat.N / 2;
    if ((rc = stage_words(words, *chunk, st))) return rc;
  }
  // per-sweep threshold tables, kStageWords / kSqaTab sweeps per chunk
  {
    constexpr int W = pc::kSqaTab;
    constexpr int kSweepsPerChunk = kStageWords / W;
    const double beta_eff = 1.0 / ((double)P * T);
    for (int s0 = 0; s0 < n_sweeps; s0 += kSweepsPerChunk) {
      const int ns = (n_sweeps - s0 < kSweepsPerChunk) ? n_sweeps - s0 : kSweepsPerChunk;
      uint32_t *tab = chunk->w;
      for (int k = 0; k < ns; ++k) {
        const int32_t jq = pc_jperp_q(gamma[s0 + k], P, T);
        for (int e = 0; e < W; ++e) tab[W * k + e] = 0u;
        for (int m = 0; m < 3; ++m)
          for (int e = 0; e < 13; ++e) tab[W * k + e + 13 * m] = sqa_threshold(beta_eff, e - 6, jq, 2 * m - 2);
      }
      chunk->off = (uint32_t)(kNoallocJnegBytes / 4 + (size_t)s0 * W);
      chunk->n = (uint32_t)(ns * W);
      if ((rc = stage_words(words, *chunk, st))) return rc;
    }
  }
  SqaArgs a;
  a.Lx = lat.L[0];
  a.Ly = lat.L[1];
  a.Lz = lat.L[2];
  a.N = lat.N;
  a.P = P;
  a.NB = P / 16;
  a.S = n_sweeps;
  a.mLx = recip32((uint32_t)a.Lx);
  a.mLy = recip32((uint32_t)a.Ly);
  a.run0 = run0;
  a.k0 = (uint32_t)(seed & 0xFFFFFFFFu);
  a.k1 = (uint32_t)(seed >> 32);
  a.jneg = reinterpret_cast<const uint16_t *>(scratch);
  a.nbonds = 3 * lat.N;
  a.table = reinterpret_cast<const uint32_t *>(scratch + kNoallocJnegBytes);
  a.E = E_dev;
  a.best = best_dev;
  a.spins = nullptr;
  a.corr = nullptr;
  a.state = nullptr;   // one CTA per run: no state scratch
  a.done = a.queue = a.err = nullptr;
  a.R = R;
  a.K = n_sweeps;
  a.n_items = R;
  a.first_item = 0;
  a.wait_ns = 0;
  return sqa_launch(a, R, st);
} catch (...) {
  return pc::fail_exception();
}
