// Batched negacyclic NTT / inverse NTT over RNS limbs.
//
// Forward: out[j] = sum_i a_i psi^(i (2 bitrev(j) + 1)) mod q, computed as
// log N Cooley-Tukey stages with the psi twist merged into the twiddles
// (twiddle of stage s, butterfly block i: psi^bitrev(2^s + i)).  Inverse:
// Gentleman-Sande stages with psi^-bitrev, then N^-1.
//
// N = 2^(L1+L2) is split in two launches.  The first L1 forward stages only
// couple elements whose index agrees modulo 2^L2 ("columns", 2^L1 words 2^L2 apart);
// the last L2 stages couple only elements inside blocks of 2^L2 consecutive words.
// What bounds a transform is instruction issue on the integer pipes (32-bit multiply-adds at half
// rate, 64-bit products at a quarter), not memory: so the layout spends as few instructions per
// butterfly as it can.
//  * A phase of L stages is two register passes of K0 = ceil(L / 2) and K1 = floor(L / 2) stages
//    (radix 16 twice for L = 8) with one exchange through shared memory between them, every thread
//    holding 2^K0 words of a column or a block (2^17: L1 = 9 in three passes of 8 words, ColGeo; L2 stays 8).
//    The 2^K1 threads of one block lie in one warp: the row phase has no CTA barrier.
//  * The first pass of the column phase and the last one read and write global memory from
//    registers (8 adjacent columns a CTA, 4 at 2^17: whole 32-byte sectors).
//  * Twiddles are (w 2^32, w 2^64) mod q pairs (mont_mul_lazy), stored per phase and block in the
//    order in which the lanes of a warp read them (tw_slot): every load is coalesced and
//    free of bank conflicts, and a block's twiddles are one run of 2^L2 pairs.
//  * Residues stay lazy (Harvey 2014).  For q < 2^57 (and at least kMinPrime, as every q) the forward stages
//    reduce nothing: the first load adds a multiple of q that keeps every difference non-negative, and the last
//    store reduces (below 112q < 2^64); larger primes reduce the first operand at every other stage (below 12q).
//    Inverse: for q < 2^55 bounds double unreduced through a phase.
// GB300, N = 2^16, against Shoup butterflies in radix-8 passes with a CTA barrier each: forward of 384 limbs
// 304 -> 216 us, HMult with rescale of 8 ciphertexts at level 23 3.28 -> 2.30 ms.  The big kernels then issue
// 0.45 - 0.50 instructions a cycle of a scheduler with the multiply pipe 74 - 81% busy, the register loop of the
// butterfly alone 0.50 and 88%: what is left is mostly their instruction count.
// Optional fusions (NttAux): the first phase may read another buffer (out of place) or compute its
// input as the fast basis conversion of a key-switching digit (ModUp fused into the load),
// the inverse may end with a per-limb factor other than N^-1, a digit's own limbs may be skipped,
// and a rescale, a ModDown or both (one transform, see ks_moddown_rescale) may be fused around a
// forward transform (conversion and spread into the first phase's load, the finish into the second
// phase's store).
#pragma once
#include <algorithm>
#include <type_traits>

#include "internal.cuh"
#include "profiler.cuh"

namespace hedap {

// ---------------------------------------------------------------- butterflies
// mont_mul_lazy returns less than 3q.  Forward (Cooley-Tukey), small primes (q < 2^57): x + t and x - t
// as they are; a stage lowers and raises the bounds by 3q, so the first load adds 3 log2(N) q and the words stay
// within [0, (9.2 + 6 log2(N)) q) < 2^64.  Seven products and eight additions, 32.9 cycles of a scheduler per warp
// in a register loop, against 40.3 with x + 3q - t and 37.2 of a Shoup butterfly that reduces x every other stage.
// Large primes: x + 3q - t, and x brought from [0, 12q) to [0, 6q] at even stages: 9q after an even
// stage, 12q < 2^64 after the odd one (and 2^32 more, see sub_if_above).
template <bool SMALL, bool EVEN>
__device__ __forceinline__ void ct_bfly(u64& x, u64& y, const ulonglong2 w, u64 q, uint32_t nqi) {
  if constexpr (!SMALL && EVEN) x = sub_if_above(x, q * 6);
  const u64 t = mont_mul_lazy(y, w.x, w.y, q, nqi);  // [0, 3q)
  y = SMALL ? x - t : x + q * 3 - t;
  x = x + t;
}
__device__ __forceinline__ bool fwd_small(u64 q) { return q < (1ull << 57); }
__device__ __forceinline__ bool inv_small(u64 q) { return q < (1ull << 55); }
// what the first load of a forward transform adds to every word
template <int LOGN>
__device__ __forceinline__ u64 fwd_bias(u64 q) { return fwd_small(q) ? q * (3 * LOGN) : 0; }
// canonical residue of a forward transform's lazy output (112q or 12q, see above)
template <bool SMALL>
__device__ __forceinline__ u64 fwd_canonical(u64 x, u64 q, uint32_t rc) {
  if constexpr (SMALL) {
    x = reduce_lazy(x, q, rc);
  } else {
    if (x >= q * 8) x -= q * 8;
    if (x >= q * 4) x -= q * 4;
    if (x >= q * 2) x -= q * 2;
  }
  return x >= q ? x - q : x;
}
// c - v for a lazy forward output v and a canonical c, as a non-negative 64-bit word
template <bool SMALL>
__device__ __forceinline__ u64 fwd_minus(u64 c, u64 v, u64 q) { return c + q * (SMALL ? 112 : 13) - v; }

// K forward stages in registers on G columns of 2^K words: stage S + u (S the global index of the
// first) pairs words 2^(K-1-u) apart; tw(u, mm) is the twiddle of sub-block mm of stage u
template <bool SMALL, int S, int K, int G, class TW>
__device__ __forceinline__ void fwd_pass(u64 (&v)[G][1 << K], u64 q, uint32_t nqi, TW tw) {
#pragma unroll
  for (int u = 0; u < K; ++u) {
#pragma unroll
    for (int mm = 0; mm < (1 << u); ++mm) {
      const ulonglong2 w = tw(u, mm);
#pragma unroll
      for (int k = 0; k < (1 << (K - 1 - u)); ++k) {
        const int m = (mm << (K - u)) + k, h = 1 << (K - 1 - u);
#pragma unroll
        for (int g = 0; g < G; ++g) {
          if ((S + u) % 2 == 0) ct_bfly<SMALL, true>(v[g][m], v[g][m + h], w, q, nqi);
          else ct_bfly<SMALL, false>(v[g][m], v[g][m + h], w, q, nqi);
        }
      }
    }
  }
}
// K inverse (Gentleman-Sande) stages in registers, the mirror image: stage u pairs words 2^u apart, its
// sub-block mm spans 2^(u+1) words, tw(u', mm) with u' = K - 1 - u as in the forward pass.  SMALL: the
// bound 2^E q doubles at every stage; otherwise (q >= 2^55) sums are brought back towards 3q and differences are taken from
// 4q: sub_if_above may leave a sum 2^32 above 3q, two such sums twice as much, so that the excess doubles at every
// stage of both phases and stays below 2^(32 + 17) < q.
template <bool SMALL, int E, int K, int G, class TW>
__device__ __forceinline__ void inv_pass(u64 (&v)[G][1 << K], u64 q, uint32_t nqi, TW tw) {
#pragma unroll
  for (int u = 0; u < K; ++u) {
#pragma unroll
    for (int mm = 0; mm < (1 << (K - 1 - u)); ++mm) {
      const ulonglong2 w = tw(K - 1 - u, mm);
#pragma unroll
      for (int k = 0; k < (1 << u); ++k) {
        const int m = (mm << (u + 1)) + k, h = 1 << u;
#pragma unroll
        for (int g = 0; g < G; ++g) {
          u64 &x = v[g][m], &y = v[g][m + h];
          const u64 off = SMALL ? q << (E + u) : q * 4;
          u64 s = x + y;
          const u64 d = x + off - y;
          if constexpr (!SMALL) s = sub_if_above(s, q * 3);
          y = mont_mul_lazy(d, w.x, w.y, q, nqi);
          x = s;
        }
      }
    }
  }
}

// ---------------------------------------------------------------- geometry
// asynchronous global -> shared copies (cp.async): every copy of a tile is in flight at once, with
// no register round trip
__device__ __forceinline__ void cp_async16(void* sdst, const void* gsrc) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(sdst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }
__device__ __forceinline__ ulonglong2 ldg2(const u64* p) { return *reinterpret_cast<const ulonglong2*>(p); }
__device__ __forceinline__ void stg2(u64* p, ulonglong2 v) { *reinterpret_cast<ulonglong2*>(p) = v; }

// A phase of L stages on 2^L words: pass 0 of K0 stages, thread `low` (of 2^K1) holding words
// m 2^K1 + low; pass 1 of K1 stages, a thread holding the 2^K1 consecutive words of GP = 2^(K0-K1) groups.
template <int L>
struct Phase {
  static constexpr int K0 = (L + 1) / 2, K1 = L / 2;
  static constexpr int M0 = 1 << K0, M1 = 1 << K1;  // words of a group in pass 0 / pass 1
  static constexpr int GP = 1 << (K0 - K1);         // pass-1 groups a thread owns
  static constexpr int PER = 32 >> K1;              // blocks a warp holds
};
// column phase, a CTA of TH threads, one column a thread, TPC threads a column: the first pass holds words m TPC + low
// (m < M0), the last one words (i TPC + low) M1 + m (i < GP, m < M1).  Word c of column cg at (c + (c >> K1)) COLS + cg (a
// row of padding every 2^K1 rows, so that the last pass's reads are free of bank conflicts).
// The 2^9 rows of N = 2^17 take three passes of three stages, 8 words a thread.  With 2^9 words in the row phase instead, a
// thread held 32 words, or 16 with their 128-bit key sums, and both spilled (the key product's 912 bytes a thread): forward
// of 160 limbs 312 -> 219 us (primes of 60 bits 363 -> 237 us), HMult of 8 ciphertexts at level 7 1263 -> 1006 us, of one
// 273 -> 175 us, rescale of 8 at level 8 with 58-bit primes 465 -> 291 us.
template <int L1, int TH>
struct ColGeo {
  static constexpr bool THREE = L1 == 9;
  static constexpr int K0 = THREE ? 3 : Phase<L1>::K0, K1 = THREE ? 3 : Phase<L1>::K1;
  static constexpr int M0 = 1 << K0, M1 = 1 << K1, TPC = (1 << L1) / M0;
  static constexpr int GP = M0 / M1;
  static constexpr int COLS = TH / TPC;
  static constexpr int XWORDS = ((1 << L1) + (1 << (L1 - K1))) * COLS;  // exchange
  static constexpr int TILE = (1 << L1) * COLS;                         // one staged tile
  // row of word c in the exchange, additive over numbers without a common bit; of a thread's offset low < TPC
  static __device__ constexpr int row(int c) { return c + (c >> K1); }
  static __device__ constexpr int low_row(int low) { return THREE ? row(low) : low; }
};
// row phase, per warp: PER blocks, two words of padding every 2^K1 words (LDS.128 of consecutive words is free
// of bank conflicts) and 2^K1 after each block when several blocks share a half-warp
template <int L2>
struct RowGeo : Phase<L2> {
  static_assert(L2 <= 8, "at most 16 words a thread; the inverse's 2^(L2+1) q stay below 2^64");
  using P = Phase<L2>;
  static constexpr int GS = P::M1 + 2;                                           // stride of a group
  static constexpr int BS = P::M0 * GS + (P::K1 < 4 ? P::M1 : 0);                // stride of a block
  static constexpr int XWORDS = P::PER * BS;
  // place of word pair e (words 2 e, 2 e + 1) of a block; additive over numbers without a common bit
  static constexpr int pair(int e) { return (e >> (P::K1 - 1)) * GS + (e & (P::M1 / 2 - 1)) * 2; }
};

// ---------------------------------------------------------------- fused loads
// true when limb li of `part` is one of its digit's own limbs (skipped, see NttAux)
__device__ __forceinline__ bool own_limb(const NttAux& A, int part, int li) {
  if (!A.own_alpha) return false;
  const int lo = (part % A.own_dn) * A.own_alpha;
  return li >= lo && li < min(lo + A.own_alpha, A.own_limit);
}
// A first phase's input words of one limb, from the words z(t) of `ns` tiles: the digit's
// coefficient-domain limbs (ModUp), the special limbs (ModDown; the last limb's coefficients as z(ns) when a
// rescale is fused) or the last limb (rescale), at most three products.  They share one Montgomery
// step.  ModUp: a term folded into the key is z itself, below the bound the key's construction checked (8q
// in all).  ModDown: q - floor(P/2) mod q plus the products (below 4.2q).  The rescale's centred last
// limb: x, plus -q_l mod q when x > q_l / 2, below 3q.  In all below 9.2q.
enum LoadKind { LOAD_PLAIN = 0, LOAD_MODUP = 1, LOAD_MODDOWN = 2, LOAD_SPREAD = 3 };
enum LastLimb { LAST_NONE = 0, LAST_RAW = 1, LAST_MONT = 2 };  // how a fused rescale's last limb enters the sum
template <int KIND>
struct FusedLoad {
  static constexpr int MAXT = 3;
  u64 f[MAXT], fb[MAXT];  // products: factor pairs
  int tile[MAXT];         // tile of product t
  u64 off, half, sub;
  PrimeDev P;
  int nm, raw, last;  // products, the tile added as it is (-1: none), LastLimb
  int ns;
  // bias: added to every word (fwd_bias)
  __device__ __forceinline__ void init(const NttAux& A, const Tables& T, const PrimeDev& p, u64 bias, int j, int li,
                                       int n_tiles) {
    P = p;
    ns = n_tiles;
    off = bias;
    half = sub = 0;
    raw = -1;
    last = LAST_NONE;
    nm = KIND == LOAD_SPREAD ? 0 : ns;
    if (KIND == LOAD_MODUP) {
      const u64* bc = A.bconv + (size_t)j * A.own_alpha * A.ext + li;
#pragma unroll
      for (int t = 0; t < MAXT; ++t)
        if (t < ns && !bc[A.bconv_b_offset + (size_t)t * A.ext]) raw = t;  // at most one
      nm = ns - (raw >= 0);
#pragma unroll
      for (int t = 0; t < MAXT; ++t) {
        tile[t] = raw >= 0 && t >= raw ? t + 1 : t;
        f[t] = t < nm ? bc[(size_t)tile[t] * A.ext] : 0;
        fb[t] = t < nm ? bc[A.bconv_b_offset + (size_t)tile[t] * A.ext] : 0;
      }
    } else if (KIND == LOAD_MODDOWN) {
#pragma unroll
      for (int t = 0; t < MAXT; ++t) {
        const bool on = t < ns;
        tile[t] = t;
        f[t] = on ? A.pconv_phat[(size_t)t * A.pconv_ld + li] : 0;
        fb[t] = on ? A.pconv_phat_b[(size_t)t * A.pconv_ld + li] : 0;
      }
      off += p.q - A.pconv_half[li];
    }
    if (KIND == LOAD_SPREAD || (KIND == LOAD_MODDOWN && A.spread)) {
      const u64 ql = T.pr[A.spread_prime].q;
      half = ql >> 1;
      sub = p.q - A.spread_sub[li];
      last = ql < 2 * p.q ? LAST_RAW : LAST_MONT;
    }
  }
  template <int NM, bool RAW, int LAST, class Z>
  __device__ __forceinline__ u64 word(Z z) const {
    const u64 q = P.q;
    u64 v = off;
    MontAcc s{0, 0};
#pragma unroll
    for (int t = 0; t < NM; ++t) mont_mac(s, z(tile[t]), f[t], fb[t]);
    if (RAW) v += z(raw);
    if (LAST != LAST_NONE) {
      const u64 x = z(KIND == LOAD_SPREAD ? 0 : ns);
      if (LAST == LAST_RAW) v += x;
      else mont_add(s, x, P.r64);
      if (x > half) v += sub;
    }
    if (NM > 0 || LAST == LAST_MONT) v += mont_finish(s, q, P.nqi);
    return v;
  }
  // calls body with a function word(z) for this limb's terms: no branch per word
  template <class F>
  __device__ __forceinline__ void apply(F body) const {
#define HEDAP_WORDS(NM, RAW, LAST) body([&](auto z) { return word<NM, RAW, LAST>(z); })
    if constexpr (KIND == LOAD_SPREAD) {
      if (last == LAST_RAW) HEDAP_WORDS(0, false, LAST_RAW);
      else HEDAP_WORDS(0, false, LAST_MONT);
    } else if constexpr (KIND == LOAD_MODUP) {
      if (raw >= 0) {
        if (nm == 1) HEDAP_WORDS(1, true, LAST_NONE);
        else if (nm == 2) HEDAP_WORDS(2, true, LAST_NONE);
        else HEDAP_WORDS(0, true, LAST_NONE);
      } else {
        if (nm == 1) HEDAP_WORDS(1, false, LAST_NONE);
        else if (nm == 2) HEDAP_WORDS(2, false, LAST_NONE);
        else HEDAP_WORDS(3, false, LAST_NONE);
      }
    } else {
      if (last == LAST_NONE) {
        if (nm == 1) HEDAP_WORDS(1, false, LAST_NONE);
        else if (nm == 2) HEDAP_WORDS(2, false, LAST_NONE);
        else HEDAP_WORDS(3, false, LAST_NONE);
      } else if (last == LAST_RAW) {
        if (nm == 1) HEDAP_WORDS(1, false, LAST_RAW);
        else if (nm == 2) HEDAP_WORDS(2, false, LAST_RAW);
        else HEDAP_WORDS(3, false, LAST_RAW);
      } else {
        if (nm == 1) HEDAP_WORDS(1, false, LAST_MONT);
        else if (nm == 2) HEDAP_WORDS(2, false, LAST_MONT);
        else HEDAP_WORDS(3, false, LAST_MONT);
      }
    }
#undef HEDAP_WORDS
  }
};

// ---------------------------------------------------------------- forward, column phase
// all passes of one limb's columns: v holds the first pass's input (row m TPC + low), o the last one's output (row
// (i TPC + low) M1 + m of this thread's column); tw: global memory (L1) or shared memory
template <bool SMALL, int L1, int TH>
__device__ __forceinline__ void fwd_cols_passes(u64 (&v)[1][ColGeo<L1, TH>::M0], u64* xs, const ulonglong2* tw, u64 q,
                                                uint32_t nqi, int low, int cg,
                                                u64 (&o)[ColGeo<L1, TH>::GP][1][ColGeo<L1, TH>::M1]) {
  using G = ColGeo<L1, TH>;
  fwd_pass<SMALL, 0, G::K0, 1>(v, q, nqi, [&](int u, int mm) { return tw[(1 << u) + mm]; });
  __syncthreads();  // the last limb's exchange has been read
#pragma unroll
  for (int m = 0; m < G::M0; ++m) xs[(G::row(m * G::TPC) + G::low_row(low)) * G::COLS + cg] = v[0][m];
  __syncthreads();
  if constexpr (G::THREE) {  // the middle pass: rows hi 64 + m 8 + low % 8
    const int hi = low >> 3;
    u64* x = xs + (hi * G::row(64) + (low & 7)) * G::COLS + cg;
#pragma unroll
    for (int m = 0; m < 8; ++m) v[0][m] = x[G::row(m * 8) * G::COLS];
    fwd_pass<SMALL, 3, 3, 1>(v, q, nqi, [&](int u, int mm) { return tw[(8 << u) + (hi << u) + mm]; });
#pragma unroll
    for (int m = 0; m < 8; ++m) x[G::row(m * 8) * G::COLS] = v[0][m];
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < G::GP; ++i) {
    const int hi = i * G::TPC + low;  // rows hi 2^K1 + m
#pragma unroll
    for (int m = 0; m < G::M1; ++m) o[i][0][m] = xs[(hi * (G::M1 + 1) + m) * G::COLS + cg];
    constexpr int GROUPS = 1 << (L1 - G::K1);
    fwd_pass<SMALL, L1 - G::K1, G::K1, 1>(o[i], q, nqi, [&](int u, int mm) {
      return tw[GROUPS + ((1 << u) - 1 + mm) * GROUPS + hi];
    });
  }
}
// the same, the output stored to global memory: out at (row 0, this thread's column)
template <bool SMALL, int L1, int L2, int TH>
__device__ __forceinline__ void fwd_cols_body(u64 (&v)[1][ColGeo<L1, TH>::M0], u64* xs, const ulonglong2* tw, u64 q,
                                              uint32_t nqi, int low, int cg, u64* out) {
  using G = ColGeo<L1, TH>;
  u64 o[G::GP][1][G::M1];
  fwd_cols_passes<SMALL, L1, TH>(v, xs, tw, q, nqi, low, cg, o);
#pragma unroll
  for (int i = 0; i < G::GP; ++i)
#pragma unroll
    for (int m = 0; m < G::M1; ++m) out[(size_t)((i * G::TPC + low) * G::M1 + m) << L2] = o[i][0][m];
}
template <int N, int TH>  // N twiddles into shared memory
__device__ __forceinline__ void stage_twiddles(ulonglong2* dst, const ulonglong2* src, int t) {
#pragma unroll
  for (int i = 0; i < (N + TH - 1) / TH; ++i)
    if (N % TH == 0 || i * TH + t < N) cp_async16(dst + i * TH + t, src + i * TH + t);
}
template <int L1, int L2, int TH, int MINB>
__global__ void __launch_bounds__(TH, MINB) k_ntt_fwd_cols(Tables T, LimbSet S, NttAux A) {
  using G = ColGeo<L1, TH>;
  extern __shared__ __align__(16) u64 sm[];
  constexpr size_t N = (size_t)1 << (L1 + L2);
  const int cg = threadIdx.x % G::COLS, low = threadIdx.x / G::COLS;
  const int y = blockIdx.y, part = y / S.n_limbs, li = S.limb_begin + y % S.n_limbs;
  if (own_limb(A, part, li)) return grid_wait();
  const int pi = S.prime(li);
  const PrimeDev P = T.pr[pi];
  const size_t col = (size_t)blockIdx.x * G::COLS + cg;
  const u64* src = (A.src ? A.src + part * A.src_stride + (size_t)li * N : S.limb(part, li, N)) + col;
  ulonglong2* tw = reinterpret_cast<ulonglong2*>(sm + G::XWORDS);
  stage_twiddles<1 << L1, TH>(tw, T.psi2 + (size_t)pi * tw_stride(L1, L2), threadIdx.x);
  cp_async_commit();
  const u64 bias = fwd_bias<L1 + L2>(P.q);
  grid_wait();
  u64 v[1][G::M0];
#pragma unroll
  for (int m = 0; m < G::M0; ++m) v[0][m] = src[(size_t)(m * G::TPC + low) << L2] + bias;
  cp_async_wait_all();
  __syncthreads();
  u64* out = S.limb(part, li, N) + col;
  if (fwd_small(P.q)) fwd_cols_body<true, L1, L2, TH>(v, sm, tw, P.q, P.nqi, low, cg, out);
  else fwd_cols_body<false, L1, L2, TH>(v, sm, tw, P.q, P.nqi, low, cg, out);
}

// The fused first phases read the same few tiles for every output limb: the ModUp of one digit its na <= 3
// coefficient-domain limbs z, the ModDown conversion the K <= 3 special-prime limbs (plus the last limb when a
// rescale is fused), the rescale spread the last limb.  A CTA stages the tiles of its TH / 2^K1 columns once
// (cp.async, straight into shared memory) and runs the column phase of `lpc` consecutive output limbs of one
// part from there.  One column a thread: with two, the tiles let only 8 warps fit an SM and the passes
// waited on their own latency (1313 against 960 us when it was tried, 770 us since; N = 2^16, 8 x 12 digits at level 23).
template <int L1, int L2, int TH, int MINB, int KIND>
__global__ void __launch_bounds__(TH, MINB) k_ntt_fwd_cols_shared(Tables T, LimbSet S, NttAux A, int lpc) {
  using G = ColGeo<L1, TH>;
  extern __shared__ __align__(16) u64 sm[];
  constexpr size_t N = (size_t)1 << (L1 + L2);
  const int cg = threadIdx.x % G::COLS, low = threadIdx.x / G::COLS;
  const int groups = (S.n_limbs + lpc - 1) / lpc;
  const int part = blockIdx.y / groups, g = blockIdx.y % groups;
  const int l0 = S.limb_begin + g * lpc, l1 = min(l0 + lpc, S.limb_begin + S.n_limbs);
  const size_t col = (size_t)blockIdx.x * G::COLS;
  u64* zt = sm + G::XWORDS;
  const int j = KIND == LOAD_MODUP ? part % A.own_dn : 0, lo = j * A.own_alpha;
  const int ns = KIND == LOAD_MODUP ? min(A.own_alpha, A.own_limit - lo) : KIND == LOAD_MODDOWN ? A.pconv_K : 0;
  const u64* base = KIND == LOAD_MODUP     ? A.z + (size_t)(part / A.own_dn) * A.z_stride + (size_t)lo * N
                    : KIND == LOAD_MODDOWN ? A.pconv + (size_t)part * A.pconv_stride
                                           : nullptr;
  const u64* last = KIND != LOAD_MODUP && A.spread ? A.spread + (size_t)part * A.spread_stride : nullptr;
  const int tiles = ns + (last ? 1 : 0);
  grid_wait();
  for (int i = threadIdx.x; i < tiles * (G::TILE / 2); i += TH) {
    const int t = i / (G::TILE / 2), e = 2 * (i % (G::TILE / 2)), row = e / G::COLS;
    const u64* src = t < ns ? base + (size_t)t * N : last;
    cp_async16(zt + (size_t)t * G::TILE + e, src + ((size_t)row << L2) + col + e % G::COLS);
  }
  cp_async_commit();
  cp_async_wait_all();
  __syncthreads();
  FusedLoad<KIND> F;
  for (int li = l0; li < l1; ++li) {
    if (own_limb(A, part, li)) continue;
    const int pi = S.prime(li);
    const PrimeDev P = T.pr[pi];
    F.init(A, T, P, fwd_bias<L1 + L2>(P.q), j, li, ns);
    u64 v[1][G::M0];
    const u64* zl = zt + low * G::COLS + cg;
    F.apply([&](auto word) {
#pragma unroll
      for (int m = 0; m < G::M0; ++m) v[0][m] = word([&](int t) { return zl[t * G::TILE + m * G::TPC * G::COLS]; });
    });
    const ulonglong2* tw = T.psi2 + (size_t)pi * tw_stride(L1, L2);
    u64* out = S.limb(part, li, N) + col + cg;
    if (fwd_small(P.q)) fwd_cols_body<true, L1, L2, TH>(v, sm, tw, P.q, P.nqi, low, cg, out);
    else fwd_cols_body<false, L1, L2, TH>(v, sm, tw, P.q, P.nqi, low, cg, out);
  }
}

// The same first phases with more than three products a word (digits of 4 to 8 primes, 4 to 8 special primes):
// the tiles would fill the shared memory, so they are read from L2 term by term into open sums (MontAcc) in registers.
// Three warps a scheduler do not hide L2 by themselves: a thread's words go in two halves, the loads of one in flight
// while the products of the other are formed (N = 2^16, 3 ciphertexts at level 18, eight primes a digit, seven
// special ones: ModUp 136 -> 130 us, ModDown with the rescale 145 -> 87 us, as against a term's words at once).
template <int L1, int L2, int TH, int MINB, int KIND>
__global__ void __launch_bounds__(TH, MINB) k_ntt_fwd_cols_wide(Tables T, LimbSet S, NttAux A) {
  using G = ColGeo<L1, TH>;
  extern __shared__ __align__(16) u64 sm[];
  constexpr size_t N = (size_t)1 << (L1 + L2);
  const int cg = threadIdx.x % G::COLS, low = threadIdx.x / G::COLS;
  const int part = blockIdx.y / S.n_limbs, li = S.limb_begin + blockIdx.y % S.n_limbs;
  grid_wait();
  if (own_limb(A, part, li)) return;
  const int pi = S.prime(li);
  const PrimeDev P = T.pr[pi];
  const u64 q = P.q;
  const size_t col = (size_t)blockIdx.x * G::COLS + cg;
  const int j = KIND == LOAD_MODUP ? part % A.own_dn : 0, lo = j * A.own_alpha;
  const int ns = KIND == LOAD_MODUP ? min(A.own_alpha, A.own_limit - lo) : A.pconv_K;
  const u64* base = (KIND == LOAD_MODUP ? A.z + (size_t)(part / A.own_dn) * A.z_stride + (size_t)lo * N
                                        : A.pconv + (size_t)part * A.pconv_stride) + ((size_t)low << L2) + col;
  u64 off = fwd_bias<L1 + L2>(q);
  if (KIND == LOAD_MODDOWN) off += q - A.pconv_half[li];
  u64 v[1][G::M0];
  MontAcc s[G::M0];
#pragma unroll
  for (int m = 0; m < G::M0; ++m) {
    v[0][m] = 0;
    s[m] = MontAcc{0, 0};
  }
  auto close = [&] {  // one Montgomery step: the column sums stay below 2^64 for four products
#pragma unroll
    for (int m = 0; m < G::M0; ++m) {
      v[0][m] += mont_finish(s[m], q, P.nqi);
      s[m] = MontAcc{0, 0};
    }
  };
  constexpr int H = G::M0 / 2;
  const u64* last =
      KIND == LOAD_MODDOWN && A.spread ? A.spread + (size_t)part * A.spread_stride + ((size_t)low << L2) + col : nullptr;
  u64 x[2][H];
  auto load = [&](const u64* z, auto half) {
#pragma unroll
    for (int m = 0; m < H; ++m) x[half()][m] = z[(size_t)((half() * H + m) * G::TPC) << L2];
  };
  const auto h0 = std::integral_constant<int, 0>{};
  const auto h1 = std::integral_constant<int, 1>{};
  const u64* fp = KIND == LOAD_MODUP ? A.bconv + (size_t)lo * A.ext + li : A.pconv_phat + li;
  const u64* fbp = KIND == LOAD_MODUP ? fp + A.bconv_b_offset : A.pconv_phat_b + li;
  const int fld = KIND == LOAD_MODUP ? A.ext : A.pconv_ld;
  load(base, h0);
  u64 f = *fp, fb = *fbp;
#pragma unroll 1
  for (int t = 0; t < ns; ++t) {
    const u64 *z = base + (size_t)t * N, *next = t + 1 < ns ? z + N : last;
    load(z, h1);
    u64 f_next = 0, fb_next = 0;
    if (t + 1 < ns) {
      f_next = fp[(size_t)(t + 1) * fld];
      fb_next = fbp[(size_t)(t + 1) * fld];
    }
    if (t == 4) close();
    auto take = [&](auto half) {
      if (KIND == LOAD_MODUP && !fb) {  // folded into the key
#pragma unroll
        for (int m = 0; m < H; ++m) v[0][half() * H + m] += x[half()][m];
      } else {
#pragma unroll
        for (int m = 0; m < H; ++m) mont_mac(s[half() * H + m], x[half()][m], f, fb);
      }
    };
    take(h0);
    if (next) load(next, h0);
    take(h1);
    f = f_next;
    fb = fb_next;
  }
  if (KIND == LOAD_MODDOWN && last) load(last, h1);
  close();
  // at most eight products (below 1.1q each, and 2q of the two steps) or a folded limb and seven: below 16q by the
  // key's construction; brought below 10q, with the bias, the ModDown's constant and the last limb below 12q
#pragma unroll
  for (int m = 0; m < G::M0; ++m) v[0][m] = off + (v[0][m] >= q * 6 ? v[0][m] - q * 6 : v[0][m]);
  if (KIND == LOAD_MODDOWN && last) {
    const u64 ql = T.pr[A.spread_prime].q, half = ql >> 1, sub = q - A.spread_sub[li];
#pragma unroll
    for (int m = 0; m < G::M0; ++m) {
      const u64 y = x[m / H][m % H];
      MontAcc a{0, 0};
      mont_add(a, y, P.r64);
      v[0][m] += mont_finish(a, q, P.nqi) + (y > half ? sub : 0);
    }
  }
  const ulonglong2* tw = T.psi2 + (size_t)pi * tw_stride(L1, L2);
  u64* out = S.limb(part, li, N) + col;
  if (fwd_small(q)) fwd_cols_body<true, L1, L2, TH>(v, sm, tw, q, P.nqi, low, cg, out);
  else fwd_cols_body<false, L1, L2, TH>(v, sm, tw, q, P.nqi, low, cg, out);
}

// ---------------------------------------------------------------- forward, row phase
// A warp owns PER blocks of 2^L2 consecutive words of one limb; 2^K1 lanes per block.
template <bool SMALL, int L1, int L2>
__device__ __forceinline__ void fwd_rows_body(u64 (&v)[1][1 << Phase<L2>::K0], u64* xs, const ulonglong2* tw,
                                              const PrimeDev& P, int low) {
  using G = RowGeo<L2>;
  const u64 q = P.q;
  fwd_pass<SMALL, L1, G::K0, 1>(v, q, P.nqi, [&](int u, int mm) { return tw[(1 << u) + mm]; });
#pragma unroll
  for (int m = 0; m < G::M0; ++m) xs[m * G::GS + low] = v[0][m];
  __syncwarp();
#pragma unroll
  for (int i = 0; i < G::GP; ++i) {
    const int hi = i * G::M1 + low;
    u64 w[1][G::M1];
#pragma unroll
    for (int m = 0; m < G::M1; m += 2) {
      const ulonglong2 x = ldg2(xs + hi * G::GS + m);
      w[0][m] = x.x;
      w[0][m + 1] = x.y;
    }
    fwd_pass<SMALL, L1 + G::K0, G::K1, 1>(w, q, P.nqi, [&](int u, int mm) {
      return tw[G::M0 + ((1 << u) - 1 + mm) * G::M0 + hi];
    });
#pragma unroll
    for (int m = 0; m < G::M1; m += 2) stg2(xs + hi * G::GS + m, ulonglong2{w[0][m], w[0][m + 1]});
  }
  __syncwarp();
}
// word pair e = k 2^K1 + low (words 2 e, 2 e + 1) of a block in the exchange buffer
template <int L2>
__device__ __forceinline__ ulonglong2 row_pair(const u64* xs, int k, int low) {
  using G = RowGeo<L2>;
  return ldg2(xs + G::pair(low) + G::pair(k * G::M1));
}
// word m 2^K1 + low of a block in the exchange buffer (lane part and compile-time part)
template <int L2>
__device__ __forceinline__ uint32_t row_word(int m, int low) {
  using G = RowGeo<L2>;
  return G::pair(low >> 1) + (low & 1) + G::pair(m * (G::M1 / 2));
}
// a caller's limbs may begin at any 8-byte boundary: the row phases then load and store single words (40 limbs of 2^16
// words forward 29 us, inverse 33 us; through an aligned buffer, two copies, 47 and 50 us)
__device__ __forceinline__ bool odd_word(const u64* p) { return reinterpret_cast<uintptr_t>(p) & 8; }
// n0: the block's first word of the limb, at: of the part
template <bool SMALL, int L1, int L2>
__device__ __forceinline__ void fwd_rows_store(const u64* xs, const NttAux& A, u64* a, uint32_t n0, size_t at, int part,
                                               int li, const PrimeDev& P, int low) {
  constexpr int LOGN = L1 + L2;
  using G = RowGeo<L2>;
  const u64 q = P.q;
  constexpr int PAIRS = G::M0 / 2;  // word pairs of a lane
  if (A.fin_w2) {  // ModDown fused with the rescale: c (P q_l)^-1 + (e - v) q_l^-1; or a rescale of c times a constant
    const u64* cp = A.fin_c + (size_t)part * A.fin_c_stride + at;
    const u64* ep = A.fin_e ? A.fin_e + (size_t)part * A.fin_e_stride + at : nullptr;
    u64* dp = A.fin_dst + (size_t)part * A.fin_dst_stride + at;
    const u64 w = A.fin_w[li], wb = A.fin_wb[li], w2 = A.fin_w2[li], w2b = A.fin_w2b[li];
    auto fin = [&](u64 c, u64 e, u64 v) {  // both products in one Montgomery step: below 4q
      MontAcc s{0, 0};
      mont_mac(s, c, w, wb);
      mont_mac(s, fwd_minus<SMALL>(e, v, q), w2, w2b);
      u64 z = mont_finish(s, q, P.nqi);
      if (z >= q * 2) z -= q * 2;
      return z >= q ? z - q : z;
    };
#pragma unroll
    for (int k = 0; k < PAIRS; ++k) {
      const int e = k * G::M1 + low;
      const ulonglong2 v = row_pair<L2>(xs, k, low), c = ldg2(cp + 2 * e);
      const ulonglong2 ee = ep ? ldg2(ep + 2 * e) : ulonglong2{0, 0};
      ulonglong2 z;
      z.x = fin(c.x, ee.x, v.x);
      z.y = fin(c.y, ee.y, v.y);
      if (A.fin_neg) {
        z.x = sub_mod(0, z.x, q);
        z.y = sub_mod(0, z.y, q);
      }
      stg2(dp + 2 * e, z);
    }
  } else if (A.fin_dst) {  // fused epilogue of a rescale / ModDown: (c - v) * w (+ dst)
    const u64* cp = A.fin_c + (size_t)part * A.fin_c_stride + at;
    const int r = A.fin_d ? part / A.fin_per : 0, rp = part - r * A.fin_per;
    u64* dp = (A.fin_d ? A.fin_dsts[r] : A.fin_dst) + (size_t)rp * A.fin_dst_stride + at;
    const u64 w = A.fin_w[li], wb = A.fin_wb[li];
    auto fin = [&](u64 c, u64 v) {  // below 3q
      u64 z = mont_mul_lazy(fwd_minus<SMALL>(c, v, q), w, wb, q, P.nqi);
      if (z >= q * 2) z -= q * 2;
      return z >= q ? z - q : z;
    };
    const bool acc = (part & 1) ? A.fin_acc_odd : A.fin_acc_even;
#pragma unroll
    for (int k = 0; k < PAIRS; ++k) {
      const int e = k * G::M1 + low;
      const ulonglong2 v = row_pair<L2>(xs, k, low), c = ldg2(cp + 2 * e);
      ulonglong2 z;
      z.x = fin(c.x, v.x);
      z.y = fin(c.y, v.y);
      if (acc) {
        ulonglong2 d;
        if (A.fin_d) {
          const u64* limb = A.fin_d + (size_t)rp * A.fin_d_stride + (at - n0);
          d = galois_pair(limb, galois_index(n0 + 2 * e, A.fin_gs[r], LOGN));
        } else {
          d = ldg2(dp + 2 * e);
        }
        z.x = add_mod(z.x, d.x, q);
        z.y = add_mod(z.y, d.y, q);
      }
      stg2(dp + 2 * e, z);
    }
  } else if (odd_word(a)) {
#pragma unroll
    for (int m = 0; m < G::M0; ++m) a[m * G::M1 + low] = fwd_canonical<SMALL>(xs[row_word<L2>(m, low)], q, P.rc);
  } else {
#pragma unroll
    for (int k = 0; k < PAIRS; ++k) {
      const int e = k * G::M1 + low;
      const ulonglong2 v = row_pair<L2>(xs, k, low);
      stg2(a + 2 * e, ulonglong2{fwd_canonical<SMALL>(v.x, q, P.rc), fwd_canonical<SMALL>(v.y, q, P.rc)});
    }
  }
}

// `ppc` parts of one limb per warp, one after the other: they share the blocks' twiddles, staged once
template <int L1, int L2, int W, int MINB>
__global__ void __launch_bounds__(32 * W, MINB) k_ntt_fwd_rows(Tables T, LimbSet S, NttAux A, int ppc) {
  using G = RowGeo<L2>;
  extern __shared__ __align__(16) u64 sm[];
  constexpr size_t N = (size_t)1 << (L1 + L2);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, low = lane % G::M1, b = lane / G::M1;
  const int pg = blockIdx.y / S.n_limbs, li = S.limb_begin + blockIdx.y % S.n_limbs;
  const int pi = S.prime(li);
  const PrimeDev P = T.pr[pi];
  const int blk = (blockIdx.x * W + warp) * G::PER + b;
  u64* xs = sm + warp * G::XWORDS + b * G::BS;
  ulonglong2* tw = reinterpret_cast<ulonglong2*>(sm + W * G::XWORDS) + (warp * G::PER << L2);  // the warp's blocks
  stage_twiddles<(G::PER << L2), 32>(tw, T.psi2 + (size_t)pi * tw_stride(L1, L2) + (1 << L1) + ((size_t)(blk - b) << L2),
                                     lane);
  cp_async_commit();
  tw += b << L2;
  const size_t j0 = (size_t)blk << L2, at = (size_t)li * N + j0;
  grid_wait();
  bool staged = false;
  for (int part = pg * ppc; part < min((pg + 1) * ppc, S.n_parts); ++part) {
    if (own_limb(A, part, li)) continue;
    u64* a = S.limb(part, li, N) + j0;
    if (A.fin_dst) {  // the epilogue's operands: fetched into L2 while the passes run (128-byte lines)
      const u64* cp = A.fin_c + (size_t)part * A.fin_c_stride + at;
      const u64* dp = A.fin_e ? A.fin_e + (size_t)part * A.fin_e_stride + at
                              : A.fin_dst + (size_t)part * A.fin_dst_stride + at;
      const bool acc = A.fin_e || (!A.fin_d && ((part & 1) ? A.fin_acc_odd : A.fin_acc_even));
      for (int idx = 16 * low; idx < (1 << L2); idx += 16 * G::M1) {
        asm volatile("prefetch.global.L2 [%0];" ::"l"(cp + idx));
        if (acc) asm volatile("prefetch.global.L2 [%0];" ::"l"(dp + idx));
      }
    }
    u64 v[1][G::M0];
#pragma unroll
    for (int m = 0; m < G::M0; ++m) v[0][m] = a[m * G::M1 + low];
    if (!staged) {
      cp_async_wait_all();
      __syncwarp();
      staged = true;
    }
    if (fwd_small(P.q)) {
      fwd_rows_body<true, L1, L2>(v, xs, tw, P, low);
      fwd_rows_store<true, L1, L2>(xs, A, a, (uint32_t)j0, at, part, li, P, low);
    } else {
      fwd_rows_body<false, L1, L2>(v, xs, tw, P, low);
      fwd_rows_store<false, L1, L2>(xs, A, a, (uint32_t)j0, at, part, li, P, low);
    }
    __syncwarp();
  }
  cp_async_wait_all();
}

// ---------------------------------------------------------------- forward, row phase fused with the key inner product
// The extended digits of a key switch are transformed and immediately consumed by the inner product
// with the switching key, so the transformed digits are never written.  A warp owns one ciphertext k, one
// extended limb t (prime pt) and KB blocks of 2^L2 words (256 words in all, 8 a lane, so that the lane's
// 16 sums of 128 bits stay in registers) and walks the dn digits: the column-phase output of digit j is copied
// into the warp's shared memory with cp.async while the previous digit computes, the passes run between
// warp barriers, and each word is multiplied by the two key words of digit j, limb t (loaded before the
// passes).  The digit owning t comes last: there the NTT-domain input d itself.  One reduction per word at the end; acc[k][0/1][t]
// are the only stores.  Modular sums do not depend on order, so the result equals the separate
// transform and inner product bit for bit.  Consecutive warps hold the batch members of one block,
// so each key word comes from L2 once per CTA and the block's twiddles, staged in shared memory once,
// serve all of them.  Words entering the products are below 112q < 2^64 with q < 2^57, or below 3.1q with
// q < 2^60.1: the sum of up to 64 products stays below 2^128.
template <int L2>
struct KskGeo {
  static constexpr int PER = 8;                             // words a lane
  static constexpr int LPB = (1 << L2) / PER;               // lanes a block
  static constexpr int KB = 32 / LPB;                       // blocks a warp
  // passes: a first one of F stages, then passes of 3
  static constexpr int F = L2 % 3 ? L2 % 3 : 3, NP = (L2 + 2) / 3;
  static constexpr int BS = (1 << L2) + 2 * (1 << L2 >> 3) + 8 * ((1 << L2) >> 6) + (L2 < 6 ? 8 : 0);
  // padded index inside a block, and of a word of the warp's run; both are additive over numbers without a common
  // bit, which keeps the lane's part out of the unrolled loops
  static constexpr int word(int x) { return x + 2 * (x >> 3) + 8 * (x >> 6); }
  static constexpr int run_word(int x) { return (x >> L2) * BS + word(x & ((1 << L2) - 1)); }
  static constexpr int XWORDS = KB * BS;
};
// twiddles of a block as staged for KskGeo's passes: those of a pass of K stages from local stage s0
// at 2^s0: entry e = (1 << u) - 1 + mm of group `high` at 2^s0 + (e << s0) + high
template <bool SMALL, int L1, int L2, int S0>
__device__ __forceinline__ void ksk_passes(u64* xs, const ulonglong2* tw, u64 q, uint32_t nqi, int ll,
                                           u64 (&out)[KskGeo<L2>::PER]) {
  using G = KskGeo<L2>;
  constexpr int K = S0 == 0 ? G::F : 3;
  constexpr int TL = 1 << (L2 - S0 - K), GPT = G::PER >> K;
  u64 v[GPT][1][1 << K];
#pragma unroll
  for (int i = 0; i < GPT; ++i) {
    const int g = TL == 1 ? ll * GPT + i : i * G::LPB + ll, low = g & (TL - 1), high = g / TL;
    const int base = high * (TL << K) + low;
    if constexpr (TL == 1 && K == 3) {
#pragma unroll
      for (int m = 0; m < 8; m += 2) {
        const ulonglong2 x = ldg2(xs + G::word(base) + m);
        v[i][0][m] = x.x;
        v[i][0][m + 1] = x.y;
      }
    } else {
#pragma unroll
      for (int m = 0; m < (1 << K); ++m) v[i][0][m] = xs[G::word(base) + G::word(m * TL)];
    }
    fwd_pass<SMALL, L1 + S0, K, 1>(v[i], q, nqi, [&](int u, int mm) {
      return tw[(1 << S0) + (((1 << u) - 1 + mm) << S0) + high];
    });
    if constexpr (TL > 1) {
#pragma unroll
      for (int m = 0; m < (1 << K); ++m) xs[G::word(base) + G::word(m * TL)] = v[i][0][m];
    } else {
#pragma unroll
      for (int m = 0; m < (1 << K); ++m) out[i * (1 << K) + m] = v[i][0][m];
    }
  }
  if constexpr (TL > 1) {
    __syncwarp();
    ksk_passes<SMALL, L1, L2, S0 + K>(xs, tw, q, nqi, ll, out);
  }
}

template <int L1, int L2, int W, int MINB>
__global__ void __launch_bounds__(32 * W, MINB) k_ntt_fwd_rows_ksk(Tables T, LimbSet S, NttAux A, KskFuse F, int nstage) {
  using G = KskGeo<L2>;
  extern __shared__ __align__(16) u64 sm[];
  constexpr size_t N = (size_t)1 << (L1 + L2);
  constexpr int GROUPS = (1 << L1) / G::KB;  // block groups of a limb
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, ll = lane % G::LPB, b = lane / G::LPB;
  const int t = S.limb_begin + blockIdx.y, pt = S.prime(t);
  const PrimeDev P = T.pr[pt];
  const u64 q = P.q;
  // warp tasks: (block group, ciphertext), ciphertext fastest; the last CTA may have idle warps
  const int task0 = blockIdx.x * W, task = task0 + warp;
  const int g0 = task0 / F.batch, gw = min(task / F.batch, GROUPS - 1);
  const bool live = task < GROUPS * F.batch;
  // the twiddles of block groups g0 .. g0 + nstage - 1, re-ordered for KskGeo's passes
  ulonglong2* tws = reinterpret_cast<ulonglong2*>(sm + W * 2 * G::XWORDS);
  {
    using R = Phase<L2>;
    const ulonglong2* src = T.psi2 + (size_t)pt * tw_stride(L1, L2) + (1 << L1);
    const int nblk = min(nstage, GROUPS - g0) * G::KB;
    for (int i = threadIdx.x; i < nblk << L2; i += 32 * W) {
      const int e = i & ((1 << L2) - 1);
      if (e == 0) continue;
      // slot e belongs to the pass from s0; its entry and group give the tree index 2^s (...) + ...
      int s0 = 0;
#pragma unroll
      for (int s = G::F; s < L2; s += 3)
        if (e >= 1 << s) s0 = s;
      const int r = e - (1 << s0), ent = (r >> s0) + 1, high = r & ((1 << s0) - 1);
      const int u = 31 - __clz(ent), mm = ent - (1 << u);
      const int tree = (((1 << s0) + high) << u) + mm;
      int slot = tree;
      if (tree >= R::M0) {
        const int s = 31 - __clz(tree), uu = s - R::K0, r2 = tree - (1 << s);
        slot = R::M0 + ((1 << uu) - 1 + (r2 & ((1 << uu) - 1))) * R::M0 + (r2 >> uu);
      }
      cp_async16(tws + i, src + ((size_t)(g0 * G::KB + (i >> L2)) << L2) + slot);
    }
  }
  const int k = task % F.batch;
  const size_t j0 = (size_t)(gw * G::KB) << L2;
  const int dn = A.own_dn;
  const int own = (A.own_alpha && t < A.own_limit) ? t / A.own_alpha : -1;
  const u64* src0 = S.limb(k * dn, t, N) + j0;  // digit j's run at + j part_stride
  const int j_first = own == 0 ? 1 : 0;
  u64* bufs = sm + warp * 2 * G::XWORDS;
  auto fetch = [&](int j, u64* dst) {
    const u64* src = src0 + (size_t)j * S.part_stride + 2 * lane;
    dst += G::run_word(2 * lane);
#pragma unroll
    for (int i = 0; i < G::PER / 2; ++i) cp_async16(dst + G::run_word(64 * i), src + i * 64);
  };
  grid_wait();
  if (live && j_first < dn) fetch(j_first, bufs);
  cp_async_commit();
  Acc128 ab[G::PER], aa[G::PER];
#pragma unroll
  for (int i = 0; i < G::PER; ++i) ab[i] = aa[i] = Acc128{0, 0};
  const ulonglong2* tw = tws + ((size_t)((gw - g0) * G::KB + b) << L2);
  const u64* kb = F.key + (size_t)pt * N + j0;
  // word pair i of the lane (words 2 i, 2 i + 1 of its PER consecutive ones) of digit j's key run (key_pair: the
  // lanes' pairs are consecutive)
  auto key_words = [&](int j, size_t part, ulonglong2 (&w)[G::PER / 2]) {
    const u64* at = kb + (size_t)j * F.key_digit_stride + part + 2 * key_pair(lane * (G::PER / 2));
#pragma unroll
    for (int i = 0; i < G::PER / 2; ++i) w[i] = __ldg(reinterpret_cast<const ulonglong2*>(at + 2 * key_pair(i)));
  };
  auto mac_words = [&](const u64 (&v)[G::PER], const ulonglong2 (&w)[G::PER / 2], Acc128 (&acc)[G::PER]) {
#pragma unroll
    for (int i = 0; i < G::PER / 2; ++i) {
      mac128(acc[2 * i], v[2 * i], w[i].x);
      mac128(acc[2 * i + 1], v[2 * i + 1], w[i].y);
    }
  };
  cp_async_wait_all();
  __syncthreads();
  if (!live) return;
  auto digits = [&](auto is_small) {
    constexpr bool SMALL = decltype(is_small)::value;
    for (int j = j_first, it = 0; j < dn; ++it) {
      const int next = j + 1 == own ? j + 2 : j + 1;
      u64* cur = bufs + (it & 1) * G::XWORDS;
      if (it) {
        cp_async_wait_all();
        __syncwarp();
      }
      if (next < dn) fetch(next, bufs + ((it + 1) & 1) * G::XWORDS);
      cp_async_commit();
      ulonglong2 wb[G::PER / 2], wa[G::PER / 2];
      key_words(j, 0, wb);
      key_words(j, F.key_a_offset, wa);
      u64 v[G::PER];
      ksk_passes<SMALL, L1, L2, 0>(cur + b * G::BS, tw, q, P.nqi, ll, v);
      if constexpr (!SMALL) {
#pragma unroll
        for (int i = 0; i < G::PER; ++i) v[i] = sub_if_above(sub_if_above(v[i], q * 6), q * 3);
      }
      mac_words(v, wb, ab);
      mac_words(v, wa, aa);
      j = next;
    }
  };
  if (fwd_small(q)) digits(std::true_type{});
  else digits(std::false_type{});
  const size_t wat = (size_t)lane * G::PER;  // this lane's words of the warp's run
  if (own >= 0) {  // the digit that owns limb t: the NTT-domain input itself
    const u64* src = F.d + (size_t)k * F.d_stride + (size_t)t * N + j0 + wat;
    u64 v[G::PER];
#pragma unroll
    for (int i = 0; i < G::PER; i += 2) {
      const ulonglong2 x = ldg2(src + i);
      v[i] = x.x;
      v[i + 1] = x.y;
    }
    ulonglong2 w[G::PER / 2];
    key_words(own, 0, w);
    mac_words(v, w, ab);
    key_words(own, F.key_a_offset, w);
    mac_words(v, w, aa);
  }
  u64* o0 = F.acc + (size_t)(2 * k) * F.acc_part_stride + (size_t)t * N + j0 + wat;
  u64* o1 = o0 + F.acc_part_stride;
#pragma unroll
  for (int i = 0; i < G::PER; i += 2) {
    stg2(o0 + i, ulonglong2{reduce128(ab[i], P), reduce128(ab[i + 1], P)});
    stg2(o1 + i, ulonglong2{reduce128(aa[i], P), reduce128(aa[i + 1], P)});
  }
}

// ---------------------------------------------------------------- inverse, row phase
// The forward row phase mirrored: the 2^K1 consecutive words of a lane's groups first, then the words
// 2^K1 apart.  Output left lazy (below 2^(L2+1) q for small primes, otherwise below 4q, see inv_pass).
template <bool SMALL, int L2>
__device__ __forceinline__ void inv_rows_passes(u64 (&v)[1][1 << Phase<L2>::K0], u64* xs, const ulonglong2* tw,
                                                const PrimeDev& P, int low) {
  using G = RowGeo<L2>;
  const u64 q = P.q;
#pragma unroll
  for (int i = 0; i < G::GP; ++i) {
    const int hi = i * G::M1 + low;
    u64 w[1][G::M1];
#pragma unroll
    for (int m = 0; m < G::M1; m += 2) {
      const ulonglong2 x = ldg2(xs + hi * G::GS + m);
      w[0][m] = x.x;
      w[0][m + 1] = x.y;
    }
    inv_pass<SMALL, 1, G::K1, 1>(w, q, P.nqi, [&](int u, int mm) {
      return tw[G::M0 + ((1 << u) - 1 + mm) * G::M0 + hi];
    });
#pragma unroll
    for (int m = 0; m < G::M1; m += 2) stg2(xs + hi * G::GS + m, ulonglong2{w[0][m], w[0][m + 1]});
  }
  __syncwarp();
#pragma unroll
  for (int m = 0; m < G::M0; ++m) v[0][m] = xs[m * G::GS + low];
  inv_pass<SMALL, 1 + G::K1, G::K0, 1>(v, q, P.nqi, [&](int u, int mm) { return tw[(1 << u) + mm]; });
}
// a block's words from global memory into the exchange buffer: j0 the block's first word of the limb
template <int L2>
__device__ __forceinline__ void inv_rows_load(const NttAux& A, const LimbSet& S, int part, int li, const u64* src, u64* xs,
                                              size_t j0, const PrimeDev& P, int low) {
  using G = RowGeo<L2>;
  if (A.pre_scale && li == S.limb_begin) {  // the first limb enters as e + x w
    const u64* ep = A.pre_e ? A.pre_e + part * A.pre_e_stride + j0 : nullptr;
#pragma unroll
    for (int k = 0; k < G::M0 / 2; ++k) {
      const int e = k * G::M1 + low;
      const ulonglong2 x = ldg2(src + 2 * e), c = ep ? ldg2(ep + 2 * e) : ulonglong2{0, 0};
      stg2(xs + G::pair(low) + G::pair(k * G::M1),
           ulonglong2{add_mod(c.x, shoup_mul(x.x, A.pre_w, A.pre_wsh, P.q), P.q),
                      add_mod(c.y, shoup_mul(x.y, A.pre_w, A.pre_wsh, P.q), P.q)});
    }
  } else if (odd_word(src)) {
#pragma unroll
    for (int m = 0; m < G::M0; ++m) xs[row_word<L2>(m, low)] = src[m * G::M1 + low];
  } else {
#pragma unroll
    for (int k = 0; k < G::M0 / 2; ++k) {
      const int e = k * G::M1 + low;
      cp_async16(xs + G::pair(low) + G::pair(k * G::M1), src + 2 * e);
    }
  }
}
template <int L1, int L2, int W, int MINB>
__global__ void __launch_bounds__(32 * W, MINB) k_ntt_inv_rows(Tables T, LimbSet S, NttAux A, int ppc) {
  using G = RowGeo<L2>;
  extern __shared__ __align__(16) u64 sm[];
  constexpr size_t N = (size_t)1 << (L1 + L2);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, low = lane % G::M1, b = lane / G::M1;
  const int pg = blockIdx.y / S.n_limbs, li = S.limb_begin + blockIdx.y % S.n_limbs;
  const int pi = S.prime(li);
  const PrimeDev P = T.pr[pi];
  const int blk = (blockIdx.x * W + warp) * G::PER + b;
  u64* xs = sm + warp * G::XWORDS + b * G::BS;
  ulonglong2* tw = reinterpret_cast<ulonglong2*>(sm + W * G::XWORDS) + (warp * G::PER << L2);  // the warp's blocks
  stage_twiddles<(G::PER << L2), 32>(tw, T.ipsi2 + (size_t)pi * tw_stride(L1, L2) + (1 << L1) + ((size_t)(blk - b) << L2),
                                     lane);
  tw += b << L2;
  const size_t j0 = (size_t)blk << L2;
  grid_wait();
  for (int part = pg * ppc; part < min((pg + 1) * ppc, S.n_parts); ++part) {
    if (own_limb(A, part, li)) continue;
    u64* a = S.limb(part, li, N) + j0;
    const u64* src = A.src ? A.src + part * A.src_stride + (size_t)li * N + j0 : a;
    inv_rows_load<L2>(A, S, part, li, src, xs, j0, P, low);
    cp_async_commit();
    cp_async_wait_all();
    __syncwarp();
    u64 v[1][G::M0];
    if (inv_small(P.q)) inv_rows_passes<true, L2>(v, xs, tw, P, low);
    else inv_rows_passes<false, L2>(v, xs, tw, P, low);
#pragma unroll
    for (int m = 0; m < G::M0; ++m) a[m * G::M1 + low] = v[0][m];
    __syncwarp();
  }
  cp_async_wait_all();
}

// ---------------------------------------------------------------- inverse, column phase (+ N^-1)
template <bool SMALL, int L1, int L2, int TH>
__device__ __forceinline__ void inv_cols_body(u64 (&w)[ColGeo<L1, TH>::GP][1][ColGeo<L1, TH>::M1], u64* a, u64* xs,
                                              const ulonglong2* tw, const PrimeDev& P, int low, int cg, u64 ni, u64 nip, u64 add) {
  using G = ColGeo<L1, TH>;
  const u64 q = P.q;
#pragma unroll
  for (int i = 0; i < G::GP; ++i) {
    const int hi = i * G::TPC + low;
    if constexpr (SMALL) {
#pragma unroll
      for (int m = 0; m < G::M1; ++m) w[i][0][m] = reduce_lazy(w[i][0][m], q, P.rc);
    }
    constexpr int GROUPS = 1 << (L1 - G::K1);
    inv_pass<SMALL, 1, G::K1, 1>(w[i], q, P.nqi, [&](int u, int mm) {
      return tw[GROUPS + ((1 << u) - 1 + mm) * GROUPS + hi];
    });
#pragma unroll
    for (int m = 0; m < G::M1; ++m) xs[(hi * (G::M1 + 1) + m) * G::COLS + cg] = w[i][0][m];
  }
  __syncthreads();
  u64 v[1][G::M0];
  if constexpr (G::THREE) {  // the middle pass, as in fwd_cols_passes
    const int hi = low >> 3;
    u64* x = xs + (hi * G::row(64) + (low & 7)) * G::COLS + cg;
#pragma unroll
    for (int m = 0; m < 8; ++m) v[0][m] = x[G::row(m * 8) * G::COLS];
    inv_pass<SMALL, 1 + G::K1, 3, 1>(v, q, P.nqi, [&](int u, int mm) { return tw[(8 << u) + (hi << u) + mm]; });
#pragma unroll
    for (int m = 0; m < 8; ++m) x[G::row(m * 8) * G::COLS] = v[0][m];
    __syncthreads();
  }
#pragma unroll
  for (int m = 0; m < G::M0; ++m) v[0][m] = xs[(G::row(m * G::TPC) + G::low_row(low)) * G::COLS + cg];
  if constexpr (SMALL && G::THREE) {  // nine doublings of 2q would pass 2^64
#pragma unroll
    for (int m = 0; m < G::M0; ++m) v[0][m] = reduce_lazy(v[0][m], q, P.rc);
  }
  inv_pass<SMALL, G::THREE ? 1 : 1 + G::K1, G::K0, 1>(v, q, P.nqi, [&](int u, int mm) { return tw[(1 << u) + mm]; });
#pragma unroll
  for (int m = 0; m < G::M0; ++m) a[(size_t)(m * G::TPC + low) << L2] = add_mod(shoup_mul(v[0][m], ni, nip, q), add, q);
}
template <int L1, int L2, int TH, int MINB>
__global__ void __launch_bounds__(TH, MINB) k_ntt_inv_cols(Tables T, LimbSet S, NttAux A) {
  using G = ColGeo<L1, TH>;
  extern __shared__ __align__(16) u64 sm[];
  constexpr size_t N = (size_t)1 << (L1 + L2);
  const int cg = threadIdx.x % G::COLS, low = threadIdx.x / G::COLS;
  const int y = blockIdx.y, part = y / S.n_limbs, li = S.limb_begin + y % S.n_limbs;
  if (own_limb(A, part, li)) return grid_wait();
  const int pi = S.prime(li);
  const PrimeDev P = T.pr[pi];
  u64* a = S.limb(part, li, N) + (size_t)blockIdx.x * G::COLS + cg;
  ulonglong2* tw = reinterpret_cast<ulonglong2*>(sm + G::XWORDS);
  stage_twiddles<1 << L1, TH>(tw, T.ipsi2 + (size_t)pi * tw_stride(L1, L2), threadIdx.x);
  cp_async_commit();
  grid_wait();
  u64 w[G::GP][1][G::M1];
#pragma unroll
  for (int i = 0; i < G::GP; ++i)
#pragma unroll
    for (int m = 0; m < G::M1; ++m) w[i][0][m] = a[(size_t)((i * G::TPC + low) * G::M1 + m) << L2];
  const int r = li - S.limb_begin;
  const u64 ni = A.post ? A.post[2 * r] : T.ninv[pi], nip = A.post ? A.post[2 * r + 1] : T.ninv_sh[pi];
  const u64 add = A.post_add ? A.post_add[r] : 0;
  cp_async_wait_all();
  __syncthreads();
  if (inv_small(P.q)) inv_cols_body<true, L1, L2, TH>(w, a, sm, tw, P, low, cg, ni, nip, add);
  else inv_cols_body<false, L1, L2, TH>(w, a, sm, tw, P, low, cg, ni, nip, add);
}

// ---------------------------------------------------------------- small rings: a whole limb per cluster
// N <= 2^13: a cluster of CTAs (1024 words and 128 threads each, 2048 and 256 at 2^13) holds a whole limb in shared memory
// and hands it from one phase to the other through distributed shared memory, so that one launch does both.  For a
// few limbs a launch costs its latency (5 us), not its work; a limb on one SM alone (N = 2^12: 10 us) loses
// what the launch saves.  8 words a thread (16 in the row phase at 2^13, where half of the threads work); the
// twiddles of the CTA's columns and blocks are staged with the first load.
template <int L1, int L2>
struct WholeGeo {
  static constexpr int CW = L1 + L2 == 13 ? 2048 : 1024;     // words of a CTA
  static constexpr int CS = (1 << (L1 + L2)) / CW;           // CTAs of a cluster
  static constexpr int TH = CW / 8, BLK = (1 << L1) / CS;    // threads, row blocks of a CTA
  using C = ColGeo<L1, TH>;
  using R = RowGeo<L2>;
  static_assert(C::COLS * CS == 1 << L2 && C::M0 == 8 && BLK * R::M1 <= TH, "8 words a thread in the column phase");
  static constexpr int YWORDS = BLK * R::BS;                 // words of the row layout, block after block
  static constexpr int XWORDS = (C::XWORDS + 1) & ~1;
  static constexpr int TW = (1 << L1) + (BLK << L2);
  static constexpr size_t SMEM = (size_t)(XWORDS + YWORDS) * 8 + (size_t)TW * 16;
};
template <int CS>
__device__ __forceinline__ void cluster_arrive() {
  if constexpr (CS > 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
template <int CS>
__device__ __forceinline__ void cluster_wait() {
  if constexpr (CS > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  else __syncthreads();
}
// the address of shared-memory word p in CTA `rank` of the cluster, and a store there
__device__ __forceinline__ uint32_t cluster_addr(const u64* p, uint32_t rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_store(uint32_t addr, u64 v) {
  asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(addr), "l"(v) : "memory");
}
template <int L1, int L2>
__global__ void __cluster_dims__(WholeGeo<L1, L2>::CS, 1, 1) __launch_bounds__(WholeGeo<L1, L2>::TH)
    k_ntt_inv_whole(Tables T, LimbSet S, NttAux A) {
  using W = WholeGeo<L1, L2>;
  using G = typename W::C;
  using R = typename W::R;
  extern __shared__ __align__(16) u64 sm[];
  constexpr size_t N = (size_t)1 << (L1 + L2);
  const int li = S.limb_begin + blockIdx.x / W::CS, rank = blockIdx.x % W::CS, part = blockIdx.y;
  if (own_limb(A, part, li)) return grid_wait();
  cluster_arrive<W::CS>();  // the others run before their shared memory is written
  const int pi = S.prime(li);
  const PrimeDev P = T.pr[pi];
  u64 *X = sm, *Y = sm + W::XWORDS;
  ulonglong2* tw = reinterpret_cast<ulonglong2*>(Y + W::YWORDS);
  const ulonglong2* src_tw = T.ipsi2 + (size_t)pi * tw_stride(L1, L2);
  stage_twiddles<1 << L1, W::TH>(tw, src_tw, threadIdx.x);
  stage_twiddles<(W::BLK << L2), W::TH>(tw + (1 << L1), src_tw + (1 << L1) + ((size_t)rank * W::BLK << L2), threadIdx.x);
  u64* a = S.limb(part, li, N);
  const u64* src = A.src ? A.src + part * A.src_stride + (size_t)li * N : a;
  const int low = threadIdx.x % R::M1, b = threadIdx.x / R::M1, blk = rank * W::BLK + b;  // row phase: block blk
  const int cg = threadIdx.x % G::COLS, clow = threadIdx.x / G::COLS;
  const bool row = b < W::BLK;
  u64* ys = Y + b * R::BS;
  grid_wait();
  if (row) inv_rows_load<L2>(A, S, part, li, src + ((size_t)blk << L2), ys, (size_t)blk << L2, P, low);
  cp_async_commit();
  const int r = li - S.limb_begin;
  const u64 ni = A.post ? A.post[2 * r] : T.ninv[pi], nip = A.post ? A.post[2 * r + 1] : T.ninv_sh[pi];
  const u64 add = A.post_add ? A.post_add[r] : 0;
  cp_async_wait_all();
  __syncthreads();
  auto body = [&](auto is_small) {
    constexpr bool SMALL = decltype(is_small)::value;
    u64 v[1][R::M0];
    if (row) inv_rows_passes<SMALL, L2>(v, ys, tw + (1 << L1) + (b << L2), P, low);
    cluster_wait<W::CS>();
    if (row) {
#pragma unroll
      for (int m = 0; m < R::M0; ++m) {  // row blk, column m 2^K1 + low
        const int col = m * R::M1 + low;
        u64* at = X + (blk + (blk >> G::K1)) * G::COLS + col % G::COLS;
        if constexpr (W::CS > 1) cluster_store(cluster_addr(at, col / G::COLS), v[0][m]);
        else *at = v[0][m];
      }
    }
    cluster_arrive<W::CS>();
    cluster_wait<W::CS>();
    u64 w[G::GP][1][G::M1];
#pragma unroll
    for (int i = 0; i < G::GP; ++i)
#pragma unroll
      for (int m = 0; m < G::M1; ++m) w[i][0][m] = X[((i * G::M1 + clow) * (G::M1 + 1) + m) * G::COLS + cg];
    // every thread writes back the words that it read: no barrier before inv_cols_body's exchange
    inv_cols_body<SMALL, L1, L2, W::TH>(w, a + rank * G::COLS + cg, X, tw, P, clow, cg, ni, nip, add);
  };
  if (inv_small(P.q)) body(std::true_type{});
  else body(std::false_type{});
}
template <int L1, int L2, int KIND>
__global__ void __cluster_dims__(WholeGeo<L1, L2>::CS, 1, 1) __launch_bounds__(WholeGeo<L1, L2>::TH)
    k_ntt_fwd_whole(Tables T, LimbSet S, NttAux A) {
  using W = WholeGeo<L1, L2>;
  using G = typename W::C;
  using R = typename W::R;
  extern __shared__ __align__(16) u64 sm[];
  constexpr size_t N = (size_t)1 << (L1 + L2);
  const int li = S.limb_begin + blockIdx.x / W::CS, rank = blockIdx.x % W::CS, part = blockIdx.y;
  if (own_limb(A, part, li)) return grid_wait();
  cluster_arrive<W::CS>();  // the others run before their shared memory is written
  const int pi = S.prime(li);
  const PrimeDev P = T.pr[pi];
  u64 *X = sm, *Y = sm + W::XWORDS;
  ulonglong2* tw = reinterpret_cast<ulonglong2*>(Y + W::YWORDS);
  const ulonglong2* src_tw = T.psi2 + (size_t)pi * tw_stride(L1, L2);
  stage_twiddles<1 << L1, W::TH>(tw, src_tw, threadIdx.x);
  stage_twiddles<(W::BLK << L2), W::TH>(tw + (1 << L1), src_tw + (1 << L1) + ((size_t)rank * W::BLK << L2), threadIdx.x);
  cp_async_commit();
  const int cg = threadIdx.x % G::COLS, clow = threadIdx.x / G::COLS;
  const int low = threadIdx.x % R::M1, b = threadIdx.x / R::M1, blk = rank * W::BLK + b;  // row phase: block blk
  const u64 bias = fwd_bias<L1 + L2>(P.q);
  u64* a = S.limb(part, li, N);
  // this thread's word of row clow; row m 2^K1 + clow is m N / M0 further
  const size_t c0 = ((size_t)clow << L2) + rank * G::COLS + cg;
  grid_wait();
  u64 v[1][G::M0];
  if constexpr (KIND == LOAD_PLAIN) {
    const u64* src = (A.src ? A.src + part * A.src_stride + (size_t)li * N : a) + c0;
#pragma unroll
    for (int m = 0; m < G::M0; ++m) v[0][m] = src[m * (N / G::M0)] + bias;
  } else {
    const int j = KIND == LOAD_MODUP ? part % A.own_dn : 0, lo = j * A.own_alpha;
    const int ns = KIND == LOAD_MODUP ? min(A.own_alpha, A.own_limit - lo) : KIND == LOAD_MODDOWN ? A.pconv_K : 0;
    const u64* base = (KIND == LOAD_MODUP     ? A.z + (size_t)(part / A.own_dn) * A.z_stride + (size_t)lo * N
                       : KIND == LOAD_MODDOWN ? A.pconv + (size_t)part * A.pconv_stride
                                              : A.spread) + c0;
    const u64* last = KIND != LOAD_MODUP && A.spread ? A.spread + (size_t)part * A.spread_stride + c0 : nullptr;
    FusedLoad<KIND> F;
    F.init(A, T, P, bias, j, li, ns);
    F.apply([&](auto word) {
#pragma unroll
      for (int m = 0; m < G::M0; ++m)
        v[0][m] = word([&](int t) { return t < ns ? base[(size_t)t * N + m * (N / G::M0)] : last[m * (N / G::M0)]; });
    });
  }
  cp_async_wait_all();
  __syncthreads();
  auto body = [&](auto is_small) {
    constexpr bool SMALL = decltype(is_small)::value;
    u64 o[G::GP][1][G::M1];
    fwd_cols_passes<SMALL, L1, W::TH>(v, X, tw, P.q, P.nqi, clow, cg, o);
    cluster_wait<W::CS>();
    const int col = rank * G::COLS + cg;
#pragma unroll
    for (int i = 0; i < G::GP; ++i)
#pragma unroll
      for (int m = 0; m < G::M1; ++m) {  // row c, this thread's column
        const int c = (i * G::M1 + clow) * G::M1 + m;
        u64* at = Y + (c % W::BLK) * R::BS + (col / R::M1) * R::GS + col % R::M1;
        if constexpr (W::CS > 1) cluster_store(cluster_addr(at, c / W::BLK), o[i][0][m]);
        else *at = o[i][0][m];
      }
    cluster_arrive<W::CS>();
    cluster_wait<W::CS>();
    if (b < W::BLK) {
      u64* ys = Y + b * R::BS;
      u64 w[1][R::M0];
#pragma unroll
      for (int m = 0; m < R::M0; ++m) w[0][m] = ys[m * R::GS + low];
      __syncwarp();
      fwd_rows_body<SMALL, L1, L2>(w, ys, tw + (1 << L1) + (b << L2), P, low);
      fwd_rows_store<SMALL, L1, L2>(ys, A, a + ((size_t)blk << L2), (uint32_t)blk << L2, (size_t)li * N + ((size_t)blk << L2),
                                    part, li, P, low);
    }
  };
  if (fwd_small(P.q)) body(std::true_type{});
  else body(std::false_type{});
}
template <int L1, int L2>
static bool launch_whole(const LimbSet& S, const Tables& T, cudaStream_t st, bool inverse, const NttAux& A,
                         const KskFuse* F) {
  if constexpr (L1 + L2 <= 13) {
    using W = WholeGeo<L1, L2>;
    const int n_prod = A.z ? std::min(A.own_alpha, A.own_limit) : A.pconv ? A.pconv_K : 0;
    if (F || !ntt_whole_limb(T, (size_t)S.n_limbs * S.n_parts, n_prod)) return false;
    static const bool attrs = [&] {
      allow_smem(k_ntt_inv_whole<L1, L2>, W::SMEM);
      allow_smem(k_ntt_fwd_whole<L1, L2, LOAD_PLAIN>, W::SMEM);
      allow_smem(k_ntt_fwd_whole<L1, L2, LOAD_MODUP>, W::SMEM);
      allow_smem(k_ntt_fwd_whole<L1, L2, LOAD_MODDOWN>, W::SMEM);
      allow_smem(k_ntt_fwd_whole<L1, L2, LOAD_SPREAD>, W::SMEM);
      return true;
    }();
    (void)attrs;
    const dim3 g((unsigned)(S.n_limbs * W::CS), (unsigned)S.n_parts);
    if (inverse) launch(k_ntt_inv_whole<L1, L2>, g, dim3(W::TH), W::SMEM, st, T, S, A);
    else if (A.z) launch(k_ntt_fwd_whole<L1, L2, LOAD_MODUP>, g, dim3(W::TH), W::SMEM, st, T, S, A);
    else if (A.pconv) launch(k_ntt_fwd_whole<L1, L2, LOAD_MODDOWN>, g, dim3(W::TH), W::SMEM, st, T, S, A);
    else if (A.spread) launch(k_ntt_fwd_whole<L1, L2, LOAD_SPREAD>, g, dim3(W::TH), W::SMEM, st, T, S, A);
    else launch(k_ntt_fwd_whole<L1, L2, LOAD_PLAIN>, g, dim3(W::TH), W::SMEM, st, T, S, A);
    HEDAP_LAUNCH_CHECK();
    prof_count_launches(1);
    return true;
  }
  return false;
}

// ---------------------------------------------------------------- dispatch
// A variant fixes the warps of a CTA and how many of them the register allocation must leave room for on an SM.
// The autotuner in ntt_tune() times every shape and keeps the fastest per role.
template <class Kernel>
static void allow_smem(Kernel kern, size_t bytes) {
  if (bytes > 48 * 1024)
    HEDAP_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
}
// fused row phase: 4 warps a CTA and 168 registers (3 CTAs an SM): 859 us for 8 x 12 digits at level 23, against
// 1195 us of the 128-thread CTAs with three barriers a digit
constexpr int kKskWarps = 4, kKskMinBlocks = 3;

// Output limbs per CTA of the shared-tile column phase: the number that minimises waves x (limbs + 0.3), the 0.3 limb
// being the staging of the tiles (an estimate, not timed apart); `ctas` CTAs per group of limbs, `slots` resident at a time.  One ciphertext at
// level 23 (N = 2^16): 9 limbs a CTA, 1.9 waves, where a fixed target of four waves gave 4 limbs and 4.4 waves.
inline int limbs_per_cta(size_t ctas, int limbs, size_t slots) {
  int best = 1;
  double best_cost = 1e300;
  for (int n = 1; n <= limbs; ++n) {
    const size_t all = ctas * (size_t)((limbs + n - 1) / n);
    const double cost = (double)((all + slots - 1) / slots) * (n + 0.3);
    if (cost < best_cost) {
      best_cost = cost;
      best = n;
    }
  }
  return best;
}
template <int L1, int L2, int WW, int WPS>
static void launch_pair(const LimbSet& S, const Tables& T, cudaStream_t st, bool inverse, const NttAux& A,
                        const KskFuse* F) {
  using RG = RowGeo<L2>;
  constexpr int TH = L1 == 9 ? 256 : std::min(32 * WW, (1 << L2) << Phase<L1>::K1);  // column phase: threads per CTA
  using CG = ColGeo<L1, TH>;
  constexpr int RW = std::min(WW, (1 << L1) / RG::PER);              // row phase: warps per CTA
  constexpr int CB = std::max(1, (WPS * 32 + TH - 1) / TH), RB = std::max(1, WPS / RW);
  const dim3 gc((unsigned)((1 << L2) / CG::COLS), (unsigned)(S.n_parts * S.n_limbs));
  const unsigned rx = (unsigned)((1 << L1) / RG::PER / RW);
  constexpr size_t smem_x = (size_t)CG::XWORDS * 8, smem_c = smem_x + ((size_t)16 << L1);
  constexpr size_t smem_r = (size_t)RW * (RG::XWORDS * 8 + (RG::PER * (size_t)16 << L2));
  if (gc.y == 0) return;
  // parts of one limb that a warp takes in turn: as many as leave about four waves of warps
  const size_t warps1 = (size_t)rx * RW * S.n_limbs * S.n_parts;
  const int ppc = (int)std::max<size_t>(1, std::min<size_t>(std::min(S.n_parts, 8), warps1 / ((size_t)152 * WPS * 4)));
  const dim3 gr(rx, (unsigned)(((S.n_parts + ppc - 1) / ppc) * S.n_limbs));
  // the first phase applies src / z / spread; the second runs in place on S (or into fin_dst)
  NttAux A2 = A;
  A2.src = nullptr;
  A2.z = nullptr;
  A2.spread = nullptr;
  A2.pconv = nullptr;
  if (!inverse) {
    // staged tiles: the digit's limbs (ModUp), the special limbs (ModDown, plus the last limb when a
    // rescale is fused) or the last limb (rescale); at most 3 products per word in the load
    const int n_prod = A.z ? std::min(A.own_alpha, A.own_limit) : A.pconv ? A.pconv_K : 0;
    const int nt = n_prod + (!A.z && A.spread ? 1 : 0);
    if (nt >= 1 && n_prod <= 3 && !A.src) {
      const size_t smem = smem_x + (size_t)nt * CG::TILE * 8;
      const int lpc = limbs_per_cta((size_t)gc.x * S.n_parts, S.n_limbs, 152 * std::min<size_t>(CB, 232448 / (smem + 1024)));
      const dim3 g2(gc.x, (unsigned)(S.n_parts * ((S.n_limbs + lpc - 1) / lpc)));
      constexpr size_t smem_max = smem_x + (size_t)4 * CG::TILE * 8;
      static const bool attrs = [&] {
        allow_smem(k_ntt_fwd_cols_shared<L1, L2, TH, CB, LOAD_MODUP>, smem_max);
        allow_smem(k_ntt_fwd_cols_shared<L1, L2, TH, CB, LOAD_MODDOWN>, smem_max);
        allow_smem(k_ntt_fwd_cols_shared<L1, L2, TH, CB, LOAD_SPREAD>, smem_max);
        return true;
      }();
      (void)attrs;
      if (A.z) launch(k_ntt_fwd_cols_shared<L1, L2, TH, CB, LOAD_MODUP>, g2, dim3(TH), smem, st, T, S, A, lpc);
      else if (A.pconv) launch(k_ntt_fwd_cols_shared<L1, L2, TH, CB, LOAD_MODDOWN>, g2, dim3(TH), smem, st, T, S, A, lpc);
      else launch(k_ntt_fwd_cols_shared<L1, L2, TH, CB, LOAD_SPREAD>, g2, dim3(TH), smem, st, T, S, A, lpc);
    } else if (n_prod > 3) {
      constexpr int WB = std::max(1, (L1 == 9 ? 16 : 12) * 32 / TH);
      if (A.z) launch(k_ntt_fwd_cols_wide<L1, L2, TH, WB, LOAD_MODUP>, gc, dim3(TH), smem_x, st, T, S, A);
      else launch(k_ntt_fwd_cols_wide<L1, L2, TH, WB, LOAD_MODDOWN>, gc, dim3(TH), smem_x, st, T, S, A);
    } else {
      launch(k_ntt_fwd_cols<L1, L2, TH, CB>, gc, dim3(TH), smem_c, st, T, S, A);
    }
    if (F) {
      using KG = KskGeo<L2>;
      constexpr int GROUPS = (1 << L1) / KG::KB;
      const int tasks = GROUPS * F->batch;
      const int nstage = std::min(kKskWarps, (kKskWarps - 2 + F->batch) / F->batch + 1);  // block groups a CTA may touch
      const size_t smem = (size_t)kKskWarps * 2 * KG::XWORDS * 8 + ((size_t)nstage * KG::KB << L2) * 16;
      static const bool attr_k = [&] {
        allow_smem(k_ntt_fwd_rows_ksk<L1, L2, kKskWarps, kKskMinBlocks>,
                   (size_t)kKskWarps * 2 * KG::XWORDS * 8 + ((size_t)kKskWarps * KG::KB << L2) * 16);
        return true;
      }();
      (void)attr_k;
      const dim3 gk((unsigned)((tasks + kKskWarps - 1) / kKskWarps), (unsigned)S.n_limbs);
      launch(k_ntt_fwd_rows_ksk<L1, L2, kKskWarps, kKskMinBlocks>, gk, dim3(32 * kKskWarps), smem, st, T, S, A2, *F, nstage);
    } else {
      static const bool attrs = [&] {
        allow_smem(k_ntt_fwd_rows<L1, L2, RW, RB>, smem_r);
        return true;
      }();
      (void)attrs;
      launch(k_ntt_fwd_rows<L1, L2, RW, RB>, gr, dim3(32 * RW), smem_r, st, T, S, A2, ppc);
    }
  } else {
    static const bool attrs = [&] {
      allow_smem(k_ntt_inv_rows<L1, L2, RW, RB>, smem_r);
      return true;
    }();
    (void)attrs;
    launch(k_ntt_inv_rows<L1, L2, RW, RB>, gr, dim3(32 * RW), smem_r, st, T, S, A, ppc);
    launch(k_ntt_inv_cols<L1, L2, TH, CB>, gc, dim3(TH), smem_c, st, T, S, A2);
  }
  HEDAP_LAUNCH_CHECK();
  prof_count_launches(2);
}

template <int L1, int L2>
static void launch_variant(int v, const LimbSet& S, const Tables& T, cudaStream_t st, bool inverse,
                           const NttAux& A, const KskFuse* F) {
  if (launch_whole<L1, L2>(S, T, st, inverse, A, F)) return;
  if (v % kNttShapes == 0) launch_pair<L1, L2, 4, 16>(S, T, st, inverse, A, F);
  else launch_pair<L1, L2, 4, 20>(S, T, st, inverse, A, F);
}

// one launch pair of the transform at N = 2^log_n (log_n 10 .. 17) with launch shape v; the
// instantiations are spread over the ntt_inst_*.cu translation units so that they compile in parallel
void ntt_launch(int log_n, int v, const LimbSet& S, const Tables& T, cudaStream_t st, bool inverse,
                const NttAux& A, const KskFuse* F);

}  // namespace hedap
