// Host orchestration of the CKKS operations of Sec. 2.1 over the device
// kernels: Add/Sub, Mul_C (tensor product + hybrid key switching), rescale,
// Mul_P by constants, Galois automorphisms (rotation, conjugation).
// Every operation works on a batch of ciphertexts at one level and scale (a
// single ciphertext is a batch of one); each launch covers the whole batch.
// Ciphertexts stay in the NTT domain; temporaries are stream-ordered on the
// context's stream.
#include <cmath>

#include "internal.cuh"
#include "kernels.cuh"
#include "profiler.cuh"

namespace hedap {

static LimbSet qset(u64* base, size_t part_stride, int n_parts, int first, int count, int prime_offset = 0) {
  return LimbSet{base, part_stride, n_parts, first, count, INT_MAX, prime_offset, 0};
}

std::unique_ptr<Ct> ct_alloc(Ctx& C, int level, int batch) {
  if (level < 0 || level > C.L()) throw Error(HEDAP_ERR_LEVEL, "level out of range");
  if (batch < 1 || batch > kMaxBatch) throw Error(HEDAP_ERR_ARG, "batch must lie in [1, 16]");
  auto c = std::make_unique<Ct>();
  c->owner = &C;
  c->N = C.N;
  c->cap = level + 1;
  c->level = level;
  c->batch = batch;
  c->scale = C.scale;
  c->buf = DevBuf(2 * (size_t)batch * (level + 1) * C.N, C.stream);
  return c;
}

// copy limbs 0..level of every part of a into a new (packed) batch
std::unique_ptr<Ct> ct_copy(Ctx& C, const Ct& a, int level) {
  if (level > a.level) throw Error(HEDAP_ERR_LEVEL, "cannot raise the level by copying");
  auto c = ct_alloc(C, level, a.batch);
  c->scale = a.scale;
  k_copy_parts(C, a.part(0), a.part_stride(), c->part(0), c->part_stride(), a.parts(), (size_t)(level + 1) * C.N);
  return c;
}
std::unique_ptr<Ct> ev_drop(Ctx& C, const Ct& a, int level) {
  if (level < 0) throw Error(HEDAP_ERR_LEVEL, "negative level");
  return ct_copy(C, a, level);
}

std::unique_ptr<Ct> batch_pack(Ctx& C, const std::vector<const Ct*>& cts) {
  if (cts.empty()) throw Error(HEDAP_ERR_ARG, "empty batch");
  const Ct& f = *cts[0];
  int total = 0;
  for (const Ct* c : cts) {
    if (c->level != f.level || c->scale != f.scale) throw Error(HEDAP_ERR_ARG, "batched ciphertexts differ in level or scale");
    total += c->batch;
  }
  auto b = ct_alloc(C, f.level, total);
  b->scale = f.scale;
  int at = 0;
  for (const Ct* c : cts) {
    k_copy_parts(C, c->part(0), c->part_stride(), b->part(2 * at), b->part_stride(), c->parts(),
                 (size_t)(f.level + 1) * C.N);
    at += c->batch;
  }
  return b;
}
std::unique_ptr<Ct> batch_slice(Ctx& C, const Ct& b, int first, int count) {
  if (first < 0 || count < 1 || first + count > b.batch) throw Error(HEDAP_ERR_ARG, "batch slice out of range");
  auto c = ct_alloc(C, b.level, count);
  c->scale = b.scale;
  k_copy_parts(C, b.part(2 * first), b.part_stride(), c->part(0), c->part_stride(), 2 * count,
               (size_t)(b.level + 1) * C.N);
  return c;
}
std::unique_ptr<Ct> batch_unpack(Ctx& C, const Ct& b, int k) {
  if (k < 0 || k >= b.batch) throw Error(HEDAP_ERR_ARG, "batch index out of range");
  auto c = ct_alloc(C, b.level, 1);
  c->scale = b.scale;
  k_copy_parts(C, b.part(2 * k), b.part_stride(), c->part(0), c->part_stride(), 2, (size_t)(b.level + 1) * C.N);
  return c;
}

static void check_scales(double a, double b) {
  if (std::fabs(a / b - 1.0) > 1e-12) throw Error(HEDAP_ERR_SCALE, "operand scales differ");
}
static void check_batches(const Ct& a, const Ct& b) {
  if (a.batch != b.batch) throw Error(HEDAP_ERR_ARG, "operands have different batch sizes");
}

std::unique_ptr<Ct> ev_add(Ctx& C, const Ct& a, const Ct& b, bool sub) {
  const int l = std::min(a.level, b.level);
  check_scales(a.scale, b.scale);
  check_batches(a, b);
  auto o = ct_alloc(C, l, a.batch);
  o->scale = a.scale;
  k_add_sub(C, a.part(0), a.part_stride(), b.part(0), b.part_stride(), o->part(0), o->part_stride(), a.parts(),
            l + 1, sub);
  return o;
}

// ------------------------------------------------------------------ level constants
const LevelConsts& level_consts(Ctx& C, int l) {
  auto it = C.lc.find(l);
  if (it != C.lc.end()) return *it->second;
  auto L = std::make_unique<LevelConsts>();
  const int a = C.alpha, dn = C.dnum(l), K = C.n_p, ext = l + 1 + K;
  const u64* q = C.primes.data();
  auto prime_of_ext = [&](int t) { return t <= l ? q[t] : q[C.n_q + (t - l - 1)]; };
  const size_t nb = (size_t)dn * a * ext;  // qhat table size; its Shoup companions follow it
  std::vector<u64> v(2 * (l + 1) + 2 * nb, 0);
  for (int j = 0; j < dn; ++j) {
    const int lo = j * a, hi = std::min(lo + a, l + 1);
    for (int i = lo; i < hi; ++i) {
      u64 h = 1;
      for (int m = lo; m < hi; ++m)
        if (m != i) h = h_mulmod(h, q[m] % q[i], q[i]);
      const u64 inv = h_invmod(h, q[i]);
      v[i] = inv;
      v[(l + 1) + i] = h_shoup(inv, q[i]);
      for (int t = 0; t < ext; ++t) {
        const u64 pt = prime_of_ext(t);
        u64 hm = 1 % pt;
        for (int m = lo; m < hi; ++m)
          if (m != i) hm = h_mulmod(hm, q[m] % pt, pt);
        v[2 * (l + 1) + ((size_t)j * a + (i - lo)) * ext + t] = hm;
        v[2 * (l + 1) + nb + ((size_t)j * a + (i - lo)) * ext + t] = h_shoup(hm, pt);
      }
    }
  }
  L->modup = DevBuf(v.size(), C.stream);
  HEDAP_CUDA(cudaMemcpyAsync(L->modup.p, v.data(), v.size() * 8, cudaMemcpyHostToDevice, C.stream));
  // the key switch's fused ModUp: every factor divided by the key's scale (Ctx::key_scale), as pairs for
  // mont_mul_lazy; the factor of the folded limb becomes 1 and is marked by a second word 0
  std::vector<u64> vk(2 * nb, 0);
  double products = 0;
  const int T = C.total_primes();
  for (int j = 0; j < dn; ++j) {
    const int lo = j * a, hi = std::min(lo + a, l + 1);
    for (int t = 0; t < ext; ++t) {
      if (t >= lo && t < hi) continue;  // the digit's own limbs are not converted
      const int gt = t <= l ? t : C.n_q + (t - l - 1);
      const u64 pt = prime_of_ext(t), un = C.key_unscale[(size_t)j * T + gt];
      const int i0 = C.key_scale_i0[(size_t)j * T + gt];
      for (int i = lo; i < hi; ++i) {
        const size_t at = 2 * (l + 1) + ((size_t)j * a + (i - lo)) * ext + t;
        const size_t to = at - 2 * (l + 1);
        const u64 f = h_mulmod(v[at], un, pt);
        vk[to] = h_mont(f, pt);
        vk[to + nb] = (i == i0 && f == 1) ? 0 : h_mont(vk[to], pt);
        products += vk[to + nb] ? 1 : 0;
      }
    }
  }
  L->modup_products = products;
  L->modup_ks = DevBuf(vk.size(), C.stream);
  HEDAP_CUDA(cudaMemcpyAsync(L->modup_ks.p, vk.data(), vk.size() * 8, cudaMemcpyHostToDevice, C.stream));
  // the key switch's inverse NTT ends with N^-1 qhat_i^-1 instead of N^-1, so that its output is the
  // first factor [x_i qhat_i^-1]_{q_i} of the fast basis conversion
  std::vector<u64> post(2 * (l + 1));
  for (int i = 0; i <= l; ++i) {
    post[2 * i] = h_mulmod(h_invmod(C.N % q[i], q[i]), v[i], q[i]);
    post[2 * i + 1] = h_shoup(post[2 * i], q[i]);
  }
  L->intt_post = DevBuf(post.size(), C.stream);
  HEDAP_CUDA(cudaMemcpyAsync(L->intt_post.p, post.data(), post.size() * 8, cudaMemcpyHostToDevice, C.stream));
  HEDAP_CUDA(cudaStreamSynchronize(C.stream));
  if (l >= 1) {
    const u64 ql = q[l];
    std::vector<u64> r(3 * (size_t)l);
    for (int i = 0; i < l; ++i) {
      L->rescale.ql_mod[i] = ql % q[i];
      L->rescale.inv[i] = h_invmod(ql % q[i], q[i]);
      L->rescale.inv_sh[i] = h_shoup(L->rescale.inv[i], q[i]);
      r[i] = L->rescale.ql_mod[i];
      r[l + i] = h_mont(L->rescale.inv[i], q[i]);
      r[2 * l + i] = h_mont(r[l + i], q[i]);
    }
    L->d_rescale = DevBuf(r.size(), C.stream);
    HEDAP_CUDA(cudaMemcpyAsync(L->d_rescale.p, r.data(), r.size() * 8, cudaMemcpyHostToDevice, C.stream));
    // ModDown fused with this level's rescale (ks_moddown_rescale)
    const int K = C.n_p;
    auto P_mod = [&](u64 m) {
      u64 v = 1 % m;
      for (int k = 0; k < K; ++k) v = h_mulmod(v, q[C.n_q + k] % m, m);
      return v;
    };
    std::vector<u64> w(2 * (size_t)l);
    for (int i = 0; i < l; ++i) {
      w[i] = h_mont(h_mulmod(h_invmod(P_mod(q[i]), q[i]), L->rescale.inv[i], q[i]), q[i]);
      w[l + i] = h_mont(w[i], q[i]);
    }
    L->d_mdr = DevBuf(w.size(), C.stream);
    HEDAP_CUDA(cudaMemcpyAsync(L->d_mdr.p, w.data(), w.size() * 8, cudaMemcpyHostToDevice, C.stream));
    MdrLast& M = L->mdr_last;
    M = MdrLast{};
    M.K = std::min(K, 8);
    const u64 pinv = h_invmod(P_mod(ql), ql);
    for (int k = 0; k < M.K; ++k) {
      const u64 pk = q[C.n_q + k];
      M.f[k] = h_invmod(pk % ql, ql);
      M.fs[k] = h_shoup(M.f[k], ql);
    }
    const u64 halfq = h_mulmod((P_mod(ql) + ql - 1) % ql, h_invmod(2, ql), ql);  // floor(P/2) mod q_l
    M.off = (ql - h_mulmod(halfq, pinv, ql)) % ql;
    M.pinv = pinv;
    M.pinv_sh = h_shoup(pinv, ql);
    std::vector<u64> mp(2 + 2 * (size_t)M.K);
    mp[0] = h_invmod(C.N % ql, ql);
    mp[1] = h_shoup(mp[0], ql);
    for (int k = 0; k < M.K; ++k) {
      mp[2 + 2 * k] = C.mdr_post[2 * k];
      mp[3 + 2 * k] = C.mdr_post[2 * k + 1];
    }
    L->mdr_post = DevBuf(mp.size(), C.stream);
    HEDAP_CUDA(cudaMemcpyAsync(L->mdr_post.p, mp.data(), mp.size() * 8, cudaMemcpyHostToDevice, C.stream));
    HEDAP_CUDA(cudaStreamSynchronize(C.stream));
  }
  auto& ref = *L;
  C.lc[l] = std::move(L);
  return ref;
}

// ------------------------------------------------------------------ key switching
// Hybrid key switching (Han-Ki 2020) of a batch of polynomials with the key for
// `galois`: iNTT, ModUp of every digit to Q_l u P, NTT, inner product with the
// key digits (each key word read once for the batch), iNTT of the P limbs,
// ModDown (rounded division by P), NTT.  The ModUp is fused into the transforms:
// the inverse NTT reads d out of place and ends with N^-1 qhat_i^-1, the forward
// NTT of each extended limb loads the basis conversion directly, and a digit's
// own limbs (whose NTT is d itself) are neither converted nor transformed.
//
// An operation's temporaries come from one allocation, in which what ends with the inner product gives its place
// to ModDown's workspace: on a small ring each allocation with its release costs the host a good part of a launch.
// What is written last is a workspace until then, so that an operation holds no more than with an allocation each: the
// coefficient-domain limbs of the ModUp lie in the sums' place (read before the first sum is stored), the polynomial
// that is switched, and ModDown's transform where the finishing store adds nothing to it, in the result's.
struct Scratch {
  DevBuf buf;
  size_t at = 0;  // set back by the caller once what lies above has been used
  Scratch(Ctx& C, size_t words) : buf(words, C.stream) {}
  u64* take(size_t words) {
    if (at + words > buf.words) throw Error(HEDAP_ERR_ARG, "scratch exhausted");
    u64* p = buf.p + at;
    at += words;
    return p;
  }
};
// words of ks_modup's extended digits; its coefficient-domain limbs (batch (l + 1) N words) fit in the sums' place
static size_t digit_words(const Ctx& C, int batch, int l) {
  return (size_t)batch * C.N * C.dnum(l) * (l + 1 + C.n_p);
}
static size_t acc_words(const Ctx& C, int batch, int l) { return (size_t)batch * 2 * (l + 1 + C.n_p) * C.N; }
// ModUp of a batch of NTT-domain polynomials d (member stride d_stride) into NTT-domain extended
// digits y [B][dn][ext][N] (a digit's own limbs are left out: they are d itself; with fuse, y holds the column phase's
// output).  dc: workspace of B (l + 1) N words, free again before the inner product.
static void ks_modup(Ctx& C, const u64* d, size_t d_stride, int batch, int l, u64* dc, u64* y,
                     const KskFuse* fuse = nullptr) {
  const size_t N = C.N, nl = (size_t)l + 1;
  const int ext = l + 1 + C.n_p, dn = C.dnum(l);
  const LevelConsts& LC = level_consts(C, l);
  NttAux inv{};
  inv.src = d;
  inv.src_stride = d_stride;
  inv.post = LC.intt_post.p;  // dc: z_i = [x_i qhat_i^-1]_{q_i}, coefficient domain
  ntt_inverse(C.tab, qset(dc, nl * N, batch, 0, l + 1), C.stream, &inv);
  NttAux up{};
  up.own_alpha = C.alpha;
  up.own_dn = dn;
  up.own_limit = l + 1;
  up.z = dc;
  up.z_stride = nl * N;
  up.bconv = LC.modup_ks.p;  // factors divided by the key's folded ones
  up.bconv_b_offset = (size_t)dn * C.alpha * ext;
  up.ext = ext;
  up.z_products = LC.modup_products * batch * (double)N;
  ntt_forward(C.tab, LimbSet{y, (size_t)ext * N, batch * dn, 0, ext, l + 1, 0, C.n_q}, C.stream, &up, fuse);
}
static const DevBuf& key_for(Ctx& C, u64 galois) {
  auto it = C.keys.find(galois);
  if (it == C.keys.end()) {
    gen_galois_key(C, galois);
    it = C.keys.find(galois);
  }
  return it->second;
}
// iNTT of the P limbs of the key-switch sums acc [batch][2][ext][N], ModDown, NTT, written to / added
// into out; v: workspace of moddown_words
static size_t moddown_words(const Ctx& C, int batch, int l) { return (size_t)batch * 2 * (l + 1) * C.N; }
// several rotations of one ciphertext at once: sums acc [count][batch][2][ext][N], rotation r's ModDown to out[r] with
// sigma_gs[r](c0) (part stride c0_stride) added to the even parts, gathered by the finishing store
struct RotationOut {
  const u64* c0;
  size_t c0_stride;
  int count;
  u64* out[kKskRotations];
  u64 gs[kKskRotations];
};
static void ks_moddown(Ctx& C, u64* acc, u64* v, int batch, int l, u64* out, size_t out_stride, bool acc0, bool acc1,
                       const RotationOut* R = nullptr) {
  const int parts = 2 * batch * (R ? R->count : 1);
  const size_t N = C.N, nl = (size_t)l + 1;
  const int K = C.n_p, ext = l + 1 + K;
  // ModDown: the special-prime limbs (at most 8) to the coefficient domain, ending with N^-1 phinv_k, the conversion
  // into every Q prime fused into the forward NTT's load, and (acc - v) P^-1 (+ out) fused into its store
  NttAux inv{};
  inv.post = C.d_moddown2.p;
  inv.post_add = C.d_moddown2.p + 2 * K + 1;
  ntt_inverse(C.tab, LimbSet{acc, (size_t)ext * N, parts, l + 1, K, l + 1, 0, C.n_q}, C.stream, &inv);
  const u64* Pinv = C.d_moddown2.p + 3 * K + 1 + 2 * (size_t)K * C.n_q;
  NttAux fw{};
  fw.pconv = acc + nl * N;
  fw.pconv_stride = (size_t)ext * N;
  fw.pconv_K = K;
  fw.pconv_ld = C.n_q;
  fw.pconv_phat = C.d_moddown2.p + 3 * K + 1;
  fw.pconv_phat_b = C.d_moddown2.p + 3 * K + 1 + (size_t)K * C.n_q;
  fw.pconv_half = C.d_moddown.p + 3 * K + (size_t)K * C.n_q + 2 * (size_t)C.n_q;
  fw.fin_dst = out;
  fw.fin_dst_stride = out_stride;
  fw.fin_c = acc;
  fw.fin_c_stride = (size_t)ext * N;
  fw.fin_w = Pinv;
  fw.fin_wb = Pinv + C.n_q;
  fw.fin_acc_even = acc0 ? 1 : 0;
  fw.fin_acc_odd = acc1 ? 1 : 0;
  if (R) {
    fw.fin_d = R->c0;
    fw.fin_d_stride = R->c0_stride;
    fw.fin_per = 2 * batch;
    std::copy_n(R->out, R->count, fw.fin_dsts);
    std::copy_n(R->gs, R->count, fw.fin_gs);
  }
  ntt_forward(C.tab, qset(v, nl * N, parts, 0, l + 1), C.stream, &fw);
}

// The key switch up to the inner product: iNTT of d, the extended digits' forward transform with the
// key inner product fused into its second phase (the transformed digits are never stored).  The
// sums acc [batch][2][ext][N] (NTT domain) go to acc; y: workspace of digit_words.
static void ks_inner(Ctx& C, const u64* d, size_t d_stride, int batch, int l, u64 galois, u64* acc, u64* y) {
  const DevBuf& key = key_for(C, galois);
  const int T = C.total_primes();
  if (C.tab.small_routes && C.log_n <= 13 && C.alpha <= 3 && ((size_t)batch * (l + 1 + C.n_p) << C.log_n) <= (size_t)1 << 18) {
    // a small ring's few limbs: the digits transformed in one launch, all of them at once, and the inner product in
    // a second; fused, one warp for 256 words would walk the digits one after the other with fewer than 1024
    // warps on the GPU.  HMult, separate against fused (us), words a digit over the batch: 12 digits, 2^10 27 K
    // 26.8 36.5, 213 K 56.1 54.4; 2^12 160 K 44.2 50.8, 319 K 73.8 71.2; 2^13 213 K 64.4 65.8, 426 K 104.9 99.5;
    // 4 digits, 2^11 41 K 28.7 30.5, 328 K 46.3 45.4; 3 digits, 2^12 197 K 37.8 38.1, 786 K 82.5 76.4.
    ks_modup(C, d, d_stride, batch, l, acc, y);
    KskInnerArgs A;
    A.count = 1;
    A.key[0] = key.p;
    A.acc[0] = acc;
    A.g[0] = 1;
    k_ksk_inner(C, y, d, d_stride, A, batch, l);
    return;
  }
  KskFuse F;
  F.d = d;
  F.d_stride = d_stride;
  F.key = key.p;
  F.key_digit_stride = (size_t)2 * T * C.N;
  F.key_a_offset = (size_t)T * C.N;
  F.acc = acc;
  F.acc_part_stride = (size_t)(l + 1 + C.n_p) * C.N;
  F.batch = batch;
  ks_modup(C, d, d_stride, batch, l, acc, y, &F);
}

// One key switch: the inner product, then ModDown.
void key_switch(Ctx& C, const u64* d, size_t d_stride, int batch, int l, u64 galois, u64* out, size_t out_stride,
                bool acc0, bool acc1) {
  Scratch S(C, acc_words(C, batch, l) + std::max(digit_words(C, batch, l), moddown_words(C, batch, l)));
  u64* acc = S.take(acc_words(C, batch, l));
  const size_t mark = S.at;
  ks_inner(C, d, d_stride, batch, l, galois, acc, S.take(digit_words(C, batch, l)));
  S.at = mark;
  ks_moddown(C, acc, S.take(moddown_words(C, batch, l)), batch, l, out, out_stride, acc0, acc1);
}

// ModDown of the key-switch sums acc added to e (NTT domain, level l, part stride e_stride), followed
// by the rescale by q_l, written to out (level l - 1).  Separately, ModDown transforms its conversion
// v back over the l + 1 limbs and the rescale transforms the spread w of the centred last limb over
// the l remaining ones; the transforms are linear, so
//   ((e + (acc - NTT(v)) P^-1) - NTT(w)) q_l^-1 = acc (P q_l)^-1 + (e - NTT(v P^-1 + w)) q_l^-1
// and one forward transform of v P^-1 + w over l limbs does both (v P^-1 is the conversion with
// constants scaled by P^-1).  The last limb's coefficients come first: INTT(e_l + acc_l P^-1) minus
// the conversion of the special limbs into q_l scaled by P^-1.  Every residue equals that of ModDown
// followed by the rescale.
// x: workspace of mdr_words; the transform runs in out's place (2 batch parts of l limbs, out_stride >= l N apart).
static size_t mdr_words(const Ctx& C, int batch) { return (size_t)2 * batch * C.N; }
static void ks_moddown_rescale(Ctx& C, u64* acc, u64* x, int batch, int l, const u64* e, size_t e_stride, u64* out,
                               size_t out_stride, bool negate = false) {
  const size_t N = C.N;
  const int K = C.n_p, ext = l + 1 + K, nq = C.n_q;
  const LevelConsts& LC = level_consts(C, l);
  // limb l of the sums enters as e_l + acc_l P^-1 and the special limbs, which follow it, end with
  // N^-1 phinv_k: one inverse transform of K + 1 limbs a part
  NttAux inv{};
  inv.post = LC.mdr_post.p;
  inv.post_add = C.d_moddown2.p + 2 * K;  // 0 for limb l, c_k for the special limbs
  inv.pre_scale = 1;
  inv.pre_e = e + (size_t)l * N;
  inv.pre_e_stride = e_stride;
  inv.pre_w = LC.mdr_last.pinv;
  inv.pre_wsh = LC.mdr_last.pinv_sh;
  ntt_inverse(C.tab, LimbSet{acc, (size_t)ext * N, 2 * batch, l, K + 1, l + 1, 0, C.n_q}, C.stream, &inv);
  k_mdr_last_coef(C, acc + (size_t)l * N, (size_t)ext * N, x, 2 * batch, l, LC.mdr_last);
  NttAux fw{};
  fw.pconv = acc + (size_t)(l + 1) * N;
  fw.pconv_stride = (size_t)ext * N;
  fw.pconv_K = K;
  fw.pconv_ld = nq;
  fw.pconv_phat = C.d_mdr.p;
  fw.pconv_phat_b = C.d_mdr.p + (size_t)K * nq;
  fw.pconv_half = C.d_mdr.p + 2 * (size_t)K * nq;
  fw.spread = x;
  fw.spread_stride = N;
  fw.spread_sub = LC.d_rescale.p;
  fw.spread_prime = l;
  fw.fin_dst = out;
  fw.fin_dst_stride = out_stride;
  fw.fin_c = acc;
  fw.fin_c_stride = (size_t)ext * N;
  fw.fin_w = LC.d_mdr.p;
  fw.fin_wb = LC.d_mdr.p + l;
  fw.fin_e = e;
  fw.fin_e_stride = e_stride;
  fw.fin_w2 = LC.d_rescale.p + l;
  fw.fin_w2b = LC.d_rescale.p + 2 * l;
  fw.fin_neg = negate ? 1 : 0;
  ntt_forward(C.tab, qset(out, out_stride, 2 * batch, 0, l), C.stream, &fw);
}

// Rotations of one (batched) ciphertext by several Galois elements sharing one ModUp of its
// second part (hoisting): the extended digits of c1 are formed once, and each rotation applies its
// automorphism to them inside the inner product.  The result differs from ev_galois (which
// converts the rotated c1) by multiples of the digit moduli in the extended basis, within the
// same noise bound.
// The inner products of the rotations gs with the digits y, in one launch: the sums of rotation r go to acc[r].
// c0: P times its rotation is added to the even parts
static void hoisted_inner(Ctx& C, const Ct& a, const u64* y, const u64* gs, int count, u64* const* acc, const u64* c0) {
  KskInnerArgs A;
  A.count = count;
  for (int r = 0; r < count; ++r) {
    A.key[r] = key_for(C, gs[r]).p;
    A.acc[r] = acc[r];
    A.g[r] = gs[r];
  }
  k_ksk_inner(C, y, a.part(1), 2 * a.part_stride(), A, a.batch, a.level, c0, 2 * a.part_stride());
}
// `chunk` rotations at a time
static std::vector<std::unique_ptr<Ct>> hoisted_chunks(Ctx& C, const Ct& a, const std::vector<u64>& gs, size_t chunk) {
  const int l = a.level;
  const size_t per = acc_words(C, a.batch, l);
  Scratch S(C, digit_words(C, a.batch, l) + chunk * (per + moddown_words(C, a.batch, l)));
  u64 *acc = S.take(chunk * per), *y = S.take(digit_words(C, a.batch, l)), *v = S.take(chunk * moddown_words(C, a.batch, l));
  ks_modup(C, a.part(1), 2 * a.part_stride(), a.batch, l, acc, y);
  std::vector<std::unique_ptr<Ct>> out;
  for (size_t first = 0; first < gs.size(); first += chunk) {
    RotationOut R{a.part(0), a.part_stride(), (int)std::min(chunk, gs.size() - first), {}, {}};
    u64* accs[kKskRotations];
    size_t out_stride = 0;
    for (int r = 0; r < R.count; ++r) {
      auto o = ct_alloc(C, l, a.batch);
      o->scale = a.scale;
      out_stride = o->part_stride();
      R.out[r] = o->part(0);
      R.gs[r] = gs[first + r];
      accs[r] = acc + r * per;
      out.push_back(std::move(o));
    }
    hoisted_inner(C, a, y, R.gs, R.count, accs, nullptr);
    ks_moddown(C, acc, v, a.batch, l, R.out[0], out_stride, true, false, &R);
  }
  return out;
}

std::vector<std::unique_ptr<Ct>> ev_galois_hoisted(Ctx& C, const Ct& a, const std::vector<u64>& gs) {
  for (u64 g : gs) key_for(C, g);
  // as many rotations at a time as about 1 GiB of sums (and 32 K limbs a launch) allows, and one ModDown for all of
  // them: a rotation's few special limbs alone fill a fraction of the GPU, and its last wave is nearly empty (five
  // rotations of two ciphertexts, N = 2^16, level 14, 1 / 2 / 3 / 5 at a time: 1074 / 961 / 905 / 836 us).  Where the
  // memory for that is not there, one at a time: the sums and the ModDown workspace of a single rotation.
  const size_t per = acc_words(C, a.batch, a.level), limbs = (size_t)2 * a.batch * (a.level + 1 + C.n_p);
  const size_t chunk =
      std::max<size_t>(1, std::min({gs.size(), (size_t)kKskRotations, ((size_t)1 << 27) / per, 32768 / limbs}));
  if (chunk > 1) {
    try {
      return hoisted_chunks(C, a, gs, chunk);
    } catch (const Error& e) {
      if (e.code != HEDAP_ERR_OOM) throw;
    }
  }
  return hoisted_chunks(C, a, gs, 1);
}

std::vector<DevBuf> ev_galois_hoisted_qp(Ctx& C, const Ct& a, const std::vector<u64>& gs) {
  for (u64 g : gs) key_for(C, g);
  std::vector<DevBuf> out(gs.size());  // every sum is kept: as many rotations to a launch as it takes
  if (gs.empty()) return out;
  out[0] = DevBuf(acc_words(C, a.batch, a.level), C.stream);
  DevBuf digits(digit_words(C, a.batch, a.level), C.stream);
  u64* y = digits.p;
  ks_modup(C, a.part(1), 2 * a.part_stride(), a.batch, a.level, out[0].p, y);
  for (size_t first = 0; first < gs.size(); first += kKskRotations) {
    const int count = (int)std::min<size_t>(kKskRotations, gs.size() - first);
    u64* accs[kKskRotations];
    for (int r = 0; r < count; ++r) {
      if (first + r) out[first + r] = DevBuf(acc_words(C, a.batch, a.level), C.stream);
      accs[r] = out[first + r].p;
    }
    hoisted_inner(C, a, y, gs.data() + first, count, accs, a.part(0));
  }
  return out;
}
void ev_moddown_into(Ctx& C, DevBuf& acc, int batch, int level, Ct& out) {
  DevBuf v(moddown_words(C, batch, level), C.stream);
  ks_moddown(C, acc.p, v.p, batch, level, out.part(0), out.part_stride(), false, false);
}

std::unique_ptr<Ct> ev_mul_relin(Ctx& C, const Ct& a, const Ct& b) {
  const int l = std::min(a.level, b.level);
  check_batches(a, b);
  auto o = ct_alloc(C, l, a.batch);
  o->scale = a.scale * b.scale;
  const size_t per = (size_t)(l + 1) * C.N;
  DevBuf d2(a.batch * per, C.stream);
  k_tensor(C, a.part(0), a.part_stride(), b.part(0), b.part_stride(), o->part(0), o->part_stride(), d2.p, a.batch,
           l + 1);
  key_switch(C, d2.p, per, a.batch, l, 0, o->part(0), o->part_stride(), true, true);
  return o;
}

// rescale by q_l: c_i <- (c_i - [c_l]_centred) * q_l^-1 mod q_i, i < l.  With K (w the per-limb constants): of the
// product c w, in the same two transforms: the last limb enters its inverse transform as c_l w_l, and the
// finish computes c_i (w_i q_l^-1) - v q_l^-1, so the product is never formed apart (one pass over the
// ciphertext less; Mul_P by a constant of 8 ciphertexts at level 23).
static std::unique_ptr<Ct> rescale_scaled(Ctx& C, const Ct& a, const LimbConsts* K) {
  const int l = a.level;
  if (l < 1) throw Error(HEDAP_ERR_LEVEL, "rescale needs level >= 1");
  const size_t N = C.N;
  const int P = a.parts();
  const LevelConsts& LC = level_consts(C, l);
  auto o = ct_alloc(C, l - 1, a.batch);
  o->scale = a.scale / (double)C.primes[l];
  // the last limb to the coefficient domain (read in place), then one forward transform whose
  // load spreads its centred residue into every other prime and whose store finishes the rescale
  Scratch S(C, (size_t)P * (l + 1) * N + (K ? 2 * (size_t)l : 0));
  u64 *last = S.take(P * N), *tmp = S.take((size_t)P * l * N);
  NttAux inv{};
  inv.src = a.part(0) + (size_t)l * N;
  inv.src_stride = a.part_stride();
  NttAux fw{};
  fw.fin_w = LC.d_rescale.p + l;
  fw.fin_wb = LC.d_rescale.p + 2 * l;
  if (K) {
    inv.pre_scale = 1;
    inv.pre_w = K->w[l];
    inv.pre_wsh = h_shoup(K->w[l], C.primes[l]);
    LimbConsts F;  // mont_mul_lazy's pairs of w_i q_l^-1
    for (int i = 0; i < l; ++i) {
      F.w[i] = h_mont(h_mulmod(K->w[i], LC.rescale.inv[i], C.primes[i]), C.primes[i]);
      F.wsh[i] = h_mont(F.w[i], C.primes[i]);
    }
    u64* factors = S.take(2 * (size_t)l);
    k_put_limbconst(C, factors, l, F);
    fw.fin_w2 = fw.fin_w;
    fw.fin_w2b = fw.fin_wb;
    fw.fin_w = factors;
    fw.fin_wb = factors + l;
  }
  ntt_inverse(C.tab, qset(last, N, P, 0, 1, l), C.stream, &inv);
  fw.spread = last;
  fw.spread_stride = N;
  fw.spread_sub = LC.d_rescale.p;
  fw.spread_prime = l;
  fw.fin_dst = o->part(0);
  fw.fin_dst_stride = o->part_stride();
  fw.fin_c = a.part(0);
  fw.fin_c_stride = a.part_stride();
  ntt_forward(C.tab, qset(tmp, (size_t)l * N, P, 0, l), C.stream, &fw);
  return o;
}
std::unique_ptr<Ct> ev_rescale(Ctx& C, const Ct& a) { return rescale_scaled(C, a, nullptr); }

static void check_terms(const std::vector<std::pair<const Ct*, double>>& terms, int level) {
  for (const auto& t : terms) {
    if (t.first->level < level) throw Error(HEDAP_ERR_LEVEL, "linear combination operand below the output level");
    if (t.first->batch != terms[0].first->batch) throw Error(HEDAP_ERR_ARG, "operands have different batch sizes");
  }
}
static void lincomb_into(Ctx& C, const std::vector<std::pair<const Ct*, double>>& terms, int level, double target,
                         double c0, Ct& o);
// A relinearised product entering a linear combination that is rescaled next, as one fused
// operation: rescale(m (d01 + ModDown(acc)) + sum_j c_j t_j + c0), m the product's integer constant.
// With m = 1 the sum e = d01 + sum_j c_j t_j + c0 is formed first (one linear-combination pass) and
// ks_moddown_rescale finishes e + ModDown(acc).  With m = -1 every other constant is negated instead
// (std::round is odd, so each integer constant is exactly negated), giving -(the sum), and the fused
// rescale stores the negated residues: the centred residue is odd for an odd q_l, so rescale(-x) =
// -rescale(x) residue for residue.  Any other m, or a chain too wide for one linear-combination pass,
// takes the unfused sequence.
std::unique_ptr<Ct> ev_mul_lincomb_rescale(Ctx& C, const Ct& a, const Ct& b, double prod_scale, double prod_coef,
                                           const std::vector<std::pair<const Ct*, double>>& terms, double target,
                                           double c0) {
  const int l = std::min(a.level, b.level);
  check_batches(a, b);
  const double m = l >= 1 ? std::round(prod_coef * target * (double)C.primes[l] / prod_scale) : 0.0;
  if (l < 1 || (m != 1.0 && m != -1.0) || l + 1 > kLcLimbs || terms.size() + 1 > kLcTerms) {
    auto pr = ev_mul_relin(C, a, b);
    pr->scale = prod_scale;
    std::vector<std::pair<const Ct*, double>> all{{pr.get(), prod_coef}};
    all.insert(all.end(), terms.begin(), terms.end());
    return ev_rescale(C, *ev_lincomb_raw(C, all, l, target, c0));
  }
  auto d01 = ct_alloc(C, l, a.batch);
  d01->scale = prod_scale;
  auto o = ct_alloc(C, l - 1, a.batch);  // holds d2 first: batch (l + 1) N of its 2 batch l N words
  const size_t per = (size_t)(l + 1) * C.N;
  Scratch S(C, acc_words(C, a.batch, l) + std::max(digit_words(C, a.batch, l), mdr_words(C, a.batch)));
  u64* acc = S.take(acc_words(C, a.batch, l));
  const size_t mark = S.at;
  u64* d2 = o->part(0);
  k_tensor(C, a.part(0), a.part_stride(), b.part(0), b.part_stride(), d01->part(0), d01->part_stride(), d2, a.batch,
           l + 1);
  ks_inner(C, d2, per, a.batch, l, 0, acc, S.take(digit_words(C, a.batch, l)));
  S.at = mark;
  std::vector<std::pair<const Ct*, double>> all{{d01.get(), m * prod_coef}};
  for (const auto& t : terms) all.emplace_back(t.first, m * t.second);
  check_terms(all, l);
  lincomb_into(C, all, l, target, m * c0, *d01);  // e, in d01's place
  const double raw = target * (double)C.primes[l];
  o->scale = raw / (double)C.primes[l];
  ks_moddown_rescale(C, acc, S.take(mdr_words(C, a.batch)), a.batch, l, d01->part(0), d01->part_stride(), o->part(0),
                     o->part_stride(), m < 0);
  return o;
}

// HMult and rescale: the tensor product, the relinearising key switch up to its inner product, then
// ModDown and the rescale in one transform (ks_moddown_rescale); equal, residue for residue, to
// ev_rescale(ev_mul_relin(a, b)).
std::unique_ptr<Ct> ev_mul(Ctx& C, const Ct& a, const Ct& b) {
  const int l = std::min(a.level, b.level);
  if (l < 1) throw Error(HEDAP_ERR_LEVEL, "rescale needs level >= 1");
  check_batches(a, b);
  const size_t per = (size_t)(l + 1) * C.N;
  auto o = ct_alloc(C, l - 1, a.batch);  // holds d2 first: batch (l + 1) N of its 2 batch l N words
  o->scale = a.scale * b.scale / (double)C.primes[l];
  Scratch S(C, 2 * a.batch * per + acc_words(C, a.batch, l) +
                   std::max(digit_words(C, a.batch, l), mdr_words(C, a.batch)));
  u64 *e = S.take(2 * a.batch * per), *acc = S.take(acc_words(C, a.batch, l));  // e: the tensor's d0, d1
  const size_t mark = S.at;
  u64* d2 = o->part(0);
  k_tensor(C, a.part(0), a.part_stride(), b.part(0), b.part_stride(), e, per, d2, a.batch, l + 1);
  ks_inner(C, d2, per, a.batch, l, 0, acc, S.take(digit_words(C, a.batch, l)));
  S.at = mark;
  ks_moddown_rescale(C, acc, S.take(mdr_words(C, a.batch)), a.batch, l, e, per, o->part(0), o->part_stride());
  return o;
}

u64 galois_for_rotation(const Ctx& C, i64 steps) {
  const i64 h = (i64)(C.N / 2);
  const i64 r = ((steps % h) + h) % h;
  return h_powmod(5, (u64)r, 2 * C.N);
}

size_t galois_words(const Ctx& C, int batch, int l) {
  return moddown_words(C, batch, l) /* the result */ + acc_words(C, batch, l) +
         std::max(digit_words(C, batch, l), moddown_words(C, batch, l));
}
std::unique_ptr<Ct> ev_galois(Ctx& C, const Ct& a, u64 g) {
  const int l = a.level;
  auto o = ct_alloc(C, l, a.batch);
  o->scale = a.scale;
  // sigma_g(c1) is switched, from the result's place; sigma_g(c0) is gathered by the ModDown's finishing store
  Scratch S(C, acc_words(C, a.batch, l) + std::max(digit_words(C, a.batch, l), moddown_words(C, a.batch, l)));
  u64* acc = S.take(acc_words(C, a.batch, l));
  const size_t mark = S.at;
  k_automorph(C, a.part(1), 2 * a.part_stride(), o->part(1), 2 * o->part_stride(), a.batch, l + 1, g);
  ks_inner(C, o->part(1), 2 * o->part_stride(), a.batch, l, g, acc, S.take(digit_words(C, a.batch, l)));
  S.at = mark;
  const RotationOut R{a.part(0), a.part_stride(), 1, {o->part(0)}, {g}};
  ks_moddown(C, acc, S.take(moddown_words(C, a.batch, l)), a.batch, l, o->part(0), o->part_stride(), true, false, &R);
  return o;
}

// key switch of (c0, c1) with the key `id` (from the secret c1 multiplies to the key's target)
std::unique_ptr<Ct> ev_switch_key(Ctx& C, const Ct& a, u64 id) {
  if (!C.keys.count(id)) throw Error(HEDAP_ERR_ARG, "switching key not generated");
  const int l = a.level;
  auto o = ct_copy(C, a, l);
  key_switch(C, o->part(1), 2 * o->part_stride(), a.batch, l, id, o->part(0), o->part_stride(), true, false);
  return o;
}

// Mul_P by a real constant c at plaintext scale target * q_l / scale, then rescale;
// the result's scale is set to exactly `target`.
// Mul_P by c without the rescale: the product is labelled target * q_l (several such products at one
// level with one target add exactly and share one rescale)
std::unique_ptr<Ct> ev_mul_const_raw(Ctx& C, const Ct& a, double c, double target) {
  const int l = a.level;
  if (l < 1) throw Error(HEDAP_ERR_LEVEL, "constant multiplication needs level >= 1");
  const double sp = target * (double)C.primes[l] / a.scale;
  const double v = std::round(c * sp);
  LimbConsts K;
  for (int i = 0; i <= l; ++i) {
    K.w[i] = h_double_to_mod(v, C.primes[i]);
    K.wsh[i] = h_shoup(K.w[i], C.primes[i]);
  }
  auto t = ct_alloc(C, l, a.batch);
  t->scale = target * (double)C.primes[l];
  k_mul_limbconst(C, a.part(0), a.part_stride(), t->part(0), t->part_stride(), a.parts(), l + 1, K);
  return t;
}
std::unique_ptr<Ct> ev_lincomb_raw(Ctx& C, const std::vector<std::pair<const Ct*, double>>& terms, int level,
                                   double target, double c0) {
  if (terms.empty()) throw Error(HEDAP_ERR_ARG, "linear combination without terms");
  if (level < 1) throw Error(HEDAP_ERR_LEVEL, "constant multiplication needs level >= 1");
  const double raw = target * (double)C.primes[level];
  const int batch = terms[0].first->batch;
  check_terms(terms, level);
  auto o = ct_alloc(C, level, batch);
  o->scale = raw;
  if (level + 1 > kLcLimbs) {  // wide chains: one product and one addition at a time
    std::unique_ptr<Ct> acc;
    for (const auto& t : terms) {
      std::unique_ptr<Ct> d = t.first->level == level ? nullptr : ev_drop(C, *t.first, level);
      auto term = ev_mul_const_raw(C, d ? *d : *t.first, t.second, target);
      acc = acc ? ev_add(C, *acc, *term, false) : std::move(term);
    }
    acc->scale = raw;
    return ev_add_const(C, *acc, c0);
  }
  lincomb_into(C, terms, level, target, c0, *o);
  return o;
}
// the sum itself, into o (at `level`, at most kLcLimbs limbs; it may be the first term: a thread reads the words that it
// writes, and only in the first launch)
static void lincomb_into(Ctx& C, const std::vector<std::pair<const Ct*, double>>& terms, int level, double target,
                         double c0, Ct& o) {
  const double raw = target * (double)C.primes[level];
  for (size_t first = 0; first < terms.size(); first += kLcTerms) {
    LinCombArgs A{};
    A.count = (int)std::min<size_t>(kLcTerms, terms.size() - first);
    A.accumulate = first > 0;
    A.add_c0 = first == 0;
    for (int j = 0; j < A.count; ++j) {
      const Ct& a = *terms[first + j].first;
      A.in[j] = a.part(0);
      A.stride[j] = a.part_stride();
      const double sp = target * (double)C.primes[level] / a.scale;  // as in ev_mul_const_raw
      const double v = std::round(terms[first + j].second * sp);
      for (int i = 0; i <= level; ++i) {
        A.w[j][i] = h_double_to_mod(v, C.primes[i]);
        A.wsh[j][i] = h_shoup(A.w[j][i], C.primes[i]);
      }
    }
    if (A.add_c0) {
      const double v0 = std::round(c0 * raw);  // as in ev_add_const on the sum
      for (int i = 0; i <= level; ++i) A.c0[i] = h_double_to_mod(v0, C.primes[i]);
    }
    k_lincomb(C, o.part(0), o.part_stride(), o.parts(), level + 1, A);
  }
}

std::unique_ptr<Ct> ev_mul_const(Ctx& C, const Ct& a, double c, double target) {
  const int l = a.level;
  if (l < 1) throw Error(HEDAP_ERR_LEVEL, "constant multiplication needs level >= 1");
  const double v = std::round(c * (target * (double)C.primes[l] / a.scale));  // as in ev_mul_const_raw
  LimbConsts K;
  for (int i = 0; i <= l; ++i) K.w[i] = h_double_to_mod(v, C.primes[i]);
  auto o = rescale_scaled(C, a, &K);
  o->scale = target;
  return o;
}

std::unique_ptr<Ct> ev_add_const(Ctx& C, const Ct& a, double c) {
  const double v = std::round(c * a.scale);
  LimbConsts K;
  for (int i = 0; i <= a.level; ++i) K.w[i] = h_double_to_mod(v, C.primes[i]);
  auto o = ct_alloc(C, a.level, a.batch);
  o->scale = a.scale;
  k_add_limbconst(C, a.part(0), a.part_stride(), o->part(0), o->part_stride(), a.parts(), a.level + 1, K);
  return o;
}

// (a + c) * m in one pass: the constant c is added at a's scale exactly as ev_add_const adds it,
// then everything is multiplied by the integer m (same residues as the two operations in turn)
std::unique_ptr<Ct> ev_add_const_mul_int(Ctx& C, const Ct& a, double c, i64 m) {
  if (a.level + 1 > kLcLimbs) return ev_mul_int(C, *ev_add_const(C, a, c), m);
  const double v = std::round(c * a.scale);
  LinCombArgs A{};
  A.count = 1;
  A.add_c0 = 1;
  A.in[0] = a.part(0);
  A.stride[0] = a.part_stride();
  for (int i = 0; i <= a.level; ++i) {
    const u64 q = C.primes[i], mm = h_smod(m, q);
    A.w[0][i] = mm;
    A.wsh[0][i] = h_shoup(mm, q);
    A.c0[i] = h_mulmod(h_double_to_mod(v, q), mm, q);
  }
  auto o = ct_alloc(C, a.level, a.batch);
  o->scale = a.scale;
  k_lincomb(C, o->part(0), o->part_stride(), o->parts(), a.level + 1, A);
  return o;
}

std::unique_ptr<Ct> ev_mul_int(Ctx& C, const Ct& a, i64 m) {
  LimbConsts K;
  for (int i = 0; i <= a.level; ++i) {
    K.w[i] = h_smod(m, C.primes[i]);
    K.wsh[i] = h_shoup(K.w[i], C.primes[i]);
  }
  auto o = ct_alloc(C, a.level, a.batch);
  o->scale = a.scale;
  k_mul_limbconst(C, a.part(0), a.part_stride(), o->part(0), o->part_stride(), a.parts(), a.level + 1, K);
  return o;
}

}  // namespace hedap
