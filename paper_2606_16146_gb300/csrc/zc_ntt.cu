// zc_ntt.cu -- NTT-form ZeroCheck prover (Fig. side-by-side-zc, left;
// Sec. 3.2).
//
//   N1  g_j <- INTT_H(e_j)                    (per column, size N)
//   N2  for each coset slice s_j = 7 w_M^j H (j < s = M/N):
//         ghat_j = NTT_N(g_j(k) (7 w_M^j)^k / N), fhat = gate(ghat),
//         qhat = fhat / z_H, with z_H constant on the slice: 7^N w_s^j - 1
//   N3  q <- INTT_D(qhat) = 7^-k M^-1 DFT_M^-1(qhat)
//   N4  root(q), z = squeeze (again while z^N = 1)
//   N5  openings g_j(z), q(z)
//
// Transforms are "four-step" (Bailey) factorisations done as passes over
// HBM; each pass runs many sub-DFTs of length L <= 4096 in shared memory
// (self-sorting Stockham stages of radix 8/4/2).  Digit orders are chosen so
// that no pass ever transposes:
//   * N1 is the reversed-input structure: its first pass reads the natural
//     evaluations with a stride (a gather), its output is natural.
//   * N2 is the natural-input structure: each slice comes out digit-reversed.
//   * The gate is pointwise, so qhat keeps that order, which is exactly the
//     input order of N3 written as a three-digit reversed-input transform
//     (slice digit outermost); N3's output, q, is natural.
// Every factor of a transform is a constant: the stages' twiddles, the
// twiddles between passes, the coset factors (7 w_M^j)^k / N of N2 with the
// conversion to Montgomery form in them (columns and coefficients are
// canonical, "level 0") and the outer twiddles of N3 with 7^-k and the
// conversion back come from tables of (w, floor(2^256 w / r)) pairs, per size
// and in the lanes' order.  Sizes whose tables do not fit the cache use
// two-level power tables of the 2^30-th root of unity
// (w^e = HI[e >> 15] * LO[e & 32767]).
#include <algorithm>
#include <cstring>

#include "zc_internal.cuh"
#include "zc_ntt_index.cuh"
#include "zc_transcript.cuh"

namespace zc {

constexpr int kLog30 = 30;
constexpr uint32_t kLoBits = 15;
constexpr uint32_t kLoMask = (1u << kLoBits) - 1;
constexpr int kMaxNttN = 24;
static_assert((uint64_t)kMaxCols << kMaxNttN < 1ull << 32, "slice strides are 32-bit");

struct NttTables {
  bool ready = false;
  fr w32h;                 // 7^((r-1)/2^32), canonical, host copy
  FrcTab dft_fwd, dft_inv; // the stages' twiddles, see stage_tab
  frc c_fwd[3], c_inv[3];  // w_8, w_4, w_8^3 of each direction (host copies, passed to the kernels by value)
  fr* wf_lo = nullptr;     // w_2^30^b, b < 2^15 (level 1)
  fr* wf_hi = nullptr;     // w_2^30^(a 2^15)
  fr* wi_lo = nullptr;     // inverse root
  fr* wi_hi = nullptr;
  fr* s7_lo = nullptr;     // 7^-b (level 0)
  fr* s7_hi = nullptr;     // 7^-(a 2^15) (level 1)
  fr* p7_lo = nullptr;     // 7^b (level 1)
  fr* p7_hi = nullptr;     // 7^(a 2^15) (level 1)
  void* mem = nullptr;
};

static NttTables g_tabs_by_dev[64];
static std::mutex g_tabs_mu;

struct NttTabArgs {
  FrcTab dft_fwd, dft_inv; fr* wf_lo; fr* wf_hi; fr* wi_lo; fr* wi_hi; fr* s7_lo; fr* s7_hi;
  fr* p7_lo; fr* p7_hi;
  fr w30;        // 2^30-th root (level 1)
  fr w30i;       // its inverse (level 1)
  fr seveninv;   // 7^-1 (level 1)
  const DevConst* C;
};

__device__ fr fr_pow_dev(fr base, uint64_t e, const DevConst* C) {  // level 1 in/out
  fr acc = C->one;
  while (e) {
    if (e & 1) acc = fr_mul(acc, base);
    base = fr_mul(base, base);
    e >>= 1;
  }
  return acc;
}

__global__ void k_ntt_tables(NttTabArgs A) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  const DevConst* C = A.C;
  if (i < kStageTab) {
    const uint32_t logNs = i < 88 ? 3 : i < 792 ? 6 : 9, e = i - stage_tab(logNs, 3), Ns = 1u << logNs;
    const uint32_t lr = e < 7 * Ns ? 3 : e < 10 * Ns ? 2 : 1, g = i - stage_tab(logNs, lr);
    const uint64_t ex = (uint64_t)((g / Ns + 1) * (g % Ns)) << (30 - logNs - lr);  // r k
    A.dft_fwd.st(i, frc_of(fr_pow_dev(A.w30, ex, C)));
    A.dft_inv.st(i, frc_of(fr_pow_dev(A.w30i, ex, C)));
  }
  if (i < (1u << kLoBits)) {
    A.wf_lo[i] = fr_pow_dev(A.w30, i, C);
    A.wf_hi[i] = fr_pow_dev(A.w30, (uint64_t)i << kLoBits, C);
    A.wi_lo[i] = fr_pow_dev(A.w30i, i, C);
    A.wi_hi[i] = fr_pow_dev(A.w30i, (uint64_t)i << kLoBits, C);
    A.s7_lo[i] = from_mont(fr_pow_dev(A.seveninv, i, C));          // level 0
    A.s7_hi[i] = fr_pow_dev(A.seveninv, (uint64_t)i << kLoBits, C);  // level 1
    A.p7_lo[i] = fr_pow_dev(C->small[7], i, C);
    A.p7_hi[i] = fr_pow_dev(C->small[7], (uint64_t)i << kLoBits, C);
  }
}

// w^e for the 2^30-th root (or its inverse), e < 2^30, level 1
__device__ __forceinline__ fr root_pow(const fr* lo, const fr* hi, uint32_t e) {
  return fr_mul(ld_fr(hi + (e >> kLoBits)), ld_fr(lo + (e & kLoMask)));
}

// ---------------------------------------------------------------- passes --

enum { PRE_NONE = 0, PRE_COSET = 1, PRE_TAB = 2 };
enum { POST_NONE = 0, POST_TW = 1, POST_OUTER = 2, POST_FINAL = 3, POST_TAB = 4 };

struct NttPassArgs {
  const fr* in[kMaxCols];
  fr* out[kMaxCols];
  uint32_t items;         // columns in this launch
  uint32_t logL;          // sub-DFT length
  uint32_t logW;          // sub-DFTs per CTA
  uint32_t B;             // sub-DFTs (a CTA's surplus ones are neither read nor written)
  uint32_t out_y, pre_y;  // slice blockIdx.y: elements from one slice's outputs, and pre factors, to the next's
  uint32_t in_y;          // ... and inputs (0: every slice reads the same)
  NttMap im, om;          // element (b, t) of a column
  FrcTab dft;             // stage twiddles, forward or inverse
  frc w8, w4, w83;        // w_8, w_4, w_8^3
  int pre;
  NttMap pm;              // PRE_TAB: factor pre_tab[pm]; PRE_COSET: k = pm, factor hi[k >> shift] lo[k & mask]
  FrcTab pre_tab;
  const fr* pre_lo;
  const fr* pre_hi;
  uint32_t pre_shift;
  int post;
  NttMap qm;              // POST_TAB: factor post_tab[qm]
  FrcTab post_tab;
  const fr* tw_lo;
  const fr* tw_hi;
  uint32_t tw_lbmod;      // POST_TW: e = (b mod 2^lbmod) * t
  uint32_t tw_shift;      // exponent in the 2^30 table: (e mod 2^(30-shift)) << shift
  uint32_t outer_lbdiv;   // POST_OUTER: e = (b >> lbdiv) * ((t << lbdiv) + (b mod 2^lbdiv))
  uint32_t fin_logN;      // POST_FINAL: k = (t << fin_logN) + b
  uint32_t* err;          // if set: the pass reads the proof's input columns, and a value >= r sets bit 0
  void use(const NttMaps& m) { logL = m.logL; im = m.im; om = m.om; pm = m.pm; qm = m.qm; }
};

// radix-2/4/8 butterflies on x[0..R) in registers, X[k] = sum_r x[r] w_R^(rk).
// Inputs are canonical.  A value that only feeds a multiplication (fr_mulc
// takes any value below 2r) is left lazily reduced in [0, 2r): the stage
// outputs (the next stage multiplies all but one of them by its twiddle and
// reduces that one, the pass's store reduces or multiplies every one), and
// the terms multiplied by w_4, w_8, w_8^3.  Every factor of a transform is a
// constant, so all of them are fr_mulc products, inlined; w_4, w_8 and w_8^3
// are kernel parameters, which the multiplier reads as operands without a
// load.
// OUT: 0 every output canonical, 1 a0 canonical and a1..a3 lazy, 2 all lazy.
template <int OUT>
__device__ __forceinline__ void dft4(fr& a0, fr& a1, fr& a2, fr& a3, const frc& w4) {
  const fr u0 = fr_add(a0, a2), u1 = fr_sub(a0, a2);
  const fr v0 = fr_add(a1, a3), v1 = fr_mulc(w4, fr_sub_lazy(a1, a3));
  a0 = OUT == 2 ? fr_add_lazy(u0, v0) : fr_add(u0, v0);
  a2 = OUT >= 1 ? fr_sub_lazy(u0, v0) : fr_sub(u0, v0);
  a1 = OUT >= 1 ? fr_add_lazy(u1, v1) : fr_add(u1, v1);
  a3 = OUT >= 1 ? fr_sub_lazy(u1, v1) : fr_sub(u1, v1);
}

// outputs lazy
__device__ __forceinline__ void dft8(fr (&x)[8], const NttPassArgs& A) {
  fr e0 = x[0], e1 = x[2], e2 = x[4], e3 = x[6];
  fr o0 = x[1], o1 = x[3], o2 = x[5], o3 = x[7];
  dft4<0>(e0, e1, e2, e3, A.w4);
  dft4<1>(o0, o1, o2, o3, A.w4);
  o1 = fr_mulc(A.w8, o1);
  o2 = fr_mulc(A.w4, o2);
  o3 = fr_mulc(A.w83, o3);
  x[0] = fr_add_lazy(e0, o0);
  x[4] = fr_sub_lazy(e0, o0);
  x[1] = fr_add_lazy(e1, o1);
  x[5] = fr_sub_lazy(e1, o1);
  x[2] = fr_add_lazy(e2, o2);
  x[6] = fr_sub_lazy(e2, o2);
  x[3] = fr_add_lazy(e3, o3);
  x[7] = fr_sub_lazy(e3, o3);
}

// The CTA tile in shared memory: element i's two 16-byte halves live in two
// planes, and the 16-byte index is XOR-swizzled (i ^ ((i >> 3) & 7)) so
// that unit-stride and radix-strided (8, 64) warp accesses spread over all
// banks.
struct SmTile {
  uint4* p;     // plane 0: p[0, T), plane 1: p[T, 2T)
  uint32_t T;
  __device__ __forceinline__ fr get(uint32_t i) const { return get_at(tile_slot(i)); }
  __device__ __forceinline__ fr get_at(uint32_t s) const {
    const uint4 a = p[s], b = p[T + s];
    fr x;
    x.v[0] = a.x; x.v[1] = a.y; x.v[2] = a.z; x.v[3] = a.w;
    x.v[4] = b.x; x.v[5] = b.y; x.v[6] = b.z; x.v[7] = b.w;
    return x;
  }
  __device__ __forceinline__ void put(uint32_t i, const fr& x) const {
    const uint32_t s = tile_slot(i);
    p[s] = make_uint4(x.v[0], x.v[1], x.v[2], x.v[3]);
    p[T + s] = make_uint4(x.v[4], x.v[5], x.v[6], x.v[7]);
  }
};

// One pass: the sub-DFTs b of length L = 2^logL over strided elements, W of
// them per CTA, blockDim.x = L W / 8 threads with 8 elements each.
//
// Every stage reads element tid + NT p of the tile into register p (NT =
// blockDim.x, p < 8), so its radix-R groups are the registers p that agree
// modulo 8 / R, whatever L, W and the stage.  The factors of a step (the pre
// table before the first stage, the twiddles before the others, the post
// table before the store) go through one copy of the code.
//
// What bounds it: the wide multiply-adds of the ~6 products per element (the
// multiplier pipe is 79 % busy in the first N2 pass at n = 20, 670 us; reading
// elements and factors one per lane it was 67 %, 769 us), then the latency of
// 16 warps per SM.  Why the pass looks as it does: 32- and 64-byte elements
// read one per lane made every request touch 16 to 32 lines (L1 75 % busy, now
// 21 %), so columns move in 16-byte halves, two lanes to an element, and
// factors lie in 16-byte planes in the order the lanes read them; products
// inlined at each use were 75 KB of instructions, more than the instruction
// cache keeps, hence the shared step; address arithmetic competes for the
// multiplier pipe, hence the FAST form (8.21 -> 8.02 ms for the proof).
// FAST: whole tiles of sub-DFTs of at least 8 points, 64 threads or more, all
// factors from tables; slot p's addresses are slot 0's plus a uniform offset.
// The general form also takes short sub-DFTs, a part-filled tile (sub-DFTs
// past the last one repeat it and are not stored) and the two-level power
// tables.
template <int MAXT, int MINB, bool FAST>
__global__ void __launch_bounds__(MAXT, MINB) k_ntt_pass(NttPassArgs A) {
  extern __shared__ __align__(16) uint4 sm_planes[];
  const uint32_t NT = blockDim.x, tid = threadIdx.x;
  const SmTile sm{sm_planes, NT * 8};
  // items (columns) vary fastest across consecutive CTAs, so the per-element
  // factor tables, shared by every column, are reused from L2
  const uint32_t item = blockIdx.x % A.items;
  const uint32_t logL = A.logL, logW = A.logW;
  const uint32_t b0 = (blockIdx.x / A.items) << logW;
  const NttTile<FAST> X(logL, logW, b0, A.B, NT, tid);
  // The column's elements come through shared memory in 16-byte halves, two
  // lanes to an element; a warp copies its own slots only.
  {
    const uint32_t half = tid & 1;
    const char* in = reinterpret_cast<const char*>(A.in[item] + (size_t)A.in_y * blockIdx.y) + 16 * half;
#pragma unroll
    for (int s = 0; s < 2; s++) {
      const uint32_t i = X.copy_elt(s);
      const char* g = in + sizeof(fr) * (size_t)X.index(A.im, i);
#pragma unroll
      for (int p = 0; p < 8; p++) {
        const uint32_t d = (uint32_t)__cvta_generic_to_shared(sm.p + sm.T * half + X.slot(i, p));
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(g + (ptrdiff_t)sizeof(fr) * X.step(A.im, i, p))
                     : "memory");
      }
    }
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
    __syncwarp();
  }
  auto get = [&](int p) { return sm.get_at(X.slot(tid, p)); };
  fr x[8];
#pragma unroll
  for (int p = 0; p < 8; p++) x[p] = get(p);
  if (A.err) {
    bool bad = false;
#pragma unroll
    for (int p = 0; p < 8; p++) bad |= !fr_is_canonical(x[p]);
    if (bad) atomicOr(A.err, 1u);
  }
  if (!FAST && A.pre == PRE_COSET) {
#pragma unroll
    for (int p = 0; p < 8; p++) {
      const uint32_t k = X.index(A.pm, tid + NT * p);
      // one slice per launch: every column uses the same tables
      x[p] = fr_mul(fr_mul(ld_fr(A.pre_hi + (k >> A.pre_shift)), ld_fr(A.pre_lo + (k & ((1u << A.pre_shift) - 1)))),
                    x[p]);
    }
  }
  const bool post_tab = A.post == POST_TAB;
  uint32_t logNs = 0;
  bool fin = false;  // the step after the last stage: the post table
#pragma unroll 1
  while (true) {
    const uint32_t lr = min(3u, logL - logNs);  // radix R as a log
    // factors: pre or post table, or the twiddles w_{Ns R}^{r k}, r = p >> lg
    // (for r = 0 the previous stage's lazy output is only reduced)
    const bool tw = !fin && logNs > 0, all = fin || (logNs == 0 && A.pre == PRE_TAB);
    if (tw || all) {
      const FrcTab base = tw ? A.dft : fin ? A.post_tab : A.pre_tab;
      const NttMap m = fin ? A.qm : A.pm;
      const FrcTab first = base.at(tw ? X.tw_first(logNs, lr)
                                     : (ptrdiff_t)X.index(m, tid) + (fin ? 0 : (ptrdiff_t)A.pre_y * blockIdx.y));
      // one load for both kinds (a load in each branch: n = 20 7.72 to 7.84 ms, this 7.61)
      auto fac = [&](int p) {
        return first.ld(tw ? (ptrdiff_t)X.tw_step(logNs, lr, p) : X.step(m, tid, p));
      };
#pragma unroll
      for (int p = 7; p >= 4; p--) x[p] = fr_mulc(fac(p), x[p]);
      if (all || lr >= 2) {
        x[3] = fr_mulc(fac(3), x[3]);
        x[2] = fr_mulc(fac(2), x[2]);
      } else {
        x[3] = fr_reduce1(x[3]);
        x[2] = fr_reduce1(x[2]);
      }
      if (all || lr == 3) x[1] = fr_mulc(fac(1), x[1]);
      else x[1] = fr_reduce1(x[1]);
      if (all) x[0] = fr_mulc(fac(0), x[0]);
      else x[0] = fr_reduce1(x[0]);
    }
    if (fin) break;
    if (lr == 3) {
      dft8(x, A);
    } else if (lr == 2) {
      dft4<2>(x[0], x[2], x[4], x[6], A.w4);
      dft4<2>(x[1], x[3], x[5], x[7], A.w4);
    } else if (lr == 1) {
#pragma unroll
      for (int g = 0; g < 4; g++) {
        const fr u = x[g], v = x[g + 4];
        x[g] = fr_add_lazy(u, v);
        x[g + 4] = fr_sub_lazy(u, v);
      }
    }
    if (logNs + lr == logL) {
      if (!post_tab) break;
      fin = true;
      continue;
    }
    __syncthreads();  // every slot has been read
#pragma unroll
    for (int p = 0; p < 8; p++) sm.put(X.exchange(logNs, lr, p), x[p]);
    __syncthreads();
#pragma unroll
    for (int p = 0; p < 8; p++) x[p] = get(p);
    logNs += lr;
  }

  // ---- store, two lanes to an element as in the load: a lane keeps one half
  // of its own element and swaps the other for that half of its neighbour's.
  // Without a post table the values are lazy: reduced, or multiplied here.
  const bool odd = tid & 1;
  char* const out = reinterpret_cast<char*>(A.out[item] + (size_t)A.out_y * blockIdx.y) + 16 * odd;
  char* const oe = out + sizeof(fr) * (size_t)X.index(A.om, tid & ~1u);  // the even lane's element
  char* const oo = out + sizeof(fr) * (size_t)X.index(A.om, tid | 1u);
#pragma unroll
  for (int p = 0; p < 8; p++) {
    fr y = x[p];
    if (!post_tab) {
      const uint32_t b = X.sub(tid + NT * p), t = X.elt(tid + NT * p);
      if (FAST || A.post == POST_NONE) {
        y = fr_reduce1(y);
      } else if (A.post == POST_FINAL) {
        const uint32_t k = (t << A.fin_logN) + b;
        y = fr_mul(fr_mul(ld_fr(A.tw_hi + (k >> kLoBits)), ld_fr(A.tw_lo + (k & kLoMask))), y);  // level 0
      } else {
        const uint32_t dm = (1u << A.outer_lbdiv) - 1;
        const uint64_t e = A.post == POST_TW ? (uint64_t)(b & ((1u << A.tw_lbmod) - 1)) * t
                                             : (uint64_t)(b >> A.outer_lbdiv) * ((t << A.outer_lbdiv) + (b & dm));
        const uint32_t ex = (uint32_t)((e << A.tw_shift) & ((1ull << kLog30) - 1));
        y = ex ? fr_mul(root_pow(A.tw_lo, A.tw_hi, ex), y) : fr_reduce1(y);
      }
    }
    uint32_t r[4];
#pragma unroll
    for (int h = 0; h < 4; h++) r[h] = __shfl_xor_sync(0xffffffffu, odd ? y.v[h] : y.v[4 + h], 1);
    if (X.stored((tid & ~1u) + NT * p))
      *reinterpret_cast<uint4*>(oe + (ptrdiff_t)sizeof(fr) * X.step(A.om, tid & ~1u, p)) =
          odd ? make_uint4(r[0], r[1], r[2], r[3]) : make_uint4(y.v[0], y.v[1], y.v[2], y.v[3]);
    if (X.stored((tid | 1u) + NT * p))
      *reinterpret_cast<uint4*>(oo + (ptrdiff_t)sizeof(fr) * X.step(A.om, tid | 1u, p)) =
          odd ? make_uint4(y.v[4], y.v[5], y.v[6], y.v[7]) : make_uint4(r[0], r[1], r[2], r[3]);
  }
}

// The same pass for launches too small to fill the GPU: two elements per
// thread and radix-2 stages, so a thread's chain is a product per stage instead
// of a dozen, on four times the threads (n = 12: a pass takes 20 to 30 us with
// eight elements per thread, of which the products in a row are most).  Element
// tid + NT p, p < 2; the stages exchange through two tiles in turn.  Whole
// tiles, 2 <= L <= 1024, all factors from tables.
__global__ void __launch_bounds__(512) k_ntt_pass_small(NttPassArgs A) {
  extern __shared__ __align__(16) uint4 sm_planes[];
  const uint32_t NT = blockDim.x, tid = threadIdx.x;
  const uint32_t item = blockIdx.x % A.items;
  const uint32_t logL = A.logL;
  const NttSmallTile X{logL, A.logW, (blockIdx.x / A.items) << A.logW, NT, tid};
  const uint32_t b = X.sub(), t0 = X.elt(0), t1 = X.elt(1);
  const fr* in = A.in[item] + (size_t)A.in_y * blockIdx.y;
  fr x0 = ld_fr(in + A.im.at(b, t0)), x1 = ld_fr(in + A.im.at(b, t1));
  if (A.err && !(fr_is_canonical(x0) && fr_is_canonical(x1))) atomicOr(A.err, 1u);
  if (A.pre == PRE_TAB) {
    const FrcTab f = A.pre_tab.at((ptrdiff_t)A.pre_y * blockIdx.y);
    x0 = fr_mulc(f.ld(A.pm.at(b, t0)), x0);
    x1 = fr_mulc(f.ld(A.pm.at(b, t1)), x1);
  }
  for (uint32_t logNs = 0; logNs < logL; logNs++) {
    if (logNs > 0) {
      x0 = fr_reduce1(x0);
      x1 = fr_mulc(A.dft.ld(X.twiddle(logNs)), x1);
    }
    const fr y0 = fr_add_lazy(x0, x1), y1 = fr_sub_lazy(x0, x1);
    if (logNs + 1 == logL) {
      x0 = y0;
      x1 = y1;
      break;
    }
    const SmTile sm{sm_planes + (logNs & 1) * 4 * NT, 2 * NT};
    sm.put(X.exchange(logNs, 0), y0);
    sm.put(X.exchange(logNs, 1), y1);
    __syncthreads();
    x0 = sm.get(tid);
    x1 = sm.get(tid + NT);
  }
  if (A.post == POST_TAB) {
    x0 = fr_mulc(A.post_tab.ld(A.qm.at(b, t0)), x0);
    x1 = fr_mulc(A.post_tab.ld(A.qm.at(b, t1)), x1);
  } else {
    x0 = fr_reduce1(x0);
    x1 = fr_reduce1(x1);
  }
  fr* out = A.out[item] + (size_t)A.out_y * blockIdx.y;
  st_fr(out + A.om.at(b, t0), x0);
  st_fr(out + A.om.at(b, t1), x1);
}

// N3's last stage for 2, 4 or 8 slices: the transform across the slices, in
// registers, one k' per thread (element k' of slice j at in[j N + k'], output t
// times post_tab[t] at out[t N + k']).  It is bound by memory (1 GB for 4
// x 2^22 elements: 158 us at the copy rate); the pass kernel's general form took
// 390 us there, the whole proof 32.27 ms against 32.05.
template <int LS>
__global__ void __launch_bounds__(256) k_ntt_cross(NttPassArgs A) {
  constexpr int S = 1 << LS;
  const uint32_t k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= A.B) return;
  fr x[8];
#pragma unroll
  for (int j = 0; j < S; j++) x[j] = ld_fr(A.in[0] + (size_t)j * A.B + k);
  if constexpr (LS == 3) {
    dft8(x, A);
  } else if constexpr (LS == 2) {
    dft4<2>(x[0], x[1], x[2], x[3], A.w4);
  } else {
    const fr u = x[0], v = x[1];
    x[0] = fr_add_lazy(u, v);
    x[1] = fr_sub_lazy(u, v);
  }
#pragma unroll
  for (int t = 0; t < S; t++)
    st_fr(A.out[0] + (size_t)t * A.B + k, t == 0 ? fr_reduce1(x[0]) : fr_mulc(A.post_tab.ld(t), x[t]));
}

// ----------------------------------------------------- per-size tables --
// For one (n, log2 s): the four-step twiddles of size N in both directions,
// the coset factors (7 w_M^j)^k / N of every slice (times R, which also
// converts canonical coefficients to Montgomery form), the outer twiddles of
// the quotient INTT with its scale 7^-k, all as constant multipliers (frc).
// The scale's other part, 7^-(N t) of the cross-slice stage's output t, is a
// table of s constants on the host.  They depend only on the sizes, so a
// context builds them on first use and reuses them.
struct NttSizeArgs {
  FrcTab tw_fwd;   // [b * L1 + t] = w_N^(b t), b < L2, t < L1
  FrcTab tw_inv;   // [b * L2 + t] = w_N^-(b t), b < L1, t < L2
  FrcTab coset;    // [j * N + pos(k)] = (7 w_M^j)^k / N, and to level 1
  FrcTab outer;    // [j * N + pos(k)] = w_M^-(j k) 7^-k, and from level 1
  uint32_t n, lb, l1, l2;
  fr ninv_l2;
  const NttTables* T;
  const DevConst* C;
};

__global__ void k_ntt_size_tables(NttSizeArgs A, NttTables T) {
  const uint64_t N = 1ull << A.n, M = N << A.lb;
  const uint32_t logm = A.n + A.lb;
  const uint64_t L1 = 1ull << A.l1, L2 = 1ull << A.l2;
  const uint64_t total = 2 * N + 2 * M;
  for (uint64_t e = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (uint64_t)gridDim.x * blockDim.x) {
    if (e < N) {
      const uint64_t b = e / L1, t = e % L1;
      const uint32_t ex = (uint32_t)((((b * t) & (N - 1)) << (kLog30 - A.n)) & ((1ull << kLog30) - 1));
      A.tw_fwd.st(e, frc_of(root_pow(T.wf_lo, T.wf_hi, ex)));
    } else if (e < 2 * N) {
      const uint64_t i = e - N, b = i / L2, t = i % L2;
      const uint32_t ex = (uint32_t)((((b * t) & (N - 1)) << (kLog30 - A.n)) & ((1ull << kLog30) - 1));
      A.tw_inv.st(i, frc_of(root_pow(T.wi_lo, T.wi_hi, ex)));
    } else if (e < 2 * N + M) {
      const uint64_t i = e - 2 * N, j = i >> A.n, k = i & (N - 1);
      const uint32_t ex = (uint32_t)(((j * k) & (M - 1)) << (kLog30 - logm));
      fr f = fr_mul(fr_mul(ld_fr(T.p7_hi + (k >> kLoBits)), ld_fr(T.p7_lo + (k & kLoMask))),
                    root_pow(T.wf_lo, T.wf_hi, ex));
      A.coset.st((j << A.n) + tab_pos(k, A.l1, A.l2), frc_of(fr_mul(f, A.ninv_l2)));
    } else {
      const uint64_t i = e - 2 * N - M, j = i >> A.n, k = i & (N - 1);
      const uint32_t ex = (uint32_t)(((j * k) & (M - 1)) << (kLog30 - logm));
      const fr s7 = fr_mul(ld_fr(T.s7_hi + (k >> kLoBits)), ld_fr(T.s7_lo + (k & kLoMask)));  // 7^-k, level 0
      A.outer.st((j << A.n) + tab_pos(k, A.l1, A.l2), frc_of(fr_mul(root_pow(T.wi_lo, T.wi_hi, ex), s7)));
    }
  }
}

// ------------------------------------------------------- per-proof kernels --

struct NttSliceTabArgs {
  fr* lo;            // [s][2^hbits] c_j^b (level 1)
  fr* hi;            // [s][2^(n-hbits)] c_j^(a 2^hbits) / N (level 2)
  frc* zinv;         // [s] (7^N w_s^j - 1)^-1 M^-1
  uint32_t s, n, hbits, logm;
  fr ninv_l2;        // N^-1 at level 2
  fr minv_l1;        // M^-1 at level 1
  const fr* wf_lo; const fr* wf_hi;
  const DevConst* C;
};

__global__ void k_ntt_slice_tables(NttSliceTabArgs A) {
  const DevConst* C = A.C;
  const uint32_t nlo = 1u << A.hbits, nhi = 1u << (A.n - A.hbits);
  const uint32_t per = nlo + nhi;
  const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < (uint64_t)A.s * per) {
    const uint32_t j = (uint32_t)(i / per), e = (uint32_t)(i % per);
    // c_j = 7 w_M^j
    const uint32_t ex = (j << (kLog30 - A.logm)) & ((1u << kLog30) - 1);
    fr cj = fr_mul(C->small[7], root_pow(A.wf_lo, A.wf_hi, ex));
    if (e < nlo) {
      A.lo[(size_t)j * nlo + e] = fr_pow_dev(cj, e, C);
    } else {
      const uint32_t a = e - nlo;
      fr v = fr_pow_dev(cj, (uint64_t)a << A.hbits, C);
      A.hi[(size_t)j * nhi + a] = fr_mul(v, A.ninv_l2);  // level 2
    }
  }
  if (i < A.s) {
    // z_H on slice j: (7 w_M^j w_N^i)^N - 1 = 7^N w_s^j - 1
    const uint32_t j = (uint32_t)i;
    fr s7n = fr_pow_dev(C->small[7], 1ull << A.n, C);
    const uint32_t ex = (j << (kLog30 - (A.logm - A.n))) & ((1u << kLog30) - 1);
    fr zj = fr_sub(fr_mul(s7n, root_pow(A.wf_lo, A.wf_hi, ex)), C->one);
    fr inv = fr_inv_binary(from_mont(zj));        // canonical
    A.zinv[j] = frc_of(fr_mul(fr_mul(inv, C->r2), A.minv_l1));
  }
}

struct NttGateArgs {      // slice blockIdx.y of the launch
  const fr* col[kMaxCols];  // slice evaluations, level 1
  uint64_t col_y;           // elements from one slice's evaluations to the next's
  fr* qhat;                 // slice output
  const frc* zinv;          // constant of this slice
  const fr* sub;            // nullptr, or values subtracted after the scaling (level 1)
  uint64_t N;
  uint32_t gate, d, c;       // gate word, degree, columns
};

// f at the slice points, times the slice constant 1 / (z_H M): Plonk; product
// q w1 .. w_{d-1} - o; sum g_1 .. g_d + g_{d+1} + .. + g_c (all at level 1).
__global__ void __launch_bounds__(256) k_ntt_gate(NttGateArgs A) {
  const frc zi = ld_frc(A.zinv + blockIdx.y);
  const uint64_t cy = A.col_y * blockIdx.y;
  auto col = [&](uint32_t j, uint64_t p) { return ld_fr(A.col[j] + cy + p); };
  for (uint64_t p = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; p < A.N;
       p += (uint64_t)gridDim.x * blockDim.x) {
    fr f;
    if (A.gate == ZC_GATE_PLONK) {
      // a (qL + qM b) + qR b + qO c with one reduction for the three products
      const fr b = col(6, p);
      const fr u = fr_add(col(0, p), fr_mul_inl(col(2, p), b));
      f = fr_mul_sum3(col(5, p), u, col(1, p), b, col(3, p), col(7, p));
      f = fr_add(f, col(4, p));
    } else {
      f = col(0, p);
      for (uint32_t j = 1; j < A.d; j++) f = fr_mul_inl(f, col(j, p));
      if (A.gate == ZC_GATE_PRODUCT) f = fr_sub(f, col(A.d, p));
      else
        for (uint32_t j = A.d; j < A.c; j++) f = fr_add(f, col(j, p));
    }
    f = fr_mulc(zi, f);
    if (A.sub) f = fr_sub(f, ld_fr(A.sub + p));
    st_fr(A.qhat + A.N * blockIdx.y + p, f);
  }
}

// ------------------------------------------------ step-radix domain --
// D = D_big u D_small, D_big = 7 <w_M> (M = 2^lb N), D_small = sigma H with
// sigma = 7 w_{2M} (Sec. 4, degree scaling: a transform of M + N points
// from power-of-two transforms plus element-wise work).  q = q_big +
// (x^M - 7^M) q_small: q_big is the INTT over D_big of qhat there; on
// D_small, x^M = sigma^M, so q_small = INTT over D_small of
// (qhat - q_big) / kappa, kappa = sigma^M - 7^M.

struct NttStepTabArgs {
  FrcTab coset;   // [pos(k)] sigma^k / N, and to level 1
  fr* unscale;    // [k] w_{2M}^-k, level 1
  uint32_t n, l1, l2, shift2m;  // exponent shift of w_{2M} in the 2^30 tables: 30 - log2(2M)
  fr ninv_l2;
  NttTables T;
};

__global__ void k_ntt_step_tables(NttStepTabArgs A) {
  const uint64_t N = 1ull << A.n;
  for (uint64_t k = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; k < N; k += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t ex = (uint32_t)((k << A.shift2m) & ((1ull << kLog30) - 1));
    const fr p7 = fr_mul(ld_fr(A.T.p7_hi + (k >> kLoBits)), ld_fr(A.T.p7_lo + (k & kLoMask)));  // 7^k
    A.coset.st(tab_pos(k, A.l1, A.l2), frc_of(fr_mul(fr_mul(p7, root_pow(A.T.wf_lo, A.T.wf_hi, ex)), A.ninv_l2)));
    st_fr(A.unscale + k, root_pow(A.T.wi_lo, A.T.wi_hi, ex));
  }
}

// q_big evaluated on D_small starts with its reduction modulo x^N - sigma^N,
// scaled by 1/kappa: rho[k] = sum_m q[k + m N] sigma^(mN) / kappa.
struct NttStepReduceArgs {
  const fr* q;       // q_big, M canonical coefficients
  fr* rho;           // N outputs, level 0
  const fr* cm;      // 2^lb constants sigma^(mN) / kappa, level 1
  uint64_t N;
  uint32_t parts;    // M / N
};

__global__ void k_ntt_step_reduce(NttStepReduceArgs A) {
  for (uint64_t k = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; k < A.N;
       k += (uint64_t)gridDim.x * blockDim.x) {
    fr acc = fr_mul(ld_fr(A.q + k), ld_fr(A.cm));
    for (uint32_t m = 1; m < A.parts; m++) acc = fr_add(acc, fr_mul(ld_fr(A.q + k + m * A.N), ld_fr(A.cm + m)));
    st_fr(A.rho + k, acc);
  }
}

// q_small[k] = w_{2M}^-k x[k] (x: the small part's INTT, which carried the
// factor 7^-k); q[M + k] = q_small[k], q[k] -= 7^M q_small[k].
struct NttStepCombineArgs {
  fr* q;             // M + N coefficients; x in q[M .. M + N)
  const fr* unscale;
  const fr* s7m;     // 7^M, level 1
  uint64_t N, M;
};

__global__ void k_ntt_step_combine(NttStepCombineArgs A) {
  const fr c = ld_fr(A.s7m);
  for (uint64_t k = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; k < A.N;
       k += (uint64_t)gridDim.x * blockDim.x) {
    const fr t = fr_mul(ld_fr(A.q + A.M + k), ld_fr(A.unscale + k));
    st_fr(A.q + A.M + k, t);
    st_fr(A.q + k, fr_sub(ld_fr(A.q + k), fr_mul(t, c)));
  }
}

struct NttZArgs {
  NttState* st;
  const uint8_t* roots;  // c column roots then root(q)
  int c;
  uint32_t n;
  uint32_t S0[8];
  fr* zpow;              // z^(2^i), i < nz (level 1)
  uint32_t nz;           // powers the openings use, z^N and z^32 among them
  const DevConst* C;
};

// Transcript up to z (two warps, see ShaPair; again while z^N = 1) and the
// powers z^(2^i), of which z^N is one.  Launched with 64 threads.
__global__ void __launch_bounds__(64) k_ntt_z(NttZArgs A) {
  __shared__ ShaPair Z;
  __shared__ uint32_t blk[32];
  __shared__ uint32_t again;
  const DevConst* C = A.C;
  uint32_t S[8];
  for (int i = 0; i < 8; i++) S[i] = A.S0[i];
  tr_absorb32(Z, blk, S, A.roots, A.c + 1);
  for (int tries = 0; tries < 64; tries++) {
    const fr raw = tr_squeeze(Z, S);
    if (threadIdx.x == 0) {
      fr p = fr_mul(raw, C->r2);
      A.st->z = p;
      for (uint32_t i = 0; i < A.nz; i++) {
        A.zpow[i] = p;
        if (i == A.n) {
          A.st->zpow_n = p;
          again = fr_equal(p, C->one) ? 1u : 0u;
        }
        p = fr_mul(p, p);
      }
    }
    __syncthreads();
    if (!again) return;
    __syncthreads();
  }
  if (threadIdx.x == 0) A.st->err |= 1u;
}

// Evaluate sum_k x[k] z^k for each item (level-0 x); every warp takes a
// contiguous segment, lane l the elements seg + l + 32 m, Horner in z^32.
struct NttOpenArgs {
  const fr* x[kMaxCols + 1];
  uint64_t len[kMaxCols + 1];
  const fr* zpow;     // z^(2^i)
  fr* partials;       // [item][blocks]
  uint32_t nblk;
  uint32_t seg;       // elements per warp segment (multiple of 32)
};

// Steps per warp segment of the openings: a segment ends in one product by
// z^base (up to log2 M products), which 128 steps hide; with fewer than ~512
// such segments in the longest vector the chain of steps is the time, so the
// segments get shorter, down to 8 steps (n = 12: one warp per column and 128
// steps took 128 us).
static uint32_t open_steps(uint64_t M) {
  const uint64_t m = M / (32 * 512);
  return (uint32_t)(m < 8 ? 8 : m > 128 ? 128 : m);
}

__device__ fr zpow_of(const fr* zp, uint64_t e, const fr& one) {
  fr acc = one;
  for (int i = 0; e; i++, e >>= 1)
    if (e & 1) acc = fr_mul(acc, ld_fr(zp + i));
  return acc;
}

__global__ void __launch_bounds__(256) k_ntt_open(NttOpenArgs A, const DevConst* C) {
  const int item = blockIdx.y;
  const fr* x = A.x[item];
  const uint64_t len = A.len[item];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const frc z32 = frc_of(ld_fr(A.zpow + 5));
  fr tot = fr_zero();
  const uint64_t nseg = (len + A.seg - 1) / A.seg;
  for (uint64_t sgi = (uint64_t)blockIdx.x * 8 + warp; sgi < nseg; sgi += (uint64_t)gridDim.x * 8) {
    const uint64_t base = sgi * A.seg;
    const uint64_t cnt = A.seg < len - base ? A.seg : len - base;
    const uint32_t mcount = (uint32_t)((cnt + 31) / 32);
    fr acc = fr_zero();
    auto value = [&](int32_t m) {
      const uint64_t k = base + lane + 32ull * (uint32_t)m;
      return m >= 0 && k < len ? ld_fr(x + k) : fr_zero();
    };
    fr nx = value((int32_t)mcount - 1);  // the next step's value is loaded during the present product
    for (int32_t m = (int32_t)mcount - 1; m >= 0; m--) {
      const fr xk = nx;
      nx = value(m - 1);
      // while the warp's accumulators and values are all zero (the zero top
      // of an honest quotient) the step would multiply zeros: skip it
      if (__all_sync(0xffffffffu, fr_is_zero(acc) && fr_is_zero(xk))) continue;
      acc = fr_add(fr_mulc(z32, acc), xk);
    }
    if (__all_sync(0xffffffffu, fr_is_zero(acc))) continue;
    acc = fr_mul(acc, zpow_of(A.zpow, base + lane, C->one));
    tot = fr_add(tot, acc);
  }
  __shared__ fr red[8];
  tot = warp_sum(tot);
  if (lane == 0) red[warp] = tot;
  __syncthreads();
  if (threadIdx.x == 0) {
    fr s = fr_zero();
    for (int w = 0; w < 8; w++) s = fr_add(s, red[w]);
    st_fr(A.partials + (size_t)item * A.nblk + blockIdx.x, s);
  }
}

struct NttFinalArgs {
  const fr* partials;
  uint32_t nblk;
  int c;
  uint32_t gate, n, d, logm;
  fr ninv_l1;
  const uint8_t* qroot;
  NttState* st;
  uint8_t* proof;
};

__global__ void k_ntt_final(NttFinalArgs A) {
  // one warp per opening: lanes add strided block partials, then shuffles
  const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int item = threadIdx.x >> 5; item <= A.c; item += nw) {
    fr s = fr_zero();
    for (uint32_t b = lane; b < A.nblk; b += 32) s = fr_add(s, ld_fr_cg(A.partials + (size_t)item * A.nblk + b));
    s = warp_sum(s);
    if (lane == 0) {
      if (item < A.c) s = fr_mul(s, A.ninv_l1);  // coefficients carry the factor N
      uint8_t* o = A.proof + 52 + 32 * item;
      for (int i = 0; i < 8; i++)
        for (int b = 0; b < 4; b++) o[4 * i + b] = (uint8_t)(s.v[i] >> (8 * b));
    }
  }
  if (threadIdx.x == 0) {
    const char* mg = A.st->err ? "ZCE!" : "ZCN1";
    for (int b = 0; b < 4; b++) A.proof[b] = (uint8_t)mg[b];
    uint32_t hv[4] = {A.gate, A.n, A.d, A.logm};
    for (int q = 0; q < 4; q++)
      for (int b = 0; b < 4; b++) A.proof[4 + 4 * q + b] = (uint8_t)(hv[q] >> (8 * b));
    for (int b = 0; b < 32; b++) A.proof[20 + b] = A.qroot[b];
  }
}

__global__ void k_ntt_state_init(NttState* st) {
  if (threadIdx.x == 0) st->err = 0;
}

// ------------------------------------------------------------------ host --

static zc_status ensure_tables(zc_ctx* ctx, cudaStream_t st, NttTables** out) {
  std::lock_guard<std::mutex> lk(g_tabs_mu);
  NttTables& T = g_tabs_by_dev[ctx->device];
  if (!T.ready) {
    const size_t n4 = kStageTab, n15 = 1u << kLoBits;
    size_t bytes = sizeof(frc) * 2 * n4 + sizeof(fr) * 8 * n15;
    if (cudaMalloc(&T.mem, bytes) != cudaSuccess) {
      cudaGetLastError();
      ctx->err = "cudaMalloc NTT tables";
      return ZC_ERR_OOM;
    }
    T.dft_fwd = FrcTab::make(T.mem, n4);
    T.dft_inv = FrcTab::make(static_cast<frc*>(T.mem) + n4, n4);
    fr* p = reinterpret_cast<fr*>(static_cast<frc*>(T.mem) + 2 * n4);
    T.wf_lo = p; p += n15;
    T.wf_hi = p; p += n15;
    T.wi_lo = p; p += n15;
    T.wi_hi = p; p += n15;
    T.s7_lo = p; p += n15;
    T.s7_hi = p; p += n15;
    T.p7_lo = p; p += n15;
    T.p7_hi = p; p += n15;
    const DevConst& C = ctx->hconst;
    // w_2^32 = 7^((r-1)/2^32); w_2^30 = (w_2^32)^4
    uint32_t e[8];
    for (int i = 0; i < 7; i++) e[i] = p_limb(i + 1);
    e[7] = 0;
    fr seven = h_from_u64(7);
    fr acc = h_from_u64(1), base = seven;
    for (int i = 0; i < 8; i++)
      for (int b = 0; b < 32; b++) {
        if ((e[i] >> b) & 1) acc = h_canon_mul(acc, base, C);
        base = h_canon_mul(base, base, C);
      }
    T.w32h = acc;
    fr w30 = h_canon_mul(acc, acc, C);
    w30 = h_canon_mul(w30, w30, C);
    NttTabArgs a{};
    a.dft_fwd = T.dft_fwd; a.dft_inv = T.dft_inv;
    a.wf_lo = T.wf_lo; a.wf_hi = T.wf_hi; a.wi_lo = T.wi_lo; a.wi_hi = T.wi_hi;
    a.s7_lo = T.s7_lo; a.s7_hi = T.s7_hi;
    a.p7_lo = T.p7_lo; a.p7_hi = T.p7_hi;
    a.w30 = fr_mul_g(w30, C.r2);
    a.w30i = fr_mul_g(h_inv(w30, C), C.r2);
    {
      const fr w8 = h_pow(w30, 1ull << 27, C), w8i = h_inv(w8, C);
      for (int q = 0; q < 3; q++) {
        T.c_fwd[q] = h_frc(h_pow(w8, q + 1, C), C);
        T.c_inv[q] = h_frc(h_pow(w8i, q + 1, C), C);
      }
    }
    a.seveninv = fr_mul_g(h_inv(seven, C), C.r2);
    a.C = ctx->dconst;
    k_ntt_tables<<<(n15 + 255) / 256, 256, 0, st>>>(a);
    if (cudaStreamSynchronize(st) != cudaSuccess) {
      ctx->err = "NTT table set-up failed";
      return ZC_ERR_CUDA;
    }
    T.ready = true;
  }
  *out = &T;
  return ZC_OK;
}

// Pass variants: 8 elements per thread, up to 512 threads, a minimum number of
// resident CTAs per SM (caps registers).  The context's tuning picks the tile
// and residency.
template <int MAXT, int MINB>
static void launch_pass_variant(const NttPassArgs& a, dim3 grid, const NttPlan& P, cudaStream_t st) {
  if (ntt_fast(P, a.logL, a.B) && a.pre != PRE_COSET && (a.post == POST_NONE || a.post == POST_TAB))
    k_ntt_pass<MAXT, MINB, true><<<grid, P.tile / 8, P.tile * sizeof(fr), st>>>(a);
  else
    k_ntt_pass<MAXT, MINB, false><<<grid, P.tile / 8, P.tile * sizeof(fr), st>>>(a);
}

static void set_pass_attributes() {
  cudaFuncSetAttribute(k_ntt_pass_small, cudaFuncAttributeMaxDynamicSharedMemorySize, 1024 * 64);
  cudaFuncSetAttribute(k_ntt_pass<128, 4, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 1024 * 32);
  cudaFuncSetAttribute(k_ntt_pass<128, 4, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 1024 * 32);
  cudaFuncSetAttribute(k_ntt_pass<256, 2, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 2048 * 32);
  cudaFuncSetAttribute(k_ntt_pass<256, 2, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 2048 * 32);
  cudaFuncSetAttribute(k_ntt_pass<256, 1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 2048 * 32);
  cudaFuncSetAttribute(k_ntt_pass<256, 1, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 2048 * 32);
  cudaFuncSetAttribute(k_ntt_pass<512, 1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 4096 * 32);
  cudaFuncSetAttribute(k_ntt_pass<512, 1, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 4096 * 32);
}

static int g_attr_done[64] = {0};
static void ensure_pass_attributes(int dev) {
  std::lock_guard<std::mutex> lk(g_tabs_mu);
  if (!g_attr_done[dev]) {
    set_pass_attributes();
    g_attr_done[dev] = 1;
  }
}

// Launches of at most this many elements take two per thread (proofs by limit
// 2^17 / 2^18 / 2^19 / 2^20: n = 14 472, 474, 461, 462 us; n = 16 834, 815,
// 822, 838; n = 17 1320, 1322, 1308, 1405; with eight always n = 12 441
// against 390).
constexpr uint64_t kSmallElems = 1ull << 19;

static void set_dft(NttPassArgs& a, const NttTables* T, bool inverse) {
  const frc* c = inverse ? T->c_inv : T->c_fwd;
  a.dft = inverse ? T->dft_inv : T->dft_fwd;
  a.w8 = c[0];
  a.w4 = c[1];
  a.w83 = c[2];
}

// launch one batched pass over `items` columns
static zc_status run_pass(zc_ctx* ctx, cudaStream_t st, NttPassArgs& a, int items, uint64_t B, uint32_t slices = 1) {
  const uint32_t logL = a.logL;
  const uint32_t tile = (uint32_t)ctx->tuned(ZC_FORM_NTT, ctx->cur_n, ZC_TUNE_NTT_TILE_LOG);
  const int minb = ctx->tuned(ZC_FORM_NTT, ctx->cur_n, ZC_TUNE_NTT_MINB);
  NttPlan P;
  // few elements, and no tile or residency asked for: two per thread
  const bool small = !tile && !minb && (uint64_t)items * slices * (B << logL) <= kSmallElems && a.pre != PRE_COSET &&
                     (a.post == POST_NONE || a.post == POST_TAB) && ntt_plan_small(logL, B, &P);
  if (!small) P = ntt_plan(logL, B, tile);
  a.logW = P.logW;
  a.items = (uint32_t)items;
  a.B = (uint32_t)B;
  const dim3 grid((uint32_t)(P.blocks * (uint64_t)items), slices);
  if (small) k_ntt_pass_small<<<grid, P.tile / 2, 2 * P.tile * sizeof(fr), st>>>(a);
  else if (P.logTile == 12) launch_pass_variant<512, 1>(a, grid, P, st);
  else if (P.logTile == 11 && minb != 1) launch_pass_variant<256, 2>(a, grid, P, st);
  else if (P.logTile == 11) launch_pass_variant<256, 1>(a, grid, P, st);
  else launch_pass_variant<128, 4>(a, grid, P, st);
  ctx->launches++;
  return ZC_OK;
}

// Room for `bytes` more of tables within the context's budget: the least
// recently used sizes go, but never one that a captured batch graph or a set
// being prepared holds.  False when that leaves too little (must: what can go
// goes, and the budget is passed by the rest).
static bool table_room(zc_ctx* ctx, size_t bytes, bool must) {
  size_t used = 0, held = 0;
  for (auto& e : ctx->ntt_cache) {
    used += e.bytes + e.step_bytes;
    if (e.own.use_count() > 1) held += e.bytes + e.step_bytes;
  }
  if (!must && held + bytes > ctx->ntt_cache_budget) return false;
  while (used + bytes > ctx->ntt_cache_budget) {
    size_t old = SIZE_MAX;
    for (size_t i = 0; i < ctx->ntt_cache.size(); i++)
      if (ctx->ntt_cache[i].own.use_count() == 1 &&
          (old == SIZE_MAX || ctx->ntt_cache[i].stamp < ctx->ntt_cache[old].stamp))
        old = i;
    if (old == SIZE_MAX) break;
    used -= ctx->ntt_cache[old].bytes + ctx->ntt_cache[old].step_bytes;
    ctx->ntt_cache.erase(ctx->ntt_cache.begin() + old);
  }
  return true;
}

// The per-size tables of (n, lb), built on first use; nullptr when they
// would exceed the context's table budget (the passes then form every factor
// from the two-level power tables instead).
static zc_ctx::NttSizeTables* size_tables(zc_ctx* user, const NttTables* T, uint32_t n, uint32_t lb,
                                          uint32_t l1, uint32_t l2, bool step, cudaStream_t st) {
  zc_ctx* ctx = user->table_owner ? user->table_owner : user;
  const uint64_t N = 1ull << n, M = N << lb;
  for (auto& e : ctx->ntt_cache)
    if (e.n == n && e.lb == lb && e.l1 == l1) {
      e.stamp = ++ctx->ntt_cache_clock;
      return &e;
    }
  const uint64_t s = 1ull << lb;
  const size_t bytes = sizeof(frc) * (2 * N + 2 * M + 2 * s);
  if (ctx->ntt_cache_frozen || bytes > ctx->ntt_cache_budget) return nullptr;
  if (!table_room(ctx, bytes, step)) return nullptr;  // a step-radix domain has no other route
  zc_ctx::NttSizeTables e;
  e.own = std::make_shared<zc_ctx::NttTableMem>();
  if (cudaMalloc(&e.own->mem, bytes) != cudaSuccess) {
    cudaGetLastError();
    e.own->mem = nullptr;
    return nullptr;
  }
  e.n = n;
  e.lb = lb;
  e.l1 = l1;
  e.bytes = bytes;
  frc* q = static_cast<frc*>(e.own->mem);
  e.tw_fwd = FrcTab::make(q, N); q += N;
  e.tw_inv = FrcTab::make(q, N); q += N;
  e.coset = FrcTab::make(q, M); q += M;
  e.outer = FrcTab::make(q, M); q += M;
  e.fin = FrcTab::make(q, s); q += s;
  e.zinv = q;
  {
    // on the host: 7^-(N t), t < s; (z_H on slice j)^-1 M^-1 = (7^N w_s^j - 1)^-1 M^-1
    const DevConst& C = ctx->hconst;
    const fr ws = h_pow(T->w32h, (1ull << 32) >> lb, C);
    const fr s7n = h_pow(h_from_u64(7), N, C), minv = h_inv(h_from_u64(M), C);
    const fr s7i = h_inv(s7n, C);
    std::vector<frc> hc(2 * s);
    fr wj = h_from_u64(1), fj = h_from_u64(1);
    for (uint64_t j = 0; j < s; j++) {
      const fr v = fr_sub_g(h_canon_mul(s7n, wj, C), h_from_u64(1));
      const frc fc = h_frc(fj, C);
      for (int h = 0; h < 4; h++)  // planes, as FrcTab
        std::memcpy(reinterpret_cast<char*>(hc.data()) + 16 * (h * s + j), reinterpret_cast<const char*>(&fc) + 16 * h, 16);
      hc[s + j] = h_frc(h_canon_mul(h_inv(v, C), minv, C), C);
      fj = h_canon_mul(fj, s7i, C);
      wj = h_canon_mul(wj, ws, C);
    }
    if (cudaMemcpyAsync(e.fin.p, hc.data(), sizeof(frc) * 2 * s, cudaMemcpyHostToDevice, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess) {
      cudaGetLastError();
      return nullptr;
    }
  }
  NttSizeArgs a{};
  a.tw_fwd = e.tw_fwd;
  a.tw_inv = e.tw_inv;
  a.coset = e.coset;
  a.outer = e.outer;
  a.n = n;
  a.lb = lb;
  a.l1 = l1;
  a.l2 = l2;
  const DevConst& C = ctx->hconst;
  a.ninv_l2 = fr_mul_g(fr_mul_g(h_inv(h_from_u64(N), C), C.r2), C.r2);
  a.C = ctx->dconst;
  const uint64_t total = 2 * N + 2 * M;
  k_ntt_size_tables<<<(unsigned)std::min<uint64_t>((total + 255) / 256, (uint64_t)ctx->sm_count * 16), 256, 0,
                      st>>>(a, *T);
  ctx->launches++;
  e.stamp = ++ctx->ntt_cache_clock;
  ctx->ntt_cache.push_back(e);
  return &ctx->ntt_cache.back();
}

static void pass_defaults(NttPassArgs& a) {
  std::memset(&a, 0, sizeof a);
}

static NttDomain domain_of(const zc_params* p) {
  NttDomain D;
  ntt_domain(p->n, p->d, p->log_blowup, &D);  // validated by check_params
  return D;
}

size_t ntt_scratch_bytes(const zc_params* p, int sm_count, bool q_direct) {
  const NttDomain D = domain_of(p);
  const uint32_t n = p->n, lb = D.k;
  const int c = gate_ncols(p->gate, p->d);
  const uint64_t N = 1ull << n, Mb = N << lb, s = 1ull << lb, M = D.M;
  const uint32_t hbits = (n + 1) / 2;
  const uint32_t nlo = 1u << hbits, nhi = 1u << (n - hbits);
  const uint32_t nblk_open = 2 * (uint32_t)sm_count;
  const size_t psize = 20 + 32 + 32 * ((size_t)c + 1);
  size_t need = 2 * align_up(sizeof(fr) * N, 256) * c;  // coefficients + slice buffer
  need += align_up(sizeof(fr) * M, 256);                  // qhat (both parts)
  if (!q_direct) need += align_up(sizeof(fr) * M, 256);   // q
  if (D.step) need += 2 * align_up(sizeof(fr) * N, 256);  // q_big reduced, and its LDE
  need += align_up(sizeof(fr) * s * (nlo + nhi), 256) + align_up(sizeof(frc) * s, 256);
  need += align_up(sizeof(fr) * (c + 1) * nblk_open, 256) + align_up(sizeof(fr) * 32, 256);
  need += align_up(sizeof(NttState), 256) + align_up(psize, 256) + align_up(32 * (size_t)(c + 1), 256);
  need += root_scratch_bytes(c, N) + root_scratch_bytes(1, M) + 8192;
  (void)Mb;
  return need;
}

// Side stream and per-column events for pipelined uploads of host columns
// (created on first use, freed by zc_destroy).
zc_status ensure_upload_stream(zc_ctx* ctx, int c) {
  if (!ctx->up_stream) {
    if (cudaStreamCreateWithFlags(&ctx->up_stream, cudaStreamNonBlocking) != cudaSuccess ||
        cudaEventCreateWithFlags(&ctx->up_fork, cudaEventDisableTiming) != cudaSuccess) {
      cudaGetLastError();
      ctx->err = "cannot create the upload stream";
      return ZC_ERR_CUDA;
    }
  }
  while ((int)ctx->up_ev.size() < c) {
    cudaEvent_t e;
    if (cudaEventCreateWithFlags(&e, cudaEventDisableTiming) != cudaSuccess) {
      cudaGetLastError();
      ctx->err = "cannot create an upload event";
      return ZC_ERR_CUDA;
    }
    ctx->up_ev.push_back(e);
  }
  return ZC_OK;
}

// Transforms of 2^n points run as two four-step passes (sub-DFTs of
// 2^ceil(n/2) and 2^floor(n/2) points) from n = 12 on (a single pass holds at
// most 2^12 points; at 2^12 the two passes' extra CTAs already win), or from
// a tuned size, else as one pass per transform.
static bool ntt_two_pass(const zc_ctx* ctx, uint32_t n) {
  if (n > 12) return true;  // one pass holds at most a 2^12 transform
  const int32_t t = ctx->tuned(ZC_FORM_NTT, n, ZC_TUNE_NTT_TWO_LOG);
  return n >= (uint32_t)(t > 0 ? t : 12) && n >= 2;
}

// coset factors (frc), unscale factors, 8 + 2^lb constants
static size_t step_table_bytes(uint32_t n, uint32_t lb) { return sizeof(fr) * ((3ull << n) + 8 + (1ull << lb)); }

// The step-radix tables of a cache entry (lb = k): built once, with the
// host-computed constants of the small part.  False if they cannot be made.
static bool step_tables(zc_ctx* user, zc_ctx::NttSizeTables*& e, const NttTables* T, cudaStream_t st) {
  if (e->step_bytes) return true;
  zc_ctx* ctx = user->table_owner ? user->table_owner : user;
  if (ctx->ntt_cache_frozen) return false;
  // room for them too, with this entry held; e moves as others go
  const std::shared_ptr<zc_ctx::NttTableMem> own = e->own;
  table_room(ctx, step_table_bytes(e->n, e->lb), true);
  for (auto& t : ctx->ntt_cache)
    if (t.own == own) e = &t;
  const uint32_t n = e->n, lb = e->lb;
  const uint64_t N = 1ull << n, M = N << lb, parts = 1ull << lb;
  if (n + lb + 1 > (uint32_t)kLog30 || parts > 64) return false;
  const size_t nconst = 8 + parts;
  const size_t bytes = step_table_bytes(n, lb);
  void* mem = nullptr;
  if (cudaMalloc(&mem, bytes) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  const FrcTab coset = FrcTab::make(mem, N);
  fr* unscale = reinterpret_cast<fr*>(static_cast<frc*>(mem) + N);
  fr* cst = unscale + N;
  const DevConst& C = ctx->hconst;
  // sigma = 7 w_{2M}; kappa = sigma^M - 7^M; z_H on D_small = sigma^N - 1
  const fr w2m = h_pow(T->w32h, (1ull << 32) >> (n + lb + 1), C);
  const fr seven = h_from_u64(7), one = h_from_u64(1);
  const fr sigma = h_canon_mul(seven, w2m, C);
  const fr s7m = h_pow(seven, M, C);
  const fr kinv = h_inv(fr_sub_g(h_pow(sigma, M, C), s7m), C);
  const fr ninv = h_inv(h_from_u64(N), C);
  const fr sn = h_pow(sigma, N, C);
  std::vector<fr> hc(nconst, fr_zero());
  const frc zi = h_frc(h_canon_mul(h_canon_mul(h_inv(fr_sub_g(sn, one), C), kinv, C), ninv, C), C);
  hc[0] = zi.w;
  hc[1] = zi.q;
  hc[2] = h_canon_mul(s7m, C.one, C);
  fr pm = one;
  for (uint64_t m = 0; m < parts; m++) {
    hc[8 + m] = h_canon_mul(h_canon_mul(pm, kinv, C), C.one, C);  // level 1
    pm = h_canon_mul(pm, sn, C);
  }
  if (cudaMemcpyAsync(cst, hc.data(), sizeof(fr) * nconst, cudaMemcpyHostToDevice, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess) {
    cudaGetLastError();
    cudaFree(mem);
    return false;
  }
  NttStepTabArgs a{};
  a.coset = coset;
  a.unscale = unscale;
  a.n = n;
  a.l1 = e->l1;
  a.l2 = n - e->l1;
  a.shift2m = kLog30 - (n + lb + 1);
  a.ninv_l2 = fr_mul_g(fr_mul_g(ninv, C.r2), C.r2);
  a.T = *T;
  k_ntt_step_tables<<<(unsigned)std::min<uint64_t>((N + 255) / 256, (uint64_t)ctx->sm_count * 16), 256, 0, st>>>(a);
  if (cudaGetLastError() != cudaSuccess) {
    cudaFree(mem);
    return false;
  }
  e->own->step_mem = mem;
  e->step_bytes = bytes;
  e->step_coset = coset;
  e->step_unscale = unscale;
  e->step_const = cst;
  user->launches++;
  return true;
}

// ---- Reed-Solomon row encoding for the hash-based commitment (zc_pcs.cu):
// row i of column j (w = 2^nc coefficients) evaluated at the W = 4w points
// 7 w_W^k, written to enc[j][k m + i].  Slice s (k = s + 4 k') is one pass
// of w-point transforms over the m rows with the factor (7 w_W^s)^l applied
// on load; canonical columns in, canonical codewords out.

struct PcsTabArgs {
  FrcTab tab;         // [s w + l] = (7 w_W^s)^l
  uint32_t nc;        // w = 2^nc
  uint32_t shiftW;    // 30 - log2 W
  NttTables T;
};

__global__ void k_pcs_tables(PcsTabArgs A) {
  const uint32_t w = 1u << A.nc, total = 4 * w;
  for (uint32_t e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
    const uint32_t s = e >> A.nc, l = e & (w - 1);
    const fr p7 = fr_mul(ld_fr(A.T.p7_hi + (l >> kLoBits)), ld_fr(A.T.p7_lo + (l & kLoMask)));  // 7^l
    const uint32_t ex = (uint32_t)((((uint64_t)s * l) << A.shiftW) & ((1ull << kLog30) - 1));
    A.tab.st(e, frc_of(fr_mul(p7, root_pow(A.T.wf_lo, A.T.wf_hi, ex))));
  }
}

zc_status pcs_encode(zc_ctx* ctx, const fr* const* cols, int c, uint32_t nr, uint32_t nc, fr* const* enc,
                     FrcTab tab, cudaStream_t st) {
  if (nc < 1 || nc > 12 || c < 1 || c > kMaxCols) {
    ctx->err = "pcs: rows of 2 .. 2^12 elements";
    return ZC_ERR_UNSUPPORTED;
  }
  ensure_pass_attributes(ctx->device);
  NttTables* T = nullptr;
  zc_status s0 = ensure_tables(ctx, st, &T);
  if (s0 != ZC_OK) return s0;
  const uint64_t w = 1ull << nc, m = 1ull << nr;
  PcsTabArgs ta{};
  ta.tab = tab;
  ta.nc = nc;
  ta.shiftW = kLog30 - (nc + 2);
  ta.T = *T;
  k_pcs_tables<<<(unsigned)std::min<uint64_t>((4 * w + 255) / 256, 1024), 256, 0, st>>>(ta);
  ctx->launches++;
  ctx->cur_n = nc;
  for (uint32_t sl = 0; sl < 4; sl++) {
    NttPassArgs a;
    pass_defaults(a);
    for (int j = 0; j < c; j++) {
      a.in[j] = cols[j];
      a.out[j] = enc[j] + sl * m;     // position k = sl + 4 k'
    }
    const NttMaps mp = maps_pcs(nr, nc);
    a.use(mp);
    set_dft(a, T, false);
    a.pre = PRE_TAB; a.pre_tab = tab.at(sl * w);
    zc_status rs = run_pass(ctx, st, a, c, mp.B);
    if (rs != ZC_OK) return rs;
  }
  return cudaGetLastError() == cudaSuccess ? ZC_OK : ZC_ERR_CUDA;
}

zc_status ntt_prepare(zc_ctx* ctx, const zc_params* p, cudaStream_t st, Holds* holds) {
  ensure_pass_attributes(ctx->device);
  NttTables* T = nullptr;
  zc_status s0 = ensure_tables(ctx, st, &T);
  if (s0 != ZC_OK) return s0;
  const NttDomain D = domain_of(p);
  const uint32_t n = p->n, lb = D.k;
  const bool two = ntt_two_pass(ctx, n);
  zc_ctx::NttSizeTables* ST = size_tables(ctx, T, n, lb, two ? (n + 1) / 2 : n, two ? n / 2 : 0, D.step, st);
  if (ST) holds->push_back(ST->own);
  if (D.step && (!ST || !step_tables(ctx, ST, T, st))) {
    ctx->err = "step-radix domain: tables unavailable";
    return ZC_ERR_OOM;
  }
  return cudaStreamSynchronize(st) == cudaSuccess ? ZC_OK : ZC_ERR_CUDA;
}

// Slices of N2 per launch: while one slice's passes have at most two waves of
// CTAs (1024 elements each, four per SM), several slices share a launch: each
// alone leaves most of the GPU idle for as long as a full one (n = 12: 3 x 54
// us of the proof's 670).
static uint32_t slices_per_launch(int sm_count, int c, uint64_t N, uint64_t s) {
  uint32_t k = 1;
  while (2 * k <= s && 2 * k * ((uint64_t)c * N / 1024 + 1) <= 8ull * sm_count) k *= 2;
  return k;
}

zc_status ntt_prove(zc_ctx* ctx, const zc_params* p, const void* const* cols, int on_dev,
                    const uint8_t (*roots)[32], cudaStream_t st, uint8_t* proof,
                    bool proof_on_dev, void* q_out, int q_on_dev) {
  const uint32_t gate = p->gate, n = p->n, d = p->d;
  ctx->cur_n = n;
  if (n > (uint32_t)kMaxNttN) {
    ctx->err = "NTT form supports n <= 24";
    return ZC_ERR_UNSUPPORTED;
  }
  const NttDomain D = domain_of(p);
  if (D.step && D.s != 0) {
    ctx->err = "step-radix domains take a small part of N points (s = 0)";
    return ZC_ERR_UNSUPPORTED;
  }
  const uint32_t lb = D.k;          // the big part 7 <w_Mb>, Mb = 2^lb N
  const uint32_t logm = n + lb;     // log2 Mb
  if (logm + (D.step ? 1 : 0) > (uint32_t)kLog30) {
    ctx->err = "domain larger than 2^30";
    return ZC_ERR_UNSUPPORTED;
  }
  const int c = gate_ncols(gate, d);
  const uint64_t N = 1ull << n, Mb = 1ull << logm, s = 1ull << lb;
  const uint64_t M = D.M;           // Mb, or Mb + N (step radix)
  const size_t psize = 20 + 32 + 32 * ((size_t)c + 1);
  ensure_pass_attributes(ctx->device);
  NttTables* T = nullptr;
  zc_status s0 = ensure_tables(ctx, st, &T);
  if (s0 != ZC_OK) return s0;

  const uint32_t hbits = (n + 1) / 2;
  const uint32_t nlo = 1u << hbits, nhi = 1u << (n - hbits);
  const uint32_t nblk_open = 2 * (uint32_t)ctx->sm_count;
  const bool q_direct = q_out && q_on_dev;
  // several slices per launch take more scratch than the proof needs: as many
  // as the arena has room for.  It is allocated larger only when it has to be
  // allocated anyway, never moved for this (a captured graph may use it), nor
  // on lanes and within the memory budget.
  const size_t need = ntt_scratch_bytes(p, ctx->sm_count, q_direct);
  const uint64_t Na = std::max<uint64_t>(N, 8);  // buffers of 256 bytes at least
  uint32_t sb = slices_per_launch(ctx->sm_count, c, N, s);
  auto more = [&] { return (size_t)(sb - 1) * c * Na * sizeof(fr); };
  if (ctx->arena.cap < need && !ctx->table_owner && !ctx->arena_borrowed && ensure_arena(ctx, need + more()) != ZC_OK)
    ctx->err.clear();
  zc_status s1 = ensure_arena(ctx, need);
  if (s1 != ZC_OK) return s1;
  while (sb > 1 && ctx->arena.cap < need + more()) sb /= 2;
  Arena& ar = ctx->arena;
  ar.reset();
  fr* coef[kMaxCols];
  fr* slb[kMaxCols];
  for (int j = 0; j < c; j++) coef[j] = ar.take<fr>(N);
  fr* const slices = ar.take<fr>((size_t)sb * c * Na);
  for (int j = 0; j < c; j++) slb[j] = slices + j * Na;
  fr* qhat = ar.take<fr>(M);
  fr* qv = q_direct ? static_cast<fr*>(q_out) : ar.take<fr>(M);
  fr* rho = D.step ? ar.take<fr>(N) : nullptr;   // q_big reduced mod x^N - sigma^N
  fr* vsm = D.step ? ar.take<fr>(N) : nullptr;   // its values on D_small
  fr* tlo = ar.take<fr>(s * nlo);
  fr* thi = ar.take<fr>(s * nhi);
  frc* zinv = ar.take<frc>(s);
  fr* opart = ar.take<fr>((size_t)(c + 1) * nblk_open);
  fr* zpow = ar.take<fr>(32);
  NttState* dstate = ar.take<NttState>(1);
  uint8_t* dproof = ar.take<uint8_t>(psize);
  uint8_t* droots = ar.take<uint8_t>(32 * (size_t)(c + 1));
  if (!droots) {
    ctx->err = "scratch arena too small";
    return ZC_ERR_OOM;
  }
  ctx->launches = 0;
  ctx->nev = 7;

  const bool two = ntt_two_pass(ctx, n);
  const uint32_t l1 = two ? (n + 1) / 2 : n;   // first digit
  const uint32_t l2 = two ? n / 2 : 0;         // second digit
  zc_status rs;
  zc_ctx::NttSizeTables* ST = size_tables(ctx, T, n, lb, l1, l2, D.step, st);
  if (D.step && (!ST || !step_tables(ctx, ST, T, st))) {
    ctx->err = "step-radix domain: per-size tables unavailable";
    return ZC_ERR_OOM;
  }
  if (!ST) sb = 1;

  // N1's first pass (rows over i2, twiddled) for the columns [j0, j1)
  auto n1_first = [&](const fr* const* in, int j0, int j1) -> zc_status {
    NttPassArgs a;
    pass_defaults(a);
    for (int j = j0; j < j1; j++) {
      a.in[j - j0] = in[j];
      a.out[j - j0] = coef[j];
    }
    const NttMaps mp = maps_n1_rows(l1, l2);
    a.use(mp);
    set_dft(a, T, true);
    a.err = &dstate->err;              // every input element passes through here once
    a.post = POST_TW; a.tw_lo = T->wi_lo; a.tw_hi = T->wi_hi;
    a.tw_lbmod = l1; a.tw_shift = kLog30 - n;
    if (ST) {
      a.post = POST_TAB; a.post_tab = ST->tw_inv;
    }
    return run_pass(ctx, st, a, j1 - j0, mp.B);
  };
  // N1's second pass (columns of length L1, in place) for the columns [j0, j1)
  auto n1_second = [&](int j0, int j1) -> zc_status {
    NttPassArgs a;
    pass_defaults(a);
    for (int j = j0; j < j1; j++) {
      a.in[j - j0] = coef[j];
      a.out[j - j0] = coef[j];
    }
    const NttMaps mp = maps_n1_cols(l1, l2);
    a.use(mp);
    set_dft(a, T, true);
    return run_pass(ctx, st, a, j1 - j0, mp.B);
  };

  k_ntt_state_init<<<1, 32, 0, st>>>(dstate);
  ctx->launches++;

  // Host columns: uploaded one by one on a side stream; with two passes the
  // first N1 pass of column j starts as soon as column j has arrived.
  const fr* src[kMaxCols];
  const bool pipelined = !on_dev && two;
  if (on_dev) {
    for (int j = 0; j < c; j++) src[j] = static_cast<const fr*>(cols[j]);
  } else if (pipelined) {
    zc_status us = ensure_upload_stream(ctx, c);
    if (us != ZC_OK) return us;
    ZC_CUDA_TRY(ctx, cudaEventRecord(ctx->up_fork, st));
    ZC_CUDA_TRY(ctx, cudaStreamWaitEvent(ctx->up_stream, ctx->up_fork, 0));
    for (int j = 0; j < c; j++) {
      ZC_CUDA_TRY(ctx, cudaMemcpyAsync(slb[j], cols[j], N * sizeof(fr), cudaMemcpyHostToDevice,
                                       ctx->up_stream));
      ZC_CUDA_TRY(ctx, cudaEventRecord(ctx->up_ev[j], ctx->up_stream));
      src[j] = slb[j];
    }
    for (int j = 0; j < c; j++) {
      ZC_CUDA_TRY(ctx, cudaStreamWaitEvent(st, ctx->up_ev[j], 0));
      if ((rs = n1_first(src, j, j + 1)) != ZC_OK) return rs;
    }
  } else {
    for (int j = 0; j < c; j++) {
      ZC_CUDA_TRY(ctx, cudaMemcpyAsync(slb[j], cols[j], N * sizeof(fr), cudaMemcpyHostToDevice, st));
      src[j] = slb[j];
    }
  }
  ZC_CUDA_TRY(ctx, cudaEventRecord(ctx->ev[0], st));
  if (roots) {
    std::memcpy(ctx->pinned, roots, 32 * (size_t)c);
    ZC_CUDA_TRY(ctx, cudaMemcpyAsync(droots, ctx->pinned, 32 * (size_t)c, cudaMemcpyHostToDevice, st));
  } else {
    zc_status rs = launch_roots(ctx, src, c, N, droots, st);
    if (rs != ZC_OK) return rs;
  }
  ZC_CUDA_TRY(ctx, cudaEventRecord(ctx->ev[1], st));

  // per-slice coset tables and z_H inverses (only without per-size tables)
  const DevConst& C = ctx->hconst;
  fr ninv = h_inv(h_from_u64(N), C), minv = h_inv(h_from_u64(M), C);
  if (!ST) {
    NttSliceTabArgs ta{};
    ta.lo = tlo;
    ta.hi = thi;
    ta.zinv = zinv;
    ta.s = (uint32_t)s;
    ta.n = n;
    ta.hbits = hbits;
    ta.logm = logm;
    ta.ninv_l2 = fr_mul_g(fr_mul_g(ninv, C.r2), C.r2);
    ta.minv_l1 = fr_mul_g(minv, C.r2);
    ta.wf_lo = T->wf_lo;
    ta.wf_hi = T->wf_hi;
    ta.C = ctx->dconst;
    uint64_t tot = s * (nlo + nhi);
    k_ntt_slice_tables<<<(unsigned)((tot + 255) / 256), 256, 0, st>>>(ta);
    ctx->launches++;
  }

  // ---- N1: g_j = DFT^-1(e_j) (the factor 1/N is applied later), natural out
  if (two) {
    if (!pipelined && (rs = n1_first(src, 0, c)) != ZC_OK) return rs;
    if ((rs = n1_second(0, c)) != ZC_OK) return rs;  // all columns in one launch
  } else {
    NttPassArgs a;
    pass_defaults(a);
    for (int j = 0; j < c; j++) {
      a.in[j] = src[j];
      a.out[j] = coef[j];
    }
    a.use(maps_one(n));
    set_dft(a, T, true);
    a.err = &dstate->err;
    if ((rs = run_pass(ctx, st, a, c, 1)) != ZC_OK) return rs;
  }
  ZC_CUDA_TRY(ctx, cudaEventRecord(ctx->ev[2], st));

  // ---- N2: per slice, coset NTT of every column, gate, divide by z_H.
  // slice_lde: the coset NTT of the `items` coefficient vectors in[] into
  // out[] on one slice, or on sb slices from j on, with the coset factor table pre (per-size tables)
  // or slice j's two-level tables (without them).
  auto slice_lde = [&](const fr* const* in, fr* const* out, int items, const FrcTab* pre, uint64_t j,
                       bool mark, uint32_t sb) -> zc_status {
    NttPassArgs a;
    pass_defaults(a);
    for (int i = 0; i < items; i++) {
      a.in[i] = in[i];
      a.out[i] = out[i];
    }
    a.pre = PRE_COSET;
    a.pre_lo = tlo + j * nlo;
    a.pre_hi = thi + j * nhi;
    a.pre_shift = hbits;
    a.out_y = (uint32_t)(c * Na);
    a.pre_y = (uint32_t)N;
    set_dft(a, T, false);
    if (two) {
      const NttMaps mc = maps_n2_cols(l1, l2), mr = maps_n2_rows(l1, l2);
      a.use(mc);
      a.post = POST_TW; a.tw_lo = T->wf_lo; a.tw_hi = T->wf_hi;
      a.tw_lbmod = l2; a.tw_shift = kLog30 - n;
      if (ST) {
        a.pre = PRE_TAB; a.pre_tab = *pre;
        a.post = POST_TAB; a.post_tab = ST->tw_fwd;
      } else {
        a.pm = mc.km;
      }
      if ((rs = run_pass(ctx, st, a, items, mc.B, sb)) != ZC_OK) return rs;
      if (mark) ZC_CUDA_TRY(ctx, cudaEventRecord(ctx->ev[7], st));
      pass_defaults(a);
      for (int i = 0; i < items; i++) {
        a.in[i] = out[i];
        a.out[i] = out[i];
      }
      a.use(mr);
      a.in_y = a.out_y = (uint32_t)(c * Na);
      set_dft(a, T, false);
      if ((rs = run_pass(ctx, st, a, items, mr.B, sb)) != ZC_OK) return rs;
    } else {
      a.use(maps_one(n));
      if (ST) {
        a.pre = PRE_TAB; a.pre_tab = *pre;
      }
      if ((rs = run_pass(ctx, st, a, items, 1, sb)) != ZC_OK) return rs;
      if (mark) ZC_CUDA_TRY(ctx, cudaEventRecord(ctx->ev[7], st));
    }
    return ZC_OK;
  };
  // gate and division by z_H (constant zi on the slice), minus sub if given
  auto slice_gate = [&](fr* out, const frc* zi, const fr* sub, uint32_t sb) {
    NttGateArgs ga{};
    for (int i = 0; i < c; i++) ga.col[i] = slb[i];
    ga.col_y = c * Na;
    ga.qhat = out;
    ga.zinv = zi;
    ga.sub = sub;
    ga.N = N;
    ga.gate = gate;
    ga.d = d;
    ga.c = (uint32_t)c;
    uint32_t gb = (uint32_t)std::min<uint64_t>((N + 255) / 256, (uint64_t)ctx->sm_count * 8);
    k_ntt_gate<<<dim3(gb, sb), 256, 0, st>>>(ga);
    ctx->launches++;
  };
  for (uint64_t j = 0; j < s; j += sb) {
    const FrcTab cs = ST ? ST->coset.at(j * N) : FrcTab();
    if ((rs = slice_lde(coef, slb, c, ST ? &cs : nullptr, j, j == 0, sb)) != ZC_OK) return rs;
    slice_gate(qhat + j * N, (ST ? ST->zinv : zinv) + j, nullptr, sb);
  }
  ZC_CUDA_TRY(ctx, cudaEventRecord(ctx->ev[3], st));

  // ---- N3: q = 7^-k M^-1 DFT_M^-1(qhat), digits (s, L1, L2) or (s, N).
  // inverse: the INTT of ns = 2^lbs slices qin[] into qout[] (natural
  // order, with the factor 7^-k; M^-1 came with the slice constants).
  auto inverse = [&](fr* qin, fr* qout, uint64_t s, uint32_t lb, uint32_t logm) -> zc_status {
  {
    NttPassArgs a;
    if (two) {
      pass_defaults(a);
      a.in[0] = qin; a.out[0] = qin;
      const NttMaps mr = maps_n3_rows(l1, l2, s), mc = maps_n3_cols(l1, l2, s);
      a.use(mr);
      set_dft(a, T, true);
      a.post = POST_TW; a.tw_lo = T->wi_lo; a.tw_hi = T->wi_hi;
      a.tw_lbmod = l1; a.tw_shift = kLog30 - n;
      if (ST) {
        a.post = POST_TAB; a.post_tab = ST->tw_inv;
      }
      if ((rs = run_pass(ctx, st, a, 1, mr.B)) != ZC_OK) return rs;
      pass_defaults(a);
      a.in[0] = qin; a.out[0] = qin;
      a.use(mc);
      set_dft(a, T, true);
      a.post = POST_OUTER; a.tw_lo = T->wi_lo; a.tw_hi = T->wi_hi;
      a.outer_lbdiv = l2; a.tw_shift = kLog30 - logm;
      if (ST) {
        if (s == 1) a.out[0] = qout;  // no cross-slice stage
        a.post = POST_TAB; a.post_tab = ST->outer;
      }
      if ((rs = run_pass(ctx, st, a, 1, mc.B)) != ZC_OK) return rs;
    } else {
      pass_defaults(a);
      a.in[0] = qin; a.out[0] = qin;
      const NttMaps mp = maps_n3_one(n, s);
      a.use(mp);
      set_dft(a, T, true);
      a.post = POST_OUTER; a.tw_lo = T->wi_lo; a.tw_hi = T->wi_hi;
      a.outer_lbdiv = 0; a.tw_shift = kLog30 - logm;
      if (ST) {
        if (s == 1) a.out[0] = qout;
        a.post = POST_TAB; a.post_tab = ST->outer;
      }
      if ((rs = run_pass(ctx, st, a, 1, mp.B)) != ZC_OK) return rs;
    }
    if (ST && s == 1) return ZC_OK;
    pass_defaults(a);
    a.in[0] = qin; a.out[0] = qout;
    const NttMaps ms = maps_n3_slices(n, lb);
    a.use(ms);
    set_dft(a, T, true);
    a.post = POST_FINAL; a.tw_lo = T->s7_lo; a.tw_hi = T->s7_hi;
    a.fin_logN = n;
    if (ST && lb <= 3) {  // in registers, with 7^-(N t)
      a.post_tab = ST->fin;
      a.B = (uint32_t)N;
      const unsigned blocks = (unsigned)((N + 255) / 256);
      if (lb == 1) k_ntt_cross<1><<<blocks, 256, 0, st>>>(a);
      else if (lb == 2) k_ntt_cross<2><<<blocks, 256, 0, st>>>(a);
      else k_ntt_cross<3><<<blocks, 256, 0, st>>>(a);
      ctx->launches++;
      return ZC_OK;
    }
    if (ST) {
      a.post = POST_TAB; a.post_tab = ST->fin;
    }
    if ((rs = run_pass(ctx, st, a, 1, ms.B)) != ZC_OK) return rs;
  }
    return ZC_OK;
  };
  if ((rs = inverse(qhat, qv, s, lb, logm)) != ZC_OK) return rs;
  if (D.step) {
    // q_big on D_small (reduce, then the slice LDE with sigma's factors),
    // the small part's gate minus it, its INTT, and q = q_big + (x^Mb -
    // 7^Mb) q_small.
    NttStepReduceArgs ra{};
    ra.q = qv;
    ra.rho = rho;
    ra.cm = ST->step_const + 8;
    ra.N = N;
    ra.parts = (uint32_t)s;
    const unsigned eg = (unsigned)std::min<uint64_t>((N + 255) / 256, (uint64_t)ctx->sm_count * 8);
    k_ntt_step_reduce<<<eg, 256, 0, st>>>(ra);
    ctx->launches++;
    const fr* rin[1] = {rho};
    fr* rout[1] = {vsm};
    if ((rs = slice_lde(rin, rout, 1, &ST->step_coset, 0, false, 1)) != ZC_OK) return rs;
    if ((rs = slice_lde(coef, slb, c, &ST->step_coset, 0, false, 1)) != ZC_OK) return rs;
    slice_gate(qhat + Mb, reinterpret_cast<const frc*>(ST->step_const), vsm, 1);
    if ((rs = inverse(qhat + Mb, qv + Mb, 1, 0, n)) != ZC_OK) return rs;
    NttStepCombineArgs ca{};
    ca.q = qv;
    ca.unscale = ST->step_unscale;
    ca.s7m = ST->step_const + 2;
    ca.N = N;
    ca.M = Mb;
    k_ntt_step_combine<<<eg, 256, 0, st>>>(ca);
    ctx->launches++;
  }
  ZC_CUDA_TRY(ctx, cudaEventRecord(ctx->ev[4], st));
  // a host q leaves on the side stream while the root and the openings run
  const bool q_async = q_out && !q_direct && !q_on_dev;
  if (q_async) {
    zc_status us = ensure_upload_stream(ctx, 1);
    if (us != ZC_OK) return us;
    ZC_CUDA_TRY(ctx, cudaStreamWaitEvent(ctx->up_stream, ctx->ev[4], 0));
    ZC_CUDA_TRY(ctx, cudaMemcpyAsync(q_out, qv, M * sizeof(fr), cudaMemcpyDeviceToHost, ctx->up_stream));
    ZC_CUDA_TRY(ctx, cudaEventRecord(ctx->up_ev[0], ctx->up_stream));
  }

  // ---- N4: root(q), z
  {
    const fr* qp[1] = {qv};
    if ((rs = launch_roots(ctx, qp, 1, M, droots + 32 * (size_t)c, st)) != ZC_OK) return rs;
    NttZArgs za{};
    za.st = dstate;
    za.roots = droots;
    za.c = c;
    za.n = n;
    transcript_init_words(za.S0, ZC_FORM_NTT, gate, n, d, D.word);
    za.zpow = zpow;
    za.nz = std::max<uint32_t>(logm + (D.step ? 1 : 0), std::max<uint32_t>(n, 5)) + 1;
    za.C = ctx->dconst;
    k_ntt_z<<<1, 64, 0, st>>>(za);
    ctx->launches++;
  }
  ZC_CUDA_TRY(ctx, cudaEventRecord(ctx->ev[5], st));

  // ---- N5, N6: openings and the proof
  {
    NttOpenArgs oa{};
    for (int j = 0; j < c; j++) {
      oa.x[j] = coef[j];
      oa.len[j] = N;
    }
    oa.x[c] = qv;
    oa.len[c] = M;
    oa.zpow = zpow;
    oa.partials = opart;
    oa.seg = 32 * open_steps(M);
    const uint32_t nblk = (uint32_t)std::min<uint64_t>(nblk_open, (M + 8ull * oa.seg - 1) / (8ull * oa.seg));
    oa.nblk = nblk;
    k_ntt_open<<<dim3(nblk, c + 1), 256, 0, st>>>(oa, ctx->dconst);
    ctx->launches++;
    NttFinalArgs fa{};
    fa.partials = opart;
    fa.nblk = nblk;
    fa.c = c;
    fa.gate = gate;
    fa.n = n;
    fa.d = d;
    fa.logm = D.word;
    fa.ninv_l1 = fr_mul_g(ninv, C.r2);
    fa.qroot = droots + 32 * (size_t)c;
    fa.st = dstate;
    fa.proof = dproof;
    k_ntt_final<<<1, 256, 0, st>>>(fa);
    ctx->launches++;
  }
  ZC_CUDA_TRY(ctx, cudaGetLastError());
  ZC_CUDA_TRY(ctx, cudaMemcpyAsync(proof, dproof, psize,
                                   proof_on_dev ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost,
                                   st));
  if (q_async) {
    ZC_CUDA_TRY(ctx, cudaStreamWaitEvent(st, ctx->up_ev[0], 0));
  } else if (q_out && !q_direct) {
    ZC_CUDA_TRY(ctx, cudaMemcpyAsync(q_out, qv, M * sizeof(fr), cudaMemcpyDeviceToHost, st));
  }
  ZC_CUDA_TRY(ctx, cudaEventRecord(ctx->ev[6], st));
  // dominant launch: one N2 column pass over all c columns of sb slices
  const double Lc = two ? (double)l1 : (double)n;
  ctx->dom_mulmods = sb * ((double)c * (double)N / 2 * Lc + (double)c * (double)N);
  ctx->dom_bytes = sb * (2.0 * 32 * c * (double)N);
  ctx->dom_a = 2;
  ctx->dom_b = 7;
  if (!proof_on_dev || !on_dev || (q_out && !q_direct)) {
    ZC_CUDA_TRY(ctx, cudaStreamSynchronize(st));
    if (std::memcmp(proof, "ZCE!", 4) == 0) {
      ctx->err = "column value >= r";
      return ZC_ERR_ARG;
    }
  }
  return ZC_OK;
}

}  // namespace zc
