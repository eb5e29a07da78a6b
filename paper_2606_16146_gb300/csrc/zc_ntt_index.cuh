// zc_ntt_index.cuh -- index arithmetic of the NTT passes: which elements a
// pass's sub-DFTs read and write, which table entries they use, and where a
// thread's eight (or two) elements lie in the tile.  Plain integer code, shared
// by the kernels, their launches and the check of every size on the host
// (tests/test_ntt_index.py).
#pragma once
#include <stddef.h>
#include <stdint.h>

#include "zc_field.cuh"  // ZC_HD

namespace zc {

// ------------------------------------------------------------ stage twiddles --

// Twiddles of the radix-R stage at stride Ns = 8, 64 or 512: w_{Ns R}^{r k},
// 1 <= r < R, k < Ns, at stage_tab + (r - 1) Ns + k, so that consecutive k are
// consecutive entries.
constexpr uint32_t kStageTab = 11 * (8 + 64 + 512);
ZC_HD uint32_t stage_tab(uint32_t logNs, uint32_t lr) {
  const uint32_t Ns = 1u << logNs;
  return 11 * ((Ns - 8) / 7) + (lr == 3 ? 0 : lr == 2 ? 7 * Ns : 10 * Ns);
}
// w_{2 Ns}^k = w_4096^(4 k'), k' = k 512 / Ns: the radix-8 table at stride 512, r = 4
ZC_HD uint32_t stage_tab2(uint32_t logNs, uint32_t k) { return stage_tab(9, 3) + 3 * 512 + (k << (9 - logNs)); }

// ------------------------------------------------------------------- strides --

// Index of element t of sub-DFT b in a column or a factor table; every stride
// is a power of two: ((b >> div) << hs) + ((b & mask) << ls) + (t << ts).
struct NttMap {
  uint32_t div, hs, mask, ls, ts;
  ZC_HD uint32_t at(uint32_t b, uint32_t t) const { return ((b >> div) << hs) + ((b & mask) << ls) + (t << ts); }
};
constexpr uint32_t kNone = 31;  // a shift that leaves nothing of b < 2^31
// b << ls, t << ts
inline NttMap map_flat(uint32_t ls, uint32_t ts) { return NttMap{kNone, 0, 0xffffffffu, ls, ts}; }
// (b >> div) << hs, (b mod 2^div) << ls, t << ts
inline NttMap map_split(uint32_t div, uint32_t hs, uint32_t ls, uint32_t ts) {
  return NttMap{div, hs, (1u << div) - 1, ls, ts};
}
// the low div bits of b only
inline NttMap map_low(uint32_t div, uint32_t ls, uint32_t ts) { return NttMap{kNone, 0, (1u << div) - 1, ls, ts}; }

// A pass: B sub-DFTs of 2^logL points, elements read at im and written at om;
// pre factor pm and post factor qm in their tables, km the number of the
// coefficient (the pre factor without tables).
struct NttMaps {
  uint32_t logL;
  uint64_t B;
  NttMap im, om, pm, qm, km;
};

// coefficient k = L2 t + b at entry L1 b + t: the passes over t read consecutive entries
ZC_HD uint64_t tab_pos(uint64_t k, uint32_t l1, uint32_t l2) { return ((k & ((1ull << l2) - 1)) << l1) + (k >> l2); }

// N = 2^(l1 + l2).  N1's rows over i2, element (i1, i2) read from e[i1 + L1 i2]; post w_N^-(i1 k2) = tw_inv[i1 L2 + k2]
inline NttMaps maps_n1_rows(uint32_t l1, uint32_t l2) {
  return NttMaps{l2, 1ull << l1, map_flat(0, l1), map_flat(l2, 0), {}, map_flat(l2, 0), {}};
}
// N1's columns of length L1, in place
inline NttMaps maps_n1_cols(uint32_t l1, uint32_t l2) {
  return NttMaps{l1, 1ull << l2, map_flat(0, l2), map_flat(0, l2), {}, {}, {}};
}
// N2's columns over k1, k = L2 k1 + k2; pre the coset factor of k at L1 k2 + k1, post w_N^(k2 i1) = tw_fwd[k2 L1 + i1]
inline NttMaps maps_n2_cols(uint32_t l1, uint32_t l2) {
  return NttMaps{l1, 1ull << l2, map_flat(0, l2), map_flat(0, l2), map_flat(l1, 0), map_flat(l1, 0), map_flat(0, l2)};
}
// N2's rows over k2
inline NttMaps maps_n2_rows(uint32_t l1, uint32_t l2) {
  return NttMaps{l2, 1ull << l1, map_flat(l2, 0), map_flat(l2, 0), {}, {}, {}};
}
// N3's rows (j, i2) over i3; post w_N^-(i2 k3) = tw_inv[(b mod L1) L2 + k3]
inline NttMaps maps_n3_rows(uint32_t l1, uint32_t l2, uint64_t s) {
  return NttMaps{l2, s << l1, map_flat(l2, 0), map_flat(l2, 0), {}, map_low(l1, l2, 0), {}};
}
// N3's columns (j, k3) over i2 within a slice; post w_M^-(j k') 7^-k', k' = L2 k2 + k3, at outer[j N + L1 k3 + k2]
inline NttMaps maps_n3_cols(uint32_t l1, uint32_t l2, uint64_t s) {
  const NttMap m = map_split(l2, l1 + l2, 0, l2);
  return NttMaps{l1, s << l2, m, m, {}, map_split(l2, l1 + l2, l1, 0), {}};
}
// one pass per transform: a whole column, and N3's row per slice
inline NttMaps maps_one(uint32_t n) {
  const NttMap m = map_flat(0, 0);
  return NttMaps{n, 1, m, m, m, {}, m};
}
inline NttMaps maps_n3_one(uint32_t n, uint64_t s) {
  const NttMap m = map_flat(n, 0);
  return NttMaps{n, s, m, m, {}, m, {}};
}
// N3 across the 2^lb slices; post 7^-(N t) = fin[t]
inline NttMaps maps_n3_slices(uint32_t n, uint32_t lb) {
  return NttMaps{lb, 1ull << n, map_flat(0, n), map_flat(0, n), {}, map_low(0, 0, 0), {}};
}
// commitment: row b of 2^nr, coefficient t of 2^nc, to position 4 t
inline NttMaps maps_pcs(uint32_t nr, uint32_t nc) {
  return NttMaps{nc, 1ull << nr, map_flat(nc, 0), map_flat(0, nr + 2), map_low(0, 0, 0), {}, {}};
}

// ------------------------------------------------------------------ launches --

// Tile of 2^(logW + logL) elements: 2^logW sub-DFTs.
struct NttPlan {
  uint32_t logW, tile;
  uint64_t blocks;   // per column
  uint32_t logTile;  // the pass variant (10, 11 or 12)
};
// logTile: 0 or the tuned one
inline NttPlan ntt_plan(uint32_t logL, uint64_t B, uint32_t logTile) {
  if (logTile < logL) logTile = logL < 10 ? 10 : logL;
  if (logTile > 12) logTile = 12;
  if (logTile < 10) logTile = 10;
  // a tile holds at least one warp's elements, sub-DFTs past the last included
  uint32_t logW = logTile - logL;
  while (logW > 0 && logW + logL > 8 && (1ull << logW) > B) logW--;
  return NttPlan{logW, 1u << (logW + logL), (B + (1ull << logW) - 1) >> logW, logTile};
}
// whole tiles of sub-DFTs of at least 8 points, 64 threads or more
inline bool ntt_fast(const NttPlan& p, uint32_t logL, uint64_t B) {
  return logL >= 3 && p.tile >= 512 && !(B & ((1ull << p.logW) - 1));
}
// the small pass: whole tiles of 256 elements (or one sub-DFT); false where they do not come out even
inline bool ntt_plan_small(uint32_t logL, uint64_t B, NttPlan* p) {
  if (logL < 1 || logL > 10) return false;
  const uint32_t lt = logL > 8 ? logL : 8;
  if ((B << logL) & ((1ull << lt) - 1)) return false;
  *p = NttPlan{lt - logL, 1u << lt, B >> (lt - logL), 0};
  return true;
}

// -------------------------------------------------------------------- passes --

// slot of tile element i (16-byte halves in two planes, XOR-swizzled)
ZC_HD uint32_t tile_slot(uint32_t i) { return i ^ ((i >> 3) & 7); }

// Thread tid's part of a tile: elements i = tid + NT p, p < 8 (NT threads).
template <bool FAST>
struct NttTile {
  uint32_t logL, logW, b0, B, NT, tid;
  uint32_t Wm = (1u << logW) - 1, tq = (1u << logL) >> 3;
  ZC_HD NttTile(uint32_t logL_, uint32_t logW_, uint32_t b0_, uint32_t B_, uint32_t NT_, uint32_t tid_)
      : logL(logL_), logW(logW_), b0(b0_), B(B_), NT(NT_), tid(tid_) {}
  // the sub-DFT and the element of tile element i
  ZC_HD uint32_t sub(uint32_t i) const {
    const uint32_t b = b0 + (i & Wm);
    return FAST || b < B ? b : B - 1;
  }
  ZC_HD uint32_t elt(uint32_t i) const { return i >> logW; }
  // index of tile element i, and from i0 to i0 + NT p (FAST: p tq elements
  // further on; otherwise it may go back)
  ZC_HD uint32_t index(const NttMap& m, uint32_t i) const { return m.at(sub(i), elt(i)); }
  ZC_HD ptrdiff_t step(const NttMap& m, uint32_t i0, int p) const {
    return FAST ? (ptrdiff_t)(p * (tq << m.ts)) : (ptrdiff_t)index(m, i0 + NT * p) - (ptrdiff_t)index(m, i0);
  }
  // slot of element i + NT p (NT is a multiple of 64 in the FAST form: the swizzle of i serves all)
  ZC_HD uint32_t slot(uint32_t i, int p) const { return FAST ? tile_slot(i) + NT * p : tile_slot(i + NT * p); }
  // the load: two lanes to an element, a warp copies its own elements i + NT p only
  ZC_HD uint32_t copy_elt(int s) const { return (tid & ~31u) + ((tid & 31) >> 1) + 16 * s; }
  // stage of radix 2^lr after strides of 2^logNs: register p is r = p >> lg of
  // group g = p mod 2^lg, lg = 3 - lr.  Entry of the twiddle w_{Ns R}^{r k}, r >=
  // 1, k = elt mod Ns: tw_first + tw_step.  Group g's sub-DFT element is j + g
  // tq; only a last stage has several groups, and there k = j.
  ZC_HD ptrdiff_t tw_first(uint32_t logNs, uint32_t lr) const {
    const uint32_t km = (1u << logNs) - 1;
    return (ptrdiff_t)(stage_tab(logNs, lr) + (FAST ? elt(tid) & km : 0)) - (ptrdiff_t)(km + 1);
  }
  ZC_HD uint32_t tw_step(uint32_t logNs, uint32_t lr, int p) const {
    const uint32_t lg = 3 - lr, g = p & ((1u << lg) - 1), r = (uint32_t)p >> lg, km = (1u << logNs) - 1;
    return (r << logNs) + (FAST ? g * tq : elt(tid + NT * g) & km);
  }
  // where register p of the stage goes: element (j, r) to (j / Ns) Ns R + j mod Ns + r Ns
  ZC_HD uint32_t exchange(uint32_t logNs, uint32_t lr, int p) const {
    const uint32_t lg = 3 - lr, ja = tid + NT * (p & ((1u << lg) - 1)), r = (uint32_t)p >> lg, ls = logNs + logW;
    return ((ja >> ls) << (ls + lr)) + (ja & ((1u << ls) - 1)) + (r << ls);
  }
  // sub-DFTs past the last repeat it and are not stored
  ZC_HD bool stored(uint32_t i) const { return FAST || b0 + (i & Wm) < B; }
};

// The small pass: elements tid and tid + NT of a tile of 2 NT, radix 2.
struct NttSmallTile {
  uint32_t logL, logW, b0, NT, tid;
  ZC_HD uint32_t sub() const { return b0 + (tid & ((1u << logW) - 1)); }  // NT is a multiple of 2^logW
  ZC_HD uint32_t elt(int p) const { return (tid + NT * p) >> logW; }
  ZC_HD uint32_t twiddle(uint32_t logNs) const { return stage_tab2(logNs, elt(0) & ((1u << logNs) - 1)); }
  ZC_HD uint32_t exchange(uint32_t logNs, int p) const {
    const uint32_t ls = logNs + logW;
    return ((tid >> ls) << (ls + 1)) + (tid & ((1u << ls) - 1)) + ((uint32_t)p << ls);
  }
};

}  // namespace zc
