// Every index of the NTT passes against its buffer and its definition, on the
// host, through the code that the kernels and their launches use.  Built and
// run by tests/test_ntt_index.py; prints "ok <passes> <threads>" or the first
// index that is wrong, with the pass it belongs to.
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <set>
#include <string>
#include <vector>

#include "../paper_2606_16146_gb300/csrc/zc_ntt_index.cuh"

using namespace zc;

static std::string where;
static uint64_t passes = 0, threads = 0;

#define CHECK(c)                                                               \
  do {                                                                         \
    if (!(c)) {                                                                \
      std::printf("%s: line %d: %s\n", where.c_str(), __LINE__, #c);           \
      std::exit(1);                                                            \
    }                                                                          \
  } while (0)

// entries of the buffers a pass uses (0: the pass does not use it)
struct Sizes {
  uint64_t in, out, pre, post, coef;
};

// some of 0..n-1: all when few, else both ends and a spread between
static std::vector<uint64_t> some(uint64_t n, uint64_t most) {
  std::vector<uint64_t> v;
  if (n <= most)
    for (uint64_t i = 0; i < n; i++) v.push_back(i);
  else
    for (uint64_t i = 0; i < most; i++) v.push_back(i < 2 ? i : i + 2 >= most ? n - (most - i) : i * 0x9E3779B97F4A7C15ull % n);
  return v;
}

// Counts the stores of whole launches (a byte per element) up to this many elements.
constexpr uint64_t kWhole = 1ull << 18;

// the tile exchanges of one stage must be a permutation of the tile
static void permutation(std::vector<uint32_t>& v, uint32_t tile) {
  std::sort(v.begin(), v.end());
  CHECK(v.size() == tile);
  for (uint32_t i = 0; i < tile; i++) CHECK(v[i] == i);
}

template <bool FAST>
static void check_pass(const NttMaps& M, const NttPlan& P, const Sizes& Z) {
  const uint32_t logL = M.logL, NT = P.tile / 8, L = 1u << logL;
  CHECK(M.B < (1ull << 31) && NT >= 1 && P.blocks >= 1 && NT % 32 == 0);
  CHECK(P.tile <= 4096 && (P.blocks << P.logW) >= M.B && ((P.blocks - 1) << P.logW) < M.B);
  CHECK(NT <= (P.logTile == 12 ? 512u : P.logTile == 11 ? 256u : 128u));  // the variant's launch bounds
  if (FAST) CHECK(NT % 64 == 0 && !(M.B & ((1ull << P.logW) - 1)) && logL >= 3);
  std::vector<uint8_t> stored;
  if ((M.B << logL) <= kWhole) stored.assign(Z.out, 0);
  const bool whole = !stored.empty();
  for (uint64_t blk : some(P.blocks, whole ? P.blocks : 6)) {
    const uint32_t b0 = (uint32_t)(blk << P.logW);
    std::vector<uint8_t> copied(2 * P.tile, 0);
    std::vector<std::vector<uint32_t>> ex(4);
    const bool all = whole || blk < 2 || NT <= 128;
    for (uint64_t t64 : some(NT, all ? NT : 64)) {
      const uint32_t tid = (uint32_t)t64;
      threads++;
      const NttTile<FAST> X(logL, P.logW, b0, (uint32_t)M.B, NT, tid);
      auto at = [&](const NttMap& m, uint32_t i) {  // the definition
        uint64_t b = (uint64_t)b0 + (i & ((1u << P.logW) - 1)), t = i >> P.logW;
        if (b >= M.B) b = M.B - 1;
        return ((b >> m.div) << m.hs) + ((b & m.mask) << m.ls) + (t << m.ts);
      };
      auto walk = [&](const NttMap& m, uint32_t i0, uint64_t size) {
        for (int p = 0; p < 8; p++) {
          const int64_t e = (int64_t)X.index(m, i0) + X.step(m, i0, p);
          CHECK(e == (int64_t)at(m, i0 + NT * p));
          CHECK(e >= 0 && (uint64_t)e < size);
        }
      };
      for (int s = 0; s < 2; s++) {  // the load
        const uint32_t i = X.copy_elt(s);
        CHECK(i / 32 == tid / 32);
        walk(M.im, i, Z.in);
        for (int p = 0; p < 8; p++) {
          CHECK(X.slot(i, p) == tile_slot(i + NT * p) && X.slot(i, p) < P.tile);
          copied[2 * X.slot(i, p) + (tid & 1)]++;
        }
      }
      for (int p = 0; p < 8; p++) CHECK(X.slot(tid, p) == tile_slot(tid + NT * p));
      if (Z.pre) walk(M.pm, tid, Z.pre);
      if (Z.post) walk(M.qm, tid, Z.post);
      if (Z.coef) walk(M.km, tid, Z.coef);
      int stage = 0;
      for (uint32_t logNs = 0; logNs < logL; stage++) {
        const uint32_t lr = std::min(3u, logL - logNs), lg = 3 - lr, Ns = 1u << logNs;
        if (logNs > 0)
          for (int p = 1 << lg; p < 8; p++) {  // r >= 1
            const uint32_t g = p & ((1u << lg) - 1), r = (uint32_t)p >> lg, k = ((tid + NT * g) >> P.logW) % Ns;
            const int64_t e = X.tw_first(logNs, lr) + X.tw_step(logNs, lr, p);
            CHECK(e == (int64_t)stage_tab(logNs, lr) + (int64_t)(r - 1) * Ns + k);
            CHECK(e >= 0 && e < (int64_t)kStageTab);
          }
        if (logNs + lr < logL)
          for (int p = 0; p < 8; p++) {
            const uint32_t g = p & ((1u << lg) - 1), r = (uint32_t)p >> lg, i = tid + NT * g;
            const uint32_t w = i & ((1u << P.logW) - 1), j = i >> P.logW;
            CHECK(j < L >> lr);
            const uint32_t q = X.exchange(logNs, lr, p);
            CHECK(q == ((((j >> logNs) << (logNs + lr)) + j % Ns + r * Ns) << P.logW) + w);
            if (all) ex[stage].push_back(q);
          }
        logNs += lr;
      }
      for (uint32_t i0 : {tid & ~1u, tid | 1u}) {  // the store: this lane writes half of both elements
        walk(M.om, i0, Z.out);
        for (int p = 0; p < 8; p++) {
          const uint32_t i = i0 + NT * p;
          CHECK(X.stored(i) == ((uint64_t)b0 + (i & ((1u << P.logW) - 1)) < M.B));
          if (whole && X.stored(i)) stored[X.index(M.om, i0) + X.step(M.om, i0, p)] += tid & 1 ? 16 : 1;
        }
      }
    }
    if (all) {
      for (uint8_t c : copied) CHECK(c == 1);
      for (auto& v : ex)
        if (!v.empty()) permutation(v, P.tile);
    }
  }
  if (whole) {  // both halves of every output element once
    uint64_t n = 0;
    for (uint8_t c : stored) {
      CHECK(c == 0 || c == 17);
      n += c == 17;
    }
    CHECK(n == M.B << logL);
  }
  passes++;
}

static void check_small(const NttMaps& M, const NttPlan& P, const Sizes& Z) {
  const uint32_t NT = P.tile / 2;
  CHECK(NT >= 128 && NT <= 512 && P.blocks << P.logW == M.B && NT % (1u << P.logW) == 0);
  std::vector<uint8_t> stored;
  if ((M.B << M.logL) <= kWhole) stored.assign(Z.out, 0);
  for (uint64_t blk : some(P.blocks, stored.empty() ? 6 : P.blocks)) {
    const uint32_t b0 = (uint32_t)(blk << P.logW);
    std::vector<std::vector<uint32_t>> ex(M.logL);
    for (uint32_t tid = 0; tid < NT; tid++) {
      threads++;
      const NttSmallTile X{M.logL, P.logW, b0, NT, tid};
      for (int p = 0; p < 2; p++) {
        const uint32_t i = tid + NT * p;
        CHECK(X.sub() == b0 + (i & ((1u << P.logW) - 1)) && X.sub() < M.B && X.elt(p) == i >> P.logW);
        CHECK(M.im.at(X.sub(), X.elt(p)) < Z.in && M.om.at(X.sub(), X.elt(p)) < Z.out);
        if (Z.pre) CHECK(M.pm.at(X.sub(), X.elt(p)) < Z.pre);
        if (Z.post) CHECK(M.qm.at(X.sub(), X.elt(p)) < Z.post);
        if (!stored.empty()) stored[M.om.at(X.sub(), X.elt(p))]++;
      }
      for (uint32_t logNs = 0; logNs < M.logL; logNs++) {
        const uint32_t Ns = 1u << logNs, j = tid >> P.logW, w = tid & ((1u << P.logW) - 1);
        // w_{2 Ns}^k as an entry (r - 1) 512 + k' of the radix-8 table at stride 512: exponent r k' of w_4096
        const uint32_t e = X.twiddle(logNs) - stage_tab(9, 3), r = e / 512 + 1, kk = e % 512;
        CHECK(X.twiddle(logNs) < kStageTab && r < 8 && r * kk == j % Ns * (2048 / Ns));
        if (logNs + 1 < M.logL)
          for (int p = 0; p < 2; p++) {
            CHECK(X.exchange(logNs, p) == ((((j >> logNs) << (logNs + 1)) + j % Ns + (p ? Ns : 0)) << P.logW) + w);
            ex[logNs].push_back(X.exchange(logNs, p));
          }
      }
    }
    for (auto& v : ex)
      if (!v.empty()) permutation(v, P.tile);
  }
  if (!stored.empty()) CHECK((uint64_t)std::count(stored.begin(), stored.end(), 1) == M.B << M.logL);
  passes++;
}

static uint32_t tiles_of(uint32_t n, uint32_t* t) {  // 0: no key set
  const uint32_t a[4] = {0, 10, 11, 12};
  const uint32_t k = n <= 14 || n == 17 || n == 20 ? 4 : 1;
  std::copy(a, a + k, t);
  return k;
}

// every form that a launch of the pass may take
static void check(uint32_t n, const char* name, const NttMaps& M, const Sizes& Z, bool cross = false) {
  uint32_t t[4];
  const uint32_t k = tiles_of(n, t);
  for (uint32_t i = 0; i < k; i++) {
    const NttPlan P = ntt_plan(M.logL, M.B, t[i]);
    where = std::string(name) + " n=" + std::to_string(n) + " logL=" + std::to_string(M.logL) +
            " B=" + std::to_string(M.B) + " tile=" + std::to_string(P.tile);
    if (ntt_fast(P, M.logL, M.B)) check_pass<true>(M, P, Z);
    check_pass<false>(M, P, Z);  // the form of the power tables, on whole tiles too
  }
  NttPlan S;
  where += " small";
  if (!cross && M.B << M.logL <= 1ull << 19 && ntt_plan_small(M.logL, M.B, &S)) check_small(M, S, Z);
}

int main() {
  // the twiddle tables: blocks of 7, 3 and 1 rows of Ns entries, one after the other
  where = "stage_tab";
  std::set<uint32_t> seen;
  for (uint32_t logNs : {3u, 6u, 9u})
    for (uint32_t lr : {3u, 2u, 1u})
      for (uint32_t e = 0; e < ((1u << lr) - 1) << logNs; e++) CHECK(seen.insert(stage_tab(logNs, lr) + e).second);
  CHECK(seen.size() == kStageTab && *seen.rbegin() == kStageTab - 1);
  for (uint32_t n = 1; n <= 24; n++) {
    const uint64_t N = 1ull << n;
    for (int two = 0; two < 2; two++) {
      if (two ? n < 2 : n > 12) continue;
      const uint32_t l1 = two ? (n + 1) / 2 : n, l2 = two ? n / 2 : 0;
      where = "tab_pos";
      if (n <= 14) {
        std::vector<uint8_t> hit(N, 0);
        for (uint64_t k = 0; k < N; k++) {
          CHECK(tab_pos(k, l1, l2) < N);
          hit[tab_pos(k, l1, l2)]++;
        }
        CHECK((uint64_t)std::count(hit.begin(), hit.end(), 1) == N);
      }
      if (two) {
        check(n, "N1 rows", maps_n1_rows(l1, l2), Sizes{N, N, 0, N, 0});
        check(n, "N1 columns", maps_n1_cols(l1, l2), Sizes{N, N, 0, 0, 0});
        const NttMaps mc = maps_n2_cols(l1, l2);
        check(n, "N2 columns", mc, Sizes{N, N, N, N, N});
        where = "N2 coset factor";
        for (uint64_t b : some(mc.B, 64))  // the table entry of the coefficient that is read
          for (uint32_t t = 0; t < 1u << l1; t++) CHECK(mc.pm.at(b, t) == tab_pos(mc.km.at(b, t), l1, l2));
        check(n, "N2 rows", maps_n2_rows(l1, l2), Sizes{N, N, 0, 0, 0});
      } else {
        check(n, "one pass", maps_one(n), Sizes{N, N, N, 0, N});
      }
      for (uint32_t lb = 0; lb <= 6 && n + lb <= 30; lb++) {
        const uint64_t s = 1ull << lb, M = N << lb;
        if (two) {
          check(n, "N3 rows", maps_n3_rows(l1, l2, s), Sizes{M, M, 0, N, 0});
          const NttMaps mc = maps_n3_cols(l1, l2, s);
          check(n, "N3 columns", mc, Sizes{M, M, 0, M, 0});
          where = "N3 outer factor";
          for (uint64_t b : some(mc.B, 64))
            for (uint32_t t = 0; t < 1u << l1; t++) {
              const uint64_t e = mc.im.at(b, t), j = e >> n;  // slice j, k' = e mod N
              CHECK(mc.qm.at(b, t) == (j << n) + tab_pos(e & (N - 1), l1, l2));
            }
        } else {
          check(n, "N3 one pass", maps_n3_one(n, s), Sizes{M, M, 0, M, 0});
        }
        if (lb > 0) check(n, "N3 slices", maps_n3_slices(n, lb), Sizes{M, M, 0, s, 0}, lb <= 3);
      }
    }
    for (uint32_t nc = 1; nc <= std::min(n, 12u) && n <= 22; nc++)  // from slice 3's first position on
      check(n, "commitment", maps_pcs(n - nc, nc), Sizes{N, 4 * N - 3 * (N >> nc), 1ull << nc, 0, 0});
  }
  std::printf("ok %llu %llu\n", (unsigned long long)passes, (unsigned long long)threads);
  return 0;
}
