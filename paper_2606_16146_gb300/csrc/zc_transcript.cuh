// zc_transcript.cuh -- Fiat-Shamir transcript on the device, word-based.
//
// The paper derives every challenge by hashing (Fig. side-by-side-zc:
// "r <- Hash([g])", "alpha_i <- Hash(G_i)").  State S is a SHA-256 digest;
// absorb(m): S = SHA-256(S | m); squeeze: S = SHA-256(S | 0x43) and the
// challenge is int_le(S) mod r.  All absorbed messages here are whole 32-bit
// words (digests and canonical field elements), so blocks are assembled as
// words: a field element's little-endian bytes are its limbs byte-swapped.
#pragma once
#include "zc_internal.cuh"

namespace zc {

#if defined(__CUDACC__)

// SHA-256 by two warps.  A transcript hash is one serial chain of
// compressions, and the 24 instructions of a round (14 of the round itself, 10
// of the message schedule) fill the ALU pipe of the SM quarter its warp runs
// on: 3130 cycles a compression.  Warp 0 runs the rounds and warp 1, on another
// quarter, the schedule: words 16..63 with their round constants, through
// shared memory, sixteen at a time.  The first sixteen rounds need only the
// message, so the schedule stays ahead, and a compression takes the rounds'
// ~1920 cycles; both loops are short enough to be cheap when their code is
// cold.  All lanes of a warp compute the same values.  The two warps meet four
// times a block: when its words are in shared memory (and the previous block's
// schedule has been read), and at each third of the schedule.
struct ShaPair {
  uint32_t kw[48];     // schedule words 16..63 plus round constants
  uint32_t sq[16];     // the squeeze block: state, 0x43, padding
};

// both warps; the id is an immediate (with an id in a register a kernel
// reserves all sixteen barriers)
__device__ __forceinline__ void pair_sync() {
  __syncwarp();
  asm volatile("bar.sync 1, 64;" ::: "memory");
}

// warp 1: the schedule of the block blk (shared memory)
__device__ __forceinline__ void sha_pair_schedule(ShaPair& Z, const uint32_t* blk) {
  uint32_t w[16];
  pair_sync();
#pragma unroll
  for (int i = 0; i < 16; i++) w[i] = blk[i];
#pragma unroll 1
  for (int q = 0; q < 3; q++) {
#pragma unroll
    for (int i = 0; i < 16; i++) Z.kw[16 * q + i] = sha_sched(w, i) + kShaK[16 * q + 16 + i];
    pair_sync();
  }
}

// warp 0: h <- compress(h, blk)
__device__ __forceinline__ void sha_pair_rounds(ShaPair& Z, const uint32_t* blk, uint32_t h[8]) {
  uint32_t v[8];
#pragma unroll
  for (int i = 0; i < 8; i++) v[i] = h[i];
  pair_sync();
#pragma unroll
  for (int i = 0; i < 16; i++) sha_round(v, kShaK[i] + blk[i]);
#pragma unroll 1
  for (int q = 0; q < 3; q++) {
    pair_sync();
#pragma unroll
    for (int i = 0; i < 16; i++) sha_round(v, Z.kw[16 * q + i]);
  }
#pragma unroll
  for (int i = 0; i < 8; i++) h[i] += v[i];
}

// One block by both warps (warp 0: h updated; warp 1: h untouched).
__device__ __forceinline__ void sha_pair_block(ShaPair& Z, const uint32_t* blk, uint32_t h[8]) {
  if (threadIdx.x < 32) sha_pair_rounds(Z, blk, h);
  else sha_pair_schedule(Z, blk);
}

// Padding of a message of nwords words at w (room for the whole last block):
// the words after the message, by the threads t, t + nt, ...
__device__ __forceinline__ uint32_t sha_blocks(uint32_t nwords) { return (nwords + 3 + 15) / 16; }
__device__ __forceinline__ void sha_pad(uint32_t* w, uint32_t nwords, uint32_t t, uint32_t nt) {
  const uint32_t end = 16 * sha_blocks(nwords);
  for (uint32_t i = nwords + t; i < end; i += nt) w[i] = i == nwords ? 0x80000000u : i == end - 1 ? 32 * nwords : 0u;
}

// int_le(digest) mod r as a canonical element (2^256 < 3r: at most two subtractions)
__device__ inline fr digest_mod_r(const uint32_t h[8]) {
  fr x;
  for (int i = 0; i < 8; i++) x.v[i] = sha_bswap(h[i]);
  for (int k = 0; k < 2; k++) {
    if (!fr_is_canonical(x)) {
      int64_t br = 0;
      for (int i = 0; i < 8; i++) {
        int64_t dd = (int64_t)x.v[i] - p_limb(i) + br;
        x.v[i] = (uint32_t)dd;
        br = dd >> 32;
      }
    }
  }
  return x;
}

// the squeeze block of the state S (warp 0's lanes; both warps call)
__device__ __forceinline__ void tr_squeeze_block(ShaPair& Z, const uint32_t S[8]) {
  if (threadIdx.x < 16) {
    const int i = threadIdx.x;
    uint32_t v = i == 8 ? 0x43800000u : i == 15 ? 33 * 8 : 0u;  // the byte 0x43, then the padding bit; the length
#pragma unroll
    for (int q = 0; q < 8; q++) v = i == q ? S[q] : v;
    Z.sq[i] = v;
  }
}

// S <- SHA-256(S | 0x43) and the canonical challenge, warps 0 and 1 (values in
// warp 0)
__device__ __forceinline__ fr tr_squeeze(ShaPair& Z, uint32_t S[8]) {
  tr_squeeze_block(Z, S);
  sha256_init(S);
  sha_pair_block(Z, Z.sq, S);
  return digest_mod_r(S);
}

// S <- SHA-256(w) for the padded message w (shared memory) of nwords words,
// then a squeeze; one copy of the compression serves both.  Warps 0 and 1
// (values in warp 0).
__device__ __forceinline__ fr tr_hash_squeeze(ShaPair& Z, const uint32_t* w, uint32_t nwords, uint32_t S[8]) {
  const uint32_t nb = sha_blocks(nwords);
  sha256_init(S);
#pragma unroll 1
  for (uint32_t b = 0; b <= nb; b++) {
    if (b == nb) {
      tr_squeeze_block(Z, S);
      sha256_init(S);
    }
    sha_pair_block(Z, b < nb ? w + 16 * b : Z.sq, S);
  }
  return digest_mod_r(S);
}

// S <- SHA-256(S | m_j) for c 32-byte messages at m (global memory), warps 0
// and 1 (S in warp 0).  blk: 32 words of shared memory.
__device__ __forceinline__ void tr_absorb32(ShaPair& Z, uint32_t* blk, uint32_t S[8], const uint8_t* m, int c) {
  if (threadIdx.x < 16) blk[16 + threadIdx.x] = threadIdx.x == 0 ? 0x80000000u : threadIdx.x == 15 ? 512 : 0u;
#pragma unroll 1
  for (int j = 0; j < 2 * c; j++) {
    if (!(j & 1)) {
      if (threadIdx.x < 16) {
        const int i = threadIdx.x;
        const uint8_t* p = m + 16 * j + 4 * (i & 7);
        uint32_t v = ((uint32_t)p[0] << 24) | ((uint32_t)p[1] << 16) | ((uint32_t)p[2] << 8) | p[3];
#pragma unroll
        for (int q = 0; q < 8; q++) v = i == q ? S[q] : v;
        blk[i] = v;
      }
      sha256_init(S);
    }
    sha_pair_block(Z, blk + 16 * (j & 1), S);
  }
}

#endif

}  // namespace zc
