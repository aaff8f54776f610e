// Entropy coding of the indices (Section 3.1, "entropy encoding codebook pointers"): index value l occurs with
// probability p_l (mass of the l-th cell of the codebook under the density of Lemma 1), so a lossless prefix code
// brings the average width from b bits towards the entropy of {p_l} (3.8 bits at b = 4, about 5 % saved).
//
// The code is given by its lengths (tq_entropy_lengths builds the Huffman lengths from the cell masses); code
// words are assigned canonically from the lengths: symbols sorted by (length, symbol) receive consecutive
// values, shifted left whenever the length grows.  Every vector is coded on its own, so rows are decoded in
// parallel.  Row stream: bit p is bit (p & 7) of byte (p >> 3); code words follow one another without gaps,
// each written from its most significant bit; a row occupies a whole number of 32-bit words.
//
//   measure   one warp per row: eight coordinates become a word of nibbles, byte permutes look up four code lengths at a time
//             and dp4a adds them; a CTA also leaves the total of its rows
//   offsets   exclusive prefix sum of the row sizes: a CTA of 1024 rows adds up the CTA totals before it, then scans its own
//   pack      one warp per row: code words are looked up two at a time, a lane joins the eight of its group, a warp scan of the
//             lengths places them in a shared-memory image of the row (atomic OR), which leaves in one coalesced sweep
//   unpack    one thread per row: a look-up on the next 10 (12) stream bits gives as many whole symbols as they hold
// Bound by instruction issue (pack: 71 % of the slots) and, in unpack (54 %), by the latency of a thread's chain of look-ups; not by
// memory.  Measured at n = 100,000, d = 1536, b = 4 (76.8 MB of indices), before -> now: measure 121 -> 34 us, offsets 83 (one
// CTA) -> 4, clearing the output 13 -> 1, pack 396 -> 113, unpack 471 -> 154.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "tq_internal.h"
#include "tq_quantize_tc.h"

namespace tq {
namespace entropy {

namespace {

constexpr int kMaxLen = 12;   // longest code word accepted (look-up table of 2^12 entries in shared memory)

struct Code {
  uint8_t len[16];
  uint16_t word[16];   // canonical code word, most significant bit first
  int bits;            // b_m
  int maxlen;
  uint32_t len4[4];    // the lengths again, four to a word
};

struct Args {
  int64_t n;
  int d;
  const uint8_t* idx;
  size_t idx_rb;
  Code code;
};

__device__ __forceinline__ uint32_t spread3(uint32_t x) {   // eight 3-bit codes (low 24 bits) as nibbles
  x = (x & 0x00000fffu) | ((x & 0x00fff000u) << 4);
  x = (x & 0x003f003fu) | ((x & 0x0fc00fc0u) << 2);
  return (x & 0x07070707u) | ((x & 0x38383838u) << 1);
}
__device__ __forceinline__ uint32_t spread2(uint32_t x) {
  x = (x & 0x000000ffu) | ((x & 0x0000ff00u) << 8);
  x = (x & 0x000f000fu) | ((x & 0x00f000f0u) << 4);
  return (x & 0x03030303u) | ((x & 0x0c0c0c0cu) << 2);
}
__device__ __forceinline__ uint32_t spread1(uint32_t x) {
  x = (x & 0x0fu) | ((x & 0xf0u) << 12);
  x = (x & 0x00030003u) | ((x & 0x000c000cu) << 6);
  return (x & 0x01010101u) | ((x & 0x02020202u) << 3);
}

// Word w of a packed row.  BYTES: the rows are not 4-byte aligned (a slice of a larger buffer) and are read byte by byte.
template <bool BYTES>
__device__ __forceinline__ uint32_t row_word(const uint8_t* __restrict__ row, int w) {
  if (!BYTES) return __ldg(reinterpret_cast<const uint32_t*>(row) + w);
  const uint8_t* b = row + 4 * w;
  return (uint32_t)__ldg(b) | ((uint32_t)__ldg(b + 1) << 8) | ((uint32_t)__ldg(b + 2) << 16) | ((uint32_t)__ldg(b + 3) << 24);
}

// Coordinates 8 g .. 8 g + 7 of a packed row of row_words words as eight nibbles (whole groups of the row lie inside it because
// its stride covers ceil(d BITS / 8) bytes rounded up to words).
template <int BITS, bool BYTES>
__device__ __forceinline__ uint32_t nibbles(const uint8_t* __restrict__ row, int row_words, int g) {
  if (BITS == 4) return row_word<BYTES>(row, g);
  const int bit = 8 * BITS * g, w = bit >> 5, sh = bit & 31;
  const uint32_t x = row_word<BYTES>(row, w);
  if (BITS == 3) return spread3(__funnelshift_r(x, sh > 8 && w + 1 < row_words ? row_word<BYTES>(row, w + 1) : 0u, sh) & 0x00ffffffu);
  return BITS == 2 ? spread2((x >> sh) & 0xffffu) : spread1((x >> sh) & 0xffu);
}

// acc + the code lengths of the eight nibbles of x.
template <int BITS>
__device__ __forceinline__ uint32_t code_bits(const Code& c, uint32_t x, uint32_t acc) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const uint32_t four = h ? x >> 16 : x;
    uint32_t v = __byte_perm(c.len4[0], c.len4[1], BITS == 4 ? four & 0x7777u : four);
    if (BITS == 4) {
      const uint32_t up = __byte_perm(0x0000ff00u, 0u, (four >> 3) & 0x1111u);
      v = (v & ~up) | (__byte_perm(c.len4[2], c.len4[3], four & 0x7777u) & up);
    }
    acc = __dp4a(v, 0x01010101u, acc);
  }
  return acc;
}

// Row sizes in bytes (multiples of 4) and the total of each CTA's 8 R rows.
template <int BITS, bool BYTES>
__global__ void __launch_bounds__(256) measure_kernel(Args a, int R, uint32_t* __restrict__ sizes, uint64_t* __restrict__ totals) {
  __shared__ uint32_t warp_tot[8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int groups = (a.d + 7) / 8, row_words = (int)(a.idx_rb / 4);
  const int absent = 8 * groups - a.d;   // coordinates of the last group past the row's end: taken off again, whatever they hold
  uint32_t tot = 0;
  for (int r = 0; r < R; ++r) {
    const int64_t row = ((int64_t)blockIdx.x * R + r) * 8 + warp;
    if (row >= a.n) break;
    const uint8_t* p = a.idx + (size_t)row * a.idx_rb;
    uint32_t bits = 0;
    for (int g0 = 0; g0 < groups; g0 += 256) {   // eight loads per lane in flight
      uint32_t x[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int g = g0 + 32 * i + lane;
        x[i] = g < groups ? nibbles<BITS, BYTES>(p, row_words, g) : 0u;
      }
#pragma unroll
      for (int i = 0; i < 8; ++i)
        if (g0 + 32 * i + lane < groups) bits = code_bits<BITS>(a.code, x[i], bits);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) bits += __shfl_xor_sync(0xffffffffu, bits, o);
    if (absent > 0) {   // their nibbles moved to the bottom, index 0 above them
      const uint32_t tail = nibbles<BITS, BYTES>(p, row_words, groups - 1) >> (4 * (8 - absent));
      bits -= code_bits<BITS>(a.code, tail, 0u) - (uint32_t)(8 - absent) * a.code.len[0];
    }
    const uint32_t bytes = (bits + 31) / 32 * 4;
    if (lane == 0) sizes[row] = bytes;
    tot += bytes;
  }
  if (lane == 0) warp_tot[warp] = tot;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint64_t t = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) t += warp_tot[w];
    totals[blockIdx.x] = t;
  }
}

__device__ __forceinline__ unsigned long long warp_inclusive(unsigned long long v, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long t = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += t;
  }
  return v;
}

// Exclusive prefix sums of `count` totals in place, by one CTA that walks them in pieces of 1024 with a carry: only for so
// many rows that every CTA of offsets_kernel adding up its predecessors' totals would cost more (see tq_entropy_measure).
__global__ void __launch_bounds__(1024) prefix_totals_kernel(uint64_t* __restrict__ totals, int64_t count) {
  __shared__ unsigned long long warp_tot[32], carry;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) carry = 0ull;
  __syncthreads();
  for (int64_t base = 0; base < count; base += 1024) {
    const int64_t i = base + threadIdx.x;
    const unsigned long long v = i < count ? totals[i] : 0ull, incl = warp_inclusive(v, lane);
    if (lane == 31) warp_tot[warp] = incl;
    __syncthreads();
    if (warp == 0) {
      const unsigned long long w = warp_tot[lane];
      warp_tot[lane] = warp_inclusive(w, lane) - w;
    }
    __syncthreads();
    const unsigned long long excl = carry + warp_tot[warp] + incl - v;
    if (i < count) totals[i] = excl;
    __syncthreads();
    if (threadIdx.x == 1023) carry = excl + v;
    __syncthreads();
  }
}

// offsets[i] = sum of sizes[0 .. i-1], offsets[n] = total; a CTA of 1024 threads takes 1024 rows.  totals[g]: bytes of rows
// [g rows_per_total, (g + 1) rows_per_total), or with `prefixed` the bytes before that group.
__global__ void __launch_bounds__(1024) offsets_kernel(const uint32_t* __restrict__ sizes, const uint64_t* __restrict__ totals,
                                                       int rows_per_total, int prefixed, int64_t n, uint64_t* __restrict__ offsets) {
  __shared__ unsigned long long warp_tot[32], before[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t base = (int64_t)blockIdx.x * 1024, first = base / rows_per_total;   // rows_per_total divides 1024
  unsigned long long b = 0ull;
  if (!prefixed)
    for (int64_t g = threadIdx.x; g < first; g += 1024) b += totals[g];
  else if (threadIdx.x == 0 && base < n) b = totals[first];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) b += __shfl_xor_sync(0xffffffffu, b, o);
  const int64_t i = base + threadIdx.x;
  const unsigned long long v = i < n ? sizes[i] : 0ull, incl = warp_inclusive(v, lane);
  if (lane == 0) before[warp] = b;
  if (lane == 31) warp_tot[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    const unsigned long long w = warp_tot[lane];
    unsigned long long s = before[lane];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    warp_tot[lane] = s + warp_inclusive(w, lane) - w;
  }
  __syncthreads();
  if (i < n) {
    const unsigned long long excl = warp_tot[warp] + incl - v;
    offsets[i] = excl;
    if (i == n - 1) offsets[n] = excl + v;
  }
  if (n == 0 && i == 0) offsets[0] = 0ull;
}

// The rare cases of pack_kernel, out of line: inside it they took 8 us of 110.
// A row that ends past the buffer (false: nothing else is to be done for it) or that the caller has given more room than any
// stream needs.  Whole warps.
__device__ __noinline__ bool unusual_row(uint64_t off, uint64_t off_end, uint8_t* out, uint64_t out_bytes, uint32_t image_bytes, int* status) {
  const int lane = threadIdx.x & 31;
  if (off_end > out_bytes || off_end < off) {
    if (lane == 0) atomicExch(status, TQ_ERR_WORKSPACE);
    for (uint64_t b = off + lane; b < out_bytes && b < off_end; b += 32) out[b] = 0;
    return false;
  }
  for (uint64_t b = off + image_bytes + 4 * lane; b + 4 <= off_end; b += 128) *reinterpret_cast<uint32_t*>(out + b) = 0u;
  return true;
}
// Zeros before the first row and behind the last one (both on word boundaries).  Whole grid.
__device__ __noinline__ void clear_rest(uint64_t first, uint64_t last, uint8_t* out, uint64_t out_bytes) {
  const uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x, step = (uint64_t)gridDim.x * blockDim.x;
  auto clear = [&](uint64_t begin, uint64_t end) {
    for (uint64_t b = begin + 4 * t; b + 4 <= end; b += 4 * step) *reinterpret_cast<uint32_t*>(out + b) = 0u;
    const uint64_t tail = begin + (end - begin) / 4 * 4 + t;
    if (tail < end) out[tail] = 0;
  };
  clear(0, min(first, out_bytes));
  if (last < out_bytes) clear(last, out_bytes);
}

// Persistent over rows.  Shared memory: 256 pairs of code words x 32 copies (no two lanes meet in a bank), then one row image
// per warp.  A pair entry holds the two code words in stream order (up to 24 bits) and their length above.  A lane takes every
// 32nd group of eight coordinates; a warp scan of the groups' lengths places them.  Everything is straight-line code: a version
// that appended to a 64-bit buffer and flushed it word by word took 1,560 instructions per row of 1536 coordinates, because
// some lane flushed at every step.
constexpr int kPackWarps = 8;
template <int BITS, bool LONG, bool BYTES>   // LONG: eight code words may take more than 64 bits (a code word of more than 8)
__global__ void __launch_bounds__(32 * kPackWarps) pack_kernel(Args a, const uint64_t* __restrict__ offsets, uint8_t* __restrict__ out,
                                                               size_t out_bytes, int image_words, int* status) {
  extern __shared__ uint32_t pack_smem[];
  uint32_t* pairs = pack_smem;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t* image = pack_smem + 256 * 32 + warp * (image_words + 4);
  for (int e = warp; e < 256; e += kPackWarps) {
    const int s0 = e & 15, s1 = e >> 4;
    const int l0 = a.code.len[s0], l1 = a.code.len[s1];
    // a code word from its most significant bit = stream order: its bits reversed into LSB-first order
    const uint32_t r0 = l0 ? __brev((uint32_t)a.code.word[s0]) >> (32 - l0) : 0u, r1 = l1 ? __brev((uint32_t)a.code.word[s1]) >> (32 - l1) : 0u;
    pairs[e * 32 + lane] = r0 | (r1 << l0) | ((uint32_t)(l0 + l1) << 24);
  }
  __syncthreads();
  const uint32_t* mine = pairs + lane;
  const bool rest = offsets[0] != 0 || offsets[a.n] < out_bytes;   // bytes of the output that belong to no row
  const uint32_t image_bytes = 4u * (uint32_t)image_words;
  const int groups = (a.d + 7) / 8, row_words = (int)(a.idx_rb / 4);
  for (int64_t row = (int64_t)blockIdx.x * kPackWarps + warp; row < a.n; row += (int64_t)gridDim.x * kPackWarps) {
    const uint64_t off = offsets[row], off_end = offsets[row + 1];
    if ((off_end > out_bytes || off_end - off > image_bytes) && !unusual_row(off, off_end, out, out_bytes, image_bytes, status)) continue;
    const int words = (int)(min(off_end - off, (uint64_t)image_bytes) / 4);
    const uint8_t* p = a.idx + (size_t)row * a.idx_rb;
    for (int w = lane; w < words; w += 32) image[w] = 0u;
    __syncwarp();
    int base = 0;   // stream bits before this sweep's groups
    uint32_t next = lane < groups ? nibbles<BITS, BYTES>(p, row_words, lane) : 0u;
    for (int g0 = 0; g0 < groups; g0 += 32) {
      const int g = g0 + lane;
      const uint32_t x = next;
      if (g + 32 < groups) next = nibbles<BITS, BYTES>(p, row_words, g + 32);   // requested one sweep ahead
      unsigned long long half[2];   // four code words each, at most 48 bits
      int len[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        uint32_t e0 = mine[((x >> (16 * h)) & 255u) * 32], e1 = mine[((x >> (16 * h + 8)) & 255u) * 32];
        if (8 * (g0 + 32) > a.d) {   // the last sweep: coordinates past the row's end have no code word
          const int left = a.d - 8 * g - 4 * h;
          const uint32_t four = x >> (16 * h);
          if (left < 4) {
            if (left <= 0) e0 = 0u;
            else if (left == 1) { const uint32_t l = a.code.len[four & 15u]; e0 = (e0 & ((1u << l) - 1u)) | (l << 24); }
            if (left <= 2) e1 = 0u;
            else { const uint32_t l = a.code.len[(four >> 8) & 15u]; e1 = (e1 & ((1u << l) - 1u)) | (l << 24); }
          }
        }
        const int l0 = (int)(e0 >> 24);
        half[h] = (unsigned long long)(e0 & 0x00ffffffu) | ((unsigned long long)(e1 & 0x00ffffffu) << l0);
        len[h] = l0 + (int)(e1 >> 24);
      }
      const int mine_bits = len[0] + len[1];
      int incl = mine_bits;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
      }
      int pos = base + incl - mine_bits;
      base += __shfl_sync(0xffffffffu, incl, 31);
      // up to 64 bits shifted by up to 31: two words, rarely a third (the image has room for zero parts past its end)
      auto place = [&](unsigned long long v) {
        const int w = pos >> 5, sh = pos & 31;
        const unsigned long long lo = v << sh;
        atomicOr(image + w, (uint32_t)lo);
        atomicOr(image + w + 1, (uint32_t)(lo >> 32));
        const uint32_t v2 = __funnelshift_l((uint32_t)(v >> 32), 0u, sh);
        if (v2) atomicOr(image + w + 2, v2);
      };
      if (LONG) {
        place(half[0]);
        pos += len[0];
        place(half[1]);
      } else {
        place(half[0] | (half[1] << len[0]));
      }
    }
    __syncwarp();
    uint32_t* dst = reinterpret_cast<uint32_t*>(out + off);
    for (int w = lane; w < words; w += 32) dst[w] = image[w];
    __syncwarp();
  }
  if (rest) clear_rest(offsets[0], offsets[a.n], out, out_bytes);
}

// One thread per row.  Look-up on the next K bits: up to 16 bits of whole symbols, their number of output bits and the stream bits
// they take.  The lanes of a warp run in step by output word, so that filling and emitting words is the same instruction for all of
// them; only the number of look-ups per word differs.
// Bound: instructions issued per look-up (a chain of shifts of two-word buffers, written out in 32-bit funnel shifts: a 64-bit shift
// by a variable is six) and the look-ups per word.  K = 12 takes 2.8 of them per word of eight 4-bit symbols, K = 10 3.7, but its 16 KB
// table is L1 that the rows' lines need, so that it pays only where one CTA of many rows has the SM to itself (five CTAs of 128
// rows with it: 322 us).  100,000 rows of d = 1536: 154 -> 142 us.
__global__ void __launch_bounds__(1024) unpack_kernel(Args a, int K, const uint64_t* __restrict__ offsets,
                                                      const uint8_t* __restrict__ packed, uint8_t* __restrict__ idx_out) {
  extern __shared__ uint32_t unpack_smem[];
  uint32_t* lut = unpack_smem;                                            // [2^K]: symbols | output bits << 16 | stream bits << 24
  uint16_t* single = reinterpret_cast<uint16_t*>(unpack_smem + (1 << K)); // [2^maxlen]: symbol | length << 8
  const int L = a.code.maxlen, bits = a.code.bits;
  for (int u = threadIdx.x; u < (1 << L); u += blockDim.x) {
    uint16_t e = 1 << 8;   // no code word (an incomplete code): one bit, symbol 0
    for (int s = 0; s < (1 << bits); ++s) {
      const int l = a.code.len[s];
      if ((u & ((1u << l) - 1u)) == __brev((unsigned)a.code.word[s]) >> (32 - l)) e = (uint16_t)(s | (l << 8));
    }
    single[u] = e;
  }
  __syncthreads();
  for (int u = threadIdx.x; u < (1 << K); u += blockDim.x) {
    uint32_t sym = 0u;
    int used = 0, produced = 0;
    while (produced + bits <= 16) {
      const uint16_t e = single[(u >> used) & ((1u << L) - 1u)];
      const int l = e >> 8;
      if (used + l > K) break;   // the word may go on past the look-up window
      sym |= (uint32_t)(e & 255u) << produced;
      used += l;
      produced += bits;
    }
    lut[u] = sym | ((uint32_t)produced << 16) | ((uint32_t)used << 24);
  }
  __syncthreads();
  const int64_t row = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (row >= a.n) return;
  const uint64_t off = offsets[row];
  const uint32_t* src = reinterpret_cast<const uint32_t*>(packed + off);
  const int nwords = (int)((offsets[row + 1] - off) / 4);
  uint32_t* dst = reinterpret_cast<uint32_t*>(idx_out + (size_t)row * a.idx_rb);
  const int row_words = (int)(a.idx_rb / 4), total_bits = a.d * bits, out_words = (total_bits + 31) / 32;
  const uint32_t last_mask = (total_bits & 31) ? (1u << (total_bits & 31)) - 1u : 0xffffffffu;
  // The stream window is filled at the start of every output word by all lanes together, and only rarely inside a word: a
  // load that some lane issues at every look-up makes the other lanes of the warp wait for it (267 against 150 us).
  uint32_t in_lo = 0u, in_hi = 0u, out_lo = 0u, out_hi = 0u;
  int have = 0, rd = 0, ofill = 0;
  const unsigned mask = (1u << K) - 1u;
  uint32_t ahead = nwords > 0 ? __ldg(src) : 0u;   // the next word, requested one word early
  auto refill = [&]() {   // (have < 32.)  Zero words past the end of the row stream only pad the look-up of its last code words
    in_lo |= ahead << have;
    in_hi |= __funnelshift_l(ahead, 0u, have);
    have += 32;
    ++rd;
    ahead = rd < nwords ? __ldg(src + rd) : 0u;
  };
  auto next_word = [&]() -> uint32_t {
    if (have < 32) refill();
    do {
      if (have < K) refill();
      const uint32_t e = lut[in_lo & mask];
      const int used = e >> 24;
      in_lo = __funnelshift_r(in_lo, in_hi, used);
      in_hi >>= used;
      have -= used;
      const uint32_t symbols = e & 0xffffu;
      out_lo |= symbols << ofill;
      out_hi |= __funnelshift_l(symbols, 0u, ofill);
      ofill += (e >> 16) & 255u;
    } while (ofill < 32);
    const uint32_t v = out_lo;
    out_lo = out_hi;
    out_hi = 0u;
    ofill -= 32;
    return v;
  };
  auto checked_word = [&](int ow) -> uint32_t {
    if (ow >= out_words) return 0u;   // pad words of the row
    const uint32_t v = next_word();
    return ow == out_words - 1 ? v & last_mask : v;   // what follows the last coordinate is not a symbol
  };
  int ow = 0;
  if (row_words % 4 == 0) {
    for (; ow + 4 <= total_bits / 32; ow += 4) {
      uint4 v;
      v.x = next_word();
      v.y = next_word();
      v.z = next_word();
      v.w = next_word();
      *reinterpret_cast<uint4*>(dst + ow) = v;
    }
  }
  for (; ow < row_words; ++ow) dst[ow] = checked_word(ow);
}

bool by_bytes(const void* idx) { return (reinterpret_cast<uintptr_t>(idx) & 3) != 0; }

using MeasureFn = void (*)(Args, int, uint32_t*, uint64_t*);
MeasureFn measure_for(int bits, bool bytes) {
  static constexpr MeasureFn fns[4][2] = {{measure_kernel<1, false>, measure_kernel<1, true>}, {measure_kernel<2, false>, measure_kernel<2, true>},
                                          {measure_kernel<3, false>, measure_kernel<3, true>}, {measure_kernel<4, false>, measure_kernel<4, true>}};
  return fns[bits - 1][bytes];
}

using PackFn = void (*)(Args, const uint64_t*, uint8_t*, size_t, int, int*);
template <bool LONG, bool BYTES>
PackFn pack_for(int bits) {
  static constexpr PackFn fns[4] = {pack_kernel<1, LONG, BYTES>, pack_kernel<2, LONG, BYTES>, pack_kernel<3, LONG, BYTES>, pack_kernel<4, LONG, BYTES>};
  return fns[bits - 1];
}

int make_code(const tq_plan* plan, const uint8_t* lengths, Code* c, const char* who) {
  const int L = 1 << plan->mse_bits;
  std::memset(c, 0, sizeof(*c));
  c->bits = plan->mse_bits;
  double kraft = 0.0;
  std::vector<std::pair<int, int>> order;
  for (int s = 0; s < L; ++s) {
    TQ_REQUIRE(lengths[s] >= 1 && lengths[s] <= kMaxLen, TQ_ERR_UNSUPPORTED, "%s: code length %d of symbol %d outside 1..%d", who,
               (int)lengths[s], s, kMaxLen);
    c->len[s] = lengths[s];
    c->len4[s >> 2] |= (uint32_t)lengths[s] << (8 * (s & 3));
    c->maxlen = std::max(c->maxlen, (int)lengths[s]);
    kraft += std::ldexp(1.0, -(int)lengths[s]);
    order.push_back({(int)lengths[s], s});
  }
  TQ_REQUIRE(kraft <= 1.0, TQ_ERR_INVALID_ARG, "%s: the lengths violate Kraft's inequality (no prefix code has them)", who);
  std::sort(order.begin(), order.end());
  unsigned code = 0;
  int prev = 0;
  for (const auto& e : order) {
    code <<= e.first - prev;
    c->word[e.second] = (uint16_t)code;
    ++code;
    prev = e.first;
  }
  return TQ_OK;
}

int check(const tq_plan* plan, const char* who, const uint8_t* lengths, int64_t n) {
  TQ_REQUIRE(plan != nullptr, TQ_ERR_INVALID_ARG, "%s: plan is NULL", who);
  int dev = -1;
  TQ_CHECK_CUDA(cudaGetDevice(&dev), who);
  TQ_REQUIRE(dev == plan->device, TQ_ERR_INVALID_ARG, "%s: plan was created on device %d, current device is %d", who, plan->device, dev);
  TQ_REQUIRE(plan->mse_bits >= 1, TQ_ERR_UNSUPPORTED, "%s: the plan has no index array (0-bit MSE stage)", who);
  TQ_REQUIRE(plan->layout == TQ_LAYOUT_CANONICAL, TQ_ERR_UNSUPPORTED, "%s: the plan must use the canonical code layout", who);
  TQ_REQUIRE(lengths != nullptr && n >= 0, TQ_ERR_INVALID_ARG, "%s: lengths is NULL or n is negative", who);
  return TQ_OK;
}

}  // namespace
}  // namespace entropy

// Mass of every cell of the codebook under the density of Lemma 1 (defined in tq_host.cu).
int cell_masses(int d, int levels, const float* centroids, double* p_out);

}  // namespace tq

using namespace tq;

extern "C" int tq_entropy_lengths(int d, int bits, const float* centroids, uint8_t* lengths) {
  const char* who = "tq_entropy_lengths";
  TQ_REQUIRE(d >= 2 && d <= TQ_MAX_D && bits >= 1 && bits <= 4, TQ_ERR_UNSUPPORTED, "%s: d=%d bits=%d unsupported", who, d, bits);
  TQ_REQUIRE(centroids != nullptr && lengths != nullptr, TQ_ERR_INVALID_ARG, "%s: NULL argument", who);
  const int L = 1 << bits;
  double p[16];
  int rc = cell_masses(d, L, centroids, p);
  if (rc) return rc;
  // Huffman: merge the two least probable nodes; among equals the one created earlier goes first
  struct Node { double p; int order; unsigned mask; };
  std::vector<Node> nodes;
  int depth[16] = {0};
  for (int s = 0; s < L; ++s) nodes.push_back({p[s], s, 1u << s});
  int created = L;
  while (nodes.size() > 1) {
    std::sort(nodes.begin(), nodes.end(), [](const Node& a, const Node& b) { return a.p != b.p ? a.p < b.p : a.order < b.order; });
    const Node a = nodes[0], b = nodes[1];
    for (int s = 0; s < L; ++s)
      if ((a.mask | b.mask) >> s & 1u) ++depth[s];
    nodes.erase(nodes.begin(), nodes.begin() + 2);
    nodes.push_back({a.p + b.p, created++, a.mask | b.mask});
  }
  for (int s = 0; s < L; ++s) lengths[s] = (uint8_t)depth[s];
  return TQ_OK;
}

// Row sizes (4 bytes each), then the totals of groups of at least eight rows (8 bytes each, with room to start them on an 8-byte
// boundary of a workspace that has only a 4-byte one).
static size_t sizes_bytes(int64_t n) { return (size_t)((n * 4 + 255) / 256 * 256); }
extern "C" size_t tq_entropy_workspace_bytes(int64_t n) {
  return n > 0 ? sizes_bytes(n) + (size_t)(((n + 7) / 8 * 8 + 4 + 255) / 256 * 256) : 0;
}

extern "C" int tq_entropy_measure(const tq_plan* plan, const uint8_t* lengths, int64_t n, const uint8_t* idx, uint64_t* row_offsets,
                                  void* workspace, size_t workspace_bytes, void* stream) {
  const char* who = "tq_entropy_measure";
  TQ_RANGE(who);
  int rc = entropy::check(plan, who, lengths, n);
  if (rc) return rc;
  TQ_REQUIRE(row_offsets != nullptr && (n == 0 || idx != nullptr), TQ_ERR_INVALID_ARG, "%s: NULL argument", who);
  TQ_REQUIRE(workspace_bytes >= tq_entropy_workspace_bytes(n) && (n == 0 || workspace != nullptr), TQ_ERR_WORKSPACE,
             "%s: workspace of %zu bytes, %zu needed", who, workspace_bytes, tq_entropy_workspace_bytes(n));
  TQ_REQUIRE((n == 0 || (reinterpret_cast<uintptr_t>(workspace) & 3) == 0) && (reinterpret_cast<uintptr_t>(row_offsets) & 7) == 0, TQ_ERR_ALIGNMENT,
             "%s: workspace / row_offsets is misaligned", who);
  entropy::Args a;
  if ((rc = entropy::make_code(plan, lengths, &a.code, who))) return rc;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  a.n = n; a.d = plan->d; a.idx = idx; a.idx_rb = plan->idx_row_bytes;
  uint32_t* sizes = static_cast<uint32_t*>(workspace);
  uint64_t* totals = reinterpret_cast<uint64_t*>((reinterpret_cast<uintptr_t>(workspace) + sizes_bytes(n) + 7) & ~(uintptr_t)7);
  // eight rows per warp once that still fills the chip four times over
  const int R = n >= (int64_t)8 * 8 * 4 * tc::sm_count() ? 8 : 1;
  const int64_t groups = (n + 8 * R - 1) / (8 * R);
  // CTA j of offsets_kernel adds up the j 1024 / (8 R) totals before it: 2^21 rows make 2,048 CTAs read 16,384 totals on
  // average (0.27 GB from L2); from there on one launch turns the totals into prefix sums first
  const int prefixed = n > ((int64_t)1 << 21) ? 1 : 0;
  if (n > 0) {
    entropy::measure_for(a.code.bits, entropy::by_bytes(idx))<<<(unsigned)groups, 256, 0, st>>>(a, R, sizes, totals);
    TQ_CHECK_CUDA(cudaGetLastError(), who);
    if (prefixed) {
      entropy::prefix_totals_kernel<<<1, 1024, 0, st>>>(totals, groups);
      TQ_CHECK_CUDA(cudaGetLastError(), who);
    }
  }
  entropy::offsets_kernel<<<(unsigned)std::max<int64_t>(1, (n + 1023) / 1024), 1024, 0, st>>>(sizes, totals, 8 * R, prefixed, n, row_offsets);
  count_launches(n > 0 ? 2 + prefixed : 1);
  TQ_CHECK_CUDA(cudaGetLastError(), who);
  return TQ_OK;
}

extern "C" int tq_entropy_pack(const tq_plan* plan, const uint8_t* lengths, int64_t n, const uint8_t* idx, const uint64_t* row_offsets,
                               uint8_t* out, size_t out_bytes, void* stream) {
  const char* who = "tq_entropy_pack";
  TQ_RANGE(who);
  int rc = entropy::check(plan, who, lengths, n);
  if (rc) return rc;
  if (n == 0) return TQ_OK;
  TQ_REQUIRE(idx != nullptr && row_offsets != nullptr && out != nullptr, TQ_ERR_INVALID_ARG, "%s: NULL argument", who);
  TQ_REQUIRE((reinterpret_cast<uintptr_t>(out) & 3) == 0, TQ_ERR_ALIGNMENT, "%s: out is not 4-byte aligned", who);
  entropy::Args a;
  if ((rc = entropy::make_code(plan, lengths, &a.code, who))) return rc;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  a.n = n; a.d = plan->d; a.idx = idx; a.idx_rb = plan->idx_row_bytes;
  const int image_words = (int)(((int64_t)a.d * a.code.maxlen + 31) / 32);   // the longest row stream
  const size_t smem = (256 * 32 + (size_t)entropy::kPackWarps * (image_words + 4)) * sizeof(uint32_t);
  const int per_sm = std::max(1, std::min(8, (int)(228 * 1024 / (smem + 1024))));
  const int64_t ctas = std::min<int64_t>((n + entropy::kPackWarps - 1) / entropy::kPackWarps, (int64_t)tc::sm_count() * per_sm);
  const bool wide = a.code.maxlen > 8, bytes = entropy::by_bytes(idx);
  const auto kernel = wide ? (bytes ? entropy::pack_for<true, true>(a.code.bits) : entropy::pack_for<true, false>(a.code.bits))
                           : (bytes ? entropy::pack_for<false, true>(a.code.bits) : entropy::pack_for<false, false>(a.code.bits));
  static std::atomic<unsigned long long> smem_devices[16];   // per instantiation
  if (smem > 48 * 1024)
    TQ_CHECK_CUDA(allow_largest_smem(reinterpret_cast<const void*>(kernel), smem_devices[a.code.bits - 1 + 4 * wide + 8 * bytes]), who);
  kernel<<<(unsigned)ctas, 32 * entropy::kPackWarps, smem, st>>>(a, row_offsets, out, out_bytes, image_words, plan->d_status);
  count_launches(1);
  TQ_CHECK_CUDA(cudaGetLastError(), who);
  return TQ_OK;
}

extern "C" int tq_entropy_unpack(const tq_plan* plan, const uint8_t* lengths, int64_t n, const uint8_t* packed,
                                 const uint64_t* row_offsets, uint8_t* idx, void* stream) {
  const char* who = "tq_entropy_unpack";
  TQ_RANGE(who);
  int rc = entropy::check(plan, who, lengths, n);
  if (rc) return rc;
  if (n == 0) return TQ_OK;
  TQ_REQUIRE(idx != nullptr && row_offsets != nullptr && packed != nullptr, TQ_ERR_INVALID_ARG, "%s: NULL argument", who);
  TQ_REQUIRE((reinterpret_cast<uintptr_t>(packed) & 3) == 0 && (reinterpret_cast<uintptr_t>(idx) & 15) == 0, TQ_ERR_ALIGNMENT,
             "%s: packed / idx is misaligned", who);
  entropy::Args a;
  if ((rc = entropy::make_code(plan, lengths, &a.code, who))) return rc;
  a.n = n; a.d = plan->d; a.idx = nullptr; a.idx_rb = plan->idx_row_bytes;
  // An SM's share of the rows as one CTA (of at most 1,024) where it is worth the larger table, else CTAs of 128 rows.  Packing and
  // unpacking, CTAs of 128 rows / of the share: 37,000 rows (256 per SM) d = 128 b = 3 67.9 / 75.7 us, d = 1536 b = 2 140 / 148; 60,000 rows
  // (416 per SM) 87.3 / 87.9 and 189 / 187; 100,000 rows d = 1536 b = 4 349 / 339.
  const int64_t share = round_up64((n + tc::sm_count() - 1) / tc::sm_count(), 32);
  const bool wide = share >= 384;
  const int threads = wide ? (int)((share + (share + 1023) / 1024 - 1) / ((share + 1023) / 1024) + 31) / 32 * 32 : 128;
  const int K = wide || a.code.maxlen > 10 ? 12 : 10;
  const size_t smem = sizeof(uint32_t) * ((size_t)1 << K) + sizeof(uint16_t) * ((size_t)1 << a.code.maxlen);   // at most 24 KB
  const int64_t ctas = (n + threads - 1) / threads;
  entropy::unpack_kernel<<<(unsigned)ctas, threads, smem, static_cast<cudaStream_t>(stream)>>>(a, K, row_offsets, packed, idx);
  count_launches(1);
  TQ_CHECK_CUDA(cudaGetLastError(), who);
  return TQ_OK;
}
