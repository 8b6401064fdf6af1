// Jiffy decoder kernel (sm_103a): the encoder's steps run backwards
// ("straightforward reversal", Sec. III-C).
//
// One warp per row item (scan t, attribute a, row r). Warps take items in
// batches from an atomic ticket, in increasing order, so every item a warp
// may wait on was handed out earlier. Rows decode independently: the row table gives each row's chunk and the residual its
// first delta continues from. What chains the frames of a call is the
// prediction of P frames (Sec. III-D): k_dec_masks undoes the XOR of the masks
// along the frames ahead of the rows, and the pixels are added up either by
// the rows, which then wait (bounded) for the same row of the frame before,
// or behind the rows by k_dec_sums (k_dec_secs says which). Small calls run
// the rows kernel alone, which then does all of it. There is no CTA-wide
// barrier: a warp never waits for another warp of its CTA.
//
// Per row:
//   all      the section (found by k_dec_secs) and the row-table entry
//   lanes    class words -> literal prefix (Sec. III-C mask code)
//   mask     a mask word (32 pixels) per lane at a time: its class code or
//            literal, XOR with the previous scan's word for P (Sec. III-D);
//            one warp scan per 32 words gives each word's first compacted
//            index
//   lanes    block headers validated and sized (Sec. II, PFOR blocks)
//   then, per 256-pixel step (lane l owning the 8 consecutive pixels
//   8l .. 8l+7 of the step), interleaved:
//   unpack   the blocks the step needs, two at a time, lane l owning the 8
//            consecutive values 8l..8l+7 of their 256 (half the instructions
//            per value of one block and 4 values): a window of the body words
//            they occupy, funnel-shift extraction, exception high parts via a
//            patch buffer, inverse ZigZag (Eq. 1); running sums and a warp
//            scan from the row's carry (inverse delta, on the kept samples
//            alone), into a ring of residuals
//   scatter  compacted index of each own pixel from its mask word's; x
//            precision (Sec. III-A); + previous pixel for P; vector stores
// The row chunk is read through L1 (bulk-prefetched into L2 at the start of
// the row); residuals pass through a small ring buffer in shared memory.
#include <algorithm>

#include "jiffy_device.cuh"
#include "jiffy_kernels.h"

namespace jiffy {

namespace {

constexpr uint32_t kDecBatch = 1;  // row items per ticket unless the launch asks otherwise (1 balances the tail best)

__device__ __forceinline__ uint32_t ld_in_u32(const uint8_t* in, unsigned long long at) {
  return __ldg(reinterpret_cast<const unsigned int*>(in + at));
}

__device__ __forceinline__ uint32_t valid_word_bits(uint32_t W, uint32_t nw, uint32_t j) {
  return (j + 1 < nw || (W & 31u) == 0) ? 0xffffffffu : ((1u << (W & 31u)) - 1u);
}

__device__ __forceinline__ uint32_t literal_bits(uint32_t cwd) { return (cwd >> 1) & ~cwd & 0x55555555u; }

// Index of the segment holding global row item key: the last i with base[i] <= key.
__device__ __forceinline__ uint32_t find_seg(const uint32_t* base, uint32_t n, uint32_t key) {
  uint32_t lo = 0, hi = n;
  while (hi - lo > 1) {
    const uint32_t mid = (lo + hi) >> 1;
    if (__ldg(base + mid) <= key) lo = mid;
    else hi = mid;
  }
  return lo;
}

}  // namespace

// Per-warp shared memory (byte offsets): a ring of 512 residuals (unpacked
// ahead of the scatter; the first 8 again behind the last), a 256-word exception patch buffer, the row's block
// descriptors, zero mask words (1 = zero sample), each mask word's first
// compacted index and literal mask words.
constexpr uint32_t kRing = 512;

struct DecWarpLayout {
  uint32_t ring, patch, desc, mw, wbase, lits, bytes;
};

__host__ __device__ inline DecWarpLayout dec_warp_layout(uint32_t W) {
  DecWarpLayout L;
  L.ring = 0;
  L.patch = L.ring + 4u * (kRing + 8u);
  L.desc = L.patch + 8u * kBlockN;
  L.mw = L.desc + ((8u * ceil_div_u32(W, kBlockN) + 15u) & ~15u);
  L.wbase = L.mw + ((4u * ceil_div_u32(W, 32u) + 15u) & ~15u);
  L.lits = L.wbase + ((4u * ceil_div_u32(W, 32u) + 15u) & ~15u);
  L.bytes = (L.lits + 4u * ceil_div_u32(W, 32u) + 15u) & ~15u;
  return L;
}

// The section of attribute a in frame t of a segment, checked (a thread, or a
// warp whose lanes do the same): frame offsets before any read, the frame
// header, on request the stream header of a stream's first frame.
__device__ __forceinline__ DecSec find_section(const DecSeg& sg, uint32_t t, uint32_t a, bool stream_header) {
  const uint32_t H = sg.H, A = sg.A;
  DecSec s{};
  const unsigned long long f0 = sg.off[t], f1 = sg.off[t + 1];
  // offsets in range before any read: 4-byte aligned, a whole frame
  // header, inside `in`, after the stream header for a stream's first frame
  const unsigned long long first = (t == 0 && sg.check_shdr) ? 16ull + 8ull * A : 0ull;
  bool bad = f0 < first || f0 > f1 || (f0 & 3ull) || f1 < f0 + sg.fhdr || f1 > sg.in_len || ((f1 - f0) >> 32);
  if (!bad) {
    unsigned long long before = 0, total = 0;
    uint32_t mine = 0;
    for (uint32_t aa = 0; aa < A; aa++) {
      const uint32_t m = ld_in_u32(sg.in, f0 + 8ull + 12ull * aa);
      const uint32_t sb = ld_in_u32(sg.in, f0 + 12ull + 12ull * aa);
      if (m > 1u || sb < 8u * H || (sb & 3u)) bad = true;
      if (aa < a) before += sb;
      if (aa == a) {
        mine = sb;
        s.mode = m & 1u;
      }
      total += sb;
    }
    const uint32_t frame_bytes = ld_in_u32(sg.in, f0), scan = ld_in_u32(sg.in, f0 + 4);
    if (frame_bytes != f1 - f0 || scan != sg.frame0 + t || total + sg.fhdr != frame_bytes) bad = true;
    if (s.mode == 1u && sg.frame0 + t == 0) bad = true;
    s.sec = f0 + sg.fhdr + before;
    if (!bad && (sg.stages & kStageZstdMask)) {  // index + frame + padding before the row chunks
      const unsigned long long idx = 4ull + 4ull * sg.zm_nblk;
      if (mine - 8ull * H < idx) {
        bad = true;
      } else {
        const uint32_t F = ld_in_u32(sg.in, s.sec + 8ull * H);
        const unsigned long long part = (idx + F + 3ull) & ~3ull;
        if (part > mine - 8ull * H) bad = true;
        else s.zpart = (uint32_t)part;
      }
    }
    s.data_len = mine - 8u * H - s.zpart;
    if (stream_header && t == 0 && a == 0 && sg.check_shdr && !bad) {
      // stream header: shape, dtypes, precisions (compared without a branch
      // in between, so that the words are read together)
      uint32_t diff = (ld_in_u32(sg.in, 0) ^ 0x3159464Au) | (ld_in_u32(sg.in, 4) ^ (1u | (A << 16))) |
                      (ld_in_u32(sg.in, 8) ^ H) | (ld_in_u32(sg.in, 12) ^ sg.W);
      for (uint32_t aa = 0; aa < A; aa++)
        diff |= (ld_in_u32(sg.in, 16 + 8ull * aa) ^ attr_header_word(sg.attrs[aa].s, sg.stages)) |
                (ld_in_u32(sg.in, 20 + 8ull * aa) ^ sg.attrs[aa].P);
      bad = diff != 0u;
    }
  }
  if (bad) s = DecSec{};
  s.bad = bad ? 1u : 0u;
  return s;
}

// k_dec_secs, ahead of everything else of a call: one CTA per attribute of a
// segment (a chain), a thread per section of it. It finds and checks the
// sections, so that the rows, which are many per section, only read the
// result; left to the rows it takes each of them three dependent rounds of
// loads (replaying 100 scans of 128 x 2048: 329 us of rows, 278 us without,
// both before the unpacking was rewritten). It also decides how the chain's P
// frames are added up, and clears what the call counts with: the ticket, the
// done flags that are waited for, a blocking call's error words.
//
// P frames (Sec. III-D) after a call's first frame need the same row of the
// frame before. Either their rows wait for it (kLinkWait), which is free as
// long as the other rows keep the GPU busy meanwhile, or they write their
// residuals and k_dec_sums adds them up (kLinkSum), which costs the P planes
// another trip through memory. A P run passes from row to row in about 6 us a
// frame, and about 5000 warps decode a row each in 10 us: the rows wait while
// the longest run of the chain takes less than the whole call.
constexpr uint32_t kSecThreads = 512;
constexpr uint32_t kRunWords = 256;        // frames looked at for the longest run: 32 of these (more: summed)
constexpr uint32_t kRowsPerLink = 3000;

__global__ void __launch_bounds__(kSecThreads) k_dec_secs(DecParams p) {
  __shared__ uint32_t s_modes[kRunWords];
  __shared__ uint32_t s_kind;
  chain_start();
  const uint32_t chain = blockIdx.x, tid = threadIdx.x;
  const DecSeg& sg = p.seg[find_seg(p.seg_chain_base, p.n_seg, chain)];
  const uint32_t H = sg.H, A = sg.A, T = sg.T, a = chain - sg.chain_base;
  if (chain == 0 && tid == 0) *p.ticket = 0u;
  if (a == 0 && tid == 0 && sg.clear_err) *sg.err = 0u;
  int any = 0;
  for (uint32_t t0 = 0; t0 < T; t0 += kSecThreads) {
    const uint32_t t = t0 + tid;
    DecSec s{};
    if (t < T) {
      s = find_section(sg, t, a, true);
      p.secs[sg.sec_base + t * A + a] = s;
    }
    const bool linked = t >= 1u && s.mode == 1u;  // needs the frame before it in this call
    any |= linked;
    const uint32_t bits = __ballot_sync(0xffffffffu, linked);
    if (lane_id() == 0 && (t >> 5) < kRunWords) s_modes[t >> 5] = bits;
  }
  any = __syncthreads_or(any);
  if (!any) {
    if (tid == 0) p.chain_p[chain] = kLinkNone;
    return;
  }
  if (tid == 0) {
    uint32_t longest = 0, run = 0;
    const uint32_t nwords = ceil_div_u32(T, 32u);
    for (uint32_t w = 0; w < min(nwords, kRunWords); w++) {
      uint32_t m = s_modes[w], left = 32u;
      while (left) {  // alternating runs of ones and zeros
        const uint32_t ones = ~m ? (uint32_t)__ffs(~m) - 1u : 32u, n1 = min(ones, left);
        run += n1;
        longest = max(longest, run);
        left -= n1;
        if (!left) break;
        m >>= n1;
        run = 0;
        const uint32_t n0 = m ? min((uint32_t)__ffs(m) - 1u, left) : left;
        left -= n0;
        m >>= n0 & 31u;
        if (n0 == 32u) m = 0;
      }
    }
    // (the test hook withholds a row's completion: its chain then waits for it)
    const bool wait = p.withhold || (nwords <= kRunWords && (unsigned long long)longest * kRowsPerLink <= p.n_items);
    s_kind = wait ? kLinkWait : kLinkSum;
    p.chain_p[chain] = s_kind;
  }
  __syncthreads();
  const uint32_t kind = s_kind;
  for (uint32_t t = tid; t < T; t += kSecThreads) {
    DecSec* s = p.secs + sg.sec_base + t * A + a;
    uint32_t link = 0;
    if (t >= 1u && s->mode == 1u) link = kind;
    if (kind == kLinkWait && t + 1u < T && s[A].mode == 1u) link |= kLinkNext;
    s->link = link;
  }
  if (kind == kLinkWait)
    for (uint32_t i = tid; i < T * H; i += kSecThreads) p.done[sg.item_base + a * T * H + i] = 0u;
}

// Waits (bounded) until the flag at p has reached v. One lane calls it.
__device__ __noinline__ bool wait_flag(const uint32_t* p, uint32_t v) {
  const volatile uint32_t* c = p;
  if (*c >= v) return true;
  const unsigned long long t0 = global_timer_ns();
  uint32_t ns = 32;
  while (*c < v) {
    __nanosleep(ns);
    if (ns < 256) ns <<= 1;
    if (global_timer_ns() - t0 > kSpinLimitNs) return false;
  }
  return true;
}

// The chains of a call whose P frames are handled in the ways `kinds` (bits
// 1 << kLinkWait, 1 << kLinkSum), 256 chains at a time, and the work items
// each of them has: CTAs of the chain kernels take items of all of them in
// turn. Every thread of a 256-thread CTA calls load; returns the items.
struct ChainList {
  uint32_t start[257], warps[8];
  template <typename Items>
  __device__ __forceinline__ uint32_t load(const DecParams& p, uint32_t base, uint32_t kinds, Items items) {
    const uint32_t tid = threadIdx.x, c = base + tid;
    __syncthreads();
    uint32_t n = 0;
    if (c < p.n_chains && ((kinds >> p.chain_p[c]) & 1u)) n = items(p.seg[find_seg(p.seg_chain_base, p.n_seg, c)]);
    const uint32_t incl = warp_incl_scan(n);
    if (lane_id() == 31u) warps[warp_id()] = incl;
    __syncthreads();
    uint32_t off = 0;
    for (uint32_t w = 0; w < warp_id(); w++) off += warps[w];
    start[tid + 1u] = off + incl;
    if (tid == 0) start[0] = 0u;
    __syncthreads();
    return start[256];
  }
  __device__ __forceinline__ uint32_t find(uint32_t i) const {  // the chain (from base) of item i
    uint32_t lo = 0, hi = 256;
    while (hi - lo > 1u) {
      const uint32_t m = (lo + hi) >> 1;
      if (start[m] <= i) lo = m;
      else hi = m;
    }
    return lo;
  }
};

// The mode of attribute a in frame t of a segment (0 past the call's frames;
// malformed sections count as I, their rows report them).
__device__ __forceinline__ uint32_t frame_mode(const DecParams& p, const DecSeg& sg, uint32_t a, uint32_t t) {
  return t < sg.T ? p.secs[sg.sec_base + t * sg.A + a].mode : 0u;
}

// k_dec_masks, ahead of the rows of a call with segments of several frames:
// the masks of P frames are chained by XOR (Sec. III-D). Left to the rows,
// every frame of a P run waits for the frame before it (6 us a frame at 64 x
// 489 with masks and pixels waited for apart, 19 us when it waited for the
// whole decode). Here CTAs take the rows of an attribute:
// a thread reads the coded mask words of one frame, and the frames are
// combined by a scan over the lanes that restarts at every I frame (and over
// the CTA's 8 warps through shared memory, 256 frames at a time). The masks
// of the P frames and of the frames before them are written; the rows then
// decode independently of one another. A warp walking the frames one by one
// took 90 us for 100 frames of 64 x 489, this takes 13 us. An attribute
// without P frames ends after reading its modes, once per CTA and not per
// row (which cost 26 us for 64 streams).
constexpr uint32_t kMaskThreads = 256;
constexpr uint32_t kMaskWarps = kMaskThreads / 32;
constexpr uint32_t kMaskPart = 32;  // mask words of a row that a CTA takes at a time (a multiple of 16)

// The coded mask words of a row, read four at a time by one thread (all
// loads of a group are requested before the first is used).
struct MaskWords {
  const uint32_t* chunk;  // class words, then literals (null: all zero)
  uint32_t words, lit;    // the chunk's words; the next literal
  const uint8_t* zrow;    // or the row's bytes of a decoded Zstandard frame
  uint32_t zrb;
  __device__ __forceinline__ void next4(uint32_t j0, uint32_t nw, uint32_t last_valid, uint32_t (&c)[4]) {
    if (zrow) {
#pragma unroll
      for (uint32_t i = 0; i < 4u; i++) {
        const uint32_t j = j0 + i;
        c[i] = 0;
        if ((zrb & 3u) == 0u) {
          if (j < nw) c[i] = __ldcg(reinterpret_cast<const uint32_t*>(zrow) + j);
        } else {
#pragma unroll
          for (uint32_t q = 0; q < 4u; q++)
            if (4u * j + q < zrb) c[i] |= (uint32_t)__ldcg(zrow + 4u * j + q) << (8u * q);
        }
      }
    } else {
      const uint32_t cw = chunk ? __ldg(chunk + (j0 >> 4)) >> (2u * (j0 & 15u)) : 0u;
#pragma unroll
      for (uint32_t i = 0; i < 4u; i++) {
        const uint32_t cls = (cw >> (2u * i)) & 3u;
        const bool l = cls == 2u;
        c[i] = l && lit < words ? __ldg(chunk + lit) : (cls == 1u ? 0xffffffffu : 0u);
        lit += l;
      }
    }
#pragma unroll
    for (uint32_t i = 0; i < 4u; i++)
      if (j0 + i + 1u >= nw) c[i] &= last_valid;
  }
};

// Undoes the XORs of mask words [j0, j1) of row r of attribute a: ONE, a warp
// (up to 32 frames), else the CTA.
template <bool ONE>
__device__ __forceinline__ void undo_masks(const DecParams& p, const DecSeg& sg, uint32_t a, uint32_t r, uint32_t j0,
                                           uint32_t j1, uint32_t* s_last, uint32_t* s_reset, uint32_t* carry) {
  const uint32_t lane = lane_id(), wp = ONE ? 0u : warp_id(), tid = ONE ? lane : threadIdx.x;
  auto sync = [] {
    if (ONE) __syncwarp();
    else __syncthreads();
  };
  if (ONE) s_last = carry;
  const uint32_t H = sg.H, W = sg.W, nw = sg.nw, ncls = sg.ncls, T = sg.T;
  const bool zmask = (sg.stages & kStageZstdMask) != 0u;
  if (tid < kMaskPart) carry[tid] = 0u;
  sync();
  if (frame_mode(p, sg, a, 0u)) {  // the zero bits of the scan before the call
    const uint32_t S = sg.attrs[a].s;
    const uint8_t* prow = sg.state[a] + (size_t)r * W * S;
    for (uint32_t j = j0 + wp; j < j1; j += ONE ? 1u : kMaskWarps) {
      const uint32_t x = 32u * j + lane;
      const uint32_t z = __ballot_sync(0xffffffffu, x < W && load_sample_cg(prow, S, x) == 0u);
      if (lane == 0) carry[j - j0] = z;
    }
  }
  sync();
  for (uint32_t T0 = 0; T0 < T; T0 += kMaskThreads) {
    const uint32_t t = T0 + tid;
    const uint32_t pm = frame_mode(p, sg, a, t);
    const bool goes_on = frame_mode(p, sg, a, t + 1u) != 0u;
    const bool need = t < T && (pm || goes_on);
    MaskWords mw{nullptr, 0u, ncls, nullptr, sg.zm_rb};
    if (need && zmask) {
      mw.zrow = p.zdec + sg.zm_base + (size_t)(t * sg.A + a) * sg.zm_stride + (size_t)r * sg.zm_rb;
    } else if (need) {
      const DecSec si = p.secs[sg.sec_base + t * sg.A + a];
      if (!si.bad) {
        const uint32_t start = r ? ld_in_u32(sg.in, si.sec + 8ull * (r - 1)) : 0u;
        const uint32_t end = ld_in_u32(sg.in, si.sec + 8ull * r);
        if (!((start | end) & 3u) && start <= end && end <= si.data_len && end - start >= 4u * ncls) {
          mw.chunk = reinterpret_cast<const uint32_t*>(sg.in + si.sec + 8ull * H + start);
          mw.words = (end - start) / 4u;
          for (uint32_t i = 0; i < (j0 >> 4); i++) mw.lit += __popc(literal_bits(__ldg(mw.chunk + i)));
        }
      }
    }
    const uint32_t needs = __ballot_sync(0xffffffffu, need);
    const uint32_t resets = __ballot_sync(0xffffffffu, !pm);
    // the lane before the first of the run that a lane belongs to (-1: lane
    // 0 starts it, 32: the run goes on from the frames before)
    const uint32_t upto = resets & (0xffffffffu >> (31u - lane));
    const int before = upto ? 30 - __clz(upto) : 32;
    auto undo = [&](uint32_t (&c)[4], const uint32_t (&from)[4]) {  // warp-wide: coded words -> masks
      uint32_t u[4];
#pragma unroll
      for (uint32_t o = 1; o < 32u; o <<= 1) {
#pragma unroll
        for (uint32_t i = 0; i < 4u; i++) u[i] = __shfl_up_sync(0xffffffffu, c[i], o);
#pragma unroll
        for (uint32_t i = 0; i < 4u; i++) c[i] ^= lane >= o ? u[i] : 0u;
      }
#pragma unroll
      for (uint32_t i = 0; i < 4u; i++) u[i] = __shfl_sync(0xffffffffu, c[i], before & 31);
#pragma unroll
      for (uint32_t i = 0; i < 4u; i++) c[i] ^= before == 32 ? from[i] : (before < 0 ? 0u : u[i]);
    };
    const uint32_t last_valid = valid_word_bits(W, nw, nw - 1u);
    if (!ONE && T - T0 > 32u) {  // the warps' last masks, as if nothing came before them; then each warp's carry
      // (where the next warp's first frame continues a run)
      if (__shfl_sync(0xffffffffu, (uint32_t)goes_on, 31)) {
        MaskWords m = mw;
        const uint32_t none[4] = {0, 0, 0, 0};
        for (uint32_t j = j0; j < j1; j += 4u) {
          uint32_t c[4] = {0, 0, 0, 0};
          if (need) m.next4(j, nw, last_valid, c);
          undo(c, none);
          if (lane == 31u) *reinterpret_cast<uint4*>(s_last + wp * kMaskPart + j - j0) = make_uint4(c[0], c[1], c[2], c[3]);
        }
      }
      if (lane == 0) s_reset[wp] = resets;
      sync();
      if (tid < kMaskPart) {
        uint32_t from = carry[tid];
        for (uint32_t w = 0; w < kMaskWarps; w++) {
          const uint32_t x = s_last[w * kMaskPart + tid] ^ (s_reset[w] ? 0u : from);
          s_last[w * kMaskPart + tid] = from;
          from = x;
        }
        carry[tid] = from;  // (of the next round)
      }
    } else if (!ONE && tid < kMaskPart) {
      s_last[tid] = carry[tid];
    }
    sync();
    if (needs) {
      uint32_t* om = p.masks + sg.mask_base + ((size_t)(a * T + t) * H + r) * nw;
      for (uint32_t j = j0; j < j1; j += 4u) {
        const uint4 f4 = *reinterpret_cast<const uint4*>(s_last + wp * kMaskPart + j - j0);
        const uint32_t from[4] = {f4.x, f4.y, f4.z, f4.w};
        uint32_t c[4] = {0, 0, 0, 0};
        if (need) mw.next4(j, nw, last_valid, c);
        undo(c, from);
        if (need)
#pragma unroll
          for (uint32_t i = 0; i < 4u; i++)
            if (j + i < nw) om[j + i] = c[i];
      }
    }
    sync();
  }
}

__global__ void __launch_bounds__(kMaskThreads) k_dec_masks(DecParams p) {
  __shared__ __align__(16) uint32_t s_last[kMaskWarps * kMaskPart];  // last masks of the warps' frames
  __shared__ uint32_t s_reset[kMaskWarps], s_carry[kMaskPart];       // the mask before the frames of a round
  __shared__ ChainList list;
  chain_wait();
  chain_start();
  for (uint32_t base = 0; base < p.n_chains; base += 256u) {
    // (up to 32 frames: a warp takes a part of a row, else the whole CTA)
    const uint32_t total = list.load(p, base, (1u << kLinkWait) | (1u << kLinkSum), [](const DecSeg& sg) {
      if (sg.stages & kStageNoMask) return 0u;
      const uint32_t parts = sg.H * ceil_div_u32(sg.nw, kMaskPart);
      return sg.T <= 32u ? ceil_div_u32(parts, kMaskWarps) : parts;
    });
    for (uint32_t i = blockIdx.x; i < total; i += gridDim.x) {
      const uint32_t c = list.find(i);
      const DecSeg& sg = p.seg[find_seg(p.seg_chain_base, p.n_seg, base + c)];
      const uint32_t a = base + c - sg.chain_base, parts = ceil_div_u32(sg.nw, kMaskPart);
      const bool one = sg.T <= 32u;
      const uint32_t k = one ? (i - list.start[c]) * kMaskWarps + warp_id() : i - list.start[c];
      const uint32_t j0 = (k % parts) * kMaskPart, j1 = min(j0 + kMaskPart, sg.nw);
      if (!one) undo_masks<false>(p, sg, a, k / parts, j0, j1, s_last, s_reset, s_carry);
      else if (k < sg.H * parts) undo_masks<true>(p, sg, a, k / parts, j0, j1, s_last, s_reset, s_last + warp_id() * kMaskPart);
      __syncthreads();
    }
  }
}

// k_dec_sums, after the rows of such a call: out_t = kept ? R_t + out_{t-1} : 0
// along the P frames of a row (Sec. III-D, modulo the sample width), R_t as
// the row items wrote it, kept out of the masks. A CTA takes 256 pixels and
// the P runs that start in a group of 32 frames (runs are independent of one
// another), a thread one pixel: neighbouring lanes neighbouring pixels, so
// any alignment of the planes is coalesced. Eight frames are loaded ahead, so
// that the chain costs a load's latency per eight frames. (A lane walking 8
// pixels frame by frame took 270 us for 100 frames of 64 x 489.)
constexpr uint32_t kSumThreads = 256;
constexpr uint32_t kSumAhead = 8;  // frames loaded ahead (divides 32)

template <typename Sample>
__device__ __forceinline__ void sum_runs(const DecParams& p, const DecSeg& sg, uint32_t a, uint32_t r, uint32_t px0,
                                         uint32_t g0, Sample** s_row, uint32_t nomask) {
  const uint32_t W = sg.W, H = sg.H, T = sg.T, A = sg.A, nw = sg.nw, lane = lane_id();
  const uint32_t x = px0 + threadIdx.x, xc = min(x, W - 1u);
  const size_t ro = (size_t)r * W + xc;
  const bool in = x < W;
  const uint32_t* mask = p.masks + sg.mask_base + ((size_t)a * T * H + r) * nw + (xc >> 5);
  const size_t mstep = (size_t)H * nw;
  Sample* const state = reinterpret_cast<Sample*>(sg.state_next[a]) + ro;
  Sample v = 0;
  bool open = false;  // in a run that started at g0 or later
  for (uint32_t t0 = g0; t0 < T; t0 += 32u) {
    // frames t0 .. t0 + 31 and the one before: their planes, their modes
    __syncthreads();
    if (threadIdx.x < 33u) {
      const uint32_t t = t0 - 1u + threadIdx.x;
      s_row[threadIdx.x] = t < T ? reinterpret_cast<Sample*>(sg.outp[t * A + a]) : nullptr;
    }
    __syncthreads();
    uint32_t ps = __ballot_sync(0xffffffffu, frame_mode(p, sg, a, t0 + lane));
    if (t0 == g0) {  // a run that goes on from before g0 belongs to another group
      if (g0 > 1u && frame_mode(p, sg, a, g0 - 1u)) ps &= ~ps ? 0xffffffffu << (__ffs(~ps) - 1) : 0u;
    } else {  // past the group: only the run that is still open
      ps = open ? (~ps ? ps & ((1u << (__ffs(~ps) - 1)) - 1u) : ps) : 0u;
    }
    if (!ps) return;
#pragma unroll 1
    for (uint32_t q0 = 0; q0 < 32u; q0 += kSumAhead) {
      const uint32_t m = (ps >> q0) & ((1u << kSumAhead) - 1u);
      if (!m) {
        open = false;
        continue;
      }
      Sample R[kSumAhead], B[kSumAhead];  // R_t; out_{t-1} where a run starts
      uint32_t z[kSumAhead];
#pragma unroll
      for (uint32_t q = 0; q < kSumAhead; q++) {
        const bool on = in && ((m >> q) & 1u);
        const bool start = on && (q ? !((m >> (q - 1u)) & 1u) : !open);
        R[q] = on ? __ldcg(s_row[q0 + q + 1u] + ro) : (Sample)0;
        B[q] = start ? __ldcg(s_row[q0 + q] + ro) : (Sample)0;
        z[q] = on && !nomask ? __ldcg(mask + (t0 + q0 + q) * mstep) : 0u;
      }
#pragma unroll
      for (uint32_t q = 0; q < kSumAhead; q++) {
        if ((m >> q) & 1u) {
          if (q ? !((m >> (q - 1u)) & 1u) : !open) v = B[q];
          v = ((z[q] >> (xc & 31u)) & 1u) ? (Sample)0 : (Sample)(R[q] + v);
          if (in) {
            s_row[q0 + q + 1u][ro] = v;
            if (t0 + q0 + q + 1u == T) *state = v;
          }
        }
      }
      open = (m >> (kSumAhead - 1u)) & 1u;
    }
    if (!open) return;
  }
}

__global__ void __launch_bounds__(kSumThreads) k_dec_sums(DecParams p) {
  __shared__ void* s_row[33];
  __shared__ ChainList list;
  chain_wait();
  chain_start();
  for (uint32_t base = 0; base < p.n_chains; base += 256u) {
    const uint32_t total = list.load(p, base, 1u << kLinkSum, [](const DecSeg& sg) {
      return sg.H * ceil_div_u32(sg.W, kSumThreads) * ceil_div_u32(sg.T - 1u, 32u);
    });
    for (uint32_t i = blockIdx.x; i < total; i += gridDim.x) {
      const uint32_t c = list.find(i);
      const DecSeg& sg = p.seg[find_seg(p.seg_chain_base, p.n_seg, base + c)];
      const uint32_t a = base + c - sg.chain_base, S = sg.attrs[a].s;
      const uint32_t cols = ceil_div_u32(sg.W, kSumThreads), k = i - list.start[c];
      const uint32_t px0 = (k % cols) * kSumThreads, r = k / cols % sg.H, g0 = 1u + 32u * (k / cols / sg.H);
      const uint32_t nomask = sg.stages & kStageNoMask;
      if (S == 4) sum_runs(p, sg, a, r, px0, g0, reinterpret_cast<uint32_t**>(s_row), nomask);
      else if (S == 2) sum_runs(p, sg, a, r, px0, g0, reinterpret_cast<uint16_t**>(s_row), nomask);
      else sum_runs(p, sg, a, r, px0, g0, reinterpret_cast<uint8_t**>(s_row), nomask);
    }
  }
}

// STAGED: the segments may have stage switches, or the test hook may be set
// (else both are read as 0). LOCAL: a small call, the rows kernel alone: each
// row finds its section itself, and the rows of a P run wait for one another,
// for the mask (done flag 1) before their own mask and for the pixels (2)
// before their own pixels.
template <bool STAGED, bool LOCAL>
__device__ __forceinline__ void decode_item(const DecParams& p, const uint32_t k, uint32_t* ring,
                                            uint32_t* patch, uint2* desc, uint32_t* mw, uint32_t* wbase,
                                            uint32_t* lits) {
  const DecSeg& sg = p.seg[find_seg(p.seg_item_base, p.n_seg, k)];
  const uint32_t lane = lane_id();
  const uint32_t H = sg.H, W = sg.W, A = sg.A, nw = sg.nw, ncls = sg.ncls;
  const uint32_t stages = STAGED ? sg.stages : 0u;
  const uint32_t niter = ceil_div_u32(W, 256u);
  const uint32_t kl = k - sg.item_base;  // item within the segment
  // row items of a segment are numbered attribute-major, (a, t, r): resident
  // warps decode one attribute's rows at a time
  const uint32_t r = kl % H, at_idx = kl / H, a = at_idx / sg.T, t = at_idx % sg.T;
  const uint32_t ta = t * A + a;
  const AttrDev at = sg.attrs[a];
  const uint32_t S = at.s;
  const size_t rowb = (size_t)W * S;

  // ---- the section (as k_dec_secs found it), the row-table entry
  DecSec si;
  if (LOCAL) {
    si = find_section(sg, t, a, r == 0);
    if (si.mode == 1u && t > 0u) si.link = kLinkWait;
    if (si.bad) {
      si.link = kLinkNext;  // (whoever waits for it is not kept waiting)
    } else if (t + 1u < sg.T) {
      const unsigned long long g0 = sg.off[t + 1], g1 = sg.off[t + 2];
      if (g1 >= g0 + sg.fhdr && g1 <= sg.in_len && !(g1 & 3ull) && ld_in_u32(sg.in, g0 + 8ull + 12ull * a) == 1u)
        si.link |= kLinkNext;
    }
  } else {
    si = p.secs[sg.sec_base + ta];
  }
  const uint32_t mode = si.mode;
  // P rows after the call's first frame: the mask comes from k_dec_masks, and
  // the row either waits for the same row of the frame before, or writes q P
  // of its residuals alone and k_dec_sums adds the frames up
  const bool chained = (si.link & 3u) != kLinkNone, summed = (si.link & 3u) == kLinkSum;
  bool bad = si.bad != 0u;
  uint32_t clen = 0, carry = 0;
  unsigned long long chunk_off = 0;
  if (!bad) {
    const uint32_t end = ld_in_u32(sg.in, si.sec + 8ull * r);
    carry = ld_in_u32(sg.in, si.sec + 8ull * r + 4);
    const uint32_t start = r ? ld_in_u32(sg.in, si.sec + 8ull * (r - 1)) : 0u;
    if (start > end || end > si.data_len || (r + 1 == H && end != si.data_len) || ((start | end) & 3u) ||
        end - start > row_bound_bytes(W) || end - start < 4u * ncls)
      bad = true;
    clen = end - start;
    chunk_off = si.sec + 8ull * H + si.zpart + start;
  }

  // ---- the chunk is read through L1: fetched into L2 in one bulk request,
  //      its lines requested for L1 by the lanes (one round)
  const uint32_t* chunk = reinterpret_cast<const uint32_t*>(sg.in + chunk_off);
  if (!bad) {
    if (lane == 0) {
      const uintptr_t c0 = reinterpret_cast<uintptr_t>(chunk), c1 = c0 + clen;
      const uintptr_t a0 = (c0 + 15u) & ~uintptr_t(15), a1 = c1 & ~uintptr_t(15);
      if (a1 > a0)
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(a0), "r"((uint32_t)(a1 - a0)) : "memory");
    }
    prefetch_l1(chunk, clen);
  }
  // ---- class words: class 3 and bits past nw are invalid; literal prefix
  uint32_t cw = 0, lit = 0;
  if (!bad && lane < ncls) {
    cw = chunk[lane];
    uint32_t used = 0xffffffffu;
    const uint32_t nslots = min(16u, nw - 16u * lane);
    if (nslots < 16u) used = (1u << (2u * nslots)) - 1u;
    lit = __popc(literal_bits(cw));
    if (((cw >> 1) & cw & 0x55555555u) || (cw & ~used)) bad = true;
  }
  const uint32_t litincl = warp_incl_scan(lit);
  const uint32_t litpre = litincl - lit;
  const uint32_t nlit = __shfl_sync(0xffffffffu, litincl, 31);
  bad = __any_sync(0xffffffffu, bad) || 4u * (ncls + nlit) > clen;
  if (!bad) {  // the row's literal mask words, one coalesced read into shared memory
    for (uint32_t i = lane; i < nlit; i += 32u) lits[i] = chunk[ncls + i];
    __syncwarp();
  }
  {  // a literal last mask word may not set bits past W
    const uint32_t j = nw - 1;
    const uint32_t cwj = __shfl_sync(0xffffffffu, cw, (j >> 4) & 31u);
    const uint32_t lpj = __shfl_sync(0xffffffffu, litpre, (j >> 4) & 31u);
    if (!bad && (W & 31u) && ((cwj >> (2u * (j & 15u))) & 3u) == 2u) {
      const uint32_t li = lpj + __popc(literal_bits(cwj) & ((1u << (2u * (j & 15u))) - 1u));
      if (lits[li] & ~valid_word_bits(W, nw, j)) bad = true;
    }
  }

  uint8_t* orow = sg.outp[ta] + r * rowb;
  uint8_t* srow = (t + 1 == sg.T && !summed) ? sg.state_next[a] + r * rowb : nullptr;
  const uint8_t* prow = (mode == 1u && !summed) ? (t > 0 ? sg.outp[ta - A] : sg.state[a]) + r * rowb : nullptr;
  const bool vec_prev = prow && vec_ok(prow, S);
  if (!bad && prow && t == 0 && lane == 0) {  // the previous scan's row, for the P sums of the scatter
    const uintptr_t c0 = reinterpret_cast<uintptr_t>(prow), c1 = c0 + rowb;
    const uintptr_t a0 = (c0 + 15u) & ~uintptr_t(15), a1 = c1 & ~uintptr_t(15);
    if (a1 > a0)
      asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(a0), "r"((uint32_t)(a1 - a0)) : "memory");
  }
  const bool vec_out = vec_ok(orow, S) && (!srow || vec_ok(srow, S));

  // ---- zero mask, a word (32 pixels) per lane at a time: class code or
  //      literal (Sec. III-C); for P (Sec. III-D) the XOR with the previous
  //      scan's mask is undone (first frame: taken from its samples; later
  //      ones: k_dec_masks has done it). Without the mask stage (no class
  //      words) every sample is coded. One warp scan per 32 words gives each
  //      word's first compacted index.
  uint32_t n = 0, late = 0;
  bool zbad = false;
  auto wait_row = [&](uint32_t v) {  // for the row of the frame before (bounded)
    if (lane == 0 && !wait_flag(p.done + (k - H), v)) {
      late = 1;
      atomicOr(sg.err, kErrTimeout);
    }
    late = __shfl_sync(0xffffffffu, late, 0);
    bad = late != 0u;
    __threadfence();
  };
  if (LOCAL && chained && !bad && !(stages & kStageNoMask)) wait_row(1u);
  if (!bad) {
    const bool nomask = (stages & kStageNoMask) != 0u;
    const bool links = LOCAL && !nomask;
    const uint32_t* pmask = (links && chained) ? p.masks + sg.mask_base + (size_t)(kl - H) * nw : nullptr;
    uint32_t* omask = (links && (si.link & kLinkNext)) ? p.masks + sg.mask_base + (size_t)kl * nw : nullptr;
    const uint32_t* fmask = (!LOCAL && chained && !nomask) ? p.masks + sg.mask_base + (size_t)kl * nw : nullptr;
    const bool prev_samples = prow && !chained && !nomask;
    // the row's coded mask bytes from the section's Zstandard frame (decoded
    // by k_zstd_dec); a bit past W is malformed
    const uint8_t* zrow = (STAGED && (stages & kStageZstdMask))
                              ? p.zdec + sg.zm_base + (size_t)ta * sg.zm_stride + (size_t)r * sg.zm_rb
                              : nullptr;
    const uint32_t zrb = sg.zm_rb;
    if (prev_samples) {  // the previous scan's zero bits, 8 pixels per lane per step, into mw
      uint8_t* pb = reinterpret_cast<uint8_t*>(mw);
      for (uint32_t it = 0; it < niter; it++) {
        const uint32_t x0 = 256u * it + 8u * lane;
        if (x0 < W) {
          const uint32_t nv = min(8u, W - x0);
          uint32_t pv[8];
          load8<true>(prow, S, x0, nv, vec_prev, pv);
          uint32_t pm = 0;
#pragma unroll
          for (int i = 0; i < 8; i++) pm |= (uint32_t)(pv[i] == 0u) << i;
          pb[x0 >> 3] = (uint8_t)pm;
        }
      }
      __syncwarp();
    }
    for (uint32_t j0 = 0; j0 < nw; j0 += 32u) {
      const uint32_t j = j0 + lane;
      const uint32_t cwj = __shfl_sync(0xffffffffu, cw, (j >> 4) & 31u);
      const uint32_t lpj = __shfl_sync(0xffffffffu, litpre, (j >> 4) & 31u);
      uint32_t kept = 0;
      if (j < nw) {
        const uint32_t valid = valid_word_bits(W, nw, j);
        uint32_t X = 0;
        if (ncls) {
          const uint32_t sl = 2u * (j & 15u), cls = (cwj >> sl) & 3u;
          if (cls == 1u) X = valid;
          else if (cls == 2u) X = lits[lpj + __popc(literal_bits(cwj) & ((1u << sl) - 1u))];
          if (LOCAL && pmask) X ^= __ldcg(pmask + j);
          else if (prev_samples) X ^= mw[j];  // bits past W are cleared below
          X &= valid;
        } else if (zrow) {
          if ((zrb & 3u) == 0u) {
            X = __ldcg(reinterpret_cast<const uint32_t*>(zrow) + j);
          } else {
            for (uint32_t q = 0; q < 4u && 4u * j + q < zrb; q++) X |= (uint32_t)__ldcg(zrow + 4u * j + q) << (8u * q);
          }
          zbad |= (X & ~valid) != 0u;
          if (LOCAL && pmask) X ^= __ldcg(pmask + j);
          else if (prev_samples) X ^= mw[j];
          X &= valid;
        }
        if (!LOCAL && fmask) X = __ldcg(fmask + j) & valid;
        if (LOCAL && omask) omask[j] = X;
        mw[j] = X;
        kept = __popc(~X & valid);
      }
      uint32_t tot;
      const uint32_t ex = warp_excl_scan(kept, tot);
      if (j < nw) wbase[j] = n + ex;
      n += tot;
    }
  }
  bad = bad || __any_sync(0xffffffffu, zbad);
  __syncwarp();
  if (LOCAL && (si.link & kLinkNext)) {  // the mask is there for the row of the next frame
    __threadfence();
    __syncwarp();
    if (lane == 0 && (!STAGED || k + 1u != p.withhold)) atomicExch(p.done + k, 1u);
  }
  const uint32_t nb = ceil_div_u32(n, kBlockN);

  // ---- block headers (lane l: blocks 4l .. 4l+3): validate, size the
  //      bodies, check they fill the chunk exactly; descriptors {body word,
  //      b | e << 8 | hb << 16 | m << 24} for the unpack
  const uint32_t hdr0 = ncls + nlit;
  if (!bad && 4u * (hdr0 + nb) > clen) bad = true;
  {
    uint32_t sz[4], hv[4], mysum = 0;
    bool lbad = false;
#pragma unroll
    for (uint32_t q = 0; q < 4; q++) {
      const uint32_t blk = 4u * lane + q;
      sz[q] = 0;
      hv[q] = 0;
      if (!bad && blk < nb) {
        const uint32_t h = chunk[hdr0 + blk];
        const uint32_t b = h & 0xffu, e = (h >> 8) & 0xffu, hb = (h >> 16) & 0xffu;
        const uint32_t m = min(kBlockN, n - blk * kBlockN);
        if ((h >> 24) || b > 32u || hb > 32u || b + hb > 32u || e > m || ((e == 0u) != (hb == 0u))) lbad = true;
        sz[q] = block_body_bytes(m, min(b, 32u), min(e, m), min(b + hb, 32u)) / 4u;
        hv[q] = (h & 0x00ffffffu) | (m << 24);
        mysum += sz[q];
      }
    }
    bad = __any_sync(0xffffffffu, bad || lbad);
    uint32_t total;
    uint32_t o = hdr0 + nb + warp_excl_scan(mysum, total);
    if (!bad && 4u * (hdr0 + nb + total) != clen) bad = true;
#pragma unroll
    for (uint32_t q = 0; q < 4; q++) {
      const uint32_t blk = 4u * lane + q;
      if (blk < nb) desc[blk] = make_uint2(o, hv[q]);
      o += sz[q];
    }
  }
  __syncwarp();

  // ---- unpack, two blocks at a time (lane l: 8 consecutive values, a
  //      register window of the body words they occupy, funnel-shift
  //      extraction; exceptions' high parts through the patch buffer;
  //      inverse ZigZag, Eq. 1; inverse delta from the running residual) into
  //      a ring of residuals, interleaved with the scatter by position: x
  //      precision (Sec. III-A), + the previous pixel for P
  if (chained && !summed && !bad) wait_row(2u);
  if (!bad) {
    const uint32_t Pq = at.P;
    const bool no_delta = (stages & kStageNoDelta) != 0u, no_zz = (stages & kStageNoZigzag) != 0u;
    const uint32_t last_word = clen / 4u - 1u;
    uint32_t erun = carry, unpacked = 0;
    bool xbad = false;
    for (uint32_t it = 0; it < niter && !xbad; it++) {
      const uint32_t x0 = 256u * it + 8u * lane;
      const uint32_t nv = x0 < W ? min(8u, W - x0) : 0u;
      // own pixels' mask byte (pixels past W count as zero samples) and the
      // compacted index of the first; the step ends at the next word group
      const uint32_t X = nv ? mw[x0 >> 5] : 0xffffffffu;
      const uint32_t nzm = ~(X >> (x0 & 31u)) & ((1u << nv) - 1u);
      const uint32_t kk = nv ? wbase[x0 >> 5] + __popc(~X & ((1u << (x0 & 31u)) - 1u)) : n;
      const uint32_t kend = 8u * it + 8u < nw ? wbase[8u * it + 8u] : n;
      while (unpacked < kend) {  // two blocks: lane l the values 8l .. 8l+7 of their 256
        const uint32_t blk = (unpacked >> 7) + (lane >> 4), l16 = lane & 15u;
        const uint2 dsc = blk < nb ? desc[blk] : make_uint2(0u, 0u);
        const uint32_t b = dsc.y & 0xffu, e = (dsc.y >> 8) & 0xffu, hb = (dsc.y >> 16) & 0xffu;
        const uint32_t bm = b >= 32u ? 0xffffffffu : ((1u << b) - 1u);
        uint32_t v[8];
        if (__all_sync(0xffffffffu, b <= 8u)) {  // 8 values in 64 bits
          const uint32_t bit0 = 8u * l16 * b, sh = bit0 & 31u, w0 = dsc.x + (bit0 >> 5);
          const uint32_t W0 = chunk[min(w0, last_word)], W1 = chunk[min(w0 + 1u, last_word)],
                         W2 = chunk[min(w0 + 2u, last_word)];
          const uint32_t A = __funnelshift_r(W0, W1, sh), B = __funnelshift_r(W1, W2, sh);
          const uint32_t C = __funnelshift_rc(A, B, 4u * b);
          v[0] = A; v[1] = A >> b; v[2] = A >> (2u * b); v[3] = A >> (3u * b);
          v[4] = C; v[5] = C >> b; v[6] = C >> (2u * b); v[7] = C >> (3u * b);
        } else {  // some block is wider: 4 values in up to 128 bits, twice
#pragma unroll
          for (uint32_t h = 0; h < 2; h++) {
            const uint32_t bit0 = (8u * l16 + 4u * h) * b, sh = bit0 & 31u, w0 = dsc.x + (bit0 >> 5);
            const uint32_t W0 = chunk[min(w0, last_word)], W1 = chunk[min(w0 + 1u, last_word)],
                           W2 = chunk[min(w0 + 2u, last_word)];
            const uint32_t A = __funnelshift_r(W0, W1, sh), B = __funnelshift_r(W1, W2, sh);
            uint32_t* q = v + 4u * h;
            if (b <= 16u) {
              const unsigned long long Y = ((unsigned long long)B << 32) | A;
              q[0] = A; q[1] = __funnelshift_r(A, B, b); q[2] = __funnelshift_rc(A, B, 2u * b);
              q[3] = (uint32_t)(Y >> (3u * b));
            } else {
              const uint32_t W3 = chunk[min(w0 + 3u, last_word)], W4 = chunk[min(w0 + 4u, last_word)];
              const uint32_t C = __funnelshift_r(W2, W3, sh), D = __funnelshift_r(W3, W4, sh);
              q[0] = A; q[1] = __funnelshift_rc(A, B, b); q[2] = __funnelshift_rc(B, C, 2u * b - 32u);
              q[3] = 3u * b <= 64u ? __funnelshift_rc(B, C, 3u * b - 32u) : __funnelshift_rc(C, D, 3u * b - 64u);
            }
          }
        }
#pragma unroll
        for (int i = 0; i < 8; i++) v[i] &= bm;  // (b = 0: all zero)
        if (__any_sync(0xffffffffu, e)) {  // exceptions: positions (ascending, < m), high parts of hb bits
          const uint32_t m = dsc.y >> 24;
          uint4* pt = reinterpret_cast<uint4*>(patch) + 2u * lane;
          pt[0] = pt[1] = make_uint4(0u, 0u, 0u, 0u);
          __syncwarp();
          const uint32_t lw = dsc.x + ((m * b + 31u) >> 5);
          const uint8_t* pos = reinterpret_cast<const uint8_t*>(chunk + lw);
          const uint32_t hw = lw + ((e + 3u) >> 2);
          const uint32_t hmask = hb >= 32u ? 0xffffffffu : ((1u << hb) - 1u);
          for (uint32_t jx = l16; jx < e; jx += 16) {
            const uint32_t ps = pos[jx];
            if (ps >= m || (jx > 0 && ps <= pos[jx - 1])) {
              xbad = true;
            } else {
              const uint32_t bit = jx * hb, wi = hw + (bit >> 5);
              const uint32_t lo = chunk[min(wi, last_word)], hi = chunk[min(wi + 1u, last_word)];
              patch[128u * (lane >> 4) + ps] = (__funnelshift_r(lo, hi, bit & 31u) & hmask) << b;
            }
          }
          __syncwarp();
          const uint4 p0 = pt[0], p1 = pt[1];
          v[0] |= p0.x; v[1] |= p0.y; v[2] |= p0.z; v[3] |= p0.w;
          v[4] |= p1.x; v[5] |= p1.y; v[6] |= p1.z; v[7] |= p1.w;
        }
        if (!no_zz) {
#pragma unroll
          for (int i = 0; i < 8; i++) v[i] = unzigzag(v[i]);
        }
        if (!no_delta) {  // deltas to residuals: running sums from the last one (values past n follow it)
          uint32_t sum = v[0];
#pragma unroll
          for (int i = 1; i < 8; i++) sum += v[i];
          uint32_t tot;
          v[0] += erun + warp_excl_scan(sum, tot);
          erun += tot;
#pragma unroll
          for (int i = 1; i < 8; i++) v[i] += v[i - 1];
        }
        const uint32_t at = (unpacked + 8u * lane) & (kRing - 1u);
        uint4* rp = reinterpret_cast<uint4*>(ring) + (at >> 2);
        rp[0] = make_uint4(v[0], v[1], v[2], v[3]);
        rp[1] = make_uint4(v[4], v[5], v[6], v[7]);
        if (at == 0u) {  // again behind the end, for the 8 pixels of a lane that run past it
          rp[kRing / 4u] = rp[0];
          rp[kRing / 4u + 1u] = rp[1];
        }
        unpacked += 2u * kBlockN;
      }
      xbad = __any_sync(0xffffffffu, xbad);
      __syncwarp();
      if (xbad) break;
      uint32_t pv[8] = {0, 0, 0, 0, 0, 0, 0, 0};
      if (prow && nv) load8<true>(prow, S, x0, nv, vec_prev, pv);
      uint32_t out[8];
      const uint32_t* res = ring + (kk & (kRing - 1u));
#pragma unroll
      for (int i = 0; i < 8; i++) {
        const bool kept = (nzm >> i) & 1u;
        out[i] = kept ? *res * Pq + pv[i] : 0u;
        res += kept ? 1 : 0;
      }
      if (nv) {
        store8(orow, S, x0, nv, vec_out, out);
        if (srow) store8(srow, S, x0, nv, vec_out, out);
      }
      __syncwarp();
    }
    bad = xbad;
  }
  if (lane == 0 && bad && !late) atomicOr(sg.err, kErrCorrupt);
  __syncwarp();
  if (si.link & kLinkNext) {  // the same row of the next frame waits for this one
    __threadfence();
    __syncwarp();
    if (lane == 0 && (!STAGED || k + 1u != p.withhold)) atomicExch(p.done + k, 2u);
  }
}

// (at most 64 registers: 32 warps per SM)
template <int WPC, bool STAGED, bool LOCAL>
__global__ void __launch_bounds__(WPC * 32, 32 / WPC) k_decode(DecParams p) {
  extern __shared__ __align__(16) uint32_t smem[];
  const uint32_t lane = lane_id();
  const DecWarpLayout lay = dec_warp_layout(p.max_W);
  uint8_t* wb = reinterpret_cast<uint8_t*>(smem) + warp_id() * lay.bytes;
  uint32_t* ring = reinterpret_cast<uint32_t*>(wb + lay.ring);
  uint32_t* patch = reinterpret_cast<uint32_t*>(wb + lay.patch);
  uint2* desc = reinterpret_cast<uint2*>(wb + lay.desc);
  uint32_t* mw = reinterpret_cast<uint32_t*>(wb + lay.mw);
  uint32_t* wbase = reinterpret_cast<uint32_t*>(wb + lay.wbase);
  uint32_t* lits = reinterpret_cast<uint32_t*>(wb + lay.lits);
  chain_wait();
  chain_start();
  while (true) {
    uint32_t kb = 0;
    if (lane == 0) kb = atomicAdd(p.ticket, p.items_per_ticket);
    kb = __shfl_sync(0xffffffffu, kb, 0);
    if (kb >= p.n_items) break;
    const uint32_t kend = min(kb + p.items_per_ticket, p.n_items);
    for (uint32_t k = kb; k < kend; k++) {
      decode_item<STAGED, LOCAL>(p, k, ring, patch, desc, mw, wbase, lits);
    }
  }
}

size_t dec_smem_bytes_host(uint32_t W) { return dec_warp_layout(W).bytes; }

constexpr size_t kDecSmemAuto = 48 * 1024;  // per CTA when picking warps per CTA by itself
constexpr size_t kDecSmemMax = 227 * 1024;

template <int WPC>
static void (*rows_kernel(const DecParams& p))(DecParams) {
  if (p.local) return p.staged ? k_decode<WPC, true, true> : k_decode<WPC, false, true>;
  return p.staged ? k_decode<WPC, true, false> : k_decode<WPC, false, false>;
}

static void (*rows_kernel(const DecParams& p, uint32_t wpc))(DecParams) {
  return wpc == 8 ? rows_kernel<8>(p) : wpc == 4 ? rows_kernel<4>(p) : wpc == 2 ? rows_kernel<2>(p) : rows_kernel<1>(p);
}

int decode_rows_launch(const DecParams& p, RowsLaunch* out) {
  const DecWarpLayout L = dec_warp_layout(p.max_W);
  if ((L.ring | L.patch | L.desc | L.mw | L.wbase | L.lits | L.bytes) & 15u) return (int)cudaErrorInvalidValue;  // 16-byte aligned regions
  uint32_t wpc = p.wpc;
  if ((wpc != 1 && wpc != 2 && wpc != 4 && wpc != 8) || wpc * L.bytes > kDecSmemMax) wpc = 0;
  if (!wpc) wpc = 4 * L.bytes <= kDecSmemAuto ? 4u : (2 * L.bytes <= kDecSmemAuto ? 2u : 1u);
  const size_t smem = (size_t)wpc * L.bytes;
  int dev = 0, sms = 0, per_sm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) {
    void (*f)(DecParams) = rows_kernel(p, wpc);
    // (the limit is the kernel's, shared by all threads: always the same one,
    // or a call of narrower rows takes it from another thread's launch)
    e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDecSmemMax);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, f, (int)wpc * 32, smem);
  }
  if (e != cudaSuccess) return (int)e;
  uint32_t ctas = (uint32_t)max(per_sm, 1);
  if (p.ctas_per_sm) ctas = min(ctas, p.ctas_per_sm);
  const uint32_t ipt = p.items_per_ticket ? min(p.items_per_ticket, 64u) : kDecBatch;
  // enough warps to fill the GPU; warps beyond the work find the ticket spent
  const uint32_t want = ceil_div_u32(p.n_items, ipt * wpc);
  out->sms = (uint32_t)sms;
  out->wpc = wpc;
  out->ctas_per_sm = ctas;
  out->items_per_ticket = ipt;
  out->grid = max(1u, min(want, ctas * (uint32_t)sms));
  return 0;
}

int launch_decode(const DecParams& p0, void* stream, void* const* ev) {
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  RowsLaunch rl{};
  int rc = decode_rows_launch(p0, &rl);
  if (rc != 0) return rc;
  DecParams p = p0;
  p.items_per_ticket = rl.items_per_ticket;
  const size_t smem = (size_t)rl.wpc * dec_warp_layout(p.max_W).bytes;
  if (ev) record_event(ev[0], st);
  if (!p.local) k_dec_secs<<<p.n_chains, kSecThreads, 0, st>>>(p);
  rc = launch_zstd_decode(p, st);
  if (rc != 0) return rc;
  cudaError_t e = cudaSuccess;
  if (!p.local) e = launch_chained(k_dec_masks, 4u * rl.sms, kMaskThreads, 0, st, p);
  if (e == cudaSuccess) e = launch_chained(rows_kernel(p, rl.wpc), rl.grid, rl.wpc * 32u, smem, st, p);
  if (!p.local && e == cudaSuccess) e = launch_chained(k_dec_sums, 4u * rl.sms, kSumThreads, 0, st, p);
  if (e != cudaSuccess) return (int)e;
  if (ev) record_event(ev[1], st);
  return (int)cudaGetLastError();
}

}  // namespace jiffy
