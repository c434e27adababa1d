// GB300 (sm_103a) kernels of the device-resident decode path.
//
// decode_kernel — one persistent launch decodes a list of segments (paper
// §3.3 full pipeline; §4 range decode; §5 chunked range decode). Each warp
// repeatedly takes the next work item from a global counter; the list is in
// level order, so every segment a warp waits for was taken earlier by a warp
// that is running (no deadlock, every source segment has a lower dependency level). Per segment (details at
// decode_segment):
//   1. rANS over the three command classes (the format's rANS coding): the 32 lanes run
//      the 32 interleaved states; each step's renormalisation words are handed
//      out in ascending lane order with a ballot + popc, from a shared-memory
//      ring that cp.async keeps filled ahead of the reader.
//   2. command parse: 32 commands at a time, positions from warp scans, every
//      command rule checked, source segments checked (level below
//      ours, present in the view).
//   3. rANS over the literal class, each literal stored straight to its
//      output position.
//   4. bounded waits on the ready flags of source segments, then match copies
//      in hazard-free rounds spread over the lanes.
//   5. publish: the warp synchronises (which orders every lane's output
//      stores before what lane 0 does next), then lane 0 stores the level and
//      epoch into the segment's flag with release semantics, a release that
//      covers the other lanes' stores through that ordering.
// staged_kernel — the same for short lists, where latency counts: a team of
// warps per segment, built in shared memory.
// batch_kernel — whole archives per CTA, or two small ones.
// Errors latch the first code into a device word; waits give up at a time
// limit (globaltimer) or as soon as another warp has latched an error.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstring>
#include <mutex>
#include <vector>

#include "kernels.h"

namespace aceapex {

namespace {

constexpr uint32_t kFull = 0xFFFFFFFFu;

__device__ __forceinline__ uint64_t ld_acquire(const uint64_t *p) {
  uint64_t v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void st_release(uint64_t *p, uint64_t v) {
  asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// the same within the CTA, on a word in shared memory
__device__ __forceinline__ uint32_t ld_acquire_cta(const uint32_t *p) {
  uint32_t v;
  asm volatile("ld.acquire.cta.shared.u32 %0, [%1];" : "=r"(v) : "r"((uint32_t)__cvta_generic_to_shared(p)) : "memory");
  return v;
}
__device__ __forceinline__ uint32_t ld_acquire_cta8(const uint8_t *p) {
  uint32_t v;
  asm volatile("ld.acquire.cta.shared.u8 %0, [%1];" : "=r"(v) : "r"((uint32_t)__cvta_generic_to_shared(p)) : "memory");
  return v;
}
__device__ __forceinline__ void st_release_cta8(uint8_t *p, uint32_t v) {
  asm volatile("st.release.cta.shared.u8 [%0], %1;" ::"r"((uint32_t)__cvta_generic_to_shared(p)), "r"(v) : "memory");
}
__device__ __forceinline__ void st_release_cta(uint32_t *p, uint32_t v) {
  asm volatile("st.release.cta.shared.u32 [%0], %1;" ::"r"((uint32_t)__cvta_generic_to_shared(p)), "r"(v) : "memory");
}

__device__ __forceinline__ uint32_t ld_relaxed(const uint32_t *p) {
  uint32_t v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ uint64_t now_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ uint32_t lanemask_lt() {
  uint32_t m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}

__device__ __forceinline__ void latch(uint32_t *err, uint32_t code) { atomicCAS(err, 0u, code); }

// address of absolute position p in view v; nullptr when p's page is absent
__device__ __forceinline__ uint8_t *at(const OutView &v, uint64_t p, uint32_t log2_S) {
  if (v.page) {
    uint32_t slot = v.page[p >> log2_S];
    if (slot == 0xFFFFFFFFu) return nullptr;
    return v.slot_base + ((uint64_t)slot << log2_S) + (p & ((uint64_t(1) << log2_S) - 1));
  }
  return v.base + ((p - v.origin) & v.mask);
}

__device__ __forceinline__ uint32_t smem_addr(const void *p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

// 16-byte asynchronous global -> shared copy (both addresses 16-byte aligned)
// with an L2 cache policy
__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, uint64_t pol) {
  asm volatile("cp.async.cg.shared.global.L2::cache_hint [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "l"(pol) : "memory");
}
// L2 policy for data read once (the payload): evicted first, so that the
// output, which matches read back, stays longer
__device__ __forceinline__ uint64_t policy_evict_first() {
  uint64_t pol;
  asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// inclusive warp scan of a 32-bit value
__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t v, int lane) {
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    uint32_t t = __shfl_up_sync(kFull, v, d);
    if (lane >= d) v += t;
  }
  return v;
}

// Wait until every lane with `need` sees *flag == epoch. False on timeout or
// when another warp has latched an error. Lane 0 reads the error word and
// the clock and decides for the warp (see take_item).
__device__ bool wait_flags(const uint64_t *flag, bool need, uint32_t epoch, uint64_t deadline, uint32_t *err,
                           int lane) {
  for (uint32_t spin = 0;; ++spin) {
    bool ok = !need || (uint32_t)ld_acquire(flag) == epoch;
    if (__all_sync(kFull, ok)) return true;
    uint32_t why = 0;
    if (lane == 0) why = ld_relaxed(err) != 0 ? 1u : now_ns() > deadline ? 2u : 0u;
    why = __shfl_sync(kFull, why, 0);
    if (why) {
      if (why == 2 && lane == 0) latch(err, kErrTimeout);
      return false;
    }
    __nanosleep(spin < 8 ? 64 : spin < 32 ? 256 : 1024);
  }
}

// The warp's next work index (lane 0's atomic on counter) and whether the
// error word is set, both read by lane 0 and broadcast, so that every lane
// takes the same branch: lanes that read the error word themselves could see
// different values while another warp latches it, and a warp whose lanes part
// there would meet at different warp-synchronous calls.
__device__ __forceinline__ uint32_t take_item(uint32_t *counter, const uint32_t *err, int lane, bool &failed) {
  uint32_t idx = 0, e = 0;
  if (lane == 0) {
    idx = atomicAdd(counter, 1u);
    e = ld_relaxed(err);
  }
  idx = __shfl_sync(kFull, idx, 0);
  failed = __shfl_sync(kFull, e, 0) != 0;
  return idx;
}

// u16 little-endian at p (2-byte aligned)
__device__ __forceinline__ uint32_t ld16(const uint8_t *p) { return *reinterpret_cast<const uint16_t *>(p); }
__device__ __forceinline__ void st16(uint8_t *p, uint32_t v) { *reinterpret_cast<uint16_t *>(p) = (uint16_t)v; }

constexpr int kViewLinear = 0, kViewRing = 1, kViewPaged = 2;

// address of source position p in view v (its page is known to be present)
template <int kMode>
__device__ __forceinline__ const uint8_t *src_at(const OutView &v, uint64_t p, uint32_t log2_S) {
  if (kMode == kViewPaged) return at(v, p, log2_S);
  if (kMode == kViewRing) return v.base + ((p - v.origin) & v.mask);
  return v.base + (p - v.origin);
}

// r = bytes c .. c+15 of the 32 bytes X || Y (bytes past the end read as 0)
__device__ __forceinline__ void realign16(uint4 X, uint4 Y, uint32_t c, uint32_t r[4]) {
  const uint32_t w[12] = {X.x, X.y, X.z, X.w, Y.x, Y.y, Y.z, Y.w, 0u, 0u, 0u, 0u};
  const uint32_t k = c >> 2, sh = 8 * (c & 3);
  uint32_t s4[8], s2[6], s1[5];
#pragma unroll
  for (int j = 0; j < 8; ++j) s4[j] = (k & 4) ? w[j + 4] : w[j];
#pragma unroll
  for (int j = 0; j < 6; ++j) s2[j] = (k & 2) ? s4[j + 2] : s4[j];
#pragma unroll
  for (int j = 0; j < 5; ++j) s1[j] = (k & 1) ? s2[j + 1] : s2[j];
#pragma unroll
  for (int j = 0; j < 4; ++j) r[j] = __funnelshift_r(s1[j], s1[j + 1], sh);
}

// Bytes [o, o + n) of the 16-byte block at `to` (16-byte aligned), n < 16, from
// the block r.
__device__ __forceinline__ void store_piece(uint8_t *to, const uint32_t r[4], uint32_t o, uint32_t n) {
  // bytes [o, o + n) of the block as naturally aligned pieces of
  // 1, 2, 4 and 8 bytes (a scattered store costs the memory
  // pipeline one pass per line it touches, whatever its width)
  auto wd = [&](uint32_t i) { return i & 2 ? (i & 1 ? r[3] : r[2]) : (i & 1 ? r[1] : r[0]); };
  if (o == 0 || o + n == 16) {
    // the first or last block of a match: one end of the bytes is
    // an end of the block, and the pieces are the set bits of n,
    // rising in size from o when the bytes end at the block's end,
    // falling from 0 when they start at its start (four store
    // instructions per warp)
    const bool rise = o != 0;
    if (n & 8) *reinterpret_cast<uint2 *>(to + (rise ? 8 : 0)) = rise ? make_uint2(r[2], r[3]) : make_uint2(r[0], r[1]);
    if (n & 4) {
      const uint32_t a = rise ? o + (n & 3) : (n & 8);
      *reinterpret_cast<uint32_t *>(to + a) = wd(a >> 2);
    }
    if (n & 2) {
      const uint32_t a = rise ? o + (n & 1) : (n & 12);
      *reinterpret_cast<uint16_t *>(to + a) = (uint16_t)(wd(a >> 2) >> (8 * (a & 2)));
    }
    if (n & 1) {
      const uint32_t a = rise ? o : (n & 14);
      to[a] = (uint8_t)(wd(a >> 2) >> (8 * (a & 3)));
    }
  } else {
    // both ends inside the block (a match shorter than 16 bytes):
    // rising in size up to the first boundary that the next piece
    // would cross, then falling (eight store instructions)
    uint32_t a = o;
    const uint32_t e = o + n;
    if ((a & 1) && a < e) { to[a] = (uint8_t)(wd(a >> 2) >> (8 * (a & 3))); a += 1; }
    if ((a & 2) && a + 2 <= e) { *reinterpret_cast<uint16_t *>(to + a) = (uint16_t)(wd(a >> 2) >> (8 * (a & 2))); a += 2; }
    if ((a & 4) && a + 4 <= e) { *reinterpret_cast<uint32_t *>(to + a) = wd(a >> 2); a += 4; }
    if ((a & 8) && a + 8 <= e) { *reinterpret_cast<uint2 *>(to + a) = make_uint2(r[2], r[3]); a += 8; }
    if (a + 8 <= e) { *reinterpret_cast<uint2 *>(to + a) = (a & 8) ? make_uint2(r[2], r[3]) : make_uint2(r[0], r[1]); a += 8; }
    if (a + 4 <= e) { *reinterpret_cast<uint32_t *>(to + a) = wd(a >> 2); a += 4; }
    if (a + 2 <= e) { *reinterpret_cast<uint16_t *>(to + a) = (uint16_t)(wd(a >> 2) >> (8 * (a & 2))); a += 2; }
    if (a < e) to[a] = (uint8_t)(wd(a >> 2) >> (8 * (a & 3)));
  }
}

// Per-warp shared table of the matches copied in one round.
struct MatchTable {
  uint64_t src[32];
  uint64_t dst[32];   // absolute positions
  uint32_t len[32];   // match length
  uint32_t start[33]; // first 16-byte unit of each lane's match in the round; start[32] = round total
  uint32_t pad[3];    // keeps the size a multiple of 16
};

// 16- and 32-bit loads through 32-bit shared-window addresses (volatile:
// they must stay behind the cp.async waits that fill the word ring)
__device__ __forceinline__ uint32_t lds_u16(uint32_t a) {
  uint16_t v;
  asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ uint32_t lds_u32(uint32_t a) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ uint32_t lds_u8(uint32_t a) {
  uint32_t v;
  asm volatile("ld.shared.u8 %0, [%1];" : "=r"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ uint4 lds_v4(uint32_t a) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
  return v;
}
__device__ __forceinline__ void sts_u8(uint32_t a, uint32_t v) {
  asm volatile("st.shared.u8 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void sts_u16(uint32_t a, uint32_t v) {
  asm volatile("st.shared.u16 [%0], %1;" ::"r"(a), "h"((uint16_t)v) : "memory");
}

// The state after decoding the symbol of table entry e (sym | bias << 8 |
// (freq - 1) << 20): freq * (x >> 12) + bias. With q = freq - 1 and e >> 8 =
// q << 12 | bias this is q * ((x >> 12) - 4096) + (x >> 12) + (e >> 8): no
// mask for the bias and no increment of q, one instruction less per step of
// an issue-bound loop (1 GiB FASTQ 1.511 -> 1.495 ms).
__device__ __forceinline__ uint32_t rans_next(uint32_t x, uint32_t e) {
  const uint32_t xh = x >> kScaleBits;
  return (e >> 20) * (xh - kScale) + (xh + (e >> 8));
}

// The command staging area of a warp: shared memory (kShared, read and
// written through its shared-window address), or a generic pointer to shared
// memory or to the warp's global slot for segments whose command streams do
// not fit. Byte offsets; the area is 4-byte aligned.
template <bool kShared>
struct Stage {
  uint8_t *p;
  uint32_t s;  // shared-window address of p (kShared)
  __device__ __forceinline__ uint32_t u16(uint32_t o) const {
    if (kShared) return lds_u16(s + o);
    return *reinterpret_cast<const uint16_t *>(p + o);
  }
  __device__ __forceinline__ uint32_t u32(uint32_t o) const {
    if (kShared) return lds_u32(s + o);
    return *reinterpret_cast<const uint32_t *>(p + o);
  }
  __device__ __forceinline__ void st8(uint32_t o, uint32_t v) const {
    if (kShared) asm volatile("st.shared.u8 [%0], %1;" ::"r"(s + o), "r"(v) : "memory");
    else p[o] = (uint8_t)v;
  }
  __device__ __forceinline__ void st16(uint32_t o, uint32_t v) const {
    if (kShared) asm volatile("st.shared.u16 [%0], %1;" ::"r"(s + o), "h"((uint16_t)v) : "memory");
    else *reinterpret_cast<uint16_t *>(p + o) = (uint16_t)v;
  }
  __device__ __forceinline__ void st32(uint32_t o, uint32_t v) const {
    if (kShared) asm volatile("st.shared.u32 [%0], %1;" ::"r"(s + o), "r"(v) : "memory");
    else *reinterpret_cast<uint32_t *>(p + o) = v;
  }
  // W-byte little-endian value at offset o (1 <= W <= 8); reads only the
  // aligned 4-byte words that hold bytes of [o, o + W), so never past the
  // word that holds byte o + W - 1
  __device__ __forceinline__ uint64_t le(uint32_t o, uint32_t W) const {
    const uint32_t a = o & ~3u, sh = 8 * (o & 3u), span = (o & 3u) + W;
    const uint32_t w0 = u32(a);
    const uint32_t w1 = span > 4 ? u32(a + 4) : 0u;
    uint64_t v = __funnelshift_r(w0, w1, sh);
    if (W > 4) {
      const uint32_t w2 = span > 8 ? u32(a + 8) : 0u;
      v |= (uint64_t)__funnelshift_r(w1, w2, sh) << 32;
    }
    return W >= 8 ? v : v & ((uint64_t(1) << (8 * W)) - 1);
  }
};

#ifdef ACEAPEX_PHASE_CLOCKS
// Warp-cycle counters per phase (instrumented build only): 0 command-class
// rANS, 1 command parse, 2 literal rANS and placement, 3 source checks of
// the match chunks,
// 4 match copies, 5 the rest of the work loop; then event counts: 6 match
// chunks, 7 copy rounds, 8 copy units, 9 segments, 10 chunks whose source
// flags were not all set at the first reading; 11 warp cycles spent waiting
// for those flags (counted apart from phase 3, the chunks' source checks).
__device__ unsigned long long g_phase_cycles[16];
#define PHASE_COUNT(i, v) \
  do {                    \
    if (lane == 0) ph[i] += (v); \
  } while (0)
#define PHASE_MARK(i)                    \
  do {                                   \
    if (lane == 0) {                     \
      const uint64_t t_ = clock64();     \
      ph[i] += t_ - ph_t;                \
      ph_t = t_;                         \
    }                                    \
  } while (0)
#else
#define PHASE_MARK(i) \
  do {                \
  } while (0)
#define PHASE_COUNT(i, v) \
  do {                    \
  } while (0)
#endif

// Decode one segment into view V and publish its ready flag.
//
// lut: the 4 x 4096-entry decode table (kSmemLut: at shared-window address
// lut_s; otherwise global lut). st: the warp's command staging area. mt: the
// warp's shared match table; ring_s: shared-window address of the warp's
// 1,280-byte renormalisation-word ring (16-byte aligned).
//
// Phases: (1) rANS over the three command classes into the staging area;
// (2) parse, scans and the checks of every command, rewriting each command's
// literal-run length in place as the inclusive literal prefix (the run's end
// in literal numbering); (3) rANS over the literal class, each literal stored
// straight to its output position: the literals of one step are consecutive
// in literal numbering, so a warp-uniform cursor walks the command boundaries
// that fall inside the step and moves the per-lane output pointers of the
// lanes past each boundary by that command's match length; (4) per 32-command
// chunk: source levels (and pages) checked, bounded waits on the source
// segments' flags, then match copies in rounds: a round copies every pending
// match whose source does not overlap the output of an earlier pending match,
// the bytes of the round spread over all lanes; (5) publish.
//
// entropy_phases is (1) to (3): false when the segment is corrupt (or its
// page absent); the command records are then in the stage.
// kStaged: the literals are only decoded, literal k to byte tot_m + k of the
// segment's copy in shared memory at out_s (tot_m: the segment's match bytes;
// place_literals moves them from there), and *progress counts the literals
// decoded so far. after_parse(ok, tot_m) is called between (2) and (3).
template <bool kSmemLut, int kMode, bool kSharedStage, bool kStaged, class AfterParse>
__device__ __forceinline__ bool entropy_phases(const DevArchive &A, const OutView &V, uint32_t seg,
                                               const uint32_t *lut, uint32_t lut_s, const Stage<kSharedStage> st,
                                               uint32_t ring_s, uint32_t out_s, uint32_t *progress,
                                               AfterParse after_parse, int lane, const SegRec &d, uint64_t *ph,
                                               uint64_t &ph_t) {
  (void)ph;
  (void)ph_t;
  const uint32_t log2_S = A.log2_S;
  const uint64_t seg_start = (uint64_t)seg << log2_S;
  const uint64_t rem = A.n - seg_start;
  const uint32_t out_size = rem < (uint64_t(1) << log2_S) ? (uint32_t)rem : (1u << log2_S);
  const uint32_t nc = d.n_cmd, nl = d.n_lit, nw = d.n_words, W = A.W, mm = A.min_match;
  const uint32_t b1 = 2 * nc, b2 = 4 * nc, b3 = (4 + W) * nc, n_sym = b3 + nl;
  // the segment's own output is contiguous in every view
  uint8_t *const out = at(V, seg_start, log2_S);
  bool ok = out != nullptr;

  // ---------------------------------------------------------------- rANS
  const uint8_t *pl = A.payload + d.payload_off;
  uint32_t x = __ldg(reinterpret_cast<const uint32_t *>(pl) + lane);
  if (!__all_sync(kFull, x >= kRansL)) ok = false;
  // Renormalisation words go through a 512-word ring in shared memory, filled
  // by cp.async in blocks of 128 words two blocks ahead of the reader, so the
  // decode never waits on a global load between block boundaries. Block slot
  // 0 is also copied to the 256 bytes after the ring (lanes 16..31 make that
  // copy), so the words of the next four steps are always contiguous from
  // the read address wr: no step masks its address. A lane copies a 16-byte
  // chunk only if it starts before the segment's last word; the payload is
  // padded to 16 bytes, so no copy leaves the archive.
  const uint8_t *wsrc = pl + 128;
  const uint64_t pol = policy_evict_first();
  auto fetch = [&](uint32_t blk) {
    const uint32_t wi = blk * 128 + (uint32_t)(lane & 15) * 8;
    const uint32_t to = ring_s + (lane < 16 ? (blk & 3) * 256 : 1024u) + (lane & 15) * 16;
    if ((lane < 16 || (blk & 3) == 0) && wi < nw) cp_async16(to, wsrc + (size_t)wi * 2, pol);
    cp_async_commit();
  };
  fetch(0);
  fetch(1);
  fetch(2);
  fetch(3);
  cp_async_wait<2>();
  __syncwarp();
  // blk: the block being read; wr: shared address of the next word; bnd: end
  // of blk's slot (wr moves on into the next slot, or into the copy of slot
  // 0, which it leaves for slot 0 itself when blk advances)
  uint32_t blk = 0, wr = ring_s, bnd = ring_s + 256;
  const uint32_t lt = lanemask_lt();
  // after the step that consumed the last word of a block: reuse its slot
  auto advance = [&]() {
    if (wr >= bnd) {
      ++blk;
      bnd += 256;
      if (bnd > ring_s + 1024) {
        wr -= 1024;
        bnd -= 1024;
      }
      __syncwarp();
      fetch(blk + 3);
      cp_async_wait<2>();
      __syncwarp();
    }
  };
  // table entry of slot (class << 12 | x mod 4096)
  auto entry = [&](uint32_t idx) -> uint32_t {
    if (kSmemLut) return lds_u32(lut_s + 4 * idx);
    return __ldg(lut + idx);
  };
  // lanes whose state fell below 2^16 read the next words in ascending lane
  // order (every lane reads a ring word; only those lanes use it)
  auto renorm = [&](bool need) {
    const uint32_t m = __ballot_sync(kFull, need);
    const uint32_t w = lds_u16(wr + 2 * __popc(m & lt));
    if (need) x = __byte_perm(w, x, 0x5410);  // x << 16 | w
    wr += 2 * __popc(m);
  };
  // one interleaved step of the command classes: lane j decodes symbol q
  auto cmd_step = [&](uint32_t q) -> uint32_t {
    const bool active = q < n_sym;
    const uint32_t cls = (uint32_t)(q >= b1) + (uint32_t)(q >= b2) + (uint32_t)(q >= b3);
    uint32_t sym = 0;
    if (active) {
      const uint32_t e = entry((cls << kScaleBits) | (x & (kScale - 1)));
      sym = e & 0xFFu;
      x = rans_next(x, e);
    }
    renorm(active && x < kRansL);
    return sym;
  };

  // Stage layout: command c's literal-run length and match length less
  // min_match as one 32-bit record (u16, u16) at 4 c, which the parse
  // replaces by the run's end in literal numbering and the match bytes of
  // commands 0..c (both below 2^16: a segment holds at most 16 KiB); at 4 nc
  // a sentinel record whose run end (65535) lies beyond every literal; the
  // W-byte offsets from 4 nc + 4. Symbol q of the command classes goes to
  // stage_off(q).
  auto stage_off = [&](uint32_t q) -> uint32_t {
    if (q < b1) return 4 * (q >> 1) + (q & 1);
    if (q < b2) return 4 * ((q - b1) >> 1) + 2 + ((q - b1) & 1);
    return q + 4;
  };
  const uint32_t offs = b2 + 4;  // the offsets' start

  // (1) command classes; the step that crosses into the literals keeps its
  // literal symbol in `pend` until the command prefixes exist. Four steps take
  // at most 128 words, so after an advance() (blocks blk and blk + 1 complete,
  // wr inside blk's slot) four steps read only those two blocks.
  uint32_t t0 = 0, pend = 0;
  if (ok) {
    // four steps inside one class: the table row is known for all lanes
    auto cls_step = [&](uint32_t row) -> uint32_t {
      const uint32_t e = entry(row | (x & (kScale - 1)));
      x = rans_next(x, e);
      renorm(x < kRansL);
      return e & 0xFFu;
    };
    for (; t0 + 128 <= b3; t0 += 128) {
      const uint32_t c_lo = (uint32_t)(t0 >= b1) + (uint32_t)(t0 >= b2);
      const uint32_t c_hi = (uint32_t)(t0 + 127 >= b1) + (uint32_t)(t0 + 127 >= b2);
      if (c_lo == c_hi) {
        const uint32_t base = c_lo == 0 ? 0u : c_lo == 1 ? b1 : b2;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const uint32_t k = t0 + 32 * u + lane - base;  // symbol number within the class
          st.st8(c_lo == 2 ? b2 + 4 + k : 4 * (k >> 1) + 2 * c_lo + (k & 1), cls_step(c_lo << kScaleBits));
        }
      } else {
#pragma unroll
        for (int u = 0; u < 4; ++u) st.st8(stage_off(t0 + 32 * u + lane), cmd_step(t0 + 32 * u + lane));
      }
      advance();
    }
    for (; t0 < b3; t0 += 32) {
      const uint32_t q = t0 + lane;
      const uint32_t sym = cmd_step(q);
      if (q < b3) st.st8(stage_off(q), sym);
      else pend = sym;
      advance();
    }
  }
  __syncwarp();
  PHASE_MARK(0);

  // (2) parse, prefixes, checks
  uint32_t tot_l = 0, tot_m = 0;
  for (uint32_t c0 = 0; ok && c0 < nc; c0 += 32) {
    const uint32_t c = c0 + lane;
    const bool valid = c < nc;
    uint32_t ll = 0, ml = 0;
    uint64_t src = 0;
    if (valid) {
      const uint32_t rec = st.u32(4 * c);
      ll = rec & 0xFFFFu;
      ml = (rec >> 16) + mm;
      src = W == 4 ? (uint64_t)st.u32(offs + 4 * c) : st.le(offs + W * c, W);  // (4-byte offsets are aligned)
    }
    const uint32_t inc_l = warp_incl_scan(ll, lane), inc_m = warp_incl_scan(ml, lane);
    const uint32_t lit_end = tot_l + inc_l, msum = tot_m + inc_m - ml;
    const uint32_t cend = lit_end + msum + ml;  // end of the command in the segment
    const uint64_t dst = seg_start + lit_end + msum;
    const bool bad = valid && ((uint64_t)cend > out_size || lit_end > nl || src + ml > dst || src + ml < src ||
                               (A.D && dst - src > A.D));
    if (__any_sync(kFull, bad)) {
      ok = false;
      break;
    }
    if (valid) st.st32(4 * c, lit_end | (msum + ml) << 16);
    tot_l += __shfl_sync(kFull, inc_l, 31);
    tot_m += __shfl_sync(kFull, inc_m, 31);
  }
  if (ok && (tot_l + tot_m > out_size || out_size - tot_m != nl)) ok = false;
  if (ok && lane == 0) st.st32(4 * nc, 0xFFFFu);
  __syncwarp();
  PHASE_MARK(1);

  after_parse(ok, tot_m);

  // (3) literals. K0: literal number of lane 0 in the current step; E: end of
  // the literal run of command cu (literal number), the next boundary; Sc:
  // match bytes before the literals from the current boundary on (the
  // cumulative match length through command cu - 1); outK: the output
  // address of literal K0 before any match byte.
  if (kStaged && ok) {
    uint32_t to = out_s + tot_m + (uint32_t)lane;  // where the lane's next literal goes
    uint32_t n_done = 0;
    auto step = [&](bool active) -> uint32_t {
      // the words from wr on, one per lane: read before the chain needs them,
      // and handed out by a shuffle, which is shorter than an indexed read
      const uint32_t words = lds_u16(wr + 2 * lane);
      uint32_t e = 0;
      if (active) {
        e = entry((3u << kScaleBits) | (x & (kScale - 1)));
        x = rans_next(x, e);
      }
      const bool need = active && x < kRansL;
      const uint32_t m = __ballot_sync(kFull, need);
      const uint32_t w = __shfl_sync(kFull, words, __popc(m & lt));
      if (need) x = __byte_perm(w, x, 0x5410);  // x << 16 | w
      wr += 2 * __popc(m);
      return e;
    };
    auto tell = [&]() {
      __syncwarp();
      if (lane == 0) st_release_cta(progress, n_done);
    };
    if (b3 & 31u) {  // the crossing step, decoded in (1): its literals are lanes b3 mod 32 on
      const uint32_t l0 = b3 & 31u;
      if ((uint32_t)lane >= l0 && t0 - 32 + lane < n_sym) sts_u8(to - l0, pend);
      n_done = min(32 - l0, nl);
      to += 32 - l0;
    }
    for (; t0 + 128 <= n_sym; t0 += 128) {
#pragma unroll
      for (int u = 0; u < 4; ++u) sts_u8(to + 32 * u, step(true));
      to += 128;
      n_done += 128;
      advance();
      tell();
    }
    for (; t0 < n_sym; t0 += 32) {
      const bool active = t0 + lane < n_sym;
      const uint32_t e = step(active);
      if (active) sts_u8(to, e);
      to += 32;
      advance();
    }
    n_done = nl;
    tell();
  } else if (ok) {
    int K0 = (b3 & 31u) ? (int)(b3 & ~31u) - (int)b3 : 0;
    uint32_t cu = 0, rec = st.u32(0), Sc = 0;
    int E = (int)(rec & 0xFFFFu);
    uint8_t *outK = out + K0;
    // The lane's offset for this step: lanes at or after a run end that lies
    // inside [K0, K0 + 32) take that command's cumulative match length.
    auto bound = [&]() -> uint32_t {
      uint32_t sl = Sc;
      while (E - K0 < 32) {
        Sc = rec >> 16;
        if (lane >= E - K0) sl = Sc;
        rec = st.u32(4 * ++cu);
        E = (int)(rec & 0xFFFFu);
      }
      return sl + (uint32_t)lane;
    };
    auto lit_rans = [&]() -> uint32_t {
      const uint32_t e = entry((3u << kScaleBits) | (x & (kScale - 1)));
      x = rans_next(x, e);
      renorm(x < kRansL);
      return e;
    };
    if (b3 & 31u) {  // the crossing step, decoded in (1)
      const uint32_t o = bound();
      if (lane >= -K0 && t0 - 32 + lane < n_sym) outK[o] = (uint8_t)pend;
      outK += 32;
      K0 += 32;
    }
    for (; t0 + 128 <= n_sym; t0 += 128) {
      if (E - K0 >= 128) {  // no run ends inside these four steps
        uint8_t *p = outK + (Sc + (uint32_t)lane);
#pragma unroll
        for (int u = 0; u < 4; ++u) p[32 * u] = (uint8_t)lit_rans();
      } else {
        // the same walk as bound(), with the next run end kept relative to
        // the block (D) and each lane's offset (ol) changed only at run ends,
        // so that a step without one costs a compare and its store
        int D = E - K0;
        uint32_t ol = Sc + (uint32_t)lane;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          uint32_t o = ol;
          while (D < 32 * (u + 1)) {  // a run end inside step u, at lane D - 32 u
            Sc = rec >> 16;
            ol = Sc + (uint32_t)lane;
            if (lane >= D - 32 * u) o = ol;
            rec = st.u32(4 * ++cu);
            E = (int)(rec & 0xFFFFu);
            D = E - K0;
          }
          outK[32 * u + o] = (uint8_t)lit_rans();
        }
      }
      K0 += 128;
      outK += 128;
      advance();
    }
    for (; t0 + 32 <= n_sym; t0 += 32) {
      const uint32_t o = bound();
      outK[o] = (uint8_t)lit_rans();
      outK += 32;
      K0 += 32;
      advance();
    }
    if (t0 < n_sym) {
      const bool active = t0 + lane < n_sym;
      const uint32_t o = bound();
      uint32_t e = 0;
      if (active) {
        e = entry((3u << kScaleBits) | (x & (kScale - 1)));
        x = rans_next(x, e);
      }
      renorm(active && x < kRansL);
      if (active) outK[o] = (uint8_t)e;
      t0 += 32;
    }
  }
  // words consumed: the blocks before the current ring cycle plus the offset
  // of wr in the ring (and its copy of slot 0)
  const uint32_t wb = (blk & ~3u) * 256 + (wr - ring_s);
  if (!__all_sync(kFull, x == kRansL) || wb != 2 * nw) ok = false;
  __syncwarp();
  PHASE_MARK(2);
  return ok;
}

// Named barriers of a team. The forms without .aligned: the code before them
// branches by lane, and a warp that reached an aligned barrier in two parts
// would be counted twice.
__device__ __forceinline__ void named_sync(uint32_t id, uint32_t threads) {
  __syncwarp();
  asm volatile("barrier.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void named_arrive(uint32_t id, uint32_t threads) {
  __syncwarp();
  asm volatile("barrier.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// A team of warps that share one segment (staged_kernel): in the shared
// memory of the CTA.
constexpr uint32_t kTeamBytes = 416;  // a segment has at most 16384 / 5 commands: 410 groups of 8
struct TeamState {
  uint32_t seg;                // segment being decoded; kNoSeg ends the team
  uint32_t fail;               // set by the warp that finds the segment corrupt or a wait too long
  uint32_t lits;               // literals decoded so far
  uint32_t tot_m;              // match bytes of the segment
  uint8_t done[kTeamBytes];    // bit k of byte j: the match of command 8 j + k is in place
};
constexpr uint32_t kNoSeg = 0xFFFFFFFFu;
constexpr uint32_t kMaxTeams = 6;  // teams of a CTA: two named barriers each, of 1 .. 15
constexpr uint32_t kMaxTeam = 16;  // warps per team
constexpr uint32_t kStagedThreads = 768;
constexpr uint32_t kStagedSmem = 228352;  // dynamic shared memory of staged_kernel; its static part is below 4 KiB

// Waits for warps of the same team are not dependency waits, which L.wait_ns
// bounds: they end by themselves, and have a limit only so that no poll is
// endless.
__device__ __forceinline__ uint64_t own_wait_ns(const DecodeLaunch &L) {
  return max(L.wait_ns, (uint64_t)2000000000);
}

__device__ __forceinline__ uint32_t ld_vol(const uint32_t *p) { return *const_cast<const volatile uint32_t *>(p); }

// The literals of a segment that a team's first warp is decoding, moved from
// byte tot_m + k of the copy at out_s to their places, 128 at a time behind
// the decoder. A literal's place is never after where it was decoded to, and
// never after an earlier literal's source, so moving the blocks in order (each
// read before it is written) keeps what is still to be moved. False when the
// decoder gave up.
__device__ __forceinline__ bool place_literals(const Stage<true> st, const TeamState *ts, uint32_t out_s, uint32_t nl,
                                               uint64_t deadline, uint32_t *err, int lane) {
  const uint32_t tot_m = ts->tot_m, from = out_s + tot_m + (uint32_t)lane;
  // rec: the next run end (literal number, match bytes through its command);
  // ahead: the record after it, read early (the stage is readable past the
  // sentinel, and what follows it is never used)
  uint32_t cu = 0, rec = st.u32(0), ahead = st.u32(4), S = 0;
  for (uint32_t K = 0; K < nl && S != tot_m; K += 128) {
    const uint32_t want = min(K + 128, nl);
    for (uint32_t spin = 0; ; ++spin) {
      if (__all_sync(kFull, ld_acquire_cta(&ts->lits) >= want)) break;
      uint32_t why = 0;
      if (lane == 0 && (spin & 63) == 63) why = ld_vol(&ts->fail) ? 1u : now_ns() > deadline ? 2u : 0u;
      why = __shfl_sync(kFull, why, 0);
      if (why) {
        if (why == 2 && lane == 0) latch(err, kErrTimeout);
        return false;
      }
      __nanosleep(40);
    }
    uint32_t v[4], o[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      v[u] = K + 32 * u + lane < nl ? lds_u8(from + K + 32 * u) : 0u;
      o[u] = S;
    }
    __syncwarp();
    while ((rec & 0xFFFFu) < K + 128) {  // a run end inside the block (the sentinel's lies beyond every literal)
      const int D = (int)((rec & 0xFFFFu) - K);
      S = rec >> 16;
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (lane + 32 * u >= D) o[u] = S;
      ++cu;
      rec = ahead;
      ahead = st.u32(4 * cu + 4);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (K + 32 * u + lane < nl) sts_u8(out_s + K + 32 * u + lane + o[u], v[u]);
    __syncwarp();
  }
  return true;
}

// Phase (4) of a segment whose entropy phases are done, by one warp, in the
// view. False when a command is corrupt or a wait gave up.
template <int kMode, bool kSharedStage>
__device__ __forceinline__ bool match_phase(const DecodeLaunch &L, const DevArchive &A, const OutView &V, uint32_t seg,
                                            uint32_t epoch, const Stage<kSharedStage> st, MatchTable *mt, int lane,
                                            uint32_t nc, uint32_t my_level, uint64_t *ph, uint64_t &ph_t) {
  (void)ph;
  (void)ph_t;
  const uint32_t log2_S = A.log2_S, W = A.W;
  const uint64_t seg_start = (uint64_t)seg << log2_S;
  const uint32_t offs = 4 * nc + 4;
  uint8_t *const out = at(V, seg_start, log2_S);
  bool ok = true;
  // aligned 16-byte blocks of the view never straddle a segment (hence no ring
  // wrap or page boundary either)
  const bool vec =
      log2_S >= 4 && (kMode == kViewPaged  ? (reinterpret_cast<uintptr_t>(V.slot_base) & 15) == 0
                      : kMode == kViewRing ? ((reinterpret_cast<uintptr_t>(V.base) | V.origin) & 15) == 0
                                           : ((reinterpret_cast<uintptr_t>(V.base) - V.origin) & 15) == 0);
  const uint64_t deadline = now_ns() + L.wait_ns;
  uint32_t mbase = 0;  // match bytes before the chunk
  for (uint32_t c0 = 0; c0 < nc; c0 += 32) {
    const uint32_t c = c0 + lane;
    const bool valid = c < nc;
    uint32_t ml = 0, lend = 0, cum = 0;
    uint64_t src = 0;
    if (valid) {
      const uint32_t rec = st.u32(4 * c);
      cum = rec >> 16;
      lend = rec & 0xFFFFu;
      src = W == 4 ? (uint64_t)st.u32(offs + 4 * c) : st.le(offs + W * c, W);  // (4-byte offsets are aligned)
    }
    // match bytes of the commands before c (the previous lane's sum, or the
    // last sum of the previous chunk); this command's length is the difference
    const uint32_t up = __shfl_up_sync(kFull, cum, 1);
    const uint32_t before = lane ? up : mbase;
    if (valid) ml = cum - before;
    const uint64_t dst = valid ? seg_start + lend + before : ~uint64_t(0);
    mbase = __shfl_sync(kFull, cum, min(nc - 1 - c0, 31u));
    const uint64_t q0 = src >> log2_S, q1 = valid ? (src + ml - 1) >> log2_S : q0;
    // start moving the chunk's source bytes (the first and the last 128-byte
    // line of each match's) toward L2 while the checks and hazards run
    if (kMode != kViewPaged && valid) {
      asm volatile("prefetch.global.L2 [%0];" ::"l"(src_at<kMode>(V, src, log2_S)));
      if (((src ^ (src + ml - 1)) >> 7) != 0)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(src_at<kMode>(V, src + ml - 1, log2_S)));
    }
    const bool need0 = valid && q0 != seg;
    const bool need1 = valid && q1 != q0 && q1 != seg;
    // A source segment must have a lower level than ours (a wait on any other
    // could not end) and, in a paged view, be present. Its level is the high
    // half of its flag word, read in the same load as its epoch.
    bool bad = false;
    uint32_t f0 = epoch, f1 = epoch;
    if (need0) {
      const uint64_t f = ld_acquire(A.flags + q0);
      bad |= (uint32_t)(f >> 32) >= my_level;
      if (kMode == kViewPaged) bad |= V.page[q0] == 0xFFFFFFFFu;
      f0 = (uint32_t)f;
    }
    if (need1) {
      const uint64_t f = ld_acquire(A.flags + q1);
      bad |= (uint32_t)(f >> 32) >= my_level;
      if (kMode == kViewPaged) bad |= V.page[q1] == 0xFFFFFFFFu;
      f1 = (uint32_t)f;
    }
    // (the hazard ranges need no flag: they are found while the loads above
    // are in flight, and the loaded values are used only after them)
    // linear view: the table holds each match's source address
    mt->src[lane] = kMode == kViewLinear ? (uint64_t)reinterpret_cast<uintptr_t>(V.base + (src - V.origin)) : src;
    mt->dst[lane] = dst;
    __syncwarp();
    // The earlier matches of this chunk whose outputs overlap this match's
    // source: outputs are disjoint and ascending, so they are the lanes j with
    // dst_j < src + ml and dst_j + ml_j > src, a contiguous range [jlo, jhi]
    // found by two binary searches (offsets from the segment start; a source
    // that ends before the segment overlaps nothing); all lie below this lane
    // because src + ml <= dst.
    uint32_t hmask = 0;
    {
      const uint64_t se = src + ml;
      const uint32_t se_rel = valid && se > seg_start ? (uint32_t)(se - seg_start) : 0u;
      const uint32_t s_rel = valid && src > seg_start ? (uint32_t)(src - seg_start) : 0u;
      const uint32_t d_off = valid ? (uint32_t)(dst - seg_start) : 0xFFFFFFFFu;
      const uint32_t d_end = valid ? d_off + ml : 0xFFFFFFFFu;
      // (no search when every source ends before the chunk's first output)
      if (__any_sync(kFull, se_rel > __shfl_sync(kFull, d_off, 0))) {
        uint32_t jh = 0, jl = 0;
#pragma unroll
        for (int s = 16; s; s >>= 1) {
          if (__shfl_sync(kFull, d_off, jh + s) < se_rel) jh += s;
          if (__shfl_sync(kFull, d_end, jl + s) <= s_rel) jl += s;
        }
        const bool any_h = __shfl_sync(kFull, d_off, jh) < se_rel;  // some output starts before the source ends
        const bool any_l = __shfl_sync(kFull, d_end, jl) <= s_rel;  // some output ends before the source starts
        const uint32_t jlo = any_l ? jl + 1 : 0;
        if (any_h && jlo <= jh) hmask = ((2u << jh) - 1u) & ~((1u << jlo) - 1u);
      }
    }
    if (__any_sync(kFull, bad)) {
      ok = false;
      break;
    }
    if (!__all_sync(kFull, f0 == epoch && f1 == epoch)) {
      PHASE_COUNT(10, 1);
      PHASE_MARK(3);
      if (!wait_flags(A.flags + (need0 ? q0 : 0), need0, epoch, deadline, L.err, lane) ||
          !wait_flags(A.flags + (need1 ? q1 : 0), need1, epoch, deadline, L.err, lane)) {
        ok = false;
        break;
      }
      PHASE_MARK(11);
    }
    PHASE_MARK(3);
    PHASE_COUNT(6, 1);
    bool pending = valid;
    for (int round = 0;; ++round) {
      const uint32_t pm = __ballot_sync(kFull, pending);
      if (!pm) break;
      // a match waits while its source overlaps the output of an earlier
      // pending match
      const bool haz = (pm & hmask) != 0;
      const bool ready = pending && !haz;
      // Units: with vec, the 16-byte-aligned blocks of each match's output
      // (a block's source bytes span at most two aligned source blocks, read
      // with two 16-byte loads and realigned in registers; a whole block is
      // stored with one 16-byte store, a partial one byte by byte); otherwise
      // 16-byte pieces copied byte by byte. Lane j copies units j, j+32, ...
      // of the round. With vec an aligned source block never leaves its
      // segment, and a segment is only read after its flag was acquired.
      const uint32_t nu = !ready ? 0 : vec ? (((uint32_t)(dst - seg_start) & 15u) + ml + 15) >> 4 : (ml + 15) >> 4;
      const uint32_t incl = warp_incl_scan(nu, lane);
      const uint32_t total = __shfl_sync(kFull, incl, 31);
      PHASE_COUNT(7, 1);
      PHASE_COUNT(8, total);
      mt->start[lane] = incl - nu;
      mt->len[lane] = ml;
      if (lane == 31) mt->start[32] = incl;
      __syncwarp();
      for (uint32_t uu = lane; uu < total; uu += 32) {
        uint32_t m = 0;
#pragma unroll
        for (int s = 16; s; s >>= 1)
          if (mt->start[m + s] <= uu) m += s;
        if (vec) {
          const uint32_t doff = (uint32_t)(mt->dst[m] - seg_start);
          const uint32_t b16 = (doff & ~15u) + ((uu - mt->start[m]) << 4);
          const uint32_t a0 = max(doff, b16), a1 = min(doff + mt->len[m], b16 + 16);
          const uint32_t o = a0 - b16, n = a1 - a0;
          uint4 X = make_uint4(0, 0, 0, 0), Y = X;
          uint32_t cc;
          if (kMode == kViewLinear) {
            const uint8_t *pa = reinterpret_cast<const uint8_t *>(mt->src[m] + (a0 - doff));
            const uint32_t dl = (uint32_t)reinterpret_cast<uintptr_t>(pa) & 15u;
            const uint4 *pb = reinterpret_cast<const uint4 *>(pa - dl);
            if (dl >= o) {
              X = pb[0];
              if (dl + n > 16) Y = pb[1];
              cc = dl - o;
            } else {
              Y = pb[0];
              cc = 16 + dl - o;
            }
          } else {
            const uint64_t P = mt->src[m] + (a0 - doff);
            const uint8_t *pa = src_at<kMode>(V, P, log2_S);
            const uint32_t dl = (uint32_t)reinterpret_cast<uintptr_t>(pa) & 15u;
            if (dl >= o) {
              X = *reinterpret_cast<const uint4 *>(pa - dl);
              if (dl + n > 16) Y = *reinterpret_cast<const uint4 *>(src_at<kMode>(V, P + (16 - dl), log2_S));
              cc = dl - o;
            } else {
              Y = *reinterpret_cast<const uint4 *>(pa - dl);
              cc = 16 + dl - o;
            }
          }
          // cc < 16 in both cases (dl, o < 16): the mask tells the compiler,
          // which drops the selection level that a shift of 16 or more needs
          uint32_t r[4];
          realign16(X, Y, cc & 15u, r);
          uint8_t *to = out + b16;
          if (n == 16) {
            *reinterpret_cast<uint4 *>(to) = make_uint4(r[0], r[1], r[2], r[3]);
          } else {
            store_piece(to, r, o, n);
          }
        } else {
          const uint32_t o = (uu - mt->start[m]) << 4;
          const uint32_t n = min(16u, mt->len[m] - o);
          const uint64_t pp = mt->src[m] + o;
          uint8_t *to = out + (mt->dst[m] - seg_start) + o;
          uint8_t v[16];
          if (kMode == kViewLinear) {
#pragma unroll
            for (int j = 0; j < 16; ++j)
              if ((uint32_t)j < n) v[j] = reinterpret_cast<const uint8_t *>(pp)[j];
          } else
#pragma unroll
          for (int j = 0; j < 16; ++j)
            if ((uint32_t)j < n) v[j] = *src_at<kMode>(V, pp + j, log2_S);
#pragma unroll
          for (int j = 0; j < 16; ++j)
            if ((uint32_t)j < n) to[j] = v[j];
        }
      }
      __syncwarp();
      pending = pending && !ready;
    }
    PHASE_MARK(4);
  }
  return ok;
}

// A match being copied by a team: ml bytes from absolute position src to
// offset doff of the segment's copy.
struct TeamMatch {
  uint64_t src;
  uint32_t doff, ml;
  // the copy's aligned 16-byte blocks that it touches
  __device__ __forceinline__ uint32_t blocks() const { return ((doff & 15u) + ml + 15) >> 4; }
};

// Blocks k0, k0 + step, ... of match m, into the segment's copy at out_s. What
// lies in this segment is read from the copy, the rest from the view. vec: the
// view's 16-byte blocks are aligned in memory, and a block is built from the
// one or two aligned blocks (each in one segment) that hold its bytes; else
// the bytes are copied one by one.
template <int kMode>
__device__ __forceinline__ void copy_blocks(const DevArchive &A, const OutView &V, uint64_t seg_start, uint32_t out_s,
                                            const TeamMatch &m, uint32_t k0, uint32_t step, bool vec) {
  if (!vec) {
#pragma unroll 1
    for (uint32_t j = k0; j < m.ml; j += step)
      sts_u8(out_s + m.doff + j, m.src + j >= seg_start ? lds_u8(out_s + (uint32_t)(m.src + j - seg_start))
                                                       : (uint32_t)*src_at<kMode>(V, m.src + j, A.log2_S));
    return;
  }
  auto block = [&](uint64_t q) -> uint4 {
    if (q >= seg_start) return lds_v4(out_s + (uint32_t)(q - seg_start));
    const uint8_t *p = src_at<kMode>(V, q, A.log2_S);
    return kMode != kViewPaged || p ? *reinterpret_cast<const uint4 *>(p) : make_uint4(0, 0, 0, 0);
  };
  for (uint32_t k = k0; k < m.blocks(); k += step) {
    const uint32_t b16 = (m.doff & ~15u) + 16 * k;
    const uint32_t a0 = max(m.doff, b16), a1 = min(m.doff + m.ml, b16 + 16), o = a0 - b16, n = a1 - a0;
    const uint64_t P = m.src + (a0 - m.doff);
    const uint32_t dl = (uint32_t)P & 15u;
    uint4 X = make_uint4(0, 0, 0, 0), Y = X;
    const uint64_t q = P - dl;
    if (dl >= o) {
      X = block(q);
      if (dl + n > 16) Y = block(q + 16);
    } else {
      Y = block(q);
    }
    uint32_t r[4];
    realign16(X, Y, (dl - o) & 15u, r);
    uint8_t *to = reinterpret_cast<uint8_t *>(__cvta_shared_to_generic(out_s + b16));
    if (n == 16) *reinterpret_cast<uint4 *>(to) = make_uint4(r[0], r[1], r[2], r[3]);
    else store_piece(to, r, o, n);
  }
}

// Phase (4) by a team of T warps, in the segment's copy in shared memory at
// out_s. Commands go to the warps in batches of B (batch j to warp j mod T,
// each warp's in order), one to a lane; B is 8, 16 or 32, the least that takes
// all commands in one batch per warp. A match is copied, by four lanes, as soon as
// its source segments are published and the earlier matches of this segment
// that it reads are in place (ts->done): it waits for nothing else, so the
// length of this phase is the longest chain of such matches and not their
// number, and since every wait is for a lower command or a lower level, the
// waits end. Matches of more than 16 blocks are copied by the whole warp.
// False when a command is corrupt or a wait gave up.
template <int kMode>
__device__ __forceinline__ bool match_phase_team(const DecodeLaunch &L, const DevArchive &A, const OutView &V,
                                                 uint32_t seg, uint32_t epoch, const Stage<true> st, int lane,
                                                 uint32_t nc, uint32_t my_level, TeamState *ts, uint32_t out_s,
                                                 uint32_t first, uint32_t T) {
  const uint32_t log2_S = A.log2_S, W = A.W, offs = 4 * nc + 4;
  const uint64_t seg_start = (uint64_t)seg << log2_S;
  const bool vec =
      log2_S >= 4 && (kMode == kViewPaged  ? (reinterpret_cast<uintptr_t>(V.slot_base) & 15) == 0
                      : kMode == kViewRing ? ((reinterpret_cast<uintptr_t>(V.base) | V.origin) & 15) == 0
                                           : ((reinterpret_cast<uintptr_t>(V.base) - V.origin) & 15) == 0);
  const uint64_t begun = now_ns();
  const uint32_t B = 8 * T >= nc ? 8u : 16 * T >= nc ? 16u : 32u;
  for (uint32_t c0 = B * first; c0 < nc; c0 += B * T) {
    const uint32_t c = c0 + (uint32_t)lane;
    bool pending = (uint32_t)lane < B && c < nc, bad = false;
    uint32_t ml = 0, doff = 0;
    uint64_t src = 0;
    // the earlier commands [jlo, jhi] whose matches this one reads
    uint32_t jlo = 1, jhi = 0;
    const uint64_t *f0 = nullptr, *f1 = nullptr;  // flags of the source segments
    if (pending) {
      const uint32_t rec = st.u32(4 * c), before = c ? st.u32(4 * c - 4) >> 16 : 0u;
      src = W == 4 ? (uint64_t)st.u32(offs + 4 * c) : st.le(offs + W * c, W);
      ml = (rec >> 16) - before;
      doff = (rec & 0xFFFFu) + before;
      const uint64_t q0 = src >> log2_S, q1 = (src + ml - 1) >> log2_S;
      // (the parse has checked the command; these bounds keep every access below in place)
      bad = q1 >= A.n_seg || ml - 1 >= 1u << log2_S || doff + ml > 1u << log2_S;
      if (!bad && q0 != seg) f0 = A.flags + q0;
      if (!bad && q1 != q0 && q1 != seg) f1 = A.flags + q1;
      if (kMode == kViewPaged) bad |= (f0 && V.page[q0] == 0xFFFFFFFFu) || (f1 && V.page[q1] == 0xFFFFFFFFu);
      if (src + ml > seg_start) {
        // command j's match ends at offset C(j) = its record's two halves:
        // jlo is the first with C > src, jhi the first with C >= src + ml,
        // or the one before if that match starts after the source
        const uint32_t s_rel = src > seg_start ? (uint32_t)(src - seg_start) : 0u;
        const uint32_t e_rel = (uint32_t)(src + ml - seg_start);
        auto end_of = [&](uint32_t j) {
          const uint32_t r = st.u32(4 * j);
          return (r & 0xFFFFu) + (r >> 16);
        };
        uint32_t a = 0, b = 0;
        for (uint32_t s = 1u << (31 - __clz(c | 1u)); s; s >>= 1) {
          if (a + s <= c && end_of(a + s - 1) <= s_rel) a += s;
          if (b + s <= c && end_of(b + s - 1) < e_rel) b += s;
        }
        // (b <= c: this command's own match starts at or after src + ml)
        if (b == c || (st.u32(4 * b) & 0xFFFFu) + (b ? st.u32(4 * b - 4) >> 16 : 0u) >= e_rel) --b;
        if ((int)a <= (int)b) jlo = a, jhi = b;
      }
    }
    bool look = true;  // read the flags (an L2 round trip) only when nothing else is left to do
    for (uint32_t spin = 0;; ++spin) {
      if (look && pending) {
        // each flag is read until it has this call's epoch; a source segment
        // must have a lower level than ours (a wait on any other could not end)
        const uint64_t v0 = f0 ? ld_acquire(f0) : epoch, v1 = f1 ? ld_acquire(f1) : epoch;
        if (f0) bad |= (uint32_t)(v0 >> 32) >= my_level;
        if (f1) bad |= (uint32_t)(v1 >> 32) >= my_level;
        if ((uint32_t)v0 == epoch) f0 = nullptr;
        if ((uint32_t)v1 == epoch) f1 = nullptr;
      }
      bool ready = pending && !f0 && !f1;
      if (ready) {
        while (jlo <= jhi) {  // (in place ones are passed for good)
          const uint32_t m = ld_acquire_cta8(ts->done + (jlo >> 3));
          if (!(m >> (jlo & 7u) & 1u)) break;
          ++jlo;
        }
        if (jlo <= jhi) ready = false;
      }
      if (__any_sync(kFull, bad)) return false;
      const uint32_t rm = __ballot_sync(kFull, ready);
      if (rm) {
        const uint32_t big = __ballot_sync(kFull, ready && TeamMatch{src, doff, ml}.blocks() > 16);
        __syncwarp();  // (lanes read behind the acquires of the lanes that hold the matches)
        auto match_of = [&](int l) {
          return TeamMatch{__shfl_sync(kFull, src, l), __shfl_sync(kFull, doff, l), __shfl_sync(kFull, ml, l)};
        };
#pragma unroll 1
        for (int g = 0; g < (int)B; g += 8) {
          const uint32_t some = rm & ~big & (0xFFu << g);
          if (!some) continue;
          const int l = g + (lane >> 2);
          const TeamMatch m = match_of(l);
          if (some >> l & 1u) copy_blocks<kMode>(A, V, seg_start, out_s, m, (uint32_t)lane & 3u, 4, vec);
          __syncwarp();
        }
#pragma unroll 1
        for (uint32_t r = big; r; r &= r - 1)
          copy_blocks<kMode>(A, V, seg_start, out_s, match_of(__ffs((int)r) - 1), (uint32_t)lane, 32, vec);
        pending = pending && !ready;
        __syncwarp();
        // (the bits of lanes beyond the list are set too)
        const uint32_t left = __ballot_sync(kFull, pending);
        if ((uint32_t)lane < B / 8) st_release_cta8(ts->done + (c0 >> 3) + lane, ~(left >> (8 * lane)));
        if (!left) break;
        look = false;
        spin = 0;
      } else {
        if (!__any_sync(kFull, pending)) break;
        if (!look) {
          look = true;
          continue;
        }
        uint32_t why = 0;
        if ((spin & 7) == 7) {
          const uint64_t limit = __any_sync(kFull, pending && (f0 || f1)) ? L.wait_ns : own_wait_ns(L);
          if (lane == 0) why = ld_vol(&ts->fail) || ld_relaxed(L.err) ? 1u : now_ns() - begun > limit ? 2u : 0u;
        }
        why = __shfl_sync(kFull, why, 0);
        if (why) {
          if (why == 2 && lane == 0) latch(L.err, kErrTimeout);
          return false;
        }
        __nanosleep(spin < 64 ? 32 : 256);
      }
    }
  }
  return true;
}

// Phase (5), by one warp after every warp that copied matches of the segment:
// no fence per lane, since the barrier that the caller passed (the warp's, or
// the team's) orders every lane's stores before lane 0's release store, and
// release is cumulative.
__device__ __forceinline__ void publish(const DecodeLaunch &L, const DevArchive &A, uint32_t seg, uint32_t level,
                                        uint32_t epoch, bool ok, int lane) {
  if (!ok && lane == 0 && ld_relaxed(L.err) == 0) latch(L.err, kErrCorrupt);
  if (lane == 0 && ok && !(A.blocked && A.blocked[seg])) st_release(A.flags + seg, (uint64_t)level << 32 | epoch);
}

// Decode one segment: its command streams are staged in the warp's shared
// area when they fit (scap bytes), else in its global slot gstage. With
// kSharedStage every segment of the launch fits (the host checked the
// archive's largest command stream), and the stage is read and written with
// shared-memory instructions.
template <bool kSmemLut, int kMode, bool kSharedStage>
__device__ __forceinline__ void decode_segment(const DecodeLaunch &L, const DevArchive &A, const OutView &V,
                                               uint32_t seg, uint32_t epoch, const uint32_t *lut, uint8_t *sstage,
                                               uint32_t scap, uint8_t *gstage, MatchTable *mt, uint16_t *ring,
                                               int lane, uint64_t *ph, uint64_t &ph_t) {
  const SegRec d = A.dir[seg];
  const uint32_t b3 = (4 + A.W) * d.n_cmd;
  uint8_t *stage = kSharedStage || b3 + 4 <= scap ? sstage : gstage;
  const Stage<kSharedStage> st{stage, kSharedStage ? smem_addr(stage) : 0u};
  const bool ok = entropy_phases<kSmemLut, kMode, kSharedStage, false>(
                      A, V, seg, lut, kSmemLut ? smem_addr(lut) : 0u, st, smem_addr(ring), 0, nullptr,
                      [](bool, uint32_t) {}, lane, d, ph, ph_t) &&
                  match_phase<kMode, kSharedStage>(L, A, V, seg, epoch, st, mt, lane, d.n_cmd, d.level, ph, ph_t);
  PHASE_COUNT(9, 1);
  __syncwarp();
  publish(L, A, seg, d.level, epoch, ok, lane);
}

// Dynamic shared memory of a decode CTA: the decode table (64 KiB), then a
// 1,280-byte word ring per warp (the 1 KiB ring and a copy of its first 256
// bytes), then a match table and a command stage per warp.
struct WarpSmem {
  uint32_t *lut;
  uint16_t *ring;
  MatchTable *mt;
  uint8_t *stage;
};
__device__ __forceinline__ WarpSmem warp_smem(uint8_t *smem, int wid) {
  constexpr uint32_t nw = kDecodeThreads / 32;
  WarpSmem w;
  w.lut = reinterpret_cast<uint32_t *>(smem);
  uint8_t *rings = smem + kLutBytes;
  w.ring = reinterpret_cast<uint16_t *>(rings + wid * 1280);
  w.mt = reinterpret_cast<MatchTable *>(rings + nw * 1280) + wid;
  w.stage = rings + nw * (1280 + sizeof(MatchTable)) + (size_t)wid * kSmemStage;
  return w;
}

#ifdef ACEAPEX_PHASE_CLOCKS
#define PHASE_DECL        \
  uint64_t ph[12] = {};   \
  uint64_t ph_t = clock64()
#define PHASE_FLUSH()                                                                               \
  do {                                                                                              \
    if (lane == 0)                                                                                  \
      for (int i_ = 0; i_ < 12; ++i_) atomicAdd(&g_phase_cycles[i_], (unsigned long long)ph[i_]); \
  } while (0)
#else
#define PHASE_DECL            \
  uint64_t *ph = nullptr;     \
  uint64_t ph_t = 0
#define PHASE_FLUSH() \
  do {                \
  } while (0)
#endif

// Persistent decode of one archive: its decode table is copied to shared
// memory once per CTA, and every warp takes the next work item.
// kMode: how the view maps positions (linear output, ring, or page table).
template <int kMode, bool kSharedStage>
__global__ void __launch_bounds__(kDecodeThreads, 1) decode_kernel(DecodeLaunch L) {
  extern __shared__ __align__(16) uint8_t smem[];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const WarpSmem ws = warp_smem(smem, wid);
  {
    const uint4 *g = reinterpret_cast<const uint4 *>(L.arc0.lut);
    uint4 *s4 = reinterpret_cast<uint4 *>(ws.lut);
    for (uint32_t i = threadIdx.x; i < kLutBytes / 16; i += blockDim.x) s4[i] = g[i];
    __syncthreads();
  }
  const uint32_t gwarp = blockIdx.x * (blockDim.x >> 5) + wid;
  if (gwarp >= L.scratch_warps || (uint32_t)wid >= L.active_warps) return;
  uint8_t *gstage = L.scratch + (size_t)gwarp * kStageBytes;
  const uint32_t epoch = ld_relaxed(L.epoch);
  PHASE_DECL;
  for (;;) {
    bool failed;
    const uint32_t idx = take_item(L.counter, L.err, lane, failed);
    if (idx >= L.n_work) break;
    if (failed) continue;  // drain the list quickly after an error
    PHASE_MARK(5);
    decode_segment<true, kMode, kSharedStage>(L, L.arc0, L.view0, L.work[idx].seg, epoch, ws.lut, ws.stage,
                                              L.stage_cap, gstage, ws.mt, ws.ring, lane, ph, ph_t);
  }
  PHASE_FLUSH();
}

// Shared memory of a team in staged_kernel: the segment's copy (rounded up to
// 16 bytes), the word ring and the command stage.
struct TeamLayout {
  uint32_t copy, stage, bytes;  // sizes of the copy and the stage, and of all
};
__host__ __device__ inline TeamLayout team_layout(uint32_t log2_S, uint32_t max_stage) {
  TeamLayout y;
  y.copy = ((1u << log2_S) + 15u) & ~15u;
  y.stage = (max_stage + 4 + 15u) & ~15u;  // (4: the record read ahead past the sentinel)
  y.bytes = y.copy + 1280u + y.stage;
  return y;
}

// Decode of a short list, for latency: a team of T warps takes a segment and
// builds it in shared memory. Its first warp decodes the entropy classes, the
// second places the literals behind it, so that the chain of rANS steps
// carries nothing else; then all copy the matches; then they write the segment
// to the view and the first warp publishes it.
//
// What bounds such a decode is one segment's rANS chain and then one match
// phase per level of the wavefront. Each SM runs the match phase only a few
// times, so that its instructions are fetched on that path: the last warp of
// each team runs it once on a made-up segment while the entropy classes are
// being decoded.
//
// Measured against a warp per segment (decode_kernel): 2,000-read FASTQ, 42
// segments in 5 levels, 137.8 -> 78.8 us (39 us of it the chain of 425 steps,
// 32 us the levels); 500 segments in 8 levels 210 -> 137 us; 1,800 segments,
// two per team, 238 -> 199 us.
template <int kMode>
__global__ void __launch_bounds__(kStagedThreads, 1) staged_kernel(DecodeLaunch L, uint32_t teams, uint32_t T) {
  extern __shared__ __align__(16) uint8_t smem[];
  __shared__ TeamState s_team[kMaxTeams + 1];
  __shared__ __align__(16) uint32_t s_warm[16 + 32];  // the made-up segment: its stage, its copy
  const int lane = threadIdx.x & 31;
  const uint32_t wid = threadIdx.x >> 5;
  const DevArchive &A = L.arc0;
  if (L.stage_need && ld_relaxed(L.stage_need) > L.max_stage) return;  // (another kernel takes the list)
  {
    const uint4 *g = reinterpret_cast<const uint4 *>(L.arc0.lut);
    uint4 *s4 = reinterpret_cast<uint4 *>(smem);
    for (uint32_t i = threadIdx.x; i < kLutBytes / 16; i += blockDim.x) s4[i] = g[i];
    // the made-up segment's two commands: 40 literals and a match of 36 from
    // 1, then 4 literals and a match of 12 from 50 (inside the first match)
    uint8_t *w = reinterpret_cast<uint8_t *>(s_warm);
    if (threadIdx.x < 64) w[threadIdx.x] = 0;
    __syncthreads();
    if (threadIdx.x == 0) {
      s_warm[0] = 40u | 36u << 16;
      s_warm[1] = 44u | 48u << 16;
      s_warm[2] = 0xFFFFu;
      w[12] = 1;
      w[12 + A.W] = 50;
    }
    __syncthreads();
  }
  // the leaders are warps 0 .. teams - 1 (spread over the SM's four
  // schedulers), then come T - 1 helpers per team
  const bool leads = wid < teams;
  const uint32_t team = leads ? wid : (wid - teams) / (T - 1);
  const uint32_t rank = leads ? 0u : 1u + (wid - teams) % (T - 1);
  TeamState *const ts = s_team + team;
  const TeamLayout y = team_layout(A.log2_S, L.max_stage);
  uint8_t *const mine = smem + kLutBytes + team * y.bytes;
  const uint32_t out_s = smem_addr(mine), ring_s = smem_addr(mine + y.copy);
  const Stage<true> st{mine + y.copy + 1280, ring_s + 1280};
  const uint32_t *const lut = reinterpret_cast<const uint32_t *>(smem);
  const uint32_t epoch = ld_relaxed(L.epoch);
  auto team_sync = [&]() { named_sync(team + 1, 32 * T); };
  // (the made-up segment is segment 0, which must be long enough)
  bool warm = rank == T - 1 && A.log2_S >= 7 && A.n >= 128;
  PHASE_DECL;
  for (;;) {
    uint32_t seg = 0, nc = 2, level = 0;
    bool bad = false;
    if (!warm) {
      if (leads) {
        uint32_t take = kNoSeg;
        for (;;) {
          bool failed;
          const uint32_t idx = take_item(L.counter, L.err, lane, failed);
          if (idx >= L.n_work) break;
          if (failed) continue;  // drain the list quickly after an error
          take = L.work[idx].seg;
          break;
        }
        PHASE_MARK(5);
        for (uint32_t j = lane; j < kTeamBytes / 4; j += 32) reinterpret_cast<uint32_t *>(ts->done)[j] = 0;
        auto begin = [&](bool ok, uint32_t tot_m) {
          if (lane == 0) {
            ts->seg = take;
            ts->fail = !ok;
            ts->lits = 0;
            ts->tot_m = tot_m;
          }
          named_arrive(team + 8, 64);
        };
        if (take != kNoSeg) {
          const SegRec d = A.dir[take];
          const bool ok = entropy_phases<true, kMode, true, true>(A, L.view0, take, lut, smem_addr(lut), st, ring_s,
                                                                  out_s, &ts->lits, begin, lane, d, ph, ph_t);
          if (!ok && lane == 0) *const_cast<volatile uint32_t *>(&ts->fail) = 1;
        } else {
          begin(false, 0);
        }
      } else if (rank == 1) {
        named_sync(team + 8, 64);
        const uint32_t s = __shfl_sync(kFull, ts->seg, 0);
        if (s < A.n_seg && !__shfl_sync(kFull, ld_vol(&ts->fail), 0) &&
            !place_literals(st, ts, out_s, A.dir[s].n_lit, now_ns() + own_wait_ns(L), L.err, lane) && lane == 0)
          *const_cast<volatile uint32_t *>(&ts->fail) = 1;
      }
      team_sync();
      seg = __shfl_sync(kFull, ts->seg, 0);
      if (seg >= A.n_seg) break;  // kNoSeg
      const SegRec d = A.dir[seg];
      nc = d.n_cmd;
      level = d.level;
      bad = __shfl_sync(kFull, ld_vol(&ts->fail), 0) != 0;  // (another warp may be setting it)
    }
    const Stage<true> wst{reinterpret_cast<uint8_t *>(s_warm), smem_addr(s_warm)};
    if (!bad &&
        !match_phase_team<kMode>(L, A, L.view0, seg, epoch, warm ? wst : st, lane, nc, level,
                                 warm ? s_team + kMaxTeams : ts, warm ? smem_addr(s_warm + 16) : out_s,
                                 warm ? 0u : rank, T) &&
        !warm && lane == 0)
      *const_cast<volatile uint32_t *>(&ts->fail) = 1;
    if (warm) {
      warm = false;
      continue;
    }
    team_sync();
    if (!ld_vol(&ts->fail)) {
      // (no warp sets fail after the barrier)
      const uint64_t seg_start = (uint64_t)seg << A.log2_S, rem = A.n - seg_start;
      const uint32_t size = rem < (uint64_t(1) << A.log2_S) ? (uint32_t)rem : 1u << A.log2_S;
      uint8_t *const out = at(L.view0, seg_start, A.log2_S);
      const uint32_t whole = (reinterpret_cast<uintptr_t>(out) & 15) == 0 ? size & ~15u : 0u;
#pragma unroll 1
      for (uint32_t i = 16 * (rank * 32 + lane); i < whole; i += 512 * T)
        *reinterpret_cast<uint4 *>(out + i) = lds_v4(out_s + i);
#pragma unroll 1
      for (uint32_t i = whole + rank * 32 + lane; i < size; i += 32 * T) out[i] = (uint8_t)lds_u8(out_s + i);
    }
    team_sync();
    PHASE_COUNT(9, leads);
    if (leads) publish(L, A, seg, level, epoch, !ld_vol(&ts->fail), lane);
  }
  PHASE_FLUSH();
}

// Batch decode (see launch_batch): whole archives, the n_large largest one per
// CTA at a time, then the others, which have at most kPairWarps segments, two
// per CTA at a time: each pair of kPairWarps warps with a decode table of its
// own, since one archive would leave most of the CTA's 32 warps idle and two
// tables are what shared memory holds beside the warps' areas.
constexpr uint32_t kPairWarps = kBatchSmall;
static_assert(2 * kLutBytes + 2 * kPairWarps * (1280 + sizeof(MatchTable) + kSmemStage) <=
                  kLutBytes + (kDecodeThreads / 32) * (1280 + sizeof(MatchTable) + kSmemStage),
              "two tables and two groups of warps fit the launch");
template <bool kSharedStage>
__global__ void __launch_bounds__(kDecodeThreads, 1) batch_kernel(DecodeLaunch L, uint32_t n_arcs, uint32_t n_large) {
  extern __shared__ __align__(16) uint8_t smem[];
  __shared__ uint32_t s_arc[2], s_next[2];
  __shared__ DevArchive s_A[2];
  __shared__ OutView s_V[2];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const uint32_t gwarp = blockIdx.x * (blockDim.x >> 5) + wid;
  uint8_t *gstage = L.scratch + (size_t)gwarp * kStageBytes;
  const uint32_t epoch = ld_relaxed(L.epoch);
  PHASE_DECL;
  // g: which group (the CTA as one group in the first pass); members: its
  // threads, me: this thread's number among them
  uint32_t g = 0, members = blockDim.x, me = threadIdx.x, warps = L.active_warps;
  WarpSmem ws = warp_smem(smem, wid);
  bool pairs = false, claimed = false;
  auto sync = [&]() {
    if (pairs) named_sync(1 + g, members);
    else __syncthreads();
  };
  for (;;) {
    if (me == 0) {
      if (!claimed) s_arc[g] = atomicAdd(L.counter, 1u);
      s_next[g] = 0;
    }
    sync();
    const uint32_t a = s_arc[g];
    if (a >= n_large && !pairs) {
      // the second pass; group 0 goes on with the archive just claimed
      __syncthreads();
      if ((uint32_t)wid >= 2 * kPairWarps) break;
      pairs = true;
      g = (uint32_t)wid / kPairWarps;
      members = 32 * kPairWarps;
      me = threadIdx.x - g * members;
      warps = min(kPairWarps, L.active_warps);
      claimed = g == 0;
      uint8_t *mine = smem + 2 * kLutBytes + (size_t)wid * (1280 + sizeof(MatchTable) + kSmemStage);
      ws.lut = reinterpret_cast<uint32_t *>(smem + g * kLutBytes);
      ws.ring = reinterpret_cast<uint16_t *>(mine);
      ws.mt = reinterpret_cast<MatchTable *>(mine + 1280);
      ws.stage = mine + 1280 + sizeof(MatchTable);
      continue;
    }
    claimed = false;
    if (a >= n_arcs) break;
    if (me == 0) {
      s_A[g] = L.arcs[a];
      s_V[g] = L.views[a];
    }
    sync();
    const DevArchive &A = s_A[g];
    const uint4 *lut = reinterpret_cast<const uint4 *>(A.lut);
    uint4 *s4 = reinterpret_cast<uint4 *>(ws.lut);
    for (uint32_t i = me; i < kLutBytes / 16; i += members) s4[i] = lut[i];
    sync();
    for (; (me >> 5) < warps;) {
      bool failed;
      const uint32_t idx = take_item(&s_next[g], L.err, lane, failed);
      if (idx >= A.n_seg) break;
      if (failed) continue;
      PHASE_MARK(5);
      decode_segment<true, kViewLinear, kSharedStage>(L, A, s_V[g], A.order[idx].seg, epoch, ws.lut, ws.stage,
                                                      L.stage_cap, gstage, ws.mt, ws.ring, lane, ph, ph_t);
    }
    sync();  // the table is replaced only after every warp left this archive
  }
  PHASE_FLUSH();
}

// One warp per window of `per` segments: the window's segments in level
// order, index order within a level (one pass over the window per level, a
// ballot placing each pass's members), into out[s0 .. s1) of the window.
__global__ void window_order_kernel(const SegRec *dir, uint64_t n_seg, uint64_t per, uint32_t max_level,
                                    WorkItem *out) {
  const uint64_t w = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5;
  const uint32_t lane = threadIdx.x & 31;
  const uint64_t s0 = w * per;
  if (s0 >= n_seg) return;  // (the whole warp)
  const uint64_t s1 = min(n_seg, s0 + per);
  const uint32_t lt = lanemask_lt();
  uint64_t pos = s0;
  for (uint32_t l = 0; l <= max_level; ++l)
    for (uint64_t b = s0; b < s1; b += 32) {
      const uint64_t s = b + lane;
      const bool take = s < s1 && dir[s].level == l;
      const uint32_t m = __ballot_sync(kFull, take);
      if (take) out[pos + __popc(m & lt)] = WorkItem{0u, (uint32_t)s};
      pos += __popc(m);
    }
}

__global__ void init_flags_kernel(uint64_t *flags, const SegRec *dir, uint64_t n) {
  const uint64_t s = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  if (s < n) flags[s] = (uint64_t)dir[s].level << 32;
}

// A range decode's list by value: writes the work list and the page table and
// starts the call, in one launch (a copy from pinned memory and two kernels
// took 8 us before the decode could start).
__global__ void __launch_bounds__(1024) begin_list_kernel(const __grid_constant__ WorkList list, WorkItem *work,
                                                          uint32_t *page, uint32_t *global_epoch, uint32_t *epoch,
                                                          uint32_t *counter) {
  if (threadIdx.x == 0) {
    *epoch = atomicAdd(global_epoch, 1u) + 1u;
    *counter = 0;
  }
  if (threadIdx.x < list.n) {
    work[threadIdx.x] = WorkItem{0u, list.seg[threadIdx.x]};
    page[list.seg[threadIdx.x]] = threadIdx.x;
  }
}

__global__ void begin_kernel(uint32_t *global_epoch, uint32_t *epoch, uint32_t *counter) {
  *epoch = atomicAdd(global_epoch, 1u) + 1u;
  *counter = 0;
}

__global__ void clear_pages_kernel(uint32_t *page, const WorkItem *work, uint32_t n) {
  uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) page[work[i].seg] = 0xFFFFFFFFu;
}

__global__ void copy_view_kernel(OutView src, OutView dst, uint32_t log2_S, uint64_t lo, uint64_t n) {
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
    const uint8_t *p = at(src, lo + i, log2_S);
    uint8_t *q = at(dst, lo + i, log2_S);
    if (p && q) *q = *p;
  }
}

// Bytes [a, b) of dst (absent pages: zeros), by one thread: what of [lo, lo + n)
// falls into one of dst's aligned 16-byte blocks. One page lookup and one
// 16-byte store per block (built from two aligned source blocks) when the
// block's source lies in one segment of at least 16 bytes, aligned in memory.
__device__ __forceinline__ void gather_block(const OutView &v, uint32_t log2_S, uint64_t lo, uint8_t *dst, uint64_t a,
                                             uint64_t b) {
  if (b - a == 16 && log2_S >= 4 && v.page && (reinterpret_cast<uintptr_t>(v.slot_base) & 15) == 0 &&
      (lo + a) >> log2_S == (lo + b - 1) >> log2_S) {
    const uint8_t *p = at(v, lo + a, log2_S);
    uint32_t r[4] = {0, 0, 0, 0};
    if (p) {
      const uint32_t dl = (uint32_t)reinterpret_cast<uintptr_t>(p) & 15u;
      const uint4 *q = reinterpret_cast<const uint4 *>(p - dl);
      realign16(q[0], dl ? q[1] : make_uint4(0, 0, 0, 0), dl, r);
    }
    *reinterpret_cast<uint4 *>(dst + a) = make_uint4(r[0], r[1], r[2], r[3]);
    return;
  }
  for (uint64_t i = a; i < b; ++i) {
    const uint8_t *p = at(v, lo + i, log2_S);
    dst[i] = p ? *p : 0;
  }
}

// [lo, lo + n) of the view into dst (any alignment): a thread per aligned
// 16-byte block of dst (a byte per thread took 25 us for 9.4 MB).
__global__ void gather_kernel(OutView v, uint32_t log2_S, uint64_t lo, uint64_t n, uint8_t *dst) {
  const uint64_t off = reinterpret_cast<uintptr_t>(dst) & 15;  // dst's place in its first block
  const uint64_t blocks = (off + n + 15) >> 4;
  for (uint64_t k = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; k < blocks;
       k += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t a = k ? 16 * k - off : 0, b = min(n, 16 * (k + 1) - off);
    gather_block(v, log2_S, lo, dst, a, b);
  }
}

// gather_kernel for a short range, and the page table's entries cleared after
// it, by one CTA
__global__ void __launch_bounds__(1024) gather_clear_kernel(OutView v, uint32_t log2_S, uint64_t lo, uint64_t n,
                                                            uint8_t *dst, uint32_t *page, const WorkItem *work,
                                                            uint32_t n_work) {
  const uint64_t off = reinterpret_cast<uintptr_t>(dst) & 15, blocks = (off + n + 15) >> 4;
  for (uint64_t k = threadIdx.x; k < blocks; k += blockDim.x)
    gather_block(v, log2_S, lo, dst, k ? 16 * k - off : 0, min(n, 16 * (k + 1) - off));
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < n_work; i += blockDim.x) page[work[i].seg] = 0xFFFFFFFFu;
}

// bases [0, n) of a FASTA region whose first base sits at lo with line phase
// `phase` (its position within a line of L bases): base i is at
// lo + i + (phase + i) / L, the newline after every L bases skipped
// (with n_work, by one CTA, which then clears the page table's entries)
__global__ void gather_bases_kernel(OutView v, uint32_t log2_S, uint64_t lo, uint32_t phase, uint32_t L, uint64_t n,
                                    uint8_t *dst, uint32_t *page, const WorkItem *work, uint32_t n_work) {
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
    const uint8_t *p = at(v, lo + i + (phase + i) / L, log2_S);
    dst[i] = p ? *p : 0;
  }
  if (n_work) {
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < n_work; i += blockDim.x) page[work[i].seg] = 0xFFFFFFFFu;
  }
}

constexpr uint64_t kGatherChunk = 65536;

__global__ void multi_gather_kernel(const GatherJob *jobs, uint32_t n_jobs, uint64_t n_chunks) {
  for (uint64_t c = blockIdx.x; c < n_chunks; c += gridDim.x) {
    // the job holding chunk c: largest j with jobs[j].chunk0 <= c
    uint32_t lo = 0, hi = n_jobs;
    while (hi - lo > 1) {
      const uint32_t mid = (lo + hi) >> 1;
      if (jobs[mid].chunk0 <= c) lo = mid;
      else hi = mid;
    }
    const GatherJob &J = jobs[lo];
    const uint64_t a = (c - J.chunk0) * kGatherChunk, b = min(J.n, a + kGatherChunk);
    // as gather_kernel: a thread per aligned 16-byte block of dst
    const uint64_t off = reinterpret_cast<uintptr_t>(J.dst + a) & 15, blocks = (off + (b - a) + 15) >> 4;
    for (uint64_t k = threadIdx.x; k < blocks; k += blockDim.x)
      gather_block(J.v, J.log2_S, J.lo, J.dst, k ? a + 16 * k - off : a, min(b, a + 16 * (k + 1) - off));
  }
}

__global__ void set_pages_kernel(uint32_t *page, const WorkItem *work, uint32_t n) {
  uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) page[work[i].seg] = i;
}

// -------------------------------------------------------- device closures
// Members are only read from list slots that an earlier launch has filled:
// found[l] counts what expanding level l added, found[top + 1] the seeds, so
// the members before level l's launch are the sum over the levels above l, all
// of them words that no warp of that launch writes. (One counter for all
// levels would rise while its launch still runs, and before the slots behind
// it are written.)
__device__ __forceinline__ uint32_t closure_settled(const ClosureDev &C, uint32_t level, uint32_t top, int lane) {
  uint32_t n = 0;
  for (uint32_t l = level + 1 + lane; l <= top + 1; l += 32) n += C.found[l];
  return __reduce_add_sync(kFull, n);
}

__global__ void closure_seed_kernel(ClosureDev C, uint32_t s_lo, uint32_t n, uint32_t top, uint32_t gen) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    C.mark[s_lo + i] = gen;
    C.list[i] = s_lo + i;
  }
  if (blockIdx.x == 0)
    for (uint32_t l = threadIdx.x; l <= top + 1; l += blockDim.x) C.found[l] = l == top + 1 ? n : 0u;
}

// One warp per member of the given level (grid-stride over the list); its
// lanes walk the member's dependency list. A dependency joins the closure
// when this warp is the first to tag it with gen; the warp reserves the list
// slots of its new members with one atomic. Members added here have lower
// levels, so the list that this level needs is complete before its launch.
__global__ void closure_expand_kernel(ClosureDev C, uint32_t level, uint32_t top, uint32_t gen) {
  const int lane = threadIdx.x & 31;
  const uint32_t warps = gridDim.x * (blockDim.x >> 5);
  const uint32_t n = closure_settled(C, level, top, lane);
  for (uint32_t i = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); i < n; i += warps) {
    const uint32_t s = C.list[i];
    if (s >= C.n_seg) {  // (a slot that nobody wrote: nothing is read through it)
      if (lane == 0) latch(C.err, kErrCorrupt);
      continue;
    }
    if (C.dir[s].level != level) continue;
    const uint64_t b = C.dep_ptr[s], e = C.dep_ptr[s + 1];
    for (uint64_t k0 = b; k0 < e; k0 += 32) {
      const uint64_t k = k0 + lane;
      uint32_t d = 0;
      bool fresh = false;
      if (k < e) {
        d = C.deps[k];
        fresh = atomicExch(C.mark + d, gen) != gen;
      }
      const uint32_t m = __ballot_sync(kFull, fresh);
      if (!m) continue;
      uint32_t base = 0;
      if (lane == 0) base = n + atomicAdd(C.found + level, (uint32_t)__popc(m));
      base = __shfl_sync(kFull, base, 0);
      if (fresh) C.list[base + __popc(m & lanemask_lt())] = d;
    }
  }
}

// one CTA: counting sort of the members by level (a level is one byte)
__global__ void __launch_bounds__(1024) closure_order_kernel(ClosureDev C, uint32_t top, WorkItem *work,
                                                             uint32_t *page, uint32_t *n_out) {
  __shared__ uint32_t off[kClosureLevels];
  const uint32_t n = closure_settled(C, 0, top, threadIdx.x & 31);
  for (uint32_t l = threadIdx.x; l < kClosureLevels; l += blockDim.x) off[l] = 0;
  __syncthreads();
  auto level_of = [&](uint32_t s) { return min((uint32_t)C.dir[s].level, kClosureLevels - 1); };
  for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) {
    const uint32_t s = C.list[i];
    if (s < C.n_seg) atomicAdd(&off[level_of(s)], 1u);
    else latch(C.err, kErrCorrupt);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t run = 0;
    for (uint32_t l = 0; l < kClosureLevels; ++l) {
      const uint32_t c = off[l];
      off[l] = run;
      run += c;
    }
    *n_out = run;
  }
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) {
    const uint32_t s = C.list[i];
    if (s >= C.n_seg) continue;
    const uint32_t pos = atomicAdd(&off[level_of(s)], 1u);
    work[pos] = WorkItem{0u, s};
    page[s] = pos;
  }
}

// ------------------------------------------------------------------- CRC-32
// Standard CRC-32 (reflected polynomial 0xEDB88320, init and xorout ~0).
// A register r advanced over a message M from r0 is shift(r0, |M|) ^ raw(M),
// where raw is the register from r0 = 0 and shift(r, n) multiplies r by
// x^(8n) mod P (n zero bytes). So raw(A||B) = shift(raw(A), |B|) ^ raw(B),
// and crc(M) = raw(M) ^ shift(~0, |M|) ^ ~0. Everything is GF(2)-linear in
// the bytes, which the kernels below use to hash pieces in any order.
//
// Table words (g_crc_tabs, filled once per device from the host):
//   [0, 4096)                slice tables T_k[b] = raw(b followed by k zero
//                            bytes), k = 0..15 (T_0 is the usual byte table)
//   4096 + 1024 k + 256 i    byte tables of shift by 2^k bytes, k = 0..47:
//                            entry v = shift(v << 8i, 2^k)
constexpr int kCrcOps = 48;
constexpr int kCrcTabWords = 4096 + kCrcOps * 1024;
constexpr int kCrcSmemOps = 10;  // shifts by 2^0 .. 2^9 bytes kept in shared memory
constexpr int kCrcSmemWords = 4096 + kCrcSmemOps * 1024;
constexpr int kCrcThreads = 512;
__device__ uint32_t g_crc_tabs[kCrcTabWords];

__device__ __forceinline__ uint32_t crc_op(const uint32_t *t, uint32_t r) {
  return t[r & 0xFFu] ^ t[256 + ((r >> 8) & 0xFFu)] ^ t[512 + ((r >> 16) & 0xFFu)] ^ t[768 + (r >> 24)];
}

// shift(r, n) with the byte tables of 2^k bytes at ops + 1024 k
__device__ __forceinline__ uint32_t crc_shift(const uint32_t *ops, uint32_t r, uint64_t n) {
  for (int k = 0; n; ++k, n >>= 1)
    if (n & 1) r = crc_op(ops + 1024 * k, r);
  return r;
}

// raw CRC of 16 bytes held little-endian in w
__device__ __forceinline__ uint32_t crc_raw16(const uint32_t *T, uint4 w) {
  const uint32_t v[4] = {w.x, w.y, w.z, w.w};
  uint32_t r = 0;
#pragma unroll
  for (int m = 0; m < 16; ++m) r ^= T[256 * (15 - m) + ((v[m >> 2] >> (8 * (m & 3))) & 0xFFu)];
  return r;
}

// CRC-32 of [lo, hi) of the ring view, written to *out by the CTA that
// finishes last. The window is read in the parts of it that lie in one aligned
// piece of 2^log2_P bytes each (crc_piece says how large), a warp per piece,
// persistent grid: in rows of 512 bytes, lane j taking the
// 16 bytes at 512 i + 16 j of row i (coalesced), whose 16-byte pieces it folds
// Horner-style with a shift of 512 bytes between rows; bytes after the last
// full row are folded per lane. Each lane then shifts its register past the
// bytes that follow its own last piece, the warp XORs the 32 registers, and
// lane 0 shifts the result past the bytes of the window after the piece: what
// all warps have XORed together is the window's raw CRC, so nothing has to be
// joined in order (a second kernel that joined 8,192 pieces of a window in one
// CTA took 31 us, beside 45 us of reading). sums: the register and the number
// of CTAs done, both zero between launches.
__global__ void __launch_bounds__(kCrcThreads, 3) window_crc_kernel(OutView v, uint32_t log2_P, uint64_t lo,
                                                                    uint64_t hi, uint32_t *sums, uint32_t *out) {
  __shared__ uint32_t tab[kCrcSmemWords];
  __shared__ uint32_t s_xor;
  if (threadIdx.x == 0) s_xor = 0;
  for (int i = threadIdx.x; i < kCrcSmemWords; i += blockDim.x) tab[i] = g_crc_tabs[i];
  __syncthreads();
  const uint32_t *ops = tab + 4096;
  const uint32_t *op512 = ops + 1024 * 9;
  const int lane = threadIdx.x & 31;
  const uint64_t P = uint64_t(1) << log2_P;
  const uint64_t first = lo >> log2_P, last = (hi - 1) >> log2_P;
  const uint64_t pieces = last - first + 1;
  const uint32_t *all_ops = g_crc_tabs + 4096;
  uint32_t sum = 0;
  for (uint64_t i = blockIdx.x * (uint64_t)(blockDim.x >> 5) + (threadIdx.x >> 5); i < pieces;
       i += (uint64_t)gridDim.x * (blockDim.x >> 5)) {
    const uint64_t s = first + i;
    const uint64_t a = (s << log2_P) > lo ? (s << log2_P) : lo;
    const uint64_t b = ((s << log2_P) + P) < hi ? ((s << log2_P) + P) : hi;
    const uint32_t len = (uint32_t)(b - a);
    const uint8_t *p = v.base + ((a - v.origin) & v.mask);
    // a piece with a full row has P >= 512; then it, and lo, start at a
    // multiple of 16 bytes of the ring (crc_piece), so p is 16-byte aligned
    const uint32_t rows = len >> 9;
    uint32_t acc = 0;
    const uint4 *p16 = reinterpret_cast<const uint4 *>(p) + lane;
    uint32_t row = 0;
    for (; row + 4 <= rows; row += 4) {
      uint4 w[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) w[u] = __ldcs(p16 + 32 * (row + u));
#pragma unroll
      for (int u = 0; u < 4; ++u) acc = crc_op(op512, acc) ^ crc_raw16(tab, w[u]);
    }
    for (; row < rows; ++row) acc = crc_op(op512, acc) ^ crc_raw16(tab, __ldcs(p16 + 32 * row));
    uint32_t r = rows ? crc_shift(ops, acc, (len - 512u * rows) + 496u - 16u * lane) : 0u;
    // bytes after the full rows: lane j takes [16 j, 16 j + 16) of the rest
    const uint32_t t = len - 512u * rows, t0 = 16u * lane;
    if (t0 < t) {
      const uint32_t tj = min(16u, t - t0);
      uint32_t x = 0;
      for (uint32_t k = 0; k < tj; ++k) x = (x >> 8) ^ tab[(x ^ p[512u * rows + t0 + k]) & 0xFFu];
      r ^= crc_shift(ops, x, t - t0 - tj);
    }
#pragma unroll
    for (int d = 16; d; d >>= 1) r ^= __shfl_xor_sync(kFull, r, d);
    if (lane == 0) sum ^= crc_shift(all_ops, r, hi - b);
  }
  if (lane == 0 && sum) atomicXor(&s_xor, sum);
  __syncthreads();
  if (threadIdx.x == 0) {
    if (s_xor) atomicXor(sums, s_xor);
    __threadfence();
    if (atomicAdd(sums + 1, 1u) == gridDim.x - 1) {  // every CTA's part is in
      __threadfence();
      const uint32_t raw = atomicExch(sums, 0u);
      sums[1] = 0;
      *out = raw ^ crc_shift(all_ops, 0xFFFFFFFFu, hi - lo) ^ 0xFFFFFFFFu;
    }
  }
}

// ------------------------------------------------- FASTQ stream separation
// A FASTQ split into its four line streams (headers, sequences, '+' lines,
// qualities) is put back together on the device: the newlines of each
// decoded stream are indexed (count per chunk, scan, positions), then warps take
// eight consecutive records at a time and copy line r of every stream to its
// place. Record r starts at the sum over the streams of the start of their line r, since every earlier
// line of every stream precedes it in the FASTQ.
constexpr uint32_t kNlChunk = 65536;

// The four streams (each starts at a multiple of 16 bytes and is readable to
// the next one) and their newline index.
struct LineStreams {
  const uint8_t *base[4];
  uint64_t len[4];
  uint32_t chunk0[5];  // first chunk of each stream in the launch, and the total
  uint32_t *counts;    // newlines of each chunk
  uint64_t *offs[4];   // newlines before each chunk of the stream, and the stream's total
  uint32_t *nl[4];     // position of the j-th newline, j < cap
  uint64_t cap[4];
};

__device__ __forceinline__ int stream_of(const LineStreams &S, uint32_t chunk) {
  return (chunk >= S.chunk0[1]) + (chunk >= S.chunk0[2]) + (chunk >= S.chunk0[3]);
}

// bit j: byte j of v is a newline
__device__ __forceinline__ uint32_t newline_mask(uint4 v) {
  auto four = [](uint32_t w) { return ((__vcmpeq4(w, 0x0A0A0A0Au) & 0x08040201u) * 0x01010101u) >> 24; };
  return four(v.x) | four(v.y) << 4 | four(v.z) << 8 | four(v.w) << 12;
}

// the newlines of the 16 bytes at position p of buf[0, end)
__device__ __forceinline__ uint32_t newlines_at(const uint8_t *buf, uint64_t p, uint64_t end) {
  if (p >= end) return 0;
  const uint32_t m = newline_mask(*reinterpret_cast<const uint4 *>(buf + p));
  return end - p < 16 ? m & ((1u << (uint32_t)(end - p)) - 1u) : m;
}

// Newlines of each chunk of the streams; one CTA of 256 threads per chunk.
// Both kernels below read 16 bytes per lane, all four streams in one launch;
// with a byte per lane and a launch per stream they took 200 and 543 us for
// 192 MiB of FASTQ.
__global__ void __launch_bounds__(256) nl_count_kernel(LineStreams S) {
  const int s = stream_of(S, blockIdx.x);
  const uint64_t c0 = (uint64_t)(blockIdx.x - S.chunk0[s]) * kNlChunk, end = min(S.len[s], c0 + kNlChunk);
  uint32_t k = 0;
#pragma unroll 4
  for (uint32_t i = threadIdx.x * 16; i < kNlChunk; i += 256 * 16) k += __popc(newlines_at(S.base[s], c0 + i, end));
  for (int d = 16; d; d >>= 1) k += __shfl_xor_sync(kFull, k, d);
  __shared__ uint32_t part[8];
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = k;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t t = 0;
    for (int w = 0; w < 8; ++w) t += part[w];
    S.counts[blockIdx.x] = t;
  }
}

// offs[c] = newlines of the stream before chunk c, and its total (one CTA per stream)
__global__ void __launch_bounds__(1024) nl_scan_kernel(LineStreams S) {
  __shared__ uint64_t part[32];
  const int s = blockIdx.x, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const uint32_t n_chunks = S.chunk0[s + 1] - S.chunk0[s];
  const uint32_t *counts = S.counts + S.chunk0[s];
  const uint32_t per = (n_chunks + blockDim.x - 1) / blockDim.x;
  const uint32_t i0 = min(threadIdx.x * per, n_chunks), i1 = min(i0 + per, n_chunks);
  uint64_t t = 0;
  for (uint32_t i = i0; i < i1; ++i) t += counts[i];
  uint64_t incl = t;
  for (int d = 1; d < 32; d <<= 1) {
    const uint64_t v = __shfl_up_sync(kFull, incl, d);
    if (lane >= d) incl += v;
  }
  if (lane == 31) part[w] = incl;
  __syncthreads();
  uint64_t run = incl - t, total = 0;
  for (int v = 0; v < 32; ++v) {
    if (v < w) run += part[v];
    total += part[v];
  }
  for (uint32_t i = i0; i < i1; ++i) {
    S.offs[s][i] = run;
    run += counts[i];
  }
  if (threadIdx.x == 0) S.offs[s][n_chunks] = total;
}

// nl[j] = position of the stream's j-th newline (j < cap; err set beyond).
// Warp w of a chunk's CTA takes the w-th eighth of the chunk in rows of 512
// bytes; a scan over the lanes places a row's newlines after the earlier ones.
__global__ void __launch_bounds__(256) nl_positions_kernel(LineStreams S, uint32_t *err) {
  const int s = stream_of(S, blockIdx.x);
  const uint32_t c = blockIdx.x - S.chunk0[s];
  const uint64_t c0 = (uint64_t)c * kNlChunk, end = min(S.len[s], c0 + kNlChunk);
  __shared__ uint32_t wcount[8];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const uint64_t w0 = c0 + wid * (kNlChunk / 8) + lane * 16;
  uint32_t mine = 0;
#pragma unroll 4
  for (uint32_t i = 0; i < kNlChunk / 8; i += 512) mine += __popc(newlines_at(S.base[s], w0 + i, end));
  for (int d = 16; d; d >>= 1) mine += __shfl_xor_sync(kFull, mine, d);
  if (lane == 0) wcount[wid] = mine;
  __syncthreads();
  uint64_t at = S.offs[s][c];
  for (int w = 0; w < wid; ++w) at += wcount[w];
  for (uint32_t i0 = 0; i0 < kNlChunk / 8; i0 += 4 * 512) {
    uint32_t row[4];  // four rows in flight
#pragma unroll
    for (int v = 0; v < 4; ++v) row[v] = newlines_at(S.base[s], w0 + i0 + 512 * v, end);
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      uint32_t m = row[v];
      const uint32_t k = __popc(m), incl = warp_incl_scan(k, lane);
      for (uint64_t j = at + incl - k; m; m &= m - 1, ++j) {
        if (j < S.cap[s]) S.nl[s][j] = (uint32_t)(w0 + i0 + 512 * v) + (uint32_t)__ffs((int)m) - 1;
        else latch(err, kErrCorrupt);
      }
      at += __shfl_sync(kFull, incl, 31);
    }
  }
}

// The four lines of a record: sources, places in the output and lengths, and
// the first 16-byte block of each in the record's list of blocks (u[4]: their
// number). A block is an aligned 16-byte block of the output that a line
// touches.
struct RecordLines {
  const uint8_t *from[4];
  uint8_t *to[4];
  uint32_t ln[4], u[5];
};
__device__ __forceinline__ void copy_line_block(const RecordLines &L, uint32_t b) {
  uint8_t *line = L.to[0];
  const uint8_t *from = L.from[0];
  uint32_t len = L.ln[0], u0 = 0;
#pragma unroll
  for (int v = 1; v < 4; ++v)
    if (b >= L.u[v]) line = L.to[v], from = L.from[v], len = L.ln[v], u0 = L.u[v];
  const LineBlock part = line_block((uint32_t)reinterpret_cast<uintptr_t>(line) & 15u, len, b - u0);
  const uint32_t o = part.o, m = part.n;
  uint8_t *const to = line + part.from - o;
  from += part.from;
  const uint32_t dl = (uint32_t)reinterpret_cast<uintptr_t>(from) & 15u;
  const uint4 *blk = reinterpret_cast<const uint4 *>(from - dl);
  uint4 X = make_uint4(0, 0, 0, 0), Y = X;
  if (dl >= o) {
    X = blk[0];
    if (dl + m > 16) Y = blk[1];
  } else {
    Y = blk[0];
  }
  uint32_t r[4];
  realign16(X, Y, (dl - o) & 15u, r);
  if (m == 16) *reinterpret_cast<uint4 *>(to) = make_uint4(r[0], r[1], r[2], r[3]);
  else store_piece(to, r, o, m);
}

// A warp takes eight consecutive records at a time (grid-stride): line r of
// stream k is [end(r - 1), end(r)) with end(r) the byte after its newline, or
// the stream's end for a last line without one. The ends of the eight
// records' lines are one load; a record's lines are copied together, a lane to
// each 16-byte block (526 us for 192 MiB with a byte per lane and line after
// line, 237 now; two records in flight per lane took 285).
__global__ void __launch_bounds__(256) interleave_kernel(LineStreams S, uint8_t *out) {
  const int lane = threadIdx.x & 31, k = lane & 3;
  const uint64_t warps = (uint64_t)gridDim.x * (blockDim.x >> 5);
  // lines of stream 0; no index entry is read from cap on (an error is latched then)
  const uint64_t n0 = min(*(S.offs[0] + (S.chunk0[1] - S.chunk0[0])), S.cap[0]);
  const uint64_t R = n0 + (S.len[0] && (n0 == 0 || S.nl[0][n0 - 1] != S.len[0] - 1) ? 1 : 0);
  const uint64_t cnt = min(*(S.offs[k] + (S.chunk0[k + 1] - S.chunk0[k])), S.cap[k]), len = S.len[k];
  auto end_of = [&](uint64_t r) { return r < cnt ? (uint64_t)S.nl[k][r] + 1 : len; };
  for (uint64_t r0 = 8 * (blockIdx.x * (uint64_t)(blockDim.x >> 5) + (threadIdx.x >> 5)); r0 < R; r0 += 8 * warps) {
    const uint64_t r_mine = r0 + (lane >> 2);
    const uint64_t e_mine = end_of(r_mine), s_mine = r_mine ? end_of(r_mine - 1) : 0;
    const uint32_t n = (uint32_t)min((uint64_t)8, R - r0);
    auto lines_of = [&](uint32_t i) {
      RecordLines L;
      uint64_t s[4], at = 0;
      L.u[0] = 0;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        s[q] = __shfl_sync(kFull, s_mine, 4 * i + q);
        const uint64_t e = __shfl_sync(kFull, e_mine, 4 * i + q);
        L.ln[q] = e > s[q] ? (uint32_t)(e - s[q]) : 0u;
        L.from[q] = S.base[q] + s[q];
        at += s[q];
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        L.to[q] = out + at;
        at += L.ln[q];
        L.u[q + 1] = L.u[q] + line_blocks((uint32_t)reinterpret_cast<uintptr_t>(L.to[q]) & 15u, L.ln[q]);
      }
      return L;
    };
#pragma unroll 1
    for (uint32_t i = 0; i < n; ++i) {
      const RecordLines L = lines_of(i);
      for (uint32_t b = lane; b < L.u[4]; b += 32) copy_line_block(L, b);
    }
  }
}
}  // namespace

// ------------------------------------------------------------------ launchers

constexpr size_t kWarpSmem = sizeof(MatchTable) + 1280 + kSmemStage;
static_assert(sizeof(MatchTable) % 16 == 0, "keeps the stages aligned");
constexpr size_t kSmemLutBytes = kLutBytes + (size_t)(kDecodeThreads / 32) * kWarpSmem;

int decode_grid(int device, int block) {
  (void)block;
  int sms = 0, a = 0, b = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
  const auto smem = [](const void *k) {
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemLutBytes);
  };
  smem((const void *)decode_kernel<kViewLinear, false>);
  smem((const void *)decode_kernel<kViewRing, false>);
  smem((const void *)decode_kernel<kViewPaged, false>);
  smem((const void *)decode_kernel<kViewLinear, true>);
  smem((const void *)decode_kernel<kViewRing, true>);
  smem((const void *)decode_kernel<kViewPaged, true>);
  for (const void *k : {(const void *)staged_kernel<kViewLinear>, (const void *)staged_kernel<kViewRing>,
                        (const void *)staged_kernel<kViewPaged>})
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kStagedSmem);
  smem((const void *)batch_kernel<false>);
  smem((const void *)batch_kernel<true>);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, decode_kernel<kViewLinear, false>, kDecodeThreads, kSmemLutBytes);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, batch_kernel<false>, kDecodeThreads, kSmemLutBytes);
  int per_sm = a < b ? a : b;
  if (per_sm < 1) per_sm = 1;
  return sms * per_sm;
}

// Teams per CTA and warps per team when staged_kernel takes a list of per_cta
// items per CTA, else no teams. Up to kMaxTeams segments' copies fit a CTA
// beside the decode table; fewer, larger teams are faster than seven of three
// warps (1,000 segments: 197 against 161 us).
//
// With more items than teams, teams decode a second segment after the first.
// That costs them another rANS chain and saves a single warp's match phase in
// each level of the wavefront, so it pays where the list is deep and has many
// commands, which the ratio of levels x commands per segment to rANS steps per
// segment tells: from 1.3 on (L.team_depth 2) for two segments per team, from
// 0.5 on (1) for one segment per CTA more than teams, below for none.
// us of decode_kernel -> staged_kernel, by that ratio:
//   1,824 segments (12 per CTA)
//   FASTQ, 8 levels: 16 KiB 235 -> 202 (3.1), 8 KiB 130 -> 118 (2.5), 4 KiB
//     79 -> 76 (2.1), 2 KiB 58 -> 56 (1.9)
//   FASTQ, 5 levels: 16 KiB 192 -> 182 (1.9), 8 KiB 107 -> 106 (1.5), 4 KiB
//     64 -> 70 (1.2), 2 KiB 46 -> 51 (1.1)
//   FASTQ, 3 levels: 16 KiB 156 -> 159 (1.1), 8 KiB 88 -> 93 (0.9)
//   genome, 2 or 3 levels: 16 KiB 87 -> 104 (0.3), 8 KiB 53 -> 69, 4 KiB
//     35 -> 43, 2 KiB 25 -> 35, 1 KiB 23 -> 29 (less)
//   950 segments (7 per CTA)
//   FASTQ, 4 levels: 16 KiB 160 -> 132 (1.3), 4 KiB 54 -> 52 (0.9)
//   FASTQ, 3 levels: 16 KiB 143 -> 120 (1.0), 4 KiB 50 -> 47 (0.7)
//   FASTQ, 2 levels: 16 KiB 125 -> 117 (0.6), 8 KiB 68 -> 69 (0.5), 4 KiB 44 -> 45
//   FASTQ, 1 level: 16 KiB 103 -> 116 (0.3), 4 KiB 38 -> 44
//   (16 KiB, 4 levels, 1,216 segments, 8 per CTA: 163 -> 154 at 1.37)
// With one segment to a team, segments of 4 KiB and more gain or lose little (us,
// 912 segments: FASTQ, 8 levels, 16 KiB 211 -> 163, 4 KiB 72 -> 62; 2 levels,
// 4 KiB 43 -> 41; genome, 16 KiB 74 -> 70, 4 KiB 34 -> 37). In smaller ones the
// chain and the match phase are short against a team's barriers and its write
// back: 2 KiB gain in deep lists (8 levels 52 -> 48, 304 segments 44 -> 41; 3
// levels 34 -> 35) and lose in others (2 levels 30 -> 32, genome 22 -> 28), 1 KiB
// lose in all (37 -> 39, 24 -> 26, 20 -> 24).
struct Teams {
  uint32_t n, warps;
};
static Teams team_shape(const DecodeLaunch &L, uint32_t per_cta) {
  const uint32_t warps = std::min(L.active_warps, kStagedThreads / 32);
  const uint32_t fit = std::min((kStagedSmem - kLutBytes) / team_layout(L.arc0.log2_S, L.max_stage).bytes, kMaxTeams);
  const bool large = L.arc0.log2_S >= 12 || (L.arc0.log2_S == 11 && L.team_depth);
  if (!large || per_cta > fit + (L.team_depth == 2 ? fit : L.team_depth) || L.max_stage > L.stage_cap) return {0, 0};
  const uint32_t n = std::min(per_cta, fit), T = std::min(kMaxTeam, warps / n);
  return T >= 2 ? Teams{n, T} : Teams{0, 0};
}

cudaError_t launch_decode(const DecodeLaunch &L0, int grid, int block, cudaStream_t st) {
  (void)block;
  if (L0.n_work == 0) return cudaSuccess;
  DecodeLaunch L = L0;
  // A list shorter than the grid's warps is spread over the SMs: warps claim
  // items as they come, and with all 32 warps of a CTA claiming, the first
  // CTAs to start would take the whole list (152 segments, one per SM instead
  // of on five SMs: 75.7 -> 56.4 us; 902 segments of a read's closure: 315 ->
  // 284 us a lookup). A CTA that starts late still finds the list's rest.
  if ((uint32_t)grid > L.n_work) grid = (int)L.n_work;
  const uint32_t per_cta = (L.n_work + grid - 1) / grid;
  const Teams teams = team_shape(L, per_cta);
  if (teams.n) {
    const size_t bytes = kLutBytes + (size_t)teams.n * team_layout(L.arc0.log2_S, L.max_stage).bytes;
    const int threads = (int)(teams.n * teams.warps * 32);
    if (L.view0.page) staged_kernel<kViewPaged><<<grid, threads, bytes, st>>>(L, teams.n, teams.warps);
    else if (L.view0.mask != ~uint64_t(0)) staged_kernel<kViewRing><<<grid, threads, bytes, st>>>(L, teams.n, teams.warps);
    else staged_kernel<kViewLinear><<<grid, threads, bytes, st>>>(L, teams.n, teams.warps);
    return cudaGetLastError();
  }
  L.active_warps = std::min(L.active_warps, per_cta);
  // every segment's command streams fit the shared stage: the stage-in-shared kernel
  const bool sh = L.max_stage <= L.stage_cap;
  if (L.view0.page) {
    if (sh) decode_kernel<kViewPaged, true><<<grid, kDecodeThreads, kSmemLutBytes, st>>>(L);
    else decode_kernel<kViewPaged, false><<<grid, kDecodeThreads, kSmemLutBytes, st>>>(L);
  } else if (L.view0.mask != ~uint64_t(0)) {
    if (sh) decode_kernel<kViewRing, true><<<grid, kDecodeThreads, kSmemLutBytes, st>>>(L);
    else decode_kernel<kViewRing, false><<<grid, kDecodeThreads, kSmemLutBytes, st>>>(L);
  } else {
    if (sh) decode_kernel<kViewLinear, true><<<grid, kDecodeThreads, kSmemLutBytes, st>>>(L);
    else decode_kernel<kViewLinear, false><<<grid, kDecodeThreads, kSmemLutBytes, st>>>(L);
  }
  return cudaGetLastError();
}

cudaError_t launch_batch(const DecodeLaunch &L, uint32_t n_arcs, uint32_t n_small, int grid, cudaStream_t st) {
  if (n_arcs == 0) return cudaSuccess;
  // (as launch_decode: the stage-in-shared kernel when every segment of every archive fits)
  // pairs only where archives wait for CTAs (512 archives of 16 KiB to 2 MiB:
  // 558 -> 505 us)
  const uint32_t n_large = n_arcs > (uint32_t)grid ? n_arcs - n_small : n_arcs;
  if (L.max_stage <= L.stage_cap) batch_kernel<true><<<grid, kDecodeThreads, kSmemLutBytes, st>>>(L, n_arcs, n_large);
  else batch_kernel<false><<<grid, kDecodeThreads, kSmemLutBytes, st>>>(L, n_arcs, n_large);
  return cudaGetLastError();
}

cudaError_t launch_window_order(const SegRec *dir, uint64_t n_seg, uint64_t per, uint32_t max_level, WorkItem *out,
                                cudaStream_t st) {
  if (!n_seg || !per) return cudaSuccess;
  const uint64_t warps = (n_seg + per - 1) / per;
  window_order_kernel<<<(unsigned)((warps + 7) / 8), 256, 0, st>>>(dir, n_seg, per, max_level, out);
  return cudaGetLastError();
}

cudaError_t launch_init_flags(uint64_t *flags, const SegRec *dir, uint64_t n, cudaStream_t st) {
  if (!n) return cudaSuccess;
  init_flags_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(flags, dir, n);
  return cudaGetLastError();
}

cudaError_t launch_begin_list(const WorkList &list, WorkItem *work, uint32_t *page, uint32_t *global_epoch,
                              uint32_t *epoch, uint32_t *counter, cudaStream_t st) {
  begin_list_kernel<<<1, 1024, 0, st>>>(list, work, page, global_epoch, epoch, counter);
  return cudaGetLastError();
}

cudaError_t launch_begin(uint32_t *global_epoch, uint32_t *epoch, uint32_t *counter, cudaStream_t st) {
  begin_kernel<<<1, 1, 0, st>>>(global_epoch, epoch, counter);
  return cudaGetLastError();
}

cudaError_t launch_clear_pages(uint32_t *page, const WorkItem *work, uint32_t n, cudaStream_t st) {
  if (!n) return cudaSuccess;
  clear_pages_kernel<<<(n + 255) / 256, 256, 0, st>>>(page, work, n);
  return cudaGetLastError();
}

cudaError_t launch_copy_view(OutView src, OutView dst, uint32_t log2_S, uint64_t lo, uint64_t hi, cudaStream_t st) {
  if (hi <= lo) return cudaSuccess;
  uint64_t n = hi - lo;
  int grid = (int)((n + 255) / 256 < 8192 ? (n + 255) / 256 : 8192);
  copy_view_kernel<<<grid, 256, 0, st>>>(src, dst, log2_S, lo, n);
  return cudaGetLastError();
}

// Ranges up to this many bytes are gathered by one CTA, which clears the page
// table too (a lookup's record or region: one launch of 3 us instead of two).
// Not after a wide closure: one CTA clears 1,024 entries in about 0.4 us, the
// kernel of its own takes 3 us for any number (a read with 5,952 segments, of
// 4 KiB: 234.8 us by one CTA, 232.7 apart; below 4,096 there is no difference).
constexpr uint64_t kShortGather = 16384;
constexpr uint32_t kShortClear = 4096;

cudaError_t launch_gather(OutView v, uint32_t log2_S, uint64_t lo, uint64_t hi, uint8_t *dst, uint32_t *page,
                          const WorkItem *work, uint32_t n_work, cudaStream_t st) {
  if (hi - lo <= kShortGather && n_work <= kShortClear) {
    gather_clear_kernel<<<1, 1024, 0, st>>>(v, log2_S, lo, hi - lo, dst, page, work, n_work);
    return cudaGetLastError();
  }
  const uint64_t n = hi - lo, want = (n / 16 + 2 + 255) / 256;  // (up to two partial blocks)
  const int grid = (int)(want < 4096 ? want : 4096);
  gather_kernel<<<grid, 256, 0, st>>>(v, log2_S, lo, n, dst);
  return launch_clear_pages(page, work, n_work, st);
}

cudaError_t launch_gather_bases(OutView v, uint32_t log2_S, uint64_t lo, uint32_t phase, uint32_t line_width,
                                uint64_t n, uint8_t *dst, uint32_t *page, const WorkItem *work, uint32_t n_work,
                                cudaStream_t st) {
  if (n <= kShortGather && n_work <= kShortClear) {
    gather_bases_kernel<<<1, 1024, 0, st>>>(v, log2_S, lo, phase, line_width, n, dst, page, work, n_work);
    return cudaGetLastError();
  }
  int grid = (int)((n + 255) / 256 < 4096 ? (n + 255) / 256 : 4096);
  gather_bases_kernel<<<grid, 256, 0, st>>>(v, log2_S, lo, phase, line_width, n, dst, nullptr, nullptr, 0);
  return launch_clear_pages(page, work, n_work, st);
}

cudaError_t launch_fastq_interleave(const uint8_t *const base[4], const uint64_t len[4], uint32_t *counts,
                                    uint64_t *offs, uint32_t *const nl[4], const uint64_t cap[4], uint32_t *err,
                                    uint8_t *out, cudaStream_t st) {
  LineStreams S{};
  uint32_t chunks = 0;
  for (int k = 0; k < 4; ++k) {
    S.base[k] = base[k];
    S.len[k] = len[k];
    S.chunk0[k] = chunks;
    S.offs[k] = offs + chunks + k;
    S.nl[k] = nl[k];
    S.cap[k] = cap[k];
    chunks += (uint32_t)((len[k] + kNlChunk - 1) / kNlChunk);
  }
  S.chunk0[4] = chunks;
  S.counts = counts;
  if (!chunks) return cudaSuccess;
  nl_count_kernel<<<chunks, 256, 0, st>>>(S);
  nl_scan_kernel<<<4, 1024, 0, st>>>(S);
  nl_positions_kernel<<<chunks, 256, 0, st>>>(S, err);
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  interleave_kernel<<<8 * sms, 256, 0, st>>>(S, out);
  return cudaGetLastError();
}

cudaError_t launch_multi_gather(const GatherJob *jobs, uint32_t n_jobs, uint64_t n_chunks, cudaStream_t st) {
  if (!n_jobs || !n_chunks) return cudaSuccess;
  const int grid = (int)(n_chunks < 4096 ? n_chunks : 4096);
  multi_gather_kernel<<<grid, 256, 0, st>>>(jobs, n_jobs, n_chunks);
  return cudaGetLastError();
}

cudaError_t launch_set_pages(uint32_t *page, const WorkItem *work, uint32_t n, cudaStream_t st) {
  if (!n) return cudaSuccess;
  set_pages_kernel<<<(n + 255) / 256, 256, 0, st>>>(page, work, n);
  return cudaGetLastError();
}

cudaError_t launch_closure_seed(ClosureDev C, uint32_t s_lo, uint32_t n, uint32_t top, uint32_t gen, cudaStream_t st) {
  closure_seed_kernel<<<(n + 255) / 256 < 1024 ? (n + 255) / 256 : 1024, 256, 0, st>>>(C, s_lo, n, top, gen);
  return cudaGetLastError();
}

cudaError_t launch_closure_expand(ClosureDev C, uint32_t level, uint32_t top, uint32_t gen, cudaStream_t st) {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  closure_expand_kernel<<<2 * sms, 512, 0, st>>>(C, level, top, gen);
  return cudaGetLastError();
}

cudaError_t launch_closure_order(ClosureDev C, uint32_t top, WorkItem *work, uint32_t *page, uint32_t *n_out,
                                 cudaStream_t st) {
  closure_order_kernel<<<1, 1024, 0, st>>>(C, top, work, page, n_out);
  return cudaGetLastError();
}

static bool g_crc_ready[64] = {};

// Fills g_crc_tabs on the current device (once per device).
static cudaError_t ensure_crc_constants() {
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 0 && dev < 64 && g_crc_ready[dev]) return cudaSuccess;
  static std::vector<uint32_t> tabs;
  static std::once_flag once;
  std::call_once(once, [] {
    tabs.assign(kCrcTabWords, 0);
    auto byte_step = [](uint32_t c) {
      for (int k = 0; k < 8; ++k) c = (c >> 1) ^ (0xEDB88320u & (0u - (c & 1u)));
      return c;
    };
    uint32_t *T = tabs.data();
    for (uint32_t b = 0; b < 256; ++b) T[b] = byte_step(b);
    for (int k = 1; k < 16; ++k)
      for (uint32_t b = 0; b < 256; ++b) {
        const uint32_t c = T[256 * (k - 1) + b];
        T[256 * k + b] = (c >> 8) ^ T[c & 0xFFu];
      }
    // col[k][i]: register 1 << i shifted by 2^k zero bytes (repeated squaring)
    std::vector<uint32_t> col(32 * kCrcOps);
    for (int i = 0; i < 32; ++i) col[i] = byte_step(1u << i);
    for (int k = 1; k < kCrcOps; ++k)
      for (int i = 0; i < 32; ++i) {
        uint32_t v = col[32 * (k - 1) + i], r = 0;
        for (int j = 0; j < 32; ++j)
          if (v >> j & 1u) r ^= col[32 * (k - 1) + j];
        col[32 * k + i] = r;
      }
    for (int k = 0; k < kCrcOps; ++k)
      for (int i = 0; i < 4; ++i)
        for (uint32_t v = 0; v < 256; ++v) {
          uint32_t r = 0;
          for (int j = 0; j < 8; ++j)
            if (v >> j & 1u) r ^= col[32 * k + 8 * i + j];
          T[4096 + 1024 * k + 256 * i + v] = r;
        }
  });
  cudaError_t e = cudaMemcpyToSymbol(g_crc_tabs, tabs.data(), tabs.size() * sizeof(uint32_t));
  if (e == cudaSuccess && dev >= 0 && dev < 64) g_crc_ready[dev] = true;
  return e;
}

// log2 of the pieces that window_crc_kernel's warps take: 16 KiB, less where a
// window has not that much for every warp of the grid, and never less than a
// segment. Each piece costs a shift of its CRC past the rest of the window, up
// to 30 dependent table steps by one lane, which is nothing beside 16 KiB and
// more than the reading of a small segment (193 MB in 128 MiB windows, segments
// of 64 bytes / 256 bytes / 1 KiB / 4 KiB: 3,049 / 896 / 306 / 175 us with a
// kernel of its own to join the segments' CRCs, 3,628 / 975 / 277 / 114 with a
// piece per segment, 98 / 97 / 98 / 97 with these). A piece lies in one part of the ring
// (both are powers of two, from origin 0), and at 16 bytes alignment when lo does.
static uint32_t crc_piece(const OutView &v, uint64_t lo, uint64_t bytes, uint32_t log2_S, uint64_t warps) {
  uint32_t log2_P = log2_S;
  if ((lo & 15) == 0 && v.origin == 0)
    while (log2_P < 14 && (uint64_t(2) << log2_P) <= v.mask + 1 && (uint64_t(2) << log2_P) * warps <= bytes) ++log2_P;
  return log2_P;
}

cudaError_t launch_window_crc(OutView v, uint64_t lo, uint64_t hi, uint32_t *crc, uint32_t *sums, uint32_t log2_S,
                              cudaStream_t st) {
  if (hi <= lo) return cudaSuccess;
  cudaError_t e = ensure_crc_constants();
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const uint32_t log2_P = crc_piece(v, lo, hi - lo, log2_S, (uint64_t)(3 * sms) * (kCrcThreads / 32));
  const uint64_t pieces = ((hi - 1) >> log2_P) - (lo >> log2_P) + 1;
  const uint64_t want = (pieces + kCrcThreads / 32 - 1) / (kCrcThreads / 32);
  const int grid = (int)(want < (uint64_t)(3 * sms) ? want : (uint64_t)(3 * sms));
  window_crc_kernel<<<grid, kCrcThreads, 0, st>>>(v, log2_P, lo, hi, sums, crc);
  return cudaGetLastError();
}

// ===================================================================
// Allocation-free whole-file decode (aceapex_decode_all_noalloc).
//
// Some callers cannot allocate device memory at decode time: a host program
// that hands the whole device to its own memory pool at start-up and forbids
// libraries from calling cudaMalloc afterwards, or a real-time pipeline that
// only permits allocation during initialisation. For them this entry point
// decodes an archive that the caller already holds in device memory into the
// caller's output buffer and allocates nothing: the scratch it needs (decode
// tables, ready flags, control words and per-warp staging) lives in one
// file-scope device array of fixed size, which every GPU that loads the
// library holds until the process exits.
//
// Limits: at most kNoAllocMaxSegments segments (1 GiB of output at 16 KiB
// segments); larger archives are rejected with ACEAPEX_ERANGE. All calls share the array and it keeps the last
// call's contents: each call clears the words that must start at zero and
// takes a fresh epoch, but calls that overlap on the GPU (on different
// streams, or from different threads) race and must not be issued.
namespace {

constexpr uint32_t kNoAllocMaxSegments = 65536;
constexpr size_t kNoAllocCtlBytes = 4096;                      // control words
constexpr size_t kNoAllocLutBytes = 4 * kScale * sizeof(uint32_t);
constexpr size_t kNoAllocFlagBytes = kNoAllocMaxSegments * sizeof(uint64_t);
constexpr size_t kNoAllocWorkBytes = kNoAllocMaxSegments * sizeof(WorkItem);
constexpr size_t kNoAllocBytes = kNoAllocCtlBytes + kNoAllocLutBytes + kNoAllocFlagBytes + kNoAllocWorkBytes;

// about 1.1 MiB per device
static __device__ __align__(256) uint8_t g_noalloc_scratch[kNoAllocBytes];

// control words at the start of the array: the work counter, the epoch, the
// error word, the classes without symbols (a bit each), the largest command
// stage of any segment, and per level the number of segments and the next
// place in the work list less the level's start
struct NoAllocCtl {
  uint32_t counter, epoch, err, empty, need, pad[3];
  uint32_t hist[256], next[256];
};
static_assert(sizeof(NoAllocCtl) <= kNoAllocCtlBytes, "the control words fit their part of the array");

constexpr uint32_t kNoAllocThreads = 1024;

// Builds the decode table from the archive's tables, checks their sums,
// clears the control words and takes the next epoch. One CTA: a thread per
// table entry for the prefix sums, then a thread per table slot, which finds
// its symbol by binary search (one thread summing 1,024 entries and writing
// runs of slots took 54 us; this takes 6).
__global__ void __launch_bounds__(kNoAllocThreads) noalloc_setup_kernel(const uint8_t *tables) {
  NoAllocCtl *ctl = reinterpret_cast<NoAllocCtl *>(g_noalloc_scratch);
  uint32_t *lut = reinterpret_cast<uint32_t *>(g_noalloc_scratch + kNoAllocCtlBytes);
  __shared__ uint32_t cum[4][257];  // cum[c][x + 1]: frequencies of symbols 0 .. x
  __shared__ uint32_t wsum[32], total[4];
  const uint32_t tid = threadIdx.x, c = tid >> 8, x = tid & 255, lane = tid & 31, w = tid >> 5;
  const uint32_t f = (uint32_t)tables[2 * tid] | (uint32_t)tables[2 * tid + 1] << 8;
  const uint32_t incl = warp_incl_scan(f, (int)lane);
  if (lane == 31) wsum[w] = incl;
  __syncthreads();
  uint32_t before = 0;
  for (uint32_t v = w & ~7u; v < w; ++v) before += wsum[v];
  cum[c][x + 1] = before + incl;
  if (x == 0) cum[c][0] = 0;
  if (x == 255) total[c] = before + incl;
  for (uint32_t i = tid; i < 256; i += kNoAllocThreads) ctl->hist[i] = ctl->next[i] = 0;
  __syncthreads();
  const bool bad = (total[0] && total[0] != kScale) || (total[1] && total[1] != kScale) ||
                   (total[2] && total[2] != kScale) || (total[3] && total[3] != kScale);
  for (uint32_t i = tid; i < 4 * kScale && !bad; i += kNoAllocThreads) {
    const uint32_t cl = i >> kScaleBits, slot = i & (kScale - 1);
    if (!total[cl]) {
      lut[i] = 0;
      continue;
    }
    uint32_t s = 0;  // the symbol with cum <= slot < cum + f: the number of later starts at or below slot
    for (uint32_t d = 128; d; d >>= 1)
      if (cum[cl][s + d] <= slot) s += d;
    lut[i] = s | (slot - cum[cl][s]) << 8 | (cum[cl][s + 1] - cum[cl][s] - 1) << 20;
  }
  if (tid == 0) {
    ctl->counter = 0;
    ctl->err = bad ? kErrCorrupt : 0u;
    ctl->empty = (total[0] ? 0u : 1u) | (total[1] ? 0u : 2u) | (total[2] ? 0u : 4u) | (total[3] ? 0u : 8u);
    ctl->need = 0;
    ctl->epoch = ctl->epoch + 1u;
  }
}

// A thread per segment: checks what the decoder relies on in its directory
// record (which was not validated on the host), sets its flag word, and counts
// the segments per level and the largest command stage.
__global__ void __launch_bounds__(kNoAllocThreads) noalloc_scan_kernel(DevArchive A, uint64_t payload_bytes,
                                                                       uint32_t max_level) {
  NoAllocCtl *ctl = reinterpret_cast<NoAllocCtl *>(g_noalloc_scratch);
  __shared__ uint32_t hist[256], need;
  for (uint32_t i = threadIdx.x; i < 256; i += blockDim.x) hist[i] = 0;
  if (threadIdx.x == 0) need = 0;
  __syncthreads();
  const uint32_t s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s < A.n_seg) {
    const SegRec d = A.dir[s];
    const uint32_t empty = ctl->empty;
    // (the payload test is written so that no sum can wrap)
    const uint64_t n_sym = (uint64_t)d.n_cmd * (4 + A.W) + d.n_lit;
    const bool sane = n_sym <= kMaxSym && (d.payload_off & 15) == 0 && d.payload_off <= payload_bytes &&
                      payload_bytes - d.payload_off >= 128 &&
                      d.n_words <= (payload_bytes - d.payload_off - 128) / 2 && d.level <= max_level &&
                      !(d.n_cmd && (empty & 7u)) && !(d.n_lit && (empty & 8u));
    if (!sane) latch(&ctl->err, kErrCorrupt);  // no segment is decoded then
    else atomicMax(&need, d.n_cmd * (4 + A.W) + 4);
    A.flags[s] = (uint64_t)d.level << 32;
    atomicAdd(&hist[min((uint32_t)d.level, 255u)], 1u);
  }
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < 256; i += blockDim.x)
    if (hist[i]) atomicAdd(&ctl->hist[i], hist[i]);
  if (threadIdx.x == 0 && need) atomicMax(&ctl->need, need);
}

// The work list in level order (any order within a level): each CTA reserves
// its segments' places of a level with one atomic.
__global__ void __launch_bounds__(kNoAllocThreads) noalloc_order_kernel(DevArchive A, WorkItem *work) {
  NoAllocCtl *ctl = reinterpret_cast<NoAllocCtl *>(g_noalloc_scratch);
  __shared__ uint32_t start[256], count[256], wsum[8];
  const uint32_t tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  uint32_t h = 0, incl = 0;
  if (tid < 256) {
    count[tid] = 0;
    h = ctl->hist[tid];
    incl = warp_incl_scan(h, (int)lane);
    if (lane == 31) wsum[w] = incl;
  }
  __syncthreads();
  const uint32_t s = blockIdx.x * blockDim.x + tid;
  uint32_t lv = 0, at = 0;
  if (s < A.n_seg) {
    lv = min((uint32_t)A.dir[s].level, 255u);
    at = atomicAdd(&count[lv], 1u);
  }
  __syncthreads();
  if (tid < 256) {
    uint32_t before = 0;
    for (uint32_t v = 0; v < w; ++v) before += wsum[v];
    start[tid] = before + incl - h + (count[tid] ? atomicAdd(&ctl->next[tid], count[tid]) : 0u);
  }
  __syncthreads();
  if (s < A.n_seg) work[start[lv] + at] = WorkItem{0u, s};
}

// Warps of a CTA, and bytes of shared command stage each: 32 with the usual
// stage when every segment of the archive fits it, else 8 with the largest
// stage that a segment can have.
constexpr uint32_t kNoAllocBigWarps = 8;
static_assert(kLutBytes + kNoAllocBigWarps * (1280 + sizeof(MatchTable) + kStageBytes) <=
                  kLutBytes + (kDecodeThreads / 32) * (1280 + sizeof(MatchTable) + kSmemStage),
              "both splits of the shared memory fit the launch");

// The whole chip, a warp per segment, in level order. (256 warps on 32 SMs,
// with the tables and the command stages in global memory and in index order,
// took 3.06 ms for 64 MiB of FASTQ.)
__global__ void __launch_bounds__(kDecodeThreads, 1) noalloc_decode_kernel(DecodeLaunch L, bool small_done) {
  extern __shared__ __align__(16) uint8_t smem[];
  const NoAllocCtl *ctl = reinterpret_cast<const NoAllocCtl *>(g_noalloc_scratch);
  const bool big = ctl->need > kSmemStage;
  if (small_done && !big) return;  // staged_kernel has decoded the list
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  {
    const uint4 *g = reinterpret_cast<const uint4 *>(L.arc0.lut);
    uint4 *s4 = reinterpret_cast<uint4 *>(smem);
    for (uint32_t i = threadIdx.x; i < kLutBytes / 16; i += blockDim.x) s4[i] = g[i];
    __syncthreads();
  }
  const uint32_t warps = big ? kNoAllocBigWarps : kDecodeThreads / 32;
  if ((uint32_t)wid >= min(warps, L.active_warps)) return;
  uint8_t *rings = smem + kLutBytes;
  uint16_t *ring = reinterpret_cast<uint16_t *>(rings + wid * 1280);
  MatchTable *mt = reinterpret_cast<MatchTable *>(rings + warps * 1280) + wid;
  uint8_t *stage = rings + warps * (1280 + sizeof(MatchTable)) + (size_t)wid * (big ? kStageBytes : kSmemStage);
  const uint32_t epoch = ld_relaxed(L.epoch);
  PHASE_DECL;
  for (;;) {
    bool failed;
    const uint32_t idx = take_item(L.counter, L.err, lane, failed);
    if (idx >= L.n_work) break;
    if (failed) continue;
    decode_segment<true, kViewLinear, true>(L, L.arc0, L.view0, L.work[idx].seg, epoch,
                                            reinterpret_cast<const uint32_t *>(smem), stage, kStageBytes, nullptr, mt,
                                            ring, lane, ph, ph_t);
  }
  PHASE_FLUSH();
}

__global__ void noalloc_status_kernel(uint32_t *status) {
  *status = reinterpret_cast<const NoAllocCtl *>(g_noalloc_scratch)->err;
}

std::mutex g_noalloc_mu;
struct NoAllocDevice {
  uint8_t *base = nullptr;  // device address of the scratch array
  int sms = 0;
} g_noalloc_dev[64];

}  // namespace

extern "C" int aceapex_decode_all_noalloc(const void *d_archive, uint64_t nbytes, void *d_out, uint64_t out_cap,
                                          uint32_t *d_status, void *stream) {
  if (!d_archive || !d_status || nbytes < kHeaderBytes + kTablesBytes ||
      (reinterpret_cast<uintptr_t>(d_archive) & 15))
    return 1;  // ACEAPEX_EINVAL
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 4;  // ACEAPEX_ECUDA
  // set-up, once per device with that device current: the device address of
  // the scratch array (its name in host code is only a stand-in) and the
  // kernels' shared-memory limits
  uint8_t *base = nullptr;
  int grid = 0;
  {
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    NoAllocDevice &D = g_noalloc_dev[dev];
    if (!D.base) {
      void *p = nullptr;
      if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p ||
          cudaDeviceGetAttribute(&D.sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
          cudaFuncSetAttribute(noalloc_decode_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)kSmemLutBytes) != cudaSuccess ||
          cudaFuncSetAttribute(staged_kernel<kViewLinear>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)kStagedSmem) != cudaSuccess)
        return 4;
      D.base = static_cast<uint8_t *>(p);
    }
    base = D.base;
    grid = D.sms;
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  // the header, read into host stack memory
  uint8_t h[kHeaderBytes];
  if (cudaMemcpyAsync(h, d_archive, kHeaderBytes, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess)
    return 4;
  auto u64 = [&](int o) { uint64_t v; std::memcpy(&v, h + o, 8); return v; };
  auto u32 = [&](int o) { uint32_t v; std::memcpy(&v, h + o, 4); return v; };
  const uint64_t n = u64(16), n_seg = u64(40), n_deps = u64(48), n_reads = u64(56);
  const uint32_t log2_B = h[24], log2_S = h[25], W = h[26], min_match = h[27], flags = h[31];
  if (std::memcmp(h, "ACEAPEX1", 8) != 0 || u32(8) != 1 || u32(12) != kHeaderBytes || h[28] != kScaleBits ||
      h[29] != kLanes || (flags & ~1u) || (!(flags & 1u) && n_reads) || log2_B < 2 || log2_B > 30 ||
      log2_S != (log2_B < kMaxLog2S ? log2_B : kMaxLog2S) || W != offset_width(n) || min_match < 1)
    return 2;  // ACEAPEX_ECORRUPT
  // counts bounded by the archive length first, so that the section offsets
  // below cannot wrap
  if (n_seg > nbytes / 24 || n_deps > nbytes / 4 || n_reads > nbytes / 8) return 2;
  const uint64_t S = uint64_t(1) << log2_S;
  const uint64_t off_dir = u64(72), off_dep_ptr = u64(80), off_deps = u64(88), off_reads = u64(96);
  const uint64_t off_payload = u64(104), payload_bytes = u64(112), total = u64(120);
  if (off_payload > nbytes || payload_bytes > nbytes || (payload_bytes & 15)) return 2;
  if (n_seg != (n + S - 1) / S || u64(64) != kHeaderBytes || off_dir != kHeaderBytes + kTablesBytes ||
      off_dep_ptr != round16(off_dir + 24 * n_seg) || off_deps != round16(off_dep_ptr + 8 * (n_seg + 1)) ||
      off_reads != round16(off_deps + 4 * n_deps) || off_payload != round16(off_reads + 8 * n_reads) ||
      total != off_payload + payload_bytes || total != nbytes)
    return 2;
  if (n_seg > kNoAllocMaxSegments) return 6;  // ACEAPEX_ERANGE: beyond the fixed scratch
  if (out_cap < n || (n && !d_out)) return 6;
  if (n == 0) return cudaMemsetAsync(d_status, 0, 4, st) == cudaSuccess ? 0 : 4;

  const uint8_t *arc = static_cast<const uint8_t *>(d_archive);
  DecodeLaunch L{};
  DevArchive &A = L.arc0;
  A.payload = arc + off_payload;
  A.dir = reinterpret_cast<const SegRec *>(arc + off_dir);
  A.lut = reinterpret_cast<const uint32_t *>(base + kNoAllocCtlBytes);
  A.flags = reinterpret_cast<uint64_t *>(base + kNoAllocCtlBytes + kNoAllocLutBytes);
  A.blocked = nullptr;
  A.n = n;
  A.D = u64(32);
  A.log2_S = log2_S;
  A.W = W;
  A.min_match = min_match;
  A.n_seg = (uint32_t)n_seg;
  L.view0.base = static_cast<uint8_t *>(d_out);
  L.view0.origin = 0;
  L.view0.mask = ~uint64_t(0);
  NoAllocCtl *ctl = reinterpret_cast<NoAllocCtl *>(base);
  WorkItem *work = reinterpret_cast<WorkItem *>(base + kNoAllocCtlBytes + kNoAllocLutBytes + kNoAllocFlagBytes);
  L.counter = &ctl->counter;
  L.epoch = &ctl->epoch;
  L.err = &ctl->err;
  L.work = work;
  L.n_work = (uint32_t)n_seg;
  L.scratch = nullptr;
  L.wait_ns = 2000000000ull;
  L.active_warps = kDecodeThreads / 32;
  L.stage_cap = L.max_stage = kSmemStage;
  L.stage_need = &ctl->need;
  L.team_depth = 2;  // (the commands are counted on the device; FASTQ is the deep case)
  const unsigned blocks = (unsigned)((n_seg + kNoAllocThreads - 1) / kNoAllocThreads);
  noalloc_setup_kernel<<<1, kNoAllocThreads, 0, st>>>(arc + kHeaderBytes);
  // (a reader that waits for a segment whose record is corrupt gives up: the
  // error is latched before any segment is taken)
  noalloc_scan_kernel<<<blocks, kNoAllocThreads, 0, st>>>(A, payload_bytes, h[30]);
  noalloc_order_kernel<<<blocks, kNoAllocThreads, 0, st>>>(A, work);
  // as launch_decode: spread a short list, and give it teams
  if ((uint64_t)grid > n_seg) grid = (int)n_seg;
  const uint32_t per_cta = (L.n_work + grid - 1) / grid;
  const Teams teams = team_shape(L, per_cta);
  if (teams.n) {
    const size_t bytes = kLutBytes + (size_t)teams.n * team_layout(log2_S, L.max_stage).bytes;
    staged_kernel<kViewLinear><<<grid, (int)(teams.n * teams.warps * 32), bytes, st>>>(L, teams.n, teams.warps);
  }
  L.active_warps = std::min(L.active_warps, per_cta);
  noalloc_decode_kernel<<<grid, kDecodeThreads, kSmemLutBytes, st>>>(L, teams.n != 0);
  noalloc_status_kernel<<<1, 1, 0, st>>>(d_status);
  return cudaGetLastError() == cudaSuccess ? 0 : 4;
}

}  // namespace aceapex

#ifdef ACEAPEX_PHASE_CLOCKS
// Instrumented build only: copies the warp cycles that the decode kernels
// spent in each phase (command-class rANS, command parse, literal rANS and
// placement, source checks, match copies, the rest of the work loop), the
// event counts (match chunks, copy rounds, copy units, segments, chunks that
// waited) and the cycles spent waiting for source segments, in that order,
// since the last reset into out[0 .. n) (n <= 12), and zeroes them when
// reset != 0.
// Synchronises the current device. Returns 0, or 4 on a CUDA error.
extern "C" int aceapex_phase_cycles(uint64_t *out, int n, int reset) {
  unsigned long long h[16] = {};
  if (cudaDeviceSynchronize() != cudaSuccess ||
      cudaMemcpyFromSymbol(h, aceapex::g_phase_cycles, sizeof(h)) != cudaSuccess)
    return 4;
  for (int i = 0; i < n && i < 12; ++i) out[i] = h[i];
  if (reset) {
    const unsigned long long z[16] = {};
    if (cudaMemcpyToSymbol(aceapex::g_phase_cycles, z, sizeof(z)) != cudaSuccess) return 4;
  }
  return 0;
}
#endif
