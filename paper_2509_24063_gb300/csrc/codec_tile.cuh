// Tile-level device functions of the batched codec (paper Sec. 2.3, steps B, C
// and D), shared by its two forms: the tile launches (codec_tiles.cu) and the
// persistent launch of an explicit schedule (batched.cu).  Matching in shared
// memory, the block scan of a tile's counts, the warps' payload stages and the
// record stash.
#pragma once

#include "codec.cuh"

namespace tera {

// hash phases take kIlp entries per thread (entry i*T + thread of the tile),
// so several independent probes / atomics are in flight per thread
constexpr u32 kIlp = 4;

__device__ __forceinline__ u64 ceil_div(u64 a, u64 b) { return (a + b - 1) / b; }

// Shared-memory matching state of the block's current pair.
struct SmemTable {
  unsigned short* tbl;  // hash table, or nullptr: the pair uses its global hash segment
  u32 mask;             // table entries - 1
  u32* bits;            // bit k: message record k was taken by a slot
};

constexpr u32 kFpBits = 3, kFpMask = (1u << kFpBits) - 1u;
constexpr u32 kTableMax = (1u << (16 - kFpBits)) - 1u;  // records of a u16 entry
__device__ __forceinline__ u32 fp_of(u64 h) { return (u32)h & kFpMask; }
__device__ __forceinline__ u32 tbl_start(u64 h, u32 mask) { return (u32)(h >> 32) & mask; }

// Exclusive block scan of packed counts (low / high 32 bits) with one
// barrier: each warp publishes its total, and after the barrier every warp
// scans the warps' totals itself.  The caller alternates `buf` (33 words)
// between consecutive scans: a buffer is written again only after the next
// scan's barrier, which every warp passes after its reads of this one.  After
// the last scan of a run, one __syncthreads() must precede other uses of buf.
__device__ __forceinline__ u64 scan_packed(u64 v, u64* buf, u64* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nwarps = (blockDim.x + 31) >> 5;
  const u64 incl = warp_incl_scan<u64>(v);
  if (lane == 31) buf[warp] = incl;
  __syncthreads();
  const u64 x = lane < nwarps ? buf[lane] : 0ull;
  const u64 xi = warp_incl_scan<u64>(x);
  *total = __shfl_sync(0xFFFFFFFFu, xi, nwarps - 1);
  return __shfl_sync(0xFFFFFFFFu, xi - x, warp) + incl - v;
}

// Each warp stages its own contiguous byte range in a private region and
// stores it with 16-byte stores inside and byte stores on the edges it shares
// with the neighbouring warps.  32 records + 16 bytes: the decode stages from
// the 16-byte boundary below its first byte, and the encode's flush reads one
// word past its last.
constexpr u32 kWarpStage = 32 * kRecBytes + 16;

// Per-thread record stash in shared memory: 16-byte part k of thread i's
// record at stash[k T + i], so each part of a warp's records is one
// contiguous 512-byte row.  It holds the record a slot or decode tile needs
// after its block scan, which would otherwise stay in registers across the
// barrier (and spill).  Only the owning thread reads its entries, so no
// barrier guards them.
template <int T>
__device__ __forceinline__ void stash_put(ulonglong2* st, const Rec& r) {
#pragma unroll
  for (int k = 0; k < 4; ++k)
    st[k * T + threadIdx.x] = make_ulonglong2(r.w[2 * k], r.w[2 * k + 1]);
}

template <int T>
__device__ __forceinline__ Rec stash_get(const ulonglong2* st) {
  Rec r;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const ulonglong2 v = st[k * T + threadIdx.x];
    r.w[2 * k] = v.x;
    r.w[2 * k + 1] = v.y;
  }
  return r;
}

// The record at g (16-byte aligned) into the stash by asynchronous
// copies; stash_wait() before reading it.
template <int T>
__device__ __forceinline__ void stash_async(ulonglong2* st, const uint8_t* g) {
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const u32 dst = (u32)__cvta_generic_to_shared(st + k * T + threadIdx.x);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" : : "r"(dst), "l"(g + 16 * k)
                 : "memory");
  }
  asm volatile("cp.async.commit_group;" : : : "memory");
}

__device__ __forceinline__ void stash_wait() { asm volatile("cp.async.wait_all;" : : : "memory"); }

// The L significant bytes of v (its higher bytes are zero) at byte offset o of
// a zeroed, 4-byte-aligned stage: ORed into the at most three 32-bit words
// they touch, so neighbouring lanes' bytes in a shared word are kept.
__device__ __forceinline__ void stage_or(uint8_t* st, u32 o, u64 v, u32 L) {
  if (L == 0) return;
  u32* w = reinterpret_cast<u32*>(st + (o & ~3u));
  const u32 sh = (o & 3u) * 8u;
  const u64 lo = v << sh;
  const u32 nb = (o & 3u) + L;  // bytes from the first word's start, at most 11
  atomicOr(&w[0], (u32)lo);
  if (nb > 4) atomicOr(&w[1], (u32)(lo >> 32));
  if (nb > 8) atomicOr(&w[2], (u32)(v >> (64u - sh)));
}

// Zero the first n bytes of a 16-byte-aligned warp stage (rounded up to 16).
__device__ __forceinline__ void warp_zero(uint8_t* wst, u32 n) {
  for (u32 c = threadIdx.x & 31; c < ((n + 15u) >> 4); c += 32)
    *reinterpret_cast<uint4*>(wst + (c << 4)) = make_uint4(0u, 0u, 0u, 0u);
}

// Store the n bytes at the start of a warp stage to gW, whatever its
// alignment: each whole 16-byte chunk of the destination is assembled from
// five 32-bit stage words by funnel shifts and stored at once; the edge
// chunks, shared with the neighbouring warps' bytes, are stored byte by byte.
// The stage has at least 16 bytes beyond n, so the fifth word stays inside it.
__device__ __forceinline__ void warp_flush(const uint8_t* wst, uint8_t* gW, u32 n) {
  const u32 s0 = (u32)((uintptr_t)gW & 15u);
  uint8_t* g16 = gW - s0;
  const u32 end = s0 + n;
  const u32 nchunks = (end + 15u) >> 4;
  const u32* w32 = reinterpret_cast<const u32*>(wst);
  for (u32 c = threadIdx.x & 31; c < nchunks; c += 32) {
    const u32 lo = c << 4, hi = lo + 16u;
    if (lo >= s0 && hi <= end) {
      const u32 o = lo - s0;  // stage offset of the chunk's first byte
      const u32 i = o >> 2, sh = (o & 3u) * 8u;
      u32 v[4];
      if (sh == 0) {
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = w32[i + k];
      } else {
        u32 a = w32[i];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const u32 b = w32[i + k + 1];
          v[k] = __funnelshift_r(a, b, sh);
          a = b;
        }
      }
      *reinterpret_cast<uint4*>(g16 + lo) = make_uint4(v[0], v[1], v[2], v[3]);
    } else {
      for (u32 x = (lo > s0 ? lo : s0); x < (hi < end ? hi : end); ++x) g16[x] = wst[x - s0];
    }
  }
}

// ---------------- match in shared memory ----------------
//
// A group of T threads carries a pair: the whole block, or (T = 32) one warp
// of a block whose warps carry a pair each.

template <int T>
__device__ __forceinline__ u32 group_thread() { return threadIdx.x & (u32)(T - 1); }

template <int T>
__device__ __forceinline__ void group_sync() {
  if constexpr (T == 32) __syncwarp();
  else __syncthreads();
}

template <int T>
__device__ __forceinline__ bool group_any(bool v) {
  if constexpr (T == 32) return __any_sync(0xFFFFFFFFu, v) != 0;
  else return __syncthreads_or(v) != 0;
}


// Index message records [0, m) of pair p.  A second record with an id already
// present is an invalid message (TERA_EINVAL) and is not indexed.
template <int T>
__device__ __forceinline__ void smem_build(const EncArgs& A, u32 p, u64 m, const SmemTable& tb) {
  const u64 g_lo = A.pair_off[p];
  for (u32 i = group_thread<T>(); i <= tb.mask; i += T) tb.tbl[i] = 0;
  for (u32 i = group_thread<T>(); i < (u32)((m + 31) / 32); i += T) tb.bits[i] = 0u;
  // message ids are read one batch ahead, so they arrive while a batch inserts
  u64 id_next[kIlp];
#pragma unroll
  for (u32 i = 0; i < kIlp; ++i) {
    const u64 k = (u64)i * T + group_thread<T>();
    id_next[i] = k < m ? msg_id(A, p, g_lo + k) : 0;
  }
  group_sync<T>();
  for (u64 k0 = 0; k0 < m; k0 += (u64)T * kIlp) {
    u64 id[kIlp];
#pragma unroll
    for (u32 i = 0; i < kIlp; ++i) {
      id[i] = id_next[i];
      const u64 k = k0 + (u64)(kIlp + i) * T + group_thread<T>();
      id_next[i] = k < m ? msg_id(A, p, g_lo + k) : 0;
    }
#pragma unroll
    for (u32 i = 0; i < kIlp; ++i) {
      const u64 k = k0 + (u64)i * T + group_thread<T>();
      if (k >= m) continue;
      const u64 h = mix64(id[i]);
      const u32 fp = fp_of(h);
      const unsigned short e = (unsigned short)(((u32)(k + 1) << kFpBits) | fp);
      u32 at = tbl_start(h, tb.mask);
      for (u32 probe = 0; probe <= tb.mask; ++probe) {
        const u32 old = atomicCAS(&tb.tbl[at], (unsigned short)0, e);
        if (old == 0u) break;
        if ((old & kFpMask) == fp && msg_id(A, p, g_lo + (old >> kFpBits) - 1) == id[i]) {
          latch(A.st, TERA_EINVAL);  // ids must be unique within a message
          break;
        }
        at = (at + 1) & tb.mask;
      }
    }
  }
}

// Message record (index in the pair) with this id, probing from `at`; kNoMatch if none.
__device__ __forceinline__ u32 smem_find(const EncArgs& A, u32 p, const SmemTable& tb, u64 g_lo,
                                         u64 id, u32 fp, u32 at) {
  for (u32 probe = 0; probe <= tb.mask; ++probe) {
    const u32 e = tb.tbl[at];
    if (e == 0u) return kNoMatch;
    if ((e & kFpMask) == fp && msg_id(A, p, g_lo + (e >> kFpBits) - 1) == id)
      return (e >> kFpBits) - 1;
    at = (at + 1) & tb.mask;
  }
  return kNoMatch;
}

// Look every slot of pair p up; slot_src[slot] = global record index or
// kNoMatch; bits mark the taken records.  Returns this thread's match count.
template <int T>
__device__ __forceinline__ u32 smem_match(const EncArgs& A, u32 p, u64 r, const SmemTable& tb) {
  // no reference (r = 0): ref_off is null and no slot is read
  const u64 ro = A.ref_off ? A.ref_off[p] : 0, g_lo = A.pair_off[p];
  u32 found = 0;
  // slot ids are read one batch ahead, so they arrive while a batch probes
  u64 id_next[kIlp];
#pragma unroll
  for (u32 i = 0; i < kIlp; ++i) {
    const u64 j = (u64)i * T + group_thread<T>();
    id_next[i] = j < r ? ref_id(A, p, ro, j) : 0;
  }
  for (u64 j0 = 0; j0 < r; j0 += (u64)T * kIlp) {
    u64 id[kIlp];
#pragma unroll
    for (u32 i = 0; i < kIlp; ++i) {
      id[i] = id_next[i];
      const u64 j = j0 + (u64)(kIlp + i) * T + group_thread<T>();
      id_next[i] = j < r ? ref_id(A, p, ro, j) : 0;
    }
    // first fingerprint hit of every slot (shared memory only), then the
    // id checks of all of them in flight together
    u32 cand[kIlp], at[kIlp], fp[kIlp];
#pragma unroll
    for (u32 i = 0; i < kIlp; ++i) {
      const u64 j = j0 + (u64)i * T + group_thread<T>();
      cand[i] = kNoMatch;
      const u64 h = mix64(id[i]);
      fp[i] = fp_of(h);
      at[i] = tbl_start(h, tb.mask);
      if (j >= r) continue;
      for (u32 probe = 0; probe <= tb.mask; ++probe) {
        const u32 e = tb.tbl[at[i]];
        if (e == 0u) break;
        if ((e & kFpMask) == fp[i]) {
          cand[i] = (e >> kFpBits) - 1;
          break;
        }
        at[i] = (at[i] + 1) & tb.mask;
      }
    }
    u64 cid[kIlp];
#pragma unroll
    for (u32 i = 0; i < kIlp; ++i) cid[i] = cand[i] != kNoMatch ? msg_id(A, p, g_lo + cand[i]) : 0;
#pragma unroll
    for (u32 i = 0; i < kIlp; ++i) {
      const u64 j = j0 + (u64)i * T + group_thread<T>();
      if (j >= r) continue;
      u32 k = cand[i];
      if (k != kNoMatch && cid[i] != id[i])  // fingerprint collision: keep probing
        k = smem_find(A, p, tb, g_lo, id[i], fp[i], (at[i] + 1) & tb.mask);
      if (k != kNoMatch) {
        const u32 bit = 1u << (k & 31u);
        if (atomicOr(&tb.bits[k >> 5], bit) & bit) {
          latch(A.st, TERA_EINVAL);  // a second slot with the same id: that slot is a hole
          k = kNoMatch;
        }
      }
      found += k != kNoMatch;
      A.slot_src[ro + j] = k != kNoMatch ? (u32)(g_lo + k) : kNoMatch;
    }
  }
  return found;
}

// ---------------- match of ascending id lists ----------------
//
// When the ids of a pair's message strictly ascend (agents kept in the order
// their ids were given, so that each list, in agent order, is in id order), a
// slot's match is found without an index: the round of reference slots from
// j0 (2 kIlp per thread) loads the message ids from kWinSlack before to
// kWinSlack after [j0 + d, j0 + d + 2 kIlp T) into shared memory, d = (message
// index - slot index) of the last match so far, and each slot searches that
// window by bisection (a slot whose id lies outside it searches all message
// ids).  Every slot is looked up by bisection, so the matches are the index's
// whatever the reference order; an ascending reference keeps the searches in
// the window.  Pairs whose message ids do not ascend take the index.

constexpr u32 kWinSlack = 64;

// The message ids of pair p strictly ascending (the same answer in every
// thread).  A reference slot whose id repeats finds a record already taken,
// which the search treats as the index does (an invalid reference; the slot
// is a hole).
template <int T>
__device__ __forceinline__ bool ids_ascending(const EncArgs& A, u32 p, u64 m) {
  const u64 g_lo = A.pair_off[p];
  int bad = 0;
  for (u64 k0 = group_thread<T>(); k0 + 1 < m; k0 += 4 * (u64)T) {
    u64 a[4], b[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const u64 k = k0 + (u64)i * T;
      a[i] = k + 1 < m ? msg_id(A, p, g_lo + k) : 0;
      b[i] = k + 1 < m ? msg_id(A, p, g_lo + k + 1) : 1;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) bad |= !(a[i] < b[i]);
  }
  return !group_any<T>(bad != 0);
}

// Every slot of pair p looked up (ascending message ids): slot_src[slot] =
// global record index or kNoMatch, and the taken bits; 2 kIlp slots per
// thread per round.  Returns this thread's match count.  win: shared memory
// for 2 kIlp T + 2 kWinSlack ids.
template <int T>
__device__ __forceinline__ u32 sorted_match(const EncArgs& A, u32 p, u64 m, u64 r,
                                            const SmemTable& tb, u64* win) {
  constexpr u32 kW = 2 * kIlp;  // slots per thread per round
  constexpr u64 kSpan = (u64)T * kW;
  // one per group: a block of warps on their own has at most eight
  __shared__ long long s_dn[T == 32 ? 8 : 1];
  __shared__ unsigned long long s_jkn[T == 32 ? 8 : 1];
  long long& s_d = s_dn[T == 32 ? threadIdx.x >> 5 : 0];
  unsigned long long& s_jk = s_jkn[T == 32 ? threadIdx.x >> 5 : 0];
  const u64 ro = A.ref_off ? A.ref_off[p] : 0, g_lo = A.pair_off[p];
  for (u32 i = group_thread<T>(); i < (u32)((m + 31) / 32); i += T) tb.bits[i] = 0u;
  if (group_thread<T>() == 0) {
    s_d = 0;
    s_jk = 0;
  }
  group_sync<T>();
  u32 found = 0;
  for (u64 j0 = 0; j0 < r; j0 += kSpan) {  // block-uniform
    const long long ws = (long long)j0 + s_d - (long long)kWinSlack;
    const u64 wlo = ws < 0 ? 0 : ((u64)ws < m ? (u64)ws : m);
    const u64 whi = wlo + kSpan + 2 * kWinSlack < m ? wlo + kSpan + 2 * kWinSlack : m;
    u64 x[kW];
#pragma unroll
    for (u32 i = 0; i < kW; ++i) {
      const u64 j = j0 + (u64)i * T + group_thread<T>();
      x[i] = j < r ? ref_id(A, p, ro, j) : 0;
    }
    for (u64 k = wlo + group_thread<T>(); k < whi; k += T) win[k - wlo] = msg_id(A, p, g_lo + k);
    group_sync<T>();  // the window is loaded
    const u64 n = whi - wlo;
    u64 last = 0;  // (slot + 1) << 32 | record of this thread's last match
#pragma unroll
    for (u32 i = 0; i < kW; ++i) {
      const u64 j = j0 + (u64)i * T + group_thread<T>();
      if (j >= r) continue;
      u32 k = kNoMatch;
      if (n > 0 && x[i] >= win[0] && x[i] <= win[n - 1]) {
        u64 lo = 0, hi = n;
        while (lo < hi) {
          const u64 mid = (lo + hi) >> 1;
          if (win[mid] < x[i]) lo = mid + 1;
          else hi = mid;
        }
        if (win[lo] == x[i]) k = (u32)(wlo + lo);
      } else {
        u64 lo = 0, hi = m;
        while (lo < hi) {
          const u64 mid = (lo + hi) >> 1;
          if (msg_id(A, p, g_lo + mid) < x[i]) lo = mid + 1;
          else hi = mid;
        }
        if (lo < m && msg_id(A, p, g_lo + lo) == x[i]) k = (u32)lo;
      }
      if (k != kNoMatch) {
        const u32 bit = 1u << (k & 31u);
        if (atomicOr(&tb.bits[k >> 5], bit) & bit) {
          latch(A.st, TERA_EINVAL);  // a second slot with the same id: that slot is a hole
          k = kNoMatch;
        }
      }
      if (k != kNoMatch) {
        ++found;
        last = ((j + 1) << 32) | k;
      }
      A.slot_src[ro + j] = k != kNoMatch ? (u32)(g_lo + k) : kNoMatch;
    }
    // the round's last match: its offset carries to the next round
    u64 wl = last;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const u64 t = __shfl_xor_sync(0xFFFFFFFFu, wl, o);
      wl = t > wl ? t : wl;
    }
    if ((group_thread<T>() & 31) == 0 && wl) atomicMax(&s_jk, wl);
    group_sync<T>();  // the window is read, s_jk is final
    if (group_thread<T>() == 0 && s_jk) {
      s_d = (long long)(s_jk & 0xFFFFFFFFull) - (long long)((s_jk >> 32) - 1);
      s_jk = 0;
    }
    group_sync<T>();
  }
  return found;
}

// ---------------- predictor ----------------

// Predictor work of a matched slot: the training sample, and the slot's
// residual payload size from the prediction the pre-pass made (predictions
// exist only with both a history and the network, and then the pre-pass has
// run).
template <bool PR>
__device__ __forceinline__ u64 pred_slot(const EncArgs& A, u32 p, u64 j, u64 r, u64 mode,
                                         const Rec& R, const Rec& M, u32 bxor) {
  u64 vres = bxor;
  if (!A.pr.hist || mode != TERA_MODE_XOR) return vres;
  if (A.pr.samples) {
    const Hist H = load_hist(A.pr.hist + kHistBytes * (A.ref_off[p] + j));
    const u32 nc = cell_count(A.pr.cseg, seg_base(A.ref_off[p], p), seg_size(r),
                              cell_key(R, A.pr));
    float f[kMlpIn];
    if (features(R, H, nc, f)) {
      float* smp = A.pr.samples + (u64)kSampleFloats * (A.ref_off[p] + j);
#pragma unroll
      for (int i = 0; i < kMlpIn; ++i) smp[i] = f[i];
#pragma unroll
      for (int a = 0; a < 3; ++a)
        smp[kMlpIn + a] = __double2float_rn(
            __dsub_rn(__longlong_as_double((long long)M.w[1 + a]),
                      __longlong_as_double((long long)R.w[1 + a])));
      smp[11] = 1.0f;
    }
  }
  if (A.pr.pre) {
    const u64* ps = A.pr.pscr + 4 * (A.ref_off[p] + j);
    if (__ldcg(ps + 3)) {
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        vres += sig_bytes(zigzag(M.w[1 + a] - __ldcg(ps + a)));
        vres -= sig_bytes(M.w[1 + a] ^ R.w[1 + a]);
      }
    }
  }
  return vres;
}

// ---------------- decode ----------------

// The L (0..8) bytes at byte offset o of an 8-byte-aligned stage, as a
// little-endian word: two aligned 8-byte loads and a funnel shift (the stage
// is followed by at least 16 bytes of shared memory, so the second load stays
// inside the allocation; bytes past the staged data are masked off).
__device__ __forceinline__ u64 stage_bytes_at(const uint8_t* st, u32 o, u32 L) {
  const u64* w = reinterpret_cast<const u64*>(st + (o & ~7u));
  const u32 sh = (o & 7u) * 8u;
  const u64 lo = w[0], hi = w[1];
  const u64 x = sh ? (lo >> sh) | (hi << (64u - sh)) : lo;
  return L >= 8u ? x : (x & ((1ull << (8u * L)) - 1ull));
}

// Facts of one entry of a decode tile from its code.
struct DecEnt {
  u32 b, vn;  // payload bytes, record decoded (not a placeholder)
  bool hole;
  bool bad;   // malformed code: not decoded, no payload
};

__device__ __forceinline__ DecEnt dec_entry(DevStatus* st, u32 code, u64 e, u64 n, u64 ns) {
  DecEnt x{0u, 0u, true, false};
  if (e < n && !check_code(code, e, ns, &x.hole, &x.b)) {
    x.bad = true;
    x.b = 0;
    latch(st, TERA_ECORRUPT);
  }
  x.vn = (e < n && !x.hole) ? 1u : 0u;
  return x;
}

}  // namespace tera
