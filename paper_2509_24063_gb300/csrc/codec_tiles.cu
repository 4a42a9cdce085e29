// Batched codec over tiles: steps a3-a5 (paper Sec. 2.3, steps B, C and D) for
// every pair of one iteration, as launches over tiles of 32 to 256 entries; only
// the match has a block or a warp a pair, and parts the large ones:
//
//   setup   per-pair facts, wire slabs and the lists of tiles
//   match   one block (a warp for a small pair) per pair: the message record of
//           every reference slot (ids in shared memory), the matches before each
//           tile and the list of the records no slot took; a big pair (more than
//           kTableMax records, or kBlockSlots slots and twice a block's share) is
//           only asked here, a tile each, whether its ids ascend, and matched by
//   bigmatch  (tiles of such pairs; does nothing without them): by bisection
//           over ascending ids, else in a global hash segment that its tiles
//           index first
//   sizes   predictor only: the payload of the XOR and of the residual form
//   encode  one tile of slots or new records: difference, code, new-reference
//           records, and the payload, packed, into the tile's own part of the
//           receive buffer (a tile's payload never exceeds its records)
//   wire    one tile: its payload's place in the message, from the counts of
//           the tiles before it, and the payload copied there; the headers of
//           the pairs without entries
//   decode  one tile of entries from the wire and the receiver's reference
//
// Only the payload's place depends on other tiles' contents, and the payload
// is a small part of the bytes moved (11 of some 330 per record), so writing
// it twice costs less than any order among the tiles: no tile waits for
// another.
//
// Why tiles: a block that carries a pair through all steps on its own (the
// persistent launch of batched.cu, used for an explicit schedule) pays every
// step's memory latency once per tile of every pair, one after the other, and
// the largest pair is the launch's length.  Measured, whole codec: uniform 100
// M agents (16.6 M records) 1.98 -> 1.45 ms, of which encode 690 us (3.58 GB,
// 77 % of the measured copy rate), decode 467 us (2.3 GB), match 179, wire 95,
// setup 17; 16 M agents kept box by box 0.93 -> 0.62 ms; a pair of 1.1 M
// records among 6.5 M: 3.3 -> 0.8 ms; 6.3 K records in 12 pairs: 92 -> 60 us.
// A look-back over the tiles in place of the second copy of the payload
// (tiles claimed in order, sums published) left encode and decode at 1.16 ms
// each; a block a tile with barriers between its steps at 0.86 and 0.74.
#include "codec_tile.cuh"

using namespace tera;

namespace {

constexpr int kT = 256;           // threads of a block
constexpr int kPerSm = 4;         // resident blocks per SM (64 registers a thread)
constexpr int kEncPerSm = 4, kDecPerSm = 3;  // (the decode's shared memory: 65 KB a block)
constexpr u32 kBigTile = kT * kIlp;  // ids of a tile of a pair matched through global memory
// Entries of a tile: 32 << 0 .. 3, the most that still gives every resident
// warp kTilesPerWarp tiles; a warp takes a tile's entries 32 at a time, so a small
// iteration's tiles are a single step (uniform 4 thousand agents: encode 23 ->
// 10 us) and a large one's are not all set-up.
constexpr u32 kMinShift = 5, kMaxShift = 8;
constexpr u64 kTilesPerWarp = 8;
// Tiles of new records: the setup plans those of the m - r records that must be
// new, and one per kNewShare tiles of records for the others, which only the
// match counts; where it finds more than kNewTiles tiles of them for each
// planned one, it adds tiles at the end of the list until there is one each.
// (16 M agents, 5.9 M records, all of other ids than the reference's: with the
// planned tiles alone, each with up to sixteen tiles' records, 2573 us an
// iteration, now 1450; three in ten of other ids, 1616 and 1360.)
constexpr u32 kNewShare = 16, kNewTiles = 2;
// Pairs of at most this many slots and records are matched by one warp, so
// that the thousands of edge and corner pairs of a large grid are in flight at
// once (13,824 pairs, 100 M agents: match 297 -> 264 us, before the ids were held
// in shared memory; now 179).  A grid with few
// pairs for the GPU's blocks gives all but the smallest a block (1 M agents,
// 936 pairs: 39 us with the higher limit, 32 with the lower).
constexpr u32 kWarpPair = 256, kWarpPairFew = 64;

// The wire launch adds up the payload bytes of a pair's tiles before each: one by
// one in pairs of at most kGroupMin tiles, else by the sums of kTileGroup tiles,
// which the encode keeps for such pairs (planned and added tiles apart).  (One by
// one in every pair, the launch grew with the square of a pair's tiles: two boxes
// of 8 M agents, 1.8 M records a pair, 219 us, now 39; of 40 M agents, 9 M records
// a pair, 328, now 78.)
constexpr u32 kGroupMin = 256;

// A pair of more slots than this, and than twice a block's share of all slots, is
// a big one whatever its message holds (a population that shrank): one block that
// looks all of them up, 2.5 us for each 1,024, would be the launch's length.  Two
// messages of some 5 K records against 450 K slots each: 1250 -> 104 us an
// iteration, against 22 K slots 108 -> 81, 11 K 80 (with the line at 8,192: 84).
// 8 M agents in 64 boxes, 26 K slots a pair, 668 (690 without the share).
constexpr u32 kBlockSlots = 16384;

// Bits beside the pair in a tile's word (pairs are below 2^29): of a pair whose
// tiles' sums the encode keeps, and a tile the match added.  In the word, so that
// the encode need not hold the pair's counts over a tile for them (34.6 against
// 37.3 us at 1 M agents).
constexpr u32 kLarge = 1u << 31, kAdded = 1u << 30, kPairMask = kAdded - 1u;

// Per-pair facts, one 64-byte line.
struct __align__(16) TilePair {
  u64 g_lo;   // first record of the message (pair_off)
  u64 ro;     // first slot of the sender reference (ref_off)
  u64 w_off;  // the message's slab
  u32 r, m;   // slots (0 when sent raw), records
  u32 unit0;  // first tile of the pair
  u32 nst, nnu;  // slot tiles, new-record units
  u32 item0;  // first match item
  u32 big0;   // first bigmatch item
  u32 nbig;   // bigmatch items
  u32 mode;   // XOR or raw
  u32 fits;   // the receiver's reference is the one the message refers to (slots, header)
};
static_assert(sizeof(TilePair) == 64, "one line per pair");

// Device scalars of one call (TS_OK: the setup accepted it; TS_EXTRA: tiles the
// match added behind the TS_UNITS planned ones).
enum { TS_UNITS = 0, TS_ITEMS, TS_BIG, TS_SMALL, TS_SHIFT, TS_TICKET_MATCH, TS_TICKET_BIG,
       TS_OK, TS_EXTRA, TS_COUNT };

struct TileArgs {
  EncArgs E;
  DecArgs D;
  TilePair* pair;
  u32* unit_pair;       // pair of each tile, and kLarge, kAdded
  u32 unit_cap;         // tiles there is room for
  u32* unit_first;      // [P] first tile of each pair
  u64* setup_state;     // look-back states of the setup (zero between calls)
  u32* setup_ticket;
  u64 limit_ns;         // of a wait
  u32* item_pair;       // pair of each match item
  u32* big_pair;        // pair of each bigmatch item
  u32* small_pair;      // pairs matched by one warp
  u32 warps;            // resident warps of a launch
  u32 warp_pair;        // slots and records of a pair matched by one warp, at most
  u32* before;          // matched slots before each slot tile (bigmatch: first, in it)
  u32* bytes;           // payload bytes of each tile
  u32* group;           // payload bytes of each kTileGroup tiles (of pairs above kGroupMin)
  u64* place;           // payload bytes of the pair before each tile
  u64* tot;             // [P * PT_COUNT] matched records, XOR and residual bytes
  u32* done;            // [P] matched tiles of a big pair
  u32* built;           // [P] indexed tiles of a big pair
  u32* unsorted;        // [P] a big pair whose message ids do not ascend
  u32* bits;            // taken records of big pairs: word (g_lo >> 5) + p of pair p
  u32* new_idx;         // new records of each pair in message order, from g_lo
  uint8_t* scratch;     // arena for the packed payload
  u32* scal;            // TS_*
  u64 P;
};

// PT_EXTRA: first added tile (behind TS_UNITS) | their number << 32
enum { PT_MATCHED = 0, PT_XOR = 1, PT_RES = 2, PT_EXTRA = 3, PT_COUNT = 4 };

// ---------------- setup ----------------

struct Facts {
  u64 r, m, rr, r_full, slab;
  bool raw;
  u64 units, items, big, small;
};

// log2 of the tiles' entries.
__device__ __forceinline__ u32 tile_shift(const TileArgs& A) {
  const u64 E = A.E.pair_off[A.P], R = A.E.ref_off ? A.E.ref_off[A.P] : 0;
  const u64 most = E > R ? E : R;
  u32 s = kMaxShift;
  while (s > kMinShift && (most >> s) < kTilesPerWarp * (u64)A.warps) --s;
  return s;
}

__device__ __forceinline__ u64 tiles(u64 entries, u32 shift) {
  return (entries + (1ull << shift) - 1ull) >> shift;
}

__device__ __forceinline__ Facts facts_of(const TileArgs& A, u64 p, int mode, u32 shift,
                                          u64 all_slots) {
  Facts f;
  f.m = A.E.pair_off[p + 1] - A.E.pair_off[p];
  f.r_full = A.E.ref_off ? A.E.ref_off[p + 1] - A.E.ref_off[p] : 0;
  f.raw = mode == TERA_MODE_RAW || A.E.reset[p];
  f.r = f.raw ? 0 : f.r_full;
  f.rr = A.D.ref_off ? A.D.ref_off[p + 1] - A.D.ref_off[p] : 0;
  f.slab = round16((u64)kHdrBytes + 4 * (f.r_full + f.m) + (u64)kRecBytes * f.m);
  const u64 sure = f.m > f.r ? f.m - f.r : 0;
  u64 nnu = tiles(sure, shift) + ceil_div(tiles(f.m, shift), kNewShare);
  // a pair without entries whose receiver holds a reference still goes
  // through the decode's header check
  if (f.r == 0 && f.m == 0 && f.rr != 0) nnu = 1;
  f.units = tiles(f.r, shift) + nnu;
  const bool big = f.m > kTableMax ||
                   (f.r > kBlockSlots && f.r * (A.warps / (kT / 32)) > 2 * all_slots);
  f.small = f.r + f.m != 0 && f.r <= A.warp_pair && f.m <= A.warp_pair;
  f.items = big ? ceil_div(f.m, kBigTile) : (f.r + f.m != 0 && !f.small ? 1 : 0);
  f.big = big ? ceil_div(f.m, kBigTile) + ceil_div(f.r, kBigTile) : 0;
  return f;
}

// The header check of the receiver's reference of pair p (rr records).
__device__ __forceinline__ bool recv_header_ok(const DecArgs& D, u64 p, u64 rr) {
  const u64* rh = reinterpret_cast<const u64*>(D.ref + (D.ref_off[p] + p) * kRecBytes);
  return (u32)rh[0] == kTaioMagic && (u32)rh[1] == D.class_id && (u32)(rh[1] >> 32) == (u32)p &&
         rh[2] == rr;
}

constexpr int kSetupT = 1024;

// out[i] = pair of item i for the items [lo, lo + n) of the block's pairs,
// first[k] (k < np) the first item of pair p0 + k counted from lo (first[np] = n).
__device__ __forceinline__ void fill_map(u32* __restrict__ out, u64 lo, u32 n, u64 cap,
                                         const u32* first, u32 np, u32 p0) {
  for (u32 i = threadIdx.x; i < n && lo + i < cap; i += kSetupT)
    out[lo + i] = p0 + upper_pair(first, 0u, np, (u64)i);
}

// One launch, kSetupT pairs a block: the pairs' facts, then their places in the
// slabs and lists by a block scan and a look-back over the blocks (four chains:
// slab bytes, tiles, match items and warp pairs in the halves of a word, items
// of big pairs).  The last block checks the capacities and writes the lists'
// lengths, all zero when a capacity is exceeded or any block's wait was cut short
// (its pairs' lines and list entries are then not written, and no launch may
// index by them).  Nothing of the caller's but the offsets is written here: the
// verdict is known at the end only, and a refused call leaves messages,
// references, reset marks and totals as they were.
__global__ void __launch_bounds__(kSetupT)
    tiles_setup_kernel(TileArgs A, int mode, u64* __restrict__ wire_off, u64 wire_cap, u64 rec_cap,
                       u64 recv_cap, u64 unit_cap, u64 item_cap, u64 big_cap, u32* epoch) {
  chain_begin();
  __shared__ U64x2 sm2[33];
  __shared__ u32 first[3][kSetupT];
  __shared__ u64 s_pre[4];
  __shared__ u32 s_block, s_fine;
  if (threadIdx.x == 0) {
    s_block = gridDim.x > 1 ? atomicAdd(A.setup_ticket, 1u) : 0u;
    s_fine = 1;
  }
  const u32 shift = tile_shift(A);
  const u64 P = A.P, E = A.E.pair_off[P];
  const u64 rmax = A.E.ref_off ? A.E.ref_off[P] : 0, dmax = A.D.ref_off ? A.D.ref_off[P] : 0;
  const u64 big = E > rmax ? (E > dmax ? E : dmax) : (rmax > dmax ? rmax : dmax);
  const bool abort = big > rec_cap || E + P > recv_cap;
  __syncthreads();
  const u32 block = s_block;
  const u64 p = (u64)block * kSetupT + threadIdx.x;
  Facts f{};
  bool recv_ok = true;
  if (p < P) {
    f = facts_of(A, p, mode, shift, rmax);
    if (!f.raw && A.D.ref && !abort) recv_ok = recv_header_ok(A.D, p, f.rr);
  }
  U64x2 ta, tb;
  const U64x2 ea = block_excl_scan2(U64x2{f.slab, f.units}, sm2, &ta);
  const U64x2 eb = block_excl_scan2(U64x2{f.items | (f.small << 32), f.big}, sm2, &tb);
  first[0][threadIdx.x] = (u32)eb.a;
  first[1][threadIdx.x] = (u32)(eb.a >> 32);
  first[2][threadIdx.x] = (u32)eb.b;
  if (threadIdx.x < 128) {  // a warp a chain
    const u32 c = threadIdx.x >> 5;
    const u64 own = c == 0 ? ta.a : (c == 1 ? ta.b : (c == 2 ? tb.a : tb.b));
    u64 pre = 0;
    if (gridDim.x > 1 && !lb_warp_sum(A.setup_state + (u64)c * gridDim.x, block, own, A.E.st, A.limit_ns,
                                      nullptr, &pre) &&
        (threadIdx.x & 31) == 0)
      s_fine = 0;
    if ((threadIdx.x & 31) == 0) s_pre[c] = pre;
  }
  __syncthreads();
  const bool fine = s_fine != 0;
  const U64x2 carry_a{s_pre[0], s_pre[1]}, carry_b{s_pre[2], s_pre[3]};
  if (fine && p < P) {
    const u64 w = carry_a.a + ea.a, g_lo = A.E.pair_off[p];
    wire_off[p] = w;
    if (A.D.recv_off) A.D.recv_off[p] = g_lo;  // receive buffers sized by the record counts
    if (!abort) {
      TilePair x;
      x.g_lo = g_lo;
      x.ro = A.E.ref_off ? A.E.ref_off[p] : 0;
      x.w_off = w;
      x.r = (u32)f.r;
      x.m = (u32)f.m;
      x.unit0 = (u32)(carry_a.b + ea.b);
      x.nst = (u32)tiles(f.r, shift);
      x.nnu = (u32)f.units - x.nst;
      x.item0 = (u32)carry_b.a + (u32)eb.a;
      x.big0 = (u32)(carry_b.b + eb.b);
      x.nbig = (u32)f.big;
      x.mode = f.raw ? TERA_MODE_RAW : TERA_MODE_XOR;
      x.fits = f.raw || (f.r == (A.D.ref ? f.rr : 0) && recv_ok) ? 1u : 0u;
      A.pair[p] = x;
      ulonglong2* tot = reinterpret_cast<ulonglong2*>(A.tot + p * PT_COUNT);
      tot[0] = make_ulonglong2(0, 0);
      tot[1] = make_ulonglong2(0, 0);
      A.done[p] = 0;
      A.built[p] = 0;
      A.unsorted[p] = 0;
      A.unit_first[p] = x.unit0;
    }
  }
  __syncthreads();
  if (fine && !abort) {
    const u64 left = P - (u64)block * kSetupT;
    const u32 np = (u32)(left < (u64)kSetupT ? left : (u64)kSetupT), p0 = block * kSetupT;
    fill_map(A.item_pair, carry_b.a & 0xFFFFFFFFull, (u32)tb.a, item_cap, first[0], np, p0);
    fill_map(A.small_pair, carry_b.a >> 32, (u32)(tb.a >> 32), P, first[1], np, p0);
    fill_map(A.big_pair, carry_b.b, (u32)tb.b, big_cap, first[2], np, p0);
  }
  if (block != gridDim.x - 1) return;
  // the words of the blocks between the first, which never waits, and this one:
  // a block that gave up has let the blocks after it go on
  bool gone = !fine;
  const u32 between = gridDim.x > 2 ? gridDim.x - 2 : 0;
  for (u32 i = threadIdx.x; i < 4 * between; i += kSetupT) {
    const u64* word = A.setup_state + (u64)(i / between) * gridDim.x + 1 + i % between;
    LbWait wait{A.limit_ns, nullptr};
    u64 state;
    while ((state = lb_get(word) >> kLbShift) < kLbSum && !wait.over(A.E.st)) {
    }
    gone |= state != kLbSum;
  }
  const bool late = __syncthreads_or(gone) != 0;
  if (threadIdx.x == 0) {
    const u32 ep = *epoch + 1u;
    *epoch = ep == 0u ? 1u : ep;
    for (int i = 0; i < TS_COUNT; ++i) A.scal[i] = 0u;
    if (late) return;  // (the timeout is latched) no tile of this call runs
    const U64x2 all_a = carry_a + ta, all_b = carry_b + tb;
    const u64 slabs = all_a.a, units = all_a.b, bigs = all_b.b;
    const u64 n_items = all_b.a & 0xFFFFFFFFull, n_small = all_b.a >> 32;
    wire_off[P] = slabs;
    if (A.D.recv_off) A.D.recv_off[P] = E;
    bool none = abort;
    if (slabs > wire_cap) {
      latch(A.E.st, TERA_ECAPACITY);
      need(A.E.st, slabs);
      none = true;
    }
    if (big > rec_cap) {
      latch(A.E.st, TERA_ECAPACITY);
      need(A.E.st, big);
    }
    if (E + P > recv_cap) {
      latch(A.E.st, TERA_ECAPACITY);
      need(A.E.st, E + P);
    }
    if (units > unit_cap || n_items > item_cap || bigs > big_cap) {
      latch(A.E.st, TERA_ECAPACITY);  // cannot happen: the lists are sized for it
      none = true;
    }
    A.scal[TS_SHIFT] = shift;
    if (none) return;
    A.scal[TS_OK] = 1u;
    A.scal[TS_UNITS] = (u32)units;
    A.scal[TS_ITEMS] = (u32)n_items;
    A.scal[TS_SMALL] = (u32)n_small;
    A.scal[TS_BIG] = (u32)bigs;
  }
}

// ---------------- match ----------------

// The next item of a list, claimed in order: thread 0 claims, every thread
// gets it (~0u when the list is done).  Ends with a block barrier; the caller
// passes another one before the next claim.
__device__ __forceinline__ u32 claim(u32* ticket, u32 n, u32* s_next) {
  if (threadIdx.x == 0) {
    const u32 t = atomicAdd(ticket, 1u);
    *s_next = t < n ? t : ~0u;
  }
  __syncthreads();
  return *s_next;
}

// Word k / 32 of the taken bits of pair p's message (global, big pairs).
__device__ __forceinline__ u32* big_bits(const TileArgs& A, const TilePair& x, u32 p) {
  return A.bits + (x.g_lo >> 5) + p;
}

// The records of pair p whose bit is not set, in message order, into
// new_idx[g_lo ..]; words of 32 records, `bits` in shared (or, G, global) memory.
template <int T, bool G>
__device__ __forceinline__ void new_list(const TileArgs& A, const TilePair& x, const u32* bits,
                                         u32* sm32) {
  // eight words a thread and round in global memory: one block lists a big
  // pair's records, and a round is two barriers
  constexpr u32 kV = G ? 8 : 1;
  const u32 words = (x.m + 31u) / 32u;
  u64 run = 0;
  for (u32 w0 = 0; w0 < words; w0 += T * kV) {  // group-uniform
    const u32 w = w0 + group_thread<T>() * kV;
    u32 free[kV], c = 0;
#pragma unroll
    for (u32 v = 0; v < kV; ++v) {
      free[v] = 0;
      if (w + v < words) {
        const u32 b = G ? __ldcg(bits + w + v) : bits[w + v];
        free[v] = ~b & ((w + v + 1u) * 32u <= x.m ? 0xFFFFFFFFu : (1u << (x.m & 31u)) - 1u);
      }
    }
#pragma unroll
    for (u32 v = 0; v < kV; ++v) c += (u32)__popc(free[v]);
    u32 tot, pos;
    if constexpr (T == 32) {
      const u32 inc = warp_incl_scan<u32>(c);
      pos = inc - c;
      tot = __shfl_sync(0xFFFFFFFFu, inc, 31);
    } else {
      pos = block_excl_scan<u32>(c, sm32, &tot);
    }
    u32* out = A.new_idx + x.g_lo + run + pos;
#pragma unroll
    for (u32 v = 0; v < kV; ++v)
      for (u32 f = free[v]; f; f &= f - 1u) *out++ = (w + v) * 32u + (u32)__ffs(f) - 1u;
    run += tot;
  }
}

// before[unit0 + t] from the matches of each of the pair's nst slot tiles
// (counts in the same places): their exclusive sums.
template <int T>
__device__ __forceinline__ void sum_tiles(const TileArgs& A, const TilePair& x, u32* sm32) {
  constexpr u32 kV = T == 32 ? 1 : 8;
  u32 run = 0;
  for (u32 t0 = 0; t0 < x.nst; t0 += T * kV) {  // group-uniform
    const u32 t = t0 + group_thread<T>() * kV;
    u32 c[kV], sum = 0;
#pragma unroll
    for (u32 v = 0; v < kV; ++v) c[v] = t + v < x.nst ? __ldcg(A.before + x.unit0 + t + v) : 0u;
#pragma unroll
    for (u32 v = 0; v < kV; ++v) sum += c[v];
    u32 tot, ex;
    if constexpr (T == 32) {
      const u32 inc = warp_incl_scan<u32>(sum);
      ex = inc - sum;
      tot = __shfl_sync(0xFFFFFFFFu, inc, 31);
    } else {
      ex = block_excl_scan<u32>(sum, sm32, &tot);
    }
#pragma unroll
    for (u32 v = 0; v < kV; ++v) {
      if (t + v < x.nst) A.before[x.unit0 + t + v] = run + ex;
      ex += c[v];
    }
    run += tot;
  }
}

// The matches of each slot tile of a pair whose slot_src this group wrote, a
// tile per warp.
template <int T>
__device__ __forceinline__ void count_tiles(const TileArgs& A, const TilePair& x, u32 shift) {
  for (u32 t = group_thread<T>() >> 5; t < x.nst; t += T / 32) {
    u32 c = 0;
    for (u32 i = threadIdx.x & 31; i < (1u << shift); i += 32) {
      const u32 j = (t << shift) + i;
      c += j < x.r && __ldcg(A.E.slot_src + x.ro + j) != kNoMatch;
    }
    c = warp_sum(c);
    if ((threadIdx.x & 31) == 0) A.before[x.unit0 + t] = c;
  }
}

// More tiles for the n_new new records of pair p when the planned ones would hold
// many tiles' records each; s_first: a word of the group's shared memory.
template <int T>
__device__ __forceinline__ void add_new_tiles(const TileArgs& A, const TilePair& x, u32 p, u32 n_new,
                                              u32 shift, u32* s_first) {
  const u32 want = (u32)tiles(n_new, shift);
  if (want <= kNewTiles * x.nnu) return;  // group-uniform
  const u32 more = want - x.nnu;
  group_sync<T>();
  if (group_thread<T>() == 0) {
    const u32 first = atomicAdd(A.scal + TS_EXTRA, more);
    A.tot[(u64)p * PT_COUNT + PT_EXTRA] = (u64)first | ((u64)more << 32);
    *s_first = first;
  }
  group_sync<T>();
  const u64 at = (u64)A.scal[TS_UNITS] + *s_first;
  for (u32 i = group_thread<T>(); i < more && at + i < A.unit_cap; i += T)
    A.unit_pair[at + i] = p | kAdded | (more > kGroupMin ? kLarge : 0u);
}

// One tile of a big pair's message: whether its ids ascend (up to the next
// tile's first), and its taken bits cleared.
__device__ __forceinline__ void big_check(const TileArgs& A, const TilePair& x, u32 p, u32 tile) {
  const u32 k0 = tile * kBigTile;
  if (threadIdx.x < kBigTile / 32) {
    const u32 w = k0 / 32 + threadIdx.x;
    if (w < (x.m + 31u) / 32u) big_bits(A, x, p)[w] = 0u;
  }
  u64 a[kIlp], b[kIlp];
#pragma unroll
  for (u32 i = 0; i < kIlp; ++i) {
    const u32 k = k0 + i * kT + threadIdx.x;
    a[i] = k + 1 < x.m ? msg_id(A.E, p, x.g_lo + k) : 0;
    b[i] = k + 1 < x.m ? msg_id(A.E, p, x.g_lo + k + 1) : 1;
  }
  bool bad = false;
#pragma unroll
  for (u32 i = 0; i < kIlp; ++i) bad |= !(a[i] < b[i]);
  if (bad) A.unsorted[p] = 1u;
}

// One tile of message ids of a big pair into its hash segment (as the
// persistent launch does).
__device__ __forceinline__ void big_build(const TileArgs& A, const TilePair& x, u32 p, u32 tile,
                                          u32 epoch) {
  const EncArgs& E = A.E;
  const u64 base = seg_base(x.g_lo, p), size = seg_size(x.m);
  const u32 k0 = tile * kBigTile;
  u64 id[kIlp], at[kIlp], cur[kIlp], prev[kIlp];
  bool live[kIlp];
#pragma unroll
  for (u32 i = 0; i < kIlp; ++i) {
    const u32 k = k0 + i * kT + threadIdx.x;
    live[i] = k < x.m;
    id[i] = live[i] ? msg_id(E, p, x.g_lo + k) : 0;
  }
#pragma unroll
  for (u32 i = 0; i < kIlp; ++i) {
    at[i] = seg_start(id[i], size);
    cur[i] = live[i] ? __ldcg(&E.seg[base + at[i]].a) : 0;
  }
#pragma unroll
  for (u32 i = 0; i < kIlp; ++i) {
    const u32 k = k0 + i * kT + threadIdx.x;
    const bool empty = live[i] && (u32)(cur[i] >> 32) != epoch;
    prev[i] = empty ? atomicCAS(&E.seg[base + at[i]].a, cur[i], ((u64)epoch << 32) | k) : ~0ull;
  }
#pragma unroll
  for (u32 i = 0; i < kIlp; ++i) {
    if (!live[i]) continue;
    const u32 k = k0 + i * kT + threadIdx.x;
    if ((u32)(cur[i] >> 32) != epoch && prev[i] == cur[i]) {
      E.seg[base + at[i]].b = id[i];
    } else {  // taken in this iteration: continue along the probe sequence
      seg_insert_from<true>(E.seg, base, size, id[i], ((u64)epoch << 32) | k, epoch,
                            at[i] + 1 == size ? 0 : at[i] + 1);
    }
  }
}

// Shared memory of a match by the whole block (four blocks per SM) and of one
// by a warp, an eighth of it: message ids, 8 bytes each, then, when they are in
// no order, a hash table of two 4-byte entries per id; the taken bits behind.
constexpr u32 kMatchArea = 50176;
constexpr u32 kIdsMax = kMatchArea / 8;     // ids that fit
constexpr u32 kHashMax = kMatchArea / 16;   // ids that fit beside their table
constexpr size_t kMatchSmem = kMatchArea + (kTableMax + 1) / 8 + 16;
constexpr u32 kWarpArea = 16 * kWarpPair;
static_assert(kMatchArea >= 4 * (kTableMax + 1), "the persistent launch's table fits");
static_assert(kMatchArea >= 8 * (2 * kIlp * kT + 2 * kWinSlack), "its id window fits");
static_assert(8 * (kWarpArea + kWarpPair / 8) <= kMatchSmem, "eight warps' shares fit");

// Every slot of pair p looked up among its message ids, held in shared memory:
// bisected when they ascend, else by a hash table.  Bits mark the taken
// records; returns this thread's match count.  (Against the message's ids in
// global memory, a window or a fingerprint check at a time: 266 -> 130 us for
// 5.9 M records in no order, 264 -> 179 for 16.6 M ascending.)
template <int T>
__device__ __forceinline__ u32 match_ids(const TileArgs& A, const TilePair& x, u32 p, bool ascending,
                                         const u64* ids, u32* tbl, u32* bits) {
  const EncArgs& E = A.E;
  const u32 m = x.m, size = 2 * m;
  for (u32 i = group_thread<T>(); i < (m + 31u) / 32u; i += T) bits[i] = 0u;
  if (!ascending) {
    for (u32 i = group_thread<T>(); i < size; i += T) tbl[i] = 0u;
    group_sync<T>();
    for (u32 k = group_thread<T>(); k < m; k += T) {
      const u64 id = ids[k];
      u32 at = (u32)seg_start(id, size);
      for (u32 probe = 0; probe < size; ++probe) {
        const u32 old = atomicCAS(tbl + at, 0u, k + 1u);
        if (old == 0u) break;
        if (ids[old - 1u] == id) {
          latch(E.st, TERA_EINVAL);  // ids must be unique within a message
          break;
        }
        at = at + 1u == size ? 0u : at + 1u;
      }
    }
  }
  group_sync<T>();
  u32 found = 0;
  for (u32 j0 = 0; j0 < x.r; j0 += T * kIlp) {  // group-uniform
    u64 id[kIlp];
    u32 k[kIlp];
#pragma unroll
    for (u32 i = 0; i < kIlp; ++i) {
      const u32 j = j0 + i * T + group_thread<T>();
      id[i] = j < x.r ? ref_id(E, p, x.ro, j) : 0;
      k[i] = kNoMatch;
    }
    if (m == 0) {
      // nothing to match
    } else if (ascending) {
      // the kIlp bisections step together, so that their reads overlap
      u32 lo[kIlp], len = m;
#pragma unroll
      for (u32 i = 0; i < kIlp; ++i) lo[i] = 0;
      while (len > 1) {  // the last id not above the slot's is in [lo, lo + len)
        const u32 half = len >> 1;
#pragma unroll
        for (u32 i = 0; i < kIlp; ++i) lo[i] = ids[lo[i] + half] <= id[i] ? lo[i] + half : lo[i];
        len -= half;
      }
#pragma unroll
      for (u32 i = 0; i < kIlp; ++i) k[i] = ids[lo[i]] == id[i] ? lo[i] : kNoMatch;
    } else {
#pragma unroll
      for (u32 i = 0; i < kIlp; ++i) {
        u32 at = (u32)seg_start(id[i], size);
        for (u32 probe = 0; probe < size; ++probe) {
          const u32 e = tbl[at];
          if (e == 0u) break;
          if (ids[e - 1u] == id[i]) {
            k[i] = e - 1u;
            break;
          }
          at = at + 1u == size ? 0u : at + 1u;
        }
      }
    }
#pragma unroll
    for (u32 i = 0; i < kIlp; ++i) {
      const u32 j = j0 + i * T + group_thread<T>();
      if (j >= x.r) continue;
      if (k[i] != kNoMatch) {
        const u32 bit = 1u << (k[i] & 31u);
        if (atomicOr(bits + (k[i] >> 5), bit) & bit) {
          latch(E.st, TERA_EINVAL);  // a second slot with the same id: that slot is a hole
          k[i] = kNoMatch;
        }
      }
      found += k[i] != kNoMatch;
      E.slot_src[x.ro + j] = k[i] != kNoMatch ? (u32)x.g_lo + k[i] : kNoMatch;
    }
  }
  return found;
}

// The matches of a pair of at most kTableMax records (T = 32: kWarpPair), by a
// group of T threads: slot_src, the new records, the matches before each slot
// tile and in all.
template <int T>
__device__ __forceinline__ void match_pair(const TileArgs& A, const TilePair& x, u32 p, u32 shift,
                                           uint8_t* area, u32* bits, u32* s_cnt, u32* sm32) {
  if (group_thread<T>() == 0) *s_cnt = 0;
  u64* ids = reinterpret_cast<u64*>(area);
  bool ascending, held = true;
  if (T == 32 || x.m <= kIdsMax) {
    for (u32 k0 = 0; k0 < x.m; k0 += 8 * T) {
      u64 v[8];
#pragma unroll
      for (u32 i = 0; i < 8; ++i) {
        const u32 k = k0 + i * T + group_thread<T>();
        v[i] = k < x.m ? msg_id(A.E, p, x.g_lo + k) : 0;
      }
#pragma unroll
      for (u32 i = 0; i < 8; ++i) {
        const u32 k = k0 + i * T + group_thread<T>();
        if (k < x.m) ids[k] = v[i];
      }
    }
    group_sync<T>();
    bool bad = false;
    for (u32 k = group_thread<T>(); k + 1 < x.m; k += T) bad |= !(ids[k] < ids[k + 1]);
    ascending = !group_any<T>(bad);
    held = T == 32 || ascending || x.m <= kHashMax;
  } else {
    group_sync<T>();
    ascending = ids_ascending<T>(A.E, p, x.m);
    held = false;
  }
  u32 c = 0;
  if (held) {
    c = match_ids<T>(A, x, p, ascending, ids, reinterpret_cast<u32*>(ids + x.m), bits);
  } else if constexpr (T != 32) {
    SmemTable tb{reinterpret_cast<unsigned short*>(area), 0u, bits};
    u32 size = 32;
    while (size < 2 * x.m) size <<= 1;
    tb.mask = size - 1;
    if (ascending) {
      if (x.r) c = sorted_match<T>(A.E, p, x.m, x.r, tb, ids);
    } else {
      smem_build<T>(A.E, p, x.m, tb);  // also finds an id that occurs twice
      group_sync<T>();
      if (x.r) c = smem_match<T>(A.E, p, x.r, tb);
    }
  }
  if (x.r == 0) return;
  c = warp_sum(c);
  if ((threadIdx.x & 31) == 0 && c) atomicAdd(s_cnt, c);
  group_sync<T>();
  const u32 matched = *s_cnt;
  if (group_thread<T>() == 0) A.tot[(u64)p * PT_COUNT + PT_MATCHED] = matched;
  if (matched < x.m) new_list<T, false>(A, x, bits, sm32);
  if (x.nst == 1) {
    if (group_thread<T>() == 0) A.before[x.unit0] = 0u;
  } else {
    __threadfence_block();
    group_sync<T>();
    count_tiles<T>(A, x, shift);
    __threadfence_block();
    group_sync<T>();
    sum_tiles<T>(A, x, sm32);
  }
  add_new_tiles<T>(A, x, p, x.m - matched, shift, s_cnt);
}

// The pair of every tile (unit_pair), which the launches after this one read:
// each warp of the launch takes a run of tiles, finds the first one's pair and
// walks on from it.
__device__ __forceinline__ void map_tiles(const TileArgs& A) {
  const u32 lane = threadIdx.x & 31;
  const u64 units = A.scal[TS_UNITS], warps = (u64)gridDim.x * (kT / 32);
  const u64 run = (ceil_div(units, warps) + 31) & ~31ull;
  const u64 a = ((u64)blockIdx.x * (kT / 32) + (threadIdx.x >> 5)) * run;
  const u64 b = a + run < units ? a + run : units;
  if (a >= b) return;
  // the last pair whose first tile is a or before it, 32 probes at a time
  u32 lo = 0, hi = (u32)A.P - 1;
  while (lo < hi) {
    const u32 step = (hi - lo + 32) / 32, at = lo + lane * step;
    const u32 bal = __ballot_sync(0xFFFFFFFFu, at <= hi && A.unit_first[at] <= a);
    const u32 k = 31u - (u32)__clz(bal | 1u);
    const u32 next = lo + k * step;
    hi = next + step - 1u < hi ? next + step - 1u : hi;
    lo = next;
    if (step == 1u) break;
  }
  u32 p = lo;
  for (u64 u = a + lane; u < b; u += 32) {
    u32 end = (u32)units;
    while (p + 1 < (u32)A.P && (end = A.unit_first[p + 1]) <= u) {
      ++p;
      end = (u32)units;
    }
    A.unit_pair[u] = p | (end - A.unit_first[p] > kGroupMin ? kLarge : 0u);
  }
}

// The pairs of the match list, a block each, claimed one by one; then the
// small ones, a warp each.
__global__ void __launch_bounds__(kT, kPerSm) codec_match_kernel(TileArgs A) {
  chain_begin();
  extern __shared__ __align__(16) uint8_t dyn[];
  __shared__ u32 sm32[33];
  __shared__ u32 s_next, s_cnt[kT / 32];
  const u32 n = A.scal[TS_ITEMS], n_small = A.scal[TS_SMALL], shift = A.scal[TS_SHIFT];
  if (blockIdx.x == 0) {  // the setup's states, zero for the next call
    const u32 blocks = (u32)((A.P + kSetupT - 1) / kSetupT);
    for (u32 i = threadIdx.x; i < 4 * blocks; i += kT) A.setup_state[i] = 0;
    if (threadIdx.x == 0) *A.setup_ticket = 0;
  }
  for (u32 i = blockIdx.x * kT + threadIdx.x; i <= A.unit_cap / kTileGroup; i += gridDim.x * kT)
    A.group[i] = 0u;
  map_tiles(A);
  if (n) {
    for (;;) {
      const u32 it = claim(A.scal + TS_TICKET_MATCH, n, &s_next);
      if (it == ~0u) break;
      const u32 p = A.item_pair[it];
      const TilePair x = A.pair[p];
      if (x.nbig) big_check(A, x, p, it - x.item0);
      else match_pair<kT>(A, x, p, shift, dyn, reinterpret_cast<u32*>(dyn + kMatchArea), s_cnt, sm32);
      __syncthreads();
    }
  }
  const u32 warp = threadIdx.x >> 5;
  uint8_t* share = dyn + warp * (kWarpArea + kWarpPair / 8);
  for (u32 i = blockIdx.x * (kT / 32) + warp; i < n_small; i += gridDim.x * (kT / 32)) {
    const u32 p = A.small_pair[i];
    const TilePair x = A.pair[p];
    match_pair<32>(A, x, p, shift, share, reinterpret_cast<u32*>(share + kWarpArea), s_cnt + warp,
                   nullptr);
    __syncwarp();
  }
}

// First message record of pair p in [lo, hi) whose id is not below v (ids
// ascending), by one warp, 32 probes at a time.
__device__ __forceinline__ u32 warp_lower_bound(const EncArgs& E, u32 p, u64 g_lo, u32 lo, u32 hi,
                                                u64 v) {
  const u32 lane = threadIdx.x & 31;
  while (lo < hi) {
    const u64 len = hi - lo;
    const bool less = msg_id(E, p, g_lo + lo + (u32)(len * lane / 32)) < v;
    const u32 c = (u32)__popc(__ballot_sync(0xFFFFFFFFu, less));
    const u32 base = lo;
    if (c < 32u) hi = base + (u32)(len * c / 32);
    if (c > 0u) lo = base + (u32)(len * (c - 1u) / 32) + 1u;
  }
  return lo;
}

// Ids of a big pair's window in shared memory: what 1024 slots of an ascending
// reference span while fewer than three in four of the records between them
// are someone else's.
constexpr u32 kBigWindow = 4096;

// The slots of an item of a big pair whose message ids ascend (live: ids id):
// the span of message records from the item's first to its last id is found by
// two warps and brought into shared memory when it fits, and every id in it
// bisected there; other ids are bisected over the whole message.  (6.5 M
// records, 1.1 M of them in one pair: 615 us of indexing and lookups in global
// hash segments before, 295 with the check and this.)
__device__ __forceinline__ void big_sorted(const TileArgs& A, const TilePair& x, u32 p, u32 j0,
                                           const u64* id, const bool* live, u64* window,
                                           u32* s_span, u32* k) {
  const EncArgs& E = A.E;
  const u32 j1 = x.r - j0 < kBigTile ? x.r - 1u : j0 + kBigTile - 1u;
  const u64 first = ref_id(E, p, x.ro, j0), last = ref_id(E, p, x.ro, j1);
  const u32 warp = threadIdx.x >> 5;
  if (warp < 2) {
    const u32 at = warp_lower_bound(E, p, x.g_lo, 0, x.m, warp == 0 ? first : last);
    if ((threadIdx.x & 31) == 0) s_span[warp] = at;
  }
  __syncthreads();
  const u32 lo = s_span[0], hi = s_span[1] + 1u < x.m ? s_span[1] + 1u : x.m;
  const bool in = first <= last && lo < hi && hi - lo <= kBigWindow;  // block-uniform
  if (in)
    for (u32 i = threadIdx.x; i < hi - lo; i += kT) window[i] = msg_id(E, p, x.g_lo + lo + i);
  __syncthreads();
#pragma unroll
  for (u32 i = 0; i < kIlp; ++i) {
    k[i] = kNoMatch;
    if (!live[i]) continue;
    if (in && id[i] >= first && id[i] <= last) {
      u32 a = 0, b = hi - lo;
      while (a < b) {
        const u32 mid = (a + b) >> 1;
        if (window[mid] < id[i]) a = mid + 1;
        else b = mid;
      }
      if (a < hi - lo && window[a] == id[i]) k[i] = lo + a;
    } else {
      u32 a = 0, b = x.m;
      while (a < b) {
        const u32 mid = a + ((b - a) >> 1);
        if (msg_id(E, p, x.g_lo + mid) < id[i]) a = mid + 1;
        else b = mid;
      }
      if (a < x.m && msg_id(E, p, x.g_lo + a) == id[i]) k[i] = a;
    }
  }
}

// The same in the pair's hash segment.
__device__ __forceinline__ void big_lookup(const TileArgs& A, const TilePair& x, u32 p,
                                           const u64* id, const bool* live, u32 epoch, u32* k) {
  const EncArgs& E = A.E;
  const u64 base = seg_base(x.g_lo, p), size = seg_size(x.m);
  u64 at[kIlp];
  U64x2 e[kIlp];
#pragma unroll
  for (u32 i = 0; i < kIlp; ++i) {
    at[i] = seg_start(id[i], size);
    e[i] = live[i] ? ldx<true>(E.seg + base + at[i]) : U64x2{0, 0};
  }
#pragma unroll
  for (u32 i = 0; i < kIlp; ++i) {
    k[i] = kNoMatch;
    if (!live[i] || (u32)(e[i].a >> 32) != epoch) continue;
    if (e[i].b == id[i]) {
      k[i] = (u32)e[i].a;
    } else {
      k[i] = seg_lookup_from<true>(E.seg, epoch, base, size, 0, id[i],
                                   at[i] + 1 == size ? 0 : at[i] + 1);
    }
  }
}

// The big pairs' items, claimed in order: a pair's message tiles (indexed when
// its ids do not ascend), then its slot tiles, which wait until the tiles
// before them are indexed (claimed earlier, so by running blocks; at most the
// context's limit, then TERA_ETIMEOUT and no match).  The taken records are marked; the
// block that finishes a pair's last tile lists its new records.
__global__ void __launch_bounds__(kT, kPerSm) codec_bigmatch_kernel(TileArgs A) {
  chain_begin();
  extern __shared__ __align__(16) uint8_t dyn[];
  __shared__ u32 sm32[33];
  __shared__ u32 s_next, s_last, s_hits[kBigTile / 32], s_span[2];
  static_assert(kBigTile == 1024, "one warp adds an item's hits up");
  const u32 n = A.scal[TS_BIG];
  if (n == 0) return;
  const u32 shift = A.scal[TS_SHIFT];
  const EncArgs& E = A.E;
  const u32 epoch = *E.epoch;
  for (;;) {
    const u32 it = claim(A.scal + TS_TICKET_BIG, n, &s_next);
    if (it == ~0u) return;
    const u32 p = A.big_pair[it];
    const TilePair x = A.pair[p];
    const u32 nbuild = (x.m + kBigTile - 1u) / kBigTile;
    const u32 tile = it - x.big0;
    const bool sorted = A.unsorted[p] == 0u;
    if (tile < nbuild) {
      if (!sorted) {
        big_build(A, x, p, tile, epoch);
        __threadfence();
      }
      __syncthreads();
      if (!sorted && threadIdx.x == 0) atomicAdd(A.built + p, 1u);
      continue;
    }
    const u32 j0 = (tile - nbuild) * kBigTile;
    u32* bits = big_bits(A, x, p);
    u64 id[kIlp];
    bool live[kIlp];
    u32 k[kIlp];
#pragma unroll
    for (u32 i = 0; i < kIlp; ++i) {
      const u32 j = j0 + i * kT + threadIdx.x;
      live[i] = j < x.r;
      id[i] = live[i] ? ref_id(E, p, x.ro, j) : 0;
    }
    if (sorted) {
      big_sorted(A, x, p, j0, id, live, reinterpret_cast<u64*>(dyn), s_span, k);
    } else {
      if (threadIdx.x == 0) {
        s_span[0] = 1u;
        LbWait wait{A.limit_ns, nullptr};
        u32 v;
        for (;;) {
          asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(A.built + p) : "memory");
          if (v >= nbuild) break;
          if (wait.over(E.st)) {
            s_span[0] = 0u;
            break;
          }
        }
      }
      __syncthreads();
      if (s_span[0]) {
        big_lookup(A, x, p, id, live, epoch, k);
      } else {
#pragma unroll
        for (u32 i = 0; i < kIlp; ++i) k[i] = kNoMatch;
      }
    }
    u32 old[kIlp];
#pragma unroll
    for (u32 i = 0; i < kIlp; ++i)
      old[i] = k[i] != kNoMatch ? atomicOr(bits + (k[i] >> 5), 1u << (k[i] & 31u)) : 0u;
#pragma unroll
    for (u32 i = 0; i < kIlp; ++i) {
      if (!live[i]) continue;
      if (k[i] != kNoMatch && ((old[i] >> (k[i] & 31u)) & 1u)) {
        latch(E.st, TERA_EINVAL);  // a second slot with the same id: that slot is a hole
        k[i] = kNoMatch;
      }
      E.slot_src[x.ro + j0 + i * kT + threadIdx.x] =
          k[i] != kNoMatch ? (u32)(x.g_lo + k[i]) : kNoMatch;
    }
    // the matches of the slot tiles this item is made of
#pragma unroll
    for (u32 i = 0; i < kIlp; ++i) {
      const u32 hits = __ballot_sync(0xFFFFFFFFu, live[i] && k[i] != kNoMatch);
      if ((threadIdx.x & 31) == 0) s_hits[i * (kT / 32) + (threadIdx.x >> 5)] = (u32)__popc(hits);
    }
    __syncthreads();
    if (threadIdx.x < kBigTile / 32) {
      const u32 mine = s_hits[threadIdx.x], per = 1u << (shift - 5);
      const u32 found = warp_sum(mine);
      u32 c = 0;
      if (threadIdx.x < kBigTile >> shift)
        for (u32 i = 0; i < per; ++i) c += s_hits[threadIdx.x * per + i];
      const u32 t = (j0 >> shift) + threadIdx.x;
      if (threadIdx.x < kBigTile >> shift && t < x.nst) A.before[x.unit0 + t] = c;
      if (threadIdx.x == 0 && found)
        atomicAdd(A.tot + (u64)p * PT_COUNT + PT_MATCHED, (u64)found);
    }
    __threadfence();  // the bits before the count of finished tiles
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(A.done + p, 1u) + 1u == x.nbig - nbuild;
    __syncthreads();
    if (s_last) {
      __threadfence();
      new_list<kT, true>(A, x, bits, sm32);
      sum_tiles<kT>(A, x, sm32);
      const u32 matched = (u32)__ldcg(A.tot + (u64)p * PT_COUNT + PT_MATCHED);
      add_new_tiles<kT>(A, x, p, x.m - matched, shift, s_span);
    }
    __syncthreads();
  }
}

// ---------------- sizes of the predictor's forms ----------------

// Predictor: the XOR and residual payload bytes of every slot tile, added up
// per pair (they choose the message mode), and the training samples.  A warp a
// tile, as the steps after it: a block a tile waited at two barriers for its
// slowest records (6.4 M slots: 310 -> 190 us, the copy rate).
__global__ void __launch_bounds__(kT, kPerSm) codec_sizes_kernel(TileArgs A) {
  chain_begin();
  const EncArgs& E = A.E;
  const u32 n = A.scal[TS_UNITS], shift = A.scal[TS_SHIFT];
  const u32 lane = threadIdx.x & 31, stride = gridDim.x * (kT / 32);
  u32 u = blockIdx.x * (kT / 32) + (threadIdx.x >> 5);
  u32 p_next = u < n ? A.unit_pair[u] : 0u;
  for (; u < n; u += stride) {
    const u32 p = p_next & kPairMask;
    if (u + stride < n) p_next = A.unit_pair[u + stride];
    const TilePair x = A.pair[p];
    const u32 tile = u - x.unit0;
    if (tile >= x.nst) continue;
    const u32 lo = tile << shift, hi = x.r - lo < (1u << shift) ? x.r : lo + (1u << shift);
    u32 bx = 0, br = 0;
    u32 g_next = lo + lane < hi ? E.slot_src[x.ro + lo + lane] : kNoMatch;
    for (u32 j = lo + lane; j < hi; j += 32) {
      const u32 g = g_next;
      g_next = j + 32 < hi ? E.slot_src[x.ro + j + 32] : kNoMatch;
      if (E.pr.samples) E.pr.samples[(u64)kSampleFloats * (x.ro + j) + 11] = 0.0f;
      if (g == kNoMatch) continue;
      const Rec R = load_rec(E.ref + (x.ro + p + 1 + j) * kRecBytes);
      const Rec M = load_rec(E.rec + ((u64)g + p + 1) * kRecBytes);
      u32 b = 0;
#pragma unroll
      for (int w = 0; w < 8; ++w) b += sig_bytes(M.w[w] ^ R.w[w]);
      bx += b;
      br += (u32)pred_slot<true>(E, p, j, x.r, x.mode, R, M, b);
    }
    __syncwarp();
    bx = warp_sum(bx);
    br = warp_sum(br);
    if (lane == 0) {
      u64* t = A.tot + (u64)p * PT_COUNT;
      if (bx) atomicAdd(t + PT_XOR, (u64)bx);
      if (br) atomicAdd(t + PT_RES, (u64)br);
    }
  }
}

// The new-record ranks [*lo, *hi) of unit i of a pair's nnu units.
__device__ __forceinline__ void new_range(u32 n_new, u32 nnu, u32 i, u32 shift, u32* lo, u32* hi) {
  u32 per = (n_new + nnu - 1u) / nnu;
  per = (per + (1u << shift) - 1u) >> shift << shift;
  const u64 a = (u64)per * i, b = a + per;
  *lo = a < n_new ? (u32)a : n_new;
  *hi = b < n_new ? (u32)b : n_new;
}

// Message record of new rank i.
__device__ __forceinline__ u64 new_record(const TileArgs& A, const TilePair& x, u32 i) {
  return x.r ? A.new_idx[x.g_lo + i] : i;
}

// ---------------- encode, wire, decode: one warp a tile ----------------
//
// A warp carries a tile in steps of 32 entries; nothing is shared between
// warps, so there are no barriers, and a pair of a few records costs one warp
// one step.  Four lanes hold a record, 16 bytes each, eight records at a time:
// a load or store of the warp then covers whole cache lines (four to eight,
// where a record a lane covers sixteen to thirty-two with every one of its four
// loads, and the L1 is what bounds the kernel), and the lanes' order is the
// order of the payload's words, so one scan over the lanes places them.

constexpr u32 kWarps = kT / 32;
// a warp's payload stage: up to 15 bytes carried from the step before, 32
// records, and what the copies read or clear past the bytes
constexpr u32 kStage = 16 + 32 * kRecBytes + 32;
constexpr u32 kRows = 32 * kRecBytes;  // a step's reference records
constexpr size_t kEncSmem = kWarps * (kStage + 2 * kRows);  // reference and message rows
constexpr size_t kDecSmem = kWarps * (2 * kStage + 2 * kRows);

__device__ __forceinline__ void copy16(void* dst, const void* src) {
  const u32 d = (u32)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" : : "r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void copies_commit() {
  asm volatile("cp.async.commit_group;" : : : "memory");
}
template <int N>
__device__ __forceinline__ void copies_wait() {  // all but the last N groups
  asm volatile("cp.async.wait_group %0;" : : "n"(N) : "memory");
}

// The tiles of the call: those the setup planned, the match's behind them.
__device__ __forceinline__ u32 tile_count(const TileArgs& A) {
  const u32 all = A.scal[TS_UNITS] + A.scal[TS_EXTRA];
  return all < A.unit_cap ? all : A.unit_cap;
}

// What a tile's warp needs of its pair.
struct Tile {
  TilePair x;
  u32 p, local;
  u32 n_new;
};

// A pair's added tiles: the first's place in the list, and how many.  Read where
// they matter only: a slot tile does not wait for them.
struct Added {
  u32 first, n;
};
__device__ __forceinline__ Added added_tiles(const TileArgs& A, u32 p) {
  const u64 extra = A.tot[(u64)p * PT_COUNT + PT_EXTRA];
  return Added{A.scal[TS_UNITS] + (u32)extra, (u32)(extra >> 32)};
}

// word: unit_pair[u].
__device__ __forceinline__ Tile tile_of(const TileArgs& A, u32 u, u32 word) {
  const u32 p = word & kPairMask;
  Tile t;
  t.p = p;
  t.x = A.pair[p];
  t.local = u - t.x.unit0;
  if (word & kAdded) t.local = t.x.nst + t.x.nnu + (u - added_tiles(A, p).first);
  t.n_new = t.x.m - (u32)A.tot[(u64)p * PT_COUNT + PT_MATCHED];
  return t;
}

template <bool PR>
__device__ __forceinline__ u64 message_mode(const TileArgs& A, const Tile& t) {
  if constexpr (PR) {
    const u64* tot = A.tot + (u64)t.p * PT_COUNT;
    if (A.E.pr.params && A.E.pr.allow_residual && t.x.mode == TERA_MODE_XOR &&
        tot[PT_RES] < tot[PT_XOR])
      return kModeResidual;
  }
  return t.x.mode;
}

// Where the records of a pair lie in an arena the size of the receive buffer
// (the receive buffer itself, which holds the payload until the decode, or the
// context's when there is no decode): the tiles' packed payload, each tile's
// from its first record's place.
__device__ __forceinline__ uint8_t* payload_place(const TileArgs& A, const Tile& t, u64 record) {
  return A.scratch + (t.x.g_lo + t.p + 1 + record) * kRecBytes;
}

// Two words of a record, and their significant bytes.
struct Piece {
  u64 a, b;
};
__device__ __forceinline__ Piece load_piece(const uint8_t* rec, u32 q) {
  const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(rec + 16 * q);
  return Piece{v.x, v.y};
}
__device__ __forceinline__ void store_piece(uint8_t* rec, u32 q, const Piece& v) {
  *reinterpret_cast<ulonglong2*>(rec + 16 * q) = make_ulonglong2(v.a, v.b);
}

// Exclusive offsets of four steps' lane counts (each below 2^16 in all), in
// the order step, lane; returns the total.  Two counts a word, so two scans.
__device__ __forceinline__ u32 scan4(const u32 c[4], u32 off[4]) {
  const u32 lo = c[0] | (c[1] << 16), hi = c[2] | (c[3] << 16);
  const u32 il = warp_incl_scan<u32>(lo), ih = warp_incl_scan<u32>(hi);
  const u32 tl = __shfl_sync(0xFFFFFFFFu, il, 31), th = __shfl_sync(0xFFFFFFFFu, ih, 31);
  const u32 t0 = tl & 0xFFFFu, t1 = t0 + (tl >> 16), t2 = t1 + (th & 0xFFFFu);
  off[0] = (il & 0xFFFFu) - c[0];
  off[1] = t0 + (il >> 16) - c[1];
  off[2] = t1 + (ih & 0xFFFFu) - c[2];
  off[3] = t2 + (ih >> 16) - c[3];
  return t2 + (th >> 16);
}

// Payload of the warp's next 32 entries (d: this lane's entry's words, code:
// their lengths, vb bytes in all) behind the *bytes already packed at out:
// whole 16-byte pieces are stored, the rest stays at the start of the stage.
// An entry a lane: neighbouring lanes' bytes are then mostly in different
// words of the stage (with two words of a record a lane the lanes' ORs met in
// the same words: 370 against 275 us on a blob population's 6.5 M records).
__device__ __forceinline__ void pack_step(uint8_t* st, uint8_t* out, const Rec& d, u32 code, u32 vb,
                                          u32* bytes) {
  const u32 lane = threadIdx.x & 31;
  const u32 incl = warp_incl_scan<u32>(vb);
  const u32 total = __shfl_sync(0xFFFFFFFFu, incl, 31);
  if (total == 0) return;
  const u32 fill = *bytes & 15u, end = fill + total;
  for (u32 c = 1 + lane; c < ((end + 15u) >> 4) + 1u; c += 32)
    *reinterpret_cast<uint4*>(st + (c << 4)) = make_uint4(0u, 0u, 0u, 0u);
  __syncwarp();
  u32 o = fill + incl - vb;
#pragma unroll
  for (int w = 0; w < 8; ++w) {
    const u32 L = (code >> (4 * w)) & 0xFu;
    if (__any_sync(0xFFFFFFFFu, L)) {
      stage_or(st, o, d.w[w], L);
      o += L;
    }
  }
  __syncwarp();
  const u32 whole = end >> 4;
  uint8_t* to = out + (*bytes - fill);
  for (u32 c = lane; c < whole; c += 32)
    *reinterpret_cast<uint4*>(to + (c << 4)) = *reinterpret_cast<const uint4*>(st + (c << 4));
  if (whole) {
    const uint4 rest = *reinterpret_cast<const uint4*>(st + (whole << 4));
    __syncwarp();
    if (lane == 0) *reinterpret_cast<uint4*>(st) = rest;
  }
  *bytes += total;
  __syncwarp();
}

// A step's records in shared memory: piece k (16 bytes) of record e at row e,
// place (k + e / 2) mod 4, so that eight lanes reading piece k of eight
// consecutive records meet no bank twice.
__device__ __forceinline__ u32 row_at(u32 e, u32 k) { return e * kRecBytes + (((k + (e >> 1)) & 3u) << 4); }

__device__ __forceinline__ Rec row_rec(const uint8_t* rows, u32 e) {
  Rec r;
#pragma unroll
  for (u32 k = 0; k < 4; ++k) {
    const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(rows + row_at(e, k));
    r.w[2 * k] = v.x;
    r.w[2 * k + 1] = v.y;
  }
  return r;
}

// The step's message records (rows) named by `hits`, in order, to the new
// sender reference from record g on, and their ids to the id column.
__device__ __forceinline__ void store_next(const EncArgs& E, u32 p, u64 g, const uint8_t* rows,
                                           u32 hits, u64 id) {
  const u32 lane = threadIdx.x & 31, q = lane & 3;
  uint8_t* to = E.ref_next + (g + p + 1) * kRecBytes;
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    const u32 e = 8 * s + (lane >> 2);
    if (!(hits >> e & 1u)) continue;
    const u32 k = (u32)__popc(hits & ((1u << e) - 1u));
    if (!in_bounds(E.st, g + k, E.pair_off[p], E.pair_off[p + 1])) continue;
    *reinterpret_cast<ulonglong2*>(to + (u64)k * kRecBytes + 16 * q) =
        *reinterpret_cast<const ulonglong2*>(rows + row_at(e, q));
  }
  if (E.ref_ids_next && (hits >> lane & 1u)) {
    const u64 k = g + (u32)__popc(hits & ((1u << lane) - 1u));
    if (in_bounds(E.st, k, E.pair_off[p], E.pair_off[p + 1])) E.ref_ids_next[k] = id;
  }
}

template <bool PR>
__global__ void __launch_bounds__(kT, kEncPerSm) codec_encode_kernel(TileArgs A) {
  chain_begin();
  extern __shared__ __align__(16) uint8_t dyn[];
  const EncArgs& E = A.E;
  const u32 warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const u32 r8 = lane >> 2, q = lane & 3;  // this lane's record of each eight, and its piece
  uint8_t* st = dyn + warp * (kStage + 2 * kRows);
  uint8_t* rows = st + kStage;
  const u32 n = tile_count(A);
  const u32 shift = A.scal[TS_SHIFT];
  const u32 epoch = *E.epoch;
  const u32 stride = gridDim.x * kWarps;
  u32 u = blockIdx.x * kWarps + warp;
  u32 p_next = u < n ? A.unit_pair[u] : 0u;
  for (; u < n; u += stride) {
    const u32 word = p_next;
    const Tile t = tile_of(A, u, word);
    if (u + stride < n) p_next = A.unit_pair[u + stride];
    const u32 p = t.p;
    u32* codes = reinterpret_cast<u32*>(E.wire + t.x.w_off + kHdrBytes);
    if (lane == 0) *reinterpret_cast<uint4*>(st) = make_uint4(0u, 0u, 0u, 0u);
    __syncwarp();
    u32 bytes = 0;
    uint8_t* out;
    if (t.local < t.x.nst) {
      const u32 j0 = t.local << shift;
      const u32 nj = t.x.r - j0 < (1u << shift) ? t.x.r - j0 : 1u << shift;
      const u32* src = E.slot_src + t.x.ro + j0;
      const uint8_t* ref = E.ref + (t.x.ro + p + 1 + j0) * kRecBytes;
      const uint8_t* rec = E.rec + ((u64)p + 1) * kRecBytes;
      u64 pos = A.before[u];
      out = payload_place(A, t, pos);
      bool residual = false;
      if constexpr (PR) residual = message_mode<PR>(A, t) == kModeResidual;
      // a step's records are asked for before the step before is packed, their
      // places a step earlier still
      const auto request = [&](u32 i0, u32 g) {
        const u32 hits = __ballot_sync(0xFFFFFFFFu, g != kNoMatch);
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          const u32 e = 8 * s + r8, gs = __shfl_sync(0xFFFFFFFFu, g, e);
          if (hits >> e & 1u) {
            copy16(rows + row_at(e, q), ref + (u64)(i0 + e) * kRecBytes + 16 * q);
            copy16(rows + kRows + row_at(e, q), rec + (u64)gs * kRecBytes + 16 * q);
          }
        }
        copies_commit();
        return hits;
      };
      u32 g_next = 32 + lane < nj ? src[32 + lane] : kNoMatch;
      u32 hits = request(0, lane < nj ? src[lane] : kNoMatch);
      for (u32 i0 = 0; i0 < nj; i0 += 32) {
        const u32 g_now = g_next;
        g_next = i0 + 64 + lane < nj ? src[i0 + 64 + lane] : kNoMatch;
        copies_wait<0>();
        __syncwarp();
        const bool hit = hits >> lane & 1u;
        Rec d{};
        u32 code = 0, vb = 0;
        u64 id = 0;
        if (hit) {
          d = row_rec(rows, lane);
          const Rec cur = row_rec(rows + kRows, lane);
          id = cur.w[0];
          const u64* ps = nullptr;
          if constexpr (PR) {
            if (E.pr.hist_next) {
              uint8_t* hn = E.pr.hist_next +
                            kHistBytes * (t.x.g_lo + pos + (u32)__popc(hits & ((1u << lane) - 1u)));
              if (E.pr.hist) {
                const Hist H = load_hist(E.pr.hist + kHistBytes * (t.x.ro + j0 + i0 + lane));
                store_hist_next(hn, &d, &H);
              } else {
                store_hist_next(hn, &d, nullptr);
              }
            }
            if (residual) {
              ps = E.pr.pscr + 4 * (t.x.ro + j0 + i0 + lane);
              if (!ps[3]) ps = nullptr;
            }
          }
#pragma unroll
          for (int w = 0; w < 8; ++w) {
            if (PR && ps && w >= 1 && w <= 3) d.w[w] = zigzag(cur.w[w] - ps[w - 1]);
            else d.w[w] ^= cur.w[w];
          }
        }
        __syncwarp();
        store_next(E, p, t.x.g_lo + pos, rows + kRows, hits, id);
        __syncwarp();  // the rows are read: the next step's may come
        u32 hits_next = 0;
        if (i0 + 32 < nj) hits_next = request(i0 + 32, g_now);
        if (hit) code = rec_code(d, &vb);
        if (i0 + lane < nj && in_bounds(E.st, j0 + i0 + lane, 0, (u64)t.x.r + t.n_new))
          codes[j0 + i0 + lane] = hit ? code : 0xFu;  // 0xF: placeholder
        pack_step(st, out, d, code, vb, &bytes);
        pos += (u32)__popc(hits);
        hits = hits_next;
      }
    } else {
      // new records: rank i's code and new-reference record have known places
      const u64 matched = (u64)t.x.m - t.n_new;
      u32 lo, hi;
      new_range(t.n_new, t.x.nnu + added_tiles(A, p).n, t.local - t.x.nst, shift, &lo, &hi);
      out = payload_place(A, t, matched + lo);
      for (u32 i0 = lo; i0 < hi; i0 += 32) {
        const u32 hits = hi - i0 >= 32 ? 0xFFFFFFFFu : (1u << (hi - i0)) - 1u;
        const u64 k = i0 + lane < hi ? new_record(A, t.x, i0 + lane) : 0;
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          const u32 e = 8 * s + r8;
          const u64 ks = __shfl_sync(0xFFFFFFFFu, k, e);
          if (i0 + e < hi)
            copy16(rows + row_at(e, q), E.rec + (t.x.g_lo + ks + p + 1) * kRecBytes + 16 * q);
        }
        copies_commit();
        copies_wait<0>();
        __syncwarp();
        Rec d{};
        u32 code = 0, vb = 0;
        if (i0 + lane < hi) {
          d = row_rec(rows, lane);
          // an id that occurs twice in a big pair's message: the other record is found
          if (t.x.nbig && A.unsorted[p] &&
              seg_lookup<true>(E.seg, epoch, p, t.x.g_lo, t.x.m, d.w[0]) != (u32)(t.x.g_lo + k))
            latch(E.st, TERA_EINVAL);
          code = rec_code(d, &vb);
          if (in_bounds(E.st, i0 + lane, 0, t.n_new)) codes[t.x.r + i0 + lane] = code;
          if constexpr (PR) {
            if (E.pr.hist_next)
              store_hist_next(E.pr.hist_next + kHistBytes * (t.x.g_lo + matched + i0 + lane),
                              nullptr, nullptr);
          }
        }
        store_next(E, p, t.x.g_lo + matched + i0, rows, hits, d.w[0]);
        pack_step(st, out, d, code, vb, &bytes);
        __syncwarp();
      }
    }
    // the last piece may carry zeros past the bytes, still inside the records' place
    if ((bytes & 15u) && lane == 0)
      *reinterpret_cast<uint4*>(out + (bytes & ~15u)) = *reinterpret_cast<const uint4*>(st);
    if (lane == 0) {
      A.bytes[u] = bytes;
      if (word & kLarge) atomicAdd(A.group + u / kTileGroup, bytes);
    }
    __syncwarp();
  }
}

// Header, padding, iteration totals and the new reference's header of a pair,
// by the warp that knows the pair's payload.
__device__ __forceinline__ void finish_message(const TileArgs& A, const Tile& t, u64 payload,
                                               u64 mode) {
  const EncArgs& E = A.E;
  const int lane = threadIdx.x & 31;
  const u32 p = t.p;
  const u64 r = t.x.r, n_new = t.n_new;
  const u64 body = (u64)kHdrBytes + 4 * (r + n_new) + payload;
  const u64 msg = round16(body);
  const u64 matched = (u64)t.x.m - n_new;
  uint8_t* w8 = E.wire + t.x.w_off;
  if (lane == 0) {
    // the message fits the slab reserved for it (checked after the fact)
    (void)in_bounds(E.st, msg, 0, E.wire_off[p + 1] - t.x.w_off + 1);
    ulonglong2* h = reinterpret_cast<ulonglong2*>(w8);
    h[0] = make_ulonglong2((u64)kWireMagic | ((u64)kVersion << 32) | ((u64)kRecBytes << 48),
                           (u64)E.class_id | (mode << 32));
    h[1] = make_ulonglong2(r, n_new);
    h[2] = make_ulonglong2(r - matched, payload);
    h[3] = make_ulonglong2((u64)p, msg);
    E.wire_len[p] = msg;
    atomicAdd(&E.stats->ref_slots, r);
    atomicAdd(&E.stats->holes, r - matched);
    atomicAdd(&E.stats->new_records, n_new);
    atomicAdd(&E.stats->payload_bytes, payload);
    atomicAdd(&E.stats->wire_bytes, msg);
    write_taio_header(E.ref_next + (t.x.g_lo + p) * kRecBytes, E.class_id, p, t.x.m);
    E.reset[p] = 0;
  }
  if (body + lane < msg) w8[body + lane] = 0;  // zero padding (< 16 bytes)
}

// This lane's share of the payload bytes of the tiles [a, b) of one pair.
__device__ __forceinline__ u64 tile_bytes(const TileArgs& A, u32 a, u32 b) {
  const u32 lane = threadIdx.x & 31;
  u64 sum = 0;
  if (b - a > kGroupMin) {
    const u32 g0 = (a + kTileGroup - 1) / kTileGroup, g1 = b / kTileGroup;
    for (u32 g = g0 + lane; g < g1; g += 32) sum += A.group[g];
    for (u32 i = a + lane; i < g0 * kTileGroup; i += 32) sum += A.bytes[i];
    a = g1 * kTileGroup;
  }
  for (u32 i = a + lane; i < b; i += 32) sum += A.bytes[i];
  return sum;
}

// The pairs without entries on either side, a thread each: headers alone.  The
// launch's last threads take them (on small iterations they have no tile).
__device__ __forceinline__ void finish_empty(const TileArgs& A) {
  const u64 threads = (u64)gridDim.x * kT;
  u64 n = 0;
  for (u64 p = threads - 1 - ((u64)blockIdx.x * kT + threadIdx.x); p < A.P; p += threads) {
    const TilePair& x = A.pair[p];
    if ((x.nst | x.nnu) != 0) continue;
    const u64 g_lo = x.g_lo, w = x.w_off;
    const u32 mode = x.mode;
    ulonglong2* h = reinterpret_cast<ulonglong2*>(A.E.wire + w);
    h[0] = make_ulonglong2((u64)kWireMagic | ((u64)kVersion << 32) | ((u64)kRecBytes << 48),
                           (u64)A.E.class_id | ((u64)mode << 32));
    h[1] = make_ulonglong2(0, 0);
    h[2] = make_ulonglong2(0, 0);
    h[3] = make_ulonglong2(p, kHdrBytes);
    A.E.wire_len[p] = kHdrBytes;
    write_taio_header(A.E.ref_next + (g_lo + p) * kRecBytes, A.E.class_id, (u32)p, 0);
    if (A.D.recv) write_taio_header(A.D.recv + (g_lo + p) * kRecBytes, A.D.class_id, (u32)p, 0);
    A.E.reset[p] = 0;
    ++n;
    if (!x.fits) latch(A.D.st, TERA_ECORRUPT);  // as the decode's header check
  }
  n = warp_sum(n);
  if ((threadIdx.x & 31) == 0 && n) atomicAdd(&A.E.stats->wire_bytes, n * kHdrBytes);
}

// A tile's payload to its place in the message, behind that of the pair's
// tiles before it (their counts added up).
template <bool PR>
__global__ void __launch_bounds__(kT, kPerSm) codec_wire_kernel(TileArgs A) {
  chain_begin();
  const EncArgs& E = A.E;
  const u32 warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const u32 n = tile_count(A);
  const u32 shift = A.scal[TS_SHIFT];
  const u32 stride = gridDim.x * kWarps;
  u32 u = blockIdx.x * kWarps + warp;
  u32 p_next = u < n ? A.unit_pair[u] : 0u;
  for (; u < n; u += stride) {
    const Tile t = tile_of(A, u, p_next);
    if (u + stride < n) p_next = A.unit_pair[u + stride];
    const u32 own = A.bytes[u];
    u64 record;
    bool last;
    if (t.local < t.x.nst) {
      record = A.before[u];
      last = t.n_new == 0 && t.local + 1 == t.x.nst;
    } else {
      u32 lo, hi;
      new_range(t.n_new, t.x.nnu + added_tiles(A, t.p).n, t.local - t.x.nst, shift, &lo, &hi);
      record = (u64)t.x.m - t.n_new + lo;
      // an entryless pair's message is its header
      last = hi == t.n_new && (lo < hi || (t.n_new == 0 && t.x.r == 0 && t.local == 0));
    }
    const u32 planned = t.x.nst + t.x.nnu, own_planned = t.local < planned ? t.local : planned;
    u64 pre = tile_bytes(A, t.x.unit0, t.x.unit0 + own_planned);
    if (t.local > planned) pre += tile_bytes(A, u - (t.local - planned), u);
    pre = warp_sum(pre);
    if (lane == 0) A.place[u] = pre;
    uint8_t* pay = E.wire + t.x.w_off + kHdrBytes + 4 * ((u64)t.x.r + t.n_new);
    if (own) {
      uint8_t* packed = payload_place(A, t, record);
      warp_flush(packed, pay + pre, own);
      if (!t.x.fits && A.D.recv) {  // a rejected pair's records will not be decoded over it
        __syncwarp();
        for (u32 c = lane; c < ((own + 15u) >> 4); c += 32)
          *reinterpret_cast<uint4*>(packed + (c << 4)) = make_uint4(0u, 0u, 0u, 0u);
      }
    }
    if (last) finish_message(A, t, pre + own, message_mode<PR>(A, t));
  }
  if (A.scal[TS_OK]) finish_empty(A);
}

// Tiles and their places are the encode's (both sides of the call run here); a
// tile's payload bytes, from the codes on the wire, have to come to the
// encode's.
template <bool PR>
__global__ void __launch_bounds__(kT, kDecPerSm) codec_decode_kernel(TileArgs A) {
  chain_begin();
  extern __shared__ __align__(16) uint8_t dyn[];
  const DecArgs& D = A.D;
  const u32 warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const u32 r8 = lane >> 2, q = lane & 3;  // this lane's record of each eight, and its piece
  uint8_t* stages = dyn + warp * (2 * kStage + 2 * kRows);
  uint8_t* rows = stages + 2 * kStage;
  const u32 n_units = tile_count(A);
  const u32 shift = A.scal[TS_SHIFT];
  const u32 stride = gridDim.x * kWarps;
  u32 u = blockIdx.x * kWarps + warp;
  u32 p_next = u < n_units ? A.unit_pair[u] : 0u;
  for (; u < n_units; u += stride) {
    const Tile t = tile_of(A, u, p_next);
    if (u + stride < n_units) p_next = A.unit_pair[u + stride];
    const u32 p = t.p;
    const u64 m = t.x.m, ns = t.x.r, n = ns + t.n_new;
    u32 lo, hi, base = 0;  // this tile's entries [lo, hi) behind the pair's entry `base`
    u64 pos;               // records before it
    if (t.local < t.x.nst) {
      lo = t.local << shift;
      hi = t.x.r - lo < (1u << shift) ? t.x.r : lo + (1u << shift);
      pos = A.before[u];
    } else {
      new_range(t.n_new, t.x.nnu + added_tiles(A, p).n, t.local - t.x.nst, shift, &lo, &hi);
      base = t.x.r;
      pos = m - t.n_new + lo;
    }
    const uint8_t* w8 = D.wire + t.x.w_off;
    u64 mode = t.x.mode;
    bool usable = t.x.fits != 0 && lo < hi;
    if (PR || t.local == 0) {
      DecHdr H;
      const u32 err = dec_read_header<false, PR>(D, p, m, &H);
      if (t.local == 0 && lane == 0) {
        if (err) latch(D.st, err);
        else if (H.ns != ns || H.nn != t.n_new) latch(D.st, TERA_ECORRUPT);
        write_taio_header(D.recv + (t.x.g_lo + p) * kRecBytes, D.class_id, p, m);
      }
      usable = usable && !err;
      mode = H.mode;
    }
    if (!usable) continue;
    const u32* codes = reinterpret_cast<const u32*>(w8 + kHdrBytes) + base;
    const uint8_t* pay = w8 + kHdrBytes + 4 * n + A.place[u];
    const u32 want = A.bytes[u];
    const u64 ro = D.ref_off ? D.ref_off[p] : 0;
    const uint8_t* ref = D.ref + (ro + p + 1) * kRecBytes;
    uint8_t* recv = D.recv + (t.x.g_lo + p + 1) * kRecBytes;
    u32 at = 0;  // payload bytes of the steps asked for
    // a step: what its codes say, and where its payload starts in the stage
    struct Step {
      u32 code, hits, records, off[4], s0;
    };
    bool broken = false;
    // asks for a step's payload and reference records (a step ahead of their use)
    const auto request = [&](u32 i0, u32 code) {
      Step x;
      x.code = code;
      const DecEnt c = dec_entry(D.st, code, i0 + lane < hi ? (u64)base + i0 + lane : n, n, ns);
      x.hits = __ballot_sync(0xFFFFFFFFu, c.vn && !c.bad);
      x.records = __ballot_sync(0xFFFFFFFFu, c.vn);
      const bool odd = ((i0 - lo) & 32u) != 0;
      uint8_t* row = rows + (odd ? kRows : 0);
      u32 b[4];
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        const u32 e = 8 * s + r8;
        const u32 y = __shfl_sync(0xFFFFFFFFu, code, e) >> (8 * q);
        const bool live = x.hits >> e & 1u;
        b[s] = live ? (y & 0xFu) + (y >> 4 & 0xFu) : 0u;
        if (live && base == 0 && i0 + e < ns)
          copy16(row + (s * 32 + lane) * 16, ref + (u64)(i0 + e) * kRecBytes + 16 * q);
      }
      const u32 total = scan4(b, x.off);
      const uint8_t* g = pay + at;
      x.s0 = (u32)((uintptr_t)g & 15u);
      // inside the tile's bytes
      if (at + total > want) broken = true;
      else if (total) {
        // the slab is 16-byte aligned and padded, so the rounded range stays
        // inside the message
        const uint8_t* g16 = g - x.s0;
        uint8_t* st = stages + (odd ? kStage : 0);
        for (u32 k = lane; k < ((x.s0 + total + 15u) >> 4); k += 32)
          copy16(st + (k << 4), g16 + (k << 4));
      }
      at += total;
      copies_commit();
      return x;
    };
    u32 c_next = lo + 32 + lane < hi ? codes[lo + 32 + lane] : 0u;
    Step now = request(lo, lo + lane < hi ? codes[lo + lane] : 0u);
    for (u32 i0 = lo; i0 < hi; i0 += 32) {
      const bool odd = ((i0 - lo) & 32u) != 0;
      const u32 code_next = c_next;
      c_next = i0 + 64 + lane < hi ? codes[i0 + 64 + lane] : 0u;
      Step next = now;
      if (i0 + 32 < hi && !broken) {
        next = request(i0 + 32, code_next);
        copies_wait<1>();
      } else {
        copies_wait<0>();
      }
      __syncwarp();
      const u32 hits = now.hits, records = now.records;
      // inside the pair's records
      if (pos + (u32)__popc(records) > m) broken = true;
      if (broken) break;
      const uint8_t* st = stages + (odd ? kStage : 0);
      const uint8_t* row = rows + (odd ? kRows : 0);
      const u32 i = i0 + lane;
      if constexpr (PR) {
        if ((hits >> lane & 1u) && D.pr.hist_next) {
          const u64 to = pos + (u32)__popc(records & ((1u << lane) - 1u));
          uint8_t* hn = D.pr.hist_next + kHistBytes * (t.x.g_lo + to);
          if (base == 0 && i < ns) {
            Rec r;
            const u64* w = reinterpret_cast<const u64*>(ref + (u64)i * kRecBytes);
            r.w[1] = w[1];
            r.w[2] = w[2];
            r.w[3] = w[3];
            Hist h;
            if (D.pr.hist) h = load_hist(D.pr.hist + kHistBytes * (ro + i));
            store_hist_next(hn, &r, D.pr.hist ? &h : nullptr);
          } else {
            store_hist_next(hn, nullptr, nullptr);
          }
        }
      }
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        const u32 e = 8 * s + r8;
        const u32 y = __shfl_sync(0xFFFFFFFFu, now.code, e) >> (8 * q);
        if (!(hits >> e & 1u)) continue;
        const u32 la = y & 0xFu, lb = y >> 4 & 0xFu;
        const u32 o = now.s0 + now.off[s];
        Piece v{stage_bytes_at(st, o, la), stage_bytes_at(st, o + la, lb)};
        if (base == 0 && i0 + e < ns) {
          const Piece R = load_piece(row + (s * 32 + r8 * 4) * 16, q);
          bool done = false;
          if constexpr (PR) {
            if (D.pr.pre && mode == kModeResidual && q < 2) {
              const u64* ps = D.pr.pscr + 4 * (ro + i0 + e);
              if (ps[3]) {  // words 1 to 3
                v.a = q ? ps[1] + unzigzag(v.a) : v.a ^ R.a;
                v.b = ps[q ? 2 : 0] + unzigzag(v.b);
                done = true;
              }
            }
          }
          if (!done) {
            v.a ^= R.a;
            v.b ^= R.b;
          }
        }
        const u64 to = pos + (u32)__popc(records & ((1u << e) - 1u));
        if (in_bounds(D.st, to, 0, m)) store_piece(recv + to * kRecBytes, q, v);
      }
      pos += (u32)__popc(records);
      now = next;
      __syncwarp();
    }
    copies_wait<0>();
    __syncwarp();
    if (lane == 0 && (broken || at != want)) latch(D.st, TERA_ECORRUPT);
  }
}

}  // namespace

namespace tera {

tera_status launch_tiles(tera_ctx* ctx, const EncArgs& E, const DecArgs& D, bool pr, int mode,
                         u64 wire_cap, u64 recv_cap, cudaStream_t s) {
  const u64 P = ctx->n_pairs;
  const bool encode_only = D.recv == nullptr;
  tera_status st;
  const unsigned grid = (unsigned)(ctx->num_sms * kPerSm);
  static PerDevice configured;
  if (configured.needed(ctx->device)) {
    const void* k[] = {reinterpret_cast<const void*>(codec_encode_kernel<false>),
                       reinterpret_cast<const void*>(codec_encode_kernel<true>),
                       reinterpret_cast<const void*>(codec_decode_kernel<false>),
                       reinterpret_cast<const void*>(codec_decode_kernel<true>)};
    if (cudaFuncSetAttribute(reinterpret_cast<const void*>(codec_match_kernel),
                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kMatchSmem) != cudaSuccess)
      return TERA_ECUDA;
    for (int i = 0; i < 4; ++i)
      if (cudaFuncSetAttribute(k[i], cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)(i < 2 ? kEncSmem : kDecSmem)) != cudaSuccess)
        return TERA_ECUDA;
    configured.done(ctx->device);
  }
  TileArgs A;
  A.E = E;
  A.D = D;
  A.pair = reinterpret_cast<TilePair*>(ctx->t_pair);
  A.unit_pair = ctx->t_unit_pair;
  A.unit_cap = (u32)(ctx->t_units < 0xFFFFFFFFull ? ctx->t_units : 0xFFFFFFFFull);
  A.unit_first = ctx->t_unit_first;
  A.setup_state = ctx->t_part;
  A.item_pair = ctx->t_item_pair;
  A.big_pair = ctx->t_big_pair;
  A.small_pair = ctx->t_small_pair;
  A.warps = (u32)(ctx->num_sms * kPerSm * (kT / 32));
  A.warp_pair = P > 8ull * grid ? kWarpPair : kWarpPairFew;
  A.before = ctx->t_before;
  A.bytes = ctx->t_bytes;
  A.group = ctx->t_group;
  A.place = ctx->t_place;
  A.tot = ctx->t_tot;
  A.done = ctx->t_done;
  A.built = ctx->t_done + P;
  A.unsorted = ctx->t_done + 2 * P;
  A.bits = ctx->t_bits;
  A.new_idx = ctx->t_new;
  A.scratch = encode_only ? ctx->t_scratch : D.recv;
  A.scal = ctx->t_scal;
  A.P = P;
  const unsigned setup = (unsigned)(P == 0 ? 1 : (P + kSetupT - 1) / kSetupT);
  const unsigned egrid = (unsigned)(ctx->num_sms * kEncPerSm), dgrid = (unsigned)(ctx->num_sms * kDecPerSm);
  A.setup_ticket = reinterpret_cast<u32*>(ctx->t_part + 4 * (u64)setup);
  A.limit_ns = ctx->wait_ns;
  prof_begin(ctx, s);
  launch_chained(tiles_setup_kernel, setup, kSetupT, 0, s, A, mode, const_cast<u64*>(E.wire_off), wire_cap,
                                               ctx->cap_records, recv_cap, ctx->t_units,
                                               ctx->t_items, ctx->t_bigs, ctx->d_epoch);
  if ((st = check_launch(ctx, "tiles_setup_kernel", s)) != TERA_OK) return st;
  prof_begin(ctx, s);
  launch_chained(codec_match_kernel, grid, kT, kMatchSmem, s, A);
  if ((st = check_launch(ctx, "codec_match_kernel", s)) != TERA_OK) return st;
  if (ctx->cap_records > kTableMax) {  // a big pair needs that many records
    prof_begin(ctx, s);
    launch_chained(codec_bigmatch_kernel, grid, kT, 8 * kBigWindow, s, A);
    if ((st = check_launch(ctx, "codec_bigmatch_kernel", s)) != TERA_OK) return st;
  }
  if (pr) {
    prof_begin(ctx, s);
    launch_chained(codec_sizes_kernel, grid, kT, 0, s, A);
    if ((st = check_launch(ctx, "codec_sizes_kernel", s)) != TERA_OK) return st;
  }
  prof_begin(ctx, s);
  if (pr) launch_chained(codec_encode_kernel<true>, egrid, kT, kEncSmem, s, A);
  else launch_chained(codec_encode_kernel<false>, egrid, kT, kEncSmem, s, A);
  if ((st = check_launch(ctx, "codec_encode_kernel", s)) != TERA_OK) return st;
  prof_begin(ctx, s);
  if (pr) launch_chained(codec_wire_kernel<true>, grid, kT, 0, s, A);
  else launch_chained(codec_wire_kernel<false>, grid, kT, 0, s, A);
  if ((st = check_launch(ctx, "codec_wire_kernel", s)) != TERA_OK) return st;
  if (encode_only) return TERA_OK;
  prof_begin(ctx, s);
  if (pr) launch_chained(codec_decode_kernel<true>, dgrid, kT, kDecSmem, s, A);
  else launch_chained(codec_decode_kernel<false>, dgrid, kT, kDecSmem, s, A);
  return check_launch(ctx, "codec_decode_kernel", s);
}

// Bounds of the lists for `cap` slots, records and pairs P (the setup's
// counts): tiles of slots, tiles of records that must be new, shares of
// records (the tiles of new records after the match are at most the records' own
// tiles and a share); match items and bigmatch items of big pairs.  Tiles below the
// largest size come with fewer than twice kTilesPerWarp per resident warp.
void tile_list_bounds(u64 cap, u64 P, u64 warps, u64* units, u64* items, u64* bigs) {
  const u64 few = 2 * kTilesPerWarp * warps;
  const u64 most = (cap >> kMaxShift) > few ? cap >> kMaxShift : few;
  *units = 2 * most + most / kNewShare + 5 * P + 64;
  *items = cap / kBigTile + 2 * P + 64;
  *bigs = 2 * (cap / kBigTile + P) + 64;
}

}  // namespace tera
