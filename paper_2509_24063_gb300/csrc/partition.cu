// Step a1 — grid classification and per-pair message lists (paper Sec. 2.1,
// "Aura Update": agents within the interaction distance of a neighbouring
// box are sent to it every iteration; the aura is narrower than the box).
//
// Kernels:
//   classify_kernel  one pass over x,y,z (coalesced 16-byte loads): owner box,
//                    26-bit aura mask, count of (agent, pair) entries of every
//                    run of 64 consecutive agents; per axis a bucket table in
//                    shared memory answers most coordinates, the exact key
//                    comparisons the rest
//   emit_kernel      stable compaction of the entries in agent order (warp
//                    scans inside a run, run bases from a scan)
//   rs_hist_kernel / rs_scatter_kernel
//                    stable LSD radix sort of the entry indices by pair
//                    index, so each pair's list keeps ascending agent order:
//                    the digit counts of every pass in one read of the keys,
//                    then a launch a pass, whose tiles (staged into shared
//                    memory by cp.async) find the digits' places by a
//                    look-back over the tiles before them; the last pass
//                    writes the agent of every record and the record index of
//                    every entry (pack reads in agent order)
//   pair_off_kernel  per-pair counts and offsets from the sorted keys
#include "classify.cuh"
#include "tera_internal.cuh"

using namespace tera;

namespace {

// One axis by the exact comparisons, out of line (few coordinates come here,
// and inlined into every round of the kernel it pushed the rounds' code out of
// the instruction cache): (box index << 2) | aura offsets (bit 0: -1, bit 1:
// +1), or ~0 outside the domain.
__device__ __noinline__ u32 axis_exact(u64 bits, int a, const SmemGrid& s) {
  int i;
  const u32 o = classify_axis(bits, a, s, &i);
  return o ? ((u32)i << 2) | (o & 1u) | ((o & 4u) >> 1) : ~0u;
}

// The same by the bucket table when the coordinate's bucket holds an answer.
// The estimate is taken only for magnitudes in the float normal range (2^-126
// <= |v| < 2^128, which also sends NaN and infinities to the exact path).
__device__ __forceinline__ u32 axis_entry(u64 bits, int a, const SmemGrid& s, const uint8_t* tab,
                                          float flo, float fs) {
  const u32 hi = (u32)(bits >> 32);
  const u32 ha = hi & 0x7FFFFFFFu;
  u32 e = kBucketExact;
  if (ha - 0x38100000u < 0x0FE00000u) {
    const float af = __uint_as_float((hi & 0x80000000u) | ((ha - 0x38000000u) << 3));
    const int j = __float2int_rz((af - flo) * fs);
    if ((u32)j < (u32)kAxisBuckets) e = tab[j];
  }
  return e & kBucketExact ? axis_exact(bits, a, s) : e;
}

// Owner and aura mask of one agent from its three axes; lut: the mask of every
// combination of the axes' offsets (bit pairs x, y, z).
__device__ __forceinline__ void agent_entry(u32 ex, u32 ey, u32 ez, int n0, int n1, const u32* lut,
                                            int* owner, u32* mask, bool* ok) {
  *ok = ex != ~0u && ey != ~0u && ez != ~0u;
  *owner = *ok ? (int)(ex >> 2) + n0 * ((int)(ey >> 2) + n1 * (int)(ez >> 2)) : -1;
  *mask = *ok ? lut[(ex & 3u) | ((ey & 3u) << 2) | ((ez & 3u) << 4)] : 0u;
}

// Each block classifies tiles of R rounds of 512 agents (tile blockIdx.x, then
// every gridDim.x-th: the grid holds the blocks resident at once, so the grid
// rows and the bucket tables are copied into shared memory once per block).
// In round k of a tile, thread t holds agents 512k + 2t and 512k + 2t + 1 (one
// 16-byte load per coordinate), so every warp load is fully coalesced, and
// each warp covers a run of kRunAgents consecutive agents per round; the
// number of (agent, pair) entries of every run is written (runs are in agent
// order).  TAB: with bucket tables (bk); else every agent takes the exact key
// comparisons.
//
// Bound: issue and HBM about equally.  338 warp instructions per 64 agents and
// the exact comparisons inlined 24 times over (3.3 stall cycles an issue on
// instruction fetches) took 689 us for 100 M agents; with the masks looked up
// and the exact path out of line 537.  (Fewer resident blocks for more
// registers: 5 per SM 752 us, 4 per SM 725; two rounds unrolled 654.)
template <bool TAB, int R>
__global__ void __launch_bounds__(kClassifyThreads, 6)
    classify_kernel(const u64* __restrict__ x, const u64* __restrict__ y,
                    const u64* __restrict__ z, u64 n, const GridTables* __restrict__ g,
                    const AxisBuckets* __restrict__ bk, u64 n_tiles, int* __restrict__ owner,
                    u32* __restrict__ mask, u32* __restrict__ run_cnt, u64 n_runs, DevStatus* st,
                    DevStats* stats, u64* __restrict__ sort_head) {
  __shared__ SmemGrid sg;
  __shared__ float s_flo[3], s_fs[3];
  __shared__ u32 s_lut[64];
  // the tables follow the grid rows (a multiple of 32 bytes) in dynamic shared memory
  uint8_t* tab = reinterpret_cast<uint8_t*>(grid_rows() + (g->n[0] + g->n[1] + g->n[2]));
  if constexpr (TAB) {
    if (threadIdx.x < 64) {
      const u32 q = threadIdx.x;
      u32 o[3];
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const u32 b = q >> (2 * a) & 3u;
        o[a] = 2u | (b & 1u) | ((b & 2u) << 1);
      }
      s_lut[q] = o[0] * spread3(o[1], 3) * spread3(o[2], 9) & ~(1u << 13);
    }
    const uint4* src = reinterpret_cast<const uint4*>(bk->tab);
    uint4* dst = reinterpret_cast<uint4*>(tab);
    for (int i = threadIdx.x; i < 3 * kAxisBuckets / 16; i += blockDim.x) dst[i] = src[i];
    if (threadIdx.x < 3) {
      s_flo[threadIdx.x] = bk->flo[threadIdx.x];
      s_fs[threadIdx.x] = bk->fs[threadIdx.x];
    }
  }
  load_grid(sg, g);  // ends with a block barrier
  chain_begin();  // (the tables are the context's: written when it was made)
  if (blockIdx.x == 0) {  // what the launches after this one find zero
    for (u32 i = threadIdx.x; i < kSortHead; i += blockDim.x) sort_head[i] = 0;
    if (threadIdx.x == 0) {
      stats->iterations += 1;
      stats->agents += n;
      st->abort = 0;
      if (n == 0) run_cnt[0] = 0;
    }
  }
  const int lane = threadIdx.x & 31;
  const int n0 = sg.n[0], n1 = sg.n[1];
  bool bad = false;
  for (u64 tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
    const u64 tile0 = tile * (2 * kClassifyThreads * R);
#pragma unroll
    for (int k = 0; k < R; ++k) {
      const u64 a0 = tile0 + (u64)k * (2 * kClassifyThreads) + 2u * threadIdx.x;
      u64 vx[2], vy[2], vz[2];
      if (a0 + 1 < n) {
        ulonglong2 tx = *reinterpret_cast<const ulonglong2*>(x + a0);
        ulonglong2 ty = *reinterpret_cast<const ulonglong2*>(y + a0);
        ulonglong2 tz = *reinterpret_cast<const ulonglong2*>(z + a0);
        vx[0] = tx.x; vx[1] = tx.y; vy[0] = ty.x; vy[1] = ty.y; vz[0] = tz.x; vz[1] = tz.y;
      } else {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          if (a0 + q < n) {
            vx[q] = x[a0 + q]; vy[q] = y[a0 + q]; vz[q] = z[a0 + q];
          } else {
            vx[q] = vy[q] = vz[q] = 0ull;
          }
        }
      }
      int o[2];
      u32 m[2];
      u32 cnt = 0;
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        bool ok;
        if constexpr (TAB)
          agent_entry(axis_entry(vx[q], 0, sg, tab, s_flo[0], s_fs[0]),
                      axis_entry(vy[q], 1, sg, tab + kAxisBuckets, s_flo[1], s_fs[1]),
                      axis_entry(vz[q], 2, sg, tab + 2 * kAxisBuckets, s_flo[2], s_fs[2]), n0, n1,
                      s_lut, &o[q], &m[q], &ok);
        else
          classify_agent(vx[q], vy[q], vz[q], sg, &o[q], &m[q], &ok);
        if (a0 + q < n) {
          bad |= !ok;
          cnt += __popc(m[q]);
        }
      }
      if (a0 + 1 < n) {
        *reinterpret_cast<int2*>(owner + a0) = make_int2(o[0], o[1]);
        *reinterpret_cast<uint2*>(mask + a0) = make_uint2(m[0], m[1]);
      } else if (a0 < n) {
        owner[a0] = o[0];
        mask[a0] = m[0];
      }
      cnt = warp_sum(cnt);
      const u64 run = (a0 - 2u * lane) / kRunAgents;
      if (lane == 0 && run < n_runs) run_cnt[run] = cnt;
    }
  }
  if (bad) latch(st, TERA_EDOMAIN);
}

// Emit (pair, agent) entries in agent order, with the rounds and runs of
// classify_kernel: run r writes its entries from run_base[r]; within a run,
// lanes are ranked by a warp scan.
template <int R>
__global__ void __launch_bounds__(kClassifyThreads)
    emit_kernel(const int* __restrict__ owner, const u32* __restrict__ mask, u64 n,
                const u64* __restrict__ run_base, u64 n_runs, u32* __restrict__ keys,
                u32* __restrict__ vals, u64 cap, DevStatus* st) {
  chain_begin();
  if (*reinterpret_cast<const volatile u32*>(&st->abort)) return;  // the scan gave up
  const u64 total = run_base[n_runs];
  const u64 n_entries = total;  // (a warp's own count below is also called total)
  if (total > cap) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      latch(st, TERA_ECAPACITY);
      need(st, total);
      atomicExch(&st->abort, 1u);
    }
    return;
  }
  const int lane = threadIdx.x & 31;
  const u64 tile0 = (u64)blockIdx.x * (2 * kClassifyThreads * R);
  for (int k = 0; k < R; ++k) {
    const u64 a0 = tile0 + (u64)k * (2 * kClassifyThreads) + 2u * threadIdx.x;
    const u64 first = a0 - 2u * lane;
    if (first >= n) break;  // warp-uniform
    u32 m[2] = {0u, 0u};
    int o[2] = {0, 0};
    if (a0 + 1 < n) {
      uint2 mm = *reinterpret_cast<const uint2*>(mask + a0);
      m[0] = mm.x; m[1] = mm.y;
      if (m[0] | m[1]) {
        int2 oo = *reinterpret_cast<const int2*>(owner + a0);
        o[0] = oo.x; o[1] = oo.y;
      }
    } else if (a0 < n) {
      m[0] = mask[a0];
      if (m[0]) o[0] = owner[a0];
    }
    const u32 c = __popc(m[0]) + __popc(m[1]);
    const u32 inc = warp_incl_scan<u32>(c);
    const u32 total = __shfl_sync(0xFFFFFFFFu, inc, 31);
    const u64 base = run_base[first / kRunAgents];
    // the run's entries written by the whole warp, lane i taking entry i of
    // each 32: its source lane is the first whose inclusive count exceeds i
    for (u32 r0 = 0; r0 < total; r0 += 32) {  // warp-uniform
      const u32 idx = r0 + (u32)lane;
      u32 src = 0;
#pragma unroll
      for (u32 b = 16; b >= 1; b >>= 1)
        if (__shfl_sync(0xFFFFFFFFu, inc, (int)(src + b - 1)) <= idx) src += b;
      const u32 s_inc = __shfl_sync(0xFFFFFFFFu, inc, (int)src);
      const u32 s_c = __shfl_sync(0xFFFFFFFFu, c, (int)src);
      const u32 s_m0 = __shfl_sync(0xFFFFFFFFu, m[0], (int)src);
      const u32 s_m1 = __shfl_sync(0xFFFFFFFFu, m[1], (int)src);
      const int s_o0 = __shfl_sync(0xFFFFFFFFu, o[0], (int)src);
      const int s_o1 = __shfl_sync(0xFFFFFFFFu, o[1], (int)src);
      if (idx >= total) continue;
      u32 k = idx - (s_inc - s_c);  // entry k of the source lane's two agents
      const u32 n0 = __popc(s_m0);
      const bool second = k >= n0;
      u32 mm = second ? s_m1 : s_m0;
      k = second ? k - n0 : k;
      for (u32 t = 0; t < k; ++t) mm &= mm - 1;
      const u32 b = (u32)(__ffs(mm) - 1);
      if (!in_bounds(st, base + idx, 0, n_entries)) continue;
      keys[base + idx] = (u32)(second ? s_o1 : s_o0) * 27u + b;
      vals[base + idx] = (u32)(first + 2u * src + (second ? 1u : 0u));  // the entry's agent
    }
  }
}

// Entries to sort: none when they exceed the capacity or the call was aborted.
__device__ __forceinline__ u64 live_entries(const u64* total_ptr, u64 cap, const DevStatus* st) {
  if (*reinterpret_cast<const volatile u32*>(&st->abort)) return 0;
  u64 t = *total_ptr;
  return t > cap ? 0 : t;
}

constexpr int kSortSub = 4;  // sub-steps of 32 entries per warp and round of a tile
constexpr int kSortRound = kSortThreads * kSortSub;
static_assert(kSortTile % kSortRound == 0, "whole rounds");

// Scratch of a sort (SortBufs::hist): counts[pass * kRadix + d] of digit d,
// then a claim ticket per pass, then the look-back states of each pass's
// tiles, state[(pass * tiles + tile) * radix + d].
__device__ __forceinline__ u64* sort_states(u64* head, u32 pass, u64 tiles, u32 radix) {
  return head + kSortHead + (u64)pass * tiles * radix;
}

// Entries of a tile: kSortTile, or a single round of it while such tiles are
// about two per SM of the 152 at most (a constant, as the host sizes the scratch by
// it without a device), so that a short list is still spread over the SMs (100
// thousand agents, 70 K entries: 103 -> 98 us per iteration.  Up to four per SM
// 1 M agents, whose tiles then wait for one another longer, lose what they
// gain: 306 -> 308).
constexpr u64 kSortFew = 300ull * kSortRound;
__host__ __device__ constexpr u32 sort_tile(u64 entries) {
  return entries <= kSortFew ? kSortRound : kSortTile;
}

// Tiles of up to cap entries, at most.
constexpr u64 sort_tiles(u64 cap) {
  const u64 few = ((cap < kSortFew ? cap : kSortFew) + kSortRound - 1) / kSortRound;
  const u64 many = (cap + kSortTile - 1) / kSortTile;
  return few > many ? few : many;
}

// Digit counts of every pass from one read of the keys, and the cleared
// look-back states of the tiles that hold entries.  Resident blocks only, each
// counting in shared memory, so that the counts cost the blocks' atomics and
// not the tiles'.
__global__ void __launch_bounds__(kSortThreads)
    rs_hist_kernel(const u32* __restrict__ keys, const u64* __restrict__ total_ptr, u64 cap,
                   u32 passes, u32 dbits, u64 tiles, u64* __restrict__ head, const DevStatus* st) {
  chain_begin();
  __shared__ u32 cnt[4 * kRadix];
  const u64 E = live_entries(total_ptr, cap, st);
  const u32 radix = 1u << dbits;
  for (u32 d = threadIdx.x; d < passes * kRadix; d += blockDim.x) cnt[d] = 0;
  __syncthreads();
  const u64 step = (u64)gridDim.x * blockDim.x;
  const u64 tid = (u64)blockIdx.x * blockDim.x + threadIdx.x;
  const bool wide = (reinterpret_cast<uintptr_t>(keys) & 15u) == 0;
  const u64 quads = wide ? E / 4 : 0;
  for (u64 i = tid; i < quads; i += step) {
    const uint4 k = reinterpret_cast<const uint4*>(keys)[i];
    for (u32 p = 0; p < passes; ++p) {
      const u32 sh = p * dbits;
      atomicAdd(&cnt[p * kRadix + ((k.x >> sh) & (radix - 1))], 1u);
      atomicAdd(&cnt[p * kRadix + ((k.y >> sh) & (radix - 1))], 1u);
      atomicAdd(&cnt[p * kRadix + ((k.z >> sh) & (radix - 1))], 1u);
      atomicAdd(&cnt[p * kRadix + ((k.w >> sh) & (radix - 1))], 1u);
    }
  }
  for (u64 i = 4 * quads + tid; i < E; i += step)
    for (u32 p = 0; p < passes; ++p)
      atomicAdd(&cnt[p * kRadix + ((keys[i] >> (p * dbits)) & (radix - 1))], 1u);
  const u32 tile = sort_tile(E);
  const u64 live = (E + tile - 1) / tile * radix;
  for (u32 p = 0; p < passes; ++p) {
    u64* s = sort_states(head, p, tiles, radix);
    for (u64 i = tid; i < live; i += step) s[i] = 0;
  }
  __syncthreads();
  for (u32 d = threadIdx.x; d < passes * kRadix; d += blockDim.x)
    if (cnt[d]) atomicAdd(head + d, (u64)cnt[d]);
}

// Stable scatter of sort tiles (sort_tile entries), claimed one after the
// other by resident blocks.  A tile counts its digits, publishes the counts,
// and while its entries are ranked the tiles before it publish theirs; thread
// d then walks back over digit d's counts (eight tiles' in flight) to the
// nearest inclusive sum (A. Adinets and D. Merrill, "Onesweep: A Faster Least
// Significant Digit Radix Sort for GPUs", 2022).  A histogram launch and a scan of three per pass did
// this before: 178 + 58 us a pass at 16.6 M entries.  The tile's input
// (keys, entry indices when given, agents) is first copied into shared memory
// in input order by cp.async in 16-byte pieces (a ragged end, or unaligned
// arrays, by plain loads), so the tile pays the latency of its global loads
// once.  The tile is then ranked in kSortPerThread / 4 rounds: in a round warp
// w takes 128 consecutive entries (4 sub-steps of 32, lane order), ranks equal
// digits with match_any against warp-private counters, and one prefix over the
// warps places them; the tile-local sorted position of every entry (digit
// start + rank) records the entry's place in the tile (inv).  The tile is
// written out in sorted order, so consecutive threads write consecutive
// addresses of a digit's run.  Each entry carries its index (vals_in ==
// nullptr on the first pass: entry i is at position i) and its agent
// (agents_in, read in input order: the entry list's agents on the first pass,
// the previous pass's output after it).  Every pass but the last writes both;
// the last writes the agent as the value (vals_out[pos] = agent) and, when
// dest is given, the entry's record index (dest[e] = pos).  kR bounds the
// radix (digit arrays in shared memory).

// Dynamic shared memory of a scatter: raw keys and agents, the sorted-position
// index, and the raw entry indices when the pass reads them.
__host__ __device__ constexpr size_t sort_smem_bytes(bool with_vals) {
  return (with_vals ? 3 : 2) * sizeof(u32) * kSortTile + sizeof(unsigned short) * kSortTile;
}

__device__ __forceinline__ void cp_async16(u32* smem_dst, const u32* gmem_src) {
  const unsigned dst = (unsigned)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" : : "r"(dst), "l"(gmem_src) : "memory");
}

template <u32 kR>
__global__ void __launch_bounds__(kSortThreads)
    rs_scatter_kernel(const u32* __restrict__ keys_in, const u32* __restrict__ vals_in,
                      const u32* __restrict__ agents_in, u32* __restrict__ keys_out,
                      u32* __restrict__ vals_out, u32* __restrict__ agents_out,
                      u32* __restrict__ dest, int last, const u64* __restrict__ total_ptr, u64 cap,
                      u32 pass, u32 shift, u32 radix, u64* __restrict__ head, u64 n_tiles,
                      u64 limit_ns, DevStatus* st) {
  chain_begin();
  constexpr int kWarps = kSortThreads / 32;
  constexpr int kRoundEntries = kSortRound;
  extern __shared__ __align__(16) u32 sort_stage[];
  u32* rkey = sort_stage;
  u32* ragt = sort_stage + kSortTile;
  unsigned short* inv = reinterpret_cast<unsigned short*>(sort_stage + 2 * kSortTile);
  u32* rval = sort_stage + 2 * kSortTile + kSortTile / 2;  // only when vals_in != nullptr
  __shared__ u32 base[kR];    // global start of each digit for this tile
  __shared__ u32 lstart[kR];  // tile-local start of each digit
  __shared__ u32 run[kR];     // entries of each digit placed in earlier rounds
  __shared__ u32 wcnt[kWarps][kR];
  __shared__ u32 sm[33];
  __shared__ u32 s_tile;
  const u64 E = live_entries(total_ptr, cap, st);
  const u32 tile_cap = sort_tile(E);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const u32 lt = (1u << lane) - 1u;
  u64* states = sort_states(head, pass, n_tiles, radix);
  // global start of this thread's digit
  u32 dstart;
  {
    u32 tot;
    dstart = block_excl_scan<u32>(
        threadIdx.x < radix ? (u32)head[pass * kRadix + threadIdx.x] : 0u, sm, &tot);
  }
  for (;;) {
  if (threadIdx.x == 0) s_tile = (u32)atomicAdd(head + 4 * kRadix + pass, 1ull);
  for (u32 d = threadIdx.x; d < radix; d += blockDim.x) run[d] = 0;
  __syncthreads();
  const u64 tile = s_tile;
  const u64 t0 = tile * tile_cap;
  if (t0 >= E) return;
  const u32 tile_n = (u32)(E - t0 < (u64)tile_cap ? E - t0 : (u64)tile_cap);
  {
    const uintptr_t al = reinterpret_cast<uintptr_t>(keys_in) |
                         reinterpret_cast<uintptr_t>(agents_in) |
                         reinterpret_cast<uintptr_t>(vals_in);
    const u32 n4 = (al & 15u) == 0 ? tile_n / 4 : 0;  // t0 is a multiple of 4 entries
    for (u32 c = threadIdx.x; c < n4; c += blockDim.x) cp_async16(rkey + 4 * c, keys_in + t0 + 4 * c);
    asm volatile("cp.async.commit_group;" : : : "memory");
    for (u32 c = threadIdx.x; c < n4; c += blockDim.x) {
      cp_async16(ragt + 4 * c, agents_in + t0 + 4 * c);
      if (vals_in) cp_async16(rval + 4 * c, vals_in + t0 + 4 * c);
    }
    asm volatile("cp.async.commit_group;" : : : "memory");
    for (u32 li = 4 * n4 + threadIdx.x; li < tile_n; li += blockDim.x) {
      rkey[li] = keys_in[t0 + li];
      ragt[li] = agents_in[t0 + li];
      if (vals_in) rval[li] = vals_in[t0 + li];
    }
  }
  asm volatile("cp.async.wait_group 1;" : : : "memory");
  __syncthreads();
  for (u32 li = threadIdx.x; li < tile_n; li += blockDim.x)
    atomicAdd(&run[(rkey[li] >> shift) & (radix - 1)], 1u);
  __syncthreads();
  const u32 mine = threadIdx.x < radix ? run[threadIdx.x] : 0u;  // this thread's digit's entries
  if (threadIdx.x < radix)
    lb_put(states + tile * radix + threadIdx.x, mine, tile ? kLbOwn : kLbSum);
  {
    u32 tot;
    const u32 ex = block_excl_scan<u32>(mine, sm, &tot);
    if (threadIdx.x < radix) {
      lstart[threadIdx.x] = ex;
      run[threadIdx.x] = 0;
    }
  }
  asm volatile("cp.async.wait_all;" : : : "memory");
  __syncthreads();
  for (u32 r0 = 0; r0 < tile_n; r0 += kRoundEntries) {  // block-uniform
    for (u32 d = lane; d < radix; d += 32) wcnt[warp][d] = 0;
    __syncwarp();
    u32 dig[kSortSub], rank[kSortSub];
#pragma unroll
    for (int q = 0; q < kSortSub; ++q) {
      const u32 li = r0 + (u32)warp * (32 * kSortSub) + (u32)q * 32 + (u32)lane;
      const bool live = li < tile_n;
      dig[q] = live ? ((rkey[li] >> shift) & (radix - 1)) : kR;  // sentinel for padding
      const u32 peers = __match_any_sync(0xFFFFFFFFu, dig[q]);
      rank[q] = (live ? wcnt[warp][dig[q]] : 0u) + __popc(peers & lt);
      __syncwarp();
      if (live && (peers & lt) == 0u) wcnt[warp][dig[q]] += __popc(peers);
      __syncwarp();
    }
    __syncthreads();
    for (u32 d = threadIdx.x; d < radix; d += blockDim.x) {
      u32 sacc = run[d];
      for (int w = 0; w < kWarps; ++w) {
        const u32 c = wcnt[w][d];
        wcnt[w][d] = sacc;
        sacc += c;
      }
      run[d] = sacc;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kSortSub; ++q) {
      if (dig[q] < kR) {
        const u32 li = r0 + (u32)warp * (32 * kSortSub) + (u32)q * 32 + (u32)lane;
        inv[lstart[dig[q]] + wcnt[warp][dig[q]] + rank[q]] = (unsigned short)li;
      }
    }
    __syncthreads();
  }
  bool gone = false;
  if (threadIdx.x < radix) {
    constexpr int kFlight = 8;
    u64 pre = 0;
    bool done = tile == 0;
    LbWait wait{limit_ns, &st->abort};
    for (long long at = (long long)tile - 1; !done && !gone;) {
      u64 v[kFlight];
#pragma unroll
      for (int i = 0; i < kFlight; ++i)
        v[i] = at - i >= 0 ? lb_get(states + (u64)(at - i) * radix + threadIdx.x) : 0ull;
      int taken = 0;
#pragma unroll
      for (int i = 0; i < kFlight; ++i) {
        const u64 state = v[i] >> kLbShift;
        if (done || gone || taken < i || state == 0) continue;
        if (state == kLbGone) {
          gone = true;
          continue;
        }
        pre += v[i] & kLbMask;
        ++taken;
        done = state == kLbSum;
      }
      at -= taken;
      if (taken == 0 && !done && !gone && wait.over(st)) gone = true;
    }
    lb_put(states + tile * radix + threadIdx.x, gone ? 0ull : pre + mine, gone ? kLbGone : kLbSum);
    base[threadIdx.x] = dstart + (u32)pre;
  }
  // (a tile that was given up sets the call's abort flag: nothing reads the lists)
  if (__syncthreads_or(gone)) return;
  for (u32 lp = threadIdx.x; lp < tile_n; lp += blockDim.x) {
    const u32 src = inv[lp];
    const u32 key = rkey[src], a = ragt[src];
    const u32 v = vals_in ? rval[src] : (u32)(t0 + src);
    const u32 d = (key >> shift) & (radix - 1);
    const u32 pos = base[d] + (lp - lstart[d]);
    if (!in_bounds(st, pos, 0, E) || !in_bounds(st, v, 0, E)) continue;
    keys_out[pos] = key;
    if (last) {
      vals_out[pos] = a;
      if (dest) dest[v] = pos;
    } else {
      vals_out[pos] = v;
      agents_out[pos] = a;
    }
  }
  __syncthreads();  // the tile's shared memory is used again
  }
}

// One probe step of a warp's search for the first of a[0, *hi) that is not
// below v, 32 probes at a time: [*lo, *hi) shrinks to a 32nd.
__device__ __forceinline__ void warp_probe(bool less, u64 len, u64* lo, u64* hi) {
  const u32 bal = __ballot_sync(0xFFFFFFFFu, less);
  const u32 c = (u32)__popc(bal);  // the probes are ascending, so these are the first
  const u64 base = *lo;
  if (c < 32u) *hi = base + len * c / 32;
  if (c > 0u) *lo = base + len * (c - 1u) / 32 + 1;
}

// First of keys[0, n) that is not below p.
__device__ __forceinline__ u64 lower_bound_u32(const u32* __restrict__ keys, u64 n, u32 p) {
  u64 lo = 0, hi = n;
  while (lo < hi) {
    const u64 mid = (lo + hi) >> 1;
    if (keys[mid] < p) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

// Offsets and counts of the pairs from the sorted keys.  WARP: a warp finds where
// pair p's and pair p + 1's entries begin, both searches a step at a time (five
// steps of 32 probes for 16 M entries); else a thread bisects for both, 24
// dependent loads twice over.  A warp is the faster while every pair has one at
// once; with more pairs their warps come in waves.  Launch times, warp against
// thread, 100 thousand and 16 M agents: 1,728 pairs 7.8 / 12.4 and 10.4 / 20.3
// us, 13,824 pairs 12.2 / 10.3 and 16.7 / 21.1 (whole partition 44 / 42 and 745 /
// 750), 19,683 pairs 16.0 / 10.9 and 18.8 / 20.4, 216,000 pairs 98 / 14 and 120 /
// 29.
constexpr u64 kWarpPairs = 16384;
template <bool WARP>
__global__ void __launch_bounds__(256)
    pair_off_kernel(const u32* __restrict__ sorted_keys, const u64* __restrict__ total_ptr, u64 cap,
                    u64 n_pairs, u64* __restrict__ pair_off, u64* __restrict__ pair_count,
                    u64* __restrict__ packable, DevStats* stats, const DevStatus* st) {
  chain_begin();
  const u64 E = live_entries(total_ptr, cap, st);
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    stats->records += E;
    // what pack_runs_kernel compares with the pairs' total: no total for lists
    // that are not there (a scan that gave up leaves run_base as it was)
    *packable = *reinterpret_cast<const volatile u32*>(&st->abort) ? ~0ull : E;
  }
  const u64 t = (u64)blockIdx.x * blockDim.x + threadIdx.x, threads = (u64)gridDim.x * blockDim.x;
  if constexpr (!WARP) {
    for (u64 p = t; p <= n_pairs; p += threads) {
      const u64 at = lower_bound_u32(sorted_keys, E, (u32)p);
      pair_off[p] = at;
      if (p < n_pairs) pair_count[p] = lower_bound_u32(sorted_keys, E, (u32)(p + 1)) - at;
    }
    return;
  }
  const u32 lane = threadIdx.x & 31;
  for (u64 p = t >> 5; p <= n_pairs; p += threads >> 5) {
    u64 lo0 = 0, hi0 = E, lo1 = 0, hi1 = E;
    while (lo0 < hi0 || lo1 < hi1) {  // warp-uniform
      const u64 len0 = hi0 - lo0, len1 = hi1 - lo1;
      const u64 m0 = lo0 + len0 * lane / 32, m1 = lo1 + len1 * lane / 32;
      const u32 k0 = len0 ? sorted_keys[m0] : 0u, k1 = len1 ? sorted_keys[m1] : 0u;
      if (len0) warp_probe(k0 < (u32)p, len0, &lo0, &hi0);
      if (len1) warp_probe(k1 < (u32)(p + 1), len1, &lo1, &hi1);
    }
    if (lane == 0) {
      pair_off[p] = lo0;
      if (p < n_pairs) pair_count[p] = lo1 - lo0;
    }
  }
}

}  // namespace

namespace tera {

// Stable LSD radix sort of entries by a u32 key (every key < key_limit),
// ceil(bits / 8) digit passes.  The entry count is read on the device
// (*total_ptr; nothing is sorted when it exceeds cap).  Pass k reads (kin, vin,
// ain) and writes the b buffers (k even) or the c buffers; the last pass
// writes the sorted keys to the buffer it does not read, vals_final[pos] =
// agent[e] for the entry e sorted to pos, and dest[e] = pos (dest may be null).
// The agents travel with the entries (read in order on every pass).
static void sort_shape(u64 key_limit, int* passes, int* dbits) {
  int bits = 1;
  while ((1ull << bits) < key_limit) ++bits;
  *passes = (bits + kRadixBits - 1) / kRadixBits;
  *dbits = (bits + *passes - 1) / *passes;
}

u64 sort_scratch(u64 cap, u64 key_limit) {
  int passes, dbits;
  sort_shape(key_limit, &passes, &dbits);
  return kSortHead + (((u64)passes * sort_tiles(cap)) << dbits);
}

tera_status radix_sort_entries(tera_ctx* ctx, const SortBufs& b, const u32* keys_in,
                               const u32* agent, u32* dest, u32* vals_final, const u64* total_ptr,
                               u64 cap, u64 key_limit, const u32** sorted_keys, cudaStream_t s) {
  int passes, dbits;
  sort_shape(key_limit, &passes, &dbits);
  const u32 radix = 1u << dbits;
  const u64 tiles = cap == 0 ? 1 : sort_tiles(cap);
  const u32* kin = keys_in;
  const u32* vin = nullptr;
  const u32* ain = agent;
  u32* kfinal = (passes & 1) ? b.keys_b : b.keys_c;
  tera_status st;
  static PerDevice smem_set;
  if (smem_set.needed(ctx->device)) {
    cudaFuncSetAttribute(rs_scatter_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)sort_smem_bytes(true));
    cudaFuncSetAttribute(rs_scatter_kernel<kRadix>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)sort_smem_bytes(true));
    smem_set.done(ctx->device);
  }
  if (cap > 0) {
    const u64 hgrid = (u64)grid_for(ctx, 4);
    prof_begin(ctx, s);
    launch_chained(rs_hist_kernel, (unsigned)(tiles < hgrid ? tiles : hgrid), kSortThreads, 0, s, 
        keys_in, total_ptr, cap, (u32)passes, (u32)dbits, tiles, b.hist, ctx->d_status);
    if ((st = check_launch(ctx, "rs_hist_kernel", s)) != TERA_OK) return st;
  }
  for (int pass = 0; pass < passes && cap > 0; ++pass) {
    const u32 shift = (u32)(pass * dbits);
    const bool last = pass + 1 == passes;
    u32* kout = last ? kfinal : ((pass & 1) ? b.keys_c : b.keys_b);
    u32* vout = last ? vals_final : ((pass & 1) ? b.vals_c : b.vals_b);
    u32* aout = last ? nullptr : ((pass & 1) ? b.agents_c : b.agents_b);
    const size_t smem = sort_smem_bytes(vin != nullptr);
    // resident blocks: six per SM on the first pass (no entry indices staged), four after it
    const u64 res = (u64)grid_for(ctx, vin ? 4 : 6);
    const unsigned grid = (unsigned)(tiles < res ? tiles : res);
    prof_begin(ctx, s);
    if (radix <= 128)
      launch_chained(rs_scatter_kernel<128>, grid, kSortThreads, smem, s, 
          kin, vin, ain, kout, vout, aout, last ? dest : nullptr, last ? 1 : 0, total_ptr, cap,
          (u32)pass, shift, radix, b.hist, tiles, ctx->wait_ns, ctx->d_status);
    else
      launch_chained(rs_scatter_kernel<kRadix>, grid, kSortThreads, smem, s, 
          kin, vin, ain, kout, vout, aout, last ? dest : nullptr, last ? 1 : 0, total_ptr, cap,
          (u32)pass, shift, radix, b.hist, tiles, ctx->wait_ns, ctx->d_status);
    if ((st = check_launch(ctx, "rs_scatter_kernel", s)) != TERA_OK) return st;
    kin = kout;
    vin = vout;
    ain = aout;
  }
  *sorted_keys = kin;
  return TERA_OK;
}

}  // namespace tera

extern "C" tera_status tera_partition(tera_ctx* ctx, const tera_soa* soa, tera_partition_out* out,
                                      void* stream) {
  TERA_CALL_RANGE("tera_partition");
  if (!ctx || !soa || !out) return TERA_EINVAL;
  if (soa->n < 0 || soa->n > (int64_t)0xFFFFFFFFll) return TERA_EINVAL;
  if (soa->n > 0 && (!soa->x || !soa->y || !soa->z)) return TERA_EINVAL;
  if (!out->owner || !out->mask || !out->pair_count || !out->pair_off ||
      (out->idx_capacity > 0 && !out->pair_idx))
    return TERA_EINVAL;
  if (out->idx_capacity > 0xFFFFFFFFull) return TERA_EINVAL;
  // 16-byte loads of x, y, z and 8-byte stores of owner / mask
  if (((uintptr_t)soa->x | (uintptr_t)soa->y | (uintptr_t)soa->z) & 15u) return TERA_EINVAL;
  if (((uintptr_t)out->owner | (uintptr_t)out->mask) & 7u) return TERA_EINVAL;
  cudaSetDevice(ctx->device);
  cudaStream_t s = (cudaStream_t)stream;
  const u64 n = (u64)soa->n;
  tera_status st;
  if ((st = ensure_agents(ctx, soa->n, s)) != TERA_OK) return st;
  if (!ctx->tile_cnt || !ctx->tile_base) return TERA_ENOMEM;
  if ((st = ensure_records(ctx, out->idx_capacity, s)) != TERA_OK) return st;
  ctx->iterations += 1;
  const int rounds = agent_rounds(ctx, n);
  const u64 per = 2ull * kClassifyThreads * rounds;
  const u64 blocks = n == 0 ? 1 : (n + per - 1) / per;
  const u64 runs = n == 0 ? 1 : (n + kRunAgents - 1) / kRunAgents;
  // resident blocks only (6 per SM): each copies the tables into shared memory once
  const size_t csmem =
      grid_smem_bytes(ctx->grid) + (ctx->d_buckets ? 3 * (size_t)kAxisBuckets : 0);
  static PerDevice csmem_set;
  if (csmem_set.needed(ctx->device)) {
    const int rows = (int)(sizeof(BoxKeys) * 3 * kMaxAxis), tabs = rows + 3 * kAxisBuckets;
    const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
    cudaFuncSetAttribute(classify_kernel<true, kAgentRounds>, attr, tabs);
    cudaFuncSetAttribute(classify_kernel<true, 1>, attr, tabs);
    cudaFuncSetAttribute(classify_kernel<false, kAgentRounds>, attr, rows);
    cudaFuncSetAttribute(classify_kernel<false, 1>, attr, rows);
    csmem_set.done(ctx->device);
  }
  const u64 cgrid = blocks < (u64)ctx->num_sms * 6 ? blocks : (u64)ctx->num_sms * 6;
  prof_begin(ctx, s);
  const auto classify = rounds == 1
                            ? (ctx->d_buckets ? classify_kernel<true, 1> : classify_kernel<false, 1>)
                            : (ctx->d_buckets ? classify_kernel<true, kAgentRounds>
                                              : classify_kernel<false, kAgentRounds>);
  launch_chained(classify, (unsigned)cgrid, kClassifyThreads, csmem, s,
      reinterpret_cast<const u64*>(soa->x), reinterpret_cast<const u64*>(soa->y),
      reinterpret_cast<const u64*>(soa->z), n, ctx->d_grid, ctx->d_buckets, blocks, out->owner,
      out->mask, ctx->tile_cnt, runs, ctx->d_status, ctx->d_stats, ctx->rs_hist);
  if ((st = check_launch(ctx, "classify_kernel", s)) != TERA_OK) return st;
  if ((st = scan_u32(ctx, ctx->tile_cnt, ctx->tile_base, nullptr, runs, s)) != TERA_OK)
    return st;

  const u64 P = ctx->n_pairs;
  const u64 cap = out->idx_capacity;
  const u64* total_ptr = ctx->tile_base + runs;
  if (cap > 0 || n > 0) {
    prof_begin(ctx, s);
    launch_chained(rounds == 1 ? emit_kernel<1> : emit_kernel<kAgentRounds>, (unsigned)blocks, kClassifyThreads, 0, s, 
        out->owner, out->mask, n, ctx->tile_base, runs, ctx->keys_a, ctx->ent_agent, cap,
        ctx->d_status);
    if ((st = check_launch(ctx, "emit_kernel", s)) != TERA_OK) return st;
  }
  const SortBufs bufs{ctx->keys_b,   ctx->keys_c,   ctx->vals_b, ctx->vals_c,
                      ctx->agents_b, ctx->agents_c, ctx->rs_hist};
  const u32* sorted = nullptr;
  if ((st = radix_sort_entries(ctx, bufs, ctx->keys_a, ctx->ent_agent, ctx->ent_dest, out->pair_idx,
                               total_ptr, cap, P, &sorted, s)) != TERA_OK)
    return st;
  ctx->rec_pair = const_cast<u32*>(sorted);
  ctx->pack_n = soa->n;
  prof_begin(ctx, s);
  const bool warp = P <= kWarpPairs;
  launch_chained(warp ? pair_off_kernel<true> : pair_off_kernel<false>,
                 (unsigned)(P / (warp ? 8 : 256) + 1), 256, 0, s,
      sorted, total_ptr, cap, P, reinterpret_cast<u64*>(out->pair_off),
      reinterpret_cast<u64*>(out->pair_count), ctx->d_total, ctx->d_stats, ctx->d_status);
  return check_launch(ctx, "pair_off_kernel", s);
}
