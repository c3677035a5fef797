// k_index.cu -- index construction on the device: position updates, Morton
// keys, radix sort of the objects, and PR-quadtree leaves.
//
// Paper steps: batch processing of updates (Sec. 2.2), Alg. 1
// (GPUcalculateMortonHash, GPUradixSort, GPUdetectQuadrants +
// CPUcheckQuadrants), uniform grid indexing (Sec. 5.2).
#include <cstddef>

#include "mqr_internal.cuh"

namespace mqr {

// ---------------------------------------------------------------------------
// a1: apply updates.  Sec. 2.2: only the most recent update of an object in a
// tick is kept.  Each update i of id carries the stamp (epoch << 32 | i); the
// largest stamp of the call wins (later call = larger epoch), then only the
// winning update writes the position.
// ---------------------------------------------------------------------------
//
// Four updates of a thread are in flight (a block apart, so that every load is
// coalesced): both kernels wait on memory, the second on two dependent steps.
constexpr uint32_t kUpdThreads = 256, kUpdItems = 4;

__global__ void __launch_bounds__(kUpdThreads)
stamp_kernel(const uint32_t *__restrict__ ids, uint32_t n, uint32_t nmax,
             unsigned long long epoch, unsigned long long *__restrict__ stamp, unsigned long long *err) {
    const uint32_t i0 = blockIdx.x * (kUpdThreads * kUpdItems) + threadIdx.x;
    if (i0 >= n) return;
    const uint32_t left = n - i0;
    uint32_t id[kUpdItems];
#pragma unroll
    for (uint32_t u = 0; u < kUpdItems; ++u)
        if (u * kUpdThreads < left) id[u] = __ldg(ids + i0 + u * kUpdThreads);
#pragma unroll
    for (uint32_t u = 0; u < kUpdItems; ++u) {
        if (u * kUpdThreads >= left) break;
        if (id[u] >= nmax) atomicOr(err, kErrBadId);
        else atomicMax(stamp + id[u], (epoch << 32) | (i0 + u * kUpdThreads));
    }
}

__global__ void __launch_bounds__(kUpdThreads)
write_winner_kernel(const uint32_t *__restrict__ ids, const float2 *__restrict__ xy,
                    uint32_t n, uint32_t nmax, unsigned long long epoch,
                    const unsigned long long *__restrict__ stamp, float2 *__restrict__ pos) {
    const uint32_t i0 = blockIdx.x * (kUpdThreads * kUpdItems) + threadIdx.x;
    if (i0 >= n) return;
    const uint32_t left = n - i0;
    uint32_t id[kUpdItems];
    float2 v[kUpdItems];
    unsigned long long s[kUpdItems];
#pragma unroll
    for (uint32_t u = 0; u < kUpdItems; ++u) {
        id[u] = 0xffffffffu;
        if (u * kUpdThreads < left) {
            id[u] = __ldg(ids + i0 + u * kUpdThreads);
            v[u] = __ldg(xy + i0 + u * kUpdThreads);
        }
    }
#pragma unroll
    for (uint32_t u = 0; u < kUpdItems; ++u)
        if (id[u] < nmax) s[u] = __ldg(stamp + id[u]);
#pragma unroll
    for (uint32_t u = 0; u < kUpdItems; ++u)
        if (id[u] < nmax && s[u] == ((epoch << 32) | (i0 + u * kUpdThreads))) pos[id[u]] = v[u];
}

void launch_apply_updates(cudaStream_t st, const uint32_t *ids, const float2 *xy, uint32_t n,
                          uint32_t nmax, unsigned long long epoch, unsigned long long *stamp,
                          float2 *pos, unsigned long long *err) {
    if (n == 0) return;
    const uint32_t per = kUpdThreads * kUpdItems, g = n / per + (n % per ? 1u : 0u);
    stamp_kernel<<<g, kUpdThreads, 0, st>>>(ids, n, nmax, epoch, stamp, err);
    write_winner_kernel<<<g, kUpdThreads, 0, st>>>(ids, xy, n, nmax, epoch, stamp, pos);
}

// Object state snapshots (checkpoint / restart): the present flags of the
// slots out of the update stamps, and stamps back from flags (a restored
// object counts as updated by the restoring call, so later calls win).
__global__ void state_flags_kernel(const unsigned long long *__restrict__ stamp, uint32_t nmax,
                                   uint8_t *__restrict__ present) {
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < nmax; i += gridDim.x * blockDim.x)
        present[i] = stamp[i] != 0ull ? 1 : 0;
}
__global__ void state_stamps_kernel(const uint8_t *__restrict__ present, uint32_t nmax, unsigned long long epoch,
                                    unsigned long long *__restrict__ stamp) {
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < nmax; i += gridDim.x * blockDim.x)
        stamp[i] = present[i] ? (epoch << 32) : 0ull;
}
void launch_state_flags(cudaStream_t st, const unsigned long long *stamp, uint32_t nmax, uint8_t *present) {
    if (nmax) state_flags_kernel<<<(nmax + 255) / 256, 256, 0, st>>>(stamp, nmax, present);
}
void launch_state_stamps(cudaStream_t st, const uint8_t *present, uint32_t nmax, unsigned long long epoch,
                         unsigned long long *stamp) {
    if (nmax) state_stamps_kernel<<<(nmax + 255) / 256, 256, 0, st>>>(present, nmax, epoch, stamp);
}

// ---------------------------------------------------------------------------
// The start of a tick: clears the arena (bytes a multiple of 16, Info first)
// and takes over the update kernels' error bits (upd_err) or, for a slot, the
// snapshot's counters and error bits (snap: n_present, n_leaves, max_level,
// err).  One launch instead of a memset and two or three small copies, each of
// which cost a dependent step of about 2 us on the stream.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256)
tick_begin_kernel(uint4 *__restrict__ arena, size_t n16, unsigned long long *upd_err,
                  const unsigned long long *__restrict__ snap) {
    constexpr size_t kInfo16 = (sizeof(Info) + 15) / 16;
    const size_t i0 = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    for (size_t i = i0; i < n16; i += (size_t)gridDim.x * blockDim.x)
        if (i >= kInfo16) arena[i] = make_uint4(0u, 0u, 0u, 0u);
    if (i0 < sizeof(Info) / 8) {
        unsigned long long v = 0;
        if (i0 == offsetof(Info, err) / 8) {
            v = snap ? snap[3] : *upd_err;
            if (!snap) *upd_err = 0;
        } else if (snap && i0 < 3) {
            v = snap[i0];
        }
        reinterpret_cast<unsigned long long *>(arena)[i0] = v;
    }
}

void launch_tick_begin(cudaStream_t st, void *arena, size_t bytes, unsigned long long *upd_err,
                       const unsigned long long *snap) {
    static_assert(offsetof(Info, n_present) == 0 && offsetof(Info, n_leaves) == 8 && offsetof(Info, max_level) == 16 &&
                      sizeof(Info) <= 256 * 8, "the counters a snapshot hands over, and one block for Info");
    const size_t n16 = bytes / 16;
    const unsigned grid = (unsigned)((n16 + 1023) / 1024 < 304 ? (n16 + 1023) / 1024 : 304);
    tick_begin_kernel<<<grid ? grid : 1, 256, 0, st>>>(reinterpret_cast<uint4 *>(arena), n16, upd_err, snap);
}

constexpr uint32_t kSortDirectGroups = 32;      // tiles add up to this many group rows themselves (see a3)

// A tile's count of one digit into the coarse rows (layout: see a3).
__device__ __forceinline__ void add_digit_count(uint32_t *group_counts, uint32_t tile, uint32_t d, uint32_t c,
                                                uint32_t n) {
    atomicAdd(group_counts + (size_t)(kSortTotalRows + tile / kSortGroup) * 256 + d, c);
    if (sort_groups(n) <= kSortDirectGroups) atomicAdd(group_counts + (tile % kSortTotalRows) * 256 + d, c);
}

// ---------------------------------------------------------------------------
// a2: Morton keys at l_max = 15 of every slot, fused with the first sort
// pass's digit counts (a block covers exactly one sort tile) and the count of
// present objects.  Bound by memory: 16 B read and 8 B written per slot (18 us
// at 4M slots, 5.3 TB/s; 24 with counts of all four digits; 105 -> 59 at 12M
// slots of 256 worlds, each block searching the worlds of its ends only).
// stamp may be null: every object is present (info may then be null too).
// ---------------------------------------------------------------------------
constexpr int kMortonBatch = 4;           // slots of a thread in flight (eight at 2 blocks per SM: 36 us against 26 at 4M)

__global__ void __launch_bounds__(kSortThreads, 3)
morton_kernel(const float2 *__restrict__ pos, const unsigned long long *__restrict__ stamp,
              uint32_t nmax, float x0, float y0, float sx, float sy, Worlds worlds,
              unsigned long long *__restrict__ keys, uint32_t *__restrict__ tile_counts,
              uint32_t *__restrict__ group_counts, Info *info) {
    __shared__ uint32_t s_hist[256];
    __shared__ uint32_t s_cnt, s_w[2];
    const int tid = threadIdx.x;
    const uint32_t base = blockIdx.x * kSortTile;
    if (tid < 256) s_hist[tid] = 0;
    if (tid == 256) s_cnt = 0;
    if (worlds.n && tid < 64) {                        // the worlds of the block's first and last slot
        const uint32_t w = world_of_warp(tid < 32 ? base : min(base + kSortTile, nmax) - 1u, worlds.obj_base, worlds.n);
        if ((tid & 31) == 0) s_w[tid >> 5] = w;
    }
    __syncthreads();
    const uint32_t w0 = worlds.n ? s_w[0] : 0u, w1 = worlds.n ? s_w[1] + 1u : 0u;
    uint32_t present = 0;
#pragma unroll 1
    for (int b = 0; b < kSortItems; b += kMortonBatch) {
        float2 p[kMortonBatch];
        unsigned long long st[kMortonBatch];
#pragma unroll
        for (int it = 0; it < kMortonBatch; ++it) {
            const uint32_t i = base + (b + it) * kSortThreads + tid;
            if (i < nmax) {
                p[it] = __ldg(pos + i);
                st[it] = stamp ? __ldg(stamp + i) : 1ull;
            }
        }
#pragma unroll
        for (int it = 0; it < kMortonBatch; ++it) {
            const uint32_t i = base + (b + it) * kSortThreads + tid;
            if (i >= nmax) break;
            uint32_t k = kAbsentKey;
            if (st[it] != 0ull) {
                uint32_t ci = cell_of(p[it].x, x0, sx), cj = cell_of(p[it].y, y0, sy);
                if (worlds.n) {
                    const uint32_t w = world_of(i, worlds.obj_base, w0, w1);
                    ci = world_cell(ci, w, worlds.bits, 0);
                    cj = world_cell(cj, w, worlds.bits, 1);
                }
                k = morton2(ci, cj);
                ++present;
            }
            keys[i] = ((unsigned long long)k << 32) | i;
            atomicAdd(&s_hist[k & 255u], 1u);
        }
    }
    present = warp_sum(present);
    if ((tid & 31) == 0 && present) atomicAdd(&s_cnt, present);
    __syncthreads();
    if (tid < 256) {
        const uint32_t c = s_hist[tid];
        tile_counts[(size_t)blockIdx.x * 256 + tid] = c;
        if (c) add_digit_count(group_counts, blockIdx.x, tid, c, nmax);
    }
    if (info && tid == 0 && s_cnt) atomicAdd(&info->n_present, (unsigned long long)s_cnt);
}

void launch_morton_keys(cudaStream_t st, const float2 *pos, const unsigned long long *stamp,
                        uint32_t nmax, float x0, float y0, float sx, float sy, Worlds worlds,
                        unsigned long long *keys, uint32_t *tile_counts, uint32_t *group_counts, Info *info) {
    if (nmax == 0) return;
    morton_kernel<<<sort_tiles(nmax), kSortThreads, 0, st>>>(pos, stamp, nmax, x0, y0, sx, sy, worlds, keys,
                                                             tile_counts, group_counts, info);
}

// ---------------------------------------------------------------------------
// a3: one pass of a stable LSD radix sort (8-bit digit at `shift`): per-tile
// digit counts, then a rank-and-scatter kernel that finds the start of every
// tile's digit runs from those counts, so no tile waits for another.
//
// Digit counts, rows of 256 adjacent words: tile_counts[t][d] for every tile
// of kSortTile keys; group_counts: kSortTotalRows rows that add up to the
// digits' totals, then a row for every kSortGroup tiles (zeroed by the caller,
// accumulated by the counting kernels; one row of totals met 1,000 additions
// per word at 4M keys: tile counts 9.4 us against 6).  A tile's run of digit d starts at
//   digit start(d) + sum of the rows of earlier groups
//                  + sum of tile_counts[t'][d], t' < t in the same group,
// the digit starts being the scan of the totals.
// Up to kSortDirectGroups groups the tile adds the rows itself (coalesced,
// independent loads); above, group_scan_kernel turns the group rows into
// starts first, so that a tile never reads more than kSortGroup rows.
//
// Measured, all four passes with their counts (before: tile counts, a scan
// kernel per digit over the tiles, match-any ranking): 0.089 -> 0.061 ms at
// 1M objects, 0.209 -> 0.149 ms at 4M, 0.534 -> 0.367 ms at 12M.
// ---------------------------------------------------------------------------

__global__ void __launch_bounds__(kSortThreads)
tile_hist_kernel(const unsigned long long *__restrict__ in, uint32_t n, int shift,
                 uint32_t *__restrict__ tile_counts, uint32_t *__restrict__ group_counts) {
    __shared__ uint32_t s_h[256];
    const int tid = threadIdx.x;
    if (tid < 256) s_h[tid] = 0;
    const uint32_t base = blockIdx.x * kSortTile;
    unsigned long long k[kSortItems];
    const bool whole = base + kSortTile <= n;
    if (whole) {                      // 16-byte loads: the tile starts at a multiple of 4,096 keys
        const ulonglong2 *in2 = reinterpret_cast<const ulonglong2 *>(in + base);
#pragma unroll
        for (int it = 0; it < kSortItems / 2; ++it) {
            const ulonglong2 v = __ldg(in2 + it * kSortThreads + tid);
            k[2 * it] = v.x;
            k[2 * it + 1] = v.y;
        }
    } else {
#pragma unroll
        for (int it = 0; it < kSortItems; ++it) {
            const uint32_t i = base + it * kSortThreads + tid;
            k[it] = i < n ? __ldg(in + i) : 0ull;
        }
    }
    __syncthreads();
#pragma unroll
    for (int it = 0; it < kSortItems; ++it)
        if (whole || base + it * kSortThreads + tid < n) atomicAdd(&s_h[(uint32_t)(k[it] >> shift) & 255u], 1u);
    __syncthreads();
    if (tid < 256) {
        const uint32_t c = s_h[tid];
        tile_counts[(size_t)blockIdx.x * 256 + tid] = c;
        if (c) add_digit_count(group_counts, blockIdx.x, tid, c, n);
    }
}

// group_counts[g][d] -> digit start(d) + the keys of digit d in earlier
// groups.  One block: thread (r, d) takes the r-th quarter of the groups.
__global__ void __launch_bounds__(1024)
group_scan_kernel(uint32_t *__restrict__ group_counts, uint32_t groups) {
    __shared__ uint32_t s_part[4][256];
    __shared__ uint32_t s_scan[256 / 32];
    const int tid = threadIdx.x, d = tid & 255, r = tid >> 8, lane = tid & 31;
    const uint32_t per = (groups + 3) / 4, g0 = min(groups, r * per), g1 = min(groups, g0 + per);
    uint32_t sum = 0;
#pragma unroll 8
    for (uint32_t g = g0; g < g1; ++g) sum += group_counts[(size_t)g * 256 + d];
    s_part[r][d] = sum;
    __syncthreads();
    uint32_t inc = 0, tot = 0;
    if (r == 0) {                     // digit starts: the scan of the 256 totals
        tot = s_part[0][d] + s_part[1][d] + s_part[2][d] + s_part[3][d];
        inc = warp_incl_scan(tot);
        if (lane == 31) s_scan[d >> 5] = inc;
    }
    __syncthreads();
    if (r == 0) {
        uint32_t run = inc - tot;
        for (int w = 0; w < (d >> 5); ++w) run += s_scan[w];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t v = s_part[k][d];
            s_part[k][d] = run;
            run += v;
        }
    }
    __syncthreads();
    uint32_t run = s_part[r][d];
#pragma unroll 8
    for (uint32_t g = g0; g < g1; ++g) {
        const uint32_t v = group_counts[(size_t)g * 256 + d];
        group_counts[(size_t)g * 256 + d] = run;
        run += v;
    }
}

// The lanes of the warp whose digit equals this lane's: one ballot per bit.
// (match-any takes a turn per distinct digit, about 80 cycles for 32 random
// ones, and bound the pass; eight ballots and their selects issue in 10.)
__device__ __forceinline__ uint32_t digit_peers(uint32_t d) {
    uint32_t m = 0xffffffffu;
#pragma unroll
    for (int b = 0; b < 8; ++b) {
        const bool p = (d >> b) & 1u;
        const uint32_t v = __ballot_sync(0xffffffffu, p);
        m &= p ? v : ~v;
    }
    return m;
}

// Rank and scatter one tile.  Warps rank their keys in private digit counts
// (stable: items in order, lanes in order); four warps turn the counts into
// positions in the tile while eight others add up the tile's output starts;
// the keys are then put in digit order in shared memory and stored run by
// run, consecutive threads to consecutive addresses.  Keys past n are all
// ones: they rank behind every key of the last digit and are not stored.
template <bool FINAL>
__global__ void __launch_bounds__(kSortThreads, 3)               // 3 tiles in flight per SM (40 registers)
sort_pass_kernel(const unsigned long long *__restrict__ in, unsigned long long *__restrict__ out,
                 uint32_t n, int shift, const uint32_t *__restrict__ tile_counts, const uint32_t *__restrict__ group_counts,
                 int groups_scanned, unsigned long long *err, const float2 *__restrict__ pos,
                 uint32_t *__restrict__ skey, uint32_t *__restrict__ sid, float2 *__restrict__ sxy) {
    constexpr int W = kSortThreads / 32;
    static_assert(kSortThreads >= 384 && W * 256 * 2 == kSortThreads * 16, "warp roles and the 16-byte clear");
    __shared__ unsigned long long s_keys[kSortTile];
    __shared__ __align__(16) uint16_t s_whist[W][256];   // per-warp digit counts, then positions in the tile
    __shared__ uint32_t s_gbase[256], s_dstart[256];
    __shared__ uint32_t s_part[4], s_part2[8];

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t tile = blockIdx.x;
    const uint32_t base = tile * kSortTile;
    const uint32_t wbase = base + warp * 32 * kSortItems;
    const uint32_t lt = lanemask_lt();

    unsigned long long k[kSortItems];
#pragma unroll
    for (int it = 0; it < kSortItems; ++it) {
        const uint32_t idx = wbase + it * 32 + lane;
        k[it] = idx < n ? in[idx] : ~0ull;
    }
    reinterpret_cast<uint4 *>(&s_whist[0][0])[tid] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    uint16_t *wh = s_whist[warp];
    uint32_t r[kSortItems / 2];                    // ranks in the warp's keys (at most 256), two to a register
#pragma unroll
    for (int it = 0; it < kSortItems; ++it) {
        const uint32_t dg = (uint32_t)(k[it] >> shift) & 255u;
        const uint32_t peers = digit_peers(dg);
        const uint32_t rank = wh[dg] + __popc(peers & lt);
        __syncwarp();
        if ((peers >> lane) == 1u) wh[dg] = (uint16_t)(rank + 1u);      // the last of its peers
        __syncwarp();
        if (it & 1) r[it / 2] |= rank << 16;
        else r[it / 2] = rank;
    }
    __syncthreads();

    if (warp < 4) {
        // digits 2 tid and 2 tid + 1, packed: the warps' exclusive counts, then the digits' starts
        uint32_t c = 0;
        uint32_t *col = reinterpret_cast<uint32_t *>(&s_whist[0][0]) + tid;
#pragma unroll
        for (int w = 0; w < W; ++w) c += col[w * 128];
        const uint32_t c0 = c & 0xffffu, c1 = c >> 16;
        const uint32_t inc = warp_incl_scan(c0 + c1);
        if (lane == 31) s_part[warp] = inc;
        asm volatile("bar.sync 1, 128;" ::: "memory");
        uint32_t d0 = inc - c0 - c1;
        for (int w = 0; w < warp; ++w) d0 += s_part[w];
        s_dstart[2 * tid] = d0;
        s_dstart[2 * tid + 1] = d0 + c0;
        uint32_t run = d0 | ((d0 + c0) << 16);         // positions are below 4,096: no carry between the halves
#pragma unroll 4
        for (int w = 0; w < W; ++w) {
            const uint32_t v = col[w * 128];
            col[w * 128] = run;
            run += v;
        }
    } else if (warp < 12) {
        const uint32_t d = tid - 128, g = tile / kSortGroup;
        uint32_t start = 0;
        if (groups_scanned) {
            start = __ldg(group_counts + (size_t)(kSortTotalRows + g) * 256 + d);
        } else {
            uint32_t total = 0, before = 0;
#pragma unroll
            for (uint32_t j = 0; j < kSortTotalRows; ++j) total += __ldg(group_counts + (size_t)j * 256 + d);
#pragma unroll 8
            for (uint32_t j = 0; j < g; ++j) before += __ldg(group_counts + (size_t)(kSortTotalRows + j) * 256 + d);
            const uint32_t inc = warp_incl_scan(total);
            if (lane == 31) s_part2[d >> 5] = inc;
            asm volatile("bar.sync 2, 256;" ::: "memory");
            start = inc - total + before;
            for (uint32_t w = 0; w < (d >> 5); ++w) start += s_part2[w];
        }
#pragma unroll 8
        for (uint32_t t = g * kSortGroup; t < tile; ++t) start += __ldg(tile_counts + (size_t)t * 256 + d);
        s_gbase[d] = start;
    }
    __syncthreads();

#pragma unroll
    for (int it = 0; it < kSortItems; ++it) {
        const uint32_t dg = (uint32_t)(k[it] >> shift) & 255u;
        s_keys[wh[dg] + ((it & 1) ? r[it / 2] >> 16 : r[it / 2] & 0xffffu)] = k[it];
    }
    if (tid < 256) s_gbase[tid] -= s_dstart[tid];
    __syncthreads();

    const uint32_t nvalid = n - base < (uint32_t)kSortTile ? n - base : (uint32_t)kSortTile;
    if constexpr (FINAL) {
        // The last pass splits keys and ids and, unless sxy is null, gathers
        // each object's position by id (random reads),
        // four gathers of a thread in flight.  (Eight at 64 registers, two
        // tiles per SM: 49 us against 45 at 4M objects, 116 against 103 at 12M.)
#pragma unroll 1
        for (int b = 0; b < kSortItems; b += 4) {
            float2 pv[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const uint32_t i = tid + (b + j) * kSortThreads;
                if (i < nvalid) {
                    const unsigned long long key = s_keys[i];
                    if (sxy && (uint32_t)(key >> 32) != kAbsentKey) pv[j] = pos[(uint32_t)key];
                }
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const uint32_t i = tid + (b + j) * kSortThreads;
                if (i >= nvalid) continue;
                const unsigned long long key = s_keys[i];
                const uint32_t o = s_gbase[(uint32_t)(key >> shift) & 255u] + i;
                if (o >= n) {
                    atomicOr(err, kErrInternal);
                    continue;
                }
                skey[o] = (uint32_t)(key >> 32);
                sid[o] = (uint32_t)key;
                if (sxy && (uint32_t)(key >> 32) != kAbsentKey) sxy[o] = pv[j];
            }
        }
    } else {
        for (uint32_t i = tid; i < nvalid; i += kSortThreads) {
            const unsigned long long key = s_keys[i];
            const uint32_t o = s_gbase[(uint32_t)(key >> shift) & 255u] + i;
            if (o >= n) {
                atomicOr(err, kErrInternal);
                continue;
            }
            out[o] = key;
        }
    }
}

void launch_sort_pass(cudaStream_t st, const unsigned long long *in, unsigned long long *out, uint32_t n,
                      int shift, uint32_t *tile_counts, uint32_t *group_counts, bool counts_ready,
                      unsigned long long *err, bool final_obj, const float2 *pos, uint32_t *skey, uint32_t *sid,
                      float2 *sxy) {
    if (n == 0) return;
    const uint32_t tiles = sort_tiles(n), groups = sort_groups(n);
    if (!counts_ready) tile_hist_kernel<<<tiles, kSortThreads, 0, st>>>(in, n, shift, tile_counts, group_counts);
    const int scanned = groups > kSortDirectGroups ? 1 : 0;
    if (scanned) group_scan_kernel<<<1, 1024, 0, st>>>(group_counts + (size_t)kSortTotalRows * 256, groups);
    if (final_obj)
        sort_pass_kernel<true><<<tiles, kSortThreads, 0, st>>>(in, out, n, shift, tile_counts, group_counts, scanned,
                                                              err, pos, skey, sid, sxy);
    else
        sort_pass_kernel<false><<<tiles, kSortThreads, 0, st>>>(in, out, n, shift, tile_counts, group_counts, scanned,
                                                               err, nullptr, nullptr, nullptr, nullptr);
}

uint32_t sort_pass_launches(uint32_t n, bool counts_ready) {
    if (n == 0) return 0;
    return 1u + (counts_ready ? 0u : 1u) + (sort_groups(n) > kSortDirectGroups ? 1u : 0u);
}

// ---------------------------------------------------------------------------
// a2 + a3 for small populations: keys and all four sort passes in one launch,
// by one thread-block cluster.  The keys never leave the SMs: every block
// ranks its keys in shared memory, the blocks read each other's 256 digit
// totals, and each key is stored into the shared memory of the block that
// holds its new position (two cluster barriers per pass).  Launches, barriers
// and latency bound a sort of this size.  Keys and sort, by events: 58 us ->
// 21 at 4,096 objects, 62 -> 27 at 16,384, 69 -> 46 at 65,536; at 131,072 the
// passes of a launch each (71 us) are faster than this kernel (75).
// ---------------------------------------------------------------------------
constexpr int kSmallThreads = 1024, kSmallWarps = kSmallThreads / 32;

__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t cluster_map(uint32_t saddr, uint32_t rank) {
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(saddr), "r"(rank));
    return a;
}

// The grid is one cluster; block r holds the positions [r * T, (r + 1) * T),
// T = 1024 * ITEMS.  stamp may be null (every object is present), sxy and
// info too (keys and ids only).
template <int ITEMS>
__global__ void __launch_bounds__(kSmallThreads, 1)
small_sort_kernel(const float2 *__restrict__ pos, const unsigned long long *__restrict__ stamp, uint32_t n,
                  float x0, float y0, float sx, float sy, Worlds worlds, uint32_t *__restrict__ skey,
                  uint32_t *__restrict__ sid, float2 *__restrict__ sxy, Info *info) {
    constexpr uint32_t T = kSmallThreads * ITEMS;
    extern __shared__ unsigned long long s_keys[];              // T keys
    __shared__ __align__(16) uint16_t s_whist[kSmallWarps][256];
    __shared__ uint32_t s_seg[8][128];                          // digit pairs: counts of eight groups of four warps
    __shared__ uint32_t s_tot[256], s_base[256], s_part[8], s_cnt;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t rank = cluster_rank(), nblocks = gridDim.x;
    const uint32_t p0 = rank * T + warp * 32 * ITEMS + lane;
    const uint32_t lt = lanemask_lt();
    const uint32_t keys_addr = (uint32_t)__cvta_generic_to_shared(s_keys);
    const uint32_t tot_addr = (uint32_t)__cvta_generic_to_shared(s_tot);
    if (tid == 0) s_cnt = 0;

    unsigned long long k[ITEMS];
    uint32_t present = 0;
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) {
        const uint32_t i = p0 + it * 32;
        k[it] = ~0ull;
        if (i < n) {
            uint32_t key = kAbsentKey;
            if (!stamp || stamp[i] != 0ull) {
                const float2 p = pos[i];
                uint32_t ci = cell_of(p.x, x0, sx), cj = cell_of(p.y, y0, sy);
                if (worlds.n) {
                    const uint32_t w = world_of(i, worlds.obj_base, 0, worlds.n);
                    ci = world_cell(ci, w, worlds.bits, 0);
                    cj = world_cell(cj, w, worlds.bits, 1);
                }
                key = morton2(ci, cj);
                ++present;
            }
            k[it] = ((unsigned long long)key << 32) | i;
        }
    }
    __syncthreads();
    if (info) {
        present = warp_sum(present);
        if (lane == 0 && present) atomicAdd(&s_cnt, present);
    }
#pragma unroll 1
    for (int shift = 32; shift < 64; shift += 8) {
        if (shift > 32) {
#pragma unroll
            for (int it = 0; it < ITEMS; ++it) k[it] = s_keys[warp * 32 * ITEMS + it * 32 + lane];
        }
        reinterpret_cast<uint4 *>(&s_whist[0][0])[tid] = make_uint4(0u, 0u, 0u, 0u);
        __syncthreads();
        uint16_t *wh = s_whist[warp];
        uint32_t r[(ITEMS + 1) / 2];                            // ranks in the warp's keys (at most 128)
#pragma unroll
        for (int it = 0; it < ITEMS; ++it) {
            const uint32_t dg = (uint32_t)(k[it] >> shift) & 255u;
            const uint32_t peers = digit_peers(dg);
            const uint32_t rk = wh[dg] + __popc(peers & lt);
            __syncwarp();
            if ((peers >> lane) == 1u) wh[dg] = (uint16_t)(rk + 1u);
            __syncwarp();
            if (it & 1) r[it / 2] |= rk << 16;
            else r[it / 2] = rk;
        }
        __syncthreads();
        // the warps' counts to the block's exclusive counts, two digits to a
        // word: thread (g, c) takes digit pair c of four warps
        {
            const int g = tid >> 7, c = tid & 127;
            uint32_t *col = reinterpret_cast<uint32_t *>(&s_whist[0][0]) + g * 4 * 128 + c;
            uint32_t v[4], sum = 0;
#pragma unroll
            for (int w = 0; w < 4; ++w) {
                v[w] = col[w * 128];
                sum += v[w];
            }
            s_seg[g][c] = sum;
            __syncthreads();
            uint32_t run = 0, tot = 0;
#pragma unroll
            for (int h = 0; h < 8; ++h) {
                const uint32_t x = s_seg[h][c];
                if (h < g) run += x;
                tot += x;
            }
#pragma unroll
            for (int w = 0; w < 4; ++w) {
                col[w * 128] = run;
                run += v[w];
            }
            if (g == 0) {
                s_tot[2 * c] = tot & 0xffffu;
                s_tot[2 * c + 1] = tot >> 16;
            }
        }
        cluster_barrier();                                      // every block's totals are out, its keys read
        uint32_t before = 0, all = 0, inc = 0;
        if (tid < 256) {
            for (uint32_t q = 0; q < nblocks; ++q) {
                uint32_t v;
                asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(cluster_map(tot_addr, q) + 4u * tid));
                if (q < rank) before += v;
                all += v;
            }
            inc = warp_incl_scan(all);
            if (lane == 31) s_part[warp] = inc;
        }
        __syncthreads();
        if (tid < 256) {
            uint32_t start = inc - all + before;
            for (int w = 0; w < warp; ++w) start += s_part[w];
            s_base[tid] = start;
        }
        __syncthreads();
#pragma unroll
        for (int it = 0; it < ITEMS; ++it) {
            const uint32_t dg = (uint32_t)(k[it] >> shift) & 255u;
            const uint32_t o = s_base[dg] + wh[dg] + ((it & 1) ? r[it / 2] >> 16 : r[it / 2] & 0xffffu);
            asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(cluster_map(keys_addr, o / T) + 8u * (o % T)),
                         "l"(k[it]) : "memory");
        }
        cluster_barrier();                                      // the keys have arrived
    }
    if (info && tid == 0 && s_cnt) atomicAdd(&info->n_present, (unsigned long long)s_cnt);
#pragma unroll 4
    for (uint32_t j = tid; j < T; j += kSmallThreads) {
        const uint32_t o = rank * T + j;
        if (o >= n) break;
        const unsigned long long key = s_keys[j];
        skey[o] = (uint32_t)(key >> 32);
        sid[o] = (uint32_t)key;
        if (sxy && (uint32_t)(key >> 32) != kAbsentKey) sxy[o] = pos[(uint32_t)key];
    }
}

// A cluster of at most 16 blocks (twice the portable size: at 32,768 objects
// 33 us against 42 with eight blocks of twice the keys).
constexpr uint32_t kSmallBlocks = 16;
static_assert(kSmallSortMax == kSmallBlocks * kSmallThreads * 4, "four items at most");

template <int ITEMS>
static cudaLaunchConfig_t small_config(uint32_t n, cudaStream_t st, cudaLaunchAttribute *attr) {
    constexpr uint32_t T = kSmallThreads * ITEMS;
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = (n + T - 1) / T;
    attr->val.clusterDim.y = attr->val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((n + T - 1) / T);
    cfg.blockDim = dim3(kSmallThreads);
    cfg.dynamicSmemBytes = T * sizeof(unsigned long long);
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

template <int ITEMS>
static bool small_ready_items() {
    if (cudaFuncSetAttribute(small_sort_kernel<ITEMS>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
        return false;
    cudaLaunchAttribute attr{};
    const cudaLaunchConfig_t cfg = small_config<ITEMS>(kSmallBlocks * kSmallThreads * ITEMS, nullptr, &attr);
    int clusters = 0;
    return cudaOccupancyMaxActiveClusters(&clusters, small_sort_kernel<ITEMS>, &cfg) == cudaSuccess && clusters > 0;
}

bool small_sort_ready() {
    static_assert(kSmallThreads * 4 * sizeof(unsigned long long) + sizeof(uint16_t) * kSmallWarps * 256 + 8192 <=
                      57344, "dynamic and static shared memory");
    const bool ok = cudaFuncSetAttribute(small_sort_kernel<4>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)(kSmallThreads * 4 * sizeof(unsigned long long))) == cudaSuccess &&
                    small_ready_items<1>() && small_ready_items<2>() && small_ready_items<4>();
    if (!ok) (void)cudaGetLastError();
    return ok;
}

template <int ITEMS>
static cudaError_t launch_small_items(cudaStream_t st, const float2 *pos, const unsigned long long *stamp, uint32_t n,
                                      float x0, float y0, float sx, float sy, Worlds worlds, uint32_t *skey,
                                      uint32_t *sid, float2 *sxy, Info *info) {
    cudaLaunchAttribute attr{};
    const cudaLaunchConfig_t cfg = small_config<ITEMS>(n, st, &attr);
    return cudaLaunchKernelEx(&cfg, small_sort_kernel<ITEMS>, pos, stamp, n, x0, y0, sx, sy, worlds, skey, sid, sxy,
                              info);
}

cudaError_t launch_small_sort(cudaStream_t st, const float2 *pos, const unsigned long long *stamp, uint32_t n,
                              float x0, float y0, float sx, float sy, Worlds worlds, uint32_t *skey, uint32_t *sid,
                              float2 *sxy, Info *info) {
    if (n == 0) return cudaSuccess;
    if (n <= kSmallBlocks * kSmallThreads)
        return launch_small_items<1>(st, pos, stamp, n, x0, y0, sx, sy, worlds, skey, sid, sxy, info);
    if (n <= kSmallBlocks * kSmallThreads * 2)
        return launch_small_items<2>(st, pos, stamp, n, x0, y0, sx, sy, worlds, skey, sid, sxy, info);
    return launch_small_items<4>(st, pos, stamp, n, x0, y0, sx, sy, worlds, skey, sid, sxy, info);
}

// ---------------------------------------------------------------------------
// a4: PR-quadtree leaves by segmented counts on the Morton-sorted keys.
//
// With K the sorted keys of the N present objects and c = leaf_cap, the node
// of level l containing K[p] holds more than c objects iff some window
// K[i..i+c] with i in [p-c, p] lies inside it, i.e. iff
// shared_depth(K[i], K[i+c]) >= l.  Hence the leaf level of object p is
//     L(p) = min(15, 1 + max_{i in [p-c, p], 0 <= i, i+c < N} d[i]),
//     d[i] = shared_depth(K[i], K[i+c]),
// and L(p) = 0 (the root is the only leaf) when N <= c.  This is exactly the
// split rule of Alg. 1 (split iff count > th_quad, keep level-l_max quadrants)
// evaluated for all levels at once, on the encoded values e[i] = 1 + d[i] (0 =
// no window).  For one capacity of 8 or more, the window of p is cut at blocks
// of eight positions: a suffix of its first block, whole blocks, a prefix of
// its last; a thread builds the prefix and suffix maxima of a block in
// registers, the whole blocks come from a sparse table (doubling) of block
// maxima, an eighth of one over positions, and eight levels are combined as
// bytes of two words (45 -> 30 us at 4M objects, 105 -> 72 at 12M: the
// table over positions cost 200 instructions an object).  Per-region
// capacities keep the table over positions.  A new leaf starts at p when
// (L, K >> 2(15-L)) changes; leaves are compacted with a single-pass scan into
// the cell boundary table in Morton order.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint8_t window_enc(const uint32_t *__restrict__ K, long i, uint32_t cap,
                                              uint32_t N) {
    if (i < 0 || (unsigned long long)i + cap >= N) return 0;
    return (uint8_t)(1u + shared_depth(K[i], K[i + cap]));
}

// Global-memory variant for large capacities: G[j] = e[j - cap - 1].
__global__ void window_enc_kernel(const uint32_t *__restrict__ K, uint32_t cap, uint32_t size,
                                  const Info *info, uint8_t *__restrict__ G) {
    uint32_t N = (uint32_t)info->n_present;
    for (uint32_t j = blockIdx.x * blockDim.x + threadIdx.x; j < size; j += gridDim.x * blockDim.x)
        G[j] = window_enc(K, (long)j - (long)cap - 1, cap, N);
}
__global__ void window_double_kernel(const uint8_t *__restrict__ a, uint8_t *__restrict__ b,
                                     uint32_t size, uint32_t step) {
    for (uint32_t j = blockIdx.x * blockDim.x + threadIdx.x; j < size; j += gridDim.x * blockDim.x) {
        uint8_t v = a[j];
        if (j + step < size) v = max(v, a[j + step]);
        b[j] = v;
    }
}

__global__ void __launch_bounds__(kLeafThreads)
leaves_kernel(const uint32_t *__restrict__ K, uint32_t cap, int uniform_grid, uint32_t grid_level,
              uint32_t min_level, uint32_t region_bits, const uint32_t *__restrict__ region_cap, int kexp,
              const uint8_t *__restrict__ Mk_global, uint32_t *status,
              uint32_t *tile_counter, uint32_t *__restrict__ leaf_lo, uint32_t *__restrict__ leaf_hi,
              uint32_t *__restrict__ leaf_beg, uint32_t *__restrict__ leaf_nsub, uint2 *__restrict__ leaf_box,
              uint32_t tstride, Info *info) {
    // dynamic shared memory: the block tables of the single capacity, or (per-region
    // capacities) two window tables of tstride bytes each
    extern __shared__ __align__(16) uint8_t dsm[];
    __shared__ __align__(8) uint8_t s_L[8 + kLeafTile];      // level of position p at p - t0 + 8; [7]: of t0 - 1
    __shared__ uint32_t s_scan[kLeafThreads / 32 + 1];
    __shared__ uint32_t s_tile, s_prefix;
    __shared__ uint32_t s_rcap[1 << (2 * kMaxRegionBits)];   // per-region capacities, loaded up front

    const int tid = threadIdx.x;
    const uint32_t N = (uint32_t)info->n_present;
    if (tid == 0) s_tile = atomicAdd(tile_counter, 1u);
    if (region_bits)
        for (uint32_t i = tid; i < (1u << (2 * region_bits)); i += kLeafThreads) s_rcap[i] = region_cap[i];
    __syncthreads();
    const uint32_t tile = s_tile;
    const long t0 = (long)tile * kLeafTile;
    if (t0 >= (long)N) return;
    const long tend = min((long)N, t0 + kLeafTile);

    const bool root_only = !uniform_grid && !region_bits && cap >= N;
    if (region_bits) {
        // Per-region capacities: the nodes of depth region_bits are regions,
        // region r (Morton prefix r) splitting its nodes at region_cap[r].
        // The positions of one region are contiguous; for each region the
        // tile meets, the window rule runs with that region's capacity.
        // Windows that leave the region share fewer than region_bits levels
        // and never raise a level above region_bits, the minimum level.
        // s_first[r - r_lo] = first position of region r (r_lo < r <= r_hi),
        // found in parallel at the positions where the region changes.
        __shared__ int s_first[(1 << (2 * kMaxRegionBits)) + 1];
        const uint32_t sh = 2u * (kLevels - region_bits);
        const long pa = t0 > 0 ? t0 - 1 : 0, pb = tend;
        const uint32_t r_lo = K[pa] >> sh, r_hi = K[pb - 1] >> sh;
        if (r_hi > r_lo) {
            for (long p = pa + 1 + tid; p < pb; p += kLeafThreads) {
                const uint32_t r0 = K[p - 1] >> sh, r1 = K[p] >> sh;
                for (uint32_t r = r0 + 1; r <= r1; ++r) s_first[r - r_lo] = (int)(p - pa);
            }
            __syncthreads();
        }
        for (uint32_t r = r_lo; r <= r_hi; ++r) {
            const long a = r == r_lo ? pa : pa + s_first[r - r_lo];
            const long b = r == r_hi ? pb : pa + s_first[r + 1 - r_lo];
            if (a < b) {
                const uint32_t rc = s_rcap[r];
                int rk = 0;
                while ((2ull << rk) <= (unsigned long long)rc + 1) ++rk;   // floor(log2(rc+1))
                const long rs = a - (long)rc;         // the window of position a starts here
                const int S = (int)(b - rs);
                uint8_t *A = dsm, *B = dsm + tstride;
                for (int j = tid; j < S; j += kLeafThreads) A[j] = window_enc(K, rs + j, rc, N);
                __syncthreads();
                for (int st = 0; st < rk; ++st) {
                    const int step = 1 << st;
                    for (int j = tid; j < S; j += kLeafThreads) {
                        uint8_t v = A[j];
                        if (j + step < S) v = max(v, A[j + step]);
                        B[j] = v;
                    }
                    __syncthreads();
                    uint8_t *t = A; A = B; B = t;
                }
                for (long p = a + tid; p < b; p += kLeafThreads) {
                    uint8_t m = max(A[p - (long)rc - rs], A[p - (1l << rk) + 1 - rs]);
                    s_L[p - t0 + 8] = m > 15 ? 15 : m;
                }
            }
            __syncthreads();
        }
    } else if (uniform_grid || root_only) {
        uint8_t lv = uniform_grid ? (uint8_t)grid_level : (uint8_t)0;
        for (int i = tid; i <= kLeafTile; i += kLeafThreads) s_L[i + 7] = lv;
    } else if (Mk_global == nullptr && cap < 8) {
        for (long p = t0 - 1 + tid; p < tend; p += kLeafThreads) {
            uint8_t m = 0;
            for (long i = p - (long)cap; i <= p; ++i) m = max(m, window_enc(K, i, cap, N));
            s_L[p - t0 + 8] = m > 15 ? 15 : m;
        }
    } else if (Mk_global == nullptr) {
        // Blocks of 8 positions from rs on; block lead is the tile's first.
        const uint32_t D = cap >> 3, rem = cap & 7u;            // a window starts D (and a part) blocks back
        const int lead = (int)((cap + 1 + 7) >> 3), nb = lead + kLeafTile / 8;
        const long rs = t0 - 8l * lead;
        unsigned long long *s_pre = reinterpret_cast<unsigned long long *>(dsm), *s_suf = s_pre + nb;
        uint8_t *A = reinterpret_cast<uint8_t *>(s_suf + nb), *B = A + nb;
        for (int blk = tid; blk < nb; blk += kLeafThreads) {
            const long j0 = rs + 8l * blk;
            uint32_t e[8];
            if (j0 >= 0 && j0 + 7 + (long)cap < (long)N) {
                uint32_t ka[8], kb[8];
                *reinterpret_cast<uint4 *>(ka) = __ldg(reinterpret_cast<const uint4 *>(K + j0));
                *reinterpret_cast<uint4 *>(ka + 4) = __ldg(reinterpret_cast<const uint4 *>(K + j0) + 1);
                if ((cap & 3u) == 0u) {
                    *reinterpret_cast<uint4 *>(kb) = __ldg(reinterpret_cast<const uint4 *>(K + j0 + cap));
                    *reinterpret_cast<uint4 *>(kb + 4) = __ldg(reinterpret_cast<const uint4 *>(K + j0 + cap) + 1);
                } else {
#pragma unroll
                    for (int i = 0; i < 8; ++i) kb[i] = __ldg(K + j0 + cap + i);
                }
#pragma unroll
                for (int i = 0; i < 8; ++i) e[i] = 1u + shared_depth(ka[i], kb[i]);
            } else {
#pragma unroll
                for (int i = 0; i < 8; ++i) e[i] = window_enc(K, j0 + i, cap, N);
            }
            uint32_t m = 0, lo = 0, hi = 0;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                m = max(m, e[i]);
                if (i < 4) lo |= m << (8 * i);
                else hi |= m << (8 * (i - 4));
            }
            s_pre[blk] = ((unsigned long long)hi << 32) | lo;
            A[blk] = (uint8_t)m;
            m = lo = hi = 0;
#pragma unroll
            for (int i = 7; i >= 0; --i) {
                m = max(m, e[i]);
                if (i < 4) lo |= m << (8 * i);
                else hi |= m << (8 * (i - 4));
            }
            s_suf[blk] = ((unsigned long long)hi << 32) | lo;
        }
        __syncthreads();
        // keep the block maxima (B) and double a copy: M[b] covers 2^kf blocks, at most D - 1
        uint8_t *M = A, *T = B, *s_m = A;
        int kf = 0;
        while ((2u << kf) <= D - 1u && D > 1u) ++kf;
        if (kf > 0) {
            s_m = B + nb;                                       // a third row
            for (int i = tid; i < nb; i += kLeafThreads) s_m[i] = A[i];
            for (int st = 0; st < kf; ++st) {
                const int step = 1 << st;
                for (int i = tid; i < nb; i += kLeafThreads) {
                    uint8_t v = M[i];
                    if (i + step < nb) v = max(v, M[i + step]);
                    T[i] = v;
                }
                __syncthreads();
                uint8_t *t = M; M = T; T = t;
            }
        }
        // the levels of block blk's eight positions, a byte each
        auto levels = [&](int blk) {
            uint32_t mid = 0;                                   // the D - 1 whole blocks before blk
            if (D > 1u) mid = max(M[blk - (int)D + 1], M[blk - (1 << kf)]);
            unsigned long long suf = s_suf[blk - (int)D];
            uint32_t mid1 = mid;
            if (rem) {                                          // the first rem positions start a block earlier
                mid1 = max(mid, (uint32_t)s_m[blk - (int)D]);
                suf = (s_suf[blk - (int)D - 1] >> (8u * (8u - rem))) | (suf << (8u * rem));
            }
            const unsigned long long pre = s_pre[blk];
            const unsigned long long head = rem ? ~0ull >> (8u * (8u - rem)) : 0ull;
            const unsigned long long mids = ((mid * 0x0101010101010101ull) & ~head) | ((mid1 * 0x0101010101010101ull) & head);
            const uint32_t lo = __vminu4(__vmaxu4(__vmaxu4((uint32_t)pre, (uint32_t)suf), (uint32_t)mids), 0x0f0f0f0fu);
            const uint32_t hi = __vminu4(__vmaxu4(__vmaxu4((uint32_t)(pre >> 32), (uint32_t)(suf >> 32)),
                                                  (uint32_t)(mids >> 32)), 0x0f0f0f0fu);
            return ((unsigned long long)hi << 32) | lo;
        };
        static_assert(kLeafTile == 8 * kLeafThreads, "a block of positions to a thread");
        *reinterpret_cast<unsigned long long *>(s_L + 8 + 8 * tid) = levels(lead + tid);
        if (tid == 0 && t0 > 0) {
            // position t0 - 1, the last of the block before: its window needs
            // blocks lead - 1 - D and, for rem > 0, nothing earlier
            uint32_t m = 0;
            for (int blk = lead - (int)D; blk < lead; ++blk) m = max(m, (uint32_t)s_m[blk]);
            const uint32_t sb = (uint32_t)(s_suf[lead - 1 - (int)D] >> (8u * (7u - rem))) & 255u;
            m = max(m, sb);
            s_L[7] = (uint8_t)min(m, 15u);
        }
    } else {
        // Global sparse table: Mk_global[j] covers e over [j-cap-1, j-cap-1+2^k).
        for (long p = t0 - 1 + tid; p < tend; p += kLeafThreads) {
            if (p < 0) continue;
            long ja = p - (long)cap + (long)cap + 1;           // position p-cap
            long jb = p - (1l << kexp) + 1 + (long)cap + 1;    // position p-2^k+1
            uint8_t m = max(Mk_global[ja], Mk_global[jb]);
            s_L[p - t0 + 8] = m > 15 ? 15 : m;
        }
    }
    __syncthreads();
    if (min_level) {           // batched worlds: no leaf above the worlds' roots
        for (int i = tid; i <= kLeafTile; i += kLeafThreads) s_L[i + 7] = max(s_L[i + 7], (uint8_t)min_level);
        __syncthreads();
    }

    // Leaf starts: thread handles positions t0 + tid*8 .. +8 (blocked).
    constexpr int PER = kLeafTile / kLeafThreads;
    const long pt = t0 + tid * PER;
    uint32_t kk[PER];
    if (pt + PER <= (long)N) {
        *reinterpret_cast<uint4 *>(kk) = __ldg(reinterpret_cast<const uint4 *>(K + pt));
        *reinterpret_cast<uint4 *>(kk + 4) = __ldg(reinterpret_cast<const uint4 *>(K + pt) + 1);
    } else {
#pragma unroll
        for (int e = 0; e < PER; ++e) kk[e] = pt + e < (long)N ? __ldg(K + pt + e) : 0u;
    }
    uint32_t kprev = pt > 0 && pt < tend ? __ldg(K + pt - 1) : 0u;
    const unsigned long long Ls = *reinterpret_cast<const unsigned long long *>(s_L + 8 + tid * PER);
    uint32_t Lprev = s_L[7 + tid * PER];
    uint32_t flags = 0, cnt = 0, maxl = 0;
#pragma unroll
    for (int e = 0; e < PER; ++e) {
        const long p = pt + e;
        const uint32_t L = (uint32_t)(Ls >> (8 * e)) & 255u;
        const uint32_t sh = 2u * (kLevels - L);
        const bool start = p == 0 || Lprev != L || (kprev >> sh) != (kk[e] >> sh);
        if (p < tend && start) {
            flags |= 1u << e;
            ++cnt;
            maxl = max(maxl, L);
        }
        kprev = kk[e];
        Lprev = L;
    }
    uint32_t total;
    uint32_t off = block_excl_scan<kLeafThreads>(cnt, &total, s_scan);
    if (tid < 32) {
        const uint32_t pre = lookback_warp<uint32_t>(status, tile, total, &info->err);
        if (tid == 0) s_prefix = pre;
    }
    __syncthreads();
    uint32_t idx = s_prefix + off;
#pragma unroll
    for (int e = 0; e < PER; ++e) {
        if (!(flags & (1u << e))) continue;
        const long p = pt + e;
        const uint32_t L = (uint32_t)(Ls >> (8 * e)) & 255u;
        const uint32_t sh = 2u * (kLevels - L);
        const uint32_t lo = (kk[e] >> sh) << sh;              // sh <= 30
        uint32_t span = sh >= 30 ? (1u << 30) - 1 : (1u << sh) - 1;
        leaf_lo[idx] = lo;
        leaf_hi[idx] = lo + span;
        leaf_beg[idx] = (uint32_t)p;
        leaf_nsub[idx] = 0;
        leaf_box[idx] = make_uint2(compact15(lo) | (compact15(lo >> 1) << 16), kLevels - L);
        ++idx;
    }
    maxl = __reduce_max_sync(0xffffffffu, maxl);
    if ((tid & 31) == 0 && maxl) atomicMax(&info->max_level, (unsigned long long)maxl);
    if (tend == (long)N && tid == 0) {
        leaf_beg[s_prefix + total] = N;
        info->n_leaves = s_prefix + total;
    }
}

// Objects per region (the Morton prefixes of length 2*region_bits) of the
// sorted keys: thread r finds the first key of regions r and r+1.
__global__ void region_counts_kernel(const uint32_t *__restrict__ K, uint32_t N, uint32_t region_bits,
                                     uint32_t *__restrict__ counts) {
    const uint32_t R = 1u << (2 * region_bits), sh = 2u * (kLevels - region_bits);
    const uint32_t r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= R) return;
    uint32_t bound[2];
    for (int e = 0; e < 2; ++e) {
        const uint32_t v = r + e;
        uint32_t a = 0, b = N;
        while (a < b) {
            const uint32_t m = a + (b - a) / 2;
            if ((K[m] >> sh) < v) a = m + 1; else b = m;
        }
        bound[e] = a;
    }
    counts[r] = bound[1] - bound[0];
}

cudaError_t launch_region_counts(cudaStream_t st, const uint32_t *skey, uint32_t n, uint32_t region_bits,
                                 uint32_t *counts) {
    const uint32_t R = 1u << (2 * region_bits);
    region_counts_kernel<<<(R + 127) / 128, 128, 0, st>>>(skey, n, region_bits, counts);
    return cudaGetLastError();
}

static constexpr size_t leaf_tables(uint32_t cap) { return (size_t)19 * (kLeafTile / 8 + (cap + 8) / 8); }

void launch_build_leaves(cudaStream_t st, const uint32_t *skey, uint32_t nmax, uint32_t cap,
                         int uniform_grid, uint32_t grid_level, uint32_t min_level, uint32_t region_bits,
                         const uint32_t *region_cap, uint8_t *mk_a, uint8_t *mk_b,
                         uint32_t *status, uint32_t *tile_counter, uint32_t *leaf_lo,
                         uint32_t *leaf_hi, uint32_t *leaf_beg, uint32_t *leaf_nsub, uint2 *leaf_box,
                         Info *info) {
    if (nmax == 0) return;
    uint32_t tiles = (nmax + kLeafTile - 1) / kLeafTile;
    int kexp = 0;
    while ((2ull << kexp) <= (unsigned long long)cap + 1) ++kexp;   // floor(log2(cap+1))
    const uint8_t *mk = nullptr;
    size_t dyn = 0;
    uint32_t tstride = 0;
    if (region_bits) {
        tstride = kLeafTile + kLeafCapSmem + 1;                   // every region capacity <= kLeafCapSmem
        dyn = 2 * (size_t)tstride;
    } else if (!uniform_grid && cap < nmax) {
        if (cap <= (uint32_t)kLeafCapSmem) {
            // prefix and suffix maxima of the blocks of 8 positions and three rows of block maxima
            dyn = leaf_tables(cap);
            static_assert(leaf_tables(kLeafCapSmem) + kLeafTile + 8 + 8 * (1 << (2 * kMaxRegionBits)) + 256 <= 48 * 1024,
                          "with the kernel's own arrays, what a launch may have without asking for more");
        } else {
            uint32_t size = nmax + cap + 1;   // cap < nmax: fits the 2*nmax+2 buffers
            window_enc_kernel<<<1024, 256, 0, st>>>(skey, cap, size, info, mk_a);
            uint8_t *a = mk_a, *b = mk_b;
            for (int s = 0; s < kexp; ++s) {
                window_double_kernel<<<1024, 256, 0, st>>>(a, b, size, 1u << s);
                uint8_t *t = a; a = b; b = t;
            }
            mk = a;
        }
    }
    leaves_kernel<<<tiles, kLeafThreads, dyn, st>>>(skey, cap, uniform_grid, grid_level, min_level, region_bits,
                                                    region_cap, kexp, mk,
                                                    status, tile_counter, leaf_lo, leaf_hi, leaf_beg,
                                                    leaf_nsub, leaf_box, tstride, info);
}

}  // namespace mqr
