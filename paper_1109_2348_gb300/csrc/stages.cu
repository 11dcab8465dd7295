// Run-length encoding and decoding of a batch (Section 3.2, Fig. 1 and
// Fig. 2 of the paper; the method of Fang et al. it describes).
//
// Encode: a byte ends a run if the next byte differs or starts another block
// (runs never cross blocks); an exclusive prefix sum of these flags gives
// every run its output slot; a run's length is the difference of consecutive
// end indices (the end before a tile's first run comes from the tiles before).
// Decode: the inclusive prefix sum of the lengths gives every run's end; flags at the last byte of every run, prefix-summed
// over the output, give every output byte its run; the byte is copied.
//
// Variable-length encoding (Section 3.4, Fig. 3; the substitution method of
// Balevic it describes): every byte is looked up in a codeword table, the
// exclusive prefix sum of the codeword lengths gives every codeword's first
// bit, and the codewords are written there (most significant bit first;
// each block's stream starts at a byte boundary).
//
// Move-to-front encoding (Section 3.3): the paper searches the list in
// parallel for one byte after another. Here blocks are cut into chunks whose
// starting lists come from the last occurrences of every byte value before
// them (one pass over the bytes, one over the chunks), and a warp encodes 32
// bytes of a chunk at once (below).
//
// GB300 layout: tiles are 4,096 elements (256 threads x 16). The run-length
// prefix sums take two passes (sums by spans, then the tiles); the codeword
// offsets a single pass with decoupled look-back between a block's tiles. A
// tile's codewords are packed into 32-bit words in shared memory and stored
// whole; only the two words a tile shares with its neighbours are merged with
// atomic ORs.
#include <algorithm>
#include <cstring>

#include "bwt.h"
#include "kernels.h"
#include "plan_internal.h"

using namespace bwt;

#define CKS(call)                                              \
    do {                                                       \
        cudaError_t _e = (call);                               \
        if (_e != cudaSuccess) return record_cuda(_e, #call);  \
    } while (0)

namespace {

constexpr int RT = 256;                 // threads per tile
constexpr int RI = 16;                  // elements per thread
constexpr uint32_t RTILE = RT * RI;     // 4096
constexpr uint32_t PART = RTILE / (RT / 32);  // a warp's share of a tile

// Block holding global position i (blocks are contiguous and cover the batch).
__device__ __forceinline__ uint32_t block_at(const BlockInfo* blocks, uint32_t nb, uint32_t i) {
    uint32_t lo = 0, hi = nb;
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (blocks[mid].off <= i) lo = mid; else hi = mid;
    }
    return lo;
}

__device__ __forceinline__ uint32_t next_tile(uint32_t* s_tile, uint32_t* counter) {
    if (threadIdx.x == 0) *s_tile = atomicAdd(counter, 1u);
    __syncthreads();
    const uint32_t t = *s_tile;
    __syncthreads();
    return t;
}

// ---- tile prefixes of the run-length stages -----------------------------------
//
// The prefix sums run in two passes: every tile's sum, with the tiles' prefixes
// by spans -- a span of consecutive tiles a CTA, at most four CTAs an SM, with
// decoupled look-back between spans -- and then the tiles, which wait for
// nothing. With the look-back between the tiles themselves (one pass, 1,200
// tiles in flight polling each other's words) 64 mixed blocks took 147 us for
// encoding and 147 for the lengths of decoding; with spans 42 + 75 and 43 + 50.
// (Tried for one pass: 128 words a look-back step, a CTA-wide look-back,
// 16,384-byte tiles: no faster. Two or eight spans an SM: 204 and 176 us a call
// where four took 179.) The second passes launch several tiles' worth of CTAs
// an SM: their tiles differ in work (encoding 161 us a call with 8, 152 with 48).

// Turns last[t] of the span's tiles [t0, t1) -- a tile's last run end, 0: none --
// into the last one before t in the span, and returns the span's last one. Ends
// increase with the tile, so both are maxima. All RT threads call.
__device__ __forceinline__ uint32_t span_last_ends(uint32_t* last, uint32_t t0, uint32_t t1, uint32_t* warp_max) {
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t run = 0;
    for (uint32_t base = t0; base < t1; base += RT) {
        const uint32_t t = base + threadIdx.x;
        uint32_t x = t < t1 ? last[t] : 0u;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x = max(x, y);
        }
        if (lane == 31) warp_max[warp] = x;
        __syncthreads();
        uint32_t ex = __shfl_up_sync(0xffffffffu, x, 1);
        ex = max(run, lane ? ex : 0u);
#pragma unroll
        for (uint32_t w = 0; w < RT / 32; ++w) {
            const uint32_t y = warp_max[w];
            if (w < warp) ex = max(ex, y);
            run = max(run, y);
        }
        if (t < t1) last[t] = ex;
        __syncthreads();
    }
    return run;
}

// Turns sums[t] of the span's tiles [t0, t1) into their exclusive prefixes over
// all tiles (mod 2^32). All RT threads call.
__device__ __forceinline__ void span_prefixes(uint32_t* sums, uint32_t t0, uint32_t t1, uint64_t* status, uint32_t span,
                                              uint32_t spin, uint32_t withhold, uint32_t* ctrl, uint32_t* scan_tmp,
                                              uint64_t* s_excl) {
    __syncthreads();  // the sums are written
    uint64_t run = 0;
    for (uint32_t base = t0; base < t1; base += RT) {
        const uint32_t t = base + threadIdx.x;
        uint32_t total;
        const uint32_t ex = block_exclusive_scan<RT>(t < t1 ? sums[t] : 0u, scan_tmp, &total);
        if (t < t1) sums[t] = (uint32_t)run + ex;
        run += total;
    }
    if (threadIdx.x < 32) {
        const uint64_t e = lookback_u64(status, span, 0, run & LB_VAL, spin, &ctrl[CTRL_ERR], withhold);
        if (threadIdx.x == 0) *s_excl = e;
    }
    __syncthreads();
    const uint32_t e = (uint32_t)*s_excl;
    for (uint32_t t = t0 + threadIdx.x; t < t1; t += RT) sums[t] += e;
}

// Bit j: byte j of a and of b differ.
__device__ __forceinline__ uint32_t bytes_differ(uint32_t a, uint32_t b) {
    return (__vsetne4(a, b) * 0x01020408u) >> 24;
}

// Run ends among the 16 bytes v at global position i0 (bit j: byte j ends a
// run), given the byte after them: the byte differs from the next one or is its
// block's last. `len` bytes of the tile at t0 are real; b0 is the block of t0,
// bend0 its end. With another block inside the tile, `starts` gets the bytes
// that start one (bit j), and b the block of i0.
__device__ __forceinline__ uint32_t run_ends(uint4 v, uint32_t after, uint32_t i0, uint32_t t0, uint32_t len, uint32_t N,
                                             const BlockInfo* __restrict__ blocks, uint32_t nb, uint32_t b0,
                                             uint32_t bend0, uint32_t& starts, uint32_t& b) {
    uint32_t flags = bytes_differ(v.x, __funnelshift_r(v.x, v.y, 8)) |
                     bytes_differ(v.y, __funnelshift_r(v.y, v.z, 8)) << 4 |
                     bytes_differ(v.z, __funnelshift_r(v.z, v.w, 8)) << 8 |
                     bytes_differ(v.w, __funnelshift_r(v.w, after, 8)) << 12;
    const uint32_t q0 = i0 - t0;
    starts = 0u;
    b = b0;
    if (bend0 < t0 + len) {  // uniform over the tile: another block starts in it
        b = i0 < N ? block_at(blocks, nb, i0) : 0u;
        uint32_t bb = b, bend = i0 < N ? blocks[b].off + blocks[b].n : 0u;
        if (i0 < N && blocks[b].off == i0) starts |= 1u;
#pragma unroll
        for (int j = 0; j < RI; ++j) {
            if (i0 + j >= N) break;
            if (i0 + j == bend) {
                ++bb;
                bend = blocks[bb].off + blocks[bb].n;
                starts |= 1u << j;
            }
            if (i0 + j + 1 == bend) flags |= 1u << j;
        }
    } else {
        if (i0 == t0 && blocks[b0].off == t0) starts = 1u;
        if (bend0 == t0 + len && bend0 - 1 - i0 < (uint32_t)RI) flags |= 1u << (bend0 - 1 - i0);
    }
    if (q0 + RI > len) flags &= q0 < len ? (1u << (len - q0)) - 1u : 0u;
    return flags;
}

// The 16 bytes at S[i], i + 16 <= N or bytes past N undefined (zero): one load
// where aligned.
__device__ __forceinline__ uint4 load16(const uint8_t* __restrict__ S, uint32_t i, uint32_t N) {
    if ((uint64_t)i + 16 <= N && (reinterpret_cast<uintptr_t>(S + i) & 15u) == 0u)
        return __ldg(reinterpret_cast<const uint4*>(S + i));
    uint32_t w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
    for (int j = 0; j < 16; ++j)
        if ((uint64_t)i + j < N) w[j / 4] |= (uint32_t)S[i + j] << (8 * (j % 4));
    return make_uint4(w[0], w[1], w[2], w[3]);
}

// Tiles of a batch so small that the second pass finds its own prefixes, a warp
// an earlier tile, and the first is left out: a launch and a look-back less (a
// 30,000-byte batch: 38.0 -> 35.5 us a call; two tiles a warp, up to 65,000
// bytes: the same to encode, 40 -> 50 to decode).
constexpr uint32_t FEW_TILES = RT / 32;

// A tile's number of run ends and its last one (end index, 0: none), or those of
// its bytes [from, to), by a warp.
__device__ __forceinline__ void tile_run_ends(const uint8_t* __restrict__ S, uint32_t N,
                                              const BlockInfo* __restrict__ blocks, uint32_t nb, uint32_t t,
                                              uint32_t& cnt, uint32_t& end, uint32_t from = 0, uint32_t to = RTILE) {
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t p0 = t * RTILE, len = min(RTILE, N - p0);
    const uint32_t b0 = block_at(blocks, nb, p0), bend0 = blocks[b0].off + blocks[b0].n;
    cnt = end = 0;
#pragma unroll 4
    for (uint32_t q = from + lane * 16; q < to; q += 512) {
        const uint32_t i0 = p0 + q;
        const uint4 v = load16(S, i0, N);
        uint32_t after = __shfl_down_sync(0xffffffffu, v.x, 1);
        if (lane == 31) after = (uint64_t)i0 + 16 < N ? S[i0 + 16] : 0u;
        uint32_t starts, b;
        const uint32_t f = run_ends(v, after, i0, p0, len, N, blocks, nb, b0, bend0, starts, b);
        cnt += __popc(f);
        if (f) end = i0 + 32u - __clz(f);
    }
    cnt = __reduce_add_sync(0xffffffffu, cnt);
    end = __reduce_max_sync(0xffffffffu, end);
}

// Encode, sums: every tile's run ends, a warp a tile (a batch of no more tiles
// than spans: a CTA a tile, as a lone warp's loads wait for each other: 400,000
// bytes 48 -> 37 us a call, decoded 53 -> 42); then the tiles' prefixes, and the
// last run ends before the tiles in their span.
__global__ void __launch_bounds__(RT) k_rle_sums(const uint8_t* __restrict__ S, uint32_t N,
                                                 const BlockInfo* __restrict__ blocks, uint32_t nb,
                                                 uint32_t* __restrict__ sums, uint32_t* __restrict__ last,
                                                 uint32_t* __restrict__ span_last, uint64_t* __restrict__ status,
                                                 uint32_t* __restrict__ counter, uint32_t* ctrl) {
    __shared__ uint32_t s_span, s_part[2], scan_tmp[32];
    __shared__ uint64_t s_excl;
    const uint32_t ntiles = (N + RTILE - 1) / RTILE, per = (ntiles + gridDim.x - 1) / gridDim.x;
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t span = next_tile(&s_span, counter);  // in start order, so that earlier spans are in flight
    const uint32_t t0 = min(ntiles, span * per), t1 = min(ntiles, t0 + per);
    if (per == 1) {
        if (threadIdx.x < 2) s_part[threadIdx.x] = 0u;
        __syncthreads();
        if (t0 < t1) {
            uint32_t cnt, end;
            tile_run_ends(S, N, blocks, nb, t0, cnt, end, warp * PART, warp * PART + PART);
            if (lane == 0) {
                atomicAdd(&s_part[0], cnt);
                atomicMax(&s_part[1], end);
            }
        }
        __syncthreads();
        if (threadIdx.x == 0 && t0 < t1) {
            sums[t0] = s_part[0];
            last[t0] = s_part[1];
        }
    } else {
        for (uint32_t t = t0 + warp; t < t1; t += RT / 32) {
            uint32_t cnt, end;
            tile_run_ends(S, N, blocks, nb, t, cnt, end);
            if (lane == 0) {
                sums[t] = cnt;
                last[t] = end;
            }
        }
    }
    span_prefixes(sums, t0, t1, status, span, ctrl[CTRL_SPIN], ctrl[CTRL_WITHHOLD], ctrl, scan_tmp, &s_excl);
    const uint32_t end = span_last_ends(last, t0, t1, scan_tmp);  // after it: later spans wait for the prefixes
    if (threadIdx.x == 0) span_last[span] = end;
}

// The last run end before tile t (a warp calls; 0 before the first): the one in
// its span, else the nearest earlier span's, 128 spans a step. There are at most
// four spans an SM, so a run over any number of tiles is a few steps: one run of
// 2^26 bytes 122 us a call, of 2^28 340. (Walking back over the tiles themselves,
// 32 a step: 615 us and 11.1 ms.)
__device__ __forceinline__ uint32_t last_end_before(const uint32_t* __restrict__ last,
                                                    const uint32_t* __restrict__ span_last, uint32_t t, uint32_t per) {
    const uint32_t lane = threadIdx.x & 31, v = last[t];
    if (v) return v;
    for (uint32_t end = t / per; end > 0; end = end > 128 ? end - 128 : 0) {
        uint32_t m = 0;
#pragma unroll
        for (uint32_t k = 0; k < 4; ++k) m = max(m, k * 32 + lane < end ? span_last[end - 1 - k * 32 - lane] : 0u);
        m = __reduce_max_sync(0xffffffffu, m);
        if (m) return m;
    }
    return 0u;
}

// Encode: run-end flags and their block scan give every run its slot; the runs'
// bytes and lengths -- the differences of consecutive end indices -- are
// compacted through shared memory so that they are written in rows.
// run_off[b] = the first run of block b (run_off[nb] = the number of runs). 64
// mixed blocks (57.6 MB, 38.5 M runs): 388 us at first, with byte loads and
// every thread writing its own runs, and 72 us for a pass over the end indices;
// 104 us with entries written one a thread, 75 four a thread.
__global__ void __launch_bounds__(RT) k_rle_encode(const uint8_t* __restrict__ S, uint32_t N,
                                                   const BlockInfo* __restrict__ blocks, uint32_t nb,
                                                   const uint32_t* __restrict__ first, const uint32_t* __restrict__ last,
                                                   const uint32_t* __restrict__ span_last, uint32_t per,
                                                   uint8_t* __restrict__ chars, uint32_t* __restrict__ lens,
                                                   uint64_t* __restrict__ run_off, uint32_t* ctrl) {
    // the tile's run bytes and end positions, from index k0 mod 4 on: a group
    // of four entries has the alignment of its place in the outputs
    __shared__ __align__(4) uint8_t sb[RTILE + 4];
    __shared__ __align__(8) uint16_t se[RTILE + 4];
    __shared__ uint8_t s_first[RT / 32 + 1];  // each warp's first byte (and the next tile's)
    __shared__ uint32_t s_prev, s_few[2 * RT / 32], scan_tmp[32];
    if (ld_volatile(&ctrl[CTRL_ERR])) return;  // a wait of the sums ran out: the prefixes are not to be used
    const uint32_t ntiles = (N + RTILE - 1) / RTILE;
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool vec = (reinterpret_cast<uintptr_t>(chars) & 3u) == 0u && (reinterpret_cast<uintptr_t>(lens) & 15u) == 0u;
    for (uint32_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const uint32_t t0 = t * RTILE, len = min(RTILE, N - t0);
        const uint32_t q0 = threadIdx.x * RI, i0 = t0 + q0;
        const uint4 v = load16(S, i0, N);
        uint32_t k0 = 0;
        const uint32_t b0 = block_at(blocks, nb, t0), bend0 = blocks[b0].off + blocks[b0].n;
        if (first) {
            k0 = first[t];
            if (warp == 1) {
                const uint32_t e = last_end_before(last, span_last, t, per);
                if (lane == 0) s_prev = e;
            }
        } else {  // few tiles: warp w counts tile w
            uint32_t cnt = 0, end = 0;
            if (warp < t) tile_run_ends(S, N, blocks, nb, warp, cnt, end);
            if (lane == 0) {
                s_few[warp] = cnt;
                s_few[RT / 32 + warp] = end;
            }
            __syncthreads();
            uint32_t prev = 0;
#pragma unroll
            for (int w = 0; w < RT / 32; ++w) {
                k0 += s_few[w];
                prev = max(prev, s_few[RT / 32 + w]);
            }
            if (threadIdx.x == 0) s_prev = prev;
        }
        if (lane == 0) s_first[warp] = (uint8_t)v.x;
        if (threadIdx.x == 0) s_first[RT / 32] = t0 + len < N ? S[t0 + len] : (uint8_t)0;
        uint32_t after = __shfl_down_sync(0xffffffffu, v.x, 1);  // its low byte follows this thread's
        __syncthreads();
        if (lane == 31) after = s_first[warp + 1];
        uint32_t starts, b;
        const uint32_t flags = run_ends(v, after, i0, t0, len, N, blocks, nb, b0, bend0, starts, b);
        uint32_t total;
        const uint32_t pre = block_exclusive_scan<RT>(__popc(flags), scan_tmp, &total);
        {
            const uint32_t w[4] = {v.x, v.y, v.z, v.w};
            uint32_t k = pre + (k0 & 3u);
#pragma unroll
            for (int j = 0; j < RI; ++j) {
                if ((flags >> j) & 1u) {
                    sb[k] = (uint8_t)(w[j / 4] >> (8 * (j % 4)));
                    se[k] = (uint16_t)(q0 + j + 1);
                    ++k;
                }
            }
        }
        __syncthreads();
        while (starts) {  // runs before the block's first byte
            const int j = __ffs(starts) - 1;
            starts &= starts - 1;
            while (blocks[b].off < i0 + j) ++b;
            run_off[b] = (uint64_t)k0 + pre + __popc(flags & ((1u << j) - 1u));
        }
        if (t + 1 == ntiles && threadIdx.x == 0) run_off[nb] = (uint64_t)k0 + total;
        // groups of four entries; g is the first one's index in the arrays
        const uint32_t a = k0 & 3u, end = a + total;
        const uint64_t base = (uint64_t)k0 - a;
        for (uint32_t g = threadIdx.x * 4; g < end; g += RT * 4) {
            const uint32_t c4 = *reinterpret_cast<const uint32_t*>(sb + g);
            const uint2 e4 = *reinterpret_cast<const uint2*>(se + g);
            const uint32_t e[4] = {e4.x & 0xffffu, e4.x >> 16, e4.y & 0xffffu, e4.y >> 16};
            uint32_t l[4];
            l[0] = g > a ? e[0] - se[g - 1] : t0 + e[0] - s_prev;
#pragma unroll
            for (int j = 1; j < 4; ++j) l[j] = g + j > a ? e[j] - e[j - 1] : t0 + e[j] - s_prev;
            if (vec && g >= a && g + 4 <= end && base + g + 4 <= N) {
                *reinterpret_cast<uint32_t*>(chars + base + g) = c4;
                *reinterpret_cast<uint4*>(lens + base + g) = make_uint4(l[0], l[1], l[2], l[3]);
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (g + j >= a && g + j < end && base + g + j < N) {
                        chars[base + g + j] = (uint8_t)(c4 >> (8 * j));
                        lens[base + g + j] = l[j];
                    }
                }
            }
        }
        __syncthreads();
    }
}

// Four lengths from k on, those past the last run (R) read as one, which is no
// input error. vec: lens is 16-byte aligned.
__device__ __forceinline__ uint4 lens4(const uint32_t* __restrict__ lens, uint64_t R, uint64_t k, bool vec) {
    if (vec && k + 4 <= R) return __ldg(reinterpret_cast<const uint4*>(lens + k));
    return make_uint4(k < R ? lens[k] : 1u, k + 1 < R ? lens[k + 1] : 1u, k + 2 < R ? lens[k + 2] : 1u,
                      k + 3 < R ? lens[k + 3] : 1u);
}

// The summed lengths of tile t of RTILE runs, or of its runs [from, to), by a
// warp; zero: one of this lane's lengths is zero (an input error). The last tile's missing entries
// count one and are subtracted, so that it takes the same eight loads in flight
// as a full one: 4 blocks of up to 415 KB waited 41 us for its lengths read one
// after the other.
__device__ __forceinline__ uint32_t tile_len_sum(const uint32_t* __restrict__ lens, uint64_t R, uint32_t t, bool vec,
                                                 bool& zero, uint32_t from = 0, uint32_t to = RTILE) {
    const uint32_t lane = threadIdx.x & 31;
    const uint64_t k0 = (uint64_t)t * RTILE, k1 = k0 + to;
    uint32_t sum = 0;
#pragma unroll 8
    for (uint32_t q = from + lane * 4; q < to; q += 128) {
        const uint4 x = lens4(lens, R, k0 + q, vec);
        zero |= x.x == 0u || x.y == 0u || x.z == 0u || x.w == 0u;
        sum += x.x + x.y + x.z + x.w;
    }
    const uint32_t pad = k1 <= R ? 0u : (uint32_t)(k1 - max(R, k0 + from));
    return __reduce_add_sync(0xffffffffu, sum) - pad;
}

// Decode, sums: the summed lengths of every tile, a warp a tile (no more tiles
// than spans: a CTA a tile), and the tiles' prefixes.
__global__ void __launch_bounds__(RT) k_rle_len_sums(const uint32_t* __restrict__ lens,
                                                     const uint64_t* __restrict__ run_off, uint32_t nb, uint32_t N,
                                                     uint32_t* __restrict__ sums, uint64_t* __restrict__ status,
                                                     uint32_t* __restrict__ counter, uint32_t* ctrl) {
    __shared__ uint32_t s_span, s_part, scan_tmp[32];
    __shared__ uint64_t s_excl;
    const uint64_t R = min(run_off[nb], (uint64_t)N);  // a run holds at least one byte
    const uint32_t ntiles = (uint32_t)((R + RTILE - 1) / RTILE), per = (ntiles + gridDim.x - 1) / gridDim.x;
    const bool vec = (reinterpret_cast<uintptr_t>(lens) & 15u) == 0u;
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t span = next_tile(&s_span, counter);
    const uint32_t t0 = min(ntiles, span * per), t1 = min(ntiles, t0 + per);
    bool zero = false;
    if (per == 1) {
        if (threadIdx.x == 0) s_part = 0u;
        __syncthreads();
        if (t0 < t1) {
            const uint32_t sum = tile_len_sum(lens, R, t0, vec, zero, warp * PART, warp * PART + PART);
            if (lane == 0) atomicAdd(&s_part, sum);
        }
        __syncthreads();
        if (threadIdx.x == 0 && t0 < t1) sums[t0] = s_part;
    } else {
        for (uint32_t t = t0 + warp; t < t1; t += RT / 32) {
            const uint32_t sum = tile_len_sum(lens, R, t, vec, zero);
            if (lane == 0) sums[t] = sum;
        }
    }
    if (zero) atomicOr(&ctrl[CTRL_ERR], ERR_INPUT);
    span_prefixes(sums, t0, t1, status, span, ctrl[CTRL_SPIN], ctrl[CTRL_WITHHOLD], ctrl, scan_tmp, &s_excl);
}

// Decode step 1: B[k] = end of run k (inclusive prefix sum of the lengths,
// global).
__global__ void __launch_bounds__(RT) k_rle_scan(const uint32_t* __restrict__ lens, const uint64_t* __restrict__ run_off,
                                                 uint32_t nb, uint32_t N, const uint32_t* __restrict__ first,
                                                 uint32_t* __restrict__ B, uint32_t* ctrl) {
    __shared__ uint32_t scan_tmp[32], s_few[RT / 32];
    const uint64_t R = min(run_off[nb], (uint64_t)N);
    const uint32_t ntiles = (uint32_t)((R + RTILE - 1) / RTILE);
    const bool vec = (reinterpret_cast<uintptr_t>(lens) & 15u) == 0u;
    for (uint32_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const uint64_t k0 = (uint64_t)t * RTILE + threadIdx.x * RI;
        uint32_t v[RI], sum = 0;
        if (vec && k0 + RI <= R) {
#pragma unroll
            for (int j = 0; j < RI; j += 4) {
                const uint4 x = __ldg(reinterpret_cast<const uint4*>(lens + k0 + j));
                v[j] = x.x;
                v[j + 1] = x.y;
                v[j + 2] = x.z;
                v[j + 3] = x.w;
            }
        } else {
#pragma unroll
            for (int j = 0; j < RI; ++j) v[j] = k0 + j < R ? lens[k0 + j] : 0u;
        }
        uint32_t f = 0;
        if (first) {
            f = first[t];
        } else {  // few tiles: warp w sums tile w; every tile looks for its own zero lengths
            bool zero = false;
            const uint32_t w = threadIdx.x >> 5, x = w < t ? tile_len_sum(lens, R, w, vec, zero) : 0u;
            if ((threadIdx.x & 31) == 0) s_few[w] = x;
            zero = false;
#pragma unroll
            for (int j = 0; j < RI; ++j) zero |= v[j] == 0u && k0 + j < R;
            if (zero) atomicOr(&ctrl[CTRL_ERR], ERR_INPUT);
            __syncthreads();
#pragma unroll
            for (int k = 0; k < RT / 32; ++k) f += s_few[k];
        }
#pragma unroll
        for (int j = 0; j < RI; ++j) sum += v[j];
        uint32_t total;
        uint32_t acc = f + block_exclusive_scan<RT>(sum, scan_tmp, &total);
#pragma unroll
        for (int j = 0; j < RI; ++j) {
            acc += v[j];
            v[j] = acc;
        }
        if (k0 + RI <= R) {  // B is the plan's, 16-byte aligned
#pragma unroll
            for (int j = 0; j < RI; j += 4)
                *reinterpret_cast<uint4*>(B + k0 + j) = make_uint4(v[j], v[j + 1], v[j + 2], v[j + 3]);
        } else {
#pragma unroll
            for (int j = 0; j < RI; ++j)
                if (k0 + j < R) B[k0 + j] = v[j];
        }
    }
}

// Decode steps 2-4: per output tile, flags at the last byte of every run that
// ends in it, their exclusive prefix sum = the run of every byte (after the
// runs that end before the tile), and the run's byte. A CTA takes a span of
// consecutive tiles: the first one's first run is searched by a warp (32
// probes a round), every later tile starts at the run the one before ended in.
// Bytes are gathered from shared memory and written 16 at a time. 64 mixed
// blocks: 366 us with a search a tile by one thread (25 dependent loads) and
// byte stores -> 90 us.
__global__ void __launch_bounds__(RT) k_rle_expand(const uint8_t* __restrict__ chars, const uint32_t* __restrict__ B,
                                                   const uint64_t* __restrict__ run_off,
                                                   const BlockInfo* __restrict__ blocks, uint32_t nb, uint32_t N,
                                                   uint8_t* __restrict__ out, uint32_t* ctrl) {
    __shared__ __align__(16) uint8_t sflag[RTILE];
    __shared__ uint8_t sc[RTILE];
    __shared__ uint32_t s_k0, scan_tmp[32];
    // the input's check: every block's runs end exactly at the block's end
    for (uint32_t b = blockIdx.x * RT + threadIdx.x; b < nb; b += gridDim.x * RT) {
        const uint64_t r0 = run_off[b], r1 = run_off[b + 1];
        const bool ok = (b > 0 || r0 == 0) && r1 > r0 && r1 <= N && B[r1 - 1] == blocks[b].off + blocks[b].n;
        if (!ok) atomicOr(&ctrl[CTRL_ERR], ERR_INPUT);
    }
    const uint64_t R = min(run_off[nb], (uint64_t)N);
    if (R == 0) return;  // no runs: the check flags the input
    const uint32_t ntiles = (N + RTILE - 1) / RTILE;
    const uint32_t span = (ntiles + gridDim.x - 1) / gridDim.x;
    const uint32_t t_end = min(ntiles, (blockIdx.x + 1) * span);
    const bool vec = (reinterpret_cast<uintptr_t>(out) & 15u) == 0u;
    if (blockIdx.x * span >= ntiles) return;
    if (threadIdx.x < 32) {  // first run ending after the span's start: runs before it end at or before it
        const uint32_t t0 = blockIdx.x * span * RTILE;
        uint64_t lo = 0, hi = R;  // B[lo - 1] <= t0 < B[hi]
        while (lo < hi) {
            const uint64_t p = lo + (hi - lo) * threadIdx.x / 32;
            const uint32_t m = __popc(__ballot_sync(0xffffffffu, B[p] <= t0));  // a prefix of the lanes
            const uint64_t nlo = m ? lo + (hi - lo) * (m - 1) / 32 + 1 : lo;
            hi = m < 32 ? lo + (hi - lo) * m / 32 : hi;
            lo = nlo;
        }
        if (threadIdx.x == 0) s_k0 = (uint32_t)lo;
    }
    __syncthreads();
    uint32_t k0 = s_k0;
    for (uint32_t t = blockIdx.x * span; t < t_end; ++t) {
        const uint32_t t0 = t * RTILE, len = min(RTILE, N - t0);
        reinterpret_cast<uint4*>(sflag)[threadIdx.x] = make_uint4(0u, 0u, 0u, 0u);
        __syncthreads();
        // the runs that reach into the tile (at most len): their bytes, and a
        // flag at each one's last byte; four a thread and step, loaded together
        constexpr int U = 4;
        for (uint32_t x0 = threadIdx.x; x0 < len; x0 += U * RT) {
            uint32_t e[U], st[U];
            uint8_t c[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint64_t k = (uint64_t)k0 + x0 + u * RT;
                const bool ok = x0 + u * RT < len && k < R;
                e[u] = ok ? B[k] : 0u;
                st[u] = ok ? (k > 0 ? B[k - 1] : 0u) : 0xffffffffu;
                c[u] = ok ? chars[k] : (uint8_t)0;
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (st[u] < t0 + len) {  // else it begins after the tile (B increases) or is none
                    sc[x0 + u * RT] = c[u];
                    if (e[u] - 1 - t0 < len) sflag[e[u] - 1 - t0] = 1;
                }
            }
            if (st[U - 1] >= t0 + len) break;
        }
        __syncthreads();
        const uint32_t q0 = threadIdx.x * RI;
        const uint4 f4 = reinterpret_cast<const uint4*>(sflag)[threadIdx.x];
        const uint32_t f[4] = {f4.x, f4.y, f4.z, f4.w};
        const uint32_t cnt = __popc(f4.x) + __popc(f4.y) + __popc(f4.z) + __popc(f4.w);
        uint32_t total;
        uint32_t r = block_exclusive_scan<RT>(cnt, scan_tmp, &total);
        uint32_t w[4];
        const uint32_t rmax = (uint32_t)min((uint64_t)RTILE - 1u, R - 1 - min((uint64_t)k0, R - 1));
#pragma unroll
        for (int j = 0; j < RI; ++j) {
            const uint32_t c = sc[min(r, rmax)];
            w[j / 4] = j % 4 ? w[j / 4] | c << (8 * (j % 4)) : c;
            r += (f[j / 4] >> (8 * (j % 4))) & 1u;
        }
        if (vec && q0 + RI <= len) {
            *reinterpret_cast<uint4*>(out + t0 + q0) = make_uint4(w[0], w[1], w[2], w[3]);
        } else {
#pragma unroll
            for (int j = 0; j < RI; ++j)
                if (q0 + j < len) out[t0 + q0 + j] = (uint8_t)(w[j / 4] >> (8 * (j % 4)));
        }
        k0 += total;
        __syncthreads();
    }
}

// ---- variable-length encoding ------------------------------------------------

// Bits of every block's stream (sum of its bytes' codeword lengths). A byte
// whose codeword length is outside 1..32 is an input error.
__global__ void __launch_bounds__(RT) k_vle_bits(const uint8_t* __restrict__ S, const TileDesc* __restrict__ tiles,
                                                 uint32_t ntiles, const uint8_t* __restrict__ len,
                                                 unsigned long long* __restrict__ block_bits, uint32_t* ctrl) {
    __shared__ uint8_t slen[256];
    __shared__ uint32_t red[RT / 32];
    slen[threadIdx.x] = len[threadIdx.x];
    __syncthreads();
    for (uint32_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const TileDesc td = tiles[t];
        uint32_t sum = 0;
        bool bad = false;
        auto add = [&](uint32_t x) {
            const uint32_t l = slen[x];
            bad |= l - 1u > 31u;
            sum += l;
        };
        // whole aligned 16-byte words by one load each, the bytes before and
        // after them one by one
        const uint32_t head = min(td.len, (uint32_t)(-reinterpret_cast<uintptr_t>(S + td.start)) & 15u);
        const uint32_t nvec = (td.len - head) / 16, tail = head + nvec * 16;
        for (uint32_t v = threadIdx.x; v < nvec; v += RT) {
            const uint4 w = __ldg(reinterpret_cast<const uint4*>(S + td.start + head) + v);
            const uint32_t x[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
            for (int j = 0; j < 16; ++j) add((x[j / 4] >> (8 * (j % 4))) & 0xffu);
        }
        if (threadIdx.x < head) add(S[td.start + threadIdx.x]);
        if (threadIdx.x < td.len - tail) add(S[td.start + tail + threadIdx.x]);
        if (bad) atomicOr(&ctrl[CTRL_ERR], ERR_INPUT);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = sum;
        __syncthreads();
        if (threadIdx.x == 0) {
            uint32_t tot = 0;
            for (int w = 0; w < RT / 32; ++w) tot += red[w];
            atomicAdd(&block_bits[td.blk], (unsigned long long)tot);
        }
        __syncthreads();
    }
}

// 64-bit block-wide exclusive scan (1024 threads).
__device__ __forceinline__ unsigned long long scan64_1024(unsigned long long v, unsigned long long* tmp,
                                                          unsigned long long* total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) tmp[warp] = x;
    __syncthreads();
    if (warp == 0) {
        unsigned long long w = tmp[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        tmp[lane] = w;
    }
    __syncthreads();
    const unsigned long long r = (warp ? tmp[warp - 1] : 0ull) + x - v;
    *total = tmp[31];
    __syncthreads();
    return r;
}

// Byte offsets of the block streams (exclusive scan of ceil(bits / 8)); the
// total goes to byte_off[nb]. The buffer must hold the total rounded up to
// whole 32-bit words. One CTA.
__global__ void __launch_bounds__(1024) k_vle_offsets(const unsigned long long* __restrict__ block_bits, uint32_t nb,
                                                      uint64_t cap, uint64_t* __restrict__ byte_off, uint32_t* ctrl) {
    __shared__ unsigned long long tmp[32];
    unsigned long long run = 0;  // the same in every thread
    for (uint32_t base = 0; base < nb; base += 1024) {
        const uint32_t b = base + threadIdx.x;
        const unsigned long long bytes = b < nb ? (block_bits[b] + 7) / 8 : 0ull;
        unsigned long long tot;
        const unsigned long long ex = scan64_1024(bytes, tmp, &tot);
        if (b < nb) byte_off[b] = run + ex;
        run += tot;
    }
    if (threadIdx.x == 0) {
        byte_off[nb] = run;
        if ((run + 3) / 4 * 4 > cap) atomicOr(&ctrl[CTRL_ERR], ERR_CAPACITY);
    }
}

// Zeroes the output words [0, ceil(byte_off[nb] / 4)) that lie inside the
// buffer (partial words at the end are merged by atomic OR, so they need it).
// Also clears the packing's look-back words.
__global__ void k_vle_zero(uint32_t* __restrict__ out32, const uint64_t* __restrict__ byte_off, uint32_t nb,
                           uint64_t cap_words, uint64_t* __restrict__ status, uint32_t ntiles) {
    for (uint32_t t = blockIdx.x * blockDim.x + threadIdx.x; t < ntiles; t += gridDim.x * blockDim.x) status[t] = 0ull;
    const uint64_t words = min((byte_off[nb] + 3) / 4, cap_words);
    for (uint64_t w = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; w < words; w += (uint64_t)gridDim.x * blockDim.x)
        out32[w] = 0u;
}

// Packs every tile's codewords: bit offsets inside the block by a block
// scan plus look-back over the block's earlier tiles, words assembled in
// shared memory (stream bit j of a word is bit 31 - j, stored byte-swapped so
// that memory order is stream order), interior words stored, edge words
// OR-ed. out32 is the output viewed as 32-bit words (4-byte aligned). A thread
// takes 16 bytes, staged by 16-byte loads, looks each up once (code and length
// share a word when no code is longer than 26 bits) and shifts its codewords
// together in a register: only its first and last words are OR-ed into shared
// memory. 38.5 M move-to-front bytes: 152 us with byte loads, two look-ups and
// an OR or two a codeword -> 96 us (five CTAs an SM; four: 102); the bits of the
// blocks 32 -> 23.
constexpr uint32_t VLE_WORDS = RTILE + 2;  // a tile spans at most 4096 * 32 bits + alignment
constexpr uint32_t VLE_PACKED = 26;        // longest code that shares a word with its length (6 bits)
constexpr size_t VLE_SMEM = VLE_WORDS * 4 + 256 * 5;
static_assert(VLE_WORDS * 4 >= RTILE + 48, "the staged bytes fit the words");

__global__ void __launch_bounds__(RT, 5) k_vle_pack(const uint8_t* __restrict__ S, const BlockInfo* __restrict__ blocks,
                                                 const TileDesc* __restrict__ tiles,
                                                 uint32_t ntiles, const uint32_t* __restrict__ code,
                                                 const uint8_t* __restrict__ len, const uint64_t* __restrict__ byte_off,
                                                 uint64_t cap_words, uint32_t* __restrict__ out32,
                                                 uint64_t* __restrict__ status, uint32_t* __restrict__ counter,
                                                 uint32_t* ctrl) {
    extern __shared__ __align__(16) unsigned char smem[];
    uint32_t* words = reinterpret_cast<uint32_t*>(smem);           // [VLE_WORDS] (the tile's bytes before)
    uint32_t* scode = words + VLE_WORDS;                           // [256] codes, masked to their lengths (| length)
    uint8_t* slen = reinterpret_cast<uint8_t*>(scode + 256);       // [256]
    __shared__ uint32_t s_tile, scan_tmp[32];
    __shared__ uint64_t s_excl;
    const uint32_t spin = ctrl[CTRL_SPIN], withhold = ctrl[CTRL_WITHHOLD];
    if (ld_volatile(&ctrl[CTRL_ERR]) & (ERR_INPUT | ERR_CAPACITY)) return;  // bad table or too small a buffer
    const uint32_t my_len = len[threadIdx.x];
    const bool packed = __syncthreads_and(my_len <= VLE_PACKED) != 0;
    {
        const uint32_t c = my_len >= 32u ? code[threadIdx.x] : code[threadIdx.x] & ((1u << my_len) - 1u);
        scode[threadIdx.x] = packed ? c << 6 | my_len : c;
        slen[threadIdx.x] = (uint8_t)my_len;
    }
    for (;;) {
        const uint32_t at = next_tile(&s_tile, counter);
        if (at >= ntiles) break;
        const TileDesc td = tiles[at];
        const uint32_t t = td.index;  // its look-back row: the table is interleaved
        const BlockInfo bi = blocks[td.blk];
        const uint32_t shift = stage_tile_bytes(S, bi, td.start - bi.off, td.len, smem, threadIdx.x, RT);
        __syncthreads();
        const uint32_t q0 = threadIdx.x * RI;
        uint32_t e[RI], lsum = 0;  // entries: code, or code and length
        uint32_t l4[RI / 4] = {};  // lengths, a byte each
        {
            uint32_t x[RI / 4 + 1];
#pragma unroll
            for (int k = 0; k < RI / 4 + 1; ++k) x[k] = words[(shift >> 2) + threadIdx.x * (RI / 4) + k];
#pragma unroll
            for (int j = 0; j < RI; ++j) {
                const uint32_t w = __funnelshift_r(x[j / 4], x[j / 4 + 1], 8 * (shift & 3u));
                const uint32_t c = (w >> (8 * (j % 4))) & 0xffu;
                uint32_t l = 0;
                e[j] = 0;
                if (q0 + j < td.len) {
                    e[j] = scode[c];
                    l = packed ? e[j] & 63u : slen[c];
                }
                l4[j / 4] |= l << (8 * (j % 4));
                lsum += l;
            }
        }
        uint32_t total;
        const uint32_t pre = block_exclusive_scan<RT>(lsum, scan_tmp, &total);  // every byte has been read
        if (threadIdx.x < 32) {
            const uint64_t ex = lookback_u64(status, t, td.firstTile, total, spin, &ctrl[CTRL_ERR], withhold);
            if (threadIdx.x == 0) s_excl = ex;
        }
        // the words the tile can touch, wherever in its first word it starts
        const uint32_t nzero = min(total / 32 + 2, VLE_WORDS);
        for (uint32_t w = threadIdx.x; w < nzero; w += RT) words[w] = 0u;
        __syncthreads();
        const uint64_t g0 = byte_off[td.blk] * 8 + s_excl;  // first bit of the tile
        const uint64_t w0 = g0 >> 5;
        if (lsum) {
            const uint32_t x0 = (uint32_t)(g0 + pre - (w0 << 5));  // this thread's first bit in the tile's words
            uint32_t wi = min(x0 >> 5, VLE_WORDS - 1), fill = x0 & 31u;
            bool whole = fill == 0u;  // the word in hand starts with this thread's bits
            uint64_t acc = 0;         // its bits, left-aligned, and the next word's
#pragma unroll
            for (int j = 0; j < RI; ++j) {
                const uint32_t L = (l4[j / 4] >> (8 * (j % 4))) & 0xffu;
                acc |= (uint64_t)(packed ? e[j] >> 6 : e[j]) << (64u - max(1u, fill + L));
                fill += L;
                if (fill >= 32u) {
                    const uint32_t v = (uint32_t)(acc >> 32);
                    if (whole) words[wi] = v;
                    else atomicOr(&words[wi], v);
                    whole = true;
                    wi = min(wi + 1, VLE_WORDS - 1);
                    acc <<= 32;
                    fill -= 32u;
                }
            }
            if (fill) atomicOr(&words[wi], (uint32_t)(acc >> 32));
        }
        __syncthreads();
        const uint32_t nwords = (uint32_t)(((g0 + total + 31) >> 5) - w0);
        for (uint32_t x = threadIdx.x; x < nwords; x += RT) {
            const uint64_t w = w0 + x;
            if (w >= cap_words) break;
            const uint32_t v = __byte_perm(words[x], 0, 0x0123);
            if (x == 0 || x + 1 == nwords) atomicOr(&out32[w], v);
            else out32[w] = v;
        }
        __syncthreads();
    }
}

// ---- move-to-front encoding ---------------------------------------------------
//
// Three launches over chunks of `mc` bytes (512 .. 4,096; chunks never cross
// blocks): the last occurrence of every byte value in every chunk, its
// running maximum over each block's chunks, and the encoding of all chunks
// at once, a warp each. A byte's code is the number of distinct bytes since
// its last occurrence, so a warp encodes 32 bytes a step from the list
// before them, with ballots in place of 32 list updates in a row.
//
// Measured on 38.5 M run bytes (64 mixed blocks): 2,117 us (one list update a
// byte, a chain of shuffles) -> 485 us for the encoding, 476 -> 24 us for the
// chunks' starting lists, 198 -> 48 us for the last occurrences. The encoding
// is bound by issue (68%, 311 warp instructions a step of 32 bytes). Chunk
// sizes: a chunk's starting list costs about 12 steps, so large batches take
// 4,096-byte chunks (565 us in all; at most twice as many chunks: 588, five
// times: 870); five CTAs an SM at 48 registers and four at 64 took the same.
constexpr int MTF_WARPS = 8;
constexpr uint32_t MTF_MIN = 512, MTF_MAX = 4096;  // chunk sizes
constexpr uint32_t MTF_CHUNKS = 16384;             // chunks shorter than MTF_MAX: at most this many

struct MtfChunk {
    uint32_t start, len, rel, n;  // global start, bytes, block-relative start, bytes of the block
};

// Chunk c: cfirst[b] = first chunk of block b (cfirst[nb] = chunks).
__device__ __forceinline__ MtfChunk mtf_chunk(const BlockInfo* __restrict__ blocks, const uint32_t* __restrict__ cfirst,
                                              uint32_t nb, uint32_t c, uint32_t mc) {
    uint32_t lo = 0, hi = nb;
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (cfirst[mid] <= c) lo = mid; else hi = mid;
    }
    const BlockInfo bi = blocks[lo];
    const uint32_t rel = (c - cfirst[lo]) * mc;
    return MtfChunk{bi.off + rel, min(mc, bi.n - rel), rel, bi.n};
}

// One warp stages S[g0 .. g0 + len) at buf[shift ..), shift = the address
// modulo 16 (returned): 16-byte loads where the aligned words around the
// range lie inside S[0 .. N), else bytes. buf is 16-byte aligned and holds
// len + 31 bytes.
__device__ __forceinline__ uint32_t warp_stage(const uint8_t* __restrict__ S, uint32_t g0, uint32_t len, uint32_t N,
                                               uint8_t* buf) {
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t shift = (uint32_t)(reinterpret_cast<uintptr_t>(S + g0) & 15u);
    const uint32_t nvec = (shift + len + 15) >> 4;
    if (g0 >= shift && (uint64_t)g0 - shift + 16ull * nvec <= N) {
        const uint4* src = reinterpret_cast<const uint4*>(S + g0 - shift);
        for (uint32_t v = lane; v < nvec; v += 32) reinterpret_cast<uint4*>(buf)[v] = __ldg(src + v);
    } else {
        for (uint32_t q = lane; q < len; q += 32) buf[shift + q] = S[g0 + q];
    }
    __syncwarp();
    return shift;
}

// Pass 1: tab[chunk][x] = block-relative position + 1 of the last x in the
// chunk, 0 if it holds none. A warp walks its chunk backwards, 32 bytes a
// step; a step whose bytes were all seen costs a look-up and a ballot.
__global__ void __launch_bounds__(MTF_WARPS * 32) k_mtf_last(const uint8_t* __restrict__ S, uint32_t N,
                                                             const BlockInfo* __restrict__ blocks, uint32_t nb,
                                                             const uint32_t* __restrict__ cfirst, uint32_t mc,
                                                             uint32_t* __restrict__ tab) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint32_t s_last[MTF_WARPS][256];
    const uint32_t lane = threadIdx.x & 31, wl = threadIdx.x >> 5;
    uint8_t* buf = smem + wl * (mc + 32);
    uint32_t* last = s_last[wl];
    const uint32_t nc = cfirst[nb];
    for (uint32_t c = blockIdx.x * MTF_WARPS + wl; c < nc; c += gridDim.x * MTF_WARPS) {
        const MtfChunk ch = mtf_chunk(blocks, cfirst, nb, c, mc);
#pragma unroll
        for (int k = 0; k < 8; ++k) last[k * 32 + lane] = 0u;
        const uint32_t shift = warp_stage(S, ch.start, ch.len, N, buf);
        for (uint32_t b = (ch.len - 1) & ~31u;; b -= 32) {
            const uint32_t q = b + lane;
            const uint32_t x = q < ch.len ? buf[shift + q] : 256u;
            const bool fresh = x < 256u && last[x] == 0u;
            if (__any_sync(0xffffffffu, fresh)) {
                const uint32_t peers = __match_any_sync(0xffffffffu, fresh ? x : 256u);
                if (fresh && (peers >> lane) == 1u) last[x] = ch.rel + q + 1;  // the highest lane of its value
                __syncwarp();
            }
            if (b == 0) break;
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) tab[(size_t)c * 256 + k * 32 + lane] = last[k * 32 + lane];
        __syncwarp();
    }
}

// Pass 2, in place: tab[chunk][x] = position + 1 of the last x before the
// chunk in its block, 0 if there is none. One CTA a block, a thread a value;
// 16 chunks' loads are in flight at once.
__global__ void __launch_bounds__(256) k_mtf_scan(const uint32_t* __restrict__ cfirst, uint32_t nb,
                                                  uint32_t* __restrict__ tab) {
    for (uint32_t b = blockIdx.x; b < nb; b += gridDim.x) {
        uint32_t run = 0;
        const uint32_t c1 = cfirst[b + 1];
        for (uint32_t c = cfirst[b]; c < c1; c += 16) {
            uint32_t v[16];
#pragma unroll
            for (int k = 0; k < 16; ++k) v[k] = c + k < c1 ? tab[(size_t)(c + k) * 256 + threadIdx.x] : 0u;
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                if (c + k < c1) tab[(size_t)(c + k) * 256 + threadIdx.x] = run;
                if (v[k]) run = v[k];  // later chunks hold later positions
            }
        }
    }
}

// The list before a chunk: the byte values by last occurrence, latest first,
// then those not seen yet in ascending order. A warp sorts (recency, value)
// descending, bitonic, eight values a lane; KeyT holds recency << 8 | value.
template <typename KeyT>
__device__ __forceinline__ void mtf_start_list(const uint32_t* __restrict__ row, uint8_t* list, uint8_t* pos) {
    const uint32_t lane = threadIdx.x & 31;
    KeyT k[8];
    const uint4 r0 = reinterpret_cast<const uint4*>(row)[lane * 2], r1 = reinterpret_cast<const uint4*>(row)[lane * 2 + 1];
    const uint32_t rec[8] = {r0.x, r0.y, r0.z, r0.w, r1.x, r1.y, r1.z, r1.w};
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const uint32_t x = lane * 8 + i, r = rec[i];
        k[i] = ((KeyT)(r ? r + 255u : 255u - x) << 8) | x;
    }
#pragma unroll
    for (uint32_t kk = 2; kk <= 256; kk <<= 1) {
#pragma unroll
        for (uint32_t j = kk >> 1; j > 0; j >>= 1) {
            if (j >= 8) {  // across lanes
#pragma unroll
                for (uint32_t i = 0; i < 8; ++i) {
                    const KeyT o = __shfl_xor_sync(0xffffffffu, k[i], j >> 3);
                    const bool down = ((lane * 8) & kk) == 0, lower = ((lane * 8) & j) == 0;
                    k[i] = (lower == down) == (k[i] > o) ? k[i] : o;
                }
            } else {
#pragma unroll
                for (uint32_t i = 0; i < 8; ++i) {
                    if ((i & j) == 0) {
                        const bool down = ((lane * 8 + i) & kk) == 0;
                        const KeyT a = k[i], b = k[i | j];
                        const bool keep = (a > b) == down;
                        k[i] = keep ? a : b;
                        k[i | j] = keep ? b : a;
                    }
                }
            }
        }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const uint32_t x = (uint32_t)k[i] & 255u;
        list[lane * 8 + i] = (uint8_t)x;
        pos[x] = (uint8_t)(lane * 8 + i);
    }
}

// Pass 3: one warp encodes a chunk from its starting list, 32 bytes a step.
// With p = a byte's position in the list before the step: a byte's first
// occurrence in the step is encoded as p plus the distinct bytes of the step
// before it that stood behind p (they have moved in front of it); a later
// occurrence as the distinct bytes since the previous one, which are the
// first ones of that stretch: those whose own previous occurrence is no
// later than its start. Both compare a small number of every lane with this
// lane's, for all lanes at once, by one ballot a bit. Then the step's bytes
// move to the front by last occurrence, and the others up to the last
// position touched move back by the step's bytes behind them.
__global__ void __launch_bounds__(MTF_WARPS * 32, 5) k_mtf_encode(const uint8_t* __restrict__ S, uint32_t N,
                                                               const BlockInfo* __restrict__ blocks, uint32_t nb,
                                                               const uint32_t* __restrict__ cfirst, uint32_t mc,
                                                               const uint32_t* __restrict__ tab,
                                                               uint8_t* __restrict__ out) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint8_t s_list[MTF_WARPS][256], s_pos[MTF_WARPS][256];
    const uint32_t lane = threadIdx.x & 31, wl = threadIdx.x >> 5, lt = lanemask_lt(), gt_lanes = ~(lt | (1u << lane));
    uint8_t* buf = smem + wl * (mc + 32);
    uint8_t *list = s_list[wl], *pos = s_pos[wl];
    const uint32_t nc = cfirst[nb];
    for (uint32_t c = blockIdx.x * MTF_WARPS + wl; c < nc; c += gridDim.x * MTF_WARPS) {
        const MtfChunk ch = mtf_chunk(blocks, cfirst, nb, c, mc);
        if (ch.n < (1u << 24) - 256u) mtf_start_list<uint32_t>(tab + (size_t)c * 256, list, pos);
        else mtf_start_list<uint64_t>(tab + (size_t)c * 256, list, pos);
        const uint32_t shift = warp_stage(S, ch.start, ch.len, N, buf);
        for (uint32_t b = 0; b < ch.len; b += 32) {
            // lanes past the end repeat the last byte: they change nothing
            const uint32_t q = min(b + lane, ch.len - 1);
            const uint32_t x = buf[shift + q];
            const uint32_t p = pos[x];
            const uint32_t maxp = __reduce_max_sync(0xffffffffu, p);
            uint32_t r = 0;
            if (maxp > 0u) {  // else 32 times the byte at the front
                // lanes with this lane's byte, and lanes whose position is greater
                uint32_t eq = 0xffffffffu, gt = 0u;
#pragma unroll
                for (int k = 7; k >= 0; --k) {
                    if (maxp >> k) {  // warp-uniform
                        const bool one = (p >> k) & 1u;
                        const uint32_t B = __ballot_sync(0xffffffffu, one);
                        const uint32_t m = one ? 0u : 0xffffffffu;
                        gt |= eq & B & m;
                        eq &= B ^ m;
                    }
                }
                const uint32_t before = eq & lt;
                const bool first = before == 0u;
                const uint32_t F = __ballot_sync(0xffffffffu, first);
                r = p + __popc(gt & F & lt);
                if (F != 0xffffffffu) {
                    const uint32_t prev = 32u - __clz(before);  // lane of the previous occurrence + 1, 0: none
                    uint32_t e2 = 0xffffffffu, less = 0u;       // lanes with an equal prev, with a smaller one
#pragma unroll
                    for (int k = 4; k >= 0; --k) {
                        const bool one = (prev >> k) & 1u;
                        const uint32_t B = __ballot_sync(0xffffffffu, one);
                        const uint32_t m = one ? 0xffffffffu : 0u;
                        less |= e2 & ~B & m;
                        e2 &= ~(B ^ m);
                    }
                    if (!first) r = __popc(less & lt & (0xffffffffu << prev));
                }
                const bool last = (eq & gt_lanes) == 0u;
                const uint32_t La = __ballot_sync(0xffffffffu, last);
                const uint32_t D = __popc(F);
                uint32_t below = D;  // the step's positions below word w
                for (int w = (int)(maxp >> 5); w >= 0; --w) {
                    const uint32_t mine = first && (int)(p >> 5) == w ? 1u << (p & 31u) : 0u;
                    const uint32_t m = __reduce_or_sync(0xffffffffu, mine);
                    below -= __popc(m);
                    const uint32_t j = w * 32 + lane;
                    const uint32_t v = list[j];
                    __syncwarp();  // the word is read before its entries move up (into this word and the next)
                    if (j <= maxp && !((m >> lane) & 1u)) {
                        const uint32_t np = j + D - below - __popc(m & lt);
                        list[np] = (uint8_t)v;
                        pos[v] = (uint8_t)np;
                    }
                }
                if (last) {
                    const uint32_t np = __popc(La & gt_lanes);
                    list[np] = (uint8_t)x;
                    pos[x] = (uint8_t)np;
                }
                __syncwarp();
            }
            if (b + lane < ch.len) buf[shift + b + lane] = (uint8_t)r;
            __syncwarp();  // the last byte is read by the lanes past the end
        }
        // out, by 16-byte words where its address has the staged alignment
        uint8_t* o = out + ch.start;
        uint32_t q0 = 0, q1 = 0;  // bytes [q0, q1) go as whole words
        if ((reinterpret_cast<uintptr_t>(o) & 15u) == shift && shift + ch.len >= 32u) {
            q0 = (16u - shift) & 15u;
            q1 = ((shift + ch.len) & ~15u) - shift;
            for (uint32_t q = q0 + lane * 16; q < q1; q += 512)
                *reinterpret_cast<uint4*>(o + q) = *reinterpret_cast<const uint4*>(buf + shift + q);
        }
        for (uint32_t q = lane; q < q0; q += 32) o[q] = buf[shift + q];
        for (uint32_t q = q1 + lane; q < ch.len; q += 32) o[q] = buf[shift + q];
        __syncwarp();
    }
}

}  // namespace

extern "C" bwt_status bwt_rle_encode(bwt_plan* p, const uint8_t* d_in, const uint64_t* offsets, uint32_t num_blocks,
                                     uint8_t* d_chars, uint32_t* d_lens, uint64_t* d_run_off, void* stream) {
    if (!p || !d_in || !offsets || !d_chars || !d_lens || !d_run_off) return BWT_EINVAL;
    bwt::NvtxRange nvtx_range("rle_encode");
    if (cudaSetDevice(p->device) != cudaSuccess) return BWT_ECUDA;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    std::memset(&p->stats, 0, sizeof(p->stats));
    bwt_status s = prepare_batch(p, offsets, num_blocks, st);
    if (s != BWT_OK) return p->last = s;
    const uint32_t N = p->total, nt = (N + RTILE - 1) / RTILE;
    const int sms = num_sms();
    const int spans = std::max(1, std::min<int>(nt, sms * 4));
    uint64_t* status = reinterpret_cast<uint64_t*>(p->status);  // the spans' words, two words a tile, a word a span
    uint32_t* sums = p->status + 2 * (size_t)spans;
    if ((s = reset_ctrl(p, st, p->status, 2 * spans)) != BWT_OK) return p->last = s;
    const bool few = nt <= FEW_TILES;
    if (!few)
        k_rle_sums<<<spans, RT, 0, st>>>(d_in, N, p->blocks, p->nb, sums, sums + nt, sums + 2 * (size_t)nt, status,
                                         p->ctrl + CTRL_TILE_CTR, p->ctrl);
    const uint32_t per = (nt + (uint32_t)spans - 1) / (uint32_t)spans;  // tiles a span, as the sums' kernel takes them
    k_rle_encode<<<std::max(1, std::min<int>(nt, sms * 48)), RT, 0, st>>>(
        d_in, N, p->blocks, p->nb, few ? nullptr : sums, sums + nt, sums + 2 * (size_t)nt, per, d_chars, d_lens, d_run_off,
        p->ctrl);
    CKS(cudaGetLastError());
    p->stats.kernel_launches = few ? 2 : 3;
    return p->last = finish_status(p, st);
}

extern "C" bwt_status bwt_rle_decode(bwt_plan* p, const uint8_t* d_chars, const uint32_t* d_lens,
                                     const uint64_t* d_run_off, const uint64_t* offsets, uint32_t num_blocks,
                                     uint8_t* d_out, void* stream) {
    if (!p || !d_chars || !d_lens || !d_run_off || !offsets || !d_out) return BWT_EINVAL;
    bwt::NvtxRange nvtx_range("rle_decode");
    if (cudaSetDevice(p->device) != cudaSuccess) return BWT_ECUDA;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    std::memset(&p->stats, 0, sizeof(p->stats));
    bwt_status s = prepare_batch(p, offsets, num_blocks, st);
    if (s != BWT_OK) return p->last = s;
    const uint32_t N = p->total, nt = (N + RTILE - 1) / RTILE;  // runs <= N, so <= nt tiles of runs
    const int sms = num_sms();
    const int spans = std::max(1, std::min<int>(nt, sms * 4));
    uint64_t* status = reinterpret_cast<uint64_t*>(p->status);  // the spans' words, then a word a tile
    uint32_t* sums = p->status + 2 * (size_t)spans;
    if ((s = reset_ctrl(p, st, p->status, 2 * spans)) != BWT_OK) return p->last = s;
    uint32_t* B = p->vals[0];
    const bool few = nt <= FEW_TILES;
    if (!few)
        k_rle_len_sums<<<spans, RT, 0, st>>>(d_lens, d_run_off, p->nb, N, sums, status, p->ctrl + CTRL_TILE_CTR,
                                             p->ctrl);
    k_rle_scan<<<std::max(1, std::min<int>(nt, sms * 24)), RT, 0, st>>>(d_lens, d_run_off, p->nb, N, few ? nullptr : sums,
                                                                        B, p->ctrl);
    k_rle_expand<<<std::max(1, std::min<int>(nt, sms * 24)), RT, 0, st>>>(d_chars, B, d_run_off,
                                                                            p->blocks, p->nb, N, d_out, p->ctrl);
    CKS(cudaGetLastError());
    p->stats.kernel_launches = few ? 3 : 4;
    return p->last = finish_status(p, st);
}

extern "C" bwt_status bwt_vle_encode(bwt_plan* p, const uint8_t* d_in, const uint64_t* offsets, uint32_t num_blocks,
                                     const uint32_t* d_code, const uint8_t* d_len, uint8_t* d_out, uint64_t out_cap,
                                     uint64_t* d_byte_off, uint64_t* d_block_bits, void* stream) {
    if (!p || !d_in || !offsets || !d_code || !d_len || !d_out || !d_byte_off || !d_block_bits) return BWT_EINVAL;
    bwt::NvtxRange nvtx_range("vle_encode");
    if ((reinterpret_cast<uintptr_t>(d_out) & 3u) != 0) return BWT_EINVAL;  // written as 32-bit words
    if (cudaSetDevice(p->device) != cudaSuccess) return BWT_ECUDA;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    std::memset(&p->stats, 0, sizeof(p->stats));
    bwt_status s = prepare_batch(p, offsets, num_blocks, st);
    if (s != BWT_OK) return p->last = s;
    if ((s = reset_ctrl(p, st)) != BWT_OK) return p->last = s;
    const uint32_t nb = p->nb, nt = p->ntiles0;
    if (p->tile > (int)RTILE) return p->last = BWT_EINVAL;
    static bool attr = [] {
        cudaFuncSetAttribute((void*)k_vle_pack, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)VLE_SMEM);
        return true;
    }();
    (void)attr;
    const int sms = num_sms();
    unsigned long long* bits = reinterpret_cast<unsigned long long*>(d_block_bits);
    CKS(cudaMemsetAsync(bits, 0, sizeof(uint64_t) * nb, st));
    k_vle_bits<<<std::max(1, std::min<int>(nt, sms * 8)), RT, 0, st>>>(d_in, p->tiles0, nt, d_len, bits, p->ctrl);
    k_vle_offsets<<<1, 1024, 0, st>>>(bits, nb, out_cap, d_byte_off, p->ctrl);
    const uint64_t cap_words = out_cap / 4;  // whole words inside the buffer
    uint64_t* status = reinterpret_cast<uint64_t*>(p->status);
    k_vle_zero<<<sms * 8, 256, 0, st>>>(reinterpret_cast<uint32_t*>(d_out), d_byte_off, nb, cap_words, status, nt);
    k_vle_pack<<<std::max(1, std::min<int>(nt, sms * 6)), RT, VLE_SMEM, st>>>(
        d_in, p->blocks, p->rtile == p->tile ? p->tiles_il : p->tiles0, nt, d_code, d_len, d_byte_off, cap_words, reinterpret_cast<uint32_t*>(d_out), status,
        p->ctrl + CTRL_TILE_CTR, p->ctrl);
    CKS(cudaGetLastError());
    p->stats.kernel_launches = 5;
    return p->last = finish_status(p, st);
}

extern "C" bwt_status bwt_mtf_encode(bwt_plan* p, const uint8_t* d_in, const uint64_t* offsets, uint32_t num_blocks,
                                     uint8_t* d_out, void* stream) {
    if (!p || !d_in || !offsets || !d_out) return BWT_EINVAL;
    bwt::NvtxRange nvtx_range("mtf_encode");
    if (cudaSetDevice(p->device) != cudaSuccess) return BWT_ECUDA;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    std::memset(&p->stats, 0, sizeof(p->stats));
    bwt_status s = prepare_batch(p, offsets, num_blocks, st);
    if (s != BWT_OK) return p->last = s;
    const uint32_t nb = p->nb, N = p->total;
    // chunk size: the smallest that leaves at most MTF_CHUNKS of them (a
    // small batch is latency: more and shorter chunks), 4,096 for large batches
    uint32_t mc = MTF_MIN;
    while (mc < MTF_MAX && N / mc > MTF_CHUNKS) mc <<= 1;
    uint32_t* h_first = p->h_inv_items;  // pinned staging, free outside the inverse
    uint32_t nc = 0;
    for (uint32_t b = 0; b < nb; ++b) {
        h_first[b] = nc;
        nc += (uint32_t)((p->h_off[b + 1] - p->h_off[b] + mc - 1) / mc);
    }
    h_first[nb] = nc;
    // scratch: 256 words a chunk, per block its first chunk: in the sort's key
    // buffers, or, for blocks of a few bytes, on its own from first use on (a
    // plan's first call on 3 blocks of 233,843 bytes: 214 us with it allocated)
    uint32_t *tab = reinterpret_cast<uint32_t*>(p->keys[0]), *cfirst = reinterpret_cast<uint32_t*>(p->keys[1]);
    const size_t room = sizeof(uint64_t) * (size_t)p->cap_n;
    if ((size_t)nc * 1024 > room || ((size_t)nb + 1) * 4 > room) {
        const size_t cap_chunks = std::min<size_t>(p->cap_n / MTF_MIN, std::max<size_t>(MTF_CHUNKS, p->cap_n / MTF_MAX)) +
                                  (size_t)p->cap_b + 1;
        if (!p->mtf_lists) CKS(cudaMalloc(&p->mtf_lists, cap_chunks * 1024 + 4 * ((size_t)p->cap_b + 1)));
        tab = reinterpret_cast<uint32_t*>(p->mtf_lists);
        cfirst = tab + cap_chunks * 256;
    }
    CKS(cudaMemcpyAsync(cfirst, h_first, sizeof(uint32_t) * (nb + 1), cudaMemcpyHostToDevice, st));
    const int sms = num_sms();
    const size_t smem = (size_t)MTF_WARPS * (mc + 32);
    const int grid = std::max(1, std::min<int>((nc + MTF_WARPS - 1) / MTF_WARPS, sms * 8));
    k_mtf_last<<<grid, MTF_WARPS * 32, smem, st>>>(d_in, N, p->blocks, nb, cfirst, mc, tab);
    k_mtf_scan<<<std::min<uint32_t>(nb, (uint32_t)sms * 8), 256, 0, st>>>(cfirst, nb, tab);
    k_mtf_encode<<<grid, MTF_WARPS * 32, smem, st>>>(d_in, N, p->blocks, nb, cfirst, mc, tab, d_out);
    CKS(cudaGetLastError());
    p->stats.kernel_launches = 3;
    CKS(cudaStreamSynchronize(st));
    return p->last = BWT_OK;
}
