// Inverse BWT of a batch on the GPU.
//
// The transform is undone from L and the primary index alone (Section 3.1).
// F, the first column, is L sorted; FL[j] is the row whose rotation starts
// one position after row j's (the occurrence of F[j] in L, counted stably).
// From row r_0 = primary (rotation 0): S[i] = F[r_i] and r_{i+1} = FL[r_i].
//
// That walk is one dependent chain per block, so it is split:
//   1. one stable pass over (L[k], k) by the byte writes P[j] = (FL << 8) | F,
//      one load per step of a walk;
//   2. walkers start at every SMP-th row and at the primary row and walk FL
//      until the next such row (each row of a cycle is visited once), storing
//      the first SBUF bytes they pass in their sample's slot;
//   3. every SUP-th sample and the primary (the "supers") walk the samples to
//      the next super, adding up lengths, and pointer jumping over the supers
//      alone, with the list cut at the primary, gives every super on the
//      primary's cycle its distance to the end, hence its text offset;
//   4. every super writes its stretch of S: the stored bytes of its samples,
//      one after the other, and the few beyond SBUF by walking P again.
// A periodic block S = u^k has k cycles of |u| rows; the primary's cycle
// gives u, and the block is u repeated.
//
// Bound by random reads: a 4-byte P entry a row from L2 in the walks, a 32-byte
// sample from memory per eight bytes in the writes. Measured on 64 mixed
// blocks of 900,000 bytes: 2,618 us with keys and values sorted, two walks of
// every row and pointer jumping over all samples -> 1,285 us (sort 316, walks
// 369, supers 95, jumping 45, writes 349, histogram 42). Strides: SMP 16 with
// 56 stored bytes 1,781 (before the one-store samples: 8 with 24 stored 1,411),
// SUP 4 / 16 +2% / +8%; walkers a thread and CTAs an SM: 4/4 1,394, 4/3 1,331,
// 3/4 1,274, 3/5 1,344, 2/6 1,314.
#include <algorithm>
#include <cstring>
#include <vector>

#include "bwt.h"
#include "kernels.h"
#include "plan_internal.h"

using namespace bwt;

#define CKI(call)                                              \
    do {                                                       \
        cudaError_t _e = (call);                               \
        if (_e != cudaSuccess) return record_cuda(_e, #call);  \
    } while (0)

namespace {

constexpr uint32_t SMP = 8;      // every SMP-th row starts a walk
constexpr uint32_t SBUF = 24;    // bytes of its walk that a sample stores (a walk's mean is SMP)
constexpr uint32_t SUP = 8;      // every SUP-th sample is a super
constexpr uint32_t END = 0xffffffffu, INVALID = 0xfffffffeu;

// Block b has m_b = ceil(n_b / SMP) strided samples and the primary's, slots
// qbase[b] .. qbase[b + 1] - 1 (the primary's last), and ceil(m_b / SUP)
// strided supers and the primary's, nodes sbase[b] .. sbase[b + 1] - 1 (last
// again). A strided sample on the primary row itself is not used.
// A sample's walk, one 32-byte memory sector, written by one store: a sector
// written in parts is first read from memory (measured with an 8-byte record
// and the bytes word by word: 1.45 GB read for 57.6 MB of blocks, 556 us for
// the walks, against 0.55 GB and 369 us).
struct __align__(32) Sample {
    uint32_t next, len;  // slot where the walk stops, its steps
    uint64_t x[3];       // its first SBUF bytes, the last of them at the top of x[2]
};
static_assert(sizeof(Sample) == 32 && SBUF == 24, "a sample is one memory sector");

__device__ __forceinline__ void store_sample(Sample* p, uint32_t next, uint32_t len, const uint32_t (&w)[6]) {
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(next), "r"(len), "r"(w[0]),
                 "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5])
                 : "memory");
}

struct InvCtx {
    const BlockInfo* blocks;
    const int32_t* primary;
    const uint32_t* qbase;  // [nb + 1]
    const uint32_t* sbase;  // [nb + 1]
    uint32_t nb;
    const void* P;          // (FL << 8) | F per row, global index: u32 for blocks under 2^24 bytes, else u64
    Sample* sample;         // per slot
    uint32_t* row;          // per slot: global row after SBUF steps (longer walks only)
    uint8_t* out;
    uint32_t* ctrl;
};

// Last b with pre[b] <= k (pre[0] = 0, k < pre[nb]).
__device__ __forceinline__ uint32_t find_block(const uint32_t* pre, uint32_t nb, uint32_t k) {
    uint32_t lo = 0, hi = nb;
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (pre[mid] <= k) lo = mid; else hi = mid;
    }
    return lo;
}

// P: one stable counting pass over the bytes of L, a tile of a block at a
// time -- the radix pass of the forward sort (ranks by peer masks, decoupled
// look-back), but reading one byte and writing one P entry a row instead of
// keys and values. PT = u32: the entry is staged whole; u64: index and byte.
template <typename PT, int TILE>
__global__ void __launch_bounds__(256, TILE >= 4096 ? 5 : 6) k_inv_sort(const uint8_t* __restrict__ L,
                                                                        const BlockInfo* __restrict__ blocks,
                                                                        const TileDesc* __restrict__ tiles,
                                                                        uint32_t num_tiles,
                                                                        const uint32_t* __restrict__ seg_base,
                                                                        uint32_t* __restrict__ status,
                                                                        uint32_t* __restrict__ counter, uint32_t* ctrl,
                                                                        PT* __restrict__ P) {
    constexpr int ITEMS = TILE / 256, WKEYS = 32 * ITEMS;
    // the tile's bytes and the warps' counts first, the staged entries over them
    constexpr size_t U0 = TILE + 48 + 8 * 256 * 2, U1 = TILE * sizeof(PT);
    __shared__ __align__(16) unsigned char smem[U0 > U1 ? U0 : U1];
    uint8_t* sb = smem;
    uint16_t* whist = reinterpret_cast<uint16_t*>(smem + TILE + 48);
    PT* sp = reinterpret_cast<PT*>(smem);
    __shared__ uint32_t digit_start[256], gbase[256], scan_tmp[32];
    __shared__ uint32_t s_tile;
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, lt = lanemask_lt();
    const uint32_t spin = ctrl[CTRL_SPIN], withhold = ctrl[CTRL_WITHHOLD];
    for (;;) {
        if (tid == 0) s_tile = atomicAdd(counter, 1u);
        __syncthreads();
        if (s_tile >= num_tiles) break;
        const TileDesc td = tiles[s_tile];
        const uint32_t t = td.index;  // its look-back row: the table is interleaved
        const BlockInfo bi = blocks[td.blk];
        const uint32_t i0 = td.start - bi.off;
        const uint32_t shift = stage_tile_bytes(L, bi, i0, td.len, sb, tid, 256);
        for (int i = tid; i < 8 * 256 / 2; i += 256) reinterpret_cast<uint32_t*>(whist)[i] = 0u;
        __syncthreads();
        // rank within the warp's digit (low 16) | digit (high 16)
        uint32_t rk[ITEMS];
        uint16_t* my = whist + warp * 256;
        const bool full = td.len == (uint32_t)TILE;
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) {
            const uint32_t idx = warp * WKEYS + j * 32 + lane;
            const bool valid = idx < td.len;
            const uint32_t d = valid ? sb[shift + idx] : 256u;
            const uint32_t peers = full ? match_label<8>(d) : match_label<9>(d);
            const uint32_t r = (valid ? my[d] : 0u) + __popc(peers & lt);
            __syncwarp();  // every peer has read the count before the last of them advances it
            if (valid && (peers >> lane) == 1u) my[d] = (uint16_t)(r + 1);
            __syncwarp();
            rk[j] = r | (d << 16);
        }
        __syncthreads();
        uint32_t cnt = 0;  // thread d: the tile's count of digit d, its prefix over the warps in place
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            const uint32_t c = whist[w * 256 + tid];
            whist[w * 256 + tid] = (uint16_t)cnt;
            cnt += c;
        }
        uint32_t total;
        const uint32_t ex = block_exclusive_scan<256>(cnt, scan_tmp, &total);
        digit_start[tid] = ex;
        const bool first = t == td.firstTile;
        uint32_t* mine = status + (size_t)t * 256 + tid;
        if (!first) st_volatile(mine, ST_AGG | cnt);
        else if (!(withhold && t == 0)) st_volatile(mine, ST_INC | cnt);
        __syncthreads();
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) {
            const uint32_t d = rk[j] >> 16;
            // destination in the tile (low 16) | digit (high 16)
            if (d < 256u) rk[j] = (digit_start[d] + whist[warp * 256 + d] + (rk[j] & 0xffffu)) | (d << 16);
            else rk[j] = 0xffffffffu;
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < ITEMS; ++j)
            if (rk[j] != 0xffffffffu)
                sp[rk[j] & 0xffffu] = ((PT)(i0 + warp * WKEYS + j * 32 + lane) << 8) | (rk[j] >> 16);
        uint32_t excl = 0;
        if (!first) {
            excl = lookback_digit(status, 256, t, td.firstTile, tid, spin, &ctrl[CTRL_ERR]);
            st_volatile(mine, ST_INC | ((excl + cnt) & ST_VALUE));
        }
        gbase[tid] = td.segStart + seg_base[(size_t)td.seg * 256 + tid] + excl - ex;
        __syncthreads();
        for (uint32_t q = tid; q < td.len; q += 256) {
            const PT v = sp[q];
            const uint32_t dst = gbase[(uint32_t)v & 255u] + q;
            BWT_DCHECK(dst - td.segStart < td.pad0, &ctrl[CTRL_ERR]);
            P[dst] = v;
        }
        __syncthreads();
    }
}

// Walks of every sample, from its row to the next sample row, recording where
// and after how many steps it stops and the bytes on the way. Walks differ a
// lot in length, so walkers are not tied to a work item: each warp takes
// ranges of CH sample ids from a global counter, and a lane starts its next
// walk as soon as one of its WALKERS walks ends. A walk is one dependent load
// per step; a walker holds only global row indices and counters, so many
// walks per SM are in flight. Runs only after the radix pass succeeded (FL is
// then a permutation of every block).
constexpr uint32_t CH = 64;
constexpr int WALKERS = 3;
constexpr int WALK_CTAS_PER_SM = 4;

template <typename PT>
__global__ void __launch_bounds__(256, WALK_CTAS_PER_SM) k_inv_walks(InvCtx c, uint32_t Q,
                                                                     uint32_t* __restrict__ counter) {
    if (ld_volatile(&c.ctrl[CTRL_ERR]) & (ERR_TIMEOUT | ERR_CAPACITY)) return;
    const PT* __restrict__ P = static_cast<const PT*>(c.P);
    const uint32_t lane = threadIdx.x & 31, lt = lanemask_lt();
    uint32_t wq = 0, wq_end = 0;  // warp-uniform range of sample ids not started yet
    uint32_t wb = 0;              // block of the range's first sample
    bool exhausted = false;
    // per walker: global row, its block's first row, global row of the
    // primary, sample slot, steps taken, block, its first SBUF bytes
    uint32_t R[WALKERS], off[WALKERS], a[WALKERS], g[WALKERS], cnt[WALKERS], blk[WALKERS], w[WALKERS][6];
    bool act[WALKERS];
#pragma unroll
    for (int j = 0; j < WALKERS; ++j) act[j] = false;
    for (;;) {
        // start a walk in every idle slot, as long as samples are left
#pragma unroll
        for (int j = 0; j < WALKERS; ++j) {
            bool need = !act[j];
            for (;;) {
                const uint32_t mask = __ballot_sync(0xffffffffu, need && !exhausted);
                if (mask == 0u) break;
                if (wq == wq_end) {
                    uint32_t q0 = 0;
                    if (lane == 0) q0 = atomicAdd(counter, CH);
                    q0 = __shfl_sync(0xffffffffu, q0, 0);
                    if (q0 >= Q) {
                        exhausted = true;
                        break;
                    }
                    wq = q0;
                    wq_end = min(q0 + CH, Q);
                    wb = find_block(c.qbase, c.nb, q0);
                    continue;
                }
                const uint32_t take = min((uint32_t)__popc(mask), wq_end - wq);
                const uint32_t rk = __popc(mask & lt);
                if (need && rk < take) {
                    const uint32_t q = wq + rk;
                    uint32_t b = wb;
                    while (c.qbase[b + 1] <= q) ++b;  // a range of CH samples spans few blocks
                    const uint32_t s = q - c.qbase[b], m = c.qbase[b + 1] - c.qbase[b] - 1;
                    const BlockInfo bi = c.blocks[b];
                    const int32_t ps = c.primary[b];
                    if (ps < 0 || (uint32_t)ps >= bi.n) {
                        if (s == 0) atomicOr(&c.ctrl[CTRL_ERR], ERR_INPUT);
                    } else {
                        const uint32_t row = s < m ? s * SMP : (uint32_t)ps;
                        if (s == m || row != (uint32_t)ps) {  // the primary row walks as slot m
                            R[j] = bi.off + row;
                            off[j] = bi.off;
                            a[j] = bi.off + (uint32_t)ps;
                            g[j] = q;
                            cnt[j] = 0;
                            blk[j] = b;
                            act[j] = true;
#pragma unroll
                            for (int k = 0; k < 6; ++k) w[j][k] = 0u;
                            need = false;
                        }
                    }
                }
                wq += take;
            }
        }
        bool any = false;
#pragma unroll
        for (int j = 0; j < WALKERS; ++j) any |= act[j];
        if (!__any_sync(0xffffffffu, any) && exhausted) break;
        // one step of every walk
        PT v[WALKERS];
#pragma unroll
        for (int j = 0; j < WALKERS; ++j) v[j] = act[j] ? P[R[j]] : (PT)0;
#pragma unroll
        for (int j = 0; j < WALKERS; ++j) {
            if (!act[j]) continue;
            const uint32_t nr = off[j] + (uint32_t)(v[j] >> 8);
            R[j] = nr;
            if (cnt[j] < SBUF) {  // shifted in at the top
#pragma unroll
                for (int k = 0; k < 5; ++k) w[j][k] = __funnelshift_r(w[j][k], w[j][k + 1], 8);
                w[j][5] = (w[j][5] >> 8) | ((uint32_t)v[j] << 24);
            }
            if (++cnt[j] == SBUF) c.row[g[j]] = nr;
            if (nr == a[j] || ((nr - off[j]) & (SMP - 1)) == 0) {
                const uint32_t base = c.qbase[blk[j]];
                store_sample(c.sample + g[j], nr == a[j] ? c.qbase[blk[j] + 1] - 1 : base + (nr - off[j]) / SMP, cnt[j],
                             w[j]);
                act[j] = false;
            }
        }
    }
}

// A super's place: block, its slots and nodes, its own slot; false if it is
// not used (its block's primary is out of range, or it sits on that row).
struct SuperAt {
    BlockInfo bi;
    uint32_t base, m, node0, nodes, slot;
};

__device__ __forceinline__ bool super_at(const InvCtx& c, uint32_t node, SuperAt& u) {
    const uint32_t b = find_block(c.sbase, c.nb, node);
    u.bi = c.blocks[b];
    const int32_t ps = c.primary[b];
    u.base = c.qbase[b];
    u.m = c.qbase[b + 1] - u.base - 1;
    u.node0 = c.sbase[b];
    u.nodes = c.sbase[b + 1] - u.node0;
    const uint32_t t = node - u.node0, s = t + 1 < u.nodes ? t * SUP : u.m;
    u.slot = u.base + s;
    return ps >= 0 && (uint32_t)ps < u.bi.n && (s == u.m || s * SMP != (uint32_t)ps);
}

// Every super walks the samples to the next super (itself at the latest).
__global__ void __launch_bounds__(256) k_inv_supers(InvCtx c, uint32_t nodes, uint32_t* __restrict__ nx,
                                                    uint32_t* __restrict__ dd) {
    if (ld_volatile(&c.ctrl[CTRL_ERR]) & (ERR_TIMEOUT | ERR_CAPACITY)) return;
    for (uint32_t node = blockIdx.x * blockDim.x + threadIdx.x; node < nodes; node += gridDim.x * blockDim.x) {
        SuperAt u;
        uint32_t next = INVALID, d = 0;
        if (super_at(c, node, u)) {
            uint32_t cur = u.slot;
            for (;;) {
                const uint2 r = *reinterpret_cast<const uint2*>(c.sample + cur);  // next, len
                d += r.y;
                cur = r.x;
                const uint32_t s = cur - u.base;
                if (s == u.m) {
                    next = END;
                    break;
                }
                if (s % SUP == 0) {
                    next = u.node0 + s / SUP;
                    break;
                }
            }
        }
        nx[node] = next;
        dd[node] = d;
    }
}

// One pointer-jumping round over the supers: dist += dist[next], next = next[next].
__global__ void __launch_bounds__(256) k_inv_jump(uint32_t nodes, const uint32_t* __restrict__ nx,
                                                  const uint32_t* __restrict__ dd, uint32_t* __restrict__ nx2,
                                                  uint32_t* __restrict__ dd2, const uint32_t* ctrl) {
    if (ld_volatile(&ctrl[CTRL_ERR]) & (ERR_TIMEOUT | ERR_CAPACITY)) return;
    for (uint32_t g = blockIdx.x * blockDim.x + threadIdx.x; g < nodes; g += gridDim.x * blockDim.x) {
        const uint32_t t = nx[g];
        const bool go = t < INVALID;
        dd2[g] = dd[g] + (go ? dd[t] : 0u);
        nx2[g] = go ? nx[t] : t;
    }
}

// All rounds of one block's supers at once, a CTA a block: the lists in
// shared memory (8 bytes a super), a thread holding up to JUMP_PER of them.
// For blocks of up to JUMP_MAX supers (1,048,504 bytes): on 64 blocks of
// 900,000 bytes (450,000 supers) 14 launches of 8 us each, on twice the supers
// one of 45 us.
constexpr uint32_t JUMP_PER = 16, JUMP_MAX = 1024 * JUMP_PER;
constexpr size_t JUMP_SMEM = (size_t)JUMP_MAX * 8;

__global__ void __launch_bounds__(1024) k_inv_jump_blocks(const uint32_t* __restrict__ sbase, uint32_t nb,
                                                          uint32_t* __restrict__ nx, uint32_t* __restrict__ dd,
                                                          const uint32_t* ctrl) {
    extern __shared__ __align__(8) uint2 list[];  // next super (relative to the block), distance
    if (ld_volatile(&ctrl[CTRL_ERR]) & (ERR_TIMEOUT | ERR_CAPACITY)) return;
    for (uint32_t b = blockIdx.x; b < nb; b += gridDim.x) {
        const uint32_t n0 = sbase[b], n = min(sbase[b + 1] - n0, JUMP_MAX);
        for (uint32_t i = threadIdx.x; i < n; i += 1024) {
            const uint32_t t = nx[n0 + i];
            list[i] = make_uint2(t < INVALID ? t - n0 : t, dd[n0 + i]);
        }
        __syncthreads();
        for (uint32_t len = 1; len <= n; len <<= 1) {  // >= log2(supers) + 1 rounds
            uint2 v[JUMP_PER];
#pragma unroll
            for (uint32_t k = 0; k < JUMP_PER; ++k) {
                const uint32_t i = k * 1024 + threadIdx.x;
                if (i < n) {
                    v[k] = list[i];
                    if (v[k].x < n) {
                        const uint2 t = list[v[k].x];
                        v[k] = make_uint2(t.x, v[k].y + t.y);
                    }
                }
            }
            __syncthreads();
#pragma unroll
            for (uint32_t k = 0; k < JUMP_PER; ++k) {
                const uint32_t i = k * 1024 + threadIdx.x;
                if (i < n) list[i] = v[k];
            }
            __syncthreads();
        }
        for (uint32_t i = threadIdx.x; i < n; i += 1024) {
            const uint2 v = list[i];
            nx[n0 + i] = v.x < INVALID ? v.x + n0 : v.x;
            dd[n0 + i] = v.y;
        }
        __syncthreads();
    }
}

// Appends bytes to consecutive addresses: whole aligned 8-byte words are
// stored at once, the first and the last by bytes.
struct ByteWriter {
    uint8_t* at;    // address of acc's byte 0 (8-byte aligned)
    uint64_t acc;
    uint32_t k;     // bytes in acc, counting the `lead` that are not ours
    uint32_t lead;

    __device__ __forceinline__ void init(uint8_t* p) {
        lead = k = (uint32_t)(reinterpret_cast<uintptr_t>(p) & 7u);
        at = p - k;
        acc = 0;
    }
    __device__ __forceinline__ void bytes(uint32_t to) {
        for (uint32_t q = lead; q < to; ++q) at[q] = (uint8_t)(acc >> (8 * q));
    }
    // the low n bytes of x (0 <= n <= 8)
    __device__ __forceinline__ void put(uint64_t x, uint32_t n) {
        if (n == 0) return;
        if (n < 8) x &= (1ull << (8 * n)) - 1ull;
        acc |= x << (8 * k);
        if (k + n < 8) {
            k += n;
            return;
        }
        if (lead) bytes(8);
        else *reinterpret_cast<uint64_t*>(at) = acc;
        lead = 0;
        at += 8;
        acc = k ? x >> (8 * (8 - k)) : 0ull;
        k = k + n - 8;
    }
    __device__ __forceinline__ void finish() { bytes(k); }
};

// Every super on the primary's cycle writes S from its text offset to the
// next super's. Each iteration a thread takes either one sample (its record
// and its stored bytes) or one step of a walk beyond them, so the threads of
// a warp wait for one load at a time, whichever they are at.
template <typename PT>
__global__ void __launch_bounds__(256) k_inv_write(InvCtx c, uint32_t nodes, const uint32_t* __restrict__ nx,
                                                   const uint32_t* __restrict__ dd) {
    if (ld_volatile(&c.ctrl[CTRL_ERR]) & (ERR_TIMEOUT | ERR_CAPACITY)) return;
    const PT* __restrict__ P = static_cast<const PT*>(c.P);
    for (uint32_t node = blockIdx.x * blockDim.x + threadIdx.x; node < nodes; node += gridDim.x * blockDim.x) {
        SuperAt u;
        if (!super_at(c, node, u) || nx[node] != END) continue;
        ByteWriter w;
        w.init(c.out + u.bi.off + (dd[u.node0 + u.nodes - 1] - dd[node]));  // cycle length - distance to the end
        uint32_t cur = u.slot, row = 0, rest = 0;
        bool more = true;
        while (more || rest) {
            ulonglong4 x = make_ulonglong4(0, 0, 0, 0);  // the sample
            PT v = 0;
            const bool walk = rest > 0;
            if (walk) v = P[row];
            if (!walk) {
                const ulonglong2* src = reinterpret_cast<const ulonglong2*>(c.sample + cur);
                const ulonglong2 lo = src[0], hi = src[1];
                x = make_ulonglong4(lo.x, lo.y, hi.x, hi.y);
            }
            if (walk) {
                w.put((uint64_t)v, 1);
                row = u.bi.off + (uint32_t)(v >> 8);
                --rest;
            } else {
                const uint32_t len = (uint32_t)(x.x >> 32);
                const uint32_t n = min(len, SBUF);  // the bytes stored: the top n of the 24
                const uint32_t low = SBUF - n;
                if (low >= 16u) x = make_ulonglong4(x.x, x.w, 0, 0);
                else if (low >= 8u) x = make_ulonglong4(x.x, x.z, x.w, 0);
                const uint32_t sh = 8u * (low & 7u);
                if (sh) {
                    x.y = (x.y >> sh) | (x.z << (64u - sh));
                    x.z = (x.z >> sh) | (x.w << (64u - sh));
                    x.w >>= sh;
                }
                w.put(x.y, min(8u, n));
                w.put(x.z, min(8u, n - min(n, 8u)));
                w.put(x.w, n - min(n, 16u));
                if (len > SBUF) {
                    rest = len - SBUF;
                    row = c.row[cur];
                }
                cur = (uint32_t)x.x;
                const uint32_t s = cur - u.base;
                more = !(s == u.m || s % SUP == 0);
            }
        }
        w.finish();
    }
}

// Periodic blocks: the primary's cycle covers one period; repeat it. A warp a
// tile: most batches have no such block, and a tile is then a few loads.
__global__ void __launch_bounds__(256) k_inv_replicate(InvCtx c, const TileDesc* __restrict__ tiles, uint32_t ntiles,
                                                       const uint32_t* __restrict__ dd) {
    if (ld_volatile(&c.ctrl[CTRL_ERR]) & (ERR_TIMEOUT | ERR_CAPACITY)) return;
    for (uint32_t t = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; t < ntiles; t += gridDim.x * blockDim.x >> 5) {
        const TileDesc td = tiles[t];
        const BlockInfo bi = c.blocks[td.blk];
        const int32_t prim_s = c.primary[td.blk];
        if (prim_s < 0 || (uint32_t)prim_s >= bi.n) continue;
        const uint32_t cyc = dd[c.sbase[td.blk + 1] - 1];
        if (cyc == 0 || cyc >= bi.n) continue;
        const uint32_t q0 = td.start - bi.off;
        for (uint32_t q = threadIdx.x & 31; q < td.len; q += 32)
            if (q0 + q >= cyc) c.out[td.start + q] = c.out[bi.off + (q0 + q) % cyc];
    }
}

template <typename PT>
void launch_inv_sort(bwt_plan* p, const uint8_t* L, uint32_t* counter, PT* P, cudaStream_t st) {
    const uint32_t nt = p->ntiles_il;
    const int sms = num_sms(), grid = std::max(1, std::min<int>((int)nt, sms * (p->rtile >= 4096 ? 5 : 6)));
    if (p->rtile == 1024)
        k_inv_sort<PT, 1024><<<grid, 256, 0, st>>>(L, p->blocks, p->tiles_il, nt, p->hist, p->status, counter, p->ctrl, P);
    else if (p->rtile == 2048)
        k_inv_sort<PT, 2048><<<grid, 256, 0, st>>>(L, p->blocks, p->tiles_il, nt, p->hist, p->status, counter, p->ctrl, P);
    else
        k_inv_sort<PT, 4096><<<grid, 256, 0, st>>>(L, p->blocks, p->tiles_il, nt, p->hist, p->status, counter, p->ctrl, P);
}

}  // namespace

extern "C" bwt_status bwt_inverse_batch(bwt_plan* p, const uint8_t* d_L, const uint64_t* offsets,
                                        uint32_t num_blocks, const int32_t* d_primary, uint8_t* d_out,
                                        void* stream) {
    if (!p || !d_L || !offsets || !d_primary || !d_out || (const void*)d_L == (const void*)d_out) return BWT_EINVAL;
    bwt::NvtxRange nvtx_range("inverse");
    if (cudaSetDevice(p->device) != cudaSuccess) return BWT_ECUDA;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    std::memset(&p->stats, 0, sizeof(p->stats));
    bwt_status s = prepare_batch(p, offsets, num_blocks, st);
    if (s != BWT_OK) return p->last = s;
    const uint32_t nb = p->nb, nt = p->ntiles0, total = p->total;
    // samples and supers per block
    uint32_t Q = 0, nodes = 0, max_nodes = 0;
    uint32_t* h_qbase = p->h_inv_items;
    uint32_t* h_sbase = p->h_inv_items + p->cap_b + 1;
    for (uint32_t b = 0; b < nb; ++b) {
        h_qbase[b] = Q;
        h_sbase[b] = nodes;
        const uint32_t m = (p->h_blocks[b].n + SMP - 1) / SMP, k = (m + SUP - 1) / SUP + 1;
        Q += m + 1;
        nodes += k;
        max_nodes = std::max(max_nodes, k);
    }
    h_qbase[nb] = Q;
    h_sbase[nb] = nodes;
    // scratch: a row a sample and 16 bytes a super in vals[0], the samples in
    // keys[0], which the inverse does not use otherwise (a plan for blocks of a
    // few bytes allocates its own on first use)
    const size_t slots = (size_t)(p->cap_n / SMP) + 2 * (size_t)p->cap_b + 1;
    const size_t sups = slots / SUP + 2 * (size_t)p->cap_b + 1;
    uint32_t* row = p->vals[0];
    if (4 * slots + 16 * sups > sizeof(uint32_t) * (size_t)p->cap_n) {
        if (!p->inv_slots) CKI(cudaMalloc(&p->inv_slots, 4 * slots + 16 * sups));
        row = p->inv_slots;
    }
    if (!p->inv_items) CKI(cudaMalloc(&p->inv_items, sizeof(uint32_t) * 2 * ((size_t)p->cap_b + 1)));
    Sample* sample = reinterpret_cast<Sample*>(p->keys[0]);
    if (slots * sizeof(Sample) > sizeof(uint64_t) * p->cap_n) {
        if (!p->inv_buf) CKI(cudaMalloc(&p->inv_buf, slots * sizeof(Sample)));
        sample = reinterpret_cast<Sample*>(p->inv_buf);
    }
    CKI(cudaMemcpyAsync(p->inv_items, h_qbase, sizeof(uint32_t) * 2 * ((size_t)p->cap_b + 1),
                        cudaMemcpyHostToDevice, st));
    if ((s = reset_ctrl(p, st)) != BWT_OK) return p->last = s;

    // 1. P by one stable pass over (L[k], k); 4 bytes a row while block rows
    //    fit in 24 bits, so twice as many blocks' tables stay in L2 during the
    //    walks
    const bool p32 = p->max_n <= (1u << 24);
    uint32_t* counters = p->ctrl + CTRL_TILE_CTR + 60;  // zeroed by reset_ctrl; no radix pass of this call uses them
    CKI(cudaMemsetAsync(p->hist, 0, sizeof(uint32_t) * 256 * nb, st));
    CKI(launch_hist_bytes(d_L, p->blocks, p->tiles0, nt, p->hist, st));
    CKI(launch_scan_rows(p->hist, 256, nullptr, 0, nb, nb, st));
    CKI(cudaMemsetAsync(p->status, 0, sizeof(uint32_t) * (size_t)p->ntiles_il * 256, st));
    if (p32) launch_inv_sort<uint32_t>(p, d_L, counters, reinterpret_cast<uint32_t*>(p->keys[1]), st);
    else launch_inv_sort<uint64_t>(p, d_L, counters, p->keys[1], st);
    CKI(cudaGetLastError());

    // 2-4. walks, supers, writes
    InvCtx c{};
    c.blocks = p->blocks;
    c.primary = d_primary;
    c.qbase = p->inv_items;
    c.sbase = p->inv_items + p->cap_b + 1;
    c.nb = nb;
    c.P = p->keys[1];
    c.row = row;
    c.sample = sample;
    c.out = d_out;
    c.ctrl = p->ctrl;
    uint32_t* nxb[2] = {c.row + slots, c.row + slots + sups};
    uint32_t* ddb[2] = {c.row + slots + 2 * sups, c.row + slots + 3 * sups};
    const int sms = num_sms();
    // walkers in flight: enough to hide latency, few enough that the blocks
    // being walked keep their tables in L2
    const int wgrid = sms * WALK_CTAS_PER_SM;
    const int grid = std::max(1, std::min<int>((int)((nodes + 255) / 256), sms * 8));
    if (p32) k_inv_walks<uint32_t><<<wgrid, 256, 0, st>>>(c, Q, counters + 1);
    else k_inv_walks<uint64_t><<<wgrid, 256, 0, st>>>(c, Q, counters + 1);
    k_inv_supers<<<grid, 256, 0, st>>>(c, nodes, nxb[0], ddb[0]);
    int src = 0, rounds = 1;
    if (max_nodes <= JUMP_MAX) {
        static const bool attr = cudaFuncSetAttribute((void*)k_inv_jump_blocks, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                      (int)JUMP_SMEM) == cudaSuccess;
        if (!attr) return p->last = record_cuda(cudaErrorInvalidValue, "cudaFuncSetAttribute");
        k_inv_jump_blocks<<<std::min<uint32_t>(nb, (uint32_t)sms), 1024, std::min<size_t>(JUMP_SMEM, 8ull * max_nodes),
                            st>>>(c.sbase, nb, nxb[0], ddb[0], p->ctrl);
    } else {
        while ((1u << (rounds - 1)) < max_nodes + 1) ++rounds;  // >= log2(supers per block) + 1
        for (int i = 0; i < rounds; ++i, src ^= 1)
            k_inv_jump<<<grid, 256, 0, st>>>(nodes, nxb[src], ddb[src], nxb[src ^ 1], ddb[src ^ 1], p->ctrl);
    }
    if (p32) k_inv_write<uint32_t><<<grid, 256, 0, st>>>(c, nodes, nxb[src], ddb[src]);
    else k_inv_write<uint64_t><<<grid, 256, 0, st>>>(c, nodes, nxb[src], ddb[src]);
    k_inv_replicate<<<std::max(1, std::min<int>((int)((nt + 7) / 8), sms * 8)), 256, 0, st>>>(c, p->tiles0, nt, ddb[src]);
    CKI(cudaGetLastError());
    p->stats.kernel_launches = 8 + rounds;
    p->stats.radix_launches = 1;
    p->stats.radix_keys = total;
    return p->last = finish_status(p, st);
}
