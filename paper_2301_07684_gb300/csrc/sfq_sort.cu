// sfq_sort.cu -- stable LSD radix sort of product records by (parent id, step, member,
// parent tag), so that runs can be compared with the oracle record by record.
//
// The key of a record is the pair of words (parent id, step << 4 | member << 2 | tag).  Only
// the bits in which the records of a call differ are sorted, eight at a time.
//   Up to SMALL_N records: one block, one launch.  It finds the differing bits, sorts 16-bit
//     indices in shared memory (digits are read from the records themselves) and permutes
//     the columns in place.
//   More: one pass over the records finds the differing bits and the host reads them.  If
//     the two windows of differing bits fit a 32- or 64-bit word together (the parent ids of
//     a population are an index range, so they nearly always do), records are sorted by that
//     composite key; the sorted keys are the sorted parent ids and steps, and only momenta
//     and meta bytes are gathered.  Else the sort runs in two stages, the secondary word
//     first, then the parent ids.
// One pass = a digit histogram per tile, one exclusive scan per digit over the tiles, and a
// stable scatter (sort_scatter_kernel).
#include <cstdint>
#include <cstring>

#include <cuda_runtime.h>

#include "sfq_internal.h"

namespace sfq {
namespace {

constexpr int RADIX = 256;
constexpr int SB = 256, SW = SB / 32, IPT = 16;          // threads and warps of a tile, records per thread
constexpr int TILE = SB * IPT;                           // records per tile

__device__ __forceinline__ uint64_t secondary(uint32_t step, uint8_t meta) {
    // member (bits 2-3) ranks before the parent tag (bits 4-5)
    return ((uint64_t)step << 4) | (((meta >> 2) & 3u) << 2) | ((meta >> 4) & 3u);
}

// The bits of the two words that are set in some record (or) and in all of them (and).
struct Bits {
    unsigned long long or_s, or_p, nand_s, nand_p;       // the complements of the ands
};
__device__ __forceinline__ void or_warp(unsigned long long &v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v |= __shfl_xor_sync(0xFFFFFFFFu, v, o);
}
__device__ __forceinline__ void accumulate(Bits &b, uint64_t s, uint64_t p) {
    b.or_s |= s; b.nand_s |= ~s;
    b.or_p |= p; b.nand_p |= ~p;
}
// Block-wide union; thread 0 gets it (ws: 4 words per warp).
__device__ __forceinline__ void or_block(Bits &b, unsigned long long *ws) {
    or_warp(b.or_s); or_warp(b.or_p); or_warp(b.nand_s); or_warp(b.nand_p);
    const int warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if ((threadIdx.x & 31) == 0) {
        ws[4 * warp] = b.or_s; ws[4 * warp + 1] = b.or_p; ws[4 * warp + 2] = b.nand_s; ws[4 * warp + 3] = b.nand_p;
    }
    __syncthreads();
    if (threadIdx.x == 0)
        for (int w = 1; w < nw; ++w) {
            b.or_s |= ws[4 * w]; b.or_p |= ws[4 * w + 1]; b.nand_s |= ws[4 * w + 2]; b.nand_p |= ws[4 * w + 3];
        }
}

// One atomic per block and word (one per warp took 37 us for 5.3e6 records, all on two words).
__global__ void __launch_bounds__(256) bits_kernel(int64_t n, const uint64_t *__restrict__ pid,
                                                   const uint32_t *__restrict__ step, const uint8_t *__restrict__ meta,
                                                   Bits *__restrict__ out) {
    __shared__ unsigned long long ws[4 * 8];
    Bits b{};
    // four records' loads in flight (past the end: the last record again, which adds nothing)
    for (int64_t i0 = blockIdx.x * 256ll + threadIdx.x; i0 < n; i0 += gridDim.x * 1024ll) {
        uint64_t p[4];
        uint32_t st[4];
        uint8_t m[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int64_t j = i0 + k * (int64_t)gridDim.x * 256, i = j < n ? j : n - 1;
            p[k] = pid[i]; st[k] = step[i]; m[k] = meta[i];
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) accumulate(b, secondary(st[k], m[k]), p[k]);
    }
    or_block(b, ws);
    if (threadIdx.x == 0) {
        atomicOr(&out->or_s, b.or_s); atomicOr(&out->or_p, b.or_p);
        atomicOr(&out->nand_s, b.nand_s); atomicOr(&out->nand_p, b.nand_p);
    }
}

// The window [lo, lo + width) of differing bits of a word; the bits outside it are `fixed` in
// every record.
struct Window {
    int lo, width;
    uint64_t fixed;
};
__host__ __device__ inline uint64_t low_bits(int w) { return w >= 64 ? ~0ull : (1ull << w) - 1ull; }
// Position of word `v` in the composite key, and back.
__device__ __forceinline__ uint64_t pack(uint64_t v, const Window &w) { return (v >> w.lo) & low_bits(w.width); }
__device__ __forceinline__ uint64_t unpack(uint64_t k, const Window &w) {
    return w.width ? ((k & low_bits(w.width)) << w.lo) | w.fixed : w.fixed;
}

// Digit counts of a tile (digit-major: counts[d * ntiles + tile]).  COMPOSE also forms the keys:
// 1 from both words, 2 the secondary word alone, 3 the parent ids in the order of `perm`.
template <typename K, int COMPOSE>
__global__ void __launch_bounds__(SB) sort_hist_kernel(int64_t n, K *__restrict__ key, const uint64_t *__restrict__ pid,
                                                       const uint32_t *__restrict__ step,
                                                       const uint8_t *__restrict__ meta,
                                                       const uint32_t *__restrict__ perm, Window ws, Window wp,
                                                       int shift, uint32_t *__restrict__ counts, int ntiles) {
    __shared__ uint32_t h[RADIX];
    for (int d = threadIdx.x; d < RADIX; d += SB) h[d] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * TILE;
    K v[IPT];                                             // the tile's loads go out together
#pragma unroll
    for (int k = 0; k < IPT; ++k) {
        const int64_t j = base + k * SB + threadIdx.x, i = j < n ? j : n - 1;
        if (COMPOSE == 1) v[k] = (K)(pack(pid[i], wp) << ws.width | pack(secondary(step[i], meta[i]), ws));
        else if (COMPOSE == 2) v[k] = (K)pack(secondary(step[i], meta[i]), ws);
        else if (COMPOSE == 3) v[k] = (K)pack(pid[perm ? perm[i] : (uint32_t)i], wp);
        else v[k] = key[i];
    }
#pragma unroll
    for (int k = 0; k < IPT; ++k) {
        const int64_t i = base + k * SB + threadIdx.x;
        if (i < n) {
            if (COMPOSE) key[i] = v[k];
            atomicAdd(&h[(uint32_t)(v[k] >> shift) & 0xFFu], 1u);
        }
    }
    __syncthreads();
    for (int d = threadIdx.x; d < RADIX; d += SB) counts[(int64_t)d * ntiles + blockIdx.x] = h[d];
}

// Exclusive scan, in place, of every digit's row of tile counts; total[d] receives the row's sum.
// One block per digit: a row of 4.2e6 records is one chunk.
constexpr int SCAN_BS = 1024;
__device__ __forceinline__ uint32_t warp_inclusive(uint32_t x, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, x, o);
        if (lane >= o) x += t;
    }
    return x;
}
__global__ void __launch_bounds__(SCAN_BS) sort_scan_kernel(uint32_t *__restrict__ counts, int ntiles,
                                                            uint32_t *__restrict__ total) {
    __shared__ uint32_t wsum[SCAN_BS / 32];
    uint32_t *row = counts + (int64_t)blockIdx.x * ntiles;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    uint32_t carry = 0;
    for (int b0 = 0; b0 < ntiles; b0 += blockDim.x) {
        const int i = b0 + threadIdx.x;
        const uint32_t v = i < ntiles ? row[i] : 0u;
        const uint32_t x = warp_inclusive(v, lane);
        if (lane == 31) wsum[warp] = x;
        __syncthreads();
        if (warp == 0) wsum[lane] = warp_inclusive(lane < nw ? wsum[lane] : 0u, lane);
        __syncthreads();
        if (i < ntiles) row[i] = carry + (warp ? wsum[warp - 1] : 0u) + x - v;
        carry += wsum[nw - 1];
        __syncthreads();                                  // wsum is rewritten by the next chunk
    }
    if (threadIdx.x == 0) total[blockIdx.x] = carry;
}

// The lanes whose record has the same digit (0 for a lane without a record): one ballot per
// digit bit.  __match_any_sync takes a step per distinct value: with 32 of them in a warp the
// scatter took 68 us a pass for 5.3e6 records.
__device__ __forceinline__ unsigned warp_peers(uint32_t d, bool valid) {
    unsigned peers = __ballot_sync(0xFFFFFFFFu, valid);
#pragma unroll
    for (int b = 0; b < 8; ++b) {
        const bool bit = (d >> b) & 1u;
        const unsigned m = __ballot_sync(0xFFFFFFFFu, bit);
        peers &= bit ? m : ~m;
    }
    return valid ? peers : 0u;
}
// Rank of each lane's record among the warp's records of its digit so far: the lowest lane of
// a digit adds its peers to the warp's count (`run`).
__device__ __forceinline__ uint32_t warp_rank(uint32_t *run, uint32_t d, bool valid, int lane) {
    const unsigned peers = warp_peers(d, valid);
    const int first = peers ? __ffs(peers) - 1 : 0;
    uint32_t before = 0;
    if (peers && lane == first) before = atomicAdd(&run[d], (uint32_t)__popc(peers));
    __syncwarp();                                         // the next round's addition follows this one
    return __shfl_sync(0xFFFFFFFFu, before, first) + __popc(peers & ((1u << lane) - 1u));
}

// Stable scatter of (key, index) pairs by one digit.  Each warp of a block ranks 512 successive
// records; the block joins the warps' counts, orders its tile in shared memory and writes it
// out as runs of equal digits.  5.3e6 records: 38 us a pass (53 to 113 us with one warp
// ranking and scattering 2048 records by itself, 47 us of which however few records there
// were: 64 rounds, each a chain of shared-memory round trips).  Issue and the phases'
// latency bound it; 64 registers for 32-bit keys keep two tiles' worth of warps on an SM
// (128 registers: 48 us).
// idx_in == NULL: the records are in their original order.
template <typename K>
struct ScatterSmem {
    uint32_t run[SW][RADIX];
    uint32_t delta[RADIX];                                // global position minus position in the tile
    uint32_t dsum[16];
    uint32_t idx[TILE];
    K key[TILE];
};
template <typename K>
__global__ void __launch_bounds__(SB, sizeof(K) == 4 ? 1024 / SB : 512 / SB)
    sort_scatter_kernel(int64_t n, const K *__restrict__ key_in, const uint32_t *__restrict__ idx_in,
                        K *__restrict__ key_out, uint32_t *__restrict__ idx_out, int shift,
                        const uint32_t *__restrict__ counts, int ntiles, const uint32_t *__restrict__ total) {
    extern __shared__ __align__(16) unsigned char smraw[];
    ScatterSmem<K> &S = *reinterpret_cast<ScatterSmem<K> *>(smraw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t base = (int64_t)blockIdx.x * TILE;
    const int m = n - base < TILE ? (int)(n - base) : TILE;
    for (int d = lane; d < RADIX; d += 32) S.run[warp][d] = 0;
    K key[IPT];
    uint32_t idx[IPT], rank[IPT];
#pragma unroll
    for (int r = 0; r < IPT; ++r) {
        const int at = (warp * IPT + r) * 32 + lane;
        key[r] = at < m ? key_in[base + at] : (K)0;
    }
    __syncwarp();
#pragma unroll
    for (int r = 0; r < IPT; ++r)
        rank[r] = warp_rank(S.run[warp], (uint32_t)(key[r] >> shift) & 0xFFu, (warp * IPT + r) * 32 + lane < m, lane);
    // the indices are fetched here, behind the ranking's registers
#pragma unroll
    for (int r = 0; r < IPT; ++r) {
        const int at = (warp * IPT + r) * 32 + lane;
        idx[r] = idx_in && at < m ? idx_in[base + at] : (uint32_t)(base + at);
    }
    __syncthreads();
    // per digit: the warps' exclusive counts, the digit's start in the tile and in the output
    uint32_t mine = 0, all = 0, in = 0, ina = 0;
    if (tid < RADIX) {
#pragma unroll
        for (int w = 0; w < SW; ++w) {
            const uint32_t t = S.run[w][tid];
            S.run[w][tid] = mine;
            mine += t;
        }
        all = total[tid];
        in = warp_inclusive(mine, lane);
        ina = warp_inclusive(all, lane);
        if (lane == 31) {
            S.dsum[warp] = in;
            S.dsum[warp + 8] = ina;
        }
    }
    __syncthreads();
    if (tid < RADIX) {
        uint32_t loc = in - mine, glob = ina - all;
        for (int w = 0; w < warp; ++w) {
            loc += S.dsum[w];
            glob += S.dsum[w + 8];
        }
#pragma unroll
        for (int w = 0; w < SW; ++w) S.run[w][tid] += loc;
        S.delta[tid] = glob + counts[(int64_t)tid * ntiles + blockIdx.x] - loc;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < IPT; ++r) {
        if ((warp * IPT + r) * 32 + lane < m) {
            const uint32_t at = S.run[warp][(uint32_t)(key[r] >> shift) & 0xFFu] + rank[r];
            S.key[at] = key[r];
            S.idx[at] = idx[r];
        }
    }
    __syncthreads();
#pragma unroll 4
    for (int j = tid; j < m; j += SB) {
        const K k = S.key[j];
        const uint32_t to = S.delta[(uint32_t)(k >> shift) & 0xFFu] + (uint32_t)j;
        if (to < n) {                                     // holds for a correct scan
            key_out[to] = k;
            idx_out[to] = S.idx[j];
        }
    }
}
static_assert(RADIX == 8 * 32 && SW >= 8, "digits are scanned by the first eight warps");

// Before they are gathered, a record's momentum and meta byte are put side by side: a gather
// then touches one 32-byte sector of a record instead of four (5.3e6 records: 102 us from
// separate columns and 20 us to copy them back), and writes the columns themselves.
template <typename T> struct Packed;
template <> struct __align__(16) Packed<float> { float x, y, z; uint32_t meta; };
template <> struct Packed<double> { double x, y, z; };   // meta bytes follow the array
template <typename T>
__global__ void __launch_bounds__(256) sort_pack_kernel(int64_t n, const T *__restrict__ px, const T *__restrict__ py,
                                                        const T *__restrict__ pz, const uint8_t *__restrict__ meta,
                                                        Packed<T> *__restrict__ out) {
    for (int64_t i = blockIdx.x * 256ll + threadIdx.x; i < n; i += gridDim.x * 256ll) {
        Packed<T> v;
        v.x = px[i]; v.y = py[i]; v.z = pz[i];
        if constexpr (sizeof(T) == 4) v.meta = meta[i];
        else reinterpret_cast<uint8_t *>(out + n)[i] = meta[i];
        out[i] = v;
    }
}
// The columns in sorted order: parent ids and steps from the sorted keys.
template <typename T, typename K>
__global__ void __launch_bounds__(256) sort_gather_kernel(int64_t n, const uint32_t *__restrict__ perm,
                                                          const K *__restrict__ key, Window ws, Window wp,
                                                          const Packed<T> *__restrict__ in, T *__restrict__ px,
                                                          T *__restrict__ py, T *__restrict__ pz,
                                                          uint8_t *__restrict__ meta, uint64_t *__restrict__ pid,
                                                          uint32_t *__restrict__ step) {
    for (int64_t i = blockIdx.x * 256ll + threadIdx.x; i < n; i += gridDim.x * 256ll) {
        const uint32_t j = perm[i];
        const uint64_t k = key[i];
        if (j < n) {                                      // perm is a permutation of [0, n)
            const Packed<T> v = in[j];
            px[i] = v.x; py[i] = v.y; pz[i] = v.z;
            if constexpr (sizeof(T) == 4) meta[i] = (uint8_t)v.meta;
            else meta[i] = reinterpret_cast<const uint8_t *>(in + n)[j];
        }
        pid[i] = unpack(ws.width < 64 ? k >> ws.width : 0ull, wp);
        step[i] = (uint32_t)(unpack(k, ws) >> 4);
    }
}

// One column in the order of `perm` (the two-stage sort).
template <typename T>
__global__ void gather_kernel(int64_t n, const uint32_t *__restrict__ perm, const T *__restrict__ src,
                              T *__restrict__ dst) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    {
        const uint32_t j = perm[i];
        dst[i] = j < n ? src[j] : T(0);
    }
}

// ---------------------------------------------------------------------------
// Up to SMALL_N records in one block: a step loop's few thousand photons, where the launches
// and the read-back of the general path are what a caller waits for.  A call with 1000 / 8000 /
// 16384 records takes 37 / 59 / 91 us from Python, 74 / 77 / 100 us through the general path,
// so the line is where one SM's latency meets it.
constexpr int SMALL_N = 16384, MB = 1024, MW = MB / 32, MR = SMALL_N / MB;
static_assert(SMALL_N <= 1 << 14 && SMALL_N / MW <= 1 << 9, "index, digit and rank share a word");
struct SmallSmem {
    uint16_t idx[2][SMALL_N];
    uint32_t run[MW][RADIX];
    uint32_t start[RADIX];
    uint32_t dsum[8];
    unsigned long long bits[4 * MW];
    Bits all;
};
template <typename T>
__global__ void __launch_bounds__(MB) small_sort_kernel(int n, T *__restrict__ px, T *__restrict__ py, T *__restrict__ pz,
                                                        uint64_t *__restrict__ pid, uint32_t *__restrict__ step,
                                                        uint8_t *__restrict__ meta) {
    extern __shared__ __align__(16) unsigned char smraw[];
    SmallSmem &S = *reinterpret_cast<SmallSmem *>(smraw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rounds = (n + MB - 1) / MB;                 // records per thread; a warp's are successive
    Bits b{};
#pragma unroll 4
    for (int r = 0; r < MR; ++r) {
        const int i = r * MB + tid < n ? r * MB + tid : n - 1;
        if (r < rounds) accumulate(b, secondary(step[i], meta[i]), pid[i]);
    }
    or_block(b, S.bits);
    if (tid == 0) S.all = b;
    __syncthreads();
    b = S.all;
    int cur = -1;                                         // the buffer that holds the order (-1: as given)
    for (int word = 0; word < 2; ++word) {
        uint64_t diff = word ? b.or_p & b.nand_p : b.or_s & b.nand_s;
        while (diff) {
            const int lo = __ffsll((long long)diff) - 1;
            diff &= ~(0xFFull << lo);
            for (int d = lane; d < RADIX; d += 32) S.run[warp][d] = 0;
            uint32_t it[MR];                              // index | digit << 14 | rank in the warp << 23
#pragma unroll
            for (int r = 0; r < MR; ++r) {
                const int at = (warp * rounds + r) * 32 + lane;
                it[r] = (uint32_t)RADIX << 14;
                if (r < rounds && at < n) {
                    const uint32_t id = cur < 0 ? (uint32_t)at : S.idx[cur][at];
                    const uint64_t v = word ? pid[id] : secondary(step[id], meta[id]);
                    it[r] = id | (uint32_t)((v >> lo) & 0xFFu) << 14;
                }
            }
            __syncwarp();
#pragma unroll
            for (int r = 0; r < MR; ++r)
                if (r < rounds) {
                    const uint32_t d = (it[r] >> 14) & 0xFFu;
                    it[r] |= warp_rank(S.run[warp], d, !((it[r] >> 22) & 1u), lane) << 23;
                }
            __syncthreads();
            uint32_t mine = 0, in = 0;
            if (tid < RADIX) {
                for (int w = 0; w < MW; ++w) {
                    const uint32_t t = S.run[w][tid];
                    S.run[w][tid] = mine;
                    mine += t;
                }
                in = warp_inclusive(mine, lane);
                if (lane == 31) S.dsum[warp] = in;
            }
            __syncthreads();
            if (tid < RADIX) {
                uint32_t loc = in - mine;
                for (int w = 0; w < warp; ++w) loc += S.dsum[w];
                S.start[tid] = loc;
            }
            __syncthreads();
            const int nxt = cur == 0 ? 1 : 0;
#pragma unroll
            for (int r = 0; r < MR; ++r)
                if (r < rounds && !((it[r] >> 22) & 1u)) {
                    const uint32_t d = (it[r] >> 14) & 0xFFu;
                    S.idx[nxt][S.start[d] + S.run[warp][d] + (it[r] >> 23)] = (uint16_t)(it[r] & 0x3FFFu);
                }
            cur = nxt;
            __syncthreads();
        }
    }
    if (cur < 0) return;
    // the columns in place: every record of a column is read before any is written
    const uint16_t *order = S.idx[cur];
#define SFQ_PERMUTE(C, col)                                                  \
    {                                                                        \
        C v[MR];                                                             \
        _Pragma("unroll") for (int r = 0; r < MR; ++r)                       \
            if (r * MB + tid < n) v[r] = col[order[r * MB + tid]];           \
        __syncthreads();                                                     \
        _Pragma("unroll") for (int r = 0; r < MR; ++r)                       \
            if (r * MB + tid < n) col[r * MB + tid] = v[r];                  \
    }
    SFQ_PERMUTE(T, px)
    SFQ_PERMUTE(T, py)
    SFQ_PERMUTE(T, pz)
    SFQ_PERMUTE(uint64_t, pid)
    SFQ_PERMUTE(uint32_t, step)
    SFQ_PERMUTE(uint8_t, meta)
#undef SFQ_PERMUTE
}

// ---------------------------------------------------------------------------
size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }

// Two buffers of keys and indices, the tile counts, and room for the gathered columns.  A
// sort ends in the first pair; what follows it (28 bytes per record or more) is then free and
// takes the columns.
struct Plan {
    size_t o_ka, o_ia, o_kb, o_ib, o_cnt, o_tot, o_bits, total;
    int ntiles;
};

Plan plan(int64_t n) {
    Plan p{};
    p.ntiles = (int)((n + TILE - 1) / TILE);
    size_t o = 0;
    p.o_bits = o; o += 256;
    p.o_tot = o; o += RADIX * 4;
    p.o_cnt = o; o += align256((size_t)p.ntiles * RADIX * 4);
    p.o_ka = o; o += align256(n * 8);
    p.o_ia = o; o += align256(n * 4);
    p.o_kb = o; o += align256(n * 8);
    p.o_ib = o; o += align256(n * 4);
    o += align256(n * 16);
    p.total = o;
    return p;
}

// The scratch a caller provides: as large as the sort's first version asked for (three 8-byte
// and two 4-byte columns, counts of 2048-record tiles and one column), which holds the plan.
size_t contract_bytes(int64_t n) {
    const int64_t ncnt = (n + 2047) / 2048 * RADIX, nchunks = (ncnt + 4095) / 4096;
    return 3 * align256(n * 8) + 2 * align256(n * 4) + align256((size_t)ncnt * 4) + align256((size_t)nchunks * 4) + 256 +
           align256(n * 8);
}

Window window_of(uint64_t or_bits, uint64_t nand_bits) {
    const uint64_t diff = or_bits & nand_bits;
    if (!diff) return Window{0, 0, ~nand_bits};
    const int lo = __builtin_ctzll(diff), width = 64 - __builtin_clzll(diff) - lo;
    return Window{lo, width, ~nand_bits & ~(low_bits(width) << lo)};
}

// LSD passes over `bits` key bits.  The keys are formed by the first histogram (COMPOSE); the
// passes alternate between the buffers so that the last one writes buffer 0.
template <typename K, int COMPOSE>
cudaError_t passes(const sfq_products &out, int64_t n, const Window &ws, const Window &wp, int bits, K *const key[2],
                   uint32_t *const idx[2], const uint32_t *perm, int from, uint32_t *cnt, uint32_t *tot, int ntiles,
                   cudaStream_t s) {
    const cudaError_t e = cudaFuncSetAttribute(sort_scatter_kernel<K>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)sizeof(ScatterSmem<K>));
    if (e != cudaSuccess) return e;
    int cur = from;
    for (int shift = 0; shift < bits; shift += 8, cur ^= 1) {
        const uint32_t *in = shift ? idx[cur] : perm;
        if (shift == 0)
            sort_hist_kernel<K, COMPOSE><<<ntiles, SB, 0, s>>>(n, key[cur], out.parent_id, out.step, out.meta, perm, ws,
                                                              wp, shift, cnt, ntiles);
        else
            sort_hist_kernel<K, 0><<<ntiles, SB, 0, s>>>(n, key[cur], nullptr, nullptr, nullptr, nullptr, ws, wp, shift,
                                                         cnt, ntiles);
        sort_scan_kernel<<<RADIX, ntiles < SCAN_BS ? (ntiles + 31) / 32 * 32 : SCAN_BS, 0, s>>>(cnt, ntiles, tot);
        sort_scatter_kernel<K><<<ntiles, SB, sizeof(ScatterSmem<K>), s>>>(n, key[cur], in, key[cur ^ 1], idx[cur ^ 1],
                                                                         shift, cnt, ntiles, tot);
    }
    return cudaGetLastError();
}

template <typename T, typename K>
cudaError_t composite_sort(const sfq_products &out, int64_t n, const Window &ws, const Window &wp, char *sc,
                           const Plan &P, cudaStream_t s, int num_sms) {
    K *key[2] = {reinterpret_cast<K *>(sc + P.o_ka), reinterpret_cast<K *>(sc + P.o_kb)};
    uint32_t *idx[2] = {reinterpret_cast<uint32_t *>(sc + P.o_ia), reinterpret_cast<uint32_t *>(sc + P.o_ib)};
    const int bits = ws.width + wp.width, np = (bits + 7) / 8;
    cudaError_t e = passes<K, 1>(out, n, ws, wp, bits, key, idx, nullptr, np & 1, reinterpret_cast<uint32_t *>(sc + P.o_cnt),
                                 reinterpret_cast<uint32_t *>(sc + P.o_tot), P.ntiles, s);
    if (e != cudaSuccess) return e;
    Packed<T> *packed = reinterpret_cast<Packed<T> *>(sc + P.o_kb);
    T *px = static_cast<T *>(out.px), *py = static_cast<T *>(out.py), *pz = static_cast<T *>(out.pz);
    const int64_t blocks = (n + 255) / 256;
    const int grid = (int)(blocks < num_sms * 8ll ? blocks : num_sms * 8ll);
    sort_pack_kernel<T><<<grid, 256, 0, s>>>(n, px, py, pz, out.meta, packed);
    sort_gather_kernel<T, K><<<grid, 256, 0, s>>>(n, idx[0], key[0], ws, wp, packed, px, py, pz, out.meta, out.parent_id,
                                                 out.step);
    return cudaGetLastError();
}

// Both words in turn (their windows do not fit 64 bits together: hashed parent ids).
cudaError_t two_stage_sort(const sfq_products &out, int64_t n, size_t elem, const Window &ws, const Window &wp, char *sc,
                           const Plan &P, cudaStream_t s, int num_sms) {
    uint64_t *key[2] = {reinterpret_cast<uint64_t *>(sc + P.o_ka), reinterpret_cast<uint64_t *>(sc + P.o_kb)};
    uint32_t *idx[2] = {reinterpret_cast<uint32_t *>(sc + P.o_ia), reinterpret_cast<uint32_t *>(sc + P.o_ib)};
    uint32_t *cnt = reinterpret_cast<uint32_t *>(sc + P.o_cnt), *tot = reinterpret_cast<uint32_t *>(sc + P.o_tot);
    const int p0 = (ws.width + 7) / 8, p1 = (wp.width + 7) / 8;
    const int mid = p1 & 1;                               // where the second stage starts, to end in buffer 0
    cudaError_t e = passes<uint64_t, 2>(out, n, ws, wp, ws.width, key, idx, nullptr, (mid ^ p0) & 1, cnt, tot, P.ntiles, s);
    if (e == cudaSuccess)
        e = passes<uint64_t, 3>(out, n, ws, wp, wp.width, key, idx, p0 ? idx[mid] : nullptr, mid, cnt, tot, P.ntiles, s);
    if (e != cudaSuccess) return e;
    void *tmp = sc + P.o_kb;
    const int grid = num_sms * 8;
#define SFQ_GATHER(T, ptr)                                                                                 \
    gather_kernel<T><<<grid, 256, 0, s>>>(n, idx[0], static_cast<const T *>(ptr), static_cast<T *>(tmp));   \
    e = cudaMemcpyAsync(ptr, tmp, (size_t)n * sizeof(T), cudaMemcpyDeviceToDevice, s);                      \
    if (e != cudaSuccess) return e;
    if (elem == 4) {
        SFQ_GATHER(float, out.px) SFQ_GATHER(float, out.py) SFQ_GATHER(float, out.pz)
    } else {
        SFQ_GATHER(double, out.px) SFQ_GATHER(double, out.py) SFQ_GATHER(double, out.pz)
    }
    SFQ_GATHER(uint64_t, out.parent_id)
    SFQ_GATHER(uint32_t, out.step)
    SFQ_GATHER(uint8_t, out.meta)
#undef SFQ_GATHER
    return cudaGetLastError();
}

template <typename T>
cudaError_t small_sort(const sfq_products &out, int n, cudaStream_t s) {
    const cudaError_t e = cudaFuncSetAttribute(small_sort_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)sizeof(SmallSmem));
    if (e != cudaSuccess) return e;
    small_sort_kernel<T><<<1, MB, sizeof(SmallSmem), s>>>(n, static_cast<T *>(out.px), static_cast<T *>(out.py),
                                                          static_cast<T *>(out.pz), out.parent_id, out.step, out.meta);
    return cudaGetLastError();
}

}  // namespace

cudaError_t sort_products(const sfq_products &out, int64_t n, size_t elem, void *scratch, cudaStream_t s,
                          int num_sms) {
    if (n <= 1) return cudaSuccess;
    // a sort reads back key bits, so it is not recorded into a graph; the one-block sort would be,
    // with its record count fixed, and is refused alike
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    cudaError_t e = cudaStreamIsCapturing(s, &cap);
    if (e != cudaSuccess) return e;
    if (cap != cudaStreamCaptureStatusNone) return cudaErrorStreamCaptureUnsupported;
    if (n <= SMALL_N) {
        // every sort waits for the stream's earlier work: the larger ones by their read-back, this
        // one only because callers rely on it (a step loop has read the record count by now and
        // finds the stream idle)
        e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) return e;
        return elem == 4 ? small_sort<float>(out, (int)n, s) : small_sort<double>(out, (int)n, s);
    }
    const Plan P = plan(n);
    char *sc = static_cast<char *>(scratch);
    Bits *bits = reinterpret_cast<Bits *>(sc + P.o_bits);
    e = cudaMemsetAsync(bits, 0, sizeof(Bits), s);
    if (e != cudaSuccess) return e;
    const int64_t blocks = (n + 256 * 8 - 1) / (256 * 8);
    bits_kernel<<<(unsigned)(blocks < num_sms * 8ll ? blocks : num_sms * 8ll), 256, 0, s>>>(n, out.parent_id, out.step,
                                                                                          out.meta, bits);
    Bits h;
    e = cudaMemcpyAsync(&h, bits, sizeof(h), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return e;
    const Window ws = window_of(h.or_s, h.nand_s), wp = window_of(h.or_p, h.nand_p);
    const int width = ws.width + wp.width;
    if (width == 0) return cudaSuccess;                   // one key: the records are in order
    if (width > 64) return two_stage_sort(out, n, elem, ws, wp, sc, P, s, num_sms);
    if (elem == 4)
        return width <= 32 ? composite_sort<float, uint32_t>(out, n, ws, wp, sc, P, s, num_sms)
                           : composite_sort<float, uint64_t>(out, n, ws, wp, sc, P, s, num_sms);
    return width <= 32 ? composite_sort<double, uint32_t>(out, n, ws, wp, sc, P, s, num_sms)
                       : composite_sort<double, uint64_t>(out, n, ws, wp, sc, P, s, num_sms);
}

size_t sort_scratch_bytes(int64_t n, size_t) {
    return n <= 1 ? 256 : contract_bytes(n);                             // plan(n).total fits it above SMALL_N
}

}  // namespace sfq
