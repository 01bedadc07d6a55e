// Sort-based bulk build (Sec. 3 "Bulk Operations"): the table is built from a
// batch by sorting the batch by hash, dropping all but the last of equal keys,
// and placing the survivors as an insertion in that order would: element i
// (in sorted order) lands at P_i = max(home_i, P_{i-1} + 1), the paper's
// "start looking at max(h(x), i)" rule.  Positions past the last cell wrap to
// the first empty cells from cell 0 on.
//
// GB300 mapping.
//   1. LSD radix sort of the (key, value) cells by the top B bits of the hash
//      (B = 32 for tables of up to 2^32 cells), 8 bits per pass: one kernel
//      counts the digits of all passes, then each pass reads and writes the
//      cells once, tiles of 4096 cells finding their places by decoupled
//      look-back.  The first pass reads the caller's key and value arrays; the
//      count notes keys 0 / ~0 (for the special slots or the reserved status
//      bit, both set only once the build is sure).
//   2. Placement as a scan: with r_i the number of survivors before i,
//      P_i = r_i + max over survivors j <= i of (home_j - r_j), so a scan of
//      (count, max) pairs under (C1, M1) + (C2, M2) = (C1 + C2,
//      max(M1, M2 - C1)) gives every position at once.  One pass reduces
//      chunks of 2048 cells (8 consecutive ones per thread), one CTA scans the
//      chunk totals, one pass writes the cells (positions rise with i: a
//      chunk's survivors are staged by rank and stored by consecutive threads).
//   3. One thread places the survivors whose position passed the last cell
//      (the tail of the sorted order) at the first empty cells from 0, in
//      order, and sets the counters and special slots.
#include "cht_internal.h"

namespace cht {
namespace {

constexpr int kSortThreads = 256;
constexpr int kPassThreads = 512;
constexpr int kSortItems = 8;
constexpr u32 kSortTile = kPassThreads * kSortItems;  // cells per radix tile
constexpr int kScanThreads = 256;
constexpr u32 kScanChunk = kScanThreads * 16;          // u32 per scan chunk
constexpr int kPlaceItems = 8;
constexpr u32 kPlaceChunk = 256 * kPlaceItems;         // cells per placement chunk
constexpr long long kNegInf = -(1ll << 62);

struct SortSrc {
    const Cell* cells;  // null: read keys / vals (the first pass)
    const u64* keys;
    const u64* vals;
};

__device__ __forceinline__ void load_src(const SortSrc& s, u64 i, u64& k, u64& v) {
    if (s.cells) {
        ld_cell_cg(s.cells + i, k, v);
    } else {
        k = s.keys[i];
        v = s.vals[i];
    }
}

// top B bits of the hash
__device__ __forceinline__ u64 sort_key(u64 k, u32 B) { return fmix64(k) >> (64u - B); }

// Inclusive sum over a 256-thread block; `total` gets the block sum.  sh:
// 8 words of shared scratch.
__device__ __forceinline__ u32 block_incl_u32(u32 x, u32& total, u32* sh) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int o = 1; o < 32; o <<= 1) {
        const u32 y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sh[w] = x;
    __syncthreads();
    u32 pre = 0, tot = 0;
    for (int j = 0; j < kScanThreads / 32; ++j) {
        if (j < w) pre += sh[j];
        tot += sh[j];
    }
    __syncthreads();
    total = tot;
    return pre + x;
}

// ---------------------------------------------------------------------------
// radix sort
// ---------------------------------------------------------------------------
constexpr int kDigits = 256;
constexpr int kMaxPasses = 5;  // sort keys of at most 40 bits

// The digit counts of every pass in one read of the keys (8 bytes a pair,
// where a count before each pass read the whole cells again).  Also notes keys
// 0 / ~0: they take the special slots (the last copy's value) or set the
// reserved status bit; they never enter the table.
__global__ void __launch_bounds__(kSortThreads) radix_count_kernel(const u64* keys, u64 n, u32 B, u32* hist,
                                                                   BuildExtra* ex, int full_keys) {
    pdl_enter();
    __shared__ u32 bins[kMaxPasses][kDigits];
    const int passes = int(B / 8);
    for (int p = 0; p < passes; ++p) bins[p][threadIdx.x] = 0;
    __syncthreads();
    const u64 step = u64(gridDim.x) * (kSortThreads * 8);
    for (u64 base = u64(blockIdx.x) * (kSortThreads * 8); base < n; base += step) {
        u64 k[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const u64 i = base + u32(q) * kSortThreads + threadIdx.x;
            k[q] = i < n ? keys[i] : 1;
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const u64 i = base + u32(q) * kSortThreads + threadIdx.x;
            if (i >= n) break;
            const u64 s = sort_key(k[q], B);
            for (int p = 0; p < passes; ++p) atomicAdd(&bins[p][u32(s >> (8 * p)) & 255u], 1u);
            if (is_reserved(k[q])) {
                if (full_keys)
                    atomicMax(&ex->sp_last[k[q] == kEmpty ? 0 : 1], i + 1);
                else
                    atomicOr(&ex->reserved, 1ull);
            }
        }
    }
    __syncthreads();
    for (int p = 0; p < passes; ++p)
        if (bins[p][threadIdx.x]) atomicAdd(&hist[p * kDigits + threadIdx.x], bins[p][threadIdx.x]);
}

// A tile's digit counts on their way to prefixes: bits 0-31 the count (of this
// tile, or of all tiles up to it), bits 32-33 which (kTileCount, kTilePrefix),
// from bit 34 the pass + 1, so that one zeroed array serves all passes.
constexpr u64 kTileCount = 1ull << 32, kTilePrefix = 2ull << 32;
constexpr u32 kMaxPolls = 1u << 22;  // a few seconds

struct PassArgs {
    SortSrc src;
    Cell* dst;
    u64 n;
    u32 B, pass;
    const u32* hist;  // this pass's digit counts
    u64* tiles;       // [tile][kDigits]
    u32* ticket;      // this pass's tile counter (zero before the launch)
};

// Digit `d` in the tiles before `tile`, counted from the cells themselves:
// what a lookback falls back on if a tile's counts never appear.
__device__ __noinline__ u32 recount_digit(const PassArgs& a, u32 tile, u32 d) {
    u32 sum = 0;
    for (u64 i = 0; i < u64(tile) * kSortTile; ++i) {
        u64 k, v;
        load_src(a.src, i, k, v);
        sum += (u32(sort_key(k, a.B) >> (8 * a.pass)) & 255u) == d;
    }
    return sum;
}

// One stable 8-bit pass.  A tile ranks its cells (warp w has 256 of them, 8
// steps of 32 consecutive ones: eight ballots give each lane the lanes with
// its digit, a per-warp counter in shared memory the count of earlier steps),
// publishes its digit counts, and gets the counts of the tiles before it by
// looking back over theirs (decoupled look-back, Merrill & Garland, "Single-pass
// Parallel Prefix Scan with Decoupled Look-back", 2016; used for radix sorting by
// Adinets & Merrill, "Onesweep", arXiv 2206.01784): one read and one write of
// the cells per pass and no count or scan kernels between.  Tiles come from a
// ticket, so those looked back at are running or done.  The tile is reordered
// by digit in shared memory (stable) and written from there: consecutive
// threads write consecutive cells of a digit's run, so the stores coalesce.
// Bound by shared memory (random 16-byte stores of the reordering).  2^25
// pairs, a pass: count + scan + scatter 390 us -> 330 us; 2048 to 8192 cells a
// tile and looking back at 1 to 24 tiles at a time are slower.
template <bool kFirst>
__global__ void __launch_bounds__(kPassThreads, 2) radix_pass_kernel(PassArgs a) {
    constexpr int kW = kPassThreads / 32;
    pdl_enter();
    extern __shared__ __align__(16) unsigned char smem[];
    Cell* const stage = reinterpret_cast<Cell*>(smem);                             // kSortTile cells
    unsigned short(*const wcnt)[kDigits + 2] = reinterpret_cast<unsigned short(*)[kDigits + 2]>(stage + kSortTile);
    u32* const goff = reinterpret_cast<u32*>(&wcnt[kW][0]);                        // place of a digit's run - its slot
    unsigned char* const sdig = reinterpret_cast<unsigned char*>(goff + kDigits);  // kSortTile
    __shared__ u32 sh[2][8];
    __shared__ u32 s_tile;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const u32 below = (1u << lane) - 1u;
    const u32 shift = 8 * a.pass;
    if (threadIdx.x == 0) s_tile = atomicAdd(a.ticket, 1u);
    for (u32 j = threadIdx.x; j < u32(kW) * (kDigits + 2) / 2; j += kPassThreads) reinterpret_cast<u32*>(wcnt)[j] = 0;
    __syncthreads();
    const u32 tile = s_tile;
    const u64 tbase = u64(tile) * kSortTile;
    const u64 base = tbase + u64(w) * (32 * kSortItems);
    u64 ks[kSortItems], vs[kSortItems];
    u32 dr[kSortItems];  // digit << 16 | rank in the warp
    // all loads first (in flight together), then the ranking votes
#pragma unroll
    for (int q = 0; q < kSortItems; ++q) {
        const u64 i = base + u64(q) * 32 + lane;
        ks[q] = 0;
        vs[q] = 0;
        if (i < a.n) {
            if (kFirst) {
                ks[q] = a.src.keys[i];
                vs[q] = a.src.vals[i];
            } else {
                ld_cell_cg(a.src.cells + i, ks[q], vs[q]);
            }
        }
    }
#pragma unroll
    for (int q = 0; q < kSortItems; ++q) {
        const bool valid = base + u64(q) * 32 + lane < a.n;
        const u32 d = u32(sort_key(ks[q], a.B) >> shift) & 255u;
        // lanes with the same digit: eight ballots, one per digit bit
        u32 peers = __ballot_sync(0xffffffffu, valid);
#pragma unroll
        for (int bit = 0; bit < 8; ++bit) {
            const u32 m = __ballot_sync(0xffffffffu, (d >> bit) & 1u);
            peers &= ((d >> bit) & 1u) ? m : ~m;
        }
        const u32 b = wcnt[w][d];
        dr[q] = (d << 16) | (b + __popc(peers & below));
        __syncwarp();
        if (valid && (peers & below) == 0u) wcnt[w][d] = (unsigned short)(b + __popc(peers));  // the lowest lane
        __syncwarp();
    }
    __syncthreads();
    if (threadIdx.x < kDigits) {
        // the tile's count of this thread's digit (and exclusive over the warps)
        const u32 d = threadIdx.x;
        u32 cnt = 0;
#pragma unroll
        for (int x = 0; x < kW; ++x) {
            const u32 t = wcnt[x][d];
            wcnt[x][d] = (unsigned short)cnt;
            cnt += t;
        }
        const u64 tag = u64(a.pass + 1) << 34;
        volatile u64* const mine = a.tiles + u64(tile) * kDigits + d;
        *mine = tag | (tile == 0 ? kTilePrefix : kTileCount) | cnt;
        // where the digit's run starts, in the tile and in the output
        const u32 h = a.hist[d];
        u32 x = cnt, g = h;
        for (int o = 1; o < 32; o <<= 1) {
            const u32 y = __shfl_up_sync(0xffffffffu, x, o), z = __shfl_up_sync(0xffffffffu, g, o);
            if (lane >= o) {
                x += y;
                g += z;
            }
        }
        if (lane == 31) {
            sh[0][w] = x;
            sh[1][w] = g;
        }
        asm volatile("bar.sync 1, 256;" ::: "memory");  // the eight warps with a digit per thread
        u32 slot = x - cnt, place = g - h;
        for (int j = 0; j < w; ++j) {
            slot += sh[0][j];
            place += sh[1][j];
        }
#pragma unroll
        for (int y = 0; y < kW; ++y) wcnt[y][d] = (unsigned short)(wcnt[y][d] + slot);
        u32 before = 0;
        if (tile > 0) {
            u32 polls = 0;
            for (u32 t = tile;;) {
                u64 v[4];  // four tiles at a time, the loads in flight together
#pragma unroll
                for (u32 u = 0; u < 4; ++u)
                    v[u] = u < t ? *(volatile u64*)(a.tiles + u64(t - 1 - u) * kDigits + d) : 0;
                bool done = false, wait = false;
                u32 used = 0;
#pragma unroll
                for (u32 u = 0; u < 4; ++u) {
                    if (done || wait) continue;
                    if ((v[u] >> 34) != a.pass + 1) {
                        wait = true;
                        continue;
                    }
                    before += u32(v[u]);
                    ++used;
                    done = (v[u] & kTilePrefix) != 0;
                }
                if (done) break;
                t -= used;
                if (wait && ++polls > kMaxPolls) {
                    before = recount_digit(a, tile, d);
                    break;
                }
            }
            *mine = tag | kTilePrefix | (before + cnt);
        }
        goff[d] = place + before - slot;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kSortItems; ++q) {
        if (base + u64(q) * 32 + lane < a.n) {
            const u32 d = dr[q] >> 16, j = wcnt[w][d] + (dr[q] & 0xffffu);
            Cell cl;
            cl.key = ks[q];
            cl.val = vs[q];
            stage[j] = cl;
            sdig[j] = (unsigned char)d;
        }
    }
    __syncthreads();
    const u32 cnt = a.n - tbase < kSortTile ? u32(a.n - tbase) : kSortTile;
    for (u32 j = threadIdx.x; j < cnt; j += kPassThreads) {
        const u32 to = goff[sdig[j]] + j;
        if (to < a.n) a.dst[to] = stage[j];
    }
}

constexpr size_t pass_smem_bytes() {
    return size_t(kSortTile) * sizeof(Cell) + size_t(kPassThreads / 32) * (kDigits + 2) * 2 + kDigits * 4 + kSortTile;
}

// ---------------------------------------------------------------------------
// exclusive scan of u32 (the digit-major histogram), in place
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kScanThreads) scan_reduce_kernel(const u32* in, u64 m, u32* part) {
    pdl_enter();
    __shared__ u32 sh[kScanThreads / 32];
    const u64 base = u64(blockIdx.x) * kScanChunk;
    u32 s = 0;
    for (int q = 0; q < 16; ++q) {
        const u64 i = base + u64(q) * kScanThreads + threadIdx.x;
        if (i < m) s += in[i];
    }
    u32 total;
    block_incl_u32(s, total, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = total;
}

__global__ void __launch_bounds__(kScanThreads) scan_partials_kernel(u32* part, u64 np) {
    pdl_enter();
    __shared__ u32 sh[kScanThreads / 32];
    u32 carry = 0;
    for (u64 b = 0; b < np; b += kScanThreads) {
        const u64 i = b + threadIdx.x;
        const u32 x = i < np ? part[i] : 0u;
        u32 total;
        const u32 incl = block_incl_u32(x, total, sh);
        if (i < np) part[i] = carry + incl - x;
        carry += total;
    }
}

__global__ void __launch_bounds__(kScanThreads) scan_apply_kernel(u32* data, u64 m, const u32* part) {
    pdl_enter();
    __shared__ u32 sh[kScanThreads / 32];
    const u64 base = u64(blockIdx.x) * kScanChunk;
    u32 carry = part[blockIdx.x];
    for (int q = 0; q < 16; ++q) {
        const u64 i = base + u64(q) * kScanThreads + threadIdx.x;
        const u32 x = i < m ? data[i] : 0u;
        u32 total;
        const u32 incl = block_incl_u32(x, total, sh);
        if (i < m) data[i] = carry + incl - x;
        carry += total;
    }
}

cudaError_t scan_exclusive(u32* data, u64 m, u32* part, cudaStream_t s) {
    const u64 nb = (m + kScanChunk - 1) / kScanChunk;
    launch_overlapped(scan_reduce_kernel, unsigned(nb), kScanThreads, 0, s, data, m, part);
    launch_overlapped(scan_partials_kernel, 1, kScanThreads, 0, s, part, nb);
    launch_overlapped(scan_apply_kernel, unsigned(nb), kScanThreads, 0, s, data, m, part);
    count_launch();
    count_launch();
    count_launch();
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// placement: scan of (count, max) pairs
// ---------------------------------------------------------------------------
struct Agg {
    u32 c;        // survivors
    long long m;  // max over survivors j of (home_j - rank_j), ranks local to the segment
};

__device__ __forceinline__ Agg agg_join(Agg a, Agg b) {
    Agg r;
    r.c = a.c + b.c;
    const long long bm = b.m - (long long)a.c;
    r.m = a.m > bm ? a.m : bm;
    return r;
}

// One past the position of the last survivor (0: none).
__device__ __forceinline__ u64 agg_end(Agg a) { return a.c ? u64((long long)a.c + a.m) : 0; }

// The cells of a dense write from w0 on that are too many for one CTA: written
// densely, 2048 at a time behind barriers, they go at a CTA's own rate.  With
// mostly distinct keys a chunk of 2048 sorted cells owns at most 16 times as
// many (build_place_dense); copies of few keys leave few survivors and long
// ranges, which the whole grid zeroes first (build_zero_kernel), and the chunk
// then writes its survivors alone.  (2^24 copies of 16 keys merged into an
// empty table of 2^25 cells: 2.88 -> 1.29 ms, 2^24 distinct ones 1.27 ms; the
// launch that finds nothing to zero costs a merge 2-4 us.)
constexpr u64 kMaxDense = 1ull << 16;
struct LongRange {
    u64 first, count;
};

// Inclusive scan of one Agg per thread over a 256-thread block; `total` gets
// the block's join.
__device__ __forceinline__ Agg block_incl_agg(Agg x, Agg& total, u32* shc, long long* shm) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int o = 1; o < 32; o <<= 1) {
        Agg y;
        y.c = __shfl_up_sync(0xffffffffu, x.c, o);
        y.m = __shfl_up_sync(0xffffffffu, x.m, o);
        if (lane >= o) x = agg_join(y, x);
    }
    if (lane == 31) {
        shc[w] = x.c;
        shm[w] = x.m;
    }
    __syncthreads();
    Agg pre = {0u, kNegInf}, tot = {0u, kNegInf};
    for (int j = 0; j < 8; ++j) {
        Agg t;
        t.c = shc[j];
        t.m = shm[j];
        if (j < w) pre = agg_join(pre, t);
        tot = agg_join(tot, t);
    }
    __syncthreads();
    total = tot;
    return agg_join(pre, x);
}

struct PlaceArgs {
    const Cell* srt;       // sorted cells
    u64 n;
    u32 B, log2c;
    Agg* parts;            // per chunk: its join (count passes), then its exclusive prefix
    unsigned char* flags;  // per sorted cell: 1 survivor, 0 not, 2 deferred
    u32* deferred;         // cells whose survivor test was deferred (count in ex->n_deferred)
    unsigned char* dirty;  // per chunk: a deferred cell of it turned out to survive
    Cell* cells;           // the table
    int dense;             // write every cell of the table, empty ones too
    LongRange* longs;      // dense: the ranges over kMaxDense (count in ex->n_long)
    Cell* ov;              // survivors past the last cell, by rank
    BuildExtra* ex;
};

// (These kernels overlap the launches before them, which write what they read:
// their loads are coherent ones, not read-only ones.)
__device__ __forceinline__ u64 ld_key(const Cell* p) {
    u64 k;
    asm volatile("ld.global.cg.u64 %0, [%1];" : "=l"(k) : "l"(p));
    return k;
}

constexpr int kRunScan = 32;  // cells a survivor test looks ahead before deferring

// Survivor test, first try.  A cell survives if its key is not reserved and
// no later cell of the same sort key (equal keys have equal hashes, so their
// copies share that run) holds the same key.  Nearly always the next cell
// decides; when a different key with the same top B hash bits sits between
// (a run mixing keys), up to kRunScan cells are looked at, after which the
// test is deferred (2) to a CTA of its own (build_resolve_kernel), so that a
// rare key inside a long run of copies of another key costs no long scan by
// one thread.
// k, s: the cell's key and sort key; kn, sn: the next cell's.
__device__ __forceinline__ unsigned char survivor_first(const PlaceArgs& a, u64 i, u64 k, u64 s, u64 kn, u64 sn) {
    if (is_reserved(k)) return 0;
    if (i + 1 >= a.n) return 1;
    if (sn != s) return 1;
    if (kn == k) return 0;
    for (u64 j = i + 2; j < a.n && j < i + 2 + kRunScan; ++j) {
        const u64 kj = ld_key(a.srt + j);
        if (sort_key(kj, a.B) != s) return 1;
        if (kj == k) return 0;
    }
    return i + 2 + kRunScan >= a.n ? 1 : 2;
}

// Count passes (MODE 0: decide survivors and write the flags; MODE 1: only
// for chunks where a deferred cell survived, recount from the flags) and the
// write pass (MODE 2).  Each thread takes kPlaceItems consecutive sorted
// cells.  The count passes store each chunk's join; the write pass turns the
// chunk's exclusive prefix plus the thread's into ranks and positions.
//
// The chunk goes through shared memory: coalesced loads in, and each thread
// reads its consecutive cells from there, one slot of padding after every
// kPlaceItems so that the threads of a warp fall on different banks.  (Loaded
// by their threads directly, every load instruction touched 32 lines, and the
// unpadded stage had 8-way bank conflicts on every store: the write pass was
// bound by shared memory, short_scoreboard 12 per issue.  2^25 cells into
// 2^26: count 170 -> 134 us, write 382 -> 313 us.)
__device__ __forceinline__ u32 padded(u32 i) { return i + i / kPlaceItems; }
constexpr u32 kPlaceWin = 2048;  // cells per window of a dense write
constexpr u32 kPlacePad = kPlaceChunk + kPlaceChunk / kPlaceItems;

template <int MODE>
__global__ void __launch_bounds__(256) build_place_kernel(PlaceArgs a) {
    pdl_enter();
    __shared__ u32 shc[8];
    __shared__ long long shm[8];
    __shared__ u32 ic[256];
    __shared__ long long im[256];
    // the write pass stages whole cells and lists the survivors by rank, the
    // count passes stage keys
    extern __shared__ __align__(16) unsigned char psm[];
    Cell* const stage = reinterpret_cast<Cell*>(psm);
    u64* const skey = reinterpret_cast<u64*>(psm);
    u64* const spos = reinterpret_cast<u64*>(stage + kPlacePad);
    unsigned short* const sidx = reinterpret_cast<unsigned short*>(spos + kPlaceChunk);
    if (MODE == 1 && a.dirty[blockIdx.x] == 0) return;
    const u64 c = 1ull << a.log2c;
    const u32 hshift = a.B - a.log2c;
    const u64 c0 = u64(blockIdx.x) * kPlaceChunk;
    const u64 i0 = c0 + u64(threadIdx.x) * kPlaceItems;
    {
        u64 k[kPlaceItems], v[kPlaceItems];
#pragma unroll
        for (int q = 0; q < kPlaceItems; ++q) {
            const u64 i = c0 + u32(q) * 256 + threadIdx.x;
            k[q] = kEmpty;
            v[q] = 0;
            if (i < a.n) {
                if (MODE == 2) ld_cell_cg(a.srt + i, k[q], v[q]);
                else k[q] = ld_key(a.srt + i);
            }
        }
#pragma unroll
        for (int q = 0; q < kPlaceItems; ++q) {
            const u32 j = padded(u32(q) * 256 + threadIdx.x);
            if (MODE == 2) {
                stage[j].key = k[q];
                stage[j].val = v[q];
            } else {
                skey[j] = k[q];
            }
        }
    }
    // the thread's eight flags are one word (flags of a chunk start 8-byte aligned)
    u64 fl = 0;
    if (MODE != 0) {
        if (i0 + kPlaceItems <= a.n) {
            fl = *reinterpret_cast<const u64*>(a.flags + i0);
        } else {
            for (int q = 0; q < kPlaceItems; ++q)
                if (i0 + q < a.n) fl |= u64(a.flags[i0 + q]) << (8 * q);
        }
    }
    __syncthreads();
    const u32 s0 = threadIdx.x * (kPlaceItems + 1);  // padded(threadIdx.x * kPlaceItems)
    u64 ks[kPlaceItems];
#pragma unroll
    for (int q = 0; q < kPlaceItems; ++q) ks[q] = MODE == 2 ? stage[s0 + q].key : skey[s0 + q];
    u64 ss[kPlaceItems];  // sort keys: each hash is computed once
#pragma unroll
    for (int q = 0; q < kPlaceItems; ++q) ss[q] = sort_key(ks[q], a.B);
    u32 sv = 0;
    if (MODE == 0) {
        u64 knext = kEmpty;
        if (i0 + kPlaceItems < a.n)
            knext = threadIdx.x < 255 ? skey[s0 + kPlaceItems + 1] : ld_key(a.srt + i0 + kPlaceItems);
        const u64 snext = sort_key(knext, a.B);
#pragma unroll
        for (int q = 0; q < kPlaceItems; ++q) {
            if (i0 + q >= a.n) continue;
            const unsigned char f =
                q + 1 < kPlaceItems
                    ? survivor_first(a, i0 + q, ks[q], ss[q], ks[(q + 1) % kPlaceItems], ss[(q + 1) % kPlaceItems])
                    : survivor_first(a, i0 + q, ks[q], ss[q], knext, snext);
            fl |= u64(f) << (8 * q);
            if (f == 1) sv |= 1u << q;
            if (f == 2) a.deferred[atomicAdd(&a.ex->n_deferred, 1u)] = u32(i0 + q);
        }
        if (i0 + kPlaceItems <= a.n) {
            *reinterpret_cast<u64*>(a.flags + i0) = fl;
        } else {
            for (int q = 0; q < kPlaceItems; ++q)
                if (i0 + q < a.n) a.flags[i0 + q] = (unsigned char)(fl >> (8 * q));
        }
    } else {
#pragma unroll
        for (int q = 0; q < kPlaceItems; ++q)
            if (((fl >> (8 * q)) & 255u) == 1u) sv |= 1u << q;
    }
    Agg loc = {0u, kNegInf};
#pragma unroll
    for (int q = 0; q < kPlaceItems; ++q) {
        if (!((sv >> q) & 1u)) continue;
        const Agg x = {1u, (long long)(ss[q] >> hshift)};
        loc = agg_join(loc, x);
    }
    Agg tot;
    const Agg incl = block_incl_agg(loc, tot, shc, shm);
    if (MODE != 2) {
        if (threadIdx.x == 0) a.parts[blockIdx.x] = tot;
        return;
    }
    ic[threadIdx.x] = incl.c;
    im[threadIdx.x] = incl.m;
    __syncthreads();
    const Agg first = a.parts[blockIdx.x];
    Agg carry = first;
    if (threadIdx.x > 0) {
        const Agg left = {ic[threadIdx.x - 1], im[threadIdx.x - 1]};
        carry = agg_join(carry, left);
    }
    // the chunk's survivors, by rank, with their positions, so that
    // consecutive threads then store consecutive survivors (rising positions)
#pragma unroll
    for (int q = 0; q < kPlaceItems; ++q) {
        if (!((sv >> q) & 1u)) continue;
        const u64 home = ss[q] >> hshift;
        const u64 rank = carry.c;
        const long long hm = (long long)home - (long long)rank;
        const long long m = carry.m > hm ? carry.m : hm;
        const u32 j = carry.c - first.c;
        spos[j] = rank + u64(m);
        sidx[j] = (unsigned short)(s0 + q);
        const Agg x = {1u, (long long)home};
        carry = agg_join(carry, x);
    }
    // the cells a dense write covers: from after the last survivor of the chunks
    // before to this chunk's last one (the last chunk: to the end of the table)
    u64 w0 = agg_end(first);
    u64 end = tot.c ? agg_end(agg_join(first, tot)) : w0;
    if (blockIdx.x + 1 == gridDim.x || end > c) end = c;
    const bool dense = a.dense && (end <= w0 || end - w0 <= kMaxDense);
    __syncthreads();
    for (u32 j = threadIdx.x; j < tot.c; j += 256) {
        const u64 p = spos[j];
        if (p < c && dense) continue;
        const Cell cl = stage[sidx[j]];
        if (p < c) {
            a.cells[p] = cl;
        } else {
            const u64 rank = u64(first.c) + j;
            a.ov[rank] = cl;
            atomicMin(&a.ex->first_ov, rank);
        }
    }
    if (!dense) return;
    // dense: a window of kPlaceWin cells at a time through a map from cell to
    // survivor
    unsigned short* const map = sidx + kPlaceChunk;
    const Cell zero = {0ull, 0ull};
    u32 j = threadIdx.x;  // this thread's next survivor
    for (; w0 < end; w0 += kPlaceWin) {
        const u32 len = end - w0 < kPlaceWin ? u32(end - w0) : kPlaceWin;
        for (u32 x = threadIdx.x; x < kPlaceWin / 4; x += 256) reinterpret_cast<u64*>(map)[x] = ~0ull;
        __syncthreads();
        for (; j < tot.c && spos[j] < w0 + len; j += 256) map[spos[j] - w0] = sidx[j];
        __syncthreads();
        for (u32 x = threadIdx.x; x < len; x += 256) {
            const unsigned short i = map[x];
            a.cells[w0 + x] = i == 0xffffu ? zero : stage[i];
        }
        __syncthreads();
    }
}

template <int MODE>
u64 place_smem_bytes() {
    return MODE == 2 ? size_t(kPlacePad) * sizeof(Cell) + size_t(kPlaceChunk) * (sizeof(u64) + 2) + kPlaceWin * 2
                     : size_t(kPlacePad) * sizeof(u64);
}

// ---------------------------------------------------------------------------
// Deferred survivor tests: one CTA per deferred cell scans the rest of its run
// 2048 cells at a time (coalesced) for another copy of its key; a survivor
// marks its chunk for the recount.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) build_resolve_kernel(PlaceArgs a) {
    pdl_enter();
    __shared__ u64 sh_found[8], sh_end[8];
    const u32 nd = a.ex->n_deferred;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (u32 d = blockIdx.x; d < nd; d += gridDim.x) {
        const u64 i = a.deferred[d];
        const u64 k = ld_key(a.srt + i);
        const u64 s = sort_key(k, a.B);
        unsigned char f = 1;
        for (u64 j0 = i + 2; j0 < a.n; j0 += kPlaceChunk) {
            u64 found = ~0ull, end = ~0ull;
            for (int q = 0; q < kPlaceItems; ++q) {
                const u64 j = j0 + u64(q) * 256 + threadIdx.x;
                if (j >= a.n) {
                    end = end < a.n ? end : a.n;
                    continue;
                }
                const u64 kj = ld_key(a.srt + j);
                if (sort_key(kj, a.B) != s) end = end < j ? end : j;
                else if (kj == k) found = found < j ? found : j;
            }
            for (int o = 16; o > 0; o >>= 1) {
                const u64 f2 = __shfl_xor_sync(0xffffffffu, found, o);
                const u64 e2 = __shfl_xor_sync(0xffffffffu, end, o);
                found = f2 < found ? f2 : found;
                end = e2 < end ? e2 : end;
            }
            if (lane == 0) {
                sh_found[w] = found;
                sh_end[w] = end;
            }
            __syncthreads();
            found = sh_found[0];
            end = sh_end[0];
            for (int v = 1; v < 8; ++v) {
                found = sh_found[v] < found ? sh_found[v] : found;
                end = sh_end[v] < end ? sh_end[v] : end;
            }
            __syncthreads();
            if (found < end) {  // a later copy inside the run
                f = 0;
                break;
            }
            if (end != ~0ull) break;  // the run ended first
        }
        if (threadIdx.x == 0) {
            a.flags[i] = f;
            if (f) a.dirty[i / kPlaceChunk] = 1;
        }
    }
}

// One CTA: exclusive prefixes of the chunk joins, the survivor count S; kScanJoins
// joins at a time through shared memory, eight consecutive ones a thread
// (padded as in the placement), one block scan for each.  (256 joins at a time
// took 69 us for 2^14 chunks, 8192 at a time by 1024 threads 30 us.)
constexpr u32 kScanJoins = 2048;

// With `longs` (a dense write follows) it also lists the chunks' ranges over
// kMaxDense, as the write pass computes them.
__global__ void __launch_bounds__(256) build_place_scan_kernel(Agg* parts, u64 np, BuildExtra* ex, LongRange* longs,
                                                               u64 c) {
    pdl_enter();
    __shared__ Agg st[kScanJoins / 8 * 9];
    __shared__ u32 shc[8];
    __shared__ long long shm[8];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    Agg carry = {0u, kNegInf};
    for (u64 b = 0; b < np; b += kScanJoins) {
#pragma unroll
        for (u32 q = 0; q < kScanJoins / 256; ++q) {
            const u32 j = q * 256 + threadIdx.x;
            st[j + j / 8] = b + j < np ? parts[b + j] : Agg{0u, kNegInf};
        }
        __syncthreads();
        Agg* const mine = st + threadIdx.x * 9;
        Agg x = mine[0];
#pragma unroll
        for (int q = 1; q < 8; ++q) x = agg_join(x, mine[q]);
        for (int o = 1; o < 32; o <<= 1) {
            Agg y;
            y.c = __shfl_up_sync(0xffffffffu, x.c, o);
            y.m = __shfl_up_sync(0xffffffffu, x.m, o);
            if (lane >= o) x = agg_join(y, x);
        }
        if (lane == 31) {
            shc[w] = x.c;
            shm[w] = x.m;
        }
        Agg left;
        left.c = __shfl_up_sync(0xffffffffu, x.c, 1);
        left.m = __shfl_up_sync(0xffffffffu, x.m, 1);
        if (lane == 0) left = {0u, kNegInf};
        __syncthreads();
        Agg pre = carry;
        for (int j = 0; j < 8; ++j) {
            const Agg t = {shc[j], shm[j]};
            if (j < w) pre = agg_join(pre, t);
            carry = agg_join(carry, t);
        }
        // the join has no inverse (max), so prefixes are carried forward
        pre = agg_join(pre, left);
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const Agg y = mine[q];
            mine[q] = pre;
            pre = agg_join(pre, y);
        }
        if (longs) {  // (the thread's eight ranges together, then each)
            const u64 j0 = b + u64(threadIdx.x) * 8;
            if (j0 < np && (j0 + 8 >= np || agg_end(pre) > agg_end(mine[0]) + kMaxDense)) {
                for (u32 q = 0; q < 8 && j0 + q < np; ++q) {
                    const u64 w0 = agg_end(mine[q]), e1 = agg_end(q < 7 ? mine[q + 1] : pre);
                    const u64 e = j0 + q + 1 == np || e1 > c ? c : e1;
                    if (e > w0 && e - w0 > kMaxDense) longs[atomicAdd(&ex->n_long, 1u)] = LongRange{w0, e - w0};
                }
            }
        }
        __syncthreads();
#pragma unroll
        for (u32 q = 0; q < kScanJoins / 256; ++q) {
            const u32 j = q * 256 + threadIdx.x;
            if (b + j < np) parts[b + j] = st[j + j / 8];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        ex->S = carry.c;
        ex->first_ov = ~0ull;
    }
}

// Zeroes the long ranges, the whole grid on each (none: returns at once).
__global__ void __launch_bounds__(256) build_zero_kernel(Cell* cells, const LongRange* longs, const BuildExtra* ex) {
    pdl_enter();
    const u32 n = ex->n_long;
    const Cell zero = {0ull, 0ull};
    for (u32 r = 0; r < n; ++r) {
        const LongRange x = longs[r];
        for (u64 i = u64(blockIdx.x) * 256 + threadIdx.x; i < x.count; i += u64(gridDim.x) * 256)
            cells[x.first + i] = zero;
    }
}

// One thread: survivors whose position passed the last cell take the first
// empty cells from cell 0 on, in sorted order (a sequential insertion wraps
// the same way; the cells before them are final); then the counters and the
// special slots (the last copy's value).
__global__ void build_finish_kernel(Cell* cells, u32 log2c, const Cell* ov, BuildExtra* ex, DevState* st,
                                    const u64* vals) {
    pdl_enter();
    if (threadIdx.x != 0) return;
    const u64 c = 1ull << log2c;
    const u64 S = ex->S;
    u64 cursor = 0;
    for (u64 r = ex->first_ov; r < S; ++r) {
        while (cursor < c && cells[cursor].key != kEmpty) ++cursor;
        if (cursor >= c) {  // cannot happen while S < c
            st->status |= kFull;
            break;
        }
        cells[cursor] = ov[r];
        ++cursor;
    }
    st->I = S;
    st->D = 0;
    if (ex->reserved) st->status |= kReserved;
    for (int sl = 0; sl < 2; ++sl) {
        const u64 last = ex->sp_last[sl];
        if (last) {
            st->sp_present[sl] = 1u;
            st->sp_val[sl] = vals[last - 1];
        }
    }
}

}  // namespace

u32 build_sort_bits(u32 log2c) { return log2c <= 32 ? 32u : 8u * ((log2c + 7u) / 8u); }

namespace {
// Scratch layout: two sort buffers, the tiles' digit prefixes, the chunk joins, the survivor flags, the deferred list, the
// chunks' recount marks, the long ranges, the counters.
constexpr u64 kCountBytes = (kMaxPasses * (kDigits + 1) * 4 + 255) & ~255ull;
struct Layout {
    u64 ntiles, nchunks;
    u64 off_buf1, off_tiles, off_parts, off_flags, off_def, off_dirty, off_long, off_ex, off_counts, total;
    explicit Layout(u64 n) {
        auto al = [](u64 x) { return (x + 255) & ~255ull; };
        ntiles = (n + kSortTile - 1) / kSortTile;
        nchunks = (n + kPlaceChunk - 1) / kPlaceChunk;
        off_buf1 = al(n * sizeof(Cell));
        off_tiles = off_buf1 + al(n * sizeof(Cell));
        off_parts = off_tiles + al(ntiles * kDigits * sizeof(u64));
        off_flags = off_parts + al(nchunks * sizeof(Agg));
        off_def = off_flags + al(n);
        off_dirty = off_def + al(n * 4);
        // (a dense write has n >= c / 8: at most c / kMaxDense long ranges)
        off_long = off_dirty + al(nchunks);
        off_ex = off_long + al((8 * n / kMaxDense + 2) * sizeof(LongRange));
        off_counts = off_ex + al(sizeof(BuildExtra));  // digit counts and tile tickets of the passes
        total = off_counts + kCountBytes;
    }
};

PlaceArgs place_args(const Cell* sorted, u64 n, u32 log2c, void* scratch, BuildExtra* ex) {
    const Layout L(n);
    unsigned char* base = static_cast<unsigned char*>(scratch);
    PlaceArgs a;
    a.srt = sorted;
    a.n = n;
    a.B = build_sort_bits(log2c);
    a.log2c = log2c;
    a.parts = reinterpret_cast<Agg*>(base + L.off_parts);
    a.flags = base + L.off_flags;
    a.deferred = reinterpret_cast<u32*>(base + L.off_def);
    a.dirty = base + L.off_dirty;
    a.cells = nullptr;
    a.dense = 0;
    a.longs = reinterpret_cast<LongRange*>(base + L.off_long);
    // the survivors past the last cell go to whichever sort buffer does not
    // hold the sorted cells
    Cell* b0 = reinterpret_cast<Cell*>(base);
    a.ov = sorted == b0 ? reinterpret_cast<Cell*>(base + L.off_buf1) : b0;
    a.ex = ex;
    return a;
}
}  // namespace

namespace {
// ---------------------------------------------------------------------------
// Merge of two runs sorted by sort key (a table's live cells and a batch), the
// first run's cells before the second's where sort keys are equal: the stable
// sort of their concatenation, in one pass.  Merge path (Green, McColl & Bader,
// "GPU Merge Path", 2012): a binary search over the cells finds where each
// tile of kPlaceChunk output cells begins in both runs (a kernel of its own,
// one thread per tile: ~25 dependent reads, which took 5/8 of the time when
// each tile's CTA waited for its own); the tile's two parts go to shared memory
// and each thread merges kPlaceItems cells of it.
// ---------------------------------------------------------------------------
struct MergeArgs {
    const Cell* x;  // nx cells
    const Cell* y;  // ny cells
    u64 nx, ny;
    u32 B;
    u32* split;  // per tile: cells of x before it
    Cell* out;
};

// How many of the first `diag` merged cells come from x.
__device__ __forceinline__ u64 merge_split(const MergeArgs& a, u64 diag) {
    u64 lo = diag > a.ny ? diag - a.ny : 0, hi = diag < a.nx ? diag : a.nx;
    while (lo < hi) {
        const u64 mid = (lo + hi) / 2;
        if (sort_key(ld_key(a.x + mid), a.B) <= sort_key(ld_key(a.y + (diag - 1 - mid)), a.B)) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

__global__ void __launch_bounds__(128) merge_split_kernel(MergeArgs a) {
    pdl_enter();
    const u64 tot = a.nx + a.ny, t = u64(blockIdx.x) * 128 + threadIdx.x, d = t * kPlaceChunk;
    if (d < tot + kPlaceChunk) a.split[t] = u32(merge_split(a, d < tot ? d : tot));
}

__global__ void __launch_bounds__(256) merge_runs_kernel(MergeArgs a) {
    pdl_enter();
    extern __shared__ __align__(16) unsigned char msm[];
    Cell* const stage = reinterpret_cast<Cell*>(msm);            // x's part, then y's
    u64* const sk = reinterpret_cast<u64*>(stage + kPlaceChunk);  // their sort keys
    unsigned short* const from = reinterpret_cast<unsigned short*>(sk + kPlaceChunk);
    const u64 tot = a.nx + a.ny;
    const u64 d0 = u64(blockIdx.x) * kPlaceChunk, d1 = d0 + kPlaceChunk < tot ? d0 + kPlaceChunk : tot;
    const u64 x0 = a.split[blockIdx.x], y0 = d0 - x0;
    const u32 nx = u32(a.split[blockIdx.x + 1] - x0), m = u32(d1 - d0), ny = m - nx;
#pragma unroll
    for (int q = 0; q < kPlaceItems; ++q) {
        const u32 j = u32(q) * 256 + threadIdx.x;
        if (j < m) {
            Cell cl;
            ld_cell_cg(j < nx ? a.x + x0 + j : a.y + y0 + (j - nx), cl.key, cl.val);
            stage[j] = cl;
            sk[j] = sort_key(cl.key, a.B);
        }
    }
    __syncthreads();
    // this thread's cells of the tile: split, then a serial merge
    const u32 g0 = threadIdx.x * kPlaceItems < m ? threadIdx.x * kPlaceItems : m;
    u32 lo = g0 > ny ? g0 - ny : 0, hi = g0 < nx ? g0 : nx;
    while (lo < hi) {
        const u32 mid = (lo + hi) / 2;
        if (sk[mid] <= sk[nx + g0 - 1 - mid]) lo = mid + 1;
        else hi = mid;
    }
    u32 i = lo, j = g0 - lo;
#pragma unroll
    for (int q = 0; q < kPlaceItems; ++q) {
        if (g0 + q < m) {
            const bool take_x = j >= ny || (i < nx && sk[i] <= sk[nx + j]);
            from[g0 + q] = (unsigned short)(take_x ? i : nx + j);
            if (take_x) ++i;
            else ++j;
        }
    }
    __syncthreads();
    for (u32 t = threadIdx.x; t < m; t += 256) a.out[d0 + t] = stage[from[t]];
}
}  // namespace

cudaError_t launch_build_merge(const Cell* x, u64 nx, const Cell* y, u64 ny, u32 log2c, void* scratch,
                               const Cell** merged, cudaStream_t s) {
    MergeArgs a;
    a.x = x;
    a.y = y;
    a.nx = nx;
    a.ny = ny;
    a.B = build_sort_bits(log2c);
    a.out = static_cast<Cell*>(scratch);
    constexpr size_t smem = size_t(kPlaceChunk) * (sizeof(Cell) + sizeof(u64) + 2);
    const cudaError_t e = cudaFuncSetAttribute(merge_runs_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
    if (e != cudaSuccess) return e;
    const u64 tot = nx + ny, tiles = (tot + kPlaceChunk - 1) / kPlaceChunk;
    // (the sort's tile prefixes are not used by a merge: 2 KB per 4096 cells)
    a.split = reinterpret_cast<u32*>(static_cast<unsigned char*>(scratch) + Layout(tot).off_tiles);
    launch_overlapped(merge_split_kernel, unsigned((tiles + 1 + 127) / 128), 128, 0, s, a);
    launch_overlapped(merge_runs_kernel, unsigned(tiles), 256, smem, s, a);
    count_launch();
    count_launch();
    *merged = a.out;
    return cudaGetLastError();
}

Cell* build_spare_cells(void* scratch, u64 n) {
    return reinterpret_cast<Cell*>(static_cast<unsigned char*>(scratch) + Layout(n).off_buf1);
}

u64 build_scratch_bytes(u64 n) { return Layout(n).total; }

u64 scan_partials(u64 m) { return (m + kScanChunk - 1) / kScanChunk; }
cudaError_t scan_exclusive_u32(u32* data, u64 m, u32* part, cudaStream_t s) { return scan_exclusive(data, m, part, s); }

cudaError_t launch_build_sort(const u64* keys, const u64* vals, u64 n, u32 log2c, int full_keys, void* scratch,
                              const Cell** sorted, BuildExtra** ex_out, cudaStream_t s) {
    const u32 B = build_sort_bits(log2c);
    const Layout L(n);
    unsigned char* base = static_cast<unsigned char*>(scratch);
    Cell* buf[2] = {reinterpret_cast<Cell*>(base), reinterpret_cast<Cell*>(base + L.off_buf1)};
    BuildExtra* ex = reinterpret_cast<BuildExtra*>(base + L.off_ex);
    u32* counts = reinterpret_cast<u32*>(base + L.off_counts);
    u64* tiles = reinterpret_cast<u64*>(base + L.off_tiles);
    cudaError_t e = cudaMemsetAsync(ex, 0, L.total - L.off_ex, s);  // ex, the counts and the tickets
    if (e == cudaSuccess) e = cudaMemsetAsync(tiles, 0, L.ntiles * kDigits * sizeof(u64), s);
    if (e != cudaSuccess) return e;
    u64 cgrid = u64(sm_count()) * 8;
    if (cgrid > (n + kSortThreads * 8 - 1) / (kSortThreads * 8)) cgrid = (n + kSortThreads * 8 - 1) / (kSortThreads * 8);
    launch_overlapped(radix_count_kernel, unsigned(cgrid), kSortThreads, 0, s, keys, n, B, counts, ex, full_keys);
    count_launch();
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    constexpr size_t smem = pass_smem_bytes();
    for (auto fn : {radix_pass_kernel<true>, radix_pass_kernel<false>}) {
        e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
        if (e != cudaSuccess) return e;
    }
    PassArgs a;
    a.src.cells = nullptr;
    a.src.keys = keys;
    a.src.vals = vals;
    a.n = n;
    a.B = B;
    a.tiles = tiles;
    int cur = 0;
    for (a.pass = 0; a.pass < B / 8; ++a.pass) {
        a.dst = buf[cur];
        a.hist = counts + a.pass * kDigits;
        a.ticket = counts + kMaxPasses * kDigits + a.pass;
        e = launch_overlapped(a.pass == 0 ? radix_pass_kernel<true> : radix_pass_kernel<false>, unsigned(L.ntiles),
                              kPassThreads, smem, s, a);
        count_launch();
        if (e == cudaSuccess) e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        a.src.cells = buf[cur];
        cur ^= 1;
    }
    *sorted = a.src.cells;
    *ex_out = ex;
    return cudaSuccess;
}

cudaError_t launch_build_count(const Cell* sorted, u64 n, u32 log2c, bool dense, void* scratch, BuildExtra* ex,
                               cudaStream_t s) {
    const Layout L(n);
    const PlaceArgs a = place_args(sorted, n, log2c, scratch, ex);
    cudaError_t e = cudaMemsetAsync(a.dirty, 0, L.nchunks, s);
    if (e != cudaSuccess) return e;
    launch_overlapped(build_place_kernel<0>, unsigned(L.nchunks), 256, place_smem_bytes<0>(), s, a);
    // deferred survivor tests (both kernels return at once when there are none)
    launch_overlapped(build_resolve_kernel, unsigned(sm_count() * 4), 256, 0, s, a);
    launch_overlapped(build_place_kernel<1>, unsigned(L.nchunks), 256, place_smem_bytes<1>(), s, a);
    launch_overlapped(build_place_scan_kernel, 1, 256, 0, s, a.parts, L.nchunks, ex,
                      dense && (1ull << log2c) > kMaxDense ? a.longs : nullptr, 1ull << log2c);
    for (int i = 0; i < 4; ++i) count_launch();
    return cudaGetLastError();
}

// New cells are written dense by a batch of at least an eighth of their
// number: whole sectors, empty cells included, so they need not be zeroed
// first (a merge of 2^25 + 2^22 pairs into 2^26 cells: 160 us of zeroing and a
// 313 us write, against one of 310 us).  Below that the ranges of most chunks
// grow past what a CTA should write; the batch's size stands for its
// distinct keys here, and chunks with too few of them are told by their range
// (kMaxDense).  Cells that are zero already take the survivors alone.
bool build_place_dense(u64 n, u32 log2c) { return n >= (1ull << log2c) / 8; }

cudaError_t launch_build_place(const Cell* sorted, u64 n, Cell* cells, u32 log2c, bool dense, void* scratch,
                               BuildExtra* ex, DevState* st, const u64* vals, cudaStream_t s) {
    const Layout L(n);
    PlaceArgs a = place_args(sorted, n, log2c, scratch, ex);
    a.cells = cells;
    a.dense = dense ? 1 : 0;
    cudaError_t e = cudaFuncSetAttribute(build_place_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         int(place_smem_bytes<2>()));
    if (e != cudaSuccess) return e;
    if (dense && (1ull << log2c) > kMaxDense) {
        launch_overlapped(build_zero_kernel, unsigned(sm_count()), 256, 0, s, cells, a.longs, ex);
        count_launch();
    }
    launch_overlapped(build_place_kernel<2>, unsigned(L.nchunks), 256, place_smem_bytes<2>(), s, a);
    launch_overlapped(build_finish_kernel, 1, 32, 0, s, cells, log2c, a.ov, ex, st, vals);
    count_launch();
    count_launch();
    return cudaGetLastError();
}

}  // namespace cht
