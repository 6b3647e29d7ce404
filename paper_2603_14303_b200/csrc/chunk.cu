// sc_chunk: delimiter-bounded chunking (Sec. 2.2, Eq. 1) as a segmented boundary scan.
//
// Per sequence position p: isd[p] = token id in the delimiter set.  A non-delimiter run starts
// at p when p == 0 or isd[p-1]; run_start(p) is the last such position at or before p, and p
// opens a segment iff isd[p] or (p - run_start(p)) % max_chunk_len == 0.  Segment offsets are
// the compacted positions of those flags.
// Two kernels.  chunk_flags: one block per 2048 tokens (per several such tiles where a sequence has more than kMaxSpans of
// them); it finds the run it starts in by looking back for the last delimiter before it, writes the flags as bits and
// counts them.  The first look is at 256 tokens and finds one in ordinary text; further looks take 16 K tokens each, and no
// more than kMaxSpans blocks of a sequence look back, so that text without delimiters costs time proportional to its length.
// chunk_write_pack: one block per sequence turns flags into offsets and packs consecutive segments into the
// <= SC_TILE_ROWS-token work tiles sc_compress consumes.
// What bounds it: launches and dependent round trips, not bytes.  Five kernels before (carry, count, scan, write, pack, with
// token ids read four times and the tile chain walked one tile at a time) took 17.8 us for 2048 tokens, 40 us for 32K,
// 30 us for 16 x 16K; these take 8.2, 12.1 and 10.5 us (back to back in a CUDA graph).  Without a delimiter in the text: 14 us for
// 32K, 31 for 128K, 196 for 1M (226 with delimiters); 55, 204 and 1877 when every look took 256 tokens.
#include "common.cuh"

namespace sc {

constexpr int kChunkThreads = 256;
constexpr int kChunkPer = 8;
constexpr int kChunkTile = kChunkThreads * kChunkPer;  // 2048 tokens per block
constexpr int kMaxSpans = 128;                         // blocks of a sequence (each may look back to its start)
constexpr int kLookUnroll = 32, kLookRounds = 2;       // tokens per thread of a further look: 64
constexpr int kPackThreads = 1024;
constexpr int kPackWindow = 4096;                      // segments packed at a time
constexpr int kPackJump = 8;                           // tiles per step of the chain walk

struct DelimSet {
    int32_t id[SC_MAX_DELIMS];
    int32_t n;
};

__device__ __forceinline__ bool in_set(int32_t tok, const DelimSet& D) {
    bool hit = false;
    for (int i = 0; i < D.n; ++i) hit |= (D.id[i] == tok);
    return hit;
}

// Maximum of one int per thread over the block, 256 threads.
__device__ __forceinline__ int block_max(int v, int* wt /*[8]*/) {
    v = warp_max_i(v);
    if ((threadIdx.x & 31) == 0) wt[threadIdx.x >> 5] = v;
    __syncthreads();
    int r = wt[0];
#pragma unroll
    for (int i = 1; i < kChunkThreads / 32; ++i) r = max(r, wt[i]);
    __syncthreads();
    return r;
}

// Last delimiter among tokens [lo, hi), as its position + 1, or 0; all threads of the block get the answer.
__device__ __noinline__ int last_delimiter(const int32_t* ids, int lo, int hi, const DelimSet& D, int* wt) {
    int last = 0;
    for (int p0 = lo + threadIdx.x; p0 < hi; p0 += kLookUnroll * kChunkThreads) {
        int32_t tok[kLookUnroll];   // requested together
#pragma unroll
        for (int i = 0; i < kLookUnroll; ++i) tok[i] = ids[min(p0 + i * kChunkThreads, hi - 1)];
        unsigned hits = 0u;
        for (int k = 0; k < D.n; ++k) {   // (one delimiter against all tokens: the other way round every comparison waits for its id)
            const int32_t id = D.id[k];
#pragma unroll
            for (int i = 0; i < kLookUnroll; ++i) hits |= (tok[i] == id ? 1u : 0u) << i;
        }
        if (hits) last = min(p0 + (31 - __clz(hits)) * kChunkThreads, hi - 1) + 1;
    }
    return block_max(last, wt);
}

// Kernel 1: segment-start flags of `span` tiles of 2048 tokens (a byte per thread and tile, bit i = token i of its eight)
// and their number per tile.  kOne: span is 1 (the loop costs 0.4 us of 12).
template <bool kOne>
__global__ void __launch_bounds__(kChunkThreads)
chunk_flags(const int32_t* __restrict__ token_ids, int n, int tps, int span, const __grid_constant__ DelimSet D, int max_len, uint8_t* __restrict__ flags,
            int32_t* __restrict__ tile_cnt) {
    __shared__ int wt[kChunkThreads / 32];
    in_stream_order();
    if (kOne) span = 1;
    const int spans = kOne ? tps : (tps + span - 1) / span;
    const int b = blockIdx.x / spans, first = (blockIdx.x - b * spans) * span, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int32_t* ids = token_ids + (int64_t)b * n;
    // start of the run that reaches into the first tile: behind the last delimiter before it
    int carry = 0;
    if (D.n > 0 && first > 0) {
        int hi = first * kChunkTile;
        const int p = hi - 1 - (int)threadIdx.x;
        carry = block_max(in_set(ids[p], D) ? p + 1 : 0, wt);
        hi -= kChunkThreads;
        while (carry == 0 && hi > 0) {
            const int lo = max(hi - kLookUnroll * kLookRounds * kChunkThreads, 0);
            carry = last_delimiter(ids, lo, hi, D, wt);
            hi = lo;
        }
    }
    for (int tile = first; kOne ? tile == first : tile < min(first + span, tps); ++tile) {
        const int p0 = tile * kChunkTile + threadIdx.x * kChunkPer;
        int32_t tok[kChunkPer];
        if (p0 + kChunkPer <= n && (reinterpret_cast<uintptr_t>(ids + p0) & 15u) == 0) {
            const int4 x = *reinterpret_cast<const int4*>(ids + p0), y = *reinterpret_cast<const int4*>(ids + p0 + 4);
            tok[0] = x.x; tok[1] = x.y; tok[2] = x.z; tok[3] = x.w; tok[4] = y.x; tok[5] = y.y; tok[6] = y.z; tok[7] = y.w;
        } else {
#pragma unroll
            for (int i = 0; i < kChunkPer; ++i) tok[i] = p0 + i < n ? ids[p0 + i] : 0;
        }
        const int32_t prev_tok = p0 > 0 && p0 - 1 < n ? ids[p0 - 1] : 0;
        unsigned isd = 0u;
#pragma unroll
        for (int i = 0; i < kChunkPer; ++i)
            if (p0 + i < n && in_set(tok[i], D)) isd |= 1u << i;
        // run starts among this thread's tokens; the last one carries over to the threads behind it
        unsigned starts = (isd << 1) & 0xffu;
        if (p0 == 0 || (p0 < n && in_set(prev_tok, D))) starts |= 1u;
        int last = starts ? p0 + 31 - __clz(starts) : -1;
        int incl = warp_scan_max(last, lane);
        if (lane == 31) wt[w] = incl;
        __syncthreads();
        int run = __shfl_up_sync(kFull, incl, 1);
        if (lane == 0) run = -1;
        run = max(run, carry);
        for (int i = 0; i < (kOne ? w : kChunkThreads / 32); ++i) {
            if (kOne || i < w) run = max(run, wt[i]);
            carry = max(carry, wt[i]);   // for the next tile
        }
        unsigned f = 0u;
#pragma unroll
        for (int i = 0; i < kChunkPer; ++i) {
            const int p = p0 + i;
            if ((starts >> i) & 1u) run = p;
            const int off = p - run;
            if (p < n && (((isd >> i) & 1u) || off == 0 || (off >= max_len && off % max_len == 0))) f |= 1u << i;
        }
        flags[((size_t)b * tps + tile) * kChunkThreads + threadIdx.x] = (uint8_t)f;
        __syncthreads();   // wt is read above
        const int c = warp_sum_i(__popc(f));
        if (lane == 0) wt[w] = c;
        __syncthreads();
        if (threadIdx.x == 0) {
            int t = 0;
#pragma unroll
            for (int i = 0; i < kChunkThreads / 32; ++i) t += wt[i];
            tile_cnt[b * tps + tile] = t;
        }
        if (!kOne) __syncthreads();   // wt is written again
    }
}

// Inclusive scan of one int per thread over 1024 threads; *total = the sum.
__device__ __forceinline__ int block_scan(int v, int* wt /*[32]*/, int* total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int s = warp_scan_add(v, lane);
    if (lane == 31) wt[w] = s;
    __syncthreads();
    const int t = warp_scan_add(wt[lane], lane);   // every warp scans the 32 totals
    *total = __shfl_sync(kFull, t, 31);
    const int before = __shfl_sync(kFull, t, max(w - 1, 0));
    __syncthreads();
    return s + (w > 0 ? before : 0);
}

// Kernel 2: one block per sequence.  Offsets from the flags; then the work tiles: as many whole segments as fit in
// SC_TILE_ROWS tokens, or one longer segment alone.  The chain tile -> next tile is sequential, but where a tile that
// starts at segment s ends does not depend on the chain: for a window of segments in shared memory every thread finds
// the end of the tile that would start at its segments (a binary search over the monotone offsets), the table is
// composed with itself three times, one thread walks the chain eight tiles per lookup, and the tiles between are
// filled in by all.
__global__ void __launch_bounds__(kPackThreads)
chunk_write_pack(const uint8_t* __restrict__ flags, const int32_t* __restrict__ tile_cnt, int B, int n, int tps,
                 int32_t* __restrict__ seg_off, int n_seg_cap, int32_t* __restrict__ seq_seg_off, int32_t* __restrict__ n_seg,
                 int32_t* __restrict__ tile_seg, int n_tile_cap, int32_t* __restrict__ seq_tile_cnt, int32_t* status) {
    __shared__ int buf[kPackWindow + 1];
    __shared__ uint16_t nxt[kPackWindow + 1], ja[kPackWindow + 1], jb[kPackWindow + 1];   // next tile's segment; jumps
    __shared__ uint16_t chain[kPackWindow / kPackJump + 2];
    __shared__ int wt[32];
    __shared__ int sh_cur, sh_nodes, sh_steps;
    const int b = blockIdx.x, tid = threadIdx.x;
    in_stream_order();
    // segments of the sequences before this one, and of this one
    int before = 0, own = 0, s0, cnt_b;
    for (int i = tid; i < b * tps; i += kPackThreads) before += tile_cnt[i];
    for (int i = tid; i < tps; i += kPackThreads) own += tile_cnt[b * tps + i];
    block_scan(before, wt, &s0);
    block_scan(own, wt, &cnt_b);
    if (tid == 0) {
        seq_seg_off[b] = s0;
        if (b == B - 1) {
            const int total = s0 + cnt_b;
            seq_seg_off[B] = total;
            *n_seg = total;
            if (total > n_seg_cap) set_status(status, SC_ERR_CAPACITY);
            else seg_off[total] = B * n;
        }
    }
    const uint32_t* words = reinterpret_cast<const uint32_t*>(flags + (size_t)b * tps * kChunkThreads);
    const int n_words = (n + 31) >> 5;
    int done = 0;   // segments written
    for (int w0 = 0; w0 < n_words; w0 += kPackThreads) {
        const int wi = w0 + tid;
        uint32_t f = wi < n_words ? words[wi] : 0u;
        int total;
        int rank = done + block_scan(__popc(f), wt, &total) - __popc(f);
        while (f) {
            const int off = b * n + wi * 32 + __ffs(f) - 1;
            f &= f - 1;
            if (s0 + rank < n_seg_cap) seg_off[s0 + rank] = off;
            if (rank <= kPackWindow) buf[rank] = off;   // the first window of the packing
            ++rank;
        }
        done += total;
    }
    __syncthreads();
    const int s1 = min(s0 + cnt_b, n_seg_cap);   // clamped when the offsets overflowed
    int32_t* out = tile_seg + (int64_t)b * (n_tile_cap + 1);
    int cur = s0, nt = 0;
    while (cur < s1) {
        const int ws = cur, cnt = min(kPackWindow, s1 - ws);
        const bool last_window = ws + cnt == s1;
        if (ws != s0) for (int i = tid; i < cnt; i += kPackThreads) buf[i] = seg_off[ws + i];
        if (tid == 0 && (ws != s0 || ws + cnt == s0 + cnt_b)) buf[cnt] = last_window ? (b + 1) * n : seg_off[ws + cnt];
        __syncthreads();
        // a tile's end is known for sure only if SC_TILE_ROWS + 1 offsets behind its start are in the window
        const int lim = last_window ? cnt : cnt - SC_TILE_ROWS;
        for (int i = tid; i <= cnt; i += kPackThreads) {
            int lo = i;   // not known (or the end): the chain stops here
            if (i < lim) {
                // largest e in (i, cnt] with buf[e] - buf[i] <= SC_TILE_ROWS, or i + 1 for a segment longer than a tile
                const int limit = buf[i] + SC_TILE_ROWS;
                int hi = min(cnt, i + SC_TILE_ROWS);   // a segment holds at least one token
                lo = i + 1;
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (buf[mid] <= limit) lo = mid; else hi = mid - 1;
                }
            }
            nxt[i] = (uint16_t)lo;
        }
        __syncthreads();
        for (int i = tid; i <= cnt; i += kPackThreads) ja[i] = nxt[nxt[i]];
        __syncthreads();
        for (int i = tid; i <= cnt; i += kPackThreads) jb[i] = ja[ja[i]];
        __syncthreads();
        for (int i = tid; i <= cnt; i += kPackThreads) ja[i] = jb[jb[i]];
        __syncthreads();
        if (tid == 0) {
            int x = 0, k = 0;
            while (x < lim) { chain[k++] = (uint16_t)x; x = ja[x]; }
            sh_cur = ws + x; sh_nodes = k;
        }
        __syncthreads();
        const int nodes = sh_nodes;
        int steps = 0;
        for (int k = tid; k < nodes; k += kPackThreads) {   // (at most one node per thread: a step passes kPackJump segments)
            int x = chain[k];
            for (steps = 0; steps < kPackJump && x < lim; ++steps) {
                const int t = nt + k * kPackJump + steps;
                if (t < n_tile_cap) out[t] = ws + x;
                x = nxt[x];
            }
            if (k == nodes - 1) sh_steps = steps;
        }
        cur = sh_cur;
        __syncthreads();
        nt += (nodes - 1) * kPackJump + sh_steps;
    }
    if (tid == 0) {
        out[min(nt, n_tile_cap)] = s1;
        seq_tile_cnt[b] = nt;
        if (nt > n_tile_cap) set_status(status, SC_ERR_CAPACITY);
    }
}

size_t chunk_ws_bytes(int32_t B, int32_t n) {
    const size_t tiles = (size_t)B * div_up(n, kChunkTile);
    return tiles * (kChunkThreads + sizeof(int32_t)) + 64;
}

cudaError_t launch_chunk(const ChunkArgs& a, cudaStream_t st) {
    const int tps = div_up(a.n, kChunkTile);
    const int tiles = a.B * tps;
    int32_t* tile_cnt = a.ws;
    uint8_t* flags = reinterpret_cast<uint8_t*>(a.ws + (tiles + 15) / 16 * 16);   // (64 spare bytes cover the padding)
    DelimSet D;
    D.n = a.n_delim;
    for (int i = 0; i < SC_MAX_DELIMS; ++i) D.id[i] = (i < a.n_delim) ? a.delim[i] : 0;
    const int span = div_up(tps, kMaxSpans), spans = div_up(tps, span);
    cudaError_t e = launch_in_order(span == 1 ? chunk_flags<true> : chunk_flags<false>, dim3(a.B * spans), kChunkThreads, 0, st, a.token_ids,
                                    a.n, tps, span, D, a.max_chunk_len, flags, tile_cnt);
    if (e != cudaSuccess) return e;
    note_launches(2);
    return launch_in_order(chunk_write_pack, dim3(a.B), kPackThreads, 0, st, (const uint8_t*)flags, (const int32_t*)tile_cnt, a.B, a.n, tps,
                                 a.seg_off, a.n_seg_cap, a.seq_seg_off, a.n_seg, a.tile_seg, a.n_tile_cap, a.seq_tile_cnt, a.status);
}

}  // namespace sc
