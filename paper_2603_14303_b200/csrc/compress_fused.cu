// Fused bf16 compress kernel (d = 128), sm_100a: Eq. 2 + Algorithm 1 + Eq. 3 in one pass over K, V.
//
// Persistent blocks (three per SM) draw work tiles from a global ticket counter.  A tile is a run of whole segments of
// at most SC_TILE_ROWS tokens of one (layer, sequence, KV head) -- K and V both staged in shared memory -- or one longer
// segment alone (K staged, then V in its place).  A block has four compute warps and a service warp; they meet
// through mbarriers only.  The service warp stages a tile as soon as the buffer is free, looks back for the tile's output
// offset, publishes the tile's prefix and draws the next ticket while the tile is pooled.
// Compute warps, per tile:
//   1. similarities (Eq. 2): the Gram matrix of the tile's keys is one 128 x 128 x 128 tcgen05.mma product in tensor
//      memory (the 128-byte-swizzled layout the TMA boxes wrote is the K-major operand layout; three such products, one
//      after the other, for a tile of 129..256 tokens).  Thread i owns row i; it reads only the columns its warp's rows
//      can need and keeps, as bits in registers, which EARLIER tokens of its segment it is similar to (Sim > tau decided as
//      |k_c| (tau |k_i|) - G < 0: half an instruction of two fmas and one funnel shift that collects its sign per pair).
//   2. Algorithm 1 for all rows at once, in rounds: a row with an earlier neighbour that is a seed is a member, a row
//      whose earlier neighbours are all members is a seed.  Both facts are final once true, the lowest open row is
//      decided in every round, so the rounds end and give exactly the sequential pass's partition; chunks that are unions
//      of cliques take two.  A member joins the earliest seed among its earlier neighbours.  The tile's cluster count is
//      published at once; every token's cluster number (rank of its seed) goes to shared memory.
//   3. Eq. 3: the members' sum of a cluster is a row of M V, M the 0/1 matrix clusters x tokens; M's fragments are made
//      from the cluster numbers (kept as bf16: comparing two of them gives the 1.0 or 0.0 the product wants), K and V come
//      transposed from their staged rows (ldmatrix.trans), mma.m16n8k16 adds up in fp32 (products with 1 and 0 are exact).
//      Sixteen clusters of more than one token at a time, over the tokens from their first seed to the end of their last
//      segment only; each warp takes a quarter of the columns.  Sums are scaled by 1/|S|, rounded once and stored.  Clusters
//      of one token are copied bit for bit; a sum that is not finite (0 * inf would reach other clusters) sends the sixteen
//      clusters to a loop over their members.
//
// What bounds it: the latency of a tile's serial steps, three tiles to an SM; an instruction of a warp takes 6 clocks (issue slots
// 36 % used, tensor pipe 27 %, shared memory about half), so chains of dependent instructions count: four shift chains
// instead of one in sim_word, four in the check of the sums and steps 1 and 2 of a short tile in line took 8 layers x 8 heads x 32K tokens
// from 303 to 291 us (one launch per layer 117 -> 110 for two, chunks of 8 tokens 345 -> 333, of 128 508 -> 485).  Nothing may spill:
// shared memory leaves the L1 cache 28 KB, a spilled word is a trip to L2, and variants with 4 to 80 bytes of stack lost 5 to 10 %.
// Copies of an earlier form with steps left out, 32 layers on resident inputs, 1105 us: 707 (loads only), 834 (loads, steps 1 and 2), 1025
// (all but the stores of the means).
// A tile of 129..256 tokens holds up the look-back of the tiles behind it with its three products.  In short inputs, whose time is one such
// tile's, steps 1 and 2 of the short tiles in line cost 0.3 to 0.6 us (8 heads x 512 tokens with chunks over 128: 12.8 us with those
// steps out of line, 13.5); 32 layers x 32K tokens gain 26 us by them, 4 x 64K in chunks of 128 23 of 547.
// Why these steps: one product per tile and decision rounds take 6.5 K warp instructions per 128 tokens, a warp per segment with
// mma.sync tiles, the greedy pass and sums of member rows on the CUDA cores took 13 K: 32 layers 1395 us; 16 sequences x 16K,
// lognormal chunks, 500 us a layer against 300; 4 x 64K in chunks of 128 794 against 578.  Sums over member rows in cluster
// order in place of the product: 1245 us.
//
// Offsets: a prefix sum over the tiles of each head by decoupled look-back over per-tile status words; tickets are handed
// out in order, so every predecessor is held by a running block and the bounded wait cannot starve.  A block draws its
// next ticket only when its tile's count is out and its offset known: drawn one tile earlier, a tile waits unstarted in a
// block that itself waits, and holds up its successors (16 x 16K, two layers 666 us against 711; chunks of 128 tokens 781
// against 884).  Tickets go round the (layer, sequence, head) units.  The last block to finish zeroes the
// status words and counters, so a workspace that was zero before the call is zero again after it.  One launch may
// serve several layers (sc_compress_layers).
#include <cuda.h>

#include <mutex>

#include "common.cuh"
#include "umma.cuh"

namespace sc {

namespace cf {

constexpr int kWarps = 4;                         // compute warps
constexpr int kThreads = (kWarps + 1) * 32;       // plus one service warp
constexpr int kTeam = kWarps * 32;
constexpr int kD = 128;
constexpr int kHalfRow = 128;                     // a staged row is two 128-byte halves (64 columns each), see tile_addr
constexpr int kBoxRows = 32;                      // rows per TMA box
constexpr int kBoxBytes = kBoxRows * kHalfRow;    // 4096
constexpr int kMaxRows = SC_MAX_CHUNK_LEN;        // 256: a long tile
constexpr int kShortRows = SC_TILE_ROWS;          // 128
constexpr int kHalfShort = kShortRows * kHalfRow; // 16384: distance between the column halves of a short tile
constexpr int kHalfLong = kMaxRows * kHalfRow;    // 32768: ... of a long one
constexpr int kVOff = 2 * kHalfShort;             // short: K | V, long = one tensor
constexpr int kNormOff = 2 * kHalfLong;           // float[256]: norms of the tile's rows
constexpr int kRankOff = kNormOff + kMaxRows * 4;            // bf16[256]: cluster of each token (whole numbers to 256 are exact), see rank_slot
constexpr int kCntOff = kRankOff + kMaxRows * 2;             // int32[256]: tokens of each cluster
constexpr int kSeedOff = kCntOff + kMaxRows * 4;             // uint8[256]: the cluster's seed
constexpr int kListOff = kSeedOff + kMaxRows;                // uint8[256]: the clusters of more than one token, in order
constexpr int kEndOff = kListOff + kMaxRows;                 // uint16[256]: end of the seed's segment
constexpr int kMiscOff = kEndOff + kMaxRows * 2;             // seeds[8], members[8]; starts[2][4]; geo[2][8]; base, P, tmem slot, flags
constexpr int kBarOff = kMiscOff + 64 + 32 + 64 + 32;
constexpr int kSmemBytes = kBarOff + 64;
constexpr int kTmemCols = 128;                    // one 128 x 128 fp32 accumulator per block (three blocks per SM: 384 of 512 columns)
constexpr int kBlocksPerSm = 3;
static_assert(kRankOff % 16 == 0 && kCntOff % 16 == 0 && kMiscOff % 16 == 0 && kBarOff % 8 == 0, "alignment");
static_assert(kSmemBytes <= 76800, "three blocks per SM need <= 75 KB each");

enum Mode { kCountOnly = 0, kLookBack = 1 };
enum Geo { gB = 0, gH = 1, gT = 2, gNseg = 3, gRow0 = 4, gR = 5, gLast = 6, gLayer = 7 };   // gT = -1: no work left

constexpr uint32_t kFlagAggregate = 1u << 30, kFlagPrefix = 2u << 30, kValueMask = (1u << 30) - 1;
constexpr unsigned long long kWaitLimitNs = 2000000000ull;   // every wait gives up after 2 s
// The look-back reads 64 predecessors per poll (4 and 8 groups measured slower, 1 slower on short chunks).
constexpr int kPollGroups = 2;
constexpr int kCtlWords = 64;                                // ticket, done counter, padding

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
// One TMA box: 32 rows x 64 columns of a [B, Hkv, n, 128] tensor, 128-byte swizzled, no multicast.
__device__ __forceinline__ void tma_box(uint32_t dst, const CUtensorMap* map, int col, int row, int h, int b, uint32_t bar) {
    asm volatile("cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];\n"
                 ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(col), "r"(row), "r"(h), "r"(b), "r"(bar) : "memory");
}
// Byte offset, inside one column half of the staged keys, of 16-byte chunk `chunk` (0..7) of row
// `row`: rows are 128 bytes apart and the chunk index is XORed with the row's low three bits (the
// TMA 128-byte swizzle), which makes ldmatrix over eight consecutive rows conflict free.
__device__ __forceinline__ uint32_t tile_addr(int row, int chunk) { return row * kHalfRow + ((chunk ^ (row & 7)) << 4); }
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// Bits of word `word` at or above position `lo` (any position of the tile); no branch.
__device__ __forceinline__ uint32_t bits_from(int lo, int word) {
    uint32_t m;
    asm("shl.b32 %0, %1, %2;\n" : "=r"(m) : "r"(0xffffffffu), "r"(max(lo - word * 32, 0)));   // (shl gives 0 for 32 and more)
    return m;
}
__device__ __forceinline__ uint32_t ld_volatile(const uint32_t* p) {
    uint32_t v;
    asm volatile("ld.volatile.global.u32 %0, [%1];\n" : "=r"(v) : "l"(p) : "memory");
    return v;
}
// The four compute warps meet ...
__device__ __forceinline__ void team_sync() { asm volatile("barrier.cta.sync 1, 128;\n" ::: "memory"); }
// ... and learn whether any of them says so.
__device__ __forceinline__ bool team_any(bool mine) {
    uint32_t out;
    asm volatile(
        "{\n"
        ".reg .pred p, r;\n"
        "setp.ne.u32 p, %1, 0;\n"
        "barrier.cta.red.or.pred r, 1, 128, p;\n"
        "selp.u32 %0, 1, 0, r;\n"
        "}\n"
        : "=r"(out) : "r"(mine ? 1u : 0u) : "memory");
    return out != 0u;
}

// One 128 x 128 block of -K.K^T of the staged keys (the product negates its first operand, so that sim_word adds pairs of
// accumulators to its products: the two-at-a-time fma takes no negated operand): rows of 128-row block mb against rows of block nb (column halves `hs` bytes
// apart).  One thread issues the eight instructions; the mbarrier gets one arrival when they are complete.
__device__ __forceinline__ void umma_gram_block(uint32_t kbase, int hs, int mb, int nb, uint32_t tmem, uint32_t bar) {
    constexpr uint32_t idesc = umma::instr_desc_bf16(128, 128, false, false, true);
#pragma unroll
    for (int ks = 0; ks < 8; ++ks) {
        const uint32_t off = (ks >> 2) * hs + (ks & 3) * 32;
        umma::mma_bf16_ss(tmem, umma::smem_desc_sw128(kbase + mb * 128 * kHalfRow + off, 16, 1024),
                          umma::smem_desc_sw128(kbase + nb * 128 * kHalfRow + off, 16, 1024), idesc, ks > 0);
    }
    umma::mma_commit(bar);
}

// Bits over 32 columns: bit c = (thr_c - G_c < 0), thr_c = norm_c * tni; g holds -G.  The sign of each difference is shifted in
// behind the others, from the last column of a byte to the first; a difference of zero (Sim == tau) and one that is not a
// number give no bit.  Two differences per instruction: 4 x 64K in chunks of 128, two layers, 553 -> 521 us (chunks of 20: the same).
__device__ __forceinline__ uint32_t sim_word(const uint32_t (&g)[32], const float* norm_c, float tni1) {
    const float2 tni = make_float2(tni1, tni1);
    uint32_t w[4] = {0u, 0u, 0u, 0u};   // a byte each: four chains of eight shifts side by side
    const float4* nc = reinterpret_cast<const float4*>(norm_c);
#pragma unroll
    for (int half = 1; half >= 0; --half)
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            const float4 nv = nc[2 * x + half];
            const uint32_t* gk = g + x * 8 + half * 4;
            const float2 hi = umma::fma2(make_float2(nv.z, nv.w), tni, make_float2(__uint_as_float(gk[2]), __uint_as_float(gk[3])));
            const float2 lo = umma::fma2(make_float2(nv.x, nv.y), tni, make_float2(__uint_as_float(gk[0]), __uint_as_float(gk[1])));
            w[x] = __funnelshift_l(__float_as_uint(hi.y), w[x], 1);
            w[x] = __funnelshift_l(__float_as_uint(hi.x), w[x], 1);
            w[x] = __funnelshift_l(__float_as_uint(lo.y), w[x], 1);
            w[x] = __funnelshift_l(__float_as_uint(lo.x), w[x], 1);
        }
    return __byte_perm(__byte_perm(w[0], w[1], 0x0040), __byte_perm(w[2], w[3], 0x0040), 0x5410);
}
// A negative threshold: a zero-norm key has Sim = 0 > tau.
__device__ __forceinline__ uint32_t sim_word_neg(const uint32_t (&g)[32], const float* norm_c, float tni) {
    uint32_t w = 0u;
#pragma unroll
    for (int k = 0; k < 32; ++k) {
        const float thr = norm_c[k] * tni;
        w |= (-__uint_as_float(g[k]) > thr || thr == 0.f ? 1u : 0u) << k;
    }
    return w;
}

// Algorithm 1 for the tile, given each row's earlier-neighbour words (rows tid + 128 r, r < NR, tile word warp + 4 r), and what
// the pooling needs: every token's cluster, and every cluster's size, seed and end of segment.  `end`: end of the rows'
// segments.  Returns the number of clusters.  All compute threads call it.
__device__ __forceinline__ int rank_slot(int i) {   // where a token's cluster number is kept: the four a lane needs for one mma
    return (i & ~15) | ((i & 6) << 1) | ((i & 8) >> 2) | (i & 1);   // fragment (2t, 2t+1, 2t+8, 2t+9 of sixteen) are together
}
template <int NR>
__device__ __forceinline__ int settle_rows(const uint32_t (&e)[NR][4 * NR], const bool (&act)[NR], const int (&end)[NR], unsigned char* smem,
                                           int warp, int lane, int32_t* as, int row0, uint32_t* publish, int* sh_p) {
    constexpr int NW = 4 * NR;
    uint32_t* seeds = reinterpret_cast<uint32_t*>(smem + kMiscOff);
    uint32_t* members = seeds + 8;
    int* cnt = reinterpret_cast<int*>(smem + kCntOff);
    bool open[NR], is_seed[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) { open[r] = act[r]; is_seed[r] = false; cnt[(warp + 4 * r) * 32 + lane] = 0; }
    uint32_t sd[NW], mb[NW];   // all lanes hold the same words
    bool more;
    // round 0 needs no words: a row without earlier neighbours is a seed
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        uint32_t any = 0u;
#pragma unroll
        for (int w = 0; w < NW; ++w) any |= e[r][w];
        if (act[r] && any == 0u) { is_seed[r] = true; open[r] = false; }
        const uint32_t ns = __ballot_sync(kFull, is_seed[r]);
        if (lane == 0) { seeds[warp + 4 * r] = ns; members[warp + 4 * r] = 0u; }
    }
    team_sync();
    for (;;) {   // the lowest open row is decided every round
#pragma unroll
        for (int w = 0; w < NW; w += 4) {
            const uint4 a = *reinterpret_cast<const uint4*>(seeds + w), b = *reinterpret_cast<const uint4*>(members + w);
            sd[w] = a.x; sd[w + 1] = a.y; sd[w + 2] = a.z; sd[w + 3] = a.w;
            mb[w] = b.x; mb[w + 1] = b.y; mb[w + 2] = b.z; mb[w + 3] = b.w;
        }
        more = false;
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            uint32_t near_seed = 0u, not_member = 0u;
#pragma unroll
            for (int w = 0; w < NW; ++w) { near_seed |= e[r][w] & sd[w]; not_member |= e[r][w] & ~mb[w]; }
            const bool to_member = open[r] && near_seed != 0u;
            const bool to_seed = open[r] && near_seed == 0u && not_member == 0u;
            if (to_member || to_seed) open[r] = false;
            if (to_seed) is_seed[r] = true;
            const uint32_t nm = __ballot_sync(kFull, to_member), ns = __ballot_sync(kFull, to_seed);
            if (lane == 0) {   // only this warp writes its words
                if (nm) members[warp + 4 * r] |= nm;
                if (ns) seeds[warp + 4 * r] |= ns;
            }
            more |= open[r];
        }
        if (!team_any(more)) break;
    }
#pragma unroll
    for (int w = 0; w < NW; w += 4) {
        const uint4 a = *reinterpret_cast<const uint4*>(seeds + w);
        sd[w] = a.x; sd[w + 1] = a.y; sd[w + 2] = a.z; sd[w + 3] = a.w;
    }
    int P = 0;
#pragma unroll
    for (int w = 0; w < NW; ++w) P += __popc(sd[w]);
    if (threadIdx.x == 0) {
        *sh_p = P;
        if (publish) atomicExch(publish, kFlagAggregate | (uint32_t)P);
    }
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        // a member joins the earliest seed among its earlier neighbours; a cluster's number is the rank of its seed
        const int i = (warp + 4 * r) * 32 + lane;
        uint32_t m = 0u, in = 0u;   // the word that holds the seed: candidates, all seeds of the word
        int at = 0, before = 0, upto = 0;
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            const uint32_t mw = is_seed[r] ? (w == warp + 4 * r ? 1u << lane : 0u) : e[r][w] & sd[w];
            const bool take = m == 0u && mw != 0u;
            m = take ? mw : m; in = take ? sd[w] : in; at = take ? w * 32 : at; upto = take ? before : upto;
            before += __popc(sd[w]);
        }
        const int bit = __ffs(m) - 1, s = at + bit, rank = upto + __popc(in & ((1u << (bit & 31)) - 1u));
        reinterpret_cast<__nv_bfloat16*>(smem + kRankOff)[rank_slot(i)] = __int2bfloat16_rn(act[r] ? rank : -1);   // -1: past the tile's end, no cluster
        if (act[r]) {
            atomicAdd(&cnt[rank], 1);
            if (is_seed[r]) {
                (smem + kSeedOff)[rank] = (uint8_t)i;
                reinterpret_cast<uint16_t*>(smem + kEndOff)[rank] = (uint16_t)end[r];
            }
            if (as) as[i] = row0 + s;
        }
    }
    team_sync();
    return P;
}

// The diagonal of a diagonal block = squared norms, negated (a key without length: zero of either sign): thread (warp q, lane) owns row 32 q + lane of the block.  `g` holds the
// 32 columns of the warp's own rows; this lane's element is picked by the bits of the lane number.
__device__ __forceinline__ float diagonal(const uint32_t (&g)[32], int lane) {
    uint32_t t[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) t[k] = (lane & 16) ? g[k + 16] : g[k];
#pragma unroll
    for (int k = 0; k < 8; ++k) t[k] = (lane & 8) ? t[k + 8] : t[k];
#pragma unroll
    for (int k = 0; k < 4; ++k) t[k] = (lane & 4) ? t[k + 4] : t[k];
    t[0] = (lane & 2) ? t[2] : t[0]; t[1] = (lane & 2) ? t[3] : t[1];
    return __uint_as_float((lane & 1) ? t[1] : t[0]);
}

// Steps 1 and 2 for a tile of up to 128 rows, thread i = row i (the product of its keys is complete).  `starts`: bit words of the
// rows that start a segment.
template <bool kAnyTau>
__device__ __forceinline__ int settle_short_tile(unsigned char* smem, const uint32_t* starts, int R, uint32_t tmem, uint32_t phase_u, float tau,
                                                 bool wait_failed, int32_t* as, int row0, uint32_t* publish, int* sh_p) {
    float* norm = reinterpret_cast<float*>(smem + kNormOff);
    const int i = threadIdx.x, lane = i & 31, q = i >> 5;
    const uint32_t lane_addr = tmem + ((uint32_t)(q * 32) << 16);
    // the segment [beg, end) of the row: the nearest start at or before it, and the next one
    int beg, end;
    {
        const uint4 sv = *reinterpret_cast<const uint4*>(starts);
        const uint32_t st[4] = {sv.x, sv.y, sv.z, sv.w};
        int last = 0, next = R;       // outside the warp's word
        uint32_t own = 0u;
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            if (w == q) own = st[w];
            if (w < q && st[w] != 0u) last = w * 32 + 31 - __clz(st[w]);
            if (3 - w > q && st[3 - w] != 0u) next = (3 - w) * 32 + __ffs(st[3 - w]) - 1;
        }
        const uint32_t upto = own & (0xffffffffu >> (31 - lane)), later = own & ~(0xffffffffu >> (31 - lane));
        beg = upto ? q * 32 + 31 - __clz(upto) : last;
        end = min(later ? q * 32 + __ffs(later) - 1 : next, R);
    }
    wait_failed = wait_failed || !umma::mbar_wait(smem_u32(smem) + kBarOff + 16, phase_u);
    __syncwarp();
    umma::fence_after_sync();
    uint32_t g[32];
    umma::tmem_ld32(lane_addr + q * 32, g);   // the columns of the warp's own rows
    umma::tmem_ld_wait();
    norm[i] = sqrtf(fabsf(diagonal(g, lane)));
    const bool act[1] = {i < R};
    if (team_any(wait_failed)) return -1;   // (the norms are in place)
    const float tni = tau * norm[i];
    const int w_lo = __reduce_min_sync(kFull, beg >> 5);   // first word any of the warp's rows needs
    uint32_t e[1][4];
#pragma unroll
    for (int c = 3; c >= 0; --c) {
        uint32_t w = 0u;
        if (c >= w_lo && c <= q) {
            if (c != q) {
                umma::tmem_ld32(lane_addr + c * 32, g);
                umma::tmem_ld_wait();
            }
            w = kAnyTau && tau < 0.f ? sim_word_neg(g, norm + c * 32, tni) : sim_word(g, norm + c * 32, tni);
            w &= bits_from(beg, c);
            if (c == q) w &= (1u << lane) - 1u;   // earlier rows only
        }
        e[0][c] = w;
    }
    umma::fence_before_sync();
    const int ends[1] = {end};
    return settle_rows<1>(e, act, ends, smem, q, lane, as, row0, publish, sh_p);
}

// Steps 1 and 2 for a tile of more than 128 rows (one segment): three products, the two diagonal ones first (they give the
// norms), each read before the next overwrites it; thread tid settles rows tid and tid + 128.
template <bool kAnyTau>
__device__ __noinline__ int settle_long_tile(unsigned char* smem, int R, uint32_t tmem, uint32_t phase_u, float tau, bool wait_failed,
                                             int32_t* as, int row0, uint32_t* publish, int* sh_p) {
    float* norm = reinterpret_cast<float*>(smem + kNormOff);
    const uint32_t sbase = smem_u32(smem), bar_u = sbase + kBarOff + 16;
    const int tid = threadIdx.x, lane = tid & 31, q = tid >> 5;
    const uint32_t lane_addr = tmem + ((uint32_t)(q * 32) << 16);
    uint32_t e[2][8], g[32];
#pragma unroll
    for (int w = 0; w < 8; ++w) e[0][w] = e[1][w] = 0u;
#pragma unroll
    for (int ps = 0; ps < 3; ++ps) {   // blocks (0, 0); (1, 1); (1, 0)
        const int mb = ps == 0 ? 0 : 1, nb = ps == 1 ? 1 : 0, i = mb * 128 + tid;
        if (team_any(wait_failed)) return -1;   // (the product before has been read)
        if (tid == 0) {
            umma::fence_after_sync();
            umma_gram_block(sbase, kHalfLong, mb, nb, tmem, bar_u);
        }
        __syncwarp();
        wait_failed = !umma::mbar_wait(bar_u, phase_u);
        phase_u ^= 1u;
        __syncwarp();
        umma::fence_after_sync();
        if (mb == nb) {
            umma::tmem_ld32(lane_addr + q * 32, g);
            umma::tmem_ld_wait();
            norm[i] = sqrtf(fabsf(diagonal(g, lane)));
            if (team_any(wait_failed)) return -1;   // (the norms are in place)
        }
        const float tni = tau * norm[i];
#pragma unroll
        for (int c = 3; c >= 0; --c) {
            if (mb == nb && c > q) continue;   // columns past the warp's rows
            if (mb != nb || c != q) {
                umma::tmem_ld32(lane_addr + c * 32, g);
                umma::tmem_ld_wait();
            }
            const float* nc = norm + nb * 128 + c * 32;
            const uint32_t w = kAnyTau && tau < 0.f ? sim_word_neg(g, nc, tni) : sim_word(g, nc, tni);
            e[mb][nb * 4 + c] = i >= R ? 0u : (mb == nb && c == q) ? w & ((1u << lane) - 1u) : w;   // earlier rows only
        }
        umma::fence_before_sync();
    }
    if (team_any(wait_failed)) return -1;
    const bool act[2] = {true, tid + 128 < R};
    const int ends[2] = {R, R};
    return settle_rows<2>(e, act, ends, smem, q, lane, as, row0, publish, sh_p);
}

// Step 3 for sixteen clusters whose sums are not all finite: each lane one column of the warp's quarter, member by member.
__device__ __noinline__ void pool_by_members(const unsigned char* tensor, int hs, const unsigned char* smem, bool listed, int m,
                                             int n_multi, int t_lo, int t_hi, __nv_bfloat16* dst, int room, int warp, int lane) {
    const int* cnt = reinterpret_cast<const int*>(smem + kCntOff);
    const int col = warp * 32 + lane;
    for (int x = 16 * m; x < min(16 * m + 16, n_multi); ++x) {
        const int c = listed ? (smem + kListOff)[x] : x;
        if (cnt[c] <= 1 || c >= room) continue;
        float sum = 0.f;
        for (int i = t_lo; i < t_hi; ++i)
            if ((int)__bfloat162float(reinterpret_cast<const __nv_bfloat16*>(smem + kRankOff)[rank_slot(i)]) == c)
                sum += __bfloat162float(*reinterpret_cast<const __nv_bfloat16*>(tensor + (col >> 6) * hs + tile_addr(i, (col & 63) >> 3) + (col & 7) * 2));
        dst[(size_t)c * kD + col] = __float2bfloat16_rn(sum * __frcp_rn((float)cnt[c]));
    }
}

// 1 where the halves are equal, else 0 (one instruction: the result is the operand the product wants).
__device__ __forceinline__ uint32_t same_as(__nv_bfloat162 a, __nv_bfloat162 b) {
    const __nv_bfloat162 r = __heq2(a, b);
    return *reinterpret_cast<const uint32_t*>(&r);
}

// Step 3 for the NT tensors staged at smem, smem + kVOff (column halves hs bytes apart): this warp's 32 columns of every cluster
// of more than one token, and the one-token clusters that are its turn.  dst[]: the tile's first core (row 0 of 128
// columns); `room`: cores that fit.
template <int NT>
__device__ __forceinline__ void pool_tile(unsigned char* smem, int hs, int P, __nv_bfloat16* dst_k, __nv_bfloat16* dst_v, int room,
                                          int warp, int lane) {
    const int g = lane >> 2, tig = lane & 3;
    const uint32_t sbase = smem_u32(smem);
    const int* cnt = reinterpret_cast<const int*>(smem + kCntOff);
    const unsigned char* seedrow = smem + kSeedOff;
    const uint16_t* seg_end = reinterpret_cast<const uint16_t*>(smem + kEndOff);
    // ldmatrix.trans: matrix j of four holds tokens 8 (j & 1) .. + 7, columns 8 (j >> 1) .. + 7 of a 16 x 16 block
    const int j = lane >> 3, r8 = lane & 7;
    const uint32_t b_row = sbase + (warp >> 1) * hs + ((j & 1) * 8 + r8) * kHalfRow;
    const uint32_t off0 = (uint32_t)((((warp & 1) * 4 + (j >> 1)) ^ r8) << 4), off1 = (uint32_t)((((warp & 1) * 4 + 2 + (j >> 1)) ^ r8) << 4);
    // the clusters of more than one token, in order (every warp writes the same list)
    unsigned char* list = smem + kListOff;
    int n_multi = NT > 1 ? 0 : P;   // (a long tile has few clusters of one token: all its clusters take part)
    for (int x0 = 0; NT > 1 && x0 < P; x0 += 32) {
        const bool multi = x0 + lane < P && cnt[x0 + lane] > 1;
        const uint32_t mm = __ballot_sync(kFull, multi);
        if (multi) list[n_multi + __popc(mm & ((1u << lane) - 1u))] = (unsigned char)(x0 + lane);
        n_multi += __popc(mm);
    }
    __syncwarp();
    for (int m = 0; m * 16 < n_multi; ++m) {
        const auto at = [&](int x) { x = min(x, n_multi - 1); return NT > 1 ? (int)list[x] : x; };   // (past the end: the last again)
        const int la = at(16 * m + g), lb = at(16 * m + 8 + g);
        const int k_lo = seedrow[at(16 * m)] >> 4, t_hi = seg_end[at(16 * m + 15)], k_hi = (t_hi + 15) >> 4;
        float acc[NT][4][4];
#pragma unroll
        for (int t = 0; t < NT; ++t)
#pragma unroll
            for (int nt = 0; nt < 4; ++nt) acc[t][nt][0] = acc[t][nt][1] = acc[t][nt][2] = acc[t][nt][3] = 0.f;
        const __nv_bfloat162 c0 = __bfloat162bfloat162(__int2bfloat16_rn(la)), c1 = __bfloat162bfloat162(__int2bfloat16_rn(lb));
#pragma unroll 2
        for (int kk = k_lo; kk < k_hi; ++kk) {
            // M's fragment: rows g and g + 8 of the sixteen clusters, tokens 2 tig, +1, +8, +9 of the sixteen
            const uint2 ranks = *reinterpret_cast<const uint2*>(smem + kRankOff + kk * 32 + 8 * tig);
            const __nv_bfloat162 r01 = *reinterpret_cast<const __nv_bfloat162*>(&ranks.x), r89 = *reinterpret_cast<const __nv_bfloat162*>(&ranks.y);
            const uint32_t a0 = same_as(r01, c0), a1 = same_as(r01, c1), a2 = same_as(r89, c0), a3 = same_as(r89, c1);
#pragma unroll
            for (int t = 0; t < NT; ++t) {
                const uint32_t row = b_row + t * kVOff + kk * 16 * kHalfRow;
                uint32_t b0, b1, b2, b3;
                ldmatrix_x4_trans(row + off0, b0, b1, b2, b3);
                mma_bf16(acc[t][0], a0, a1, a2, a3, b0, b1);
                mma_bf16(acc[t][1], a0, a1, a2, a3, b2, b3);
                ldmatrix_x4_trans(row + off1, b0, b1, b2, b3);
                mma_bf16(acc[t][2], a0, a1, a2, a3, b0, b1);
                mma_bf16(acc[t][3], a0, a1, a2, a3, b2, b3);
            }
        }
        float check[4] = {0.f, 0.f, 0.f, 0.f};   // stay zero as long as every sum is finite
#pragma unroll
        for (int t = 0; t < NT; ++t)
#pragma unroll
            for (int nt = 0; nt < 4; ++nt)
#pragma unroll
                for (int x = 0; x < 4; ++x) check[x] = fmaf(acc[t][nt][x], 0.f, check[x]);
        if (__any_sync(kFull, !((check[0] + check[1]) + (check[2] + check[3]) == 0.f))) {
            const int t_lo = k_lo * 16;
            pool_by_members(smem, hs, smem, NT > 1, m, n_multi, t_lo, t_hi, dst_k, room, warp, lane);
            if (NT > 1) pool_by_members(smem + kVOff, hs, smem, NT > 1, m, n_multi, t_lo, t_hi, dst_v, room, warp, lane);
        } else {
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {
                const int c = hh ? lb : la;
                const int n = 16 * m + 8 * hh + g < n_multi ? cnt[c] : 0;
                if (n > 1 && c < room) {
                    const float inv = __frcp_rn((float)n);
                    const size_t o = (size_t)c * kD + warp * 32 + 2 * tig;
#pragma unroll
                    for (int t = 0; t < NT; ++t)
#pragma unroll
                        for (int nt = 0; nt < 4; ++nt) {
                            const __nv_bfloat162 v = __floats2bfloat162_rn(acc[t][nt][2 * hh] * inv, acc[t][nt][2 * hh + 1] * inv);
                            *reinterpret_cast<__nv_bfloat162*>((t ? dst_v : dst_k) + o + nt * 8) = v;
                        }
                }
            }
        }
    }
    // clusters of one token: bit for bit, sixteen lanes a row
    const int t = lane >> 4, chunk = lane & 15;
    for (int c0 = 0; c0 < P; c0 += 32) {
        const bool single = c0 + lane < P && c0 + lane < room && cnt[c0 + lane] == 1;
        uint32_t todo = __ballot_sync(kFull, single) & (0x11111111u << warp);
        while (todo) {
            const int c = c0 + __ffs(todo) - 1;
            todo &= todo - 1;
            if (t < NT)
                *reinterpret_cast<uint4*>((t ? dst_v : dst_k) + (size_t)c * kD + chunk * 8) =
                    *reinterpret_cast<const uint4*>(smem + t * kVOff + (chunk >> 3) * hs + tile_addr(seedrow[c], chunk & 7));
        }
    }
}

// What differs between the layers of a multi-layer launch (sc_compress_layers); a one-layer launch has one.
struct LayerRefs {
    CUtensorMap map_k, map_v;   // [B, Hkv, n, 128] bf16, boxes of 32 rows x 64 columns, 128-byte swizzle
    __nv_bfloat16* core_k; __nv_bfloat16* core_v; int32_t* count; int32_t* core_len; int32_t* assign;
};
constexpr int kMaxLayers = 64;   // layers per launch (the launch parameters hold their tensor maps)

template <int NL>
struct Params {
    int B, Hkv, n, L;
    const int32_t* seg_off; const int32_t* tile_seg; const int32_t* seq_tile_cnt; int n_tile_cap;
    float tau;
    int cap;
    int32_t* ctl;            // [0] ticket counter, [1] blocks finished
    uint32_t* tile_state;    // [L][B*Hkv][n_tile_cap]
    int32_t* status;
    const float* tau_dev;    // threshold in device memory (budget search), or null: use tau
    const int32_t* skip;     // device flag: nonzero = this launch has nothing to do (budget search), or null
    int overlap;             // SC_FLAG_OVERLAP_PREV
    int count_into_len;      // kCountOnly: add the tile's cluster count to core_len instead of recording it per tile
    LayerRefs layer[NL];
};

// The service warp draws the next ticket, turns it into a tile (layer, sequence, head, tile index, rows) and marks the rows
// that start a segment.  Tickets go round the (layer, sequence, head) units: ticket w is tile w / units of unit
// w % units, so a tile's predecessor has usually published its cluster count (and often its prefix) by the time
// the tile looks back.  A unit with fewer tiles skips its surplus tickets.
// geo[gT] = -1 when no work is left (max_nt = most tiles any sequence has).
template <int NL>
__device__ __forceinline__ void fetch_tile(const Params<NL>& p, int lane, int max_nt, int* geo, uint32_t* starts) {
    const int pairs = p.B * p.Hkv, units = pairs * p.L;
    int b, h, t, nt, ly;
    for (;;) {
        int w = 0;
        if (lane == 0) w = atomicAdd(&p.ctl[0], 1);
        w = __shfl_sync(kFull, w, 0);
        t = w / units;
        if (t >= max_nt) {
            if (lane == 0) geo[gT] = -1;
            __syncwarp();
            return;
        }
        const int unit = w - t * units;
        ly = unit / pairs;
        const int bh = unit - ly * pairs;
        b = bh / p.Hkv;
        h = bh - b * p.Hkv;
        nt = min(p.seq_tile_cnt[b], p.n_tile_cap);
        if (t < nt) break;
    }
    const int32_t* ts = p.tile_seg + (size_t)b * (p.n_tile_cap + 1);
    const int s_begin = ts[t], s_end = ts[t + 1];
    const int nseg = max(min(s_end - s_begin, kShortRows), 1);
    const int g_row0 = p.seg_off[s_begin];
    const int R = max(min(p.seg_off[s_begin + nseg] - g_row0, kMaxRows), 1);
    if (lane < 4) starts[lane] = 0u;
    __syncwarp();
    if (R <= kShortRows)
        for (int i = lane; i < nseg; i += 32) {
            const int a = min(p.seg_off[s_begin + i] - g_row0, kShortRows - 1);
            atomicOr(&starts[a >> 5], 1u << (a & 31));
        }
    if (lane == 0) {
        geo[gB] = b; geo[gH] = h; geo[gT] = t; geo[gNseg] = nseg; geo[gRow0] = g_row0 - b * p.n; geo[gR] = R;
        geo[gLast] = (t == nt - 1);
        geo[gLayer] = ly;
    }
    __syncwarp();
}

// Stages the rows of a tile of one tensor with TMA: one box of 32 rows x 64 columns per lane (R <= 256 needs at most 16 boxes for
// both column halves), the halves `hs` bytes apart at `dst`.  Rows past R inside the last box are the cache's next rows,
// or zeros past the end of the sequence; no cluster holds them.
__device__ __forceinline__ void stage_rows(uint32_t dst, int hs, const CUtensorMap* map, const int* geo, uint32_t bar, int lane) {
    const int nb = (geo[gR] + kBoxRows - 1) / kBoxRows;
    if (lane == 0) umma::mbar_expect_tx(bar, (uint32_t)(2 * nb * kBoxBytes));
    __syncwarp();
    if (lane < 2 * nb) {
        const int half = lane >= nb, i = lane - half * nb;
        tma_box(dst + half * hs + i * kBoxBytes, map, half * 64, geo[gRow0] + i * kBoxRows, geo[gH], geo[gB], bar);
    }
}

// Look-back by one warp: clusters of tiles 0 .. t - 1 of a head (their counts may still be on their way).
// Reads kPollGroups x 32 status words at a time, nearest first, until one that holds a full prefix.
__device__ __forceinline__ int look_back(const uint32_t* stt, int t, int lane, int32_t* status) {
    int upto = t, sum = 0;   // tiles [0, upto) still to be accounted for
    bool done = false;
    unsigned long long t0 = 0;
    while (upto > 0 && !done) {
        uint32_t v[kPollGroups];
#pragma unroll
        for (int j = 0; j < kPollGroups; ++j) {
            const int k = upto - 1 - lane - 32 * j;
            v[j] = (k >= 0) ? ld_volatile(&stt[k]) : kFlagPrefix;   // before tile 0: prefix 0
        }
        bool stalled = false, progressed = false;
#pragma unroll
        for (int j = 0; j < kPollGroups; ++j) {
            if (done || stalled) continue;
            const uint32_t ready = __ballot_sync(kFull, (v[j] >> 30) != 0u);
            const uint32_t pref = __ballot_sync(kFull, (v[j] >> 30) == 2u);
            // usable run: lanes 0..m-1 all ready, stopping at the first that holds a full prefix
            const int first_unready = (ready == kFull) ? 32 : __ffs(~ready) - 1;
            const int first_pref = pref ? __ffs(pref) - 1 : 32;
            const int take = min(first_unready, first_pref + 1);
            sum += warp_sum_i((lane < take) ? (int)(v[j] & kValueMask) : 0);
            if (first_pref < first_unready) { done = true; continue; }   // reached an inclusive prefix
            upto -= take;
            progressed |= take > 0;
            stalled = take < 32;
        }
        if (!done && !progressed) {
            const unsigned long long now = __shfl_sync(kFull, umma::global_ns(), 0);   // one clock for the warp
            if (t0 == 0) t0 = now;
            else if (now - t0 > kWaitLimitNs) { set_status(status, SC_ERR_TIMEOUT); return 0; }
            __nanosleep(64);
        }
    }
    return sum;
}

// kAnyTau: the threshold may be negative (the code for it costs the other case registers).
template <int kMode, int NL, bool kAnyTau>
__global__ void __launch_bounds__(kThreads, kBlocksPerSm) compress_fused_kernel(const __grid_constant__ Params<NL> p) {
    extern __shared__ __align__(1024) unsigned char smem[];   // the swizzle pattern repeats every 1024 bytes
    uint32_t* starts_buf = reinterpret_cast<uint32_t*>(smem + kMiscOff + 64);   // [2][4] rows that start a segment
    int* geo_buf = reinterpret_cast<int*>(smem + kMiscOff + 96);                // [2][8]
    volatile int* sh_base = reinterpret_cast<volatile int*>(smem + kMiscOff + 160);   // first core of the tile
    int* sh_p = reinterpret_cast<int*>(smem + kMiscOff + 164);                        // its clusters
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem + kMiscOff + 168);
    int* last_block = reinterpret_cast<int*>(smem + kMiscOff + 172);
    const uint32_t sbase = smem_u32(smem);
    // keys landed; values landed; product done; offset known; count known; buffer free; (long tile) keys spent
    const uint32_t bar_k = sbase + kBarOff, bar_v = bar_k + 8, bar_u = bar_k + 16, bar_base = bar_k + 24, bar_p = bar_k + 32,
                   bar_free = bar_k + 40, bar_half = bar_k + 48;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool service = warp == kWarps;   // the fifth warp
    int max_nt = 0;                        // most tiles any sequence has

    // An ordinary launch waits here for the kernel before it; an overlapped one waits for its predecessor only at its very end.
    if (!p.overlap) asm volatile("griddepcontrol.wait;\n" ::: "memory");
    if (p.skip != nullptr && *p.skip != 0) return;   // uniform over the grid: nothing touched, nothing to clean
    // (+ 0: a threshold of -0.0 becomes +0.0; its sign would reach the differences of sim_word)
    const float tau = (p.tau_dev != nullptr ? *p.tau_dev : p.tau) + 0.f;
    if (tid == 0) {
        umma::mbar_init(bar_k, 1);
        umma::mbar_init(bar_v, 1);
        umma::mbar_init(bar_u, 1);
        umma::mbar_init(bar_base, 1);
        umma::mbar_init(bar_p, 1);
        umma::mbar_init(bar_free, kWarps);
        umma::mbar_init(bar_half, kWarps);
        umma::mbar_fence_init();
        if ((sbase & 1023u) != 0u) set_status(p.status, SC_ERR_CUDA);   // the swizzled addressing assumes this
    }
    umma::fence_async_proxy();
    // Tensor memory for the product of a tile's keys: allocated once per (persistent) block by the service warp,
    // which then gives up the permit (a block may not allocate again after that, so it is not done per tile).
    if (service) umma::tmem_alloc(sbase + kMiscOff + 168, kTmemCols);
    umma::fence_before_sync();
    for (int b = lane; b < p.B; b += 32) max_nt = max(max_nt, min(p.seq_tile_cnt[b], p.n_tile_cap));
    max_nt = warp_max_i(max_nt);
    __syncthreads();
    umma::fence_after_sync();
    const uint32_t tmem = *tmem_slot;
    // The next kernel may be set up (under an overlapped launch of it: run) beside this one from here on, and not earlier: a block of
    // it that took the tensor memory first would keep this block waiting for it, while itself waiting for this kernel.
    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
    bool failed = false;

    if (service) {
        fetch_tile(p, lane, max_nt, geo_buf, starts_buf);
        uint32_t n_half = 0;
        for (uint32_t it = 0;; ++it) {
            const int* geo = geo_buf + (it & 1) * 8;
            // the buffer is free: the compute warps are through with the tile before
            if (it > 0 && !umma::mbar_wait(bar_free, (it - 1) & 1)) { failed = true; break; }
            if (geo[gT] < 0) {
                if (lane == 0) umma::mbar_arrive(bar_k);
                break;
            }
            const LayerRefs& lr = p.layer[NL == 1 ? 0 : geo[gLayer]];
            const bool long_tile = geo[gR] > kShortRows;
            stage_rows(sbase, long_tile ? kHalfLong : kHalfShort, &lr.map_k, geo, bar_k, lane);
            if (kMode != kCountOnly && !long_tile) stage_rows(sbase + kVOff, kHalfShort, &lr.map_v, geo, bar_v, lane);
            if (kMode != kCountOnly) {
                const int bh = geo[gB] * p.Hkv + geo[gH];
                uint32_t* stt = p.tile_state + (size_t)((NL == 1 ? 0 : geo[gLayer]) * p.B * p.Hkv + bh) * p.n_tile_cap;
                const int base = look_back(stt, geo[gT], lane, p.status);
                if (lane == 0) {
                    *sh_base = base;
                    umma::mbar_arrive(bar_base);
                }
                if (!umma::mbar_wait(bar_p, it & 1)) { failed = true; break; }
                if (lane == 0) {
                    const int upto = base + *sh_p;
                    atomicExch(&stt[geo[gT]], kFlagPrefix | (uint32_t)upto);
                    if (geo[gLast]) {
                        lr.core_len[bh] = upto;
                        if (upto > p.cap) set_status(p.status, SC_ERR_CAPACITY);
                    }
                }
                if (long_tile) {   // V takes the place of K
                    if (!umma::mbar_wait(bar_half, n_half & 1)) { failed = true; break; }
                    ++n_half;
                    stage_rows(sbase, kHalfLong, &lr.map_v, geo, bar_v, lane);
                }
            }
            // drawn now, not earlier: a tile drawn by a block that is still waiting would hold up its successors
            fetch_tile(p, lane, max_nt, geo_buf + ((it & 1) ^ 1) * 8, starts_buf + ((it & 1) ^ 1) * 4);
        }
    } else {
        uint32_t phase_u = 0;
        bool bad = false;   // a wait of this warp gave up
        for (uint32_t it = 0;; ++it) {
            const int* geo = geo_buf + (it & 1) * 8;
            const uint32_t par = it & 1;
            bad = !umma::mbar_wait(bar_k, par) || bad;   // the keys have landed (or there is no more work)
            if (!bad && geo[gT] < 0) break;
            const int R = bad ? 1 : geo[gR], row0 = geo[gRow0], bh = geo[gB] * p.Hkv + geo[gH], ly = NL == 1 || bad ? 0 : geo[gLayer];
            const LayerRefs& lr = p.layer[ly];
            int32_t* as = (lr.assign && !p.count_into_len) ? lr.assign + (size_t)bh * p.n + row0 : nullptr;
            uint32_t* publish = kMode == kCountOnly && p.count_into_len
                                    ? nullptr : p.tile_state + (size_t)(ly * p.B * p.Hkv + bh) * p.n_tile_cap + geo[gT];
            const bool long_tile = R > kShortRows;
            int P;
            if (!long_tile) {
                if (tid == 0 && !bad) {
                    umma::fence_after_sync();
                    umma_gram_block(sbase, kHalfShort, 0, 0, tmem, bar_u);
                }
                __syncwarp();
                P = settle_short_tile<kAnyTau>(smem, starts_buf + par * 4, R, tmem, phase_u, tau, bad, as, row0, publish, sh_p);
                phase_u ^= 1u;
            } else {
                P = settle_long_tile<kAnyTau>(smem, R, tmem, phase_u, tau, bad, as, row0, publish, sh_p);
                phase_u ^= 1u;   // three products
            }
            if (P < 0) { failed = true; break; }   // a wait for the product gave up
            if (kMode == kCountOnly) {
                if (tid == 0 && p.count_into_len) atomicAdd(&lr.core_len[bh], P);
            } else {
                if (tid == 0) umma::mbar_arrive(bar_p);
                bad = !umma::mbar_wait(bar_base, par) || bad;
                if (!long_tile) bad = !umma::mbar_wait(bar_v, par) || bad;
                __syncwarp();
                const int base = *sh_base, room = bad ? 0 : p.cap - base;   // a wait that gave up: nothing is stored
                const size_t first = (size_t)bh * p.cap + base;
                for (int c = tid; c < P && c < room; c += kTeam) lr.count[first + c] = reinterpret_cast<const int*>(smem + kCntOff)[c];
                if (!long_tile) {
                    pool_tile<2>(smem, kHalfShort, P, lr.core_k + first * kD, lr.core_v + first * kD, room, warp, lane);
                } else {
                    pool_tile<1>(smem, kHalfLong, P, lr.core_k + first * kD, nullptr, room, warp, lane);
                    umma::fence_async_proxy();   // the values' copies overwrite what ordinary accesses read
                    __syncwarp();
                    if (lane == 0) umma::mbar_arrive(bar_half);
                    bad = !umma::mbar_wait(bar_v, par) || bad;
                    __syncwarp();
                    pool_tile<1>(smem, kHalfLong, P, lr.core_v + first * kD, nullptr, bad ? 0 : room, warp, lane);
                }
            }
            umma::fence_async_proxy();   // the next tile's copies overwrite what ordinary accesses read
            __syncwarp();
            if (lane == 0) umma::mbar_arrive(bar_free);
        }
        failed = failed || bad;
    }

    // ---- exit: the last block to finish leaves the workspace zeroed for the next call ----
    if (failed) {   // a wait gave up: report it, and give copies that may still be in flight one more bounded
                    // wait (either parity: whichever phase is open) before the block's shared memory goes away
        set_status(p.status, SC_ERR_TIMEOUT);
        for (uint32_t ph = 0; ph < 2; ++ph) {
            umma::mbar_wait(bar_k, ph);
            umma::mbar_wait(bar_v, ph);
            umma::mbar_wait(bar_u, ph);
        }
    }
    umma::fence_before_sync();
    __syncthreads();
    if (service) umma::tmem_dealloc(tmem, kTmemCols);
    // Under an overlapped launch a block does not finish before the kernel enqueued ahead of this one has
    // completed, so completion is transitive along a run of overlapped launches (a no-op otherwise).
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
    if (tid == 0) {
        __threadfence();
        const int done = atomicAdd(&p.ctl[1], 1);
        *last_block = (done == (int)gridDim.x - 1);
    }
    __syncthreads();
    if (*last_block) {
        __threadfence();
        if (kMode != kCountOnly) {   // the words of tiles that exist
            const int units = p.L * p.B * p.Hkv;
            for (int u = warp; u < units; u += kWarps + 1)
                for (int i = lane; i < max_nt; i += 32) p.tile_state[(size_t)u * p.n_tile_cap + i] = 0u;
        }
        if (tid == 0) { p.ctl[0] = 0; p.ctl[1] = 0; }
    }
}

}  // namespace cf

namespace {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// cuTensorMapEncodeTiled, looked up through the runtime (the library does not link the driver).
EncodeTiledFn encode_tiled() {
    static EncodeTiledFn fn = nullptr;
    if (fn == nullptr) {
        void* ptr = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(ptr);
    }
    return fn;
}

// [B, Hkv, n, 128] bf16 with element strides st, read in boxes of 32 rows x 64 columns.
bool make_map(CUtensorMap* map, const void* base, const sc_strides& st, int B, int Hkv, int n) {
    EncodeTiledFn enc = encode_tiled();
    if (enc == nullptr) return false;
    const cuuint64_t dims[4] = {(cuuint64_t)cf::kD, (cuuint64_t)n, (cuuint64_t)Hkv, (cuuint64_t)B};
    const cuuint64_t strides[3] = {(cuuint64_t)st.n * 2, (cuuint64_t)(Hkv > 1 ? st.h : st.n * n) * 2,
                                   (cuuint64_t)(B > 1 ? st.b : st.n * n * (int64_t)Hkv) * 2};
    const cuuint32_t box[4] = {64, (cuuint32_t)cf::kBoxRows, 1, 1};
    const cuuint32_t elem[4] = {1, 1, 1, 1};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides, box, elem,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

bool compress_fused_supported(const CompressArgs& a) {
    // ticket arithmetic is 32-bit; TMA strides are below 2^40 bytes
    const int64_t lim = (int64_t)1 << 39;
    return a.dt == SC_BF16 && a.d == cf::kD && a.n_tile_cap >= 1 &&
           (int64_t)a.B * a.Hkv * (int64_t)a.n_tile_cap < (int64_t)1 << 30 && a.st.n > 0 && a.st.n < lim &&
           a.st.h >= 0 && a.st.h < lim && a.st.b >= 0 && a.st.b < lim && encode_tiled() != nullptr;
}

size_t compress_fused_ws_bytes(int32_t B, int32_t Hkv, int32_t n) {
    const size_t tiles = 2 * (size_t)div_up(n, SC_TILE_ROWS) + 1;
    return sizeof(uint32_t) * ((size_t)B * Hkv * tiles + cf::kCtlWords) + 256;
}

namespace {

// Blocks that are resident at once on the current device (one persistent block each), set up on first use.
int resident_blocks() {
    static int grid_of[64] = {0};
    int dev = 0;
    cudaGetDevice(&dev);
    dev &= 63;
    if (grid_of[dev] == 0) {
        cudaFuncSetAttribute(cf::compress_fused_kernel<cf::kCountOnly, 1, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, cf::kSmemBytes);
        cudaFuncSetAttribute(cf::compress_fused_kernel<cf::kCountOnly, 1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, cf::kSmemBytes);
        cudaFuncSetAttribute(cf::compress_fused_kernel<cf::kLookBack, 1, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, cf::kSmemBytes);
        cudaFuncSetAttribute(cf::compress_fused_kernel<cf::kLookBack, 1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, cf::kSmemBytes);
        cudaFuncSetAttribute(cf::compress_fused_kernel<cf::kLookBack, cf::kMaxLayers, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, cf::kSmemBytes);
        cudaFuncSetAttribute(cf::compress_fused_kernel<cf::kLookBack, cf::kMaxLayers, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, cf::kSmemBytes);
        // Blocks per SM by construction: launch bounds (registers), 75 KB of shared memory and 128 of the 512
        // tensor-memory columns each.  (The occupancy query answers 1 for a kernel that allocates tensor memory.)
        // Launching more blocks than are resident would be harmless: a block draws its first ticket when it starts.
        int sms = 0;
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        grid_of[dev] = (sms < 1 ? 1 : sms) * cf::kBlocksPerSm;
    }
    return grid_of[dev];
}

template <int NL>
void fill_common(cf::Params<NL>& p, const CompressArgs& a, int L) {
    p.B = a.B; p.Hkv = a.Hkv; p.n = a.n; p.L = L;
    p.seg_off = a.seg_off; p.tile_seg = a.tile_seg; p.seq_tile_cnt = a.seq_tile_cnt; p.n_tile_cap = a.n_tile_cap;
    p.tau = a.tau; p.cap = a.cap;
    p.tau_dev = a.tau_dev; p.skip = a.skip; p.count_into_len = a.count_only ? 1 : 0;
    p.overlap = 0;
    p.ctl = (int32_t*)a.ws;
    p.tile_state = (uint32_t*)a.ws + cf::kCtlWords;
    p.status = a.status;
}

bool fill_layer(cf::LayerRefs& r, const CompressArgs& a, const void* K, const void* V, void* core_k, void* core_v,
                int32_t* count, int32_t* core_len, int32_t* assign) {
    r.core_k = (__nv_bfloat16*)core_k; r.core_v = (__nv_bfloat16*)core_v; r.count = count; r.core_len = core_len;
    r.assign = assign;
    return make_map(&r.map_k, K, a.st, a.B, a.Hkv, a.n) && make_map(&r.map_v, V, a.st, a.B, a.Hkv, a.n);
}

}  // namespace

cudaError_t launch_compress_fused(const CompressArgs& a, cudaStream_t st) {
    const int resident = resident_blocks();
    cf::Params<1> p;
    fill_common(p, a, 1);
    if (!fill_layer(p.layer[0], a, a.K, a.V, a.core_k, a.core_v, a.count, a.core_len, a.assign))
        return cudaErrorNotSupported;   // a layout TMA cannot describe: the caller takes the generic kernels
    // no more blocks than there can be tiles
    const int64_t max_tiles = (int64_t)a.B * a.Hkv * a.n_tile_cap;
    const int grid = (int)(max_tiles < resident ? max_tiles : resident);
    const bool any_tau = a.tau < 0.f;   // (of a search: its lowest threshold)
    const auto count = any_tau ? cf::compress_fused_kernel<cf::kCountOnly, 1, true> : cf::compress_fused_kernel<cf::kCountOnly, 1, false>;
    const auto full = any_tau ? cf::compress_fused_kernel<cf::kLookBack, 1, true> : cf::compress_fused_kernel<cf::kLookBack, 1, false>;
    if (a.count_only) {   // budget search: per-head cluster counts only
        note_launches(1);
        return launch_in_order(count, dim3(grid), cf::kThreads, cf::kSmemBytes, st, p);
    } else if (a.flags & SC_FLAG_TWO_PASS) {
        cf::Params<1> pc = p;
        pc.layer[0].assign = nullptr;
        note_launches(2);
        const cudaError_t e = launch_in_order(count, dim3(grid), cf::kThreads, cf::kSmemBytes, st, pc);
        return e != cudaSuccess ? e : launch_in_order(full, dim3(grid), cf::kThreads, cf::kSmemBytes, st, p);
    } else {
        // With SC_FLAG_OVERLAP_PREV the kernel may start while the one enqueued before it on the stream is
        // still draining (the caller has promised they share nothing either writes): the tail of one
        // layer's persistent blocks then overlaps the start of the next layer's.
        p.overlap = (a.flags & SC_FLAG_OVERLAP_PREV) ? 1 : 0;
        note_launches(1);
        return launch_in_order(full, dim3(grid), cf::kThreads, cf::kSmemBytes, st, p);
    }
}

// Several layers in one launch (sc_compress_layers): the (layer, sequence, head) units take the tickets in turn,
// so consecutive tiles of one head are L*B*Hkv tickets apart and a tile's predecessor has usually published its
// prefix long before the tile looks back.  `a` describes what the layers share (a.K .. a.assign are not used).
cudaError_t launch_compress_fused_layers(const CompressArgs& a, const sc_compress_layer* layers, int32_t L, cudaStream_t st) {
    if (L < 1 || L > cf::kMaxLayers) return cudaErrorInvalidValue;
    const int resident = resident_blocks();
    static cf::Params<cf::kMaxLayers> p;   // 20 KB: kept off the stack; filled and passed by value under the lock
    static std::mutex lock;
    std::lock_guard<std::mutex> guard(lock);
    fill_common(p, a, L);
    for (int l = 0; l < L; ++l)
        if (!fill_layer(p.layer[l], a, layers[l].K, layers[l].V, layers[l].core_k, layers[l].core_v, layers[l].count,
                        layers[l].core_len, layers[l].assign))
            return cudaErrorNotSupported;
    for (int l = L; l < cf::kMaxLayers; ++l) p.layer[l] = p.layer[0];
    const int64_t max_tiles = (int64_t)L * a.B * a.Hkv * a.n_tile_cap;
    const int grid = (int)(max_tiles < resident ? max_tiles : resident);
    const auto full = a.tau < 0.f ? cf::compress_fused_kernel<cf::kLookBack, cf::kMaxLayers, true> : cf::compress_fused_kernel<cf::kLookBack, cf::kMaxLayers, false>;
    note_launches(1);
    return launch_in_order(full, dim3(grid), cf::kThreads, cf::kSmemBytes, st, p);
}

size_t compress_fused_layers_ws_bytes(int32_t L, int32_t B, int32_t Hkv, int32_t n) {
    const size_t tiles = 2 * (size_t)div_up(n, SC_TILE_ROWS) + 1;
    return sizeof(uint32_t) * ((size_t)L * B * Hkv * tiles + cf::kCtlWords) + 256;
}

}  // namespace sc
