// Tensor-core bf16 decode attention for Eq. 4 (d = 128, query group G <= 8), sm_100a.
//
// One block serves one (sequence, KV head, split): its warps stream 16-row tiles of the head's
// cores through private cp.async rings in shared memory (16-byte chunks, XOR-swizzled so that
// ldmatrix is conflict free) and fold the whole GQA group into one pass:
//     S^T[16 keys x 8 heads]   = K_tile . q^T                (mma.m16n8k16, keys on M, heads on N)
//     x = S^T * scale*log2(e) + log2(count)                  (Proportional Attention, base 2)
//     P^T = 2^(x - m)  (online softmax; the running max is per head, common to the warp, and
//                       raised only when a score overtakes it by a margin)
//     O^T[128 dims x 8 heads] += V_tile^T . P^T              (ldmatrix.trans, P^T via movmatrix,
//                                                             as a bf16 pair: leading part + remainder)
// Warps are merged in a fixed order through shared memory into one (m, l, O) partial per block.
// The splits of a head form a thread-block cluster and fold their partials through distributed shared memory, each
// block its own slice of the output (no partial leaves the SMs).  Where a head has several clusters, or blocks outside
// clusters, partials go to global memory and the last one to arrive (atomic ticket, no waiting) merges them, slice by slice
// where there are counters enough, else a head at once.
// How many splits: plan_for.  In a batch the blocks that the plan gives a head are one unit; a head much longer than the mean
// of the launch gets more units (plan_units), so that a long sequence among short ones is not streamed by a few blocks.
// Every order is fixed, so results are bit-reproducible.
//
// Launch modes: ordinary; overlapped with the preceding kernel (programmatic stream
// serialization), where every global write waits for that kernel's completion; and chained, where
// in addition q is read only after that wait (q is the preceding kernel's product) while the cores
// were requested before it.
#include <cooperative_groups.h>

#include <mutex>

#include "decode_fold.cuh"

namespace sc {

namespace dm {

namespace cg = cooperative_groups;

enum LaunchMode { kOrdinary = 0, kOverlapped = 1, kChained = 2 };

constexpr int kWarps = 4;
constexpr int kStages = 3;
constexpr int kTile = 16;                       // rows per warp tile
constexpr int kD = 128;
constexpr int kRowBytes = kD * 2;               // 256
constexpr int kTileBytes = kTile * kRowBytes;   // 4096 per K or V tile
constexpr int kStageBytes = 2 * kTileBytes + 64;  // K, V, 16 counts
constexpr int kWarpBytes = kStages * kStageBytes;
constexpr int kRecvBytes = (8 * (kD / 4) + 16) * 16 + 16 * 64;   // what the blocks of a cluster hand each other: slices of O (rounded up), m and l
constexpr int kSmemBytes = kWarps * kWarpBytes + kRecvBytes;
constexpr int kPartStride = 8 * kD + 16;        // floats per (b, h, split): acc[8 heads][128], m[8], l[8]
constexpr int kCtasPerSm = 2;                   // two kernels (consecutive layers) can be co-resident
constexpr float kMaxSlack = 8.f;                // log2 units a score may exceed the running maximum before it is raised
constexpr int kMergeGroup = 16;                 // cluster partials folded per round by the merging block
constexpr int kCapRowsPerBlock = 1408;          // rows of capacity per block from which a head gets another cluster (heads are usually half full or less)
constexpr int kMaxSlots = 160;                  // partials in global memory over the launch's own units (at least one per head)
constexpr int kMaxTickets = 512;                // arrival counters: one per head and slice where these are enough, else one per head

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, int src_bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_async4(uint32_t dst, const void* src, int src_bytes) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

__device__ __forceinline__ void ldmatrix_x4(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}
__device__ __forceinline__ uint32_t movmatrix_trans(uint32_t a) {
    uint32_t d;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;\n" : "=r"(d) : "r"(a));
    return d;
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}
__device__ __forceinline__ float bf16_lo(uint32_t v) { return __uint_as_float(v << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t v) { return __uint_as_float(v & 0xffff0000u); }
__device__ __forceinline__ float fast_log2(float x) {
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;\n" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ void store_out4(__nv_bfloat16* dst, const float4& acc, float inv) {
    __nv_bfloat162 lo = __floats2bfloat162_rn(acc.x * inv, acc.y * inv);
    __nv_bfloat162 hi = __floats2bfloat162_rn(acc.z * inv, acc.w * inv);
    uint2 pk;
    pk.x = *reinterpret_cast<uint32_t*>(&lo);
    pk.y = *reinterpret_cast<uint32_t*>(&hi);
    *reinterpret_cast<uint2*>(dst) = pk;
}

// Copies rows [row0, row0+16) of one head's cores into a stage; rows >= len are zero-filled.  Lane l
// moves 16-byte chunk l & 15 of rows 2i + (l >> 4), i = 0..7, to its swizzled place soff[i] (the same
// for every tile, so the caller computes the eight offsets once).  A tile that lies wholly inside the
// head -- all but the last one -- needs no per-row test.
__device__ __forceinline__ void issue_tile(uint32_t stage, const __nv_bfloat16* __restrict__ kh,
                                           const __nv_bfloat16* __restrict__ vh, const int32_t* __restrict__ ch,
                                           int row0, int len, int lane, const uint32_t (&soff)[8]) {
    const size_t g0 = (size_t)(row0 + (lane >> 4)) * kD + (lane & 15) * 8;
    if (row0 + kTile <= len) {
        const __nv_bfloat16* ks = kh + g0;
        const __nv_bfloat16* vs = vh + g0;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            cp_async16(stage + soff[i], ks + i * 2 * kD, 16);
            cp_async16(stage + kTileBytes + soff[i], vs + i * 2 * kD, 16);
        }
        if (ch != nullptr && lane < kTile) cp_async4(stage + 2 * kTileBytes + lane * 4, ch + row0 + lane, 4);
        return;
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const bool ok = row0 + 2 * i + (lane >> 4) < len;
        const size_t goff = ok ? g0 + (size_t)i * 2 * kD : 0;
        cp_async16(stage + soff[i], kh + goff, ok ? 16 : 0);
        cp_async16(stage + kTileBytes + soff[i], vh + goff, ok ? 16 : 0);
    }
    if (ch != nullptr && lane < kTile) {
        const int row = row0 + lane;
        const bool ok = row < len;
        cp_async4(stage + 2 * kTileBytes + lane * 4, ch + (ok ? row : 0), ok ? 4 : 0);
    }
}

// Several partials per head in global memory (one per cluster, or per block outside clusters).  The blocks that hold the same
// elements [e_lo, e_hi) of them share a ticket; the last one to arrive merges the `n_parts` partials' elements: the first
// `n_first` partials lie in the slots from `first` on, the others from `more` on.  All threads of the block call it.  The fence and the
// barrier order this block's partial stores before its ticket, whose release makes them visible to whoever reads
// the ticket with acquire (the last arrival); that block's other threads are ordered behind its thread 0 by the second barrier
// and read the partials from L2.
template <bool kSpares>
__device__ __forceinline__ void ticket_and_merge(const float* __restrict__ part, int first, int more, int n_first, int n_parts, int32_t* __restrict__ ticket,
                                                 int arrivals, int e_lo, int e_hi, int bh, int G, __nv_bfloat16* __restrict__ out, int* sh_last_p) {
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        int t;
        asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], 1;\n" : "=r"(t) : "l"(ticket) : "memory");
        *sh_last_p = (t == arrivals - 1);
        if (*sh_last_p) *ticket = 0;   // leave the counter ready for the next call
    }
    __syncthreads();
    if (!*sh_last_p) return;
    // One thread per (head, four output columns); the partials are folded sixteen at a time, all of a
    // group's loads in flight together (one round trip to L2 per group).
    for (int e4 = e_lo + threadIdx.x; e4 < e_hi; e4 += kWarps * 32) {
        const int hd = e4 / (kD / 4), d4 = (e4 % (kD / 4)) * 4;
        float gm = -INFINITY, lsum = 0.f;
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int s0 = 0; s0 < n_parts; s0 += kMergeGroup) {
            float mv[kMergeGroup], lv[kMergeGroup];
            float4 ov[kMergeGroup];
#pragma unroll
            for (int j = 0; j < kMergeGroup; ++j) {
                const bool ok = s0 + j < n_parts;
                const int s = ok ? s0 + j : 0, slot = s + (!kSpares || s < n_first ? first : more - n_first);
                const float* sp = part + (size_t)slot * kPartStride;
                mv[j] = ok ? __ldcg(sp + 8 * kD + hd) : -INFINITY;
                lv[j] = ok ? __ldcg(sp + 8 * kD + 8 + hd) : 0.f;
                ov[j] = ok ? __ldcg(reinterpret_cast<const float4*>(sp + hd * kD + d4)) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
            float cm = mv[0];
#pragma unroll
            for (int j = 1; j < kMergeGroup; ++j) cm = fmaxf(cm, mv[j]);
            const float ngm = fmaxf(gm, cm);
            if (ngm == -INFINITY) continue;   // nothing but empty splits so far
            const float c = (gm == -INFINITY) ? 0.f : fast_exp2(gm - ngm);
            lsum *= c; acc.x *= c; acc.y *= c; acc.z *= c; acc.w *= c;
            gm = ngm;
#pragma unroll
            for (int j = 0; j < kMergeGroup; ++j) {
                const float w = (mv[j] == -INFINITY) ? 0.f : fast_exp2(mv[j] - gm);
                lsum = fmaf(w, lv[j], lsum);
                acc.x = fmaf(w, ov[j].x, acc.x); acc.y = fmaf(w, ov[j].y, acc.y);
                acc.z = fmaf(w, ov[j].z, acc.z); acc.w = fmaf(w, ov[j].w, acc.w);
            }
        }
        const float inv = lsum > 0.f ? 1.f / lsum : 0.f;
        store_out4(out + ((size_t)bh * G + hd) * kD + d4, acc, inv);
    }
}

// Units of a batched launch.  Every head has its own; a head of more than one and a half times the mean number of tiles gets as
// many more, from a pool of as many spare units as there are heads, as brings its units nearest to the mean.  Worked out by
// every warp from the lengths alone (one round trip for all of them, beside the block's own): head `want` has units
// 1 + extra, its extra units are numbers [begin, begin + extra) of the pool.  For a spare unit (`spare` >= 0) `want` is found
// first: the head that unit belongs to, or -1.  16 sequences x 8 heads, one of 32 K rows among 1 K: 134 us with equal
// shares, 72 with shares cut by capacity and used as a head's length warranted, 43 like this.
struct Units { int head, extra, begin; };
__device__ __forceinline__ Units plan_units(const int32_t* __restrict__ core_len, int heads, int cap, int want, int spare, int lane) {
    auto tiles_of = [&](int i) { return i < heads ? (max(min(core_len[i], cap), 0) + kTile - 1) / kTile : 0; };
    int sum = 0;
#pragma unroll 4
    for (int i = lane; i < heads; i += 32) sum += tiles_of(i);
    sum = max(__reduce_add_sync(kFull, sum), 1);
    // units nearest to tiles * heads / sum, at least one
    auto extra_of = [&](int i) {
        const long long x2 = 2ll * tiles_of(i) * heads;
        return x2 < 3ll * sum ? 0 : (int)((x2 + sum) / (2ll * sum)) - 1;
    };
    Units u = {want, want >= 0 ? extra_of(want) : 0, 0};
    if (want >= 0 && u.extra == 0) return u;
    int before = 0;
    for (int i0 = 0; i0 < heads; i0 += 32) {
        const int mine = extra_of(i0 + lane), upto = before + warp_scan_add(mine, lane);
        const unsigned here = __ballot_sync(kFull, want >= 0 ? i0 + lane == want : (mine > 0 && spare < upto));
        if (here) {
            const int src = __ffs(here) - 1;
            u.head = i0 + src;
            u.extra = __shfl_sync(kFull, mine, src);
            u.begin = __shfl_sync(kFull, upto, src) - u.extra;
            return u;
        }
        before = __shfl_sync(kFull, upto, 31);
    }
    return u;
}

// kSpares: the launch has spare units (the code for them costs the others 0.2 us).
// kPair: up to four query heads.  The second product's eight columns then hold the heads' leading parts and, four columns on, their
// remainders, so one product does for both; the queries stand in the first product's columns twice, which gives the lanes
// of either half the scores they need.  The remainders' part then has accumulators of its own, which rounds less: of 98304 outputs over 4 x 64K
// raw rows 246 are not the bf16 nearest to the value in 64 bits, 410 with both parts in one accumulator (16 x 16K cores: 930 and 966 of 393216).
template <bool kSpares, bool kPair>
__global__ void __launch_bounds__(kWarps * 32, kCtasPerSm)
decode_mma_kernel(const __nv_bfloat16* __restrict__ q, int Hq, int Hkv, const __nv_bfloat16* __restrict__ core_k,
                  const __nv_bfloat16* __restrict__ core_v, const int32_t* __restrict__ count, int cap,
                  const int32_t* __restrict__ core_len, float scale_log2, int B, int mode,
                  __nv_bfloat16* __restrict__ out, float* __restrict__ part, int32_t* __restrict__ tickets, int32_t* status) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ float sh_m[kWarps][8];
    __shared__ float sh_l[kWarps][8];
    __shared__ int sh_last;
    __shared__ __align__(8) unsigned long long sh_bar;   // what the cluster's blocks hand this one has arrived

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int g = lane >> 2, tig = lane & 3;
    const int G = Hq / Hkv;
    // Block r of the cluster folds slice r of the head's (head, column) pairs, [e_lo, e_hi), and is handed that slice by every
    // block (see the fold).
    const int csize = (int)cg::this_cluster().num_blocks(), crank = (int)cg::this_cluster().block_rank();
    const int slice = (G * (kD / 4) + csize - 1) / csize;
    const int e_lo = min(crank * slice, G * (kD / 4)), e_hi = min(e_lo + slice, G * (kD / 4));
    const auto set_up = [&] {
        if (threadIdx.x == 0) {
            umma::mbar_init(smem_u32(&sh_bar), 1);
            umma::mbar_fence_init();
            umma::mbar_expect_tx(smem_u32(&sh_bar), (uint32_t)(csize * ((e_hi - e_lo) * 16 + 64)));   // (m and l come to a block without a slice too)
        }
        __syncwarp();
        asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");   // (the wait is in front of the first access to another block's shared memory)
    };
    // An ordinary launch waits here for the kernel before it.  Under an overlapped one the next kernel may start beside
    // this one, and whatever this block reads before its own griddepcontrol.wait below (core_len, cores, counts) must not
    // be written by a kernel that may still be running then; that is the caller's promise when it asks for one.  An ordinary
    // launch sets its barrier up before it waits (200 calls over 8 x 0.5 K rows from a graph 4.13 -> 3.72 us each, 4.32 when
    // the fold read the members' shared memory), an overlapped one lets the next kernel in first (32 dependent layers 325, 332 the other way).
    if (mode == kOrdinary) {
        set_up();
        asm volatile("griddepcontrol.wait;\n" ::: "memory");
    }
    // Where there are spare units the next kernel is let in only when they have gone: its blocks would find both slots of some
    // SMs taken by them, and settle unevenly (128 raw heads x 8 K rows: 80 us, 92 with the next kernel let in at once).
    if (!kSpares) asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
    if (mode != kOrdinary) set_up();
    // the block's head, and its place among the head's blocks
    int bh = blockIdx.z * Hkv + blockIdx.y, split = blockIdx.x, n_split = gridDim.x;   // as if every head had one unit
    Units u = {bh, 0, 0};
    if (kSpares) {
        const int heads = B * Hkv, spare = bh - heads;
        u = plan_units(core_len, heads, cap, spare < 0 ? bh : -1, spare, lane);
        if (u.head < 0) return;   // a spare unit that no head needs: nothing read, nothing written
        n_split *= 1 + u.extra;
        if (spare >= 0) split += (1 + spare - u.begin) * (int)gridDim.x;
        bh = u.head;
    }
    const int len = max(min(core_len[bh], cap), 0);
    const int tiles_total = (len + kTile - 1) / kTile;
    const int tiles_per_split = (tiles_total + n_split - 1) / n_split;
    const int t0 = min(split * tiles_per_split, tiles_total);
    const int t1 = min(t0 + tiles_per_split, tiles_total);
    // this warp's tiles: t0 + warp, t0 + warp + kWarps, ...
    const int my_tiles = (t1 - t0 - warp + kWarps - 1) / kWarps;   // may be <= 0

    const __nv_bfloat16* kh = core_k + (size_t)bh * cap * kD;
    const __nv_bfloat16* vh = core_v + (size_t)bh * cap * kD;
    const int32_t* ch = count ? count + (size_t)bh * cap : nullptr;
    const uint32_t wbase = smem_u32(smem) + warp * kWarpBytes;

    uint32_t soff[8];   // this lane's eight chunk places inside a K or V tile (see issue_tile)
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int r = 2 * i + (lane >> 4), c = lane & 15;
        soff[i] = r * kRowBytes + ((c ^ (r & 7)) << 4);
    }

    // prologue: fill the whole ring (under a chained launch this is what is in shared memory when the wait ends)
#pragma unroll
    for (int s = 0; s < kStages; ++s) {
        if (s < my_tiles) issue_tile(wbase + s * kStageBytes, kh, vh, ch, (t0 + warp + s * kWarps) * kTile, len, lane, soff);
        cp_async_commit();
    }

    // Chained launch (SC_FLAG_OVERLAP_CHAIN): q is the preceding kernel's product.  The cores' first
    // tiles are on their way to shared memory; only now wait
    // for that kernel to complete (and its writes to be visible), then read q.
    if (mode == kChained) asm volatile("griddepcontrol.wait;\n" ::: "memory");

    // q^T as the B operand of every k-step: b0 = q[head g][16ks + 2tig, +1], b1 = same + 8
    uint32_t qb[8][2];
    {
        const int hd = kPair ? g & 3 : g;
        const __nv_bfloat16* qh = q + ((size_t)bh * G + hd) * kD;
#pragma unroll
        for (int ks = 0; ks < 8; ++ks) {
            // read through L2: under a chained launch q was written while this kernel was already running
            qb[ks][0] = (hd < G) ? __ldcg(reinterpret_cast<const uint32_t*>(qh + ks * 16 + 2 * tig)) : 0u;
            qb[ks][1] = (hd < G) ? __ldcg(reinterpret_cast<const uint32_t*>(qh + ks * 16 + 2 * tig + 8)) : 0u;
        }
    }
    float o[8][4];
#pragma unroll
    for (int mt = 0; mt < 8; ++mt) { o[mt][0] = o[mt][1] = o[mt][2] = o[mt][3] = 0.f; }
    float m0 = -INFINITY, m1 = -INFINITY, l0 = 0.f, l1 = 0.f;   // columns 2tig and 2tig+1

    // per-lane ldmatrix row/chunk selectors
    const int lm_j = lane >> 3, lm_r = lane & 7;
    const int k_row = lm_r + ((lm_j & 1) << 3), k_csel = lm_j >> 1;    // K: matrices (r0-7,c), (r8-15,c), (r0-7,c+1), (r8-15,c+1)
    const int v_row = lm_r + ((lm_j >> 1) << 3), v_csel = lm_j & 1;    // V^T: (r0-7,c), (r0-7,c+1), (r8-15,c), (r8-15,c+1)

    for (int i = 0; i < my_tiles; ++i) {
        cp_async_wait<kStages - 1>();   // tile i has landed; tiles i+1, i+2 are on their way
        __syncwarp();

        const uint32_t st = wbase + (i % kStages) * kStageBytes;
        const int row0 = (t0 + warp + i * kWarps) * kTile;

        // S^T = K . q^T, four accumulator chains
        float sa[4] = {0.f, 0.f, 0.f, 0.f}, sb[4] = {0.f, 0.f, 0.f, 0.f};
        float sc2[4] = {0.f, 0.f, 0.f, 0.f}, sd[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int ks = 0; ks < 8; ++ks) {
            uint32_t a0, a1, a2, a3;
            const int c = 2 * ks + k_csel;
            ldmatrix_x4(st + k_row * kRowBytes + ((c ^ (k_row & 7)) << 4), a0, a1, a2, a3);
            if ((ks & 3) == 0) mma_bf16(sa, a0, a1, a2, a3, qb[ks][0], qb[ks][1]);
            else if ((ks & 3) == 1) mma_bf16(sb, a0, a1, a2, a3, qb[ks][0], qb[ks][1]);
            else if ((ks & 3) == 2) mma_bf16(sc2, a0, a1, a2, a3, qb[ks][0], qb[ks][1]);
            else mma_bf16(sd, a0, a1, a2, a3, qb[ks][0], qb[ks][1]);
        }
        float lc_lo = 0.f, lc_hi = 0.f;
        if (ch != nullptr) {
            const int* cs = reinterpret_cast<const int*>(smem + warp * kWarpBytes + (i % kStages) * kStageBytes + 2 * kTileBytes);
            lc_lo = fast_log2((float)max(cs[g], 1));
            lc_hi = fast_log2((float)max(cs[g + 8], 1));
        }
        const bool ok_lo = row0 + g < len, ok_hi = row0 + g + 8 < len;
        const float x0 = ok_lo ? fmaf((sa[0] + sb[0]) + (sc2[0] + sd[0]), scale_log2, lc_lo) : -INFINITY;
        const float x1 = ok_lo ? fmaf((sa[1] + sb[1]) + (sc2[1] + sd[1]), scale_log2, lc_lo) : -INFINITY;
        const float x2 = ok_hi ? fmaf((sa[2] + sb[2]) + (sc2[2] + sd[2]), scale_log2, lc_hi) : -INFINITY;
        const float x3 = ok_hi ? fmaf((sa[3] + sb[3]) + (sc2[3] + sd[3]), scale_log2, lc_hi) : -INFINITY;
        // The running maxima m0, m1 are common to the warp.  They are raised only when some lane meets a
        // score more than kMaxSlack above them (one vote per tile instead of a shuffle reduction): the
        // weights 2^(x - m) then stay below 2^kMaxSlack, which fp32 sums and bf16 weights carry without loss.
        const float lx0 = fmaxf(x0, x2), lx1 = fmaxf(x1, x3);
        if (__any_sync(kFull, (lx0 > m0 + kMaxSlack) || (lx1 > m1 + kMaxSlack))) {
            float mx0 = lx0, mx1 = lx1;
#pragma unroll
            for (int off = 4; off < 32; off <<= 1) {
                mx0 = fmaxf(mx0, __shfl_xor_sync(kFull, mx0, off));
                mx1 = fmaxf(mx1, __shfl_xor_sync(kFull, mx1, off));
            }
            const float mn0 = fmaxf(m0, mx0), mn1 = fmaxf(m1, mx1);   // finite: a tile has a valid row
            const float c0 = fast_exp2(m0 - mn0), c1 = fast_exp2(m1 - mn1);
            l0 *= c0; l1 *= c1;
#pragma unroll
            for (int mt = 0; mt < 8; ++mt) { o[mt][0] *= c0; o[mt][2] *= c0; o[mt][1] *= c1; o[mt][3] *= c1; }
            m0 = mn0; m1 = mn1;
        }
        // The weights enter the second product as bf16 pairs (leading part + remainder), which keeps
        // sixteen bits of each: a single bf16 rounding of P would be the largest error of the whole path.
        const float w0 = fast_exp2(x0 - m0), w1 = fast_exp2(x1 - m1);   // row g
        const float w2 = fast_exp2(x2 - m0), w3 = fast_exp2(x3 - m1);   // row g + 8
        const uint32_t p_lo = pack_bf16x2(w0, w1), p_hi = pack_bf16x2(w2, w3);
        const uint32_t r_lo = pack_bf16x2(w0 - bf16_lo(p_lo), w1 - bf16_hi(p_lo));
        const uint32_t r_hi = pack_bf16x2(w2 - bf16_lo(p_hi), w3 - bf16_hi(p_hi));
        l0 += (bf16_lo(p_lo) + bf16_lo(r_lo)) + (bf16_lo(p_hi) + bf16_lo(r_hi));
        l1 += (bf16_hi(p_lo) + bf16_hi(r_lo)) + (bf16_hi(p_hi) + bf16_hi(r_hi));
        const uint32_t pb0 = movmatrix_trans(kPair && tig >= 2 ? r_lo : p_lo), pb1 = movmatrix_trans(kPair && tig >= 2 ? r_hi : p_hi);
        const uint32_t rb0 = kPair ? 0u : movmatrix_trans(r_lo), rb1 = kPair ? 0u : movmatrix_trans(r_hi);

        // O^T += V^T . P^T
#pragma unroll
        for (int mt = 0; mt < 8; ++mt) {
            uint32_t a0, a1, a2, a3;
            const int c = 2 * mt + v_csel;
            ldmatrix_x4_trans(st + kTileBytes + v_row * kRowBytes + ((c ^ (v_row & 7)) << 4), a0, a1, a2, a3);
            mma_bf16(o[mt], a0, a1, a2, a3, pb0, pb1);
            if (!kPair) mma_bf16(o[mt], a0, a1, a2, a3, rb0, rb1);
        }
        __syncwarp();
        // the stage just consumed takes the tile three ahead
        const int nxt = i + kStages;
        if (nxt < my_tiles)
            issue_tile(wbase + (i % kStages) * kStageBytes, kh, vh, ch, (t0 + warp + nxt * kWarps) * kTile, len, lane, soff);
        cp_async_commit();
        if (kSpares && i == 0) asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
    }
    cp_async_wait<0>();

    // ---- merge the warps of this block (fixed order) ----
    // lane-local l covers rows g, g+8 of every tile: sum over the 8 row groups
#pragma unroll
    for (int off = 4; off < 32; off <<= 1) {
        l0 += __shfl_xor_sync(kFull, l0, off);
        l1 += __shfl_xor_sync(kFull, l1, off);
    }
    if (g == 0) {
        sh_m[warp][2 * tig] = m0; sh_m[warp][2 * tig + 1] = m1;
        sh_l[warp][2 * tig] = l0; sh_l[warp][2 * tig + 1] = l1;
    }
    __syncthreads();   // every warp is done with its ring; reuse it as [warp][8 heads][128] fp32
    float bm0 = -INFINITY, bm1 = -INFINITY;
#pragma unroll
    for (int w2 = 0; w2 < kWarps; ++w2) { bm0 = fmaxf(bm0, sh_m[w2][2 * tig]); bm1 = fmaxf(bm1, sh_m[w2][2 * tig + 1]); }
    const float f0 = (m0 == -INFINITY) ? 0.f : fast_exp2(m0 - bm0);
    const float f1 = (m1 == -INFINITY) ? 0.f : fast_exp2(m1 - bm1);
    float* slab = reinterpret_cast<float*>(smem) + warp * (8 * kD);
#pragma unroll
    for (int mt = 0; mt < 8; ++mt) {
        const int d0 = mt * 16 + g;
        slab[(2 * tig) * kD + d0] = o[mt][0] * f0;
        slab[(2 * tig + 1) * kD + d0] = o[mt][1] * f1;
        slab[(2 * tig) * kD + d0 + 8] = o[mt][2] * f0;
        slab[(2 * tig + 1) * kD + d0 + 8] = o[mt][3] * f1;
    }
    __syncthreads();
    // ---- the splits of one thread-block cluster are folded through distributed shared memory ----
    // Block r of the cluster folds slice r of the (head, column) pairs.  Every block adds up its warps' slabs and hands each slice, and
    // its m and l, straight to the block that folds it (st.async, counted by that block's mbarrier): a block waits for what it
    // folds and for nothing else, reads it from its own shared memory and may leave.  32 dependent layers of 8 heads x
    // 8.3 K rows 325 us; with plain stores and a cluster barrier 339; reading out of the members' shared memory between two
    // cluster barriers 350.  28 layers of 4 x 34 K rows 499, 501, 520; one call over 8 x 0.5 K rows 5.2 each.
    float4* recv_o = reinterpret_cast<float4*>(smem + kWarps * kWarpBytes);   // [csize][slice]
    float* recv_ml = reinterpret_cast<float*>(smem + kWarps * kWarpBytes + (8 * (kD / 4) + 16) * 16);   // [csize][m of 8 heads, l of 8 heads]
    asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");   // every block of the cluster has started
    const float* slabs = reinterpret_cast<const float*>(smem);
    for (int e4 = threadIdx.x; e4 < G * (kD / 4); e4 += kWarps * 32) {
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int w2 = 0; w2 < kWarps; ++w2) {
            const float4 v = *reinterpret_cast<const float4*>(slabs + w2 * (8 * kD) + e4 * 4);
            acc.x += v.x; acc.y += v.y; acc.z += v.z; acc.w += v.w;
            if (kPair) {   // the remainders' part
                const float4 r = *reinterpret_cast<const float4*>(slabs + w2 * (8 * kD) + 4 * kD + e4 * 4);
                acc.x += r.x; acc.y += r.y; acc.z += r.z; acc.w += r.w;
            }
        }
        const int to = e4 / slice;
        const uint32_t bar_to = mapa(smem_u32(&sh_bar), to), dst = mapa(smem_u32(recv_o + crank * slice + (e4 - to * slice)), to);
        hand_over(dst, bar_to, acc);
    }
    for (int x = threadIdx.x; x < csize * 8; x += kWarps * 32) {
        const int hd = x & 7;
        float bm = -INFINITY, bl = 0.f;
#pragma unroll
        for (int w2 = 0; w2 < kWarps; ++w2) bm = fmaxf(bm, sh_m[w2][hd]);
#pragma unroll
        for (int w2 = 0; w2 < kWarps; ++w2) {
            const float mw = sh_m[w2][hd];
            bl += (mw == -INFINITY) ? 0.f : sh_l[w2][hd] * fast_exp2(mw - bm);
        }
        const uint32_t bar_to = mapa(smem_u32(&sh_bar), x >> 3), dst = mapa(smem_u32(recv_ml + crank * 16 + hd * 2), x >> 3);
        hand_over(dst, bar_to, bm, bl);
    }
    const int n_clusters = n_split / csize, cidx = split / csize;   // clusters of the head, this one's index
    // partials: every head's own unit in turn, then the spare units; a unit leaves one for each of its clusters
    const int per_unit = kSpares ? (int)gridDim.x / csize : n_clusters;
    const int first = bh * per_unit, more = (B * Hkv + u.begin) * per_unit;
    float* my_part = part + (size_t)(cidx + (!kSpares || cidx < per_unit ? first : more - per_unit)) * kPartStride;
    const bool direct = n_clusters == 1;   // this cluster holds the whole head: its fold is the result
    if (direct && warp > 0 && e_lo + warp * 32 >= e_hi) return;   // nothing to fold for this warp (one stays until all has arrived)
    const bool got = slices_arrived(smem_u32(&sh_bar));
    // Nothing has been written to global memory so far (the block partials live in shared memory).  Under
    // an overlapped launch every global write of this kernel (out, cluster partials, arrival counters) is
    // ordered behind the completion of the kernel before it, which ordered its own writes behind its
    // predecessor in the same way: completion is transitive along a run of overlapped launches, and they
    // may share workspace and out buffers.  (A no-op for an ordinary launch and after the wait above.)
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
    if (!got) set_status(status, SC_ERR_TIMEOUT);
    for (int e4 = e_lo + threadIdx.x; e4 < e_hi; e4 += kWarps * 32) {
        const int hd = e4 / (kD / 4), d4 = (e4 % (kD / 4)) * 4;
        const Folded f = fold_slices(recv_o, recv_ml, csize, slice, e4 - e_lo, hd, got);
        if (direct) {
            const float inv = f.l > 0.f ? 1.f / f.l : 0.f;
            store_out4(out + ((size_t)bh * G + hd) * kD + d4, f.o, inv);
        } else {
            *reinterpret_cast<float4*>(my_part + hd * kD + d4) = f.o;
            if (d4 == 0 || e4 == e_lo) { my_part[8 * kD + hd] = f.m; my_part[8 * kD + 8 + hd] = f.l; }   // (the same values from every slice of the head)
        }
    }
    if (direct && __all_sync(kFull, got)) return;   // (as good as always: 0.1 us less here than behind the code for several partials)

    // ---- several partials per head: the last block to arrive merges them, slice by slice where there are counters enough ----
    if (!direct) {
        const bool by_slice = B * Hkv * csize <= kMaxTickets;
        ticket_and_merge<kSpares>(part, first, more, per_unit, n_clusters, tickets + (by_slice ? bh * csize + crank : bh), by_slice ? n_clusters : n_clusters * csize,
                                  by_slice ? e_lo : 0, by_slice ? e_hi : G * (kD / 4), bh, G, out, &sh_last);
    }
    outlast_cluster(smem_u32(&sh_bar), got);
}

// Block split of one head: how many blocks stream it, and how they are grouped into clusters.
struct SplitPlan { int n_split, cluster; };
// Largest number of clusters of c blocks (c = 2..16) that are resident at once, two blocks per SM: fit[c].
struct Resident { int sms; int fit[kMaxCluster + 1]; };

inline int head_slots(long long heads, int cap) {   // most partials the own unit of a head can leave in global memory
    const int by_rows = (cap + 63) / 64;
    const int s = heads >= kMaxSlots ? 1 : (int)(kMaxSlots / heads);
    return s < by_rows ? s : (by_rows < 1 ? 1 : by_rows);
}
// Partials a launch can leave, the spare units' among them.  It grows with the number of heads and with the capacity, so that a
// workspace for the largest batch serves every smaller one.
inline size_t all_slots(long long heads, int cap) {
    const long long by_rows = cap < 64 ? 1 : (cap + 63) / 64, split = heads * by_rows;
    const long long several = split < kMaxSlots ? split : kMaxSlots, own = heads < kMaxTickets ? heads : kMaxTickets;
    return 2 * (size_t)(several > own ? several : own);
}

// The rules and what they were measured against (us per layer, Llama-shaped heads of 128 columns, 2 x 148 block slots; "->" is
// from a plan that took splits from the capacity alone, in several waves, and asked L2 for each block's rows in advance):
//   - one cluster per head, as wide as lets the clusters of all heads be resident at once: 128 heads x 3.4 K rows, 2 blocks
//     each, 51.6 -> 41.2; 56 heads x 6.3 K, 5, 43.7 -> 33.9; 32 x 6.3 K, 8, 31.9 -> 22.5; 24 x 12.6 K, 10, 45.7 -> 31.9; 16 x 25 K, 12,
//     47.0 -> 36.0; 8 x 34 K, 16, 40.2 -> 27.8.  More than 12 only where 16 would fit: 16 heads, for which 13 do and 14 do not, 13
//     blocks against 12: 4 to 25 K rows 1 to 2 % faster, 2.1 K rows 8.9 against 8.3.
//   - fewer blocks for short capacities, whose time is the fold and the barrier: 8 heads x 0.5 K rows of 1 K capacity: 9 blocks
//     4.5, 16 blocks 5.0; x 2.1 K of 4 K: 12 blocks 6.1, 16 blocks 6.6; from 8 K of capacity on 16.
//   - several clusters per head where few heads would leave blocks with thousands of rows: 4 heads x 34 K rows, 3 x 16, 19.7 (one: 21;
//     21.1 to 43.6 before); not below, the ticket and the merge cost 2: 4 heads x 8.5 K, one cluster 9.2, three 11.1.
//   - more heads than any cluster width fits: one block per head (256 heads x 3.4 K rows: 82.1, split in two 83.2); where they
//     are up to 15 % more than two per SM, which leaves a last round nearly empty, clusters of three (one block and three: 320
//     heads x 7 K rows 210, 176; 368 214, 204, but with 3.4 K rows 110, 120; 320 x 2 K rows of 4 K 68, 74).
//   - a cache without counts is a raw one, whose heads are mostly full: one block per SM outside clusters keeps HBM
//     busiest (32 heads x 64 K rows, 4 each, 157; 8 each in clusters 166; 8 heads x 131 K: 83.5 against 116.9).  From 75
//     heads on that is one block each; where it leaves more SMs idle in its last round than clusters of two or three would,
//     those are taken (one block and two or three: 76 heads x 8 K rows 60.7, 54.4; 88 63.3, 60.3; 176 123, 113; 200 137, 131; 320
//     232, 206; at 104 to 152 and 296 heads one block is best).
inline SplitPlan plan_for(long long heads, int cap, bool raw, const Resident& res) {
    const int by_rows = (cap + 4 * kTile - 1) / (4 * kTile);   // at least 64 rows per split
    if (raw && cap >= 8192) {
        int s = heads >= res.sms ? 1 : (int)(res.sms / heads);
        if (s == 1) {   // one block each, or a cluster of two or three where its rounds of one block per SM are a tenth fuller
            const auto rounds = [&](long long blocks) { return (blocks + res.sms - 1) / res.sms; };
            for (int w = 2; w <= 3; ++w)
                if ((heads <= res.fit[w] || 20 * heads > 21 * res.sms) && 10 * w * rounds(heads * s) > 11 * s * rounds(heads * w)) s = w;
            return {s, s};
        }
        const int slots = head_slots(heads, cap);
        s = s < 16 ? s : 16 * (s / 16);
        if (s > slots) s = slots;
        return {s, s == 2 && heads <= res.fit[2] ? 2 : 1};
    }
    int limit = 8 + cap / 1024;
    if (limit > by_rows) limit = by_rows;
    if (limit > kMaxCluster) limit = kMaxCluster;
    int c = 1;
    for (int w = 2; w <= limit; ++w)
        if (heads <= res.fit[w] && (w <= 12 || heads <= res.fit[kMaxCluster])) c = w;
    if (heads > 2 * res.sms && 20 * heads <= 46 * res.sms && cap >= 8192) c = 3;
    if (c < kMaxCluster) return {c, c};
    int k = (cap + kMaxCluster * kCapRowsPerBlock - 1) / (kMaxCluster * kCapRowsPerBlock);   // clusters per head
    if (k > res.fit[c] / heads) k = (int)(res.fit[c] / heads);
    const int slots = head_slots(heads, cap);
    if (k > slots) k = slots;
    return {c * (k < 1 ? 1 : k), c};
}

// Spare units (plan_units) for a batch whose blocks may otherwise get thousands of rows to stream.  Among equal heads they cost
// 0.3 to 0.7 us (16 x 8 heads of 8 K capacity 42.9 -> 43.4; raw, 8 K rows, 40 to 72 heads up to 7 %); wide clusters find no room beside
// the others and come last (4 x 8 heads of 13 K, eight blocks each, 13.7 -> 14.4), so they need more rows to be worth it.  One
// sequence long, the others short, 16 x 8 heads: 32 K of 32 K 134 -> 43 us, 4 K of 4 K 22.6 -> 18.9, raw 32 K 220 -> 57; 4 x 8 heads,
// 32 K 46.7 -> 33.8.  Not for two sequences, whose longer one can only gain half (34.8 -> 34.3), and for heads of one block each only
// from 8 K on (344 heads x 2 K of 4 K 69.5 -> 71.4).
inline bool has_spares(int B, int Hkv, int cap, int n_split, bool raw) {
    return B > 2 && (long long)B * Hkv <= kMaxTickets && cap >= (n_split == 1 ? 8192 : 4096) && cap > (raw || n_split <= 2 ? 1024 : 2048) * n_split;
}

}  // namespace dm

bool decode_mma_supported(const DecodeArgs& a) {
    return a.dt == SC_BF16 && a.d == dm::kD && (a.Hq / a.Hkv) <= 8 && a.cap > 0 && a.Hkv <= 65535 && a.B <= 65535;
}

// Bytes at the front of the workspace that hold the arrival counters (zero between calls): the same for every shape, so that
// no call's partials lie where another one's counters are.
size_t decode_mma_counter_bytes() { return sizeof(int32_t) * dm::kMaxTickets; }

size_t decode_mma_ws_bytes(int32_t B, int32_t Hq, int32_t Hkv, int32_t d, int32_t cap) {
    (void)Hq; (void)d;
    // arrival counters (zero between calls) + partials
    return 256 + decode_mma_counter_bytes() + sizeof(float) * dm::all_slots((long long)B * Hkv, cap) * dm::kPartStride;
}

cudaError_t launch_decode_mma(const DecodeArgs& a, cudaStream_t st) {
    // per device: SM count, the opt-ins, and how many clusters of each width can be resident at once
    static dm::Resident res_of[64];
    static std::once_flag once_of[64];
    int dev = 0;
    cudaGetDevice(&dev);
    dev &= 63;
    dm::Resident& res = res_of[dev];
    std::call_once(once_of[dev], [&res, dev] {
        int v = 0;
        cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
        res.sms = v < 1 ? 1 : v;
        bool wide = true;
        for (auto kernel : {dm::decode_mma_kernel<false, false>, dm::decode_mma_kernel<true, false>, dm::decode_mma_kernel<false, true>,
                            dm::decode_mma_kernel<true, true>}) {
            cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, dm::kSmemBytes);
            wide = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess && wide;
        }
        for (int c = 2; c <= dm::kMaxCluster; ++c) {
            cudaLaunchConfig_t probe = {};
            probe.gridDim = dim3(c, 1, 1);
            probe.blockDim = dim3(dm::kWarps * 32);
            probe.dynamicSmemBytes = dm::kSmemBytes;
            cudaLaunchAttribute pa[1];
            pa[0].id = cudaLaunchAttributeClusterDimension;
            pa[0].val.clusterDim.x = c; pa[0].val.clusterDim.y = 1; pa[0].val.clusterDim.z = 1;
            probe.attrs = pa;
            probe.numAttrs = 1;
            int n_clusters = 0;
            res.fit[c] = 0;
            if ((c <= 8 || wide) && cudaOccupancyMaxActiveClusters(&n_clusters, dm::decode_mma_kernel<false, false>, &probe) == cudaSuccess) res.fit[c] = n_clusters;
        }
        (void)cudaGetLastError();   // a refused opt-in or probe is not an error of this call
    });
    const dm::SplitPlan plan = dm::plan_for((long long)a.B * a.Hkv, a.cap, a.count == nullptr, res);
    int32_t* tickets = (int32_t*)a.ws;
    float* part = (float*)((char*)a.ws + decode_mma_counter_bytes());
    const float scale = (a.scale == 0.f ? 1.f / sqrtf((float)a.d) : a.scale) * 1.4426950408889634f;
    cudaLaunchConfig_t cfg = {};
    const bool spares = dm::has_spares(a.B, a.Hkv, a.cap, plan.n_split, a.count == nullptr);
    cfg.gridDim = dim3(plan.n_split, a.Hkv, spares ? 2 * a.B : a.B);
    cfg.blockDim = dim3(dm::kWarps * 32);
    cfg.dynamicSmemBytes = dm::kSmemBytes;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = plan.cluster; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    const int mode = (a.flags & SC_FLAG_OVERLAP_CHAIN) ? dm::kChained : (a.flags & SC_FLAG_OVERLAP_PREV) ? dm::kOverlapped : dm::kOrdinary;
    const bool pair = a.Hq / a.Hkv <= 4;
    const auto kernel = spares ? (pair ? dm::decode_mma_kernel<true, true> : dm::decode_mma_kernel<true, false>)
                               : (pair ? dm::decode_mma_kernel<false, true> : dm::decode_mma_kernel<false, false>);
    note_launches(1);
    return own_error(cudaLaunchKernelEx(&cfg, kernel, (const __nv_bfloat16*)a.q, a.Hq, a.Hkv,
                                        (const __nv_bfloat16*)a.core_k, (const __nv_bfloat16*)a.core_v, a.count, a.cap,
                                        a.core_len, scale, a.B, mode, (__nv_bfloat16*)a.out, part, tickets, a.status));
}

}  // namespace sc
