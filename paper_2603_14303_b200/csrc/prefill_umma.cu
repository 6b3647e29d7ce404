// Multi-query Proportional Attention (Sec. 2.4, Eq. 4 as printed, with a block of m queries per head):
//     O = softmax(Q K_c^T * scale + ln s) V_c      Q: [m, d] per query head, K_c/V_c: the head's cores
// for chunked prefill or speculative decoding over a compressed cache.  Unlike the one-query decode
// step this is a dense contraction: the G query heads that share a KV head times the m queries give
// G*m rows against the same cores, so it runs on the tcgen05 tensor cores (bf16, d = 128):
//   one CTA = 128 query rows of one (sequence, KV head), walking the head's cores 128 at a time;
//   warps 0, 2 TMA: the query tile once, then K and V tiles into rings of three (128-byte swizzle); warp 2 log2(count) too;
//   warp 1     issues the MMAs: S = Q K^T into one of three score buffers in tensor memory (three tiles ahead
//              of the weighted sum), then O += P V with P read from tensor memory and V as an MN-major
//              operand straight from its [keys x dims] tile;
//   warps 4-19 softmax, two groups of eight warps that take the key tiles in turn (one, warps 4-11, where there is one tile), two threads per query row
//              (= tensor-memory lane; each owns half of the tile's keys):
//              x = S * scale*log2(e) + log2(count), masks (head length, optional causal tail), P = 2^(x - m) as a bf16 pair
//              (leading part + remainder) written back over the scores it came from: the 32 fp32 columns of a chunk of scores
//              become 16 columns of packed leading parts and 16 of remainders, so P never touches shared memory.
//              The row's reference m is raised lazily (the accumulator row is rescaled in tensor memory only then; the
//              tile's maximum is taken as a bound: largest raw product * scale + largest log2(count) of the tile) and is
//              settled tile by tile: a group looks at its tile's maxima, waits until the other has settled the tile before,
//              settles its own and goes on to the weights beside the other group; finally O / l -> bf16 -> global.
// When the launch has too few CTAs to fill the GPU (few query rows: speculative decoding, short chunks), the keys
// of a head are split over the CTAs of a thread-block cluster: each walks its share of the key tiles, leaves its
// unnormalised (m, l, O) in its own shared memory, and after a cluster barrier every CTA folds a slice of the
// query rows out of all members' shared memory (distributed shared memory) and writes that slice of the output.
// What bounds it: shared memory.  A key tile's operands (64 KB for the scores, twice 32 KB for the pair of weights) and its copies
// (64 KB) are 1536 clocks at 128 bytes, and the tensor cores need 1632; the MMA warp is busy 2300 of the 2530 clocks a tile takes.
// 4 layers x 512 causal queries per head over 8.5 K cores 520 -> 467 us, one layer x 256 65 -> 54 against two score buffers and eight
// softmax warps on one tile at a time, whose softmax (3500 clocks with one warp-instruction every 3 clocks per scheduler) was
// the bound.  Two query tiles per CTA with a score buffer and an accumulator each: 480; the same with a 64-key
// double buffer 562.  MMAs issued by a branch of one thread take 62 clocks each, by an elected lane of a converged warp 27.
// Cluster width: as many CTAs per query tile as let every cluster of the launch be resident at once (asked of the
// occupancy query: on this GPU 15 clusters of 8 or 9, 11 of 10, 7 of 11 to 16); powers of two up to 8 before.  8 queries per
// head, 8 KV heads: 10 instead of 8 CTAs, 29 -> 24 us per layer with the above (four replicas of the rows, see kRep: 19); 16 clusters: 7 instead of 8 (which took
// two waves), 64 queries per head 190 -> 132 us for 4 layers.
// Every wait is bounded; a wait that gives up is reported through the status word.
// A CUDA-core kernel (one warp per query) serves other dtypes and head sizes.
#include <cooperative_groups.h>

#include <algorithm>
#include <mutex>
#include <type_traits>

#include "common.cuh"
#include "umma.cuh"

namespace sc {

namespace pf {

using namespace umma;
namespace cg = cooperative_groups;

constexpr int kT = 128;                       // query rows per CTA, keys per tile
constexpr int kHalf = kT * 128;               // 16384 bytes: one 64-column half of a [128 x 128] bf16 tile
constexpr int kTile = 2 * kHalf;              // 32768
constexpr int kTmemCols = 512;                // S0 | S1 | S2 | O (128 columns each; P overwrites S in place)
constexpr int kColS = 0, kColO = 384;
constexpr int kStages = 3;                    // K and V rings, score buffers
constexpr int kSmQ = 0, kSmK = kTile, kSmV = (1 + kStages) * kTile, kSmLc = (1 + 2 * kStages) * kTile, kSmMx = kSmLc + kStages * kT * 4,
              kSmBar = kSmMx + 2 * kT * 4;
constexpr int kSmemBytes = kSmBar + 304;
constexpr int kMaxSplit = 16;                 // CTAs that share one query tile: a cluster (more than 8 needs the non-portable opt-in)
constexpr float kMaxSlack = 8.f;              // log2 units a score may exceed the running maximum before it is raised
static_assert(kSmemBytes <= 232448, "shared memory of one CTA");

struct Params {
    CUtensorMap map_q, map_k, map_v;          // rows x 128 bf16, boxes of 128 rows x 64 columns
    const int32_t* count; const int32_t* core_len;
    __nv_bfloat16* out;
    int Hq, Hkv, m, cap, causal, n_split;   // n_split: CTAs (= cluster size) that share the keys of one query tile
    float scale_log2;
    int32_t* status;
};

__device__ __forceinline__ float ex2(float x) { float y; asm("ex2.approx.ftz.f32 %0, %1;\n" : "=f"(y) : "f"(x)); return y; }
__device__ __forceinline__ float lg2(float x) { float y; asm("lg2.approx.ftz.f32 %0, %1;\n" : "=f"(y) : "f"(x)); return y; }
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
        "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};\n"
        ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
          "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]),
          "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]),
          "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
        : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t (&r)[8]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};\n"
                 ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]) : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};\n"
        ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
          "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
}
// D[tmem] (+)= A[tmem] * B[smem]: A's rows are tensor-memory lanes, two 16-bit elements of the contraction
// axis per 32-bit column; a whole converged warp calls it, one elected lane issues.
__device__ __forceinline__ void mma_bf16_ts_warp(uint32_t tmem_d, uint32_t tmem_a, uint64_t bdesc, uint32_t idesc, bool accumulate) {
    asm volatile("{\n.reg .pred p, e;\nelect.sync _|e, 0xffffffff;\nsetp.ne.b32 p, %4, 0;\n@e tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n"
                 ::"r"(tmem_d), "r"(tmem_a), "l"(bdesc), "r"(idesc), "r"((uint32_t)accumulate) : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory"); }
__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}
// r0 = w0 - low bf16 of ph, r1 = w1 - high bf16 of ph, with the mixed-precision fma (the bf16 operands are taken
// as they are: (-1) * h + w, one rounding -- what unpacking and subtracting gives, in half the instructions).
__device__ __forceinline__ void remainders(uint32_t ph, float w0, float w1, float& r0, float& r1) {
    asm("{\n.reg .b16 lo, hi, m1;\nmov.b32 {lo, hi}, %2;\nmov.b16 m1, 0xBF80;\n"
        "fma.rn.f32.bf16 %0, lo, m1, %3;\nfma.rn.f32.bf16 %1, hi, m1, %4;\n}\n"
        : "=f"(r0), "=f"(r1) : "r"(ph), "f"(w0), "f"(w1));
}

__device__ __forceinline__ float max3(float a, float b, float c) {
    float y;
    asm("max.f32 %0, %1, %2, %3;\n" : "=f"(y) : "f"(a), "f"(b), "f"(c));
    return y;
}
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
    float2 y;
    asm("{\n.reg .b64 a, b, y;\nmov.b64 a, {%2, %3};\nmov.b64 b, {%4, %5};\nadd.rn.f32x2 y, a, b;\nmov.b64 {%0, %1}, y;\n}\n"
        : "=f"(y.x), "=f"(y.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return y;
}

// kRep: how often the query rows stand in the tile's 128 lanes.  Up to 32 (64) rows they do so four times (twice), and each
// replica takes a quarter (half) of every key tile -- its weights of the other keys are zero --, so that all softmax warps work
// and a thread has 16 (32) scores a tile instead of 64; the replicas are folded at the end like the CTAs of a split.
// kGroups: groups of softmax warps, one or two.
template <int kRep, int kGroups>
__global__ void __launch_bounds__(128 + 256 * kGroups, 1) prefill_umma_kernel(const __grid_constant__ Params p) {
    extern __shared__ __align__(1024) unsigned char smem[];   // the swizzle pattern repeats every 1024 bytes
    const int n_split = p.n_split, split = blockIdx.x % n_split;   // the CTAs of a cluster are consecutive in x
    const int qt = blockIdx.x / n_split, h = blockIdx.y, b = blockIdx.z;
    const int G = p.Hq / p.Hkv, bh = b * p.Hkv + h;
    const int rows_total = G * p.m;                           // query rows of this (sequence, KV head)
    const uint32_t sbase = smem_u32(smem);
    float* lc_s = reinterpret_cast<float*>(smem + kSmLc);     // [3][128] log2(count) of a tile's keys
    const uint32_t bar0 = sbase + kSmBar;
    // three of each, by key tile: K, V, log2(count) landed; K spent; scores ready; weights ready; weights (and V) spent, O holds the tile
    const uint32_t q_full = bar0, k_full0 = bar0 + 8, v_full0 = bar0 + 32, lc_full0 = bar0 + 56, k_empty0 = bar0 + 80, s_full0 = bar0 + 104,
                   p_full0 = bar0 + 128, pv_done0 = bar0 + 152, ref0 = bar0 + 176;   // ref: [4 x 32 rows][tile & 1] the tile's reference is settled
    float* lcm_s = reinterpret_cast<float*>(smem + kSmBar + 240);                      // [3] largest log2(count) of a tile
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem + kSmBar + 252);
    volatile int* sh_fail = reinterpret_cast<volatile int*>(smem + kSmBar + 256);
    volatile int* sh_issued = reinterpret_cast<volatile int*>(smem + kSmBar + 260);   // key tiles whose K, and whose V, was requested
    volatile int* sh_fail_pair = reinterpret_cast<volatile int*>(smem + kSmBar + 268);   // [8] set by the two warps of 32 rows of a group

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (warp == 0) {
        if (lane < 30) mbar_init(bar0 + 8 * lane, lane >= 22 ? 2 : lane >= 16 && lane < 19 ? 8 : 1);   // ref: a row's two warps; weights: a group's eight
        mbar_fence_init();
        if (lane < 8) sh_fail_pair[lane] = 0;
        if (lane == 0) { *sh_fail = 0; sh_issued[0] = 0; sh_issued[1] = 0; }
    } else if (warp == 2 && lane < 3) {
        prefetch_map(lane == 0 ? &p.map_q : lane == 1 ? &p.map_k : &p.map_v);
    }
    if (warp == 1) tmem_alloc(sbase + kSmBar + 252, kTmemCols);
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const uint32_t tmem = *tmem_slot;

    in_stream_order();   // everything above needs nothing from the kernel before
    const int len = max(min(p.core_len[bh], p.cap), 0);
    const int nt_all = (len + kT - 1) / kT;                   // key tiles of the head
    const int per_split = (nt_all + n_split - 1) / n_split;
    const int t_lo = min(split * per_split, nt_all);          // this CTA's tiles: [t_lo, t_lo + nt)
    const int nt = min(t_lo + per_split, nt_all) - t_lo;
    const long long q_row0 = ((long long)b * p.Hq + (long long)h * G) * p.m + (long long)qt * kT;
    if ((sbase & 1023u) != 0u) {   // the swizzled addressing assumes this; uniform over the block
        if (tid == 0) set_status(p.status, SC_ERR_CUDA);
        __syncthreads();
        if (warp == 1) tmem_dealloc(tmem, kTmemCols);
        return;
    }
    if (warp == 0) {
        if (lane == 0 && nt > 0) {   // ---- TMA producer: queries and keys (a key tile's place is free long before a value tile's) ----
            mbar_expect_tx(q_full, kTile);
            for (int c = 0; c < kRep; ++c) {   // (boxes of 128 / kRep rows)
                tma_load_4d(sbase + kSmQ + c * (kHalf / kRep), &p.map_q, 0, (int)q_row0, 0, 0, q_full);
                tma_load_4d(sbase + kSmQ + kHalf + c * (kHalf / kRep), &p.map_q, 64, (int)q_row0, 0, 0, q_full);
            }
            for (int t = 0; t < nt; ++t) {
                const int s = t % kStages, round = t / kStages, at = bh * p.cap + (t_lo + t) * kT;
                if (round > 0 && !mbar_wait(k_empty0 + 8 * s, (round - 1) & 1)) { *sh_fail = 1; break; }
                mbar_expect_tx(k_full0 + 8 * s, kTile);
                tma_load_4d(sbase + kSmK + s * kTile, &p.map_k, 0, at, 0, 0, k_full0 + 8 * s);
                tma_load_4d(sbase + kSmK + s * kTile + kHalf, &p.map_k, 64, at, 0, 0, k_full0 + 8 * s);
                sh_issued[0] = t + 1;
            }
        }
    } else if (warp == 2) {
        // ---- TMA producer: values; and log2(count) of the tile's keys, whose counts are requested a tile ahead ----
        const int32_t* cnt = p.count ? p.count + (size_t)bh * p.cap : nullptr;
        int c[4];
        auto request_counts = [&](int t) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int j = (t_lo + t) * kT + u * 32 + lane;
                c[u] = cnt != nullptr && t < nt && j < len ? cnt[j] : 1;
            }
        };
        request_counts(0);
        for (int t = 0; t < nt; ++t) {
            const int s = t % kStages, round = t / kStages, at = bh * p.cap + (t_lo + t) * kT;
            // (when the weighted sum of the tile before in this place is complete, its counts have been read as well)
            if (round > 0 && !__all_sync(kFull, mbar_wait(pv_done0 + 8 * s, (round - 1) & 1))) { *sh_fail = 1; break; }
            if (lane == 0) {
                mbar_expect_tx(v_full0 + 8 * s, kTile);
                tma_load_4d(sbase + kSmV + s * kTile, &p.map_v, 0, at, 0, 0, v_full0 + 8 * s);
                tma_load_4d(sbase + kSmV + s * kTile + kHalf, &p.map_v, 64, at, 0, 0, v_full0 + 8 * s);
                sh_issued[1] = t + 1;
            }
            int top = 0;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float lc = lg2((float)max(c[u], 1));
                lc_s[s * kT + u * 32 + lane] = lc;
                top = max(top, __float_as_int(lc));   // lc >= 0: the bits order like the values
            }
            top = __reduce_max_sync(kFull, top);
            if (lane == 0) lcm_s[s] = __int_as_float(top);
            __syncwarp();
            if (lane == 0) mbar_arrive(lc_full0 + 8 * s);
            request_counts(t + 1);
        }
    } else if (warp == 1) {
        if (nt > 0) {   // ---- MMA issuer (the whole warp, one elected lane) ----
            constexpr uint32_t idesc_qk = instr_desc_bf16(kT, kT, false, false);   // Q and K both K-major
            constexpr uint32_t idesc_pv = instr_desc_bf16(kT, kT, false, true);    // P K-major (tensor memory), V MN-major
            const auto arrived = [&](uint32_t bar, int parity) { return __all_sync(kFull, mbar_wait(bar, parity & 1)); };
            auto issue_qk = [&](int s) {   // S = Q K^T
                const uint64_t qd = smem_desc_sw128(sbase + kSmQ, 16, 1024), kd = smem_desc_sw128(sbase + kSmK + s * kTile, 16, 1024);
#pragma unroll
                for (int ks = 0; ks < 8; ++ks) {
                    const uint32_t off = ((ks >> 2) * kHalf + (ks & 3) * 32) >> 4;
                    mma_bf16_ss_warp(tmem + kColS + s * kT, qd + off, kd + off, idesc_qk, ks > 0);
                }
                mma_commit_warp(k_empty0 + 8 * s);
                mma_commit_warp(s_full0 + 8 * s);
            };
            bool ok = arrived(q_full, 0);
            for (int t = 0; t < min(nt, kStages) && ok; ++t) {
                ok = arrived(k_full0 + 8 * t, 0);
                if (!ok) break;
                fence_after_sync();
                issue_qk(t);
            }
            for (int t = 0; t < nt && ok; ++t) {
                const int s = t % kStages, round = t / kStages;
                ok = arrived(v_full0 + 8 * s, round) && arrived(p_full0 + 8 * s, round);   // the weights of tile t are in tensor memory
                if (!ok) break;
                fence_after_sync();
                const uint64_t vd = smem_desc_sw128(sbase + kSmV + s * kTile, kHalf, 1024);   // MN-major, 16 key rows a step
                const uint32_t pcol = tmem + kColS + s * kT;
#pragma unroll
                for (int ks = 0; ks < 8; ++ks) {   // sixteen keys per instruction: eight packed columns of P
                    const uint32_t pa = pcol + (ks >> 1) * 32 + (ks & 1) * 8;                  // leading parts; remainders 16 columns on
                    mma_bf16_ts_warp(tmem + kColO, pa, vd + ((ks * 16 * 128) >> 4), idesc_pv, t > 0 || ks > 0);
                    mma_bf16_ts_warp(tmem + kColO, pa + 16, vd + ((ks * 16 * 128) >> 4), idesc_pv, true);
                }
                mma_commit_warp(pv_done0 + 8 * s);   // P of this buffer and V of this stage are spent, O holds tile t
                if (t + kStages < nt) {   // the scores three tiles ahead go where this tile's scores and weights were
                    ok = arrived(k_full0 + 8 * s, round + 1) && arrived(pv_done0 + 8 * s, round);
                    if (!ok) break;
                    fence_after_sync();
                    issue_qk(s);
                }
            }
            if (!ok && lane == 0) *sh_fail = 1;
        }
    } else if (warp >= 4) {
        // ---- softmax: warps 4-11 take the even key tiles, warps 12-19 the odd ones (one group: all); two threads per query row (= tensor-memory
        //      lane), each owning half of a tile's keys (of the replica's share) ----
        const int grp = kGroups == 1 ? 0 : (warp - 4) >> 3, q = warp & 3, r = q * 32 + lane, wg = ((warp - 4) >> 2) & 1;
        constexpr int kRows = kT / kRep, kKeys = 64 / kRep;   // rows of a replica; keys of a tile per thread
        constexpr int kHold = kKeys > 32 ? 32 : kKeys;        // scores kept in registers (the others are read again)
        const int col0 = (r / kRows) * kRows + wg * kKeys;    // the first of them (a replica has as many keys as rows)
        const int row = qt * kT + r % kRows;                  // row among the G*m of this head group
        const bool row_ok = row < rows_total;
        const int qi = row % p.m;                             // which of the m queries
        const int vis = p.causal ? len - (p.m - 1 - qi) : len;   // keys this row sees: [0, vis)
        const uint32_t lane_addr = tmem + ((uint32_t)(q * 32) << 16);
        const int pair = grp * 4 + q;                         // the two warps of these 32 rows in this group
        float* ref_s = reinterpret_cast<float*>(smem + kSmMx);      // [128] the rows' references
        float* mx_s = ref_s + kT;                                   // [128] a maximum on its way, where a reference is raised
        float m_mine = -INFINITY, l_run = 0.f;                // l_run: the weights of this thread's keys, relative to m_mine
        bool failed = false;
        const bool idle = qt * kT + (q * 32) % kRows >= rows_total;     // none of the warp's rows exists: it only keeps step
        const float2 scale2 = make_float2(p.scale_log2, p.scale_log2);
        const auto pair_sync = [&] { asm volatile("bar.sync %0, 64;\n" ::"r"(1 + pair) : "memory"); };
        const auto pair_any = [&](bool mine) {
            uint32_t out;
            asm volatile("{\n.reg .pred p, r;\nsetp.ne.u32 p, %1, 0;\nbarrier.cta.red.or.pred r, %2, 64, p;\nselp.u32 %0, 1, 0, r;\n}\n"
                         : "=r"(out) : "r"(mine ? 1u : 0u), "r"(1 + pair) : "memory");
            return out != 0u;
        };
        for (int t = grp; t < nt; t += kGroups) {
            const int s = t % kStages, round = t / kStages, j0 = (t_lo + t) * kT, jw = j0 + col0;   // jw: first key of this thread
            const uint32_t s_addr = lane_addr + kColS + s * kT + col0;
            bool lost = !mbar_wait(s_full0 + 8 * s, round & 1) || !mbar_wait(lc_full0 + 8 * s, round & 1);
            __syncwarp();
            fence_after_sync();
            // pass 1: the largest raw product of the thread's keys.  That times the scale plus the tile's largest log2(count) bounds
            // its largest score: any reference at or above the true maximum serves the softmax, and this one is at most log2 of
            // the largest count above it.  (A scale that is not positive takes the smallest product.)
            uint32_t g[kHold];
            const bool all_seen = __all_sync(kFull, jw + kKeys <= vis);   // none of these keys is masked for any row of the warp
            float mx = -INFINITY;
            if (!idle) {
#pragma unroll
                for (int c = kKeys / kHold - 1; c >= 0; --c) {   // (the first piece stays in registers, the other is read again)
                    if constexpr (kHold == 16) tmem_ld16(s_addr, g);
                    else tmem_ld32(s_addr + c * 32, g);
                    tmem_ld_wait();
                    if (!(p.scale_log2 > 0.f)) {
#pragma unroll
                        for (int k = 0; k < kHold; ++k)
                            if (jw + c * 32 + k < vis) mx = fmaxf(mx, -__uint_as_float(g[k]));
                    } else if (all_seen) {
                        float m4[4] = {mx, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
                        for (int k = 0; k < kHold; k += 8)
#pragma unroll
                            for (int x = 0; x < 4; ++x) m4[x] = max3(m4[x], __uint_as_float(g[k + x]), __uint_as_float(g[k + 4 + x]));
                        mx = fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3]));
                    } else {
#pragma unroll
                        for (int k = 0; k < kHold; ++k)
                            if (jw + c * 32 + k < vis) mx = fmaxf(mx, __uint_as_float(g[k]));
                    }
                }
                if (mx != -INFINITY) mx = fmaf(mx, fabsf(p.scale_log2), lcm_s[s]);
            }
            // Rows of the stage past the head's end hold whatever lies behind the cores (0 * NaN would poison
            // the second product): this row's threads clear its V row.  K rows need nothing, their scores are masked.
            if (j0 + kT > len) {
                lost = !mbar_wait(v_full0 + 8 * s, round & 1) || lost;
                if (j0 + r >= len) {
#pragma unroll
                    for (int u = 0; u < 8; ++u)
                        *reinterpret_cast<uint4*>(smem + kSmV + s * kTile + wg * kHalf + r * 128 + u * 16) = make_uint4(0u, 0u, 0u, 0u);
                }
                fence_async_proxy();   // for the tensor core's reads
                __syncwarp();
            }
            // The row's reference is settled tile by tile, by either group in its turn: the tile before has settled its own.
            if (t > 0) lost = !mbar_wait(ref0 + 16 * q + 8 * ((t - 1) & 1), ((t - 1) >> 1) & 1) || lost;
            float m = t > 0 ? ref_s[r] : -INFINITY;
            if (lost) { *sh_fail = 1; sh_fail_pair[pair] = 1; }
            if (t == 0) (wg == 0 ? mx_s : ref_s)[r] = mx;       // (there is no reference to read yet)
            const bool raise_any = pair_any(!idle && mx > m + kMaxSlack);   // also the first finite score (m = -inf)
            if (sh_fail_pair[pair]) { failed = true; break; }
            if (raise_any) {
                if (t > 0) {
                    (wg == 0 ? mx_s : ref_s)[r] = mx;           // (both threads of the row have read the reference, nobody else does yet)
                    pair_sync();
                }
                mx = fmaxf(mx, (wg == 0 ? ref_s : mx_s)[r]);
                const bool raise = mx > m + kMaxSlack;          // same in the row's two threads
                const float f = raise ? ex2(m - mx) : 1.f;      // 0 when nothing had been seen
                if (raise) m = mx;
                if (wg == 0) ref_s[r] = m;
                // the accumulator may be touched only between two weighted sums: the one before must be complete (this tile's
                // cannot start before this warp has handed in its weights)
                if (t > 0 && !idle) {
                    if (!mbar_wait(pv_done0 + 8 * ((t - 1) % kStages), ((t - 1) / kStages) & 1)) { *sh_fail = 1; sh_fail_pair[pair] = 1; }
                    __syncwarp();
                    fence_after_sync();
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        uint32_t o[16];
                        tmem_ld16(lane_addr + kColO + wg * 64 + c * 16, o);
                        tmem_ld_wait();
#pragma unroll
                        for (int k = 0; k < 16; ++k) o[k] = __float_as_uint(__uint_as_float(o[k]) * f);
                        tmem_st16(lane_addr + kColO + wg * 64 + c * 16, o);
                    }
                    tmem_st_wait();
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(ref0 + 16 * q + 8 * (t & 1));
            if (!idle) {
                if (m != m_mine) {   // the row sum follows the reference
                    l_run = m_mine == -INFINITY ? 0.f : l_run * ex2(m_mine - m);
                    m_mine = m;
                }
                if (kRep > 1) {   // the weights of the other replicas' keys
                    const uint32_t zero[16] = {0u};
#pragma unroll
                    for (int c = kRows; c < kT; c += 32) tmem_st16(lane_addr + kColS + s * kT + (((r / kRows) * kRows + c) & (kT - 1)) + wg * 16, zero);
                }
                // pass 2: weights, as bf16 pairs (leading part + remainder), back into the score buffer's columns: the 32 score
                // columns of a chunk become 16 columns of packed leading parts and 16 of remainders
                const float mref = m == -INFINITY ? 0.f : m;
                const float2 nref2 = make_float2(-mref, -mref);
                // (the row sum takes the weights before the split: the pair carries sixteen bits of each, the difference
                // is below 2^-17 of the sum)
                float2 l2[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
                for (int c = 0; c < kKeys / 16; ++c) {
                    if (kKeys > kHold && c == kHold / 16) {
                        if constexpr (kHold == 32) tmem_ld32(s_addr + 32, g);
                        tmem_ld_wait();
                    }
                    uint32_t hi[8], lo[8];
#pragma unroll
                    for (int k = 0; k < 16; k += 4) {
                        const float4 lc = *reinterpret_cast<const float4*>(lc_s + s * kT + col0 + c * 16 + k);
                        const uint32_t* gk = g + (c * 16) % kHold + k;
                        const float2 x0 = add2(fma2(make_float2(__uint_as_float(gk[0]), __uint_as_float(gk[1])), scale2, make_float2(lc.x, lc.y)), nref2);
                        const float2 x1 = add2(fma2(make_float2(__uint_as_float(gk[2]), __uint_as_float(gk[3])), scale2, make_float2(lc.z, lc.w)), nref2);
                        float2 w0 = make_float2(ex2(x0.x), ex2(x0.y)), w1 = make_float2(ex2(x1.x), ex2(x1.y));
                        if (!all_seen) {
                            const int j = jw + c * 16 + k;
                            w0.x = j < vis ? w0.x : 0.f; w0.y = j + 1 < vis ? w0.y : 0.f;
                            w1.x = j + 2 < vis ? w1.x : 0.f; w1.y = j + 3 < vis ? w1.y : 0.f;
                        }
                        l2[0] = add2(l2[0], w0); l2[1] = add2(l2[1], w1);
                        const uint32_t p0 = pack2(w0.x, w0.y), p1 = pack2(w1.x, w1.y);
                        float r0, r1, r2, r3;
                        remainders(p0, w0.x, w0.y, r0, r1);
                        remainders(p1, w1.x, w1.y, r2, r3);
                        hi[k >> 1] = p0; hi[(k >> 1) + 1] = p1;
                        lo[k >> 1] = pack2(r0, r1); lo[(k >> 1) + 1] = pack2(r2, r3);
                    }
                    // (sixteen keys: half a chunk of 32 columns, which the two threads of a row share where there are four replicas)
                    const uint32_t at = lane_addr + kColS + s * kT + (col0 & ~31) + (c >> 1) * 32 + ((kRep == 4 ? wg : c) & 1) * 8;
                    tmem_st8(at, hi);
                    tmem_st8(at + 16, lo);
                }
                l_run += (l2[0].x + l2[0].y) + (l2[1].x + l2[1].y);
                tmem_st_wait();
            }
            fence_before_sync();      // this thread's accesses to tensor memory
            __syncwarp();
            if (lane == 0) mbar_arrive(p_full0 + 8 * s);
        }
        // ---- O / l -> bf16 -> global: each thread 32 (one group: 64) columns of its row; l is the sum of the row's four (two) partial sums ----
        // The group that took the last tile waits for the last weighted sum.  (The other one could not: while the sum three tiles
        // before is not complete, the parity of that place's barrier reads as if the last one were.)  It knows through rows_sync.
        if (nt > 0 && !failed && grp == (nt - 1) % kGroups) {
            if (!__all_sync(kFull, mbar_wait(pv_done0 + 8 * ((nt - 1) % kStages), ((nt - 1) / kStages) & 1))) { *sh_fail = 1; sh_fail_pair[pair] = 1; }
            fence_after_sync();
            fence_before_sync();
        }
        const auto rows_sync = [&] { asm volatile("bar.sync %0, %1;\n" ::"r"(9 + q), "n"(64 * kGroups) : "memory"); };   // the warps of these 32 rows
        rows_sync();   // the last reference is settled, O is complete
        fence_after_sync();
        const bool ok = nt > 0 && !sh_fail_pair[q] && !sh_fail_pair[4 + q];
        const float m_row = nt > 0 ? ref_s[r] : -INFINITY;
        float* ls_s = reinterpret_cast<float*>(smem + kSmK + 2 * kTile);   // [2 kGroups][128] (all keys are spent)
        ls_s[(grp * 2 + wg) * kT + r] = m_mine == -INFINITY ? 0.f : l_run * ex2(m_mine - m_row);
        rows_sync();
        const float l_row = kGroups == 1 ? ls_s[r] + ls_s[kT + r] : (ls_s[r] + ls_s[kT + r]) + (ls_s[2 * kT + r] + ls_s[3 * kT + r]);
        constexpr int kOut = 64 / kGroups;   // columns of a thread
        const int ocol = (grp * 2 + wg) * kOut;
        uint32_t o[kOut];
        if (ok) {
#pragma unroll
            for (int c = 0; c < kOut; c += 32) tmem_ld32(lane_addr + kColO + ocol + c, *reinterpret_cast<uint32_t(*)[32]>(&o[c]));
            tmem_ld_wait();
        } else {
#pragma unroll
            for (int k = 0; k < kOut; ++k) o[k] = 0u;
        }
        if (kRep == 1 && n_split == 1) {
            __nv_bfloat16* orow = p.out + (size_t)(q_row0 + r) * 128 + ocol;
            const float inv = l_row > 0.f ? 1.f / l_row : 0.f;
            if (row_ok) {
#pragma unroll
                for (int u = 0; u < kOut / 8; ++u) {
                    uint4 v;
                    v.x = pack2(__uint_as_float(o[8 * u]) * inv, __uint_as_float(o[8 * u + 1]) * inv);
                    v.y = pack2(__uint_as_float(o[8 * u + 2]) * inv, __uint_as_float(o[8 * u + 3]) * inv);
                    v.z = pack2(__uint_as_float(o[8 * u + 4]) * inv, __uint_as_float(o[8 * u + 5]) * inv);
                    v.w = pack2(__uint_as_float(o[8 * u + 6]) * inv, __uint_as_float(o[8 * u + 7]) * inv);
                    *reinterpret_cast<uint4*>(orow + u * 8) = v;
                }
            }
        } else {
            // this CTA's share of the keys: unnormalised O, m and l into its own shared memory (the K ring is spent)
            float* part_o = reinterpret_cast<float*>(smem + kSmK);      // [128 rows][32 float4], float4 index ^ (row & 31)
            float* part_ml = reinterpret_cast<float*>(smem + kSmV);     // [128] m, [128] l; the folded replicas' [128] m, [128] l
#pragma unroll
            for (int u = 0; u < kOut / 4; ++u) {
                const int c4 = ocol / 4 + u;
                *reinterpret_cast<uint4*>(part_o + r * 128 + ((c4 ^ (r & 31)) << 2)) = make_uint4(o[4 * u], o[4 * u + 1], o[4 * u + 2], o[4 * u + 3]);
            }
            if (grp == 0 && wg == 0) { part_ml[r] = ok ? m_row : -INFINITY; part_ml[kT + r] = ok ? l_row : 0.f; }
            if (kRep > 1) {   // the replicas of a row into the first, one thread per (row, four output columns)
                asm volatile("bar.sync 13, %0;\n" ::"n"(256 * kGroups) : "memory");
                for (int it = tid - 128; it < kRows * 32; it += 256 * kGroups) {
                    const int fr = it >> 5, c4 = it & 31;
                    float gm = -INFINITY, lsum = 0.f;
                    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                    for (int j = 0; j < kRep; ++j) gm = fmaxf(gm, part_ml[fr + kRows * j]);
#pragma unroll
                    for (int j = 0; j < kRep; ++j) {
                        const float mj = part_ml[fr + kRows * j], w = mj == -INFINITY ? 0.f : ex2(mj - gm);
                        const float4 ov = *reinterpret_cast<const float4*>(part_o + (fr + kRows * j) * 128 + ((c4 ^ (fr & 31)) << 2));
                        lsum = fmaf(w, part_ml[kT + fr + kRows * j], lsum);
                        acc.x = fmaf(w, ov.x, acc.x); acc.y = fmaf(w, ov.y, acc.y);
                        acc.z = fmaf(w, ov.z, acc.z); acc.w = fmaf(w, ov.w, acc.w);
                    }
                    *reinterpret_cast<float4*>(part_o + fr * 128 + ((c4 ^ (fr & 31)) << 2)) = acc;   // (read by this thread only)
                    if (c4 == 0) { part_ml[2 * kT + fr] = gm; part_ml[3 * kT + fr] = lsum; }
                }
            }
        }
    }
    if (kRep > 1 || n_split > 1) {
        cg::cluster_group cluster = cg::this_cluster();
        __syncwarp();
        fence_before_sync();
        cluster.sync();   // every member's partial is in its shared memory
        if (warp >= 4) {
            // this CTA folds query rows [split * R, (split + 1) * R) of the tile, R = 128 / n_split rounded up: one thread per
            // (row, four output columns), reading that piece of every member's partial, four or eight members at a time
            const float* part_o = reinterpret_cast<const float*>(smem + kSmK);
            const float* part_ml = reinterpret_cast<const float*>(smem + kSmV) + (kRep > 1 ? 2 * kT : 0);
            constexpr int kRows = kT / kRep;
            const int R = (kRows + n_split - 1) / n_split, r_end = min(min((split + 1) * R, kRows), rows_total - qt * kT);
            const auto fold_rows = [&](auto width) {   // `width` partials at a time
                constexpr int kFold = decltype(width)::value;
                for (int it = tid - 128; it < R * 32; it += 256 * kGroups) {
                    const int r = split * R + (it >> 5), c4 = it & 31;
                    if (r >= r_end) break;
                    float gm = -INFINITY, lsum = 0.f;
                    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
                    for (int j0 = 0; j0 < n_split; j0 += kFold) {
                        float mv[kFold], lv[kFold];
                        float4 ov[kFold];
#pragma unroll
                        for (int j = 0; j < kFold; ++j) {   // requested together
                            const bool on = j0 + j < n_split;
                            const float* ml = cluster.map_shared_rank(part_ml, on ? j0 + j : 0);
                            const float* po = cluster.map_shared_rank(part_o, on ? j0 + j : 0);
                            mv[j] = on ? ml[r] : -INFINITY;
                            lv[j] = on ? ml[kT + r] : 0.f;
                            ov[j] = on ? *reinterpret_cast<const float4*>(po + r * 128 + ((c4 ^ (r & 31)) << 2)) : make_float4(0.f, 0.f, 0.f, 0.f);
                        }
                        float top = gm;
#pragma unroll
                        for (int j = 0; j < kFold; ++j) top = fmaxf(top, mv[j]);
                        if (top == -INFINITY) continue;   // nothing but empty shares so far
                        const float f = gm == -INFINITY ? 0.f : ex2(gm - top);
                        lsum *= f; acc.x *= f; acc.y *= f; acc.z *= f; acc.w *= f;
                        gm = top;
#pragma unroll
                        for (int j = 0; j < kFold; ++j) {
                            const float w = (mv[j] == -INFINITY) ? 0.f : ex2(mv[j] - gm);
                            lsum = fmaf(w, lv[j], lsum);
                            acc.x = fmaf(w, ov[j].x, acc.x); acc.y = fmaf(w, ov[j].y, acc.y);
                            acc.z = fmaf(w, ov[j].z, acc.z); acc.w = fmaf(w, ov[j].w, acc.w);
                        }
                    }
                    const float inv = lsum > 0.f ? 1.f / lsum : 0.f;
                    uint2 v;
                    v.x = pack2(acc.x * inv, acc.y * inv);
                    v.y = pack2(acc.z * inv, acc.w * inv);
                    *reinterpret_cast<uint2*>(p.out + (size_t)(q_row0 + r) * 128 + c4 * 4) = v;
                }
            };
            if (n_split <= 4) fold_rows(std::integral_constant<int, 4>());
            else fold_rows(std::integral_constant<int, 8>());
        }
        __syncwarp();
        cluster.sync();   // every member's shared memory has been read: they may leave
    }
    __syncthreads();
    if (*sh_fail) {   // a wait gave up: report it and give copies still in flight one more bounded wait
        if (tid == 0) {
            set_status(p.status, SC_ERR_TIMEOUT);
            if (nt > 0) mbar_wait(q_full, 0);
            for (int u = 0; u < 2; ++u) {
                const int issued = sh_issued[u];
                for (int t = max(issued - kStages, 0); t < issued; ++t) mbar_wait((u ? v_full0 : k_full0) + 8 * (t % kStages), (t / kStages) & 1);
            }
        }
        __syncthreads();
    }
    fence_before_sync();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem, kTmemCols);
}

// Any dtype, any d <= 256: one warp per (sequence, query head, query), online softmax in fp32.
template <typename T>
__global__ void __launch_bounds__(128) prefill_generic_kernel(const T* __restrict__ q, int B, int Hq, int Hkv, int m, int d,
                                                              const T* __restrict__ core_k, const T* __restrict__ core_v,
                                                              const int32_t* __restrict__ count, int cap,
                                                              const int32_t* __restrict__ core_len, float scale_log2, int causal,
                                                              T* __restrict__ out) {
    in_stream_order();
    const int lane = threadIdx.x & 31;
    const long long it = (long long)blockIdx.x * 4 + (threadIdx.x >> 5);
    if (it >= (long long)B * Hq * m) return;
    const int i = (int)(it % m), hq = (int)((it / m) % Hq), b = (int)(it / ((long long)m * Hq));
    const int h = hq / (Hq / Hkv);
    const int len = max(min(core_len[b * Hkv + h], cap), 0);
    const int vis = causal ? len - (m - 1 - i) : len;
    const T* qr = q + it * d;
    const long long cbase = ((long long)b * Hkv + h) * cap;
    float qv[8], acc[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const int c = lane + 32 * u;
        qv[u] = c < d ? Elem<T>::load(qr + c) * scale_log2 : 0.f;
        acc[u] = 0.f;
    }
    float mx = -INFINITY, lsum = 0.f;
    for (int t = 0; t < vis; ++t) {
        const T* kr = core_k + (cbase + t) * d;
        const T* vr = core_v + (cbase + t) * d;
        float s = 0.f;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int c = lane + 32 * u;
            if (c < d) s = fmaf(qv[u], Elem<T>::load(kr + c), s);
        }
        s = warp_sum(s);
        if (count != nullptr) s += log2f((float)max(count[cbase + t], 1));
        const float mn = fmaxf(mx, s);
        const float corr = exp2f(mx - mn), pw = exp2f(s - mn);
        lsum = lsum * corr + pw;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int c = lane + 32 * u;
            if (c < d) acc[u] = acc[u] * corr + pw * Elem<T>::load(vr + c);
        }
        mx = mn;
    }
    const float inv = lsum > 0.f ? 1.f / lsum : 0.f;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const int c = lane + 32 * u;
        if (c < d) Elem<T>::store(out + it * d + c, acc[u] * inv);
    }
}

}  // namespace pf

cudaError_t launch_prefill(const PrefillArgs& a, cudaStream_t st) {
    using namespace pf;
    const float scale_log2 = (a.scale == 0.f ? 1.f / sqrtf((float)a.d) : a.scale) * 1.4426950408889634f;
    const int causal = (a.flags & SC_FLAG_CAUSAL_TAIL) ? 1 : 0;
    const int G = a.Hq / a.Hkv;
    const long long q_rows = (long long)a.B * a.Hq * a.m, c_rows = (long long)a.B * a.Hkv * a.cap;
    if (a.dt == SC_BF16 && a.d == 128 && !(a.flags & SC_FLAG_GENERIC) && a.cap > 0 && q_rows < 0x7fffffff &&
        c_rows < 0x7fffffff && a.Hkv <= 65535 && a.B <= 65535) {
        // per device: the opt-ins, and how many clusters of each size (one CTA per SM) can be resident at once
        static int fit_of[64][kMaxSplit + 1] = {{0}};
        static std::once_flag once_of[64];
        int dev = 0;
        cudaGetDevice(&dev);
        dev &= 63;
        int* fit = fit_of[dev];
        std::call_once(once_of[dev], [&] {
            bool wide = true;
            for (auto kernel : {prefill_umma_kernel<1, 2>, prefill_umma_kernel<2, 2>, prefill_umma_kernel<4, 2>, prefill_umma_kernel<1, 1>, prefill_umma_kernel<2, 1>,
                                prefill_umma_kernel<4, 1>}) {
                cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
                wide = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess && wide;
            }
            for (int c = 2; c <= (wide ? kMaxSplit : 8); ++c) {
                cudaLaunchConfig_t probe = {};
                probe.gridDim = dim3(c, 1, 1);
                probe.blockDim = dim3(128 + 256 * 2);
                probe.dynamicSmemBytes = kSmemBytes;
                cudaLaunchAttribute pa[1];
                pa[0].id = cudaLaunchAttributeClusterDimension;
                pa[0].val.clusterDim.x = c; pa[0].val.clusterDim.y = 1; pa[0].val.clusterDim.z = 1;
                probe.attrs = pa;
                probe.numAttrs = 1;
                int n_clusters = 0;
                if (cudaOccupancyMaxActiveClusters(&n_clusters, prefill_umma_kernel<1, 2>, &probe) == cudaSuccess) fit[c] = n_clusters;
            }
            (void)cudaGetLastError();   // a refused opt-in or probe is not an error of this call
        });
        Params p;
        p.count = a.count; p.core_len = a.core_len; p.out = (__nv_bfloat16*)a.out;
        p.Hq = a.Hq; p.Hkv = a.Hkv; p.m = a.m; p.cap = a.cap; p.causal = causal; p.scale_log2 = scale_log2; p.status = a.status;
        // Replicas: the tile's chain of steps is the time of a launch with few rows, and most of it is a thread's scores.  8 layers of
        // 8 tokens verified and accepted (32 rows): 214 us with one, 180 with four; of 9 tokens (36 rows) 220 with one, 190 with
        // two; of 16 (64 rows) 247 and 219.
        const int rep = G * a.m <= 32 ? 4 : G * a.m <= 64 ? 2 : 1;
        if (make_map_bf16_rows(&p.map_q, a.q, 0, 0, 128, 1, 1, q_rows, kT / rep) &&
            make_map_bf16_rows(&p.map_k, a.core_k, 0, 0, 128, 1, 1, c_rows, kT) &&
            make_map_bf16_rows(&p.map_v, a.core_v, 0, 0, 128, 1, 1, c_rows, kT)) {
            // Few query tiles (short chunks, speculative decoding): the keys are split over a cluster.  Of the widths whose clusters
            // all fit at once, the narrowest that leaves a CTA the fewest key tiles of a head that fills half the capacity (as
            // compressed heads do or less): a wider one has the same tiles to walk and more partials to fold.  8 heads x 4 K
            // rows of 8 K, 128 query rows: 8 CTAs 16.6 us, 10 CTAs 17.5; 8 K rows of 16 K: 23.5 and 23.1; 500 rows of 1 K: 4 CTAs 10.6,
            // 2 CTAs 14.6.  Fewer than four are not worth their fold (3 us with two) for less than eight tiles, unless the
            // rows stand in the tile more than once and the fold is short.
            const long long ctas = (long long)((G * a.m + kT - 1) / kT) * a.Hkv * a.B;
            const int half_tiles = ((a.cap + kT - 1) / kT + 1) / 2;
            int n_split = 1;
            for (int c = rep == 1 && half_tiles < 8 ? 4 : 2; c <= kMaxSplit; ++c) {
                if (c > 8 && half_tiles < (c < 12 ? 2 * c : c)) continue;   // a second round of the fold for less than a tile
                if (ctas <= fit[c] && (half_tiles + c - 1) / c < (half_tiles + n_split - 1) / n_split) n_split = c;
            }
            p.n_split = n_split;
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3((unsigned)((G * a.m + kT - 1) / kT) * n_split, a.Hkv, a.B);
            // One group of softmax warps where a CTA is likely to have a single key tile, or two of few rows folded over a cluster anyway:
            // 384 threads start 0.3 us sooner than 640, and a second group has nothing, or little, to do.  8 heads, one query over 266
            // rows of 512: 8.3 us with two groups, 8.0 with one; 128 causal ones over 394: 11.9, 11.4; 28 rows over 2162 on 16 CTAs 9.5, 9.1.  With more tiles two: 32 queries
            // over 2162 rows 14.3, 14.6; 64 over 130, two tiles of one CTA, 9.8, 10.5.  Likely: five eighths of the capacity, a
            // little more than the half that compressed heads fill, and a causal block's own tokens.
            const long long likely = (causal ? (long long)std::max(a.cap - a.m, 0) * 5 / 8 + a.m : (long long)a.cap * 5 / 8);
            const long long each = ((likely + kT - 1) / kT + n_split - 1) / n_split;
            const bool one_group = each <= (rep > 1 && n_split > 1 ? 2 : 1);
            cfg.blockDim = dim3(128 + 256 * (one_group ? 1 : 2));
            cfg.dynamicSmemBytes = kSmemBytes;
            cfg.stream = st;
            cudaLaunchAttribute attr[2];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = n_split; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
            attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
            attr[1].val.programmaticStreamSerializationAllowed = 1;
            cfg.attrs = attr;
            cfg.numAttrs = 2;
            note_launches(1);
            return own_error(cudaLaunchKernelEx(&cfg, one_group ? (rep == 4 ? prefill_umma_kernel<4, 1> : rep == 2 ? prefill_umma_kernel<2, 1> : prefill_umma_kernel<1, 1>)
                                                         : (rep == 4 ? prefill_umma_kernel<4, 2> : rep == 2 ? prefill_umma_kernel<2, 2> : prefill_umma_kernel<1, 2>), p));
        }
    }
    const unsigned blocks = (unsigned)((q_rows + 3) / 4);
    note_launches(1);
    if (a.dt == SC_BF16)
        return launch_in_order(prefill_generic_kernel<__nv_bfloat16>, dim3(blocks), 128, 0, st, (const __nv_bfloat16*)a.q, a.B, a.Hq, a.Hkv, a.m,
                               a.d, (const __nv_bfloat16*)a.core_k, (const __nv_bfloat16*)a.core_v, a.count, a.cap, a.core_len, scale_log2,
                               causal, (__nv_bfloat16*)a.out);
    return launch_in_order(prefill_generic_kernel<float>, dim3(blocks), 128, 0, st, (const float*)a.q, a.B, a.Hq, a.Hkv, a.m, a.d,
                           (const float*)a.core_k, (const float*)a.core_v, a.count, a.cap, a.core_len, scale_log2, causal, (float*)a.out);
}

}  // namespace sc
