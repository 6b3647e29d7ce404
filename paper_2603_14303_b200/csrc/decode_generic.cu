// Generic decode path for Eq. 4 (any dtype, d <= 256 multiple of 8).  One block serves one (sequence, KV head, split of
// its cores, up to four of its query heads); its warps take 32-row tiles in turn: eight lanes per row form the
// scores (four rows at a time, sixteen requested ahead), one lane per row takes part in the online softmax in
// fp32, and for the weighted sum a lane owns four columns of every row, sixteen rows requested together.  A second kernel combines the splits in order.
// Serves SC_F32 and cross-checks the tensor-core bf16 kernel.
// Bounded by the latency of its loads: 2162 cores x 8 heads of fp32, 16 splits: 217 + 18 us when a warp served one query
// head row by row (each row a dependent chain of load, five shuffles and two exponentials), 14 + 7 us like this (37 + 7 with
// eight rows requested at a time).  Eight warps or four per block: see run().
#include "common.cuh"

namespace sc {

constexpr int kCombineWarps = 4;
constexpr int kDecHeads = 4;    // query heads per block
constexpr int kDecMaxD = 256;

__host__ __device__ inline int generic_splits(int cap) {
    int s = (cap + 511) / 512;
    return s < 1 ? 1 : (s > 64 ? 64 : s);
}

// NC: the most 32-column pieces a row has (4 or 8).
// Eight warps have an SM to themselves (bounds (256, 1); left to itself the compiler takes 80 registers and spills: 23 us for 16).
template <typename T, int NC, int kDecWarps>
__global__ void __launch_bounds__(kDecWarps * 32, kDecWarps == 8 ? 1 : 0)
decode_generic(const T* __restrict__ q, int Hq, int Hkv, int d, const T* __restrict__ core_k,
               const T* __restrict__ core_v, const int32_t* __restrict__ count, int cap,
               const int32_t* __restrict__ core_len, float scale_log2, int n_split, float* __restrict__ part) {
    constexpr int kPer = NC / 4;
    __shared__ __align__(16) float sq[kDecHeads][kDecMaxD];              // scaled queries
    __shared__ __align__(16) float4 sp[kDecWarps][32];                   // scores, then weights, of a tile: [row][head]
    __shared__ __align__(16) float so[kDecWarps][kDecHeads][kDecMaxD];   // the warps' sums
    __shared__ float sm[kDecWarps][kDecHeads], sl[kDecWarps][kDecHeads];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, sub = lane & 7, rsub = lane >> 3;
    in_stream_order();
    const int G = Hq / Hkv, groups = (G + kDecHeads - 1) / kDecHeads;
    // blockIdx.x = ((b * Hkv + h) * groups + group) * n_split + split
    const int split = blockIdx.x % n_split, hg = (blockIdx.x / n_split) % (Hkv * groups), b = blockIdx.x / n_split / (Hkv * groups);
    const int h = hg / groups, g0 = (hg - h * groups) * kDecHeads, nh = min(kDecHeads, G - g0);
    const int len = max(min(core_len[b * Hkv + h], cap), 0);
    const int per_split = (len + n_split - 1) / n_split;
    const int t0 = min(split * per_split, len), t1 = min(t0 + per_split, len);
    const int hq0 = b * Hq + h * G + g0;   // first query head of the block
    const size_t cbase = ((size_t)b * Hkv + h) * cap;
    for (int i = threadIdx.x; i < kDecHeads * kDecMaxD; i += kDecWarps * 32) {
        const int g = i / kDecMaxD, c = i % kDecMaxD;
        sq[g][c] = g < nh && c < d ? Elem<T>::load(q + (size_t)(hq0 + g) * d + c) * scale_log2 : 0.f;
    }
    __syncthreads();
    float m[kDecHeads], l[kDecHeads], acc[kDecHeads][kPer][4];
#pragma unroll
    for (int g = 0; g < kDecHeads; ++g) {
        m[g] = -INFINITY; l[g] = 0.f;   // l: this lane's rows only
#pragma unroll
        for (int u = 0; u < kPer; ++u) acc[g][u][0] = acc[g][u][1] = acc[g][u][2] = acc[g][u][3] = 0.f;
    }
    for (int tb = t0 + w * 32; tb < t1; tb += kDecWarps * 32) {
        const int nr = min(32, t1 - tb);
        // ln s, in base-2 units (a valid row has count >= 1)
        const float lc = count != nullptr && lane < nr ? log2f((float)max(count[cbase + tb + lane], 1)) : 0.f;
#pragma unroll (16 / NC)
        for (int it = 0; it < 8; ++it) {   // four rows at a time
            const int r = it * 4 + rsub;
            const T* kr = core_k + (cbase + tb + min(r, nr - 1)) * d;
            float4 kv[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                const int col = (c * 8 + sub) * 4;
                kv[c] = col < d ? load4(kr + col) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
            float s[kDecHeads];
#pragma unroll
            for (int g = 0; g < kDecHeads; ++g) {
                s[g] = 0.f;
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    const float4 qv = *reinterpret_cast<const float4*>(&sq[g][(c * 8 + sub) * 4]);
                    s[g] = fmaf(qv.x, kv[c].x, fmaf(qv.y, kv[c].y, fmaf(qv.z, kv[c].z, fmaf(qv.w, kv[c].w, s[g]))));
                }
            }
#pragma unroll
            for (int o = 1; o < 8; o <<= 1)
#pragma unroll
                for (int g = 0; g < kDecHeads; ++g) s[g] += __shfl_xor_sync(kFull, s[g], o);
            if (sub == 0) sp[w][r] = make_float4(s[0], s[1], s[2], s[3]);
        }
        __syncwarp();
        {
            const float4 xs = sp[w][lane];
            const float x[kDecHeads] = {xs.x, xs.y, xs.z, xs.w};
            float pw[kDecHeads];
#pragma unroll
            for (int g = 0; g < kDecHeads; ++g) {
                const float xg = lane < nr ? x[g] + lc : -INFINITY;
                const float mn = fmaxf(m[g], warp_max(xg));
                const float corr = exp2f(m[g] - mn);   // m = -inf on the first tile gives 0
                pw[g] = exp2f(xg - mn);
                l[g] = l[g] * corr + pw[g];
#pragma unroll
                for (int u = 0; u < kPer; ++u) { acc[g][u][0] *= corr; acc[g][u][1] *= corr; acc[g][u][2] *= corr; acc[g][u][3] *= corr; }
                m[g] = mn;
            }
            __syncwarp();
            sp[w][lane] = make_float4(pw[0], pw[1], pw[2], pw[3]);
        }
        __syncwarp();
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
            const int col = (u * 32 + lane) * 4;
            if (col >= d) continue;
            const T* vc = core_v + (cbase + tb) * d + col;
            for (int r0 = 0; r0 < nr; r0 += 16) {   // sixteen rows requested together
                float4 vv[16];
#pragma unroll
                for (int j = 0; j < 16; ++j) vv[j] = r0 + j < nr ? load4(vc + (size_t)(r0 + j) * d) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    const float4 pv = sp[w][r0 + j];
                    const float pg[kDecHeads] = {pv.x, pv.y, pv.z, pv.w};
#pragma unroll
                    for (int g = 0; g < kDecHeads; ++g) {
                        acc[g][u][0] = fmaf(pg[g], vv[j].x, acc[g][u][0]); acc[g][u][1] = fmaf(pg[g], vv[j].y, acc[g][u][1]);
                        acc[g][u][2] = fmaf(pg[g], vv[j].z, acc[g][u][2]); acc[g][u][3] = fmaf(pg[g], vv[j].w, acc[g][u][3]);
                    }
                }
            }
        }
        __syncwarp();   // the next tile's scores overwrite the weights
    }
    // the warps' (m, l, O), in order
#pragma unroll
    for (int g = 0; g < kDecHeads; ++g) {
        const float lw = warp_sum(l[g]);
        if (lane == 0) { sm[w][g] = m[g]; sl[w][g] = lw; }
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
            const int col = (u * 32 + lane) * 4;
            *reinterpret_cast<float4*>(&so[w][g][col]) = make_float4(acc[g][u][0], acc[g][u][1], acc[g][u][2], acc[g][u][3]);
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nh * (d / 2); i += kDecWarps * 32) {
        const int g = i / (d / 2), c = (i - g * (d / 2)) * 2;
        float mm = -INFINITY;
#pragma unroll
        for (int j = 0; j < kDecWarps; ++j) mm = fmaxf(mm, sm[j][g]);
        float ls = 0.f;
        float2 o = make_float2(0.f, 0.f);
#pragma unroll
        for (int j = 0; j < kDecWarps; ++j) {
            if (sm[j][g] == -INFINITY) continue;   // a warp without rows
            const float f = exp2f(sm[j][g] - mm);
            ls += f * sl[j][g];
            o.x = fmaf(f, so[j][g][c], o.x); o.y = fmaf(f, so[j][g][c + 1], o.y);
        }
        float* pr = part + ((size_t)(hq0 + g) * n_split + split) * (d + 2);
        *reinterpret_cast<float2*>(pr + c) = o;
        if (c == 0) *reinterpret_cast<float2*>(pr + d) = make_float2(mm, ls);
    }
}

// One warp per query head: the splits' weights from one pair of loads per lane, then their sums in order.
template <typename T>
__global__ void __launch_bounds__(kCombineWarps * 32)
combine_generic(int64_t heads, int d, int n_split, const float* __restrict__ part, T* __restrict__ out) {
    __shared__ float sw[kCombineWarps][64];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t hd = (int64_t)blockIdx.x * kCombineWarps + w;
    in_stream_order();
    if (hd >= heads) return;
    const float* pr = part + hd * n_split * (d + 2);
    float2 ml[2];   // (m, l) of splits lane, lane + 32
#pragma unroll
    for (int k = 0; k < 2; ++k)
        ml[k] = lane + 32 * k < n_split ? __ldcg(reinterpret_cast<const float2*>(pr + (size_t)(lane + 32 * k) * (d + 2) + d))
                                        : make_float2(-INFINITY, 0.f);
    const float m = warp_max(fmaxf(ml[0].x, ml[1].x));
    float lsum = 0.f;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const float wgt = ml[k].x == -INFINITY ? 0.f : exp2f(ml[k].x - m);   // 0: an empty split
        sw[w][lane + 32 * k] = wgt;
        lsum += wgt * ml[k].y;
    }
    lsum = warp_sum(lsum);
    __syncwarp();
    const float inv = lsum > 0.f ? 1.f / lsum : 0.f;
    for (int c = lane * 2; c < d; c += 64) {
        float2 acc = make_float2(0.f, 0.f);
        for (int s0 = 0; s0 < n_split; s0 += 8) {
            float2 v[8];
#pragma unroll
            for (int j = 0; j < 8; ++j)
                v[j] = s0 + j < n_split && sw[w][s0 + j] != 0.f ? __ldcg(reinterpret_cast<const float2*>(pr + (size_t)(s0 + j) * (d + 2) + c))
                                                                : make_float2(0.f, 0.f);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const float wgt = s0 + j < n_split ? sw[w][s0 + j] : 0.f;
                acc.x = fmaf(wgt, v[j].x, acc.x); acc.y = fmaf(wgt, v[j].y, acc.y);
            }
        }
        Elem<T>::store(out + hd * d + c, acc.x * inv);
        Elem<T>::store(out + hd * d + c + 1, acc.y * inv);
    }
}

size_t decode_generic_ws_bytes(int32_t B, int32_t Hq, int32_t Hkv, int32_t d, int32_t cap) {
    (void)Hkv;
    return decode_mma_counter_bytes() + sizeof(float) * (size_t)B * Hq * generic_splits(cap) * (d + 2) + 256;
}

template <typename T>
static cudaError_t run(const DecodeArgs& a, cudaStream_t st) {
    const int n_split = generic_splits(a.cap);
    const float scale = (a.scale == 0.f ? 1.f / sqrtf((float)a.d) : a.scale) * 1.4426950408889634f;
    const int groups = div_up(a.Hq / a.Hkv, kDecHeads);
    const int64_t blocks = (int64_t)n_split * a.Hkv * groups * a.B;
    if (blocks > 0x7fffffff) return cudaErrorInvalidConfiguration;
    const unsigned grid = (unsigned)blocks;
    // Partials lie behind the tensor-core kernel's counters, which have to stay zero for a later call with this workspace.  They
    // are read and written in pairs of floats; a workspace need only be aligned to one (256 spare bytes cover the step).
    float* part = reinterpret_cast<float*>((reinterpret_cast<uintptr_t>(a.ws) + decode_mma_counter_bytes() + 7) & ~(uintptr_t)7);
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // A launch of no more blocks than SMs leaves each block an SM, which eight warps use better: float32, 8 heads x 4 K rows of 8 K
    // 19.7 -> 16.1 us, bf16 with d = 256 38.3 -> 29.4.  Where there are more, blocks of four warps, of which an SM holds three
    // to five with their starts and folds beside the others' loads: 16 sequences x 8 heads x 4 K rows, float32 211 -> 135, bf16
    // with d = 64 283 -> 113, with d = 256 429 -> 282; just above the line, 10 heads x 4 K rows, 23.9 -> 22.7.
    const bool alone = blocks <= sms;
    const auto kernel = a.d <= 128 ? (alone ? decode_generic<T, 4, 8> : decode_generic<T, 4, 4>)
                                   : (alone ? decode_generic<T, 8, 8> : decode_generic<T, 8, 4>);
    cudaError_t e = launch_in_order(kernel, dim3(grid), (alone ? 8 : 4) * 32, 0, st,
                                    (const T*)a.q, a.Hq, a.Hkv, a.d, (const T*)a.core_k, (const T*)a.core_v, a.count, a.cap,
                                    a.core_len, scale, n_split, part);
    if (e != cudaSuccess) return e;
    const int64_t heads = (int64_t)a.B * a.Hq;
    e = launch_in_order(combine_generic<T>, dim3(div_up(heads, kCombineWarps)), kCombineWarps * 32, 0, st, heads, a.d, n_split,
                              (const float*)part, (T*)a.out);
    if (e != cudaSuccess) return e;
    note_launches(2);
    return cudaSuccess;
}

cudaError_t launch_decode_generic(const DecodeArgs& a, cudaStream_t st) {
    return a.dt == SC_BF16 ? run<__nv_bfloat16>(a, st) : run<float>(a, st);
}

}  // namespace sc
