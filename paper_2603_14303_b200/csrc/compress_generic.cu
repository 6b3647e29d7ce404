// Generic compress path (any dtype, any d <= 256 that is a multiple of 8, any strides):
// three kernels per layer -- GSC per segment, prefix sum of cluster counts per (b, head),
// mean-pool merge per segment.  CUDA-core arithmetic in fp32; serves SC_F32 and is the
// cross-check of the fused bf16 path.
// One warp per segment, a block of its own (blocks of four warps ran as long as their longest segment, in two uneven waves: scheduler
// partitions were busy 17 to 52 thousand of 62 thousand clocks; the whole path for 8 heads x 8K tokens 89.9 -> 85.3 us).
// Bounded by the latency of its loads, so all rows of a segment of up to 32 tokens are in flight at
// once: clustering keeps them in registers for every seed, the merge takes them in the order of their clusters, eight at a time.
// 8 heads x 8K tokens of fp32, chunks of 20 / 8 tokens (caches cold): clustering 43 / 34 us -> 29 / 20
// against eight and four rows in flight (101 us with one row at a time).  Clustering: 128 registers of rows leave three warps per scheduler; four spill, +8 %.
// The eight lanes of a row group share out the sums of their rows (seven shuffles and one division for eight rows; with
// 24 and eight, 34 / 39 us).  Merge: in cluster order a sum is one set of registers; added to the clusters' sums in shared memory
// row by row (a load, an addition and a store that wait for one another) the path takes 85.8 us against 80.4; K and V of
// a segment in one warp 82.4, and chunks of 128 tokens 280 against 250 (they leave too few warps).
#include <algorithm>
#include <type_traits>

#include "common.cuh"

namespace sc {

constexpr int kGenWarps = 1;
constexpr int kGenBlocks = 12;     // per SM (168 registers a thread): a short segment's rows are kept in registers
constexpr int kShortSeg = 32;      // rows of a short segment (d <= 128)
constexpr int kMergeRows = 8;     // rows of a short segment requested together
constexpr int kMergeBlocks = 24;

// Sums over the eight lanes of a row group: x[q] of every lane in, the sum for q = lane % R out (R = 8, 4, 2).
template <int R>
__device__ __forceinline__ float group_sums(float (&x)[R], int lane) {
#pragma unroll
    for (int o = 1; o < R; o <<= 1) {   // halve the number of sums a lane holds
        const bool odd = lane & o;
#pragma unroll
        for (int q = 0; q < R / (2 * o); ++q) {
            const float give = odd ? x[2 * q] : x[2 * q + 1], keep = odd ? x[2 * q + 1] : x[2 * q];
            x[q] = keep + __shfl_xor_sync(kFull, give, o);
        }
    }
#pragma unroll
    for (int o = R; o < 8; o <<= 1) x[0] += __shfl_xor_sync(kFull, x[0], o);
    return x[0];
}

// A vote of lanes that decide for row (their group of eight) R + lane % R, as bits by row.
template <int R>
__device__ __forceinline__ unsigned by_row(unsigned votes) {
    if (R == 4) return (votes & 15u) | ((votes >> 4) & 0xf0u) | ((votes >> 8) & 0xf00u) | ((votes >> 12) & 0xf000u);
    if (R == 2) return (votes & 3u) | ((votes >> 6) & 12u) | ((votes >> 12) & 48u) | ((votes >> 18) & 192u);
    return votes;
}

// Algorithm 1 for a segment of at most 4 R rows: all of them are requested at once and stay in registers, R per group of
// eight lanes; only the seeds' rows are read again.  A lane decides for row (its group) R + lane % R.  Same sums in the
// same order as the loop for longer ones.
template <int R, int NC, typename Load, typename Dot>
__device__ __forceinline__ int short_segment(int l, float tau, int32_t* as, int r, int lane, const Load& load_row, const Dot& dot) {
    const int row0 = (lane >> 3) * R;
    float4 v[R][NC];
    float x[R];
#pragma unroll
    for (int q = 0; q < R; ++q) load_row(row0 + q, row0 + q < l, v[q]);
#pragma unroll
    for (int q = 0; q < R; ++q) x[q] = dot(v[q], v[q]);
    const float nj = sqrtf(group_sums<R>(x, lane));
    unsigned open = 0xffffffffu >> (32 - l);
    int p = 0, mine = 0;   // mine: seed of token `lane`
    while (open) {
        const int i = __ffs(open) - 1;
        ++p;
        open &= open - 1;
        if (lane == i) mine = i;
        if (!open) break;
        float4 seed[NC];
        load_row(i, true, seed);
        const float ni = __shfl_sync(kFull, nj, (i / R) * 8 + i % R);
#pragma unroll
        for (int q = 0; q < R; ++q) x[q] = dot(seed, v[q]);
        const float prod = group_sums<R>(x, lane);
        const float sim = (ni == 0.f || nj == 0.f) ? 0.f : prod / (ni * nj);
        const unsigned hits = by_row<R>(__ballot_sync(kFull, sim > tau)) & open;
        if ((hits >> lane) & 1u) mine = i;
        open &= ~hits;
    }
    if (lane < l) as[lane] = r + mine;
    return p;
}

// Algorithm 1 for one segment per warp.  Longer segments' rows are read straight from global memory, 32 at a time, eight lanes a
// row, against the seed's row, which they hold in registers; rows already assigned are not read.  The whole path for
// 8 heads x 8K tokens of fp32 in chunks of 128: eight rows at a time 250 us, sixteen 200, 32 178; of 60: 169, 148, 139.  Where d > 128
// sixteen rows of fp32 (8 x 8K in chunks of 128 on the average: eight 482 us, sixteen 384), but eight for segments of up to 32 rows, whose
// places in a batch are mostly empty (8 heads x 128 tokens in chunks of 8: eight 24.4, sixteen 26.3), and eight of bf16, which
// spends its time on instructions and not on loads (4 x 8 x 8K, chunks of 8: 489 and 590; of 128: 848 and 944).  NC:
// the most 32-column pieces a row has (4 or 8).
template <typename T, int NC>
__global__ void __launch_bounds__(kGenWarps * 32, kGenBlocks)
gsc_generic(const T* __restrict__ K, sc_strides st, int B, int Hkv, int n, int d,
            const int32_t* __restrict__ seg_off, const int32_t* __restrict__ n_seg_p, int seg_stride,
            float tau_host, const float* __restrict__ tau_dev, const int32_t* __restrict__ skip,
            int32_t* __restrict__ assign, int32_t* __restrict__ seg_p) {
    __shared__ float norms[kGenWarps][SC_MAX_CHUNK_LEN];
    in_stream_order();
    if (skip != nullptr && *skip != 0) return;
    const float tau = tau_dev != nullptr ? *tau_dev : tau_host;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, sub = lane & 7, rsub = lane >> 3;
    const int n_seg = min(*n_seg_p, seg_stride);
    const int64_t items = (int64_t)n_seg * Hkv, warps = (int64_t)gridDim.x * kGenWarps;
    // two segments in a row per warp and step: runs and the delimiters between them alternate
    for (int64_t it = ((int64_t)blockIdx.x * kGenWarps + w) * 2; it < items; it += (it & 1) ? 2 * warps - 1 : 1) {
        const int s = (int)(it % n_seg), h = (int)(it / n_seg);
        const int a = seg_off[s], e = seg_off[s + 1];
        const int b = a / n, r = a - b * n, l = min(e - a, SC_MAX_CHUNK_LEN);
        const T* Kb = K + b * st.b + h * st.h + (int64_t)r * st.n + sub * 4;   // this lane's first columns of the segment's first row
        int32_t* as = assign + ((int64_t)b * Hkv + h) * n + r;
        // sum over the row's columns of x.y, x = row j (skipped where !on), the same in the row's eight lanes
        auto load_row = [&](int j, bool on, float4 (&v)[NC]) {
            const T* row = Kb + (int64_t)j * st.n;
#pragma unroll
            for (int c = 0; c < NC; ++c) v[c] = on && (c * 8 + sub) * 4 < d ? load4(row + c * 32) : make_float4(0.f, 0.f, 0.f, 0.f);
        };
        auto dot = [&](const float4 (&x)[NC], const float4 (&y)[NC]) {
            float acc = 0.f;
#pragma unroll
            for (int c = 0; c < NC; ++c) acc = fmaf(x[c].x, y[c].x, fmaf(x[c].y, y[c].y, fmaf(x[c].z, y[c].z, fmaf(x[c].w, y[c].w, acc))));
            return acc;
        };
        if (l == 1) {
            if (lane == 0) { as[0] = r; seg_p[(int64_t)h * seg_stride + s] = 1; }
            continue;
        }
        if constexpr (NC == 4) {
            if (l <= kShortSeg) {
                const int p = l <= 8 ? short_segment<2, NC>(l, tau, as, r, lane, load_row, dot)
                              : l <= 16 ? short_segment<4, NC>(l, tau, as, r, lane, load_row, dot)
                                        : short_segment<8, NC>(l, tau, as, r, lane, load_row, dot);
                if (lane == 0) seg_p[(int64_t)h * seg_stride + s] = p;
                continue;
            }
        }
        // longer: 4 R rows at a time; a lane decides for row j0 + row_of (in pairs of lanes, or fours)
        const auto longer = [&](auto rows_per_group) {
            constexpr int R = decltype(rows_per_group)::value, kRows = 4 * R;
            const int row_of = rsub * R + lane % R;
            const bool speaks = sub < R;   // one lane of those that decide for the same row
            for (int j0 = 0; j0 < l; j0 += kRows) {
                float4 v[R][NC];
                float x[R];
    #pragma unroll
                for (int q = 0; q < R; ++q) load_row(j0 + rsub * R + q, j0 + rsub * R + q < l, v[q]);
    #pragma unroll
                for (int q = 0; q < R; ++q) x[q] = dot(v[q], v[q]);
                const float nn = group_sums<R>(x, lane);
                if (speaks && j0 + row_of < l) norms[w][j0 + row_of] = sqrtf(nn);
            }
            __syncwarp();
            unsigned word = 0;  // lane c holds the assigned bits of tokens 32c .. 32c+31
            int p = 0;
            for (int i = 0; i < l; ++i) {
                const unsigned wi = __shfl_sync(kFull, word, i >> 5);
                if ((wi >> (i & 31)) & 1u) continue;
                ++p;
                if (lane == (i >> 5)) word |= 1u << (i & 31);
                if (lane == 0) as[i] = r + i;
                if (i + 1 >= l) break;
                float4 seed[NC];
                load_row(i, true, seed);
                const float ni = norms[w][i];
                for (int j0 = (i + 1) & ~(kRows - 1); j0 < l; j0 += kRows) {   // kRows tokens of one word
                    unsigned open = (~__shfl_sync(kFull, word, j0 >> 5)) >> (j0 & 31) & (0xffffffffu >> (32 - kRows));
                    if (j0 <= i) open &= ~0u << (i + 1 - j0);
                    if (l - j0 < kRows) open &= (1u << (l - j0)) - 1u;
                    if (open == 0u) continue;
                    float4 v[R][NC];
                    float x[R];
    #pragma unroll
                    for (int q = 0; q < R; ++q) load_row(j0 + rsub * R + q, (open >> (rsub * R + q)) & 1u, v[q]);
    #pragma unroll
                    for (int q = 0; q < R; ++q) x[q] = dot(seed, v[q]);
                    const float prod = group_sums<R>(x, lane), nj = j0 + row_of < l ? norms[w][j0 + row_of] : 0.f;
                    const float sim = (ni == 0.f || nj == 0.f) ? 0.f : prod / (ni * nj);
                    const unsigned hits = by_row<R>(__ballot_sync(kFull, sim > tau)) & open;
                    if (lane == (j0 >> 5)) word |= hits << (j0 & 31);
                    if (speaks && ((hits >> row_of) & 1u)) as[j0 + row_of] = r + i;
                }
            }
            return p;
        };
        int p;
        if constexpr (NC == 4) p = longer(std::integral_constant<int, 8>());
        else if constexpr (sizeof(T) == 2) p = longer(std::integral_constant<int, 2>());
        else p = l <= 32 ? longer(std::integral_constant<int, 2>()) : longer(std::integral_constant<int, 4>());
        if (lane == 0) seg_p[(int64_t)h * seg_stride + s] = p;
        __syncwarp();
    }
}

// Exclusive prefix sum of the per-segment cluster counts inside each (b, head).
__global__ void __launch_bounds__(256)
scan_generic(int Hkv, const int32_t* __restrict__ seq_seg_off, int seg_stride,
             const int32_t* __restrict__ seg_p, int32_t* __restrict__ seg_core_off,
             int32_t* __restrict__ core_len, int cap, int32_t* status, const int32_t* __restrict__ skip,
             int count_only) {
    __shared__ int wt[8];
    in_stream_order();
    if (skip != nullptr && *skip != 0) return;
    const int b = blockIdx.x / Hkv, h = blockIdx.x % Hkv;
    const int s0 = min(seq_seg_off[b], seg_stride), s1 = min(seq_seg_off[b + 1], seg_stride);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int carry = 0;
    for (int base = s0; base < s1; base += 256) {
        int s = base + threadIdx.x;
        int v = (s < s1) ? seg_p[(int64_t)h * seg_stride + s] : 0;
        int incl = warp_scan_add(v, lane);
        if (lane == 31) wt[w] = incl;
        __syncthreads();
        int pre = 0, tot = 0;
        for (int i = 0; i < 8; ++i) { if (i < w) pre += wt[i]; tot += wt[i]; }
        __syncthreads();
        if (s < s1) seg_core_off[(int64_t)h * seg_stride + s] = carry + pre + incl - v;
        carry += tot;
    }
    if (threadIdx.x == 0) {
        core_len[b * Hkv + h] = carry;
        if (carry > cap && !count_only) set_status(status, SC_ERR_CAPACITY);
    }
}

// Eq. 3 for one segment of K or of V per warp: fp32 sums in token order, one divide, one rounding.  A lane owns four
// columns (eight where d > 128).  Beyond 32 tokens or 128 columns a cluster's members come from ballots over the segment's
// assignments, four rows requested together.
template <typename T, int kPer>
__global__ void __launch_bounds__(kGenWarps * 32, kMergeBlocks)
merge_generic(const T* __restrict__ K, const T* __restrict__ V, sc_strides st, int B, int Hkv, int n, int d,
              const int32_t* __restrict__ seg_off, const int32_t* __restrict__ n_seg_p, int seg_stride,
              const int32_t* __restrict__ assign, const int32_t* __restrict__ seg_core_off,
              T* __restrict__ core_k, T* __restrict__ core_v, int32_t* __restrict__ count, int cap) {
    constexpr int kWords = SC_MAX_CHUNK_LEN / 32;
    __shared__ uint8_t order[kGenWarps][32];
    in_stream_order();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int n_seg = min(*n_seg_p, seg_stride);
    const int64_t segs = (int64_t)n_seg * Hkv, warps = (int64_t)gridDim.x * kGenWarps / 2;   // per tensor
    const int64_t me = (int64_t)blockIdx.x * kGenWarps + w;
    const bool is_v = me & 1;
    for (int64_t it = (me >> 1) * 2; it < segs; it += (it & 1) ? 2 * warps - 1 : 1) {   // two segments in a row, as above
        const int s = (int)(it % n_seg), h = (int)(it / n_seg);
        const int a = seg_off[s], e = seg_off[s + 1];
        const int b = a / n, r = a - b * n, l = min(e - a, SC_MAX_CHUNK_LEN), nw = (l + 31) >> 5;
        const T* rows = (is_v ? V : K) + b * st.b + h * st.h + (int64_t)r * st.n + lane * 4;
        const int32_t* as = assign + ((int64_t)b * Hkv + h) * n + r;
        int row = seg_core_off[(int64_t)h * seg_stride + s];
        const int64_t obase = ((int64_t)b * Hkv + h) * cap;
        T* cores = (is_v ? core_v : core_k) + obase * d + lane * 4;
        if (l == 1) {   // as it is (delimiters, and whatever stands between two of them)
            if (row >= cap) continue;
#pragma unroll
            for (int u = 0; u < kPer; ++u)
                if ((u * 32 + lane) * 4 < d) store4(cores + (int64_t)row * d + u * 128, load4(rows + u * 128));
            if (lane == 0 && !is_v) count[obase + row] = 1;
            continue;
        }
        if constexpr (kPer == 1) {
            if (l <= kShortSeg) {
                // the tokens in order of their clusters: place p of that order holds a token and whether it is its cluster's last
                const int own = lane < l ? as[lane] - r : -1;
                int before = 0, place = 0, last = 0;
                for (unsigned todo = __ballot_sync(kFull, own == lane); todo; todo &= todo - 1) {
                    const unsigned members = __ballot_sync(kFull, own == __ffs(todo) - 1);
                    if ((members >> lane) & 1u) { place = before + __popc(members & ((1u << lane) - 1u)); last = members >> lane == 1u ? 32 : 0; }
                    before += __popc(members);
                }
                if (lane < l) order[w][place] = (uint8_t)(lane | last);
                __syncwarp();
                const int at = order[w][lane];   // (places from l on are not used)
                // rows in that order, eight requested together: a cluster's sum needs one register set, a first row starts it
                const bool on = lane * 4 < d;
                float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
                int cnt = 0;
                for (int p0 = 0; p0 < l; p0 += kMergeRows) {
                    float4 v[kMergeRows];
#pragma unroll
                    for (int x = 0; x < kMergeRows; ++x) {
                        const int token = __shfl_sync(kFull, at, (p0 + x) & 31) & 31;
                        v[x] = on && p0 + x < l ? load4(rows + (int64_t)token * st.n) : make_float4(0.f, 0.f, 0.f, 0.f);
                    }
#pragma unroll
                    for (int x = 0; x < kMergeRows; ++x) {
                        if (p0 + x >= l) break;
                        sum = cnt == 0 ? v[x] : make_float4(sum.x + v[x].x, sum.y + v[x].y, sum.z + v[x].z, sum.w + v[x].w);
                        ++cnt;
                        if (!(__shfl_sync(kFull, at, (p0 + x) & 31) & 32)) continue;
                        if (row < cap) {
                            if (cnt > 1) {
                                const float fc = (float)cnt;
                                sum = make_float4(sum.x / fc, sum.y / fc, sum.z / fc, sum.w / fc);
                            }
                            if (on) store4(cores + (int64_t)row * d, sum);
                            if (lane == 0 && !is_v) count[obase + row] = cnt;
                        }
                        cnt = 0;
                        ++row;
                    }
                }
                __syncwarp();   // the order is read: the next segment's may be written
                continue;
            }
        }
        int mine[kWords];   // seed (relative) of tokens 32 k + lane
#pragma unroll
        for (int k = 0; k < kWords; ++k) mine[k] = 32 * k + lane < l ? as[32 * k + lane] - r : -1;
        for (int ws = 0; ws < nw; ++ws) {
            int own = -1;
#pragma unroll
            for (int k = 0; k < kWords; ++k) if (k == ws) own = mine[k];
            unsigned seeds = __ballot_sync(kFull, own == 32 * ws + lane);
            while (seeds) {
                const int i = 32 * ws + __ffs(seeds) - 1;
                seeds &= seeds - 1;
                float4 sum[kPer];
#pragma unroll
                for (int u = 0; u < kPer; ++u) sum[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                int cnt = 0;
#pragma unroll
                for (int k = 0; k < kWords; ++k) {
                    if (k < ws || k >= nw) continue;
                    unsigned mem = __ballot_sync(kFull, mine[k] == i);
                    cnt += __popc(mem);
                    while (mem) {   // four members at a time
                        int j[4];
#pragma unroll
                        for (int x = 0; x < 4; ++x) { j[x] = mem ? 32 * k + __ffs(mem) - 1 : -1; mem &= mem - 1; }
#pragma unroll
                        for (int u = 0; u < kPer; ++u) {
                            float4 v[4];
#pragma unroll
                            for (int x = 0; x < 4; ++x)
                                v[x] = j[x] >= 0 && (u * 32 + lane) * 4 < d ? load4(rows + (int64_t)j[x] * st.n + u * 128)
                                                                            : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                            for (int x = 0; x < 4; ++x) { sum[u].x += v[x].x; sum[u].y += v[x].y; sum[u].z += v[x].z; sum[u].w += v[x].w; }
                        }
                    }
                }
                if (row < cap) {
                    const float fc = (float)cnt;
#pragma unroll
                    for (int u = 0; u < kPer; ++u) {
                        if ((u * 32 + lane) * 4 >= d) continue;
                        const float4 v = cnt == 1 ? load4(rows + (int64_t)i * st.n + u * 128)   // as it is
                                                  : make_float4(sum[u].x / fc, sum[u].y / fc, sum[u].z / fc, sum[u].w / fc);
                        store4(cores + (int64_t)row * d + u * 128, v);
                    }
                    if (lane == 0 && !is_v) count[obase + row] = cnt;
                }
                ++row;
            }
        }
    }
}

size_t compress_generic_ws_bytes(int32_t B, int32_t Hkv, int32_t n) {
    // assign (when the caller passes none) + seg_p + seg_core_off, each B*Hkv*n int32
    return sizeof(int32_t) * 3 * (size_t)B * Hkv * n + 256;
}

template <typename T>
static cudaError_t run(const CompressArgs& a, cudaStream_t st) {
    const size_t per = (size_t)a.B * a.Hkv * a.n;
    int32_t* ws = (int32_t*)a.ws;
    int32_t* seg_p = ws;
    int32_t* seg_core_off = ws + per;
    int32_t* assign = (a.assign && !a.count_only) ? a.assign : ws + 2 * per;
    const int seg_stride = a.B * a.n;  // capacity of the segment axis
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // A warp takes two segments in turn; how many there are is known on the device only.  A run and its delimiter are three rows or
    // more as a rule (where they are not, a warp takes further ones), and blocks without any cost 0.5 us per thousand: 8 heads x 64
    // tokens of float32 8.6 us for the three kernels, 22 with 64 blocks per SM whatever the input; a pair to four rows 11.8, a
    // pair to two the same as to three up to 128 tokens and 0.1 to 1.5 us more above.
    const int64_t pairs = (int64_t)a.B * a.Hkv * a.n / 3 + 1, most = (int64_t)sms * 64;
    const unsigned gsc_grid = (unsigned)std::min(pairs, most), merge_grid = (unsigned)std::min(2 * pairs, most);
    auto gsc = a.d <= 128 ? gsc_generic<T, 4> : gsc_generic<T, 8>;
    cudaError_t e = launch_in_order(gsc, dim3(gsc_grid), kGenWarps * 32, 0, st, (const T*)a.K, a.st, a.B, a.Hkv, a.n, a.d, a.seg_off,
                                    a.n_seg, seg_stride, a.tau, a.tau_dev, a.skip, assign, seg_p);
    if (e != cudaSuccess) return e;
    e = launch_in_order(scan_generic, dim3(a.B * a.Hkv), 256, 0, st, a.Hkv, a.seq_seg_off, seg_stride, (const int32_t*)seg_p,
                              seg_core_off, a.core_len, a.cap, a.status, a.skip, a.count_only);
    if (e != cudaSuccess) return e;
    if (a.count_only) {   // budget search: per-head cluster counts only
        note_launches(2);
        return cudaSuccess;
    }
    e = launch_in_order(a.d <= 128 ? merge_generic<T, 1> : merge_generic<T, 2>, dim3(merge_grid), kGenWarps * 32, 0, st, (const T*)a.K,
                              (const T*)a.V, a.st, a.B, a.Hkv, a.n, a.d, a.seg_off, a.n_seg, seg_stride, (const int32_t*)assign,
                              (const int32_t*)seg_core_off, (T*)a.core_k, (T*)a.core_v, a.count, a.cap);
    if (e != cudaSuccess) return e;
    note_launches(3);
    return cudaSuccess;
}

cudaError_t launch_compress_generic(const CompressArgs& a, cudaStream_t st) {
    return a.dt == SC_BF16 ? run<__nv_bfloat16>(a, st) : run<float>(a, st);
}

}  // namespace sc
