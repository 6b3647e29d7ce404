// The fold of the decode kernel's clusters: every block hands each slice of its partial (m, l, O), through distributed shared
// memory, to the block that folds that slice.
#pragma once

#include "common.cuh"
#include "umma.cuh"

namespace sc {
namespace dm {

constexpr int kMaxCluster = 16;                 // blocks per cluster (more than 8 needs the non-portable opt-in)

__device__ __forceinline__ float fast_exp2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;\n" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ uint32_t mapa(uint32_t addr, int rank) {
    uint32_t a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(a) : "r"(addr), "r"(rank));
    return a;
}
// Stores to the shared memory of a block of the cluster, counted by that block's mbarrier (addresses from mapa).
__device__ __forceinline__ void hand_over(uint32_t dst, uint32_t bar, const float4& v) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];\n"
                 ::"r"(dst), "r"(__float_as_uint(v.x)), "r"(__float_as_uint(v.y)), "r"(__float_as_uint(v.z)), "r"(__float_as_uint(v.w)), "r"(bar) : "memory");
}
__device__ __forceinline__ void hand_over(uint32_t dst, uint32_t bar, float x, float y) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.b32 [%0], {%1, %2}, [%3];\n"
                 ::"r"(dst), "r"(__float_as_uint(x)), "r"(__float_as_uint(y)), "r"(bar) : "memory");
}

// Waits until everything the cluster's blocks hand this one has arrived.  The limit is by the clock, which runs on while a context is
// switched off: a wait that ran out of it is given one more.
__device__ __forceinline__ bool slices_arrived(uint32_t bar, unsigned long long limit_ns = umma::kWaitLimitNs) {
    bool got = false;
#pragma unroll 1
    for (int turn = 0; turn < 2 && !got; ++turn) got = umma::mbar_wait<true>(bar, 0, limit_ns);
    return got;
}

// Element `at` (four columns of head `hd`) of this block's slice from all `csize` partials, in order: recv_o [csize][slice],
// recv_ml [csize][8 heads][m, l].  Where they have not all arrived the sums are not a number, in whatever they are merged into too.
struct Folded { float4 o; float m, l; };
__device__ __forceinline__ Folded fold_slices(const float4* recv_o, const float* recv_ml, int csize, int slice, int at, int hd, bool arrived) {
    float mv[kMaxCluster], lv[kMaxCluster];
    float4 ov[kMaxCluster];
#pragma unroll
    for (int j = 0; j < kMaxCluster; ++j) {
        mv[j] = j < csize ? recv_ml[j * 16 + 2 * hd] : -INFINITY;
        lv[j] = j < csize ? recv_ml[j * 16 + 2 * hd + 1] : 0.f;
        ov[j] = j < csize ? recv_o[j * slice + at] : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    Folded f = {make_float4(0.f, 0.f, 0.f, 0.f), mv[0], 0.f};
#pragma unroll
    for (int j = 1; j < kMaxCluster; ++j) f.m = fmaxf(f.m, mv[j]);
#pragma unroll
    for (int j = 0; j < kMaxCluster; ++j) {
        const float w = (mv[j] == -INFINITY) ? 0.f : fast_exp2(mv[j] - f.m);
        f.l = fmaf(w, lv[j], f.l);
        f.o.x = fmaf(w, ov[j].x, f.o.x); f.o.y = fmaf(w, ov[j].y, f.o.y);
        f.o.z = fmaf(w, ov[j].z, f.o.z); f.o.w = fmaf(w, ov[j].w, f.o.w);
    }
    if (!arrived) {
        const float nan = __int_as_float(0x7fffffff);
        f.o = make_float4(nan, nan, nan, nan);
        f.m = 0.f;   // (a partial without rows would be passed over)
    }
    return f;
}

// The last step of a warp; does something where slices_arrived gave up for one of its threads: the block's shared memory stays until
// the cluster's other blocks have left (each of their waits ends, and a thread that has left is not waited for) and what they
// handed over has landed.
__device__ __forceinline__ void outlast_cluster(uint32_t bar, bool arrived, unsigned long long limit_ns = umma::kWaitLimitNs) {
    if (__all_sync(kFull, arrived)) return;
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
    umma::mbar_wait<true>(bar, 0, limit_ns);
}

}  // namespace dm
}  // namespace sc
