// One cluster of two blocks and the decode kernel's fold: block 1 hands its half to block 0 after `delay_ns` (or never, below 0),
// block 0 waits with `limit_ns`.  Every wait here ends: the delay and the limits are clocked, a block that left is not waited for.
#include "decode_fold.cuh"

namespace {

constexpr int kSlice = 4;   // groups of four columns, all of head 0

__global__ void __cluster_dims__(2) __launch_bounds__(32) probe(long long delay_ns, unsigned long long limit_ns, float* out, int32_t* status,
                                                                unsigned long long* left) {
    using namespace sc;
    __shared__ __align__(16) float4 recv_o[2 * kSlice];
    __shared__ __align__(16) float recv_ml[2 * 16];
    __shared__ __align__(8) unsigned long long bar;
    const uint32_t bar_s = umma::smem_u32(&bar);
    const int rank = blockIdx.x, lane = threadIdx.x;
    if (lane < 2 * kSlice) recv_o[lane] = make_float4(0.f, 0.f, 0.f, 0.f);
    recv_ml[lane] = 0.f;
    if (lane == 0) {
        umma::mbar_init(bar_s, 1);
        umma::mbar_fence_init();
        if (rank == 0) umma::mbar_expect_tx(bar_s, 2 * (kSlice * 16 + 8));
    }
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
    const unsigned long long t0 = umma::global_ns();
    if (rank == 1) {
        while (delay_ns > 0 && umma::global_ns() - t0 < (unsigned long long)delay_ns) {}
        __syncwarp();
    }
    if (rank == 0 || delay_ns >= 0) {   // m = 0, l = 1 and O = 1 (block 0), 3 (block 1): 2 on the average
        const uint32_t to = dm::mapa(bar_s, 0);
        const float v = rank == 0 ? 1.f : 3.f;
        if (lane < kSlice) dm::hand_over(dm::mapa(umma::smem_u32(recv_o + rank * kSlice + lane), 0), to, make_float4(v, v, v, v));
        if (lane == 0) dm::hand_over(dm::mapa(umma::smem_u32(recv_ml + rank * 16), 0), to, 0.f, 1.f);
    }
    __syncwarp();
    if (rank == 0) {
        const bool got = dm::slices_arrived(bar_s, limit_ns);
        if (!got) set_status(status, SC_ERR_TIMEOUT);
        if (lane < kSlice) {
            const dm::Folded f = dm::fold_slices(recv_o, recv_ml, 2, kSlice, lane, 0, got);
            *reinterpret_cast<float4*>(out + lane * 4) = make_float4(f.o.x / f.l, f.o.y / f.l, f.o.z / f.l, f.o.w / f.l);
            if (lane == 0) out[4 * kSlice] = f.m;
        }
        __syncwarp();
        dm::outlast_cluster(bar_s, got, limit_ns);
    }
    __syncwarp();
    if (lane == 0) left[rank] = umma::global_ns();
}

}  // namespace

extern "C" int run_probe(long long delay_ns, unsigned long long limit_ns, float* out, int32_t* status, unsigned long long* left, void* stream) {
    probe<<<2, 32, 0, (cudaStream_t)stream>>>(delay_ns, limit_ns, out, status, left);
    return (int)cudaGetLastError();
}
