// Blocked running DFT over the design box.  After cnt steps n0..n0+cnt-1 (n0 = ctl[3]), the block sums
// sum_s E^{n0+s+1} (cos, -sin)(w_f (n0+s+1) dt) are formed in T and added to the FP64 accumulators, which
// are read and written once per block of steps instead of every step.
//
// A snapshot slot and an accumulator frequency are both 3 nd consecutive samples, so a block takes
// kDftChunk consecutive samples whatever their component, and a thread two of them, 256 apart (whole
// sectors for the 16-byte accumulators, paired FP32 arithmetic for the sums).
//
// The kernel reads up to 16 + 8 streams tens of MB apart; what bounds it is how they reach DRAM.  With the
// snapshots loaded straight into registers, a warp's 128 or 256 bytes of each stream at a time, it ran
// slower the more loads were in flight (128^3 voxels, three frequencies: 0.24 to 0.39 ms from 5 to 3
// resident blocks).  So the chunk of each snapshot comes as one bulk copy of kDftChunk samples into shared
// memory, all of a block's copies completing on one mbarrier, and the chunk of each accumulator frequency is
// brought into L2 by one bulk prefetch, ahead of the wait for the last step.  The block's phases are staged
// in shared memory in the operand form of the paired instructions.  Measured per launch, before (one voxel
// a thread, 48 snapshot values in registers) and after: 128^3 voxels, 3 frequencies 0.213 -> 0.169 ms (5.9
// TB/s); 256 x 256 x 192, 3 frequencies 1.155 -> 0.911 ms (6.6 TB/s); 26 x 101 x 101, 8 frequencies 0.091 ->
// 0.076 ms (its FP64 additions and conversions alone take 0.04).  Resident blocks 3 / 4 / 5 / 6: 0.203 /
// 0.179 / 0.169 / 0.186 ms.
#pragma once
#include "fdtd_step.cuh"

namespace fdtd {

constexpr int kDftThreads = 256;
constexpr int kDftChunk = 2 * kDftThreads;   // samples per block

template <typename T>
struct DftSmem {
    static constexpr size_t snaps = (size_t)kMaxSnap * kDftChunk * sizeof(T);
    static constexpr size_t phases = (size_t)kMaxFreq * kMaxSnap * 4 * sizeof(T);
    static constexpr size_t total = snaps + phases + 16;
};

__device__ __forceinline__ void bulk_load(void* dst, const void* src, unsigned bytes, uint64_t* bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_addr(dst)),
                 "l"(src), "r"(bytes), "r"(smem_addr(bar))
                 : "memory");
}

__device__ __forceinline__ void bulk_prefetch_l2(const void* src, unsigned bytes)
{
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}

template <typename T>
__global__ void __launch_bounds__(kDftThreads, sizeof(T) == 4 ? 5 : 2) dft_kernel(const DParams<T> d, int cnt)
{
    using V = typename Pair<T>::V;
    extern __shared__ __align__(128) unsigned char dft_smem[];
    T* es = (T*)dft_smem;                                              // [slot][kDftChunk]
    T* sph = (T*)(dft_smem + DftSmem<T>::snaps);                       // [f][s]: cos, cos, -sin, -sin
    uint64_t* bar = (uint64_t*)(dft_smem + DftSmem<T>::snaps + DftSmem<T>::phases);
    const int tid = threadIdx.x;
    const long long ne = 3 * d.nd, q0 = (long long)blockIdx.x * kDftChunk;
    const int len = (int)(ne - q0 < kDftChunk ? ne - q0 : kDftChunk);  // samples of this block
    if (tid == 0) {
        mbar_init(bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_async_shared();
        for (int f = 0; f < d.nf; ++f) bulk_prefetch_l2(d.dft + f * ne + q0, (unsigned)len * (unsigned)sizeof(double2));
    }
    pdl_wait();                                    // the snapshots of the block's last step
    pdl_trigger();
    const int n0 = __ldcg(d.ctl + 3);
    if (tid == 0) {
        // slots are padded to a multiple of 16 bytes, so the last chunk's copy may be rounded up to one
        const unsigned bytes = ((unsigned)len * (unsigned)sizeof(T) + 15u) / 16u * 16u;
        mbar_expect_tx(bar, bytes * (unsigned)cnt);
        for (int s = 0; s < cnt; ++s)
            bulk_load(es + s * kDftChunk, d.snap + (long long)((n0 + s) % d.K) * d.snap_stride + q0, bytes, bar);
    }
    for (int t = tid; t < cnt * d.nf; t += kDftThreads) {
        const auto ph = __ldg(d.ph + (long long)(n0 + 1) * d.nf + t);
        const int s = t / d.nf, f = t - s * d.nf;
        T* o = sph + (f * kMaxSnap + s) * 4;
        o[0] = o[1] = ph.x;
        o[2] = o[3] = -ph.y;                       // e (-sin) = -(e sin) exactly
    }
    __syncthreads();
    if (!patient_wait([&] { return mbar_try_wait(bar, 0); }, [] { return global_ns(); }, kWaitNs)) {
        if (tid == 0) atomicOr(d.ctl + 2, 4);
        return;
    }
    const bool on0 = tid < len, on1 = tid + kDftThreads < len;
    if (!on0) return;
    V e[kMaxSnap];
#pragma unroll
    for (int s = 0; s < kMaxSnap; ++s)
        if (s < cnt) e[s] = pv<V>(es[s * kDftChunk + tid], on1 ? es[s * kDftChunk + kDftThreads + tid] : T(0));
    for (int f = 0; f < d.nf; ++f) {
        double2* acc = d.dft + f * ne + q0 + tid;
        double2 a0 = acc[0], a1 = on1 ? acc[kDftThreads] : double2{0.0, 0.0};
        V re = pv<V>(T(0), T(0)), im = re;
#pragma unroll
        for (int s = 0; s < kMaxSnap; ++s) {
            if (s < cnt) {
                const T* o = sph + (f * kMaxSnap + s) * 4;
                re = p_fma(e[s], ld2<V>(o), re);
                im = p_fma(e[s], ld2<V>(o + 2), im);
            }
        }
        a0.x += (double)re.x;
        a0.y += (double)im.x;
        acc[0] = a0;
        if (on1) {
            a1.x += (double)re.y;
            a1.y += (double)im.y;
            acc[kDftThreads] = a1;
        }
    }
}

}  // namespace fdtd
