// Launch wrappers and helper kernels; explicit FP32 / FP64 instantiations.
#include <mutex>
#include <utility>

#include "fdtd_design2.cuh"
#include "fdtd_dft.cuh"
#include "fdtd_kernels.cuh"
#include "fdtd_launch.h"
#include "fdtd_shell2.cuh"
#include "fdtd_step.cuh"

namespace fdtd {

__global__ void gap_gather_kernel(const double2* dft, long long nd, int nf, int d0, int d2, int d4, int dnx, int dny,
                                  int g0, int g1, int g2, int g3, int g4, int g5, double2* out)
{
    const int gnx = g1 - g0, gny = g3 - g2, gnz = g5 - g4;
    const long long ng = (long long)gnx * gny * gnz;
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= ng * 3 * nf) return;
    const long long gv = t % ng;
    const long long fc = t / ng;
    const int i = g0 + (int)(gv % gnx), j = g2 + (int)((gv / gnx) % gny), k = g4 + (int)(gv / ((long long)gnx * gny));
    const long long dv = ((long long)(k - d4) * dny + (j - d2)) * dnx + (i - d0);
    out[t] = dft[fc * nd + dv];
}

// Density import: float / double source -> T, with a range / finiteness check (flag bit 1).
template <typename T, typename S>
__global__ void rho_import_kernel(const S* src, long long n, T* dst, int* flag)
{
    const long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= n) return;
    const S r = src[v];
    if (!(r >= S(0) && r <= S(1))) atomicOr(flag, 2);
    dst[v] = (T)r;
}

template <typename T>
__global__ void to_double_kernel(const T* src, long long n, double* dst)
{
    const long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (v < n) dst[v] = (double)src[v];
}

// Integer maps from the same index helpers the update kernels use.
template <typename T>
__global__ void index_map_kernel(const KParams<T> p, int which, int32_t* out)
{
    const int i = blockIdx.x * kBX + threadIdx.x;
    const int j = blockIdx.y * kBY + threadIdx.y;
    const int k = blockIdx.z;
    if (i >= p.nx || j >= p.ny) return;
    const long long id = ((long long)k * p.ny + j) * p.nx + i;
    const bool in_d = in_box(p.db, i, j, k);
    const bool in_g = in_d && in_box(p.gb, i, j, k);
    if (which == 2) {
        out[id] = in_d ? (int32_t)(((long long)(k - p.db[4]) * p.dny + (j - p.db[2])) * p.dnx + (i - p.db[0])) : -1;
        return;
    }
    if (which == 3) {
        out[id] = in_g ? (int32_t)(((long long)(k - p.gb[4]) * p.gny + (j - p.gb[2])) * p.gnx + (i - p.gb[0])) : -1;
        return;
    }
    const int l[3] = {i, j, k};
    const int sl[3] = {slab_index(i, p.cpl[0], p.cph[0], p.nx), slab_index(j, p.cpl[1], p.cph[1], p.ny),
                       slab_index(k, p.cpl[2], p.cph[2], p.nz)};
    for (int c = 0; c < 3; ++c) {
        int32_t v = 0;
        for (int t = 0; t < 2; ++t) {
            const int a = (c + 1 + t) % 3;
            const T* tab = (which == 0) ? p.pmlE[a] : p.pmlH[a];
            if (sl[a] >= 0 && tab[4 * sl[a] + 2] != T(0)) v |= 1 << (3 + t);
        }
        if (which == 0) {
            v |= in_g ? 2 : ((in_d && in_box(p.mb[c], i, j, k)) ? 1 : 0);
            bool fixed = false;
            for (int a = 0; a < 3; ++a)
                if (a != c && l[a] == 0) fixed = true;
            if (fixed) v |= 4;
            if (p.nb > 0 && in_box(p.sb, i, j, k)) {
                const long long lv = ((long long)(k - p.sb[4]) * (p.sb[3] - p.sb[2]) + (j - p.sb[2])) * (p.sb[1] - p.sb[0]) + (i - p.sb[0]);
                if (p.src_r[(lv * 3 + c) * p.nb] != T(0)) v |= 32;
            }
        }
        out[(long long)c * p.ncell + id] = v;
    }
}

static dim3 grid3(int nx, int ny, int nz) { return dim3((nx + kBX - 1) / kBX, (ny + kBY - 1) / kBY, nz); }

// Launch of a kernel of the step chain; pdl: as a programmatic dependent launch (its blocks may start
// before the kernel before it in the stream has completed; see pdl_wait / pdl_trigger).
template <typename... KArgs, typename... Args>
static cudaError_t launch_chain(void (*k)(KArgs...), dim3 g, dim3 b, size_t smem, cudaStream_t s, bool pdl,
                                Args&&... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = g;
    cfg.blockDim = b;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k, std::forward<Args>(args)...);
}

int pole_bucket(int max_poles)
{
    return max_poles == 0 ? 0 : max_poles <= 4 ? 4 : max_poles <= 8 ? 8 : 16;
}

// Dynamic shared memory limits of the kernels that need them raised, once per device and type.
template <typename T>
cudaError_t prepare_step(int device)
{
    static std::mutex mutex;
    static unsigned long long done = 0;   // bit per device (ordinals below 64)
    std::lock_guard<std::mutex> lock(mutex);
    if (done >> device & 1) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(dft_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)DftSmem<T>::total);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(step_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)StepSmem<T>::total);
    if (e == cudaSuccess) done |= 1ull << device;
    return e;
}

// A kernel node of a step graph (no dependencies yet; the host adds them).
template <typename... KArgs, typename... Args>
static cudaError_t graph_kernel(cudaGraph_t g, cudaGraphNode_t* node, void (*k)(KArgs...), dim3 grid, dim3 block,
                                size_t smem, Args... args)
{
    void* ptrs[] = {(void*)&args...};
    cudaKernelNodeParams kp = {};
    kp.func = (void*)k;
    kp.gridDim = grid;
    kp.blockDim = block;
    kp.sharedMemBytes = (unsigned)smem;
    kp.kernelParams = ptrs;
    return cudaGraphAddKernelNode(node, g, nullptr, 0, &kp);
}

template <typename T>
cudaError_t graph_step(cudaGraph_t g, cudaGraphNode_t* node, const KParams<T>& p, const StepMaps& m)
{
    const dim3 grid((p.ib[1] - p.ib[0] + kTX - 1) / kTX, (p.ib[3] - p.ib[2] + kTY - 1) / kTY, (p.ib[5] - p.ib[4] + p.kc - 1) / p.kc);
    return graph_kernel(g, node, step_kernel<T>, grid, dim3(kPX, kTY), StepSmem<T>::total, p, m);
}

template <typename T>
cudaError_t graph_shell(cudaGraph_t g, cudaGraphNode_t* node, const KParams<T>& p, const ShellBoxes& s, bool e_part)
{
    const dim3 grid(s.first[s.n]), b(kBX, kShellBY);
    if constexpr (sizeof(T) == 4) {
        if (s.pair)
            return e_part ? graph_kernel(g, node, shell_e2_kernel, grid, b, 0, p, s)
                          : graph_kernel(g, node, shell_h2_kernel, grid, b, 0, p, s);
    }
    if constexpr (sizeof(T) == 4) {
        if (s.pz == 1)
            return e_part ? graph_kernel(g, node, shell_e_kernel<T, 1>, grid, b, 0, p, s)
                          : graph_kernel(g, node, shell_h_kernel<T, 1>, grid, b, 0, p, s);
    }
    return e_part ? graph_kernel(g, node, shell_e_kernel<T, 2>, grid, b, 0, p, s)
                  : graph_kernel(g, node, shell_h_kernel<T, 2>, grid, b, 0, p, s);
}

// Grid of the design-E kernel: one block per (p.edz planes, component) of 256 columns (column pairs for
// the paired kernel) in row order.
template <typename T>
static dim3 design_grid(const KParams<T>& p, int nt = kBX * kBY)
{
    const unsigned nxy = (unsigned)((p.db[1] - p.db[0]) / (p.ed_pair ? 2 : 1)) * (unsigned)(p.db[3] - p.db[2]);
    const unsigned nz = (unsigned)(p.db[5] - p.db[4]);
    return dim3((nxy + nt - 1) / nt, 1, 3 * ((nz + p.edz - 1) / p.edz));
}

template <typename T>
cudaError_t graph_e_design(cudaGraph_t g, cudaGraphNode_t* node, const KParams<T>& p, const PoleTable<T>& tab, int bucket)
{
    const dim3 b(kBX, kBY), grid = design_grid(p);
    if constexpr (sizeof(T) == 4) {
        if (p.ed_pair) switch (bucket) {
            case 0: return graph_kernel(g, node, e_design2_kernel<0>, grid, b, 0, p, tab);
            case 4: return graph_kernel(g, node, e_design2_kernel<4>, grid, b, 0, p, tab);
            case 8: return graph_kernel(g, node, e_design2_kernel<8>, grid, b, 0, p, tab);
            default: return cudaErrorInvalidValue;   // the host pairs only up to 8 poles a component
            }
    }
    switch (bucket) {
    case 0: return graph_kernel(g, node, e_design_kernel<T, 0>, grid, b, 0, p, tab);
    case 4: return graph_kernel(g, node, e_design_kernel<T, 4>, grid, b, 0, p, tab);
    case 8: return graph_kernel(g, node, e_design_kernel<T, 8>, grid, b, 0, p, tab);
    default: return graph_kernel(g, node, e_design_kernel<T, 16>, grid, b, 0, p, tab);
    }
}

// The E phase as one launch (FP32, up to 4 poles a component), where the launches are what the phase costs: columns
// of one plane and, with the one-sample design kernel, blocks that are resident at once; false: it takes two.
// 48^3 step 7.6 -> 7.25 us, 56^3 8.35 -> 8.05, 64^3 10.4 -> 9.8, 96 x 64 x 48 10.65 -> 10.2, 44^3 (one-sample) 7.0 -> 6.5.
// With longer columns the design box's blocks only hold the shell's up (72^3 11.2 -> 12.0), and so do the one-sample
// kernel's past one round (56^3 8.45 -> 8.85).
template <typename T>
bool graph_e_phase(cudaGraph_t g, cudaGraphNode_t* node, const KParams<T>& p, const ShellBoxes& s, const PoleTable<T>& tab,
                   int bucket, cudaError_t* e)
{
    if constexpr (sizeof(T) == 4) {
        const dim3 dg = design_grid(p, kShellNT), grid(dg.x * dg.z + s.first[s.n]), b(kBX, kShellBY);
        if (bucket > 4 || s.kz > 1 || (!p.ed_pair && grid.x > 8 * 152)) return false;
        void (*k)(KParams<float>, ShellBoxes, PoleTable<float>, unsigned, unsigned);
        if (bucket == 0)
            k = p.ed_pair ? (s.pair ? e_phase_kernel<true, true, 0> : e_phase_kernel<false, true, 0>)
                          : (s.pair ? e_phase_kernel<true, false, 0> : e_phase_kernel<false, false, 0>);
        else
            k = p.ed_pair ? (s.pair ? e_phase_kernel<true, true, 4> : e_phase_kernel<false, true, 4>)
                          : (s.pair ? e_phase_kernel<true, false, 4> : e_phase_kernel<false, false, 4>);
        *e = graph_kernel(g, node, k, grid, b, 0, p, s, tab, dg.x, dg.z);
        return true;
    }
    return false;
}

template <typename T>
static dim3 dft_grid(const DParams<T>& d)
{
    return dim3((unsigned)((3 * d.nd + kDftChunk - 1) / kDftChunk));
}

template <typename T>
cudaError_t graph_dft(cudaGraph_t g, cudaGraphNode_t* node, const DParams<T>& d, int cnt)
{
    return graph_kernel(g, node, dft_kernel<T>, dft_grid(d), dim3(kDftThreads), DftSmem<T>::total, d, cnt);
}

// One thread each: the first step of a block of steps for its DFT launch, and the step counter moved on.
__global__ void block_begin_kernel(int* ctl) { ctl[3] = ctl[0]; }
__global__ void block_end_kernel(int* ctl, int cnt)
{
    pdl_wait();
    ctl[0] += cnt;
}

cudaError_t graph_block_begin(cudaGraph_t g, cudaGraphNode_t* node, int* ctl)
{
    return graph_kernel(g, node, block_begin_kernel, dim3(1), dim3(1), 0, ctl);
}

cudaError_t graph_block_end(cudaGraph_t g, cudaGraphNode_t* node, int* ctl, int cnt)
{
    return graph_kernel(g, node, block_end_kernel, dim3(1), dim3(1), 0, ctl, cnt);
}

template <typename T>
cudaError_t launch_step(const KParams<T>& p, const StepMaps& m, cudaStream_t s, bool pdl)
{
    const dim3 g((p.ib[1] - p.ib[0] + kTX - 1) / kTX, (p.ib[3] - p.ib[2] + kTY - 1) / kTY, (p.ib[5] - p.ib[4] + p.kc - 1) / p.kc);
    return launch_chain(step_kernel<T>, g, dim3(kPX, kTY), StepSmem<T>::total, s, pdl, p, m);
}

// Shape of the shell launches: z planes per thread, by an estimate of the busiest SM's time.  A column is a serial
// chain: with c blocks resident a plane (FP64: its arithmetic's latency) waits L and a plane takes c t of the SM; an SM
// runs its b blocks C at a time, and every block costs the launch g.  L, t, g (us) and C are read off steps of
// 48^3 to 192^3 grids and of 96 x 170 x 170 with every depth from 1 to 16.  What it decides: one full round of long
// columns instead of one and a little (96 x 170 x 170: depth 9, 1216 blocks, a step 55.6 us; depth 8, 68 before), and
// short columns where a grid has few of them (48^3: depth 1 7.3 us, 2 8.2, 4 11.2).  Past three rounds only L/C + t a
// plane matters, which the depth does not change, and it stays at kLongColumn.
// Beside an interior kernel (FP32) the estimate is kept unless it takes shorter columns than kLongColumn in more than one
// round and those of kLongColumn would not leave a round nearly empty (1.2 to 1.6 rounds of blocks): it counts every column at full depth, while most are
// the few planes of a z slab, which no depth changes.  A step with the estimate's depth / with 8 (rounds of 8): 216^3, 4-cell
// CPML (0.9) 129.6 / 126.4 us; 244 x 247 x 247, 4 (1.1) 200 / 192; 220 x 260 x 240, 2 (1.2) 195 / 186; 328 x 376 x 306, 4 (1.8)
// 524 / 502; 260 x 252 x 240, 10 (2.3) 224 / 219; but 296^3, 4 (1.3) 313 / 316, 244^3, 4 (1.3) 191 / 195, 252^3, 4 (1.4) 215 / 216,
// 228 x 204 x 224, 8 (1.5) 195.4 / 196.5, 280^3, 4 (1.5) 268 / 272, and 128^3, 8 (0.9 rounds of the estimate's 4) 42.3 / 47.4.
// Blocks of 128 threads, not 256: they spread more evenly over the SMs (FP64 32^3 step 12.2 -> 10.8 us,
// 88^3 19.8 -> 15.5, 121 x 81 x 95 23.9 -> 23.2, 75 x 61 x 83 11.9 -> 11.5, 128^3 and up within 1%).
void shell_shape(ShellBoxes& s, int type_bytes, size_t ncell, bool beside)
{
    const bool f64 = type_bytes == 8;
    s.pz = f64 || ncell >= kShellTwoPlaneCells ? 2 : 1;
    const double L = f64 ? 1.2 : 0.7, t = f64 ? 1.65 : (s.pair ? 0.225 : 0.125), g = 0.001;
    const unsigned C = f64 ? 4 : 8, sms = 152;
    auto blocks = [&](int kz) {
        unsigned n = 0;
        for (int q = 0; q < s.n; ++q) {
            const int* B = s.b[q];
            const unsigned wxy = (unsigned)(B[1] - B[0]) / (s.pair ? 2u : 1u) * (unsigned)(B[3] - B[2]);
            s.first[q] = n;
            n += (wxy + kShellNT - 1) / kShellNT * (unsigned)((B[5] - B[4] + kz - 1) / kz);
        }
        s.first[s.n] = n;
        return n;
    };
    constexpr int kLongColumn = 8;
    double best = 0.0;
    s.kz = 0;
    for (int kz = 1; kz <= kShellKZ; ++kz) {
        const unsigned nb = blocks(kz), b = (nb + sms - 1) / sms;
        if (kz > kLongColumn && b > 3 * C) continue;
        const double cost = (b / C) * (kz * L + kz * C * t) + (b % C ? kz * L + kz * (b % C) * t : 0.0) + g * nb;
        if (s.kz == 0 || cost < best) {
            best = cost;
            s.kz = kz;
        }
    }
    if (const unsigned round = C * sms; beside && !f64 && s.kz < kLongColumn && blocks(s.kz) > round) {
        const unsigned n = blocks(kLongColumn);
        if (n <= round * 6 / 5 || n >= round * 8 / 5) s.kz = kLongColumn;
    }
    blocks(s.kz);
}

template <typename T>
cudaError_t launch_shell(const KParams<T>& p, const ShellBoxes& s, bool e_part, cudaStream_t st, bool pdl)
{
    const unsigned nb = s.first[s.n];
    if (nb == 0) return cudaSuccess;
    const dim3 b(kBX, kShellBY);
    if constexpr (sizeof(T) == 4) {
        if (s.pair)
            return e_part ? launch_chain(shell_e2_kernel, dim3(nb), b, 0, st, pdl, p, s)
                          : launch_chain(shell_h2_kernel, dim3(nb), b, 0, st, pdl, p, s);
    }
    if constexpr (sizeof(T) == 4) {
        if (s.pz == 1)
            return e_part ? launch_chain(shell_e_kernel<T, 1>, dim3(nb), b, 0, st, pdl, p, s)
                          : launch_chain(shell_h_kernel<T, 1>, dim3(nb), b, 0, st, pdl, p, s);
    }
    return e_part ? launch_chain(shell_e_kernel<T, 2>, dim3(nb), b, 0, st, pdl, p, s)
                  : launch_chain(shell_h_kernel<T, 2>, dim3(nb), b, 0, st, pdl, p, s);
}

template <typename T>
cudaError_t launch_e_design(const KParams<T>& p, const PoleTable<T>& tab, int bucket, cudaStream_t s, bool pdl)
{
    if (p.nd == 0) return cudaSuccess;
    const dim3 b(kBX, kBY), g = design_grid(p);
    if constexpr (sizeof(T) == 4) {
        if (p.ed_pair) switch (bucket) {
            case 0: return launch_chain(e_design2_kernel<0>, g, b, 0, s, pdl, p, tab);
            case 4: return launch_chain(e_design2_kernel<4>, g, b, 0, s, pdl, p, tab);
            case 8: return launch_chain(e_design2_kernel<8>, g, b, 0, s, pdl, p, tab);
            default: return cudaErrorInvalidValue;   // the host pairs only up to 8 poles a component
            }
    }
    switch (bucket) {
    case 0: return launch_chain(e_design_kernel<T, 0>, g, b, 0, s, pdl, p, tab);
    case 4: return launch_chain(e_design_kernel<T, 4>, g, b, 0, s, pdl, p, tab);
    case 8: return launch_chain(e_design_kernel<T, 8>, g, b, 0, s, pdl, p, tab);
    default: return launch_chain(e_design_kernel<T, 16>, g, b, 0, s, pdl, p, tab);
    }
}

template <typename T>
cudaError_t launch_dft(const DParams<T>& d, int cnt, cudaStream_t s, bool pdl)
{
    if (d.nd == 0 || cnt <= 0) return cudaSuccess;
    return launch_chain(dft_kernel<T>, dft_grid(d), dim3(kDftThreads), DftSmem<T>::total, s, pdl, d, cnt);
}


cudaError_t launch_block_begin(int* ctl, cudaStream_t s)
{
    block_begin_kernel<<<1, 1, 0, s>>>(ctl);
    return cudaGetLastError();
}

cudaError_t launch_block_end(int* ctl, int cnt, cudaStream_t s)
{
    block_end_kernel<<<1, 1, 0, s>>>(ctl, cnt);
    return cudaGetLastError();
}

// Planes per thread of the design-E kernel.  FP32: short columns spread evenly and leave more loads in flight,
// long ones prefetch their next plane, which counts the more the less of the box L2 holds.  Steps measured with 1, 2, 3,
// 5, 8 planes, by the rounds (of 4 blocks an SM) that a launch of one-plane columns takes: 112^3 (2 rounds) 25.3 25.3
// 25.7 27.6 30.2 us; 96 x 170 x 170 (3) 60.5 60.2 60.6 60.3 63.0; 128^3 (3) 36.7 36.2 36.3 37.5 39.9; 192^3 (9) 124.1
// 120.5 120.6 121.3 123.3; 256^3 (20) 276.7 268.6 268.3 269.3 271.5; 512 x 512 x 384 (121) 1794 1691 1658 1644 1649.
// other_blocks: the shell's blocks of kShellNT threads, where the E phase is one launch: two planes where that makes it
// one round (64^3, 1024 of them: a step 8.1 -> 7.55 us).
// FP64: columns of kEdZ planes, halved while the launch has fewer than five blocks an SM.
int design_planes(int columns, int dnz, bool f64, unsigned other_blocks)
{
    constexpr unsigned sms = 152;
    const unsigned gxy = ((unsigned)columns + kBX * kBY - 1) / (kBX * kBY), one = gxy * 3 * (unsigned)dnz;
    if (f64) {
        int edz = kEdZ;
        while (edz > 1 && gxy * 3 * (((unsigned)dnz + edz - 1) / edz) < 5 * sms) edz = (edz + 1) / 2;
        return edz;
    }
    if (other_blocks) {
        const unsigned g = ((unsigned)columns + kShellNT - 1) / kShellNT;
        if (other_blocks + 3 * g * dnz > 8 * sms && other_blocks + 3 * g * ((dnz + 1) / 2) <= 8 * sms) return 2;
    }
    return one < 2 * 4 * sms ? 1 : (one < 12 * 4 * sms ? 2 : (one < 40 * 4 * sms ? 3 : 5));
}

template <typename T>
cudaError_t launch_grad(const GParams<T>& g, unsigned nblocks, cudaStream_t s)
{
    grad_kernel<T><<<nblocks, kReduceThreads, 0, s>>>(g);
    return cudaGetLastError();
}

cudaError_t launch_gap_gather(const double2* dft, long long nd, int nf, const int* db, int dnx, int dny, const int* gb,
                              double2* out, cudaStream_t s)
{
    const long long ng = (long long)(gb[1] - gb[0]) * (gb[3] - gb[2]) * (gb[5] - gb[4]);
    const long long nt = ng * 3 * nf;
    if (nt == 0) return cudaSuccess;
    gap_gather_kernel<<<(unsigned)((nt + 255) / 256), 256, 0, s>>>(dft, nd, nf, db[0], db[2], db[4], dnx, dny, gb[0], gb[1],
                                                                   gb[2], gb[3], gb[4], gb[5], out);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_rho_import(const void* src, int dtype, long long n, T* dst, int* flag, cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    const unsigned nb = (unsigned)((n + 255) / 256);
    if (dtype == 0)
        rho_import_kernel<T, float><<<nb, 256, 0, s>>>((const float*)src, n, dst, flag);
    else
        rho_import_kernel<T, double><<<nb, 256, 0, s>>>((const double*)src, n, dst, flag);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_to_double(const T* src, long long n, double* dst, cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    to_double_kernel<T><<<(unsigned)((n + 255) / 256), 256, 0, s>>>(src, n, dst);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_index_map(const KParams<T>& p, int which, int32_t* out, cudaStream_t s)
{
    index_map_kernel<T><<<grid3(p.nx, p.ny, p.nz), dim3(kBX, kBY), 0, s>>>(p, which, out);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_gather_design_e(const KParams<T>& p, T* out, cudaStream_t s)
{
    if (p.nd == 0) return cudaSuccess;
    gather_design_e_kernel<T><<<(unsigned)((p.nd + 255) / 256), 256, 0, s>>>(p, out);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_paper_drive(const T* gh, T* drive, int M, int ns, double eps0, cudaStream_t s)
{
    const long long n = (long long)M * ns;
    if (n == 0) return cudaSuccess;
    paper_drive_kernel<T><<<(unsigned)((n + 255) / 256), 256, 0, s>>>(gh, drive, M, ns, eps0);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_paper_grad(const PParams<T>& g, cudaStream_t s)
{
    if (g.nd == 0) return cudaSuccess;
    paper_grad_kernel<T><<<(unsigned)((g.nd + 255) / 256), 256, 0, s>>>(g);
    return cudaGetLastError();
}

// Gradient sums times the cell volume, in the caller's type.
template <typename O>
__global__ void paper_scale_kernel(const double* __restrict__ g, double dV, long long n, O* __restrict__ out)
{
    const long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (v < n) out[v] = (O)(g[v] * dV);
}

cudaError_t launch_paper_scale(const double* g, double dV, long long n, void* out, int dtype, cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    const unsigned nb = (unsigned)((n + 255) / 256);
    if (dtype == 1)
        paper_scale_kernel<double><<<nb, 256, 0, s>>>(g, dV, n, (double*)out);
    else
        paper_scale_kernel<float><<<nb, 256, 0, s>>>(g, dV, n, (float*)out);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_rho_scatter(const void* src, int dtype, long long n, const long long off[4], const int md[3][3],
                               int dnx, int dny, long long nd, T* dst, int* flag, cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    const int3 m0 = make_int3(md[0][0], md[0][1], md[0][2]), m1 = make_int3(md[1][0], md[1][1], md[1][2]);
    const int3 m2 = make_int3(md[2][0], md[2][1], md[2][2]);
    const unsigned nb = (unsigned)((n + 255) / 256);
    if (dtype == 0)
        rho_scatter_kernel<T, float><<<nb, 256, 0, s>>>((const float*)src, n, off[1], off[2], m0, m1, m2, dnx, dny, nd, dst, flag);
    else
        rho_scatter_kernel<T, double><<<nb, 256, 0, s>>>((const double*)src, n, off[1], off[2], m0, m1, m2, dnx, dny, nd, dst, flag);
    return cudaGetLastError();
}

#define FDTD_INSTANTIATE(T)                                                                              \
    template cudaError_t prepare_step<T>(int);                                                           \
    template cudaError_t graph_step<T>(cudaGraph_t, cudaGraphNode_t*, const KParams<T>&, const StepMaps&); \
    template cudaError_t graph_shell<T>(cudaGraph_t, cudaGraphNode_t*, const KParams<T>&, const ShellBoxes&, bool); \
    template cudaError_t graph_e_design<T>(cudaGraph_t, cudaGraphNode_t*, const KParams<T>&, const PoleTable<T>&, int); \
    template bool graph_e_phase<T>(cudaGraph_t, cudaGraphNode_t*, const KParams<T>&, const ShellBoxes&, const PoleTable<T>&, int, \
                                   cudaError_t*);                                                        \
    template cudaError_t graph_dft<T>(cudaGraph_t, cudaGraphNode_t*, const DParams<T>&, int);           \
    template cudaError_t launch_step<T>(const KParams<T>&, const StepMaps&, cudaStream_t, bool);         \
    template cudaError_t launch_shell<T>(const KParams<T>&, const ShellBoxes&, bool, cudaStream_t, bool); \
    template cudaError_t launch_e_design<T>(const KParams<T>&, const PoleTable<T>&, int, cudaStream_t, bool); \
    template cudaError_t launch_dft<T>(const DParams<T>&, int, cudaStream_t, bool);                      \
    template cudaError_t launch_grad<T>(const GParams<T>&, unsigned, cudaStream_t);                      \
    template cudaError_t launch_rho_import<T>(const void*, int, long long, T*, int*, cudaStream_t);      \
    template cudaError_t launch_rho_scatter<T>(const void*, int, long long, const long long*, const int (*)[3], int, \
                                               int, long long, T*, int*, cudaStream_t);                   \
    template cudaError_t launch_to_double<T>(const T*, long long, double*, cudaStream_t);                \
    template cudaError_t launch_index_map<T>(const KParams<T>&, int, int32_t*, cudaStream_t);            \
    template cudaError_t launch_gather_design_e<T>(const KParams<T>&, T*, cudaStream_t);                  \
    template cudaError_t launch_paper_drive<T>(const T*, T*, int, int, double, cudaStream_t);             \
    template cudaError_t launch_paper_grad<T>(const PParams<T>&, cudaStream_t);

FDTD_INSTANTIATE(float)
FDTD_INSTANTIATE(double)

}  // namespace fdtd
