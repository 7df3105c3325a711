// Density filter, smoothed-Heaviside projection and their chain rule (the paper's Sec. "Filtering and
// projection", Eqs. (FilterFunction), (Projection), (GradientsFiltered)) on the design box.
//
// The cone filter is a 3-D correlation with w(d) = R - |d| over |d| < R (voxels), neighbourhoods cut at
// the box faces.  A weight depends on the offset's row only through r2 = dy^2 + dz^2, so the rows of one r2 are
// added first and then correlated along x once: at R = 12 the sphere's 7153 taps in 437 rows become 58
// short correlations of 986 taps in all, and with the rows of +-dz added once per plane, 230 row additions.
// cone_kernel, a block: one z plane of 32 x 8 outputs, a warp per output row.
//   1. The planes z + dz and z - dz are added, for every |dz|, over the tile with its halo (zero outside the
//      box) into shared memory.
//   2. Per warp, 8 values of r2 at a time: the row sums of the warp's output row over the tile's x window, half a
//      warp an r2; then each of the 8 is correlated by four lanes of eight x-adjacent outputs, a sliding
//      window of inputs and four taps' weights at a time: two 16-byte shared loads feed 32 FMAs.
//   3. The eight partial sums of an output meet by shuffles.
// What the blocks share (weights, offsets) is made once per call by table_kernel.  At R = 12 two blocks of 106 KB
// share an SM, and it is their 16 warps' latencies that bound it (instructions issue in 54% of the cycles, the
// shared-memory pipe is 51% busy, the FMA pipe 23%).  Measured, a filter with its normalising sums (the
// chain rule takes as long): 128^3, R = 12 2.6 ms with every tap summed by a sliding window, 0.58 now; 64^3, R = 12
// 0.09 ms; 25 x 100 x 100, R = 3.5 0.025 ms (0.1 before, most of it on the host: the sums' table made there,
// copied from pageable memory and waited for).
//
// The normalising sums (the cone summed over the part of the sphere inside the box) depend only on each
// voxel's distances to the box faces: norm_sum takes them from a summed-volume table of the weights by
// inclusion-exclusion where they are used.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <mutex>
#include <string>

#include "fdtd_ccpr.h"
#include "fdtd_kernels.cuh"

namespace fdtd {
void set_thread_error(const std::string& msg);
}

namespace {

constexpr int kMaxHalo = 11;                   // R <= 12
constexpr int kOX = 32, kTY = 8;               // outputs of a block: kOX x kTY of one z plane
constexpr int kThreads = 32 * kTY;             // a warp per output row
constexpr int kBatch = 8;                      // values of r2 in hand at a time
constexpr int kMaxRows = 64, kMaxCombo = 128;  // values of r2, pairs (|dz|, |dy|) (R = 12: 58 and 121)
constexpr int kWPitch = 28;                    // weights of one r2 (at most 24)

__host__ __device__ constexpr int up4(int v) { return (v + 3) / 4 * 4; }

// Cone weight of squared distance d2: R - |d| inside the sphere |d| < R, else 0.
__host__ __device__ inline float cone_weight(int d2, float R)
{
    const float d = sqrtf((float)d2);
    return d < R ? R - d : 0.f;
}

// The sphere's rows by r2 = dy^2 + dz^2, ascending: half width m (taps |dx| <= m, which falls with r2), and the
// pairs (|dz|, |dy|) with that r2 in first[r] .. first[r + 1].
struct ConeRows {
    int n, nrows;
    short r2[kMaxRows], m[kMaxRows], first[kMaxRows + 1];
    unsigned char dz[kMaxCombo], dy[kMaxCombo];
};

ConeRows cone_rows(float R, int n)
{
    ConeRows c{};
    c.n = n;
    int k = 0;
    for (int r2 = 0; r2 <= 2 * n * n; ++r2) {
        if (!(cone_weight(r2, R) > 0.f)) break;
        const int k0 = k;
        for (int dz = 0; dz <= n; ++dz)
            for (int dy = 0; dy <= n; ++dy)
                if (dz * dz + dy * dy == r2) {
                    c.dz[k] = (unsigned char)dz;
                    c.dy[k++] = (unsigned char)dy;
                }
        if (k == k0) continue;
        int m = 0;
        while (m < n && cone_weight(r2 + (m + 1) * (m + 1), R) > 0.f) ++m;
        c.r2[c.nrows] = (short)r2;
        c.m[c.nrows] = (short)m;
        c.first[c.nrows++] = (short)k0;
    }
    c.first[c.nrows] = (short)k;
    return c;
}

// Layout of a tile in shared memory.  Window: from x0 - up4(n), far enough right for the last four taps.
struct ConeTile {
    int n4, w, ly;       // left halo, window, rows with halo
    int pitch;           // of a row sum: 4 mod 8, so that two r2's windows fall on different banks
    size_t planes, sums, meta;   // floats: planes [|dz|][ly][w] and kTY rows of zeros, row sums [warp][kBatch][pitch]
    __host__ __device__ explicit ConeTile(int n)
    {
        n4 = up4(n);
        w = kOX + n4 + up4(n + 1);
        ly = kTY + 2 * n;
        pitch = w % 8 == 4 ? w : w + 4;
        planes = (size_t)((n + 1) * ly + kTY) * w;
        sums = (size_t)kTY * kBatch * pitch;
        meta = (planes + sums) * sizeof(float);
    }
};

// What the blocks of a radius share, made once per call by table_kernel: the rows' weights from tap -up4(m) of
// their batch's first row (the widest) and zeros beyond |m|; per pair the plane offsets of its rows y + dy and
// y - dy (of the zeros for dy = 0) from the output's row; the pairs of a row; the batches' m.
struct __align__(16) ConeMeta {
    float w[kMaxRows * kWPitch];
    int2 pair[kMaxCombo];
    int first[kMaxRows + 1];
    int m[kMaxRows / kBatch];
};

// Summed-volume table of the weights in units of 2^-24, T[c][b][a] = sum over dz < c, dy < b, dx < a (offsets
// from -n): exact integers, as a weight of a sphere wider than one voxel (n > 0: R > 1) is a difference of
// two floats of at least 1, a multiple of 2^-23 whatever its rounding.  (FP64 sums are as exact, but GB300 does
// two a clock and SM.)
constexpr float kUnit = 1.f / (1 << 24);

// Normalising sum of a voxel: offsets dx in [-min(x, n), min(nx-1-x, n)] and likewise in y, z, by
// inclusion-exclusion; a voxel n or more from every face takes the whole sum.  One rounding, to float.
__device__ __forceinline__ float norm_sum(const long long* __restrict__ T, int n, float R, int x, int y, int z, int nx,
                                          int ny, int nz)
{
    if (n == 0) return R;                     // the voxel alone
    const int E = 2 * n + 2;                  // table extent per axis
    const int a0 = n - min(x, n), a1 = n + min(nx - 1 - x, n) + 1;
    const int b0 = n - min(y, n), b1 = n + min(ny - 1 - y, n) + 1;
    const int c0 = n - min(z, n), c1 = n + min(nz - 1 - z, n) + 1;
    auto t = [&](int c, int b, int a) { return __ldg(T + (c * E + b) * E + a); };
    long long s = t(c1, b1, a1);
    if (a0 + b0 + c0 != 0 || a1 + b1 + c1 != 3 * (E - 1))
        s += t(c0, b0, a1) + t(c0, b1, a0) + t(c1, b0, a0) - t(c0, b1, a1) - t(c1, b0, a1) - t(c1, b1, a0) - t(c0, b0, a0);
    return __ll2float_rn(s) * kUnit;
}

__host__ __device__ inline size_t table_words(int n) { return (size_t)(2 * n + 2) * (2 * n + 2) * (2 * n + 2); }

// One block: the shared data of the radius; the table: the weights of a row (c, b) summed along a in its thread,
// then along b and c in shared memory.
__global__ void __launch_bounds__(1024) table_kernel(long long* __restrict__ T, const __grid_constant__ ConeRows rows, float R)
{
    extern __shared__ long long tab[];
    const int n = rows.n;
    ConeMeta* meta = (ConeMeta*)(T + table_words(n));
    const ConeTile tile(n);
    for (int q = threadIdx.x; q < rows.nrows * kWPitch; q += blockDim.x) {
        const int r = q / kWPitch, m = rows.m[r], dx = q - r * kWPitch - up4(rows.m[r / kBatch * kBatch]);
        meta->w[q] = dx >= -m && dx <= m ? cone_weight(rows.r2[r] + dx * dx, R) : 0.f;
    }
    for (int q = threadIdx.x; q < rows.first[rows.nrows]; q += blockDim.x) {
        const int base = rows.dz[q] * tile.ly * tile.w, dy = rows.dy[q];
        meta->pair[q] = make_int2(base + (n + dy) * tile.w, dy ? base + (n - dy) * tile.w : (n + 1) * tile.ly * tile.w);
    }
    for (int q = threadIdx.x; q <= rows.nrows; q += blockDim.x) {
        meta->first[q] = rows.first[q];
        if (q < rows.nrows && q % kBatch == 0) meta->m[q / kBatch] = rows.m[q];
    }
    if (n == 0) return;                       // the sums are the voxel's own weight
    const int E = 2 * n + 2, E2 = E * E;
    for (int l = threadIdx.x; l < E2; l += blockDim.x) {
        const int c = l / E - 1 - n, b = l % E - 1 - n;
        long long s = 0;
        tab[l * E] = 0;
        for (int a = -n; a <= n; ++a) {
            if (c >= -n && b >= -n) s += (long long)(cone_weight(a * a + b * b + c * c, R) * (1.f / kUnit));
            tab[l * E + a + n + 1] = s;
        }
    }
    for (int axis = 1; axis < 3; ++axis) {
        __syncthreads();
        const int step = axis == 1 ? E : E2;
        for (int l = threadIdx.x; l < E2; l += blockDim.x) {
            int q = axis == 1 ? l / E * E2 + l % E : l;
            long long s = 0;
            for (int k = 0; k < E; ++k, q += step) {
                s += tab[q];
                tab[q] = s;
            }
        }
    }
    __syncthreads();
    for (int q = threadIdx.x; q < E * E2; q += blockDim.x) T[q] = tab[q];
}

struct ConvArgs {
    const float* in;
    float* out;
    const ConeMeta* meta;
    const long long* table;   // optional: out = sum / normalising sum
    float* proj;           // optional: projection of out
    int nx, ny, nz, n, nrows;
    float R, beta, eta, pden;
};

// Four inputs of a row from column x, zero outside [0, nx).  VEC: nx and x are multiples of four and the row
// starts on 16 bytes, so the four are inside or outside together.
template <bool VEC>
__device__ __forceinline__ float4 load4(const float* row, int x, int nx)
{
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (VEC) {
        if ((unsigned)x < (unsigned)nx) v = __ldg(reinterpret_cast<const float4*>(row + x));
        return v;
    }
    if ((unsigned)x < (unsigned)nx) v.x = __ldg(row + x);
    if ((unsigned)(x + 1) < (unsigned)nx) v.y = __ldg(row + x + 1);
    if ((unsigned)(x + 2) < (unsigned)nx) v.z = __ldg(row + x + 2);
    if ((unsigned)(x + 3) < (unsigned)nx) v.w = __ldg(row + x + 3);
    return v;
}

__device__ __forceinline__ float4 add4(float4 a, float4 b)
{
    const float2 l = __fadd2_rn(make_float2(a.x, a.y), make_float2(b.x, b.y));
    const float2 h = __fadd2_rn(make_float2(a.z, a.w), make_float2(b.z, b.w));
    return make_float4(l.x, l.y, h.x, h.y);
}

// Eight outputs of a lane from one tap: window values j .. j + 7.
__device__ __forceinline__ void tap8(float w, const float* v, int j, float (&acc)[8])
{
#pragma unroll
    for (int k = 0; k < 8; ++k) acc[k] = fmaf(w, v[k + j], acc[k]);
}

// The batch's correlation of a lane: its r2's row sums from p, weights from w, taps 0 .. last.  GUARD: a zero
// weight, which pads the row's taps, leaves its inputs out (they are not the output's; only their being
// infinite, NaN or huge would show).
template <bool GUARD>
__device__ __forceinline__ void correlate8(const float* p, const float* w, int last, float (&acc)[8])
{
    float v[12];
    *reinterpret_cast<float4*>(v) = *reinterpret_cast<const float4*>(p);
    *reinterpret_cast<float4*>(v + 4) = *reinterpret_cast<const float4*>(p + 4);
#pragma unroll
    for (int t = 0; t < 24; t += 4) {        // unrolled, so that the window moves by renaming
        if (t > last) break;
        const float4 wt = *reinterpret_cast<const float4*>(w + t);
        *reinterpret_cast<float4*>(v + 8) = *reinterpret_cast<const float4*>(p + t + 8);
        if (!GUARD || wt.x != 0.f) tap8(wt.x, v, 0, acc);
        if (!GUARD || wt.y != 0.f) tap8(wt.y, v, 1, acc);
        if (!GUARD || wt.z != 0.f) tap8(wt.z, v, 2, acc);
        if (!GUARD || wt.w != 0.f) tap8(wt.w, v, 3, acc);
#pragma unroll
        for (int k = 0; k < 8; ++k) v[k] = v[k + 4];
    }
}

__device__ __forceinline__ bool small4(float4 v)
{
    return fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w))) <= 1e37f && v.x == v.x && v.y == v.y &&
           v.z == v.z && v.w == v.w;
}

template <bool VEC>
__global__ void __launch_bounds__(kThreads, 2) cone_kernel(const ConvArgs a)
{
    extern __shared__ __align__(16) float cone_smem[];
    const ConeTile tile(a.n);
    const int n = a.n, W = tile.w, W4 = W / 4, ly = tile.ly;
    float *planes = cone_smem, *sums = planes + tile.planes;
    ConeMeta* meta = (ConeMeta*)((unsigned char*)cone_smem + tile.meta);
    const int tid = threadIdx.x, lane = tid & 31, ty = tid >> 5;
    const int ntx = (a.nx + kOX - 1) / kOX, z = blockIdx.x / ntx;
    const int x0 = (blockIdx.x - z * ntx) * kOX, y0 = blockIdx.y * kTY;
    for (int q = tid; q < (int)(sizeof(ConeMeta) / 16); q += kThreads)
        reinterpret_cast<float4*>(meta)[q] = __ldg(reinterpret_cast<const float4*>(a.meta) + q);
    for (int q = tid; q < kTY * W4; q += kThreads) reinterpret_cast<float4*>(planes)[(n + 1) * ly * W4 + q] = float4{};
    // half a warp a row (W4 <= 14), row (dz, ry) after row
    const int half = tid >> 4, x4 = tid & 15;
    const long long plane = (long long)a.ny * a.nx;
    bool large = false;
    if (x4 < W4) {
        const int xl = x0 - tile.n4 + 4 * x4;
        for (int r = half, dz = r / ly, ry = r - dz * ly; dz <= n; r += kThreads / 16) {
            const int yl = y0 - n + ry;
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if ((unsigned)yl < (unsigned)a.ny) {
                const float* row = a.in + z * plane + (long long)yl * a.nx;
                if (z + dz < a.nz) v = load4<VEC>(row + dz * plane, xl, a.nx);
                if (dz && z >= dz) v = add4(v, load4<VEC>(row - dz * plane, xl, a.nx));
                large |= !small4(v);
            }
            reinterpret_cast<float4*>(planes)[r * W4 + x4] = v;
            for (ry += kThreads / 16; ry >= ly; ry -= ly) ++dz;
        }
    }
    const bool guard = __syncthreads_or(large);
    const int y = y0 + ty;
    if (y >= a.ny) return;                       // whole warps; no block barrier below
    float* ws = sums + ty * kBatch * tile.pitch;
    const float* prow = planes + ty * W + 4 * x4;
    const int g = lane >> 2, o = 8 * (lane & 3);  // this lane's r2 of the batch, its first output
    float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    for (int r0 = 0; r0 < a.nrows; r0 += kBatch) {
        const int nb = min(kBatch, a.nrows - r0);
        __syncwarp();
        if (x4 < W4)
            for (int b = lane >> 4; b < nb; b += 2) {    // half a warp an r2
                float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
                const int k1 = meta->first[r0 + b + 1];
                for (int k = meta->first[r0 + b]; k < k1; ++k) {
                    const int2 off = meta->pair[k];
                    s = add4(s, add4(*reinterpret_cast<const float4*>(prow + off.x),
                                     *reinterpret_cast<const float4*>(prow + off.y)));
                }
                *reinterpret_cast<float4*>(ws + b * tile.pitch + 4 * x4) = s;
            }
        __syncwarp();
        if (g < nb) {
            const int m = meta->m[r0 / kBatch], m4 = up4(m);
            const float *p = ws + g * tile.pitch + tile.n4 - m4 + o, *w = meta->w + (r0 + g) * kWPitch;
            if (guard)
                correlate8<true>(p, w, m4 + m, acc);
            else
                correlate8<false>(p, w, m4 + m, acc);
        }
    }
    float s = 0.f;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
#pragma unroll
        for (int d = 4; d < 32; d *= 2) acc[k] += __shfl_xor_sync(0xffffffffu, acc[k], d);
        if (k == g) s = acc[k];                  // lane (g, o / 8) keeps output o + g
    }
    const int x = x0 + o + g;
    if (x >= a.nx) return;
    const long long v = ((long long)z * a.ny + y) * a.nx + x;
    if (a.table) s /= norm_sum(a.table, n, a.R, x, y, z, a.nx, a.ny, a.nz);
    a.out[v] = s;
    if (a.proj) a.proj[v] = (tanhf(a.beta * a.eta) + tanhf(a.beta * (s - a.eta))) / a.pden;
}

// g = dF/drho_b * drho_b/drho_t / W  (the input of the transposed filter)
__global__ void chain_pre_kernel(const float* dFb, const float* rho_t, const long long* T, int n, float R, float* g, int nx,
                                 int ny, int nz, float beta, float eta, float pden)
{
    const long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= (long long)nx * ny * nz) return;
    const int x = (int)(v % nx), y = (int)((v / nx) % ny), z = (int)(v / ((long long)nx * ny));
    const float t = tanhf(beta * (rho_t[v] - eta));
    g[v] = dFb[v] * beta * (1.f - t * t) / pden / norm_sum(T, n, R, x, y, z, nx, ny, nz);
}

fdtd_status fail(fdtd_status c, const std::string& m)
{
    fdtd::set_thread_error(m);
    return c;
}

fdtd_status check(int nx, int ny, int nz, double R, double beta, double eta)
{
    if (nx < 1 || ny < 1 || nz < 1) return fail(FDTD_ERR_ARG, "filter: empty box");
    if (!(R > 0.0 && R <= kMaxHalo + 1)) return fail(FDTD_ERR_ARG, "filter: radius must be in (0, 12] voxels");
    if (!(beta > 0.0) || !(eta >= 0.0 && eta <= 1.0)) return fail(FDTD_ERR_ARG, "projection: beta > 0, eta in [0,1]");
    return FDTD_OK;
}

int halo(double R) { return (int)std::ceil(R) - 1; }

// The scratch of a radius: the normalising sums' table, the blocks' shared data (16-byte aligned: 8 | table words).
size_t table_bytes(int n) { return table_words(n) * sizeof(long long) + sizeof(ConeMeta); }

// A kernel's limit of dynamic shared memory is the device's, whoever launches: every call sets it to the largest
// radius's need, so that no call can lower it between another thread's setting and its launch.
template <typename K>
cudaError_t allow_smem(K kernel, size_t most)
{
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
}

size_t cone_smem_bytes(int n) { return ConeTile(n).meta + sizeof(ConeMeta); }
size_t table_smem_bytes(int n) { return table_words(n) * sizeof(long long); }

cudaError_t conv(const float* in, float* out, const long long* T, bool normalise, float* proj, int nx, int ny, int nz,
                 double R, double beta, double eta, const ConeRows& rows, cudaStream_t s)
{
    ConvArgs a;
    a.in = in;
    a.out = out;
    a.meta = (const ConeMeta*)(T + table_words(rows.n));
    a.table = normalise ? T : nullptr;
    a.proj = proj;
    a.nx = nx;
    a.ny = ny;
    a.nz = nz;
    a.n = rows.n;
    a.nrows = rows.nrows;
    a.R = (float)R;
    a.beta = (float)beta;
    a.eta = (float)eta;
    a.pden = (float)(std::tanh(beta * eta) + std::tanh(beta * (1.0 - eta)));
    const bool vec = nx % 4 == 0 && (uintptr_t)in % 16 == 0;
    const auto k = vec ? cone_kernel<true> : cone_kernel<false>;
    cudaError_t e = allow_smem(k, cone_smem_bytes(kMaxHalo));
    if (e != cudaSuccess) return e;
    const dim3 g((unsigned)((nx + kOX - 1) / kOX) * (unsigned)nz, (ny + kTY - 1) / kTY);   // z in grid x: no limit of 65535
    k<<<g, kThreads, cone_smem_bytes(rows.n), s>>>(a);
    return cudaGetLastError();
}

cudaError_t build_table(long long* T, const ConeRows& rows, double R, cudaStream_t s)
{
    cudaError_t e = allow_smem(table_kernel, table_smem_bytes(kMaxHalo));
    if (e != cudaSuccess) return e;
    table_kernel<<<1, 1024, table_smem_bytes(rows.n), s>>>(T, rows, (float)R);
    return cudaGetLastError();
}

// Scratch of one call, from a pool per device that keeps at most kKeepBytes between calls (the default pool
// gives its memory back at every synchronisation, and mapping it anew cost a call most of its time).
constexpr int kMaxDevices = 64;
constexpr uint64_t kKeepBytes = 64ull << 20;
std::mutex g_pool_mutex;
cudaMemPool_t g_pool[kMaxDevices] = {};

cudaError_t scratch(void** p, size_t bytes, cudaStream_t s)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    cudaMemPool_t pool = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_pool_mutex);
        if (!g_pool[dev]) {
            cudaMemPoolProps props{};
            props.allocType = cudaMemAllocationTypePinned;
            props.handleTypes = cudaMemHandleTypeNone;
            props.location.type = cudaMemLocationTypeDevice;
            props.location.id = dev;
            if ((e = cudaMemPoolCreate(&pool, &props)) != cudaSuccess) return e;
            uint64_t keep = kKeepBytes;
            if ((e = cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep)) != cudaSuccess) {
                cudaMemPoolDestroy(pool);
                return e;
            }
            g_pool[dev] = pool;
        }
        pool = g_pool[dev];
    }
    return cudaMallocFromPoolAsync(p, bytes, pool, s);
}

}  // namespace

extern "C" fdtd_status fdtd_filter_project(const float* rho, float* rho_t, float* rho_b, int nx, int ny, int nz,
                                           double R, double beta, double eta, void* cuda_stream)
{
    if (!rho || !rho_t || !rho_b) return fail(FDTD_ERR_ARG, "filter: null pointer");
    if (fdtd_status st = check(nx, ny, nz, R, beta, eta)) return st;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    const ConeRows rows = cone_rows((float)R, halo(R));
    long long* T = nullptr;
    cudaError_t e = scratch((void**)&T, table_bytes(rows.n), s);
    if (e != cudaSuccess) return fail(FDTD_ERR_OOM, std::string("filter: ") + cudaGetErrorString(e));
    e = build_table(T, rows, R, s);
    if (e == cudaSuccess) e = conv(rho, rho_t, T, true, rho_b, nx, ny, nz, R, beta, eta, rows, s);   // filter + project
    cudaFreeAsync(T, s);
    if (e != cudaSuccess) return fail(FDTD_ERR_CUDA, std::string("filter: ") + cudaGetErrorString(e));
    return FDTD_OK;
}

extern "C" fdtd_status fdtd_filter_project_grad(const float* rho_t, const float* dF_drho_b, float* dF_drho, int nx,
                                                int ny, int nz, double R, double beta, double eta, void* cuda_stream)
{
    if (!rho_t || !dF_drho_b || !dF_drho) return fail(FDTD_ERR_ARG, "filter grad: null pointer");
    if (fdtd_status st = check(nx, ny, nz, R, beta, eta)) return st;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    const size_t nv = (size_t)nx * ny * nz, gb = (nv * sizeof(float) + 255) / 256 * 256;
    const ConeRows rows = cone_rows((float)R, halo(R));
    float* g = nullptr;
    cudaError_t e = scratch((void**)&g, gb + table_bytes(rows.n), s);
    if (e != cudaSuccess) return fail(FDTD_ERR_OOM, std::string("filter grad: ") + cudaGetErrorString(e));
    long long* T = (long long*)((char*)g + gb);
    const float pden = (float)(std::tanh(beta * eta) + std::tanh(beta * (1.0 - eta)));
    e = build_table(T, rows, R, s);
    if (e == cudaSuccess) {
        chain_pre_kernel<<<(unsigned)((nv + 255) / 256), 256, 0, s>>>(dF_drho_b, rho_t, T, rows.n, (float)R, g, nx, ny, nz, (float)beta,
                                                                       (float)eta, pden);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = conv(g, dF_drho, T, false, nullptr, nx, ny, nz, R, beta, eta, rows, s);   // transposed filter
    cudaFreeAsync(g, s);
    if (e != cudaSuccess) return fail(FDTD_ERR_CUDA, std::string("filter grad: ") + cudaGetErrorString(e));
    return FDTD_OK;
}
