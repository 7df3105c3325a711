// Design-E kernel on x-adjacent sample pairs (FP32): the E update inside the design box of Eqs.
// (Maxwells)a,b with (eps_mixed), (sigma_mixed), (Poles_mixed) and the pole recursion, as in
// e_design_column, with each thread updating the samples of component C at (i, j, k) and (i+1, j, k):
// 8-byte loads and stores of fields, densities and snapshots, 16-byte loads and stores of the two
// samples' pole currents, and Blackwell's paired FP32 instructions.  Samples outside their component's sample
// box or in the gap, point sources and the TF/SF plane are handled within the pair; pairs on a PEC wall and the
// per-sample records of paper mode take e_design_column sample by sample.
//
// Used when nx and the working box's x origin and extent are even (the host checks), so that a pair's two
// samples are adjacent, and 8-byte aligned, in every array (the density too, in either layout).
#pragma once
#include "fdtd_shell2.cuh"

namespace fdtd {

// L2 prefetch of the rows of the plane FDTD_ED2_PF ahead (0: none); measured 0.0718 -> 0.0699 ms on the
// config-2 design box (3 poles), 0.697 -> 0.653 ms on the config-3 one (6 poles, two blocks per SM)
#ifndef FDTD_ED2_PF
#define FDTD_ED2_PF 1
#endif

__device__ __forceinline__ float4 ldq_pre(const cpx<float>* p) { return __ldcg(reinterpret_cast<const float4*>(p)); }
__device__ __forceinline__ void stq(cpx<float>* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }

template <int MP, int C>
__device__ __forceinline__ float design_pair_column(const KParams<float>& p, const PoleTable<float>& tab, int i, int j,
                                                    int k0, int k1, int n)
{
    constexpr int ca = C == 0 ? 2 : C - 1, cb = C == 2 ? 0 : C + 1;
    constexpr int MQ = MP > 0 ? MP : 1;
    const float* Ha = p.Hn[ca];
    const float* Hb = p.Hn[cb];
    const float* Ec = p.E[C];
    const float* rc = p.rhoc[C];
    const unsigned nx = (unsigned)p.nx, plane = (unsigned)p.plane, col = (unsigned)j * nx + (unsigned)i;
    const long long dcol = (long long)(j - p.db[2]) * p.dnx + (i - p.db[0]);
    // which of the two samples lie in the component's sample box and in the gap box, in x and y
    const bool iny = j >= p.mb[C][2] && j < p.mb[C][3], gy = j >= p.gb[2] && j < p.gb[3];
    const bool m0 = iny && i >= p.mb[C][0] && i < p.mb[C][1], m1 = iny && i + 1 >= p.mb[C][0] && i + 1 < p.mb[C][1];
    const bool g0 = gy && i >= p.gb[0] && i < p.gb[1], g1 = gy && i + 1 >= p.gb[0] && i + 1 < p.gb[1];
    // per-sample cases for the whole column: paper-mode records, the PEC walls at x = 0 (C = 1, 2), y = 0 (C = 0, 2)
    const bool col_scalar = p.td_acc || p.hist_dq || ((C == 1 || C == 2) && i == 0) || (C != 1 && j == 0);
    const long long slot0 = (long long)((n - p.snap0) % p.K) * p.snap_stride + C * p.nd;
    const int P = p.P[C], P1 = p.P1[C];
    const float2 idx2 = f2(p.inv_dx, p.inv_dx), one2 = f2(1.f, 1.f);
    const float2 D1 = f2(p.D1[C], p.D1[C]), dD = f2(p.dD[C], p.dD[C]), N1 = f2(p.N1[C], p.N1[C]),
                 dN = f2(p.dN[C], p.dN[C]), hg = f2(p.hg, p.hg);
    float emax = 0.f;
    for (int k = k0; k < k1; ++k) {
        const bool in_gz = k >= p.gb[4] && k < p.gb[5];
        const bool src = p.nb > 0 && k >= p.sb[4] && k < p.sb[5] && j >= p.sb[2] && j < p.sb[3] && i + 1 >= p.sb[0] &&
                         i < p.sb[1];
        // per-sample cases of this plane: the PEC wall at z = 0 (C = 0, 1)
        if (col_scalar || (C != 2 && k == 0)) {
            pdl_wait();   // (returns at once when the phase before is complete)
            pdl_trigger();
#pragma unroll 1
            for (int e = 0; e < 2; ++e) emax = fmaxf(emax, e_design_column<float, MP, C>(p, tab, i + e, j, k, k + 1, n));
            continue;
        }
        const unsigned id = (unsigned)k * plane + col;
        const long long dv = (long long)(k - p.db[4]) * p.dplane + dcol;
        // Samples at the box's rim and in the gap take the background's update, chosen per sample at the end: one
        // chain a pair whatever its samples are.  (Each such sample's update in turn, behind the wait, was the
        // launch's longest chain: 48^3 step 8.7 -> 7.6 us, 128^3 37.3 -> 36.1.)
        const bool inz = k >= p.mb[C][4] && k < p.mb[C][5], d0 = m0 && inz && !(g0 && in_gz), d1 = m1 && inz && !(g1 && in_gz);
        const float2 e0 = ldp_pre(Ec + id), rho = ldp_pre(rc + dv);
        float4 q[MQ];
#pragma unroll
        for (int pp = 0; pp < MQ; ++pp)
            if (pp < P) q[pp] = ldq_pre(p.Q[C] + pp * p.nd + dv);
        if (k == k0) {
            pdl_wait();
            pdl_trigger();
        }
        if (FDTD_ED2_PF > 0 && k + FDTD_ED2_PF < k1) {   // the rows of a coming plane into L2
            const unsigned ip = id + FDTD_ED2_PF * plane;
            const long long dp = dv + FDTD_ED2_PF * p.dplane;
            pf_l2(Ha + ip);
            pf_l2(Hb + ip);
            pf_l2(Ec + ip);
            pf_l2(rc + dp);
#pragma unroll
            for (int pp = 0; pp < MQ; ++pp)
                if (pp < P) pf_l2(reinterpret_cast<const float*>(p.Q[C] + pp * p.nd + dp));
        }
        // (curl H)_C = (Ha - Ha(-1 along la)) - (Hb - Hb(-1 along lb)); along x the pair's lower neighbour is
        // its first sample's
        const float2 ha = ldp(Ha + id), hb = ldp(Hb + id);
        float2 ham, hbm;
        if (C == 0) {
            ham = ldp(Ha + id - nx);       // H_z along y
            hbm = ldp(Hb + id - plane);    // H_y along z
        } else if (C == 1) {
            ham = ldp(Ha + id - plane);    // H_x along z
            hbm = f2(Hb[id - 1], hb.x);    // H_z along x
        } else {
            ham = f2(Ha[id - 1], ha.x);    // H_y along x
            hbm = ldp(Hb + id - nx);       // H_x along y
        }
        // drive and the blended update, per element the operations of design_update
        float2 d = p_mul(p_sub(p_sub(ha, ham), p_sub(hb, hbm)), idx2);
        if (C == 2 && (i == p.tfsf_i0 || i + 1 == p.tfsf_i0)) {   // the TF/SF plane
            const float h = __ldg(p.hinc + n) * p.inv_dx;
            (i == p.tfsf_i0 ? d.x : d.y) -= h;
        }
        if (src) {
#pragma unroll 1
            for (int s = 0; s < 2; ++s)
                if (in_box(p.sb, i + s, j, k)) (s ? d.y : d.x) += point_drive(p, i + s, j, k, C, n);
        }
        const float2 gm = p_mul(p_mul(hg, rho), p_sub(one2, rho));
        const float2 D = p_add(p_fma(rho, dD, D1), gm);
        const float2 N = p_sub(p_fma(rho, dN, N1), gm);
        float2 sq = f2(0.f, 0.f);
#pragma unroll
        for (int pp = 0; pp < MQ; ++pp) {
            if (pp < P) {
                const float2 kap = pp < P1 ? p_sub(one2, rho) : rho;
                const cpx<float> g = tab.g[C][pp];
                const float2 qre = f2(q[pp].x, q[pp].z), qim = f2(q[pp].y, q[pp].w);
                sq = p_fma(kap, p_sub(p_mul(f2(g.re, g.re), qre), p_mul(f2(g.im, g.im), qim)), sq);
            }
        }
        const float2 num = p_sub(p_fma(N, e0, d), sq);
        const float2 eb = p_fma(f2(p.bg_ca[C], p.bg_ca[C]), e0, p_mul(f2(p.bg_cb[C], p.bg_cb[C]), d));
        const float2 e = f2(d0 ? div_t(num.x, D.x) : eb.x, d1 ? div_t(num.y, D.y) : eb.y);
        // (a background sample's currents follow its E and are read by nothing: masking them takes 128^3 from 36.1 to
        // 37.1 us a step)
        const float2 es = p_add(e, e0);
#pragma unroll
        for (int pp = 0; pp < MQ; ++pp) {
            if (pp < P) {
                const cpx<float> a = tab.am1[C][pp], b = tab.beta[C][pp];
                const float2 qre = f2(q[pp].x, q[pp].z), qim = f2(q[pp].y, q[pp].w);
                const float2 vre = p_fma(f2(b.re, b.re), es, p_add(qre, p_sub(p_mul(f2(a.re, a.re), qre), p_mul(f2(a.im, a.im), qim))));
                const float2 vim = p_fma(f2(b.im, b.im), es, p_add(qim, p_fma(f2(a.re, a.re), qim, p_mul(f2(a.im, a.im), qre))));
                stq(p.Q[C] + pp * p.nd + dv, make_float4(vre.x, vim.x, vre.y, vim.y));
            }
        }
        stp(p.En[C] + id, e);
        // read again only by the DFT, up to 16 steps on: out of L2 first (128^3 step 37.7 -> 37.2 us)
        __stcs(reinterpret_cast<float2*>(p.snap + slot0 + dv), e);
        emax = fmaxf(emax, fmaxf(fabsf(e.x), fabsf(e.y)));
    }
    return emax;
}

// Resident blocks per SM the register allocation is held to (the pole currents of a pair take twice
// the registers of a sample's).
template <int MP>
constexpr int ed2_min_blocks()
{
#ifdef FDTD_ED2_MINB
    return FDTD_ED2_MINB;
#else
    return MP <= 4 ? 4 : 2;   // MP <= 8
#endif
}

// One block: 256 column pairs in row order of component blockIdx.z % 3, p.edz planes each.  Every lane is
// busy whatever the box's width (tiles of 32 x 8 pairs before: 96 x 84 x 108 voxels 38.8 -> 36.0 us a
// launch, 32^3 voxels 9.4 -> 8.5 us).
// block (bx, bz) of a launch with nz blocks in z, of nt threads
template <int MP>
__device__ __forceinline__ void e_design2_block(const KParams<float>& p, const PoleTable<float>& tab, unsigned bx, unsigned bz,
                                                unsigned nz, int nt)
{
    const int b = (int)phase_block(p, bz, nz), zc = b / 3, c = b - 3 * zc;
    const int wx = (p.db[1] - p.db[0]) / 2;
    const int col = (int)bx * nt + threadIdx.y * kBX + threadIdx.x;
    const int y = col / wx;
    const int i = p.db[0] + 2 * (col - y * wx);
    const int j = p.db[2] + y;
    const int k0 = p.db[4] + zc * p.edz, k1 = min(p.db[5], k0 + p.edz);
    const int n = read_step(p);
    if (j >= p.db[3]) return;
    const float emax = c == 0 ? design_pair_column<MP, 0>(p, tab, i, j, k0, k1, n)
                     : c == 1 ? design_pair_column<MP, 1>(p, tab, i, j, k0, k1, n)
                              : design_pair_column<MP, 2>(p, tab, i, j, k0, k1, n);
    if (!(emax < p.blowup)) atomicOr(p.ctl + 2, 1);
}

template <int MP>
__global__ void __launch_bounds__(kBX * kBY, ed2_min_blocks<MP>()) e_design2_kernel(const KParams<float> p,
                                                                                         const PoleTable<float> tab)
{
    e_design2_block<MP>(p, tab, blockIdx.x, blockIdx.z, gridDim.z, kBX * kBY);
}

// The whole E phase in one launch (SP, DP: paired shell and design kernels): the design box's blocks, gx column
// groups by gz z chunks and components, then the shell's.
template <bool SP, bool DP, int MP>
__global__ void __launch_bounds__(kShellNT, 8) e_phase_kernel(const KParams<float> p, const ShellBoxes s, const PoleTable<float> tab,
                                                              unsigned gx, unsigned gz)
{
    const unsigned nd = gx * gz;
    if (blockIdx.x < nd) {
        const unsigned bz = blockIdx.x / gx, bx = blockIdx.x - bz * gx;
        if constexpr (DP)
            e_design2_block<MP>(p, tab, bx, bz, gz, kShellNT);
        else
            e_design_block<float, MP>(p, tab, bx, bz, gz, kShellNT);
    } else if constexpr (SP) {
        shell_e2_block(p, s, blockIdx.x - nd);
    } else {
        shell_e_block<float, 1>(p, s, blockIdx.x - nd);   // columns of one plane
    }
}

}  // namespace fdtd
