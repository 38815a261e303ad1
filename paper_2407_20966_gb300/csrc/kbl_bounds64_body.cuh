// kbl_bounds64_body.cuh -- device code of the FP64 kinetic bounds (and helpers the other
// bounds kernels share), used by the FR kernels (kbl_bounds.cu) and by the explicit-stencil
// kernels (kbl_stencil.cu).  See kbl_bounds.cu for the steps and their equations.
#pragma once

#include <cfloat>

#include "kbl_bounds_body.cuh"

namespace kbl_dev {

constexpr int CH = 16;  // states per table chunk

// ---------------------------------------------------------------------------
// shared helpers
// ---------------------------------------------------------------------------
struct StatePrim {
    double U[2];
    double th;     // theta
    double sq;     // sqrt(theta)
    double A;      // rho (2 pi theta)^(-d/2)
    double C;      // theta delta / 2
};

template <int DIM>
__device__ __forceinline__ bool prim_of(const double* q, const Phys& ph, StatePrim& s)
{
    const double rho = q[0];
    const double P = kbl_pressure<DIM>(q, ph.gamma - 1.0);
    if (!(rho > 0.0) || !(P > 0.0)) return false;
    const double th = P / rho;
    s.U[0] = q[1] / rho;
    s.U[1] = (DIM == 2) ? q[2] / rho : 0.0;
    s.th = th;
    s.sq = sqrt(th);
    s.A = (DIM == 1) ? rho / sqrt(2.0 * KBL_PI * th) : rho / (2.0 * KBL_PI * th);
    s.C = 0.5 * (2.0 / (ph.gamma - 1.0) - DIM) * th;
    return true;
}

// Block-wide sum of K doubles per thread; result valid in thread 0.
template <int K, int NT>
__device__ __forceinline__ void block_sum_f64(double (&a)[K], double* sred /* [NT/32][K] */)
{
    constexpr int NW = (NT + 31) / 32;
#pragma unroll
    for (int k = 0; k < K; k++) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) a[k] += __shfl_xor_sync(0xffffffffu, a[k], o);
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (NW > 1) {
        if (lane == 0) {
#pragma unroll
            for (int k = 0; k < K; k++) sred[wid * K + k] = a[k];
        }
        __syncthreads();
        if (threadIdx.x == 0) {
#pragma unroll
            for (int k = 0; k < K; k++) {
                double s = sred[k];
                for (int q = 1; q < NW; q++) s += sred[q * K + k];
                a[k] = s;
            }
        }
    }
}

// Compensated block-wide sum of K floats per thread (hi + lo pairs);
// result (as doubles) valid in thread 0.
template <int K, int NT>
__device__ __forceinline__ void block_sum_f32c(const float (&a)[K], double (&out)[K], float* sred /* [NW][2K] */)
{
    constexpr int NW = (NT + 31) / 32;
    float hi[K], lo[K];
#pragma unroll
    for (int k = 0; k < K; k++) {
        hi[k] = a[k];
        lo[k] = 0.0f;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
        for (int k = 0; k < K; k++) {
            const float oh = __shfl_xor_sync(0xffffffffu, hi[k], o);
            const float ol = __shfl_xor_sync(0xffffffffu, lo[k], o);
            float s, e;
            two_sum(hi[k], oh, s, e);
            hi[k] = s;
            lo[k] = __fadd_rn(__fadd_rn(lo[k], ol), e);
        }
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (NW > 1) {
        if (lane == 0) {
#pragma unroll
            for (int k = 0; k < K; k++) {
                sred[wid * 2 * K + k] = hi[k];
                sred[wid * 2 * K + K + k] = lo[k];
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) {
#pragma unroll
            for (int k = 0; k < K; k++) {
                double s = 0.0;
                for (int q = 0; q < NW; q++) s += (double)sred[q * 2 * K + k] + (double)sred[q * 2 * K + K + k];
                out[k] = s;
            }
        }
    } else {
#pragma unroll
        for (int k = 0; k < K; k++) out[k] = (double)hi[k] + (double)lo[k];
    }
}

// Final bounds from the raw sums (see the header comment, step 5-6).
// raw (1D): [Tlo, Thi, nx_hi, nx_lo, px_lo, px_hi, E_lo, E_hi]
// raw (2D): [Tlo, Thi, nx_hi, nx_lo, px_lo, px_hi, ny_hi, ny_lo, py_lo, py_hi, E_lo, E_hi]
template <int DIM>
__device__ __forceinline__ void finalize_bounds(const double* raw, double scale, const Phys& ph,
                                                double* bnd, int E, int e)
{
    constexpr int NV = DIM + 2;
    const double rm = 1.0 - ph.r_fac, rp = 1.0 + ph.r_fac;
    double lo[NV], hi[NV];
    lo[0] = rm * (scale * raw[0]);
    hi[0] = rp * (scale * raw[1]);
#pragma unroll
    for (int d = 0; d < DIM; d++) {
        const double* m = raw + 2 + 4 * d;
        lo[1 + d] = rp * (scale * m[0]) + rm * (scale * m[2]);
        hi[1 + d] = rm * (scale * m[1]) + rp * (scale * m[3]);
    }
    lo[NV - 1] = rm * (scale * raw[2 + 4 * DIM]);
    hi[NV - 1] = rp * (scale * raw[3 + 4 * DIM]);
    if (lo[0] < ph.rho_floor) lo[0] = ph.rho_floor;
#pragma unroll
    for (int v = 0; v < NV; v++) {
        bnd[(size_t)v * E + e] = lo[v];
        bnd[((size_t)NV + v) * E + e] = hi[v];
    }
}

__device__ __forceinline__ unsigned long long umin64(unsigned long long a, unsigned long long b) { return a < b ? a : b; }
__device__ __forceinline__ unsigned long long umax64(unsigned long long a, unsigned long long b) { return a > b ? a : b; }

// ---------------------------------------------------------------------------
// 2D, FP64 arithmetic throughout: row tables by the product recurrence of kbl_gauss_segment,
// products and envelopes in FP64 (min/max as unsigned 64-bit compares of the bit patterns: all
// values are >= +0, where integer order is value order; the internal weights C, of one sign for all
// states and negative for gamma > 2, enter as |C|).  Bound by the FP64 pipe: two products per
// (state, node) at 1.7 lanes per clock per SM.  Runs the grids the pairs below do not cover.
// ---------------------------------------------------------------------------
template <int NST, int NX, int NW>
struct F64Tables {
    double ex[CH][NX], exc[CH][NX], ey[CH][NX];
    double u[2][NX], w[2][NX];
    double box[4], gh[2];
    double red[NW * 12];
    StatePrim P[NST];
};

// Bounds of the states S[NST][4]: one block of NT threads, each with TX x TY velocity nodes.
template <int NST, int NX, int TX, int TY, int NT, int NW>
__device__ __forceinline__ void bounds2d_f64_states(const double (*S)[4], F64Tables<NST, NX, NW>& sm, int E, int e,
                                                    const Phys& ph, double* __restrict__ bnd, DevFlags* flags)
{
    constexpr int TPX = NX / TX, ACT = TPX * (NX / TY);
    const int tid = threadIdx.x;
    int bad = 0;
    for (int i = tid; i < NST; i += NT)
        if (!prim_of<2>(S[i], ph, sm.P[i])) bad = 1;
    if (__syncthreads_or(bad)) {
        if (tid == 0) {
            write_nan(bnd, E, e, 4);
            atomicOr(&flags->nonphysical, 1);
        }
        return;
    }
    if (tid < 4) {
        const int d = tid >> 1, up = tid & 1;
        double b = up ? sm.P[0].U[d] + ph.k * sm.P[0].sq : sm.P[0].U[d] - ph.k * sm.P[0].sq;
        for (int i = 1; i < NST; i++) {
            const double c = up ? sm.P[i].U[d] + ph.k * sm.P[i].sq : sm.P[i].U[d] - ph.k * sm.P[i].sq;
            b = up ? fmax(b, c) : fmin(b, c);
        }
        sm.box[tid] = b;
    }
    __syncthreads();
    const int nu = ph.nu[0];   // nodes per axis; tile nodes j >= nu sit on the box end with weight 0
    if (tid < 2) sm.gh[tid] = (sm.box[2 * tid + 1] - sm.box[2 * tid]) / (nu - 1);
    __syncthreads();
    for (int j = tid; j < 2 * NX; j += NT) {
        const int d = j / NX, jj = j % NX;
        sm.u[d][jj] = sm.box[2 * d] + min(jj, nu - 1) * sm.gh[d];
        sm.w[d][jj] = kbl_qweight(ph, jj, nu) * sm.gh[d];
    }
    const int tx = tid % TPX, ty = tid / TPX;
    unsigned long long tlo[TX][TY], thi[TX][TY], ilo[TX][TY], ihi[TX][TY];
#pragma unroll
    for (int a = 0; a < TX; a++)
#pragma unroll
        for (int b = 0; b < TY; b++) {
            tlo[a][b] = ~0ull; ilo[a][b] = ~0ull;
            thi[a][b] = 0ull; ihi[a][b] = 0ull;
        }
    for (int c0 = 0; c0 < NST; c0 += CH) {
        const int nc = min(CH, NST - c0);
        __syncthreads();
        // row tables by segments of SEG nodes (product recurrence, a few exponentials per segment)
        constexpr int SEG = NX < 16 ? NX : (NX % 16 ? 8 : 16), NSG = NX / SEG;
        for (int task = tid; task < nc * 2 * NSG; task += NT) {
            const int i = task / (2 * NSG), axis = (task / NSG) & 1, jb = (task % NSG) * SEG;
            const StatePrim& s = sm.P[c0 + i];
            if (axis == 0)
                kbl_gauss_segment(s.A, s.U[0], s.th, sm.box[0], sm.gh[0], nu, jb, jb + SEG, [&](int j, double v) {
                    sm.ex[i][j] = v;
                    sm.exc[i][j] = fabs(s.C) * v;
                });
            else
                kbl_gauss_segment(1.0, s.U[1], s.th, sm.box[2], sm.gh[1], nu, jb, jb + SEG,
                                  [&](int j, double v) { sm.ey[i][j] = v; });
        }
        __syncthreads();
        for (int i = 0; i < nc && tid < ACT; i++) {
            double ex[TX], exc[TX], ey[TY];
#pragma unroll
            for (int a = 0; a < TX; a++) {
                ex[a] = sm.ex[i][tx * TX + a];
                exc[a] = sm.exc[i][tx * TX + a];
            }
#pragma unroll
            for (int b = 0; b < TY; b++) ey[b] = sm.ey[i][ty * TY + b];
#pragma unroll
            for (int a = 0; a < TX; a++)
#pragma unroll
                for (int b = 0; b < TY; b++) {
                    const unsigned long long g = __double_as_longlong(ex[a] * ey[b]);
                    const unsigned long long cg = __double_as_longlong(exc[a] * ey[b]);
                    tlo[a][b] = umin64(tlo[a][b], g);
                    thi[a][b] = umax64(thi[a][b], g);
                    ilo[a][b] = umin64(ilo[a][b], cg);
                    ihi[a][b] = umax64(ihi[a][b], cg);
                }
        }
    }
    double acc[12];
#pragma unroll
    for (int k = 0; k < 12; k++) acc[k] = 0.0;
    if (tid < ACT) {
#pragma unroll
        for (int a = 0; a < TX; a++)
#pragma unroll
            for (int b = 0; b < TY; b++) {
                const int jx = tx * TX + a, jy = ty * TY + b;
                const double M = sm.w[0][jx] * sm.w[1][jy];
                const double ux = sm.u[0][jx], uy = sm.u[1][jy];
                const double Tl = __longlong_as_double(tlo[a][b]), Th = __longlong_as_double(thi[a][b]);
                const double i0 = __longlong_as_double(ilo[a][b]), i1 = __longlong_as_double(ihi[a][b]);
                const bool neg = ph.half_delta2 < 0.0;
                const double Il = neg ? -i1 : i0, Ih = neg ? -i0 : i1;
                acc[0] += M * Tl;
                acc[1] += M * Th;
                if (ux < 0.0) { acc[2] += M * Th * ux; acc[3] += M * Tl * ux; }
                else { acc[4] += M * Tl * ux; acc[5] += M * Th * ux; }
                if (uy < 0.0) { acc[6] += M * Th * uy; acc[7] += M * Tl * uy; }
                else { acc[8] += M * Tl * uy; acc[9] += M * Th * uy; }
                const double ke = 0.5 * ux * ux + 0.5 * uy * uy;
                acc[10] += M * (Tl * ke + Il);
                acc[11] += M * (Th * ke + Ih);
            }
    }
    block_sum_f64<12, NT>(acc, sm.red);
    if (tid == 0) finalize_bounds<2>(acc, 1.0, ph, bnd, E, e);
}

// Launch shape: 2 x 2 nodes per thread; 4 resident blocks at 32 nodes (64 registers) measured 7%
// faster than the 2 that 128 registers allow.
template <int NX>
struct B2f64 {
    static constexpr int TX = 2, ACT = (NX / TX) * (NX / TX), NT = (ACT + 31) / 32 * 32;
    static constexpr int MINB = NT <= 256 ? 4 : 1;
};

template <int NST, int NX>
struct Bounds2dF64Smem {
    F64Tables<NST, NX, B2f64<NX>::NT / 32> t;
    double S[NST][4];
};

// Bounds of element e from a stencil of NST states, one block of B2f64<NX>::NT threads: gather(S)
// fills S[NST][4]; the bounds go to column e of bnd[2][4][E].
template <int NST, int NX, typename Gather>
__device__ __forceinline__ void bounds2d_f64_core(Bounds2dF64Smem<NST, NX>& sm, Gather gather, int E, int e,
                                                  const Phys& ph, double* __restrict__ bnd, DevFlags* flags)
{
    constexpr int NT = B2f64<NX>::NT;
    gather(sm.S);
    __syncthreads();
    bounds2d_f64_states<NST, NX, B2f64<NX>::TX, B2f64<NX>::TX, NT>(sm.S, sm.t, E, e, ph, bnd, flags);
}

// ---------------------------------------------------------------------------
// 2D, full precision, on pairs of floats
//
// GB300 runs FP64 at 1.7 lanes per clock per SM and FP32 at 128, so the envelopes of the FP64 mode
// are formed on unevaluated sums of two floats (hi + lo, 48-49 significant bits) and the FP64 pipe
// keeps what decides the result's accuracy per state (the primitive state, the velocity box, the
// exponents' coefficients) and per sum (the moments).  Errors against extended precision, every bound
// relative to itself (a momentum to the magnitudes it sums), rms; the kernel above in brackets, its
// tables drift along the recurrence: vortex 2.2e-16 (2.5e-16), smooth waves 1.9e-16 (2.4e-16), blast
// 2.0e-16 (2.6e-16), scattered node sets 2.0e-16 (2.1e-16); blast, 48 nodes 1.7e-16 (2.3e-16), 33 nodes
// by Romberg 2.3e-16 (2.6e-16).  States that differ by factors within a stencil: lower density and
// energy 3.3e-16 (1.8e-16), all bounds 2.6e-16 (1.9e-16), since their envelope's minimum lives on few
// nodes and the tables' 2^-49 average out less.
//
//   row tables   a_i(u) = A_i 2^-t(u), c_i = C_i a_i, b_i(v) = 2^-t(v), t = (u - U)^2 log2(e)/(2 theta),
//                t in 64-bit fixed point by second differences (exact additions), 2^-t by a table of
//                128 exact knots and a polynomial on float pairs
//   pass 1       M = max_i fl(a_hi b_hi) (min alike; c b alike): the FP32 envelope
//   pass 2       E = max_i [a_hi b_hi - M + a_hi b_lo + a_lo b_hi] by FMAs, the first of which forms
//                a_hi b_hi - M with one rounding: the envelope is M + E, its winner decided to
//                2^-47, its value off by as little
//   moments      the nodes' values in error-free FP32 sums along rows and columns, those in FP64;
//                the quadrature weights are in the tables already
//
// Measured at 128^2 P3, 32^2 grid: 0.83 ms per launch (0.85 while table entries carried their rounding
// errors along the row, the base of the figures that follow); 0.87 with both axes' grid coefficients in one
// thread per state, 0.95 with the y table's values stored twice (a
// 128-bit shared load takes four wavefronts however many lanes share its addresses, and the passes
// wait on them: 6.9k of 19k clocks per element), 1.08 with the moments node by node in FP64 and the
// states' constants in two passes over shared memory, 6.52 for the FP64 kernel above (86% of the FP64
// pipe).  33^2 Romberg grid (46 x 27 P4): 0.21 ms on a 40-node tile, 2.77 ms on the FP64 kernel's 64.
// Five blocks per SM (96 registers): 0.90 ms against 0.85 (kernel alone) at 48 states, 0.54 against
// 0.57 at 24.
// What bounds it: per (state, node) 14 FP32 products/FMAs (packed two to an instruction, two
// neighbouring x nodes) and four three-input min/max, 7 + 4 issue slots: about half the launch; the
// states' FP64 chains, tables and sums the other half.  Counters at 64^2 P3: issue slots 56% busy, FP64
// pipe 46%, ALU 34%, FMA pipe 30%; 128 registers, four blocks per SM.
//
// Elements outside the range of the pairs (a state more than 2^240 below its peak inside the box,
// constants beyond +-2^60 of the largest, a lower density sum below 2^-40 of the largest state's)
// run on the FP64 pipe instead (bounds2d_f64_states), decided per element.
// ---------------------------------------------------------------------------

// 2^(-k/128), k = 0..127, rounded to a pair of floats (bits), and -log2(that pair) - k/128 in units
// of 2^-55, so that the knot is exact to the exponents' resolution.
struct Exp2Knot {
    unsigned hi, lo;
    int f;
};
__device__ const Exp2Knot kbl_exp2_knots[128] = {
    {0x3f800000u, 0x00000000u, 0}, {0x3f7e9e11u, 0x32b8f71fu, 6}, {0x3f7d3e0cu, 0x314f486cu, 1},
    {0x3f7bdfedu, 0x32d9cbe1u, 21}, {0x3f7a83b3u, 0xb2123758u, 2}, {0x3f79295au, 0xb2894457u, 43},
    {0x3f77d0dfu, 0x32e615a2u, 45}, {0x3f767a41u, 0x32d8e67fu, 3}, {0x3f75257du, 0x31a92436u, 9},
    {0x3f73d290u, 0xb2071670u, 20}, {0x3f728177u, 0x327167ffu, -11}, {0x3f713231u, 0xb2b0a5edu, -45},
    {0x3f6fe4bau, 0xb2c8464au, -8}, {0x3f6e9910u, 0xb2cfe4bau, 2}, {0x3f6d4f30u, 0x31f6cca1u, 9},
    {0x3f6c0719u, 0xb29367c7u, 48}, {0x3f6ac0c7u, 0xb1c116deu, -5}, {0x3f697c38u, 0x3280d89fu, 10},
    {0x3f68396au, 0x32a07898u, -28}, {0x3f66f85bu, 0xb2aa23c0u, -40}, {0x3f65b907u, 0xb1c41be6u, 7},
    {0x3f647b6du, 0xb2bf9185u, 33}, {0x3f633f89u, 0x32e57d15u, -31}, {0x3f62055bu, 0xabbe164cu, 0},
    {0x3f60ccdfu, 0xb19eab59u, 1}, {0x3f5f9613u, 0xb2051c3fu, 3}, {0x3f5e60f5u, 0xb2fb43e3u, 14},
    {0x3f5d2d82u, 0xb2f5ef9bu, -43}, {0x3f5bfbb8u, 0xb2d04a1cu, 46}, {0x3f5acb94u, 0x32de5594u, -44},
    {0x3f599d16u, 0xb2761d41u, 20}, {0x3f587039u, 0x3298db66u, 38}, {0x3f5744fdu, 0xb254a58au, -18},
    {0x3f561b5eu, 0xafb03219u, 0}, {0x3f54f35bu, 0xb2a86024u, -5}, {0x3f53ccf1u, 0xb2ccf4cau, -53},
    {0x3f52a81eu, 0xb2dc1daau, -24}, {0x3f5184dfu, 0x32c4a2d3u, 24}, {0x3f506334u, 0xb2144353u, -23},
    {0x3f4f4319u, 0xb2439b9cu, 22}, {0x3f4e248cu, 0x31a8fc24u, 1}, {0x3f4d078cu, 0xb2f35f84u, -45},
    {0x3f4bec15u, 0xaf86c6c2u, 0}, {0x3f4ad226u, 0x32bc8521u, -8}, {0x3f49b9beu, 0xb2f323a2u, 36},
    {0x3f48a2d8u, 0x32b91ffcu, 41}, {0x3f478d75u, 0xb25d5119u, -14}, {0x3f467991u, 0xb294abb7u, -30},
    {0x3f45672au, 0x318aa837u, -5}, {0x3f44563fu, 0xb24eb32du, 11}, {0x3f4346cdu, 0xb2176da2u, -26},
    {0x3f4238d2u, 0x324478f6u, -24}, {0x3f412c4du, 0xb256663eu, 19}, {0x3f40213bu, 0xb2bc1e5fu, 13},
    {0x3f3f179au, 0xb2930b1au, 16}, {0x3f3e0f68u, 0x31186099u, 4}, {0x3f3d08a4u, 0xb2c14fe8u, 53},
    {0x3f3c034au, 0x32fde5d4u, -5}, {0x3f3aff5bu, 0xb29bd983u, -57}, {0x3f39fcd2u, 0x328a5817u, 30},
    {0x3f38fbafu, 0x328ec5f7u, 31}, {0x3f37fbf0u, 0xb255cd70u, 31}, {0x3f36fd92u, 0xb1e6b974u, -9},
    {0x3f360094u, 0xb2af4254u, -9}, {0x3f3504f3u, 0x324fe77au, -28}, {0x3f340aafu, 0xb2bb3569u, 25},
    {0x3f3311c4u, 0x31954889u, 5}, {0x3f321a32u, 0xb2b333ceu, -2}, {0x3f3123f6u, 0xb2fc5aa8u, 39},
    {0x3f302f0eu, 0xb251247fu, 6}, {0x3f2f3b79u, 0xb2a52debu, -64}, {0x3f2e4934u, 0x32a5946bu, 59},
    {0x3f2d583fu, 0xb1adeaf6u, 11}, {0x3f2c6897u, 0xb2b68380u, -24}, {0x3f2b7a3au, 0xb294ad82u, -48},
    {0x3f2a8d26u, 0x32a5d921u, -11}, {0x3f29a15bu, 0xb2962b08u, 16}, {0x3f28b6d5u, 0x31b3d990u, 15},
    {0x3f27cd94u, 0xb2962d36u, 59}, {0x3f26e595u, 0xb240445eu, -23}, {0x3f25fed7u, 0xb2ac9d5eu, 63},
    {0x3f251958u, 0xb2f282c2u, -14}, {0x3f243516u, 0xb2a3ec33u, 1}, {0x3f23520fu, 0x32d1d005u, 67},
    {0x3f227043u, 0x3043125au, 0}, {0x3f218fafu, 0xb255eaedu, -10}, {0x3f20b051u, 0x317b9715u, 0},
    {0x3f1fd228u, 0x32159003u, 34}, {0x3f1ef532u, 0x32c12342u, 21}, {0x3f1e196eu, 0x31c4ea39u, 5},
    {0x3f1d3edau, 0xb2b1a601u, 65}, {0x3f1c6573u, 0x32d05d86u, 52}, {0x3f1b8d3au, 0xb28c5563u, -51},
    {0x3f1ab62bu, 0xb05ac01eu, -2}, {0x3f19e046u, 0xb2d9be90u, -7}, {0x3f190b88u, 0xb1ecc9f4u, 12},
    {0x3f1837f0u, 0x32a31b71u, 50}, {0x3f17657du, 0x3293e2f5u, 59}, {0x3f16942du, 0x325c8061u, 32},
    {0x3f15c3ffu, 0xb2f25267u, 0}, {0x3f14f4f0u, 0xb2ae0212u, 12}, {0x3f1426ffu, 0x317ab1c0u, 6},
    {0x3f135a2bu, 0x323c4f9cu, -29}, {0x3f128e72u, 0x32fb2a64u, -8}, {0x3f11c3d3u, 0x32e75624u, -77},
    {0x3f10fa4du, 0xb2e82237u, 63}, {0x3f1031dcu, 0x328628cdu, 64}, {0x3f0f6a81u, 0x31bf3647u, 7},
    {0x3f0ea43au, 0xb2e97465u, -57}, {0x3f0ddf04u, 0x32008b9au, 38}, {0x3f0d1adfu, 0x32b6fcb7u, 55},
    {0x3f0c57cau, 0xb26e6e43u, 18}, {0x3f0b95c2u, 0xb1e0aba1u, -12}, {0x3f0ad4c6u, 0x328a58e5u, 12},
    {0x3f0a14d5u, 0x32ea92deu, -3}, {0x3f0955eeu, 0x30586398u, 0}, {0x3f08980fu, 0xb2feda4bu, 7},
    {0x3f07db35u, 0x32ffed32u, -55}, {0x3f071f62u, 0xb2d2c2e6u, 22}, {0x3f066491u, 0x32b7247fu, 80},
    {0x3f05aac3u, 0x32cf9891u, -7}, {0x3f04f1f6u, 0x32ac6f38u, 36}, {0x3f043a29u, 0xb2714c87u, 0},
    {0x3f038359u, 0x329ddf6eu, -25}, {0x3f02cd87u, 0xb2cea7a9u, 48}, {0x3f0218afu, 0x3286e7f8u, 54},
    {0x3f0164d2u, 0xb1443fd0u, 11}, {0x3f00b1edu, 0x329fb333u, 62},
};

__device__ __forceinline__ float2 f2dup(float x) { return make_float2(x, x); }
__device__ __forceinline__ float2 f2neg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 f2sub(float2 a, float2 b) { return __ffma2_rn(b, f2dup(-1.0f), a); }
__device__ __forceinline__ void f2two_sum(float2 a, float2 b, float2& s, float2& e)
{
    s = __fadd2_rn(a, b);
    const float2 bp = f2sub(s, a);
    e = __fadd2_rn(f2sub(a, f2sub(s, bp)), f2sub(b, bp));
}

// Numbers as three floats, the third the rounding error of the second; two of them side by side.
struct Triple {
    float h, l, r;
};
struct Triple2 {
    float2 h, l, r;
};

// p + (a + b + c) for |a|, |b|, |c| of the order of p's last bit, with further terms in f: h and l
// rounded once, r what l lost
__device__ __forceinline__ Triple2 triple_of(float2 p, float2 a, float2 b, float2 c, float2 f)
{
    float2 m, e1, n, e2;
    f2two_sum(a, b, m, e1);
    f2two_sum(m, c, n, e2);
    f = __fadd2_rn(f, __fadd2_rn(e1, e2));
    Triple2 y;
    y.h = __fadd2_rn(p, n);
    const float2 d = f2sub(n, f2sub(y.h, p));
    y.l = __fadd2_rn(d, f);
    y.r = f2sub(f, f2sub(y.l, d));
    return y;
}

// y b
__device__ __forceinline__ Triple2 triple_mul(const Triple2& y, float2 bh, float2 bl, float2 br)
{
    const float2 p = __fmul2_rn(y.h, bh), q = __fmul2_rn(y.l, bh), s = __fmul2_rn(y.h, bl);
    float2 f = __ffma2_rn(y.l, bh, f2neg(q));
    f = __fadd2_rn(f, __ffma2_rn(y.h, bl, f2neg(s)));
    f = __ffma2_rn(y.l, bl, f);
    f = __ffma2_rn(y.h, br, f);
    f = __ffma2_rn(y.r, bh, f);
    return triple_of(p, __ffma2_rn(y.h, bh, f2neg(p)), q, s, f);
}

// Part of exp2_pair on the integer pipe: knot and remainder (as hi + lo) of t.
__device__ __forceinline__ void exp2_reduce(long long t, const float2* kT, const int* kF, int& n, float2& T, float& rh,
                                            float& rl)
{
    const unsigned long long tt = (unsigned long long)t + (1ull << 47);
    const unsigned th = (unsigned)(tt >> 32);
    n = (int)(th >> 23);
    const int k = (int)((th >> 16) & 127u);
    T = kT[k];
    const long long r = t - ((long long)(th >> 16) << 48) - kF[k];
    const int x = (int)((r + (1ll << 24)) >> 25);
    rh = (float)x * 0x1p-30f;
    rl = (float)(int)((unsigned)r - ((unsigned)x << 25)) * 0x1p-55f;
}

// y = 2^-(t + n) for t in units of 2^-55, 0 <= t < 256: n the whole part (rounded to 1/128); two at a
// time.  2^-r - 1 of the remainder |r| <= 2^-8 by its Taylor series on float pairs.  Against extended
// precision h + l is 0.65 2^-50 off (rms; a correctly rounded pair 0.64 2^-50), max 2.5 2^-50.
__device__ __forceinline__ Triple2 exp2_pair(long long t0, long long t1, const float2* kT, const int* kF, int& n0, int& n1)
{
    float2 T0, T1, rh, rl;
    exp2_reduce(t0, kT, kF, n0, T0, rh.x, rl.x);
    exp2_reduce(t1, kT, kF, n1, T1, rh.y, rl.y);
    const float2 Th = make_float2(T0.x, T1.x), Tl = make_float2(T0.y, T1.y);
    const float2 C1H = f2dup(-0.6931472f), C1L = f2dup(1.9046542e-09f);     // -ln 2
    const float2 C2H = f2dup(0.2402265f), C2L = f2dup(-2.2778894e-10f);     // ln^2 2 / 2
    const float2 p = __fmul2_rn(C1H, rh);
    float2 pe = __ffma2_rn(C1H, rh, f2neg(p));
    pe = __ffma2_rn(C1L, rh, pe);
    pe = __ffma2_rn(C1H, rl, pe);
    const float2 s = __fmul2_rn(rh, rh);
    float2 se = __ffma2_rn(rh, rh, f2neg(s));
    se = __ffma2_rn(__fadd2_rn(rh, rh), rl, se);
    const float2 q = __fmul2_rn(C2H, s);
    float2 qe = __ffma2_rn(C2H, s, f2neg(q));
    qe = __ffma2_rn(C2L, s, qe);
    qe = __ffma2_rn(C2H, se, qe);
    qe = __ffma2_rn(f2dup(-0.16651233f), __fmul2_rn(s, rl), qe);   // the cube's -ln^3 2 / 2 r_hi^2 r_lo
    // -ln^3 2 / 6 + ln^4 2 / 24 r - ln^5 2 / 120 r^2
    const float2 g = __ffma2_rn(__ffma2_rn(f2dup(-0.0013333558f), rh, f2dup(0.009618129f)), rh, f2dup(-0.05550411f));
    const float2 cub = __fmul2_rn(__fmul2_rn(s, rh), g);
    const float2 Ph = __fadd2_rn(p, q);
    const float2 Pl = __fadd2_rn(__fadd2_rn(f2sub(q, f2sub(Ph, p)), __fadd2_rn(pe, qe)), cub);
    const float2 w = __fmul2_rn(Th, Ph);
    float2 we = __ffma2_rn(Th, Ph, f2neg(w));
    we = __ffma2_rn(Th, Pl, we);
    we = __ffma2_rn(Tl, Ph, we);
    const float2 yh = __fadd2_rn(Th, w);
    return triple_of(yh, f2sub(w, f2sub(yh, Th)), Tl, we, f2dup(0.0f));
}

// y scaled by sc (powers of two; 0 for a node without weight, whose pair is then 0 and 0).  The third
// float, at most half a last place of the second, is dropped: handing it on to a later node of the row
// to even out the row's sum leaves an error of this node's size in one that may be far smaller, where
// it decides the lower envelope (1e-10 of a lower density across two separated streams).
__device__ __forceinline__ void triple_store(const Triple2& y, float2 sc, float2& h, float2& l)
{
    h = __fmul2_rn(y.h, sc);
    l = __fmul2_rn(y.l, sc);
}

// x in units of 2^-58, rounded; |x| < 32.
__device__ __forceinline__ long long fixed58(double x)
{
    const long long b = __double_as_longlong(x);
    const int ex = (int)((b >> 52) & 0x7ff) - 1017;     // the significand's shift
    const long long m = (b & 0xfffffffffffffll) | (1ll << 52);
    long long v;
    if (ex >= 0) v = m << min(ex, 10);
    else if (ex > -54) v = (m + (1ll << (-ex - 1))) >> -ex;
    else v = 0;
    return b < 0 ? -v : v;
}

// Whether x > 0 lies within 2^+-900.
__device__ __forceinline__ bool exponent_ok(double x) { return (unsigned)((__double2hiint(x) >> 20) - 123) <= 1800u; }

// a / b from inv = 1 / b correctly rounded: the corrected product is the correctly rounded quotient
// (Markstein) while nothing over- or underflows.
__device__ __forceinline__ double quotient_of(double a, double b, double inv)
{
    const double t = a * inv;
    return fma(fma(-t, b, a), inv, t);
}

// sqrt(x) from rs = rsqrt(x): one step of Heron's (Newton's) iteration on x rs, its residual by an FMA.
__device__ __forceinline__ double sqrt_of(double x, double rs)
{
    const double s = x * rs;
    return fma(fma(-s, s, x), 0.5 * rs, s);
}

// What rs = rsqrt(x), rounded, misses of 1 / sqrt(x).
__device__ __forceinline__ double rsqrt_rest(double x, double rs)
{
    const double r2 = rs * rs;
    return (0.5 * rs) * fma(-x, fma(rs, rs, -r2), fma(-x, r2, 1.0));
}

// x as the nearest float, the rest's, and the rest's.
__device__ __forceinline__ Triple split_f32(double x)
{
    Triple t;
    t.h = (float)x;
    const double e = x - f64_widen(t.h);
    t.l = (float)e;
    t.r = (float)(e - f64_widen(t.l));
    return t;
}

// Order-preserving integer key of a finite double, and back: minima and maxima on the integer pipe.
__device__ __forceinline__ long long key64(double x)
{
    const long long b = __double_as_longlong(x);
    return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}
__device__ __forceinline__ double unkey64(long long k)
{
    return __longlong_as_double(k ^ ((k >> 63) & 0x7fffffffffffffffll));
}

// Per-state constants of the pair tables: with z = (u - U) sqrt(log2(e) / (2 theta)), z at node
// (nu - 1) / 2 and its step per node, on both axes, in units of 2^-58; A and C, scaled.
struct PairState {
    long long z[2], dz[2];
    Triple A, C;
};

// Launch shape of the pair kernel for a tile of NX nodes per axis: a thread owns 4 x 2 nodes.
// At 32 nodes 128 threads with 8 nodes each hold 64 envelope registers and four blocks fit an SM.
template <int NX>
struct B2pair {
    static constexpr int TX = 4, TY = 2;
    static constexpr int TPX = NX / TX, TPY = NX / TY;
    static constexpr int ACT = TPX * TPY;               // threads that own nodes
    static constexpr int NT = (ACT + 31) / 32 * 32;
    static constexpr int MINB = NT >= 512 ? 1 : 512 / NT;
};

// Shared memory (dynamic) of one element's bounds on float pairs.
template <int NST_, int NX>
struct Bounds2dPairSmem {
    static constexpr int NST = NST_, NSTP = (NST + 1) & ~1, NT = B2pair<NX>::NT, NW = NT / 32;
    union __align__(16) {
        struct {
            float x[NSTP][4][NX];     // a_hi, a_lo, c_hi, c_lo
            float y[NSTP][2][NX];     // b_hi, b_lo
        } tab;
        F64Tables<NST, NX, NW> gen;   // an element out of the pairs' range
    } u;
    double S[NST][4];                 // the stencil
    PairState P[NST];
    float2 kT[128];                   // kbl_exp2_knots
    int kF[128];
    double wt[2][3][NX];              // per axis and node: u times the relaxation of the lower and of the
                                      // upper momentum bound, u^2 / 2 (velocities scaled)
    double red[NW][8];
    Triple q[NX];                     // quadrature weights (a table's: the trapezoidal ones are in the code)
    long long kbox[NW][4];
    int kmax[NW];
    double lo[2], hi[2], h[2], c[2];  // velocity box, grid spacing and node (nu - 1) / 2 per axis
};

template <int NST, int NX>
__device__ __noinline__ void bounds2d_pair_redo(Bounds2dPairSmem<NST, NX>& sm, int E, int e, const Phys& ph,
                                                double* __restrict__ bnd, DevFlags* flags)
{
    bounds2d_f64_states<NST, NX, B2pair<NX>::TX, B2pair<NX>::TY, B2pair<NX>::NT>(sm.S, sm.u.gen, E, e, ph, bnd,
                                                                                         flags);
}

// FP64 value of a float; a zero (or subnormal) gives +-2^-127 or less, next to sums of order 1.
__device__ __forceinline__ double widen_fast(float x)
{
    const int b = __float_as_int(x);
    return __hiloint2double(((b >> 3) & (int)0x8fffffff) + 0x38000000, b << 29);
}

// Column k of the warps' sums, pairwise: one after the other their roundings add up at full size.
template <int NW>
__device__ __forceinline__ double sum_warps(const double (*red)[8], int k)
{
    double a[NW];
#pragma unroll
    for (int q = 0; q < NW; q++) a[q] = red[q][k];
#pragma unroll
    for (int d = 1; d < NW; d *= 2)
#pragma unroll
        for (int q = 0; q + d < NW; q += 2 * d) a[q] += a[q + d];
    return a[0];
}

// Sums of envelope values -M + E (the passes keep the negated M): -m - e + r + q with m the FP32 sum of
// the M, e its error, r the FP32 sum of the E, q its error.
struct Sum4 {
    float m, e, r, q;
    __device__ __forceinline__ double value() const
    {
        return (widen_fast(-m) + widen_fast(-e)) + (widen_fast(r) + widen_fast(q));
    }
};
struct Sum4x2 {
    float2 m, e, r, q;
};
// without q (two summands: one rounding)
struct Sum3 {
    float m, e, r;
    __device__ __forceinline__ double value() const { return (widen_fast(-m) + widen_fast(-e)) + widen_fast(r); }
};
__device__ __forceinline__ Sum4x2 sum_pairs(float2 Ma, float2 Ea, float2 Mb, float2 Eb)
{
    Sum4x2 s;
    f2two_sum(Ma, Mb, s.m, s.e);
    f2two_sum(Ea, Eb, s.r, s.q);
    return s;
}
__device__ __forceinline__ Sum4x2 sum_sums(const Sum4x2& a, const Sum4x2& b)
{
    Sum4x2 s;
    f2two_sum(a.m, b.m, s.m, s.e);
    s.e = __fadd2_rn(s.e, __fadd2_rn(a.e, b.e));
    f2two_sum(a.r, b.r, s.r, s.q);
    s.q = __fadd2_rn(s.q, __fadd2_rn(a.q, b.q));
    return s;
}
__device__ __forceinline__ Sum4 sum_lanes(const Sum4x2& a)
{
    Sum4 s;
    two_sum(a.m.x, a.m.y, s.m, s.e);
    s.e = __fadd_rn(s.e, __fadd_rn(a.e.x, a.e.y));
    two_sum(a.r.x, a.r.y, s.r, s.q);
    s.q = __fadd_rn(s.q, __fadd_rn(a.q.x, a.q.y));
    return s;
}

// Sums of any number of envelope values -M + E over the lanes of a warp, error-free: -m + r + q with m
// the FP32 sum of the M; r that of the E less the errors of m; q what r lost (2^-48 of the values, so
// that its own roundings are of no account).  Two sums side by side.
struct LaneSum2 {
    float2 m, r, q;
};
struct LaneSum {
    float m, r, q;
    __device__ __forceinline__ double value() const { return widen_fast(-m) + (widen_fast(r) + widen_fast(q)); }
};
__device__ __forceinline__ LaneSum2 lane_pair(float2 Ma, float2 Ea, float2 Mb, float2 Eb)
{
    LaneSum2 s;
    float2 e, r, q1, q2;
    f2two_sum(Ma, Mb, s.m, e);
    f2two_sum(Ea, Eb, r, q1);
    f2two_sum(r, f2neg(e), s.r, q2);
    s.q = __fadd2_rn(q1, q2);
    return s;
}
__device__ __forceinline__ LaneSum2 lane_merge(const LaneSum2& a, const LaneSum2& b)
{
    LaneSum2 s = lane_pair(a.m, a.r, b.m, b.r);
    s.q = __fadd2_rn(s.q, __fadd2_rn(a.q, b.q));
    return s;
}
// (a.x, b.x) or (a.y, b.y)
__device__ __forceinline__ LaneSum2 lane_x(const LaneSum2& a, const LaneSum2& b)
{
    return {make_float2(a.m.x, b.m.x), make_float2(a.r.x, b.r.x), make_float2(a.q.x, b.q.x)};
}
__device__ __forceinline__ LaneSum2 lane_y(const LaneSum2& a, const LaneSum2& b)
{
    return {make_float2(a.m.y, b.m.y), make_float2(a.r.y, b.r.y), make_float2(a.q.y, b.q.y)};
}
// A step of a reduce-scatter: the lanes with up keep hi and the others lo, each plus its partner's.
__device__ __forceinline__ LaneSum2 lane_exchange(const LaneSum2& lo, const LaneSum2& hi, bool up, int off)
{
    auto swap = [&](float l, float h, float& keep) {
        keep = up ? h : l;
        return __shfl_xor_sync(0xffffffffu, up ? l : h, off);
    };
    LaneSum2 k, o;
    o.m.x = swap(lo.m.x, hi.m.x, k.m.x);
    o.m.y = swap(lo.m.y, hi.m.y, k.m.y);
    o.r.x = swap(lo.r.x, hi.r.x, k.r.x);
    o.r.y = swap(lo.r.y, hi.r.y, k.r.y);
    o.q.x = swap(lo.q.x, hi.q.x, k.q.x);
    o.q.y = swap(lo.q.y, hi.q.y, k.q.y);
    return lane_merge(k, o);
}

// 2^k for |k| <= 1000
__device__ __forceinline__ double pow2_f64(int k) { return __hiloint2double((1023 + k) << 20, 0); }

// Bounds of element e from a stencil of NST states, one block of B2pair<NX>::NT threads: gather(S)
// fills S[NST][4]; the bounds go to column e of bnd[2][4][E].
template <int NST, int NX, typename Gather>
__device__ __forceinline__ void bounds2d_pair_core(Bounds2dPairSmem<NST, NX>& sm, Gather gather, int E, int e,
                                                   const Phys& ph, double* __restrict__ bnd, DevFlags* flags)
{
    using SM = Bounds2dPairSmem<NST, NX>;
    using SH = B2pair<NX>;
    constexpr int NT = SH::NT, NW = SM::NW, NSTP = SM::NSTP, TX = SH::TX, TY = SH::TY;
    static_assert(TX == 4, "two packed pairs of x nodes per thread");
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    static_assert(NST <= NT, "a thread per state");
    const int nu = ph.nu[0];   // nodes per axis; tile nodes j >= nu carry no weight
    gather(sm.S);              // thread i fills S[i]
    for (int k = tid; k < 128; k += NT) {
        const Exp2Knot q = kbl_exp2_knots[k];
        sm.kT[k] = make_float2(__uint_as_float(q.hi), __uint_as_float(q.lo));
        sm.kF[k] = q.f;
    }

    // 1. primitive states in FP64, one thread each.  With inv = 1 / rho correctly rounded, the
    //    corrected product a inv is the correctly rounded a / rho (Markstein), within the exponent
    //    range checked first.
    long long klo[2] = {0x7fffffffffffffffll, 0x7fffffffffffffffll}, khi[2] = {-0x7fffffffffffffffll, -0x7fffffffffffffffll};
    int kA = 0, bad = 0, out_of_range = 0;
    double th = 0.0, rs = 0.0, U[2] = {0.0, 0.0}, A = 0.0;
    double(*kap)[4] = reinterpret_cast<double(*)[4]>(&sm.u.tab);   // per state kappa and U, until the tables
    if (tid < NST) {
        const double rho = sm.S[tid][0], mx = sm.S[tid][1], my = sm.S[tid][2], En = sm.S[tid][3];
        if (exponent_ok(rho) && exponent_ok(En)) {
            const double inv = 1.0 / rho;
            auto over_rho = [&](double a) { return quotient_of(a, rho, inv); };
            double mm = mx * mx;
            mm += my * my;
            const double P = (ph.gamma - 1.0) * (En - over_rho(0.5 * mm));
            bad = !(P > 0.0);
            th = over_rho(P);
            U[0] = over_rho(mx);
            U[1] = over_rho(my);
            rs = rsqrt(th);
            double sq = sqrt_of(th, rs);
            const double it = rs * rs;
            A = rho * it;                           // rho / theta (1 / (2 pi) is in the exponents)
            A = fma(fma(-A, th, rho), it, A);
#pragma unroll
            for (int d = 0; d < 2; d++) {
                klo[d] = key64(fma(-ph.k, sq, U[d]));
                khi[d] = key64(fma(ph.k, sq, U[d]));
            }
            kA = __double2hiint(A);
            out_of_range = !exponent_ok(th);
            // kappa = sqrt(log2(e) / 2) / sqrt(theta) as kh + kl
            const double rl = rsqrt_rest(th, rs);
            const double kh = 0.8493218002880191 * rs;
            kap[tid][0] = kh;
            kap[tid][1] =
                fma(0.8493218002880191, rs, -kh) + fma(-2.5959464104597403e-17, rs, 0.8493218002880191 * rl);
            kap[tid][2] = U[0];
            kap[tid][3] = U[1];
        } else {
            bad = !(rho > 0.0) || !(kbl_pressure<2>(sm.S[tid], ph.gamma - 1.0) > 0.0);
            out_of_range = 1;
            kap[tid][0] = kap[tid][1] = kap[tid][2] = kap[tid][3] = 0.0;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
        for (int d = 0; d < 2; d++) {
            klo[d] = min(klo[d], __shfl_xor_sync(0xffffffffu, klo[d], o));
            khi[d] = max(khi[d], __shfl_xor_sync(0xffffffffu, khi[d], o));
        }
        kA = max(kA, __shfl_xor_sync(0xffffffffu, kA, o));
    }
    if (lane == 0) {
        sm.kbox[wid][0] = klo[0]; sm.kbox[wid][1] = khi[0];
        sm.kbox[wid][2] = klo[1]; sm.kbox[wid][3] = khi[1];
        sm.kmax[wid] = kA;
    }
    if (__syncthreads_or(bad)) {
        if (tid == 0) {
            write_nan(bnd, E, e, 4);
            atomicOr(&flags->nonphysical, 1);
        }
        return;
    }
    if (tid < 2) {
        long long a = sm.kbox[0][2 * tid], b = sm.kbox[0][2 * tid + 1];
#pragma unroll
        for (int q = 1; q < NW && 32 * q < NST; q++) {
            a = min(a, sm.kbox[q][2 * tid]);
            b = max(b, sm.kbox[q][2 * tid + 1]);
        }
        const double la = unkey64(a), lb = unkey64(b);
        const double hd = (lb - la) / (nu - 1);
        sm.lo[tid] = la;
        sm.hi[tid] = lb;
        sm.h[tid] = hd;
        sm.c[tid] = fma((double)((nu - 1) / 2), hd, la);
    }
    kA = sm.kmax[0];
#pragma unroll
    for (int q = 1; q < NW && 32 * q < NST; q++) kA = max(kA, sm.kmax[q]);
    __syncthreads();
    // exact powers of two that bring A and the velocities to order 1
    const int eA = (kA >> 20) - 1023;
    int kU = 0;
#pragma unroll
    for (int d = 0; d < 2; d++)
        kU = max(kU, max(__double2hiint(sm.lo[d]) & 0x7fffffff, __double2hiint(sm.hi[d]) & 0x7fffffff));
    const int eU = (kU >> 20) - 1022;
    if (abs(eA) > 900 || abs(eU) > 450) out_of_range = 1;
    const double sA = pow2_f64(abs(eA) > 900 ? 0 : -eA), sU = pow2_f64(abs(eU) > 450 ? 0 : -eU);

    // 2. scaled constants, and the velocity grid's coefficients: a thread per state and axis where the
    //    block has as many (FP64 instructions take as long for half a warp as for a whole one, and the
    //    chain is shorter: 128^2 P3 step 3.01 -> 2.95 ms against a thread per state)
    if (tid < NST) {
        const Triple At = split_f32(A * sA), Ct = split_f32(ph.half_delta2 * th * (sU * sU));
        sm.P[tid].A = At;
        sm.P[tid].C = Ct;
        if (!(At.h >= 0x1p-60f) || !(Ct.h == 0.0f || (Ct.h >= 0x1p-30f && Ct.h < 0x1p60f))) out_of_range = 1;
    }
    auto grid_coefficients = [&](int i, int d) {
        const double kh = kap[i][0], kl = kap[i][1], hd = sm.h[d], dc = sm.c[d] - kap[i][2 + d];
        const double zh = dc * kh, dh = hd * kh;
        // the low parts, below 2^-48, in units of 2^-58 like the high ones
        const double zl = fma(dc, kl, fma(dc, kh, -zh)), dl = fma(hd, kl, fma(hd, kh, -dh));
        sm.P[i].z[d] = fixed58(zh) + fixed58(zl);
        sm.P[i].dz[d] = fixed58(dh) + fixed58(dl);
        // the largest exponent over the box, in FP32 with a margin
        if (!(fabsf(f32_trunc(zh)) + f32_trunc(dh) * (float)(nu / 2 + 1) < 15.5f)) out_of_range = 1;
    };
    if constexpr (2 * NST <= NT) {
        if (tid < 2 * NST) grid_coefficients(tid < NST ? tid : tid - NST, tid < NST ? 0 : 1);
    } else if (tid < NST) {
#pragma unroll
        for (int d = 0; d < 2; d++) grid_coefficients(tid, d);
    }
    for (int j = NT - 1 - tid; j < 2 * NX; j += NT) {   // from the last thread: the first hold states
        const int d = j / NX, jj = j % NX;
        const double u = sm.lo[d] + min(jj, nu - 1) * sm.h[d];
        const double us = u * sU;
        const bool neg = __double2hiint(us) < 0;
        sm.wt[d][0][jj] = us * (neg ? ph.rel_hi : ph.rel_lo);
        sm.wt[d][1][jj] = us * (neg ? ph.rel_lo : ph.rel_hi);
        sm.wt[d][2][jj] = 0.5 * us * us;
        if (ph.qw && d == 0) sm.q[jj] = split_f32(kbl_qweight(ph, jj, nu));
    }
    if (__syncthreads_or(out_of_range)) {
        bounds2d_pair_redo<NST, NX>(sm, E, e, ph, bnd, flags);
        return;
    }

    // 3. row tables: runs of 8 nodes, t by second differences
    constexpr int SEG = 8, NSG = NX / SEG;
    for (int task = tid; task < NSTP * 2 * NSG; task += NT) {
        const int axis = task >= NSTP * NSG, i = (task / NSG) % NSTP, jb = (task % NSG) * SEG;   // x rows first
        const PairState& s = sm.P[i < NST ? i : NST - 1];
        // t = z^2 and its differences in units of 2^-55, rounded to nearest (their errors add up over
        // the run; the tail of a padded tile may wrap: it carries no weight)
        const long long dz = s.dz[axis], z = s.z[axis] + (jb - (nu - 1) / 2) * dz;
        const unsigned long long z4 = 4ull * (unsigned long long)(z < 0 ? -z : z);
        long long t = (long long)((__umul64hi(z4, z4) + 1ull) >> 1);
        long long dt = (__mul64hi(2 * z + dz, 16 * dz) + 1) >> 1;   // (2 z + dz) dz
        const long long dd = (__mul64hi(8 * dz, 4 * dz) + 1) >> 1;
        if (axis == 0) t += 95530215845326779ll;   // log2(2 pi): the Maxwellian's 1 / (2 pi)
        const Triple A = s.A, C = s.C;
#pragma unroll 1
        for (int j = jb; j < jb + SEG; j += 2) {
            int n0, n1;
            const long long t1 = t + dt;
            Triple2 y = exp2_pair(t < 0 ? 0 : t, t1 < 0 ? 0 : t1, sm.kT, sm.kF, n0, n1);
            float2 sc = make_float2(n0 < 120 && j < nu ? __uint_as_float((unsigned)(127 - n0) << 23) : 0.0f,
                                    n1 < 120 && j + 1 < nu ? __uint_as_float((unsigned)(127 - n1) << 23) : 0.0f);
            // the node's quadrature weight scales every state alike, so the envelopes carry it
            if (ph.qw) {
                const Triple q0 = sm.q[j], q1 = sm.q[j + 1];
                y = triple_mul(y, make_float2(q0.h, q1.h), make_float2(q0.l, q1.l), make_float2(q0.r, q1.r));
            } else {
                if (j == 0) sc.x *= 0.5f;
                if (j == nu - 1) sc.x *= 0.5f;
                if (j + 1 == nu - 1) sc.y *= 0.5f;
            }
            float2 h, l;
            if (axis == 0) {
                y = triple_mul(y, f2dup(A.h), f2dup(A.l), f2dup(A.r));
                triple_store(y, sc, h, l);
                *(float2*)&sm.u.tab.x[i][0][j] = h;
                *(float2*)&sm.u.tab.x[i][1][j] = l;
                y = triple_mul(y, f2dup(C.h), f2dup(C.l), f2dup(C.r));
                triple_store(y, sc, h, l);
                *(float2*)&sm.u.tab.x[i][2][j] = h;
                *(float2*)&sm.u.tab.x[i][3][j] = l;
            } else {
                triple_store(y, sc, h, l);
                *(float2*)&sm.u.tab.y[i][0][j] = h;
                *(float2*)&sm.u.tab.y[i][1][j] = l;
            }
            dt += dd;
            t = t1 + dt;
            dt += dd;
        }
    }
    __syncthreads();

    // 4. envelopes of the thread's 4 x TY nodes, [y][pair of x]
    const int tx = tid % SH::TPX, ty = tid / SH::TPX;
    double acc[8];   // rho lower/upper, m_x, m_y, E
#pragma unroll
    for (int k = 0; k < 8; k++) acc[k] = 0.0;
    if (tid < SH::ACT) {
        float2 tlo[TY][2], thi[TY][2], ilo[TY][2], ihi[TY][2];
#pragma unroll
        for (int b = 0; b < TY; b++)
#pragma unroll
            for (int p = 0; p < 2; p++) {
                tlo[b][p] = ilo[b][p] = f2dup(FLT_MAX);
                thi[b][p] = ihi[b][p] = f2dup(0.0f);
            }
#pragma unroll 2
        for (int i = 0; i < NSTP; i += 2) {
            const float4 a0 = *(const float4*)&sm.u.tab.x[i][0][4 * tx], a1 = *(const float4*)&sm.u.tab.x[i + 1][0][4 * tx];
            const float4 c0 = *(const float4*)&sm.u.tab.x[i][2][4 * tx], c1 = *(const float4*)&sm.u.tab.x[i + 1][2][4 * tx];
            const float2 A0[2] = {make_float2(a0.x, a0.y), make_float2(a0.z, a0.w)};
            const float2 A1[2] = {make_float2(a1.x, a1.y), make_float2(a1.z, a1.w)};
            const float2 C0[2] = {make_float2(c0.x, c0.y), make_float2(c0.z, c0.w)};
            const float2 C1[2] = {make_float2(c1.x, c1.y), make_float2(c1.z, c1.w)};
            const float2 b0 = *(const float2*)&sm.u.tab.y[i][0][ty * TY], b1 = *(const float2*)&sm.u.tab.y[i + 1][0][ty * TY];
#pragma unroll
            for (int b = 0; b < TY; b++) {
                const float2 y0 = f2dup(b ? b0.y : b0.x), y1 = f2dup(b ? b1.y : b1.x);
#pragma unroll
                for (int p = 0; p < 2; p++) {
                    const float2 g0 = __fmul2_rn(A0[p], y0), g1 = __fmul2_rn(A1[p], y1);
                    tlo[b][p].x = fmin3(tlo[b][p].x, g0.x, g1.x);
                    tlo[b][p].y = fmin3(tlo[b][p].y, g0.y, g1.y);
                    thi[b][p].x = fmax3(thi[b][p].x, g0.x, g1.x);
                    thi[b][p].y = fmax3(thi[b][p].y, g0.y, g1.y);
                    const float2 k0 = __fmul2_rn(C0[p], y0), k1 = __fmul2_rn(C1[p], y1);
                    ilo[b][p].x = fmin3(ilo[b][p].x, k0.x, k1.x);
                    ilo[b][p].y = fmin3(ilo[b][p].y, k0.y, k1.y);
                    ihi[b][p].x = fmax3(ihi[b][p].x, k0.x, k1.x);
                    ihi[b][p].y = fmax3(ihi[b][p].y, k0.y, k1.y);
                }
            }
        }
        float2 etl[TY][2], eth[TY][2], eil[TY][2], eih[TY][2];
#pragma unroll
        for (int b = 0; b < TY; b++)
#pragma unroll
            for (int p = 0; p < 2; p++) {
                tlo[b][p] = f2neg(tlo[b][p]); thi[b][p] = f2neg(thi[b][p]);
                ilo[b][p] = f2neg(ilo[b][p]); ihi[b][p] = f2neg(ihi[b][p]);
                etl[b][p] = eil[b][p] = f2dup(FLT_MAX);
                eth[b][p] = eih[b][p] = f2dup(-FLT_MAX);
            }
#pragma unroll 1
        for (int i = 0; i < NSTP; i += 2) {
            float2 X[2][4][2];   // [state][a_hi, a_lo, c_hi, c_lo][pair]
#pragma unroll
            for (int s = 0; s < 2; s++)
#pragma unroll
                for (int k = 0; k < 4; k++) {
                    const float4 v = *(const float4*)&sm.u.tab.x[i + s][k][4 * tx];
                    X[s][k][0] = make_float2(v.x, v.y);
                    X[s][k][1] = make_float2(v.z, v.w);
                }
            float2 Y[2][2];      // [state][b_hi, b_lo] of both y nodes
#pragma unroll
            for (int s = 0; s < 2; s++)
#pragma unroll
                for (int k = 0; k < 2; k++) Y[s][k] = *(const float2*)&sm.u.tab.y[i + s][k][ty * TY];
#pragma unroll
            for (int b = 0; b < TY; b++) {
                const float2 bh0 = f2dup(b ? Y[0][0].y : Y[0][0].x), bl0 = f2dup(b ? Y[0][1].y : Y[0][1].x);
                const float2 bh1 = f2dup(b ? Y[1][0].y : Y[1][0].x), bl1 = f2dup(b ? Y[1][1].y : Y[1][1].x);
#pragma unroll
                for (int p = 0; p < 2; p++) {
                    // a b - M of both states
                    auto res = [&](int s, int k, float2 M) {
                        const float2 bh = s ? bh1 : bh0, bl = s ? bl1 : bl0;
                        const float2 r = __ffma2_rn(X[s][k][p], bh, M);
                        return __ffma2_rn(X[s][k + 1][p], bh, __ffma2_rn(X[s][k][p], bl, r));
                    };
                    float2 r0 = res(0, 0, tlo[b][p]), r1 = res(1, 0, tlo[b][p]);
                    etl[b][p].x = fmin3(etl[b][p].x, r0.x, r1.x);
                    etl[b][p].y = fmin3(etl[b][p].y, r0.y, r1.y);
                    r0 = res(0, 0, thi[b][p]), r1 = res(1, 0, thi[b][p]);
                    eth[b][p].x = fmax3(eth[b][p].x, r0.x, r1.x);
                    eth[b][p].y = fmax3(eth[b][p].y, r0.y, r1.y);
                    r0 = res(0, 2, ilo[b][p]), r1 = res(1, 2, ilo[b][p]);
                    eil[b][p].x = fmin3(eil[b][p].x, r0.x, r1.x);
                    eil[b][p].y = fmin3(eil[b][p].y, r0.y, r1.y);
                    r0 = res(0, 2, ihi[b][p]), r1 = res(1, 2, ihi[b][p]);
                    eih[b][p].x = fmax3(eih[b][p].x, r0.x, r1.x);
                    eih[b][p].y = fmax3(eih[b][p].y, r0.y, r1.y);
                }
            }
        }

        if constexpr (SH::TPX == 8 && SH::ACT == NT && NST <= 40) {
            // 5. moments, a lane's nodes 4 x 2 and a warp's 32 x 8: the envelopes' two floats meet in
            //    error-free FP32 sums, first a lane's, then by a reduce-scatter over the warp -- rows
            //    (weights in v) and the internal energy over the eight lanes of a row, columns (weights
            //    in u) over the four lanes of a column -- so that a lane ends with one row or energy sum
            //    and one column: 12 FP64 instructions a thread instead of 42, for 200 FP32 ones and
            //    shuffles.  Pays where few states leave the passes short beside the FP64 pipe.  Launch with
            //    it / without, 16,384 elements: 16 states 421 / 471 us, 20 (P1 quads) 500 / 516, 24 531 / 552,
            //    33 (P2 quads) 676 / 711; 48 states 844 / 826 (P3 quads 846 / 830): the passes set the pace,
            //    and the line lies between the two
            LaneSum2 V[2], C[2][2], I[2];   // V: both rows of a lower or upper envelope, C: [pair of columns]
#pragma unroll
            for (int s = 0; s < 2; s++) {
                const float2(&M)[TY][2] = s ? thi : tlo;
                const float2(&r)[TY][2] = s ? eth : etl;
                const LaneSum2 v0 = lane_pair(M[0][0], r[0][0], M[0][1], r[0][1]);
                const LaneSum2 v1 = lane_pair(M[1][0], r[1][0], M[1][1], r[1][1]);
                V[s] = lane_merge(lane_x(v0, v1), lane_y(v0, v1));
                LaneSum2 ci[2];
#pragma unroll
                for (int p = 0; p < 2; p++) {
                    C[p][s] = lane_pair(M[0][p], r[0][p], M[1][p], r[1][p]);
                    ci[p] = s ? lane_pair(ihi[0][p], eih[0][p], ihi[1][p], eih[1][p])
                              : lane_pair(ilo[0][p], eil[0][p], ilo[1][p], eil[1][p]);
                }
                I[s] = lane_merge(ci[0], ci[1]);
            }
            const LaneSum2 both = lane_merge(lane_x(I[0], I[1]), lane_y(I[0], I[1]));
            // lanes with bit 2: energy, lower or upper by bit 0 (none with bit 1); the others: row bit 0,
            // lower or upper by bit 1
            const LaneSum2 none = {f2dup(0.0f), f2dup(0.0f), f2dup(0.0f)};
            LaneSum2 t = lane_exchange(lane_exchange(V[0], both, lane & 4, 4), lane_exchange(V[1], none, lane & 4, 4),
                                       lane & 2, 2);
            t = lane_exchange(t, lane_y(t, t), lane & 1, 1);
            const bool energy = lane & 4, up = lane & (energy ? 1 : 2);
            const int jy = ty * TY + (lane & 1);
            const double val = LaneSum{t.m.x, t.r.x, t.q.x}.value();
            const double v0 = sm.wt[1][0][jy], v1 = sm.wt[1][1][jy], kv = sm.wt[1][2][jy];
            // v < 0: the lower sum takes the upper envelope
            const bool lower = up == (__double2hiint(v0) < 0);
            const double mv = (lower ? v0 : v1) * val, ev = (energy ? (lane & 2 ? 0.0 : 1.0) : kv) * val;
            acc[0] = energy || up ? 0.0 : val;
            acc[1] = !energy && up ? val : 0.0;
            acc[4] = !energy && lower ? mv : 0.0;
            acc[5] = energy || lower ? 0.0 : mv;
            // a column's lower and upper sum: column 2 (bit 4) + bit 3 of the lane's four
            const LaneSum2 c0 = lane_exchange(C[0][0], C[1][0], lane & 16, 16);
            const LaneSum2 c1 = lane_exchange(C[0][1], C[1][1], lane & 16, 16);
            const LaneSum2 c = lane_exchange(lane_x(c0, c1), lane_y(c0, c1), lane & 8, 8);
            const int jx = 4 * tx + ((lane >> 3) & 1) + 2 * (lane >> 4);
            const double lo = LaneSum{c.m.x, c.r.x, c.q.x}.value(), hi = LaneSum{c.m.y, c.r.y, c.q.y}.value();
            const double u0 = sm.wt[0][0][jx], u1 = sm.wt[0][1][jx], ku = sm.wt[0][2][jx];
            const bool neg = __double2hiint(u0) < 0;
            acc[2] = u0 * (neg ? hi : lo);
            acc[3] = u1 * (neg ? lo : hi);
            acc[6] = fma(ku, lo, up ? 0.0 : ev);
            acc[7] = fma(ku, hi, up ? ev : 0.0);
        } else {
            // 5. moments: the envelopes' two floats meet in error-free FP32 sums (a row over x for the weights
            //    in v, a column over y for those in u, everything for I), which then enter FP64: a third of
            //    the FP64 instructions that node by node takes (8.4k clocks per element on that pipe before)
            Sum4 V[TY][2], I[2];
            Sum3 C[TX][2];
    #pragma unroll
            for (int s = 0; s < 2; s++) {
    #pragma unroll
                for (int b = 0; b < TY; b++) {
                    const float2(&M)[2] = s ? thi[b] : tlo[b];
                    const float2(&r)[2] = s ? eth[b] : etl[b];
                    V[b][s] = sum_lanes(sum_pairs(M[0], r[0], M[1], r[1]));
                }
                Sum4x2 ci[2];
    #pragma unroll
                for (int p = 0; p < 2; p++) {
                    float2 m, e;
                    f2two_sum(s ? thi[0][p] : tlo[0][p], s ? thi[1][p] : tlo[1][p], m, e);
                    const float2 r = __fadd2_rn(s ? eth[0][p] : etl[0][p], s ? eth[1][p] : etl[1][p]);
                    C[2 * p][s] = Sum3{m.x, e.x, r.x};
                    C[2 * p + 1][s] = Sum3{m.y, e.y, r.y};
                    ci[p] = s ? sum_pairs(ihi[0][p], eih[0][p], ihi[1][p], eih[1][p])
                              : sum_pairs(ilo[0][p], eil[0][p], ilo[1][p], eil[1][p]);
                }
                I[s] = sum_lanes(sum_sums(ci[0], ci[1]));
            }
            double vs[TY][2];
    #pragma unroll
            for (int b = 0; b < TY; b++) {
                const int jy = ty * TY + b;
                const double v0 = sm.wt[1][0][jy], v1 = sm.wt[1][1][jy], kv = sm.wt[1][2][jy];
                const bool neg = __double2hiint(v0) < 0;   // v < 0: the lower sum takes the upper envelope
    #pragma unroll
                for (int s = 0; s < 2; s++) vs[b][s] = V[b][s].value();
                acc[4] = fma(v0, neg ? vs[b][1] : vs[b][0], acc[4]);
                acc[5] = fma(v1, neg ? vs[b][0] : vs[b][1], acc[5]);
                acc[6] = fma(kv, vs[b][0], acc[6]);
                acc[7] = fma(kv, vs[b][1], acc[7]);
            }
            acc[0] = vs[0][0] + vs[1][0];
            acc[1] = vs[0][1] + vs[1][1];
            acc[6] += I[0].value();
            acc[7] += I[1].value();
    #pragma unroll
            for (int a = 0; a < TX; a++) {
                const int jx = 4 * tx + a;
                const double u0 = sm.wt[0][0][jx], u1 = sm.wt[0][1][jx], ku = sm.wt[0][2][jx];
                const bool neg = __double2hiint(u0) < 0;
                const double c0 = C[a][0].value(), c1 = C[a][1].value();
                acc[2] = fma(u0, neg ? c1 : c0, acc[2]);
                acc[3] = fma(u1, neg ? c0 : c1, acc[3]);
                acc[6] = fma(ku, c0, acc[6]);
                acc[7] = fma(ku, c1, acc[7]);
            }
        }
    }
    // 6. warp reduce-scatter of the eight sums (lane 4 k holds sum k), then the warps
#pragma unroll
    for (int step = 0; step < 3; step++) {
        const int off = 16 >> step, n = 4 >> step;
        const bool up = lane & off;
#pragma unroll
        for (int k = 0; k < 4; k++) {
            if (k >= n) break;
            const double keep = up ? acc[n + k] : acc[k], send = up ? acc[k] : acc[n + k];
            acc[k] = keep + __shfl_xor_sync(0xffffffffu, send, off);
        }
    }
#pragma unroll
    for (int off = 2; off > 0; off >>= 1) acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], off);
    if ((lane & 3) == 0) sm.red[wid][lane >> 2] = acc[0];
    __syncthreads();
    int redo = 0;
    if (tid < 8) {
        double s = sum_warps<NW>(sm.red, tid);
        // sum k: rho, m_x, m_y, E (k >> 1), lower then upper
        const int v = tid >> 1, up = tid & 1;
        if (tid == 0 && !(s >= 0x1p-40)) redo = 1;
        // times h_x h_y and the relaxation (in the momentum weights already), rounded once
        const double hh = sm.h[0] * sm.h[1], p = s * hh;
        const double rest = fma(s, fma(sm.h[0], sm.h[1], -hh), fma(s, hh, -p));
        const double rel = v == 0 || v == 3 ? (up ? ph.rel_hi : ph.rel_lo) : 1.0;
        double val = fma(rel, p, rel * rest) * pow2_f64(eA) * (v == 0 ? 1.0 : v == 3 ? pow2_f64(2 * eU) : pow2_f64(eU));
        if (tid == 0 && val < ph.rho_floor) val = ph.rho_floor;
        bnd[((size_t)up * 4 + v) * E + e] = val;
    }
    if (__syncthreads_or(redo)) {
        bounds2d_pair_redo<NST, NX>(sm, E, e, ph, bnd, flags);
    }
}

// ---------------------------------------------------------------------------
// 1D, full precision: every Maxwellian of a node as three floats (exp2_pair on fixed-point
// exponents), the envelopes by comparing those, the sums in FP64
// ---------------------------------------------------------------------------
// Per-state constants: as PairState, the step in units of 2^-(58 + floor(log2 nu)).
struct LineState {
    long long z, dz;
    Triple A, C;
};

// The larger (UP) or smaller of best and x, decided on all three floats: of states equal to 1e-15 or so
// the leading two cannot tell the extreme one, and the lower bounds came out 3e-16 high, the upper ones
// as much low.
template <bool UP>
__device__ __forceinline__ void triple_extreme(Triple& best, const Triple& x)
{
    const float d = __fadd_rn(__fsub_rn(x.h, best.h), __fadd_rn(__fsub_rn(x.l, best.l), __fsub_rn(x.r, best.r)));
    if (UP ? d > 0.0f : d < 0.0f) best = x;
}
__device__ __forceinline__ double triple_value(const Triple& a)
{
    return widen_fast(a.h) + (widen_fast(a.l) + widen_fast(a.r));
}

// Add node u's terms to the raw sums of finalize_bounds<1>.
__device__ __forceinline__ void line_moments(double (&acc)[8], double u, double Tl, double Th, double Il, double Ih)
{
    acc[0] += Tl;
    acc[1] += Th;
    if (u < 0.0) { acc[2] = fma(Th, u, acc[2]); acc[3] = fma(Tl, u, acc[3]); }
    else { acc[4] = fma(Tl, u, acc[4]); acc[5] = fma(Th, u, acc[5]); }
    const double ke = 0.5 * u * u;
    acc[6] += fma(Tl, ke, Il);
    acc[7] += fma(Th, ke, Ih);
}

// Raw sums of one thread's nodes by FP64 exponentials: stencils out of the floats' range.
struct LineSums {
    double v[8];
};
template <int NST>
__device__ __noinline__ LineSums bounds1d_f64_nodes(const StatePrim* sP, const Phys& ph, double lo, double h, int tid,
                                                    int nt)
{
    LineSums s;
#pragma unroll
    for (int k = 0; k < 8; k++) s.v[k] = 0.0;
    for (int j = tid; j < ph.nu[0]; j += nt) {
        const double u = lo + j * h, q = kbl_qweight(ph, j, ph.nu[0]);
        double Tl = DBL_MAX, Th = 0.0, Il = DBL_MAX, Ih = -DBL_MAX;
        for (int i = 0; i < NST; i++) {
            const double d = u - sP[i].U[0];
            const double g = sP[i].A * exp(-(d * d) / (2.0 * sP[i].th));
            const double cg = sP[i].C * g;
            Tl = fmin(Tl, g); Th = fmax(Th, g);
            Il = fmin(Il, cg); Ih = fmax(Ih, cg);
        }
        line_moments(s.v, u, q * Tl, q * Th, q * Il, q * Ih);
    }
    return s;
}

template <int NST, int NT>
struct Bounds1dSmem {
    double S[NST][3];
    LineState P[NST];
    StatePrim G[NST];      // the FP64 path's
    float2 kT[128];        // kbl_exp2_knots
    int kF[128];
    double lo, h, c;       // box end, spacing and node (nu - 1) / 2
    int eA, eU;            // exponents taken out of A and of the velocities
    double red[NT / 32][8];
};

// Bounds of element e, one block of NT threads, sm.S filled by the threads of warp 0 (or with a
// barrier after).
template <int NST, int NT>
__device__ __forceinline__ void bounds1d_core(Bounds1dSmem<NST, NT>& sm, int E, int e, const Phys& ph,
                                              double* __restrict__ bnd, DevFlags* flags)
{
    static_assert(NST <= 32, "the states of one warp");
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nu = ph.nu[0], jc = (nu - 1) / 2;
    const int sh = 31 - __clz(nu);
    for (int k = tid; k < 128; k += NT) {
        const Exp2Knot q = kbl_exp2_knots[k];
        sm.kT[k] = make_float2(__uint_as_float(q.hi), __uint_as_float(q.lo));
        sm.kF[k] = q.f;
    }
    int bad = 0, out_of_range = 0;
    if (wid == 0) {   // the states, one lane each; the other warps wait
        double th = 1.0, rs = 1.0, U = 0.0, rho = 1.0;
        long long klo = 0x7fffffffffffffffll, khi = -0x7fffffffffffffffll;
        if (lane < NST) {
            rho = sm.S[lane][0];
            const double mx = sm.S[lane][1], En = sm.S[lane][2];
            if (exponent_ok(rho) && exponent_ok(En)) {
                const double inv = 1.0 / rho;
                const double P = (ph.gamma - 1.0) * (En - quotient_of(0.5 * (mx * mx), rho, inv));
                bad = !(P > 0.0);
                th = quotient_of(P, rho, inv);
                U = quotient_of(mx, rho, inv);
                out_of_range = !exponent_ok(th);
            } else {
                bad = !(rho > 0.0) || !(kbl_pressure<1>(sm.S[lane], ph.gamma - 1.0) > 0.0);
                out_of_range = 1;
            }
            rs = rsqrt(th);
            double sq = sqrt_of(th, rs);
            klo = key64(fma(-ph.k, sq, U));
            khi = key64(fma(ph.k, sq, U));
        }
        const double A = rho * rs;                    // 1 / sqrt(2 pi) is in the exponents
        int kA = lane < NST ? __double2hiint(A) : 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            klo = min(klo, __shfl_xor_sync(0xffffffffu, klo, o));
            khi = max(khi, __shfl_xor_sync(0xffffffffu, khi, o));
            kA = max(kA, __shfl_xor_sync(0xffffffffu, kA, o));
        }
        const double la = unkey64(klo), lb = unkey64(khi), h = (lb - la) / (nu - 1), c = fma((double)jc, h, la);
        const int eA = (kA >> 20) - 1023;
        const int eU = (max(__double2hiint(la) & 0x7fffffff, __double2hiint(lb) & 0x7fffffff) >> 20) - 1022;
        if (abs(eA) > 900 || abs(eU) > 450) out_of_range = 1;
        const double sA = pow2_f64(abs(eA) > 900 ? 0 : -eA), sU = pow2_f64(abs(eU) > 450 ? 0 : -eU);
        const double rl = rsqrt_rest(th, rs);
        Triple At = split_f32(A * sA);
        At.r += (float)(fma(rho, rs, -A) * sA + rho * rl * sA);
        const Triple Ct = split_f32(ph.half_delta1 * th * (sU * sU));
        const double kh = 0.8493218002880191 * rs;
        const double kl = fma(0.8493218002880191, rs, -kh) + fma(-2.5959464104597403e-17, rs, 0.8493218002880191 * rl);
        const double dc = c - U, zh = dc * kh, dh = h * kh;
        const double zl = fma(dc, kl, fma(dc, kh, -zh)), dl = fma(h, kl, fma(h, kh, -dh));
        const double up = pow2_f64(sh);
        if (lane < NST) {
            sm.P[lane].z = fixed58(zh) + fixed58(zl);
            sm.P[lane].dz = fixed58(dh * up) + fixed58(dl * up);   // below 31 by the range test
            sm.P[lane].A = At;
            sm.P[lane].C = Ct;
            const float tm = fabsf(f32_trunc(zh)) + f32_trunc(dh) * (float)(nu / 2 + 1);
            if (!(tm < 15.5f) || !(At.h >= 0x1p-60f) || !(Ct.h == 0.0f || (Ct.h >= 0x1p-30f && Ct.h < 0x1p60f)))
                out_of_range = 1;
        }
        if (lane == 0) {
            sm.lo = la;
            sm.h = h;
            sm.c = c;
            sm.eA = eA;
            sm.eU = eU;
        }
    }
    if (__syncthreads_or(bad)) {
        if (tid == 0) {
            write_nan(bnd, E, e, 3);
            atomicOr(&flags->nonphysical, 1);
        }
        return;
    }
    bool pairs = !__syncthreads_or(out_of_range);
    for (;;) {
        double acc[8];
#pragma unroll
        for (int k = 0; k < 8; k++) acc[k] = 0.0;
        const double lo = sm.lo, h = sm.h;
        if (pairs) {
            const double sU = pow2_f64(-sm.eU);
            for (int j = tid; j < nu; j += NT) {
                Triple Tl, Th, Il, Ih;
                const long long k = (long long)(j - jc) << (63 - sh);
#pragma unroll 1
                for (int i = 0; i < NST; i += 2) {
                    const LineState& s0 = sm.P[i];
                    const LineState& s1 = sm.P[i + 1 < NST ? i + 1 : i];
                    auto exponent = [&](const LineState& s) {
                        const long long z = s.z + 2 * __mul64hi(s.dz, k);
                        const unsigned long long z4 = 4ull * (unsigned long long)(z < 0 ? -z : z);
                        return (long long)((__umul64hi(z4, z4) + 1ull) >> 1) + 47765107922663390ll;   // log2(2 pi) / 2
                    };
                    int n0, n1;
                    Triple2 y = exp2_pair(exponent(s0), exponent(s1), sm.kT, sm.kF, n0, n1);
                    const float2 sc = make_float2(n0 < 120 ? __uint_as_float((unsigned)(127 - n0) << 23) : 0.0f,
                                                  n1 < 120 ? __uint_as_float((unsigned)(127 - n1) << 23) : 0.0f);
                    y = triple_mul(y, make_float2(s0.A.h, s1.A.h), make_float2(s0.A.l, s1.A.l),
                                   make_float2(s0.A.r, s1.A.r));
                    const Triple2 c = triple_mul(y, make_float2(s0.C.h, s1.C.h), make_float2(s0.C.l, s1.C.l),
                                                 make_float2(s0.C.r, s1.C.r));
                    const Triple T0 = {y.h.x * sc.x, y.l.x * sc.x, y.r.x * sc.x}, T1 = {y.h.y * sc.y, y.l.y * sc.y, y.r.y * sc.y};
                    const Triple I0 = {c.h.x * sc.x, c.l.x * sc.x, c.r.x * sc.x}, I1 = {c.h.y * sc.y, c.l.y * sc.y, c.r.y * sc.y};
                    if (i == 0) { Tl = Th = T0; Il = Ih = I0; }
                    else {
                        triple_extreme<false>(Tl, T0); triple_extreme<true>(Th, T0);
                        triple_extreme<false>(Il, I0); triple_extreme<true>(Ih, I0);
                    }
                    triple_extreme<false>(Tl, T1); triple_extreme<true>(Th, T1);
                    triple_extreme<false>(Il, I1); triple_extreme<true>(Ih, I1);
                }
                const double u = (lo + j * h) * sU, q = kbl_qweight(ph, j, nu);
                line_moments(acc, u, q * triple_value(Tl), q * triple_value(Th), q * triple_value(Il), q * triple_value(Ih));
            }
        } else {
            if (tid < NST) prim_of<1>(sm.S[tid], ph, sm.G[tid]);
            __syncthreads();
            if (tid == 0) {   // the box of the states as they are
                double a = sm.G[0].U[0] - ph.k * sm.G[0].sq, b = sm.G[0].U[0] + ph.k * sm.G[0].sq;
                for (int i = 1; i < NST; i++) {
                    a = fmin(a, sm.G[i].U[0] - ph.k * sm.G[i].sq);
                    b = fmax(b, sm.G[i].U[0] + ph.k * sm.G[i].sq);
                }
                sm.lo = a;
                sm.h = (b - a) / (nu - 1);
            }
            __syncthreads();
            const LineSums s = bounds1d_f64_nodes<NST>(sm.G, ph, sm.lo, sm.h, tid, NT);
#pragma unroll
            for (int k = 0; k < 8; k++) acc[k] = s.v[k];
        }
        // warp reduce-scatter (lane 4 k holds sum k), then the warps
#pragma unroll
        for (int step = 0; step < 3; step++) {
            const int off = 16 >> step, n = 4 >> step;
            const bool up = lane & off;
#pragma unroll
            for (int k = 0; k < 4; k++) {
                if (k >= n) break;
                const double keep = up ? acc[n + k] : acc[k], send = up ? acc[k] : acc[n + k];
                acc[k] = keep + __shfl_xor_sync(0xffffffffu, send, off);
            }
        }
#pragma unroll
        for (int off = 2; off > 0; off >>= 1) acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], off);
        if ((lane & 3) == 0) sm.red[wid][lane >> 2] = acc[0];
        __syncthreads();
        int redo = 0;
        if (tid < 8) {
            double s = sum_warps<NT / 32>(sm.red, tid);
            if (pairs) {
                if (tid == 0 && !(s >= 0x1p-40)) redo = 1;   // sums of floats that may have underflowed
                s *= pow2_f64(sm.eA) * (tid < 2 ? 1.0 : tid < 6 ? pow2_f64(sm.eU) : pow2_f64(2 * sm.eU));
            }
            // times h and the relaxation of the sum's envelope, rounded once
            const double r = (0xa6 >> tid) & 1 ? ph.rel_hi : ph.rel_lo, p = s * sm.h;
            s = fma(r, p, r * fma(s, sm.h, -p));
            // raw sums: Tlo, Thi, n_hi, n_lo, p_lo, p_hi, E_lo, E_hi; lane 2 + 4 and 3 + 5 make the momentum
            const double t = __shfl_down_sync(0xffu, s, 2);
            if (tid == 0 && s < ph.rho_floor) s = ph.rho_floor;
            if (tid == 2 || tid == 3) s += t;
            if (tid < 4 || tid > 5) bnd[((size_t)(tid & 1) * 3 + (tid < 2 ? 0 : tid < 4 ? 1 : 2)) * E + e] = s;
        }
        if (!__syncthreads_or(redo)) break;
        pairs = false;
    }
}

// The block's dynamic shared memory as one object.
template <typename SM>
__device__ __forceinline__ SM& kbl_dyn_smem()
{
    extern __shared__ __align__(16) unsigned char kbl_smem_bytes[];
    return *reinterpret_cast<SM*>(kbl_smem_bytes);
}

// Launch one block per element with a shared-memory object SM (above 48 KB by opt-in); with pdl, as a
// programmatic dependent (kbl_launch).
template <typename SM, typename... KArgs, typename... Args>
void kbl_launch_dyn(void (*kernel)(KArgs...), int grid, int block, cudaStream_t s, bool pdl, Args... args)
{
    if (sizeof(SM) > 48 * 1024)
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SM));
    kbl_launch(kernel, grid, block, sizeof(SM), s, pdl, args...);
}

}  // namespace kbl_dev

// Whether a grid of nu nodes per axis over k thermal units either side runs on float pairs: where their
// errors are no larger than the FP64 kernel's.  A pair's rounding (2^-49 per table entry) averages out
// over the nodes, so the density of the grid decides; the FP64 kernel's tables drift along their
// recurrence, over 16 nodes on its tiles of 32 and more but over 8 on that of 24.  Error of every bound
// relative to itself, rms over vortex, wave, blast, shock-vortex and node-set stencils, pairs / FP64, in
// units of 1e-16:
//   nodes per thermal unit  3.6 (30 nodes, k = 4) 2.1 / 2.0, 2.9 (48, 8) 2.4 / 2.1, 3.55 (33 Romberg, 4.5)
//                           2.6 / 2.3; at the line 3.75 (31, 4) 2.0 / 2.3, 3.8 (40, 5.2) 2.1 / 2.3; above
//                           it 3.9 (32, 4) 2.0 / 2.5, 4 (33 Romberg, 4) 2.4 / 2.6, 5.9 (48, 4) 1.8 / 2.4
//   24 nodes and fewer      24, k = 3 2.0 / 1.4; 24, 2 1.8 / 1.5; 20, 2.5 2.1 / 1.5; 17 Romberg, 2 2.6 / 1.9;
//                           25 nodes, k = 3 1.9 / 2.0
// Launch at 48 states, 8,192 elements, pairs / FP64: 32 nodes 0.42 / 3.3 ms, 24 nodes 0.42 / 2.6,
// 40 nodes 0.84 / 8.4, 48 nodes 1.4 / 8.1.
inline bool kbl_pair_grid(int nu, double k) { return nu - 1 >= 7.5 * k && nu > 24; }

// Run a statement with NX the smallest tile that holds NU nodes per axis: of the pair kernels, or of
// the FP64 ones.
#define KBL_TILE64_CASE(N_, ...) if (kbl_nu_ <= N_) { constexpr int NX = N_; __VA_ARGS__; }
#define KBL_DISPATCH_PAIR(NU, ...)                 \
    do {                                           \
        const int kbl_nu_ = (NU);                  \
        KBL_TILE64_CASE(32, __VA_ARGS__)           \
        KBL_TILE64_CASE(40, __VA_ARGS__)           \
        KBL_TILE64_CASE(48, __VA_ARGS__)           \
        KBL_TILE64_CASE(64, __VA_ARGS__)           \
    } while (0)
#define KBL_DISPATCH_TILE64(NU, ...)               \
    do {                                           \
        const int kbl_nu_ = (NU);                  \
        KBL_TILE64_CASE(8, __VA_ARGS__)            \
        KBL_TILE64_CASE(16, __VA_ARGS__)           \
        KBL_TILE64_CASE(24, __VA_ARGS__)           \
        KBL_TILE64_CASE(32, __VA_ARGS__)           \
        KBL_TILE64_CASE(48, __VA_ARGS__)           \
        KBL_TILE64_CASE(64, __VA_ARGS__)           \
    } while (0)
