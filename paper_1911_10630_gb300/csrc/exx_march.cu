// exx_march.cu -- the pair pipeline (Sec. III.C Steps III-V) with the
// multigrid-preconditioned FP32 CG of exx_march.cuh inside FP64 refinement.
//
// One persistent CTA per pair, the CTA sized to the ball: NT threads hold one
// column each, 128 registers a thread, so an SM holds 512 threads (a multiple
// of 128 a CTA: tensor memory ties a warp to a quarter of the SM). Per-pair
// radii run as one launch per CTA size, each over its run of the order.
//
// The FP64 phases around the PCG are bound by the FP64 pipe (two lanes a clock
// and SM) and by latency at 16 warps an SM, so they spend few FP64 operations
// and keep several loads in flight: row sums and shell values at z and -z
// together, the shell's 1 / r from a table, the refinement's residuals by an
// exact integer stencil. On the water-like box (256 orbitals at R_PE 24, 10,707
// pairs) they take 126 ms of 341; 196 of 402 as the phases of pair_kernel,
// which took 479 ms in all.
#include <cuda_runtime.h>

#include <algorithm>

#include "exx_march.cuh"
#include "exx_phases.cuh"

namespace exx {

// The PCG's solution is d + al p (d: NULL before the second iteration).
struct MarchSolution {
    const float4* d;
    const float4* p;
    float al;
};

// The PCG on the PE ball: the right-hand side in r (quads), rr its squared
// norm. Returns the iteration count.
template <int NT>
__device__ __forceinline__ int march_pcg(const SolveParams& P, const MarchGeo& M, const MGGeo& MG, float target2,
                                         int max_iter, float (*red)[33], int& flip, MarchSolution& sol) {
    float be = 0.f, al = 0.f, rz = 0.f;
    int it = 0;
    // r.r and the restricted residual of the start, then of every iteration
    for (;;) {
        const float rr = block_sum<NT, float>(pass_r<NT>(P, M, 0, al, it), red, flip);
        if (it > 0 && (!(rr > target2) || it >= max_iter)) break;
        march_coarse<NT>(P, M, MG);
        const float rzn = block_sum<NT, float>(pass_z<NT>(P, M, 0, it), red, flip);
        be = it > 0 ? rzn / rz : 0.f;
        rz = rzn;
        const float pap = block_sum<NT, float>(pass_p<NT>(P, M, be, al, it), red, flip);
        al = rz / pap;
        ++it;
    }
    sol.d = it > 1 ? hot_slot(P) + kMarchD * 2 * march_row(NT) : nullptr;
    sol.p = hot_slot(P) + (kMarchP + (M.lv[0].groups > 1 ? it & 1 : 0)) * 2 * march_row(NT);
    sol.al = al;
    return it;
}

// What a pair's phases share: in shared memory, so that the passes of the PCG
// have the registers to themselves.
struct PairState {
    PairRec pr;
    int pidx, iters, refines;
    int fix;               // the FP64 residuals come from the fixed-point copy of v
    int ovf;               // a value of v did not fit it
    double bb, rn_prev;
    double scale;          // the PCG's right-hand side over the residual: a power of 2 (exact)
    double s2E, finvE;     // fixed-point scale of v, and of its integer stencil's sums
    double vnear;          // largest |v| on the shell layer that the stencil reads
    long long clk[3], tr;
    double M[kNMono], T[kNMono];
    MarchSolution sol;
};

__device__ __forceinline__ double* slot_f64(const SolveParams& P, size_t off) {
    return reinterpret_cast<double*>(P.ws + (size_t)blockIdx.x * P.slot_bytes + off);
}

// Largest of the CTA's values, in every thread.
template <int NT>
__device__ __forceinline__ double block_max(double v, double (*red)[33], int& flip) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    double* buf = red[flip];
    flip ^= 1;
    if ((threadIdx.x & 31) == 0) buf[threadIdx.x >> 5] = v;
    __syncthreads();
    double m = buf[0];
#pragma unroll
    for (int w = 1; w < NT / 32; ++w) m = fmax(m, buf[w]);
    return m;
}

// Steps 1 to 3 of the pipeline (exx_solve.cu): gather, moments, shell values;
// then the PCG's shared memory.
template <int NT>
static __device__ __noinline__ void march_setup(const SolveParams& P, PairState& S, unsigned ring, double (*red)[33],
                                                int& flip) {
    const BallGeo& G = P.geos[S.pr.geo];
    const MarchGeo& M = P.march[S.pr.geo];
    const double* xp = P.pow_tab;  // power tables of the offsets (global, cached)
    const int t = threadIdx.x;
    double *rho = slot_f64(P, P.off_rho), *vc = slot_f64(P, P.off_vcube), *rowS = slot_f64(P, P.off_rows);
    double *V = slot_f64(P, P.off_sy), *U64 = slot_f64(P, P.off_ush);
    float* U32 = reinterpret_cast<float*>(U64 + (size_t)kNU * G.n_rows_me);
    const double rm = block_max<NT>(P.box_org ? gather_wide<true>(P, G, S.pr, rho, vc, t, NT)
                                              : gather_wide<false>(P, G, S.pr, rho, vc, t, NT), red, flip);
    moment_rows_folded(P, G, rho, rowS, t, NT);
    __syncthreads();
    // shared memory: plane sums [(2 R_PE + 1) 28]
    moment_finish<NT>(P, G, rowS, xp, xp + (2 * P.Rc + 1) * 8, reinterpret_cast<double*>(march_sm), S.M, S.T);
    shell_planes(P, G, S.T, V, t, NT);
    __syncthreads();
    shell_coeffs(P, G, V, U64, U32, t, NT);
    __syncthreads();
    const double vn = block_max<NT>(shell_values(P, G, U64, U32, vc, t, NT), red, flip);
    if (threadIdx.x == 0) {
        // any power of 2 near the residual's size does: FP32 has the range
        int e = 0;
        (void)frexp(rm, &e);
        S.scale = rm > 0.0 && rm < 1e300 ? ldexp(1.0, e < -900 ? 900 : -e) : 1.0;
        S.vnear = vn;
        S.fix = P.fixres;
        S.ovf = 0;
    }
    march_init<NT>(P, M, ring);
    if (P.n_geo > 1) {  // another ball's residual: zero off this one
        float4* rq = hot_slot(P) + kMarchR * 2 * march_row(NT);
        for (int k = threadIdx.x; k < M.lv[0].nq; k += NT) rq[k] = rq[march_row(NT) + k] = f4zero();
    }
    __syncthreads();
}

// FP64 residual r = 4 pi rho + lap v (v: current iterate on PE, shell values
// outside) into the PCG's right-hand side (times scale, FP32 quads); this
// thread's share of ||r||^2, and of the right-hand side's square.
// The first one, with v = 0 on the PE ball: the rim points (whose stencils
// reach the shell) take the stencil, the others r = 4 pi rho, each in dense
// warps.
template <int NT>
static __device__ __noinline__ double march_residual0(const SolveParams& P, const PairState& S, float& rr) {
    const MarchGeo& M = P.march[S.pr.geo];
    const BallGeo& G = P.geos[S.pr.geo];
    const int* __restrict__ cube = G.pt_cube;
    const int* __restrict__ list = G.rim;
    const int* __restrict__ qidx = M.qidx;
    const double* __restrict__ vc = slot_f64(P, P.off_vcube);
    const double* __restrict__ rho = slot_f64(P, P.off_rho);
    float* __restrict__ rq = reinterpret_cast<float*>(hot_slot(P) + kMarchR * 2 * march_row(NT));
    const Stencil<double> st = P.st64;
    const int side = P.S, n = G.n_pe, nrim = G.n_rim;
    const long long S2 = P.S2;
    const double scale = S.scale;
    double acc = 0.0;
    float a32 = 0.f;
    for (int t = threadIdx.x; t < n; t += NT) {
        const int k = __ldg(list + t);
        double r = kFourPi * rho[k];
        if (t < nrim) r += lap19<double>(vc, __ldg(cube + k), side, S2, st);
        if (P.dbg_b) P.dbg_b[k] = r;
        const float f = (float)(r * scale);
        rq[__ldg(qidx + k)] = f;
        acc = fma(r, r, acc);
        a32 = fmaf(f, f, a32);
    }
    rr = a32;
    return acc;
}

// 180 delta^2 lap v on a fixed-point copy of v: an exact integer sum.
__device__ __forceinline__ long long lap_int(const long long* __restrict__ f, int c, int S, int S2) {
    long long s1 = 0, s2 = 0, s3 = 0;
    const long long m = f[c];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const int st = a == 0 ? S2 : (a == 1 ? S : 1);
        s1 += f[c + st] + f[c - st];
        s2 += f[c + 2 * st] + f[c - 2 * st];
        s3 += f[c + 3 * st] + f[c - 3 * st];
    }
    return 270 * s1 - 27 * s2 + 2 * s3 - 1470 * m;
}

// FIX: lap v from the fixed-point copy (isotropic grids): the weights of Eq.
// d2_1 times 180 delta^2 are the integers -490, 270, -27 and 2, so the sum is
// exact, and three FP64 operations a point remain of 21. The copy rounds v at
// 2^-51 to 2^-50 of its largest value, which bounds the residual at 1e-14 (R_PE 16) to
// 1e-13 (R_PE 32) of the right-hand side; the FP64 stencil reaches 1e-14 throughout. A
// pair whose residual does not halve goes on with the FP64 stencil.
template <int NT, bool FIX>
static __device__ __noinline__ double march_residual(const SolveParams& P, const PairState& S, float& rr) {
    const BallGeo& G = P.geos[S.pr.geo];
    const int* __restrict__ cube = G.pt_cube;
    const int* __restrict__ qidx = P.march[S.pr.geo].qidx;
    const double* __restrict__ vc = slot_f64(P, P.off_vcube);
    const long long* __restrict__ vf = reinterpret_cast<const long long*>(slot_f64(P, P.off_vfix));
    const double* __restrict__ rho = slot_f64(P, P.off_rho);
    float* __restrict__ rq = reinterpret_cast<float*>(hot_slot(P) + kMarchR * 2 * march_row(NT));
    const int n = G.n_pe, side = P.S;
    const long long S2 = P.S2;
    const Stencil<double> st = P.st64;
    const double scale = S.scale, finv = S.finvE;
    double acc = 0.0;
    float a32 = 0.f;
#pragma unroll 2
    for (int k = threadIdx.x; k < n; k += NT) {
        const int c = __ldg(cube + k);
        double lap;
        if constexpr (FIX) lap = (double)lap_int(vf, c, side, (int)S2) * finv;
        else lap = lap19<double>(vc, c, side, S2, st);
        const double r = fma(kFourPi, rho[k], lap);
        const float f = (float)(r * scale);
        rq[__ldg(qidx + k)] = f;
        acc = fma(r, r, acc);
        a32 = fmaf(f, f, a32);
    }
    rr = a32;
    return acc;
}

__device__ __forceinline__ long long march_fix(double v, double s2E, int& ovf) {
    const double x = v * s2E;
    if (!(fabs(x) <= 2251799813685248.0)) {  // 2^51: a stencil sum stays below 2^63
        ovf = 1;
        return 0;
    }
    return __double2ll_rn(x);
}

// v += (d + al p) / scale, with the fixed-point copy (fix2: its scale stands);
// this thread's largest |v|.
template <int NT>
static __device__ __noinline__ double march_update(const SolveParams& P, PairState& S, bool fix2) {
    const BallGeo& G = P.geos[S.pr.geo];
    const int* __restrict__ cube = G.pt_cube;
    const int* __restrict__ qidx = P.march[S.pr.geo].qidx;
    double* __restrict__ vc = slot_f64(P, P.off_vcube);
    long long* __restrict__ vf = reinterpret_cast<long long*>(slot_f64(P, P.off_vfix));
    const float* __restrict__ dq = reinterpret_cast<const float*>(S.sol.d);
    const float* __restrict__ pq = reinterpret_cast<const float*>(S.sol.p);
    const float al = S.sol.al;
    const double f = 1.0 / S.scale, s2E = S.s2E;
    double big = 0.0;
    int ovf = 0;
#pragma unroll 4
    for (int k = threadIdx.x; k < G.n_pe; k += NT) {
        const int q = __ldg(qidx + k), c = __ldg(cube + k);
        const float dk = fmaf(al, __ldcg(pq + q), dq ? __ldcg(dq + q) : 0.f);
        const double v = fma(f, (double)dk, vc[c]);
        vc[c] = v;
        if (fix2) vf[c] = march_fix(v, s2E, ovf);
        big = fmax(big, fabs(v));
    }
    if (ovf) S.ovf = 1;
    return big;
}

// The fixed-point copy of v on the PE ball and the layer around it.
template <int NT>
static __device__ __noinline__ void march_copy_fix(const SolveParams& P, PairState& S) {
    const BallGeo& G = P.geos[S.pr.geo];
    const double* __restrict__ vc = slot_f64(P, P.off_vcube);
    long long* __restrict__ vf = reinterpret_cast<long long*>(slot_f64(P, P.off_vfix));
    const double s2E = S.s2E;
    int ovf = 0;
#pragma unroll 4
    for (int k = threadIdx.x; k < G.n_pe; k += NT) {
        const int c = __ldg(G.pt_cube + k);
        vf[c] = march_fix(vc[c], s2E, ovf);
    }
    for (int q = threadIdx.x; q < G.n_layer; q += NT) {
        const int pk = __ldg(G.layer + q), z = pk & 255;
        const RowRec R = G.rows_me[pk >> 8];
        const long long c = (long long)(R.ox + P.Rc) * P.S2 + (long long)(R.oy + P.Rc) * P.S + P.Rc;
        vf[c + z] = march_fix(vc[c + z], s2E, ovf);
        vf[c - z] = march_fix(vc[c - z], s2E, ovf);
    }
    if (ovf) S.ovf = 1;
}

// E_ij over the PE ball (this thread's share).
template <int NT>
static __device__ __noinline__ double march_energy(const SolveParams& P, const PairState& S) {
    const BallGeo& G = P.geos[S.pr.geo];
    const int* __restrict__ cube = G.pt_cube;
    const double* __restrict__ vc = slot_f64(P, P.off_vcube);
    const double* __restrict__ rho = slot_f64(P, P.off_rho);
    double e = 0.0;
#pragma unroll 4
    for (int k = threadIdx.x; k < G.n_pe; k += NT) e = fma(rho[k], vc[__ldg(cube + k)], e);
    return e;
}

template <int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB) march_kernel(const __grid_constant__ SolveParams P) {
    __shared__ double red[2][33];
    __shared__ float red32[2][33];
    __shared__ PairState S;
    __shared__ int s_item;
    __shared__ unsigned s_ring;
    int flip = 0, flip32 = 0;
    ring_alloc<NT>(&s_ring);

    for (;;) {
        if (threadIdx.x == 0) s_item = atomicAdd(P.queue, 1);
        __syncthreads();
        if (s_item >= *P.n_pair) break;
        if (threadIdx.x == 0) {
            S.pidx = P.order ? P.order[(P.item_base ? *P.item_base : 0) + s_item] : s_item;
            S.pr = P.pairs[S.pidx];
            S.iters = S.refines = 0;
            S.bb = -1.0;
            S.rn_prev = 1e300;
            S.tr = 0;
            S.clk[0] = clock64();
        }
        __syncthreads();
        march_setup<NT>(P, S, s_ring, red, flip);
        if (threadIdx.x == 0) S.clk[1] = clock64();

        bool conv = true;
        for (;;) {
            const long long tu = clock64();
            float r32 = 0.f;
            double part;
            if (S.refines == 0) part = march_residual0<NT>(P, S, r32);
            else if (S.fix) part = march_residual<NT, true>(P, S, r32);
            else part = march_residual<NT, false>(P, S, r32);
            const double rn2 = block_sum<NT, double>(part, red, flip);
            const float rr32 = block_sum<NT, float>(r32, red32, flip32);
            if (threadIdx.x == 0) {
                S.tr += clock64() - tu;
                if (S.bb < 0.0) S.bb = rn2;
            }
            __syncthreads();
            if (rn2 <= P.tol * P.tol * S.bb) break;
            const double rn = sqrt(rn2);
            if (S.fix && S.refines > 0 && !(rn < 0.5 * S.rn_prev)) {
                // the copy's rounding may bound this residual: the FP64 stencil from here on
                __syncthreads();
                if (threadIdx.x == 0) {
                    S.fix = 0;
                    S.rn_prev = 1e300;
                }
                __syncthreads();
                continue;
            }
            if (S.refines >= P.max_refine || S.iters >= P.max_iter || !(rn < S.rn_prev)) {
                conv = false;
                break;
            }
            double eta = 0.3 * P.tol * sqrt(S.bb) / rn;
            eta = eta > P.inner_tol ? eta : P.inner_tol;
            const int budget = min(P.inner_max_iter, P.max_iter - S.iters);
            MarchSolution sol;
            const int it = march_pcg<NT>(P, P.march[S.pr.geo], P.mg[S.pr.geo], (float)(eta * eta) * rr32, budget, red32,
                                         flip32, sol);
            __syncthreads();
            if (threadIdx.x == 0) {
                S.iters += it;
                ++S.refines;
                S.rn_prev = rn;
                S.sol = sol;
            }
            __syncthreads();
            const bool fix2 = S.fix && S.refines > 1;
            const double vm = march_update<NT>(P, S, fix2);
            if (S.fix && !fix2) {  // the first iterate: its largest value sets the fixed-point scale
                const double big = fmax(block_max<NT>(vm, red, flip), S.vnear);
                if (threadIdx.x == 0) {
                    int e = 0;
                    (void)frexp(1.03125 * big, &e);
                    if (P.fixres == 2) e -= 60;  // test mode: the copy overflows, the pair falls back
                    if (!(big < 1e300)) S.fix = 0;
                    S.s2E = ldexp(1.0, 51 - e);
                    S.finvE = ldexp(P.fix_inv, e - 51);
                }
                __syncthreads();
                if (S.fix) march_copy_fix<NT>(P, S);
            }
            __syncthreads();
            if (threadIdx.x == 0) {
                if (S.ovf) S.fix = S.ovf = 0;  // beyond the copy's range: the FP64 stencil from here on
                // The next residual's norm lies between eta times this one's and, where the
                // inner solve stopped short, this one's: with eta at 2^-24 or more (what FP32
                // can gain) its squares stay within FP32's range. From the residual itself,
                // not from the last scale: solves that keep stopping short do not add up.
                int e = 0;
                (void)frexp(rn * fmax(eta, 5.9604644775390625e-8), &e);
                S.scale = ldexp(1.0, -min(max(e, -900), 900));
            }
            __syncthreads();
        }
        if (threadIdx.x == 0) S.clk[2] = clock64();
        const double e = block_sum<NT, double>(march_energy<NT>(P, S), red, flip);
        if (threadIdx.x == 0) {
            P.e_pair[S.pidx] = e * P.dV;
            P.iters[S.pidx] = S.iters;
            if (P.refines) P.refines[S.pidx] = S.refines;
            if (!conv) atomicAdd(P.nonconv, 1);
        }
        scatter_wide(P, P.geos[S.pr.geo], S.pr, slot_f64(P, P.off_vcube), threadIdx.x, NT);
        if (!conv) {  // an infinite or NaN al leaves NaN in the residual's quads off the ball, where zeros belong
            float4* rq = hot_slot(P) + kMarchR * 2 * march_row(NT);
            for (int k = threadIdx.x; k < (kMarchP - kMarchR) * 2 * march_row(NT); k += NT) rq[k] = f4zero();
        }
        __syncthreads();
        if (P.phase_clk && threadIdx.x == 0) {
            const long long t3 = clock64();
            atomicAdd(P.phase_clk + 0, (unsigned long long)(S.clk[1] - S.clk[0]));
            atomicAdd(P.phase_clk + 1, (unsigned long long)S.tr);
            atomicAdd(P.phase_clk + 2, (unsigned long long)(S.clk[2] - S.clk[1] - S.tr));
            atomicAdd(P.phase_clk + 3, (unsigned long long)(t3 - S.clk[2]));
        }
    }
    __syncthreads();
    ring_free<NT>(s_ring);
}

// ---- host side ----
cudaError_t set_multipole_const_march(const MultipoleConst& mc) {
    return cudaMemcpyToSymbol(c_mp, &mc, sizeof(MultipoleConst));
}

static const void* march_fn(int threads) {
    switch (threads) {
        case 128: return (const void*)march_kernel<128, 4>;
        case 256: return (const void*)march_kernel<256, 2>;
        default: return (const void*)march_kernel<512, 1>;
    }
}

// Resident CTAs per SM. The runtime's occupancy query answers 1 for a kernel
// that allocates tensor memory, whatever it allocates, so this counts registers,
// shared memory, tensor memory and threads.
cudaError_t march_occupancy(int threads, size_t smem, int* blocks_per_sm) {
    const void* f = march_fn(threads);
    cudaError_t e = raise_smem_limit(f, smem);
    if (e != cudaSuccess) return e;
    cudaFuncAttributes at;
    if ((e = cudaFuncGetAttributes(&at, f)) != cudaSuccess) return e;
    int dev = 0, regs = 0, bytes = 0, most = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
        (e = cudaDeviceGetAttribute(&regs, cudaDevAttrMaxRegistersPerMultiprocessor, dev)) != cudaSuccess ||
        (e = cudaDeviceGetAttribute(&bytes, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev)) != cudaSuccess ||
        (e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxThreadsPerMultiProcessor, dev)) != cudaSuccess)
        return e;
    const int warp_regs = (at.numRegs * 32 + 255) & ~255;
    const int tm = threads == 128 ? ring_columns<128>() : threads == 256 ? ring_columns<256>() : ring_columns<512>();
    const int cta = (int)((smem + at.sharedSizeBytes + 1024 + 127) & ~(size_t)127);
    *blocks_per_sm = std::min(std::min(regs / (warp_regs * (threads / 32)), bytes / cta), std::min(most / threads, 512 / tm));
    return cudaSuccess;
}

cudaError_t launch_march_kernel(const SolveParams& P, int threads, int grid, size_t smem, cudaStream_t st) {
    void* args[1] = {(void*)&P};
    return cudaLaunchKernel(march_fn(threads), dim3(grid), dim3(threads), args, smem, st);
}

}  // namespace exx
