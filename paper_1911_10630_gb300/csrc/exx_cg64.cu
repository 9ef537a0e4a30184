// exx_cg64.cu -- the pair pipeline (Sec. III.C Steps III-V) with the plain FP64
// CG, a team of 1 to 8 CTAs (a thread-block cluster) per pair.
//
// The steps are those of exx_solve.cu's pair_kernel and the iteration is its
// cg_ball. GB300 issues FP64 at two lanes a clock and SM, which bounds cg_ball:
// 24 operations per point and iteration, 19 of them the stencil. On isotropic
// grids A p is formed in integers instead: the weights of Eq. d2_1 times
// 180 delta^2 are -490, 270, -27 and 2, and p is kept a second time as a 60-bit
// fixed-point number under a bound B that the CG's own reductions give each
// iteration (a power of 2, up to 4 times the largest |p|). The sum is exact but for
// its last 8 of 71 bits, and one conversion turns it back: 7 FP64 operations a point
// in all. The copy is truncated at 2^-59 B, so A p is off by (3264 + 256) 2^-59 B over
// 180 delta^2 at most, 2^-47 B: values below 2^-6 B have fewer bits in it than in FP64.
// Over the directions of CGs on balls of R_PE 8, 16 and 24 the error of A p (2-norm)
// is 4e-17 to 5e-16 of it; the FP64 stencil's, whose rounded weights do not sum to
// zero, 2e-16 to 6e-15.
//
// Two points along z share their loads (17 of 16 bytes instead of 38 of 8). What
// is left is bound by latency and DRAM: 100 bytes a point and iteration, two
// thirds of the copy rate, and A p's loads. Several CTAs on a pair keep all SMs
// busy on few pairs.
//
// Milliseconds, 64 orbitals at R_PE 24 (755 pairs, 158 iterations) / 8 orbitals
// at R_PE 16 (36 pairs, 134): cg_ball 358 / 20.1; integers one point at a time,
// 10 FP64 operations 186 / 4.2 (teams of 2 / 4); 7 operations 176 / 3.9; in
// pairs 165 / 3.4; the sums' additions on one warp 155 / 3.2. Of 165, A p took 81, the
// residual 33, the direction 37 and the team's barriers 17.
#include <cuda_runtime.h>

#include "exx_phases.cuh"

namespace exx {

constexpr int kTeam = 8;  // most CTAs of a team

__device__ __forceinline__ int team_size() {
    int r;
    asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ int team_rank() {
    int r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// Barrier of the team's threads; global writes before it are seen after it.
__device__ __forceinline__ void team_sync(int C) {
    if (C == 1) {
        __syncthreads();
    } else {
        asm volatile("barrier.cluster.arrive.release;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    }
}
__device__ __forceinline__ unsigned team_address(const void* p, int rank) {
    unsigned a = (unsigned)__cvta_generic_to_shared(p), r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}

struct TeamShared {
    double red[2][kTeam * 32];
    unsigned top[2][kTeam * 32];
    double M[kNMono], T[kNMono];
    double sum;
    unsigned max;
    int item;
};

// What the CG's passes read, per thread. Vectors hold pairs of points.
struct TeamSlot {
    const int* duo;
    double2 *r, *x, *q, *p;
    longlong2* f;  // fixed-point p, zero off the ball (FIX), or p itself
    int j0, j1;    // the CTA's pairs
    int S;
};

// Sum of v and maximum of top over the team, in every thread; a team barrier.
// Fixed order: the same value in every thread and run. An FP64 addition takes a warp
// 16 clocks of the SM's pipe, so warps without a share add nothing and one warp adds
// the partial sums: with all 16 warps at both, the two sums took a quarter of a small
// ball's iteration (CG of 10 pairs at R_PE 4, anisotropic: 0.344 ms, now 0.274).
template <int NT>
__device__ __forceinline__ double team_sum(double v, unsigned& top, TeamShared& T, int C, int& flip) {
    constexpr int W = NT / 32;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (__any_sync(0xffffffffu, v != 0.0)) v = warp_sum(v);
    top = __reduce_max_sync(0xffffffffu, top);
    double* red = T.red[flip];
    unsigned* tp = T.top[flip];
    flip ^= 1;
    if (lane < C) {
        const int at = team_rank() * W + w;
        asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(team_address(red + at, lane)), "d"(v) : "memory");
        asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(team_address(tp + at, lane)), "r"(top) : "memory");
    }
    team_sync(C);
    if (w == 0) {
        double s = 0.0;
        unsigned m = 0u;
        for (int i = lane; i < C * W; i += 32) {
            s += red[i];
            m = max(m, tp[i]);
        }
        m = __reduce_max_sync(0xffffffffu, m);
        s = warp_sum(s);
        if (lane == 0) {  // read by all before the next sum's barrier
            T.sum = s;
            T.max = m;
        }
    }
    __syncthreads();
    top = T.max;
    return T.sum;
}

// High word of |v|: ordered as |v| is. bound_of gives the least value above
// every |v| with that high word (infinite or NaN stay so).
__device__ __forceinline__ unsigned high_of(double v) { return (unsigned)__double2hiint(v) & 0x7fffffffu; }
__device__ __forceinline__ double bound_of(unsigned top) {
    return top < 0x7ff00000u ? __hiloint2double((int)(top + 1u), 0) : __hiloint2double((int)top, 0);
}

// The fixed-point copy of v: v 2^k truncated, |v 2^k| <= 2^59 (k of either sign).
// The scale is added to v's exponent (a zero or denormal v stays below 1/2; an
// infinite or NaN v becomes 0: its pair ends on the sums of r and p).
__device__ __forceinline__ long long to_fixed(double v, int k) {
    const int h = __double2hiint(v);
    const int e = (h >> 20) & 0x7ff;
    const unsigned long long m = ((unsigned long long)(unsigned)((h & 0xfffff) | 0x100000) << 32 | (unsigned)__double2loint(v)) << 7;
    const long long t = (long long)(m >> min((unsigned)(1082 - k - e), 63u));
    return h < 0 ? -t : t;
}

// -180 delta^2 / 2^8 times lap p from the fixed-point copy, in units of the
// copy: m the value, s1 to s3 the sums of its neighbours at distance 1 to 3
// (they fit 64 bits). The weighted sum (71 bits) is formed in two limbs and
// loses its last 8 bits.
__device__ __forceinline__ double weigh_fixed(long long m, long long s1, long long s2, long long s3) {
    const auto lo = [](long long v) { return (long long)(unsigned)v; };
    const auto hi = [](long long v) { return (long long)(int)(v >> 32); };
    const long long h = hi(m) * 1470 - hi(s1) * 270 + hi(s2) * 27 - hi(s3) * 2;
    const long long l = lo(m) * 1470 - lo(s1) * 270 + lo(s2) * 27 - lo(s3) * 2;
    return (double)((h << 24) + (l >> 8));
}

// q = A p on the CTA's pairs (FIX: over its unit); this thread's share of p.q.
// Both points of a pair share the 16-byte loads: 17 instead of 38 of 8 bytes.
template <int NT, bool FIX>
static __device__ __noinline__ double team_apply(const TeamSlot& s, const Stencil<double>& neg) {
    const int j1 = s.j1, Sy = (s.S + 1) / 2, Sx = s.S * Sy;  // pairs per row and plane
    const int* __restrict__ duo = s.duo;
    const longlong2* f = s.f;
    const double2* p = s.p;
    double2* q = s.q;
    double acc = 0.0;
#pragma unroll 1
    for (int j = s.j0 + (int)threadIdx.x; j < j1; j += NT) {
        const int pk = __ldg(duo + j);
        const double2 pj = __ldcg(p + j);
        double a0, a1;
        if constexpr (FIX) {
            const longlong2* c = f + (pk >> 3);
            const longlong2 m = c[0], z0 = c[-2], z1 = c[-1], z2 = c[1], z3 = c[2];
            long long u1 = z1.y + m.y, u2 = z1.x + z2.x, u3 = z0.y + z2.y;
            long long w1 = m.x + z2.x, w2 = z1.y + z2.y, w3 = z1.x + z3.x;
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                const longlong2* d = c + (a & 1 ? -1 : 1) * (a < 2 ? Sy : Sx);
                const int st = (a & 1 ? -1 : 1) * (a < 2 ? Sy : Sx);
                const longlong2 d1 = d[0], d2 = d[st], d3 = d[2 * st];
                u1 += d1.x;
                w1 += d1.y;
                u2 += d2.x;
                w2 += d2.y;
                u3 += d3.x;
                w3 += d3.y;
            }
            a0 = weigh_fixed(m.x, u1, u2, u3);
            a1 = weigh_fixed(m.y, w1, w2, w3);
        } else {
            const double2* c = reinterpret_cast<const double2*>(f) + (pk >> 3);
            const double2 m = c[0], z0 = c[-2], z1 = c[-1], z2 = c[1], z3 = c[2];
            a0 = fma(neg.cz[0], z1.y + m.y, neg.c0 * m.x);
            a0 = fma(neg.cz[1], z1.x + z2.x, a0);
            a0 = fma(neg.cz[2], z0.y + z2.y, a0);
            a1 = fma(neg.cz[0], m.x + z2.x, neg.c0 * m.y);
            a1 = fma(neg.cz[1], z1.y + z2.y, a1);
            a1 = fma(neg.cz[2], z1.x + z3.x, a1);
#pragma unroll
            for (int n = 1; n <= 3; ++n) {
                const double2 y0 = c[-n * Sy], y1 = c[n * Sy], x0 = c[-n * Sx], x1 = c[n * Sx];
                a0 = fma(neg.cy[n - 1], y0.x + y1.x, a0);
                a1 = fma(neg.cy[n - 1], y0.y + y1.y, a1);
                a0 = fma(neg.cx[n - 1], x0.x + x1.x, a0);
                a1 = fma(neg.cx[n - 1], x0.y + x1.y, a1);
            }
        }
        if (!(pk & 1)) a0 = 0.0;
        if (!(pk & 2)) a1 = 0.0;
        q[j] = make_double2(a0, a1);
        acc = fma(pj.x, a0, acc);
        acc = fma(pj.y, a1, acc);
    }
    return acc;
}

// r -= al q; this thread's share of r.r, and its largest |r|.
template <int NT>
static __device__ __noinline__ double team_residual(const TeamSlot& s, double al, unsigned& top) {
    const int j1 = s.j1;
    double2* r = s.r;
    const double2* q = s.q;
    double acc = 0.0;
    unsigned t = 0u;
#pragma unroll 4
    for (int j = s.j0 + (int)threadIdx.x; j < j1; j += NT) {
        const double2 a = __ldcg(q + j);
        double2 v = __ldcg(r + j);
        v.x = fma(-al, a.x, v.x);
        v.y = fma(-al, a.y, v.y);
        r[j] = v;
        acc = fma(v.x, v.x, acc);
        acc = fma(v.y, v.y, acc);
        t = max(t, max(high_of(v.x), high_of(v.y)));
    }
    top = t;
    return acc;
}

// x += al p, p = r + be p and its copy, scaled by 2^sh (FIRST: p = r, x = 0);
// this thread's largest |p|.
template <int NT, bool FIX, bool FIRST>
static __device__ __noinline__ unsigned team_direction(const TeamSlot& s, double al, double be, int sh) {
    const int j1 = s.j1;
    const int* __restrict__ duo = s.duo;
    const double2* r = s.r;
    double2 *x = s.x, *p = s.p;
    longlong2* f = s.f;
    unsigned t = 0u;
#pragma unroll 2
    for (int j = s.j0 + (int)threadIdx.x; j < j1; j += NT) {
        const int c = __ldg(duo + j) >> 3;
        double2 v = __ldcg(r + j);
        if constexpr (FIRST) {
            x[j] = make_double2(0.0, 0.0);
        } else {
            const double2 o = __ldcg(p + j);
            double2 w = __ldcg(x + j);
            w.x = fma(al, o.x, w.x);
            w.y = fma(al, o.y, w.y);
            x[j] = w;
            v.x = fma(be, o.x, v.x);
            v.y = fma(be, o.y, v.y);
        }
        p[j] = v;
        if constexpr (FIX) f[c] = make_longlong2(to_fixed(v.x, sh), to_fixed(v.y, sh));
        else reinterpret_cast<double2*>(f)[c] = v;
        t = max(t, max(high_of(v.x), high_of(v.y)));
    }
    return t;
}

template <int NT, bool FIX>
__global__ void __launch_bounds__(NT, 1024 / NT) cg64_kernel(const __grid_constant__ SolveParams P) {
    extern __shared__ double team_dyn[];  // plane sums [(2 R_PE + 1) 28]
    __shared__ TeamShared T;
    const int C = team_size(), rank = team_rank(), tid = threadIdx.x;
    const int gt = rank * NT + tid, gn = C * NT;
    int flip = 0;
    char* slot = P.ws + (size_t)(blockIdx.x / C) * P.slot_bytes;
    TeamSlot s;
    double* vc = reinterpret_cast<double*>(slot + P.off_vcube);
    double* rho = reinterpret_cast<double*>(slot + P.off_rho);
    s.f = reinterpret_cast<longlong2*>(slot + P.off_pcube);
    s.r = reinterpret_cast<double2*>(slot + P.off_r);
    s.x = reinterpret_cast<double2*>(slot + P.off_d);
    s.q = reinterpret_cast<double2*>(slot + P.off_ap);
    s.p = reinterpret_cast<double2*>(slot + P.off_vfix);
    s.S = P.S;
    double* rowS = reinterpret_cast<double*>(slot + P.off_rows);
    double* V = reinterpret_cast<double*>(slot + P.off_sy);
    double* U64 = reinterpret_cast<double*>(slot + P.off_ush);
    const Stencil<double> neg = negated(P.st64);
    const double* xp = P.pow_tab;
    const int np = *P.n_pair;
    const bool lead = rank == 0 && tid == 0;

    team_sync(C);  // every CTA of the team has started: its shared memory may be written
    for (;;) {
        if (lead) {
            const int i = atomicAdd(P.queue, 1);
            for (int j = 0; j < C; ++j)
                asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(team_address(&T.item, j)), "r"(i) : "memory");
        }
        team_sync(C);
        const int item = T.item;
        if (item >= np) break;
        const int pidx = P.order ? P.order[(P.item_base ? *P.item_base : 0) + item] : item;
        const PairRec pr = P.pairs[pidx];
        const BallGeo& G = P.geos[pr.geo];
        s.duo = G.duo;
        s.j0 = (int)((long long)G.n_duo * rank / C);
        s.j1 = (int)((long long)G.n_duo * (rank + 1) / C);
        const bool clk = P.phase_clk && lead;
        const long long t0 = clk ? clock64() : 0;
        float* U32 = reinterpret_cast<float*>(U64 + (size_t)kNU * G.n_rows_me);

        // gather, moments, shell values
        (void)(P.box_org ? gather_wide<true>(P, G, pr, rho, vc, gt, gn) : gather_wide<false>(P, G, pr, rho, vc, gt, gn));
        team_sync(C);
        moment_rows_folded(P, G, rho, rowS, gt, gn);
        team_sync(C);
        moment_finish<NT>(P, G, rowS, xp, xp + (2 * P.Rc + 1) * 8, team_dyn, T.M, T.T);
        shell_planes(P, G, T.T, V, gt, gn);
        team_sync(C);
        shell_coeffs(P, G, V, U64, U32, gt, gn);
        team_sync(C);
        (void)shell_values(P, G, U64, U32, vc, gt, gn);
        team_sync(C);
        const long long t1 = clk ? clock64() : 0;

        // right-hand side
        double acc = 0.0;
        unsigned top = 0u;
#pragma unroll 1
        for (int j = s.j0 + tid; j < s.j1; j += NT) {
            const int2 kk = __ldg(G.duo_k + j);
            double b[2] = {0.0, 0.0};
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int k = u ? kk.y : kk.x;
                if (k < 0) continue;
                b[u] = fma(kFourPi, rho[k], lap19<double>(vc, __ldg(G.pt_cube + k), P.S, P.S2, P.st64));
                if (P.dbg_b) P.dbg_b[k] = b[u];
                acc = fma(b[u], b[u], acc);
                top = max(top, high_of(b[u]));
            }
            s.r[j] = make_double2(b[0], b[1]);
        }
        double rr = team_sum<NT>(acc, top, T, C, flip);
        const double target2 = P.tol * P.tol * rr;
        const long long t2 = clk ? clock64() : 0;

        // CG
        double al = 0.0, unit = 1.0;
        int sh = 0;
        const auto scale_for = [&](double bound) {  // |p| <= bound: |p 2^sh| <= 2^59
            int e = 0;
            (void)frexp(bound, &e);
            sh = 59 - min(max(e, -900), 900);
            unit = ldexp(P.fix_inv, 8 - sh);
        };
        int it = 0;
        bool open = false;  // x lacks al p
        if (FIX) scale_for(bound_of(top));
        unsigned ptop = team_direction<NT, FIX, true>(s, 0.0, 0.0, sh);
        team_sync(C);
        while (rr > target2 && it < P.max_iter) {
            const double pap = unit * team_sum<NT>(team_apply<NT, FIX>(s, neg), ptop, T, C, flip);
            al = rr / pap;
            const double rrn = team_sum<NT>(team_residual<NT>(s, al * unit, top), top, T, C, flip);
            ++it;
            if (rrn <= target2 || !(rrn == rrn)) {
                rr = rrn;
                open = true;
                break;
            }
            const double be = rrn / rr;
            rr = rrn;
            if (FIX) scale_for(bound_of(top) + be * bound_of(ptop));
            ptop = team_direction<NT, FIX, false>(s, al, be, sh);
            team_sync(C);
        }
        double e = 0.0;
        for (int j = s.j0 + tid; j < s.j1; j += NT) {
            const int2 kk = __ldg(G.duo_k + j);
            double2 v = s.x[j];
            if (open) {
                const double2 p = s.p[j];
                v.x = fma(al, p.x, v.x);
                v.y = fma(al, p.y, v.y);
            }
            if (kk.x >= 0) {
                vc[__ldg(G.pt_cube + kk.x)] = v.x;
                e = fma(rho[kk.x], v.x, e);
            }
            if (kk.y >= 0) {
                vc[__ldg(G.pt_cube + kk.y)] = v.y;
                e = fma(rho[kk.y], v.y, e);
            }
        }
        e = team_sum<NT>(e, top, T, C, flip);
        const long long t3 = clk ? clock64() : 0;
        if (lead) {
            P.e_pair[pidx] = e * P.dV;
            P.iters[pidx] = it;
            if (P.refines) P.refines[pidx] = 1;
            if (!(rr <= target2)) atomicAdd(P.nonconv, 1);
        }
        scatter_wide(P, G, pr, vc, gt, gn);
        if (P.n_geo > 1)  // the next pair may have another ball: the copy is zero off it
            for (int j = s.j0 + tid; j < s.j1; j += NT) s.f[__ldg(s.duo + j) >> 3] = make_longlong2(0, 0);
        if (clk) {
            const long long t4 = clock64();
            atomicAdd(P.phase_clk + 0, (unsigned long long)(t1 - t0));
            atomicAdd(P.phase_clk + 1, (unsigned long long)(t2 - t1));
            atomicAdd(P.phase_clk + 2, (unsigned long long)(t3 - t2));
            atomicAdd(P.phase_clk + 3, (unsigned long long)(t4 - t3));
        }
        team_sync(C);
    }
    team_sync(C);  // no CTA leaves while another may still write to its shared memory
}

cudaError_t set_multipole_const_cg64(const MultipoleConst& mc) { return cudaMemcpyToSymbol(c_mp, &mc, sizeof(mc)); }

static const void* cg64_fn(int threads, bool fix) {
    switch (threads) {
        case 256: return fix ? (const void*)cg64_kernel<256, true> : (const void*)cg64_kernel<256, false>;
        case 1024: return fix ? (const void*)cg64_kernel<1024, true> : (const void*)cg64_kernel<1024, false>;
        default: return fix ? (const void*)cg64_kernel<512, true> : (const void*)cg64_kernel<512, false>;
    }
}

size_t cg64_smem(int r_pe) { return sizeof(double) * 28 * (size_t)(2 * r_pe + 1); }

cudaError_t cg64_occupancy(int threads, bool fix, size_t smem, int* blocks_per_sm) {
    const void* f = cg64_fn(threads, fix);
    cudaError_t e = raise_smem_limit(f, smem);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, f, threads, smem);
}

cudaError_t launch_cg64_kernel(const SolveParams& P, int threads, bool fix, int teams, int team, size_t smem, cudaStream_t st) {
    const void* f = cg64_fn(threads, fix);
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)team;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(teams * team));
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    void* args[] = {const_cast<SolveParams*>(&P)};
    return cudaLaunchKernelExC(&cfg, f, args);
}

}  // namespace exx
