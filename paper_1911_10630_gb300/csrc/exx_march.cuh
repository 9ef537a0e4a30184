// exx_march.cuh -- the FP32 multigrid PCG of Step IV (Sec. III.C) as passes
// that march through a ball plane by plane.
//
// The same iteration as mg_pcg in exx_solve.cu (CG preconditioned by one
// symmetric V-cycle with a weighted-Jacobi sweep each way), arranged so that
// each fine-level vector moves as rarely as the data flow allows. The sweeps
// of a V-cycle are pointwise but for three stencils, and every other operand
// of a stencil's input can be formed on the way:
//   pass P: p = z + beta p, A p, p.Ap, and d += alpha p of the last iteration
//           (reads z, p, d; writes p, d, Ap),
//   pass R: r -= alpha Ap, r.r, the residual after the first Jacobi sweep,
//           T = r - A (w D^-1 r), and its restriction (reads r, Ap; writes r),
//   pass Z: Z = w D^-1 r + P zc, z = Z + w D^-1 (r - A Z), r.z (reads r;
//           writes z): 44 bytes per point and iteration.
// The sweeps kept apart move 102 bytes, and 168 counted by the hardware.
//
// Layout: a ball's rows along z are cut into 16-byte quads (z a multiple of
// 4). A thread owns the quads of two rows, (y, z..z+3) and (y + 1, z..z+3), y
// even, and walks x: a column. Columns are sorted by how far they reach in
// |x|, so the columns of plane x are a prefix of the list and a vector is
// stored plane by plane, row j of column c of plane x at quad j nq + pst[x] + c:
// every access is a contiguous run of 16-byte quads with no index table, and
// the elements of a quad outside the ball hold zero.
//
// The x legs of the stencil are the thread's own column at six other planes: a
// ring in tensor memory (56 columns of 32-bit cells a thread; an access costs
// no shared-memory bandwidth and no register), one slot rewritten per plane.
// The y and z legs come from the centre plane in shared memory (two buffers,
// one barrier per plane), the two rows sharing their y legs: 14 16-byte loads
// and two stores per 8 points instead of 152 loads. FP32 operations are issued
// in pairs; the next planes are staged by cp.async.
//
// What bounds it: latency. A plane is one step, with a barrier, of every thread of the
// pair; over the kernel the counters give 24 % of the DRAM rate, 0.8 instructions a
// clock and SM, and the waits on staged planes and on the barrier as the first stalls. 128 registers a thread
// leave 16 warps to an SM to cover them. Per pair and iteration
// at R_PE 24, microseconds of an SM: 340 for the sweeps kept apart (the
// pair_kernel form); 225 with one row per column; 190 with the ring in
// registers or in shared memory; 150 as it is, of which the coarse levels
// take a fifth.
#pragma once

#include "exx_kernels.cuh"

namespace exx {

// The CTA's dynamic shared memory, addressed by float index: a 32-bit register
// an address, and loads known to be shared in the out-of-line passes too.
extern __shared__ __align__(16) float march_sm[];
__device__ __forceinline__ float4& s4(int i) { return *reinterpret_cast<float4*>(march_sm + i); }
__device__ __forceinline__ ulonglong2 s2(int i) { return *reinterpret_cast<const ulonglong2*>(march_sm + i); }
__device__ __forceinline__ float& s1(int i) { return march_sm[i]; }
__device__ __forceinline__ int& si(int i) { return reinterpret_cast<int*>(march_sm)[i]; }

// A group of threads marching one slab of planes. With one group the vectors
// are updated in place; with more, the halo planes of a slab are formed again
// from the neighbours' inputs, so the caller passes separate outputs.
struct MarchGroup {
    int t;          // thread within the group (its column), -1: no group
    int nthr;       // threads of the group (a multiple of 32), named barrier bar
    int bar;
    int Xs, Xe;     // coarse planes of the slab; it owns the planes [2 Xs, 2 Xe) of the ball
    __device__ __forceinline__ int index() const { return t < 0 ? 0 : bar - 1; }
};

__device__ __forceinline__ void group_sync(const MarchGroup& g) {
    asm volatile("bar.sync %0, %1;" ::"r"(g.bar), "r"(g.nthr) : "memory");
}

// Groups of level L's columns among the CTA's threads.
__device__ __forceinline__ MarchGroup march_groups(const MarchLv& L) {
    const int n32 = (L.ncol + 31) & ~31;
    const int nX = 2 * ((L.R + 1) / 2) + 1;
    const int G = L.groups;
    MarchGroup g;
    const int k = (int)threadIdx.x / n32;
    g.nthr = n32;
    g.bar = 1 + k;
    g.t = k < G ? (int)threadIdx.x - k * n32 : -1;
    g.Xs = -(nX / 2) + k * nX / G;
    g.Xe = -(nX / 2) + (k + 1) * nX / G;
    return g;
}

// One column of a level: index of its first row's quad in a plane buffer, and
// the reach in |x| of each element (byte e: largest |x| + 1, 0 = never).
struct MarchCol {
    int sm, y, z0;
    unsigned xm[2];
    int xmax, xfull;  // largest |x| of any element and of all eight (-1: never)
};

__device__ __forceinline__ MarchCol march_col(const MarchLv& L, int t) {
    MarchCol c;
    c.xmax = c.xfull = -1;
    c.sm = L.org;  // any place whose neighbours are in the buffer
    c.y = c.z0 = 0;
    c.xm[0] = c.xm[1] = 0u;
    if (t >= 0 && t < L.ncol) {
        const int4 q = __ldg(L.col + t);
        c.sm = q.x & 0xffff;
        c.y = ((q.x >> 16) & 0xff) - 64;
        c.z0 = ((q.x >> 24) & 0xff) - 64;
        c.xm[0] = (unsigned)q.y;
        c.xm[1] = (unsigned)q.z;
        int mx = 0, mn = 255;
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int b = (int)((c.xm[j] >> (8 * e)) & 255u);
                mx = max(mx, b);
                mn = min(mn, b);
            }
        c.xmax = mx - 1;
        c.xfull = mn - 1;
    }
    return c;
}

// Two rows' quads.
struct F8 {
    float4 r[2];
};

__device__ __forceinline__ float4 f4zero() { return make_float4(0.f, 0.f, 0.f, 0.f); }
__device__ __forceinline__ F8 f8zero() {
    F8 v;
    v.r[0] = v.r[1] = f4zero();
    return v;
}

// Two FP32 operations per instruction, each rounded as the scalar one.
__device__ __forceinline__ unsigned long long pack2(float a, float b) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(unsigned long long v, float& a, float& b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b) {
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

__device__ __forceinline__ float4 f4fma(unsigned long long a2, const float4& x, const float4& y) {  // a2: a twice
    float4 v;
    unpack2(fma2(a2, pack2(x.x, x.y), pack2(y.x, y.y)), v.x, v.y);
    unpack2(fma2(a2, pack2(x.z, x.w), pack2(y.z, y.w)), v.z, v.w);
    return v;
}
__device__ __forceinline__ F8 f8fma(float a, const F8& x, const F8& y) {
    const unsigned long long a2 = pack2(a, a);
    F8 v;
    v.r[0] = f4fma(a2, x.r[0], y.r[0]);
    v.r[1] = f4fma(a2, x.r[1], y.r[1]);
    return v;
}

// acc += w (a + b), w given twice.
__device__ __forceinline__ void f4legs(float4& acc, unsigned long long w2, const float4& a, const float4& b) {
    unpack2(fma2(w2, add2(pack2(a.x, a.y), pack2(b.x, b.y)), pack2(acc.x, acc.y)), acc.x, acc.y);
    unpack2(fma2(w2, add2(pack2(a.z, a.w), pack2(b.z, b.w)), pack2(acc.z, acc.w)), acc.z, acc.w);
}

__device__ __forceinline__ float f4dot(const float4& a, const float4& b, float s) {
    return fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, fmaf(a.x, b.x, s))));
}
__device__ __forceinline__ float f8dot(const F8& a, const F8& b, float s) {
    return f4dot(a.r[1], b.r[1], f4dot(a.r[0], b.r[0], s));
}

// Zero outside the ball at plane |x| = ax.
__device__ __forceinline__ void f4mask(float4& v, unsigned xm, int ax) {
    if (!((int)(xm & 255u) > ax)) v.x = 0.f;
    if (!((int)((xm >> 8) & 255u) > ax)) v.y = 0.f;
    if (!((int)((xm >> 16) & 255u) > ax)) v.z = 0.f;
    if (!((int)(xm >> 24) > ax)) v.w = 0.f;
}
__device__ __forceinline__ void f8mask(F8& v, const MarchCol& c, int ax) {
    if (ax > c.xfull) {
        f4mask(v.r[0], c.xm[0], ax);
        f4mask(v.r[1], c.xm[1], ax);
    }
}

// Quads k and k + nq of the pair's slot (one base pointer, 32-bit quad
// offsets). They are copied to a place of the thread's own in shared memory one
// step before they are used: no registers hold them meanwhile, and a column
// outside the ball gets zeros.
__device__ __forceinline__ void stage16(int to, const float4* from, bool on) {
    const unsigned dst = (unsigned)__cvta_generic_to_shared(march_sm + to);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(from), "r"(on ? 16 : 0) : "memory");
}
template <int RS>
__device__ __forceinline__ void f8stage(int to, int n, const float4* from, bool on) {
    stage16(to, from, on);
    stage16(to + 4 * n, from + RS, on);
}
__device__ __forceinline__ void stage_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void stage_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }
__device__ __forceinline__ void stage_wait_but_last() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }
__device__ __forceinline__ F8 f8staged(int at, int n) {
    F8 v;
    v.r[0] = s4(at);
    v.r[1] = s4(at + 4 * n);
    return v;
}
template <int RS>
__device__ __forceinline__ void f8store(float4* to, const F8& a) {
    to[0] = a.r[0];
    to[RS] = a.r[1];
}

// The thread's own column over the planes x - 3 .. x + 2, in tensor memory:
// eight columns of the thread's lane a plane, a[i] the address of plane
// x - 3 + i. x + 3 is in registers until the step's end, when it takes the place
// of x - 3. Tensor memory is as private as registers and as cheap to read as
// shared memory, whose pipe the y and z legs already fill.
__device__ __forceinline__ void tm_put(unsigned at, const F8& v) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(at),
                 "r"(__float_as_uint(v.r[0].x)), "r"(__float_as_uint(v.r[0].y)), "r"(__float_as_uint(v.r[0].z)),
                 "r"(__float_as_uint(v.r[0].w)), "r"(__float_as_uint(v.r[1].x)), "r"(__float_as_uint(v.r[1].y)),
                 "r"(__float_as_uint(v.r[1].z)), "r"(__float_as_uint(v.r[1].w))
                 : "memory");
}
// Starts the load; the values are there after ring_wait on them.
__device__ __forceinline__ void tm_get(unsigned at, F8& v) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(v.r[0].x), "=f"(v.r[0].y), "=f"(v.r[0].z), "=f"(v.r[0].w), "=f"(v.r[1].x), "=f"(v.r[1].y),
                   "=f"(v.r[1].z), "=f"(v.r[1].w)
                 : "r"(at)
                 : "memory");
}
struct MarchRing {
    unsigned a[6];
    __device__ __forceinline__ void put(const F8& v) {
        tm_put(a[0], v);
        turn();
    }
    __device__ __forceinline__ void turn() {
        const unsigned t = a[0];
#pragma unroll
        for (int i = 0; i < 5; ++i) a[i] = a[i + 1];
        a[5] = t;
    }
    __device__ __forceinline__ void get(int i, F8& v) const { tm_get(a[i], v); }
};
__device__ __forceinline__ void ring_wait(F8& u, F8& v) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+f"(u.r[0].x), "+f"(u.r[0].y), "+f"(u.r[0].z), "+f"(u.r[0].w), "+f"(u.r[1].x), "+f"(u.r[1].y),
                   "+f"(u.r[1].z), "+f"(u.r[1].w), "+f"(v.r[0].x), "+f"(v.r[0].y), "+f"(v.r[0].z), "+f"(v.r[0].w),
                   "+f"(v.r[1].x), "+f"(v.r[1].y), "+f"(v.r[1].z), "+f"(v.r[1].w)::"memory");
}
__device__ __forceinline__ void ring_wait(F8& u) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+f"(u.r[0].x), "+f"(u.r[0].y), "+f"(u.r[0].z), "+f"(u.r[0].w), "+f"(u.r[1].x), "+f"(u.r[1].y),
                   "+f"(u.r[1].z), "+f"(u.r[1].w)::"memory");
}
// The stores of earlier steps are complete (before the step's first load).
__device__ __forceinline__ void ring_stored() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Tensor memory of a CTA: 56 columns for each warp of a lane quarter, six
// planes and one value more (slot 6) that a pass keeps from step to step.
template <int NT>
constexpr int ring_columns() {
    int n = 32;
    while (n < 56 * ((NT / 32 + 3) / 4)) n *= 2;
    return n;
}
// The base address, in shared memory (one warp allocates; the caller synchronises).
template <int NT>
__device__ __forceinline__ void ring_alloc(unsigned* at) {
    if (threadIdx.x < 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         (unsigned)__cvta_generic_to_shared(at)),
                     "r"(ring_columns<NT>())
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
}
template <int NT>
__device__ __forceinline__ void ring_free(unsigned base) {
    if (threadIdx.x < 32)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(base), "r"(ring_columns<NT>()));
}
__device__ __forceinline__ unsigned ring_of_warp(unsigned base) {
    const unsigned w = threadIdx.x >> 5;
    return base + ((w & 3u) << 21) + 56u * (w >> 2);  // lanes 32 (w mod 4) .., 56 columns a warp
}

__device__ __forceinline__ void quad_z_legs(const float4& w, float4& acc, const float4& l, const float4& c,
                                            const float4& r) {
    acc.x = fmaf(w.x, c.y + l.w, fmaf(w.y, c.z + l.z, fmaf(w.z, c.w + l.y, acc.x)));
    acc.y = fmaf(w.x, c.z + c.x, fmaf(w.y, c.w + l.w, fmaf(w.z, r.x + l.z, acc.y)));
    acc.z = fmaf(w.x, c.w + c.y, fmaf(w.y, r.x + c.x, fmaf(w.z, r.y + l.w, acc.z)));
    acc.w = fmaf(w.x, r.x + c.z, fmaf(w.y, r.y + c.y, fmaf(w.z, r.z + c.x, acc.w)));
}

// The 19-point stencil of a column's two quads: x legs from the ring (and p3,
// plane x + 3), y and z legs from the centre plane (pl: at the first row's
// quad). Every lane of the warp takes part; one without points gets a value
// that its caller drops.
__device__ __forceinline__ F8 column_lap(int op, int pl, int pitch, const MarchRing& q, const F8& c, const F8& p3) {
    F8 acc, a, b, e;
    q.get(0, e);
    q.get(1, a);
    q.get(5, b);
    const float4 wz = s4(op + 24);  // legs 1, 2, 3 along z, the centre
#pragma unroll
    for (int j = 0; j < 2; ++j) acc.r[j] = make_float4(wz.w * c.r[j].x, wz.w * c.r[j].y, wz.w * c.r[j].z, wz.w * c.r[j].w);
    const ulonglong2 wy = s2(op + 12);  // legs 1 and 2 along y, each twice
    // rows y - 3 .. y + 4; y and y + 1 are the column's own
    const float4 m1 = s4(pl - pitch), n2 = s4(pl + 2 * pitch);
    f4legs(acc.r[0], wy.x, m1, c.r[1]);
    f4legs(acc.r[1], wy.x, c.r[0], n2);
    const float4 m2 = s4(pl - 2 * pitch), n3 = s4(pl + 3 * pitch);
    f4legs(acc.r[0], wy.y, m2, n2);
    f4legs(acc.r[1], wy.y, m1, n3);
    const float4 m3 = s4(pl - 3 * pitch), n4 = s4(pl + 4 * pitch);
    f4legs(acc.r[0], s2(op + 16).x, m3, n3);
    f4legs(acc.r[1], s2(op + 16).x, m2, n4);
    const ulonglong2 wx = s2(op);
    ring_wait(a, b);
    ring_wait(e);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        f4legs(acc.r[j], s2(op + 4).x, e.r[j], p3.r[j]);
        f4legs(acc.r[j], wx.y, a.r[j], b.r[j]);
    }
    q.get(2, a);
    q.get(4, b);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const float4 l = s4(pl + j * pitch - 4), r = s4(pl + j * pitch + 4);
        quad_z_legs(wz, acc.r[j], l, c.r[j], r);
    }
    ring_wait(a, b);
#pragma unroll
    for (int j = 0; j < 2; ++j) f4legs(acc.r[j], wx.x, a.r[j], b.r[j]);
    return acc;
}

// The march common to the passes: column g.t of level L, planes [x0, x1),
// begun at plane xb <= x0 - 6 to fill the ring. make(x) forms the stencil's
// input of a plane from what fetch(x) staged one step before; pre(x) runs
// (with whether the warp is live) before the step's barrier, mid(x) after it; step(x, pl, q, c, p3) once plane x
// is in shared memory (pl: the column's place), c and p3 the column's values
// of planes x and x + 3. A warp whose columns reach |x| = r at most only keeps
// the barriers but from plane -r - before to r + after: both plane buffers hold
// zeros in its columns otherwise. step gets whether any of the warp's columns
// has points on plane x.
template <class Fetch, class Make, class Pre, class Mid, class Step>
__device__ __forceinline__ void march_planes(const MarchLv& L, const MarchGroup& g, const MarchCol& c, int sm, unsigned ring,
                                             int xb, int x0, int x1, int before, int after, Fetch fetch, Make make, Pre pre,
                                             Mid mid, Step step) {
    MarchRing q;
#pragma unroll
    for (int i = 0; i < 6; ++i) q.a[i] = ring + 8 * i;
#pragma unroll
    for (int i = 0; i < 6; ++i) q.put(f8zero());
    const int reach = __reduce_max_sync(0xffffffffu, c.xmax);
    fetch(xb + 3);
#pragma unroll 1
    for (int x = xb; x < x0; ++x) {
        const F8 p3 = make(x + 3);
        fetch(x + 4);
        pre(x, true);
        group_sync(g);
        __syncwarp();
        q.put(p3);
    }
    // a thread without a column writes its zeros into the buffer's padding
    const int own = sm + c.sm, to = c.xmax >= 0 ? own : sm, dy = c.xmax >= 0 ? L.pitch : 0;
#pragma unroll 1
    for (int x = x0; x < x1; ++x) {
        const int odd = (x & 1) * L.planef;
        const bool live = (x >= -reach - before && x <= reach + after) || x - x0 < 2;
        F8 cq, p3;
        if (live) {
            p3 = make(x + 3);
            fetch(x + 4);
            __syncwarp();  // tensor memory is read and written by whole warps
            ring_stored();
            q.get(3, cq);
            ring_wait(cq);
            s4(to + odd) = cq.r[0];
            s4(to + odd + dy) = cq.r[1];
        }
        pre(x, live);
        group_sync(g);
        mid(x);
        if (live) {
            __syncwarp();
            step(x, abs(x) <= reach, own + odd, q, cq, p3);
            __syncwarp();
            q.put(p3);
        } else {
            q.turn();
        }
    }
    stage_wait();  // no copy in flight when the space changes hands
}

// Pass P. it = 0: p = z and d is not touched; it = 1: d = alpha p_old; later d += alpha p_old.
template <int RS>
__device__ __forceinline__ float march_p(int op, const MarchLv L, const MarchGroup g, int sm, unsigned ring, int st, int st2,
                                         float4* hot, int po, int pn, float be, float al, int it) {
    float sum = 0.f;
    if (g.t < 0) return sum;
    const MarchCol c = march_col(L, g.t);
    const int R = L.R;
    const int xs = max(2 * g.Xs, -R), xe = min(2 * g.Xe, R + 1);
    const int pst = L.sm_pst + R;
    const int n = g.nthr;
    auto fetch = [&](int x) {
        const bool on = abs(x) <= c.xmax;
        const float4* a = hot + (on ? si(pst + x) + g.t : 0);
        f8stage<RS>(st, n, a + kMarchZ * 2 * RS, on);
        if (it) f8stage<RS>(st + 8 * n, n, a + po, on);
        if (it > 1) f8stage<RS>(st2, n, a + kMarchD * 2 * RS, on);
    };
    auto make = [&](int x) {
        stage_wait();
        F8 v = f8staged(st, n);
        const bool own = x >= xs && x < xe && abs(x) <= c.xmax;
        float4* a = hot + (own ? si(pst + x) + g.t : 0);
        if (it) {
            const F8 p = f8staged(st + 8 * n, n);
            v = f8fma(be, p, v);
            if (own) f8store<RS>(a + kMarchD * 2 * RS, f8fma(al, p, it > 1 ? f8staged(st2, n) : f8zero()));
        }
        if (own) f8store<RS>(a + pn, v);
        return v;
    };
    auto none = [](int, bool) {};
    march_planes(L, g, c, sm, ring, xs > -R ? xs - 6 : xs - 3, xs, xe, 4, 2, fetch, make, none, [](int) {},
                 [&](int x, bool any, int pl, const MarchRing& q, const F8& cq, const F8& p3) {
                     if (!any) return;
                     F8 a = column_lap(op, pl, L.pitch, q, cq, p3);
                     if (abs(x) > c.xmax) return;
                     f8mask(a, c, abs(x));
                     f8store<RS>(hot + kMarchAp * 2 * RS + si(pst + x) + g.t, a);
                     sum = f8dot(cq, a, sum);
                 });
    return sum;
}

// Where a level's restricted residual goes: quads of the next marching level,
// or the zero-padded cube of the first level kept in shared memory.
struct MarchDown {
    int rhs;            // next marching level's right-hand side, or -1
    int org, plane, pitch;  // shared-memory cube, index org + X plane + Y pitch + Z
};

// Pass R on level L (next level N; wd the Jacobi factor times A's spacing,
// the same on every level; sS: a plane buffer for the sums to restrict). upd:
// r -= al ap and ro = r (level 0), else r is taken as it is. Returns the
// thread's share of r.r over the slab's planes.
template <int RS>
__device__ __forceinline__ float march_r(int op, float wd, const MarchLv L, const MarchLv N, const MarchDown dn,
                                         const MarchGroup g, int sm, int sS, unsigned ring, int st, float4* hot, int r, int ro,
                                         float al, bool upd) {
    float sum = 0.f;
    if (g.t < 0) return sum;
    const MarchCol c = march_col(L, g.t);
    const int R = L.R;
    const int xs = max(2 * g.Xs, -R), xe = min(2 * g.Xe, R + 1);
    const int x0 = 2 * g.Xs - 1, x1 = 2 * g.Xe;  // T of the planes [x0, x1)
    const int pst = L.sm_pst + R;
    // zero but for the columns, which write it at every odd plane (first after two barriers)
    for (int k = 4 * g.t; k < L.planef; k += 4 * g.nthr) s4(sS + k) = f4zero();
    const int n = g.nthr;
    auto fetch = [&](int x) {
        const bool on = abs(x) <= c.xmax;
        const float4* a = hot + (on ? si(pst + x) + g.t : 0);
        f8stage<RS>(st, n, a + r, on);
        if (upd) f8stage<RS>(st + 8 * n, n, a + kMarchAp * 2 * RS, on);
    };
    auto make = [&](int x) {
        stage_wait();
        F8 v = f8staged(st, n);
        if (upd) {
            v = f8fma(-al, f8staged(st + 8 * n, n), v);
            if (x >= xs && x < xe && abs(x) <= c.xmax) {
                f8store<RS>(hot + ro + si(pst + x) + g.t, v);
                sum = f8dot(v, v, sum);
            }
        }
        return v;
    };
    // full weighting onto coarse plane X: 0.5, 1, 0.5 along each axis over 8
    // (the coarse level has at most as many columns as the group has threads)
    const MarchCol cc = march_col(N, g.t);
    const int s0 = sS + L.org + 2 * cc.y * L.pitch + 2 * cc.z0;
    const int cube0 = dn.org + cc.y * dn.pitch + cc.z0;
    auto gather = [&](int X) {
        const int ax = abs(X);
        if (ax > cc.xmax) return;
        F8 o = f8zero();
#pragma unroll
        for (int ey = -1; ey <= 3; ++ey) {
            const int s = s0 + ey * L.pitch;
            const float b = s1(s - 1);
            const float4 u = s4(s), v = s4(s + 4);
            const float4 t = make_float4(fmaf(0.5f, b + u.y, u.x), fmaf(0.5f, u.y + u.w, u.z), fmaf(0.5f, u.w + v.y, v.x),
                                         fmaf(0.5f, v.y + v.w, v.z));
            if (ey <= 1) o.r[0] = f4fma(ey == 0 ? pack2(0.125f, 0.125f) : pack2(0.0625f, 0.0625f), t, o.r[0]);
            if (ey >= 1) o.r[1] = f4fma(ey == 2 ? pack2(0.125f, 0.125f) : pack2(0.0625f, 0.0625f), t, o.r[1]);
        }
        f8mask(o, cc, ax);
        if (dn.rhs >= 0) {
            f8store<RS>(hot + dn.rhs + si(N.sm_pst + N.R + X) + g.t, o);
        } else {
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int w = cube0 + X * dn.plane + j * dn.pitch;
                if ((int)(cc.xm[j] & 255u) > ax) s1(w) = o.r[j].x;
                if ((int)((cc.xm[j] >> 8) & 255u) > ax) s1(w + 1) = o.r[j].y;
                if ((int)((cc.xm[j] >> 16) & 255u) > ax) s1(w + 2) = o.r[j].z;
                if ((int)(cc.xm[j] >> 24) > ax) s1(w + 3) = o.r[j].w;
            }
        }
    };
    tm_put(ring + 48, f8zero());
    // the gather of a coarse plane: its sums were stored before this step's barrier
    auto mid = [&](int x) {
        if (!(x & 1) && x > x0 + 1) gather(x / 2 - 1);
    };
    const int oS = c.xmax >= 0 ? sS + c.sm : sS, dy = c.xmax >= 0 ? L.pitch : 0;
    march_planes(L, g, c, sm, ring, xs > -R ? x0 - 6 : min(x0, -R) - 3, x0, x1, 4, 4, fetch, make, [](int, bool) {}, mid,
                 [&](int x, bool any, int pl, const MarchRing& q, const F8& cq, const F8& p3) {
                     F8 T = f8zero(), acc;
                     if (any) {
                         T = f8fma(-wd, column_lap(op, pl, L.pitch, q, cq, p3), cq);
                         f8mask(T, c, abs(x));
                     }
                     // slot 6: T(2X) + T(2X - 1) / 2 of the coarse plane being summed
                     __syncwarp();
                     tm_get(ring + 48, acc);
                     ring_wait(acc);
                     if (x & 1) {
                         if (x > x0) {
                             const F8 v = f8fma(0.5f, T, acc);
                             s4(oS) = v.r[0];
                             s4(oS + dy) = v.r[1];
                         }
                         acc = f8fma(0.5f, T, f8zero());
                     } else {
                         acc = f8fma(1.f, T, acc);
                     }
                     __syncwarp();
                     tm_put(ring + 48, acc);
                 });
    group_sync(g);
    gather(g.Xe - 1);
    return sum;
}

// The next coarser level's correction: its quads (a marching level N, staged
// plane by plane through two plane buffers of N's layout), or the zero-padded
// cube of a level in shared memory. Index of (X, Y, Z): org + X plane + Y
// pitch + Z, with X & 1 in place of X for the staged planes.
struct MarchUp {
    int quads;            // -1: cube
    int cube;             // the two plane buffers
    int org, plane, pitch, R;
};

// Pass Z on level L (Jacobi factor wdl): z as quads. Returns the thread's
// share of r.z.
template <int RS>
__device__ __forceinline__ float march_z(int op, float wd, const MarchLv L, const MarchLv N, const MarchUp up,
                                         const MarchGroup g, int sm, unsigned ring, int st, float4* hot, int r, int z, float wdl) {
    float sum = 0.f;
    if (g.t < 0) return sum;
    const MarchCol c = march_col(L, g.t);
    const int R = L.R;
    const int xs = max(2 * g.Xs, -R), xe = min(2 * g.Xe, R + 1);
    const int pst = L.sm_pst + R;
    // the correction on coarse plane X, interpolated in y and z to the column's rows
    const int u0 = up.cube + up.org + c.y / 2 * up.pitch + c.z0 / 2;  // y even
    auto interp = [&](int X) {
        F8 v = f8zero();
        if (abs(X) <= up.R && c.xmax >= 0) {
            const int u = u0 + (up.quads >= 0 ? X & 1 : X) * up.plane;
            const float a = s1(u), b = s1(u + 1), e = s1(u + 2);
            const float a1 = s1(u + up.pitch), b1 = s1(u + up.pitch + 1), e1 = s1(u + up.pitch + 2);
            v.r[0] = make_float4(a, 0.5f * (a + b), b, 0.5f * (b + e));
            const float am = 0.5f * (a + a1), bm = 0.5f * (b + b1), em = 0.5f * (e + e1);
            v.r[1] = make_float4(am, 0.5f * (am + bm), bm, 0.5f * (bm + em));
        }
        return v;
    };
    // staging: the copy of coarse plane X is issued at the even step 2 X - 6
    // (plane X - 2 of the same buffer was last read two barriers before),
    // complete by the next step's barrier and read at step 2 X - 4
    MarchCol cc;
    cc.xmax = -1;
    cc.sm = 0;
    auto cload = [&](int X) {
        if (g.t < N.ncol) {
            const bool on = abs(X) <= cc.xmax;
            const int k = on ? up.quads + si(N.sm_pst + N.R + X) + g.t : 0, to = up.cube + (X & 1) * up.plane + cc.sm;
            stage16(to, hot + k, on);
            stage16(to + up.pitch, hot + k + RS, on);
        }
    };
    if (up.quads >= 0) {
        for (int k = 4 * g.t; k < 2 * N.planef; k += 4 * g.nthr) s4(up.cube + k) = f4zero();
        group_sync(g);
        cc = march_col(N, g.t);
    }
    const int n = g.nthr;
    auto fetch = [&](int x) {  // first r of the step's centre plane again, read seven planes ago
        const bool oc = abs(x - 4) <= c.xmax, on = x >= xs - 3 && abs(x) <= c.xmax;
        f8stage<RS>(st + 8 * n, n, hot + r + (oc ? si(pst + x - 4) + g.t : 0), oc);
        stage_commit();
        f8stage<RS>(st, n, hot + r + (on ? si(pst + x) + g.t : 0), on);
        stage_commit();
    };
    tm_put(ring + 48, f8zero());
    auto make = [&](int x) {  // consecutive x: slot 6 holds the coarse plane floor(x / 2) before the call
        F8 v;
        __syncwarp();
        ring_stored();
        tm_get(ring + 48, v);
        if (x & 1) {
            const F8 i1 = interp((x + 1) / 2);
            ring_wait(v);
#pragma unroll
            for (int j = 0; j < 2; ++j)
                v.r[j] = make_float4(0.5f * (v.r[j].x + i1.r[j].x), 0.5f * (v.r[j].y + i1.r[j].y),
                                     0.5f * (v.r[j].z + i1.r[j].z), 0.5f * (v.r[j].w + i1.r[j].w));
            __syncwarp();
            tm_put(ring + 48, i1);
        } else {
            ring_wait(v);
        }
        stage_wait();
        v = f8fma(wdl, f8staged(st, n), v);
        f8mask(v, c, abs(x));
        return v;
    };
    auto pre = [&](int x, bool live) {
        if (up.quads < 0) return;
        if (!(x & 1)) cload(x / 2 + 3);
        else if (!live) stage_wait();  // a live warp has waited in make
    };
    // odd; the coarse planes of the first two made planes are staged by then
    const int xb = ((xs > -R ? xs - 10 : xs - 7)) | 1;
    if (up.quads >= 0) {
        cload((xb + 5) / 2);
        stage_wait();
        group_sync(g);
    }
    march_planes(L, g, c, sm, ring, xb, xs, xe, 5, 2, fetch, make, pre, [](int) {},
                 [&](int x, bool any, int pl, const MarchRing& q, const F8& cq, const F8& p3) {
                     if (!any) return;
                     F8 v = column_lap(op, pl, L.pitch, q, cq, p3);
                     if (abs(x) > c.xmax) return;
                     stage_wait_but_last();
                     const F8 rc = f8staged(st + 8 * n, n);
                     v = f8fma(-wd, v, f8fma(wdl, rc, cq));
                     f8mask(v, c, abs(x));
                     f8store<RS>(hot + z + si(pst + x) + g.t, v);
                     sum = f8dot(rc, v, sum);
                 });
    return sum;
}

// ---- the levels kept in shared memory (radius <= kMarchSmem) --------------
// Each in a zero-padded cube whose rows share their padding: index
// org + X plane + Y pitch + Z. On entry the first one's cube holds its
// right-hand side; on return its correction.

__device__ __forceinline__ int small_idx(const MarchSmall& s, int pk) {
    return s.org + off_x(pk) * s.plane + off_y(pk) * s.pitch + off_z(pk);
}

__device__ __forceinline__ float small_lap(const Stencil<float>& A, const float* f, int plane, int pitch) {
    float acc = A.c0 * f[0];
#pragma unroll
    for (int q = 1; q <= 3; ++q) {
        acc = fmaf(A.cx[q - 1], f[q * plane] + f[-q * plane], acc);
        acc = fmaf(A.cy[q - 1], f[q * pitch] + f[-q * pitch], acc);
        acc = fmaf(A.cz[q - 1], f[q] + f[-q], acc);
    }
    return acc;
}

template <int NT>
__device__ __forceinline__ void march_small(const SolveParams& P, const MarchGeo& M, const MGGeo& MG) {
    const Stencil<float>& A = P.mg_a32[0];
    const float wd = P.mg_wd32[0];
    const int t = threadIdx.x;
    float* sm = march_sm;
    for (int l = M.nm; l < M.L; ++l) {
        const MarchSmall s = M.sl[l];
        const int* __restrict__ off = MG.lv[l].off;
        const int n = MG.lv[l].n;
        float* cube = sm + s.cube;
        float* rhs = sm + s.rhs;
        float T[kMarchPts];
#pragma unroll
        for (int i = 0; i < kMarchPts; ++i) {
            const int k = t + i * NT;
            if (k < n) {
                const float* f = cube + small_idx(s, __ldg(off + k));
                rhs[k] = f[0];
                T[i] = fmaf(-wd, small_lap(A, f, s.plane, s.pitch), f[0]);
            }
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < kMarchPts; ++i) {
            const int k = t + i * NT;
            if (k < n) cube[small_idx(s, __ldg(off + k))] = T[i];
        }
        __syncthreads();
        const MarchSmall sn = M.sl[l + 1];
        for (int k = t; k < MG.lv[l + 1].n; k += NT) {
            const int pk = __ldg(MG.lv[l + 1].off + k);
            const float* f = cube + s.org + 2 * (off_x(pk) * s.plane + off_y(pk) * s.pitch + off_z(pk));
            float acc = 0.f;
#pragma unroll
            for (int ex = -1; ex <= 1; ++ex)
#pragma unroll
                for (int ey = -1; ey <= 1; ++ey) {
                    const float* u = f + ex * s.plane + ey * s.pitch;
                    const float w = (ex ? 0.5f : 1.f) * (ey ? 0.5f : 1.f);
                    acc = fmaf(w, fmaf(0.5f, u[-1] + u[1], u[0]), acc);
                }
            sm[sn.cube + small_idx(sn, pk)] = 0.125f * acc;
        }
        __syncthreads();
    }
    {  // the coarsest level: its dense inverse (symmetric: read by columns), the sums split over the threads
        const MarchSmall s = M.sl[M.L];
        const int n = MG.lv[M.L].n;
        const int* __restrict__ off = MG.lv[M.L].off;
        float* rhs = sm + s.rhs;            // [128] right-hand side, then [NP][128] partial sums
        constexpr int NP = NT < 256 ? 1 : NT / 128, NK = NT < 128 ? NT : 128;
        const int part = t / NK;
        for (int k = t; k < n; k += NT) rhs[k] = sm[s.cube + small_idx(s, __ldg(off + k))];
        __syncthreads();
        if (part < NP)
            for (int k = t % NK; k < n; k += NK) {
                const float* __restrict__ m = MG.minv32 + k;
                float acc = 0.f;
#pragma unroll 8
                for (int j = part; j < n; j += NP) acc = fmaf(__ldg(m + j * n), rhs[j], acc);
                rhs[128 + part * 128 + k] = acc;
            }
        __syncthreads();
        for (int k = t; k < n; k += NT) {
            float acc = 0.f;
#pragma unroll
            for (int p = 0; p < NP; ++p) acc += rhs[128 + p * 128 + k];
            sm[s.cube + small_idx(s, __ldg(off + k))] = acc;
        }
        __syncthreads();
    }
    for (int l = M.L - 1; l >= M.nm; --l) {
        const MarchSmall s = M.sl[l], sn = M.sl[l + 1];
        const int* __restrict__ off = MG.lv[l].off;
        const int n = MG.lv[l].n;
        float* cube = sm + s.cube;
        const float* rhs = sm + s.rhs;
        const float* zc = sm + sn.cube + sn.org;
        const float wdl = P.mg_wd32[l];
        for (int k = t; k < n; k += NT) {
            const int pk = __ldg(off + k);
            const int x = off_x(pk), y = off_y(pk), z = off_z(pk);
            const int xo = x & 1, yo = y & 1, zo = z & 1;
            const float* f = zc + ((x - xo) / 2) * sn.plane + ((y - yo) / 2) * sn.pitch + (z - zo) / 2;
            // trilinear: the mean over the one or two coarse neighbours along each axis
            float acc = 0.f;
            for (int cx = 0; cx <= xo; ++cx)
                for (int cy = 0; cy <= yo; ++cy) {
                    const float* u = f + cx * sn.plane + cy * sn.pitch;
                    acc += zo ? 0.5f * (u[0] + u[1]) : u[0];
                }
            acc *= (xo ? 0.5f : 1.f) * (yo ? 0.5f : 1.f);
            cube[small_idx(s, pk)] = fmaf(wdl, rhs[k], acc);
        }
        __syncthreads();
        float T[kMarchPts];
#pragma unroll
        for (int i = 0; i < kMarchPts; ++i) {
            const int k = t + i * NT;
            if (k < n) {
                const float* f = cube + small_idx(s, __ldg(off + k));
                T[i] = fmaf(-wd, small_lap(A, f, s.plane, s.pitch), fmaf(wdl, rhs[k], f[0]));
            }
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < kMarchPts; ++i) {
            const int k = t + i * NT;
            if (k < n) cube[small_idx(s, __ldg(off + k))] = T[i];
        }
        __syncthreads();
    }
}

// Shared-memory places: level l's plane buffers, its extra buffer (the sums to
// restrict, or the staged planes of the level below) and rings, each per group;
// the thread's own place for staged inputs.
__device__ __forceinline__ int march_buf(const MarchLv& L, const MarchGroup& g) { return L.sm + g.index() * 2 * L.planef; }
__device__ __forceinline__ int march_extra(const MarchLv& L, const MarchGroup& g) { return L.sm_x + g.index() * L.xfloats; }
__device__ __forceinline__ int march_stage(const MarchLv& L, const MarchGroup& g) { return L.stage + g.index() * 16 * g.nthr + 4 * g.t; }
__device__ __forceinline__ unsigned march_ring(const MarchGeo& M) { return ring_of_warp((unsigned)si(M.sm_op + 28)); }

// The passes of level l (0: the PE ball), out of line: each has the registers
// to itself. The operator comes from shared memory, three 16-byte loads a step
// in place of ten registers. it picks level 0's buffers: r and p alternate
// between two where the ball is marched by more than one group.
__device__ __forceinline__ float4* hot_slot(const SolveParams& P) {
    return reinterpret_cast<float4*>(P.ws_hot + (size_t)blockIdx.x * P.hot_bytes);
}

template <int NT>
static __device__ __noinline__ float pass_r(const SolveParams& P, const MarchGeo& M, int l, float al, int it) {
    const MarchLv& L = M.lv[l];
    const MarchGroup g = march_groups(L);
    const bool two = L.groups > 1;
    MarchDown dn;
    dn.rhs = l + 1 < M.nm ? M.lv[l + 1].rhs_off : -1;
    const MarchSmall& s = M.sl[M.nm];
    dn.org = s.cube + s.org;
    dn.plane = s.plane;
    dn.pitch = s.pitch;
    return march_r<march_row(NT)>(M.sm_op, P.mg_wd32[0], L, M.lv[l + 1], dn, g, march_buf(L, g), march_extra(L, g), march_ring(M),
                   march_stage(L, g), hot_slot(P), l ? L.rhs_off : (kMarchR + (two && it > 0 ? (it - 1) & 1 : 0)) * 2 * march_row(NT),
                   (kMarchR + (two ? it & 1 : 0)) * 2 * march_row(NT),
                   al, l == 0 && it > 0);
}

template <int NT>
static __device__ __noinline__ float pass_z(const SolveParams& P, const MarchGeo& M, int l, int it) {
    const MarchLv& L = M.lv[l];
    const MarchGroup g = march_groups(L);
    MarchUp u;
    if (l + 1 < M.nm) {
        const MarchLv& N = M.lv[l + 1];
        u.quads = N.z_off;
        u.cube = march_extra(L, g);
        u.org = N.org;
        u.plane = N.planef;
        u.pitch = N.pitch;
        u.R = N.R;
    } else {
        const MarchSmall& s = M.sl[l + 1];
        u.quads = -1;
        u.cube = s.cube;
        u.org = s.org;
        u.plane = s.plane;
        u.pitch = s.pitch;
        u.R = s.R;
    }
    return march_z<march_row(NT)>(M.sm_op, P.mg_wd32[0], L, M.lv[l + 1], u, g, march_buf(L, g), march_ring(M), march_stage(L, g), hot_slot(P),
                   l ? L.rhs_off : (kMarchR + (L.groups > 1 ? it & 1 : 0)) * 2 * march_row(NT),
                   l ? L.z_off : kMarchZ * 2 * march_row(NT), P.mg_wd32[l]);
}

template <int NT>
static __device__ __noinline__ float pass_p(const SolveParams& P, const MarchGeo& M, float be, float al, int it) {
    const MarchLv& L = M.lv[0];
    const MarchGroup g = march_groups(L);
    const bool two = L.groups > 1;
    return march_p<march_row(NT)>(M.sm_op, L, g, march_buf(L, g), march_ring(M), march_stage(L, g), march_extra(L, g) + 4 * g.t, hot_slot(P),
                   (kMarchP + (two ? it & 1 : 0)) * 2 * march_row(NT), (kMarchP + (two ? (it + 1) & 1 : 0)) * 2 * march_row(NT), be,
                   al, it);
}

template <int NT>
__device__ __forceinline__ void zero_floats(int at, int n) {  // multiples of 4
    for (int k = 4 * threadIdx.x; k < n; k += 4 * NT) s4(at + k) = f4zero();
}

// The V-cycle below level 0: on entry level 1's right-hand side is complete
// (and visible); on return its correction is. Marching coarse levels work in
// the space of level 0's buffers, idle meanwhile, whose planes are zero again
// on return.
template <int NT>
__device__ __noinline__ void march_coarse(const SolveParams& P, const MarchGeo& M, const MGGeo& MG) {
    if (M.nm > 1) {
        zero_floats<NT>(0, M.coarse_floats);
        __syncthreads();
    }
    for (int l = 1; l < M.nm; ++l) {
        pass_r<NT>(P, M, l, 0.f, 0);
        __syncthreads();
    }
    march_small<NT>(P, M, MG);
    for (int l = M.nm - 1; l >= 1; --l) {
        pass_z<NT>(P, M, l, 0);
        __syncthreads();
    }
    if (M.nm > 1) {
        zero_floats<NT>(0, M.planes_floats);
        __syncthreads();
    }
}

// Zeroes the shared memory of ball M and writes its plane starts and level 0's
// operator -lap (the other levels' are powers of 4 of it): legs 1, 2, 3 along x
// (each twice), along y (twice), along z and the centre; then the rings'
// address in tensor memory.
template <int NT>
__device__ __forceinline__ void march_init(const SolveParams& P, const MarchGeo& M, unsigned ring) {
    if (threadIdx.x == 0) {
        const Stencil<float>& S = P.mg_a32[0];
        s4(M.sm_op) = make_float4(S.cx[0], S.cx[0], S.cx[1], S.cx[1]);
        s4(M.sm_op + 4) = make_float4(S.cx[2], S.cx[2], 0.f, 0.f);
        s4(M.sm_op + 12) = make_float4(S.cy[0], S.cy[0], S.cy[1], S.cy[1]);
        s4(M.sm_op + 16) = make_float4(S.cy[2], S.cy[2], 0.f, 0.f);
        s4(M.sm_op + 24) = make_float4(S.cz[0], S.cz[1], S.cz[2], S.c0);
        si(M.sm_op + 28) = (int)ring;
    }
    zero_floats<NT>(0, M.smem_zero);
    for (int l = 0; l <= M.nm; ++l)
        for (int k = threadIdx.x; k < 2 * M.lv[l].R + 1; k += NT) si(M.lv[l].sm_pst + k) = __ldg(M.lv[l].pst + k);
}

}  // namespace exx
