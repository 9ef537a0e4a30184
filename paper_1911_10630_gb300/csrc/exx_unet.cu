// exx_unet.cu -- the learned CG warm start: a 3D U-Net that maps the pair
// density rho_ij on a cube around the pair centre to a guess of v_ij.
//
// The paper starts each CG from a guess and names better guesses as the way to
// fewer iterations (Sec. III.C Step IV and the conclusions); the network is
// this library's own addition. Four levels (widths 16/32/64/128), two 3x3x3
// convolutions per level with ReLU, 2x2x2 average pooling down, nearest
// up-sampling and concatenation with the skip tensor up, a 1x1x1 head.
// Activations and weights are BF16 in channels-last layout, accumulation FP32.
//
// The 3x3x3 convolutions (all but the 3-channel input layer) are implicit GEMMs
// on the tcgen05 tensor cores: persistent CTAs, one per SM, compute 16 (H) x 8 (W)
// x DT (D) output tiles of a slice of the output channels. The input halo tile and
// the weights of one 16-channel chunk are staged in shared memory as 8-row core
// matrices, and each of the 27 taps is one MMA (M = 128 voxels, N = the slice,
// K = 16; three depth taps in one for up to 32 channels) whose A operand is the same
// staged tile seen through a shifted descriptor. The up-path layers read the
// up-sampled and the skip tensor in place of a concatenated one. The accumulators
// live in tensor memory and are read back with tcgen05.ld for the bias / ReLU / mask
// epilogue.
#include "exx_unet.cuh"
#include "exx_unet_tc.cuh"
#include "exx_phases.cuh"  // the multipole constants (this unit's copy of c_mp)

#include <algorithm>
#include <cmath>
#include <cstring>

namespace exx {
namespace unet {

namespace {

constexpr int kTH = 16, kTW = 8, kHH = kTH + 2, kWW = kTW + 2;
constexpr int kWaitLimit = 1 << 22;

__device__ __forceinline__ float bf2f(__nv_bfloat16 v) { return __bfloat162float(v); }
__device__ __forceinline__ __nv_bfloat16 f2bf(float v) { return __float2bfloat16_rn(v); }

constexpr int kStages = 4;
struct ConvArgs {
    const __nv_bfloat16* x;
    const __nv_bfloat16* low;  // the first cl input channels come from here, at half the resolution (cl = 0: none)
    const __nv_bfloat16* wp;
    const float* bias;
    const __nv_bfloat16* mask;
    __nv_bfloat16* y;
    int B, D, H, W, cin, cl, cout;
    int nb, nsplit;  // output channels per tile: nb of cout, nsplit slices
    int epi, DT, ncols, acc_cols, n_acc, n_stage;
    int fold;  // the three depth taps of a (dh, dw) in one MMA of N = 3 cout (depth-shifted TMEM slices)
    int tiles_d, tiles_h, tiles_w, n_tiles;
    int resident;  // all weights stay in shared memory
    uint32_t itile, wtile, stage;
    int* err;
};

// Persistent CTAs, one per SM, each over the tiles t, t + grid, ...: warps 0-7
// empty the accumulators (epilogue), one thread of warp 8 issues the MMAs, warps
// 9-16 stage the input halo tiles and weights. A unit is one 16-channel chunk of a
// tile; units pass through n_stage shared-memory stages (full / empty barriers),
// tiles through n_acc accumulators in tensor memory. One CTA per tile that staged,
// multiplied and stored in turn left the tensor cores 5 to 10 % busy: the 13
// convolutions of 32 cubes of 48 took 2.36 ms; with cheaper staging and two CTAs a
// SM 1.2; like this 0.85.
constexpr int kEpilogue = 256, kProducers = 256, kConvThreads = kEpilogue + 32 + kProducers;

// Index: of a voxel within a sample, long long for samples beyond 2^31 elements (in the
// staging warps, whose address arithmetic then costs 2 % of the forward pass).
template <typename Index>
__global__ void __launch_bounds__(kConvThreads, 1) conv3_tc_kernel(const __grid_constant__ ConvArgs a) {
    extern __shared__ unsigned char smem_dyn[];
    __shared__ uint64_t full[kStages], empty[kStages], acc_full[2], acc_empty[2], wres;
    __shared__ uint32_t s_tmem;
    __shared__ __align__(16) float s_bias[256];
    unsigned char* base =
        reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_dyn) + 127) & ~uintptr_t(127));
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int DT = a.DT, nch = a.cin / 16, NS = a.n_stage, NA = a.n_acc;
    if (tid == 0) {
        for (int s = 0; s < kStages; ++s) {
            tc::mbar_init(&full[s], kProducers / 32 + (a.resident ? 0 : 1));
            tc::mbar_init(&empty[s], 1);
        }
        for (int s = 0; s < 2; ++s) {
            tc::mbar_init(&acc_full[s], 1);
            tc::mbar_init(&acc_empty[s], kEpilogue);
        }
        tc::mbar_init(&wres, 1);
        tc::mbar_init_fence();
    }
    for (int i = tid; i < a.cout; i += kConvThreads) s_bias[i] = a.bias ? a.bias[i] : 0.0f;
    if (warp == 0) tc::tmem_alloc(&s_tmem, (uint32_t)a.ncols);
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tbase = s_tmem;
    if (a.fold) {  // every slice accumulates from several MMAs: start from zero
        if (warp < 4) {  // a warp reaches the 32 lanes of its number modulo 4
            for (int c0 = 0; c0 < a.ncols; c0 += 16) tc::tmem_st16_zero(tbase + ((uint32_t)(warp * 32) << 16) + c0);
            tc::tmem_wait_st();
        }
        tc::fence_before_sync();
        __syncthreads();
        tc::fence_after_sync();
    }
    unsigned char* stages = base + (a.resident ? (size_t)nch * a.wtile : 0);
    // tile t: w fastest, then h, d, sample, slice of the output channels
    const auto place = [&](int t, int& b, int& d0, int& h0, int& w0, int& n0) {
        w0 = t % a.tiles_w * kTW;
        t /= a.tiles_w;
        h0 = t % a.tiles_h * kTH;
        t /= a.tiles_h;
        d0 = t % a.tiles_d * DT;
        t /= a.tiles_d;
        b = t % a.B;
        n0 = t / a.B * a.nb;
    };
    bool ok = true;
    if (warp > kEpilogue / 32) {  // staging
        const int pt = tid - kEpilogue - 32, items = (DT + 2) * kHH * kWW * 2;
        const bool delay = NS >= 3;
        const auto finish = [&](int s) {
            tc::fence_proxy_async();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&full[s]);
        };
        if (a.resident && pt == 0) {
            tc::mbar_expect(&wres, (uint32_t)nch * a.wtile);
            for (int c = 0; c < nch; ++c)
                tc::bulk_load(base + (size_t)c * a.wtile, reinterpret_cast<const unsigned char*>(a.wp) + (size_t)c * a.wtile,
                              a.wtile, &wres);
        }
        int s = 0, k = 0, before = 0;
        uint32_t ph = 1;  // parity of the stage's last release
        for (int t = blockIdx.x; t < a.n_tiles && ok; t += gridDim.x) {
            int b, d0, h0, w0, n0;
            place(t, b, d0, h0, w0, n0);
            for (int c = 0; c < nch; ++c, ++k) {
                if (k >= NS) {
                    ok = __all_sync(0xffffffffu, tc::mbar_wait(&empty[s], ph, kWaitLimit));
                    if (!ok) break;
                }
                unsigned char* st = stages + (size_t)s * a.stage;
                if (!a.resident && pt == 0) {
                    // weights of chunk c: [27][cout/8][2][8][8] BF16
                    const unsigned char* src = reinterpret_cast<const unsigned char*>(a.wp) + (size_t)c * 27 * a.cout * 32;
                    unsigned char* dst = st + 2 * (size_t)a.itile;
                    tc::mbar_expect(&full[s], a.wtile);
                    if (a.nsplit == 1) {
                        tc::bulk_load(dst, src, a.wtile, &full[s]);
                    } else {
                        for (int tap = 0; tap < 27; ++tap)
                            tc::bulk_load(dst + (size_t)tap * a.nb * 32, src + ((size_t)tap * a.cout + n0) * 32,
                                          (uint32_t)a.nb * 32u, &full[s]);
                    }
                }
                // input halo tile: two channel octets, [DT+2][18][10] voxels x 16 B each
                const bool lo = c * 16 < a.cl;
                const int sh = lo ? 1 : 0, D = a.D >> sh, H = a.H >> sh, W = a.W >> sh;
                const int ch = lo ? a.cl : a.cin - a.cl;
                const __nv_bfloat16* xb =
                    (lo ? a.low : a.x) + (size_t)b * D * H * W * ch + (lo ? c * 16 : c * 16 - a.cl);
#pragma unroll 2
                for (int u = pt; u < items; u += kProducers) {
                    const int row = u / (2 * kWW), e = u - row * (2 * kWW), o = e & 1, wx = e >> 1;
                    const int dz = row / kHH, hy = row - dz * kHH;
                    const int d = d0 - 1 + dz, h = h0 - 1 + hy, w = w0 - 1 + wx;
                    const bool in =
                        (unsigned)d < (unsigned)a.D && (unsigned)h < (unsigned)a.H && (unsigned)w < (unsigned)a.W;
                    const __nv_bfloat16* src =
                        in ? xb + (size_t)(((Index)(d >> sh) * H + (h >> sh)) * W + (w >> sh)) * ch + o * 8 : a.x;
                    tc::cp_async16(st + (size_t)o * a.itile + (size_t)(row * kWW + wx) * 16, src, in ? 16u : 0u);
                }
                tc::cp_async_commit();
                if (!delay) {
                    tc::cp_async_wait<0>();
                    finish(s);
                } else if (k > 0) {  // one unit behind: its loads ran while this one's were issued
                    tc::cp_async_wait<1>();
                    finish(before);
                }
                before = s;
                if (++s == NS) {
                    s = 0;
                    ph ^= 1u;
                }
            }
        }
        if (delay && k > 0) {
            tc::cp_async_wait<0>();
            finish(before);
        }
    } else if (warp == kEpilogue / 32) {
        if (lane == 0) {
            const uint32_t idesc = tc::idesc_bf16_f32(128, a.fold ? 3 * a.nb : a.nb);
            const uint32_t bs = (uint32_t)(a.fold ? 3 : 1) * a.nb * 2;  // 16-byte words of weights per MMA
            if (a.resident && !tc::mbar_wait(&wres, 0, kWaitLimit)) ok = false;
            int s = 0, i = 0;
            uint32_t ph = 0;
            for (int t = blockIdx.x; t < a.n_tiles && ok; t += gridDim.x, ++i) {
                const int ab = NA == 2 ? i & 1 : 0;
                if (i >= NA && !tc::mbar_wait(&acc_empty[ab], (uint32_t)((i / NA - 1) & 1), kWaitLimit)) {
                    ok = false;
                    break;
                }
                const uint32_t acc = tbase + (uint32_t)(ab * a.acc_cols);
                for (int c = 0; c < nch; ++c) {
                    if (!tc::mbar_wait(&full[s], ph, kWaitLimit)) {
                        ok = false;
                        break;
                    }
                    tc::fence_after_sync();
                    unsigned char* st = stages + (size_t)s * a.stage;
                    const uint64_t ad0 = tc::sdesc(tc::smem_addr(st), a.itile, kWW * 16);
                    const uint64_t bd0 = tc::sdesc(
                        tc::smem_addr(a.resident ? base + (size_t)c * a.wtile : st + 2 * (size_t)a.itile), 128, 256);
                    if (a.fold) {
                        // input slice u (depth d0 - 1 + u) feeds the outputs tt = u - dz,
                        // dz = 2, 1, 0: TMEM slices u .. u + 2 (slice = tt + 2), with the
                        // weights of (dh, dw) packed as three N-blocks in that order
                        for (int u = 0; u < DT + 2; ++u) {
                            const uint64_t ad = ad0 + (uint32_t)(u * kHH * kWW);
#pragma unroll
                            for (int hw = 0; hw < 9; ++hw)
                                tc::mma_bf16(acc + (uint32_t)(u * a.nb), ad + (uint32_t)((hw / 3) * kWW + hw % 3),
                                             bd0 + hw * bs, idesc, 1u);
                        }
                    } else {
                        for (int tt = 0; tt < DT; ++tt) {
#pragma unroll 1
                            for (int dd = 0; dd < 3; ++dd) {
                                const uint64_t ad = ad0 + (uint32_t)((tt + dd) * kHH * kWW), bd = bd0 + dd * 9 * bs;
#pragma unroll
                                for (int hw = 0; hw < 9; ++hw)
                                    tc::mma_bf16(acc + (uint32_t)(tt * a.nb), ad + (uint32_t)((hw / 3) * kWW + hw % 3),
                                                 bd + hw * bs, idesc, (c > 0 || dd > 0 || hw > 0) ? 1u : 0u);
                            }
                        }
                    }
                    tc::commit(&empty[s]);
                    if (++s == NS) {
                        s = 0;
                        ph ^= 1u;
                    }
                }
                if (ok) tc::commit(&acc_full[ab]);
            }
        }
        __syncwarp();
    } else {
        const int m = (warp & 3) * 32 + lane;  // accumulator row = TMEM lane
        const uint32_t row = (uint32_t)((warp & 3) * 32) << 16;
        int i = 0;
        for (int t = blockIdx.x; t < a.n_tiles; t += gridDim.x, ++i) {
            int b, d0, h0, w0, n0;
            place(t, b, d0, h0, w0, n0);
            const int ab = NA == 2 ? i & 1 : 0;
            ok = __all_sync(0xffffffffu, tc::mbar_wait(&acc_full[ab], (uint32_t)((i / NA) & 1), kWaitLimit));
            if (!ok) break;
            tc::fence_after_sync();
            const uint32_t acc = tbase + row + (uint32_t)(ab * a.acc_cols + (a.fold ? 2 * a.nb : 0));
            const int h = h0 + (m >> 3), w = w0 + (m & 7);
            for (int tt = warp >> 2; tt < DT; tt += kEpilogue / 128) {
                const int d = d0 + tt;
                const bool live = d < a.D && h < a.H && w < a.W;
                const size_t vox = (((size_t)b * a.D + d) * a.H + h) * a.W + w;
                for (int c0 = 0; c0 < a.nb; c0 += 16) {
                    float v[16];
                    __syncwarp();
                    tc::tmem_ld16(acc + (uint32_t)(tt * a.nb + c0), v);
                    if (a.fold) tc::tmem_st16_zero(acc + (uint32_t)(tt * a.nb + c0));
                    if (!live) continue;
                    const size_t at = vox * a.cout + n0 + c0;
                    if (a.bias) {
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const float4 f = *reinterpret_cast<const float4*>(s_bias + n0 + c0 + 4 * k);
                            v[4 * k] += f.x;
                            v[4 * k + 1] += f.y;
                            v[4 * k + 2] += f.z;
                            v[4 * k + 3] += f.w;
                        }
                    }
                    if (a.epi == 1) {
#pragma unroll
                        for (int k = 0; k < 16; ++k) v[k] = fmaxf(v[k], 0.0f);
                    } else if (a.epi == 2) {
                        const uint4* mp = reinterpret_cast<const uint4*>(a.mask + at);
                        uint4 mm[2] = {mp[0], mp[1]};
                        const __nv_bfloat16* mb = reinterpret_cast<const __nv_bfloat16*>(mm);
#pragma unroll
                        for (int k = 0; k < 16; ++k) v[k] = bf2f(mb[k]) > 0.0f ? v[k] : 0.0f;
                    }
                    uint4 o[2];
                    __nv_bfloat16* ob = reinterpret_cast<__nv_bfloat16*>(o);
#pragma unroll
                    for (int k = 0; k < 16; ++k) ob[k] = f2bf(v[k]);
                    uint4* yp = reinterpret_cast<uint4*>(a.y + at);
                    yp[0] = o[0];
                    yp[1] = o[1];
                }
            }
            __syncwarp();
            if (a.fold) tc::tmem_wait_st();
            tc::fence_before_sync();
            tc::mbar_arrive(&acc_empty[ab]);
        }
    }
    ok = __syncthreads_and(ok);
    if (!ok && tid == 0) {
        atomicExch(a.err, 1);
        // let MMAs and copies still in flight finish before their memory goes back
        for (int s = 0; s < kStages; ++s) {
            tc::mbar_wait(&empty[s], 0, 256);
            tc::mbar_wait(&full[s], 0, 256);
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) tc::tmem_free(tbase, (uint32_t)a.ncols);
}

// ---- packing ---------------------------------------------------------------

// Packed operand: [K/16][27][N/8][2][8 n][8 k], k = 16 chunk + 8 half + e.
// Forward: K = cin, N = cout, value W[tap][k][n]. Data gradient (flip): the
// convolution maps cout -> cin channels, K = cout, N = cin, value
// W[26 - tap][n][k]. Depth-folded (fold): the 27 slots of a chunk are taken
// as [9 (dh, dw)][3], slot 3 hw + b holding the tap of depth offset dz = 2 - b.
__global__ void pack_kernel(const float* __restrict__ w, __nv_bfloat16* __restrict__ wp, int cin, int cout,
                            int flip, int fold) {
    const int K = flip ? cout : cin, N = flip ? cin : cout;
    const long long total = 27LL * K * N;
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
         idx += (long long)gridDim.x * blockDim.x) {
        long long r = idx;
        const int e = (int)(r % 8);
        r /= 8;
        const int nl = (int)(r % 8);
        r /= 8;
        const int half = (int)(r % 2);
        r /= 2;
        const int ng = (int)(r % (N / 8));
        r /= (N / 8);
        const int slot = (int)(r % 27);
        const int tap = fold ? (2 - slot % 3) * 9 + slot / 3 : slot;
        const int chunk = (int)(r / 27);
        const int k = chunk * 16 + half * 8 + e, n = ng * 8 + nl;
        const float v = flip ? w[((size_t)(26 - tap) * cin + n) * cout + k] : w[((size_t)tap * cin + k) * cout + n];
        wp[idx] = f2bf(v);
    }
}

// ---- CUDA-core layers ------------------------------------------------------

// Input layer: kIn FP32 channels -> 16, ReLU; S a multiple of 4. A thread makes 4
// voxels along x: a weight read from shared memory (broadcast) serves 4 FMAs and an
// input 48, which leaves the FMAs as the bound (1,296 a voxel: 0.12 ms on 32 cubes
// of 48; one voxel per thread took 0.42 ms, this 0.23).
// W16: in is 16-byte aligned (a caller's need not be).
template <bool W16>
__global__ void __launch_bounds__(128, 4) conv_first_kernel(const float* __restrict__ in, const float* __restrict__ w,
                                                         const float* __restrict__ bias, __nv_bfloat16* __restrict__ y,
                                                         int B, int S) {
    constexpr int CI = kIn;
    __shared__ __align__(16) float ws[27 * CI * 16 + 16];
    for (int i = threadIdx.x; i < 27 * CI * 16; i += blockDim.x) ws[i] = w[i];
    if (threadIdx.x < 16) ws[27 * CI * 16 + threadIdx.x] = bias[threadIdx.x];
    __syncthreads();
    const int S4 = S / 4;
    const long long nq = (long long)B * S * S * S4;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < nq; q += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(q % S4) * 4;
        const long long row = q / S4;  // (b S + z) S + y
        const int yy = (int)(row % S), z = (int)((row / S) % S);
        float acc[4][16];
#pragma unroll
        for (int c = 0; c < 16; ++c)
#pragma unroll
            for (int v = 0; v < 4; ++v) acc[v][c] = ws[27 * CI * 16 + c];
#pragma unroll 1
        for (int zy = 0; zy < 9; ++zy) {
            const int dz = zy / 3 - 1, dy = zy % 3 - 1;
            if (z + dz < 0 || z + dz >= S || yy + dy < 0 || yy + dy >= S) continue;
            const float* iv = in + ((row + dz * S + dy) * S + x) * CI;
            float a[6 * CI];  // voxels x - 1 .. x + 4
#pragma unroll
            for (int k = 0; k < CI; ++k) {
                float4 f;
                if constexpr (W16) f = *reinterpret_cast<const float4*>(iv + 4 * k);
                else f = make_float4(iv[4 * k], iv[4 * k + 1], iv[4 * k + 2], iv[4 * k + 3]);
                a[CI + 4 * k] = f.x;
                a[CI + 4 * k + 1] = f.y;
                a[CI + 4 * k + 2] = f.z;
                a[CI + 4 * k + 3] = f.w;
                a[k] = x > 0 ? iv[k - CI] : 0.0f;
                a[5 * CI + k] = x + 4 < S ? iv[4 * CI + k] : 0.0f;
            }
            const float4* wr = reinterpret_cast<const float4*>(ws + zy * 3 * CI * 16);
#pragma unroll
            for (int e = 0; e < 3 * CI; ++e)  // (dx, ci)
#pragma unroll
                for (int c4 = 0; c4 < 4; ++c4) {
                    const float4 f = wr[e * 4 + c4];
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
                        acc[v][4 * c4 + 0] = fmaf(a[v * CI + e], f.x, acc[v][4 * c4 + 0]);
                        acc[v][4 * c4 + 1] = fmaf(a[v * CI + e], f.y, acc[v][4 * c4 + 1]);
                        acc[v][4 * c4 + 2] = fmaf(a[v * CI + e], f.z, acc[v][4 * c4 + 2]);
                        acc[v][4 * c4 + 3] = fmaf(a[v * CI + e], f.w, acc[v][4 * c4 + 3]);
                    }
                }
        }
        uint4* yp = reinterpret_cast<uint4*>(y + (row * S + x) * 16);
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            uint4 o[2];
            __nv_bfloat16* ob = reinterpret_cast<__nv_bfloat16*>(o);
#pragma unroll
            for (int c = 0; c < 16; ++c) ob[c] = f2bf(fmaxf(acc[v][c], 0.0f));
            yp[2 * v] = o[0];
            yp[2 * v + 1] = o[1];
        }
    }
}

// 1x1x1 head: out = b + sum_c y0[c] w[c] (FP32).
__global__ void head_kernel(const __nv_bfloat16* __restrict__ y0, const float* __restrict__ hw, float* __restrict__ out,
                            long long nv) {
    for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < nv;
         v += (long long)gridDim.x * blockDim.x) {
        const uint4* p = reinterpret_cast<const uint4*>(y0 + v * 16);
        uint4 q[2] = {p[0], p[1]};
        const __nv_bfloat16* qb = reinterpret_cast<const __nv_bfloat16*>(q);
        float acc = hw[16];
#pragma unroll
        for (int c = 0; c < 16; ++c) acc = fmaf(bf2f(qb[c]), hw[c], acc);
        out[v] = acc;
    }
}

// Loss L = sum_v m_v (out_v - t_v)^2 / (B S^3), m_v = input mask channel; the
// head's gradients, and the gradient at y0 masked by ReLU (y0 > 0). Each block
// writes its partial sums (16 weights, bias, loss) to part[block][18]; they are
// added in block order by reduce_parts_kernel, so the result does not depend
// on the order in which blocks run.
__global__ void head_backward_kernel(const float* __restrict__ in, const float* __restrict__ target,
                                     const float* __restrict__ out, const __nv_bfloat16* __restrict__ y0,
                                     const float* __restrict__ hw, __nv_bfloat16* __restrict__ g_y0,
                                     float* __restrict__ part, long long nv, float inv_n) {
    __shared__ float red[17][8];
    float lsum = 0.0f, gw[17];
#pragma unroll
    for (int c = 0; c < 17; ++c) gw[c] = 0.0f;
    for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < nv;
         v += (long long)gridDim.x * blockDim.x) {
        const float m = in[kIn * v + kMaskChannel] > 0.5f ? 1.0f : 0.0f;
        const float diff = out[v] - target[v];
        lsum += m * diff * diff;
        const float g = 2.0f * m * diff * inv_n;
        const uint4* p = reinterpret_cast<const uint4*>(y0 + v * 16);
        uint4 q[2] = {p[0], p[1]};
        const __nv_bfloat16* qb = reinterpret_cast<const __nv_bfloat16*>(q);
        uint4 o[2];
        __nv_bfloat16* ob = reinterpret_cast<__nv_bfloat16*>(o);
#pragma unroll
        for (int c = 0; c < 16; ++c) {
            const float yv = bf2f(qb[c]);
            gw[c] = fmaf(g, yv, gw[c]);
            ob[c] = f2bf(yv > 0.0f ? g * hw[c] : 0.0f);
        }
        gw[16] += g;
        uint4* gp = reinterpret_cast<uint4*>(g_y0 + v * 16);
        gp[0] = o[0];
        gp[1] = o[1];
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int c = 0; c < 17; ++c) {
        float s = gw[c];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) red[c][wid] = s;
    }
    for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
    __shared__ float lred[8];
    if (lane == 0) lred[wid] = lsum;
    __syncthreads();
    float* mine = part + (size_t)blockIdx.x * 18;
    if (threadIdx.x < 17) {
        float s = 0.0f;
        for (int k = 0; k < (int)(blockDim.x >> 5); ++k) s += red[threadIdx.x][k];
        mine[threadIdx.x] = s;
    }
    if (threadIdx.x == 32) {
        float s = 0.0f;
        for (int k = 0; k < (int)(blockDim.x >> 5); ++k) s += lred[k];
        mine[17] = s * inv_n;
    }
}

// out[i] = sum over s of part[s * stride + i], s < n_parts (the fixed-order
// second stage of every gradient and loss reduction): 32 outputs to a block, K
// threads to an output, thread k adding the parts k, k + K, ...; the K
// sums are added in order. One thread per output left a chain of up to 2,432 loads
// (190 us; 14 now, for the head's 18 values).
template <int K>
__global__ void __launch_bounds__(32 * K) reduce_parts_kernel(const float* __restrict__ part, int n_parts,
                                                            long long stride, int count, float* __restrict__ out) {
    __shared__ float sum[K][33];
    const int i = blockIdx.x * 32 + threadIdx.x;
    float s = 0.0f;
    if (i < count) {
#pragma unroll 4
        for (int k = threadIdx.y; k < n_parts; k += K) s += __ldg(part + (size_t)k * stride + i);
    }
    sum[threadIdx.y][threadIdx.x] = s;
    __syncthreads();
    if (threadIdx.y == 0 && i < count) {
        float t = 0.0f;
#pragma unroll
        for (int k = 0; k < K; ++k) t += sum[k][threadIdx.x];
        out[i] = t;
    }
}
cudaError_t reduce_parts(const float* part, int n_parts, long long stride, int count, float* out, cudaStream_t st) {
    // 32 threads an output only for long chains (19 parts of 442,000 outputs: 56 us with
    // 32 threads, 20 with 4); 8 up to 128 parts
    if (n_parts > 128) reduce_parts_kernel<32><<<(count + 31) / 32, dim3(32, 32), 0, st>>>(part, n_parts, stride, count, out);
    else reduce_parts_kernel<8><<<(count + 31) / 32, dim3(32, 8), 0, st>>>(part, n_parts, stride, count, out);
    return cudaGetLastError();
}

// 2x2x2 average pooling, channels last; one thread per (coarse voxel, 8 channels).
__global__ void pool_kernel(const __nv_bfloat16* __restrict__ x, __nv_bfloat16* __restrict__ y, int B, int S, int C) {
    const int s = S / 2, g8 = C / 8;
    const long long total = (long long)B * s * s * s * g8;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x) {
        const int g = (int)(i % g8);
        long long p = i / g8;
        const int px = (int)(p % s), py = (int)((p / s) % s), pz = (int)((p / ((long long)s * s)) % s);
        const long long bb = p / ((long long)s * s * s);
        float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        for (int k = 0; k < 8; ++k) {
            const long long v = ((bb * S + 2 * pz + (k >> 2)) * S + 2 * py + ((k >> 1) & 1)) * S + 2 * px + (k & 1);
            const uint4 q = *reinterpret_cast<const uint4*>(x + v * C + g * 8);
            const __nv_bfloat16* qb = reinterpret_cast<const __nv_bfloat16*>(&q);
#pragma unroll
            for (int c = 0; c < 8; ++c) acc[c] += bf2f(qb[c]);
        }
        uint4 o;
        __nv_bfloat16* ob = reinterpret_cast<__nv_bfloat16*>(&o);
#pragma unroll
        for (int c = 0; c < 8; ++c) ob[c] = f2bf(0.125f * acc[c]);
        *reinterpret_cast<uint4*>(y + p * C + g * 8) = o;
    }
}

// Gradient at the up-sampled input: dlow[p] = sum over the 8 children of
// dcat[child][0:Cl], masked by ReLU (low > 0).
__global__ void upcat_back_low_kernel(const __nv_bfloat16* __restrict__ dcat, const __nv_bfloat16* __restrict__ low,
                                      __nv_bfloat16* __restrict__ dlow, int B, int S, int Cl, int Cs) {
    const int C = Cl + Cs, s = S / 2, g8 = Cl / 8;
    const long long total = (long long)B * s * s * s * g8;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x) {
        const int g = (int)(i % g8);
        const long long p = i / g8;
        const int px = (int)(p % s), py = (int)((p / s) % s), pz = (int)((p / ((long long)s * s)) % s);
        const long long bb = p / ((long long)s * s * s);
        float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        for (int k = 0; k < 8; ++k) {
            const long long v = ((bb * S + 2 * pz + (k >> 2)) * S + 2 * py + ((k >> 1) & 1)) * S + 2 * px + (k & 1);
            const uint4 q = *reinterpret_cast<const uint4*>(dcat + v * C + g * 8);
            const __nv_bfloat16* qb = reinterpret_cast<const __nv_bfloat16*>(&q);
#pragma unroll
            for (int c = 0; c < 8; ++c) acc[c] += bf2f(qb[c]);
        }
        const uint4 lq = *reinterpret_cast<const uint4*>(low + p * Cl + g * 8);
        const __nv_bfloat16* lb = reinterpret_cast<const __nv_bfloat16*>(&lq);
        uint4 o;
        __nv_bfloat16* ob = reinterpret_cast<__nv_bfloat16*>(&o);
#pragma unroll
        for (int c = 0; c < 8; ++c) ob[c] = f2bf(bf2f(lb[c]) > 0.0f ? acc[c] : 0.0f);
        *reinterpret_cast<uint4*>(dlow + p * Cl + g * 8) = o;
    }
}

// Gradient at a skip tensor: from the pooling (dpool[parent] / 8) and from the
// concatenation (dcat[v][Cl:]), masked by ReLU (skip > 0).
__global__ void skip_back_kernel(const __nv_bfloat16* __restrict__ dpool, const __nv_bfloat16* __restrict__ dcat,
                                 const __nv_bfloat16* __restrict__ skip, __nv_bfloat16* __restrict__ dskip, int B,
                                 int S, int Cl, int Cs) {
    const int C = Cl + Cs, s = S / 2, g8 = Cs / 8;
    const long long total = (long long)B * S * S * S * g8;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x) {
        const int g = (int)(i % g8);
        const long long v = i / g8;
        const int x = (int)(v % S), y = (int)((v / S) % S), z = (int)((v / ((long long)S * S)) % S);
        const long long bb = v / ((long long)S * S * S);
        const long long p = ((bb * s + z / 2) * s + y / 2) * s + x / 2;
        const uint4 a = *reinterpret_cast<const uint4*>(dpool + p * Cs + g * 8);
        const uint4 c = *reinterpret_cast<const uint4*>(dcat + v * C + Cl + g * 8);
        const uint4 k = *reinterpret_cast<const uint4*>(skip + v * Cs + g * 8);
        const __nv_bfloat16 *ab = reinterpret_cast<const __nv_bfloat16*>(&a),
                            *cb = reinterpret_cast<const __nv_bfloat16*>(&c),
                            *kb = reinterpret_cast<const __nv_bfloat16*>(&k);
        uint4 o;
        __nv_bfloat16* ob = reinterpret_cast<__nv_bfloat16*>(&o);
#pragma unroll
        for (int e = 0; e < 8; ++e) ob[e] = f2bf(bf2f(kb[e]) > 0.0f ? 0.125f * bf2f(ab[e]) + bf2f(cb[e]) : 0.0f);
        *reinterpret_cast<uint4*>(dskip + v * Cs + g * 8) = o;
    }
}

// Weight gradient of a 3x3x3 layer, dW[tap][ci][co] = sum over samples and
// voxels of x[v + tap - 1][ci] g[v][co], on the tensor cores: with K the voxels, A =
// x^T (16 ci) seen through the tap's shift and B = g (NB co), both read from their
// [voxel][channel] tiles by transposing matrix loads. tcgen05 takes M of 64 or 128
// rows under one address, which 16 channels a tap do not make; mma.sync's 16 x 8 x
// 16 fits them. A block stages voxel tiles (4 x 4 x 8: a 6 x 6 x 10 halo of x, the
// first cl channels from low at half the resolution, and the tile of g; BF16, rows
// padded so that 8 of them lie in distinct banks) through two buffers; warp (dz, dy)
// holds the sums of its three taps. The products are exact; a tile's 128 are summed
// in the tensor core from zero and the tiles' sums added in FP32, so that chains
// are shorter than one FMA per voxel. Grid: x = tile split (split s takes the tiles
// [s T / nsplit, (s + 1) T / nsplit)), y = ci block, z = co block; each split
// writes its sums to its own slice of part ([split][27 cin cout + cout]). The FMAs
// took 5.4 ms on 32 cubes of 32; this 0.7.
constexpr int kDwD = 4, kDwH = 4, kDwW = 8, kDwVox = kDwD * kDwH * kDwW;
constexpr int kDwHD = kDwD + 2, kDwHH = kDwH + 2, kDwHW = kDwW + 2, kDwHalo = kDwHD * kDwHH * kDwHW;
constexpr int kDwThreads = 9 * 32;
constexpr int kDwXRow = 48;  // bytes of a voxel's 16 channels and padding
constexpr int dw_grow(int nb) { return 2 * nb + 16; }
constexpr int dw_stage(int nb) { return kDwHalo * kDwXRow + kDwVox * dw_grow(nb); }
constexpr int dw_nb(int cout) { return cout % 32 ? 16 : 32; }

template <int NB>
__global__ void __launch_bounds__(kDwThreads) dw_kernel(const __nv_bfloat16* __restrict__ x,
                                                        const __nv_bfloat16* __restrict__ low, int cl,
                                                        const __nv_bfloat16* __restrict__ g,
                                                        float* __restrict__ part, int B, int S, int cin, int cout,
                                                        int nsplit) {
    extern __shared__ __align__(16) unsigned char dw_smem[];
    constexpr int GROW = dw_grow(NB), NJ = NB / 8, P = kDwThreads / NB;
    const int cib = blockIdx.y, cob = blockIdx.z, split = blockIdx.x;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int dz = warp / 3, dy = warp % 3;
    const int td = (S + kDwD - 1) / kDwD, th = (S + kDwH - 1) / kDwH, tw = (S + kDwW - 1) / kDwW;
    const long long T = (long long)B * td * th * tw;
    const long long t0 = T * split / nsplit, t1 = T * (split + 1) / nsplit;
    const bool lo = cib * 16 < cl;
    const int sh = lo ? 1 : 0, Sx = S >> sh, ch = lo ? cl : cin - cl;
    const __nv_bfloat16* xc = lo ? low + cib * 16 : x + cib * 16 - cl;
    const auto stage = [&](long long t, int buf) {
        long long r = t;
        const int w0 = (int)(r % tw) * kDwW;
        r /= tw;
        const int h0 = (int)(r % th) * kDwH;
        r /= th;
        const int d0 = (int)(r % td) * kDwD;
        const int b = (int)(r / td);
        unsigned char* xs = dw_smem + buf * dw_stage(NB);
        unsigned char* gs = xs + kDwHalo * kDwXRow;
        for (int u = tid; u < 2 * kDwHalo; u += kDwThreads) {
            const int half = u & 1, vx = u >> 1;
            const int d = d0 - 1 + vx / (kDwHH * kDwHW), h = h0 - 1 + (vx / kDwHW) % kDwHH, w = w0 - 1 + vx % kDwHW;
            const bool in = (unsigned)d < (unsigned)S && (unsigned)h < (unsigned)S && (unsigned)w < (unsigned)S;
            const __nv_bfloat16* src =
                in ? xc + ((((long long)b * Sx + (d >> sh)) * Sx + (h >> sh)) * Sx + (w >> sh)) * ch + half * 8 : x;
            tc::cp_async16(xs + vx * kDwXRow + half * 16, src, in ? 16u : 0u);
        }
        for (int u = tid; u < kDwVox * NJ; u += kDwThreads) {
            const int o = u % NJ, vx = u / NJ;
            const int d = d0 + vx / (kDwH * kDwW), h = h0 + (vx / kDwW) % kDwH, w = w0 + vx % kDwW;
            const bool in = d < S && h < S && w < S;
            const __nv_bfloat16* src =
                in ? g + ((((long long)b * S + d) * S + h) * S + w) * cout + cob * NB + o * 8 : g;
            tc::cp_async16(gs + vx * GROW + o * 16, src, in ? 16u : 0u);
        }
        tc::cp_async_commit();
    };
    float sum[3][NJ][4], bsum = 0.0f;
#pragma unroll
    for (int i = 0; i < 3 * NJ * 4; ++i) (&sum[0][0][0])[i] = 0.0f;
    // lane's row of the transposing loads: voxel w = lane & 7 of tile row 2 ks + hi
    const int xrow = lane >> 4, xcol = ((lane >> 3) & 1) * 16;
    const int grow = (lane >> 3) & 1, gcol = (lane >> 4) * 16;
    const uint32_t base = tc::smem_addr(dw_smem);
    if (t0 < t1) stage(t0, 0);
    for (long long t = t0; t < t1; ++t) {
        const int buf = (int)((t - t0) & 1);
        if (t + 1 < t1) {
            stage(t + 1, buf ^ 1);
            tc::cp_async_wait<1>();
        } else {
            tc::cp_async_wait<0>();
        }
        __syncthreads();
        const uint32_t xs = base + buf * dw_stage(NB), gs = xs + kDwHalo * kDwXRow;
        float c[3][NJ][4];
#pragma unroll
        for (int i = 0; i < 3 * NJ * 4; ++i) (&c[0][0][0])[i] = 0.0f;
#pragma unroll
        for (int ks = 0; ks < kDwVox / 16; ++ks) {
            const int rx = 2 * ks + xrow, rg = 2 * ks + grow;
            uint32_t bf[NJ / 2][4];
#pragma unroll
            for (int j = 0; j < NJ / 2; ++j)
                tc::ldmatrix4_trans(gs + (rg * kDwW + (lane & 7)) * GROW + gcol + j * 32, bf[j]);
#pragma unroll
            for (int dx = 0; dx < 3; ++dx) {
                uint32_t af[4];
                tc::ldmatrix4_trans(
                    xs + (((rx / kDwH + dz) * kDwHH + rx % kDwH + dy) * kDwHW + (lane & 7) + dx) * kDwXRow + xcol, af);
#pragma unroll
                for (int j = 0; j < NJ; ++j)
                    tc::mma16816(c[dx][j], af, bf[j / 2][(j & 1) * 2], bf[j / 2][(j & 1) * 2 + 1]);
            }
        }
#pragma unroll
        for (int i = 0; i < 3 * NJ * 4; ++i) (&sum[0][0][0])[i] += (&c[0][0][0])[i];
        if (cib == 0 && tid < P * NB) {
            const unsigned char* gp = dw_smem + buf * dw_stage(NB) + kDwHalo * kDwXRow + (tid % NB) * 2;
            for (int vx = tid / NB; vx < kDwVox; vx += P)
                bsum += bf2f(*reinterpret_cast<const __nv_bfloat16*>(gp + vx * GROW));
        }
        __syncthreads();  // the buffer is staged again
    }
    float* dw = part + (size_t)split * ((size_t)27 * cin * cout + cout);
#pragma unroll
    for (int dx = 0; dx < 3; ++dx)
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
            float* row = dw + ((size_t)(warp * 3 + dx) * cin + cib * 16 + (lane >> 2)) * cout + cob * NB + j * 8 + (lane & 3) * 2;
            row[0] = sum[dx][j][0];
            row[1] = sum[dx][j][1];
            row[(size_t)8 * cout] = sum[dx][j][2];
            row[(size_t)8 * cout + 1] = sum[dx][j][3];
        }
    if (cib == 0) {
        float* bs = reinterpret_cast<float*>(dw_smem);
        bs[tid] = bsum;
        __syncthreads();
        if (tid < NB) {
            float s = 0.0f;
            for (int p = 0; p < P; ++p) s += bs[p * NB + tid];
            dw[(size_t)27 * cin * cout + cob * NB + tid] = s;
        }
    }
}

// Weight gradient of the FP32 input layer: 27 x kIn x 16 weights and 16 biases,
// with dw_kernel's voxel tiles. A block stages a tile (the halo of in and the tile
// of g) and 4 groups of 81 threads (tap, ci) take 4 of its 16 rows each, 16 FMAs
// to one value of in and a broadcast row of g; 16 more threads add g up. Split s
// takes the tiles [s T / nsplit, (s + 1) T / nsplit); the groups' sums are added in
// order into part[s][27 kIn 16 + 16]. One thread per weight running over the
// voxels, its indices divided out of each, took 10.2 ms on a batch of 32 cubes of
// 32; this 0.2.
constexpr int kDwFirstTap = 27 * kIn, kDwFirstGroups = 4;
constexpr int kDwFirstThreads = (kDwFirstTap * kDwFirstGroups + 16 + 31) / 32 * 32;

__global__ void __launch_bounds__(kDwFirstThreads) dw_first_kernel(const float* __restrict__ in,
                                                                   const __nv_bfloat16* __restrict__ g,
                                                                   float* __restrict__ part, int B, int S, int nsplit) {
    constexpr int CI = kIn, NW = 27 * CI * 16, HW = kDwHW * CI;
    __shared__ float xs[kDwHD * kDwHH * HW];
    __shared__ __align__(16) float gs[kDwVox][16];
    __shared__ float sum[kDwFirstTap][17];
    const int tid = threadIdx.x;
    const int group = tid / kDwFirstTap, w = tid - group * kDwFirstTap;
    const int tap = w / CI, ci = w - tap * CI;
    const int dz = tap / 9, dy = (tap / 3) % 3, dx = tap % 3;
    const bool acc_thread = group < kDwFirstGroups;
    const int bias = tid - kDwFirstTap * kDwFirstGroups;  // 0 .. 15: adds g
    const int td = (S + kDwD - 1) / kDwD, th = (S + kDwH - 1) / kDwH, tw = (S + kDwW - 1) / kDwW;
    const long long T = (long long)B * td * th * tw;
    const long long t0 = T * blockIdx.x / nsplit, t1 = T * (blockIdx.x + 1) / nsplit;
    float acc[16], bacc = 0.0f;
#pragma unroll
    for (int k = 0; k < 16; ++k) acc[k] = 0.0f;
    for (long long t = t0; t < t1; ++t) {
        long long r = t;
        const int w0 = (int)(r % tw) * kDwW;
        r /= tw;
        const int h0 = (int)(r % th) * kDwH;
        r /= th;
        const int d0 = (int)(r % td) * kDwD;
        const int b = (int)(r / td);
        __syncthreads();  // the previous tile's values are no longer read
        for (int u = tid; u < kDwHD * kDwHH * HW; u += kDwFirstThreads) {
            const int row = u / HW, e = u - row * HW;
            const int d = d0 - 1 + row / kDwHH, h = h0 - 1 + row % kDwHH, x = w0 - 1 + e / CI;
            const bool live = d >= 0 && d < S && h >= 0 && h < S && x >= 0 && x < S;
            xs[u] = live ? in[((((long long)b * S + d) * S + h) * S + x) * CI + e % CI] : 0.0f;
        }
        for (int u = tid; u < 2 * kDwVox; u += kDwFirstThreads) {
            const int half = u & 1, vx = u >> 1;
            const int d = d0 + vx / (kDwH * kDwW), h = h0 + (vx / kDwW) % kDwH, x = w0 + vx % kDwW;
            uint4 q = make_uint4(0u, 0u, 0u, 0u);
            if (d < S && h < S && x < S)
                q = *reinterpret_cast<const uint4*>(g + ((((long long)b * S + d) * S + h) * S + x) * 16 + half * 8);
            const __nv_bfloat16* qb = reinterpret_cast<const __nv_bfloat16*>(&q);
#pragma unroll
            for (int e = 0; e < 8; ++e) gs[vx][half * 8 + e] = bf2f(qb[e]);
        }
        __syncthreads();
        if (acc_thread) {
#pragma unroll
            for (int q = 0; q < kDwD * kDwH / kDwFirstGroups; ++q) {
                const int row = group + q * kDwFirstGroups, vd = row / kDwH, vh = row % kDwH;
                const float* xrow = xs + ((vd + dz) * kDwHH + vh + dy) * HW + dx * CI + ci;
                const float4* grow = reinterpret_cast<const float4*>(gs[row * kDwW]);
#pragma unroll
                for (int vw = 0; vw < kDwW; ++vw) {
                    const float xv = xrow[vw * CI];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const float4 gq = grow[vw * 4 + k];
                        acc[4 * k + 0] = fmaf(xv, gq.x, acc[4 * k + 0]);
                        acc[4 * k + 1] = fmaf(xv, gq.y, acc[4 * k + 1]);
                        acc[4 * k + 2] = fmaf(xv, gq.z, acc[4 * k + 2]);
                        acc[4 * k + 3] = fmaf(xv, gq.w, acc[4 * k + 3]);
                    }
                }
            }
        } else if (bias < 16) {
            for (int vx = 0; vx < kDwVox; ++vx) bacc += gs[vx][bias];
        }
    }
    float* dw = part + (size_t)blockIdx.x * (NW + 16);
    for (int q = 0; q < kDwFirstGroups; ++q) {
        __syncthreads();
        if (acc_thread && group == q) {
#pragma unroll
            for (int k = 0; k < 16; ++k) sum[w][k] = q ? sum[w][k] + acc[k] : acc[k];
        }
    }
    __syncthreads();
    for (int u = tid; u < NW; u += kDwFirstThreads) dw[u] = sum[u / 16][u % 16];
    if (!acc_thread && bias < 16) dw[NW + bias] = bacc;
}

__global__ void adam_kernel(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                            float* __restrict__ v, long long n, float lr, float b1, float b2, float eps, float c1,
                            float c2) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.0f - b1) * gi;
        const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        p[i] -= lr * (mi * c1) / (sqrtf(vi * c2) + eps);
    }
}

__global__ void zero_f32_kernel(float* p, long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        p[i] = 0.0f;
}

int grid_for(long long n, int n_sm) {
    long long g = (n + 255) / 256;
    const long long cap = 16LL * n_sm;
    return (int)(g < 1 ? 1 : (g > cap ? cap : g));
}

#define UCK(x)                            \
    do {                                  \
        cudaError_t e_ = (x);             \
        if (e_ != cudaSuccess) return e_; \
    } while (0)

}  // namespace

size_t param_offset(int layer) {
    size_t off = 0;
    for (int l = 0; l < layer; ++l)
        off += (l == kHead ? (size_t)kCin[l] : (size_t)27 * kCin[l]) * kCout[l] + kCout[l];
    return off;
}
size_t param_count() { return param_offset(kLayers); }

// Whether a convolution with n_out output channels folds its depth taps (one
// MMA of N = 3 n_out per (dh, dw)): N <= 256 and the depth-shifted TMEM slices
// of a tile within 256 columns, so that two accumulators fit.
static bool conv_folds(int n_out) { return n_out <= 32; }

cudaError_t pack_weights(const float* w, __nv_bfloat16* wp, int cin, int cout, int flip, cudaStream_t st) {
    const long long total = 27LL * cin * cout;
    pack_kernel<<<(int)((total + 255) / 256), 256, 0, st>>>(w, wp, cin, cout, flip,
                                                            conv_folds(flip ? cin : cout) ? 1 : 0);
    return cudaGetLastError();
}

// As conv3_tc of the header, with the first cl of the cin channels from low
// (half the resolution, nearest up-sampling).
static cudaError_t conv3_up(const __nv_bfloat16* x, const __nv_bfloat16* low, int cl, const __nv_bfloat16* wp,
                            const float* bias, const __nv_bfloat16* mask, __nv_bfloat16* y, int B, int D, int H, int W,
                            int cin, int cout, int epi, int* err, int n_sm, cudaStream_t st) {
    if (cin % 16 || cout % 16 || cout < 16 || cout > 256 || B < 1) return cudaErrorInvalidValue;
    ConvArgs a;
    a.x = x;
    a.low = low;
    a.cl = cl;
    a.wp = wp;
    a.bias = bias;
    a.mask = mask;
    a.y = y;
    a.B = B;
    a.D = D;
    a.H = H;
    a.W = W;
    a.cin = cin;
    a.cout = cout;
    a.epi = epi;
    a.err = err;
    a.fold = conv_folds(cout) ? 1 : 0;
    // At most 64 output channels a tile: two stages with 27 taps of weights fit,
    // and the deepest level has tiles for all SMs.
    a.nsplit = 1;
    while (cout / a.nsplit > 64 || cout % (16 * a.nsplit)) ++a.nsplit;
    // 80, 112, 176 and 208 have no even split but slices of 16, each of which would stage
    // the input again: one slice and one stage (exx_unet_conv3d, 112 to 112 channels on
    // 3 x 200 x 200: 0.26 ms, 0.51 in slices).
    if (cout / a.nsplit < 32 && cout > 64) a.nsplit = 1;
    a.nb = cout / a.nsplit;
    a.wtile = 27u * (uint32_t)a.nb * 32u;
    a.tiles_w = (W + kTW - 1) / kTW;
    a.tiles_h = (H + kTH - 1) / kTH;
    const size_t room = 227 * 1024 - 4096;
    const int nch = cin / 16;
    a.resident = a.nsplit == 1 && (size_t)nch * a.wtile <= 64 * 1024;
    // Depth of the tiles: the deeper, the less halo per output; the shallower, the
    // evener the SMs' shares. The cost (clocks) of a chunk is its MMAs' (an operand
    // read of 4 KB or N / 2 columns each) or its staging's, whichever is longer.
    const int most = a.fold ? (cout <= 16 ? 8 : 4) : 4;
    double best = 0.0;
    long long tiles = 0;
    for (int DT = 1; DT <= most && DT <= D && (a.fold || DT * a.nb <= 512); ++DT) {
        const long long n = (long long)a.tiles_w * a.tiles_h * ((D + DT - 1) / DT) * B * a.nsplit;
        const double mma = (a.fold ? 9.0 * (DT + 2) : 27.0 * DT) * std::max(40.0, 0.55 * a.nb * (a.fold ? 3 : 1));
        const double load = 110.0 * (DT + 2) + (a.resident ? 0.0 : a.wtile / 64.0);
        const double cost = (double)((n + n_sm - 1) / n_sm) * (nch * std::max(mma, load) + 1000.0);
        if (DT == 1 || cost < best) {
            best = cost;
            a.DT = DT;
            tiles = n;
        }
    }
    if (tiles > 0x7fffffffLL) return cudaErrorInvalidValue;
    a.n_tiles = (int)tiles;
    a.tiles_d = (D + a.DT - 1) / a.DT;
    a.acc_cols = (a.DT + (a.fold ? 4 : 0)) * a.nb;
    a.n_acc = 2 * a.acc_cols <= 512 ? 2 : 1;
    a.ncols = 32;
    while (a.ncols < a.n_acc * a.acc_cols) a.ncols *= 2;
    a.itile = (uint32_t)(a.DT + 2) * kHH * kWW * 16;
    a.stage = 2 * a.itile + (a.resident ? 0u : a.wtile);
    const size_t fixed = a.resident ? (size_t)nch * a.wtile : 0;
    a.n_stage = (int)std::min<size_t>(kStages, (room - fixed) / a.stage);
    if (a.n_stage < 1 || a.ncols > 512) return cudaErrorInvalidValue;
    const size_t smem = fixed + (size_t)a.n_stage * a.stage + 128;
    const auto kernel = (long long)D * H * W * cin > 0x7fffffffLL ? conv3_tc_kernel<long long> : conv3_tc_kernel<int>;
    UCK(raise_smem_limit((const void*)kernel, smem));
    kernel<<<std::min(a.n_tiles, n_sm), kConvThreads, smem, st>>>(a);
    return cudaGetLastError();
}

cudaError_t conv3_tc(const __nv_bfloat16* x, const __nv_bfloat16* wp, const float* bias, const __nv_bfloat16* mask,
                     __nv_bfloat16* y, int B, int D, int H, int W, int cin, int cout, int epi, int* err, int n_sm,
                     cudaStream_t st) {
    return conv3_up(x, nullptr, 0, wp, bias, mask, y, B, D, H, W, cin, cout, epi, err, n_sm, st);
}

// ---- network driver --------------------------------------------------------

// Voxel-tile splits of a weight-gradient launch: about four blocks per SM over
// the (ci, co) blocks, and no split without a tile.
static int dw_splits(int B, int S, int cin, int cout, int n_sm) {
    const long long tiles = (long long)B * ((S + kDwD - 1) / kDwD) * ((S + kDwH - 1) / kDwH) * ((S + kDwW - 1) / kDwW);
    const long long cb = (long long)(cin / 16) * (cout / dw_nb(cout));
    const long long want = std::max(1LL, 4LL * n_sm / cb);
    return (int)std::max(1LL, std::min(tiles, want));
}

cudaError_t create(Net& n, int S, int Bmax) {
    n.S = S;
    n.Bmax = Bmax;
    int dev = 0;
    UCK(cudaGetDevice(&dev));
    UCK(cudaDeviceGetAttribute(&n.n_sm, cudaDevAttrMultiProcessorCount, dev));
    n.nparam = param_count();
    auto alloc = [&](void** p, size_t bytes) -> cudaError_t {
        cudaError_t e = cudaMalloc(p, bytes);
        if (e == cudaSuccess) n.bufs.push_back(*p);
        return e;
    };
    UCK(alloc((void**)&n.params, n.nparam * 4));
    UCK(alloc((void**)&n.grads, n.nparam * 4));
    UCK(alloc((void**)&n.adam_m, n.nparam * 4));
    UCK(alloc((void**)&n.adam_v, n.nparam * 4));
    UCK(cudaMemset(n.adam_m, 0, n.nparam * 4));
    UCK(cudaMemset(n.adam_v, 0, n.nparam * 4));
    UCK(cudaMemset(n.params, 0, n.nparam * 4));
    for (int l = 1; l < kHead; ++l) {
        const size_t e = (size_t)27 * kCin[l] * kCout[l] * sizeof(__nv_bfloat16);
        UCK(alloc((void**)&n.wfwd[l], e));
        UCK(alloc((void**)&n.wbwd[l], e));
    }
    const size_t v0 = (size_t)Bmax * S * S * S, v1 = v0 / 8, v2 = v1 / 8, v3 = v2 / 8;
    auto act = [&](__nv_bfloat16** p, size_t vox, int C) { return alloc((void**)p, vox * C * 2); };
    UCK(act(&n.x0a, v0, 16));
    UCK(act(&n.x0, v0, 16));
    UCK(act(&n.p0, v1, 16));
    UCK(act(&n.x1a, v1, 32));
    UCK(act(&n.x1, v1, 32));
    UCK(act(&n.p1, v2, 32));
    UCK(act(&n.x2a, v2, 64));
    UCK(act(&n.x2, v2, 64));
    UCK(act(&n.p2, v3, 64));
    UCK(act(&n.x3a, v3, 128));
    UCK(act(&n.x3, v3, 128));
    UCK(act(&n.y2a, v2, 64));
    UCK(act(&n.y2, v2, 64));
    UCK(act(&n.y1a, v1, 32));
    UCK(act(&n.y1, v1, 32));
    UCK(act(&n.y0a, v0, 16));
    UCK(act(&n.y0, v0, 16));
    UCK(act(&n.g_y0, v0, 16));
    UCK(act(&n.g_y0a, v0, 16));
    UCK(act(&n.g_c0, v0, 48));
    UCK(act(&n.g_y1, v1, 32));
    UCK(act(&n.g_y1a, v1, 32));
    UCK(act(&n.g_c1, v1, 96));
    UCK(act(&n.g_y2, v2, 64));
    UCK(act(&n.g_y2a, v2, 64));
    UCK(act(&n.g_c2, v2, 192));
    UCK(act(&n.g_x3, v3, 128));
    UCK(act(&n.g_x3a, v3, 128));
    UCK(act(&n.g_p2, v3, 64));
    UCK(act(&n.g_x2, v2, 64));
    UCK(act(&n.g_x2a, v2, 64));
    UCK(act(&n.g_p1, v2, 32));
    UCK(act(&n.g_x1, v1, 32));
    UCK(act(&n.g_x1a, v1, 32));
    UCK(act(&n.g_p0, v1, 16));
    UCK(act(&n.g_x0, v0, 16));
    UCK(act(&n.g_x0a, v0, 16));
    UCK(alloc((void**)&n.out, v0 * 4));
    // partial sums of the gradient reductions: the largest of the head's
    // per-block sums, the input layer's and every 3x3x3 layer's per-split sums
    {
        size_t need = (size_t)18 * 16 * n.n_sm;
        need = std::max(need, (size_t)4 * n.n_sm * (27 * kIn * 16 + 16));
        const int lvl[kLayers] = {0, 0, 1, 1, 2, 2, 3, 3, 2, 2, 1, 1, 0, 0, 0};
        for (int l = 1; l < kHead; ++l)
            need = std::max(need, (size_t)dw_splits(Bmax, S >> lvl[l], kCin[l], kCout[l], n.n_sm) *
                                      ((size_t)27 * kCin[l] * kCout[l] + kCout[l]));
        UCK(alloc((void**)&n.gpart, need * 4));
    }
    UCK(alloc((void**)&n.d_loss, 4));
    UCK(alloc((void**)&n.d_err, 4));
    UCK(cudaMemset(n.d_err, 0, 4));
    return cudaSuccess;
}

void destroy(Net& n) {
    for (void* p : n.bufs) cudaFree(p);
    n.bufs.clear();
}

cudaError_t pack(Net& n, cudaStream_t st) {
    for (int l = 1; l < kHead; ++l) {
        const float* w = n.params + param_offset(l);
        UCK(pack_weights(w, n.wfwd[l], kCin[l], kCout[l], 0, st));
        UCK(pack_weights(w, n.wbwd[l], kCin[l], kCout[l], 1, st));
    }
    n.packed = true;
    return cudaSuccess;
}

static const float* bias_of(const Net& n, int l) { return n.params + param_offset(l) + (size_t)27 * kCin[l] * kCout[l]; }

cudaError_t forward(Net& n, const float* in, int B, cudaStream_t st) {
    if (B < 1 || B > n.Bmax) return cudaErrorInvalidValue;
    if (!n.packed) UCK(pack(n, st));
    const int S = n.S, S1 = S / 2, S2 = S / 4, S3 = S / 8;
    const long long v0 = (long long)B * S * S * S, v1 = v0 / 8, v2 = v1 / 8, v3 = v2 / 8;
    auto conv_up = [&](const __nv_bfloat16* x, const __nv_bfloat16* low, int cl, __nv_bfloat16* y, int l, int s) {
        return conv3_up(x, low, cl, n.wfwd[l], bias_of(n, l), nullptr, y, B, s, s, s, kCin[l], kCout[l], 1, n.d_err,
                        n.n_sm, st);
    };
    auto conv = [&](const __nv_bfloat16* x, __nv_bfloat16* y, int l, int s) { return conv_up(x, nullptr, 0, y, l, s); };
    const auto first = reinterpret_cast<uintptr_t>(in) % 16 ? conv_first_kernel<false> : conv_first_kernel<true>;
    first<<<(unsigned)((v0 / 4 + 127) / 128), 128, 0, st>>>(in, n.params, bias_of(n, 0), n.x0a, B, S);
    UCK(cudaGetLastError());
    UCK(conv(n.x0a, n.x0, 1, S));
    pool_kernel<<<grid_for(v1 * 2, n.n_sm), 256, 0, st>>>(n.x0, n.p0, B, S, 16);
    UCK(conv(n.p0, n.x1a, 2, S1));
    UCK(conv(n.x1a, n.x1, 3, S1));
    pool_kernel<<<grid_for(v2 * 4, n.n_sm), 256, 0, st>>>(n.x1, n.p1, B, S1, 32);
    UCK(conv(n.p1, n.x2a, 4, S2));
    UCK(conv(n.x2a, n.x2, 5, S2));
    pool_kernel<<<grid_for(v3 * 8, n.n_sm), 256, 0, st>>>(n.x2, n.p2, B, S2, 64);
    UCK(conv(n.p2, n.x3a, 6, S3));
    UCK(conv(n.x3a, n.x3, 7, S3));
    UCK(conv_up(n.x2, n.x3, 128, n.y2a, 8, S2));
    UCK(conv(n.y2a, n.y2, 9, S2));
    UCK(conv_up(n.x1, n.y2, 64, n.y1a, 10, S1));
    UCK(conv(n.y1a, n.y1, 11, S1));
    UCK(conv_up(n.x0, n.y1, 32, n.y0a, 12, S));
    UCK(conv(n.y0a, n.y0, 13, S));
    head_kernel<<<grid_for(v0, n.n_sm), 256, 0, st>>>(n.y0, n.params + param_offset(kHead), n.out, v0);
    return cudaGetLastError();
}

cudaError_t backward(Net& n, const float* in, const float* target, int B, cudaStream_t st) {
    const int S = n.S, S1 = S / 2, S2 = S / 4, S3 = S / 8;
    const long long v0 = (long long)B * S * S * S, v1 = v0 / 8, v2 = v1 / 8, v3 = v2 / 8;
    zero_f32_kernel<<<grid_for((long long)n.nparam, n.n_sm), 256, 0, st>>>(n.grads, (long long)n.nparam);
    {
        const int nblk = grid_for(v0, n.n_sm);
        float* ghw = n.grads + param_offset(kHead);
        head_backward_kernel<<<nblk, 256, 0, st>>>(in, target, n.out, n.y0, n.params + param_offset(kHead), n.g_y0,
                                                   n.gpart, v0, 1.0f / (float)v0);
        UCK(reduce_parts(n.gpart, nblk, 18, 17, ghw, st));
        UCK(reduce_parts(n.gpart + 17, nblk, 18, 1, n.d_loss, st));
    }
    UCK(cudaGetLastError());
    // data gradient through layer l: from g (cout channels) to cin channels,
    // masked by ReLU of the layer's input when that input is a ReLU output
    auto dconv = [&](const __nv_bfloat16* g, const __nv_bfloat16* xmask, __nv_bfloat16* dx, int l, int s) {
        return conv3_tc(g, n.wbwd[l], nullptr, xmask, dx, B, s, s, s, kCout[l], kCin[l], xmask ? 2 : 0, n.d_err,
                        n.n_sm, st);
    };
    auto dweight_up = [&](const __nv_bfloat16* x, const __nv_bfloat16* low, int cl, const __nv_bfloat16* g, int l, int s) {
        const int nsplit = dw_splits(B, s, kCin[l], kCout[l], n.n_sm);
        const int nb = dw_nb(kCout[l]), smem = 2 * dw_stage(nb);
        const auto f = nb == 16 ? dw_kernel<16> : dw_kernel<32>;
        UCK(raise_smem_limit((const void*)f, smem));
        dim3 grid(nsplit, kCin[l] / 16, kCout[l] / nb);
        const int count = 27 * kCin[l] * kCout[l] + kCout[l];
        f<<<grid, kDwThreads, smem, st>>>(x, low, cl, g, n.gpart, B, s, kCin[l], kCout[l], nsplit);
        UCK(cudaGetLastError());
        return reduce_parts(n.gpart, nsplit, count, count, n.grads + param_offset(l), st);
    };
    auto dweight = [&](const __nv_bfloat16* x, const __nv_bfloat16* g, int l, int s) {
        return dweight_up(x, nullptr, 0, g, l, s);
    };
    // level 0, up path
    UCK(dweight(n.y0a, n.g_y0, 13, S));
    UCK(dconv(n.g_y0, n.y0a, n.g_y0a, 13, S));
    UCK(dweight_up(n.x0, n.y1, 32, n.g_y0a, 12, S));
    UCK(dconv(n.g_y0a, nullptr, n.g_c0, 12, S));
    upcat_back_low_kernel<<<grid_for(v1 * 4, n.n_sm), 256, 0, st>>>(n.g_c0, n.y1, n.g_y1, B, S, 32, 16);
    // level 1, up path
    UCK(dweight(n.y1a, n.g_y1, 11, S1));
    UCK(dconv(n.g_y1, n.y1a, n.g_y1a, 11, S1));
    UCK(dweight_up(n.x1, n.y2, 64, n.g_y1a, 10, S1));
    UCK(dconv(n.g_y1a, nullptr, n.g_c1, 10, S1));
    upcat_back_low_kernel<<<grid_for(v2 * 8, n.n_sm), 256, 0, st>>>(n.g_c1, n.y2, n.g_y2, B, S1, 64, 32);
    // level 2, up path
    UCK(dweight(n.y2a, n.g_y2, 9, S2));
    UCK(dconv(n.g_y2, n.y2a, n.g_y2a, 9, S2));
    UCK(dweight_up(n.x2, n.x3, 128, n.g_y2a, 8, S2));
    UCK(dconv(n.g_y2a, nullptr, n.g_c2, 8, S2));
    upcat_back_low_kernel<<<grid_for(v3 * 16, n.n_sm), 256, 0, st>>>(n.g_c2, n.x3, n.g_x3, B, S2, 128, 64);
    // bottleneck
    UCK(dweight(n.x3a, n.g_x3, 7, S3));
    UCK(dconv(n.g_x3, n.x3a, n.g_x3a, 7, S3));
    UCK(dweight(n.p2, n.g_x3a, 6, S3));
    UCK(dconv(n.g_x3a, nullptr, n.g_p2, 6, S3));
    // level 2, down path
    skip_back_kernel<<<grid_for(v2 * 8, n.n_sm), 256, 0, st>>>(n.g_p2, n.g_c2, n.x2, n.g_x2, B, S2, 128, 64);
    UCK(dweight(n.x2a, n.g_x2, 5, S2));
    UCK(dconv(n.g_x2, n.x2a, n.g_x2a, 5, S2));
    UCK(dweight(n.p1, n.g_x2a, 4, S2));
    UCK(dconv(n.g_x2a, nullptr, n.g_p1, 4, S2));
    // level 1, down path
    skip_back_kernel<<<grid_for(v1 * 4, n.n_sm), 256, 0, st>>>(n.g_p1, n.g_c1, n.x1, n.g_x1, B, S1, 64, 32);
    UCK(dweight(n.x1a, n.g_x1, 3, S1));
    UCK(dconv(n.g_x1, n.x1a, n.g_x1a, 3, S1));
    UCK(dweight(n.p0, n.g_x1a, 2, S1));
    UCK(dconv(n.g_x1a, nullptr, n.g_p0, 2, S1));
    // level 0, down path
    skip_back_kernel<<<grid_for(v0 * 2, n.n_sm), 256, 0, st>>>(n.g_p0, n.g_c0, n.x0, n.g_x0, B, S, 32, 16);
    UCK(dweight(n.x0a, n.g_x0, 1, S));
    UCK(dconv(n.g_x0, n.x0a, n.g_x0a, 1, S));
    {
        const int nsplit = 4 * n.n_sm;
        const int count = 27 * kIn * 16 + 16;
        dw_first_kernel<<<nsplit, kDwFirstThreads, 0, st>>>(in, n.g_x0a, n.gpart, B, S, nsplit);
        UCK(cudaGetLastError());
        UCK(reduce_parts(n.gpart, nsplit, count, count, n.grads + param_offset(0), st));
    }
    return cudaGetLastError();
}

cudaError_t adam_step(Net& n, float lr, cudaStream_t st) {
    n.adam_t += 1;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.0f / (1.0f - std::pow(b1, (float)n.adam_t));
    const float c2 = 1.0f / (1.0f - std::pow(b2, (float)n.adam_t));
    adam_kernel<<<grid_for((long long)n.nparam, n.n_sm), 256, 0, st>>>(n.params, n.grads, n.adam_m, n.adam_v,
                                                                      (long long)n.nparam, lr, b1, b2, 1e-8f, c1, c2);
    UCK(cudaGetLastError());
    return pack(n, st);
}

cudaError_t check_error(Net& n, cudaStream_t st) {
    int h = 0;
    UCK(cudaMemcpyAsync(&h, n.d_err, 4, cudaMemcpyDeviceToHost, st));
    UCK(cudaStreamSynchronize(st));
    return h ? cudaErrorLaunchTimeout : cudaSuccess;
}

}  // namespace unet
}  // namespace exx

namespace exx {
namespace unet {

// ---- pair samples ------------------------------------------------------------

namespace {


// Index of the Cartesian monomial x^a y^b z^c, l = a + b + c, in the
// library's order (degree ascending, then a descending, then b descending).
__host__ __device__ constexpr int mono_index(int a, int b, int c) {
    return (a + b + c) * (a + b + c + 1) * (a + b + c + 2) / 6 + (b + c) * (b + c + 1) / 2 + c;
}

// One network sample per pair (one CTA of 256 threads per pair):
//   channel 0: rho / s on the PE ball (s = max |rho| there), 0 elsewhere;
//   channel 1: on the cube outside the PE ball, the multipole expansion of
//     Eq. me evaluated from the moments of rho / s on the ball (Eq. mepole,
//     l <= lmax; FP32, Cartesian form with the library's K_l matrices), over
//     delta^2: the boundary values the solver imposes, in the target's units;
//   channel 2: the ball mask;
// and with vcache the target v / (s delta^2) on the ball.
__global__ void __launch_bounds__(256) sample_prep_kernel(const double* __restrict__ phi, int N0, int N1, int N2,
                                                          const PairRec* __restrict__ pairs, int k0, int S,
                                                          const BallGeo G, float* __restrict__ input,
                                                          float* __restrict__ scale, float* __restrict__ target,
                                                          const float* __restrict__ vcache, double d2, float dx,
                                                          float dy, float dz, float dV, int lmax,
                                                          const int* __restrict__ box_org, int3 bdim,
                                                          long long ostride) {
    constexpr int NM = kNMono;
    __shared__ double red[8];
    __shared__ float s_Mw[8][NM];
    __shared__ float s_M[NM], s_T[NM];
    const int k = k0 + blockIdx.x;
    const PairRec pr = pairs[k];
    const double* pi = phi + (long long)pr.i * ostride;
    const double* pj = phi + (long long)pr.j * ostride;
    const int N[3] = {N0, N1, N2}, bd[3] = {bdim.x, bdim.y, bdim.z};
    // rho at offset o of the pair's grid point (zero where o leaves a box)
    auto rho_at = [&](int ox, int oy, int oz) -> double {
        const int packed = (ox + 128) | ((oy + 128) << 8) | ((oz + 128) << 16);
        const long long ii = orb_index(N, pr.g, packed, box_org, bd, pr.i);
        const long long ij = orb_index(N, pr.g, packed, box_org, bd, pr.j);
        return (ii >= 0 && ij >= 0) ? pi[ii] * pj[ij] : 0.0;
    };
    const int R = G.r_pe, h = S / 2, S3 = S * S * S;
    double mx = 0.0;
    for (int v = threadIdx.x; v < S3; v += blockDim.x) {
        const int ox = v / (S * S) - h, oy = (v / S) % S - h, oz = v % S - h;
        if (ox * ox + oy * oy + oz * oz > R * R) continue;
        mx = fmax(mx, fabs(rho_at(ox, oy, oz)));
    }
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
    __syncthreads();
    double s = red[0];
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) s = fmax(s, red[w]);
    if (!(s > 0.0)) s = 1.0;
    const double inv = 1.0 / s, tinv = 1.0 / (s * d2);
    float* in = input + (size_t)blockIdx.x * S3 * kIn;
    float* tg = target ? target + (size_t)blockIdx.x * S3 : nullptr;
    const float* vc = vcache ? vcache + (size_t)k * G.n_pe : nullptr;
    const int W = 2 * R + 1;
    for (int v = threadIdx.x; v < S3; v += blockDim.x) {
        const int ox = v / (S * S) - h, oy = (v / S) % S - h, oz = v % S - h;
        float r = 0.0f, m = 0.0f, t = 0.0f;
        if (ox * ox + oy * oy + oz * oz <= R * R) {
            r = (float)(rho_at(ox, oy, oz) * inv);
            m = 1.0f;
            if (tg && vc) {
                const RowRec Rw = G.rows_pe[G.row_of[(ox + R) * W + (oy + R)]];
                t = (float)(vc[Rw.pe_start + oz + Rw.zpe] * tinv);
            }
        }
        in[kIn * v] = r;
        in[kIn * v + 1] = 0.0f;
        in[kIn * v + kMaskChannel] = m;
        if (tg) tg[v] = t;
    }
    if (threadIdx.x == 0) scale[blockIdx.x] = (float)s;
    __syncthreads();

    // Moments M_abc = sum rho/s x^a y^b z^c dV over the ball points of the
    // cube: one thread per cube row (x, y), row sums S_c = sum_z rho/s z^c,
    // then every monomial; per-thread partials added in a fixed order.
    float M[NM];
#pragma unroll
    for (int q = 0; q < NM; ++q) M[q] = 0.0f;
    for (int row = threadIdx.x; row < S * S; row += blockDim.x) {
        const int ox = row / S - h, oy = row % S - h;
        const int rem = R * R - ox * ox - oy * oy;
        if (rem < 0) continue;
        int zr = (int)sqrtf((float)rem);
        while ((zr + 1) * (zr + 1) <= rem) ++zr;
        while (zr * zr > rem) --zr;
        const int zlo = max(-zr, -h), zhi = min(zr, h - 1);
        float sc[kLmaxMax + 1];
#pragma unroll
        for (int c = 0; c <= kLmaxMax; ++c) sc[c] = 0.0f;
        const float* rp = in + (size_t)row * S * kIn;
        for (int z = zlo; z <= zhi; ++z) {
            float p = rp[(z + h) * kIn];
            const float zz = (float)z * dz;
#pragma unroll
            for (int c = 0; c <= kLmaxMax; ++c) {
                sc[c] += p;
                p *= zz;
            }
        }
        float xa[kLmaxMax + 1], yb[kLmaxMax + 1];
        xa[0] = yb[0] = 1.0f;
#pragma unroll
        for (int e = 1; e <= kLmaxMax; ++e) {
            xa[e] = xa[e - 1] * ((float)ox * dx);
            yb[e] = yb[e - 1] * ((float)oy * dy);
        }
#pragma unroll
        for (int l = 0; l <= kLmaxMax; ++l)
#pragma unroll
            for (int a = l; a >= 0; --a)
#pragma unroll
                for (int b = l - a; b >= 0; --b) {
                    const int c = l - a - b;
                    M[mono_index(a, b, c)] = fmaf(xa[a] * yb[b], sc[c], M[mono_index(a, b, c)]);
                }
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int q = 0; q < NM; ++q) {
        float v = M[q];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) s_Mw[wid][q] = v;
    }
    __syncthreads();
    if (threadIdx.x < NM) {
        const int q = threadIdx.x;
        float t = 0.0f;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += s_Mw[w][q];
        const int l = c_mp.mono[q][0] + c_mp.mono[q][1] + c_mp.mono[q][2];
        s_M[q] = l <= lmax ? t * dV : 0.0f;
    }
    __syncthreads();
    // T = K M (the polynomials P_l of the expansion, K_l from the host tables)
    if (threadIdx.x < NM) {
        const int q = threadIdx.x;
        const int l = c_mp.mono[q][0] + c_mp.mono[q][1] + c_mp.mono[q][2];
        const int nl = (l + 1) * (l + 2) / 2, r0 = c_mp.mono_off[l];
        const double* Kr = c_mp.K + c_mp.k_off[l] + (q - r0) * nl;
        float acc = 0.0f;
        for (int t = 0; t < nl; ++t) acc = fmaf((float)Kr[t], s_M[r0 + t], acc);
        s_T[q] = acc;
    }
    __syncthreads();
    // channel 1 on the cube points outside the ball: v = sum_l P_l / r^(2l+1),
    // with P_l = sum_c U_{l,c}(x, y) z^c formed once per row
    const float id2 = (float)(1.0 / d2);
    for (int row = threadIdx.x; row < S * S; row += blockDim.x) {
        const int ox = row / S - h, oy = row % S - h;
        const int rxy = ox * ox + oy * oy;
        if (rxy + h * h <= R * R) continue;  // the whole row inside the ball
        const float x = (float)ox * dx, y = (float)oy * dy;
        float xa[kLmaxMax + 1], yb[kLmaxMax + 1];
        xa[0] = yb[0] = 1.0f;
#pragma unroll
        for (int e = 1; e <= kLmaxMax; ++e) {
            xa[e] = xa[e - 1] * x;
            yb[e] = yb[e - 1] * y;
        }
        float U[kNU];
#pragma unroll
        for (int l = 0; l <= kLmaxMax; ++l)
#pragma unroll
            for (int c = 0; c <= l; ++c) {
                float u = 0.0f;
#pragma unroll
                for (int a = l - c; a >= 0; --a) u = fmaf(s_T[mono_index(a, l - c - a, c)], xa[a] * yb[l - c - a], u);
                U[l * (l + 1) / 2 + c] = u;
            }
        const float rxy2 = x * x + y * y;
        float* rp = in + (size_t)row * S * kIn;
        for (int z = -h; z < h; ++z) {
            if (rxy + z * z <= R * R) continue;
            const float zz = (float)z * dz;
            const float ir = rsqrtf(fmaf(zz, zz, rxy2));
            const float ir2 = ir * ir;
            float acc = 0.0f;
#pragma unroll
            for (int l = kLmaxMax; l >= 0; --l) {
                float pl = U[l * (l + 1) / 2 + l];
#pragma unroll
                for (int c = l - 1; c >= 0; --c) pl = fmaf(pl, zz, U[l * (l + 1) / 2 + c]);
                acc = fmaf(acc, ir2, pl);
            }
            rp[(z + h) * kIn + 1] = acc * ir * id2;
        }
    }
}

__global__ void __launch_bounds__(256) guess_scatter_kernel(const float* __restrict__ out,
                                                            const float* __restrict__ scale, int k0, int S,
                                                            const BallGeo G, double d2, float* __restrict__ vguess) {
    const int b = blockIdx.x, h = S / 2, S3 = S * S * S;
    const float f = (float)(scale[b] * d2);
    const float* o = out + (size_t)b * S3;
    float* vg = vguess + (size_t)(k0 + b) * G.n_pe;
    for (int p = threadIdx.x; p < G.n_pe; p += blockDim.x) {
        const int pk = G.pt_off[p];
        const int ox = (pk & 255) - 128 + h, oy = ((pk >> 8) & 255) - 128 + h, oz = ((pk >> 16) & 255) - 128 + h;
        float v = 0.0f;
        if (ox >= 0 && ox < S && oy >= 0 && oy < S && oz >= 0 && oz < S) v = o[(ox * S + oy) * S + oz] * f;
        vg[p] = v;
    }
}

}  // namespace

cudaError_t sample_prep(const double* phi, const int N[3], const PairRec* pairs, int k0, int nk, int S,
                        const BallGeo& G, float* input, float* scale, float* target, const float* vcache, double d2,
                        const double delta[3], double dV, int lmax, const int* box_org, const int bdim[3],
                        long long ostride, cudaStream_t st) {
    if (nk <= 0) return cudaSuccess;
    sample_prep_kernel<<<nk, 256, 0, st>>>(phi, N[0], N[1], N[2], pairs, k0, S, G, input, scale, target, vcache, d2,
                                           (float)delta[0], (float)delta[1], (float)delta[2], (float)dV, lmax,
                                           box_org, make_int3(bdim[0], bdim[1], bdim[2]), ostride);
    return cudaGetLastError();
}

cudaError_t set_multipole_const_unet(const MultipoleConst& mc) {
    return cudaMemcpyToSymbol(c_mp, &mc, sizeof(MultipoleConst));
}

cudaError_t guess_scatter(const float* out, const float* scale, int k0, int nk, int S, const BallGeo& G, double d2,
                          float* vguess, cudaStream_t st) {
    if (nk <= 0) return cudaSuccess;
    guess_scatter_kernel<<<nk, 256, 0, st>>>(out, scale, k0, S, G, d2, vguess);
    return cudaGetLastError();
}

}  // namespace unet
}  // namespace exx

// ---- C ABI -----------------------------------------------------------------

#include "exx_guess.h"
#include <string>

namespace exx {
void set_global_error(const std::string& msg);  // defined in exx_api.cu
}

struct exx_guess {
    exx::unet::Net net;
};

namespace {

exx_status gfail(exx_status s, const std::string& m) {
    exx::set_global_error(m);
    return s;
}

exx_status gcuda(cudaError_t e, const char* what) {
    if (e == cudaSuccess) return EXX_OK;
    (void)cudaGetLastError();
    if (e == cudaErrorLaunchTimeout)
        return gfail(EXX_ECUDA, std::string(what) + ": a tensor-core wait timed out");
    return gfail(e == cudaErrorMemoryAllocation ? EXX_ENOMEM : EXX_ECUDA,
                 std::string(what) + ": " + cudaGetErrorString(e));
}

}  // namespace

extern "C" size_t exx_guess_param_count(void) { return exx::unet::param_count(); }

extern "C" exx_status exx_guess_create(exx_guess** out, int S, int batch_max) {
    if (!out) return gfail(EXX_EINVAL, "exx_guess_create: out is NULL");
    *out = nullptr;
    if (S < 16 || S > 64 || S % 8) return gfail(EXX_EINVAL, "exx_guess_create: S must be a multiple of 8 in [16, 64]");
    if (batch_max < 1 || batch_max > 1024) return gfail(EXX_EINVAL, "exx_guess_create: batch_max must be in [1, 1024]");
    exx_guess* g = new exx_guess();
    cudaError_t e = exx::unet::create(g->net, S, batch_max);
    if (e != cudaSuccess) {
        exx::unet::destroy(g->net);
        delete g;
        return gcuda(e, "exx_guess_create");
    }
    *out = g;
    return EXX_OK;
}

extern "C" exx_status exx_guess_set_params(exx_guess* g, const float* params, size_t n) {
    if (!g || !params) return gfail(EXX_EINVAL, "exx_guess_set_params: NULL argument");
    if (n != g->net.nparam) return gfail(EXX_EINVAL, "exx_guess_set_params: wrong parameter count");
    exx_status s = gcuda(cudaMemcpy(g->net.params, params, n * 4, cudaMemcpyHostToDevice), "exx_guess_set_params");
    if (s != EXX_OK) return s;
    g->net.packed = false;
    return gcuda(exx::unet::pack(g->net, nullptr), "exx_guess_set_params");
}

extern "C" exx_status exx_guess_get_params(exx_guess* g, float* params, size_t n) {
    if (!g || !params) return gfail(EXX_EINVAL, "exx_guess_get_params: NULL argument");
    if (n != g->net.nparam) return gfail(EXX_EINVAL, "exx_guess_get_params: wrong parameter count");
    return gcuda(cudaMemcpy(params, g->net.params, n * 4, cudaMemcpyDeviceToHost), "exx_guess_get_params");
}

extern "C" exx_status exx_guess_forward(exx_guess* g, const float* input, float* output, int batch, void* stream) {
    if (!g || !input || !output) return gfail(EXX_EINVAL, "exx_guess_forward: NULL argument");
    if (batch < 1 || batch > g->net.Bmax) return gfail(EXX_EINVAL, "exx_guess_forward: batch out of range");
    cudaStream_t st = (cudaStream_t)stream;
    exx_status s = gcuda(exx::unet::forward(g->net, input, batch, st), "exx_guess_forward");
    if (s != EXX_OK) return s;
    const size_t bytes = (size_t)batch * g->net.S * g->net.S * g->net.S * 4;
    s = gcuda(cudaMemcpyAsync(output, g->net.out, bytes, cudaMemcpyDeviceToDevice, st), "exx_guess_forward");
    if (s != EXX_OK) return s;
    return gcuda(exx::unet::check_error(g->net, st), "exx_guess_forward");
}

extern "C" exx_status exx_guess_gradient(exx_guess* g, const float* input, const float* target, int batch, float* loss,
                                         float* grad, void* stream) {
    if (!g || !input || !target) return gfail(EXX_EINVAL, "exx_guess_gradient: NULL argument");
    if (batch < 1 || batch > g->net.Bmax) return gfail(EXX_EINVAL, "exx_guess_gradient: batch out of range");
    cudaStream_t st = (cudaStream_t)stream;
    exx_status s = gcuda(exx::unet::forward(g->net, input, batch, st), "exx_guess_gradient");
    if (s == EXX_OK) s = gcuda(exx::unet::backward(g->net, input, target, batch, st), "exx_guess_gradient");
    if (s == EXX_OK) s = gcuda(exx::unet::check_error(g->net, st), "exx_guess_gradient");
    if (s == EXX_OK && loss)
        s = gcuda(cudaMemcpy(loss, g->net.d_loss, 4, cudaMemcpyDeviceToHost), "exx_guess_gradient");
    if (s == EXX_OK && grad)
        s = gcuda(cudaMemcpy(grad, g->net.grads, g->net.nparam * 4, cudaMemcpyDeviceToHost), "exx_guess_gradient");
    return s;
}

extern "C" exx_status exx_guess_train_step(exx_guess* g, const float* input, const float* target, int batch, float lr,
                                           float* loss, void* stream) {
    if (!g || !input || !target) return gfail(EXX_EINVAL, "exx_guess_train_step: NULL argument");
    if (batch < 1 || batch > g->net.Bmax) return gfail(EXX_EINVAL, "exx_guess_train_step: batch out of range");
    if (!(lr > 0.0f)) return gfail(EXX_EINVAL, "exx_guess_train_step: lr must be positive");
    cudaStream_t st = (cudaStream_t)stream;
    exx_status s = gcuda(exx::unet::forward(g->net, input, batch, st), "exx_guess_train_step");
    if (s == EXX_OK) s = gcuda(exx::unet::backward(g->net, input, target, batch, st), "exx_guess_train_step");
    if (s == EXX_OK) s = gcuda(exx::unet::adam_step(g->net, lr, st), "exx_guess_train_step");
    if (s == EXX_OK && loss)
        s = gcuda(cudaMemcpyAsync(loss, g->net.d_loss, 4, cudaMemcpyDeviceToHost, st), "exx_guess_train_step");
    if (s == EXX_OK) s = gcuda(exx::unet::check_error(g->net, st), "exx_guess_train_step");
    return s;
}

extern "C" void exx_guess_destroy(exx_guess* g) {
    if (!g) return;
    exx::unet::destroy(g->net);
    delete g;
}

extern "C" exx_status exx_unet_conv3d(const void* x, const float* w, const float* bias, const void* mask, void* y,
                                      int batch, int D, int H, int W, int cin, int cout, int mode, void* stream) {
    if (!x || !w || !y) return gfail(EXX_EINVAL, "exx_unet_conv3d: NULL argument");
    if (cin % 16 || cout % 16 || cin < 16 || cout < 16 || cin > 256 || cout > 256)
        return gfail(EXX_EINVAL, "exx_unet_conv3d: channels must be multiples of 16 in [16, 256]");
    if (batch < 1 || D < 1 || H < 1 || W < 1 || mode < 0 || mode > 2)
        return gfail(EXX_EINVAL, "exx_unet_conv3d: bad size or mode");
    cudaStream_t st = (cudaStream_t)stream;
    int dev = 0, nsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    __nv_bfloat16* wp = nullptr;
    int* err = nullptr;
    exx_status s = gcuda(cudaMalloc(&wp, (size_t)27 * cin * cout * 2), "exx_unet_conv3d");
    if (s == EXX_OK) s = gcuda(cudaMalloc(&err, 4), "exx_unet_conv3d");
    if (s == EXX_OK) s = gcuda(cudaMemsetAsync(err, 0, 4, st), "exx_unet_conv3d");
    const int flip = mode == 2 ? 1 : 0;
    if (s == EXX_OK) s = gcuda(exx::unet::pack_weights(w, wp, cin, cout, flip, st), "exx_unet_conv3d");
    if (s == EXX_OK) {
        const int ci = flip ? cout : cin, co = flip ? cin : cout;
        const int epi = mode == 1 ? 1 : (mode == 2 && mask ? 2 : 0);
        s = gcuda(exx::unet::conv3_tc((const __nv_bfloat16*)x, wp, flip ? nullptr : bias,
                                      (const __nv_bfloat16*)mask, (__nv_bfloat16*)y, batch, D, H, W, ci, co, epi, err,
                                      nsm, st),
                  "exx_unet_conv3d");
    }
    int h = 0;
    if (s == EXX_OK) s = gcuda(cudaMemcpyAsync(&h, err, 4, cudaMemcpyDeviceToHost, st), "exx_unet_conv3d");
    if (s == EXX_OK) s = gcuda(cudaStreamSynchronize(st), "exx_unet_conv3d");
    if (s == EXX_OK && h) s = gfail(EXX_ECUDA, "exx_unet_conv3d: a tensor-core wait timed out");
    cudaFree(wp);
    cudaFree(err);
    return s;
}
