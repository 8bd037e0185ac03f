// The coarse operator with 16-bit links (the precision split of Sec. 2.2 taken
// one level further: the coarse operator D_c = P^dag D P of Eq. 2.5 stored in
// bfloat16 or IEEE half, one FP32 scale per 2N_tv x 2N_tv link block, every
// product accumulated in FP32).
//
//   compress_coarse        FP32 blocks Dc[d][site][col][row] -> 16-bit planes
//                          L[d][site][re|im][row][col] (entries divided by the
//                          block's largest |re|, |im|) and scale[d][site]
//   coarse_apply_links16   y = (Q_c - sigma) x, one right-hand side, thread per
//                          coarse row
//   coarse_apply_nrhs      Y = (Q_c - sigma) X for nrhs <= 16 right-hand sides
//                          on the tensor cores (mma.sync m16n8k16, BF16 in, FP32
//                          accumulate): per coarse site
//                              [P | Q] = [Ar ; Ai] (s_d [Xr | Xi]) summed over the
//                          nine hops d, Yr = P_r - Q_i, Yi = P_i + Q_r (complex
//                          product from real 40 x 40 planes), the per-link scale
//                          s_d folded into the staged right-hand sides
#include <algorithm>

#include "half16.cuh"
#include "internal.h"

namespace mgeig {

// ---------------------------------------------------------------------------
// compression: one CTA per (direction, coarse site) block

template <typename H>
__global__ void __launch_bounds__(256) compress_coarse_kernel(int n2, const float2 *__restrict__ Dc, H *__restrict__ L,
                                                              float *__restrict__ scale) {
    const size_t blk = blockIdx.x;
    const float2 *src = Dc + blk * n2 * n2;   // column-major: src[col * n2 + row]
    H *dst = L + blk * 2 * n2 * n2;           // [re|im][row][col]
    float m = 0.f;
    for (int e = threadIdx.x; e < n2 * n2; e += blockDim.x) {
        const float2 v = src[e];
        m = fmaxf(m, fmaxf(fabsf(v.x), fabsf(v.y)));
    }
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    __shared__ float wm[8];
    if ((threadIdx.x & 31) == 0) wm[threadIdx.x >> 5] = m;
    __syncthreads();
    float s = 0.f;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s = fmaxf(s, wm[w]);
    if (!(s > 0.f)) s = 1.f;
    const float inv = 1.f / s;
    for (int e = threadIdx.x; e < n2 * n2; e += blockDim.x) {
        const int col = e / n2, row = e % n2;
        const float2 v = src[e];
        dst[(size_t)row * n2 + col] = H16<H>::from(v.x * inv);
        dst[(size_t)n2 * n2 + (size_t)row * n2 + col] = H16<H>::from(v.y * inv);
    }
    if (threadIdx.x == 0) scale[blk] = s;
}

void compress_coarse(Ctx &c) {
    const int n2 = 2 * c.prm.n_tv;
    const size_t nblk = (size_t)9 * c.nagg;
    c.Dc16.alloc(nblk * 2 * n2 * n2 * sizeof(__half));
    c.Dcs.alloc(nblk * sizeof(float));
    TimeScope ts(c.timer, K_COARSE_BUILD, (double)nblk * n2 * n2 * (8 + 4));
    if (c.prm.coarse_links == MGEIG_LINKS_BF16)
        compress_coarse_kernel<__nv_bfloat16><<<(int)nblk, 256, 0, c.stream>>>(n2, c.Dc.as<float2>(),
                                                                              c.Dc16.as<__nv_bfloat16>(),
                                                                              c.Dcs.as<float>());
    else
        compress_coarse_kernel<__half><<<(int)nblk, 256, 0, c.stream>>>(n2, c.Dc.as<float2>(), c.Dc16.as<__half>(),
                                                                       c.Dcs.as<float>());
    MG_CHECK_LAUNCH();
}

// ---------------------------------------------------------------------------
// one right-hand side, FP32 arithmetic: thread per (coarse site, row).  A thread reads its own row
// of a link, so neighbouring threads' reads lie a row apart and the sectors they touch have to
// stay in L1 until the row is read: W column pairs (16, 8 or 4 bytes, as the rows' starts are
// aligned) come at a time.  IEEE half, N_tv = 20, one vector: 16^3 x 32 24.6 us with 4 bytes at
// a time, 18.5 now; 32^3 x 64 135 and 90 us.

template <int W> struct Words;
template <> struct Words<1> { typedef uint32_t T; };
template <> struct Words<2> { typedef uint2 T; };
template <> struct Words<4> { typedef uint4 T; };

template <typename H, int W>
__global__ void coarse_apply16_kernel(int nagg, int ntv, const H *__restrict__ L, const float *__restrict__ scale,
                                      const int *__restrict__ nbr, float sigma, const float2 *__restrict__ x,
                                      float2 *__restrict__ y) {
    using HP = typename H16<H>::P;
    using V = typename Words<W>::T;
    const int n2 = 2 * ntv;
    const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (size_t)nagg * n2) return;
    const int a = (int)(t / n2), row = (int)(t % n2);
    float ar = 0.f, ai = 0.f;
    int b = __ldg(nbr + a);
    for (int d = 0; d < 9; ++d) {
        const size_t blk = (size_t)d * nagg + a;
        const int ahead = d < 8 ? __ldg(nbr + blk + nagg) : 0;   // the next hop's neighbour, a hop before its vector is read
        const V *pr = reinterpret_cast<const V *>(L + blk * 2 * n2 * n2 + (size_t)row * n2);
        const V *pi = reinterpret_cast<const V *>(L + blk * 2 * n2 * n2 + (size_t)n2 * n2 + (size_t)row * n2);
        const float4 *xb = reinterpret_cast<const float4 *>(x + (size_t)b * n2);
        float dr = 0.f, di = 0.f;
        for (int p = 0; p < ntv / W; ++p) {
            const V re = __ldg(pr + p), im = __ldg(pi + p);
#pragma unroll
            for (int w = 0; w < W; ++w) {
                const float2 r = H16<H>::pair(reinterpret_cast<const HP *>(&re)[w]),
                             m = H16<H>::pair(reinterpret_cast<const HP *>(&im)[w]);
                const float4 xv = xb[p * W + w];   // two entries of x
                dr = fmaf(r.x, xv.x, dr); dr = fmaf(-m.x, xv.y, dr);
                di = fmaf(r.x, xv.y, di); di = fmaf(m.x, xv.x, di);
                dr = fmaf(r.y, xv.z, dr); dr = fmaf(-m.y, xv.w, dr);
                di = fmaf(r.y, xv.w, di); di = fmaf(m.y, xv.z, di);
            }
        }
        const float s = __ldg(scale + blk);
        ar = fmaf(s, dr, ar);
        ai = fmaf(s, di, ai);
        b = ahead;
    }
    const float2 xt = x[t];
    if (row >= ntv) { ar = -ar; ai = -ai; }
    y[t] = make_float2(ar - sigma * xt.x, ai - sigma * xt.y);
}

template <typename H>
static void launch_apply16(Ctx &c, double sigma, const float2 *x, float2 *y) {
    const int ntv = c.prm.n_tv;
    const int nb = grid_for((size_t)c.nagg * 2 * ntv, 128);
    const H *L = c.Dc16.as<H>();
    const float *s = c.Dcs.as<float>();
    const int *nbr = c.cnbr.as<int>();
    if (ntv % 4 == 0) coarse_apply16_kernel<H, 4><<<nb, 128, 0, c.stream>>>(c.nagg, ntv, L, s, nbr, (float)sigma, x, y);
    else if (ntv % 2 == 0) coarse_apply16_kernel<H, 2><<<nb, 128, 0, c.stream>>>(c.nagg, ntv, L, s, nbr, (float)sigma, x, y);
    else coarse_apply16_kernel<H, 1><<<nb, 128, 0, c.stream>>>(c.nagg, ntv, L, s, nbr, (float)sigma, x, y);
}

void coarse_apply_links16(Ctx &c, double sigma, const void *x, void *y) {
    const int ntv = c.prm.n_tv, n2 = 2 * ntv;
    MG_REQUIRE(n2 % 2 == 0 && c.Dc16.p && c.cnbr.p, MGEIG_ENOTSETUP);
    TimeScope ts(c.timer, K_COARSE_APPLY, (double)c.nagg * (9.0 * (2 * n2 * n2 * 2 + 4) + 2.0 * n2 * 8));
    const float2 *xv = static_cast<const float2 *>(x);
    if (c.prm.coarse_links == MGEIG_LINKS_BF16) launch_apply16<__nv_bfloat16>(c, sigma, xv, static_cast<float2 *>(y));
    else launch_apply16<__half>(c, sigma, xv, static_cast<float2 *>(y));
    MG_CHECK_LAUNCH();
}

// ---------------------------------------------------------------------------
// nrhs right-hand sides on the tensor cores (BF16 links)

constexpr int TC_WARPS = 6;                  // warp w: row tile w / 2, plane w % 2
constexpr int TC_THREADS = 32 * TC_WARPS;
constexpr int TC_MAXN = 16;                  // right-hand sides per launch
constexpr int TC_BP = 56;                    // staged B pitch (halves): conflict-free ldmatrix phases
constexpr int TC_K = 48;                     // staged rows of B
// pitch of the accumulators in shared memory: two-way bank conflicts at most
constexpr int TC_CP(int ncols) { return ncols + 2; }
constexpr int TC_SLACK = 16 * 48 + 64;       // zero halves after the last plane (rows / columns to 48)

__device__ __forceinline__ void mma_bf16_16816(float c[4], const uint32_t a[4], const uint32_t b[2]) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

__device__ __forceinline__ void cp_async16(void *smem, const void *gmem) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem));
}

__device__ __forceinline__ void ldmatrix_x4(uint32_t r[4], const void *row) {
    const unsigned a = (unsigned)__cvta_generic_to_shared(row);
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a));
}
__device__ __forceinline__ void ldmatrix_x2(uint32_t r[2], const void *row) {
    const unsigned a = (unsigned)__cvta_generic_to_shared(row);
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];\n" : "=r"(r[0]), "=r"(r[1]) : "r"(a));
}

// What bounds it: the instruction issue of many small steps per site, not the tensor pipe.
// So the right-hand sides are staged two rows at a time in packed BF16, and fragments come by
// ldmatrix (the links' rows where they start on 16 bytes, N_tv a multiple of 4; 4 bytes at a
// time otherwise).  12 right-hand sides at 32^3 x 64: 233 us before (22 k warp instructions a
// site), 199 now.  All nine hops staged at once, two CTAs an SM, took 348 us: too few warps.
//
// Shared memory of one CTA (one coarse site), n2 = 2 N_tv <= 48 rows:
//   As  a ring of two hop buffers: one link block's planes as stored in global
//       memory ([re|im][row][col], n2 x n2 each, row pitch n2 halves) plus TC_SLACK
//       zero halves (the row and column tiles run to the next multiple of 16, the
//       extra columns read finite entries of the next row that meet zero rows of
//       B, and the extra rows are dropped).  Hop d + 1 is copied (cp.async) while
//       hop d is multiplied
//   Bs  [d][column n < 8 NT][k < 48] staged s_d [Xr | Xi], zero for k >= n2
//   Cs  (after the products) [plane][48][2 nrhs] accumulators
template <int NT>
__global__ void __launch_bounds__(TC_THREADS, 5)
coarse_apply_nrhs_tc_kernel(int nagg, int ntv, int nrhs, const __nv_bfloat16 *__restrict__ L,
                            const float *__restrict__ scale, const int *__restrict__ nbr, float sigma,
                            const float2 *__restrict__ X, float2 *__restrict__ Y) {
    extern __shared__ __align__(16) unsigned char tc_smem[];
    const int n2 = 2 * ntv;
    const int site = blockIdx.x;
    const size_t plane = (size_t)n2 * n2;
    __nv_bfloat16 *As = reinterpret_cast<__nv_bfloat16 *>(tc_smem);
    const size_t hop_elems = ((2 * plane + TC_SLACK + 7) / 8) * 8;   // one ring buffer (16-byte multiple)
    __nv_bfloat16 *Bs = As + 2 * hop_elems;
    constexpr int ncols = 8 * NT;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // 1. the link block of hop d (contiguous 2 n2^2 halves) into ring buffer d & 1
    //    by 16-byte async copies, one commit group per hop
    const int chunks_per_blk = (int)(2 * plane * 2 / 16);
    auto copy_hop = [&](int d) {
        const __nv_bfloat16 *src = L + ((size_t)d * nagg + site) * 2 * plane;
        __nv_bfloat16 *dst = As + (size_t)(d & 1) * hop_elems;
        for (int q = threadIdx.x; q < chunks_per_blk; q += blockDim.x)
            cp_async16(dst + (size_t)q * 8, src + (size_t)q * 8);
        asm volatile("cp.async.commit_group;\n" ::);
    };
    copy_hop(0);
    for (int e = threadIdx.x; e < TC_SLACK; e += blockDim.x) {
        As[2 * plane + e] = __float2bfloat16_rn(0.f);
        As[hop_elems + 2 * plane + e] = __float2bfloat16_rn(0.f);
    }
    // 2. right-hand sides of the nine neighbours, scaled by the link's scale, in BF16: a warp
    //    takes a hop d and a right-hand side r, a lane two rows k; columns r (real parts)
    //    and nrhs + r (imaginary)
#pragma unroll 3
    for (int dr = w; dr < 9 * nrhs; dr += TC_WARPS) {
        const int d = dr / nrhs, r = dr - d * nrhs;
        const size_t blk = (size_t)d * nagg + site;
        const int b = __ldg(nbr + blk);
        const float sc = __ldg(scale + blk);
        if (lane < TC_K / 2) {
            float2 x0 = make_float2(0.f, 0.f), x1 = x0;
            if (lane < ntv) {
                const float2 *xr = X + ((size_t)r * nagg + b) * n2 + 2 * lane;
                x0 = xr[0];
                x1 = xr[1];
            }
            __nv_bfloat162 *br = reinterpret_cast<__nv_bfloat162 *>(Bs + ((size_t)d * ncols + r) * TC_BP) + lane;
            br[0] = __floats2bfloat162_rn(sc * x0.x, sc * x1.x);
            br[nrhs * (TC_BP / 2)] = __floats2bfloat162_rn(sc * x0.y, sc * x1.y);
        }
    }
    // the padding columns 2 nrhs .. 8 NT - 1 of every hop are zero
    const int npad = ncols - 2 * nrhs;
    for (int q = w; q < 9 * npad; q += TC_WARPS) {
        const int d = q / npad, col = 2 * nrhs + q - d * npad;
        if (lane < TC_K / 2)
            reinterpret_cast<__nv_bfloat162 *>(Bs + ((size_t)d * ncols + col) * TC_BP)[lane] = __floats2bfloat162_rn(0.f, 0.f);
    }
    // 3. products: warp w takes rows 16 (w / 2) .. +15 of plane w % 2, every column tile
    const int g = lane >> 2, tq = lane & 3;
    const int mt = w >> 1, pl = w & 1;
    const bool rows16 = n2 % 8 == 0;   // the links' rows start on 16 bytes
    float acc[NT][4];
#pragma unroll
    for (int j = 0; j < NT; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f;
    for (int d = 0; d < 9; ++d) {
        // hop d + 1 streams in while hop d is multiplied
        if (d + 1 < 9) {
            copy_hop(d + 1);
            asm volatile("cp.async.wait_group 1;\n" ::);
        } else {
            asm volatile("cp.async.wait_group 0;\n" ::);
        }
        __syncthreads();   // hop d (and, for d = 0, the staged B and the slack) visible to all
        if (16 * mt < n2) {
            const __nv_bfloat16 *Ap = As + (size_t)(d & 1) * hop_elems + (size_t)pl * plane + (size_t)16 * mt * n2;
            const __nv_bfloat16 *Bp = Bs + (size_t)d * ncols * TC_BP + (lane & 7) * TC_BP;
            uint32_t b[NT][6];   // k 0-7, 8-15, ... of every column tile
#pragma unroll
            for (int j = 0; j < NT; ++j) {
                ldmatrix_x4(b[j], Bp + 8 * j * TC_BP + 8 * (lane >> 3));
                ldmatrix_x2(b[j] + 4, Bp + 8 * j * TC_BP + 32 + 8 * ((lane >> 3) & 1));
            }
#pragma unroll
            for (int ks = 0; ks < 3; ++ks) {
                if (16 * ks >= n2) continue;
                uint32_t a[4];
                if (rows16) {
                    ldmatrix_x4(a, Ap + ((lane & 7) + 8 * ((lane >> 3) & 1)) * n2 + 8 * (lane >> 4) + 16 * ks);
                } else {
                    const __nv_bfloat16 *ar = Ap + g * n2 + 16 * ks + 2 * tq;
                    a[0] = *reinterpret_cast<const uint32_t *>(ar);
                    a[1] = *reinterpret_cast<const uint32_t *>(ar + 8 * n2);
                    a[2] = *reinterpret_cast<const uint32_t *>(ar + 8);
                    a[3] = *reinterpret_cast<const uint32_t *>(ar + 8 * n2 + 8);
                }
#pragma unroll
                for (int j = 0; j < NT; ++j) mma_bf16_16816(acc[j], a, b[j] + 2 * ks);
            }
        }
        __syncthreads();   // every read of ring buffer d & 1 is done before hop d + 2 overwrites it
    }
    // every read of As / Bs is done (the last barrier of the loop): the accumulators reuse the space
    float *Cs = reinterpret_cast<float *>(tc_smem);   // [plane][48][ncols]
    if (16 * mt < n2) {
#pragma unroll
        for (int j = 0; j < NT; ++j) {
            float *cp = Cs + (pl * 48 + 16 * mt + g) * TC_CP(ncols) + 8 * j + 2 * tq;
            *reinterpret_cast<float2 *>(cp) = make_float2(acc[j][0], acc[j][1]);
            *reinterpret_cast<float2 *>(cp + 8 * TC_CP(ncols)) = make_float2(acc[j][2], acc[j][3]);
        }
    }
    __syncthreads();
    // 4. Yr = Ar Xr - Ai Xi, Yi = Ar Xi + Ai Xr; then gamma5^c and the shift
    constexpr int cpitch = TC_CP(ncols);
    const float *Cr = Cs, *Ci = Cs + 48 * cpitch;
    for (int e = threadIdx.x; e < nrhs * n2; e += blockDim.x) {
        const int r = e / n2, row = e - r * n2;
        float yr = Cr[row * cpitch + r] - Ci[row * cpitch + nrhs + r];
        float yi = Cr[row * cpitch + nrhs + r] + Ci[row * cpitch + r];
        if (row >= ntv) { yr = -yr; yi = -yi; }
        const size_t idx = ((size_t)r * nagg + site) * n2 + row;
        const float2 xv = X[idx];
        Y[idx] = make_float2(yr - sigma * xv.x, yi - sigma * xv.y);
    }
}

size_t coarse_nrhs_tc_smem(int n2, int NT) {
    const size_t hop_elems = ((2 * (size_t)n2 * n2 + TC_SLACK + 7) / 8) * 8;
    const size_t a = 2 * hop_elems * 2;
    const size_t b = (size_t)9 * 8 * NT * TC_BP * 2;
    const size_t cbytes = (size_t)2 * 48 * TC_CP(8 * NT) * 4;
    return std::max(a + b, cbytes);
}

template <int NT>
static void launch_nrhs_tc(Ctx &c, double sigma, const float2 *X, float2 *Y, int nrhs) {
    const int n2 = 2 * c.prm.n_tv;
    const size_t smem = coarse_nrhs_tc_smem(n2, NT);
    MG_CUDA(cudaFuncSetAttribute(coarse_apply_nrhs_tc_kernel<NT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smem));
    // algorithmic bytes: the 16-bit links and scales once, every right-hand side read
    // (nine neighbours from L2, counted once) and written once
    TimeScope ts(c.timer, K_COARSE_APPLY,
                 (double)c.nagg * (9.0 * (2 * n2 * n2 * 2 + 4) + (double)nrhs * 2 * n2 * 8));
    coarse_apply_nrhs_tc_kernel<NT><<<c.nagg, TC_THREADS, smem, c.stream>>>(
        c.nagg, c.prm.n_tv, nrhs, c.Dc16.as<__nv_bfloat16>(), c.Dcs.as<float>(), c.cnbr.as<int>(), (float)sigma, X, Y);
    MG_CHECK_LAUNCH();
}

void coarse_apply_nrhs(Ctx &c, double sigma, const void *X, void *Y, int nrhs) {
    const int ntv = c.prm.n_tv, n2 = 2 * ntv;
    MG_REQUIRE(nrhs >= 1 && nrhs <= TC_MAXN, MGEIG_EINVAL);
    MG_REQUIRE(c.cnbr.p && c.Dc.p, MGEIG_ENOTSETUP);
    const size_t vb = (size_t)c.nagg * n2 * sizeof(float2);
    if (c.prm.coarse_links == MGEIG_LINKS_LEVEL) {
        coarse_apply_many<float>(c, sigma, X, Y, nrhs);
        return;
    }
    if (c.prm.coarse_links == MGEIG_LINKS_F16) {
        // the CUDA-core kernel, one right-hand side after another
        for (int r = 0; r < nrhs; ++r)
            coarse_apply_links16(c, sigma, static_cast<const char *>(X) + vb * r, static_cast<char *>(Y) + vb * r);
        return;
    }
    MG_REQUIRE(n2 <= 48 && c.Dc16.p, MGEIG_EINVAL);
    const float2 *x = static_cast<const float2 *>(X);
    float2 *y = static_cast<float2 *>(Y);
    switch ((2 * nrhs + 7) / 8) {
        case 1: launch_nrhs_tc<1>(c, sigma, x, y, nrhs); break;
        case 2: launch_nrhs_tc<2>(c, sigma, x, y, nrhs); break;
        case 3: launch_nrhs_tc<3>(c, sigma, x, y, nrhs); break;
        default: launch_nrhs_tc<4>(c, sigma, x, y, nrhs); break;
    }
}

}  // namespace mgeig
