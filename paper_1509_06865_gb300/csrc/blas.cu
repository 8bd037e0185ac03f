// BLAS-1 on flat complex arrays (fine spinors of one precision share one
// layout, so element-wise operations ignore it; coarse vectors are flat).
//
// Reductions are deterministic two-level trees: a fixed grid of 256-thread blocks
// accumulates grid-stride partial sums (per thread in the array's own precision, then
// in FP64 across the block), writes one partial per block, and the last block to
// finish adds the partials in a fixed order.  Inner products of many vectors against
// one vector, and updates by many vectors, are one launch: blockIdx.y cuts the vectors
// of an inner product into chunks that share one read of y per block (the Arnoldi /
// Gram-Schmidt steps of GMRES, FGMRES and Algorithm 1), an update keeps y in registers.
//
// The FP64 pipe takes half a lane a cycle and scheduler, so a warp's FP64 addition costs
// 64 cycles of it: the block sums exchange halves of the value list between lanes (31
// additions for 32 values; a shuffle tree per value takes 160, which was 10 us a launch).
// A projection (inner products with all vectors to the host, then the update) at 16^3 x 32, before
// with a launch per chunk of vectors, a second kernel for the sums and uploaded coefficients,
// and now: 20 FP64 vectors 528 us, 388 us; 32 FP32 vectors 348 us, 252 us.
#include <algorithm>

#include "ds.cuh"
#include "internal.h"

namespace mgeig {

constexpr int RED_THREADS = 256;
constexpr int RED_MAXBLOCKS = 1024;
constexpr int MAXVEC = MAX_ITERATED + 8;   // pointer slots per launch; more vectors take more launches
static_assert(MAXVEC % 8 == 0, "a double-float update is rounded after every eight vectors");
// vectors that share one read of y: 16 in FP32 (bandwidth bound); 8 in FP64 and in
// double-float arithmetic, where the arithmetic bounds the kernel and 16 accumulators cost
// occupancy
template <typename R> struct Chunk { static constexpr int n = sizeof(R) == 4 ? 16 : 8; };

template <typename R> struct V2;
template <> struct V2<double> { typedef double2 T; };
template <> struct V2<float> { typedef float2 T; };

struct PtrPack { const void *p[MAXVEC]; };

// FP32 arrays of an even number of complex values on 16-byte boundaries are
// processed two values per float4 access
template <typename R>
static bool vec4_ok(const PtrPack &pk, int k, const void *y, size_t n) {
    if (sizeof(R) != 4 || (n & 1)) return false;
    if (reinterpret_cast<uintptr_t>(y) & 15) return false;
    for (int j = 0; j < k; ++j)
        if (reinterpret_cast<uintptr_t>(pk.p[j]) & 15) return false;
    return true;
}

// reduction grids: one block per 4 * 256 elements, at most 4 blocks per SM (or
// blas_blocks per SM when the context sets it) and 1024 in all.  Measured on
// GB300 (16 FP32 or 8 double-float vectors per launch): 4 per SM beat 1024
// blocks by 1.1-1.35x at 16^3 x 32 and 32^3 x 64 (fewer block epilogues and
// partial sums)
static int red_grid(const Ctx &c, size_t n, int per_sm = 4) {
    size_t b = (n + RED_THREADS * 4 - 1) / (RED_THREADS * 4);
    b = std::min<size_t>(b, (size_t)c.sms * (c.prm.blas_blocks > 0 ? c.prm.blas_blocks : per_sm));
    if (b < 1) b = 1;
    if (b > RED_MAXBLOCKS) b = RED_MAXBLOCKS;
    return (int)b;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Sums v[0..N) (N a power of two <= 32) over the warp: lane l ends with the sum of
// value l / (32 / N).  While more than one value is left, each step hands half of them
// to the partner lane instead of adding all of them on both sides.
template <int N>
__device__ __forceinline__ double warp_sum_many(double (&v)[N]) {
    const int lane = threadIdx.x & 31;
    int m = N;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        if (m > 1) {
            m >>= 1;
            const bool up = lane & o;
#pragma unroll
            for (int i = 0; i < N / 2; ++i) {
                if (i < m) {
                    const double give = up ? v[i] : v[i + m], keep = up ? v[i + m] : v[i];
                    v[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
                }
            }
        } else {
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
        }
    }
    return v[0];
}

// Where the sums of a reduction go: partial[vector][RED_MAXBLOCKS], one ticket per chunk
// (zero between launches), and the results.
struct RedOut {
    double2 *partial;
    unsigned int *ticket;
    double2 *out;
};

// v = (re, im) of N / 2 values per thread -> their sums over the grid at out[j0 ..
// j0 + cnt): block sums to the partials, and the last block of the chunk adds those
template <int N>
__device__ __forceinline__ void grid_reduce(double (&v)[N], int j0, int cnt, const RedOut &r) {
    __shared__ double sh[RED_THREADS / 32][N];
    __shared__ bool last;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const double mine = warp_sum_many<N>(v);
    if (lane % (32 / N) == 0) sh[w][lane / (32 / N)] = mine;
    __syncthreads();
    if (threadIdx.x < 2 * cnt) {
        double a = 0;
        for (int i = 0; i < RED_THREADS / 32; ++i) a += sh[i][threadIdx.x];
        const size_t slot = (size_t)(j0 + threadIdx.x / 2) * RED_MAXBLOCKS + blockIdx.x;
        reinterpret_cast<double *>(r.partial)[2 * slot + (threadIdx.x & 1)] = a;
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(r.ticket + blockIdx.y, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    // a warp per value, its lanes for four groups of 32 residues mod 128, the groups in order:
    // the order of the sums is part of the result (see the note on 16-bit links at the
    // persistent coarse solver)
    for (int j = w; j < cnt; j += RED_THREADS / 32) {
        const double2 *p = r.partial + (size_t)(j0 + j) * RED_MAXBLOCKS;
        double q[8];
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            double a = 0, b = 0;
            for (int i = lane + 32 * m; i < (int)gridDim.x; i += 128) {
                const double2 t = __ldcg(p + i);
                a += t.x;
                b += t.y;
            }
            q[2 * m] = a;
            q[2 * m + 1] = b;
        }
        const double mine = warp_sum_many<8>(q);   // lane 8 m: re of group m, lane 8 m + 4: im
        double a = 0;
#pragma unroll
        for (int m = 0; m < 4; ++m) a += __shfl_sync(0xffffffffu, mine, 8 * m + (lane & 4));
        if (lane == 0) r.out[j0 + j].x = a;
        if (lane == 4) r.out[j0 + j].y = a;
    }
    if (threadIdx.x == 0) r.ticket[blockIdx.y] = 0;
}

// real values of C complex sums, filled up to a power of two
template <int C> constexpr int VALUES = C <= 1 ? 2 : C <= 2 ? 4 : C <= 4 ? 8 : C <= 8 ? 16 : 32;

// Blocks an SM that a kernel for C vectors leaves registers for: four (the grid's) where its
// sums and loads in flight are few, two or three where they are many
template <typename R, int C, bool batch> constexpr int dot_blocks() {
    return !batch ? (sizeof(R) == 8 ? 2 : 4) : C * sizeof(R) <= 32 ? 4 : sizeof(R) == 4 ? 2 : 3;
}

// <X_j, y> for the chunk j = per * blockIdx.y .. of at most C vectors.  VEC: two complex values
// per 16-byte load (FP32, n even, 16-byte aligned arrays).  A kernel for C vectors costs
// every call the registers and the FP64 additions of C sums (the FP64 pipe also takes its time
// for operations that are predicated off), so there are kernels for fewer: one vector of
// 12.6 M values took 105 us with the kernel for 16 in FP32, now 45; 255 us in
// double-float arithmetic and 754 in FP64 with the kernels for 8, now 92 and 207.
template <typename R, int C, bool VEC>
__global__ void __launch_bounds__(RED_THREADS, dot_blocks<R, C, VEC>())
multidot_kernel(PtrPack X, int k, int per, const void *__restrict__ yv, size_t n, RedOut out) {
    typedef typename V2<R>::T T;
    const int j0 = blockIdx.y * per;
    k = min(per, k - j0);
    R ar[C], ai[C];
#pragma unroll
    for (int j = 0; j < C; ++j) { ar[j] = 0; ai[j] = 0; }
    if constexpr (VEC) {
        const float4 *y4 = static_cast<const float4 *>(yv);
        for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n / 2; i += (size_t)gridDim.x * blockDim.x) {
            const float4 b = y4[i];
            float4 av[C];   // loaded before they are used
#pragma unroll
            for (int j = 0; j < C; ++j)
                if (j < k) av[j] = static_cast<const float4 *>(X.p[j0 + j])[i];
#pragma unroll
            for (int j = 0; j < C; ++j) {
                if (j < k) {
                    const float4 a = av[j];
                    ar[j] = fmaf(a.x, b.x, ar[j]); ar[j] = fmaf(a.y, b.y, ar[j]);
                    ar[j] = fmaf(a.z, b.z, ar[j]); ar[j] = fmaf(a.w, b.w, ar[j]);
                    ai[j] = fmaf(a.x, b.y, ai[j]); ai[j] = fmaf(-a.y, b.x, ai[j]);
                    ai[j] = fmaf(a.z, b.w, ai[j]); ai[j] = fmaf(-a.w, b.z, ai[j]);
                }
            }
        }
    } else {
        const T *y = static_cast<const T *>(yv);
        for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
            const T b = y[i];
#pragma unroll
            for (int j = 0; j < C; ++j) {
                if (j < k) {
                    const T a = static_cast<const T *>(X.p[j0 + j])[i];
                    ar[j] = fma(a.x, b.x, ar[j]); ar[j] = fma(a.y, b.y, ar[j]);
                    ai[j] = fma(a.x, b.y, ai[j]); ai[j] = fma(-a.y, b.x, ai[j]);
                }
            }
        }
    }
    double v[VALUES<C>] = {};
#pragma unroll
    for (int j = 0; j < C; ++j) { v[2 * j] = ar[j]; v[2 * j + 1] = ai[j]; }
    grid_reduce<VALUES<C>>(v, j0, k, out);
}

template <typename R>
__global__ void __launch_bounds__(RED_THREADS) norm2_kernel(const void *__restrict__ xv, size_t n, RedOut out) {
    typedef typename V2<R>::T T;
    const T *x = static_cast<const T *>(xv);
    R acc = 0;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        T a = x[i];
        acc = fma(a.x, a.x, acc); acc = fma(a.y, a.y, acc);
    }
    double v[2] = {(double)acc, 0.0};
    grid_reduce<2>(v, 0, 1, out);
}

__global__ void __launch_bounds__(RED_THREADS) resid_norm2_kernel(const double2 *__restrict__ qv,
                                                                  const double2 *__restrict__ w,
                                                                  const double2 *__restrict__ lam, size_t n, RedOut out) {
    const double l = lam[0].x;
    double acc = 0;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        double2 a = qv[i], b = w[i];
        double rx = fma(-l, b.x, a.x), ry = fma(-l, b.y, a.y);
        acc = fma(rx, rx, acc); acc = fma(ry, ry, acc);
    }
    double v[2] = {acc, 0.0};
    grid_reduce<2>(v, 0, 1, out);
}

// ---------------------------------------------------------------------------
// FP64 arrays, FP32 arithmetic: the double-float dot product and axpy.
//
// The FP64 pipe of this GPU issues about 1/64 of the FP32 rate, so the FP64
// multidot / multi_axpy (4 FP64 FMAs per complex element and vector) are bound
// by it at about a third of the memory rate.  These kernels read the same FP64
// arrays and compute in FP32 with error-free transformations:
//  * each double d becomes the unevaluated sum hi + lo of two floats by bit
//    manipulation only (hi: sign, exponent and the leading 24 significant bits;
//    lo: the next 23 bits), so |d - hi - lo| < 2^-46 |d| (Dekker's double-length
//    representation, built here by truncation instead of rounding);
//  * a product of two such numbers is hi*hi exactly as p + e (TwoProduct with
//    one FMA) plus the cross terms hi*lo + lo*hi in FP32 (lo*lo < 2^-46 of the
//    product is dropped);
//  * p is added to the running high word by Knuth's TwoSum (exact: s + err), err,
//    e and the cross terms to the low word.
// This is the compensated dot product Dot2 of Ogita, Rump and Oishi (SIAM J.
// Sci. Comput. 26, 2005) on double-float inputs: the result is as accurate as a
// sum in 47-bit arithmetic, i.e. within a few 2^-46 sum|a_i b_i| of the exact
// value (FP64 arithmetic: 2^-53 per operation).  The per-thread sums go to FP64
// for the block and grid reductions.
//
// Range: elements with |d| < 2^-126 count as 0 and the low word is dropped below
// 2^-80 (absolute errors below 2^-103 |d|-units); |d| >= 2^128 becomes +-inf (the
// orthonormal vectors, Krylov vectors and iterates these kernels serve stay far
// inside the range).  Every addition and multiplication below uses the _rn
// intrinsics, which the compiler never contracts into an FMA.

// (h, l) += (uh + ul)(vh + vl)
__device__ __forceinline__ void ds_mac(float &h, float &l, float uh, float ul, float vh, float vl) {
    const float p = __fmul_rn(uh, vh);
    float e = fmaf(uh, vh, -p);
    e = fmaf(uh, vl, e);
    e = fmaf(ul, vh, e);
    const float s = __fadd_rn(h, p);
    const float bv = __fsub_rn(s, h);
    const float err = __fadd_rn(__fsub_rn(h, __fsub_rn(s, bv)), __fsub_rn(p, bv));
    h = s;
    l = __fadd_rn(l, __fadd_rn(err, e));
}

template <int C>
__global__ void __launch_bounds__(RED_THREADS, dot_blocks<double, C, true>())
multidot_ds_kernel(PtrPack X, int k, int per, const double2 *__restrict__ y, size_t n, RedOut out) {
    const int j0 = blockIdx.y * per;
    k = min(per, k - j0);
    float rh[C], rl[C], ih[C], il[C];
#pragma unroll
    for (int j = 0; j < C; ++j) { rh[j] = rl[j] = ih[j] = il[j] = 0.0f; }
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const double2 b = y[i];
        double2 a[C];
#pragma unroll
        for (int j = 0; j < C; ++j)
            if (j < k) a[j] = static_cast<const double2 *>(X.p[j0 + j])[i];
        float brh, brl, bih, bil;
        ds_split(b.x, brh, brl);
        ds_split(b.y, bih, bil);
#pragma unroll
        for (int j = 0; j < C; ++j) {
            if (j < k) {
                float arh, arl, aih, ail;
                ds_split(a[j].x, arh, arl);
                ds_split(a[j].y, aih, ail);
                // conj(a) b = (ar br + ai bi) + i (ar bi - ai br)
                ds_mac(rh[j], rl[j], arh, arl, brh, brl);
                ds_mac(rh[j], rl[j], aih, ail, bih, bil);
                ds_mac(ih[j], il[j], arh, arl, bih, bil);
                ds_mac(ih[j], il[j], -aih, -ail, brh, brl);
            }
        }
    }
    double v[VALUES<C>] = {};
#pragma unroll
    for (int j = 0; j < C; ++j) {
        v[2 * j] = f2d_exact(rh[j]) + f2d_exact(rl[j]);
        v[2 * j + 1] = f2d_exact(ih[j]) + f2d_exact(il[j]);
    }
    grid_reduce<VALUES<C>>(v, j0, k, out);
}

static RedOut red_out_at(Ctx &c, cpx<double> *d_out) {
    double2 *p = c.red_partial.as<double2>();
    return {p, reinterpret_cast<unsigned int *>(p + (size_t)MAXVEC * RED_MAXBLOCKS), reinterpret_cast<double2 *>(d_out)};
}

template <typename R, int C>
static void launch_multidot(Ctx &c, const PtrPack &pk, int k, int per, const void *y, size_t n, const RedOut &out) {
    if constexpr (C <= Chunk<R>::n && C * sizeof(R) >= 16) {
        // FP32 vectors below 8 M complex values (a 16^3 x 32 spinor is 1.6 M): 2 blocks
        // per SM and chunk, 1.3x faster there than 4 (measured); the others 4.  The grid does not
        // depend on k, so that a thread's sums do not either
        const dim3 grid(red_grid(c, n, (sizeof(R) == 4 && n < ((size_t)8 << 20)) ? 2 : 4), (k + per - 1) / per);
        if constexpr (sizeof(R) == 4) {
            if (vec4_ok<R>(pk, k, y, n)) {
                multidot_kernel<R, C, true><<<grid, RED_THREADS, 0, c.stream>>>(pk, k, per, y, n, out);
                return;
            }
        } else if (c.ds_blas()) {
            multidot_ds_kernel<C><<<grid, RED_THREADS, 0, c.stream>>>(pk, k, per, static_cast<const double2 *>(y), n, out);
            return;
        }
        if constexpr (C <= 8) multidot_kernel<R, C, false><<<grid, RED_THREADS, 0, c.stream>>>(pk, k, per, y, n, out);
    }
}

template <typename R>
void blas_multidot(Ctx &c, const void *const *X, int k, const void *y, size_t n, cpx<double> *d_out) {
    for (; k > MAXVEC; k -= MAXVEC, X += MAXVEC, d_out += MAXVEC) blas_multidot<R>(c, X, MAXVEC, y, n, d_out);
    if (k < 1) return;
    PtrPack pk{};
    for (int j = 0; j < k; ++j) pk.p[j] = X[j];
    // 8-byte loads: eight vectors at most (12 vectors of 12.6 M values: 350 us with sixteen, whose
    // registers leave too few warps an SM, 252 so)
    const int most = vec4_ok<R>(pk, k, y, n) ? Chunk<R>::n : 8;
    const int chunks = (k + most - 1) / most, per = (k + chunks - 1) / chunks;
    TimeScope ts(c.timer, sizeof(R) == 8 ? K_BLAS_F64 : K_BLAS_LOW, (double)(k + 1) * n * 2 * sizeof(R));
    const RedOut out = red_out_at(c, d_out);
    if (sizeof(R) == 8 && per <= 2) launch_multidot<R, 2>(c, pk, k, per, y, n, out);
    else if (per <= 4) launch_multidot<R, 4>(c, pk, k, per, y, n, out);
    else if (per <= 6) launch_multidot<R, 6>(c, pk, k, per, y, n, out);
    else if (per <= 8) launch_multidot<R, 8>(c, pk, k, per, y, n, out);
    else launch_multidot<R, 16>(c, pk, k, per, y, n, out);
    MG_CHECK_LAUNCH();
}

template <typename R>
void blas_norm2(Ctx &c, const void *x, size_t n, cpx<double> *d_out) {
    TimeScope ts(c.timer, sizeof(R) == 8 ? K_BLAS_F64 : K_BLAS_LOW, (double)n * 2 * sizeof(R));
    norm2_kernel<R><<<red_grid(c, n), RED_THREADS, 0, c.stream>>>(x, n, red_out_at(c, d_out));
    MG_CHECK_LAUNCH();
}

void blas_resid_norm2(Ctx &c, const void *qv, const void *v, const cpx<double> *d_lambda, size_t n, cpx<double> *d_out) {
    TimeScope ts(c.timer, K_BLAS_F64, (double)n * 32);
    resid_norm2_kernel<<<red_grid(c, n), RED_THREADS, 0, c.stream>>>(
        static_cast<const double2 *>(qv), static_cast<const double2 *>(v), reinterpret_cast<const double2 *>(d_lambda), n,
        red_out_at(c, d_out));
    MG_CHECK_LAUNCH();
}

// The coefficients of an update: in device memory (results of a reduction) or, for
// callers that hold them on the host, in the launch's parameters
struct DevCoef {
    const double2 *p;
    __device__ __forceinline__ double2 operator[](int j) const { return p[j]; }
};
constexpr int HOST_COEFS = 32;
struct HostCoef {
    double2 v[HOST_COEFS];
    __device__ __forceinline__ double2 operator[](int j) const { return v[j]; }
};

// vectors of an update that are loaded before they are used.  Double-float arithmetic: kernels
// for fewer vectors, with fewer registers and more warps an SM (one vector of 12.6 M values 177 us
// with the kernel for 8, 150 now); FP32, one value per access: twice as many
constexpr int AXPY_BATCH = 8;

// y += sign * sum_j coef[j] X_j, y and X_j FP64, double-float arithmetic; B vectors at a time,
// LOOP: as often as it takes (without: k <= B)
template <typename Coef, int B, bool LOOP>
__global__ void __launch_bounds__(256) multi_axpy_ds_kernel(double2 *__restrict__ y, PtrPack X, int k, Coef coef,
                                                            double sign, size_t n) {
    __shared__ float4 cf[MAXVEC];   // (re high, re low, im high, im low)
    if (threadIdx.x < k) {
        const double2 t = coef[threadIdx.x];
        float4 f;
        ds_split(sign * t.x, f.x, f.y);
        ds_split(sign * t.y, f.z, f.w);
        cf[threadIdx.x] = f;
    }
    __syncthreads();
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const double2 t = y[i];
        float rh, rl, ih, il;
        ds_split(t.x, rh, rl);
        ds_split(t.y, ih, il);
        for (int j0 = 0; j0 < (LOOP ? k : 1); j0 += B) {
            double2 a[B];
#pragma unroll
            for (int j = 0; j < B; ++j)
                if (j0 + j < k) a[j] = static_cast<const double2 *>(X.p[j0 + j])[i];
            if (j0) {   // y is rounded to FP64 after every eight vectors
                ds_split(f2d_exact(rh) + f2d_exact(rl), rh, rl);
                ds_split(f2d_exact(ih) + f2d_exact(il), ih, il);
            }
#pragma unroll
            for (int j = 0; j < B; ++j) {
                if (j0 + j < k) {
                    float arh, arl, aih, ail;
                    ds_split(a[j].x, arh, arl);
                    ds_split(a[j].y, aih, ail);
                    const float4 c = cf[j0 + j];
                    // c a = (cr ar - ci ai) + i (cr ai + ci ar)
                    ds_mac(rh, rl, c.x, c.y, arh, arl);
                    ds_mac(rh, rl, -c.z, -c.w, aih, ail);
                    ds_mac(ih, il, c.x, c.y, aih, ail);
                    ds_mac(ih, il, c.z, c.w, arh, arl);
                }
            }
        }
        y[i] = make_double2(f2d_exact(rh) + f2d_exact(rl), f2d_exact(ih) + f2d_exact(il));
    }
}

// y += sign * sum_j coef[j] X_j; B: AXPY_BATCH for one value per access
template <typename R, typename Coef, int B>
__global__ void __launch_bounds__(256) multi_axpy_kernel(void *__restrict__ yv, PtrPack X, int k, Coef coef, double sign,
                                                         size_t n, bool vec4) {
    typedef typename V2<R>::T T;
    T *y = static_cast<T *>(yv);
    __shared__ T cf[MAXVEC];
    if (threadIdx.x < k) {
        const double2 t = coef[threadIdx.x];
        T f;
        f.x = (R)(sign * t.x);
        f.y = (R)(sign * t.y);
        cf[threadIdx.x] = f;
    }
    __syncthreads();
    if constexpr (sizeof(R) == 4) {
        if (vec4) {   // two complex values per 16-byte access
            float4 *y4 = static_cast<float4 *>(yv);
            for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n / 2; i += (size_t)gridDim.x * blockDim.x) {
                float4 acc = y4[i];
                for (int j0 = 0; j0 < k; j0 += AXPY_BATCH) {
                    float4 a[AXPY_BATCH];
#pragma unroll
                    for (int j = 0; j < AXPY_BATCH; ++j)
                        if (j0 + j < k) a[j] = static_cast<const float4 *>(X.p[j0 + j])[i];
#pragma unroll
                    for (int j = 0; j < AXPY_BATCH; ++j) {
                        if (j0 + j < k) {
                            const T c = cf[j0 + j];
                            acc.x = fmaf(c.x, a[j].x, acc.x); acc.x = fmaf(-c.y, a[j].y, acc.x);
                            acc.y = fmaf(c.x, a[j].y, acc.y); acc.y = fmaf(c.y, a[j].x, acc.y);
                            acc.z = fmaf(c.x, a[j].z, acc.z); acc.z = fmaf(-c.y, a[j].w, acc.z);
                            acc.w = fmaf(c.x, a[j].w, acc.w); acc.w = fmaf(c.y, a[j].z, acc.w);
                        }
                    }
                }
                y4[i] = acc;
            }
            return;
        }
    }
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        T acc = y[i];
        for (int j0 = 0; j0 < k; j0 += B) {
            T a[B];
#pragma unroll
            for (int j = 0; j < B; ++j)
                if (j0 + j < k) a[j] = static_cast<const T *>(X.p[j0 + j])[i];
#pragma unroll
            for (int j = 0; j < B; ++j) {
                if (j0 + j < k) {
                    const T c = cf[j0 + j];
                    acc.x = fma(c.x, a[j].x, acc.x); acc.x = fma(-c.y, a[j].y, acc.x);
                    acc.y = fma(c.x, a[j].y, acc.y); acc.y = fma(c.y, a[j].x, acc.y);
                }
            }
        }
        y[i] = acc;
    }
}

// element-wise grids: one thread per element up to per_sm blocks per SM (or
// blas_blocks per SM when the context sets it).  The FP32 multi-vector update
// runs best at 4 per SM (1.5x over 16 at 16^3 x 32), the double-float one,
// bound by its FP32 arithmetic, at 16
static int ew_grid(const Ctx &c, size_t n, int per_sm = 16) {
    size_t b = (n + 255) / 256;
    const size_t cap = (size_t)c.sms * (c.prm.blas_blocks > 0 ? c.prm.blas_blocks : per_sm);
    return (int)(b < cap ? (b < 1 ? 1 : b) : cap);
}

template <typename R, typename Coef>
static void launch_multi_axpy(Ctx &c, void *y, const void *const *X, int k, const Coef &coef, double sign, size_t n) {
    TimeScope ts(c.timer, sizeof(R) == 8 ? K_BLAS_F64 : K_BLAS_LOW, (double)(k + 2) * n * 2 * sizeof(R));
    PtrPack pk{};
    for (int j = 0; j < k; ++j) pk.p[j] = X[j];
    if (sizeof(R) == 8 && c.ds_blas()) {
        double2 *y2 = static_cast<double2 *>(y);
        const int nb = ew_grid(c, n);
        if (k <= 2) multi_axpy_ds_kernel<Coef, 2, false><<<nb, 256, 0, c.stream>>>(y2, pk, k, coef, sign, n);
        else if (k <= 4) multi_axpy_ds_kernel<Coef, 4, false><<<nb, 256, 0, c.stream>>>(y2, pk, k, coef, sign, n);
        else if (k <= 6) multi_axpy_ds_kernel<Coef, 6, false><<<nb, 256, 0, c.stream>>>(y2, pk, k, coef, sign, n);
        else multi_axpy_ds_kernel<Coef, AXPY_BATCH, true><<<nb, 256, 0, c.stream>>>(y2, pk, k, coef, sign, n);
    } else {
        const bool v4 = vec4_ok<R>(pk, k, y, n);
        const int nb = ew_grid(c, v4 ? n / 2 : n, sizeof(R) == 4 ? 4 : 16);
        if (sizeof(R) == 4 && !v4 && k > AXPY_BATCH)
            multi_axpy_kernel<R, Coef, sizeof(R) == 4 ? 2 * AXPY_BATCH : AXPY_BATCH>
                <<<nb, 256, 0, c.stream>>>(y, pk, k, coef, sign, n, v4);
        else multi_axpy_kernel<R, Coef, AXPY_BATCH><<<nb, 256, 0, c.stream>>>(y, pk, k, coef, sign, n, v4);
    }
    MG_CHECK_LAUNCH();
}

template <typename R>
void blas_multi_axpy(Ctx &c, void *y, const void *const *X, int k, const cpx<double> *d_coef, double sign, size_t n) {
    for (; k > 0; k -= MAXVEC, X += MAXVEC, d_coef += MAXVEC)
        launch_multi_axpy<R>(c, y, X, std::min(k, MAXVEC), DevCoef{reinterpret_cast<const double2 *>(d_coef)}, sign, n);
}

// k <= 32 coefficients from the host, in the launch's parameters (no upload)
template <typename R>
void blas_multi_axpy_host(Ctx &c, void *y, const void *const *X, int k, const double *coef, size_t n) {
    MG_REQUIRE(k >= 1 && k <= HOST_COEFS, MGEIG_EINVAL);
    HostCoef h;
    for (int j = 0; j < k; ++j) h.v[j] = make_double2(coef[2 * j], coef[2 * j + 1]);
    launch_multi_axpy<R>(c, y, X, k, h, 1.0, n);
}
template void blas_multi_axpy_host<double>(Ctx &, void *, const void *const *, int, const double *, size_t);
template void blas_multi_axpy_host<float>(Ctx &, void *, const void *const *, int, const double *, size_t);

template <typename R>
__global__ void axpy_kernel(double ar, double ai, const void *__restrict__ xv, void *__restrict__ yv, size_t n) {
    typedef typename V2<R>::T T;
    const T *x = static_cast<const T *>(xv);
    T *y = static_cast<T *>(yv);
    const R a = (R)ar, b = (R)ai;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        T u = x[i], v = y[i];
        v.x = fma(a, u.x, v.x); v.x = fma(-b, u.y, v.x);
        v.y = fma(a, u.y, v.y); v.y = fma(b, u.x, v.y);
        y[i] = v;
    }
}

template <typename R>
__global__ void scale_kernel(double ar, double ai, void *__restrict__ xv, size_t n) {
    typedef typename V2<R>::T T;
    T *x = static_cast<T *>(xv);
    const R a = (R)ar, b = (R)ai;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        T u = x[i];
        T v;
        v.x = a * u.x - b * u.y;
        v.y = a * u.y + b * u.x;
        x[i] = v;
    }
}

template <typename R>
void blas_axpy(Ctx &c, cpx<double> a, const void *x, void *y, size_t n) {
    TimeScope ts(c.timer, sizeof(R) == 8 ? K_BLAS_F64 : K_BLAS_LOW, 3.0 * n * 2 * sizeof(R));
    axpy_kernel<R><<<ew_grid(c, n), 256, 0, c.stream>>>(a.re, a.im, x, y, n);
    MG_CHECK_LAUNCH();
}

template <typename R>
void blas_scale(Ctx &c, cpx<double> a, void *x, size_t n) {
    TimeScope ts(c.timer, sizeof(R) == 8 ? K_BLAS_F64 : K_BLAS_LOW, 2.0 * n * 2 * sizeof(R));
    scale_kernel<R><<<ew_grid(c, n), 256, 0, c.stream>>>(a.re, a.im, x, n);
    MG_CHECK_LAUNCH();
}

template <typename R>
void blas_copy(Ctx &c, const void *x, void *y, size_t n) {
    MG_CUDA(cudaMemcpyAsync(y, x, n * 2 * sizeof(R), cudaMemcpyDeviceToDevice, c.stream));
}

template <typename R>
void blas_zero(Ctx &c, void *x, size_t n) {
    MG_CUDA(cudaMemsetAsync(x, 0, n * 2 * sizeof(R), c.stream));
}

// y (FP64 fine layout) += a * x (fine layout of precision R)
template <typename R>
__global__ void axpy_to_f64_fine_kernel(int V, double ar, double ai, const void *__restrict__ x, double2 *__restrict__ y) {
    int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= V) return;
    cpx<R> v[12];
    Spinor<R>::load(x, V, s, v);
#pragma unroll
    for (int k = 0; k < 12; ++k) {
        double2 t = y[(size_t)k * V + s];
        double xr = v[k].re, xi = v[k].im;
        t.x = fma(ar, xr, t.x); t.x = fma(-ai, xi, t.x);
        t.y = fma(ar, xi, t.y); t.y = fma(ai, xr, t.y);
        y[(size_t)k * V + s] = t;
    }
}

template <typename R>
void blas_axpy_to_f64(Ctx &c, cpx<double> a, const void *x, void *y64, size_t n) {
    const int V = (int)(n / 12);
    TimeScope ts(c.timer, K_BLAS_F64, (double)n * (2 * sizeof(R) + 32));
    axpy_to_f64_fine_kernel<R><<<grid_for(V, 256), 256, 0, c.stream>>>(V, a.re, a.im, x, static_cast<double2 *>(y64));
    MG_CHECK_LAUNCH();
}

// y = A x and ys = s * y for a small row-major k x k matrix A (k <= 64), one
// thread per row; A, x, y and ys live on the device (no host round trip)
__global__ void small_gemv_kernel(const double2 *__restrict__ A, int k, const double2 *__restrict__ x, double s,
                                  double2 *__restrict__ y, double2 *__restrict__ ys) {
    const int i = threadIdx.x;
    if (i >= k) return;
    double re = 0, im = 0;
    for (int l = 0; l < k; ++l) {
        const double2 a = A[(size_t)i * k + l], b = x[l];
        re = fma(a.x, b.x, re); re = fma(-a.y, b.y, re);
        im = fma(a.x, b.y, im); im = fma(a.y, b.x, im);
    }
    y[i] = make_double2(re, im);
    ys[i] = make_double2(s * re, s * im);
}

void small_gemv(Ctx &c, const cpx<double> *A, int k, const cpx<double> *x, double s, cpx<double> *y, cpx<double> *ys) {
    MG_REQUIRE(k >= 1 && k <= 64, MGEIG_EINVAL);
    TimeScope ts(c.timer, K_BLAS_F64, (double)k * (k + 3) * 16);
    small_gemv_kernel<<<1, 64, 0, c.stream>>>(reinterpret_cast<const double2 *>(A), k, reinterpret_cast<const double2 *>(x),
                                              s, reinterpret_cast<double2 *>(y), reinterpret_cast<double2 *>(ys));
    MG_CHECK_LAUNCH();
}

#define INST(R)                                                                                             \
    template void blas_multidot<R>(Ctx &, const void *const *, int, const void *, size_t, cpx<double> *);    \
    template void blas_multi_axpy<R>(Ctx &, void *, const void *const *, int, const cpx<double> *, double, size_t); \
    template void blas_norm2<R>(Ctx &, const void *, size_t, cpx<double> *);                                     \
    template void blas_axpy<R>(Ctx &, cpx<double>, const void *, void *, size_t);                          \
    template void blas_scale<R>(Ctx &, cpx<double>, void *, size_t);                                       \
    template void blas_copy<R>(Ctx &, const void *, void *, size_t);                                       \
    template void blas_zero<R>(Ctx &, void *, size_t);                                                     \
    template void blas_axpy_to_f64<R>(Ctx &, cpx<double>, const void *, void *, size_t);
INST(double)
INST(float)
#undef INST

}  // namespace mgeig
