// Two-grid kernels (Sec. 2 of arXiv:1509.06865, Eqs. 2.3-2.6):
//   build_interp   aggregation interpolation P (Eq. 2.4): per aggregate and
//                  chirality, Gram-Schmidt (twice) of the N_tv test vectors, FP64
//   restrict_vec   r_c = P^dag r          (CTAs per aggregate and part of the test vectors)
//   prolong_vec    e = P e_c              (one or two threads per fine site)
//   build_coarse   D_c = P^dag D P as nine per-direction blocks (Eq. 2.5)
//   coarse_apply_many  y = gamma5^c D_c x - sigma x = (Q_c - sigma) x (Eq. 2.6), n vectors
//   sap_sweep      one colour of the Schwarz alternating procedure on
//                  D_sigma = D - sigma gamma5: block-local minimal residual with
//                  Dirichlet block boundaries, block vector staged in shared memory
//
// P is stored as N_tv fine spinors in the internal spinor layout (column (a, c, j)
// of P = spinor j restricted to aggregate a and chirality c).  Coarse vectors are
// [coarse site][c][j] complex; coarse blocks are column-major:
// Dc[d][a][col][row], d = 0 self, 1 + 2 mu = +mu, 2 + 2 mu = -mu.
#include <algorithm>

#include "internal.h"

namespace mgeig {

struct AggGeom {
    int agg[4];     // aggregate (or SAP block) extent
    int cdims[4];   // number of aggregates per direction
    int vol;        // sites per aggregate
    int n;          // number of aggregates
};

static AggGeom make_agg(const Ctx &c, const int *blk) {
    AggGeom a;
    a.vol = 1;
    a.n = 1;
    for (int mu = 0; mu < 4; ++mu) {
        a.agg[mu] = blk[mu];
        a.cdims[mu] = c.dims[mu] / blk[mu];
        a.vol *= blk[mu];
        a.n *= a.cdims[mu];
    }
    return a;
}

// fine site of local site l in aggregate a; local coords in lc
__device__ __forceinline__ int agg_site(const Geom &g, const AggGeom &A, int a, int l, int lc[4]) {
    int ac[4];
    ac[0] = a % A.cdims[0]; a /= A.cdims[0];
    ac[1] = a % A.cdims[1]; a /= A.cdims[1];
    ac[2] = a % A.cdims[2];
    ac[3] = a / A.cdims[2];
    lc[0] = l % A.agg[0]; l /= A.agg[0];
    lc[1] = l % A.agg[1]; l /= A.agg[1];
    lc[2] = l % A.agg[2];
    lc[3] = l / A.agg[2];
    int s = 0;
    for (int mu = 3; mu >= 0; --mu) s = s * g.L[mu] + ac[mu] * A.agg[mu] + lc[mu];
    return s;
}

__device__ __forceinline__ int agg_of_site(const Geom &g, const AggGeom &A, const int c[4]) {
    int a = 0;
    for (int mu = 3; mu >= 0; --mu) a = a * A.cdims[mu] + c[mu] / A.agg[mu];
    return a;
}

// 16 bytes of an array of complex values of precision R
template <typename R> struct V16Of { typedef float4 T; };
template <> struct V16Of<double> { typedef double2 T; };

struct PtrList { const void *p[24]; };
struct MutPtrList { void *p[24]; };

// ---------------------------------------------------------------------------
// interpolation: classical Gram-Schmidt (twice) per (aggregate, chirality),
// arithmetic in precision R (FP64 for the all-FP64 path; FP32 for the mixed
// path, whose P is stored in FP32).  Test vectors are read in FP64.  One CTA per
// (aggregate, chirality); all <q_i, w> of one pass share one block reduction.

constexpr int PB_THREADS = 256;
constexpr int PB_MAXS = 4;    // sites per thread (aggregates of up to 1024 sites)
constexpr int PB_MAXN = 24;   // test vectors

// Block Gram-Schmidt of the test vectors on one aggregate and chirality, two
// passes per vector.  Sums run in the level precision R: in the mixed path the
// FP64 warp reductions of an earlier form (1/64 of the FP32 rate here) took
// half of the kernel's time, and P is stored in FP32 anyway.
template <typename R>
__global__ void __launch_bounds__(PB_THREADS) interp_kernel(Geom g, AggGeom A, PtrList W, int ntv, MutPtrList P) {
    __shared__ R sh[PB_THREADS / 32][2 * PB_MAXN];
    __shared__ R hs[2 * PB_MAXN];
    const int a = blockIdx.x >> 1, chir = blockIdx.x & 1;
    const int V = g.V;
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    int sites[PB_MAXS];
    int ns = 0;
    for (int l = threadIdx.x; l < A.vol && ns < PB_MAXS; l += blockDim.x) {
        int lc[4];
        sites[ns++] = agg_site(g, A, a, l, lc);
    }
    // block-reduce cnt complex values parked per warp in sh -> hs (all threads)
    auto reduce = [&](int cnt) {
        __syncthreads();
        for (int i = threadIdx.x; i < 2 * cnt; i += blockDim.x) {
            R s = 0;
            for (int w = 0; w < nw; ++w) s += sh[w][i];
            hs[i] = s;
        }
        __syncthreads();
    };
    auto warp_sum = [&](R v) {
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        return v;
    };
    for (int j = 0; j < ntv; ++j) {
        cpx<R> w[PB_MAXS][6];
        const double2 *src = static_cast<const double2 *>(W.p[j]);
        for (int i = 0; i < PB_MAXS; ++i)
            for (int k = 0; k < 6; ++k) {
                if (i < ns) { double2 t = src[(size_t)(chir * 6 + k) * V + sites[i]]; w[i][k] = cpx<R>((R)t.x, (R)t.y); }
                else w[i][k] = cpx<R>();
            }
        for (int pass = 0; pass < 2 && j > 0; ++pass) {
#pragma unroll 4
            for (int q = 0; q < j; ++q) {
                const cpx<R> *pq = static_cast<const cpx<R> *>(P.p[q]);
                cpx<R> d;
                for (int i = 0; i < ns; ++i)
                    for (int k = 0; k < 6; ++k) cmac_conj(d, Spinor<R>::comp(pq, V, chir * 6 + k, sites[i]), w[i][k]);
                const R re = warp_sum(d.re), im = warp_sum(d.im);
                if (lane == 0) { sh[wp][2 * q] = re; sh[wp][2 * q + 1] = im; }
            }
            reduce(j);
            for (int q = 0; q < j; ++q) {
                const cpx<R> *pq = static_cast<const cpx<R> *>(P.p[q]);
                const cpx<R> hc((R)hs[2 * q], (R)hs[2 * q + 1]);
                for (int i = 0; i < ns; ++i)
                    for (int k = 0; k < 6; ++k) w[i][k] = w[i][k] - hc * Spinor<R>::comp(pq, V, chir * 6 + k, sites[i]);
            }
        }
        R nn = 0;
        for (int i = 0; i < ns; ++i)
            for (int k = 0; k < 6; ++k) nn += w[i][k].re * w[i][k].re + w[i][k].im * w[i][k].im;
        nn = warp_sum(nn);
        if (lane == 0) { sh[wp][0] = nn; sh[wp][1] = 0; }
        reduce(1);
        const R inv = hs[0] > 0 ? R(1) / sqrt(hs[0]) : R(0);
        cpx<R> *dst = static_cast<cpx<R> *>(P.p[j]);
        for (int i = 0; i < ns; ++i)
            for (int k = 0; k < 6; ++k) Spinor<R>::comp(dst, V, chir * 6 + k, sites[i]) = inv * w[i][k];
    }
}

// P (ntv spinors of precision R) from the FP64 test vectors W64
template <typename R>
void build_interp(Ctx &c, const void *const *W64, int ntv, void *const *P) {
    AggGeom A = make_agg(c, c.prm.agg);
    MG_REQUIRE(A.vol <= PB_THREADS * PB_MAXS && ntv <= PB_MAXN, MGEIG_EINVAL);
    PtrList w{};
    MutPtrList p{};
    for (int j = 0; j < ntv; ++j) { w.p[j] = W64[j]; p.p[j] = P[j]; }
    const int threads = A.vol < PB_THREADS ? ((A.vol + 31) / 32) * 32 : PB_THREADS;
    TimeScope ts(c.timer, K_PBUILD, (double)ntv * c.g.V * 12 * (16 + 2 * sizeof(R)));
    interp_kernel<R><<<A.n * 2, threads, 0, c.stream>>>(c.g, A, w, ntv, p);
    MG_CHECK_LAUNCH();
}
template void build_interp<double>(Ctx &, const void *const *, int, void *const *);
template void build_interp<float>(Ctx &, const void *const *, int, void *const *);

// ---------------------------------------------------------------------------
// restriction r_c = P^dag r: CTA (a, y) takes aggregate a and the test vectors y per .. y per +
// per - 1; how they are cut does not change a sum
template <typename R>
__global__ void restrict_kernel(Geom g, AggGeom A, PtrList P, int ntv, int per, const void *__restrict__ r,
                                cpx<R> *__restrict__ rc) {
    extern __shared__ unsigned char smem_raw[];
    R *sh = reinterpret_cast<R *>(smem_raw);   // [nwarps][2*per][2]
    const int a = blockIdx.x, j0 = blockIdx.y * per, nj = min(per, ntv - j0);
    const int V = g.V;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int n2 = 2 * per;
    // one site per thread (aggregates of at most blockDim sites, the usual case):
    // r is loaded once and kept in registers for all test vectors; otherwise each
    // thread visits its sites once per j
    const bool one = A.vol <= (int)blockDim.x;
    int s1 = -1;
    cpx<R> x1[12];
    if (one && (int)threadIdx.x < A.vol) {
        int lc[4];
        s1 = agg_site(g, A, a, threadIdx.x, lc);
        Spinor<R>::load(r, V, s1, x1);
    }
#pragma unroll 2
    for (int j = 0; j < nj; ++j) {
        cpx<R> d0, d1;
        if (one) {
            if (s1 >= 0) {
                cpx<R> p[12];
                Spinor<R>::load(P.p[j0 + j], V, s1, p);
#pragma unroll
                for (int k = 0; k < 6; ++k) { cmac_conj(d0, p[k], x1[k]); cmac_conj(d1, p[6 + k], x1[6 + k]); }
            }
        } else {
            for (int l = threadIdx.x; l < A.vol; l += blockDim.x) {
                int lc[4];
                const int s = agg_site(g, A, a, l, lc);
                cpx<R> x[12], p[12];
                Spinor<R>::load(r, V, s, x);
                Spinor<R>::load(P.p[j0 + j], V, s, p);
#pragma unroll
                for (int k = 0; k < 6; ++k) { cmac_conj(d0, p[k], x[k]); cmac_conj(d1, p[6 + k], x[6 + k]); }
            }
        }
        for (int o = 16; o > 0; o >>= 1) {
            d0.re += __shfl_xor_sync(0xffffffffu, d0.re, o); d0.im += __shfl_xor_sync(0xffffffffu, d0.im, o);
            d1.re += __shfl_xor_sync(0xffffffffu, d1.re, o); d1.im += __shfl_xor_sync(0xffffffffu, d1.im, o);
        }
        if (lane == 0) {
            sh[(w * n2 + j) * 2] = d0.re; sh[(w * n2 + j) * 2 + 1] = d0.im;
            sh[(w * n2 + per + j) * 2] = d1.re; sh[(w * n2 + per + j) * 2 + 1] = d1.im;
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 2 * nj; i += blockDim.x) {
        const int chir = i >= nj, j = i - chir * nj, v = chir * per + j;
        cpx<R> t;
        for (int q = 0; q < nw; ++q) { t.re += sh[(q * n2 + v) * 2]; t.im += sh[(q * n2 + v) * 2 + 1]; }
        rc[(size_t)a * 2 * ntv + chir * ntv + j0 + j] = t;
    }
}

static int agg_threads(int vol) {
    if (vol >= 256) return 256;
    return ((vol + 31) / 32) * 32;
}

template <typename R>
void restrict_vec(Ctx &c, const void *const *P, const void *r, void *rc) {
    AggGeom A = make_agg(c, c.prm.agg);
    const int ntv = c.prm.n_tv;
    PtrList p{};
    for (int j = 0; j < ntv; ++j) p.p[j] = P[j];
    const int threads = agg_threads(A.vol);
    // parts of the test vectors so that there are up to six CTAs an SM: with one CTA an aggregate a
    // coarse grid of few aggregates left SMs idle (FP64, 8^3 x 16, 32 aggregates: 99 us, and the
    // prolongation, then a thread a site, 70 us; the cycle 2040 -> 1948 us with both cut).  Two
    // CTAs an SM or six are alike; 512 aggregates at 16^3 x 32 take one part, as before.  Every
    // part reads r again: in FP32 the line below keeps one part where there is not much more than
    // that to read (256 aggregates, N_tv = 4: 9.5 us in one part, 11 in two; 320, N_tv = 20: 35
    // and 37.5; 256, N_tv = 20: 33 and in three parts 29)
    int parts = std::min(ntv, std::max(1, 6 * c.sms / A.n));
    if (sizeof(R) == 4 && A.vol <= 256 && 10 * A.n >= c.sms * ntv) parts = 1;
    const int per = (ntv + parts - 1) / parts;
    const size_t smem = (size_t)(threads / 32) * 2 * per * 2 * sizeof(R);
    TimeScope ts(c.timer, K_RESTRICT, (double)(ntv + 1) * c.g.V * 24 * sizeof(R));
    restrict_kernel<R><<<dim3(A.n, (ntv + per - 1) / per), threads, smem, c.stream>>>(c.g, A, p, ntv, per, r,
                                                                                     static_cast<cpx<R> *>(rc));
    MG_CHECK_LAUNCH();
}

// ---------------------------------------------------------------------------
// prolongation e = P e_c: a thread per fine site and NC chiralities (NC = 1: blockIdx.y is the
// chirality)

template <typename R, int NC>
__global__ void prolong_kernel(Geom g, AggGeom A, PtrList P, int ntv, const cpx<R> *__restrict__ ec, void *__restrict__ e) {
    using V16 = typename V16Of<R>::T;
    constexpr int N = NC * 6 * (int)sizeof(cpx<R>) / 16;   // 16-byte planes of a thread's components
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= g.V) return;
    int c[4];
    site_coords(g, s, c);
    const int chir = blockIdx.y;
    const size_t V = g.V, first = (size_t)chir * N * V + s;
    const cpx<R> *ea = ec + (size_t)agg_of_site(g, A, c) * 2 * ntv + chir * ntv;
    cpx<R> out[6 * NC];
    for (int j = 0; j < ntv; ++j) {
        const V16 *src = static_cast<const V16 *>(P.p[j]) + first;
        V16 v[N];
#pragma unroll
        for (int q = 0; q < N; ++q) v[q] = src[q * V];
        const cpx<R> *p = reinterpret_cast<const cpx<R> *>(v);
#pragma unroll
        for (int h = 0; h < NC; ++h) {
            const cpx<R> ej = ea[h * ntv + j];
#pragma unroll
            for (int k = 6 * h; k < 6 * h + 6; ++k) cmac(out[k], p[k], ej);
        }
    }
    V16 *dst = static_cast<V16 *>(e) + first;
#pragma unroll
    for (int q = 0; q < N; ++q) dst[q * V] = reinterpret_cast<const V16 *>(out)[q];
}

template <typename R>
void prolong_vec(Ctx &c, const void *const *P, const void *ec, void *e) {
    AggGeom A = make_agg(c, c.prm.agg);
    const int ntv = c.prm.n_tv;
    PtrList p{};
    for (int j = 0; j < ntv; ++j) p.p[j] = P[j];
    TimeScope ts(c.timer, K_PROLONG, (double)(ntv + 1) * c.g.V * 24 * sizeof(R));
    // a thread per site and chirality where a thread a site gives less than four CTAs an SM (FP64,
    // 8^3 x 16: 70 us with a thread a site); at 16^3 x 32 the HBM bound form with a thread a
    // site is 9 % faster in FP32 (5.9 TB/s, 5.4 with two threads)
    const int nb = grid_for(c.g.V, 128);
    const cpx<R> *x = static_cast<const cpx<R> *>(ec);
    if (nb < 4 * c.sms) prolong_kernel<R, 1><<<dim3(nb, 2), 128, 0, c.stream>>>(c.g, A, p, ntv, x, e);
    else prolong_kernel<R, 2><<<nb, 128, 0, c.stream>>>(c.g, A, p, ntv, x, e);
    MG_CHECK_LAUNCH();
}

// ---------------------------------------------------------------------------
// coarse operator build: one CTA per (aggregate, direction)

constexpr int CB_THREADS = 256;
constexpr int CB_CHUNK = 8;   // fine sites staged per step
constexpr int CB_MAXO = 9;    // outputs per thread: (2*24)^2 / 256

// keeps chirality cp of a spinor (components 6 cp .. 6 cp + 5) and zeroes the
// other, with compile-time indices only
template <typename R>
__device__ __forceinline__ void zero_other_chirality(cpx<R> psi[12], int cp) {
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        if (cp == 0) psi[6 + k] = cpx<R>();
        else psi[k] = cpx<R>();
    }
}

// directional fine operator applied to column (cp, jp) of P at fine site s:
// d = 0: local term + hops that stay inside the aggregate; d = 1 + 2mu / 2 + 2mu:
// the single hop leaving the aggregate through its upper / lower mu face.
template <typename R>
__device__ void directional_column(const Geom &g, const AggGeom &A, const void *U, const void *clov, const void *Pj,
                                   int cp, int d, int s, const int c[4], cpx<R> out[12]) {
    const int V = g.V;
    cpx<R> up[6], lo[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) { up[k] = cpx<R>(); lo[k] = cpx<R>(); }
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
#pragma unroll
        for (int f = 0; f < 2; ++f) {
            const bool fwd = f == 0;
            const int lm = c[mu] % A.agg[mu];
            const bool leaves = fwd ? (lm == A.agg[mu] - 1) : (lm == 0);
            const int want = fwd ? 1 + 2 * mu : 2 + 2 * mu;
            if (d == 0 ? leaves : (d != want)) continue;
            int ph;
            const int n = neighbor(g, s, c, mu, fwd, &ph);
            cpx<R> u[9], psi[12];
            Gauge<R>::load(U, V, mu, fwd ? s : n, u);
            Spinor<R>::load(Pj, V, n, psi);
            zero_other_chirality(psi, cp);
            hop_accumulate<R>(mu, fwd, u, psi, (R)ph, up, lo);
        }
    }
    const R half = R(0.5);
    if (d == 0) {
        cpx<R> psi[12];
        Spinor<R>::load(Pj, V, s, psi);
        zero_other_chirality(psi, cp);
        clover_apply<R>(clov, V, s, psi, out);
    } else {
#pragma unroll
        for (int k = 0; k < 12; ++k) out[k] = cpx<R>();
    }
#pragma unroll
    for (int k = 0; k < 6; ++k) { out[k] = out[k] - half * up[k]; out[6 + k] = out[6 + k] - half * lo[k]; }
}

template <typename R>
__global__ void __launch_bounds__(CB_THREADS) coarse_build_kernel(Geom g, AggGeom A, const void *__restrict__ U,
                                                                  const void *__restrict__ clov, PtrList P, int ntv,
                                                                  cpx<R> *__restrict__ Dc) {
    extern __shared__ unsigned char smem_raw[];
    const int a = blockIdx.x / 9, d = blockIdx.x % 9;
    const int n2 = 2 * ntv;
    // component-major within a staged site ([CHUNK][12][ntv]): the threads of a warp
    // take consecutive rows, i.e. consecutive test vectors, so their reads of sP are
    // consecutive words (a [CHUNK][ntv][12] layout had 4-way bank conflicts)
    cpx<R> *sP = reinterpret_cast<cpx<R> *>(smem_raw);           // [CHUNK][12][ntv]
    cpx<R> *sH = sP + (size_t)CB_CHUNK * ntv * 12;               // [CHUNK][n2][12]
    const int V = g.V;
    // sites of this direction: all sites (d = 0) or the face l_mu = agg-1 / 0
    const int mu = d == 0 ? -1 : (d - 1) / 2;
    const int nsite = d == 0 ? A.vol : A.vol / A.agg[mu];
    cpx<R> acc[CB_MAXO];
#pragma unroll
    for (int q = 0; q < CB_MAXO; ++q) acc[q] = cpx<R>();
    for (int base = 0; base < nsite; base += CB_CHUNK) {
        const int cnt = nsite - base < CB_CHUNK ? nsite - base : CB_CHUNK;
        // stage P(x) rows and H(x) columns
        for (int t = threadIdx.x; t < cnt * (ntv + n2); t += blockDim.x) {
            const int sl = t % cnt, item = t / cnt;
            // face site enumeration: local index over the face, expanded to the aggregate
            int l = base + sl;
            if (d != 0) {
                // local coordinates with l_mu fixed (no run-time indexed arrays)
                int rem = l, ln = 0, st = 1;
#pragma unroll
                for (int nu = 0; nu < 4; ++nu) {
                    int x;
                    if (nu == mu) {
                        x = (d & 1) ? A.agg[nu] - 1 : 0;
                    } else {
                        x = rem % A.agg[nu];
                        rem /= A.agg[nu];
                    }
                    ln += x * st;
                    st *= A.agg[nu];
                }
                l = ln;
            }
            int lc[4], c[4];
            const int s = agg_site(g, A, a, l, lc);
            site_coords(g, s, c);
            cpx<R> v[12];
            if (item < ntv) {
                Spinor<R>::load(P.p[item], V, s, v);
                for (int k = 0; k < 12; ++k) sP[((size_t)sl * 12 + k) * ntv + item] = v[k];
            } else {
                const int col = item - ntv, cp = col / ntv, jp = col % ntv;
                directional_column<R>(g, A, U, clov, P.p[jp], cp, d, s, c, v);
                for (int k = 0; k < 12; ++k) sH[((size_t)sl * n2 + col) * 12 + k] = v[k];
            }
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < CB_MAXO; ++q) {
            const int o = threadIdx.x + q * blockDim.x;
            if (o < n2 * n2) {
                const int row = o % n2, col = o / n2;
                const int cr = row / ntv, jr = row % ntv;
                cpx<R> t = acc[q];
                for (int sl = 0; sl < cnt; ++sl) {
                    const cpx<R> *pr = sP + ((size_t)sl * 12 + cr * 6) * ntv + jr;   // component k at pr[k * ntv]
                    const cpx<R> *hc = sH + ((size_t)sl * n2 + col) * 12 + cr * 6;
#pragma unroll
                    for (int k = 0; k < 6; ++k) cmac_conj(t, pr[(size_t)k * ntv], hc[k]);
                }
                acc[q] = t;
            }
        }
        __syncthreads();
    }
    cpx<R> *out = Dc + ((size_t)d * A.n + a) * n2 * n2;
#pragma unroll
    for (int q = 0; q < CB_MAXO; ++q) {
        const int o = threadIdx.x + q * blockDim.x;
        if (o < n2 * n2) out[o] = acc[q];   // o = col*n2 + row: column-major block
    }
}

template <typename R>
void build_coarse(Ctx &c, const void *const *P, void *Dc) {
    AggGeom A = make_agg(c, c.prm.agg);
    const int ntv = c.prm.n_tv;
    MG_REQUIRE(4 * ntv * ntv <= CB_THREADS * CB_MAXO, MGEIG_EINVAL);
    PtrList p{};
    for (int j = 0; j < ntv; ++j) p.p[j] = P[j];
    const size_t smem = (size_t)CB_CHUNK * (ntv + 2 * ntv) * 12 * sizeof(cpx<R>);
    MG_CUDA(cudaFuncSetAttribute(coarse_build_kernel<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    const void *U = sizeof(R) == 8 ? c.U64.p : c.U32.p;
    const void *C = sizeof(R) == 8 ? c.clov64.p : c.clov32.p;
    TimeScope ts(c.timer, K_COARSE_BUILD, (double)ntv * c.g.V * 24 * sizeof(R) * 2);
    coarse_build_kernel<R><<<A.n * 9, CB_THREADS, smem, c.stream>>>(c.g, A, U, C, p, ntv, static_cast<cpx<R> *>(Dc));
    MG_CHECK_LAUNCH();
}

// ---------------------------------------------------------------------------
// coarse apply Y = (Q_c - sigma) X = (gamma5^c D_c - sigma) X of n vectors at once
//
// One CTA per coarse site.  A thread owns 16 bytes of rows (two FP32 rows, one FP64 row) and
// RPT of the vectors and goes through the columns of all nine hops in order, one running
// sum per row and vector; a link block and the neighbour's vectors come to shared memory
// one hop ahead of their use, so a link is read from memory once for all vectors.  FMAs and
// shared-memory reads take about the same time (per two columns and warp 64 FMA
// instructions and 6 reads at RPT = 4), the links of 16^3 x 32 (59 MB) as long as either
// from HBM.  The former form, one thread per row, read every link once per vector.  12
// vectors at 16^3 x 32: 391 us -> 22.4 us.

// asynchronous copy of B bytes
template <int B>
__device__ __forceinline__ void copy_async(void *smem, const void *gmem) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    if constexpr (B == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem));
    else asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(s), "l"(gmem), "n"(B));
}

template <typename R, int RPT>
__global__ void __launch_bounds__(sizeof(R) == 4 ? 160 : 576)
coarse_apply_many_kernel(int nagg, int ntv, int n, bool x16, const cpx<R> *__restrict__ Dc, const int *__restrict__ nbr,
                         R sigma, const cpx<R> *__restrict__ X, cpx<R> *__restrict__ Y) {
    using V16 = typename V16Of<R>::T;
    constexpr int ROWS = 16 / (int)sizeof(cpx<R>);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int n2 = 2 * ntv, units = n2 / ROWS, site = blockIdx.x;
    const int blk = n2 * n2, hop = blk + n * n2;   // values of one hop's buffer: links, then the vectors [r][n2]
    cpx<R> *buf = reinterpret_cast<cpx<R> *>(smem_raw);
    auto fetch_hop = [&](int d) {
        cpx<R> *dst = buf + (size_t)(d & 1) * hop;
        const cpx<R> *src = Dc + ((size_t)d * nagg + site) * blk;
        for (int e = threadIdx.x; e < blk / ROWS; e += blockDim.x) copy_async<16>(dst + e * ROWS, src + e * ROWS);
        const cpx<R> *x = X + (size_t)__ldg(nbr + (size_t)d * nagg + site) * n2;
        dst += blk;
        if (sizeof(R) == 8 || x16) {
            for (int e = threadIdx.x; e < n * units; e += blockDim.x) {
                const int r = e / units, j = (e - r * units) * ROWS;
                copy_async<16>(dst + r * n2 + j, x + (size_t)r * nagg * n2 + j);
            }
        } else {
            for (int e = threadIdx.x; e < n * n2; e += blockDim.x) {
                const int r = e / n2, j = e - r * n2;
                copy_async<8>(dst + e, x + (size_t)r * nagg * n2 + j);
            }
        }
        asm volatile("cp.async.commit_group;\n" ::);
    };
    fetch_hop(0);
    const int g = threadIdx.x / units, p = threadIdx.x - g * units;
    const bool on = g * RPT < n;
    int ro[RPT];   // where the thread's vectors start in a hop's buffer (repeats for vectors beyond n)
#pragma unroll
    for (int r = 0; r < RPT; ++r) ro[r] = blk + min(g * RPT + r, n - 1) * n2;
    cpx<R> acc[RPT][ROWS];
    for (int d = 0; d < 9; ++d) {
        if (d < 8) {
            fetch_hop(d + 1);
            asm volatile("cp.async.wait_group 1;\n" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;\n" ::: "memory");
        }
        __syncthreads();
        const cpx<R> *h = buf + (size_t)(d & 1) * hop;
        if (on) {
#pragma unroll 2
            for (int j = 0; j < n2; j += ROWS) {   // as many columns as a 16-byte read of a vector holds
                V16 b[ROWS];
#pragma unroll
                for (int u = 0; u < ROWS; ++u) b[u] = reinterpret_cast<const V16 *>(h)[(j + u) * units + p];
#pragma unroll
                for (int r = 0; r < RPT; ++r) {
                    const V16 xv = *reinterpret_cast<const V16 *>(h + ro[r] + j);
                    const cpx<R> *xc = reinterpret_cast<const cpx<R> *>(&xv);
#pragma unroll
                    for (int u = 0; u < ROWS; ++u) {
                        const cpx<R> *bc = reinterpret_cast<const cpx<R> *>(&b[u]);
#pragma unroll
                        for (int q = 0; q < ROWS; ++q) cmac(acc[r][q], bc[q], xc[u]);
                    }
                }
            }
        }
        __syncthreads();   // the buffer is free for hop d + 2
    }
    if (!on) return;
#pragma unroll
    for (int r = 0; r < RPT; ++r) {
        if (g * RPT + r >= n) break;
#pragma unroll
        for (int q = 0; q < ROWS; ++q) {
            const int row = p * ROWS + q;
            const size_t o = ((size_t)(g * RPT + r) * nagg + site) * n2 + row;
            cpx<R> t = acc[r][q];
            if (row >= ntv) t = -t;
            Y[o] = t - sigma * X[o];
        }
    }
}

template <typename R, int RPT>
static void launch_coarse_many(Ctx &c, double sigma, const cpx<R> *X, cpx<R> *Y, int n) {
    const int ntv = c.prm.n_tv, n2 = 2 * ntv;
    const int threads = (n2 * (int)sizeof(cpx<R>) / 16 * ((n + RPT - 1) / RPT) + 31) / 32 * 32;
    const size_t smem = (size_t)2 * (n2 + n) * n2 * sizeof(cpx<R>);
    MG_CUDA(cudaFuncSetAttribute(coarse_apply_many_kernel<R, RPT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    TimeScope ts(c.timer, K_COARSE_APPLY, (double)c.nagg * (9.0 * n2 * n2 + (double)n * 2 * n2) * sizeof(cpx<R>));
    coarse_apply_many_kernel<R, RPT><<<c.nagg, threads, smem, c.stream>>>(
        c.nagg, ntv, n, (reinterpret_cast<uintptr_t>(X) & 15) == 0, static_cast<const cpx<R> *>(c.Dc.p), c.cnbr.as<int>(),
        (R)sigma, X, Y);
    MG_CHECK_LAUNCH();
}

// Y = (Q_c - sigma) X for n vectors back to back (24 a launch at most), the operator in the
// level precision.  Fewer vectors a thread where there are few of them, so that the threads
// of a site do not run out
template <typename R>
void coarse_apply_many(Ctx &c, double sigma, const void *Xv, void *Yv, int n) {
    MG_REQUIRE(c.cnbr.p != nullptr && c.Dc.p != nullptr, MGEIG_ENOTSETUP);
    for (int r0 = 0; r0 < n; r0 += 24) {
        const int m = std::min(24, n - r0);
        const cpx<R> *x = static_cast<const cpx<R> *>(Xv) + (size_t)r0 * c.coarse_ncpx();
        cpx<R> *y = static_cast<cpx<R> *>(Yv) + (size_t)r0 * c.coarse_ncpx();
        if (m <= 4) launch_coarse_many<R, 1>(c, sigma, x, y, m);
        else if (sizeof(R) == 8 || m <= 8) launch_coarse_many<R, 2>(c, sigma, x, y, m);
        else if constexpr (sizeof(R) == 4) launch_coarse_many<R, 4>(c, sigma, x, y, m);
    }
}
template void coarse_apply_many<float>(Ctx &, double, const void *, void *, int);
template void coarse_apply_many<double>(Ctx &, double, const void *, void *, int);

// one vector, the operator in the form the context stores it
template <typename R>
void coarse_apply(Ctx &c, double sigma, const void *x, void *y) {
    if (sizeof(R) == 4 && c.prm.coarse_links != MGEIG_LINKS_LEVEL) coarse_apply_links16(c, sigma, x, y);
    else coarse_apply_many<R>(c, sigma, x, y, 1);
}

// ---------------------------------------------------------------------------
// SAP: one colour of blocks; CTA = one block, thread = one site (FP64: or a cluster, below)

// FP32: the block's forward links (two rows, 3 float4 per link) are staged in
// shared memory once and serve every MR step (the backward link of an in-block
// hop is the forward link of the in-block neighbour); two CTAs fit an SM.
// FP64: the links come from L2, an MR step's FP64 arithmetic takes far longer.
template <typename R> struct SapBounds { static constexpr int minb = 1; };
template <> struct SapBounds<float> { static constexpr int minb = 2; };

template <typename R>
__global__ void __launch_bounds__(256, SapBounds<R>::minb)
sap_kernel(Geom g, AggGeom B, int colour, R sigma, const void *__restrict__ U,
           const void *__restrict__ clov, const void *__restrict__ rhs, int rhs_g5, void *z, int mr_iters) {
    constexpr bool stage = sizeof(R) == 4;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    // component-major (rho[k][vol], slink[mu][3][vol]): consecutive threads read
    // consecutive words, without the 4-way bank conflicts of a site-major layout
    cpx<R> *rho = reinterpret_cast<cpx<R> *>(smem_raw);       // [12][vol]
    float4 *slink = reinterpret_cast<float4 *>(smem_raw + (size_t)B.vol * 12 * sizeof(cpx<R>));   // [4][3][vol]
    const int bv = B.vol;
    __shared__ R red[3 * 32];   // MR step sums, in the kernel's precision
    // the grid covers the blocks of one colour: blocks 2i and 2i + 1 differ in
    // colour (an even number of blocks per direction), CTA i takes the one of
    // this sweep's colour
    int b = 2 * blockIdx.x;
    {
        int r = b, bsum = 0;
        for (int mu = 0; mu < 4; ++mu) { bsum += r % B.cdims[mu]; r /= B.cdims[mu]; }
        if ((bsum & 1) != colour) b += 1;
    }
    const int V = g.V;
    const int l = threadIdx.x;
    const bool active = l < B.vol;
    int lc[4] = {0, 0, 0, 0}, c[4] = {0, 0, 0, 0}, s = 0;
    if (active) {
        s = agg_site(g, B, b, l, lc);
        site_coords(g, s, c);
    }
    cpx<R> e[12];
#pragma unroll
    for (int k = 0; k < 12; ++k) e[k] = cpx<R>();
    if (stage && active) {
        const float4 *ug = static_cast<const float4 *>(U);
        for (int mu = 0; mu < 4; ++mu)
            for (int e = 0; e < 3; ++e) slink[(mu * 3 + e) * bv + l] = ug[((size_t)mu * 3 + e) * V + s];
    }
    // residual of D_sigma z = rhs on this block (z read with its global neighbours)
    if (active) {
        cpx<R> up[6], lo[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) { up[k] = cpx<R>(); lo[k] = cpx<R>(); }
#pragma unroll
        for (int mu = 0; mu < 4; ++mu) {
            int ph;
            cpx<R> u[9], psi[12];
            int n = neighbor(g, s, c, mu, true, &ph);
            Gauge<R>::load(U, V, mu, s, u);
            Spinor<R>::load(z, V, n, psi);
            hop_accumulate<R>(mu, true, u, psi, (R)ph, up, lo);
            n = neighbor(g, s, c, mu, false, &ph);
            Gauge<R>::load(U, V, mu, n, u);
            Spinor<R>::load(z, V, n, psi);
            hop_accumulate<R>(mu, false, u, psi, (R)ph, up, lo);
        }
        cpx<R> zs[12], dz[12], bb[12];
        Spinor<R>::load(z, V, s, zs);
        clover_apply<R>(clov, V, s, zs, dz);
        Spinor<R>::load(rhs, V, s, bb);
        const R half = R(0.5);
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            cpx<R> du = dz[k] - half * up[k] - sigma * zs[k];
            cpx<R> dl = dz[6 + k] - half * lo[k] + sigma * zs[6 + k];
            cpx<R> bu = bb[k], bl = rhs_g5 ? -bb[6 + k] : bb[6 + k];
            rho[k * bv + l] = bu - du;
            rho[(6 + k) * bv + l] = bl - dl;
        }
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    for (int it = 0; it < mr_iters; ++it) {
        // q = D_sigma restricted to the block (Dirichlet) applied to rho
        cpx<R> q[12], rl[12];
        R qr_re = 0, qr_im = 0, qq = 0;
        if (active) {
            cpx<R> up[6], lo[6];
#pragma unroll
            for (int k = 0; k < 6; ++k) { up[k] = cpx<R>(); lo[k] = cpx<R>(); }
#pragma unroll
            for (int mu = 0; mu < 4; ++mu) {
#pragma unroll
                for (int f = 0; f < 2; ++f) {
                    const bool fwd = f == 0;
                    const int lm = lc[mu] + (fwd ? 1 : -1);
                    if (lm < 0 || lm >= B.agg[mu]) continue;
                    int ln = l + (fwd ? 1 : -1) * (mu == 0 ? 1 : mu == 1 ? B.agg[0] : mu == 2 ? B.agg[0] * B.agg[1]
                                                                                              : B.agg[0] * B.agg[1] * B.agg[2]);
                    cpx<R> u[9], psi[12];
                    if constexpr (stage) {
                        const float4 *q = slink + (size_t)mu * 3 * bv + (fwd ? l : ln);
                        const float4 a = q[0], b = q[bv], cc = q[2 * bv];
                        u[0] = cpx<R>(a.x, a.y); u[1] = cpx<R>(a.z, a.w); u[2] = cpx<R>(b.x, b.y);
                        u[3] = cpx<R>(b.z, b.w); u[4] = cpx<R>(cc.x, cc.y); u[5] = cpx<R>(cc.z, cc.w);
                        u[6] = conj(u[1] * u[5] - u[2] * u[4]);
                        u[7] = conj(u[2] * u[3] - u[0] * u[5]);
                        u[8] = conj(u[0] * u[4] - u[1] * u[3]);
                    } else {
                        int ph;
                        Gauge<R>::load(U, V, mu, fwd ? s : neighbor(g, s, c, mu, false, &ph), u);
                    }
#pragma unroll
                    for (int k = 0; k < 12; ++k) psi[k] = rho[k * bv + ln];
                    hop_accumulate<R>(mu, fwd, u, psi, (R)1, up, lo);
                }
            }
#pragma unroll
            for (int k = 0; k < 12; ++k) rl[k] = rho[k * bv + l];
            clover_apply<R>(clov, V, s, rl, q);
            const R half = R(0.5);
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                q[k] = q[k] - half * up[k] - sigma * rl[k];
                q[6 + k] = q[6 + k] - half * lo[k] + sigma * rl[6 + k];
            }
#pragma unroll
            for (int k = 0; k < 12; ++k) {
                qr_re += q[k].re * rl[k].re + q[k].im * rl[k].im;
                qr_im += q[k].re * rl[k].im - q[k].im * rl[k].re;
                qq += q[k].re * q[k].re + q[k].im * q[k].im;
            }
        }
        for (int o = 16; o > 0; o >>= 1) {
            qr_re += __shfl_xor_sync(0xffffffffu, qr_re, o);
            qr_im += __shfl_xor_sync(0xffffffffu, qr_im, o);
            qq += __shfl_xor_sync(0xffffffffu, qq, o);
        }
        if (lane == 0) { red[3 * w] = qr_re; red[3 * w + 1] = qr_im; red[3 * w + 2] = qq; }
        __syncthreads();   // all reads of rho for this step are done, partials visible
        R A_re = 0, A_im = 0, A_qq = 0;
        for (int i = 0; i < nw; ++i) { A_re += red[3 * i]; A_im += red[3 * i + 1]; A_qq += red[3 * i + 2]; }
        const cpx<R> alpha = A_qq > 0 ? cpx<R>(A_re / A_qq, A_im / A_qq) : cpx<R>();
        if (active) {
#pragma unroll
            for (int k = 0; k < 12; ++k) {
                cmac(e[k], alpha, rl[k]);
                rho[k * bv + l] = rl[k] - alpha * q[k];
            }
        }
        __syncthreads();
    }
    if (active) {
        cpx<R> zs[12];
        Spinor<R>::load(z, V, s, zs);
#pragma unroll
        for (int k = 0; k < 12; ++k) zs[k] = zs[k] + e[k];
        Spinor<R>::store(z, V, s, zs);
    }
}

// FP64 where there are few blocks.  What bounds a sweep is the FP64 pipe (a warp's instruction
// holds its scheduler for 64 clocks) of the schedulers that have work: 16 blocks of 256 sites at
// 8^3 x 16 took 464 us a sweep as 16 CTAs with a thread a site.  So a block is a cluster of CTAs
// with 32 sites each, and a site's work is cut into four threads of four warps: warp w takes the
// two hops of direction w and then the three components 3w .. 3w + 2 of everything else.  A
// sweep at 8^3 x 16 takes 147 us in this form (240 in clusters with a thread a site).
// A neighbour in another CTA of the cluster is read from that one's shared memory; every
// thread gets the sums of the MR step in the same order.
__device__ __forceinline__ unsigned cluster_map(unsigned smem_addr, int rank) {
    unsigned a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_addr), "r"(rank));
    return a;
}
__device__ __forceinline__ cpx<double> ld_cluster(unsigned a) {
    cpx<double> v;
    asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];" : "=d"(v.re), "=d"(v.im) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ double ld_cluster1(unsigned a) {
    double v;
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// out = rows I0 .. I0 + 2 of a 6x6 Hermitian block (packed as in hermitian6_apply, entry pairs V
// apart) times x
template <int I0>
__device__ __forceinline__ void hermitian6_rows(const double2 *p, int V, const cpx<double> x[6], cpx<double> out[3]) {
    const double2 d0 = p[(size_t)(I0 / 2) * V], d1 = p[(size_t)(I0 / 2 + 1) * V];
    const double dg[3] = {I0 ? d0.y : d0.x, I0 ? d1.x : d0.y, I0 ? d1.y : d1.x};
#pragma unroll
    for (int i = I0; i < I0 + 3; ++i) {
        cpx<double> acc = dg[i - I0] * x[i];
#pragma unroll
        for (int j = 0; j < 6; ++j) {
            if (j == i) continue;
            const double2 t = p[(size_t)(3 + (i < j ? offdiag_index(i, j) : offdiag_index(j, i))) * V];
            if (i < j) cmac(acc, cpx<double>(t.x, t.y), x[j]);
            else cmac_conj(acc, cpx<double>(t.x, t.y), x[j]);
        }
        out[i - I0] = acc;
    }
}

// The components 6 blk + I0 .. + 2 of D_sigma x: x the six components of chirality blk, hops the
// sites' four hop sums, [direction][12][32]
template <int I0>
__device__ __forceinline__ void dsigma_rows(const double2 *clov, int V, int blk, double sigma, const cpx<double> *hops,
                                            const cpx<double> x[6], cpx<double> out[3]) {
    hermitian6_rows<I0>(clov + (size_t)blk * 18 * V, V, x, out);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const cpx<double> *h = hops + (6 * blk + I0 + j) * 32;
        const cpx<double> t = (h[0] + h[12 * 32]) + (h[24 * 32] + h[36 * 32]);
        out[j] = out[j] - 0.5 * t - (blk ? -sigma : sigma) * x[I0 + j];
    }
}

// The hops of direction mu, without the -1/2: part[k * 32] for the 12 components.  f and b say
// which of them there are, phase_f and phase_b are 1 or -1, psi_f(k) and psi_b(k) the
// neighbours' components
template <class PF, class PB>
__device__ __forceinline__ void sap_hops(int mu, bool f, bool b, int phase_f, int phase_b, const void *U, int V, int s,
                                         int sb, PF psi_f, PB psi_b, cpx<double> *part) {
    using C = cpx<double>;
    C hf[6], hb[6], u[9], psi[12], t[6], h[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) hf[k] = hb[k] = C();
    if (f) {
        Gauge<double>::load(U, V, mu, s, u);
#pragma unroll
        for (int k = 0; k < 12; ++k) psi[k] = psi_f(k);
        spin_B<double>(mu, psi + 6, t);
#pragma unroll
        for (int k = 0; k < 6; ++k) h[k] = psi[k] - t[k];
        su3_mul<double>(u, h, hf);
        su3_mul<double>(u, h + 3, hf + 3);
        if (phase_f < 0) {
#pragma unroll
            for (int k = 0; k < 6; ++k) hf[k] = -hf[k];
        }
    }
    if (b) {
        Gauge<double>::load(U, V, mu, sb, u);
#pragma unroll
        for (int k = 0; k < 12; ++k) psi[k] = psi_b(k);
        spin_B<double>(mu, psi + 6, t);
#pragma unroll
        for (int k = 0; k < 6; ++k) h[k] = psi[k] + t[k];
        su3_dag_mul<double>(u, h, hb);
        su3_dag_mul<double>(u, h + 3, hb + 3);
        if (phase_b < 0) {
#pragma unroll
            for (int k = 0; k < 6; ++k) hb[k] = -hb[k];
        }
    }
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        part[k * 32] = hf[k] + hb[k];
        h[k] = hb[k] - hf[k];
    }
    spin_Bdag<double>(mu, h, t);
#pragma unroll
    for (int k = 0; k < 6; ++k) part[(6 + k) * 32] = t[k];
}

__global__ void __launch_bounds__(128, 2)
sap_f64_cluster_kernel(Geom g, AggGeom B, int colour, double sigma, const void *__restrict__ U, const double2 *__restrict__ clov,
               const cpx<double> *__restrict__ rhs, int rhs_g5, cpx<double> *z, int mr_iters, int cs) {
    using C = cpx<double>;
    __shared__ double2 rho_s[12 * 32], part_s[4 * 12 * 32];
    __shared__ double red[4 * 3];   // the warps' sums of the MR step
    C *rho = reinterpret_cast<C *>(rho_s), *part = reinterpret_cast<C *>(part_s);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int rank = blockIdx.x % cs;
    int b = 2 * (blockIdx.x / cs);   // of blocks b and b + 1 the one of this sweep's colour
    {
        int r = b, bsum = 0;
        for (int mu = 0; mu < 4; ++mu) { bsum += r % B.cdims[mu]; r /= B.cdims[mu]; }
        if ((bsum & 1) != colour) b += 1;
    }
    const int V = g.V, l = rank * 32 + lane;
    const bool active = l < B.vol;
    const int blk = w >> 1, k0 = 3 * w;   // own components: chirality blk, k0 .. k0 + 2
    int lc[4] = {0, 0, 0, 0}, c[4] = {0, 0, 0, 0}, s = 0;
    // the in-block neighbours of direction w, -1 where there is none
    int lf = -1, lb = -1, sb = 0;
    C x[6], q[3], e[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) e[j] = q[j] = C();
    // residual of D_sigma z = rhs on this block (z read with its global neighbours)
    if (active) {
        s = agg_site(g, B, b, l, lc);
        site_coords(g, s, c);
        const int step = w == 0 ? 1 : w == 1 ? B.agg[0] : w == 2 ? B.agg[0] * B.agg[1] : B.agg[0] * B.agg[1] * B.agg[2];
        const int lw = w == 0 ? lc[0] : w == 1 ? lc[1] : w == 2 ? lc[2] : lc[3];
        if (lw + 1 < B.agg[w]) lf = l + step;
        if (lw > 0) lb = l - step;
        int pf, pb;
        const int sf = neighbor(g, s, c, w, true, &pf);
        sb = neighbor(g, s, c, w, false, &pb);
        sap_hops(w, true, true, pf, pb, U, V, s, sb, [&](int k) { return z[(size_t)k * V + sf]; },
                 [&](int k) { return z[(size_t)k * V + sb]; }, part + w * 12 * 32 + lane);
    }
    __syncthreads();
    if (active) {
#pragma unroll
        for (int k = 0; k < 6; ++k) x[k] = z[(size_t)(6 * blk + k) * V + s];
        if (w & 1) dsigma_rows<3>(clov + s, V, blk, sigma, part + lane, x, q);
        else dsigma_rows<0>(clov + s, V, blk, sigma, part + lane, x, q);
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const C r = rhs[(size_t)(k0 + j) * V + s];
            rho[(k0 + j) * 32 + lane] = (rhs_g5 && blk ? -r : r) - q[j];
        }
    }
    cluster_sync();
    const unsigned rho0 = (unsigned)__cvta_generic_to_shared(rho), red0 = (unsigned)__cvta_generic_to_shared(red);
    const unsigned nf = lf >= 0 ? cluster_map(rho0, lf >> 5) + (lf & 31) * (unsigned)sizeof(C) : 0;
    const unsigned nb = lb >= 0 ? cluster_map(rho0, lb >> 5) + (lb & 31) * (unsigned)sizeof(C) : 0;
    for (int it = 0; it < mr_iters; ++it) {
        // q = D_sigma restricted to the block (Dirichlet) applied to rho
        if (active)
            sap_hops(w, lf >= 0, lb >= 0, 1, 1, U, V, s, sb,
                     [&](int k) { return ld_cluster(nf + k * 32 * (unsigned)sizeof(C)); },
                     [&](int k) { return ld_cluster(nb + k * 32 * (unsigned)sizeof(C)); }, part + w * 12 * 32 + lane);
        __syncthreads();
        double qr_re = 0, qr_im = 0, qq = 0;
        if (active) {
#pragma unroll
            for (int k = 0; k < 6; ++k) x[k] = rho[(6 * blk + k) * 32 + lane];
            if (w & 1) dsigma_rows<3>(clov + s, V, blk, sigma, part + lane, x, q);
            else dsigma_rows<0>(clov + s, V, blk, sigma, part + lane, x, q);
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const C r = w & 1 ? x[3 + j] : x[j];
                qr_re += q[j].re * r.re + q[j].im * r.im;
                qr_im += q[j].re * r.im - q[j].im * r.re;
                qq += q[j].re * q[j].re + q[j].im * q[j].im;
            }
        }
        for (int o = 16; o > 0; o >>= 1) {
            qr_re += __shfl_xor_sync(0xffffffffu, qr_re, o);
            qr_im += __shfl_xor_sync(0xffffffffu, qr_im, o);
            qq += __shfl_xor_sync(0xffffffffu, qq, o);
        }
        if (lane == 0) { red[3 * w] = qr_re; red[3 * w + 1] = qr_im; red[3 * w + 2] = qq; }
        cluster_sync();   // all reads of rho for this step are done, partials visible
        // lane 8 v + r: value v of CTA r (cs <= 8), then over the CTAs; alpha = (re, im) / qq
        // with one division for both
        const int v = lane >> 3, r = lane & 7;
        double t = 0;
        if (v < 3 && r < cs) {
            const unsigned a = cluster_map(red0, r) + v * (unsigned)sizeof(double);
            t = (ld_cluster1(a) + ld_cluster1(a + 24)) + (ld_cluster1(a + 48) + ld_cluster1(a + 72));
        }
        for (int o = 4; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        const double A_qq = __shfl_sync(0xffffffffu, t, 16);
        t = A_qq > 0 ? t / A_qq : 0.0;
        const C alpha(__shfl_sync(0xffffffffu, t, 0), __shfl_sync(0xffffffffu, t, 8));
        if (active) {
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const C r = w & 1 ? x[3 + j] : x[j];
                cmac(e[j], alpha, r);
                rho[(k0 + j) * 32 + lane] = r - alpha * q[j];
            }
        }
        cluster_sync();
    }
    if (active) {
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            C &zk = z[(size_t)(k0 + j) * V + s];
            zk = zk + e[j];
        }
    }
}

// Whether an FP64 sweep of nblk blocks of nw groups of 32 sites takes the form in clusters.  Its
// work is about 1.4 times that of the form with a thread a site (sums of the hops' parts,
// distributed shared memory), but the groups are spread evenly over the SMs; there a group is a
// warp, an SM gets whole blocks, and fewer than four warps leave schedulers idle.  Both sides count
// the groups of the SM that has most.  Measured, a sweep (a thread a site, in clusters):
//   8^3 x 16 in 4^4 blocks 466, 146 us     8^3 x 16 in 2^4 blocks 232, 148 us
//   16^2 x 8 x 16 in 4^4 466, 298 us       16^3 x 24 in 4^4 930, 793 us
//   16^4 in 4^4 467, 568 us                16^3 x 32 in 4^4 932, 1064 us
//   12^3 x 24 in 3^4 360, 438 us           24^3 x 48 in 4^4 4191, 5166 us
static bool sap_in_clusters(int nblk, int nw, int sms) {
    const int site = std::max(4, (nblk + sms - 1) / sms * nw), cluster = (nblk * nw + sms - 1) / sms;
    return 7 * cluster < 5 * site;
}

template <typename R>
void sap_sweep(Ctx &c, int colour, double sigma, const void *rhs, bool rhs_gamma5, void *z) {
    AggGeom B = make_agg(c, c.prm.sap_block);
    MG_REQUIRE(B.vol <= 1024, MGEIG_EINVAL);
    const int nw = (B.vol + 31) / 32;
    MG_REQUIRE(nw <= 8, MGEIG_ECUDA);   // 256 threads a CTA, eight CTAs a cluster
    // half the sites: z read+write, rhs, links, clover (from HBM once per sweep)
    const double site_bytes = 12 * 2 * sizeof(R) * 3 + (sizeof(R) == 8 ? 576 : 192) + 72 * sizeof(R);
    TimeScope ts(c.timer, sizeof(R) == 8 ? K_SAP_F64 : K_SAP_F32, site_bytes * c.g.V / 2);
    MG_REQUIRE(B.cdims[0] % 2 == 0, MGEIG_EINVAL);
    if (sizeof(R) == 8 && sap_in_clusters(B.n / 2, nw, c.sms)) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(B.n / 2 * nw);
        cfg.blockDim = dim3(128);
        cfg.stream = c.stream;
        cudaLaunchAttribute at = {};
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = nw;
        at.val.clusterDim.y = at.val.clusterDim.z = 1;
        cfg.attrs = &at;
        cfg.numAttrs = 1;
        MG_CUDA(cudaLaunchKernelEx(&cfg, sap_f64_cluster_kernel, c.g, B, colour, sigma, (const void *)c.U64.p,
                                   (const double2 *)c.clov64.p, (const cpx<double> *)rhs, rhs_gamma5 ? 1 : 0,
                                   (cpx<double> *)z, c.prm.sap_mr_iters, nw));
    } else {
        const size_t smem = (size_t)B.vol * 12 * (sizeof(cpx<R>) + (sizeof(R) == 4 ? sizeof(float4) : 0));
        MG_CUDA(cudaFuncSetAttribute(sap_kernel<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        sap_kernel<R><<<B.n / 2, nw * 32, smem, c.stream>>>(c.g, B, colour, (R)sigma, sizeof(R) == 8 ? c.U64.p : c.U32.p,
                                                            sizeof(R) == 8 ? c.clov64.p : c.clov32.p, rhs,
                                                            rhs_gamma5 ? 1 : 0, z, c.prm.sap_mr_iters);
    }
    MG_CHECK_LAUNCH();
}

#define INST(R)                                                                              \
    template void restrict_vec<R>(Ctx &, const void *const *, const void *, void *);         \
    template void prolong_vec<R>(Ctx &, const void *const *, const void *, void *);          \
    template void build_coarse<R>(Ctx &, const void *const *, void *);                       \
    template void coarse_apply<R>(Ctx &, double, const void *, void *);                      \
    template void sap_sweep<R>(Ctx &, int, double, const void *, bool, void *);
INST(double)
INST(float)
#undef INST

}  // namespace mgeig
