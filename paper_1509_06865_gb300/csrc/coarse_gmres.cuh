// Coarse-grid solve of the two-grid cycle (Sec. 2: restarted GMRES as the
// coarse solver for Q_c) as ONE persistent cooperative launch: every Arnoldi
// step runs on the device, with no host round trip.
//
// It solves (Q_c - sigma) e = r_c, A = Q_c - sigma = gamma5^c D_c - sigma.
//  * Deflation (k > 0): W = [P^dag w_1 .. P^dag w_k] are the coarse images of the
//    test vectors (the current eigenvector approximations of Algorithm 1), the
//    directions on which A becomes nearly singular when sigma approaches their
//    eigenvalues.  With E^-1 = (W^dag A W)^-1 (host-computed) and
//    Pi = 1 - A W E^-1 W^dag:  e = W E^-1 W^dag r_c + (1 - W E^-1 W^dag A) y,
//    where Pi A y = Pi r_c.
//  * GMRES runs on gamma5^c Pi A y = gamma5^c Pi r_c, i.e. on the D_c form
//    (gamma5^c A = D_c - sigma gamma5^c, Eq. 2.6 with a shift), whose spectrum
//    lies in the right half plane instead of around the origin.
//
// Everything is kept in the D_c form (g5 = gamma5^c): gA v = g5 A v = D_c v - sigma g5 v,
// GW_l = g5 W_l, GAW_l = g5 A W_l (signs only, so no value changes).
//
// Grid: G co-resident blocks; block b owns a contiguous slice of rb coarse rows.  Every vector the block only ever reads or writes on its own rows (the
// Krylov basis V_i, the products GU_i = gA s_i V_i, the right-hand side, the iterate,
// a work vector, and when room is left GW and GAW) lives in the block's shared
// memory (in a per-block slice of global scratch when the coarse grid is too large
// for that); only the vector being multiplied goes to global memory (`pub`), where
// the matvecs of the neighbouring blocks read it.
//
// One Arnoldi step, classical Gram-Schmidt with a second pass, two grid-wide
// reductions:
//   gu    = gA s_j V_j                         (matvec of pub, see below)
//   R1:   a_l = <GW_l, gu>, b_i = <s_i V_i, gu>, f_l = <s_j V_j, GAW_l>
//   t     = E^-1 a;  h1_i = b_i - sum_l F_il t_l   (F_il = <s_i V_i, GAW_l>)
//   w1    = gu - GAW t - sum_i h1_i s_i V_i;  pub <- w1
//   R2:   h2_i = <s_i V_i, w1>, ||w1||^2  (||w2||^2 = ||w1||^2 - ||h2||^2)
//   V_j+1 = w1 - sum_i h2_i s_i V_i  (own rows only)
// The next matvec reads w1 from pub, complete on every block after the R2
// barrier, and corrects it on its own rows with the stored products:
// gA s_j+1 V_j+1 = s_j+1 (gA w1 - sum_i h2_i GU_i).  So no block ever reads a
// vector that another block is still writing, with two grid barriers per step.
//
// The matvec does not need what follows from R2, so after that barrier the block
// splits: CG_MV threads multiply, the others gather R2, finish V_j+1 (slices in shared
// memory; else all threads do, after the matvec) and run the Givens rotations (a serial
// chain) beside them.
//
// What bounds it: latency.  At 16^3 x 32 (20480 rows, 59 MB of FP32 links, L2 resident)
// a step of the former kernel took 48 us: 18 in a matvec whose eight lanes a row went
// through the nine hops one after another, twice (135 rows on 128 groups); 9 in the two
// barriers; 8 gathering partial sums that lay [block][value], a sector a value; 6 in three
// rounds of inner products; the rest in serial scalar work.  In this form it takes 18 us
// (5 in the matvec, 4 in the barriers; a whole solve of 24 steps 1.12 -> 0.44 ms).  Blocks of
// more rows are bound by memory: at 24^3 x 48 (683 rows, slices in global memory) a step takes
// 92 us, at 32^3 x 64 (2156 rows) 273, of which the links need 139 at the HBM rate.
//
// Partial sums go to a [slot][G] buffer (consecutive reductions use disjoint
// slots): after each barrier a few lanes a value read them contiguously, in the same
// order in every block, so all blocks hold bit-identical scalars and run the Givens
// rotations and the triangular solve redundantly.  Basis vectors stay unnormalised
// with one scale factor each.
//
// The grid barrier counts arrivals and spins on the count with a clock64() budget; on
// expiry it raises a sticky error word (the kernel then returns without further
// waits) that the host reads at its next synchronisation (MGEIG_ETIMEOUT).
#pragma once

#include <type_traits>

#include "half16.cuh"
#include "internal.h"

namespace mgeig {

constexpr int CG_THREADS = 640;                   // 96 registers a thread: a matvec thread has 12 loads in flight
constexpr int CG_MV = 544;                        // threads of the matvec (eight for each of 68 row pairs); the others
                                                  // finish the step before
constexpr int CG_POST = CG_THREADS - CG_MV;
constexpr int CG_MAXG = 256;                      // blocks at most
constexpr int CG_NBR_SITES = 64;                  // coarse sites of a block's staged neighbour table
constexpr int CG_MAXM = COARSE_PERSISTENT_MAXM;   // restart length limit
constexpr int CG_MAXK = 24;                       // deflation vectors (= max N_tv)
static_assert(CG_MAXM <= 32, "one lane per Hessenberg row");
// partial-sum regions of consecutive reductions never overlap
constexpr int WS = 2 * CG_MAXK + CG_MAXM + 2;     // values of one reduction
constexpr int OFF_S1 = 0, OFF_S2 = WS, OFF_N = 2 * WS, OFF_P = 2 * WS + 2;
constexpr int CG_SLOTS = OFF_P + CG_MAXK;
// shared memory a block may use in all (static + dynamic), with a reserve
constexpr size_t CG_SMEM_LIMIT = 227 * 1024 - 1024;

struct CGState {
    unsigned int count;   // barrier arrivals of the running launch (0 between launches)
    unsigned int exits;   // blocks that have left it (0 between launches)
    int status;           // sticky: 0 ok, 1 barrier timeout, 2 breakdown
    int iters;            // accumulated Arnoldi steps of all solves
};
static_assert(sizeof(CGState) == 16, "CGState lives in one reduction slot");

template <typename R> struct Pod2;
template <> struct Pod2<float> { using T = float2; };
template <> struct Pod2<double> { using T = double2; };

__host__ __device__ constexpr size_t align16(size_t b) { return (b + 15) / 16 * 16; }

template <typename R>
struct CGArgs {
    int nagg, ntv, n;              // coarse sites, test vectors, rows = nagg * 2 ntv
    int rb;                        // rows per block (the last block may own fewer)
    int nslice;                    // owned-row vectors per block: V (m+1), GU (m), rhs, x, w
    int slices;                    // matvec threads that share a row; 1: none do
    int stage_sites;               // coarse sites whose neighbour vectors are staged at a time (0: none)
    int part_size;                 // values of the matvec's parts in shared memory (0: none)
    int smem_slices, smem_defl;    // 1: the slices / copies of GW, GAW live in shared memory
    const cpx<R> *Dc;              // [9][nagg][col][row]
    const void *L16;               // 16-bit links [9][nagg][re|im][row][col] (16-bit kernels)
    const float *Ls;               // their scales [9][nagg]
    const int *nbr;                // [9][nagg] neighbour aggregates
    R sigma;
    const cpx<R> *b;               // r_c
    cpx<R> *x;                     // e (output)
    cpx<R> *pub;                   // the vector being multiplied (n)
    cpx<R> *gslices;               // nslice vectors, block by block, when the slices are not in shared memory
    int k;                         // deflation vectors (0: none)
    const cpx<R> *W, *AW;          // k x n each
    const double2 *Einv;           // k x k, row-major
    typename Pod2<R>::T *partial;  // [CG_SLOTS][G]
    CGState *st;
    int m, maxiter;
    double tol;
    long long timeout;
};

// Barrier number *bar of a launch: every block adds one to the count and waits for
// G times the barrier's number.  One atomic without a reply and one 16-byte poll that
// brings the status along (the former arrive, reset, release and status read were
// four round trips to L2).  Returns false once the status is set.
__device__ __forceinline__ bool grid_sync(CGState *st, unsigned int nblocks, unsigned int &bar, long long timeout) {
    __syncthreads();
    __shared__ int ok;
    bar += nblocks;
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(&st->count, 1u);
        const long long t0 = clock64();
        int status;
        for (;;) {
            int4 s;   // the words of the state in order
            asm volatile("ld.volatile.global.v4.u32 {%0, %1, %2, %3}, [%4];"
                         : "=r"(s.x), "=r"(s.y), "=r"(s.z), "=r"(s.w) : "l"(st) : "memory");
            status = s.z;
            if (status != 0 || (int)((unsigned int)s.x - bar) >= 0) break;
            if (clock64() - t0 > timeout) { status = 1; atomicCAS(&st->status, 0, 1); break; }
        }
        __threadfence();
        ok = status == 0;
    }
    __syncthreads();
    return ok;
}

// Loads of data other blocks wrote before the last grid barrier bypass the
// (non-coherent) L1: ld.global.cg.
__device__ __forceinline__ cpx<float> ldcg(const cpx<float> *p) {
    float2 v = __ldcg(reinterpret_cast<const float2 *>(p));
    return cpx<float>(v.x, v.y);
}
__device__ __forceinline__ cpx<double> ldcg(const cpx<double> *p) {
    double2 v = __ldcg(reinterpret_cast<const double2 *>(p));
    return cpx<double>(v.x, v.y);
}

// The neighbour aggregate of hop d of site `site`: from the block's staged table
// (sites s0 .. s0 + CG_NBR_SITES - 1) when there is one, else from global memory.
template <typename R>
__device__ __forceinline__ int hop_nbr(const CGArgs<R> &a, const int *snb, int s0, int d, int site) {
    return snb ? snb[d * CG_NBR_SITES + site - s0] : __ldg(a.nbr + (size_t)d * a.nagg + site);
}

// The order of the FP32 sums is fixed, whatever the number of threads: the columns of a row
// and the vectors of a sum over vectors are added by residue mod 8, the rows of an inner
// product and the blocks of a grid-wide sum by residue mod 32 (a residue's terms one after
// another, then the residues in a tree), over rb = ceil(n / blocks) rows a block, one block
// per 128 rows at most.  The preconditioner's bits enter the setup's test vectors, and
// through them the 16-bit links, whose rounding turns a last-bit difference into one of
// 2^-9; and a truncated solve multiplies it by the condition number.  So every split below
// hands whole residues to its threads.

// the sum over LANES neighbouring lanes, pairs of neighbours first
template <int LANES>
__device__ __forceinline__ cpx<float> group_sum_up(cpx<float> v) {
#pragma unroll
    for (int o = 1; o < LANES; o <<= 1) {
        v.re += __shfl_xor_sync(0xffffffffu, v.re, o);
        v.im += __shfl_xor_sync(0xffffffffu, v.im, o);
    }
    return v;
}

// The sums over the columns of all nine hop blocks, (D_c v)[row], for the owned rows: eight
// threads share a pair of rows (16 bytes of a column; pairs start on even rows, so a block's
// first and last pair may be half its own), one column residue each, whose sums go to
// part[residue][row].  Consecutive threads take consecutive pairs of a column.  The block's
// neighbour vectors are staged in shared memory (xs [hop][site][n2]) while the first links
// are on their way, and a hop's links are loaded while the hop before is multiplied: the
// registers go to links in flight.  tid < CG_MV, all of them.
// FULL: n2 = 8 U, every load is unconditional.
template <int U, bool FULL>   // U: columns of one residue in a block, at least n2 / 8
__device__ __forceinline__ void qmatvec_pairs(const CGArgs<float> &a, const cpx<float> *v, cpx<float> *xs,
                                              cpx<float> *part, int r0, int nr, const int *snb, int s0, int nsites,
                                              int tid) {
    const int n2 = FULL ? 8 * U : 2 * a.ntv, ntv = n2 / 2, np = (nr + (r0 & 1) + 1) >> 1;
    const bool on = tid < 8 * np;                 // the threads left over repeat thread 0's loads
    const int q = on ? tid / np : 0, p = on ? tid - q * np : 0;
    const int row = (r0 & ~1) + 2 * p, site = row / n2;
    const size_t hop = (size_t)a.nagg * n2 * ntv;   // in units of 16 bytes
    const float4 *pb = reinterpret_cast<const float4 *>(a.Dc) + ((size_t)site * n2 + q) * ntv + ((row - site * n2) >> 1);
    float4 b0[U], b1[U];
    auto load = [&](float4(&w)[U]) {
#pragma unroll
        for (int u = 0; u < U; ++u)
            w[u] = FULL || 8 * u + q < n2 ? __ldcg(pb + 4 * u * n2) : make_float4(0.f, 0.f, 0.f, 0.f);
        pb += hop;
    };
    load(b0);
    for (int e = tid; e < 9 * nsites * ntv; e += CG_MV) {   // 16 bytes (two columns) at a time
        const int ds = e / ntv, j = e - ds * ntv, d = ds / nsites, sq = ds - d * nsites;
        reinterpret_cast<float4 *>(xs)[e] =
            __ldcg(reinterpret_cast<const float4 *>(v + (size_t)hop_nbr(a, snb, s0, d, s0 + sq) * n2) + j);
    }
    asm volatile("bar.sync 2, %0;" ::"n"(CG_MV) : "memory");
    cpx<float> t0[2], t1[2];   // the pair's rows, even and odd terms
    const cpx<float> *px = xs + (size_t)(site - s0) * n2 + q;
    auto multiply = [&](const float4(&w)[U]) {
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (FULL || 8 * u + q < n2) {
                const cpx<float> x = px[8 * u];
                cmac(t0[u & 1], cpx<float>(w[u].x, w[u].y), x);
                cmac(t1[u & 1], cpx<float>(w[u].z, w[u].w), x);
            }
        px += (size_t)nsites * n2;
    };
#pragma unroll 1
    for (int d = 0; d < 8; d += 2) {
        load(b1);
        multiply(b0);
        load(b0);
        multiply(b1);
    }
    multiply(b0);
    if (!on) return;
    const int i = row - r0;
    if (i >= 0) part[(size_t)q * nr + i] = t0[0] + t0[1];
    if (i + 1 < nr) part[(size_t)q * nr + i + 1] = t1[0] + t1[1];
}

// The neighbour vectors of the ns sites from c0 on to shared memory, [hop][site][n2], 16 bytes
// (two columns) at a time
__device__ __forceinline__ void stage_neighbours(const CGArgs<float> &a, const cpx<float> *v, cpx<float> *xs,
                                                 const int *snb, int s0, int c0, int ns, int tid) {
    const int ntv = a.ntv;
    for (int e = tid; e < 9 * ns * ntv; e += CG_MV) {
        const int ds = e / ntv, j = e - ds * ntv, d = ds / ns, sq = ds - d * ns;
        const unsigned to = (unsigned)__cvta_generic_to_shared(reinterpret_cast<float4 *>(xs) + e);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(to),
                     "l"(reinterpret_cast<const float4 *>(v + (size_t)hop_nbr(a, snb, s0, d, c0 + sq) * 2 * ntv) + j)
                     : "memory");
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
}

// The same for blocks of more rows, a chunk of coarse sites at a time (as many as there is room
// for the neighbour vectors), in passes of CG_MV / T pairs, T threads a pair with 8 / T residues
// each.  The links come from HBM here, so one or two hops are in flight while one is
// multiplied, across the passes too.  PART: consecutive threads take consecutive pairs, so that a
// column is read in one piece, and the residues meet in part[8][rows of a chunk] after the
// last pass; else, where there is no room for that, a pair's threads are neighbouring lanes
// and add with shuffles.  The sums go to out.  At 32^3 x 64 (2156 rows a block, 943 MB of links)
// a product takes 154 us, 6.1 TB/s; with a thread a row, four loads at a time, it took 258,
// with a pair's threads on neighbouring lanes 240, with a barrier after each pass 233.
template <int U, bool FULL, int T, bool PART>
__device__ __forceinline__ void qmatvec_passes(const CGArgs<float> &a, const cpx<float> *v, cpx<float> *xs,
                                               cpx<float> *part, cpx<float> *out, int r0, int nr, const int *snb, int s0,
                                               int nsites, int tid) {
    constexpr int PAIRS = CG_MV / T, PASS = 2 * PAIRS, RES = 8 / T;   // pairs and rows of a pass, residues of a thread
    constexpr int AHEAD = FULL ? 2 : 1;   // hops in flight while one is multiplied, as the registers go
    const int n2 = FULL ? 8 * U : 2 * a.ntv, ntv = n2 / 2, q = PART ? tid / PAIRS : tid % T;
    const size_t hop = (size_t)a.nagg * n2 * ntv;   // in units of 16 bytes
    const float4 *D4 = reinterpret_cast<const float4 *>(a.Dc), *pb;
    const int prows = a.stage_sites * n2;   // rows of a chunk at most
    float4 buf[AHEAD + 1][RES * U];
    auto seek = [&](int row) {
        const int site = row / n2;
        pb = D4 + ((size_t)site * n2 + q) * ntv + ((row - site * n2) >> 1);
    };
    auto load = [&](float4(&w)[RES * U]) {
#pragma unroll
        for (int e = 0; e < RES * U; ++e)
            w[e] = FULL || T * e + q < n2 ? __ldcg(pb + T * e * ntv) : make_float4(0.f, 0.f, 0.f, 0.f);
        pb += hop;
    };
    for (int c0 = s0; c0 < s0 + nsites; c0 += a.stage_sites) {
        const int ns = min(a.stage_sites, s0 + nsites - c0);
        const int first = max(r0 & ~1, c0 * n2), last = min(r0 + nr, (c0 + ns) * n2);
        if (c0 > s0) asm volatile("bar.sync 2, %0;" ::"n"(CG_MV) : "memory");   // xs is free
        int row = first + 2 * (PART ? tid % PAIRS : tid / T);
        seek(min(row, last - 1) & ~1);   // the threads left over repeat the last pair's loads
        load(buf[0]);
        if (AHEAD == 2) load(buf[1]);
        stage_neighbours(a, v, xs, snb, s0, c0, ns, tid);
        asm volatile("bar.sync 2, %0;" ::"n"(CG_MV) : "memory");
        for (int p0 = first; p0 < last; p0 += PASS, row += PASS) {
            cpx<float> t0[RES][2], t1[RES][2];   // the pair's rows, even and odd terms of a residue
            const cpx<float> *px = xs + (size_t)((min(row, last - 1) & ~1) / n2 - c0) * n2 + q;
            auto multiply = [&](const float4(&w)[RES * U]) {
#pragma unroll
                for (int e = 0; e < RES * U; ++e)   // column T e + q
                    if (FULL || T * e + q < n2) {
                        const cpx<float> x = px[T * e];
                        const int r = e % RES, u = e / RES;
                        cmac(t0[r][u & 1], cpx<float>(w[e].x, w[e].y), x);
                        cmac(t1[r][u & 1], cpx<float>(w[e].z, w[e].w), x);
                    }
                px += (size_t)ns * n2;
            };
            const bool more = p0 + PASS < last;
            auto next_pass = [&] { if (more) seek(min(row + PASS, last - 1) & ~1); };
            if constexpr (AHEAD == 2) {   // hop d in buffer d mod 3
#pragma unroll 1
                for (int d = 0; d < 6; d += 3) {
                    load(buf[2]);
                    multiply(buf[0]);
                    load(buf[0]);
                    multiply(buf[1]);
                    load(buf[1]);
                    multiply(buf[2]);
                }
                load(buf[2]);
                next_pass();
                multiply(buf[0]);
                if (more) load(buf[0]);
                multiply(buf[1]);
                if (more) load(buf[1]);
                multiply(buf[2]);
            } else {
#pragma unroll 1
                for (int d = 0; d < 8; d += 2) {
                    load(buf[1]);
                    multiply(buf[0]);
                    load(buf[0]);
                    multiply(buf[1]);
                }
                next_pass();
                if (more) load(buf[1]);
                multiply(buf[0]);
#pragma unroll
                for (int e = 0; e < RES * U; ++e) buf[0][e] = buf[1][e];
            }
            if constexpr (PART) {
                cpx<float> *mine = part + (size_t)q * prows + row - first;
                if (row < last) {
#pragma unroll
                    for (int r = 0; r < RES; ++r) {
                        mine[(size_t)r * T * prows] = t0[r][0] + t0[r][1];
                        mine[(size_t)r * T * prows + 1] = t1[r][0] + t1[r][1];
                    }
                }
            } else {
                cpx<float> y0[RES], y1[RES];
#pragma unroll
                for (int r = 0; r < RES; ++r) {
                    y0[r] = group_sum_up<T>(t0[r][0] + t0[r][1]);
                    y1[r] = group_sum_up<T>(t1[r][0] + t1[r][1]);
                }
#pragma unroll
                for (int o = 1; o < RES; o <<= 1)
#pragma unroll
                    for (int r = 0; r < RES; r += 2 * o) { y0[r] = y0[r] + y0[r + o]; y1[r] = y1[r] + y1[r + o]; }
                const int i = row - r0;
                if (q == 0 && row < last) {
                    if (i >= 0) out[i] = y0[0];
                    if (i + 1 < nr) out[i + 1] = y1[0];
                }
            }
        }
        if constexpr (PART) {
            asm volatile("bar.sync 2, %0;" ::"n"(CG_MV) : "memory");
            for (int t = max(r0, first) + tid; t < last; t += CG_MV) {
                const cpx<float> *pp = part + t - first;
                auto p2 = [&](int r) { return pp[(size_t)r * prows] + pp[(size_t)(r + 1) * prows]; };
                out[t - r0] = (p2(0) + p2(2)) + (p2(4) + p2(6));
            }
        }
    }
}

__device__ __forceinline__ void qmatvec_part(const CGArgs<float> &a, const cpx<float> *v, cpx<float> *xs,
                                             cpx<float> *part, cpx<float> *out, int r0, int nr, const int *snb, int s0,
                                             int nsites, int tid) {
    if (a.slices == 8) {
        if (a.ntv == 20) qmatvec_pairs<5, true>(a, v, xs, part, r0, nr, snb, s0, nsites, tid);   // the default
        else qmatvec_pairs<6, false>(a, v, xs, part, r0, nr, snb, s0, nsites, tid);
    } else {
        auto passes = [&](auto part_room) {
            constexpr bool P = decltype(part_room)::value;
            if (a.ntv == 20) qmatvec_passes<5, true, 8, P>(a, v, xs, part, out, r0, nr, snb, s0, nsites, tid);
            else if (a.ntv <= 8) qmatvec_passes<2, false, 4, P>(a, v, xs, part, out, r0, nr, snb, s0, nsites, tid);
            else if (a.ntv <= 16) qmatvec_passes<4, false, 8, P>(a, v, xs, part, out, r0, nr, snb, s0, nsites, tid);
            else qmatvec_passes<6, false, 8, P>(a, v, xs, part, out, r0, nr, snb, s0, nsites, tid);
        };
        if (a.part_size > 0) passes(std::true_type{});
        else passes(std::false_type{});
    }
}

// FP64: the columns of a row are cut into a.slices contiguous parts, each of them one thread's, so
// that a whole matvec is one run of independent loads per thread, or a few such runs that leave
// few threads without work in the last.
__device__ __forceinline__ void qmatvec_part(const CGArgs<double> &a, const cpx<double> *v, cpx<double> *,
                                             cpx<double> *part, cpx<double> *out, int r0, int nr, const int *snb, int s0,
                                             int, int tid) {
    constexpr int U = 2;
    const int ntv = a.ntv, n2 = 2 * ntv, CP = 9 * ntv, S = a.slices;
    const double2 *D2 = reinterpret_cast<const double2 *>(a.Dc), *v2 = reinterpret_cast<const double2 *>(v);
    const size_t next_hop = (size_t)(a.nagg - 1) * n2 * n2;
    int sl = tid / nr, p = tid - sl * nr;   // the thread's part and row
#pragma unroll 1
    for (; sl < S; p += CG_MV, sl += p / nr, p %= nr) {
        const int q0 = sl * CP / S, q1 = (sl + 1) * CP / S;
        const int row = r0 + p, site = row / n2, rin = row - site * n2;
        int d = q0 / ntv, jp = q0 - d * ntv;
        const double2 *pb = D2 + (((size_t)d * a.nagg + site) * n2 + 2 * jp) * n2 + rin;
        const double2 *px = v2 + (size_t)hop_nbr(a, snb, s0, d, site) * n2 + 2 * jp;
        cpx<double> t0, t1;
        for (int q = q0; q < q1; q += U) {
            double2 b0[U], b1[U], x0[U], x1[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (q + u < q1) {
                    b0[u] = __ldcg(pb);
                    b1[u] = __ldcg(pb + n2);
                    x0[u] = __ldcg(px);
                    x1[u] = __ldcg(px + 1);
                    pb += 2 * n2;
                    px += 2;
                    if (++jp == ntv && ++d < 9) {
                        jp = 0;
                        pb += next_hop;
                        px = v2 + (size_t)hop_nbr(a, snb, s0, d, site) * n2;
                    }
                } else {
                    b0[u] = b1[u] = x0[u] = x1[u] = make_double2(0.0, 0.0);
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                cmac(t0, cpx<double>(b0[u].x, b0[u].y), cpx<double>(x0[u].x, x0[u].y));
                cmac(t1, cpx<double>(b1[u].x, b1[u].y), cpx<double>(x1[u].x, x1[u].y));
            }
        }
        (S > 1 ? part + (size_t)sl * nr : out)[p] = t0 + t1;
    }
}

// The same sums with 16-bit links (FP32 vectors and arithmetic): eight lanes share a row,
// lane q takes the column pairs p = q (mod 8) of the real and imaginary planes, and every hop
// block's sum is multiplied by the block's scale.  Passes, staged neighbour vectors and two
// hops in flight as above.  At 32^3 x 64 a product takes 128 us (472 MB of links), at 24^3 x 48
// 44; 192 and 65 with one hop in flight and the vectors read from L2, 242 and 86 with none.
template <typename H>
__device__ __forceinline__ void qmatvec16(const CGArgs<float> &a, const cpx<float> *v, cpx<float> *xs, cpx<float> *out,
                                          int r0, int nr, const int *snb, int s0, int nsites, int tid) {
    using HP = typename H16<H>::P;
    constexpr int PASS = CG_MV / 8, U = (CG_MAXK + 7) / 8;   // pairs per lane (n2 / 2 <= CG_MAXK)
    struct Hop {
        HP re[U], im[U];
        float scale;
    };
    const int n2 = 2 * a.ntv, np = a.ntv, q = tid & 7;
    const size_t hop = (size_t)a.nagg * n2 * n2;   // in units of pairs
    const HP *pb;
    const float *ps;
    Hop b0, b1, b2;
    auto seek = [&](int row) {
        const int site = row / n2;
        pb = static_cast<const HP *>(a.L16) + ((size_t)site * 2 * n2 + row - site * n2) * np + q;
        ps = a.Ls + site;
    };
    auto load = [&](Hop &w) {
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (q + 8 * u < np) {
                w.re[u] = pb[8 * u];
                w.im[u] = pb[n2 * np + 8 * u];
            }
        w.scale = __ldg(ps);
        pb += hop;
        ps += a.nagg;
    };
    for (int c0 = s0; c0 < s0 + nsites; c0 += a.stage_sites) {
        const int ns = min(a.stage_sites, s0 + nsites - c0);
        const int first = max(r0, c0 * n2), last = min(r0 + nr, (c0 + ns) * n2);
        if (c0 > s0) asm volatile("bar.sync 2, %0;" ::"n"(CG_MV) : "memory");   // xs is free
        int row = first + (tid >> 3);
        seek(min(row, last - 1));   // the threads left over repeat the last row's loads
        load(b0);
        load(b1);
        stage_neighbours(a, v, xs, snb, s0, c0, ns, tid);
        asm volatile("bar.sync 2, %0;" ::"n"(CG_MV) : "memory");
        for (int p0 = first; p0 < last; p0 += PASS, row += PASS) {
            float ar = 0.f, ai = 0.f;
            const float4 *px = reinterpret_cast<const float4 *>(xs) + (size_t)(min(row, last - 1) / n2 - c0) * np + q;
            auto multiply = [&](const Hop &w) {
                float dr = 0.f, di = 0.f;
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    if (q + 8 * u < np) {
                        const float2 r = H16<H>::pair(w.re[u]), im = H16<H>::pair(w.im[u]);
                        const float4 x = px[8 * u];
                        dr = fmaf(r.x, x.x, dr); dr = fmaf(-im.x, x.y, dr);
                        di = fmaf(r.x, x.y, di); di = fmaf(im.x, x.x, di);
                        dr = fmaf(r.y, x.z, dr); dr = fmaf(-im.y, x.w, dr);
                        di = fmaf(r.y, x.w, di); di = fmaf(im.y, x.z, di);
                    }
                }
                ar = fmaf(w.scale, dr, ar);
                ai = fmaf(w.scale, di, ai);
                px += (size_t)ns * np;
            };
#pragma unroll 1
            for (int d = 0; d < 6; d += 3) {
                load(b2);
                multiply(b0);
                load(b0);
                multiply(b1);
                load(b1);
                multiply(b2);
            }
            load(b2);
            const bool more = p0 + PASS < last;
            if (more) seek(min(row + PASS, last - 1));
            multiply(b0);
            if (more) load(b0);
            multiply(b1);
            if (more) load(b1);
            multiply(b2);
            const cpx<float> y = group_sum_up<8>(cpx<float>(ar, ai));
            if (q == 0 && row < last) out[row - r0] = y;
        }
    }
}

// the sums of the kernel's link format LK (0: level precision, 1: BF16, 2: FP16)
template <typename R, int LK>
__device__ __forceinline__ void matvec_part(const CGArgs<R> &a, const cpx<R> *v, cpx<R> *xs, cpx<R> *part, cpx<R> *out,
                                            int r0, int nr, const int *snb, int s0, int nsites, int tid) {
    if constexpr (LK == 0) qmatvec_part(a, v, xs, part, out, r0, nr, snb, s0, nsites, tid);
    else if constexpr (LK == 1) qmatvec16<__nv_bfloat16>(a, v, xs, out, r0, nr, snb, s0, nsites, tid);
    else qmatvec16<__half>(a, v, xs, out, r0, nr, snb, s0, nsites, tid);
}

template <typename R>
__device__ __forceinline__ cpx<R> group_sum(cpx<R> v, int lanes) {
    for (int o = lanes >> 1; o > 0; o >>= 1) {
        v.re += __shfl_xor_sync(0xffffffffu, v.re, o);
        v.im += __shfl_xor_sync(0xffffffffu, v.im, o);
    }
    return v;
}

// How inner products and sums are shared among lanes.
//
// FP32: eight lanes an inner product or a grid-wide sum, each with four residues mod 32;
// L = 4 or 1 lanes a sum over vectors, with 8 / L residues mod 8.
//
// FP64: the pipe takes half a lane a cycle and scheduler, a warp's FP64 instruction 64
// cycles of it, so shuffle sums (an addition per lane and level) and half-empty warps are
// what costs: four lanes share each sum, in an order of their own.
template <typename R> struct Lanes;
template <> struct Lanes<float> {
    static constexpr int dot = 8, long_dot = 8;
    // sum over t < n of term(t, acc), q = lane in its group
    template <int L, typename F> __device__ __forceinline__ static cpx<float> dot_sum(int q, int n, F term) {
        static_assert(L == 8);
        cpx<float> r[4];
        for (int t = q; t < n; t += 32)
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (t + 8 * i < n) term(t + 8 * i, r[i]);
        return group_sum((r[0] + r[2]) + (r[1] + r[3]), 8);
    }
    // sum over t < n of conj(X[t]) Y[t] in the same order, sixteen loads at a time; the sign is changed in
    // rows from place `flip` on of their coarse site (row 0 is at place p0 of n2)
    __device__ __forceinline__ static cpx<float> dot_global(int q, int n, int p0, int n2, int flip, const cpx<float> *X,
                                                            const cpx<float> *Y) {
        cpx<float> r[4];
        const int step = 8 % n2;
        int p = (p0 + q) % n2;
        auto add = [&](cpx<float> &acc, cpx<float> x, cpx<float> y) {
            if (p >= flip) x = -x;
            p += step;
            if (p >= n2) p -= n2;
            acc.re += x.re * y.re + x.im * y.im;
            acc.im += x.re * y.im - x.im * y.re;
        };
        int t = q;
        for (; t + 56 < n; t += 64) {
            cpx<float> x[8], y[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) { x[i] = X[t + 8 * i]; y[i] = Y[t + 8 * i]; }
#pragma unroll
            for (int i = 0; i < 8; ++i) add(r[i & 3], x[i], y[i]);
        }
#pragma unroll
        for (int i = 0; i < 7; ++i)
            if (t + 8 * i < n) add(r[i & 3], X[t + 8 * i], Y[t + 8 * i]);
        return group_sum((r[0] + r[2]) + (r[1] + r[3]), 8);
    }
    // sum over the blocks b < G of the contiguous values src[b]
    __device__ __forceinline__ static cpx<float> grid_sum(const float2 *src, unsigned int G, int q, bool on) {
        cpx<float> r[4];
        constexpr int B = 5;   // all values of up to 160 blocks are loaded before they are added
        if (on)
            for (unsigned int b0 = 0; b0 < G; b0 += 32 * B) {
                float2 pv[4][B];
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int u = 0; u < B; ++u) {
                        const unsigned int b = b0 + q + 8 * i + 32 * u;
                        pv[i][u] = b < G ? __ldcg(src + b) : make_float2(0.f, 0.f);
                    }
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int u = 0; u < B; ++u) { r[i].re += pv[i][u].x; r[i].im += pv[i][u].y; }
            }
        return group_sum((r[0] + r[2]) + (r[1] + r[3]), 8);
    }
    // sum over l < n of term(l, acc): L lanes, two accumulators a residue (dual) or one
    template <int L, bool dual, typename F> __device__ __forceinline__ static cpx<float> vec_sum(int q, int n, F term) {
        cpx<float> r[8 / L];
        if constexpr (L == 1) {   // eight terms at a time, so that their loads are in flight together
            cpx<float> odd[8];
            auto eight = [&](int l, cpx<float>(&acc)[8]) {
                if (l + 4 <= n) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) term(l + i, acc[i]);
                    if (l + 8 <= n) {
#pragma unroll
                        for (int i = 4; i < 8; ++i) term(l + i, acc[i]);
                    } else {
#pragma unroll
                        for (int i = 4; i < 7; ++i)
                            if (l + i < n) term(l + i, acc[i]);
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < 3; ++i)
                        if (l + i < n) term(l + i, acc[i]);
                }
            };
            for (int l = 0; l < n; l += dual ? 16 : 8) {
                eight(l, r);
                if (dual && l + 8 < n) eight(l + 8, odd);
            }
            if (dual) {
#pragma unroll
                for (int i = 0; i < 8; ++i) r[i] = r[i] + odd[i];
            }
        } else {
#pragma unroll
            for (int i = 0; i < 8 / L; ++i) {
                cpx<float> a0, a1;
                int l = q + L * i;
                if (dual) {
                    for (; l + 8 < n; l += 16) { term(l, a0); term(l + 8, a1); }
                    if (l < n) term(l, a0);
                    r[i] = a0 + a1;
                } else {
                    for (; l < n; l += 8) term(l, a0);
                    r[i] = a0;
                }
            }
        }
#pragma unroll
        for (int o = 1; o < L; o <<= 1)
#pragma unroll
            for (int i = 0; i < 8 / L; ++i) {
                r[i].re += __shfl_xor_sync(0xffffffffu, r[i].re, o);
                r[i].im += __shfl_xor_sync(0xffffffffu, r[i].im, o);
            }
#pragma unroll
        for (int o = 1; o < 8 / L; o <<= 1)
#pragma unroll
            for (int i = 0; i < 8 / L; i += 2 * o) r[i] = r[i] + r[i + o];
        return r[0];
    }
};
template <> struct Lanes<double> {
    static constexpr int dot = 4, long_dot = 8;   // eight where a block has more rows, for more warps with work
    template <int L, typename F> __device__ __forceinline__ static cpx<double> dot_sum(int q, int n, F term) {
        cpx<double> r;
        for (int t = q; t < n; t += L) term(t, r);
        return group_sum(r, L);
    }
    __device__ __forceinline__ static cpx<double> dot_global(int q, int n, int p0, int n2, int flip, const cpx<double> *X,
                                                             const cpx<double> *Y) {
        constexpr int L = long_dot;
        cpx<double> r;
        const int step = L % n2;
        int p = (p0 + q) % n2;
        for (int t = q; t < n; t += L) {
            cpx<double> x = X[t];
            const cpx<double> y = Y[t];
            if (p >= flip) x = -x;
            p += step;
            if (p >= n2) p -= n2;
            r.re += x.re * y.re + x.im * y.im;
            r.im += x.re * y.im - x.im * y.re;
        }
        return group_sum(r, L);
    }
    __device__ __forceinline__ static cpx<double> grid_sum(const double2 *src, unsigned int G, int q, bool on) {
        cpx<double> r;
        constexpr int B = 8;
        if (on)
            for (unsigned int b0 = 0; b0 < G; b0 += 4 * B) {
                double2 pv[B];
#pragma unroll
                for (int u = 0; u < B; ++u) {
                    const unsigned int b = b0 + q + 4 * u;
                    pv[u] = b < G ? __ldcg(src + b) : make_double2(0.0, 0.0);
                }
#pragma unroll
                for (int u = 0; u < B; ++u) { r.re += pv[u].x; r.im += pv[u].y; }
            }
        return group_sum(r, 4);
    }
    template <int L, bool dual, typename F> __device__ __forceinline__ static cpx<double> vec_sum(int q, int n, F term) {
        cpx<double> r;
        for (int l = q; l < n; l += L) term(l, r);
        return group_sum(r, L);
    }
};

// Scalars (partial sums, Hessenberg matrix, Givens rotations, E^-1) are kept in
// the solver's own precision R: FP32 in the mixed-precision preconditioner,
// where FP64 arithmetic (1/64 of the FP32 rate on this part) held most warps at
// block barriers, FP64 in the all-FP64 path.
template <typename R, int LK>
__global__ void __launch_bounds__(CG_THREADS, 1) coarse_gmres_kernel(CGArgs<R> a) {
    using P = typename Pod2<R>::T;
    auto P2 = [](R x, R y) { return P{x, y}; };
    extern __shared__ __align__(16) unsigned char cg_dyn[];
    __shared__ P h[WS];                        // grid-wide sums of the first reduction (and of the single ones)
    __shared__ P hp[CG_MAXM + 2];              // of the second: the coefficients of the second pass, ||w1||^2
    __shared__ P F[CG_MAXM * CG_MAXK];         // F_il = <s_i V_i, GAW_l>
    __shared__ P hc[CG_MAXM];                  // h1_i s_i
    __shared__ P Rm[(CG_MAXM + 1) * CG_MAXM];  // rotated Hessenberg, column-major
    __shared__ R cs[CG_MAXM];
    __shared__ P sn[CG_MAXM], g[CG_MAXM + 1], y[CG_MAXM];
    __shared__ R scale[CG_MAXM + 1];
    __shared__ P Ei[CG_MAXK * CG_MAXK], t0[CG_MAXK], tc[CG_MAXK];
    __shared__ R bnorm, beta, nsum[32];
    __shared__ int stop;
    const unsigned int G = gridDim.x;
    const int tid = threadIdx.x, lane = tid & 31;
    const int rb = a.rb;
    const int r0 = min(a.n, (int)blockIdx.x * rb);
    const int r1 = min(a.n, r0 + rb);
    const int nr = r1 - r0;
    const int m = a.m, k = a.k, n2 = 2 * a.ntv;
    P *mypart = a.partial + blockIdx.x;   // value i of this block at mypart[i * G]
    unsigned int bar = 0;

    // owned-row slices: V_0..V_m, GU_0..GU_m-1, rhs, x, w
    cpx<R> *S = a.smem_slices ? reinterpret_cast<cpx<R> *>(cg_dyn) : a.gslices + (size_t)a.nslice * r0;
    const int ld = a.smem_slices ? rb : nr;
    auto Vv = [&](int i) { return S + (size_t)i * ld; };
    auto Uv = [&](int i) { return S + (size_t)(m + 1 + i) * ld; };
    cpx<R> *rhs = S + (size_t)(2 * m + 1) * ld;
    cpx<R> *xs = rhs + ld;
    cpx<R> *ws = xs + ld;
    // then the staged neighbour vectors (FP32), the matvec's parts ([slices][nr] when a.slices > 1)
    // and GW, GAW
    cpx<R> *stage = reinterpret_cast<cpx<R> *>(cg_dyn + (a.smem_slices ? align16((size_t)a.nslice * rb * sizeof(cpx<R>)) : 0));
    cpx<R> *part = stage + (size_t)9 * a.stage_sites * n2;
    cpx<R> *Dl = a.smem_defl ? part + a.part_size : nullptr;
    auto g5 = [&](int i, cpx<R> v) { return ((r0 + i) % n2) >= a.ntv ? -v : v; };
    // element i of GW_l and GAW_l
    auto GW = [&](int l, int i) { return Dl ? Dl[(size_t)l * rb + i] : g5(i, a.W[(size_t)l * a.n + r0 + i]); };
    auto GAW = [&](int l, int i) { return Dl ? Dl[(size_t)(k + l) * rb + i] : g5(i, a.AW[(size_t)l * a.n + r0 + i]); };

    // the neighbour table of the block's coarse sites, staged once
    __shared__ int snb[9 * CG_NBR_SITES];
    const int s0 = nr > 0 ? r0 / n2 : 0;
    const int nsites = nr > 0 ? (r1 - 1) / n2 - s0 + 1 : 0;
    const int *snb_p = nsites <= CG_NBR_SITES ? snb : nullptr;
    if (snb_p)
        for (int e = tid; e < 9 * nsites; e += CG_THREADS) {
            const int d = e / nsites, sl = e % nsites;
            snb[d * CG_NBR_SITES + sl] = __ldg(a.nbr + (size_t)d * a.nagg + s0 + sl);
        }
    for (int i = tid; i < k * k; i += CG_THREADS) Ei[i] = P2((R)a.Einv[i].x, (R)a.Einv[i].y);
    if (tid < CG_MAXK) { tc[tid] = P2(0, 0); t0[tid] = P2(0, 0); }
    if (Dl)
        for (int e = tid; e < k * nr; e += CG_THREADS) {
            const int l = e / nr, i = e % nr;
            Dl[(size_t)l * rb + i] = g5(i, a.W[(size_t)l * a.n + r0 + i]);
            Dl[(size_t)(k + l) * rb + i] = g5(i, a.AW[(size_t)l * a.n + r0 + i]);
        }

    // partial slot off + i <- sc(i) times the sum of val(i, t) over the owned rows t, i < cnt
    const bool wide = 4 * nr <= CG_THREADS;
    auto dots_by = [&](auto lanes, int off, int cnt, auto val, auto sc) {
        constexpr int L = decltype(lanes)::value, ngrp = CG_THREADS / L;
        for (int ib = 0; ib < cnt; ib += ngrp) {
            const int i = ib + tid / L;
            const cpx<R> acc =
                Lanes<R>::template dot_sum<L>(tid % L, i < cnt ? nr : 0, [&](int t, cpx<R> &r) { val(i, t, r); });
            if (i < cnt && tid % L == 0) mypart[(size_t)(off + i) * G] = P2(acc.re * sc(i), acc.im * sc(i));
        }
    };
    auto dots = [&](int off, int cnt, auto val, auto sc) {
        constexpr std::integral_constant<int, Lanes<R>::dot> few{};
        constexpr std::integral_constant<int, Lanes<R>::long_dot> many{};
        if (few.value == many.value || wide) dots_by(few, off, cnt, val, sc);
        else if constexpr (few.value != many.value) dots_by(many, off, cnt, val, sc);
    };
    // r += conj(p) q
    auto cdot = [](cpx<R> p, cpx<R> q, cpx<R> &r) {
        r.re += p.re * q.re + p.im * q.im;
        r.im += p.re * q.im - p.im * q.re;
    };
    // partial slot off + i <- sc(i) <X, Y> of the vectors that pick(i, X, Y, flip) names, i < cnt, `flip`: with the
    // sign of gamma5
    auto dots_global = [&](int off, int cnt, auto pick, auto sc) {
        constexpr int L = Lanes<R>::long_dot, ngrp = CG_THREADS / L;
        for (int ib = 0; ib < cnt; ib += ngrp) {
            const int i = ib + tid / L;
            const cpx<R> *X, *Y;
            bool flip;
            pick(min(i, cnt - 1), X, Y, flip);
            const cpx<R> acc = Lanes<R>::dot_global(tid % L, i < cnt ? nr : 0, r0 % n2, n2, flip ? a.ntv : n2, X, Y);
            if (i < cnt && tid % L == 0) mypart[(size_t)(off + i) * G] = P2(acc.re * sc(i), acc.im * sc(i));
        }
    };
    // dst[i] = sum of value off + i over the blocks, i < cnt, by `threads` threads, t < threads
    auto gather = [&](int off, int cnt, P *dst, int t, int threads) {
        constexpr int L = Lanes<R>::dot;
        const int ngrp = threads / L;
        for (int ib = 0; ib < cnt; ib += ngrp) {
            const int i = ib + t / L;
            const cpx<R> acc = Lanes<R>::grid_sum(a.partial + (size_t)(off + min(i, cnt - 1)) * G, G, t % L, i < cnt);
            if (i < cnt && t % L == 0) dst[i] = P2(acc.re, acc.im);
        }
    };
    // the partial sums of the block are in their slots: barrier, h = grid sums
    auto reduce = [&](int off, int cnt) -> bool {
        if (!grid_sync(a.st, G, bar, a.timeout)) return false;
        gather(off, cnt, h, tid, CG_THREADS);
        __syncthreads();
        return true;
    };
    // f(i, s) with s = sum of term(l, i, s) over l < cnt, once per owned row i: four lanes a
    // row where the threads suffice, else one
    auto rows_by = [&](auto lanes, auto dual, int t, int threads, int cnt, auto term, auto f) {
        constexpr int L = decltype(lanes)::value;
        for (int ib = 0; ib < nr; ib += threads / L) {
            const int i = ib + t / L;
            const cpx<R> s = Lanes<R>::template vec_sum<L, decltype(dual)::value>(
                t % L, i < nr ? cnt : 0, [&](int l, cpx<R> &acc) { term(l, i, acc); });
            if (i < nr && t % L == 0) f(i, s);
        }
    };
    constexpr std::integral_constant<int, 4> L4{};
    constexpr std::integral_constant<int, 1> L1{};
    constexpr std::true_type dual{};
    constexpr std::false_type single{};
    auto rows = [&](int cnt, auto term, auto f) {
        if (wide) rows_by(L4, dual, tid, CG_THREADS, cnt, term, f);
        else rows_by(L1, dual, tid, CG_THREADS, cnt, term, f);
    };
    auto C = [](P p) { return cpx<R>(p.x, p.y); };
    // finishes out = gA (s v): the parts (or the sum) of D_c v, the shift (own = v's owned
    // rows), minus sum_l h2_l s GU_l of the l < nu earlier products
    auto matvec_end = [&](R s, cpx<R> *out, const cpx<R> *own, int nu) {
        const int np = a.slices;
        auto base = [&](int i) {
            cpx<R> acc;
            if (np == 1) {
                acc = out[i];
            } else if (sizeof(R) == 8) {
                for (int l = 0; l < np; ++l) acc = acc + part[(size_t)l * nr + i];
            } else {   // the eight residues
                auto p2 = [&](int l) { return part[(size_t)l * nr + i] + part[(size_t)(l + 1) * nr + i]; };
                acc = (p2(0) + p2(2)) + (p2(4) + p2(6));
            }
            const R sg = ((r0 + i) % n2) >= a.ntv ? -a.sigma : a.sigma;
            return s * acc - (sg * s) * own[i];
        };
        rows(nu, [&](int l, int i, cpx<R> &acc) { cmac(acc, s * C(hp[l]), Uv(l)[i]); },
             [&](int i, cpx<R> u) { out[i] = base(i) - u; });
        __syncthreads();
    };
    // out = gA v of the published vector whose owned rows are `own`
    auto matvec = [&](cpx<R> *out, const cpx<R> *own) {
        if (tid < CG_MV) matvec_part<R, LK>(a, a.pub, stage, part, out, r0, nr, snb_p, s0, nsites, tid);
        __syncthreads();
        matvec_end(R(1), out, own, 0);
    };
    // dst = E^-1 h
    auto einv_h = [&](P *dst) {
        if constexpr (sizeof(R) == 4) {
            for (int i = tid; i < k; i += CG_THREADS) {
                R sr = 0, si = 0;
                for (int l = 0; l < k; ++l) {
                    P e = Ei[i * k + l], d = h[l];
                    sr += e.x * d.x - e.y * d.y;
                    si += e.x * d.y + e.y * d.x;
                }
                dst[i] = P2(sr, si);
            }
        } else {
            for (int ib = 0; ib < k; ib += CG_THREADS / 4) {
                const int i = ib + tid / 4;
                const cpx<R> t = Lanes<R>::template vec_sum<4, false>(
                    tid % 4, i < k ? k : 0, [&](int l, cpx<R> &acc) { cmac(acc, C(Ei[i * k + l]), C(h[l])); });
                if (i < k && tid % 4 == 0) dst[i] = P2(t.re, t.im);
            }
        }
        __syncthreads();
    };
    // column j of the Hessenberg matrix after the first pass, h1_i = b_i - sum_l F_il t_l, and h1_i s_i
    auto first_pass = [&](int j) {
        auto done = [&](int i, P b) {
            Rm[j * (CG_MAXM + 1) + i] = b;
            hc[i] = P2(b.x * scale[i], b.y * scale[i]);
        };
        if constexpr (sizeof(R) == 4) {
            for (int i = tid; i <= j; i += CG_THREADS) {
                P b = h[k + i];
                for (int l = 0; l < k; ++l) {
                    P f = F[i * CG_MAXK + l], t = tc[l];
                    b.x -= f.x * t.x - f.y * t.y;
                    b.y -= f.x * t.y + f.y * t.x;
                }
                done(i, b);
            }
        } else {
            const int i = tid / 4;   // j < 32: one pass
            const cpx<R> s = Lanes<R>::template vec_sum<4, false>(
                tid % 4, i <= j ? k : 0, [&](int l, cpx<R> &acc) { cmac(acc, C(F[i * CG_MAXK + l]), C(tc[l])); });
            if (i <= j && tid % 4 == 0) done(i, P2(h[k + i].x - s.re, h[k + i].y - s.im));
        }
        __syncthreads();
    };
    auto one = [](int) { return R(1); };
    // tc = E^-1 W^dag A x from the product gx = gA x
    auto deflation_coeffs = [&](const cpx<R> *gx) -> bool {
        dots(OFF_P, k, [&](int l, int t, cpx<R> &acc) { cdot(GW(l, t), gx[t], acc); }, one);
        if (!reduce(OFF_P, k)) return false;
        einv_h(tc);
        return true;
    };
    // sums over l of tc_l AW_l, from which those of GAW follow by a sign
    auto aw_t = [&](int l, int i, cpx<R> &acc) {
        cmac(acc, C(tc[l]), Dl ? Dl[(size_t)(k + l) * rb + i] : a.AW[(size_t)l * a.n + r0 + i]);
    };
    auto to_gaw = [&](int i, cpx<R> s) { return Dl ? s : g5(i, s); };
    auto publish = [&](const cpx<R> *v) {
        for (int i = tid; i < nr; i += CG_THREADS) a.pub[r0 + i] = v[i];
    };
    // partial slot <- ||v||^2 over the owned rows: sums of warps of 32 rows (of every 1024),
    // then the warps one after another
    auto norm_to = [&](const cpx<R> *v, int slot) {
        for (int w = tid >> 5; w < 32; w += CG_THREADS / 32) {
            R acc = 0;
            for (int t = 32 * w + lane; t < nr; t += 1024) {
                const cpx<R> q = v[t];
                acc += q.re * q.re + q.im * q.im;
            }
            for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            if (lane == 0) nsum[w] = acc;
        }
        __syncthreads();
        if (tid == 0) {
            R s2 = 0;
            for (int w = 0; w < 32; ++w) s2 += nsum[w];
            mypart[(size_t)slot * G] = P2(s2, 0);
        }
    };

    // rhs = gamma5^c Pi r_c, t0 = E^-1 W^dag r_c, x = 0.  The tolerance refers
    // to ||r_c||: when r_c lies mostly in span(W) the projected right-hand side
    // is small and needs no further reduction.
    for (int i = tid; i < nr; i += CG_THREADS) { rhs[i] = g5(i, a.b[r0 + i]); xs[i] = cpx<R>(); }
    __syncthreads();
    // ||r_c||^2 and W^dag r_c in one reduction
    dots(OFF_S1, k, [&](int l, int t, cpx<R> &acc) { cdot(GW(l, t), rhs[t], acc); }, one);
    norm_to(rhs, OFF_S1 + k);
    if (!reduce(OFF_S1, k + 1)) return;
    if (tid == 0) {
        bnorm = sqrt(h[k].x);
        stop = !(bnorm > 0) || !isfinite(bnorm);
    }
    if (k > 0) einv_h(t0);
    __syncthreads();
    if (k > 0) {
        rows(k, [&](int l, int i, cpx<R> &acc) { cmac(acc, C(t0[l]), GAW(l, i)); },
             [&](int i, cpx<R> s) { rhs[i] = rhs[i] - s; });
        __syncthreads();
    }
    const R tol_abs = (R)a.tol * bnorm;

    // V_j+1 = w1 - sum_i h2_i s_i V_i in place: a term, the end of a row
    auto v_term = [&](int l, int i, cpx<R> &acc) { cmac(acc, scale[l] * C(hp[l]), Vv(l)[i]); };
    auto v_put = [&](cpx<R> *vn) { return [vn](int i, cpx<R> s) { vn[i] = vn[i] - s; }; };
    // what follows the second reduction of step j, by the threads that do not multiply:
    // the coefficients, V_j+1 = w1 - sum_i h2_i s_i V_i on the owned rows (in place), and
    // in the last warp the Hessenberg column, its rotations and the stop test
    auto post = [&](int j) {
        const int t = tid - CG_MV;
        gather(OFF_S2, j + 2, hp, t, CG_POST);
        asm volatile("bar.sync 1, %0;" ::"n"(CG_POST) : "memory");
        cpx<R> *vn = Vv(j + 1);
        if (t < CG_POST - 32) {
            if (!a.smem_slices) return;   // all threads do it after the matvec
            if (sizeof(R) == 8) rows_by(L4, dual, t, CG_POST - 32, j + 1, v_term, v_put(vn));
            else rows_by(L1, dual, t, CG_POST - 32, j + 1, v_term, v_put(vn));
            return;
        }
        P *col = Rm + j * (CG_MAXM + 1);
        if constexpr (sizeof(R) == 4) {
            if (lane != 0) return;
            R n2s = hp[j + 1].x;
            for (int i = 0; i <= j; ++i) {
                col[i] = P2(col[i].x + hp[i].x, col[i].y + hp[i].y);
                n2s -= hp[i].x * hp[i].x + hp[i].y * hp[i].y;
            }
            const R nrm = sqrt(n2s > 0 ? n2s : R(0));
            P p = col[0], q;
            for (int i = 0; i < j; ++i) {   // previous rotations
                q = col[i + 1];
                const P sv = sn[i];
                const R c = cs[i];
                col[i] = P2(c * p.x + (sv.x * q.x - sv.y * q.y), c * p.y + (sv.x * q.y + sv.y * q.x));
                p = P2(c * q.x - (sv.x * p.x + sv.y * p.y), c * q.y - (sv.x * p.y - sv.y * p.x));
            }
            q = P2(nrm, 0);
            R ap = hypot(p.x, p.y), aq = hypot(q.x, q.y);
            R c, sr, si;
            if (aq == 0) { c = 1; sr = 0; si = 0; }
            else if (ap == 0) { c = 0; sr = 1; si = 0; }
            else {
                R tt = hypot(ap, aq);
                c = ap / tt;
                R ur = p.x / ap, ui = p.y / ap;          // s = (p/|p|) conj(q) / t
                sr = (ur * q.x + ui * q.y) / tt;
                si = (ui * q.x - ur * q.y) / tt;
            }
            cs[j] = c;
            sn[j] = P2(sr, si);
            col[j] = P2(c * p.x + (sr * q.x - si * q.y), c * p.y + (sr * q.y + si * q.x));
            col[j + 1] = P2(0, 0);
            P gj = g[j];
            g[j + 1] = P2(-(sr * gj.x + si * gj.y), -(sr * gj.y - si * gj.x));
            g[j] = P2(c * gj.x, c * gj.y);
            const R est = hypot(g[j + 1].x, g[j + 1].y);
            if (!isfinite(nrm) || !isfinite(est)) atomicCAS(&a.st->status, 0, 2);
            scale[j + 1] = nrm > 0 ? R(1) / nrm : R(0);
            stop = (est <= tol_abs) || nrm == 0 || !isfinite(est);
        } else {
            // the same on one warp with few FP64 instructions (64 cycles each here): lane c of
            // four takes component c of a rotation (0, 1: the rotated entry, 2, 3: the one
            // carried on), and the new rotation needs three reciprocal square roots
            R n2s = 0;
            if (lane <= j) {
                const P v = hp[lane];
                col[lane] = P2(col[lane].x + v.x, col[lane].y + v.y);
                n2s = v.x * v.x + v.y * v.y;
            }
            for (int o = 16; o > 0; o >>= 1) n2s += __shfl_xor_sync(0xffffffffu, n2s, o);
            n2s = hp[j + 1].x - n2s;
            if (!(n2s > 0) && isfinite(n2s)) n2s = 0;
            __syncwarp();
            const int c4 = lane & 3;
            R px = col[0].x, py = col[0].y;
            for (int i = 0; i < j; ++i) {   // previous rotations
                const P q = col[i + 1], sv = sn[i];
                // 0: c px + sx qx - sy qy   1: c py + sx qy + sy qx   2: c qx - sx px - sy py   3: c qy - sx py + sy px
                const R u = c4 == 0 ? px : c4 == 1 ? py : c4 == 2 ? q.x : q.y;
                const R v = c4 == 0 ? q.x : c4 == 1 ? q.y : c4 == 2 ? -px : -py;
                const R w = c4 == 0 ? -q.y : c4 == 1 ? q.x : c4 == 2 ? -py : px;
                const R r = fma(cs[i], u, fma(sv.x, v, sv.y * w));
                const R re = __shfl_sync(0xffffffffu, r, 0), im = __shfl_sync(0xffffffffu, r, 1);
                px = __shfl_sync(0xffffffffu, r, 2);
                py = __shfl_sync(0xffffffffu, r, 3);
                if (lane == 0) col[i] = P2(re, im);
            }
            const R ap2 = px * px + py * py, t2 = ap2 + n2s;
            const R it = rsqrt(t2), in = rsqrt(n2s), ia = rsqrt(ap2);
            const R nrm = n2s > 0 ? n2s * in : n2s;   // 0, inf and NaN stay
            R c = 1, sr = 0, si = 0, re = px, im = py;
            if (n2s != 0) {
                if (ap2 == 0) {
                    c = 0; sr = 1; re = nrm; im = 0;
                } else {
                    const R ait = ia * it, f = nrm * ait, d = t2 * ait;
                    c = ap2 * ait;               // |p| / t
                    sr = px * f; si = py * f;    // (p / |p|) nrm / t
                    re = px * d; im = py * d;    // (p / |p|) t
                }
            }
            if (lane == 0) {
                cs[j] = c;
                sn[j] = P2(sr, si);
                col[j] = P2(re, im);
                col[j + 1] = P2(0, 0);
                const P gj = g[j];
                const P gn = P2(-(sr * gj.x + si * gj.y), si * gj.x - sr * gj.y);
                g[j + 1] = gn;
                g[j] = P2(c * gj.x, c * gj.y);
                const R est = sqrt(gn.x * gn.x + gn.y * gn.y);
                if (!isfinite(nrm) || !isfinite(est)) atomicCAS(&a.st->status, 0, 2);
                scale[j + 1] = nrm > 0 ? in : R(0);
                stop = (est <= tol_abs) || nrm == 0 || !isfinite(est);
            }
        }
    };

    int its = 0;
    bool have_x = false;
    while (!stop && its < a.maxiter) {
        cpx<R> *v0 = Vv(0);
        // V0 = rhs - op(x)  (or rhs)
        if (have_x) {
            publish(xs);
            if (!grid_sync(a.st, G, bar, a.timeout)) return;   // x complete everywhere
            matvec(v0, xs);
            if (k > 0) {
                if (!deflation_coeffs(v0)) return;             // its barrier also ends the reads of pub
            } else if (!grid_sync(a.st, G, bar, a.timeout)) {
                return;                                        // every matvec done before pub changes
            }
            rows(k, aw_t, [&](int i, cpx<R> s) { v0[i] = rhs[i] - (v0[i] - to_gaw(i, s)); });
        } else {
            for (int i = tid; i < nr; i += CG_THREADS) v0[i] = rhs[i];
        }
        __syncthreads();
        publish(v0);
        for (int i = tid; i < nr; i += CG_THREADS) ws[i] = v0[i];
        norm_to(v0, OFF_N);
        if (!reduce(OFF_N, 1)) return;                         // also makes V0 visible in pub
        if (tid == 0) {
            beta = sqrt(h[0].x);
            stop = !(beta > tol_abs) || !isfinite(beta);
            if (!isfinite(beta)) atomicCAS(&a.st->status, 0, 2);
            scale[0] = beta > 0 ? R(1) / beta : R(0);
            g[0] = P2(beta, 0);
            for (int i = 1; i <= CG_MAXM; ++i) g[i] = P2(0, 0);
        }
        __syncthreads();
        if (stop) break;
        const int mm = min(m, a.maxiter - its);
        int kk = 0;
        bool conv = false;
        for (int j = 0;; ++j) {
            // GU_j = gA s_j V_j: the matvec of pub (= V_j before its second pass) while the
            // other threads finish step j - 1, then the correction by its second-pass
            // coefficients.  When step j - 1 was the last the product is not used (a faster
            // block may already write x to pub meanwhile)
            cpx<R> *uj = Uv(min(j, m - 1));
            if (tid < CG_MV) {
                if (j < mm) matvec_part<R, LK>(a, a.pub, stage, part, uj, r0, nr, snb_p, s0, nsites, tid);
            } else if (j > 0) {
                post(j - 1);
            }
            __syncthreads();
            kk = j;
            if (j > 0 && stop) { conv = true; break; }
            if (j == mm) break;
            // V_j, which with the slices in global memory would take the 64 threads of post() longer
            // than the matvec
            if (j > 0 && !a.smem_slices) rows(j, v_term, v_put(Vv(j)));
            matvec_end((R)scale[j], uj, ws, j);
            // reduction 1: a_l = <GW_l, gu>, b_i = <s_i V_i, gu>, f_l = <s_j V_j, GAW_l>
            const cpx<R> *vj = Vv(j);
            if (Dl) {   // value l is <X, Y> of two vectors in shared memory
                dots(OFF_S1, 2 * k + j + 1, [&](int l, int t, cpx<R> &acc) {
                    const cpx<R> *X = l < k ? Dl + (size_t)l * rb : l <= k + j ? Vv(l - k) : vj;
                    const cpx<R> *Y = l <= k + j ? uj : Dl + (size_t)(l - j - 1) * rb;
                    cdot(X[t], Y[t], acc);
                }, [&](int l) { return l < k ? R(1) : scale[l <= k + j ? l - k : j]; });
            } else {   // W and AW in global memory: the sign of gamma5 from the row's place in its site
                dots_global(OFF_S1, 2 * k + j + 1, [&](int l, const cpx<R> *&X, const cpx<R> *&Y, bool &flip) {
                    flip = l < k || l > k + j;
                    X = l < k ? a.W + (size_t)l * a.n + r0 : l <= k + j ? Vv(l - k) : vj;
                    Y = l <= k + j ? uj : a.AW + (size_t)(l - k - j - 1) * a.n + r0;
                }, [&](int l) { return l < k ? R(1) : scale[l <= k + j ? l - k : j]; });
            }
            if (!reduce(OFF_S1, 2 * k + j + 1)) return;
            // t = E^-1 a ; F row j ; h1_i = b_i - sum_l F_il t_l
            for (int l = tid; l < k; l += CG_THREADS) F[j * CG_MAXK + l] = h[k + j + 1 + l];
            if (k > 0) einv_h(tc);
            else __syncthreads();
            first_pass(j);
            // w1 = gu - GAW t - sum_i h1_i s_i V_i, published for the next matvec
            cpx<R> *vn = Vv(j + 1);
            auto hv = [&](int l, int i, cpx<R> &acc) { cmac(acc, C(hc[l]), Vv(l)[i]); };
            auto put = [&](int i, cpx<R> w) {
                vn[i] = w;
                ws[i] = w;
                a.pub[r0 + i] = w;
            };
            if (!wide) {   // two sums, each of one accumulator a residue
                rows_by(L1, single, tid, CG_THREADS, k, aw_t, [&](int i, cpx<R> s) {
                    const cpx<R> t = Lanes<R>::template vec_sum<1, false>(0, j + 1, [&](int l, cpx<R> &acc) { hv(l, i, acc); });
                    put(i, uj[i] - to_gaw(i, s) - t);
                });
            } else if constexpr (sizeof(R) == 4) {
                rows_by(L4, single, tid, CG_THREADS, k, aw_t, [&](int i, cpx<R> s) { vn[i] = uj[i] - to_gaw(i, s); });
                rows_by(L4, single, tid, CG_THREADS, j + 1, hv, [&](int i, cpx<R> s) { put(i, vn[i] - s); });
            } else {
                rows_by(L4, dual, tid, CG_THREADS, k + j + 1,
                        [&](int l, int i, cpx<R> &acc) {
                            if (l < k) cmac(acc, C(tc[l]), GAW(l, i));
                            else hv(l - k, i, acc);
                        },
                        [&](int i, cpx<R> s) { put(i, uj[i] - s); });
            }
            __syncthreads();
            // reduction 2: h2_i = <s_i V_i, w1>, ||w1||^2 (gathered in post)
            auto h2_scale = [&](int l) { return l <= j ? scale[l] : R(1); };
            if (a.smem_slices)
                dots(OFF_S2, j + 2, [&](int l, int t, cpx<R> &acc) { cdot((l <= j ? Vv(l) : ws)[t], ws[t], acc); }, h2_scale);
            else
                dots_global(OFF_S2, j + 2, [&](int l, const cpx<R> *&X, const cpx<R> *&Y, bool &flip) {
                    flip = false;
                    X = l <= j ? Vv(l) : ws;
                    Y = ws;
                }, h2_scale);
            if (!grid_sync(a.st, G, bar, a.timeout)) return;
        }
        if (tid == 0) {   // y = R^-1 g
            for (int i = kk - 1; i >= 0; --i) {
                P sacc = g[i];
                for (int l = i + 1; l < kk; ++l) {
                    P r = Rm[l * (CG_MAXM + 1) + i], yl = y[l];
                    sacc.x -= r.x * yl.x - r.y * yl.y;
                    sacc.y -= r.x * yl.y + r.y * yl.x;
                }
                P d = Rm[i * (CG_MAXM + 1) + i];
                R dd = d.x * d.x + d.y * d.y;
                y[i] = dd > 0 ? P2((sacc.x * d.x + sacc.y * d.y) / dd, (sacc.y * d.x - sacc.x * d.y) / dd)
                              : P2(0, 0);
            }
        }
        __syncthreads();
        rows(kk, [&](int l, int i, cpx<R> &acc) { cmac(acc, scale[l] * C(y[l]), Vv(l)[i]); },
             [&](int i, cpx<R> s) { xs[i] = xs[i] + s; });
        __syncthreads();
        have_x = true;
        its += kk;
        if (conv) break;
        if (tid == 0) stop = 0;
        __syncthreads();
    }
    // e = y + W (t0 - E^-1 W^dag A y)
    if (k > 0) {
        publish(xs);
        if (!grid_sync(a.st, G, bar, a.timeout)) return;
        matvec(ws, xs);
        if (!deflation_coeffs(ws)) return;
        rows(k, [&](int l, int i, cpx<R> &acc) { cmac(acc, C(t0[l]) - C(tc[l]), GW(l, i)); },
             [&](int i, cpx<R> s) { xs[i] = xs[i] + g5(i, s); });
        __syncthreads();
    }
    for (int i = tid; i < nr; i += CG_THREADS) a.x[r0 + i] = xs[i];
    if (tid == 0) {
        if (blockIdx.x == 0) atomicAdd(&a.st->iters, its);
        // the last block to leave (none waits any more) resets the counters for the next launch
        if (atomicAdd(&a.st->exits, 1u) == G - 1) {
            atomicExch(&a.st->count, 0u);
            atomicExch(&a.st->exits, 0u);
        }
    }
}

// the kernel's instances, in files of their own (half a minute of compilation each)
const void *coarse_gmres_kernel_f32();
const void *coarse_gmres_kernel_f64();
const void *coarse_gmres_kernel_bf16();
const void *coarse_gmres_kernel_f16();

}  // namespace mgeig
