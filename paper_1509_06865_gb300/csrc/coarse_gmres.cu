// Host side of the persistent coarse GMRES (coarse_gmres.cuh: the kernel and what it does): the
// launch plan, the scratch and the launch; and the kernel's FP32 instance.
#include <algorithm>
#include <array>
#include <map>
#include <mutex>

#include "coarse_gmres.cuh"

namespace mgeig {

const void *coarse_gmres_kernel_f32() { return (const void *)coarse_gmres_kernel<float, 0>; }

// ---------------------------------------------------------------------------
// host side: the launch plan (grid, slices in shared or global memory) and the
// global scratch it needs

namespace {

struct CGPlan {
    int G, rb, nslice, m, slices, stage_sites, part_size;
    bool smem_slices, smem_defl;
    size_t dyn_smem;          // dynamic shared memory per block
    size_t off_slices, off_partial, scratch_bytes;   // global scratch layout
};

size_t align256(size_t b) { return (b + 255) / 256 * 256; }

// Bytes of a block's slices (2 restart + 5 vectors of ceil(n / G) rows, at most one block
// per 128 rows) up to which they live in shared memory: the line that
// mgeig_mg_cycle_dev_noalloc's scratch limit is drawn by.  So it stays where it is although the
// kernel changes: 24912 and 47504 bytes of static shared memory are the most that the line
// leaves room for (the kernels take 24272 and 46224 now), and the 2 m + 4 vectors that a block
// keeps leave the neighbour vectors of one site room beside them, 3456 bytes at most, where the
// line is nearest (restart 32: 374 rows, 3696 bytes left).
template <typename R> struct SliceBudget { static constexpr size_t bytes = CG_SMEM_LIMIT - 24912; };
template <> struct SliceBudget<double> { static constexpr size_t bytes = CG_SMEM_LIMIT - 47504; };
// Rows an FP64 block has at least: its blocks may be more and smaller (no order to keep).
// Measured on a two-grid cycle at 8^3 x 16 (SAP included): 107 blocks of 12 rows 2.20 ms, 32
// of 40 2.38, 10 of 128 3.76
constexpr int MIN_ROWS_F64 = 12;

// the kernel instance for the context's precision and link format
template <typename R>
const void *kernel_for(Ctx &c) {
    if (sizeof(R) == 8) return coarse_gmres_kernel_f64();
    switch (c.prm.coarse_links) {
        case MGEIG_LINKS_BF16: return coarse_gmres_kernel_bf16();
        case MGEIG_LINKS_F16: return coarse_gmres_kernel_f16();
        default: return coarse_gmres_kernel_f32();
    }
}

template <typename R>
CGPlan compute_plan(Ctx &c, int k, int m) {
    using P = typename Pod2<R>::T;
    CGPlan p;
    const int n = c.nagg * 2 * c.prm.n_tv;
    const size_t elem = sizeof(cpx<R>);
    cudaFuncAttributes fa;
    const void *kern = kernel_for<R>(c);
    MG_CUDA(cudaFuncGetAttributes(&fa, kern));
    int cap = std::min(c.sms, CG_MAXG);
    if (c.prm.coarse_blocks > 0) cap = std::min(cap, c.prm.coarse_blocks);
    // where the slices live, and the scratch the documented layout takes
    const int g128 = std::max(1, std::min((n + 127) / 128, cap)), rows = (n + g128 - 1) / g128;
    const int restart = std::min(c.prm.coarse_restart, CG_MAXM);
    const size_t slice_b = (size_t)(2 * restart + 5) * rows * elem;
    p.smem_slices = slice_b <= SliceBudget<R>::bytes;
    p.m = m;
    p.nslice = 2 * m + 4;
    p.rb = rows;
    if (sizeof(R) == 8 && p.smem_slices) p.rb = std::min(n, std::max(MIN_ROWS_F64, (n + cap - 1) / cap));
    p.G = (n + p.rb - 1) / p.rb;   // every block owns at least one row
    const size_t room = CG_SMEM_LIMIT - fa.sharedSizeBytes;
    size_t used = p.smem_slices ? align16((size_t)p.nslice * p.rb * elem) : 0;
    MG_REQUIRE(used <= room, MGEIG_ECUDA);
    // Threads that share a row of the matvec and leave the sum of their parts to its end: 8 (of a row
    // pair) in FP32 with level links where one pass takes all rows, 1 in the forms with several
    // passes (and with 16-bit links, whose lanes share a row already).  FP64: up to 24, as far as
    // one run of CG_MV threads and the room go (every part costs the end of the matvec an addition
    // per row); with more rows than threads the count whose runs cost least, in FP64 instructions
    // (24^3 x 48, 683 rows: a matvec 324 us with one part, whose second run is a quarter full, 272
    // with fifteen)
    auto fits = [&](int threads, int q, size_t stage) {
        return threads <= CG_MV && used + stage + (size_t)q * p.rb * elem <= room;
    };
    p.slices = 1;
    p.stage_sites = p.part_size = 0;
    if (sizeof(R) == 8) {
        const int most = std::min(24, 9 * c.prm.n_tv);
        while (p.slices < most && fits((p.slices + 1) * p.rb, p.slices + 1, 0)) ++p.slices;
        long long best = 0;
        for (int q = 1; p.rb > CG_MV && q <= most && fits(0, q, 0); ++q) {
            const long long runs = ((long long)q * p.rb + CG_MV - 1) / CG_MV, row_groups = (p.rb + 31) / 32;
            const long long cost = runs * 72 * c.prm.n_tv * (CG_MV / 32) / q + 2 * q * row_groups;
            if (q == 1 || cost < best) { best = cost; p.slices = q; }
        }
    } else {
        const int n2 = 2 * c.prm.n_tv, sites = (p.rb + n2 - 2) / n2 + 1;   // that rb rows can touch
        const size_t site_b = (size_t)9 * n2 * elem;
        auto chunk = [&](size_t bytes) {   // coarse sites at a time, chunks of about the same size
            const int most = (int)std::min((size_t)sites, (room - used) / bytes);
            return most > 0 ? (sites + (sites + most - 1) / most - 1) / ((sites + most - 1) / most) : 0;
        };
        // level links: one pass of all rows (rb of them lie in rb / 2 + 1 pairs at most); else several,
        // with their parts where that leaves room for four sites
        const bool level = c.prm.coarse_links == MGEIG_LINKS_LEVEL;
        const int with_parts = level ? chunk(site_b + 8 * n2 * elem) : 0;
        if (level && fits(8 * (p.rb / 2 + 1), 8, sites * site_b)) {
            p.slices = 8;
            p.stage_sites = sites;
        } else if (level && with_parts >= std::min(sites, 4)) {
            p.stage_sites = with_parts;
            p.part_size = 8 * with_parts * n2;
        } else {
            p.stage_sites = chunk(site_b);
        }
        MG_REQUIRE(p.stage_sites > 0, MGEIG_ECUDA);
        used += p.stage_sites * site_b;
    }
    if (p.slices > 1) p.part_size = p.slices * p.rb;
    used += (size_t)p.part_size * elem;
    p.smem_defl = p.smem_slices && k > 0 && used + (size_t)2 * k * p.rb * elem <= room;
    if (p.smem_defl) used += (size_t)2 * k * p.rb * elem;
    p.dyn_smem = used;
    // global scratch: pub | slices (when not in shared memory) | partial sums
    p.off_slices = align256((size_t)n * elem);
    const size_t slices = p.smem_slices ? 0 : align256((size_t)((n + rows - 1) / rows) * slice_b);
    p.off_partial = p.off_slices + slices;
    const int gmax = std::max(p.G, (n + rows - 1) / rows);
    p.scratch_bytes = p.off_partial + align256((size_t)gmax * CG_SLOTS * sizeof(P));
    MG_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)p.dyn_smem));
    int per_sm = 0;
    MG_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, CG_THREADS, p.dyn_smem));
    MG_REQUIRE(per_sm >= 1 && p.G <= c.sms * per_sm, MGEIG_ECUDA);
    return p;
}

// plans depend only on the device and the problem shape: computed once each
template <typename R>
CGPlan make_plan(Ctx &c, int k) {
    static std::mutex mu;
    static std::map<std::array<int, 9>, CGPlan> cache;
    // no basis longer than the steps a solve may take
    const int m = std::min({c.prm.coarse_restart, CG_MAXM, c.prm.coarse_maxiter});
    const std::array<int, 9> key{c.device, c.nagg, c.prm.n_tv, std::min(c.prm.coarse_restart, CG_MAXM), m, k,
                                 (int)sizeof(R), sizeof(R) == 4 ? c.prm.coarse_links : 0, c.prm.coarse_blocks};
    std::lock_guard<std::mutex> lock(mu);
    auto it = cache.find(key);
    if (it != cache.end()) return it->second;
    const CGPlan p = compute_plan<R>(c, k, m);
    cache.emplace(key, p);
    return p;
}

}  // namespace

// A device's SM clock rate in kHz, asked once: the driver takes 0.6 ms to answer, as
// long as half of a coarse solve at 16^3 x 32 (with the query in every coarse solve a
// two-grid cycle there took 2.04 ms, without it 1.48 ms)
static int sm_clock_khz(int device) {
    static std::mutex mu;
    static std::map<int, int> khz;
    std::lock_guard<std::mutex> lock(mu);
    auto it = khz.find(device);
    if (it != khz.end()) return it->second;
    int v = 0;
    MG_CUDA(cudaDeviceGetAttribute(&v, cudaDevAttrClockRate, device));
    return khz[device] = v > 0 ? v : 2000000;
}

// the barrier budget in SM clock cycles
long long barrier_cycles(Ctx &c) {
    const int khz = sm_clock_khz(c.device);
    return std::max(1LL, (long long)(c.prm.barrier_timeout * khz * 1e3));
}

size_t coarse_gmres_scratch_bytes(Ctx &c, int k) {
    return c.mixed() ? make_plan<float>(c, k).scratch_bytes : make_plan<double>(c, k).scratch_bytes;
}

// The persistent coarse solve with its global scratch (coarse_gmres_scratch_bytes)
// at a caller-given device address and the CGState word block (16 bytes, zero on
// entry) at `state`.
template <typename R>
void coarse_gmres_at(Ctx &c, double sigma, const void *rc, void *ec, void *scratch, void *state, int k,
                     const void *W, const void *AW, const void *Einv) {
    MG_REQUIRE(k <= CG_MAXK && k <= c.prm.n_tv, MGEIG_EINVAL);
    const CGPlan p = make_plan<R>(c, k);
    char *sc = static_cast<char *>(scratch);
    CGArgs<R> a;
    a.nagg = c.nagg; a.ntv = c.prm.n_tv; a.n = c.nagg * 2 * c.prm.n_tv;
    a.rb = p.rb; a.nslice = p.nslice; a.slices = p.slices; a.stage_sites = p.stage_sites;
    a.part_size = p.part_size;
    a.smem_slices = p.smem_slices; a.smem_defl = p.smem_defl;
    a.Dc = static_cast<const cpx<R> *>(c.Dc.p);
    a.L16 = c.Dc16.p;
    a.Ls = c.Dcs.as<float>();
    MG_REQUIRE(sizeof(R) == 8 || c.prm.coarse_links == MGEIG_LINKS_LEVEL || c.Dc16.p, MGEIG_ENOTSETUP);
    a.nbr = c.cnbr.as<int>();
    a.sigma = (R)sigma;
    a.b = static_cast<const cpx<R> *>(rc);
    a.x = static_cast<cpx<R> *>(ec);
    a.pub = reinterpret_cast<cpx<R> *>(sc);
    a.gslices = p.smem_slices ? nullptr : reinterpret_cast<cpx<R> *>(sc + p.off_slices);
    a.k = k;
    a.W = static_cast<const cpx<R> *>(W);
    a.AW = static_cast<const cpx<R> *>(AW);
    a.Einv = static_cast<const double2 *>(Einv);
    a.partial = reinterpret_cast<typename Pod2<R>::T *>(sc + p.off_partial);
    a.st = static_cast<CGState *>(state);
    a.m = p.m;
    a.maxiter = c.prm.coarse_maxiter;
    a.tol = c.prm.coarse_tol;
    a.timeout = barrier_cycles(c);
    void *args[] = {&a};
    // the dynamic shared-memory limit is an attribute of the kernel, not of the
    // plan: plans of other problem shapes may have changed it since
    const void *kern = kernel_for<R>(c);
    MG_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)p.dyn_smem));
    TimeScope ts(c.timer, K_COARSE_SOLVE, 0);
    MG_CUDA(cudaLaunchCooperativeKernel(kern, dim3(p.G), dim3(CG_THREADS), args,
                                        p.dyn_smem, c.stream));
    ++c.launches;
}

template void coarse_gmres_at<float>(Ctx &, double, const void *, void *, void *, void *, int, const void *,
                                     const void *, const void *);
template void coarse_gmres_at<double>(Ctx &, double, const void *, void *, void *, void *, int, const void *,
                                      const void *, const void *);

// Launch the persistent coarse solve for (Q_c - sigma) e_c = r_c with scratch
// owned by the context.
template <typename R>
void coarse_gmres_persistent(Ctx &c, const CoarseSolveBufs &B, double sigma, const void *rc, void *ec) {
    B.scratch->alloc(coarse_gmres_scratch_bytes(c, B.k));
    coarse_gmres_at<R>(c, sigma, rc, ec, B.scratch->p, B.state, B.k, B.W, B.AW, B.Einv);
}

template void coarse_gmres_persistent<float>(Ctx &, const CoarseSolveBufs &, double, const void *, void *);
template void coarse_gmres_persistent<double>(Ctx &, const CoarseSolveBufs &, double, const void *, void *);

}  // namespace mgeig
