// Host-side launch of the stage kernels for one arithmetic type: table
// conversion, schedule (strip width, segment height, grid), kernel selection.
#pragma once
#include <algorithm>
#include <atomic>
#include <cmath>

#include "list.cuh"
#include "plan.h"
#include "stage.cuh"
#include "tile.cuh"

namespace gpweno {

// Block size of the 3D z-marching kernel (contiguous runs of 256 xy-columns; FP32 also runs of 128, see launch_stagez).
constexpr int kNTz = 256;
// CTAs of a 3D launch that marches `groups` groups (strips of planes, runs of columns) of n layers each, and an
// estimate of its time in layer iterations.  The layers of all groups, end to end, are cut into equal
// ranges; a range evaluates five layers of faces before its first, and again where it enters another group.
// With m ranges per group none does: ceil(n/m) + 5 iterations.  An iteration of an SM with 4 or 8 warps
// takes the same time (a chain of one thread's instructions), with 12 about 1.2 and with 16 (all that are
// resident) 1.5 times that.  Taken against the cut into as many ranges of at least eight layers as fit at once
// (`full`).  Measured steps, R = 3: 32^3 152 -> 103, 56^3 238 -> 160,
// 64^3 252 -> 215, 80^3 348 -> 342, 96^3 507 -> 424 us.
struct Cut3D {
    int grid;
    double cost;
};
inline Cut3D cut3d(long long groups, int n, int occ, int num_sms, int block)
{
    auto pace = [&](long long ctas) {
        const long long warps = std::min<long long>(occ, (ctas + num_sms - 1) / num_sms) * (block / 32);
        return warps <= 8 ? 1.0 : (warps <= 12 ? 1.2 : 1.5);
    };
    const long long slots = (long long)occ * num_sms, total = groups * n;
    const long long full = std::max(1LL, std::min(slots, total / 8));
    Cut3D best = {(int)full, ((total + full - 1) / full + (total % full || n % (total / full) ? 10 : 5)) * pace(full)};
    for (long long m = 1; m <= n && groups * m <= slots; ++m) {
        const double cost = ((n + m - 1) / m + 5) * pace(groups * m);
        if (cost < best.cost) best = {(int)(groups * m), cost};
    }
    return best;
}
// Block size of the xy-sweeping kernels (2D stage, 3D plane).  FP32: 128 threads
// and four CTAs per SM, with the same 128 registers per thread as two 256-thread
// CTAs.  A strip is then at most 123 columns, so every warp of a CTA evaluates
// faces and each of the four SM sub-partitions holds four busy warps.  With 256
// threads and strips narrower than 251 columns (205 at nx = 1024) the eighth warp
// of each CTA idles.  Its sub-partition then carries half the load of the others,
// and a row takes as long as the busiest sub-partition needs.  Measured on GB300:
// +8 % at 1024^2, +6 % at 2048^2, +1 % at 4096^2.  FP64 (255 registers, one
// 256-thread CTA per SM) keeps 256: 128 threads measured 4 % slower.
template <typename T>
constexpr int kNTxy = sizeof(T) == 4 ? 128 : 256;
constexpr int kNT1D = 128;

template <typename T, int R, int VAR>
FaceTables<T, R> make_tables(const gpweno_plan_s *p)
{
    FaceTables<T, R> t;
    constexpr int S = R + 1, UL = kUnitL<R>, UR = kUnitR<R>;
    const GpTables &g = p->tab;
    for (int k = 0; k <= S; ++k) {   // window k: the left side's sub-stencil k, the last one the right side's
        const double *w = k < S ? g.wl + k * S : g.wr + R * S;
        for (int j = 0; j < S; ++j) t.w[k][j] = (T)w[j];
        t.s1[k] = (T)(k < S ? g.sl1[k] : g.sr1[R]);
    }
    for (int m = 0; m < S; ++m) {
        t.gl[m] = (T)(g.gl[m] / g.gl[UL]);
        t.gr[m] = (T)(g.gr[m] / g.gr[UR - 1]);
    }
    const double unit = kUnitDifference<T, R, VAR> ? g.fa : 1.0;   // the scale of the smoothness indicators
    t.A = (T)(g.fA / unit);
    t.B = (T)(g.fB / unit);
    t.D = (T)(g.fD / unit);
    t.a = (T)(g.fa / unit);
    t.kb = (T)(g.fkb / unit);
    t.kd = (T)(g.fkd / unit);
    t.pA = (T)(g.fpA / unit);
    t.pD = (T)(g.fpD / unit);
    // eps in that scale; FP32: at least the floor, so that (eps + beta)^-2 stays in range
    t.eps = (T)(std::max(p->opts.eps, (double)Num<T>::kEpsFloor) / (unit * unit));
    // FP64: an eps whose eps^-p is finite stays so in that scale (down to it beta is lost against no data above 1e-70)
    if (std::is_same<T, double>::value) t.eps = (T)std::max((double)t.eps, p->opts.p == 2 ? 1e-150 : 1e-300);
    t.gm1 = (T)(p->gamma - 1.0);
    t.igm1 = (T)(1.0 / (p->gamma - 1.0));
    t.hgm1 = (T)(0.5 * (p->gamma - 1.0));
    t.gamma = (T)p->gamma;
    t.p = p->opts.p;
    t.flux = p->opts.flux_form;
    return t;
}

// Whether an FP32 plan's weights stay in range in the scale of kUnitDifference: the floor of eps + beta becomes
// floor / a^2, the largest weight (a^2 / floor)^p and the largest sum of weights that times the sum of the linear weights
// over their unit, which has to stay below 2^126 for its reciprocal to be a normal number.  (Where a weight is
// that large the data, and so the predictions summed with it, are below 1e-8.)  a^2 <= 6.3 at R = 2 and 5.1 at
// R = 3 for the default eps and long l, that is sigma <= 4.9 and 6.5 dx; any sigma for p = 1.
inline bool unit_scale_fits(const gpweno_plan_s *p)
{
    if (p->R == 1) return true;   // no kernel takes it
    const GpTables &g = p->tab;
    const int ul = p->R == 2 ? kUnitL<2> : kUnitL<3>, ur = p->R == 2 ? kUnitR<2> : kUnitR<3>;
    double l = 0.0, r = 0.0;
    for (int m = 0; m <= p->R; ++m) {
        l += std::fabs(g.gl[m] / g.gl[ul]);
        r += std::fabs(g.gr[m] / g.gr[ur - 1]);
    }
    const double x = g.fa * g.fa / std::max(p->opts.eps, (double)Num<float>::kEpsFloor);
    return (p->opts.p == 2 ? x * x : x) * std::max(l, r) <= 8.5e37;
}

// Tables of a scheme variant: GP-AO adds its own on top of the GP-WENO ones.
template <typename T, int R, int VAR>
TablesFor<T, R, VAR> make_tables_var(const gpweno_plan_s *p)
{
    if constexpr ((VAR & kVarAo) != 0) {
        using AT = AoFaceTables<T, R>;
        constexpr int NH = AT::NH, NL = AT::NL;
        AT t;
        std::memset(&t, 0, sizeof(t));
        static_cast<FaceTables<T, R> &>(t) = make_tables<T, R, VAR>(p);
        const AoTables &a = p->ao;
        for (int j = 0; j < NH; ++j) {
            t.whl[j] = (T)a.w_hi_l[j];
            t.whr[j] = (T)a.w_hi_r[j];
        }
        t.shl = (T)a.s_hi_l;
        t.shr = (T)a.s_hi_r;
        if (R == 3) {
            for (int j = 0; j < NL; ++j) {
                t.wll[j] = (T)a.w_lo_l[j];
                t.wlr[j] = (T)a.w_lo_r[j];
            }
            t.sll = (T)a.s_lo_l;
            t.slr = (T)a.s_lo_r;
            for (int k = 0; k < NL; ++k) {
                for (int j = 0; j < (NL + 1) / 2; ++j) t.Plo[k][j] = (T)a.Ph_lo[k * NL + j];
                t.Psum_lo[k] = (T)a.Psum_lo[k];
            }
        }
        for (int m = 0; m < 3; ++m) {
            for (int j = 0; j < 3; ++j) {
                t.w3l[m][j] = (T)a.w3_l[3 * m + j];
                t.w3r[m][j] = (T)a.w3_r[3 * m + j];
            }
            t.s3l[m] = (T)a.s3_l[m];
            t.s3r[m] = (T)a.s3_r[m];
        }
        for (int k = 0; k < NH; ++k) {
            for (int j = 0; j < (NH + 1) / 2; ++j) t.Phi[k][j] = (T)a.Ph_hi[k * NH + j];
            t.Psum_hi[k] = (T)a.Psum_hi[k];
        }
        for (int k = 0; k < 3; ++k) {
            for (int j = 0; j < 2; ++j) t.P3[k][j] = (T)a.Ph_3[k * 3 + j];
            t.Psum3[k] = (T)a.Psum_3[k];
        }
        const double gh = p->opts.ao_gamma_hi, gl = p->opts.ao_gamma_lo;
        t.eps_ao = (T)p->opts.eps;
        t.g_hi = (T)gh;
        t.g_hi1 = (T)(1.0 - gh);
        t.ig_hi = (T)(1.0 / gh);
        t.g3[0] = t.g3[2] = (T)(0.5 * (1.0 - gh) * (1.0 - gl));
        t.g3[1] = (T)((1.0 - gh) * gl);
        return t;
    } else {
        return make_tables<T, R, VAR>(p);
    }
}

// Schedule of the 2D kernel: strips as wide as the block allows (balanced
// widths), one CTA per resident slot, each CTA an equal share of the strips'
// rows (at least 8 rows, so the 5 warm-up y-face rows stay a minor cost).
inline Schedule schedule2d(int nx, int ny, int nt, int slots)
{
    Schedule s;
    const int wmax = nt - 5;
    s.nstrips = (nx + wmax - 1) / wmax;
    s.W = (nx + s.nstrips - 1) / s.nstrips;
    const long long rows = (long long)s.nstrips * ny;
    s.grid = (int)std::max(1LL, std::min<long long>(slots, rows / 8));
    s.H = (int)((rows + s.grid - 1) / s.grid);
    s.nseg = 0;
    return s;
}

// Block size of the tile kernel: two CTAs of 256 threads per SM; the R = 3 faces of GP-AO and FD-Flux fit 384 threads at
// 168 registers (one CTA per SM; GP-AO step of 256^2 53 -> 42 us, of 1000 x 900 453 -> 438 against 256 threads).
constexpr int kNTtile = 256;
constexpr int kTileSmem = 100 * 1024;   // most shared memory of a tile
template <int R, int VAR>
constexpr int kTileThreads = R == 3 && (VAR & (kVarAo | kVarFdFlux)) != 0 ? 384 : kNTtile;

// Strip marching's CTAs of eight rows per SM (the most it makes) below which an FP32 2D grid is tiled.  Measured
// times, marching / tiles, at 512^2 (2.1 CTAs per SM), 777 x 613 (3.5), 768^2 (4.4), 1000 x 900 (6.7), 1024^2 (7.6), 1500^2 (16):
//   HLLC step  R = 1  84/53  94/94   111/103 152/164 168/189 312/397 us    R = 2 100/62  113/110 130/127 179/182 201/217 382/453
//              R = 3 125/76  144/131 176/159 242/225 268/256 499/538
//   FD-Flux    R = 1  95/59  108/103 123/115 170/178 192/202 367/427       R = 2 137/90  158/167 182/190 252/291 283/347 547/790
//              R = 3 170/111 245/205 295/254 395/375 445/430 873/967
//   GP-AO      R = 2 154/82  182/149 212/174 301/254 334/303 649/648       R = 3 203/131 303/238 359/297 518/438 580/504 1125/1097
//   RHS alone  R = 1  23/16   27/29   31/31   43/45   47/53   84/107       R = 2  29/21   33/33   37/37   51/53   57/62  109/123
//              R = 3  37/25   43/39   51/47   72/68   79/76  143/155
// The lines were drawn with marching kernels that were 6 to 13 % slower (before they were compiled per stage), hence
// within 7 % of break-even where they lie past it (R = 1 and FD-Flux R = 2 at 3.5).  Steps of the default scheme
// (72/49, 88/57, 115/70 us at 512^2, 98/94, 116/117, 162/146 at 768^2, 146/170, 178/198, 247/235 at 1024^2) end at two CTAs
// per SM, below 512^2, not by these times: their schedule of strips is what gpweno_plan_schedule reports from there on.
template <int R, int VAR>
constexpr int kTileLimit = (VAR & kVarAo) != 0 ? 16 : ((VAR & kVarFdFlux) != 0 && R == 2 ? 4 : (R == 1 ? 5 : (R == 2 ? 6 : 8)));
constexpr int kTileLimitStep = 2, kTileLimitMost = 16;
inline bool few_rows(int nx, int ny, int num_sms, int per_sm)
{
    const int strips = (nx + kNTxy<float> - 6) / (kNTxy<float> - 5);
    return (long long)strips * ny / 8 < (long long)per_sm * num_sms;
}

// Tiles of a small FP32 2D grid, or none (TX = 0).  The tile minimises the busiest SM's
// work and depth: it evaluates `work` warps of faces, at 230 cycles each when
// its issue slots are full, and a CTA's list is `depth` faces deep, at 1500 cycles each.  The estimate takes two CTAs
// of 256 threads per SM; FD-Flux R = 2 (130 registers) has one, as have the 384-thread builds.
inline Tile2D choose_tile(int nx, int ny, int R, int num_sms)
{
    Tile2D best;
    if (!few_rows(nx, ny, num_sms, kTileLimitMost)) return best;
    double least = 0.0;
    for (int TX = 4; TX <= 64; ++TX)
        for (int TY = 4; TY <= 64; ++TY) {
            const long G = R + 3;
            const long elems = (TX + 2 * G) * (TY + 2 * G) + 2 * ((TX + 5L) * TY + TX * (TY + 5L));
            if (elems * 16 > kTileSmem) break;   // two CTAs per SM
            const int tx = (nx + TX - 1) / TX, ty = (ny + TY - 1) / TY;
            const long tiles = (long)tx * ty, per_sm = (tiles + num_sms - 1) / num_sms;
            const long warps = ((TX + 5L) * TY + TX * (TY + 5L) + 31) / 32;
            const long work = per_sm * warps, depth = (per_sm + 1) / 2 * ((warps + kNTtile / 32 - 1) / (kNTtile / 32));
            const double cost = std::max(230.0 * work, 1500.0 * depth) + 0.2 * std::min(230.0 * work, 1500.0 * depth);
            if (best.TX == 0 || cost < least) {
                least = cost;
                best.TX = TX;
                best.TY = TY;
                best.nx = tx;
                best.ny = ty;
            }
        }
    return best;
}

template <typename T>
StageArgs<T> base_args(const gpweno_plan_s *p)
{
    StageArgs<T> a;
    std::memset(&a, 0, sizeof(a));
    for (int d = 0; d < 3; ++d) {
        a.n[d] = p->dims.n[d];
        a.per[d] = p->dims.bc_lo[d] == GPWENO_BC_PERIODIC ? 1 : 0;
        a.idx[d] = (T)(1.0 / p->dims.dx[d]);
    }
    a.flags = reinterpret_cast<int *>(p->ws + 3);
    a.cstride = p->ncell;
    a.P = nullptr;
    const int sd = p->dims.ndim - 1;   // the slab dimension: the slowest one
    a.ext[0] = p->dims.bc_lo[sd] == GPWENO_BC_EXTERNAL;
    a.ext[1] = p->dims.bc_hi[sd] == GPWENO_BC_EXTERNAL;
    a.slab_dim = (a.ext[0] || a.ext[1]) ? sd : -1;
    a.halo[0] = static_cast<const T *>(p->halo[0]);
    a.halo[1] = static_cast<const T *>(p->halo[1]);
    return a;
}

// Shared memory to ask for so that a launch of `ctas` CTAs spreads evenly: the hardware fills an SM with as
// many CTAs as fit before it moves on, so a kernel of which four fit per SM leaves SMs idle when it is
// launched with two or three per SM.  Asking for more than a (k+1)-th of the SM's 228 KB (1 KB of it
// reserved per CTA) lets k = ceil(ctas / SMs) in.  Measured: R = 1 512^2 step 101 -> 81 us (three of four).
template <typename T>
constexpr int kSpreadSmem = sizeof(T) == 4 ? 116 * 1024 : 0;   // the most it asks for (FP32 kernels only)
inline size_t spread_smem(long ctas, int num_sms, size_t smem)
{
    const long k = (ctas + num_sms - 1) / num_sms;
    if (k > 3) return smem;
    const size_t want = (228 * 1024 / (k + 1) - 1024 + 16) / 16 * 16 + 16;
    return std::max(smem, want);
}

constexpr int kAnyResident = 1 << 20;   // no cap
// Resident CTAs per SM of one kernel, by device: its limit on dynamic shared memory belongs to a device as well and is
// raised there before the first launch.  Any number of threads may ask at once: each finds the same value,
// and only the final one (capped at `most`) is ever stored.
class Residency {
public:
    template <typename K>
    gpweno_status get(K kern, int block, size_t smem, size_t smem_limit, int most, const char *what, int &ctas)
    {
        int device = -1;   // the current one, which the attribute is set on, also where a caller left another than the plan's
        cudaError_t e = cudaGetDevice(&device);
        if (e != cudaSuccess) return cuda_fail(e, what);
        const bool cached = device >= 0 && device < kDevices;
        ctas = cached ? of_[device].load(std::memory_order_acquire) : 0;
        if (ctas) return GPWENO_OK;
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)std::max(smem, smem_limit));
        if (e != cudaSuccess) return cuda_fail(e, what);
        int n = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, block, smem);
        if (e != cudaSuccess || n < 1) return cuda_fail(e == cudaSuccess ? cudaErrorInvalidConfiguration : e, what);
        ctas = std::min(n, most);
        if (cached) of_[device].store(ctas, std::memory_order_release);
        return GPWENO_OK;
    }

private:
    static constexpr int kDevices = 64;   // beyond it every launch asks
    std::atomic<int> of_[kDevices] = {};
};

// Rows per CTA below which FP32 R = 2 grids take the three-CTA-per-SM build of the 2D kernel.
constexpr int kWideRows = 24;
// Rows per CTA between which R = 3 grids take it (below 16 rows they keep the four-CTA schedule that
// gpweno_plan_schedule has reported for them, 1024^2 among them).
constexpr int kMidRows = 16, kLongRows = 96;

// One launch of the 2D stage kernel built for MINB resident CTAs per SM: occupancy (queried
// once per instantiation), the one-wave schedule, the launch.
template <typename T, int R, int NT, int VAR, int MINB, int SPEC>
gpweno_status launch_stage2d_spec(gpweno_plan p, StageArgs<T> a, const TablesFor<T, R, VAR> &tb, cudaStream_t st)
{
    const size_t smem = stage2d_smem_bytes<T, R, NT>();
    auto kern = stage2d_kernel<T, R, NT, VAR, MINB, SPEC>;
    static Residency residency;   // per instantiation
    int occ;
    // at most MINB: R = 1's three-CTA build needs 120 registers at most and would fit four times
    const gpweno_status r = residency.get(kern, NT, smem, kSpreadSmem<T>, MINB, "stage2d occupancy", occ);
    if (r != GPWENO_OK) return r;
    Schedule s = schedule2d(a.n[0], a.n[1], NT, occ * p->num_sms);
    s.ctas_per_sm = occ;
    a.W = s.W;
    a.nstrips = s.nstrips;
    a.H = s.H;
    a.nseg = s.nseg;
    p->sched = s;
    cudaError_t e = launch_pdl(kern, s.grid, NT, sizeof(T) == 4 ? spread_smem(s.grid, p->num_sms, smem) : smem, st, a, tb);
    if (e != cudaSuccess) return cuda_fail(e, "stage2d kernel launch");
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "stage kernel launch");
    return GPWENO_OK;
}

// Whether the kernels are compiled for each stage.  FP64 ones are not: their time is the FP64 pipe's.
template <typename T>
constexpr bool kPerStage = std::is_same<T, float>::value;

// The same by stage.
template <typename T, int R, int NT, int VAR, int MINB>
gpweno_status launch_stage2d(gpweno_plan p, const StageArgs<T> &a, const TablesFor<T, R, VAR> &tb, cudaStream_t st)
{
    if constexpr (kPerStage<T>) {
        if (a.mode == kModeRHS) return launch_stage2d_spec<T, R, NT, VAR, MINB, kSpecRHS>(p, a, tb, st);
        if (a.mode == kModeFinal) return launch_stage2d_spec<T, R, NT, VAR, MINB, kSpecFinal>(p, a, tb, st);
        if (a.u0_is_stencil && !a.Din) return launch_stage2d_spec<T, R, NT, VAR, MINB, kSpecFirst>(p, a, tb, st);
        return launch_stage2d_spec<T, R, NT, VAR, MINB, kSpecSecond>(p, a, tb, st);
    } else {
        return launch_stage2d_spec<T, R, NT, VAR, MINB, kSpecAny>(p, a, tb, st);
    }
}

// The z-marching launch of a 3D stage: L = P - div_z/dz and the stage update.
template <typename T, int R, int VAR, int SPEC, int NT = kNTz>
gpweno_status launch_stagez(gpweno_plan p, const StageArgs<T> &a, const TablesFor<T, R, VAR> &tb, cudaStream_t st)
{
    const size_t smem = stagez_smem_bytes<T, R, NT>();
    auto kern = stagez_kernel<T, R, NT, VAR, SPEC>;
    static Residency residency;
    int occ;
    const gpweno_status r = residency.get(kern, NT, smem, kSpreadSmem<T>, kAnyResident, "stagez occupancy", occ);
    if (r != GPWENO_OK) return r;
    const long long plane = (long long)a.n[0] * a.n[1];
    const Cut3D cut = cut3d((plane + NT - 1) / NT, a.n[2], occ, p->num_sms, NT);
    if constexpr (NT == kNTz && std::is_same<T, float>::value) {
        // runs of half the columns where the SMs are then busy for less time (twice the CTAs resident)
        constexpr int half = kNTz / 2;
        if (cut3d((plane + half - 1) / half, a.n[2], 2 * occ, p->num_sms, half).cost < cut.cost)
            return launch_stagez<T, R, VAR, SPEC, half>(p, a, tb, st);
    }
    const int grid = cut.grid;
    cudaError_t e = launch_pdl(kern, grid, NT, std::is_same<T, float>::value ? spread_smem(grid, p->num_sms, smem) : smem,
                               st, a, tb);
    if (e != cudaSuccess) return cuda_fail(e, "stagez kernel launch");
    return GPWENO_OK;
}

// Band geometry of the face-list stages (list.cuh) for layers [l0, l0 + nb) of the slowest dimension.
template <typename T>
FaceBand<T> face_band(const gpweno_plan_s *p, int l0, int nb)
{
    FaceBand<T> b;
    std::memset(&b, 0, sizeof(b));
    const int nd = p->dims.ndim;
    b.buf = static_cast<T *>(p->face_ws);
    b.size = (long)(p->face_ws_bytes / sizeof(T));
    b.l0 = l0;
    b.l1 = l0 + nb;
    long off = 0;
    for (int d = 0; d < nd; ++d) {
        const bool slow = d == nd - 1;
        b.wrap[d] = p->dims.bc_lo[d] == GPWENO_BC_PERIODIC && (!slow || nb == p->dims.n[d]);
        for (int e = 0; e < 3; ++e) b.ext[d][e] = e == nd - 1 ? nb : (e < nd ? p->dims.n[e] : 1);
        if (!b.wrap[d]) b.ext[d][d] += 5;
        b.lo[d] = b.wrap[d] ? 0 : (slow ? l0 - 3 : -3);
        b.n[d] = (long)b.ext[d][0] * b.ext[d][1] * b.ext[d][2];
        b.off[d] = off;
        off += 2 * (nd + 2) * b.n[d];
    }
    return b;
}

// One stage as face and update launches, band by band.
template <typename T, int R, int NC, int VAR>
gpweno_status launch_list(gpweno_plan p, StageArgs<T> a, const TablesFor<T, R, VAR> &tb, cudaStream_t st)
{
    constexpr int NT = 256;   // one CTA per SM (255 registers)
    const Schedule s = schedule2d(a.n[0], a.n[1], NT, p->num_sms);
    a.W = s.W;
    a.nstrips = s.nstrips;
    const int layers = a.n[NC - 3];
    for (int l0 = 0; l0 < layers; l0 += p->face_ws_layers) {
        const FaceBand<T> b = face_band<T>(p, l0, std::min(p->face_ws_layers, layers - l0));
        long items = 0;
        for (int d = 0; d < NC - 2; ++d) items += (b.n[d] + 31) / 32;
        const int grid = (int)std::min<long>(p->num_sms, items);
        cudaError_t e = launch_pdl(face_list_kernel<T, NC, R, VAR, NT>, grid, NT, 0, st, a, b, tb);
        if (e != cudaSuccess) return cuda_fail(e, "face list kernel launch");
        const long rows = (long)(b.l1 - b.l0) * (NC == 5 ? a.n[1] : 1) * a.nstrips;
        e = launch_pdl(face_update_kernel<T, NC, VAR, NT>, (int)std::min<long>(rows, 8L * p->num_sms), NT, 0, st, a, b,
                       (T)p->gamma);
        if (e != cudaSuccess) return cuda_fail(e, "face update kernel launch");
        count_launch(2);
        if (NC == 4) {
            p->sched = s;
            p->sched.grid = grid;
            p->sched.ctas_per_sm = 1;
        }
    }
    return GPWENO_OK;
}

// VAR: the scheme variant (kVarMean: non-zero-mean smoothness indicators,
// kVarFdFlux: the FD-Flux form), a compile-time switch so that the default
// kernels keep their register budget.
template <typename T, int R, int VAR>
gpweno_status launch_stage_R(gpweno_plan p, const StageArgs<T> &a0, bool use_list, cudaStream_t st)
{
    StageArgs<T> a = a0;
    const TablesFor<T, R, VAR> tb = make_tables_var<T, R, VAR>(p);
    // FP64 2D and 3D: face lists wherever the plan has their workspace (measurements in list.cuh); the
    // marching kernels serve plans without one and the allocation-free step
    if constexpr (std::is_same<T, double>::value) {
        if (use_list && p->dims.ndim == 3) return launch_list<T, R, 5, VAR>(p, a, tb, st);
        if (use_list && p->dims.ndim == 2) return launch_list<T, R, 4, VAR>(p, a, tb, st);
    }
    if (p->dims.ndim == 3) {
        // (1) xy-plane kernel: P = -(div_x/dx + div_y/dy)
        {
            constexpr int NT = kNTxy<T>;
            const size_t smem = stage2d_smem_bytes<T, R, NT, 5>();
            auto kern = plane3d_kernel<T, R, NT, VAR>;
            static Residency residency;
            int occ;
            const gpweno_status r = residency.get(kern, NT, smem, kSpreadSmem<T>, kAnyResident, "plane3d occupancy", occ);
            if (r != GPWENO_OK) return r;
            StageArgs<T> pa = a;
            const int wmax = NT - 5;
            pa.nstrips = (a.n[0] + wmax - 1) / wmax;
            pa.W = (a.n[0] + pa.nstrips - 1) / pa.nstrips;
            pa.mode = kModePartial;
            pa.out = const_cast<T *>(a.P);
            pa.rate = nullptr;
            const int grid = cut3d((long long)pa.nstrips * a.n[2], a.n[1], occ, p->num_sms, NT).grid;
            cudaError_t e = launch_pdl(
                kern, grid, NT, std::is_same<T, float>::value ? spread_smem(grid, p->num_sms, smem) : smem, st, pa, tb);
            if (e != cudaSuccess) return cuda_fail(e, "plane3d kernel launch");
            count_launch(1);
        }
        // (2) z-marching kernel
        gpweno_status r;
        if constexpr (kPerStage<T>) {
            if (a.mode == kModeRHS) r = launch_stagez<T, R, VAR, kSpecRHS>(p, a, tb, st);
            else if (a.mode == kModeFinal) r = launch_stagez<T, R, VAR, kSpecFinal>(p, a, tb, st);
            else if (a.u0_is_stencil && !a.Din) r = launch_stagez<T, R, VAR, kSpecFirst>(p, a, tb, st);
            else r = launch_stagez<T, R, VAR, kSpecSecond>(p, a, tb, st);
        } else {
            r = launch_stagez<T, R, VAR, kSpecAny>(p, a, tb, st);
        }
        if (r != GPWENO_OK) return r;
    } else if (p->dims.ndim == 2) {
        constexpr int NT = kNTxy<T>;
        if constexpr (std::is_same<T, float>::value) {
            const int limit = VAR == 0 && a.mode != kModeRHS ? kTileLimitStep : kTileLimit<R, VAR>;
            if (p->tile.TX && few_rows(a.n[0], a.n[1], p->num_sms, limit)) {
                constexpr int NTt = kTileThreads<R, VAR>;
                auto kern = tile2d_kernel<R, NTt, VAR>;
                const size_t smem = tile2d_elems<R>(p->tile.TX, p->tile.TY) * sizeof(float4);
                static Residency residency;   // at the largest tile; never lowered for a plan of smaller ones
                int occ;
                const gpweno_status r = residency.get(kern, NTt, kTileSmem, kTileSmem, kAnyResident, "tile2d occupancy", occ);
                if (r != GPWENO_OK) return r;
                cudaError_t e = launch_pdl(kern, p->tile.nx * p->tile.ny, NTt, smem, st, a, p->tile, tb);
                if (e != cudaSuccess) return cuda_fail(e, "tile2d kernel launch");
                p->sched = Schedule();
                p->sched.W = p->tile.TX;
                p->sched.nstrips = p->tile.nx;
                p->sched.grid = p->tile.nx * p->tile.ny;
                p->sched.ctas_per_sm = occ;
                count_launch(1);
                return GPWENO_OK;
            }
        }
        // FP32, default scheme (also with slab halos): the build for three CTAs per SM (more
        // registers per thread: 120 to 134 at R = 2, 142 to 156 at R = 3 by stage, the four-CTA build's 128 being the
        // limit there; R = 1 needs 108 to 120 either way) is faster where
        // the four-CTA schedule cannot fill four CTAs per SM (the grid is row-limited), and for
        // R = 2, whose four-CTA build is register-capped, where it leaves a CTA fewer than
        // kWideRows rows (three CTAs per SM: fewer, taller segments, fewer warm-up rows).
        // Measured on GB300 (same-box A/B, bitwise-identical results): R = 2 x1.10 at 512^2,
        // x1.05 at 768^2, x1.017 at 1024^2; R = 1 x1.14 at 700 x 640, x1.05 at 777 x 613; R = 3 x1.10 at
        // 777 x 613, x1.05 at 1024 x 512, x1.03 at 1501 x 1100, x1.016 at 2048^2 (HLLC x1.013, x1.005).  Not
        // taken where it lost: R = 2 at 1536^2 (x0.995) and 4096^2 (x0.98), R = 1 at 1024^2 (x0.98).
        constexpr bool kHasWide = std::is_same<T, float>::value && (VAR & ~(kVarSlab | kVarFlux | kVarRange)) == 0;
        if constexpr (kHasWide) {
            const int slots4 = 512 / NT * p->num_sms;
            const Schedule s4 = schedule2d(a.n[0], a.n[1], NT, slots4);
            const long long rows = (long long)s4.nstrips * a.n[1];
            const bool row_limited = s4.grid < slots4;
            const bool short_segments = R == 2 && rows < (long long)kWideRows * s4.grid;
            const bool mid_segments =
                R == 3 && rows >= (long long)kMidRows * s4.grid && rows < (long long)kLongRows * s4.grid;
            if (row_limited || short_segments || mid_segments) {
                gpweno_status r = launch_stage2d<T, R, NT, VAR, 3>(p, a, tb, st);
                if (r != GPWENO_OK) return r;
                count_launch(1);
                return GPWENO_OK;
            }
        }
        gpweno_status r = launch_stage2d<T, R, NT, VAR, kResident<T, R, VAR> / NT>(p, a, tb, st);
        if (r != GPWENO_OK) return r;
    } else {
        cudaError_t e = cudaSuccess;
        auto launch = [&](auto kern, int cells, int nt, size_t smem) {
            a.nstrips = (a.n[0] + cells - 1) / cells;
            a.W = (a.n[0] + a.nstrips - 1) / a.nstrips;
            a.H = 1;
            a.nseg = 1;
            e = launch_pdl(kern, a.nstrips, nt, smem, st, a, tb);
        };
        // FP64: field-split CTAs up to three per SM (12 K cells).  Measured steps, split and plain, R = 1, 2, 3:
        // 8208 cells (two per SM) 35.7, 42.9, 52.5 and 53.4, 66.4, 84.8 us; 12312 cells (three) 48.3, 59.5, 74.2
        // and 53.0, 65.9, 84.6 us; a fourth would draw level
        constexpr bool kSplit = std::is_same<T, double>::value && (VAR & (kVarAo | kVarFdFlux)) == 0;
        if (kSplit && (a.n[0] + 26) / 27 <= 3 * p->num_sms) {
            if constexpr (kSplit) launch(stage1d_split_kernel<T, R, VAR>, 27, 96, 0);
        } else {
            launch(stage1d_kernel<T, R, kNT1D, VAR>, kNT1D - 5, kNT1D, stage1d_smem_bytes<T, R, kNT1D>());
        }
        if (e != cudaSuccess) return cuda_fail(e, "stage1d kernel launch");
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "stage kernel launch");
    count_launch(1);
    return GPWENO_OK;
}

template <typename T, int VAR>
gpweno_status launch_stage_T(gpweno_plan p, const StageIO &io, cudaStream_t st)
{
    StageArgs<T> a = base_args<T>(p);
    a.U = static_cast<const T *>(io.U);
    a.U0 = static_cast<const T *>(io.U0);
    a.Din = static_cast<const T *>(io.Din);
    a.Dout = static_cast<T *>(io.Dout);
    a.Vout = static_cast<T *>(io.Vout);
    a.out = static_cast<T *>(io.out);
    a.P = static_cast<const T *>(io.P);
    a.lo = static_cast<T *>(io.lo);
    a.u0_is_stencil = io.U0 == io.U ? 1 : 0;
    a.b = (T)io.b;
    a.mode = io.mode;
    a.dt = io.dt;
    a.dt_dev = io.dt_dev;
    a.rate = io.want_rate ? p->ws : nullptr;
    const bool use_list = !io.no_workspace && p->claim_face_ws();
    switch (p->R) {
    case 1:
        if constexpr ((VAR & kVarAo) != 0) {
            set_error("GP-AO needs R = 2 or 3");
            return GPWENO_ERR_ARG;
        } else {
            return launch_stage_R<T, 1, VAR>(p, a, use_list, st);
        }
    case 2: return launch_stage_R<T, 2, VAR>(p, a, use_list, st);
    case 3: return launch_stage_R<T, 3, VAR>(p, a, use_list, st);
    default: set_error("R=%d not compiled", p->R); return GPWENO_ERR_ARG;
    }
}

// Workspace of the FP64 face-list stages: layers per band and bytes, chosen at plan creation.  Bands are equal, of up
// to 24 layers, or of more as far as 32 MiB go, which keeps their face fluxes in L2; equal means that a band has more than
// half of that: five faces of every 24 (a fifth of one direction) are repeated by neighbouring bands at best, of 13
// where 25 layers make two.  32 MiB is 256 K cells in 2D, over fifty warps of faces per SM.  Grids whose 24 layers need more than 1 GiB (3D from 420^2 per plane, 2D
// from 300 K columns) keep the marching kernels.
inline void size_face_workspace(gpweno_plan_s *p)
{
    const int n = p->dims.n[p->dims.ndim - 1];
    auto bytes = [&](int nb) {
        const FaceBand<double> b = face_band<double>(p, 0, nb);
        long e = 0;
        for (int d = 0; d < p->dims.ndim; ++d) e += 2L * (p->dims.ndim + 2) * b.n[d];
        return e * (long)sizeof(double);
    };
    int nb = std::min(n, 24);
    if (bytes(nb) > (1L << 30)) return;
    while (nb < n && bytes(std::min(n, 2 * nb)) <= (32L << 20)) nb = std::min(n, 2 * nb);
    const int bands = (n + nb - 1) / nb;
    p->face_ws_layers = (n + bands - 1) / bands;
    p->face_ws_bytes = (size_t)std::max(bytes(p->face_ws_layers), bytes(nb));
}

template <typename T>
gpweno_status launch_max_rate_T(gpweno_plan p, const void *U, cudaStream_t st)
{
    StageArgs<T> a = base_args<T>(p);
    a.rate = p->ws;
    const int blocks = (int)std::min<long>((p->ncell + 255) / 256, 4L * p->num_sms);
    if (p->dims.ndim == 3)
        max_rate_kernel<T, 5><<<blocks, 256, 0, st>>>(static_cast<const T *>(U), p->ncell, a, (T)p->gamma);
    else if (p->dims.ndim == 2)
        max_rate_kernel<T, 4><<<blocks, 256, 0, st>>>(static_cast<const T *>(U), p->ncell, a, (T)p->gamma);
    else
        max_rate_kernel<T, 3><<<blocks, 256, 0, st>>>(static_cast<const T *>(U), p->ncell, a, (T)p->gamma);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "max-rate kernel launch");
    count_launch(1);
    return GPWENO_OK;
}

}  // namespace gpweno
