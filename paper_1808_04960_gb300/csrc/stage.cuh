// Fused GP-WENO stage kernels: RHS (Eq. disc_fd with the corrected fluxes of
// Eq. numFlux_cor) fused with the SSP-RK3 stage combination.
//
// 2D design ("column-strip marching").  A CTA owns a strip of W <= NT-5
// columns and a segment of rows [y0, y1).  It walks the y-faces s+1/2 from
// s = y0-3 to y1+1 once each:
//   * each thread owns one column and keeps the last five y-face fluxes of
//     that column in registers, so every y-face is evaluated exactly once and
//     the y-correction (five neighbouring faces) needs no shared memory;
//   * the rows of the strip (with R+3 ghost columns per side, boundary
//     conditions applied on load) stream through a small shared-memory ring
//     filled by cp.async one row ahead of use;
//   * for the output row r = s-2, the W+5 x-faces of that row are evaluated
//     from the ring (one per thread), staged in shared memory, corrected,
//     differenced, and combined with the y-part and the RK stage update;
//     the result is stored once (coalesced).
// Per output row a CTA evaluates W y-faces and W+5 x-faces, so the only
// redundant face work is 5 x-faces per row per strip and 5 warm-up y-faces
// per column per segment.
//
// HBM traffic per cell and stage: the stage input state once (ring rows are
// read once per strip; ghost columns come from L2), U^n once for stages 2-3,
// the output once.
#pragma once
#include "face.cuh"

namespace gpweno {

// Stage modes.  The SSP-RK3 step is carried in increment form,
//   D_1 = dt L(U^n),  D_2 = 1/4 (D_1 + dt L(U^n + D_1)),  D_3 = 2/3 (D_2 + dt L(U^n + D_2)),
//   U^{n+1} = U^n + D_3,
// which is the Shu-Osher form rewritten with U^(k) = U^n + D_k: increments are
// stored with their own relative precision, and the final sum is compensated
// (TwoSum) with a running remainder `lo`, so state rounding does not
// accumulate over many steps.
enum StageMode { kModeRHS = 0, kModeIncrement = 1, kModeFinal = 2, kModePartial = 3 };
// What a stage reads and writes, as a template parameter (SPEC) of the kernels that are compiled per stage:
// kSpecAny leaves it to StageArgs.  kSpecFirst: increment with U^n = the stencil state and no earlier
// increment; kSpecSecond: increment on top of an earlier one; kSpecFinal: the last stage; kSpecPartial: kModePartial.
// The row loop keeps two faces in flight per thread, so each register and instruction beside them counts:
// without the tests and loads of the other stages R = 2 needs 116-128 registers (128, capped, with them).
// Measured per step: R = 1/2/3 at 1024^2 164/198/261 -> 142/179/246 us, 4096^2 R = 2 2421 -> 2218 us.
enum StageSpec { kSpecAny = -1, kSpecRHS = 0, kSpecFirst = 1, kSpecSecond = 2, kSpecFinal = 3, kSpecPartial = 4 };
// kModePartial (3D only): the xy-plane kernel writes its part of L, -(div_x/dx + div_y/dy),
// to `out`; the z-marching kernel adds the z part and applies modes 0-2.

template <typename T>
struct StageArgs {
    const T *U;                // stencil state of this stage, SoA [nc][nz][ny][nx]
    const T *U0;               // U^n at the output cell (modes 1, 2); may equal U
    const T *Din;              // previous increment at the output cell (null = 0)
    T *Dout;                   // mode 1: D_k = b (Din + dt L); may equal Din
    T *Vout;                   // mode 1: U^n + D_k (next stage's stencil state)
    T *out;                    // mode 0: L(U); mode 2: U^{n+1} (may equal U0)
    T *lo;                     // mode 2: compensation remainder in/out (null: none)
    int n[3];                  // cells per dimension (x, y, z)
    int per[3];                // periodic flag per dimension
    T idx[3];                  // 1/dx per dimension
    T b;                       // stage weight b_k
    int mode;                  // StageMode
    int u0_is_stencil;         // U0 == U: take U^n from the staged stencil data
    long cstride;              // distance between components (cells of the whole grid)
    const T *P;                // z kernel: x+y part of L written by the plane kernel
    const double *dt_dev;      // device dt (or null: use dt)
    double dt;
    unsigned long long *rate;  // if non-null: atomic max of (|u_d| + c)/dx_d of the result (double bits)
    int *flags;                // bit 0: non-physical state met
    int W, nstrips, H, nseg;   // schedule: strip width, #strips, segment height, #segments
    // Slab decomposition: along the slowest dimension (slab_dim = ndim-1, or -1 if no side is
    // external) the ghost layers of an external side come from a caller-filled halo buffer of
    // G = R+3 layers, [nc][G][layer], layer k = the k-th cell beyond the side in increasing order.
    int slab_dim;
    int ext[2];                // low / high side external
    const T *halo[2];          // halo buffers of the low / high side
};

// Source of layer g (a cell index along the slab dimension, possibly a ghost) of a
// state whose layers are `unit` cells apart: the state itself, or an external halo.
// `cs` receives the distance between components at that source.
template <typename T>
__device__ __forceinline__ const T *layer_src(const StageArgs<T> &a, const T *U, int g, int n, int per, long unit,
                                              int G, long &cs)
{
    if (g < 0 && a.ext[0]) {
        cs = (long)G * unit;
        return a.halo[0] + (long)(g + G) * unit;
    }
    if (g >= n && a.ext[1]) {
        cs = (long)G * unit;
        return a.halo[1] + (long)(g - n) * unit;
    }
    cs = a.cstride;
    return U + (long)bc_map(g, n, per) * unit;
}

__device__ __forceinline__ unsigned smem_u32(const void *p)
{
    return static_cast<unsigned>(__cvta_generic_to_shared(p));
}

template <typename T>
__device__ __forceinline__ void cp_async_elem(T *dst, const T *src)
{
    static_assert(sizeof(T) == 4 || sizeof(T) == 8, "element size");
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(smem_u32(dst)), "l"(src), "n"(sizeof(T)));
}

__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;\n" ::); }

// Bounds-checked build (-DGPWENO_CHECKED; the tests build it as a library of its own): every
// shared-memory and global access of the stage kernels is first checked against the extent of
// its array; a violation sets bit `site` of the plan's flag word and skips the access (a read
// yields zero).  The default build compiles the checks away.
#ifdef GPWENO_CHECKED
constexpr bool kChecked = true;
#else
constexpr bool kChecked = false;
#endif
enum CheckSite {
    kChkRingWrite = 1,   // staging copy into the shared ring (2D, xy-planes)
    kChkStateRead = 2,   // global source of a staging copy (stage state or halo buffer)
    kChkRingRead = 3,    // stencil or U^n read from the ring
    kChkFaceWrite = 4,   // staged x-face fluxes
    kChkFaceRead = 5,
    kChkEpiRead = 6,     // U^n, increment, remainder or partial L of an output cell
    kChkEpiWrite = 7,    // stage outputs
    kChkZRing = 8,       // z kernel: shared ring
    kChkZState = 9,      // z kernel: staging source
    kChkLine = 10,       // 1D kernel: shared row and face arrays
    kChkLineState = 11   // 1D kernel: staging source
};

__device__ __forceinline__ bool chk(long long i, long long n, int site, int *flags)
{
    if constexpr (kChecked) {
        if (i < 0 || i >= n) {
            atomicOr(flags, 1 << site);
            return false;
        }
    }
    return true;
}

// Checked build: does p point into the stage state (ext_state elements) or into a registered
// halo buffer (ext_halo elements each)?
template <typename T>
__device__ __forceinline__ bool src_ok(const StageArgs<T> &a, const T *p, long ext_state, long ext_halo, int site)
{
    if constexpr (kChecked) {
        const bool in = (p >= a.U && p < a.U + ext_state) ||
                        (a.halo[0] != nullptr && p >= a.halo[0] && p < a.halo[0] + ext_halo) ||
                        (a.halo[1] != nullptr && p >= a.halo[1] && p < a.halo[1] + ext_halo);
        if (!in) atomicOr(a.flags, 1 << site);
        return in;
    }
    return true;
}

// Ring geometry of the 2D kernel for radius R and block size NT.
template <int R, int NT>
struct Ring2D {
    static constexpr int G = R + 3;                      // ghost layers
    static constexpr int LOW = R > 2 ? R : 2;            // rows below s still in use
    static constexpr int NEEDED = LOW + R + 3;           // rows s-LOW .. s+R+2 (one prefetched)
    static constexpr int ROWS = NEEDED <= 8 ? 8 : 16;    // power of two: slot = row & (ROWS-1)
    static constexpr int STRIDE = NT - 5 + 2 * G;        // elements per ring row and component
    static constexpr int WMAX = NT - 5;
    static __device__ __forceinline__ int slot(int g) { return g & (ROWS - 1); }
};

template <typename T, int R, int NT, int NC = 4>
constexpr size_t stage2d_smem_bytes()
{
    using RG = Ring2D<R, NT>;
    return sizeof(T) * (size_t)(RG::ROWS * NC * RG::STRIDE + 2 * NC * NT);
}

// Error-free sum a + b = s + e (Knuth's TwoSum).
template <typename T>
__device__ __forceinline__ T two_sum(T a, T b, T &e)
{
    const T s = a + b;
    const T bb = s - a;
    e = (a - (s - bb)) + (b - bb);
    return s;
}

// Epilogue of one cell and component: L is the RHS, u the stencil-state value of
// the cell, u0/din/lo the prefetched U^n, previous increment and remainder.
// Returns the value whose wavespeed the CFL reduction sees (mode 2: U^{n+1}).
template <typename T, int SPEC = kSpecAny>
__device__ __forceinline__ T stage_epilogue(const StageArgs<T> &a, long cell, T L, T u0, T din, T lo, T dt,
                                            long extent)
{
    if (!chk(cell, extent, kChkEpiWrite, a.flags)) return L;
    if (SPEC == kSpecAny ? a.mode == kModeRHS : SPEC == kSpecRHS) {
        a.out[cell] = L;
        return L;
    }
    // uncontracted, so that every kernel adds the same rounded increment
    const T inc = Num<T>::mul_rn(a.b, fma(dt, L, din));
    if (SPEC == kSpecAny ? a.mode == kModeIncrement : SPEC != kSpecFinal) {
        a.Dout[cell] = inc;
        a.Vout[cell] = u0 + inc;
        return u0 + inc;
    }
    if (a.lo) {
        T e;
        const T t = inc + lo;
        const T snew = two_sum<T>(u0, t, e);
        a.out[cell] = snew;
        a.lo[cell] = e;
        return snew;
    }
    const T snew = u0 + inc;
    a.out[cell] = snew;
    return snew;
}

// Rate (|u_d| + c) / dx_d of a natural-order 2D state.
template <typename T>
__device__ __forceinline__ void rates2d(const T (&u)[4], T gam, const T (&idx)[3], T &rx, T &ry)
{
    T ir = Num<T>::rcp_ieee(u[0]);
    T vx = u[1] * ir, vy = u[2] * ir;
    T pr = (gam - T(1)) * (u[3] - T(0.5) * (u[1] * vx + u[2] * vy));
    T c = Num<T>::sqrt_ieee(Num<T>::fmax(gam * pr * ir, T(0)));
    rx = (Num<T>::fabs(vx) + c) * idx[0];
    ry = (Num<T>::fabs(vy) + c) * idx[1];
}

// One segment: rows [y0, y1) of strip `strip` of the xy-plane starting at cell offset zoff.
// NC = 4 (2D) or 5 (an xy-plane of a 3D grid).
// ONE_SITE: evaluate the y- and x-face through one copy of the face routine (a
// loop of two passes) instead of two inlined copies.  Two copies let the compiler
// interleave the two independent faces (faster for the 2D kernels, the FP32 batch
// included, and in 3D at R = 1 and 2); one copy halves the code, which pays in the FP64 batch (fewer spills
// with three radii in one kernel) and in 3D at R = 3.
template <typename T, int R, int NT, int NC = 4, int VAR = 0, bool ONE_SITE = false, int SPEC = kSpecAny, bool P5 = false>
__device__ __forceinline__ void stage2d_segment(const StageArgs<T> &a, const FaceTables<T, R> &tb, int strip, int y0,
                                                int y1, T *smem, T dt, T &rmx, T &rmy, Physical<T> &ph, long zoff = 0)
{
    using RG = Ring2D<R, NT>;
    constexpr int G = RG::G, ROWS = RG::ROWS, STRIDE = RG::STRIDE;
    constexpr int NS = 2 * R + 2;
    // FP32 2D kernel: the four components of a ring element and of a staged face flux sit side
    // by side (one 16-byte shared load per stencil cell or face flux); otherwise one array per
    // component.  The one-site loop (3D planes, FP64 batches), the FD-Flux form and GP-AO keep the
    // per-component arrays: there the aligned register quads of 16-byte loads cost spills.
    constexpr bool VEC = std::is_same<T, float>::value && NC == 4 && !ONE_SITE && (VAR & (kVarFdFlux | kVarAo)) == 0;
    T *ring = smem;                              // [ROWS][NC][STRIDE], or [ROWS][STRIDE][4] (VEC)
    T *FA = smem + ROWS * NC * STRIDE;           // [NC][NT] (or [NT][4]): x-face A (flux relative to cell s)
    T *FM = FA + NC * NT;                        // [NC][NT] (or [NT][4]): x-face M (relative to cell s+1)
    // offset of component c of element col in the ring row starting at `base`, and of a face flux
    auto ro = [](int base, int col, int c) { return VEC ? base + col * 4 + c : base + c * STRIDE + col; };
    auto fo = [](int t, int c) { return VEC ? t * 4 + c : c * NT + t; };
    // the NC values of element col of a ring row (VEC: one 16-byte load)
    auto ring_elem = [&](int base, int col, T (&v)[NC]) {
        if constexpr (kChecked) {
            const int first = VEC ? base + col * 4 : base + col, last = VEC ? first + 3 : first + (NC - 1) * STRIDE;
            if (!chk(first, ROWS * NC * STRIDE, kChkRingRead, a.flags) ||
                !chk(last, ROWS * NC * STRIDE, kChkRingRead, a.flags)) {
#pragma unroll
                for (int c = 0; c < NC; ++c) v[c] = T(0);
                return;
            }
        }
        if constexpr (VEC) {
            const float4 q = *reinterpret_cast<const float4 *>(ring + base + col * 4);
            v[0] = q.x;
            v[1] = q.y;
            v[2] = q.z;
            v[3] = q.w;
        } else {
#pragma unroll
            for (int c = 0; c < NC; ++c) v[c] = ring[base + c * STRIDE + col];
        }
    };
    // one ring element (checked build: in bounds or zero)
    auto ring_at = [&](int i) -> T { return chk(i, ROWS * NC * STRIDE, kChkRingRead, a.flags) ? ring[i] : T(0); };
    auto stage_face = [&](T *F, int t, const T (&v)[NC]) {
        if (!chk(t, NT, kChkFaceWrite, a.flags)) return;
        if constexpr (VEC) {
            *reinterpret_cast<float4 *>(F + t * 4) = make_float4(v[0], v[1], v[2], v[3]);
        } else {
#pragma unroll
            for (int c = 0; c < NC; ++c) F[c * NT + t] = v[c];
        }
    };
    const int tid = threadIdx.x;
    const int nx = a.n[0], ny = a.n[1];
    const long plane = a.cstride;
    const int x0 = strip * a.W;
    const int Wc = min(a.W, nx - x0);
    const int s_begin = y0 - 3, s_end = y1 + 1;
    const int rowlen = Wc + 2 * G;
    const T idx[3] = {a.idx[0], a.idx[1], a.idx[2]};

    // one staging copy (checked build: destination in the ring, source in the state or a halo)
    auto stage_copy = [&](T *dst, const T *src) {
        if (!chk(dst - ring, ROWS * NC * STRIDE, kChkRingWrite, a.flags) ||
            !src_ok<T>(a, src, (long)NC * plane, (long)NC * G * nx, kChkStateRead))
            return;
        cp_async_elem(dst, src);
    };
    // grid columns of this thread's ring elements (the same for every row)
    const int gx0 = bc_map(x0 - G + min(tid, rowlen - 1), nx, a.per[0]);
    const int gx1 = bc_map(x0 - G + min(tid + NT, rowlen - 1), nx, a.per[0]);
    auto load_row = [&](int g) {
        T *dst = ring + RG::slot(g) * (NC * STRIDE);
        if ((VAR & kVarSlab) != 0 && NC == 4 && a.slab_dim == 1 && ((g < 0 && a.ext[0]) || (g >= ny && a.ext[1]))) {
            // a ghost row of an external side: from the halo buffer [nc][G][nx]
            const T *src = g < 0 ? a.halo[0] + (long)(g + G) * nx : a.halo[1] + (long)(g - ny) * nx;
            for (int col = tid; col < rowlen; col += NT) {
                const int gx = col == tid ? gx0 : gx1;
#pragma unroll
                for (int c = 0; c < NC; ++c) stage_copy(dst + ro(0, col, c), src + (long)c * G * nx + gx);
            }
            return;
        }
        const int gy = bc_map(g, ny, a.per[1]);
        const T *src = a.U + zoff + (long)gy * nx;
        static_assert(STRIDE <= 2 * NT, "a ring row is at most two elements per thread");
        for (int col = tid; col < rowlen; col += NT) {
            const int gx = col == tid ? gx0 : gx1;
#pragma unroll
            for (int c = 0; c < NC; ++c) stage_copy(dst + ro(0, col, c), src + c * plane + gx);
        }
    };

    // prologue: rows needed by the first y-face
    for (int g = s_begin - R; g <= s_begin + 1 + R; ++g) load_row(g);
    cp_async_commit();
    cp_async_wait_all();
    __syncthreads();

    // per column: partial sums of the next four rows' corrected y-differences (Divergence::march), the
    // difference of output row r, and M of the previous y-face
    using Dv = Divergence<T, VAR>;
    T acc[NC][4], divy[NC], Mp[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        acc[c][0] = acc[c][1] = acc[c][2] = acc[c][3] = T(0);
        divy[c] = Mp[c] = T(0);
    }

    for (int s = s_begin; s <= s_end; ++s) {
        if (s < s_end) load_row(s + 2 + R);
        cp_async_commit();
        const int r = s - 2;
        const bool out_row = r >= y0;
        const bool col_ok = tid < Wc;

        // U^n, previous increment and remainder of this thread's output cell,
        // in flight during the face work
        T u0[NC], din[NC], lov[NC];
        const long cell = zoff + (long)r * nx + x0 + tid;
        constexpr bool kAny = SPEC == kSpecAny;
        const bool epi = out_row && col_ok && (kAny ? a.mode == kModeIncrement || a.mode == kModeFinal : SPEC != kSpecRHS && SPEC != kSpecPartial);
        const bool rd_u0 = kAny ? !a.u0_is_stencil : SPEC >= kSpecSecond;
        const bool rd_din = kAny ? a.Din != nullptr : SPEC >= kSpecSecond;
        const bool rd_lo = a.lo && (kAny ? a.mode == kModeFinal : SPEC == kSpecFinal);
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const bool in = !epi || chk(c * plane + cell, (long)NC * plane, kChkEpiRead, a.flags);
            u0[c] = (epi && in && rd_u0) ? a.U0[c * plane + cell] : T(0);
            din[c] = (epi && in && rd_din) ? a.Din[c * plane + cell] : T(0);
            lov[c] = (epi && in && rd_lo) ? a.lo[c * plane + cell] : T(0);
        }

        if constexpr (ONE_SITE) {
            // ---- y-face s+1/2 of column tid (pass 0) and x-face tid of output row r (pass 1),
            // through one copy of the face routine ------------------------------
            const bool do_y = col_ok, do_x = out_row && tid < Wc + 5;
#pragma unroll 1
            for (int pass = 0; pass < 2; ++pass) {
                if (pass == 0 ? !do_y : !do_x) continue;
                // stencil element (q, c): ring + off[q] + comp[c] * STRIDE, normal-first
                static_assert(!VEC, "the one-site loop keeps one array per component");
                int off[NS];
#pragma unroll
                for (int q = 0; q < NS; ++q)
                    off[q] = pass == 0 ? RG::slot(s - R + q) * (NC * STRIDE) + G + tid : RG::slot(r) * (NC * STRIDE) + tid + q;
                T st[NS][NC];
#pragma unroll
                for (int q = 0; q < NS; ++q)
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        // a y-face's normal is the second velocity: (rho, rho v, rho u, [rho w], E)
                        const int cc = pass == 0 ? (c == 1 ? 2 : (c == 2 ? 1 : c)) : c;
                        st[q][c] = ring_at(off[q] + cc * STRIDE);
                    }
                T An[NC], Mn[NC];
                face_eval<T, NC, R, VAR, P5>(st, tb, An, Mn, ph);
                if (pass == 0) {
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        const int pc = c == 1 ? 2 : (c == 2 ? 1 : c);   // back to natural order
                        divy[c] = Dv::march(acc[c], An[pc] - Mp[c]);    // jump across row s (valid once s > s_begin)
                        Mp[c] = Mn[pc];
                    }
                } else {
                    stage_face(FA, tid, An);
                    stage_face(FM, tid, Mn);
                }
            }
        } else {
            // ---- y-face s+1/2 of column tid --------------------------------
            if (col_ok) {
                T st[NS][NC];
#pragma unroll
                for (int q = 0; q < NS; ++q) {
                    const int base = RG::slot(s - R + q) * (NC * STRIDE);
                    // normal-first for a y-face: (rho, rho v, rho u, [rho w], E)
                    if constexpr (VEC) {
                        T v[NC];
                        ring_elem(base, G + tid, v);
#pragma unroll
                        for (int c = 0; c < NC; ++c) st[q][c] = v[c == 1 ? 2 : (c == 2 ? 1 : c)];
                    } else {
#pragma unroll
                        for (int c = 0; c < NC; ++c) st[q][c] = ring_at(ro(base, G + tid, c == 1 ? 2 : (c == 2 ? 1 : c)));
                    }
                }
                T An[NC], Mn[NC];
                face_eval<T, NC, R, VAR, P5>(st, tb, An, Mn, ph);
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    const int pc = c == 1 ? 2 : (c == 2 ? 1 : c);   // back to natural order
                    divy[c] = Dv::march(acc[c], An[pc] - Mp[c]);    // jump across row s (valid once s > s_begin)
                    Mp[c] = Mn[pc];
                }
            }
            // ---- x-faces of output row r ----------------------------------
            if (out_row && tid < Wc + 5) {
                const int base = RG::slot(r) * (NC * STRIDE);
                T st[NS][NC];
#pragma unroll
                for (int q = 0; q < NS; ++q) ring_elem(base, tid + q, st[q]);
                T An[NC], Mn[NC];
                face_eval<T, NC, R, VAR, P5>(st, tb, An, Mn, ph);
                stage_face(FA, tid, An);
                stage_face(FM, tid, Mn);
            }
        }
        __syncthreads();
        // ---- divergence and stage combination -------------------------
        if (out_row && col_ok && chk(tid + 5, NT, kChkFaceRead, a.flags)) {
            const int ubase = RG::slot(r) * (NC * STRIDE);
            T un4[NC];
            if constexpr (VEC) {
                if (!rd_u0) ring_elem(ubase, G + tid, un4);
            }
            // x-faces t = tid..tid+5 are s' = x-3..x+2 around cell x = x0 + tid; the flux jumps
            // dF_k = A_{k+1} - M_k across the five cells around x (VEC: all components from
            // 16-byte loads; otherwise one component at a time)
            T dxk[VEC ? 5 : 1][NC];
            if constexpr (VEC) {
#pragma unroll
                for (int k = 0; k < 5; ++k) {
                    const float4 q = *reinterpret_cast<const float4 *>(FA + (tid + k + 1) * 4);
                    const float4 m = *reinterpret_cast<const float4 *>(FM + (tid + k) * 4);
                    dxk[k][0] = q.x - m.x;
                    dxk[k][1] = q.y - m.y;
                    dxk[k][2] = q.z - m.z;
                    dxk[k][3] = q.w - m.w;
                }
            }
            T res[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                T dx[5];
#pragma unroll
                for (int k = 0; k < 5; ++k) dx[k] = VEC ? dxk[VEC ? k : 0][c] : FA[fo(tid + k + 1, c)] - FM[fo(tid + k, c)];
                const T L = -fma(Dv::of(dx), idx[0], divy[c] * idx[1]);
                if (SPEC == kSpecPartial || (kAny && a.mode == kModePartial)) {
                    if (chk(c * plane + cell, (long)NC * plane, kChkEpiWrite, a.flags)) a.out[c * plane + cell] = L;
                    res[c] = L;
                } else {
                    const T un = !rd_u0 ? (VEC ? un4[c] : ring_at(ro(ubase, G + tid, c))) : u0[c];
                    res[c] = stage_epilogue<T, SPEC>(a, c * plane + cell, L, un, din[c], lov[c], dt, (long)NC * plane);
                }
            }
            if (NC == 4 && a.rate && (kAny ? a.mode == kModeFinal : SPEC == kSpecFinal)) {
                T rx, ry;
                rates2d<T>(reinterpret_cast<const T(&)[4]>(res), tb.gamma, idx, rx, ry);
                rmx = Num<T>::fmax(rmx, rx);
                rmy = Num<T>::fmax(rmy, ry);
            }
        }
        cp_async_wait_all();
        __syncthreads();
    }
}

template <typename T>
__device__ __forceinline__ void finish_block(const StageArgs<T> &a, T r0, T r1, T r2, bool ok)
{
    if (a.rate) {
        double v0 = (double)r0, v1 = (double)r1, v2 = (double)r2;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            v0 = fmax(v0, __shfl_xor_sync(0xffffffffu, v0, o));
            v1 = fmax(v1, __shfl_xor_sync(0xffffffffu, v1, o));
            v2 = fmax(v2, __shfl_xor_sync(0xffffffffu, v2, o));
        }
        if ((threadIdx.x & 31) == 0) {
            // non-negative doubles order like their bit patterns; NaN wins (all ones exponent)
            atomicMax(a.rate + 0, (unsigned long long)__double_as_longlong(v0));
            atomicMax(a.rate + 1, (unsigned long long)__double_as_longlong(v1));
            atomicMax(a.rate + 2, (unsigned long long)__double_as_longlong(v2));
        }
    }
    if (__any_sync(0xffffffffu, !ok) && (threadIdx.x & 31) == 0) atomicOr(a.flags, 1);
}

// Programmatic dependent launch: wait until the stream's preceding grid has
// finished and its writes are visible (a no-op without a programmatic
// dependency), then allow the stream's next kernel to be scheduled, so that its
// launch overlaps this grid's tail.  Every global access comes after this.
__device__ __forceinline__ void pdl_enter()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// First row of CTA b in the cost-balanced split of the strip-major row order
// [0, total) over `grid` CTAs.  A row costs 2 (one x- and one y-face per
// column) and every strip start inside a range costs 5 more (the warm-up
// y-face rows of a new segment), so rows [0, u) cost 2u + 5 floor((u-1)/ny);
// CTA b starts at the first row where that reaches b/grid of the total.
// Non-decreasing in b, 0 at b = 0 and total at b = grid, so the ranges
// [start(b), start(b+1)) partition the rows.
__device__ __forceinline__ long long balanced_start(int b, int grid, long long total, int ny, int nstrips)
{
    if (b <= 0) return 0;
    if (b >= grid) return total;
    const long long ctot = 2 * total + 5 * ((total - 1) / ny);
    const long long c = (ctot * b + grid / 2) / grid;
    for (int k = 0; k < nstrips; ++k) {
        const long long lo = (long long)k * ny, hi = lo + ny;
        if (2 * hi + 5LL * k >= c) return min(max((c - 5LL * k + 1) / 2, lo), hi);
    }
    return total;
}

// Resident threads per SM the 2D kernel's register budget is cut for: 512 in FP32 (128 registers), 256 in
// FP64 (255).  GP-AO and FD-Flux faces hold more at once (two stencil sizes, the two split fluxes) and
// spill there: 384 (168 registers) for R = 1, 2 and 256 for R = 3.  Measured, step on a four-quadrant grid of
// 1000 x 900: GP-AO R = 3 656 -> 543 us, R = 2 349 -> 340; FD-Flux R = 3 508 -> 412, R = 2 295 -> 281,
// R = 1 200 -> 195 us; R = 2 with 256 threads loses (430 and 357 us).  The 3D kernels, with one face in
// flight per thread, need the 512 threads also where they spill (128^3 GP-AO R = 3 2358 us, 2735 with 256).
template <typename T, int R, int VAR>
constexpr int kResident = sizeof(T) == 8 ? 256 : ((VAR & (kVarAo | kVarFdFlux)) == 0 ? 512 : (R == 3 ? 256 : 384));

// MINB: resident CTAs per SM the register budget is cut for (the default four 128-thread CTAs
// in FP32 at 128 registers; three give the compiler ~150 registers, which pays on small grids,
// see the host's choice in launch_stage_R).
template <typename T, int R, int NT, int VAR = 0, int MINB = kResident<T, R, VAR> / NT, int SPEC = kSpecAny>
__global__ void __launch_bounds__(NT, MINB) stage2d_kernel(StageArgs<T> a, TablesFor<T, R, VAR> tb)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *smem = reinterpret_cast<T *>(smem_raw);
    pdl_enter();
    const T dt = a.dt_dev ? (T)(*a.dt_dev) : (T)a.dt;
    T rmx = T(0), rmy = T(0);
    Physical<T> ph;
    // Persistent schedule: the strips' rows, laid end to end (strip-major),
    // are split into gridDim.x ranges of equal estimated cost; a range that
    // crosses a strip boundary becomes two segments.
    const int ny = a.n[1];
    const long long total = (long long)a.nstrips * ny;
    long long u = balanced_start(blockIdx.x, gridDim.x, total, ny, a.nstrips);
    const long long uend = balanced_start(blockIdx.x + 1, gridDim.x, total, ny, a.nstrips);
    while (u < uend) {
        const int strip = (int)(u / ny);
        const int y0 = (int)(u - (long long)strip * ny);
        const int y1 = (int)min((long long)ny, y0 + (uend - u));
        stage2d_segment<T, R, NT, 4, VAR, false, SPEC>(a, tb, strip, y0, y1, smem, dt, rmx, rmy, ph);
        u += y1 - y0;
    }
    finish_block<T>(a, rmx, rmy, T(0), ph.good());
}

// ---------------------------------------------------------------------------
// 3D.  Each stage is two launches: the xy-plane kernel below runs the 2D
// column-strip marching routine (5 components) on every z-plane and writes
// -(div_x/dx + div_y/dy) to a stage buffer P; the z-marching kernel then walks
// contiguous runs of xy-columns along z, evaluates each z-face once, adds
// -div_z/dz to P and applies the stage update.  P is a buffer the update later
// overwrites cell by cell (each cell reads its own P first), so 3D needs no
// scratch beyond 2D's.
//
// Form of the 3D kernels by radius (FP32, default faces), measured on shock boxes, step us: two inlined faces per row of the
// plane kernel and packed fields in both kernels at R = 1 (256^3 3688 -> 3476), two faces and packed fields in
// the z kernel only at R = 2 (4671 -> 4575; 4940 with packed planes), neither at R = 3, where the
// registers run out (6168; 6314 with two faces, 6493 packed).
template <typename T, int R, int VAR>
constexpr bool kOneSitePlane = sizeof(T) == 8 || R == 3 || (VAR & (kVarAo | kVarFdFlux)) != 0;
template <typename T, int R>
constexpr bool kPackPlane = R == 1;
template <typename T, int R>
constexpr bool kPackZ = R <= 2;

template <typename T, int R, int NT, int VAR = 0>
__global__ void __launch_bounds__(NT, (sizeof(T) == 4 ? 512 : 256) / NT) plane3d_kernel(StageArgs<T> a, TablesFor<T, R, VAR> tb)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *smem = reinterpret_cast<T *>(smem_raw);
    pdl_enter();
    T rmx = T(0), rmy = T(0);
    Physical<T> ph;
    const int nx = a.n[0], ny = a.n[1], nz = a.n[2];
    const long per_plane = (long)a.nstrips * ny;
    const long total = per_plane * nz;
    long long u = (long long)total * blockIdx.x / gridDim.x;
    const long long uend = (long long)total * (blockIdx.x + 1) / gridDim.x;
    while (u < uend) {
        const int z = (int)(u / per_plane);
        const long rem = u - (long long)z * per_plane;
        const int strip = (int)(rem / ny);
        const int y0 = (int)(rem - (long)strip * ny);
        const int y1 = (int)min((long long)ny, y0 + (uend - u));
        stage2d_segment<T, R, NT, 5, VAR, kOneSitePlane<T, R, VAR>, kSpecPartial, kPackPlane<T, R>>(a, tb, strip, y0, y1, smem, T(0), rmx, rmy, ph, (long)z * nx * ny);
        u += y1 - y0;
    }
    if (__any_sync(0xffffffffu, !ph.good()) && (threadIdx.x & 31) == 0) atomicOr(a.flags, 1);
}

template <int R>
struct RingZ {
    static constexpr int LOW = R > 2 ? R : 2;
    static constexpr int NEEDED = LOW + R + 3;
    static constexpr int ROWS = NEEDED <= 8 ? 8 : 16;
    static __device__ __forceinline__ int slot(int g) { return g & (ROWS - 1); }
};

template <typename T, int R, int NT>
constexpr size_t stagez_smem_bytes()
{
    return sizeof(T) * (size_t)(RingZ<R>::ROWS * 5 * NT);
}

template <typename T>
__device__ __forceinline__ void rates3d(const T (&u)[5], T gam, const T (&idx)[3], T &rx, T &ry, T &rz)
{
    const T ir = Num<T>::rcp_ieee(u[0]);
    const T vx = u[1] * ir, vy = u[2] * ir, vz = u[3] * ir;
    const T pr = (gam - T(1)) * (u[4] - T(0.5) * (u[1] * vx + u[2] * vy + u[3] * vz));
    const T c = Num<T>::sqrt_ieee(Num<T>::fmax(gam * pr * ir, T(0)));
    rx = (Num<T>::fabs(vx) + c) * idx[0];
    ry = (Num<T>::fabs(vy) + c) * idx[1];
    rz = (Num<T>::fabs(vz) + c) * idx[2];
}

// z-marching over columns [c0, c0+NT) of the flattened xy-plane, planes [z0, z1).
template <typename T, int R, int NT, int VAR = 0, int SPEC = kSpecAny>
__device__ __forceinline__ void stagez_segment(const StageArgs<T> &a, const FaceTables<T, R> &tb, long c0, int z0,
                                               int z1, T *ring, T dt, T (&rm)[3], Physical<T> &ph)
{
    using RZ = RingZ<R>;
    constexpr int NC = 5, NS = 2 * R + 2;
    const int tid = threadIdx.x;
    const int nz = a.n[2];
    const long plane = (long)a.n[0] * a.n[1];
    const long cs = a.cstride;
    const long col = c0 + tid;
    const bool col_ok = col < plane;
    const int s_begin = z0 - 3, s_end = z1 + 1;
    const T idx[3] = {a.idx[0], a.idx[1], a.idx[2]};

    auto load_plane = [&](int g) {
        if (!col_ok) return;
        constexpr int G = R + 3;
        T *dst = ring + RZ::slot(g) * (NC * NT) + tid;
        long ccs = cs;
        const T *src = ((VAR & kVarSlab) != 0 && a.slab_dim == 2 ? layer_src<T>(a, a.U, g, nz, a.per[2], plane, G, ccs)
                                                                 : a.U + (long)bc_map(g, nz, a.per[2]) * plane) +
                       col;
#pragma unroll
        for (int c = 0; c < NC; ++c)
            if (chk(dst + c * NT - ring, RZ::ROWS * NC * NT, kChkZRing, a.flags) &&
                src_ok<T>(a, src + c * ccs, NC * cs, (long)NC * G * plane, kChkZState))
                cp_async_elem(dst + c * NT, src + c * ccs);
    };
    for (int g = s_begin - R; g <= s_begin + 1 + R; ++g) load_plane(g);
    cp_async_commit();
    cp_async_wait_all();
    __syncthreads();

    using Dv = Divergence<T, VAR>;
    T acc[NC][4], divz[NC], Mp[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        acc[c][0] = acc[c][1] = acc[c][2] = acc[c][3] = T(0);
        divz[c] = Mp[c] = T(0);
    }

    for (int s = s_begin; s <= s_end; ++s) {
        if (s < s_end) load_plane(s + 2 + R);
        cp_async_commit();
        const int r = s - 2;
        const bool out = r >= z0 && col_ok;
        const long cell = (long)r * plane + col;
        T pv[NC], u0[NC], din[NC], lov[NC];
        constexpr bool kAny = SPEC == kSpecAny;
        const bool epi = out && (kAny ? a.mode == kModeIncrement || a.mode == kModeFinal : SPEC != kSpecRHS);
        const bool rd_u0 = kAny ? !a.u0_is_stencil : SPEC >= kSpecSecond;
        const bool rd_din = kAny ? a.Din != nullptr : SPEC >= kSpecSecond;
        const bool rd_lo = a.lo && (kAny ? a.mode == kModeFinal : SPEC == kSpecFinal);
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const bool in = !out || chk(c * cs + cell, NC * cs, kChkEpiRead, a.flags);
            pv[c] = (out && in) ? a.P[c * cs + cell] : T(0);
            u0[c] = (epi && in && rd_u0) ? a.U0[c * cs + cell] : T(0);
            din[c] = (epi && in && rd_din) ? a.Din[c * cs + cell] : T(0);
            lov[c] = (epi && in && rd_lo) ? a.lo[c * cs + cell] : T(0);
        }
        if (col_ok) {
            // normal-first for a z-face: (rho, rho w, rho u, rho v, E)
            T st[NS][NC];
#pragma unroll
            for (int q = 0; q < NS; ++q) {
                const T *rowp = ring + RZ::slot(s - R + q) * (NC * NT) + tid;
                if (!chk(rowp + 4 * NT - ring, RZ::ROWS * NC * NT, kChkZRing, a.flags)) rowp = ring;
                st[q][0] = rowp[0];
                st[q][1] = rowp[3 * NT];
                st[q][2] = rowp[1 * NT];
                st[q][3] = rowp[2 * NT];
                st[q][4] = rowp[4 * NT];
            }
            T An[NC], Mn[NC];
            face_eval<T, NC, R, VAR, kPackZ<T, R>>(st, tb, An, Mn, ph);
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                const int pc = c == 0 || c == 4 ? c : (c == 3 ? 1 : c + 1);   // back to natural order
                divz[c] = Dv::march(acc[c], An[pc] - Mp[c]);
                Mp[c] = Mn[pc];
            }
        }
        if (out) {
            const T *urow = ring + RZ::slot(r) * (NC * NT) + tid;
            if (!chk(urow + 4 * NT - ring, RZ::ROWS * NC * NT, kChkZRing, a.flags)) urow = ring;
            T res[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                const T L = fma(-divz[c], idx[2], pv[c]);
                const T un = !rd_u0 ? urow[c * NT] : u0[c];
                res[c] = stage_epilogue<T, SPEC>(a, c * cs + cell, L, un, din[c], lov[c], dt, NC * cs);
            }
            if (a.rate && (kAny ? a.mode == kModeFinal : SPEC == kSpecFinal)) {
                T rx, ry, rz;
                rates3d<T>(res, tb.gamma, idx, rx, ry, rz);
                rm[0] = Num<T>::fmax(rm[0], rx);
                rm[1] = Num<T>::fmax(rm[1], ry);
                rm[2] = Num<T>::fmax(rm[2], rz);
            }
        }
        cp_async_wait_all();
        __syncthreads();
    }
}

template <typename T, int R, int NT, int VAR = 0, int SPEC = kSpecAny>
__global__ void __launch_bounds__(NT, (sizeof(T) == 4 ? 512 : 256) / NT) stagez_kernel(StageArgs<T> a, TablesFor<T, R, VAR> tb)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *ring = reinterpret_cast<T *>(smem_raw);
    pdl_enter();
    const T dt = a.dt_dev ? (T)(*a.dt_dev) : (T)a.dt;
    T rm[3] = {T(0), T(0), T(0)};
    Physical<T> ph;
    const int nz = a.n[2];
    const long plane = (long)a.n[0] * a.n[1];
    const long groups = (plane + NT - 1) / NT;
    const long long total = (long long)groups * nz;
    long long u = total * blockIdx.x / gridDim.x;
    const long long uend = total * (blockIdx.x + 1) / gridDim.x;
    while (u < uend) {
        const long g = (long)(u / nz);
        const int z0 = (int)(u - (long long)g * nz);
        const int z1 = (int)min((long long)nz, z0 + (uend - u));
        stagez_segment<T, R, NT, VAR, SPEC>(a, tb, g * NT, z0, z1, ring, dt, rm, ph);
        u += z1 - z0;
    }
    finish_block<T>(a, rm[0], rm[1], rm[2], ph.good());
}

// ---------------------------------------------------------------------------
// 1D: a CTA owns a segment of W <= NT-5 cells; the segment and its ghost
// cells are staged in shared memory, the W+5 faces evaluated one per thread,
// corrected, differenced and combined.
template <typename T, int R, int NT>
constexpr size_t stage1d_smem_bytes()
{
    return sizeof(T) * (size_t)(3 * (NT - 5 + 2 * (R + 3)) + 2 * 3 * NT);
}

template <typename T, int R, int NT, int VAR = 0>
__global__ void __launch_bounds__(NT) stage1d_kernel(StageArgs<T> a, TablesFor<T, R, VAR> tb)
{
    constexpr int G = R + 3, NC = 3, NS = 2 * R + 2;
    constexpr int STRIDE = NT - 5 + 2 * G;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *row = reinterpret_cast<T *>(smem_raw);  // [NC][STRIDE]
    T *FA = row + NC * STRIDE;                 // [NC][NT]
    T *FM = FA + NC * NT;                      // [NC][NT]
    pdl_enter();
    const T dt = a.dt_dev ? (T)(*a.dt_dev) : (T)a.dt;
    const int tid = threadIdx.x;
    const int nx = a.n[0];
    T rmx = T(0);
    Physical<T> ph;
    for (int item = blockIdx.x; item < a.nstrips; item += gridDim.x) {
        const int x0 = item * a.W;
        const int Wc = min(a.W, nx - x0);
        for (int col = tid; col < Wc + 2 * G; col += NT) {
            long cs = nx;
            const T *src = (VAR & kVarSlab) != 0 && a.slab_dim == 0
                               ? layer_src<T>(a, a.U, x0 - G + col, nx, a.per[0], 1, G, cs)
                               : a.U + bc_map(x0 - G + col, nx, a.per[0]);
#pragma unroll
            for (int c = 0; c < NC; ++c)
                if (chk(col, STRIDE, kChkLine, a.flags) &&
                    src_ok<T>(a, src + c * cs, (long)NC * nx, (long)NC * G, kChkLineState))
                    row[c * STRIDE + col] = src[c * cs];
        }
        __syncthreads();
        if (tid < Wc + 5 && chk(tid + NS - 1, STRIDE, kChkLine, a.flags) && chk(tid, NT, kChkLine, a.flags)) {
            T st[NS][NC];
#pragma unroll
            for (int q = 0; q < NS; ++q)
#pragma unroll
                for (int c = 0; c < NC; ++c) st[q][c] = row[c * STRIDE + tid + q];
            T An[NC], Mn[NC];
            face_eval<T, NC, R, VAR>(st, tb, An, Mn, ph);
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                FA[c * NT + tid] = An[c];
                FM[c * NT + tid] = Mn[c];
            }
        }
        __syncthreads();
        if (tid < Wc && chk(tid + 5, NT, kChkLine, a.flags) && chk(G + tid, STRIDE, kChkLine, a.flags)) {
            T res[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                const T *fa = FA + c * NT + tid;
                const T *fm = FM + c * NT + tid;
                T dx[5];
#pragma unroll
                for (int k = 0; k < 5; ++k) dx[k] = fa[k + 1] - fm[k];
                const T L = -Divergence<T, VAR>::of(dx) * a.idx[0];
                const long cell = (long)c * nx + x0 + tid;
                const bool epi = a.mode != kModeRHS && chk(cell, (long)NC * nx, kChkEpiRead, a.flags);
                const T u0 = a.u0_is_stencil ? row[c * STRIDE + G + tid] : (epi ? a.U0[cell] : T(0));
                const T din = (epi && a.Din) ? a.Din[cell] : T(0);
                const T lov = (epi && a.lo && a.mode == kModeFinal) ? a.lo[cell] : T(0);
                res[c] = stage_epilogue<T>(a, cell, L, u0, din, lov, dt, (long)NC * nx);
            }
            if (a.rate && a.mode == kModeFinal) {
                T ir = Num<T>::rcp_ieee(res[0]);
                T vx = res[1] * ir;
                T pr = (tb.gamma - T(1)) * (res[2] - T(0.5) * res[1] * vx);
                T cc = Num<T>::sqrt_ieee(Num<T>::fmax(tb.gamma * pr * ir, T(0)));
                rmx = Num<T>::fmax(rmx, (Num<T>::fabs(vx) + cc) * a.idx[0]);
            }
        }
        __syncthreads();
    }
    finish_block<T>(a, rmx, T(0), T(0), ph.good());
}

// The same for short FP64 grids: a CTA of three warps owns W <= 27 cells and its W+5 <= 32 faces, warp k
// evaluating characteristic field k of every face (the Roe average by all three, each cell's own part of
// it once, the primitive differences in turns), then the left state, the right state and the neighbour flux, then
// component k of the flux.  A warp passes one FP64 instruction per 64 cycles, independent or not and however
// many of its lanes are active, and an SM one per 19 (measured with chains of fma), so a grid of a few
// warps is as slow as one face's instructions in a row: 17 us per stage of 256 cells at R = 2.  Three warps
// on one SM lose nothing to each other and split that row.
// Measured: 256-cell step R = 2 60.0 -> 36.7 us by fields, 33.3 us with the shared parts.
template <typename T, int R, int VAR>
__global__ void __launch_bounds__(96) stage1d_split_kernel(StageArgs<T> a, TablesFor<T, R, VAR> tb)
{
    constexpr int G = R + 3, NC = 3, NS = 2 * R + 2, NF = 32, E = 2;
    constexpr bool MEAN = (VAR & kVarMean) != 0;
    __shared__ T row[NC][NF + NS];        // staged cells x0-G .. x0+W+G-1
    __shared__ T part0[8][NF + NS];       // of each cell: 1/rho and CellPart
    __shared__ T dVs[2 * R][NC][NF];      // primitive differences of the cells beyond the neighbours
    __shared__ T q[2][NC][NF];            // left and right states in characteristic fields
    __shared__ T part[2][3 * NC + 2][NF]; // left, right: w, G, c, u, a
    __shared__ T nb[NC][NF];              // neighbour flux difference
    __shared__ T FA[NC][NF], FM[NC][NF];
    const int lane = threadIdx.x & 31, k = threadIdx.x >> 5, nx = a.n[0];
    pdl_enter();
    const T dt = a.dt_dev ? (T)(*a.dt_dev) : (T)a.dt;
    const int x0 = blockIdx.x * a.W, Wc = min(a.W, nx - x0);
    for (int col = lane; col < Wc + 2 * G; col += 32) {
        long cs = nx;
        const T *src = (VAR & kVarSlab) != 0 && a.slab_dim == 0 ? layer_src<T>(a, a.U, x0 - G + col, nx, a.per[0], 1, G, cs)
                                                                : a.U + bc_map(x0 - G + col, nx, a.per[0]);
        if (chk(col, NF + NS, kChkLine, a.flags) && src_ok<T>(a, src + k * cs, (long)NC * nx, (long)NC * G, kChkLineState))
            row[k][col] = src[k * cs];
    }
    __syncthreads();
    if (const int col = threadIdx.x; col < Wc + 2 * G && chk(col, NF + NS, kChkLine, a.flags)) {
        const T U[NC] = {row[0][col], row[1][col], row[2][col]};
        const CellPart<T, NC> cp = cell_part(U, tb);
        const T v[8] = {Num<T>::rcp(U[0]), cp.rs, cp.ir, cp.s, cp.u[0], cp.p, cp.hp, cp.c2};
#pragma unroll
        for (int c = 0; c < 8; ++c) part0[c][col] = v[c];
    }
    __syncthreads();
    const bool face = lane < Wc + 5 && chk(lane + NS - 1, NF + NS, kChkLine, a.flags);
    Physical<T> ph;
    FaceRoe<T, NC> f;
    if (face) {
        const int s = lane + R;
        const T uL[NC] = {row[0][s], row[1][s], row[2][s]}, uR[NC] = {row[0][s + 1], row[1][s + 1], row[2][s + 1]};
        CellPart<T, NC> L = {}, Rt = {};
        L.rs = part0[1][s];
        L.ir = part0[2][s];
        L.s = part0[3][s];
        L.u[0] = part0[4][s];
        L.p = part0[5][s];
        L.hp = part0[6][s];
        L.c2 = part0[7][s];
        Rt.rs = part0[1][s + 1];
        Rt.ir = part0[2][s + 1];
        Rt.s = part0[3][s + 1];
        f = face_roe<T, NC, true>(uL, uR, tb, L, Rt);
        // warp k takes every third of the other cells
        for (int i = k; i < 2 * R; i += NC) {
            const int j = lane + (i < R ? i : i + 2);
            const T uj[NC] = {row[0][j], row[1][j], row[2][j]};
            T dV[NC];
            f.prim_diff(uj, uL, part0[0][j], dV);
#pragma unroll
            for (int c = 0; c < NC; ++c) dVs[i][c][lane] = dV[c];
        }
    }
    __syncthreads();
    T us[NC], ur[NC];
    if (face) {
        T dV[NS][NC], d[NS];
#pragma unroll
        for (int j = 0; j < NS; ++j)
#pragma unroll
            for (int c = 0; c < NC; ++c)
                dV[j][c] = j == R ? T(0) : (j == R + 1 ? f.dVn[c] : dVs[j < R ? j : j - 2][c][lane]);
        // the rows of L_V: (0, -an, ap), (1, 0, -ie), (0, an, ap)
#pragma unroll
        for (int j = 0; j < NS; ++j)
            d[j] = j == R ? T(0) : (k == 0 ? f.lrow(0, dV[j]) : (k == 1 ? f.lrow(1, dV[j]) : f.lrow(E, dV[j])));
        const T fc = k == 0 ? f.lrow(0, f.Vs) : (k == 1 ? f.lrow(1, f.Vs) : f.lrow(E, f.Vs));
        T qL, qR;
        weno_states<T, R, MEAN, kUnitDifference<T, R, VAR>>(tb, d, fc, qL, qR);
        q[0][k][lane] = qL;
        q[1][k][lane] = qR;
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            us[c] = row[c][lane + R];
            ur[c] = row[c][lane + R + 1];
        }
    }
    __syncthreads();
    if (face && k < 2) {
        const T dq[NC] = {q[k][0][lane], q[k][1][lane], q[k][2][lane]};
        T w[NC], Gf[NC], cw[NC], un, cs;
        if (k == 0) f.left_state(dq, w);
        else f.right_state(dq, w);
        prim_pert<T, NC>(f.ref, w, tb.gamma, tb.igm1, Gf, cw, un, cs, ph);
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            part[k][c][lane] = w[c];
            part[k][NC + c][lane] = Gf[c];
            part[k][2 * NC + c][lane] = cw[c];
        }
        part[k][3 * NC][lane] = un;
        part[k][3 * NC + 1][lane] = cs;
    } else if (face) {
        T B[NC];
        f.flux_difference(us, ur, B);
        ph.need(f.c2, f.ref.p + f.dVn[E]);
#pragma unroll
        for (int c = 0; c < NC; ++c) nb[c][lane] = B[c];
    }
    __syncthreads();
    if (face) {
        const T uL = part[0][3 * NC][lane], aL = part[0][3 * NC + 1][lane];
        const T uR = part[1][3 * NC][lane], aR = part[1][3 * NC + 1][lane];
        T Ak;
        if (tb.flux == 0) {   // Lax-Friedrichs, component k alone (as face_flux)
            const T alpha = Num<T>::pmax(Num<T>::fabs(uL) + aL, Num<T>::fabs(uR) + aR);
            Ak = fma(-alpha, part[1][2 * NC + k][lane] - part[0][2 * NC + k][lane],
                     part[0][NC + k][lane] + part[1][NC + k][lane]);
        } else {
            T w[2][NC], Gf[2][NC], cw[2][NC], A[NC];
#pragma unroll
            for (int s = 0; s < 2; ++s)
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    w[s][c] = part[s][c][lane];
                    Gf[s][c] = part[s][NC + c][lane];
                    cw[s][c] = part[s][2 * NC + c][lane];
                }
            face_flux<T, NC, false>(f, tb, w[0], w[1], Gf[0], Gf[1], cw[0], cw[1], uL, uR, aL, aR, A);
            Ak = k == 0 ? A[0] : (k == 1 ? A[1] : A[2]);
        }
        FA[k][lane] = Ak;
        FM[k][lane] = fma(T(-2), nb[k][lane], Ak);
    }
    __syncthreads();
    T rmx = T(0);
    if (lane < Wc && chk(lane + 5, NF, kChkLine, a.flags)) {
        T dx[5];
#pragma unroll
        for (int j = 0; j < 5; ++j) dx[j] = FA[k][lane + j + 1] - FM[k][lane + j];
        const T L = -Divergence<T, VAR>::of(dx) * a.idx[0];
        const long cell = (long)k * nx + x0 + lane;
        const bool epi = a.mode != kModeRHS && chk(cell, (long)NC * nx, kChkEpiRead, a.flags);
        const T u0 = a.u0_is_stencil ? row[k][G + lane] : (epi ? a.U0[cell] : T(0));
        const T din = (epi && a.Din) ? a.Din[cell] : T(0);
        const T lov = (epi && a.lo && a.mode == kModeFinal) ? a.lo[cell] : T(0);
        q[0][k][lane] = stage_epilogue<T>(a, cell, L, u0, din, lov, dt, (long)NC * nx);
    }
    __syncthreads();
    if (a.rate && a.mode == kModeFinal && k == 0 && lane < Wc) {
        const T res[NC] = {q[0][0][lane], q[0][1][lane], q[0][2][lane]};
        const T ir = Num<T>::rcp_ieee(res[0]);
        const T vx = res[1] * ir;
        const T pr = (tb.gamma - T(1)) * (res[2] - T(0.5) * res[1] * vx);
        const T cc = Num<T>::sqrt_ieee(Num<T>::fmax(tb.gamma * pr * ir, T(0)));
        rmx = (Num<T>::fabs(vx) + cc) * a.idx[0];
    }
    finish_block<T>(a, rmx, T(0), T(0), ph.good());
}

// Maximum of (|u_d| + c)/dx_d over all cells (for the CFL time step).
template <typename T, int NC>
__global__ void __launch_bounds__(256) max_rate_kernel(const T *U, long ncell, StageArgs<T> a, T gam)
{
    T r[3] = {T(0), T(0), T(0)};
    for (long l = blockIdx.x * (long)blockDim.x + threadIdx.x; l < ncell; l += (long)gridDim.x * blockDim.x) {
        T u[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) u[c] = U[c * ncell + l];
        T ir = Num<T>::rcp_ieee(u[0]);
        T m2 = T(0);
#pragma unroll
        for (int d = 1; d < NC - 1; ++d) m2 = fma(u[d], u[d], m2);
        T pr = (gam - T(1)) * (u[NC - 1] - T(0.5) * m2 * ir);
        T c = Num<T>::sqrt_ieee(Num<T>::fmax(gam * pr * ir, T(0)));
#pragma unroll
        for (int d = 0; d < NC - 2; ++d) r[d] = Num<T>::fmax(r[d], (Num<T>::fabs(u[1 + d] * ir) + c) * a.idx[d]);
    }
    finish_block<T>(a, r[0], r[1], r[2], true);
}

// dt = cfl / sum_d rate_d, then the rate accumulators are cleared for the next use.
__global__ void dt_from_rate_kernel(unsigned long long *rate, int ndim, double cfl, double *dt_dev);

}  // namespace gpweno
