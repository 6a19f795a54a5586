// FP64 stages of 2D and 3D grids as two launches: every face of a band of the grid once (face_list_kernel,
// flux jumps' ingredients to the plan's workspace), then the divergence and the stage update
// (face_update_kernel).
//
// FP64 arithmetic is the whole cost on this part (two FP64 lanes per SM; a warp instruction holds
// the SM's pipe for 16 cycles), and a cell's face fluxes, written and read once, are some 130 bytes
// against over a thousand FP64 instructions.  So the split is made for the instruction count:
//   * no face is evaluated twice (the strip-marching kernel repeats 5 x-faces per strip row and 5 y-face
//     rows per segment: 25 % of the work at 512^2, several times the work on smaller grids);
//   * faces are numbered along x through the whole band, so all warps but the last of a direction
//     are full, whatever nx is;
//   * one CTA per SM takes an equal share of the band's warps of faces, so small grids use all SMs.
// The band (of the slowest dimension) bounds the workspace; consecutive bands repeat the five
// faces around their border.
// Measured on GB300 (strip marching -> this, equal bits): step of 128^2 R = 3 2351 -> 216 us, of 512^2 R = 2
// 2702 -> 1877 us, 3D right-hand side of 70x61x45 R = 2 2132 -> 948 us.  FP32 keeps marching: its faces
// are sixty times cheaper, and the fluxes' trip through memory would cost more than the repeated faces.
#pragma once
#include "stage.cuh"

namespace gpweno {

// Face arrays of one band.  Direction d holds n[d] = ext[d][0] ext[d][1] ext[d][2] faces numbered along x
// first, with ext[d][d] = cnt[d] faces along d starting at face lo[d] + 1/2, and 2 NC values of each
// ([A or M][component][face], natural component order) from element off[d] of buf.
template <typename T>
struct FaceBand {
    T *buf;
    long size;        // elements of buf
    long n[3], off[3];
    int ext[3][3];
    int lo[3];
    int wrap[3];      // 1: faces 0 .. n-1 of a periodic dimension, numbered modulo n
    int l0, l1;       // layers [l0, l1) of the slowest dimension
};

// One warp per 32 consecutive faces; CTA b takes items [b/grid, (b+1)/grid) of all directions' items.
template <typename T, int NC, int R, int VAR, int NT>
__global__ void __launch_bounds__(NT, 1) face_list_kernel(StageArgs<T> a, FaceBand<T> fb, TablesFor<T, R, VAR> tb)
{
    constexpr int ND = NC - 2, NS = 2 * R + 2, G = R + 3;
    pdl_enter();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    long items[ND], total = 0;
#pragma unroll
    for (int d = 0; d < ND; ++d) total += items[d] = (fb.n[d] + 31) / 32;
    const long first = total * blockIdx.x / gridDim.x, last = total * (blockIdx.x + 1) / gridDim.x;
    Physical<T> ph;
    for (long it = first + warp; it < last; it += NT / 32) {
        int d = 0;
        long f = it;
        while (d < ND - 1 && f >= items[d]) f -= items[d++];
        f = f * 32 + lane;
        if (f >= fb.n[d]) continue;
        // position: coordinates of the face's cell s, x first
        int pos[3];
        const int e0 = fb.ext[d][0], e1 = fb.ext[d][1];
        const long fr = f / e0;
        pos[0] = (int)(f - fr * e0);
        pos[2] = ND == 3 ? (int)(fr / e1) : 0;
        pos[1] = (int)(fr - (long)pos[2] * e1);
        const int s = fb.lo[d] + pos[d];
        if (d != ND - 1) pos[ND - 1] += fb.l0;
        const long stride = d == 0 ? 1 : (d == 1 ? (long)a.n[0] : (long)a.n[0] * a.n[1]);
        long base = 0;   // the cells of the line through the face, without its coordinate along d
        if (d != 0) base += pos[0];
        if (d != 1) base += (long)pos[1] * a.n[0];
        if (ND == 3 && d != 2) base += (long)pos[2] * a.n[0] * a.n[1];
        // normal-first component order of the marching kernels: (n, other two in order)
        int perm[NC];
        perm[0] = 0;
        perm[1] = 1 + d;
        perm[2] = d == 0 ? 2 : 1;
        if (ND == 3) perm[3] = d == 2 ? 2 : 3;
        perm[NC - 1] = NC - 1;
        T st[NS][NC];
#pragma unroll
        for (int q = 0; q < NS; ++q) {
            const int g = s - R + q;
            long cs = a.cstride;
            const T *src;
            if ((VAR & kVarSlab) != 0 && d == ND - 1) {
                src = layer_src<T>(a, a.U, g, a.n[d], a.per[d], stride, G, cs) + base;
            } else {
                src = a.U + (long)bc_map(g, a.n[d], a.per[d]) * stride + base;
            }
#pragma unroll
            for (int c = 0; c < NC; ++c)
                st[q][c] = src_ok<T>(a, src + perm[c] * cs, (long)NC * a.cstride, (long)NC * G * (a.cstride / a.n[ND - 1]),
                                     kChkStateRead)
                               ? src[perm[c] * cs]
                               : T(0);
        }
        T A[NC], M[NC];
        face_eval<T, NC, R, VAR>(st, tb, A, M, ph);
        T *dst = fb.buf + fb.off[d] + f;
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            if (!chk(dst + (NC + perm[c]) * fb.n[d] - fb.buf, fb.size, kChkFaceWrite, a.flags)) continue;
            dst[perm[c] * fb.n[d]] = A[c];
            dst[(NC + perm[c]) * fb.n[d]] = M[c];
        }
    }
    if (__any_sync(0xffffffffu, !ph.good()) && lane == 0) atomicOr(a.flags, 1);
}

// Divergence and stage update of the band's cells: one CTA per strip (at most NT columns) of a row.
template <typename T, int NC, int VAR, int NT>
__global__ void __launch_bounds__(NT) face_update_kernel(StageArgs<T> a, FaceBand<T> fb, T gamma)
{
    constexpr int ND = NC - 2;
    pdl_enter();
    const T dt = a.dt_dev ? (T)(*a.dt_dev) : (T)a.dt;
    const T idx[3] = {a.idx[0], a.idx[1], a.idx[2]};
    T rm[3] = {T(0), T(0), T(0)};
    const long rows = (long)(fb.l1 - fb.l0) * (ND == 3 ? a.n[1] : 1);
    for (long w = blockIdx.x; w < rows * a.nstrips; w += gridDim.x) {
        const long row = w / a.nstrips;
        const int x0 = (int)(w - row * a.nstrips) * a.W;
        const int x = x0 + threadIdx.x;
        if ((int)threadIdx.x >= a.W || x >= a.n[0]) continue;
        // position within the band, and the cell
        const int z = ND == 3 ? (int)(row / a.n[1]) : 0;
        const int pos[3] = {x, ND == 3 ? (int)(row - (long)z * a.n[1]) : (int)row, z};
        const long cell = ((ND == 3 ? (long)(fb.l0 + z) * a.n[1] + pos[1] : (long)fb.l0 + row)) * a.n[0] + x;
        long at[ND][6];   // the faces around the cell in each direction
#pragma unroll
        for (int d = 0; d < ND; ++d) {
            const int ext0 = fb.ext[d][0], ext1 = fb.ext[d][1];
            const long stride = d == 0 ? 1 : (d == 1 ? (long)ext0 : (long)ext0 * ext1);
            long base = 0;
            if (d != 0) base += pos[0];
            if (d != 1) base += (long)pos[1] * ext0;
            if (ND == 3 && d != 2) base += (long)pos[2] * ext0 * ext1;
            const int c = pos[d] + (d == ND - 1 ? fb.l0 : 0);
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                const int s = c - 3 + k;
                at[d][k] = base + (long)(fb.wrap[d] ? bc_map(s, a.n[d], 1) : s - fb.lo[d]) * stride;
            }
        }
        T res[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            T div[3];
#pragma unroll
            for (int d = 0; d < ND; ++d) {
                const T *A = fb.buf + fb.off[d] + c * fb.n[d], *M = A + NC * fb.n[d];
                T dx[5];
#pragma unroll
                for (int k = 0; k < 5; ++k) {
                    const bool in = chk(at[d][k + 1], fb.n[d], kChkFaceRead, a.flags) &&
                                    chk(at[d][k], fb.n[d], kChkFaceRead, a.flags);
                    dx[k] = in ? A[at[d][k + 1]] - M[at[d][k]] : T(0);
                }
                div[d] = Divergence<T, VAR>::of(dx);
            }
            T L = -fma(div[0], idx[0], div[1] * idx[1]);
            if constexpr (ND == 3) L = fma(-div[2], idx[2], L);
            const long i = c * a.cstride + cell;
            const bool epi = a.mode != kModeRHS && chk(i, (long)NC * a.cstride, kChkEpiRead, a.flags);
            const T u0 = epi ? (a.u0_is_stencil ? a.U[i] : a.U0[i]) : T(0);
            const T din = (epi && a.Din) ? a.Din[i] : T(0);
            const T lov = (epi && a.lo && a.mode == kModeFinal) ? a.lo[i] : T(0);
            res[c] = stage_epilogue<T>(a, i, L, u0, din, lov, dt, (long)NC * a.cstride);
        }
        if (a.rate && a.mode == kModeFinal) {
            T r[3] = {T(0), T(0), T(0)};
            if constexpr (ND == 3) rates3d<T>(res, gamma, idx, r[0], r[1], r[2]);
            else rates2d<T>(res, gamma, idx, r[0], r[1]);
#pragma unroll
            for (int d = 0; d < ND; ++d) rm[d] = Num<T>::fmax(rm[d], r[d]);
        }
    }
    finish_block<T>(a, rm[0], rm[1], rm[2], true);
}

}  // namespace gpweno
