// 2D stage kernel of small FP32 grids: one CTA per tile of TX x TY cells.
//
// On a grid that gives the strip-marching kernel fewer than two CTAs per SM its time is a chain: a CTA of
// eight rows passes thirteen row iterations one after the other, with most of the chip idle.  Here a CTA
// stages its tile with ghosts once, evaluates all of its x- and y-faces as one list (full warps, every
// thread a face), and then updates its cells: two or three faces deep instead of twenty-one.  The price is
// the five extra faces per tile row and column, (TX+5)/TX and (TY+5)/TY of the work, which is
// why larger grids march.  choose_tile (dispatch.cuh) sizes the tiles for the SM count.
// Measured on GB300 per step, R = 2 (marching -> tiles, equal bits): 256^2 51 -> 25 us, 384^2 67 -> 39,
// 480^2 69 -> 53, 1000 x 200 68 -> 48; 64^2 45 -> 12 us (the launches).  At 2048^2 tiles lose:
// 753 us against 585.
#pragma once
#include "plan.h"
#include "stage.cuh"

namespace gpweno {

// float4 elements of shared memory: the staged tile, then A and M of the x- and y-faces
template <int R>
constexpr __host__ __device__ size_t tile2d_elems(int TX, int TY)
{
    constexpr int G = R + 3;
    return (size_t)(TX + 2 * G) * (TY + 2 * G) + 2 * ((size_t)(TX + 5) * TY + (size_t)TX * (TY + 5));
}

template <int R, int NT, int VAR>
__global__ void __launch_bounds__(NT, NT == 384 ? 1 : kResident<float, R, VAR> / NT)
    tile2d_kernel(StageArgs<float> a, Tile2D t, TablesFor<float, R, VAR> tb)
{
    constexpr int G = R + 3, NS = 2 * R + 2, NC = 4;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int tid = threadIdx.x;
    const int nx = a.n[0], ny = a.n[1];
    const long plane = a.cstride;
    const int tile_y = blockIdx.x / t.nx;
    const int x0 = (blockIdx.x - tile_y * t.nx) * t.TX, y0 = tile_y * t.TY;
    const int Wc = min(t.TX, nx - x0), Hc = min(t.TY, ny - y0);
    const int cols = Wc + 2 * G, rows = Hc + 2 * G;
    const int nfx = (Wc + 5) * Hc, nf = nfx + Wc * (Hc + 5);
    float4 *raw = reinterpret_cast<float4 *>(smem_raw);   // [rows][cols]
    float4 *FA = raw + rows * cols;                       // [x-faces, row by row][y-faces, row by row]
    float4 *FM = FA + nf;
    [[maybe_unused]] const long elems = (long)tile2d_elems<R>(t.TX, t.TY);   // checked build

    pdl_enter();
    const float dt = a.dt_dev ? (float)(*a.dt_dev) : (float)a.dt;
    for (int r = tid / 32; r < rows; r += NT / 32) {
        const int gy = y0 - G + r;
        long cs = plane;
        const float *src = (VAR & kVarSlab) != 0 && a.slab_dim == 1 ? layer_src<float>(a, a.U, gy, ny, a.per[1], nx, G, cs)
                                                                    : a.U + (long)bc_map(gy, ny, a.per[1]) * nx;
        for (int c = tid & 31; c < cols; c += 32) {
            const int gx = bc_map(x0 - G + c, nx, a.per[0]);
            float *dst = reinterpret_cast<float *>(raw + r * cols + c);
#pragma unroll
            for (int k = 0; k < NC; ++k)
                if (chk(r * cols + c, elems, kChkRingWrite, a.flags) &&
                    src_ok<float>(a, src + k * cs + gx, (long)NC * plane, (long)NC * G * nx, kChkStateRead))
                    cp_async_elem(dst + k, src + k * cs + gx);
        }
    }
    cp_async_commit();
    cp_async_wait_all();
    __syncthreads();

    Physical<float> ph;
    for (int f = tid; f < nf; f += NT) {
        // cell s of the face in the staged tile: x-face i of row j lies between columns G-3+i and G-2+i of
        // row G+j, y-face j of column i between rows G-3+j and G-2+j of column G+i
        const bool yface = f >= nfx;
        const int w = yface ? Wc : Wc + 5, g = yface ? f - nfx : f;
        const int j = g / w, i = g - j * w;
        const int step = yface ? cols : 1;
        const int first = (yface ? (j + G - 3) * cols + i + G : (j + G) * cols + i + G - 3) - R * step;
        float st[NS][NC];
#pragma unroll
        for (int q = 0; q < NS; ++q) {
            const bool in = chk(first + q * step, (long)rows * cols, kChkRingRead, a.flags);
            const float4 v = in ? raw[first + q * step] : make_float4(1.f, 0.f, 0.f, 1.f);
            st[q][0] = v.x;   // normal-first
            st[q][1] = yface ? v.z : v.y;
            st[q][2] = yface ? v.y : v.z;
            st[q][3] = v.w;
        }
        float A[NC], M[NC];
        face_eval<float, NC, R, VAR>(st, tb, A, M, ph);
        if (chk(rows * cols + nf + f, elems, kChkFaceWrite, a.flags)) {
            FA[f] = make_float4(A[0], yface ? A[2] : A[1], yface ? A[1] : A[2], A[3]);
            FM[f] = make_float4(M[0], yface ? M[2] : M[1], yface ? M[1] : M[2], M[3]);
        }
    }
    __syncthreads();

    const float idx[3] = {a.idx[0], a.idx[1], a.idx[2]};
    float rmx = 0.f, rmy = 0.f;
    for (int g = tid; g < Wc * Hc; g += NT) {
        const int j = g / Wc, i = g - j * Wc;
        const long cell = (long)(y0 + j) * nx + x0 + i;
        float u0[NC], din[NC], lov[NC];
        const bool epi = a.mode != kModeRHS;
        const float4 u = raw[(j + G) * cols + i + G];
        const float us[NC] = {u.x, u.y, u.z, u.w};
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const bool in = epi && chk(c * plane + cell, (long)NC * plane, kChkEpiRead, a.flags);
            u0[c] = a.u0_is_stencil ? us[c] : (in ? a.U0[c * plane + cell] : 0.f);
            din[c] = (in && a.Din) ? a.Din[c * plane + cell] : 0.f;
            lov[c] = (in && a.lo && a.mode == kModeFinal) ? a.lo[c * plane + cell] : 0.f;
        }
        // the flux jumps across the five cells around this one in each direction
        float dx[NC][5], dy[NC][5];
        const int fx = j * (Wc + 5) + i, fy = nfx + j * Wc + i;
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            const bool in = chk(fx + k + 1, nf, kChkFaceRead, a.flags) && chk(fy + (k + 1) * Wc, nf, kChkFaceRead, a.flags);
            const float4 p = in ? FA[fx + k + 1] : u, m = in ? FM[fx + k] : u;
            const float4 q = in ? FA[fy + (k + 1) * Wc] : u, n = in ? FM[fy + k * Wc] : u;
            dx[0][k] = p.x - m.x;
            dx[1][k] = p.y - m.y;
            dx[2][k] = p.z - m.z;
            dx[3][k] = p.w - m.w;
            dy[0][k] = q.x - n.x;
            dy[1][k] = q.y - n.y;
            dy[2][k] = q.z - n.z;
            dy[3][k] = q.w - n.w;
        }
        float res[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            using Dv = Divergence<float, VAR>;
            const float L = -fma(Dv::of(dx[c]), idx[0], Dv::of(dy[c]) * idx[1]);
            res[c] = stage_epilogue<float>(a, c * plane + cell, L, u0[c], din[c], lov[c], dt, (long)NC * plane);
        }
        if (a.rate && a.mode == kModeFinal) {
            float rx, ry;
            rates2d<float>(res, tb.gamma, idx, rx, ry);
            rmx = fmaxf(rmx, rx);
            rmy = fmaxf(rmy, ry);
        }
    }
    finish_block<float>(a, rmx, rmy, 0.f, ph.good());
}

}  // namespace gpweno
