// Direct solve of L e = r on a box without solid cells, the correction of the
// pressure solve (Section 2) there and, with solid cells, the preconditioner of
// its conjugate gradients: L is a sum of three 1D operators whose
// eigenvectors are known (cosines on a Neumann axis, the real Fourier basis on
// a periodic one), so e is r transformed along x and y, a three-point equation
// along z per (kx, ky), and transformed back.  One application in FP32 leaves
// 1e-4 .. 5e-7 of the residual (its rounding times the conditioning of L), so
// one to three applications inside the float-float refinement (64^3: one or two,
// 256^3: two or three) reach what five BiCGStab iterations with two V-cycles each
// reach.
//
// Transforms (k_dir_xy).  Both bases split into vectors even and odd under
// j -> n-1-j, so a line folded into its sums and differences takes two
// products of half the length, and a plane four independent ones (quadrants:
// even / odd in y, even / odd in x).  One CTA holds a plane (or a block of its
// columns) in shared memory: fold (or read the quadrants), multiply by the x
// matrix, multiply by the y matrix, write the quadrants (or unfold).  The
// spectral plane keeps the even modes of an axis first, then the odd ones.
// Planes that do not fit go one axis at a time (k_dir_x, k_dir_y).
//
// Along z (k_dir_z).  With rho + 1/rho = 2 + h_z^2 (lam_x + lam_y), rho <= 1,
// the three-point operator is (1 - rho S)(1 - rho S^-1) / rho: a recursion up
// and one down the column, started from the values that the mirrored
// (Neumann) or wrapped (periodic) column gives.  A thread holds one chunk of a
// column in registers; the chunks' ends are combined through shared memory.
#pragma once

#include <cmath>
#include <vector>

#include "ns_mg_cluster.cuh"

namespace nsk {

constexpr int DIR_MAX_THREADS = 512;
constexpr size_t DIR_MAX_SMEM = 227 * 1024;
constexpr int DIR_ZC = 8;        // cells per chunk of a column
constexpr int DIR_ZC_LONG = 16;  // the same where nz needs more than 16 chunks
constexpr int DIR_ZX = 32;       // columns per CTA of k_dir_z

// DM_CORRECT: corrections in the grid's precision; DM_PRECOND: the preconditioner
// of the conjugate gradients below; DM_MIXED: FP32 corrections of an FP64
// grid's iterate and residual.
enum { DM_CORRECT = 0, DM_PRECOND = 1, DM_MIXED = 2 };

template <typename T>
struct DirPlan {
    int nx, ny, nz, per_z;
    int mode;      // DM_*: what the application is part of
    int hx, hy;    // even modes (= length of the folded line) along x, y
    int hxp;       // hx rounded up to 4
    int rb, ncol;  // rows and columns per thread of k_dir_xy
    int hyp;       // hy rounded up to rb
    int ldf;       // column stride of the folded plane in shared memory
    int cb, xb;    // columns per CTA (of a half), CTAs per plane
    int nt;        // threads of k_dir_xy
    int log2n;     // of the cells, rounded down
    int lines;     // > 0: one axis at a time, lines per block of k_dir_x / k_dir_y
    int ntx, nty;  // their threads
    int zm, zc;    // k_dir_z: cells per chunk, chunks per column
    long long cells;
    const T* rx[2];  // x matrices, forward and inverse: [parity][hxp][hxp]
    const T* ly[2];  // y matrices, forward and inverse: [parity][hyp][hyp]
    const T* col;    // per column [5][ny nx]: rho, c1, c2, rho^nz, -rho h_z^2
};

// Most threads of k_dir_z: 16 chunks of 8 cells, or 32 (FP64, whose registers
// hold half as many: 16) of 16.
template <typename T>
constexpr int dir_z_threads(int zm) {
    return DIR_ZX * (zm == DIR_ZC || sizeof(T) == 8 ? 16 : 32);
}

// Whether the state takes part in the current application: FP32+refine while
// its outer residual is above the target; otherwise while it iterates.
template <typename T> __device__ __forceinline__ bool dir_active(const SliceCtl* c, int mode) {
    if (sizeof(T) == 8 || mode != DM_CORRECT) return c->status == ST_ITER;
    return c->o_status == OS_REFINE && c->status != ST_NONFINITE;
}

// FP32 corrections live in a ring of DIR_RING buffers, one per application;
// the pressure is the warm start plus the applications not yet folded into it
// (the last three at most).  The residual is scaled by a power of two on its
// way into the transforms and e unscaled on its way out, so that neither
// underflows however far the refinement has come (a preconditioned residual
// carries its scale already; it and an FP64 grid's corrections have one buffer).
constexpr int DIR_RING = 4;
template <typename T>
__device__ __forceinline__ int dir_slot(const SliceCtl* c, int mode) {
    return sizeof(T) == 4 && mode == DM_CORRECT ? c->o_steps & (DIR_RING - 1) : 0;
}
// log2 of the scale that brings a residual of squared norm rr to an RMS of order
// one, from the exponents of rr and of the cells (no FP64 root or quotient: one
// thread computes it at the end of a kernel that everything waits for).  `top`
// keeps the scale itself in range.
__device__ __forceinline__ int dir_shift(double rr, int log2n, int top) {
    if (!(rr > 0.0) || !isfinite(rr)) return 0;
    const int e = (int)((__double_as_longlong(rr) >> 52) & 0x7ff) - 1023;
    return -max(-top, min(top, (e - log2n) / 2));
}
// The same for the FP64 residuals that FP32 corrections are made of: none where
// the residual is within 2^24 of one, FP32's range having room for that.
__device__ __forceinline__ int dir_shift64(double rr, int log2n) {
    const int e = dir_shift(rr, log2n, 500);
    return e >= -24 && e <= 24 ? 0 : e;
}
inline int dir_log2(long long n) {
    int l = 0;
    while (n >> (l + 1)) ++l;
    return l;
}
template <typename T>
__device__ __forceinline__ double dir_scale(const SliceCtl* c, bool inv, const DirPlan<T>& P) {
    if (sizeof(T) == 8 || P.mode == DM_PRECOND) return 1.0;
    // (an FP64 grid's e stays scaled: unscaled it may be out of FP32's range)
    if (P.mode == DM_MIXED) return inv ? 1.0 : ldexp(1.0, dir_shift64(c->rr, P.log2n));
    return inv ? 1.0f / c->o_fsc : c->o_fsc;
}

// acc[n][i] += sum_k L[k][i] R[k][n dc], i < RB, n < NC, k ascending; rows of L
// (16-byte aligned) are ldl apart, of R ldr.  Neighbouring threads hold
// neighbouring columns of R, so the reads of L are broadcasts and those of R
// without conflict: RB / 4 + NC shared-memory cycles per RB NC products of a
// warp (four per cycle and SM).
template <typename T, int RB, int NC>
__device__ __forceinline__ void dir_cols(const T* L, int ldl, const T* R, int ldr, int dc, int K,
                                         T (&acc)[NC][RB]) {
#pragma unroll 4
    for (int k = 0; k < K; ++k) {
        T r[NC];
#pragma unroll
        for (int n = 0; n < NC; ++n) r[n] = R[n * dc];
#pragma unroll
        for (int b = 0; b < RB / 4; ++b) {
            const Q4<T> l = q4_ld<T>(L + 4 * b);
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int n = 0; n < NC; ++n)
                    acc[n][4 * b + q] = fma(l.v[q], r[n], acc[n][4 * b + q]);
        }
        L += ldl;
        R += ldr;
    }
}

// An element of the source: FP64 values are scaled before they become FP32.
template <typename T, typename S>
__device__ __forceinline__ T dir_in(S v, double scale) {
    return sizeof(S) > sizeof(T) ? T(v * S(scale)) : T(v);
}

// Copies n elements (a multiple of 4, both sides 16-byte aligned) to shared
// memory.
template <typename T>
__device__ __forceinline__ void dir_copy(T* d, const T* __restrict__ g, int n, int t, int nt) {
    for (int q = 4 * t; q < n; q += 4 * nt) q4_st<T>(d + q, q4_ld<T>(g + q));
}

// Shared memory of k_dir_xy in elements: x matrices of the column block, y
// matrices, the folded plane (columns of rows), the product of the first stage.
template <typename T>
inline size_t dir_smem_elems(const DirPlan<T>& P) {
    return 2 * (size_t)P.hxp * P.cb + 2 * (size_t)P.hyp * P.hyp + 4 * (size_t)P.hxp * P.ldf +
           4 * (size_t)P.hyp * P.cb;
}

// Forward (INV false): src [nz][ny][nx] cells -> dst [nz][ky][kx].  Inverse:
// src [nz][ky][kx] -> dst cells (FP32: the application's slot of the ring,
// slots `ring` elements apart).  blockIdx.x = plane and column block,
// blockIdx.y = state.  Bound by instruction issue (FP64: by the FP64 pipe).
// 64^3 x 32 states, FP32: 57 us with 4 x 4 tiles of operands both read per
// thread -> 46 us.
template <typename T, bool INV, int RB, int NC, typename S = T>
__global__ void __launch_bounds__(DIR_MAX_THREADS)
    k_dir_xy(DirPlan<T> P, const SliceCtl* __restrict__ ctl, const S* __restrict__ src,
             T* __restrict__ dst, long long ring) {
    pdl_wait();
    const long long s = blockIdx.y;
    if (!dir_active<T>(ctl + s, P.mode)) return;
    const double dscale = dir_scale<T>(ctl + s, INV, P);
    const T scale = sizeof(S) > sizeof(T) ? T(1) : T(dscale);  // (else applied to S)
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int nx = P.nx, ny = P.ny, hx = P.hx, hy = P.hy, hxp = P.hxp, hyp = P.hyp;
    const int ldf = P.ldf, cb = P.cb;
    T* R = reinterpret_cast<T*>(smem_raw);
    T* Lm = R + 2 * hxp * cb;
    T* F = Lm + 2 * hyp * hyp;
    T* T1 = F + 4 * hxp * ldf;
    const int z = (int)blockIdx.x / P.xb;
    const int c0 = ((int)blockIdx.x - z * P.xb) * cb;
    const int t = (int)threadIdx.x, nt = (int)blockDim.x;
    const S* __restrict__ a = src + s * P.cells + (long long)z * nx * ny;
    T* __restrict__ o = dst + (INV ? dir_slot<T>(ctl + s, P.mode) * ring : 0) + s * P.cells +
                        (long long)z * nx * ny;
    // the plane: four rows of one column at a time (F[quadrant][column][row]);
    // rows and columns beyond the halves are zero
    for (int w = t; w < hxp * (hyp / 4); w += nt) {
        const int y0 = 4 * (w / hxp), j = w - (y0 / 4) * hxp;
        // (loads without conditions, so that they are issued together)
        const int jj = min(j, hx - 1), xm = INV ? hx + min(jj, nx - hx - 1) : nx - 1 - jj;
        Q4<T> q[4];  // (y, x) parity: ee, eo, oe, oo
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int y = min(y0 + r, hy - 1), ym = INV ? hy + min(y, ny - hy - 1) : ny - 1 - y;
            q[0].v[r] = dir_in<T>(a[y * nx + jj], dscale);
            q[1].v[r] = dir_in<T>(a[y * nx + xm], dscale);
            q[2].v[r] = dir_in<T>(a[ym * nx + jj], dscale);
            q[3].v[r] = dir_in<T>(a[ym * nx + xm], dscale);
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int y = y0 + r;
            const bool ye = y < hy, xe = j < hx;
            if (!INV) {
                // the middle of an odd extent: itself in the sum, zero in the
                // difference
                const bool xp = xm != jj, yp = ny - 1 - y != y;
                const T a00 = q[0].v[r], a01 = q[1].v[r], a10 = q[2].v[r], a11 = q[3].v[r];
                const T e0 = xp ? a00 + a01 : a00, o0 = xp ? a00 - a01 : T(0);
                const T e1 = xp ? a10 + a11 : a10, o1 = xp ? a10 - a11 : T(0);
                const bool in = ye && xe;
                q[0].v[r] = in ? scale * (yp ? e0 + e1 : e0) : T(0);
                q[1].v[r] = in ? scale * (yp ? o0 + o1 : o0) : T(0);
                q[2].v[r] = in && yp ? scale * (e0 - e1) : T(0);
                q[3].v[r] = in && yp ? scale * (o0 - o1) : T(0);
            } else {
                const bool yo = y < ny - hy, xo = j < nx - hx;
                if (!(ye && xe)) q[0].v[r] = T(0);
                if (!(ye && xo)) q[1].v[r] = T(0);
                if (!(yo && xe)) q[2].v[r] = T(0);
                if (!(yo && xo)) q[3].v[r] = T(0);
            }
        }
#pragma unroll
        for (int h = 0; h < 4; ++h) q4_st<T>(F + (h * hxp + j) * ldf + y0, q[h]);
    }
    // the matrices (the broadcast one by columns: the other direction's rows)
    const T* __restrict__ rx = P.rx[INV ? 1 : 0];
    dir_copy<T>(Lm, P.ly[INV ? 0 : 1], 2 * hyp * hyp, t, nt);
    if (cb == hxp) {
        dir_copy<T>(R, rx, 2 * hxp * hxp, t, nt);
    } else {
        const int cq = cb / 4;
        for (int q = t; q < 2 * hxp * cq; q += nt) {
            const int row = q / cq, c = 4 * (q - row * cq);
            Q4<T> v{{T(0), T(0), T(0), T(0)}};
            if (c0 + c < hxp) v = q4_ld<T>(rx + row * hxp + c0 + c);
            q4_st<T>(R + row * cb + c, v);
        }
    }
    __syncthreads();
    // A thread holds RB rows of NC columns (dc apart) of a quadrant: w = (row
    // block, quadrant, column).
    const int dc = cb / NC, cols = 4 * dc, items = cols * (hyp / RB);
    // along x: T1[q][row][c] = sum_j F[q][j][row] R[px][j][c]
    for (int w = t; w < items; w += nt) {
        const int rb = w / cols, fc = w - rb * cols, q = fc / dc, c = fc - q * dc;
        T acc[NC][RB] = {};
        dir_cols<T, RB, NC>(F + q * hxp * ldf + rb * RB, ldf, R + (q & 1) * hxp * cb + c, cb, dc,
                            hx, acc);
        T* d = T1 + (q * hyp + rb * RB) * cb + c;
#pragma unroll
        for (int i = 0; i < RB; ++i)
#pragma unroll
            for (int n = 0; n < NC; ++n) d[i * cb + n * dc] = acc[n][i];
    }
    __syncthreads();
    // along y: out[q][row][c] = sum_y Lm[py][y][row] T1[q][y][c]
    for (int w = t; w < items; w += nt) {
        const int rb = w / cols, fc = w - rb * cols, q = fc / dc, c = fc - q * dc;
        T acc[NC][RB] = {};
        dir_cols<T, RB, NC>(Lm + (q >> 1) * hyp * hyp + rb * RB, hyp, T1 + q * hyp * cb + c, cb,
                            dc, hy, acc);
        if (INV) {
            // (the folded plane is no longer read)
            T* d = F + (q * hyp + rb * RB) * cb + c;
#pragma unroll
            for (int i = 0; i < RB; ++i)
#pragma unroll
                for (int n = 0; n < NC; ++n) d[i * cb + n * dc] = acc[n][i];
        } else {
            const int cy = (q >> 1) ? ny - hy : hy, cx = (q & 1) ? nx - hx : hx;
            const int oy = (q >> 1) ? hy : 0, ox = (q & 1) ? hx : 0;
            T* d = o + (oy + rb * RB) * nx + ox + c0 + c;
#pragma unroll
            for (int i = 0; i < RB; ++i)
#pragma unroll
                for (int n = 0; n < NC; ++n)
                    if (rb * RB + i < cy && c0 + c + n * dc < cx) d[i * nx + n * dc] = acc[n][i];
        }
    }
    if (INV) {
        __syncthreads();
        const int cw = min(cb, hx - c0);  // columns of this block
        const int rpp = nt / cb, y0 = t / cb, j = t - y0 * cb;
        if (y0 < rpp && j < cw) {
            const int x = c0 + j, xm = nx - 1 - x;
            for (int y = y0; y < hy; y += rpp) {
                const int ym = ny - 1 - y;
                const T ee = scale * F[y * cb + j], eo = scale * F[(hyp + y) * cb + j];
                const T oe = scale * F[(2 * hyp + y) * cb + j];
                const T oo = scale * F[(3 * hyp + y) * cb + j];
                const T pe = ee + oe, po = eo + oo, me = ee - oe, mo = eo - oo;
                o[y * nx + x] = pe + po;
                if (xm != x) o[y * nx + xm] = pe - po;
                if (ym != y) {
                    o[ym * nx + x] = me + mo;
                    if (xm != x) o[ym * nx + xm] = me - mo;
                }
            }
        }
    }
}

// Planes too large for one CTA's shared memory: the same transforms one axis at
// a time, in persistent CTAs that keep the axis's matrices (both parities) in
// shared memory and run over blocks of P.lines lines.  A thread holds DIR_LRB
// rows of DIR_LNC columns in both parities, so folding and unfolding need no
// exchange.  256 x 256 planes, FP32: 128 products per value and axis, bound by
// the FP32 pipe and the shared-memory reads that feed it (4 of each per 16
// products): 483 to 518 us per axis for 67e6 cells, floor of the pipe alone 221 us
// (16 rows per thread, half the warps: 545 to 919 us).
constexpr int DIR_LRB = 8, DIR_LNC = 2;

template <typename T>
inline size_t dir_x_elems(const DirPlan<T>& P) {
    return 2 * (size_t)P.hxp * P.hxp + 2 * (size_t)P.hxp * (P.lines + 4);
}
template <typename T>
inline size_t dir_y_elems(const DirPlan<T>& P) {
    return 2 * (size_t)P.hyp * P.hyp + 2 * (size_t)P.hyp * P.lines;
}

template <typename T>
__device__ __forceinline__ bool dir_any_active(const SliceCtl* ctl, int batch, int mode) {
    for (int s = 0; s < batch; ++s)
        if (dir_active<T>(ctl + s, mode)) return true;
    return false;
}

// Along x: rows of src to rows of dst (INV: the application's slot of the
// ring), P.lines rows at a time.
template <typename T, bool INV, typename S = T>
__global__ void __launch_bounds__(DIR_MAX_THREADS)
    k_dir_x(DirPlan<T> P, const SliceCtl* __restrict__ ctl, const S* __restrict__ src,
            T* __restrict__ dst, long long ring, int batch) {
    pdl_wait();
    if (!dir_any_active<T>(ctl, batch, P.mode)) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int nx = P.nx, hx = P.hx, hxp = P.hxp, L = P.lines, ldf = L + 4;
    T* R = reinterpret_cast<T*>(smem_raw);
    T* F = R + 2 * hxp * hxp;  // [parity][column][row]
    const int t = (int)threadIdx.x, nt = (int)blockDim.x;
    dir_copy<T>(R, P.rx[INV ? 1 : 0], 2 * hxp * hxp, t, nt);
    const int rows = P.ny * P.nz, blocks = (rows + L - 1) / L, dc = hxp / DIR_LNC;
    for (long long it = blockIdx.x; it < (long long)blocks * batch; it += gridDim.x) {
        const int s = (int)(it / blocks), r0 = (int)(it - (long long)s * blocks) * L;
        if (!dir_active<T>(ctl + s, P.mode)) continue;
        const double dscale = dir_scale<T>(ctl + s, INV, P);
        const T scale = sizeof(S) > sizeof(T) ? T(1) : T(dscale);
        const S* __restrict__ a = src + s * P.cells + (long long)r0 * nx;
        T* __restrict__ o = dst + (INV ? dir_slot<T>(ctl + s, P.mode) * ring : 0) + s * P.cells +
                            (long long)r0 * nx;
        const int nr = min(L, rows - r0);
        __syncthreads();  // the previous block's lines are read
#pragma unroll 2
        for (int w = t; w < hxp * (L / 4); w += nt) {
            const int y0 = 4 * (w / hxp), j = w - (y0 / 4) * hxp;
            // (loads without conditions, so that they are issued together)
            const int jj = min(j, hx - 1), xm = INV ? hx + min(jj, nx - hx - 1) : nx - 1 - jj;
            Q4<T> e, d;
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const S* __restrict__ line = a + min(y0 + r, nr - 1) * nx;
                e.v[r] = dir_in<T>(line[jj], dscale);
                d.v[r] = dir_in<T>(line[xm], dscale);
            }
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const bool in = y0 + r < nr && j < hx;
                const T a0 = in ? e.v[r] : T(0);
                T a1 = in ? d.v[r] : T(0);
                if (!INV) {
                    // the middle of an odd extent: itself in the sum, zero in
                    // the difference
                    e.v[r] = scale * (xm != jj ? a0 + a1 : a0);
                    d.v[r] = xm != jj ? scale * (a0 - a1) : T(0);
                } else {
                    e.v[r] = a0;
                    d.v[r] = j < nx - hx ? a1 : T(0);
                }
            }
            q4_st<T>(F + j * ldf + y0, e);
            q4_st<T>(F + (hxp + j) * ldf + y0, d);
        }
        __syncthreads();
        for (int w = t; w < dc * (L / DIR_LRB); w += nt) {
            const int rb = w / dc, c = w - rb * dc;
            T e[DIR_LNC][DIR_LRB] = {}, d[DIR_LNC][DIR_LRB] = {};
            dir_cols<T, DIR_LRB, DIR_LNC>(F + rb * DIR_LRB, ldf, R + c, hxp, dc, hx, e);
            dir_cols<T, DIR_LRB, DIR_LNC>(F + hxp * ldf + rb * DIR_LRB, ldf, R + hxp * hxp + c,
                                          hxp, dc, hx, d);
#pragma unroll
            for (int i = 0; i < DIR_LRB; ++i) {
                const int row = rb * DIR_LRB + i;
                if (row >= nr) break;
                T* line = o + row * nx;
#pragma unroll
                for (int n = 0; n < DIR_LNC; ++n) {
                    const int x = c + n * dc, xm = nx - 1 - x;
                    if (x >= hx) continue;
                    if (!INV) {
                        line[x] = e[n][i];
                        if (x < nx - hx) line[hx + x] = d[n][i];
                    } else {
                        line[x] = scale * (e[n][i] + d[n][i]);
                        if (xm != x) line[xm] = scale * (e[n][i] - d[n][i]);
                    }
                }
            }
        }
    }
}

// Along y, in place: P.lines columns of a plane at a time.
template <typename T, bool INV>
__global__ void __launch_bounds__(DIR_MAX_THREADS)
    k_dir_y(DirPlan<T> P, const SliceCtl* __restrict__ ctl, T* __restrict__ spec, int batch) {
    pdl_wait();
    if (!dir_any_active<T>(ctl, batch, P.mode)) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int nx = P.nx, ny = P.ny, hy = P.hy, hyp = P.hyp, L = P.lines;
    T* Lm = reinterpret_cast<T*>(smem_raw);
    T* F = Lm + 2 * hyp * hyp;  // [parity][row][column]
    const int t = (int)threadIdx.x, nt = (int)blockDim.x;
    dir_copy<T>(Lm, P.ly[INV ? 0 : 1], 2 * hyp * hyp, t, nt);
    const int xb = (nx + L - 1) / L, blocks = xb * P.nz, dc = L / DIR_LNC;
    for (long long it = blockIdx.x; it < (long long)blocks * batch; it += gridDim.x) {
        const int s = (int)(it / blocks), r = (int)(it - (long long)s * blocks);
        if (!dir_active<T>(ctl + s, P.mode)) continue;
        const int z = r / xb, x0 = (r - z * xb) * L, nc = min(L, nx - x0);
        T* __restrict__ a = spec + s * P.cells + (long long)z * nx * ny + x0;
        __syncthreads();
#pragma unroll 8
        for (int q = t; q < hy * L; q += nt) {
            const int y = q / L, c = q - y * L;
            const int ym = INV ? hy + min(y, ny - hy - 1) : ny - 1 - y, cc = min(c, nc - 1);
            const T a0 = a[y * nx + cc], a1 = a[ym * nx + cc];
            const T e = INV ? a0 : (ym != y ? a0 + a1 : a0);
            const T d = INV ? (y < ny - hy ? a1 : T(0)) : (ym != y ? a0 - a1 : T(0));
            F[q] = e;
            F[hyp * L + q] = d;
        }
        __syncthreads();
        for (int w = t; w < dc * (hyp / DIR_LRB); w += nt) {
            const int rb = w / dc, c = w - rb * dc;
            T e[DIR_LNC][DIR_LRB] = {}, d[DIR_LNC][DIR_LRB] = {};
            dir_cols<T, DIR_LRB, DIR_LNC>(Lm + rb * DIR_LRB, hyp, F + c, L, dc, hy, e);
            dir_cols<T, DIR_LRB, DIR_LNC>(Lm + hyp * hyp + rb * DIR_LRB, hyp, F + hyp * L + c, L,
                                          dc, hy, d);
#pragma unroll
            for (int i = 0; i < DIR_LRB; ++i) {
                const int ky = rb * DIR_LRB + i, ym = ny - 1 - ky;
                if (ky >= hy) break;
#pragma unroll
                for (int n = 0; n < DIR_LNC; ++n) {
                    const int x = c + n * dc;
                    if (x >= nc) continue;
                    if (!INV) {
                        a[ky * nx + x] = e[n][i];
                        if (ky < ny - hy) a[(hy + ky) * nx + x] = d[n][i];
                    } else {
                        a[ky * nx + x] = e[n][i] + d[n][i];
                        if (ym != ky) a[ym * nx + x] = e[n][i] - d[n][i];
                    }
                }
            }
        }
    }
}

// The three-point equations along z of every column (kx, ky), in place.
// blockDim = (32 columns, chunks), blockIdx.y = state.  y' and x' below are
// the up and down recursions divided by rho: y'_k = r_k + rho y'_(k-1),
// x'_k = y'_k + rho x'_(k+1), e_k = -rho h_z^2 x'_k.
template <typename T, int ZM>
__global__ void __launch_bounds__(dir_z_threads<T>(ZM))
    k_dir_z(DirPlan<T> P, SliceCtl* __restrict__ ctl, T* __restrict__ a) {
    pdl_wait();
    const long long s = blockIdx.y;
    if (!dir_active<T>(ctl + s, P.mode)) return;
    __shared__ T sY[32][DIR_ZX], sL[32][DIR_ZX], sP[32][DIR_ZX], sX[32][DIR_ZX], sE[DIR_ZX];
    const int lane = (int)threadIdx.x, ch = (int)threadIdx.y, C = (int)blockDim.y;
    const int cols = P.nx * P.ny, nz = P.nz;
    const int q = (int)blockIdx.x * DIR_ZX + lane;
    const bool ok = q < cols;
    const int qc = ok ? q : 0;
    const T rho = P.col[qc], c1 = P.col[cols + qc], c2 = P.col[2 * cols + qc],
            rn = P.col[3 * cols + qc], sc = P.col[4 * cols + qc];
    const int k0 = ch * ZM, len = max(0, min(ZM, nz - k0));
    T* __restrict__ p = a + s * P.cells + (long long)k0 * cols + q;
    T f[ZM];
#pragma unroll
    for (int i = 0; i < ZM; ++i) f[i] = (ok && i < len) ? p[(long long)i * cols] : T(0);
    // the chunk's sums from below and from above, rho^len
    T up = T(0), dn = T(0), pw = T(1);
#pragma unroll
    for (int i = 0; i < ZM; ++i)
        if (i < len) {
            up = fma(rho, up, f[i]);
            pw *= rho;
        }
#pragma unroll
    for (int i = ZM - 1; i >= 0; --i) dn = fma(rho, dn, f[i]);
    sY[ch][lane] = up;
    sL[ch][lane] = dn;
    sP[ch][lane] = pw;
    __syncthreads();
    T carry = T(0), below = T(1), Y = T(0), Lt = T(0);
    for (int c = 0; c < C; ++c) {
        if (c == ch) carry = Y;
        if (c < ch) below *= sP[c][lane];
        Y = fma(sP[c][lane], Y, sY[c][lane]);
    }
    for (int c = C - 1; c >= 0; --c) Lt = fma(sP[c][lane], Lt, sL[c][lane]);
    // y'_(-1): of the mirrored column, or of the wrapped one (the constant
    // mode has c1 = 0: the sums of a mean-free column start from 0)
    const T first = P.per_z ? c1 * Y : c1 * fma(rn, Y, Lt);
    T prev = fma(below, first, carry);
    if (q == 0) {
        // the constant (kx, ky) mode: the column's mean is out of L's range;
        // without it the sums end at zero
        const T mean = Y / T(nz);
        prev -= mean * T(k0);
#pragma unroll
        for (int i = 0; i < ZM; ++i)
            if (i < len) f[i] -= mean;
    }
#pragma unroll
    for (int i = 0; i < ZM; ++i)
        if (i < len) {
            prev = fma(rho, prev, f[i]);
            f[i] = prev;
        }
    T xd = T(0);
#pragma unroll
    for (int i = ZM - 1; i >= 0; --i) xd = fma(rho, xd, f[i]);
    sX[ch][lane] = xd;
    if (k0 < nz && k0 + len == nz) sE[lane] = prev;
    __syncthreads();
    T xn = T(0);
    if (!P.per_z) {
        xn = c2 * sE[lane];
    } else {
        for (int c = C - 1; c >= 0; --c) xn = fma(sP[c][lane], xn, sX[c][lane]);
        if (q == 0) {
            // the constant mode of a periodic column: shift y' so that its sum
            // is zero (x' then returns to its start)
            const T shift = -xn / T(nz);
#pragma unroll
            for (int i = 0; i < ZM; ++i)
                if (i < len) f[i] += shift;
            xn = T(0);
            for (int c = C - 1; c > ch; --c)
                xn += sX[c][lane] + shift * T(max(0, min(ZM, nz - c * ZM)));
        } else {
            xn *= c2;
        }
    }
    if (!(P.per_z && q == 0))
        for (int c = C - 1; c > ch; --c) xn = fma(sP[c][lane], xn, sX[c][lane]);
#pragma unroll
    for (int i = ZM - 1; i >= 0; --i)
        if (i < len) {
            xn = fma(rho, xn, f[i]);
            if (ok) p[(long long)i * cols] = sc * xn;
        }
    if (blockIdx.x == 0 && lane == 0 && ch == 0) {
        // an application counts as an iteration (no other CTA reads these)
        if (sizeof(T) == 4 && P.mode == DM_CORRECT) {
            ctl[s].it_cur = 1;
            ctl[s].total_iters += 1;
        }
    }
}

// ---------------------------------------------------------------------------
// the FP32+refine step around the direct solve (boxes without solid cells):
// start of the solve, outer correction, velocity correction.  Everything per
// cell runs in FP32 and float-float: GB300's FP64 pipe is 1/64 of its FP32
// one, and a handful of conversions and FP64 sums per cell made each of these
// passes FP64-bound.
// ---------------------------------------------------------------------------

// Tiling: a CTA of 128 threads covers w x r columns (w the width of the x
// tiles, r = 128 / w rows) and lz cells along z, in batches of DIR_ZB whose
// loads are issued together.
struct DirTile {
    int w, r, bx, by, lz, ctas;
    int log2n;     // of the cells, rounded down
    double inv_n;  // 1 / cells
};
constexpr int DIR_ZB = 4;

__device__ __forceinline__ bool dir_origin(const DirTile& t, const int* n, int& i, int& j,
                                           int& k0) {
    const int cta = (int)blockIdx.x;
    const int q = cta / t.bx, tx = cta - q * t.bx;
    const int tz = q / t.by, ty = q - tz * t.by;
    const int th = tid_flat(), y = th / t.w, x = th - y * t.w;
    i = tx * t.w + x;
    j = ty * t.r + y;
    k0 = tz * t.lz;
    return y < t.r && i < n[0] && j < n[1];
}

// DIR_ZB cells of a column with their neighbours: c[1 + q] cell q, c[0] the
// one below the first, c[DIR_ZB + 1] the one above the last (cells beyond the
// tile repeat its last neighbour and are not used).
struct DirSlab {
    float c[DIR_ZB + 2], xl[DIR_ZB], xh[DIR_ZB], yl[DIR_ZB], yh[DIR_ZB];
};

__device__ __forceinline__ int dir_zwrap(const Lev& L, int k) {
    if (k < 0) return L.bc[2] == BC_PERIODIC ? L.n[2] - 1 : 0;
    if (k >= L.n[2]) return L.bc[2] == BC_PERIODIC ? 0 : L.n[2] - 1;
    return k;
}

__device__ __forceinline__ void dir_load(const Lev& L, const NbrXY& xy, int kb, int k1,
                                         const float* __restrict__ a, DirSlab& v) {
    const int plane = L.n[0] * L.n[1];
#pragma unroll
    for (int q = 0; q < DIR_ZB + 2; ++q)
        v.c[q] = a[dir_zwrap(L, min(kb + q - 1, k1)) * plane + xy.base];
#pragma unroll
    for (int q = 0; q < DIR_ZB; ++q) {
        const float* __restrict__ p = a + min(kb + q, k1 - 1) * plane + xy.base;
        v.xl[q] = p[xy.xl];
        v.xh[q] = p[xy.xh];
        v.yl[q] = p[xy.yl];
        v.yh[q] = p[xy.yh];
    }
}

__device__ __forceinline__ FF dir_lap_ff(const Lev& L, const DirSlab& v, int q) {
    const float eh[3] = {v.xh[q], v.yh[q], v.c[q + 2]};
    const float el[3] = {v.xl[q], v.yl[q], v.c[q]};
    return lap_ff6(L, eh, el, v.c[q + 1]);
}

// a b with a float, b float-float; both float-float.
__device__ __forceinline__ FF ff_mul_f(float a, FF b) {
    const float p = a * b.hi;
    return ff_norm(p, fmaf(a, b.hi, -p) + a * b.lo);
}
__device__ __forceinline__ FF ff_mul(FF a, FF b) {
    const float p = a.hi * b.hi;
    return ff_norm(p, fmaf(a.hi, b.hi, -p) + (a.hi * b.lo + a.lo * b.hi));
}

// The last CTA of the start or of an outer correction: target met, out of
// corrections, or on.
__device__ __forceinline__ void dir_decide(SliceCtl* c, double rr, double otol2, int log2n,
                                           int max_outer) {
    c->o_rr = rr;
    c->p_final = 0;
    c->o_fsc = ldexpf(1.0f, dir_shift(rr, log2n, 100));
    c->status = ST_IDLE;
    if (!isfinite(rr)) {
        c->o_status = OS_NONFINITE;
    } else if (rr <= otol2 * c->o_bb) {
        c->o_status = OS_DONE;
    } else if (c->o_steps >= max_outer) {
        c->o_status = OS_FAIL;
    } else {
        c->o_status = OS_REFINE;
        c->status = ST_ITER;
    }
}

// The pressure of the caller (FP64) as warm start and as last pressure.
__global__ void __launch_bounds__(NTHREADS)
    k_dir_load_p(long long n, const double* __restrict__ p, FFBuf f) {
    pdl_wait();
    const long long q = (long long)blockIdx.x * NTHREADS + tid_flat();
    if (q >= n) return;
    const FF v = ff_from_double(p[q]);
    f.w_hi[q] = v.hi;
    f.w_lo[q] = v.lo;
    f.q_hi[q] = v.hi;
    f.q_lo[q] = v.lo;
}

// Start of a step's solve: b = D F* / dt (WITH_U: of u + increment, the
// stored u differenced exactly), r = b - L w.  The mean of r (rounding, the
// fluxes of b cancel) is left in r and taken out by the next residual.
template <bool WITH_U>
__global__ void __launch_bounds__(NTHREADS)
    k_dir_start(Lev L, DirTile t, SliceCtl* __restrict__ ctl, const float* __restrict__ fu,
                const float* __restrict__ fv, const float* __restrict__ fw,
                const float* __restrict__ u, const float* __restrict__ v,
                const float* __restrict__ w, const float* __restrict__ w_hi,
                const float* __restrict__ w_lo, FFBuf f, FF inv_dt, FF ihx, FF ihy, FF ihz,
                long long cu, long long cv, long long cw, double* __restrict__ part,
                unsigned int* __restrict__ counter, double otol2, int max_outer) {
    pdl_wait();
    const long long s = blockIdx.y;
    SliceCtl* c = ctl + s;
    const long long off = s * L.cells;
    const int ex = L.n[0] + (L.bc[0] != BC_PERIODIC), ey = L.n[1] + (L.bc[1] != BC_PERIODIC);
    int i, j, k0;
    SqAcc arr, abb;
    float sb = 0.0f;
    FF sr{0.0f, 0.0f}, sw{0.0f, 0.0f};
    if (dir_origin(t, L.n, i, j, k0)) {
        const int k1 = min(k0 + t.lz, L.n[2]);
        const NbrXY xy = make_nbr_xy(L, i, j);
        const int plane = L.n[0] * L.n[1];
        const int ip = i + 1 == ex ? 0 : i + 1, jp = j + 1 == ey ? 0 : j + 1;
        // faces of the cell: u at (i, ip), v at (j, jp), w at (k, k + 1)
        const long long u0 = (long long)j * ex, v0 = (long long)j * L.n[0] + i,
                        v1 = (long long)jp * L.n[0] + i;
        const long long pu = (long long)L.n[1] * ex, pv = (long long)ey * L.n[0];
        const int ez = L.n[2] + (L.bc[2] != BC_PERIODIC);
        auto div3 = [&](const float* __restrict__ a, const float* __restrict__ b,
                        const float* __restrict__ d, int k, float (&q)[6]) {
            const int kp = k + 1 == ez ? 0 : k + 1;
            q[0] = a[s * cu + k * pu + u0 + ip];
            q[1] = a[s * cu + k * pu + u0 + i];
            q[2] = b[s * cv + k * pv + v1];
            q[3] = b[s * cv + k * pv + v0];
            q[4] = d[s * cw + (long long)kp * plane + xy.base];
            q[5] = d[s * cw + (long long)k * plane + xy.base];
        };
        for (int kb = k0; kb < k1; kb += DIR_ZB) {
            DirSlab wh, wl;
            float fa[DIR_ZB][6];
            dir_load(L, xy, kb, k1, w_hi + off, wh);
            dir_load(L, xy, kb, k1, w_lo + off, wl);
#pragma unroll
            for (int q = 0; q < DIR_ZB; ++q) div3(fu, fv, fw, min(kb + q, k1 - 1), fa[q]);
#pragma unroll
            for (int q = 0; q < DIR_ZB; ++q) {
                if (kb + q >= k1) break;
                // the increment's divergence in FP32 (its differences carry no
                // cancellation against u)
                float dv = (fa[q][0] - fa[q][1]) * ihx.hi;
                dv += (fa[q][2] - fa[q][3]) * ihy.hi;
                dv += (fa[q][4] - fa[q][5]) * ihz.hi;
                FF b;
                if (WITH_U) {
                    float ua[6];
                    div3(u, v, w, kb + q, ua);
                    FF d{dv, 0.0f};
                    const FF ih[3] = {ihx, ihy, ihz};
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        FF g;
                        two_sum(ua[2 * a], -ua[2 * a + 1], g.hi, g.lo);
                        d = ff_add(d, ff_mul(g, ih[a]));
                    }
                    b = ff_mul(d, inv_dt);
                } else {
                    b = ff_mul_f(dv, inv_dt);
                }
                const float ll = lap7<float>(L, wl.xh[q], wl.xl[q], wl.yh[q], wl.yl[q],
                                             wl.c[q + 2], wl.c[q], wl.c[q + 1]);
                const FF lp = ff_add_f(dir_lap_ff(L, wh, q), ll);
                const FF r = ff_add(b, ff_neg(lp));
                const long long id = off + (long long)(kb + q) * plane + xy.base;
                f.r_hi[id] = r.hi;
                f.r_lo[id] = r.lo;
                arr.add(r.hi);
                abb.add(b.hi);
                sb += b.hi;
                sr = ff_add(sr, r);
                sw = ff_add(sw, FF{wh.c[q + 1], wl.c[q + 1]});
            }
        }
    }
    float acc[5] = {arr.big, arr.small, abb.big, abb.small, sb};
    const FF ffs[2] = {sr, sw};
    double tot[7];
    if (partials_arrive_ff<5, 2>(acc, ffs, part + s * t.ctas * 7, counter + s, t.ctas, tot) &&
        tid_flat() == 0) {
        const double in = t.inv_n;
        const double rr = tot[0] + tot[1] * 0x1p-128, bb = tot[2] + tot[3] * 0x1p-128;
        const FF rm = ff_from_double(tot[5] * in);
        c->rmean_hi = rm.hi;
        c->rmean_lo = rm.lo;
        c->sx = tot[6];
        const FF mean = ff_from_double(tot[6] * in);
        c->mean_hi = mean.hi;
        c->mean_lo = mean.lo;
        c->o_steps = 0;
        c->o_bb = fmax(bb - tot[4] * tot[4] * in, 0.0);
        // a NaN stays one
        const double r0 = rr - tot[5] * tot[5] * in;
        dir_decide(c, r0 < 0.0 ? 0.0 : r0, otol2, t.log2n, max_outer);
    }
}

// Outer correction with the application e just made: r <- r - mean(r) - L e
// (L e in float-float), its norm, the decision.  p is not touched: the warm
// start `base` and the last applications together are the pressure (from the
// fourth application on the oldest one still apart is folded into base).
__global__ void __launch_bounds__(NTHREADS)
    k_dir_refine(Lev L, DirTile t, SliceCtl* __restrict__ ctl, const float* __restrict__ ring,
                 long long stride, float* __restrict__ base_hi, float* __restrict__ base_lo,
                 FFBuf f, double* __restrict__ part, unsigned int* __restrict__ counter,
                 double otol2, int max_outer) {
    pdl_wait();
    const long long s = blockIdx.y;
    SliceCtl* c = ctl + s;
    if (!dir_active<float>(c, DM_CORRECT)) return;
    const long long off = s * L.cells;
    const int step = c->o_steps;
    const float* __restrict__ e = ring + (step & (DIR_RING - 1)) * stride + off;
    const float* __restrict__ old = ring + ((step + 1) & (DIR_RING - 1)) * stride + off;
    const FF neg_rmean{-c->rmean_hi, -c->rmean_lo};
    int i, j, k0;
    SqAcc arr;
    FF sr{0.0f, 0.0f}, se{0.0f, 0.0f};
    if (dir_origin(t, L.n, i, j, k0)) {
        const int k1 = min(k0 + t.lz, L.n[2]);
        const NbrXY xy = make_nbr_xy(L, i, j);
        const int plane = L.n[0] * L.n[1];
        for (int kb = k0; kb < k1; kb += DIR_ZB) {
            DirSlab ev;
            FF ro[DIR_ZB];
            dir_load(L, xy, kb, k1, e, ev);
#pragma unroll
            for (int q = 0; q < DIR_ZB; ++q) {
                const long long id = off + (long long)min(kb + q, k1 - 1) * plane + xy.base;
                ro[q] = FF{f.r_hi[id], f.r_lo[id]};
            }
#pragma unroll
            for (int q = 0; q < DIR_ZB; ++q) {
                if (kb + q >= k1) break;
                const long long id = off + (long long)(kb + q) * plane + xy.base;
                const FF le = dir_lap_ff(L, ev, q);
                const FF r = ff_add(ff_add(ro[q], neg_rmean), ff_neg(le));
                f.r_hi[id] = r.hi;
                f.r_lo[id] = r.lo;
                arr.add(r.hi);
                sr = ff_add(sr, r);
                se = ff_add_f(se, ev.c[q + 1]);
                if (step >= DIR_RING - 1) {
                    const FF b = ff_add_f(FF{base_hi[id], base_lo[id]}, old[id - off]);
                    base_hi[id] = b.hi;
                    base_lo[id] = b.lo;
                }
            }
        }
    }
    float acc[2] = {arr.big, arr.small};
    const FF ffs[2] = {sr, se};
    double tot[4];
    if (partials_arrive_ff<2, 2>(acc, ffs, part + s * t.ctas * 4, counter + s, t.ctas, tot) &&
        tid_flat() == 0) {
        const double in = t.inv_n;
        const FF rm = ff_from_double(tot[2] * in);
        c->rmean_hi = rm.hi;
        c->rmean_lo = rm.lo;
        c->sx += tot[3];
        const FF mean = ff_from_double(c->sx * in);
        c->mean_hi = mean.hi;
        c->mean_lo = mean.lo;
        c->o_steps = step + 1;
        const double r0 = tot[0] + tot[1] * 0x1p-128 - tot[2] * tot[2] * in;
        dir_decide(c, r0 < 0.0 ? 0.0 : r0, otol2, t.log2n, max_outer);
    }
}

// Velocity correction u = u + (increment - dt G p) (INCR) or F* - dt G p, p =
// base + the applications still apart; p_out (may be null) = p - mean in FP64;
// with w_hi given the next warm start w = 2 (p - mean) - q (not in base's
// buffers, which neighbouring cells still read) and q = p - mean.
template <bool INCR>
__global__ void __launch_bounds__(NTHREADS)
    k_dir_correct(Lev L, DirTile t, const SliceCtl* __restrict__ ctl, const float* fu,
                  const float* fv, const float* fw, float* u, float* v, float* w, FFBuf f,
                  const float* base_hi, const float* base_lo, const float* __restrict__ ring,
                  long long stride, float* __restrict__ w_hi, float* __restrict__ w_lo,
                  double* __restrict__ p_out, float3 dt_ih, long long cu, long long cv,
                  long long cw) {
    pdl_wait();
    const long long s = blockIdx.y;
    const SliceCtl* c = ctl + s;
    const long long off = s * L.cells;
    const int step = c->o_steps, ne = min(step, DIR_RING - 1);
    const float* bh = base_hi + off;
    const float* bl = base_lo + off;
    // applications that do not exist are read from the base and dropped, so
    // that no load waits behind a condition
    auto app = [&](int n) -> const float* {
        return ne >= n ? ring + ((step - n) & (DIR_RING - 1)) * stride + off : bh;
    };
    const float* e0 = app(1);
    const float* e1 = app(2);
    const float* e2 = app(3);
    const FF neg_mean{-c->mean_hi, -c->mean_lo};
    const bool keep = w_hi != nullptr;
    int i, j, k0;
    if (!dir_origin(t, L.n, i, j, k0)) return;
    const int nx = L.n[0], ny = L.n[1], nz = L.n[2], plane = nx * ny;
    const int wx = L.bc[0] != BC_PERIODIC, wy = L.bc[1] != BC_PERIODIC, wz = L.bc[2] != BC_PERIODIC;
    const int k1 = min(k0 + t.lz, nz);
    const int base = j * nx + i;
    const int xl = i > 0 ? base - 1 : (wx ? base : base + nx - 1);
    const int yl = j > 0 ? base - nx : (wy ? base : base + (ny - 1) * nx);
    struct Raw {
        float h, l, a, b, c;
    };
    auto raw = [&](int q) -> Raw { return Raw{bh[q], bl[q], e0[q], e1[q], e2[q]}; };
    // p at a cell: the newest application is the smallest, so it is added last
    auto sum = [&](const Raw& v) -> FF {
        FF p{v.h, v.l};
        if (ne > 2) p = ff_add_f(p, v.c);
        if (ne > 1) p = ff_add_f(p, v.b);
        if (ne > 0) p = ff_add_f(p, v.a);
        return p;
    };
    FF pz = sum(raw((k0 > 0 ? k0 - 1 : (wz ? 0 : nz - 1)) * plane + base));
    const long long ru = s * cu + (long long)j * (nx + wx) + i, pu = (long long)ny * (nx + wx);
    const long long rv = s * cv + (long long)j * nx + i, pv = (long long)(ny + wy) * nx;
    const long long rw = s * cw + base;
    const bool ax = i > 0 || !wx, ay = j > 0 || !wy;
    constexpr int ZB = 2;
    for (int kb = k0; kb < k1; kb += ZB) {
        Raw rc[ZB], rx[ZB], ry[ZB];
        FF pc[ZB], px[ZB], py[ZB], qv[ZB];
        float fa[ZB][3], oa[ZB][3];
#pragma unroll
        for (int q = 0; q < ZB; ++q) {
            const int k = min(kb + q, k1 - 1);
            rc[q] = raw(k * plane + base);
            rx[q] = raw(k * plane + xl);
            ry[q] = raw(k * plane + yl);
            fa[q][0] = fu[ru + k * pu];
            fa[q][1] = fv[rv + k * pv];
            fa[q][2] = fw[rw + (long long)k * plane];
            if (INCR) {
                oa[q][0] = u[ru + k * pu];
                oa[q][1] = v[rv + k * pv];
                oa[q][2] = w[rw + (long long)k * plane];
            }
            if (keep) {
                const long long id = off + (long long)k * plane + base;
                qv[q] = FF{f.q_hi[id], f.q_lo[id]};
            }
        }
#pragma unroll
        for (int q = 0; q < ZB; ++q) {
            pc[q] = sum(rc[q]);
            px[q] = sum(rx[q]);
            py[q] = sum(ry[q]);
        }
#pragma unroll
        for (int q = 0; q < ZB; ++q) {
            const int k = kb + q;
            if (k >= k1) break;
            auto corr = [&](int d, FF lo, float dt_h) -> float {
                const float dgp = ((pc[q].hi - lo.hi) + (pc[q].lo - lo.lo)) * dt_h;
                return INCR ? oa[q][d] + (fa[q][d] - dgp) : fa[q][d] - dgp;
            };
            u[ru + k * pu] = ax ? corr(0, px[q], dt_ih.x) : 0.0f;
            v[rv + k * pv] = ay ? corr(1, py[q], dt_ih.y) : 0.0f;
            w[rw + (long long)k * plane] = (k > 0 || !wz) ? corr(2, pz, dt_ih.z) : 0.0f;
            // the high wall faces hold zero
            if (wx && i == nx - 1) u[ru + k * pu + 1] = 0.0f;
            if (wy && j == ny - 1) v[rv + k * pv + nx] = 0.0f;
            if (wz && k == nz - 1) w[rw + (long long)nz * plane] = 0.0f;
            const long long id = off + (long long)k * plane + base;
            const FF pg = ff_add(pc[q], neg_mean);
            if (p_out) p_out[id] = ff_to_double(pg);
            if (keep) {
                const FF wn = ff_add(FF{2.0f * pg.hi, 2.0f * pg.lo}, ff_neg(qv[q]));
                w_hi[id] = wn.hi;
                w_lo[id] = wn.lo;
                f.q_hi[id] = pg.hi;
                f.q_lo[id] = pg.lo;
            }
            pz = pc[q];
        }
    }
}
// FP64: x += e, r -= L e + mean(r), (r, r), sum x; the last CTA decides.  The
// mean of the residual, made by rounding, is out of every correction's reach
// (L has no range there): it is taken out of the next residual, or it would
// be the floor of a solve whose right side is itself close to rounding.
// E = float: the FP32 corrections of DM_MIXED, L e in float-float (48 bits of a
// correction's own size; FP32 pipe), both still in the scale that the transforms
// gave the residual (a power of two: exact).
template <typename E>
__device__ __forceinline__ double dir_lap64(const Lev& L, const Vals7<E>& v);
template <>
__device__ __forceinline__ double dir_lap64<double>(const Lev& L, const Vals7<double>& v) {
    return lap_vals<double>(L, v);
}
template <>
__device__ __forceinline__ double dir_lap64<float>(const Lev& L, const Vals7<float>& v) {
    return ff_to_double(lap_ff_vals(L, v));
}
template <typename E>
__global__ void __launch_bounds__(NTHREADS)
    k_dir_update(Lev L, MgBuf<double> mb, SliceCtl* __restrict__ ctl,
                 const E* __restrict__ evec, double* __restrict__ part, double tol2,
                 int maxit, int nfluid, int log2n) {
    pdl_wait();
    const long long s = blockIdx.y;
    SliceCtl* c = ctl + s;
    if (c->status != ST_ITER) return;
    const long long off = s * L.cells;
    const E* __restrict__ e = evec + off;
    double* __restrict__ x = mb.x + off;
    double* __restrict__ r = mb.r + off;
    int i, j, k0;
    lev_origin(L, blockIdx.x, i, j, k0);
    const double rmean = c->rmean;
    const double unscale = sizeof(E) == 4 ? ldexp(1.0, -dir_shift64(c->rr, log2n)) : 1.0;
    double rr = 0.0, sx = 0.0, sr = 0.0;
    if (i < L.n[0] && j < L.n[1]) {
        const int k1 = min(k0 + L.tz, L.n[2]);
        const NbrXY xy = make_nbr_xy(L, i, j);
        const int plane = L.n[0] * L.n[1];
        for (int kb = k0; kb < k1; kb += MG_ZB) {
            Vals7<E> ev[MG_ZB];
            double xo[MG_ZB], ro[MG_ZB];
#pragma unroll
            for (int q = 0; q < MG_ZB; ++q) {
                if (kb + q < k1) {
                    const Nbr nb = nbr_at(L, xy, kb + q);
                    ev[q] = load7<E>(nb, e);
                    xo[q] = x[nb.c];
                    ro[q] = r[nb.c];
                }
            }
#pragma unroll
            for (int q = 0; q < MG_ZB; ++q) {
                if (kb + q < k1) {
                    const int id = (kb + q) * plane + xy.base;
                    const double le = dir_lap64<E>(L, ev[q]);
                    const double xv = fma(double(ev[q].c), unscale, xo[q]);
                    const double rv = fma(-le, unscale, ro[q]) - rmean;
                    x[id] = xv;
                    r[id] = rv;
                    rr += rv * rv;
                    sx += xv;
                    sr += rv;
                }
            }
        }
    }
    double acc[3] = {rr, sx, sr};
    double tot[3];
    if (partials_and_arrive<3>(acc, part + s * L.ctas * 3, mb.counter + s, L.ctas, tot) &&
        tid_flat() == 0) {
        c->it_cur += 1;
        c->total_iters += 1;
        bicg_decide(c, tot[0], tot[0], tot[1], tol2, maxit);
        c->rmean = c->status == ST_ITER ? tot[2] / nfluid : 0.0;
    }
}

// ---------------------------------------------------------------------------
// solid cells: conjugate gradients preconditioned by the direct solve
// ---------------------------------------------------------------------------

// With solid cells L (minus it is symmetric and semidefinite) is the Neumann
// operator of the fluid cells; z = the fluid part of the box solution of r (zero
// in solid cells) preconditions it with a condition number that depends on the
// obstacles' shapes and not on the grid (an extension of a fluid field into a
// solid has at most a fixed multiple of its energy).  An iteration is one
// application and three passes, 56 B/cell next to the transforms.  128^3 x 8
// states, 8 boxes, two steps: 21.5 working iterations of 553 us a step (transforms
// 286, columns 49, the passes 218) and 8 launched for states that had converged,
// 85 us each: 31.4 ms; with BiCGStab, whose V-cycles know the solids on the finest
// level only, 47 ms.
//
// The direction survives the outer corrections, which replace r by the true
// residual: beta = -(z, q) / (p, q) makes the next one conjugate to the last and
// alpha = (r, p) / (p, q) whatever r is (a restart after each correction took 23
// iterations per solve).
//
// beta from the last iteration's q = L p.
template <typename T>
__global__ void __launch_bounds__(NTHREADS)
    k_cg_dot(Lev L, MgBuf<T> mb, const T* __restrict__ zvec, SliceCtl* __restrict__ ctl,
             double* __restrict__ part) {
    pdl_wait();
    const long long s = blockIdx.y;
    SliceCtl* c = ctl + s;
    if (c->status != ST_ITER) return;
    const bool first = c->it_cur == 0 && c->o_steps == 0;
    const T* __restrict__ q = mb.V[0] + s * L.cells;
    const T* __restrict__ z = zvec + s * L.cells;
    T acc[1] = {T(0)};
    int i, j, k0;
    lev_origin(L, blockIdx.x, i, j, k0);
    if (!first && i < L.n[0] && j < L.n[1]) {
        const int k1 = min(k0 + L.tz, L.n[2]), plane = L.n[0] * L.n[1];
        const int base = lindex(L, i, j, 0);
#pragma unroll 4
        for (int k = k0; k < k1; ++k) acc[0] += q[base + k * plane] * z[base + k * plane];
    }
    double tot[1];
    if (partials_arrive<T, 1>(acc, part + s * L.ctas, mb.counter + s, L.ctas, tot) &&
        tid_flat() == 0)
        c->beta = first ? 0.0 : -tot[0] / c->rho[1];
}

// p = z + beta p (zero in solid cells; into the other parity's buffer, the
// neighbours still read this one's), q = L p, alpha.
template <typename T>
__global__ void __launch_bounds__(NTHREADS)
    k_cg_lap(Lev L, MgBuf<T> mb, const T* __restrict__ zvec, SliceCtl* __restrict__ ctl,
             double* __restrict__ part) {
    pdl_wait();
    const long long s = blockIdx.y;
    SliceCtl* c = ctl + s;
    if (c->status != ST_ITER) return;
    const long long off = s * L.cells;
    const int par = (int)(c->total_iters & 1);
    const bool first = c->it_cur == 0 && c->o_steps == 0;
    const T beta = T(c->beta);
    const T* __restrict__ r = mb.r + off;
    const T* __restrict__ z = zvec + off;
    const T* __restrict__ po = mb.P[par ^ 1] + off;
    T* __restrict__ p = mb.P[par] + off;
    T* __restrict__ q = mb.V[0] + off;
    T acc[2] = {T(0), T(0)};
    int i, j, k0;
    lev_origin(L, blockIdx.x, i, j, k0);
    if (i < L.n[0] && j < L.n[1]) {
        const int k1 = min(k0 + L.tz, L.n[2]);
        const NbrXY xy = make_nbr_xy(L, i, j);
        constexpr int ZB = 2;
        for (int kb = k0; kb < k1; kb += ZB) {
            Vals7<T> zv[ZB], pv[ZB];
            T rv[ZB];
            int id[ZB];
            bool fl[ZB];
#pragma unroll
            for (int u = 0; u < ZB; ++u) {
                const Nbr nb = nbr_at(L, xy, min(kb + u, k1 - 1));
                id[u] = nb.c;
                fl[u] = lev_fluid(L, nb.c);
                zv[u] = load7<T>(nb, z);
                rv[u] = r[nb.c];
                // (the first iteration's buffer holds anything)
                pv[u] = first ? Vals7<T>{} : load7<T>(nb, po);
            }
#pragma unroll
            for (int u = 0; u < ZB; ++u) {
                if (kb + u >= k1) break;
                Vals7<T> v;
                v.c = fma(beta, pv[u].c, zv[u].c);
                v.xh = fma(beta, pv[u].xh, zv[u].xh);
                v.xl = fma(beta, pv[u].xl, zv[u].xl);
                v.yh = fma(beta, pv[u].yh, zv[u].yh);
                v.yl = fma(beta, pv[u].yl, zv[u].yl);
                v.zh = fma(beta, pv[u].zh, zv[u].zh);
                v.zl = fma(beta, pv[u].zl, zv[u].zl);
                // (a solid cell's neighbours are clamped to itself: q = 0)
                const T lq = lap_vals<T>(L, v);
                const T pc = fl[u] ? v.c : T(0);
                p[id[u]] = pc;
                q[id[u]] = lq;
                acc[0] += pc * lq;
                acc[1] += pc * rv[u];
            }
        }
    }
    double tot[2];
    if (partials_arrive<T, 2>(acc, part + s * L.ctas * 2, mb.counter + s, L.ctas, tot) &&
        tid_flat() == 0) {
        c->rho[1] = tot[0];
        c->alpha = tot[1] / tot[0];
    }
}

// x += alpha p (from zero in a solve's first iteration), r -= alpha q, (r, r),
// sum x, the decision.
template <typename T>
__global__ void __launch_bounds__(NTHREADS)
    k_cg_update(Lev L, MgBuf<T> mb, SliceCtl* __restrict__ ctl, double* __restrict__ part,
                double tol2, int maxit) {
    pdl_wait();
    const long long s = blockIdx.y;
    SliceCtl* c = ctl + s;
    if (c->status != ST_ITER) return;
    const long long off = s * L.cells;
    const bool first = c->it_cur == 0;
    const T alpha = T(c->alpha);
    const T* __restrict__ p = mb.P[c->total_iters & 1] + off;
    const T* __restrict__ q = mb.V[0] + off;
    T* __restrict__ x = mb.x + off;
    T* __restrict__ r = mb.r + off;
    T acc[2] = {T(0), T(0)};
    int i, j, k0;
    lev_origin(L, blockIdx.x, i, j, k0);
    if (i < L.n[0] && j < L.n[1]) {
        const int k1 = min(k0 + L.tz, L.n[2]), plane = L.n[0] * L.n[1];
        const int base = lindex(L, i, j, 0);
        for (int kb = k0; kb < k1; kb += MG_ZB) {
            T xo[MG_ZB], ro[MG_ZB], pv[MG_ZB], qv[MG_ZB];
#pragma unroll
            for (int u = 0; u < MG_ZB; ++u) {
                const int id = base + min(kb + u, k1 - 1) * plane;
                xo[u] = first ? T(0) : x[id];
                ro[u] = r[id];
                pv[u] = p[id];
                qv[u] = q[id];
            }
#pragma unroll
            for (int u = 0; u < MG_ZB; ++u) {
                if (kb + u >= k1) break;
                const int id = base + (kb + u) * plane;
                const T xv = fma(alpha, pv[u], xo[u]);
                const T rv = fma(-alpha, qv[u], ro[u]);
                x[id] = xv;
                r[id] = rv;
                acc[0] += rv * rv;
                acc[1] += xv;
            }
        }
    }
    double tot[2];
    if (partials_arrive<T, 2>(acc, part + s * L.ctas * 2, mb.counter + s, L.ctas, tot) &&
        tid_flat() == 0) {
        c->it_cur += 1;
        c->total_iters += 1;
        c->rr = tot[0];
        c->sx = tot[1];
        // (a breakdown, (p, q) = 0 with r != 0, ends as non-finite too)
        if (!isfinite(tot[0]) || !isfinite(c->alpha))
            c->status = ST_NONFINITE;
        else if (tot[0] <= fmax(tol2, c->tol2_in) * c->bb)
            c->status = ST_CONV;
        else if (c->it_cur >= maxit)
            c->status = ST_MAXIT;
    }
}

// ---------------------------------------------------------------------------
// host side: the plan and its tables
// ---------------------------------------------------------------------------

// Eigenvectors and eigenvalues (of minus the unscaled second difference) of
// one axis: even ones first; q[m * n + j] = value of vector m at cell j.
inline void dir_basis(int n, bool periodic, std::vector<double>& q, std::vector<double>& lam) {
    const double pi = 3.14159265358979323846;
    const int h = (n + 1) / 2, period = 4 * n;
    // every value is a cosine of a multiple of pi / (2 n)
    std::vector<double> cs(period);
    for (int m = 0; m < period; ++m) cs[m] = std::cos(pi * m / (2.0 * n));
    q.assign((size_t)n * n, 0.0);
    lam.assign(n, 0.0);
    for (int m = 0; m < n; ++m) {
        const bool even = m < h;
        const int i = even ? m : m - h;  // index within its parity
        double norm = std::sqrt(2.0 / n);
        bool sine = false;
        int w;  // of the mode, in pi / n
        if (!periodic) {
            w = even ? 2 * i : 2 * i + 1;
            if (w == 0) norm = std::sqrt(1.0 / n);
        } else {
            // cosines 0 .. h-1, sines 1 .. n/2 (the highest mode of an even n
            // is the sine pi (j + 1/2))
            const int k = even ? i : i + 1;
            w = 2 * k;
            sine = !even;
            if (k == 0 || 2 * k == n) norm = std::sqrt(1.0 / n);
        }
        const double sh = std::sin(0.5 * pi * w / n);
        lam[m] = 4.0 * sh * sh;
        for (int j = 0; j < n; ++j) {
            // w pi / n (j + 1/2), a sine as a cosine a quarter turn earlier
            const long long at = (long long)w * (2 * j + 1) + (sine ? 3 * n : 0);
            q[(size_t)m * n + j] = norm * cs[at % period];
        }
    }
}

// Stride of rows of w elements (a multiple of 4): an odd number of 16-byte
// units, so that eight threads' 16-byte stores hit different banks.
inline int dir_odd(int w) { return (w / 4) % 2 ? w : w + 4; }

// Sizes of the transforms one axis at a time; false where an axis's matrices
// do not fit.
template <typename T>
inline bool dir_line_sizes(DirPlan<T>& P) {
    P.rb = DIR_LRB;
    P.hyp = (P.hy + DIR_LRB - 1) / DIR_LRB * DIR_LRB;
    for (P.lines = 64; P.lines >= 32; P.lines /= 2)
        if (dir_x_elems(P) * sizeof(T) <= DIR_MAX_SMEM &&
            dir_y_elems(P) * sizeof(T) <= DIR_MAX_SMEM) {
            auto threads = [](int items) {
                const int nt = (items + 31) / 32 * 32;
                return nt > DIR_MAX_THREADS ? DIR_MAX_THREADS : nt;
            };
            P.ntx = threads(P.hxp / DIR_LNC * (P.lines / DIR_LRB));
            P.nty = threads(P.lines / DIR_LNC * (P.hyp / DIR_LRB));
            return true;
        }
    return false;
}

// Fills P's sizes for n cells; false where neither the plane nor an axis's
// matrices fit shared memory, or a column does not fit the chunks of one CTA.
template <typename T>
inline bool dir_sizes(const int n[3], bool per_z, int planes, DirPlan<T>& P) {
    P = DirPlan<T>{};
    P.nx = n[0];
    P.ny = n[1];
    P.nz = n[2];
    P.per_z = per_z ? 1 : 0;
    P.cells = (long long)n[0] * n[1] * n[2];
    P.log2n = dir_log2(P.cells);
    P.hx = (n[0] + 1) / 2;
    P.hy = (n[1] + 1) / 2;
    P.hxp = (P.hx + 3) / 4 * 4;
    // rows and columns per thread: shared-memory cycles of a block of 16 rows
    // (with the padded rows), (rows / 4 + columns) / columns; a call of about
    // one plane per SM prefers more threads.  FP32, us per transform with more
    // threads / fewer: 152 planes of 45 x 37 9.8 / 12.2, of 64 x 64 11.7 / 12.2, of
    // 96 x 64 14.5 / 15.5, of 96 x 96 20.9 / 18.3; 192 planes 10.9 / 12.2, 14.2 /
    // 14.2, 20.4 / 18.3, 31.1 / 28.7: past one plane per SM the large planes, which
    // hold most of the time, turn (planes below 64 x 64 do not; FP64 ones of 45 x 37
    // take 59 / 77 there)
    const bool few = planes < 176;
    P.ncol = few ? 1 : 2;
    P.rb = 4;
    for (int rb = 8; rb <= (few ? 8 : 16); rb *= 2) {
        auto cost = [&](int r) { return (P.hy + r - 1) / r * (r / 4 + P.ncol); };
        if (cost(rb) <= cost(P.rb)) P.rb = rb;
    }
    P.hyp = (P.hy + P.rb - 1) / P.rb * P.rb;
    P.ldf = dir_odd(P.hyp);
    P.zm = n[2] <= 16 * DIR_ZC ? DIR_ZC : DIR_ZC_LONG;
    P.zc = (n[2] + P.zm - 1) / P.zm;
    if (P.zc * DIR_ZX > dir_z_threads<T>(P.zm)) return false;
    // column blocks: as few as shared memory allows, two at least where the
    // planes of a call would leave SMs idle
    for (int xb = planes < 152 && P.hxp > 4 ? 2 : 1; xb <= P.hxp / 4; ++xb) {
        P.cb = (P.hxp / 4 + xb - 1) / xb * 4;
        P.xb = (P.hxp + P.cb - 1) / P.cb;
        if (dir_smem_elems(P) * sizeof(T) <= DIR_MAX_SMEM) {
            const int items = 4 * (P.cb / P.ncol) * (P.hyp / P.rb);
            P.nt = (items + 31) / 32 * 32;
            P.nt = P.nt < 64 ? 64 : P.nt;
            P.nt = P.nt < P.cb ? (P.cb + 31) / 32 * 32 : P.nt;
            P.nt = P.nt > DIR_MAX_THREADS ? DIR_MAX_THREADS : P.nt;
            if (P.nt >= P.cb) return true;
        }
    }
    return dir_line_sizes<T>(P);
}

// The tables of a plan: x matrices (forward, inverse), y matrices (forward,
// inverse), columns; offsets in elements to off[5].
template <typename T>
inline std::vector<T> dir_tables(const DirPlan<T>& P, const int bc[3], const double ih2[3],
                                 size_t off[5]) {
    std::vector<double> qx, lx, qy, ly;
    dir_basis(P.nx, bc[0] == BC_PERIODIC, qx, lx);
    dir_basis(P.ny, bc[1] == BC_PERIODIC, qy, ly);
    const size_t mx = 2 * (size_t)P.hxp * P.hxp, my = 2 * (size_t)P.hyp * P.hyp;
    const size_t cols = (size_t)P.nx * P.ny;
    off[0] = 0;
    off[1] = mx;
    off[2] = 2 * mx;
    off[3] = 2 * mx + my;
    off[4] = 2 * mx + 2 * my;
    std::vector<T> v(off[4] + 5 * cols, T(0));
    for (int p = 0; p < 2; ++p) {
        const int nm = p ? P.nx - P.hx : P.hx;
        for (int m = 0; m < nm; ++m)
            for (int j = 0; j < P.hx; ++j) {
                // the middle of an odd extent is not folded: its odd values are 0
                const T x = (p && 2 * j + 1 == P.nx) ? T(0) : (T)qx[(size_t)(p * P.hx + m) * P.nx + j];
                v[off[0] + ((size_t)p * P.hxp + j) * P.hxp + m] = x;  // rows j, columns m
                v[off[1] + ((size_t)p * P.hxp + m) * P.hxp + j] = x;  // rows m, columns j
            }
        const int nmy = p ? P.ny - P.hy : P.hy;
        for (int m = 0; m < nmy; ++m)
            for (int j = 0; j < P.hy; ++j) {
                const T y = (p && 2 * j + 1 == P.ny) ? T(0) : (T)qy[(size_t)(p * P.hy + m) * P.ny + j];
                v[off[2] + ((size_t)p * P.hyp + m) * P.hyp + j] = y;  // rows m, columns j
                v[off[3] + ((size_t)p * P.hyp + j) * P.hyp + m] = y;  // rows j, columns m
            }
    }
    T* c = v.data() + off[4];
    for (int ky = 0; ky < P.ny; ++ky)
        for (int kx = 0; kx < P.nx; ++kx) {
            const size_t q = (size_t)ky * P.nx + kx;
            const double sig = (lx[kx] * ih2[0] + ly[ky] * ih2[1]) / ih2[2];
            const double rho = 1.0 / (1.0 + 0.5 * sig + std::sqrt(sig + 0.25 * sig * sig));
            double rn = 1.0, base = rho;
            for (int e = P.nz; e > 0; e >>= 1, base *= base)
                if (e & 1) rn *= base;
            double c1 = 0.0, c2 = 0.0;
            if (q != 0) {
                c1 = 1.0 / (P.per_z ? 1.0 - rn : 1.0 - rn * rn);
                c2 = P.per_z ? c1 : 1.0 / (1.0 - rho);
            }
            c[q] = (T)rho;
            c[cols + q] = (T)c1;
            c[2 * cols + q] = (T)c2;
            c[3 * cols + q] = (T)rn;
            c[4 * cols + q] = (T)(-rho / ih2[2]);
        }
    return v;
}

// Tiling of the step kernels: x tiles of about 32 columns; along z (where tile_z
// does not give it) the longest march of 64 cells or less that leaves the SMs
// eight CTAs deep, 4 below that.  A CTA's sums end in FP64, which a longer march
// pays less often: 64^3 x 32 states, 8 -> 32 cells: start 137 -> 115 us,
// correction of r 73 -> 66, of u 143 -> 136; with a warp per sum in the last CTA
// and the loads before any condition 109, 60 and 120.  The capacity decides, so
// grids of different capacity add a state's partials in different orders.
inline DirTile dir_tile_of(const int n[3], int cap, int tile_z) {
    DirTile t;
    const int xt = (n[0] + 31) / 32;
    t.w = (n[0] + xt - 1) / xt;
    t.r = NTHREADS / t.w;
    t.bx = (n[0] + t.w - 1) / t.w;
    t.by = (n[1] + t.r - 1) / t.r;
    t.lz = 4;
    for (int lz = 64; lz >= 8 && t.lz == 4; lz /= 2)
        if (lz <= n[2] && (long long)t.bx * t.by * ((n[2] + lz - 1) / lz) * cap >= 152 * 8)
            t.lz = lz;
    if (tile_z > 0) t.lz = tile_z < n[2] ? tile_z : n[2];
    t.ctas = t.bx * t.by * ((n[2] + t.lz - 1) / t.lz);
    t.inv_n = 1.0 / ((double)n[0] * n[1] * n[2]);
    t.log2n = dir_log2((long long)n[0] * n[1] * n[2]);
    return t;
}

// Condition number of L on its range (its largest over its smallest nonzero
// eigenvalue).
inline double dir_condition(const int n[3], const int bc[3], const double ih2[3]) {
    const double pi = 3.14159265358979323846;
    double top = 0.0, low = 0.0;
    for (int d = 0; d < 3; ++d) {
        const double s = std::sin(bc[d] == BC_PERIODIC ? pi / n[d] : 0.5 * pi / n[d]);
        const double l = 4.0 * s * s * ih2[d];
        top += 4.0 * ih2[d];
        low = (d == 0 || l < low) ? l : low;
    }
    return top / low;
}

}  // namespace nsk
