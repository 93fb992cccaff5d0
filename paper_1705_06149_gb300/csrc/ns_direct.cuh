// Direct solve of L e = r on a box without solid cells, the correction of the
// pressure solve (Section 2) there: L is a sum of three 1D operators whose
// eigenvectors are known (cosines on a Neumann axis, the real Fourier basis on
// a periodic one), so e is r transformed along x and y, a three-point equation
// along z per (kx, ky), and transformed back.  One application in FP32 leaves
// 1e-4 .. 5e-7 of the residual (its rounding times the conditioning of L), so
// two applications inside the float-float refinement reach what five BiCGStab
// iterations with two V-cycles each reach.
//
// Transforms (k_dir_xy).  Both bases split into vectors even and odd under
// j -> n-1-j, so a line folded into its sums and differences takes two
// products of half the length, and a plane four independent ones (quadrants:
// even / odd in y, even / odd in x).  One CTA holds a plane (or a block of its
// columns) in shared memory: fold (or read the quadrants), multiply by the x
// matrix, multiply by the y matrix, write the quadrants (or unfold).  The
// spectral plane keeps the even modes of an axis first, then the odd ones.
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

template <typename T>
struct DirPlan {
    int nx, ny, nz, per_z;
    int hx, hy;    // even modes (= length of the folded line) along x, y
    int hxp, hyp;  // the same rounded up to 4
    int ldx, ldy;  // shared-memory row strides of the folded plane / the y matrix
    int cb, xb;    // columns per CTA (of a half), CTAs per plane
    int nt;        // threads of k_dir_xy
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
// its outer residual is above the target, FP64 while it iterates.
template <typename T> __device__ __forceinline__ bool dir_active(const SliceCtl* c);
template <> __device__ __forceinline__ bool dir_active<float>(const SliceCtl* c) {
    return c->o_status == OS_REFINE && c->status != ST_NONFINITE;
}
template <> __device__ __forceinline__ bool dir_active<double>(const SliceCtl* c) {
    return c->status == ST_ITER;
}

// acc[i][j] += sum_k L[i rs][k] R[k][j], i, j < 4, k ascending (K a multiple
// of 4; rows of L are rs apart so that neighbouring threads read
// neighbouring rows).
template <typename T>
__device__ __forceinline__ void dir_tile(const T* L, int rs, const T* R, int ldr, int K,
                                         T (&acc)[4][4]) {
    for (int k = 0; k < K; k += 4) {
        Q4<T> l[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) l[i] = q4_ld<T>(L + i * rs + k);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
            const Q4<T> r = q4_ld<T>(R + (k + kk) * ldr);
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fma(l[i].v[kk], r.v[j], acc[i][j]);
        }
    }
}

// Shared memory of k_dir_xy in elements: x matrices of the column block, y
// matrices, the folded plane, the product of the first stage.
template <typename T>
inline size_t dir_smem_elems(const DirPlan<T>& P) {
    return 2 * (size_t)P.hxp * P.cb + 2 * (size_t)P.hyp * P.ldy + 4 * (size_t)P.hyp * P.ldx +
           4 * (size_t)P.hyp * P.cb;
}

// Forward (INV false): src [nz][ny][nx] cells -> dst [nz][ky][kx].  Inverse:
// src [nz][ky][kx] -> dst cells.  blockIdx.x = plane and column block,
// blockIdx.y = state.
template <typename T, bool INV>
__global__ void __launch_bounds__(DIR_MAX_THREADS)
    k_dir_xy(DirPlan<T> P, const SliceCtl* __restrict__ ctl, const T* __restrict__ src,
             T* __restrict__ dst) {
    pdl_wait();
    const long long s = blockIdx.y;
    if (!dir_active<T>(ctl + s)) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int nx = P.nx, ny = P.ny, hx = P.hx, hy = P.hy, hxp = P.hxp, hyp = P.hyp;
    const int ldx = P.ldx, ldy = P.ldy, cb = P.cb;
    T* R = reinterpret_cast<T*>(smem_raw);
    T* Lm = R + 2 * hxp * cb;
    T* F = Lm + 2 * hyp * ldy;
    T* T1 = F + 4 * hyp * ldx;
    const int z = (int)blockIdx.x / P.xb;
    const int c0 = ((int)blockIdx.x - z * P.xb) * cb;
    const int t = (int)threadIdx.x, nt = (int)blockDim.x;
    const T* __restrict__ a = src + s * P.cells + (long long)z * nx * ny;
    T* __restrict__ o = dst + s * P.cells + (long long)z * nx * ny;
    {
        // the plane: thread (row, column j) of a pass; rows and columns beyond
        // the halves are zero
        const int rpp = nt / hxp, y0 = t / hxp, j = t - y0 * hxp;
        if (y0 < rpp) {
#pragma unroll 4
            for (int y = y0; y < hyp; y += rpp) {
                T q[4] = {T(0), T(0), T(0), T(0)};  // (y, x) parity: ee, eo, oe, oo
                if (!INV) {
                    if (y < hy && j < hx) {
                        const int ym = ny - 1 - y, xm = nx - 1 - j;
                        const T a00 = a[y * nx + j];
                        const T a01 = xm != j ? a[y * nx + xm] : T(0);
                        const T a10 = ym != y ? a[ym * nx + j] : T(0);
                        const T a11 = (xm != j && ym != y) ? a[ym * nx + xm] : T(0);
                        // the middle of an odd extent: itself in the sum, zero
                        // in the difference
                        const T e0 = a00 + a01, o0 = xm != j ? a00 - a01 : T(0);
                        const T e1 = a10 + a11, o1 = xm != j ? a10 - a11 : T(0);
                        q[0] = e0 + e1;
                        q[1] = o0 + o1;
                        q[2] = ym != y ? e0 - e1 : T(0);
                        q[3] = ym != y ? o0 - o1 : T(0);
                    }
                } else {
                    const bool ye = y < hy, yo = y < ny - hy, xe = j < hx, xo = j < nx - hx;
                    if (ye && xe) q[0] = a[y * nx + j];
                    if (ye && xo) q[1] = a[y * nx + hx + j];
                    if (yo && xe) q[2] = a[(hy + y) * nx + j];
                    if (yo && xo) q[3] = a[(hy + y) * nx + hx + j];
                }
#pragma unroll
                for (int h = 0; h < 4; ++h) F[(h * hyp + y) * ldx + j] = q[h];
            }
        }
        // the matrices
        const T* __restrict__ rx = P.rx[INV ? 1 : 0];
        const T* __restrict__ ly = P.ly[INV ? 1 : 0];
        const int cq = cb / 4, yq = hyp / 4;
        for (int q = t; q < 2 * hxp * cq; q += nt) {
            const int row = q / cq, c = 4 * (q - row * cq);
            Q4<T> v{{T(0), T(0), T(0), T(0)}};
            if (c0 + c < hxp) v = q4_ld<T>(rx + row * hxp + c0 + c);
            q4_st<T>(R + row * cb + c, v);
        }
        for (int q = t; q < 2 * hyp * yq; q += nt) {
            const int row = q / yq, c = 4 * (q - row * yq);
            q4_st<T>(Lm + row * ldy + c, q4_ld<T>(ly + row * hyp + c));
        }
    }
    __syncthreads();
    const int nty = hyp / 4, ntx = cb / 4, tiles = 4 * nty * ntx;
    // along x: T1[q][row][c] = sum_j F[q][row][j] R[px][j][c]
    for (int w = t; w < tiles; w += nt) {
        const int r = w / nty, mr = w - r * nty, q = r / ntx, nc = r - q * ntx;
        T acc[4][4] = {};
        dir_tile<T>(F + (q * hyp + mr) * ldx, nty * ldx, R + (q & 1) * hxp * cb + 4 * nc, cb, hxp,
                    acc);
#pragma unroll
        for (int i = 0; i < 4; ++i)
            q4_st<T>(T1 + (q * hyp + mr + i * nty) * cb + 4 * nc,
                     Q4<T>{{acc[i][0], acc[i][1], acc[i][2], acc[i][3]}});
    }
    __syncthreads();
    // along y: out[q][row][c] = sum_y Lm[py][row][y] T1[q][y][c]
    for (int w = t; w < tiles; w += nt) {
        const int r = w / nty, mr = w - r * nty, q = r / ntx, nc = r - q * ntx;
        T acc[4][4] = {};
        dir_tile<T>(Lm + ((q >> 1) * hyp + mr) * ldy, nty * ldy, T1 + q * hyp * cb + 4 * nc, cb,
                    hyp, acc);
        if (INV) {
            // (the folded plane is no longer read)
#pragma unroll
            for (int i = 0; i < 4; ++i)
                q4_st<T>(F + (q * hyp + mr + i * nty) * cb + 4 * nc,
                         Q4<T>{{acc[i][0], acc[i][1], acc[i][2], acc[i][3]}});
        } else {
            const int cy = (q >> 1) ? ny - hy : hy, cx = (q & 1) ? nx - hx : hx;
            const int oy = (q >> 1) ? hy : 0, ox = (q & 1) ? hx : 0;
            const int c = c0 + 4 * nc;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int ky = mr + i * nty;
                if (ky >= cy) continue;
                T* row = o + (oy + ky) * nx + ox + c;
                if (c + 4 <= cx && ((nx | hx) & 3) == 0) {
                    q4_st<T>(row, Q4<T>{{acc[i][0], acc[i][1], acc[i][2], acc[i][3]}});
                } else {
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        if (c + j < cx) row[j] = acc[i][j];
                }
            }
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
                const T ee = F[y * cb + j], eo = F[(hyp + y) * cb + j];
                const T oe = F[(2 * hyp + y) * cb + j], oo = F[(3 * hyp + y) * cb + j];
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

// The three-point equations along z of every column (kx, ky), in place.
// blockDim = (32 columns, chunks), blockIdx.y = state.  y' and x' below are
// the up and down recursions divided by rho: y'_k = r_k + rho y'_(k-1),
// x'_k = y'_k + rho x'_(k+1), e_k = -rho h_z^2 x'_k.
template <typename T, int ZM>
__global__ void __launch_bounds__(dir_z_threads<T>(ZM))
    k_dir_z(DirPlan<T> P, SliceCtl* __restrict__ ctl, T* __restrict__ a) {
    pdl_wait();
    const long long s = blockIdx.y;
    if (!dir_active<T>(ctl + s)) return;
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
        if (sizeof(T) == 4) {
            ctl[s].it_cur = 1;
            ctl[s].total_iters += 1;
        }
    }
}

// FP64: x += e, r -= L e + mean(r), (r, r), sum x; the last CTA decides.  The
// mean of the residual, made by rounding, is out of every correction's reach
// (L has no range there): it is taken out of the next residual, or it would
// be the floor of a solve whose right side is itself close to rounding.
__global__ void __launch_bounds__(NTHREADS)
    k_dir_update(Lev L, MgBuf<double> mb, SliceCtl* __restrict__ ctl,
                 const double* __restrict__ evec, double* __restrict__ part, double tol2,
                 int maxit, int nfluid) {
    pdl_wait();
    const long long s = blockIdx.y;
    SliceCtl* c = ctl + s;
    if (c->status != ST_ITER) return;
    const long long off = s * L.cells;
    const double* __restrict__ e = evec + off;
    double* __restrict__ x = mb.x + off;
    double* __restrict__ r = mb.r + off;
    int i, j, k0;
    lev_origin(L, blockIdx.x, i, j, k0);
    const double rmean = c->rmean;
    double rr = 0.0, sx = 0.0, sr = 0.0;
    if (i < L.n[0] && j < L.n[1]) {
        const int k1 = min(k0 + L.tz, L.n[2]);
        const NbrXY xy = make_nbr_xy(L, i, j);
        const int plane = L.n[0] * L.n[1];
        for (int kb = k0; kb < k1; kb += MG_ZB) {
            Vals7<double> ev[MG_ZB];
            double xo[MG_ZB], ro[MG_ZB];
#pragma unroll
            for (int q = 0; q < MG_ZB; ++q) {
                if (kb + q < k1) {
                    const Nbr nb = nbr_at(L, xy, kb + q);
                    ev[q] = load7<double>(nb, e);
                    xo[q] = x[nb.c];
                    ro[q] = r[nb.c];
                }
            }
#pragma unroll
            for (int q = 0; q < MG_ZB; ++q) {
                if (kb + q < k1) {
                    const int id = (kb + q) * plane + xy.base;
                    const double xv = xo[q] + ev[q].c;
                    const double rv = ro[q] - lap_vals<double>(L, ev[q]) - rmean;
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
// host side: the plan and its tables
// ---------------------------------------------------------------------------

// Eigenvectors and eigenvalues (of minus the unscaled second difference) of
// one axis: even ones first; q[m * n + j] = value of vector m at cell j.
inline void dir_basis(int n, bool periodic, std::vector<double>& q, std::vector<double>& lam) {
    const double pi = 3.14159265358979323846;
    const int h = (n + 1) / 2;
    q.assign((size_t)n * n, 0.0);
    lam.assign(n, 0.0);
    for (int m = 0; m < n; ++m) {
        const bool even = m < h;
        const int i = even ? m : m - h;  // index within its parity
        double w, norm = std::sqrt(2.0 / n);
        bool sine = false;
        if (!periodic) {
            const int k = even ? 2 * i : 2 * i + 1;
            w = pi * k / n;
            if (k == 0) norm = std::sqrt(1.0 / n);
        } else {
            // cosines m = 0 .. h-1, sines m = 1 .. n/2 (the highest mode of an
            // even n is the sine pi (j + 1/2))
            const int k = even ? i : i + 1;
            w = 2.0 * pi * k / n;
            sine = !even;
            if (k == 0 || 2 * k == n) norm = std::sqrt(1.0 / n);
        }
        const double sh = std::sin(0.5 * w);
        lam[m] = 4.0 * sh * sh;
        for (int j = 0; j < n; ++j)
            q[(size_t)m * n + j] = norm * (sine ? std::sin(w * (j + 0.5)) : std::cos(w * (j + 0.5)));
    }
}

// Fills P's sizes for n cells; false where the plane does not fit shared
// memory or a column the chunks of one CTA.
template <typename T>
inline bool dir_sizes(const int n[3], bool per_z, int planes, DirPlan<T>& P) {
    P = DirPlan<T>{};
    P.nx = n[0];
    P.ny = n[1];
    P.nz = n[2];
    P.per_z = per_z ? 1 : 0;
    P.cells = (long long)n[0] * n[1] * n[2];
    P.hx = (n[0] + 1) / 2;
    P.hy = (n[1] + 1) / 2;
    P.hxp = (P.hx + 3) / 4 * 4;
    P.hyp = (P.hy + 3) / 4 * 4;
    // rows an odd number of 16-byte units apart: eight rows' reads then hit
    // different banks
    auto odd = [](int w) { return (w / 4) % 2 ? w : w + 4; };
    P.ldx = odd(P.hxp);
    P.ldy = odd(P.hyp);
    P.zm = n[2] <= 16 * DIR_ZC ? DIR_ZC : DIR_ZC_LONG;
    P.zc = (n[2] + P.zm - 1) / P.zm;
    if (P.zc * DIR_ZX > dir_z_threads<T>(P.zm)) return false;
    // column blocks: as few as shared memory allows, two at least where the
    // planes of a call would leave SMs idle
    for (int xb = planes < 152 && P.hxp > 4 ? 2 : 1; xb <= P.hxp / 4; ++xb) {
        P.cb = (P.hxp / 4 + xb - 1) / xb * 4;
        P.xb = (P.hxp + P.cb - 1) / P.cb;
        if (dir_smem_elems(P) * sizeof(T) <= DIR_MAX_SMEM) {
            const int tiles = P.hyp * P.cb / 4;
            P.nt = (tiles + 31) / 32 * 32;
            P.nt = P.nt < 64 ? 64 : P.nt;
            P.nt = P.nt < P.hxp ? (P.hxp + 31) / 32 * 32 : P.nt;
            P.nt = P.nt > DIR_MAX_THREADS ? DIR_MAX_THREADS : P.nt;
            return P.nt >= P.hxp;
        }
    }
    return false;
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
            const double rn = std::pow(rho, P.nz);
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
