// Kernels of one forward-Euler Chorin-Temam projection step on the MAC grid
// (Croce, Ruprecht & Krause, Section 2) for a batch of independent states,
// the BiCGStab pressure solve (FP64, or FP32 inner iterations inside an FP64
// iterative refinement), and the Parareal update of Eq. 6.
//
// Every kernel runs one CTA per (tile, state): blockIdx.y is the state and
// blockIdx.x the tile inside it, so the per-state reductions (dot products,
// means) are sums over a fixed set of CTAs in a fixed order, independent of the
// batch size.  Per-state Krylov scalars live in SliceCtl; partial sums of each
// phase are reduced redundantly by every CTA of the next phase, so one
// iteration needs three launches and no host round trip.
#pragma once

#include "ns_device.cuh"

namespace nsk {

enum { ST_ITER = 0, ST_CONV = 1, ST_MAXIT = 2, ST_NONFINITE = 3, ST_IDLE = 4 };
enum { OS_REFINE = 0, OS_DONE = 1, OS_FAIL = 2, OS_NONFINITE = 3 };

struct SliceCtl {
    int status;        // ST_*: state of the current Krylov solve
    int it_cur;        // iterations completed (written by phase C / init)
    int it_next;       // iteration in progress (written by phase A)
    int restart;       // phase A restarted the recurrence (p := r)
    double rho[2];     // (r_hat, r) of the last two iterations, by parity
    double alpha, omega;
    double bb;         // ||b||^2 of the current solve
    double rr;         // ||r||^2 when the solve stopped
    double sx;         // sum of the solution over the state when the solve stopped
    int o_status;      // OS_*: FP32+refine outer loop
    int o_steps;       // outer corrections applied
    int p_final;       // FP32+refine: p64 buffer holding the result
    int fail;          // graph-resident solves: sticky bits, 1 not converged, 2 non-finite
    double o_bb, o_rr;
    long long total_iters;  // Krylov iterations accumulated over solves
    double beta;       // multigrid path: beta of the next iteration
    long long total_outer;  // graph-resident solves: refinement steps accumulated
    long long total_solves; // graph-resident solves: solves finished
    double o_scale;    // FP32+refine: power of two the inner solve's right side carries
    float o_funs;      // FP32+refine: 1 / that scale, for the next outer correction
    float o_fsc;       // FP32+refine: the scale the next correction gives its right side
    float mean_hi, mean_lo;  // FP32+refine: the fluid mean of the iterate, float-float
    float rmean_hi, rmean_lo;  // FP32+refine: the fluid mean of the outer residual
    double rmean;      // FP64 direct corrections: mean of the residual, 0 outside a solve
    double tol2_in;    // FP32+refine: squared relative tolerance of the inner solve in
                       // progress, when looser than the launch's (else 0)
};

template <typename T>
struct KBuf {       // Krylov vectors of all states, [batch][cells]
    T* x;           // solution (FP64 mode) / inner correction e (FP32 mode)
    T* r;           // residual (FP32 mode: the outer residual r32 in place)
    T* rhat;        // shadow residual
    T* P[2];        // search direction, ping-pong by iteration parity
    T* V[2];        // L P, ping-pong by iteration parity
    T* t;           // L s
};

// ---------------------------------------------------------------------------
// predictor  F* = u + dt (Re^-1 lap u - div(u u))
// ---------------------------------------------------------------------------

// Tiled predictor: a CTA owns PX x PY columns and PZ cells along z.  It marches
// in z with a ring of PT_RING planes of u, v, w in shared memory (tile and a
// halo of two positions, ghost values applied while staging; the plane three
// ahead is loaded during a step and stored at its end) and evaluates every face
// flux once: a thread owns the column (x, y) and computes the fluxes through
// its cell's high faces; the low ones are the left lane's (a shuffle), the
// lower row's (through shared memory; one barrier per z step) and the ones of
// the cell below (carried).  The fluxes through the tile's low x and y faces
// are computed by other threads in turn.
// Faces owned by the tile: the low face of each of its cells along each
// component's axis, plus the high wall face of the last cell of the domain.
// predict_tile_auto chooses the tile, or the tile autotuner among the shapes
// of PT_X columns.
// Bound: FP64, the FP64 pipe (a warp instruction holds it 16 cycles, so the
// face value is selected by integer comparisons and costs four FP64
// operations); FP32, instruction issue (hence the march: staging a tile with
// its z halo at once took half of all instructions) with 16 warps per SM (24
// with a third of the registers less: 168 us against 156).
// Measured against evaluating every y flux twice and the face value by
// comparisons, from 32 x 8 x 4 tiles staged at once: 64^3 x 32 states FP32
// 280 -> 159 us (164 with the low parts of the coefficients, 18 more multiply-adds
// a cell), 64^3 FP32 27 -> 12 us, 64^3 x 4 FP64 747 -> 282 us, 16^3 FP64 121 -> 16
// us.
constexpr int PT_X = 32, PT_Y = 8, PT_Z = 4;
constexpr int PT_THREADS = PT_X * PT_Y;
constexpr int PH = 2;       // halo
#ifdef __CUDACC__
#define NS_MIN_CTAS(...) , __VA_ARGS__
#else
#define NS_MIN_CTAS(...)
#endif
constexpr int PT_RING = 5;  // planes z-1 .. z+2 in use, z+3 being stored

// Staged elements of one component for a PX x PY x PZ tile (whatever PZ).
template <int PY, int PZ, int PX = PT_X>
constexpr int ptile_elems() {
    return (PX + 2 * PH) * (PY + 2 * PH) * PT_RING;
}

template <typename T, bool INCR, int PY = PT_Y, int PZ = PT_Z, int PX = PT_X>
__global__ void __launch_bounds__(PX * PY NS_MIN_CTAS(512 / (PX * PY)))
    k_predict_tile(Geo g, const T* __restrict__ u, const T* __restrict__ v,
                   const T* __restrict__ w, T* __restrict__ fu, T* __restrict__ fv,
                   T* __restrict__ fw, double dt, int tbx, int tby) {
    pdl_wait();
    constexpr int NT = PX * PY;
    constexpr int SX = PX + 2 * PH, SY = PY + 2 * PH;
    constexpr int PLANE = SX * SY, SN = PLANE * PT_RING;
    constexpr int PER = (PLANE + NT - 1) / NT;
    static_assert(PER <= 5, "two flag bits per staged position and component");
    extern __shared__ __align__(16) unsigned char psm_raw[];
    T* sm = reinterpret_cast<T*>(psm_raw);  // [3][PT_RING][SY][SX]
    // fluxes through the tile's low x / y faces and the rows' high y faces, by
    // parity of the z step
    __shared__ T xlo[2][3][PY], ylo[2][3][PX], yex[2][3][PY][PX];
    // dt / (2 h) (the fluxes are twice the convective ones) and dt / (Re h^2),
    // then what their rounding to T left
    __shared__ T coef[12];
    __shared__ int zsrc[3][PZ + 4];  // z index a staged plane comes from, ~ of it: sign -1
    const long long s = blockIdx.y;
    const T* vel3[3] = {u + s * g.cnt[0], v + s * g.cnt[1], w + s * g.cnt[2]};
    T* out[3] = {fu + s * g.cnt[0], fv + s * g.cnt[1], fw + s * g.cnt[2]};
    const int cta = blockIdx.x;
    const int tyz = cta / tbx, tz = tyz / tby;
    const int i0 = (cta - tyz * tbx) * PX;
    const int j0 = (tyz - tz * tby) * PY;
    const int k0 = tz * PZ;
    const int t = threadIdx.x;
    const int zn = min(PZ, g.n[2] - k0);
    // (one warp: a warp's FP64 operation holds the pipe whatever its lanes)
    if (t < 6) {
        const int d = t < 3 ? t : t - 3;
        const double k = dt * (t < 3 ? 0.5 * g.ih[d] : g.inv_re * g.ih2[d]);
        coef[t] = T(k);
        coef[6 + t] = T(k - double(T(k)));
    }
    for (int q = t; q < 3 * (PZ + 4); q += NT) {
        const int c = q / (PZ + 4), gk = k0 - PH + q - c * (PZ + 4);
        int qk = gk;
        T sign = T(1), add = T(0);
        ghost_axis(g, c, 2, qk, sign, add);
        // (positions further out are staged from anywhere and not used)
        if (gk >= g.ext[c][2] + PH) qk = 0;
        zsrc[c][q - c * (PZ + 4)] = sign < T(0) ? ~qk : qk;
    }
    // The plane positions this thread stages: offset in the plane, and flags
    // (1: sign of the ghost rule, 2: the lid's ghost)
    unsigned off[PER][3], flags = 0;
#pragma unroll
    for (int h = 0; h < PER; ++h) {
        const int pq = t + h * NT;
        const int py = pq / SX, px = pq - py * SX;
        const int gi = i0 - PH + px, gj = j0 - PH + py;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const int e0 = g.ext[c][0], e1 = g.ext[c][1];
            int qi = gi, qj = gj;
            T sign = T(1), add = T(0);
            // only positions up to two beyond the stored range are ever read
            const bool near = pq < PLANE && gi < e0 + PH && gj < e1 + PH;
            ghost_axis(g, c, 0, qi, sign, add);
            ghost_axis(g, c, 1, qj, sign, add);
            off[h][c] = near ? (unsigned)qj * (unsigned)e0 + (unsigned)qi : 0u;
            const bool lid = near && c == 0 && gj >= e1 && g.bc[1] == BC_WALL;
            flags |= ((near && sign < T(0) ? 1u : 0u) | (lid ? 2u : 0u)) << (2 * (3 * h + c));
        }
    }
    const T lid2 = T(2.0 * g.u_lid);
    __syncthreads();
    T val[PER][3];
    unsigned zneg = 0;
    // plane z (from k0 - 2) into registers; then into the ring, ghost values
    // (the lid) + sign * mirror applied
    auto load_plane = [&](int z) {
        zneg = 0;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const int zs = zsrc[c][z];
            if (zs < 0) zneg |= 1u << c;
            const T* __restrict__ a =
                vel3[c] + (long long)(zs < 0 ? ~zs : zs) * (g.ext[c][1] * g.ext[c][0]);
#pragma unroll
            for (int h = 0; h < PER; ++h) val[h][c] = a[off[h][c]];
        }
    };
    auto put_plane = [&](int slot) {
        if ((flags | zneg) != 0) {
#pragma unroll
            for (int h = 0; h < PER; ++h)
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    const unsigned f = flags >> (2 * (3 * h + c));
                    if (((f ^ (zneg >> c)) & 1u) != 0) val[h][c] = -val[h][c];
                    if (f & 2u) val[h][c] += lid2;
                }
        }
#pragma unroll
        for (int h = 0; h < PER; ++h)
            if ((h + 1) * NT <= PLANE || t + h * NT < PLANE) {
#pragma unroll
                for (int c = 0; c < 3; ++c) sm[c * SN + slot + t + h * NT] = val[h][c];
            }
    };
#pragma unroll 1
    for (int z = 0; z < PT_RING; ++z) {
        load_plane(z);
        put_plane(z * PLANE);
    }
    __syncthreads();
    const int y = t / PX, x = t - y * PX;
    // this thread's column in the ring's planes z - 1 .. z + 2, and the offset
    // of the plane being stored
    const T* qm = sm + (y + PH) * SX + x + PH + PLANE;
    const T* q0 = qm + PLANE;
    const T* q1 = q0 + PLANE;
    const T* q2 = q1 + PLANE;
    int pn = 0;
    // the low face this thread also computes (from the last thread on, the
    // first ones stage more): component, position, transport
    constexpr int NE = 3 * (PX + PY), EPER = (NE + NT - 1) / NT;
    int eb[EPER], et[EPER], el[EPER];
    T* eo[EPER];
    bool ey[EPER];
#pragma unroll
    for (int h = 0; h < EPER; ++h) {
        const int q = min(NT - 1 - t + h * NT, NE - 1);
        const bool yf = q < 3 * PX;
        const int r = yf ? q : q - 3 * PX, len = yf ? PX : PY;
        const int c = r >= 2 * len ? 2 : (r >= len ? 1 : 0), e = r - c * len;
        const int at = yf ? (PH - 1) * SX + e + PH : (e + PH) * SX + PH - 1;
        eb[h] = c * SN + at;
        et[h] = (yf ? SN : 0) + at + (yf ? SX : 1);
        // its transport's low neighbour: one back along c
        el[h] = c == 0 ? 1 : (c == 1 ? SX : 0);
        eo[h] = yf ? &ylo[0][c][e] : &xlo[0][c][e];
        ey[h] = yf;
    }
    const T kc[3] = {coef[0], coef[1], coef[2]}, kd[3] = {coef[3], coef[4], coef[5]};
    // FP32: the coefficients carry their rounding (up to 6e-8 of every increment
    // of a run, which a functional of the state would show undamped).
    constexpr bool LOW = sizeof(T) == 4;
    const T lc[3] = {coef[6], coef[7], coef[8]}, ld[3] = {coef[9], coef[10], coef[11]};
    const int i = i0 + x, j = j0 + y;
    T fz[3], zm[3], zc[3], zp[3];
    T* dst[3];
    // twice the flux through the low z face of the tile's first cell
    {
        const T w0 = q0[2 * SN];
        const T tr[3] = {q0[2 * SN - 1] + w0, q0[2 * SN - SX] + w0, qm[2 * SN] + w0};
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            zm[c] = qm[c * SN];
            zc[c] = q0[c * SN];
            zp[c] = q1[c * SN];
            fz[c] = mul_rounded(tr[c], smart_phi(tr[c], qm[c * SN - PLANE], zm[c], zc[c], zp[c]));
            dst[c] = out[c] + vindex(g, c, i, j, k0);
        }
    }
    __syncthreads();
    const bool in_xy = i < g.n[0] && j < g.n[1];
    // faces on the walls: the low one, and the high one beside the last cell
    const bool wlo[2] = {g.bc[0] != BC_PERIODIC && i == 0, g.bc[1] != BC_PERIODIC && j == 0};
    const bool whi[2] = {g.bc[0] != BC_PERIODIC && i == g.n[0] - 1,
                         g.bc[1] != BC_PERIODIC && j == g.n[1] - 1};
#pragma unroll 1
    for (int z = 0; z < zn; ++z) {
        const int par = z & 1;
        const bool more = z + 1 < zn;
        if (more) load_plane(z + 5);
#pragma unroll
        for (int h = 0; h < EPER; ++h)
            if (NT - 1 - t + h * NT < NE) {
                const int p0 = (int)(q0 - (sm + (y + PH) * SX + x + PH));
                const int pm = (int)(qm - (sm + (y + PH) * SX + x + PH));
                const T* sc = sm + eb[h] + p0;
                const T* st = sm + et[h];
                const int sd = ey[h] ? SX : 1;
                const T tl = el[h] == 0 ? st[pm] : st[p0 - el[h]];
                const T tr = tl + st[p0];
                eo[h][par * (ey[h] ? 3 * PX : 3 * PY)] =
                    mul_rounded(tr, smart_phi(tr, sc[-sd], sc[0], sc[sd], sc[2 * sd]));
            }
        T inc[3], tx[3], ty[3], px[3], py[3], fxl[3];
        const T uh = q0[1], vh = q0[SN + SX], wh = zp[2];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const T a = zc[c];
            const T xl = q0[c * SN - 1], xh = c == 0 ? uh : q0[c * SN + 1];
            const T yl = q0[c * SN - SX], yh = c == 1 ? vh : q0[c * SN + SX], zpp = q2[c * SN];
            // transport sums of the high x, y, z faces, face values
            tx[c] = uh + (c == 0 ? a : (c == 1 ? q0[1 - SX] : qm[1]));
            ty[c] = vh + (c == 1 ? a : (c == 0 ? q0[SN + SX - 1] : qm[SN + SX]));
            const T tw = wh + (c == 2 ? a : q1[2 * SN - (c == 0 ? 1 : SX)]);
            px[c] = smart_phi(tx[c], xl, a, xh, q0[c * SN + 2]);
            py[c] = smart_phi(ty[c], yl, a, yh, q0[c * SN + 2 * SX]);
            const T pz = smart_phi(tw, zm[c], a, zp[c], zpp);
            yex[par][c][y][x] = mul_rounded(ty[c], py[c]);
            fxl[c] = __shfl_up_sync(0xffffffffu, mul_rounded(tx[c], px[c]), 1);
            // (fma by fma: every tile shape rounds alike; the cell's own high
            // flux enters unrounded)
            const T d2[3] = {(xh - a) - (a - xl), (yh - a) - (a - yl),
                             (zp[c] - a) - (a - zm[c])};
            const T dz = -fma(tw, pz, -fz[c]);
            if (LOW) {
                const T low = fma(d2[2], ld[2], fma(d2[1], ld[1], d2[0] * ld[0]));
                inc[c] = fma(d2[1], kd[1], fma(d2[0], kd[0], fma(dz, lc[2], low)));
            } else {
                inc[c] = fma(d2[1], kd[1], d2[0] * kd[0]);
            }
            inc[c] = fma(dz, kc[2], fma(d2[2], kd[2], inc[c]));
            fz[c] = mul_rounded(tw, pz);
            zm[c] = a;
            zc[c] = zp[c];
            zp[c] = zpp;
        }
        if (more) put_plane(pn);
        __syncthreads();
        const int k = k0 + z;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const T xl = x == 0 ? xlo[par][c][y] : fxl[c];
            const T yl = y == 0 ? ylo[par][c][x] : yex[par][c][y > 0 ? y - 1 : 0][x];
            const T dx = -fma(tx[c], px[c], -xl), dy = -fma(ty[c], py[c], -yl);
            const T low = LOW ? fma(dy, lc[1], fma(dx, lc[0], inc[c])) : inc[c];
            const T incr = fma(dy, kc[1], fma(dx, kc[0], low));
            const bool wall = g.bc[c] != BC_PERIODIC;
            const bool lo = c < 2 ? wlo[c < 2 ? c : 0] : (wall && k == 0);
            // the high wall face of the last cell along c is inactive: zero it
            const bool hi = c < 2 ? whi[c < 2 ? c : 0] : (wall && k == g.n[2] - 1);
            if (in_xy) {
                *dst[c] = lo ? T(0) : (INCR ? incr : zm[c] + incr);
                if (hi)
                    dst[c][c == 0 ? 1 : (c == 1 ? g.ext[1][0] : g.ext[2][0] * g.ext[2][1])] = T(0);
            }
            dst[c] += g.ext[c][0] * g.ext[c][1];
        }
        const int qn = (int)(qm - (sm + (y + PH) * SX + x + PH));
        qm = q0;
        q0 = q1;
        q1 = q2;
        q2 = sm + (y + PH) * SX + x + PH + pn;
        pn = qn;
    }
}

// ---------------------------------------------------------------------------
// predictor with solid cells: one thread per face, stencil arms that stop at
// walls and solid surfaces
// ---------------------------------------------------------------------------

// Value of component c at offset m (|m| <= 2) from face f along axis d, as f's
// stencil arm sees it: stored values up to the first interface (an inactive
// face for the normal arm; a position past a wall or inside a solid for a
// tangential arm), reflected across it beyond -- odd about the interface face
// (normal), 2 u_wall - mirror (tangential; u_wall = 0 at solids, +mirror at a
// slip wall).
template <typename T>
__device__ __forceinline__ T arm_value_dev(const Geo& g, int c, const T* a, const int f[3], int d,
                                           int m) {
    if (m == 0) return a[vindex(g, c, f[0], f[1], f[2])];
    const int sg = m > 0 ? 1 : -1;
    const int am = m > 0 ? m : -m;
    const int n = g.ext[c][d];
    for (int s = 1; s <= am; ++s) {
        int q[3] = {f[0], f[1], f[2]};
        q[d] += sg * s;
        if (g.bc[d] == BC_PERIODIC) q[d] = q[d] < 0 ? q[d] + n : (q[d] >= n ? q[d] - n : q[d]);
        if (c == d) {
            if (q[d] < 0 || q[d] >= n) break;
            if (!face_active_dev(g, c, q)) {
                if (s == am) return T(0);
                int r[3] = {f[0], f[1], f[2]};
                r[d] += sg * (2 * s - am);
                return -vel(g, c, a, r[0], r[1], r[2]);
            }
        } else {
            const bool outside = q[d] < 0 || q[d] >= n;
            if (outside || face_in_solid_dev(g, c, q)) {
                int r[3] = {f[0], f[1], f[2]};
                r[d] += sg * (2 * s - 1 - am);
                const T mirror = vel(g, c, a, r[0], r[1], r[2]);
                if (outside) {
                    if (g.bc[d] == BC_SLIP) return mirror;
                    const bool hi = q[d] >= n;
                    const T uw = (c == 0 && d == 1 && hi) ? T(g.u_lid) : T(0);
                    return T(2) * uw - mirror;
                }
                return -mirror;
            }
        }
    }
    int q[3] = {f[0], f[1], f[2]};
    q[d] += m;
    return vel(g, c, a, q[0], q[1], q[2]);
}

// F* (or its increment) of one stored face.
template <typename T, bool INCR>
__device__ __forceinline__ T predict_masked_face(const Geo& g, int c, const int (&f)[3],
                                                 const T* const (&vel3)[3], T tdt) {
    if (!face_active_dev(g, c, f)) return T(0);
    T conv = T(0), diff = T(0);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        T a[5];
#pragma unroll
        for (int m = 0; m < 5; ++m) a[m] = arm_value_dev(g, c, vel3[c], f, d, m - 2);
        T up, um;
        if (d == c) {
            up = T(0.5) * (a[2] + a[3]);
            um = T(0.5) * (a[1] + a[2]);
        } else {
            int q0[3] = {f[0], f[1], f[2]};
            int q1[3] = {f[0], f[1], f[2]};
            q0[c] = f[c] - 1;
            q0[d] = f[d] + 1;
            q1[d] = f[d] + 1;
            up = T(0.5) * (vel(g, d, vel3[d], q0[0], q0[1], q0[2]) +
                           vel(g, d, vel3[d], q1[0], q1[1], q1[2]));
            q0[d] = f[d];
            q1[d] = f[d];
            um = T(0.5) * (vel(g, d, vel3[d], q0[0], q0[1], q0[2]) +
                           vel(g, d, vel3[d], q1[0], q1[1], q1[2]));
        }
        const T fp = smart_flux(up, a[1], a[2], a[3], a[4]);
        const T fm = smart_flux(um, a[0], a[1], a[2], a[3]);
        conv += (fp - fm) * g_ih<T>(g, d);
        diff += (a[3] - T(2) * a[2] + a[1]) * g_ih2<T>(g, d);
    }
    const T incr = tdt * (g_inv_re<T>(g) * diff - conv);
    return INCR ? incr : vel3[c][vindex(g, c, f[0], f[1], f[2])] + incr;
}

template <typename T, bool INCR>
__global__ void __launch_bounds__(NTHREADS)
    k_predict_masked(Geo g, const T* __restrict__ u, const T* __restrict__ v,
                     const T* __restrict__ w, T* __restrict__ fu, T* __restrict__ fv,
                     T* __restrict__ fw, double dt) {
    pdl_wait();
    const long long s = blockIdx.y;
    const T* const vel3[3] = {u + s * g.cnt[0], v + s * g.cnt[1], w + s * g.cnt[2]};
    T* out[3] = {fu + s * g.cnt[0], fv + s * g.cnt[1], fw + s * g.cnt[2]};
    int i, j, k0;
    tile_origin(g, blockIdx.x, g.fbx, g.fby, i, j, k0);
    const int k1 = min(k0 + g.tz, g.n[2] + 1);
    const T tdt = T(dt);
    for (int k = k0; k < k1; ++k) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            if (!(i < g.ext[c][0] && j < g.ext[c][1] && k < g.ext[c][2])) continue;
            const int f[3] = {i, j, k};
            out[c][vindex(g, c, i, j, k)] = predict_masked_face<T, INCR>(g, c, f, vel3, tdt);
        }
    }
}

// Does a solid cell take part in face f of component c: f does not move, or an
// arm of its stencil meets a solid surface.  Every other face is one that
// k_predict_tile, which knows walls only, evaluates as k_predict_masked does.
__device__ __forceinline__ bool face_near_solid(const Geo& g, int c, const int (&f)[3]) {
    const bool edge = g.bc[c] != BC_PERIODIC && (f[c] == 0 || f[c] == g.n[c]);
    if (edge) return false;
    if (!face_active_dev(g, c, f)) return true;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const int n = g.ext[c][d];
#pragma unroll
        for (int sg = -1; sg <= 1; sg += 2)
            for (int m = 1; m <= 2; ++m) {
                int q[3] = {f[0], f[1], f[2]};
                q[d] += sg * m;
                if (g.bc[d] == BC_PERIODIC)
                    q[d] = q[d] < 0 ? q[d] + n : (q[d] >= n ? q[d] - n : q[d]);
                if (q[d] < 0 || q[d] >= n) break;  // a wall comes first
                if (c == d) {
                    if (g.bc[d] != BC_PERIODIC && (q[d] == 0 || q[d] == g.n[d])) break;
                    if (!face_active_dev(g, c, q)) return true;
                } else if (face_in_solid_dev(g, c, q)) {
                    return true;
                }
            }
    }
    return false;
}

// The faces near solid cells: counted (list null), or their numbers (over u, v
// and w of one state) listed, in any order (every face is evaluated by itself).
static __global__ void __launch_bounds__(256)
    k_list_faces(Geo g, long long* __restrict__ list, unsigned long long* __restrict__ count) {
    const long long total = g.cnt[0] + g.cnt[1] + g.cnt[2];
    const long long q = blockIdx.x * 256ll + threadIdx.x;
    if (q >= total) return;
    const int c = q < g.cnt[0] ? 0 : (q < g.cnt[0] + g.cnt[1] ? 1 : 2);
    const long long l = q - (c > 0 ? g.cnt[0] : 0) - (c > 1 ? g.cnt[1] : 0);
    const long long r = l / g.ext[c][0];
    const int f[3] = {int(l - r * g.ext[c][0]), int(r % g.ext[c][1]), int(r / g.ext[c][1])};
    if (!face_near_solid(g, c, f)) return;
    const unsigned long long at = atomicAdd(count, 1ull);
    if (list) list[at] = q;
}

// The listed faces of every state, over what k_predict_tile left there.
// Bound by the latency of the scattered reads (128^3 x 8 states, 8 boxes, 4 %
// of the faces: 188 us; with the tiles 0.48 ms, against 4.9 ms with every face
// by these rules).
template <typename T, bool INCR>
__global__ void __launch_bounds__(NTHREADS)
    k_predict_faces(Geo g, const T* __restrict__ u, const T* __restrict__ v,
                    const T* __restrict__ w, T* __restrict__ fu, T* __restrict__ fv,
                    T* __restrict__ fw, double dt, const long long* __restrict__ list,
                    long long count) {
    pdl_wait();
    const long long s = blockIdx.y, at = blockIdx.x * (long long)NTHREADS + tid_flat();
    if (at >= count) return;
    const T* const vel3[3] = {u + s * g.cnt[0], v + s * g.cnt[1], w + s * g.cnt[2]};
    T* out[3] = {fu + s * g.cnt[0], fv + s * g.cnt[1], fw + s * g.cnt[2]};
    const long long q = list[at];
    const T tdt = T(dt);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const long long l = q - (c > 0 ? g.cnt[0] : 0) - (c > 1 ? g.cnt[1] : 0);
        if (l < 0 || l >= g.cnt[c]) continue;
        const long long r = l / g.ext[c][0];
        const int f[3] = {int(l - r * g.ext[c][0]), int(r % g.ext[c][1]), int(r / g.ext[c][1])};
        out[c][l] = predict_masked_face<T, INCR>(g, c, f, vel3, tdt);
    }
}

// ---------------------------------------------------------------------------
// b = D F* / dt, per-CTA partial sums of b (for the fluid mean)
// ---------------------------------------------------------------------------

// With u, v, w non-null (the increment form's first step) the divergence is
// that of (u + F*) -- F* then holds the increment -- each part differenced
// exactly in FP64.
template <typename T>
__global__ void __launch_bounds__(NTHREADS)
    k_divergence(Geo g, const T* __restrict__ fu, const T* __restrict__ fv,
                 const T* __restrict__ fw, const T* __restrict__ u, const T* __restrict__ v,
                 const T* __restrict__ w, double* __restrict__ b, double* __restrict__ part,
                 double inv_dt) {
    pdl_wait();
    const long long s = blockIdx.y;
    fu += s * g.cnt[0];
    fv += s * g.cnt[1];
    fw += s * g.cnt[2];
    const bool with_u = u != nullptr;
    if (with_u) {
        u += s * g.cnt[0];
        v += s * g.cnt[1];
        w += s * g.cnt[2];
    }
    b += s * g.cnt[3];
    int i, j, k0;
    tile_origin(g, blockIdx.x, g.bx, g.by, i, j, k0);
    double acc[1] = {0.0};
    if (i < g.n[0] && j < g.n[1]) {
        const int k1 = min(k0 + g.tz, g.n[2]);
        const int ip = (g.bc[0] == BC_PERIODIC && i + 1 == g.n[0]) ? 0 : i + 1;
        const int jp = (g.bc[1] == BC_PERIODIC && j + 1 == g.n[1]) ? 0 : j + 1;
        // a batch of DIV_ZB cells' face values is loaded before any of them
        // is differenced, so the loads of the batch are in flight together
        constexpr int DIV_ZB = 4;
        for (int kb = k0; kb < k1; kb += DIV_ZB) {
            T fa[DIV_ZB][6];
#pragma unroll
            for (int z = 0; z < DIV_ZB; ++z) {
                const int k = kb + z;
                if (k < k1) {
                    const int kp = (g.bc[2] == BC_PERIODIC && k + 1 == g.n[2]) ? 0 : k + 1;
                    fa[z][0] = fu[vindex(g, 0, ip, j, k)];
                    fa[z][1] = fu[vindex(g, 0, i, j, k)];
                    fa[z][2] = fv[vindex(g, 1, i, jp, k)];
                    fa[z][3] = fv[vindex(g, 1, i, j, k)];
                    fa[z][4] = fw[vindex(g, 2, i, j, kp)];
                    fa[z][5] = fw[vindex(g, 2, i, j, k)];
                }
            }
#pragma unroll
            for (int z = 0; z < DIV_ZB; ++z) {
                const int k = kb + z;
                if (k >= k1) break;
                const int kp = (g.bc[2] == BC_PERIODIC && k + 1 == g.n[2]) ? 0 : k + 1;
                // D of the stored F* (or increment) in the storage precision; in
                // FP32 this is the increment, whose differences carry no
                // cancellation against u
                T dt_ = (fa[z][0] - fa[z][1]) * g_ih<T>(g, 0);
                dt_ += (fa[z][2] - fa[z][3]) * g_ih<T>(g, 1);
                dt_ += (fa[z][4] - fa[z][5]) * g_ih<T>(g, 2);
                double dv = double(dt_);
                if (with_u) {
                    // the stored u itself: differences taken exactly in FP64
                    double du =
                        (double(u[vindex(g, 0, ip, j, k)]) - double(u[vindex(g, 0, i, j, k)])) *
                        g.ih[0];
                    du += (double(v[vindex(g, 1, i, jp, k)]) - double(v[vindex(g, 1, i, j, k)])) *
                          g.ih[1];
                    du += (double(w[vindex(g, 2, i, j, kp)]) - double(w[vindex(g, 2, i, j, k)])) *
                          g.ih[2];
                    dv += du;
                }
                const double bv = cell_solid(g, i, j, k) ? 0.0 : dv * inv_dt;
                b[cindex(g, i, j, k)] = bv;
                acc[0] += bv;
            }
        }
    }
    write_partials<1>(acc, part + (s * g.ctas + blockIdx.x));
}

// partial sums of a cell field (for the mean of a caller-supplied right side)
static __global__ void __launch_bounds__(NTHREADS)
    k_sum_cells(Geo g, const double* __restrict__ x, double* __restrict__ part) {
    const long long s = blockIdx.y;
    x += s * g.cnt[3];
    int i, j, k0;
    tile_origin(g, blockIdx.x, g.bx, g.by, i, j, k0);
    double acc[1] = {0.0};
    if (i < g.n[0] && j < g.n[1]) {
        const int k1 = min(k0 + g.tz, g.n[2]);
        for (int k = k0; k < k1; ++k) acc[0] += x[cindex(g, i, j, k)];
    }
    write_partials<1>(acc, part + (s * g.ctas + blockIdx.x));
}

// ---------------------------------------------------------------------------
// BiCGStab (van der Vorst), three phases per iteration
// ---------------------------------------------------------------------------

// Start of a solve with a warm start x0 (FP64 mode): b <- b - mean(b);
// x = x0; r = b - L x0; r_hat = r.  Partials: (r_hat,r), (r,r), sum x, (b,b).
template <typename T>
__global__ void __launch_bounds__(NTHREADS)
    k_bicg_init_warm(Geo g, KBuf<T> kb, SliceCtl* __restrict__ ctl,
                     const double* __restrict__ part_b, T* __restrict__ bvec,
                     const T* __restrict__ x0, double* __restrict__ part_c) {
    const long long s = blockIdx.y;
    double sb[1];
    reduce_partials<1>(part_b + s * g.ctas, g.ctas, sb);
    const T mean = T(sb[0] / g.n_fluid);
    const long long off = s * g.cnt[3];
    T* b = bvec + off;
    const T* xs = x0 + off;
    T* x = kb.x + off;
    T* r = kb.r + off;
    T* rh = kb.rhat + off;
    int i, j, k0;
    tile_origin(g, blockIdx.x, g.bx, g.by, i, j, k0);
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    if (i < g.n[0] && j < g.n[1]) {
        const int k1 = min(k0 + g.tz, g.n[2]);
        auto xv = [&](int a, int bb, int c) { return xs[cindex(g, a, bb, c)]; };
        for (int k = k0; k < k1; ++k) {
            const long long id = cindex(g, i, j, k);
            const bool sol = cell_solid(g, i, j, k);
            const T bv = sol ? T(0) : b[id] - mean;
            const T xc = sol ? T(0) : xs[id];
            const T rv = bv - lap_cell(g, xv, i, j, k, xc);
            b[id] = bv;
            x[id] = xc;
            r[id] = rv;
            rh[id] = rv;
            acc[1] += double(rv) * double(rv);
            acc[2] += double(xc);
            acc[3] += double(bv) * double(bv);
        }
    }
    acc[0] = acc[1];
    write_partials<4>(acc, part_c + (s * g.ctas + blockIdx.x) * 4);
    if (blockIdx.x == 0 && tid_flat() == 0) {
        SliceCtl* c = ctl + s;
        c->status = ST_ITER;
        c->it_cur = 0;
        c->it_next = 0;
        c->omega = 1.0;
        c->alpha = 1.0;
    }
}

// Phase A of iteration i (parity par = i & 1): convergence test on the
// residual of iteration i-1, then p = r + beta (p - omega v) (or p = r on a
// (re)start), v = L p.  Partial: (r_hat, v).
template <typename T>
__global__ void __launch_bounds__(NTHREADS)
    k_bicg_A(Geo g, KBuf<T> kb, SliceCtl* __restrict__ ctl, const double* __restrict__ part_c,
             double* __restrict__ part_a, double tol2, int maxit, int par) {
    const long long s = blockIdx.y;
    SliceCtl* c = ctl + s;
    if (c->status != ST_ITER) return;
    double red[4];
    reduce_partials<4>(part_c + s * g.ctas * 4, g.ctas, red);
    const int done = c->it_cur;
    const int it = done + 1;
    double rho = red[0];
    const double rr = red[1];
    const double bb = it == 1 ? red[3] : c->bb;
    const bool lead = blockIdx.x == 0 && tid_flat() == 0;
    if (!isfinite(rr) || !isfinite(rho)) {
        if (lead) {
            c->status = ST_NONFINITE;
            c->rr = rr;
        }
        return;
    }
    if (rr <= tol2 * bb) {
        if (lead) {
            c->status = ST_CONV;
            c->rr = rr;
            c->sx = red[2];
            if (it == 1) c->bb = bb;
        }
        return;
    }
    if (done >= maxit) {
        if (lead) {
            c->status = ST_MAXIT;
            c->rr = rr;
            if (it == 1) c->bb = bb;
        }
        return;
    }
    const bool restart = it == 1 || rho == 0.0 || c->omega == 0.0;
    double beta = 0.0;
    if (restart)
        rho = rr;
    else
        beta = (rho / c->rho[par ^ 1]) * (c->alpha / c->omega);
    if (lead) {
        c->rho[par] = rho;
        c->it_next = it;
        c->restart = restart ? 1 : 0;
        if (it == 1) c->bb = bb;
    }
    const T tb = T(beta), tw = T(c->omega);
    const long long off = s * g.cnt[3];
    const T* r = kb.r + off;
    T* rh = kb.rhat + off;
    const T* po = kb.P[par ^ 1] + off;
    const T* vo = kb.V[par ^ 1] + off;
    T* pn = kb.P[par] + off;
    T* vn = kb.V[par] + off;
    int i, j, k0;
    tile_origin(g, blockIdx.x, g.bx, g.by, i, j, k0);
    double acc[1] = {0.0};
    if (i < g.n[0] && j < g.n[1]) {
        const int k1 = min(k0 + g.tz, g.n[2]);
        auto pnew = [&](int a, int b, int cc) {
            const long long q = cindex(g, a, b, cc);
            return restart ? r[q] : r[q] + tb * (po[q] - tw * vo[q]);
        };
        for (int k = k0; k < k1; ++k) {
            const long long id = cindex(g, i, j, k);
            const T pc = pnew(i, j, k);
            const T lv = lap_cell(g, pnew, i, j, k, pc);
            pn[id] = pc;
            vn[id] = lv;
            T rhv;
            if (restart && it > 1) {
                rhv = r[id];
                rh[id] = rhv;
            } else {
                rhv = restart ? r[id] : rh[id];
            }
            acc[0] += double(rhv * lv);
        }
    }
    write_partials<1>(acc, part_a + (s * g.ctas + blockIdx.x));
}

// Phase B: alpha = rho / (r_hat, v); s = r - alpha v; t = L s.
// Partials: (t, s), (t, t).
template <typename T>
__global__ void __launch_bounds__(NTHREADS)
    k_bicg_B(Geo g, KBuf<T> kb, SliceCtl* __restrict__ ctl, const double* __restrict__ part_a,
             double* __restrict__ part_b, int par) {
    const long long s = blockIdx.y;
    SliceCtl* c = ctl + s;
    if (c->status != ST_ITER) return;
    double red[1];
    reduce_partials<1>(part_a + s * g.ctas, g.ctas, red);
    const double alpha = c->rho[par] / red[0];
    if (blockIdx.x == 0 && tid_flat() == 0) c->alpha = alpha;
    const T ta = T(alpha);
    const long long off = s * g.cnt[3];
    const T* r = kb.r + off;
    const T* vn = kb.V[par] + off;
    T* t = kb.t + off;
    int i, j, k0;
    tile_origin(g, blockIdx.x, g.bx, g.by, i, j, k0);
    double acc[2] = {0.0, 0.0};
    if (i < g.n[0] && j < g.n[1]) {
        const int k1 = min(k0 + g.tz, g.n[2]);
        auto sv = [&](int a, int b, int cc) {
            const long long q = cindex(g, a, b, cc);
            return r[q] - ta * vn[q];
        };
        for (int k = k0; k < k1; ++k) {
            const long long id = cindex(g, i, j, k);
            const T sc = sv(i, j, k);
            const T tv = lap_cell(g, sv, i, j, k, sc);
            t[id] = tv;
            acc[0] += double(tv * sc);
            acc[1] += double(tv * tv);
        }
    }
    write_partials<2>(acc, part_b + (s * g.ctas + blockIdx.x) * 2);
}

// Phase C: omega = (t,s)/(t,t); x += alpha p + omega s; r = s - omega t.
// Partials: (r_hat, r), (r, r), sum x.
template <typename T>
__global__ void __launch_bounds__(NTHREADS)
    k_bicg_C(Geo g, KBuf<T> kb, SliceCtl* __restrict__ ctl, const double* __restrict__ part_b,
             double* __restrict__ part_c, int par) {
    const long long s = blockIdx.y;
    SliceCtl* c = ctl + s;
    if (c->status != ST_ITER) return;
    double red[2];
    reduce_partials<2>(part_b + s * g.ctas * 2, g.ctas, red);
    const double omega = red[1] != 0.0 ? red[0] / red[1] : 0.0;
    const double alpha = c->alpha;
    if (blockIdx.x == 0 && tid_flat() == 0) {
        c->omega = omega;
        c->it_cur = c->it_next;
        c->total_iters += 1;
    }
    const T ta = T(alpha), tw = T(omega);
    const long long off = s * g.cnt[3];
    T* x = kb.x + off;
    T* r = kb.r + off;
    const T* rh = kb.rhat + off;
    const T* pn = kb.P[par] + off;
    const T* vn = kb.V[par] + off;
    const T* t = kb.t + off;
    int i, j, k0;
    tile_origin(g, blockIdx.x, g.bx, g.by, i, j, k0);
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    if (i < g.n[0] && j < g.n[1]) {
        const int k1 = min(k0 + g.tz, g.n[2]);
        for (int k = k0; k < k1; ++k) {
            const long long id = cindex(g, i, j, k);
            const T sc = r[id] - ta * vn[id];
            const T xv = x[id] + (ta * pn[id] + tw * sc);
            const T rv = sc - tw * t[id];
            x[id] = xv;
            r[id] = rv;
            acc[0] += double(rh[id] * rv);
            acc[1] += double(rv * rv);
            acc[2] += double(xv);
        }
    }
    write_partials<4>(acc, part_c + (s * g.ctas + blockIdx.x) * 4);
}

// ---------------------------------------------------------------------------
// FP32 storage + FP64 iterative refinement of the pressure solve
// ---------------------------------------------------------------------------

// Outer start: b <- b - mean(b) (FP64); p64 = p; r64 = b - L p (FP64);
// r32 = float(r64).  Partials: (r,r), (b,b), sum p.
static __global__ void __launch_bounds__(NTHREADS)
    k_refine_init(Geo g, SliceCtl* __restrict__ ctl, const double* __restrict__ part_b,
                  double* __restrict__ bvec, const double* __restrict__ p_in,
                  double* __restrict__ p64, float* __restrict__ r32, double* __restrict__ part_r) {
    const long long s = blockIdx.y;
    double sb[1];
    reduce_partials<1>(part_b + s * g.ctas, g.ctas, sb);
    const double mean = sb[0] / g.n_fluid;
    const long long off = s * g.cnt[3];
    double* b = bvec + off;
    const double* ps = p_in + off;
    double* pd = p64 + off;
    float* r = r32 + off;
    int i, j, k0;
    tile_origin(g, blockIdx.x, g.bx, g.by, i, j, k0);
    double acc[3] = {0.0, 0.0, 0.0};
    if (i < g.n[0] && j < g.n[1]) {
        const int k1 = min(k0 + g.tz, g.n[2]);
        auto pv = [&](int a, int bb, int c) { return ps[cindex(g, a, bb, c)]; };
        for (int k = k0; k < k1; ++k) {
            const long long id = cindex(g, i, j, k);
            const bool sol = cell_solid(g, i, j, k);
            const double bv = sol ? 0.0 : b[id] - mean;
            const double pc = sol ? 0.0 : ps[id];
            const double rv = bv - lap_cell(g, pv, i, j, k, pc);
            b[id] = bv;
            pd[id] = pc;
            r[id] = float(rv);
            acc[0] += rv * rv;
            acc[1] += bv * bv;
            acc[2] += pc;
        }
    }
    write_partials<3>(acc, part_r + (s * g.ctas + blockIdx.x) * 3);
    if (blockIdx.x == 0 && tid_flat() == 0) {
        SliceCtl* c = ctl + s;
        c->o_status = OS_REFINE;
        c->o_steps = 0;
        c->p_final = 0;
        c->status = ST_IDLE;
    }
}

// Outer convergence test for outer step m, then the start of the inner FP32
// solve of L e = r32 from e = 0: r_hat = r32, e = 0.
static __global__ void __launch_bounds__(NTHREADS)
    k_inner_init(Geo g, KBuf<float> kb, SliceCtl* __restrict__ ctl,
                 const double* __restrict__ part_r, double* __restrict__ part_c, double tol2,
                 int m, int max_outer) {
    const long long s = blockIdx.y;
    SliceCtl* c = ctl + s;
    if (c->o_status != OS_REFINE) return;
    double red[3];
    reduce_partials<3>(part_r + s * g.ctas * 3, g.ctas, red);
    const double rr = red[0];
    const double bb = m == 0 ? red[1] : c->o_bb;
    const bool lead = blockIdx.x == 0 && tid_flat() == 0;
    if (!isfinite(rr)) {
        if (lead) {
            c->o_status = OS_NONFINITE;
            c->o_rr = rr;
            c->status = ST_IDLE;
        }
        return;
    }
    if (rr <= tol2 * bb) {
        if (lead) {
            c->o_status = OS_DONE;
            c->o_rr = rr;
            c->o_bb = bb;
            c->p_final = m & 1;
            c->sx = red[2];
            c->status = ST_IDLE;
        }
        return;
    }
    if (m >= max_outer) {
        if (lead) {
            c->o_status = OS_FAIL;
            c->o_rr = rr;
            c->o_bb = bb;
            c->status = ST_IDLE;
        }
        return;
    }
    const long long off = s * g.cnt[3];
    const float* r = kb.r + off;
    float* rh = kb.rhat + off;
    float* e = kb.x + off;
    int i, j, k0;
    tile_origin(g, blockIdx.x, g.bx, g.by, i, j, k0);
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    if (i < g.n[0] && j < g.n[1]) {
        const int k1 = min(k0 + g.tz, g.n[2]);
        for (int k = k0; k < k1; ++k) {
            const long long id = cindex(g, i, j, k);
            const float rv = r[id];
            rh[id] = rv;
            e[id] = 0.0f;
            acc[1] += double(rv) * double(rv);
        }
    }
    acc[0] = acc[1];
    acc[3] = acc[1];
    write_partials<4>(acc, part_c + (s * g.ctas + blockIdx.x) * 4);
    if (lead) {
        c->status = ST_ITER;
        c->it_cur = 0;
        c->it_next = 0;
        c->omega = 1.0;
        c->alpha = 1.0;
        c->o_steps = m;
        if (m == 0) c->o_bb = bb;
    }
}

// Outer correction: p_new = p_old + e (FP64); r64 = b - L p_new (FP64, p_new
// recomputed at the neighbours); r32 = float(r64).  Partials: (r,r), 0, sum p.
static __global__ void __launch_bounds__(NTHREADS)
    k_refine_update(Geo g, SliceCtl* __restrict__ ctl, const double* __restrict__ bvec,
                    const double* __restrict__ p_old, double* __restrict__ p_new,
                    const float* __restrict__ e_in, float* __restrict__ r32,
                    double* __restrict__ part_r) {
    const long long s = blockIdx.y;
    SliceCtl* c = ctl + s;
    if (c->o_status != OS_REFINE) return;
    if (c->status == ST_NONFINITE) {
        if (blockIdx.x == 0 && tid_flat() == 0) c->o_status = OS_NONFINITE;
        return;
    }
    // a converged inner solve, or one stopped at its iteration limit, still
    // improves p; the outer residual test decides when to stop
    const long long off = s * g.cnt[3];
    const double* b = bvec + off;
    const double* po = p_old + off;
    double* pn = p_new + off;
    const float* e = e_in + off;
    float* r = r32 + off;
    int i, j, k0;
    tile_origin(g, blockIdx.x, g.bx, g.by, i, j, k0);
    double acc[3] = {0.0, 0.0, 0.0};
    if (i < g.n[0] && j < g.n[1]) {
        const int k1 = min(k0 + g.tz, g.n[2]);
        auto pv = [&](int a, int bb, int cc) {
            const long long q = cindex(g, a, bb, cc);
            return po[q] + double(e[q]);
        };
        for (int k = k0; k < k1; ++k) {
            const long long id = cindex(g, i, j, k);
            const double pc = pv(i, j, k);
            const double rv = b[id] - lap_cell(g, pv, i, j, k, pc);
            pn[id] = pc;
            r[id] = float(rv);
            acc[0] += rv * rv;
            acc[2] += pc;
        }
    }
    write_partials<3>(acc, part_r + (s * g.ctas + blockIdx.x) * 3);
}

// ---------------------------------------------------------------------------
// velocity correction u = F* - dt G p and the gauged pressure p - mean(p)
// ---------------------------------------------------------------------------

// x0/x1 select the solution buffer of each state: FP64 mode passes the same
// pointer twice; FP32+refine passes p64[0], p64[1] and the state's
// SliceCtl.p_final picks one.  fs == vel is allowed (in-place projection).
// INCR = false: u = F* - dt G p.  INCR = true: fs holds the increment F* - u
// and u = u + (increment - dt G p).
template <typename T, bool INCR>
__global__ void __launch_bounds__(NTHREADS)
    k_correct(Geo g, const SliceCtl* __restrict__ ctl, const T* fu, const T* fv, const T* fw,
              T* u, T* v, T* w, const double* __restrict__ x0, const double* __restrict__ x1,
              double* __restrict__ p_out, double dt, double* __restrict__ p_keep = nullptr) {
    pdl_wait();
    const long long s = blockIdx.y;
    const SliceCtl* c = ctl + s;
    const double* x = (c->p_final ? x1 : x0) + s * g.cnt[3];
    const double mean = c->sx / g.n_fluid;
    const T* f3[3] = {fu + s * g.cnt[0], fv + s * g.cnt[1], fw + s * g.cnt[2]};
    T* o3[3] = {u + s * g.cnt[0], v + s * g.cnt[1], w + s * g.cnt[2]};
    const double dtih[3] = {dt * g.ih[0], dt * g.ih[1], dt * g.ih[2]};
    int i, j, k0;
    tile_origin(g, blockIdx.x, g.fbx, g.fby, i, j, k0);
    const int k1 = min(k0 + g.tz, g.n[2] + 1);
    for (int k = k0; k < k1; ++k) {
        const int q[3] = {i, j, k};
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            if (i < g.ext[d][0] && j < g.ext[d][1] && k < g.ext[d][2]) {
                const long long id = vindex(g, d, i, j, k);
                const bool active = face_active_dev(g, d, q);
                if (!active) {
                    o3[d][id] = T(0);
                } else {
                    int lo[3] = {i, j, k};
                    lo[d] = q[d] == 0 ? g.n[d] - 1 : q[d] - 1;
                    // dt (G p) in FP64 (dt / h folded into one factor); in the
                    // increment form u + (increment - dt G p) is rounded once
                    const double dgp =
                        (x[cindex(g, i, j, k)] - x[cindex(g, lo[0], lo[1], lo[2])]) * dtih[d];
                    if (INCR)
                        o3[d][id] = o3[d][id] + (f3[d][id] - T(dgp));
                    else
                        o3[d][id] = f3[d][id] - T(dgp);
                }
            }
        }
        if (p_out && i < g.n[0] && j < g.n[1] && k < g.n[2]) {
            const long long id = cindex(g, i, j, k);
            const double pn = cell_solid(g, i, j, k) ? 0.0 : x[id] - mean;
            // p_keep (optional) receives the next solve's warm start, the
            // linear extrapolation 2 p^(n+1) - p^n
            if (p_keep) p_keep[s * g.cnt[3] + id] = 2.0 * pn - p_out[s * g.cnt[3] + id];
            p_out[s * g.cnt[3] + id] = pn;
        }
    }
}

// ---------------------------------------------------------------------------
// Parareal update (Eq. 6): y_next = F + (G_new - G_old), G_old <- G_new,
// defect = max |y_next - y_next_previous| (FP64, atomic max on the bits of a
// non-negative double, so the result does not depend on the order).
// ---------------------------------------------------------------------------

template <typename T>
__global__ void __launch_bounds__(256)
    k_parareal_update(long long n, const T* __restrict__ fy, const T* __restrict__ gnew,
                      T* __restrict__ gold, T* __restrict__ y, unsigned long long* defect) {
    pdl_wait();
    double dmax = 0.0;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n;
         q += (long long)gridDim.x * blockDim.x) {
        const T gn = gnew[q];
        const T nv = fy[q] + (gn - gold[q]);
        const double d = fabs(double(nv) - double(y[q]));
        dmax = (d > dmax || d != d) ? d : dmax;
        y[q] = nv;
        gold[q] = gn;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double other = __shfl_xor_sync(0xffffffffu, dmax, o);
        dmax = (other > dmax || other != other) ? other : dmax;
    }
    if ((threadIdx.x & 31) == 0)
        atomicMax(defect, (unsigned long long)__double_as_longlong(dmax));
}

}  // namespace nsk
