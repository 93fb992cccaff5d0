// Discrete adjoint of the fine step (Section 2 discretisation), for the
// gradient of J = 1/2 sum over active faces of component^2 hx hy hz.
//
// One step is u+ = P(u + dt R(u; u_lid)), P = I - G L^-1 D (the projection,
// symmetric since D = -G^T), R = Re^-1 lap_h u - div_h(u u) with SMART faces.
// Its adjoint maps lambda = dJ/du+ to
//   mu = P lambda,   dJ/du = mu + dt (dR/du)^T mu,   dJ/du_lid += dt (dR/du_lid)^T mu.
// (dR/du)^T mu is gathered: every stored value sums the derivatives of the
// stencil terms that read it (directly, or through the ghost rule of a wall
// reading it as a mirror), each interface flux weighted by the difference of
// mu on its two faces.  Every output is written by one thread in a fixed
// order, so the gradient does not depend on scheduling.  SMART takes the
// branch the forward kernel took (comparisons equal up to rounding); a
// flux with zero transporting velocity takes the derivative of its
// left-upwind form.  T = double (FP64 grids) or float (FP32 storage; the lid
// derivative and J are summed in FP64).
#pragma once

#include "ns_kernels.cuh"

namespace nsk {

// partial derivatives of smart_face(U, C, D), branch by branch
template <typename T>
__device__ __forceinline__ void smart_partials(T U, T C, T D, T& dU, T& dC, T& dD) {
    dU = dC = dD = T(0);
    const T dd = D - U;
    const T cc = C - U;
    if (dd == T(0)) {
        dC = T(1);
        return;
    }
    const T a = dd > T(0) ? cc : -cc;
    const T b = fabs(dd);
    if (a < T(0) || a > b) {
        dC = T(1);
    } else if (T(6) * a <= b) {
        dU = T(-2);
        dC = T(3);
    } else if (T(6) * a <= T(5) * b) {
        dU = T(-0.125);
        dC = T(0.75);
        dD = T(0.375);
    } else {
        dD = T(1);
    }
}

// flux uf * phi between b (lower) and f (higher): d/d uf and d/d (bb, b, f, ff)
template <typename T>
__device__ __forceinline__ void flux_partials(T uf, T bb, T b, T f, T ff, T& duf, T (&d4)[4]) {
    T dU, dC, dD;
    d4[0] = d4[1] = d4[2] = d4[3] = T(0);
    if (uf < T(0)) {
        duf = smart_face(ff, f, b);
        smart_partials(ff, f, b, dU, dC, dD);
        d4[3] = uf * dU;
        d4[2] = uf * dC;
        d4[1] = uf * dD;
    } else {
        duf = smart_face(bb, b, f);
        smart_partials(bb, b, f, dU, dC, dD);
        d4[0] = uf * dU;
        d4[1] = uf * dC;
        d4[2] = uf * dD;
    }
}

// mu of component c at f (f[d] may lie outside the stored range along d):
// wrapped along a periodic axis, zero outside the stored range and on
// inactive (wall-normal boundary) faces.
template <typename T>
__device__ __forceinline__ T adj_mu_at(const Geo& g, int c, const T* __restrict__ mu, int d,
                                       const int f[3]) {
    int q[3] = {f[0], f[1], f[2]};
    const int e = g.ext[c][d];
    if (q[d] < 0 || q[d] >= e) {
        if (g.bc[d] != BC_PERIODIC) return T(0);
        q[d] = q[d] < 0 ? q[d] + e : q[d] - e;
    }
    const bool active = g.bc[c] == BC_PERIODIC || (q[c] > 0 && q[c] < g.n[c]);
    return active ? mu[vindex(g, c, q[0], q[1], q[2])] : T(0);
}

// Is p an interface of component c along d that a forward flux is evaluated
// at (between positions p and p+1)?  Periodic axes wrap p.  Normal
// component: between the active faces 1..n-1 and their neighbours (0..n-1);
// tangential: -1..n-1 (the edges on the walls included).
__device__ __forceinline__ bool adj_iface(const Geo& g, int c, int d, int& p) {
    if (g.bc[d] == BC_PERIODIC) {
        const int e = g.ext[c][d];
        p = p < 0 ? p + e : (p >= e ? p - e : p);
        return true;
    }
    return d == c ? (p >= 0 && p <= g.n[d] - 1) : (p >= -1 && p <= g.n[d] - 1);
}

// Derivatives of the forward flux of component c through the interface
// between f and f + e_d (f[d] = p): with respect to its transporting
// velocity (duf) and to the four values at f - e_d .. f + 2 e_d (d4).
template <typename T>
__device__ __forceinline__ void adj_iface_flux(const Geo& g, int c, int d,
                                               const T* const (&vel3)[3], const int f[3],
                                               T& duf, T (&d4)[4]) {
    T a[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        int r[3] = {f[0], f[1], f[2]};
        r[d] += q - 1;
        a[q] = vel(g, c, vel3[c], r[0], r[1], r[2]);
    }
    T uf;
    if (d == c) {
        uf = T(0.5) * (a[1] + a[2]);
    } else {
        int q0[3] = {f[0], f[1], f[2]};
        int q1[3] = {f[0], f[1], f[2]};
        q0[c] -= 1;
        q0[d] += 1;
        q1[d] += 1;
        uf = T(0.5) * (vel(g, d, vel3[d], q0[0], q0[1], q0[2]) +
                       vel(g, d, vel3[d], q1[0], q1[1], q1[2]));
    }
    flux_partials(uf, a[0], a[1], a[2], a[3], duf, d4);
}

// (dR/du)^T mu at the stored value t of component c, and its share of
// (dR/du_lid)^T mu (returned in dl).
template <typename T>
__device__ __forceinline__ T adj_gather(const Geo& g, int c, const int t[3],
                                        const T* const (&vel3)[3], const T* const (&mu3)[3],
                                        double& dl) {
    T acc = T(0);
    const T inv_re = g_inv_re<T>(g);
#pragma unroll 1
    for (int d = 0; d < 3; ++d) {
        const T ih = g_ih<T>(g, d), ih2 = g_ih2<T>(g, d);
        const int n = g.n[d], x = t[d];
        // the positions whose value is t's: t itself and the ghosts that
        // mirror it (sign, and the lid's coefficient in the ghost value)
        int r[3];
        T sg[3];
        T lid[3];
        int nim = 0;
        r[nim] = x;
        sg[nim] = T(1);
        lid[nim++] = T(0);
        if (g.bc[d] != BC_PERIODIC) {
            if (d == c) {
                if (x >= 1 && x <= 2) {
                    r[nim] = -x;
                    sg[nim] = T(-1);
                    lid[nim++] = T(0);
                }
                if (x >= n - 2 && x <= n - 1 && x >= 0) {
                    r[nim] = 2 * n - x;
                    sg[nim] = T(-1);
                    lid[nim++] = T(0);
                }
            } else {
                const T s = g.bc[d] == BC_SLIP ? T(1) : T(-1);
                if (x <= 1) {
                    r[nim] = -x - 1;
                    sg[nim] = s;
                    lid[nim++] = T(0);
                }
                if (x >= n - 2) {
                    r[nim] = 2 * n - 1 - x;
                    sg[nim] = s;
                    lid[nim++] = (g.bc[d] == BC_WALL && c == 0 && d == 1) ? T(2) : T(0);
                }
            }
        }
#pragma unroll 1
        for (int m = 0; m < nim; ++m) {
            int f[3] = {t[0], t[1], t[2]};
            // diffusion Re^-1 (a3 - 2 a2 + a1) / h^2 of the faces r+1, r, r-1
            T sd = T(0);
#pragma unroll
            for (int o = -1; o <= 1; ++o) {
                f[d] = r[m] + o;
                sd += (o == 0 ? T(-2) : T(1)) * adj_mu_at(g, c, mu3[c], d, f);
            }
            T tot = inv_re * ih2 * sd;
            // convection -(F(p) - F(p-1)) / h: the interfaces p = r - k that
            // read r in role k (k = -1: far upwind below, 0, 1, 2)
#pragma unroll 1
            for (int k = -1; k <= 2; ++k) {
                int p = r[m] - k;
                if (!adj_iface(g, c, d, p)) continue;
                f[d] = p + 1;
                const T hi = adj_mu_at(g, c, mu3[c], d, f);
                f[d] = p;
                const T lo = adj_mu_at(g, c, mu3[c], d, f);
                const T nu = (hi - lo) * ih;
                if (nu == T(0)) continue;
                T duf, d4[4];
                adj_iface_flux(g, c, d, vel3, f, duf, d4);
                T w = d4[k + 1];
                if (d == c && (k == 0 || k == 1)) w += T(0.5) * duf;
                tot += nu * w;
            }
            acc += sg[m] * tot;
            dl += double(lid[m]) * double(tot);
        }
    }
    // t as the transporting velocity of the other components' fluxes along
    // its own axis: the interfaces of faces t - e_c and t - e_c + e_c2
#pragma unroll 1
    for (int c2 = 0; c2 < 3; ++c2) {
        if (c2 == c) continue;
        const int d = c;
        const T ih = g_ih<T>(g, d);
#pragma unroll 1
        for (int cand = 0; cand < 2; ++cand) {
            int f[3] = {t[0], t[1], t[2]};
            int p = f[d] - 1;
            if (!adj_iface(g, c2, d, p)) continue;
            f[d] = p;
            if (cand) {
                f[c2] += 1;
                if (f[c2] >= g.ext[c2][c2]) {
                    if (g.bc[c2] != BC_PERIODIC) continue;
                    f[c2] -= g.ext[c2][c2];
                }
            }
            int fh[3] = {f[0], f[1], f[2]};
            fh[d] += 1;
            const T nu = (adj_mu_at(g, c2, mu3[c2], d, fh) - adj_mu_at(g, c2, mu3[c2], d, f)) * ih;
            if (nu == T(0)) continue;
            T duf, d4[4];
            adj_iface_flux(g, c2, d, vel3, f, duf, d4);
            acc += T(0.5) * nu * duf;
        }
    }
    return acc;
}

// out = (dR/du)^T mu for every state of the batch (blockIdx.y), every stored
// value written once, component blockIdx.z; each thread gathers ADJ_TZ
// positions along z of a 32 x 4 column tile (the gather is latency-bound, so
// the launch spreads over many CTAs).  Per-CTA partial sums of
// (dR/du_lid)^T mu go to part_lid[state][component][cta] (summed in a fixed
// order by k_adj_sum).
constexpr int ADJ_TZ = 2;

template <typename T>
__global__ void __launch_bounds__(NTHREADS)
    k_adj_rhs(Geo g, const T* __restrict__ u, const T* __restrict__ v, const T* __restrict__ w,
              const T* __restrict__ mu_u, const T* __restrict__ mu_v, const T* __restrict__ mu_w,
              T* __restrict__ ou, T* __restrict__ ov, T* __restrict__ ow,
              double* __restrict__ part_lid) {
    const long long s = blockIdx.y;
    const int c = blockIdx.z;
    const T* const vel3[3] = {u + s * g.cnt[0], v + s * g.cnt[1], w + s * g.cnt[2]};
    const T* const mu3[3] = {mu_u + s * g.cnt[0], mu_v + s * g.cnt[1], mu_w + s * g.cnt[2]};
    T* const out = (c == 0 ? ou : (c == 1 ? ov : ow)) + s * g.cnt[c];
    const int cta = blockIdx.x;
    const int i = (cta % g.fbx) * TX + (int)threadIdx.x;
    const int r = cta / g.fbx;
    const int j = (r % g.fby) * TY + (int)threadIdx.y;
    const int k0 = (r / g.fby) * ADJ_TZ;
    const int k1 = min(k0 + ADJ_TZ, g.ext[c][2]);
    double dl = 0.0;
    if (i < g.ext[c][0] && j < g.ext[c][1]) {
        for (int k = k0; k < k1; ++k) {
            const int t[3] = {i, j, k};
            out[vindex(g, c, i, j, k)] = adj_gather(g, c, t, vel3, mu3, dl);
        }
    }
    double v1[1] = {dl};
    write_partials<1>(v1, part_lid + (s * 3 + c) * (long long)gridDim.x + blockIdx.x);
}

// out[s] (+)= sum of part[s][0..n-1] in order, one thread per state.
__global__ void __launch_bounds__(32)
    k_adj_sum(const double* __restrict__ part, int n, int batch, double* __restrict__ out,
              int add) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= batch) return;
    double acc = 0.0;
    for (int q = 0; q < n; ++q) acc += part[(long long)s * n + q];
    out[s] = add ? out[s] + acc : acc;
}

// lambda = mu + dt * acc on active faces, 0 elsewhere; acc is zeroed for reuse.
template <typename T>
__global__ void __launch_bounds__(256)
    k_adj_finish(Geo g, int c, long long n_total, const T* __restrict__ mu,
                 T* __restrict__ acc, T* __restrict__ lam, double dt) {
    const T tdt = T(dt);
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n_total;
         q += (long long)gridDim.x * blockDim.x) {
        const long long local = q % g.cnt[c];
        const int i = int(local % g.ext[c][0]);
        const int j = int((local / g.ext[c][0]) % g.ext[c][1]);
        const int k = int(local / ((long long)g.ext[c][0] * g.ext[c][1]));
        const int f[3] = {i, j, k};
        const bool active = g.bc[c] == BC_PERIODIC || (f[c] > 0 && f[c] < g.n[c]);
        lam[q] = active ? mu[q] + tdt * acc[q] : T(0);
        acc[q] = T(0);
    }
}

// lambda = u * vol on active faces (0 elsewhere; skipped when lam is null)
// and the per-CTA partial sums of J = 1/2 sum u^2 vol in part[state][cta]
// (blockIdx.y = state; the CTAs of the three components at offsets
// c * gridDim.x).
template <typename T>
__global__ void __launch_bounds__(NTHREADS)
    k_adj_terminal(Geo g, int c, const T* __restrict__ u, T* __restrict__ lam,
                   double* __restrict__ part, double vol) {
    const long long s = blockIdx.y;
    const long long per = g.cnt[c];
    const T* us = u + s * per;
    T* ls = lam ? lam + s * per : nullptr;
    const T tvol = T(vol);
    double acc = 0.0;
    for (long long q = blockIdx.x * (long long)NTHREADS + tid_flat(); q < per;
         q += (long long)gridDim.x * NTHREADS) {
        const int i = int(q % g.ext[c][0]);
        const int j = int((q / g.ext[c][0]) % g.ext[c][1]);
        const int k = int(q / ((long long)g.ext[c][0] * g.ext[c][1]));
        const int f[3] = {i, j, k};
        const bool active = g.bc[c] == BC_PERIODIC || (f[c] > 0 && f[c] < g.n[c]);
        const T x = active ? us[q] : T(0);
        if (ls) ls[q] = x * tvol;
        acc += 0.5 * double(x) * double(x) * vol;
    }
    double v1[1] = {acc};
    write_partials<1>(v1, part + s * 3LL * gridDim.x + (long long)c * gridDim.x + blockIdx.x);
}

// ---------------------------------------------------------------------------
// the reverse step from shared memory, and the wide sum
// ---------------------------------------------------------------------------

// Tile of k_adj_tile: 32 x 4 columns, AT_Z cells along z, halo 3.
constexpr int AT_Z = 4, AT_H = 3;
constexpr int AT_SX = TX + 2 * AT_H, AT_SY = TY + 2 * AT_H, AT_SZ = AT_Z + 2 * AT_H;
constexpr int AT_PLANE = AT_SX * AT_SY, AT_N = AT_PLANE * AT_SZ;

// Where position i of component c along axis d is read from: the stored index,
// ~index with the ghost rule's sign -1, AT_NONE beyond the two ghosts of a
// wall.  lid: the ghost adds twice the lid speed.
constexpr int AT_NONE = -(1 << 30);
__device__ __forceinline__ int adj_src(const Geo& g, int c, int d, int i, bool& lid) {
    const int e = g.ext[c][d], n = g.n[d];
    if (g.bc[d] == BC_PERIODIC) return ((i % e) + e) % e;
    if (i >= 0 && i < e) return i;
    if (i < -2 || i > e + 1) return AT_NONE;
    const bool hi = i >= e;
    int q;
    bool neg = true;
    if (d == c) {
        q = hi ? 2 * n - i : -i;
    } else {
        q = hi ? 2 * n - 1 - i : -i - 1;
        neg = g.bc[d] == BC_WALL;
        if (neg && c == 0 && d == 1 && hi) lid = true;
    }
    if (q < 0 || q >= e) return AT_NONE;
    return neg ? ~q : q;
}

// The same for mu: AT_NONE (zero) outside the stored range and on inactive
// faces.
__device__ __forceinline__ int adj_mu_src(const Geo& g, int c, int d, int i) {
    const int e = g.ext[c][d];
    if (g.bc[d] == BC_PERIODIC) return ((i % e) + e) % e;
    if (d == c) return i > 0 && i < g.n[d] ? i : AT_NONE;
    return i >= 0 && i < e ? i : AT_NONE;
}

// Face value of a line bb, b, f, ff transported by uf, and its derivatives by
// the four values: the branch the forward kernel takes (the smallest of 2 |k|,
// |k|/8 + 3|g|/8 and |g| as in smart_phi).
template <typename T>
__device__ __forceinline__ T adj_face(T uf, T bb, T b, T f, T ff, T (&d4)[4]) {
    const bool neg = uf < T(0);
    const T U = neg ? ff : bb, C = neg ? f : b, D = neg ? b : f;
    const T k = C - U, g = D - C;
    const T q = fma(T(0.375), g, T(0.125) * k);
    const T ak = fabs(k + k), aq = fabs(q), ag = fabs(g);
    const bool flat = (k == T(0) && g == T(0)) || (k < T(0) && g > T(0)) || (k > T(0) && g < T(0));
    const bool steep = !flat && ak <= aq && ak <= ag;
    const bool down = !flat && !steep && ag <= aq;
    const bool quick = !flat && !steep && !down;
    const T dU = steep ? T(-2) : (quick ? T(-0.125) : T(0));
    const T dC = steep ? T(3) : (quick ? T(0.75) : (down ? T(0) : T(1)));
    const T dD = quick ? T(0.375) : (down ? T(1) : T(0));
    d4[0] = neg ? T(0) : dU;
    d4[1] = neg ? dD : dC;
    d4[2] = neg ? dC : dD;
    d4[3] = neg ? dU : T(0);
    return flat ? C : (steep ? C + (k + k) : (down ? D : C + q));
}

// lambda = mu + dt (dR/du)^T mu on active faces (zero on wall faces) of a
// tile, every stored value written once; per-CTA partial sums of
// dt (dR/du_lid)^T mu in part_lid[state][cta].  The velocity with its ghost values
// and mu (zero outside) are staged once, so an interior value is a fixed set
// of 16 face evaluations without a boundary rule: interfaces that do not exist
// have mu differences of zero.  The ghosts that mirror a value add their part
// in the threads next to a wall.  Bound: instruction issue (each face is
// evaluated by the values that read it).  64^3, one state, FP32: 305 us
// gathering from global memory with the rules at every read -> 92 us.
template <typename T>
__global__ void __launch_bounds__(NTHREADS)
    k_adj_tile(Geo g, const T* __restrict__ u, const T* __restrict__ v, const T* __restrict__ w,
               const T* __restrict__ mu_u, const T* __restrict__ mu_v, const T* __restrict__ mu_w,
               T* __restrict__ lu, T* __restrict__ lv, T* __restrict__ lw, double dt, int tbx,
               int tby, double* __restrict__ part_lid) {
    extern __shared__ __align__(16) unsigned char asm_raw[];
    T* sv = reinterpret_cast<T*>(asm_raw);  // [3][AT_SZ][AT_SY][AT_SX]
    T* sm = sv + 3 * AT_N;                  // the same of mu
    __shared__ int zv[3][AT_SZ], zu[3][AT_SZ];
    // the forward step's coefficients, dt / h and dt / (Re h^2), then what
    // their rounding to T left
    __shared__ T coef[12];
    const long long s = blockIdx.y;
    const T* const vel3[3] = {u + s * g.cnt[0], v + s * g.cnt[1], w + s * g.cnt[2]};
    const T* const mu3[3] = {mu_u + s * g.cnt[0], mu_v + s * g.cnt[1], mu_w + s * g.cnt[2]};
    T* const out[3] = {lu + s * g.cnt[0], lv + s * g.cnt[1], lw + s * g.cnt[2]};
    const int cta = blockIdx.x, r = cta / tbx, tz = r / tby;
    const int i0 = (cta - r * tbx) * TX, j0 = (r - tz * tby) * TY, k0 = tz * AT_Z;
    const int t = tid_flat();
    if (t < 6) {
        const int d = t < 3 ? t : t - 3;
        const double k = dt * (t < 3 ? g.ih[d] : g.inv_re * g.ih2[d]);
        coef[t] = T(k);
        coef[6 + t] = T(k - double(T(k)));
    }
    for (int q = t; q < 3 * AT_SZ; q += NTHREADS) {
        const int c = q / AT_SZ, z = q - c * AT_SZ;
        bool lid = false;
        zv[c][z] = adj_src(g, c, 2, k0 - AT_H + z, lid);
        zu[c][z] = adj_mu_src(g, c, 2, k0 - AT_H + z);
    }
    __syncthreads();
    const T lid2 = T(2.0 * g.u_lid);
    for (int pq = t; pq < AT_PLANE; pq += NTHREADS) {
        const int py = pq / AT_SX, px = pq - py * AT_SX;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const int e0 = g.ext[c][0];
            const long long plane = (long long)e0 * g.ext[c][1];
            bool lid = false;
            const int qi = adj_src(g, c, 0, i0 - AT_H + px, lid);
            const int qj = adj_src(g, c, 1, j0 - AT_H + py, lid);
            const int mi = adj_mu_src(g, c, 0, i0 - AT_H + px);
            const int mj = adj_mu_src(g, c, 1, j0 - AT_H + py);
            const bool ok = qi != AT_NONE && qj != AT_NONE, mok = mi >= 0 && mj >= 0;
            const bool nxy = (qi < 0) != (qj < 0);
            const int o = ok ? (qj < 0 ? ~qj : qj) * e0 + (qi < 0 ? ~qi : qi) : 0;
            const int m = mok ? mj * e0 + mi : 0;
#pragma unroll
            for (int z = 0; z < AT_SZ; ++z) {
                const int a = zv[c][z], b = zu[c][z];
                T x = T(0);
                if (ok && a != AT_NONE) {
                    x = vel3[c][(a < 0 ? ~a : a) * plane + o];
                    if (nxy != (a < 0)) x = -x;
                    if (lid) x += lid2;
                }
                sv[c * AT_N + z * AT_PLANE + pq] = x;
                sm[c * AT_N + z * AT_PLANE + pq] =
                    (mok && b >= 0) ? mu3[c][b * plane + m] : T(0);
            }
        }
    }
    __syncthreads();
    constexpr int strd[3] = {1, AT_SX, AT_PLANE};
    // coefficient d of the list times a value (FP32: with its rounding)
    auto scaled = [&](int d, T v) -> T {
        return sizeof(T) == 4 ? fma(coef[d], v, coef[6 + d] * v) : coef[d] * v;
    };
    const int x0 = (int)threadIdx.x, y0 = (int)threadIdx.y;
    double dl = 0.0;
    if (i0 + x0 < g.n[0] && j0 + y0 < g.n[1]) {
        const int zn = min(AT_Z, g.n[2] - k0);
        for (int z = 0; z < zn; ++z) {
            const int f[3] = {i0 + x0, j0 + y0, k0 + z};
            const int o = ((z + AT_H) * AT_SY + y0 + AT_H) * AT_SX + x0 + AT_H;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const T* a = sv + c * AT_N + o;
                const T* mc = sm + c * AT_N + o;
                T acc = T(0);
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    const int sd = strd[d];
                    acc += scaled(3 + d, mc[sd] - T(2) * mc[0] + mc[-sd]);
                    // the ghosts that mirror this value, as offsets from it
                    // (0: none): beyond the low and the high wall
                    int lo = 0, hi = 0;
                    T sg = T(-1);
                    const int n = g.n[d], x = f[d];
                    if (g.bc[d] != BC_PERIODIC) {
                        if (d == c) {
                            if (x == 1) lo = -2;
                            if (x == n - 1) hi = 2;
                        } else {
                            if (g.bc[d] == BC_SLIP) sg = T(1);
                            if (x <= 1) lo = -2 * x - 1;
                            if (x >= n - 2) hi = 2 * (n - x) - 1;
                        }
                    }
                    const bool lid = c == 0 && d == 1 && g.bc[1] == BC_WALL;
                    T top = T(0);  // the high ghost's part, before its sign
                    if (d != c) {
                        if (lo == -1) acc += sg * scaled(3 + d, mc[0]);
                        if (hi == 1) top += scaled(3 + d, mc[0]);
                    }
#pragma unroll
                    for (int q = -2; q <= 1; ++q) {
                        // interface between the values at q and q + 1
                        const T nu = scaled(d, mc[(q + 1) * sd] - mc[q * sd]);
                        const T b = a[q * sd], fw = a[(q + 1) * sd];
                        const T* tr = sv + d * AT_N + o + (q + 1) * sd;
                        const T uf = d == c ? T(0.5) * (b + fw) : T(0.5) * (tr[-strd[c]] + tr[0]);
                        T d4[4];
                        const T phi = adj_face(uf, a[(q - 1) * sd], b, fw, a[(q + 2) * sd], d4);
                        T wt = uf * d4[1 - q];
                        if (d == c && (q == 0 || q == -1)) wt += T(0.5) * phi;
                        acc += nu * wt;
                        if (lo != 0) {
                            const int role = lo - q + 1;
#pragma unroll
                            for (int e = 0; e < 4; ++e)
                                if (role == e) acc += sg * (nu * (uf * d4[e]));
                        }
                        if (hi != 0) {
                            const int role = hi - q + 1;
#pragma unroll
                            for (int e = 0; e < 4; ++e)
                                if (role == e) top += nu * (uf * d4[e]);
                        }
                    }
                    acc += sg * top;
                    if (lid && hi != 0) dl += 2.0 * double(top);
                }
                // as the transport of the other components along c
                const int sc = strd[c];
#pragma unroll
                for (int c2 = 0; c2 < 3; ++c2) {
                    if (c2 == c) continue;
                    const int s2 = strd[c2];
#pragma unroll
                    for (int cand = 0; cand < 2; ++cand) {
                        const int at = o - sc + (cand ? s2 : 0);  // the interface's low value
                        const T* l = sv + c2 * AT_N + at;
                        const T* m2 = sm + c2 * AT_N + at;
                        const T nu = scaled(c, m2[sc] - m2[0]);
                        const T* tr = sv + c * AT_N + at + sc;
                        const T uf = T(0.5) * (tr[-s2] + tr[0]);
                        T d4[4];
                        acc += T(0.5) * nu * adj_face(uf, l[-sc], l[0], l[sc], l[2 * sc], d4);
                    }
                }
                const long long id = vindex(g, c, f[0], f[1], f[2]);
                const bool wall = g.bc[c] != BC_PERIODIC;
                out[c][id] = (wall && f[c] == 0) ? T(0) : mc[0] + acc;
                if (wall && f[c] == g.n[c] - 1) {
                    int h[3] = {f[0], f[1], f[2]};
                    h[c] += 1;
                    out[c][vindex(g, c, h[0], h[1], h[2])] = T(0);
                }
            }
        }
    }
    double v1[1] = {dl};
    write_partials<1>(v1, part_lid + s * (long long)gridDim.x + blockIdx.x);
}

// out[s] (+)= sum of part[s][0..n-1], one CTA per state, in a fixed order.
// One thread per state (k_adj_sum) reads its partials one after another, 279
// us for 5000; up to ADJ_SERIAL_SUM of them it is as fast.
constexpr int ADJ_SERIAL_SUM = 32;
__global__ void __launch_bounds__(NTHREADS)
    k_adj_sum_block(const double* __restrict__ part, int n, double* __restrict__ out, int add) {
    const int s = blockIdx.x;
    double v[1] = {0.0};
    for (int q = tid_flat(); q < n; q += NTHREADS) v[0] += part[(long long)s * n + q];
    block_sum<1>(v);
    if (tid_flat() == 0) out[s] = add ? out[s] + v[0] : v[0];
}

}  // namespace nsk
