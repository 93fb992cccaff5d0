// Driver of the host emulation of the kernels that apply a direct solve's
// result (test support), one state, every CTA as host threads.
//
// usage: direct_krylov_emu update f|d nx ny nz bcx bcy bcz rr rmean in.bin out.bin
//   k_dir_update: in.bin: x, r [C] FP64, e [C] (f: FP32, d: FP64); out.bin: x, r,
//   then rr, sx, rmean, status, it_cur (FP64).
// usage: direct_krylov_emu cg nx ny nz bcx bcy bcz its restart in.bin out.bin
//   conjugate gradients: its iterations of k_cg_dot, k_cg_lap, k_cg_update with
//   z = d r, then r replaced (an outer correction) and restart more.  in.bin:
//   face codes [C] (bytes), FP32: r, d, the second r, z of solid cells (all [C]);
//   out.bin: FP32 x [C] of each solve, r [C] of each; FP64 (r, r), sum x of each.

#include <functional>

static void launch(int gx, const std::function<void()>& body) {
    for (int bx = 0; bx < gx; ++bx) {
        std::barrier<> bar(NTHREADS);
        emu_cta_barrier = &bar;
        for (int w = 0; w < NWARPS; ++w) emu_warp_barrier[w] = new std::barrier<>(32);
        std::vector<std::thread> th;
        for (int t = 0; t < NTHREADS; ++t)
            th.emplace_back([&, t, bx]() {
                threadIdx.x = (unsigned)(t % TX);
                threadIdx.y = (unsigned)(t / TX);
                blockIdx.x = (unsigned)bx;
                blockIdx.y = 0;
                body();
                emu_warp_barrier[t / 32]->arrive_and_drop();
                bar.arrive_and_drop();
            });
        for (auto& x : th) x.join();
        for (int w = 0; w < NWARPS; ++w) delete emu_warp_barrier[w];
    }
}

static Lev level(char** a) {
    Lev L{};
    for (int d = 0; d < 3; ++d) {
        L.n[d] = atoi(a[d]);
        L.bc[d] = atoi(a[3 + d]);
        L.ih2[d] = 1.0 * L.n[d] * L.n[d];
        L.fih2[d] = (float)L.ih2[d];
        L.lih2[d] = (float)(L.ih2[d] - (double)L.fih2[d]);
    }
    L.cells = (long long)L.n[0] * L.n[1] * L.n[2];
    L.tz = std::min(8, L.n[2]);
    L.bx = (L.n[0] + TX - 1) / TX;
    L.by = (L.n[1] + TY - 1) / TY;
    L.bz = (L.n[2] + L.tz - 1) / L.tz;
    L.ctas = L.bx * L.by * L.bz;
    return L;
}

template <typename T>
static std::vector<T> take(FILE* f, size_t n) {
    std::vector<T> v(n);
    if (fread(v.data(), sizeof(T), n, f) != n) exit(4);
    return v;
}

template <typename E>
static int update(const Lev& L, double rr, double rmean, const char* in, const char* out) {
    const size_t C = (size_t)L.cells;
    FILE* f = fopen(in, "rb");
    if (!f) return 3;
    auto x = take<double>(f, C), r = take<double>(f, C);
    auto e = take<E>(f, C);
    fclose(f);
    unsigned counter = 0;
    std::vector<double> part(3 * (size_t)L.ctas);
    MgBuf<double> mb{};
    mb.x = x.data();
    mb.r = r.data();
    mb.counter = &counter;
    SliceCtl c{};
    c.status = ST_ITER;
    c.rr = rr;
    c.bb = 1e300;
    c.rmean = rmean;
    launch(L.ctas, [&] {
        k_dir_update<E>(L, mb, &c, e.data(), part.data(), 0.0, 40, (int)C, dir_log2(L.cells));
    });
    f = fopen(out, "wb");
    fwrite(x.data(), 8, C, f);
    fwrite(r.data(), 8, C, f);
    const double num[5] = {c.rr, c.sx, c.rmean, (double)c.status, (double)c.it_cur};
    fwrite(num, 8, 5, f);
    fclose(f);
    return 0;
}

static int cg(Lev L, int its, int more, const char* in, const char* out) {
    const size_t C = (size_t)L.cells;
    FILE* f = fopen(in, "rb");
    if (!f) return 3;
    auto code = take<uint8_t>(f, C);
    auto r = take<float>(f, C), d = take<float>(f, C), r2 = take<float>(f, C), zs = take<float>(f, C);
    fclose(f);
    L.fcode = code.data();
    std::vector<float> p[2], q(C, NAN), x(C, NAN), z(C);
    for (auto& v : p) v.assign(C, NAN);
    unsigned counter = 0;
    std::vector<double> part(2 * (size_t)L.ctas);
    MgBuf<float> mb{};
    mb.x = x.data();
    mb.r = r.data();
    mb.P[0] = p[0].data();
    mb.P[1] = p[1].data();
    mb.V[0] = q.data();
    mb.counter = &counter;
    SliceCtl c{};
    c.bb = 1e30;
    f = fopen(out, "wb");
    std::vector<double> num;
    for (int solve = 0; solve < 2; ++solve) {
        if (solve) r = r2, mb.r = r.data();
        c.o_steps = solve;
        c.it_cur = 0;
        const int n = solve ? more : its;
        for (int it = 0; it < n; ++it) {
            c.status = ST_ITER;
            for (size_t k = 0; k < C; ++k) z[k] = code[k] & FC_FLUID ? d[k] * r[k] : zs[k];
            launch(L.ctas, [&] { k_cg_dot<float>(L, mb, z.data(), &c, part.data()); });
            launch(L.ctas, [&] { k_cg_lap<float>(L, mb, z.data(), &c, part.data()); });
            launch(L.ctas, [&] { k_cg_update<float>(L, mb, &c, part.data(), 0.0, n); });
            const int want = it + 1 < n ? ST_ITER : ST_MAXIT;
            if (c.status != want || c.it_cur != it + 1) return 5;
        }
        fwrite(x.data(), 4, C, f);
        fwrite(r.data(), 4, C, f);
        num.push_back(c.rr);
        num.push_back(c.sx);
    }
    fwrite(num.data(), 8, num.size(), f);
    fclose(f);
    return 0;
}

int main(int argc, char** argv) {
    if (argc == 13 && !strcmp(argv[1], "update")) {
        const Lev L = level(argv + 3);
        const double rr = atof(argv[9]), rmean = atof(argv[10]);
        return argv[2][0] == 'f' ? update<float>(L, rr, rmean, argv[11], argv[12])
                                 : update<double>(L, rr, rmean, argv[11], argv[12]);
    }
    if (argc == 12 && !strcmp(argv[1], "cg"))
        return cg(level(argv + 2), atoi(argv[8]), atoi(argv[9]), argv[10], argv[11]);
    return 1;
}
