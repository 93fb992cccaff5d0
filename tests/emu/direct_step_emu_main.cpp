// Driver of the host emulation of the FP32+refine step kernels around the
// direct solve (test support): k_dir_load_p, k_dir_start (with and without the
// stored velocity), k_dir_refine and k_dir_correct, one state, every CTA as
// host threads.
//
// usage: direct_step_emu nx ny nz bcx bcy bcz lbox dt steps tile_z in.bin out.bin
//   steps: applications already made when k_dir_refine runs (its slot and the
//   folded one follow).  in.bin (cells C, faces Fu, Fv, Fw): p [C] FP64, then
//   FP32: increments, velocities [Fu, Fv, Fw each], ring [4][C].
//   out.bin: FP32 start without u: r_hi r_lo; start with u: r_hi r_lo; refine:
//   r_hi r_lo base_hi base_lo; correct: u v w w_hi w_lo q_hi q_lo; FP64: p_out,
//   then o_bb, o_rr (start with u), o_rr, sx (refine), o_steps, o_status.

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

int main(int argc, char** argv) {
    if (argc != 13) return 1;
    int n[3], bc[3];
    Lev L{};
    const double lbox = atof(argv[7]), dt = atof(argv[8]);
    const int steps = atoi(argv[9]);
    FF ih[3];
    auto ff = [](double d) { return FF{(float)d, (float)(d - (double)(float)d)}; };
    for (int a = 0; a < 3; ++a) {
        n[a] = atoi(argv[1 + a]);
        bc[a] = atoi(argv[4 + a]);
        const double h = lbox / n[a];
        L.n[a] = n[a];
        L.bc[a] = bc[a];
        L.ih2[a] = 1.0 / (h * h);
        L.fih2[a] = (float)L.ih2[a];
        L.lih2[a] = (float)(L.ih2[a] - (double)L.fih2[a]);
        ih[a] = ff(1.0 / h);
    }
    L.cells = (long long)n[0] * n[1] * n[2];
    const size_t C = (size_t)L.cells;
    size_t F[3];
    for (int c = 0; c < 3; ++c) {
        F[c] = 1;
        for (int a = 0; a < 3; ++a) F[c] *= n[a] + (c == a && bc[a] != BC_PERIODIC ? 1 : 0);
    }
    std::vector<double> p(C), pout(C, -1.0);
    std::vector<float> inc[3], vel[3], ring(4 * C);
    FILE* f = fopen(argv[11], "rb");
    if (!f) return 3;
    bool ok = fread(p.data(), 8, C, f) == C;
    for (auto* v : {inc, vel})
        for (int c = 0; c < 3; ++c) {
            v[c].resize(F[c]);
            ok = ok && fread(v[c].data(), 4, F[c], f) == F[c];
        }
    ok = ok && fread(ring.data(), 4, 4 * C, f) == 4 * C;
    fclose(f);
    if (!ok) return 4;
    const DirTile t = dir_tile_of(n, 1, atoi(argv[10]));
    std::vector<float> a[8];
    for (auto& v : a) v.assign(C, 0.0f);
    FFBuf fb{a[0].data(), a[1].data(), a[2].data(), a[3].data(),
             a[4].data(), a[5].data(), a[6].data(), a[7].data()};
    std::vector<double> part((size_t)t.ctas * 7);
    unsigned counter = 0;
    SliceCtl ctl{};
    FILE* out = fopen(argv[12], "wb");
    auto put = [&](const std::vector<float>& v) { fwrite(v.data(), 4, v.size(), out); };
    std::vector<double> num;
    launch((int)((C + NTHREADS - 1) / NTHREADS), [&] { k_dir_load_p((long long)C, p.data(), fb); });
    const FF idt = ff(1.0 / dt);
    launch(t.ctas, [&] {
        k_dir_start<false>(L, t, &ctl, inc[0].data(), inc[1].data(), inc[2].data(), nullptr,
                           nullptr, nullptr, fb.w_hi, fb.w_lo, fb, idt, ih[0], ih[1], ih[2],
                           (long long)F[0], (long long)F[1], (long long)F[2], part.data(),
                           &counter, 1e-20, 40);
    });
    put(a[2]);
    put(a[3]);
    launch(t.ctas, [&] {
        k_dir_start<true>(L, t, &ctl, inc[0].data(), inc[1].data(), inc[2].data(), vel[0].data(),
                          vel[1].data(), vel[2].data(), fb.w_hi, fb.w_lo, fb, idt, ih[0], ih[1],
                          ih[2], (long long)F[0], (long long)F[1], (long long)F[2], part.data(),
                          &counter, 1e-20, 40);
    });
    put(a[2]);
    put(a[3]);
    num.push_back(ctl.o_bb);
    num.push_back(ctl.o_rr);
    ctl.o_steps = steps;
    launch(t.ctas, [&] {
        k_dir_refine(L, t, &ctl, ring.data(), (long long)C, fb.w_hi, fb.w_lo, fb, part.data(),
                     &counter, 1e-20, 40);
    });
    for (int q : {2, 3, 4, 5}) put(a[q]);
    num.push_back(ctl.o_rr);
    num.push_back(ctl.sx);
    num.push_back(ctl.o_steps);
    num.push_back(ctl.o_status);
    const float3 dth{(float)(dt * (double)ih[0].hi), (float)(dt * (double)ih[1].hi),
                     (float)(dt * (double)ih[2].hi)};
    launch(t.ctas, [&] {
        k_dir_correct<true>(L, t, &ctl, inc[0].data(), inc[1].data(), inc[2].data(),
                            vel[0].data(), vel[1].data(), vel[2].data(), fb, fb.w_hi, fb.w_lo,
                            ring.data(), (long long)C, fb.p_hi, fb.p_lo, pout.data(), dth,
                            (long long)F[0], (long long)F[1], (long long)F[2]);
    });
    for (int c = 0; c < 3; ++c) put(vel[c]);
    for (int q : {0, 1, 6, 7}) put(a[q]);
    fwrite(pout.data(), 8, C, out);
    fwrite(num.data(), 8, num.size(), out);
    fclose(out);
    return 0;
}
