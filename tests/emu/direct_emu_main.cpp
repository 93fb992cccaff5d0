// Driver of the host emulation of the direct solve (test support): builds the
// plan and tables of a grid as the library does, runs the forward transforms,
// the columns and the inverse transforms of two states (the second one
// inactive), every CTA as host threads, and writes e.
//
// usage: direct_emu T nx ny nz bcx bcy bcz lx ly lz planes in.bin out.bin
//   planes: of a call, 0: the transforms one axis at a time; T: f, d, or m (an FP64
//   residual, FP32 transforms); in.bin: r, two states; out.bin: e, two states (the inactive
//   one's untouched zeros).

#include <functional>
#include <type_traits>

static void launch(int gx, int bx, int by, size_t smem, const std::function<void()>& body,
                   int states = 2) {
    const int n = bx * by;
    blockDim = EmuDim3{(unsigned)bx, (unsigned)by, 1};
    gridDim = EmuDim3{(unsigned)gx, (unsigned)states, 1};
    for (int st = 0; st < states; ++st)
        for (int c = 0; c < gx; ++c) {
            std::barrier<> bar(n);
            emu_cta_barrier = &bar;
            std::vector<unsigned char> sm(smem + 16, 0xff);  // NaN where nothing is written
            const size_t mis = (16 - (size_t)sm.data() % 16) % 16;
            emu_smem = sm.data() + mis;
            std::vector<std::thread> th;
            for (int t = 0; t < n; ++t)
                th.emplace_back([&, t]() {
                    threadIdx = EmuDim3{(unsigned)(t % bx), (unsigned)(t / bx), 0};
                    blockIdx = EmuDim3{(unsigned)c, (unsigned)st, 0};
                    body();
                    bar.arrive_and_drop();
                });
            for (auto& x : th) x.join();
        }
}

template <typename T, typename S>
static int run(char** argv) {
    int n[3], bc[3];
    double ih2[3];
    for (int a = 0; a < 3; ++a) {
        n[a] = atoi(argv[2 + a]);
        bc[a] = atoi(argv[5 + a]);
        const double h = atof(argv[8 + a]) / n[a];
        ih2[a] = 1.0 / (h * h);
    }
    DirPlan<T> P;
    const int planes = atoi(argv[11]);
    if (!dir_sizes<T>(n, bc[2] == BC_PERIODIC, planes ? planes : 500, P)) return 2;
    if (!planes && !dir_line_sizes<T>(P)) return 2;
    size_t off[5];
    std::vector<T> tab = dir_tables<T>(P, bc, ih2, off);
    P.rx[0] = tab.data() + off[0];
    P.rx[1] = tab.data() + off[1];
    P.ly[0] = tab.data() + off[2];
    P.ly[1] = tab.data() + off[3];
    P.col = tab.data() + off[4];
    const size_t N = (size_t)P.cells;
    std::vector<S> r(2 * N);
    std::vector<T> spec(2 * N, T(0)), e(2 * N, T(0));
    FILE* f = fopen(argv[12], "rb");
    if (!f || fread(r.data(), sizeof(S), 2 * N, f) != 2 * N) return 3;
    fclose(f);
    SliceCtl ctl[2] = {};
    ctl[0].status = ST_ITER;
    ctl[0].o_status = OS_REFINE;
    ctl[0].o_fsc = 4.0f;  // the scale FP32 residuals carry through the transforms
    ctl[1].o_fsc = 4.0f;
    if (sizeof(S) > sizeof(T)) {  // scaled from the residual's norm
        P.mode = DM_MIXED;
        ctl[0].o_status = OS_DONE;
        for (size_t q = 0; q < N; ++q) ctl[0].rr += double(r[q]) * double(r[q]);
    }
    ctl[1].status = ST_CONV;
    ctl[1].o_status = OS_DONE;
    const size_t smem = dir_smem_elems(P) * sizeof(T);
    auto xy = [&](auto inv, const auto* src, T* dst) {
        constexpr bool INV = decltype(inv)::value;
        auto go = [&](auto rb, auto nc) {
            launch(P.nz * P.xb, P.nt, 1, smem,
                   [&] { k_dir_xy<T, INV, decltype(rb)::value, decltype(nc)::value>(P, ctl, src, dst, 0); });
        };
        // one axis at a time: CTAs of each kernel take several blocks of lines
        auto x = [&] {
            launch(3, P.ntx, 1, dir_x_elems(P) * sizeof(T),
                   [&] { k_dir_x<T, INV>(P, ctl, src, dst, 0, 2); }, 1);
        };
        auto y = [&] {
            launch(2, P.nty, 1, dir_y_elems(P) * sizeof(T),
                   [&] { k_dir_y<T, INV>(P, ctl, spec.data(), 2); }, 1);
        };
        if (P.lines) {
            if (INV) y();
            x();
            if (!INV) y();
        } else {
            using One = std::integral_constant<int, 1>;
            using Two = std::integral_constant<int, 2>;
            using R4 = std::integral_constant<int, 4>;
            using R8 = std::integral_constant<int, 8>;
            if (P.rb == 16) go(std::integral_constant<int, 16>{}, Two{});
            else if (P.rb == 8) P.ncol == 2 ? go(R8{}, Two{}) : go(R8{}, One{});
            else P.ncol == 2 ? go(R4{}, Two{}) : go(R4{}, One{});
        }
    };
    xy(std::false_type{}, r.data(), spec.data());
    const int zg = (P.nx * P.ny + DIR_ZX - 1) / DIR_ZX;
    launch(zg, DIR_ZX, P.zc, 0, [&] {
        if (P.zm == DIR_ZC)
            k_dir_z<T, DIR_ZC>(P, ctl, spec.data());
        else
            k_dir_z<T, DIR_ZC_LONG>(P, ctl, spec.data());
    });
    xy(std::true_type{}, spec.data(), e.data());
    f = fopen(argv[13], "wb");
    fwrite(e.data(), sizeof(T), 2 * N, f);
    fclose(f);
    printf("%d %d %d %d %d\n", P.xb, P.cb, P.nt, P.zm, P.zc);
    return 0;
}

int main(int argc, char** argv) {
    if (argc != 14) return 1;
    return argv[1][0] == 'f' ? run<float, float>(argv)
                             : argv[1][0] == 'd' ? run<double, double>(argv) : run<float, double>(argv);
}
