"""Rules and arithmetic of the library that the CPU can check. CPU only."""
from tests import host_cc


def test_only_memory_of_the_graphs_device_is_used_in_place(tmp_path):
    """Kernels take a caller's array in place only from their own device (or managed memory) and only
    aligned to its elements; a peer's memory, host memory and a byte offset are copied. An id array
    that shares bytes with a result is told apart from one that ends where the result begins."""
    out = host_cc.run(tmp_path, r"""
int main()
{
    auto at = [](uintptr_t a) { return reinterpret_cast<const void*>(a); };
    const cudaMemoryType D = cudaMemoryTypeDevice, M = cudaMemoryTypeManaged, H = cudaMemoryTypeHost,
                         U = cudaMemoryTypeUnregistered;
    printf("%d%d%d", rd::usable_in_place(D, 0, 0, at(4096), 8), rd::usable_in_place(D, 2, 2, at(4104), 8),
           rd::usable_in_place(M, 1, 0, at(4096), 8));
    printf("%d%d%d%d ", rd::usable_in_place(D, 1, 0, at(4096), 8), rd::usable_in_place(D, 0, 1, at(4096), 8),
           rd::usable_in_place(H, 0, 0, at(4096), 8), rd::usable_in_place(U, 0, 0, at(4096), 8));
    printf("%d%d%d ", rd::usable_in_place(D, 0, 0, at(4100), 8), rd::usable_in_place(D, 0, 0, at(4100), 4),
           rd::usable_in_place(M, 0, 0, at(4098), 4));
    printf("%d%d%d%d", rd::ranges_overlap(at(4096), 16, at(4108), 4), rd::ranges_overlap(at(4096), 16, at(4112), 4),
           rd::ranges_overlap(at(4112), 4, at(4096), 17), rd::ranges_overlap(at(4096), 16, nullptr, 4));
}
""", headers=("rd_internal.cuh",))
    assert out == "1110000 010 1010"


def test_packed_double_float_rounds_as_the_scalar_operations(tmp_path):
    """The row epilogue's packed arithmetic (two columns an operation) is the scalar double-float
    arithmetic bit for bit -- every product normalised before it goes into a sum or another product --
    and so are the accumulations; 200,000 random operands of mixed size and sign."""
    out = host_cc.run(tmp_path, r"""
using namespace rd;
int main()
{
    std::mt19937_64 g(12);
    auto num = [&]() {
        const double m = std::uniform_real_distribution<double>(-1.0, 1.0)(g);
        return df64(std::ldexp(m, (int)(g() % 24) - 16));
    };
    auto same = [](df64 a, df64 b) { return a.hi == b.hi && a.lo == b.lo; };
    long bad = 0;
    for (int i = 0; i < 200000; ++i) {
        const df64 invd = num(), du = num();
        df64 acc[2] = {num(), num()}, bt[2] = {num(), num()}, qp[2] = {num(), num()}, qc[2] = {num(), num()};
        df64 sa[2] = {num(), num()}, sb[2] = {num(), num()}, sc[2] = {num(), num()};
        const df64x2 w2 = df_row(invd, df_pack(acc[0], acc[1]), df_pack(bt[0], bt[1]), df_pack(qp[0], qp[1]));
        df64x2 sa2 = df_pack(sa[0], sa[1]), sb2 = df_pack(sb[0], sb[1]), sc2 = df_pack(sc[0], sc[1]);
        df_row_sums(du, w2, df_pack(qc[0], qc[1]), sa2, sb2, sc2);
        df64 w[2], a[2], b[2], c[2], x[2] = {acc[0], acc[1]}, y[2] = {acc[0], acc[1]};
        df_unpack(w2, w[0], w[1]);
        df_unpack(sa2, a[0], a[1]);
        df_unpack(sb2, b[0], b[1]);
        df_unpack(sc2, c[0], c[1]);
        acc_mul_add_w(x, bt[0].hi, df_pack(qp[0], qp[1]));
        acc_add(y, df_pack(qp[0], qp[1]));
        for (int k = 0; k < 2; ++k) {
            const df64 ws = invd * acc[k] - bt[k] * qp[k], dw = du * ws;
            df64 xs = acc[k], ys = acc[k];
            acc_mul_add_w(xs, bt[0].hi, qp[k]);
            acc_add(ys, qp[k]);
            bad += !(same(w[k], ws) && same(a[k], sa[k] + dw * qc[k]) && same(b[k], sb[k] + dw * ws) &&
                     same(c[k], sc[k] + dw) && same(x[k], xs) && same(y[k], ys));
        }
    }
    printf("%ld", bad);
}
""")
    assert out == "0"


def test_error_estimate_of_increments_of_any_size(tmp_path):
    """The geometric tail estimate against its definition in long double, for increments that fall (or
    rise) at any ratio from their first size to the last denormal: no NaN, and the same value."""
    out = host_cc.run(tmp_path, r"""
int main()
{
    std::mt19937_64 g(5);
    double worst = 0.0;
    long n = 0, bad = 0;
    for (double ratio : {1e-3, 0.3, 0.499, 0.5, 0.501, 0.6, 0.9, 0.99, 0.9999, 1.0, 1.2})
        for (int k = 0; k < 4000; ++k) {
            // a stretch that starts at 2^-1074 .. 1, its ratios a little uneven
            double i[4];
            i[3] = std::ldexp(1.0 + (double)(g() >> 12) * 0x1p-52, -(int)(g() % 1075));
            for (int q = 2; q >= 0; --q) i[q] = i[q + 1] * ratio * (1.0 + 1e-3 * ((double)(g() % 2001) - 1000.0) * 1e-3);
            const double S = 0.5 + (double)(g() % 1000);
            const double est = rd::tail_estimate(i[0], i[1], i[2], i[3], S);
            long double rho = 0.5L;
            for (int q = 0; q < 3; ++q)
                if (i[q + 1] != 0.0) rho = std::fmax(rho, (long double)i[q] / (long double)i[q + 1]);
                else if (i[q] != 0.0) rho = INFINITY;
            const long double ref = rho < 1.0L ? (long double)i[0] * rho / ((1.0L - rho) * (1.0L - rho)) / S : INFINITY;
            ++n;
            if (std::isnan(est) || std::isinf(est) != std::isinf((double)ref)) { ++bad; continue; }
            if (std::isinf(est)) continue;
            // the last digits of a denormal estimate are its spacing's; (1 - rho)^-2 magnifies rounding
            const long double tol = 0x1p-1073L + std::fabs(ref) * 16 * 0x1p-52L / (rho < 1.0L ? 1.0L - rho : 1.0L);
            worst = std::fmax(worst, (double)(std::fabs((long double)est - ref) / tol));
        }
    printf("%ld %ld %d", n, bad, worst <= 1.0);
}
""", headers=("scalars.cuh",))
    assert out == "44000 0 1"


def test_root_and_inverse_within_rounding(tmp_path):
    """beta and 1/beta from one reciprocal square root: with that root off by up to two units in its last place
    either way (CUDA states one), both come out within one unit in the last place of the root and of the
    reciprocal of the root as rounded (what a square root and a division give within half a unit), over
    the whole range of exponents."""
    out = host_cc.run(tmp_path, r"""
int main()
{
    std::mt19937_64 g(7);
    double worst_root = 0.0, worst_inv = 0.0;
    for (int i = 0; i < 300000; ++i) {
        const double x = std::ldexp(1.0 + (double)(g() >> 12) * 0x1p-52, (int)(g() % 2040) - 1019);
        rsqrt_off = (int)(g() % 5) - 2;
        double root, inv;
        rd::root_and_inverse(x, &root, &inv);
        const long double s = std::sqrt((long double)x), q = 1.0L / root;  // the reciprocal of beta as rounded
        worst_root = std::fmax(worst_root, (double)(std::fabs(root - s) / (std::nextafter((double)s, INFINITY) - (double)s)));
        worst_inv = std::fmax(worst_inv, (double)(std::fabs(inv - q) / (std::nextafter((double)q, INFINITY) - (double)q)));
    }
    double root, inv;
    rd::root_and_inverse(-1e-20, &root, &inv);
    const bool neg = root == 0.0;
    rd::root_and_inverse(4e-310, &root, &inv);
    printf("%d %d %d %d", worst_root <= 1.0, worst_inv <= 1.0, neg, root == std::sqrt(4e-310));
}
""", headers=("scalars.cuh",))
    assert out == "1 1 1 1"
