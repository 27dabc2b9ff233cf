"""The scalar helpers that build FP64 and FP32 values from their bits (fp64.cuh)
against CUDA's own conversions and extended precision on the host: the ends of the
ranges, subnormals, halfway cases, infinities and NaN."""
import native_program
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SOURCE = r'''
#include <cmath>
#include <cstdio>
#include <cstring>
#include <limits>
#include <random>
#include <vector>
#include "fp64.cuh"
using namespace sim;
typedef long double L;
template <class T> T of_bits(unsigned long long b) { T v; memcpy(&v, &b, sizeof v); return v; }
template <class T> bool same(T a, T b) { return (std::isnan(a) && std::isnan(b)) || memcmp(&a, &b, sizeof a) == 0; }

template <class In, class Out, class F> __global__ void k_map(const In* x, Out* y, int n, F f) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = f(x[i]);
}
template <class Out, class In, class F> std::vector<Out> map(const std::vector<In>& x, F f) {
    In* dx;
    Out* dy;
    std::vector<Out> y(x.size());
    SIM_CUDA(cudaMalloc(&dx, x.size() * sizeof(In)));
    SIM_CUDA(cudaMalloc(&dy, x.size() * sizeof(Out)));
    SIM_CUDA(cudaMemcpy(dx, x.data(), x.size() * sizeof(In), cudaMemcpyHostToDevice));
    k_map<<<(int)(x.size() + 255) / 256, 256>>>(dx, dy, (int)x.size(), f);
    SIM_CUDA(cudaMemcpy(y.data(), dy, x.size() * sizeof(Out), cudaMemcpyDeviceToHost));
    SIM_CUDA(cudaFree(dx));
    SIM_CUDA(cudaFree(dy));
    return y;
}
struct Widen { __device__ double operator()(float f) const { return widen(f); } };
struct WidenCuda { __device__ double operator()(float f) const { return (double)f; } };
struct Narrow { __device__ float operator()(double d) const { return narrow(d); } };
struct NarrowCuda { __device__ float operator()(double d) const { return (float)d; } };
struct Rsqrt { __device__ double operator()(double d) const { return rsqrt_nr(d); } };
struct Recip { template <class C> __device__ C operator()(C a) const { return crecip(a); } };
struct Scale { __device__ double operator()(double2 v) const { return scale2(v.x, (int)v.y); } };

std::mt19937_64 gen(1);
unsigned long long u64() { return gen(); }

// largest error of 1 / a in units of u = eps/2 of |1/a|, normwise; results below the
// normal range are allowed the last place of a subnormal in either component
template <class C, class R> double recip_error(const std::vector<C>& a, const std::vector<C>& y) {
    double worst = 0;
    for (size_t i = 0; i < a.size(); ++i) {
        const L s = std::max(std::fabs((L)a[i].x), std::fabs((L)a[i].y));
        const L x = a[i].x / s, z = a[i].y / s, d = (x * x + z * z) * s, ex = x / d, ey = -z / d;
        const L norm = std::sqrt(ex * ex + ey * ey);
        if (std::max(std::fabs(ex), std::fabs(ey)) > (L)std::numeric_limits<R>::max() / 2) {
            if (std::isnan(y[i].x) && std::isnan(y[i].y)) return INFINITY;  // overflow: infinite, not undefined
            continue;
        }
        L err = std::hypot((L)y[i].x - ex, (L)y[i].y - ey);
        const L tiny = 3 * (L)std::numeric_limits<R>::denorm_min();
        err = norm < 8 * (L)std::numeric_limits<R>::min() ? std::max<L>(0, err - tiny) : err;
        const double e = (double)(err / norm / ((L)std::numeric_limits<R>::epsilon() / 2));
        if (!(e <= worst)) worst = e;
    }
    return worst;
}

int main() {
    std::vector<float> f{0.f, -0.f, INFINITY, -INFINITY, NAN};
    for (int e = 0; e < 256; ++e)
        for (unsigned m : {0u, 1u, 2u, 0x400000u, 0x7ffffeu, 0x7fffffu})
            for (unsigned s : {0u, 1u}) f.push_back(of_bits<float>((unsigned long long)(s << 31 | (unsigned)e << 23 | m)));
    for (int i = 0; i < 200000; ++i) f.push_back(of_bits<float>(u64() & 0xffffffffu));
    int bad = 0;
    auto w = map<double>(f, Widen()), wc = map<double>(f, WidenCuda());
    for (size_t i = 0; i < f.size(); ++i) bad += !same(w[i], wc[i]);
    printf("widen %d\n", bad);

    std::vector<double> d{0.0, -0.0, INFINITY, -INFINITY, NAN};
    for (int e : {0, 1, 800, 872, 873, 874, 895, 896, 897, 898, 899, 1022, 1023, 1024, 1148, 1149, 1150, 1151, 2046, 2047})
        for (unsigned long long top : {0ull, 1ull, 2ull, 3ull, 0x7ffffeull, 0x7fffffull})
            for (unsigned long long low : {0ull, 1ull, 0xfffffffull, 0x10000000ull, 0x10000001ull, 0x1fffffffull})  // below, at and above half
                for (unsigned long long s : {0ull, 1ull}) d.push_back(of_bits<double>(s << 63 | (unsigned long long)e << 52 | top << 29 | low));
    for (int i = 0; i < 200000; ++i) {
        d.push_back(of_bits<double>(u64()));
        d.push_back(of_bits<double>((u64() & 0x800fffffffffffffull) | (880 + u64() % 290) << 52));
        d.push_back(of_bits<double>((u64() & 0x800fffffe0000000ull) | (880 + u64() % 290) << 52 | 0x10000000ull));
    }
    auto nr = map<float>(d, Narrow()), nc = map<float>(d, NarrowCuda());
    bad = 0;
    for (size_t i = 0; i < d.size(); ++i) bad += !same(nr[i], nc[i]);
    printf("narrow %d\n", bad);

    std::vector<double> r{1.0, 2.0, 4.0, std::nextafter(1.0, 0), std::nextafter(4.0, 0), std::nextafter(2.0, 0), 1.1e-280, 0.9e280};
    for (int i = 0; i < 400000; ++i) r.push_back(of_bits<double>((u64() & 0xfffffffffffffull) | (95 + u64() % 1855) << 52));
    auto rs = map<double>(r, Rsqrt());
    double worst = 0;
    for (size_t i = 0; i < r.size(); ++i) {
        const L ex = 1 / std::sqrt((L)r[i]);
        worst = std::fmax(worst, (double)(std::fabs(rs[i] - ex) / ex * 0x1p53L));
    }
    printf("rsqrt %.3f\n", worst);

    std::vector<double2> sc;
    for (int e : {0, 1, 2, 52, 1023, 2045, 2046})
        for (int k : {-2045, -1023, -53, -1, 0, 1, 53, 959, 1022})
            for (unsigned long long m : {0ull, 1ull, 0xfffffffffffffull})
                if (e + k <= 2046) sc.push_back(make_double2(of_bits<double>((unsigned long long)e << 52 | m), k));
    auto ss = map<double>(sc, Scale());
    bad = 0;
    for (size_t i = 0; i < sc.size(); ++i) {
        // (a result just below the normal range would round up into it)
        const L ex = std::ldexp((L)sc[i].x, (int)sc[i].y);
        bad += ss[i] != (double)(std::isnormal(sc[i].x) && ex >= (L)std::numeric_limits<double>::min() ? ex : 0);
    }
    printf("scale %d\n", bad);

    std::vector<double2> a;
    std::vector<float2> b;
    auto md = [&](int e) { return of_bits<double>((u64() & 0x800fffffffffffffull) | (unsigned long long)e << 52); };
    auto mf = [&](int e) { return of_bits<float>((u64() & 0x807fffffull) | (unsigned long long)e << 23); };
    for (int e = 0; e < 2047; ++e)
        for (int i = 0; i < 60; ++i) {
            a.push_back(make_double2(md(e), md((int)(u64() % (e + 1)))));
            a.push_back(make_double2(md(std::max(0, e - i)), md(e)));
        }
    for (int e = 0; e < 255; ++e)
        for (int i = 0; i < 400; ++i) {
            b.push_back(make_float2(mf(e), mf((int)(u64() % (e + 1)))));
            b.push_back(make_float2(mf(std::max(0, e - i % 30)), mf(e)));
        }
    for (double2 v : {make_double2(1, 0), make_double2(0, -1), make_double2(0x1p-1074, 0), make_double2(0, 0x1p1023), make_double2(1e308, 1e308)}) a.push_back(v);
    printf("recip %.3f\n", recip_error<double2, double>(a, map<double2>(a, Recip())));
    printf("recipf %.3f\n", recip_error<float2, float>(b, map<float2>(b, Recip())));
    std::vector<double2> odd{make_double2(INFINITY, 1), make_double2(-3, -INFINITY), make_double2(INFINITY, INFINITY), make_double2(NAN, 1)};
    for (double2 v : map<double2>(odd, Recip())) printf("odd %g %g\n", std::fabs(v.x), std::fabs(v.y));
}
'''


def test_helpers_against_cuda_and_extended_precision(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    rows = [r.split() for r in native_program.run(tmp_path, SOURCE).splitlines()]
    got = {r[0]: float(r[1]) for r in rows if r[0] != "odd"}
    print(got)
    assert got["widen"] == got["narrow"] == got["scale"] == 0
    # in units of u: d y0 rounded, then the sum y0 + y0 t (1/2 + ..): u/2 + u, and the
    # series' remainder (2^-60)
    assert got["rsqrt"] <= 1.6
    # |a|^2 two roundings, its reciprocal one, the product with the component one;
    # second-order terms
    assert got["recip"] <= 4.1
    assert got["recipf"] <= 4.1
    odd = [r[1:] for r in rows if r[0] == "odd"]
    assert odd[:3] == [["0", "0"]] * 3 and odd[3] == ["nan", "nan"]
