// fx_line_host.cu -- the fixed-point line transforms compiled for the host:
// the library's own scale rules, conversions, register DFTs, twiddles and
// exchanges (fx.cuh, fx_line.cuh, fast.cuh, fast_fx.cuh), the threads of a
// line taken one after the other.
#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

#include <utility>
#include <vector>

// the device intrinsics those headers use
template <typename T, typename F> static __host__ __device__ T bits_as(F f) {
    T t;
    memcpy(&t, &f, sizeof(t));
    return t;
}
static __host__ __device__ long long round_ll(double x) {
    double r = floor(x + 0.5);
    if (x + 0.5 == r && fmod(r, 2.0) != 0.0) r -= 1.0;
    return (long long)(fabs(x) < 4503599627370496.0 ? r : x);
}
#define __double2hiint(x) ((int)(bits_as<long long>((double)(x)) >> 32))
#define __double2loint(x) ((int)bits_as<long long>((double)(x)))
#define __hiloint2double(h, l) (bits_as<double>((long long)(((unsigned long long)(unsigned)(h) << 32) | (unsigned)(l))))
#define __double_as_longlong(x) (bits_as<long long>((double)(x)))
#define __longlong_as_double(x) (bits_as<double>((long long)(x)))
#define __float_as_int(x) (bits_as<int>((float)(x)))
#define __int_as_float(x) (bits_as<float>((int)(x)))
#define __uint_as_float(x) (bits_as<float>((unsigned)(x)))
#define __clzll(x) ((x) == 0 ? 64 : __builtin_clzll((unsigned long long)(x)))
#define __double2ll_rn(x) round_ll(x)
#define __ll2double_rn(x) ((double)(x))
#define __ldg(p) (*(p))
// named by parts of the headers that are not called here
#define __ldcg(p) (*(p))
#define __umulhi(a, b) ((unsigned)(((unsigned long long)(a) * (b)) >> 32))
#define __syncthreads() ((void)0)
#define __syncwarp() ((void)0)
#define __shfl_sync(m, v, l) (v)
#define __shfl_xor_sync(m, v, l) (v)
#undef __device__
#define __device__ __attribute__((device)) __attribute__((host))
#include "fast_fx.cuh"

using namespace fsp;
using namespace fsp::fast;

namespace {

std::vector<fxw> roots(int n) {
    std::vector<fxw> w(n);
    for (int e = 0; e < n; ++e) {
        // exact on the axes, so that no factor is above 1
        const long double a = 2.0L * 3.14159265358979323846264338327950288L * e / n;
        const long long c = llroundl(ldexpl(4 * e == n || 4 * e == 3 * n ? 0.0L : cosl(a), 62));
        const long long s = llroundl(ldexpl(2 * e == n || e == 0 ? 0.0L : -sinl(a), 62));
        w[e] = fxw{fx_hi(c), fx_lo(c), fx_hi(s), fx_lo(s)};
    }
    return w;
}

// A line of a column pass on the shape of its length: in (n or n / 2 values)
// -> out (n), D = -1 with the upper half zero or D = +1.
template <int D, int n, int V, int L, int R1, int R2, int R3, bool HZ>
void line(const double *in, double *out, const fxw *tw) {
    constexpr int TPL = n / V, NT = R3 > 1 ? 2 : 1, RL = LastR<R1, R2, R3>::value, RH = HZ ? R1 / 2 : R1;
    using X = Fxc<n, V, L>;
    using F = Fst<D, n, V, L>;
    std::vector<cfx> v(n), buf(n * (L + 1));
    float s = 0.f;
    int h = 0;
    for (int t = 0; t < TPL; ++t)
        for (int k = 0; k < V / R1; ++k)
            for (int r = 0; r < RH; ++r) {
                const int p = t + k * TPL + r * (n / R1);
                v[t * V + k * R1 + r] = fx_raw(double2{in[2 * p], in[2 * p + 1]});
                fx_bound(v[t * V + k * R1 + r], s, h);
            }
    const FxScale sc = fx_scale<R1, R2, R3, HZ, 62>(s, h);
    for (int t = 0; t < TPL; ++t) {
        for (int k = 0; k < V / R1; ++k)
            for (int r = 0; r < RH; ++r) v[t * V + k * R1 + r] = fx_conv<true, false>(v[t * V + k * R1 + r], sc);
        F::template compute<R1, 1, HZ, false>(&v[t * V], t, tw);
    }
    for (int t = 0; t < TPL; ++t) X::template store_out<R1, 1>(buf.data(), &v[t * V], t, 0);
    for (int t = 0; t < TPL; ++t) {
        X::template load_in<R2>(&v[t * V], buf.data(), t, 0);
        F::template compute<R2, R1, false, false>(&v[t * V], t, tw);
    }
    if constexpr (R3 > 1) {
        for (int t = 0; t < TPL; ++t) X::template store_out<R2, R1>(buf.data(), &v[t * V], t, 0);
        for (int t = 0; t < TPL; ++t) {
            X::template load_in<R3>(&v[t * V], buf.data(), t, 0);
            F::template compute<R3, R1 * R2, false, false>(&v[t * V], t, tw);
        }
    }
    const FxOut<true, false> to(2 * NT - sc.ke, sc.bad);
    for (int t = 0; t < TPL; ++t)
        for (int k = 0; k < V / RL; ++k)
            for (int r = 0; r < RL; ++r) {
                const double2 q = to(v[t * V + k * RL + r]);
                const int p = t + k * TPL + r * (n / RL);
                out[2 * p] = q.x, out[2 * p + 1] = q.y;
            }
}
template <int n> void lines(int sign, int count, const double *in, double *out) {
    using K = CfgX<n>;
    const std::vector<fxw> tw = roots(n);
    for (int i = 0; i < count; ++i) {
        if (sign < 0)
            line<-1, n, K::V, K::L, K::R1, K::R2, K::R3, true>(in + 2LL * n * i, out + 2LL * n * i, tw.data());
        else
            line<+1, n, K::V, K::L, K::R1, K::R2, K::R3, false>(in + 2LL * n * i, out + 2LL * n * i, tw.data());
    }
}

// A line of the generic engine: 5s, 3s, 8s, a last 4 or 2.
template <int D, int R> void stage(std::vector<cfx> &v, int n, int Ns, const fxw *tw) {
    std::vector<cfx> o(n);
    for (int b = 0; b < n / R; ++b) {
        cfx q[R];
        const int j = b % Ns;
        for (int r = 0; r < R; ++r) q[r] = v[b + r * (n / R)];
        if (Ns > 1) {
            q[0] = tw_of<fx>::quarter(q[0]);
            for (int r = 1; r < R; ++r) q[r] = tw_of<fx>::template mul<D>(q[r], tw[r * j * (n / (Ns * R))]);
        }
        RD<fx, D>::template dft<R, false, false>(q);
        for (int r = 0; r < R; ++r) o[(b - j) * R + j + r * Ns] = q[r];
    }
    v = o;
}
template <int D> void generic_line(const Stages &st, const double *in, double *out, const fxw *tw) {
    const int n = st.n;
    std::vector<cfx> v(n);
    float s = 0.f;
    int h = 0;
    for (int p = 0; p < n; ++p) {
        v[p] = fx_raw(double2{in[2 * p], in[2 * p + 1]});
        fx_bound(v[p], s, h);
    }
    const int em = fx_em(h), eL = em - 16 + fx_clog2(1.5f * (float)tile_units(s, em) + 1e-30f);  // as tile_scale
    const FxScale sc{tile_ke(st, em, eL, 62), false, false};
    for (int p = 0; p < n; ++p) v[p] = fx_conv<true, false>(v[p], sc);
    int Ns = 1;
    for (int i = 0; i < st.n5; ++i, Ns *= 5) stage<D, 5>(v, n, Ns, tw);
    for (int i = 0; i < st.n3; ++i, Ns *= 3) stage<D, 3>(v, n, Ns, tw);
    for (int i = 0; i < st.n8; ++i, Ns *= 8) stage<D, 8>(v, n, Ns, tw);
    if (st.last == 4) stage<D, 4>(v, n, Ns, tw);
    if (st.last == 2) stage<D, 2>(v, n, Ns, tw);
    const FxOut<true, false> to(tile_div(st) - sc.ke, false);
    for (int p = 0; p < n; ++p) {
        const double2 q = to(v[p]);
        out[2 * p] = q.x, out[2 * p + 1] = q.y;
    }
}

}  // namespace

extern "C" {

// `count` lines of n complex doubles on the specialised shape of n; sign < 0:
// the forward transform of lines whose upper half is zero
int fx_lines(int n, int sign, int count, const double *in, double *out) {
    switch (n) {
    case 64: lines<64>(sign, count, in, out); return 0;
    case 96: lines<96>(sign, count, in, out); return 0;
    case 128: lines<128>(sign, count, in, out); return 0;
    case 192: lines<192>(sign, count, in, out); return 0;
    case 256: lines<256>(sign, count, in, out); return 0;
    case 384: lines<384>(sign, count, in, out); return 0;
    case 512: lines<512>(sign, count, in, out); return 0;
    case 1024: lines<1024>(sign, count, in, out); return 0;
    }
    return 1;
}
int fx_lines_generic(int n, int sign, int count, const double *in, double *out) {
    Stages st{n, 0, 0, 0, 0};
    int m = n;
    for (; m % 5 == 0; m /= 5) ++st.n5;
    for (; m % 3 == 0; m /= 3) ++st.n3;
    for (; m % 8 == 0; m /= 8) ++st.n8;
    if (m > 1) st.last = m;
    if (m != 1 && m != 2 && m != 4) return 1;
    const std::vector<fxw> tw = roots(n);
    for (int i = 0; i < count; ++i) {
        if (sign < 0)
            generic_line<-1>(st, in + 2LL * n * i, out + 2LL * n * i, tw.data());
        else
            generic_line<+1>(st, in + 2LL * n * i, out + 2LL * n * i, tw.data());
    }
    return 0;
}
}
