// fast_fx.cuh -- the FP64 solve passes P1..P5 in 64-bit fixed point (fx.cuh):
// arrays, spectrum and results are doubles, the transform of each line runs
// in integers at the line's own scale.
//
// A kernel loads its line's doubles, reduces their 1-norm and largest
// exponent over the threads of the line, converts, transforms, and converts
// back on the store.  P3 does so once more in the middle: the products with
// the spectrum are rescaled before the inverse.  A line that holds an
// infinity or a NaN comes out as NaN, as it does in floating point.
#pragma once
#include "fast.cuh"
#include "fx_line.cuh"

namespace fsp {
namespace fast {

// Bound on every stage's output of schedule R1, R2, R3 (first radix with half
// its inputs zero if HZ): modulus <= 2^B (61, or 62 where nothing but twiddles
// and the radices' own factors comes after), where the inputs' components are
// below 2^em, the 1-norm is below 2^eL, and each twiddled stage divides by 4.
template <int R1, int R2, int R3, bool HZ, int B> __device__ __forceinline__ int fx_ke(int em, int eL) {
    constexpr int g0 = fx_grow(HZ ? R1 / 2 : R1), g1 = g0 + fx_grow(R2), g2 = g1 + fx_grow(R3);
    int eb = max(min(em + 1 + g0, eL), min(em + 1 + g1, eL) - 2);
    if (R3 > 1) eb = max(eb, min(em + 1 + g2, eL) - 4);
    return B - eb;
}
template <int R1, int R2, int R3, bool HZ, int B> __device__ __forceinline__ FxScale fx_scale(float l1, int hmax) {
    constexpr int cnt = fx_grow(HZ ? R1 / 2 : R1) + fx_grow(R2) + fx_grow(R3) + 1;
    FxScale s;
    const int em = fx_em(hmax);
    s.bad = (hmax >> 20) == 0x7ff;
    s.any = fx_far(em);
    const int eL = s.any ? em + cnt : fx_clog2(1.5f * l1);
    s.ke = fx_ke<R1, R2, R3, HZ, B>(em, eL);
    return s;
}

// Sum of s and maxima of h and m over the threads of each line (thread = t L + l).
// sm: NTH / 32 * L entries, used once per kernel.
template <int L, int NTH> __device__ __forceinline__ void fx_reduce(float &s, int &h, int &m, int4 *sm) {
    constexpr int NW = NTH / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, l = threadIdx.x % L;
#pragma unroll
    for (int o = L; o < 32; o *= 2) {
        s += __shfl_xor_sync(0xffffffffu, s, o);
        h = max(h, __shfl_xor_sync(0xffffffffu, h, o));
        m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    }
    if constexpr (NW == 1) {
        __syncwarp();
    } else {
        if (lane < L) sm[warp * L + l] = make_int4(__float_as_int(s), h, m, 0);
        __syncthreads();
        s = 0.f;
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            const int4 q = sm[w * L + l];
            s += __int_as_float(q.x);
            h = max(h, q.y);
            m = max(m, q.z);
        }
    }
}
template <int L, int NTH> __device__ __forceinline__ void fx_reduce(float &s, int &h, int4 *sm) {
    int m = 0;
    fx_reduce<L, NTH>(s, h, m, sm);
}

template <int D, int n, int V, int L> struct Fst {
    static constexpr int TPL = n / V, LD = L + 1;
    template <int R, int Ns, bool HZ, bool HO>
    static __device__ __forceinline__ void compute(cfx *v, int t, const fxw *__restrict__ tw) {
        static_assert(V % R == 0, "radix must divide the values per thread");
        StaticFor<0, V / R>::run([&](auto kc) {
            constexpr int k = decltype(kc)::value;
            if constexpr (Ns > 1) {
                const unsigned j = (unsigned)(t + k * TPL) % (unsigned)Ns;
                constexpr int tws = n / (Ns * R);
                v[k * R].x = fx_quarter(v[k * R].x), v[k * R].y = fx_quarter(v[k * R].y);
#pragma unroll
                for (int r = 1; r < R; ++r) {
                    const int4 q = __ldg(reinterpret_cast<const int4 *>(tw) + r * j * tws);
                    v[k * R + r] = fx_twiddle<D>(v[k * R + r], fxw{q.x, q.y, q.z, q.w});
                }
            }
            RD<fx, D>::template dft<R, HZ, HO>(v + k * R);
        });
    }
};

// The exchanges between stages.  With 8 or more lines a quarter warp (what
// shared memory serves at once, 8 lanes of 16 bytes) stays within one
// position and the pitch L + 1 does.  With 4 lines it covers two positions of
// consecutive threads: a pitch of 5 would make every access a two-way
// conflict, so the pitch is 4 and a position's lowest bit is flipped where
// bits 3 and 4 differ, which puts positions 8 or 16 apart (the first stage's
// stores) into different halves of a 128-byte row and leaves neighbours
// there.  The flip depends on t and compile-time constants alone, so the
// offsets of a thread's accesses stay immediates.  FP64 N = 256 1.95 -> 1.90
// ms, N = 512 18.8 -> 18.0.
template <int n, int V, int L> struct Fxc : Stg<fx, +1, n, V, L> {
    static constexpr size_t smem = sizeof(cfx) * n * (L + 1);
};
template <int n, int V> struct Fxc<n, V, 4> {
    static constexpr int TPL = n / V;
    static constexpr size_t smem = sizeof(cfx) * n * 4;
    static_assert(TPL % 32 == 0, "t alone decides the flips");
    template <int R, int Ns> static __device__ __forceinline__ void store_out(cfx *buf, const cfx *v, int t, int l) {
        static_assert((Ns == 1 && (R == 8 || R == 16)) || (R == 8 && (Ns == 8 || Ns == 16)), "flips worked out for these");
        // position (t + k TPL - j) R + j + r Ns, j = t mod Ns; the flip is g,
        // for odd h(r) 1 - g, with h a constant of r
        const int j = t % Ns;
        const int g = Ns == 1 ? (R == 8 ? (t ^ (t >> 1)) & 1 : t & 1) : Ns == 16 ? (j >> 3) & 1 : 0;
        const int at = ((t - j) * R + j) * 4 + l;
        StaticFor<0, V / R>::run([&](auto kc) {
            constexpr int k = decltype(kc)::value;
            StaticFor<0, R>::run([&](auto rc) {
                constexpr int r = decltype(rc)::value, c = k * TPL * R + r * Ns;
                constexpr int h = Ns == 1 ? (r >> 3) & 1 : Ns == 16 ? r & 1 : (r ^ (r >> 1)) & 1;
                const int f = h ? 1 - g : g;
                if constexpr (Ns == 1)  // the lowest bit of the position is r's
                    buf[at + c * 4 + (r & 1 ? -4 * f : 4 * f)] = v[k * R + r];
                else  // ... is j's
                    buf[(at ^ (f * 4)) + c * 4] = v[k * R + r];
            });
        });
    }
    template <int R> static __device__ __forceinline__ void load_in(cfx *v, const cfx *buf, int t, int l) {
        static_assert((n / R) % 32 == 0, "t alone decides the flip");
        const cfx *b = buf + ((t ^ (((t >> 3) ^ (t >> 4)) & 1)) * 4 + l);
#pragma unroll
        for (int k = 0; k < V / R; ++k)
#pragma unroll
            for (int r = 0; r < R; ++r) v[k * R + r] = b[(k * TPL + r * (n / R)) * 4];
    }
};

// stages 1.. of the schedule after stage 0 in registers (run_rest of fast.cuh)
template <int D, int n, int V, int L, int R1, int R2, int R3, bool HO_LAST>
__device__ __forceinline__ void fx_rest(cfx *v, cfx *buf, int t, int l, const fxw *tw, bool first_sync) {
    using X = Fxc<n, V, L>;
    using F = Fst<D, n, V, L>;
    if (first_sync) __syncthreads();
    X::template store_out<R1, 1>(buf, v, t, l);
    __syncthreads();
    X::template load_in<R2>(v, buf, t, l);
    if constexpr (R3 == 1) {
        F::template compute<R2, R1, false, HO_LAST>(v, t, tw);
    } else {
        F::template compute<R2, R1, false, false>(v, t, tw);
        __syncthreads();
        X::template store_out<R2, R1>(buf, v, t, l);
        __syncthreads();
        X::template load_in<R3>(v, buf, t, l);
        F::template compute<R3, R1 * R2, false, HO_LAST>(v, t, tw);
    }
}

// Column passes: tiles, geometry and Nyquist blocks as in fast_col_body.inc.
template <int n, int V, int L, int R1, int R2, int R3, int MODE, bool RG, int MINB>
__global__ void __launch_bounds__(L *(n / V), MINB) k_fx_col(const ColArgs a) {
    pdl_wait();
    using G = ColGeo<n, MODE>;
    constexpr int TPL = n / V, N = G::N, NTH = L * TPL;
    constexpr int RL = LastR<R1, R2, R3>::value, NT = R3 > 1 ? 2 : 1;
    const long long IN_POS = RG ? a.in_pos : G::IN_POS, IN_BATCH = RG ? a.in_batch : G::IN_BATCH;
    const long long OUT_POS = RG ? a.out_pos : G::OUT_POS, OUT_BATCH = RG ? a.out_batch : G::OUT_BATCH;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cfx *buf = reinterpret_cast<cfx *>(smem_raw);
    __shared__ int4 red[G::ZL ? 2 : 1][(NTH / 32) * L];
    const int l = threadIdx.x % L, t = threadIdx.x / L;
    int line;
    long long bt;
    if constexpr (!RG) {
        constexpr int X = G::ZL ? 2 : 1;
        if ((int)blockIdx.y >= X) {
            line = blockIdx.x * L + l;
            bt = blockIdx.y - X;
        } else {
            line = N;
            bt = ((long long)blockIdx.y * (N / L) + blockIdx.x) * L + l;
        }
    } else {
        if ((int)blockIdx.y >= a.xrows) {
            line = blockIdx.x * L + l;
            bt = blockIdx.y - a.xrows;
        } else {
            const long long q = (long long)blockIdx.y * gridDim.x + blockIdx.x;
            if (q * L >= a.nbatch) return;  // the whole block: before any barrier
            line = a.nlines - 1;
            bt = q * L + l;
        }
    }
    const fxw *tw = reinterpret_cast<const fxw *>(a.tw);
    const double2 *in_t = reinterpret_cast<const double2 *>(a.in) + bt * IN_BATCH + line + (long long)t * IN_POS;
    double2 *out_t = reinterpret_cast<double2 *>(a.out) + bt * OUT_BATCH + line + (long long)t * OUT_POS;
    constexpr bool HZ0 = MODE != COL_INV;
    constexpr int D0 = MODE == COL_INV ? +1 : -1, RH = HZ0 ? R1 / 2 : R1;
    cfx v[V];
    float s = 0.f;
    int h = 0;
    StaticFor<0, V / R1>::run([&](auto kc) {
        constexpr int k = decltype(kc)::value;
        StaticFor<0, RH>::run([&](auto rc) {
            constexpr int r = decltype(rc)::value;
            constexpr long long c = k * TPL + r * (n / R1);
            v[k * R1 + r] = fx_raw(__ldcg(in_t + c * IN_POS));
        });
    });
    StaticFor<0, V / R1>::run([&](auto kc) {
        constexpr int k = decltype(kc)::value;
#pragma unroll
        for (int r = 0; r < RH; ++r) fx_bound(v[k * R1 + r], s, h);
    });
    fx_reduce<L, NTH>(s, h, red[0]);
    const FxScale sc = fx_scale<R1, R2, R3, HZ0, G::ZL ? 61 : 62>(s, h);
#pragma unroll
    for (int k = 0; k < V / R1; ++k)
#pragma unroll
        for (int r = 0; r < RH; ++r) v[k * R1 + r] = fx_conv<true, MODE != COL_INV>(v[k * R1 + r], sc);
    Fst<D0, n, V, L>::template compute<R1, 1, HZ0, false>(v, t, tw);
    fx_rest<D0, n, V, L, R1, R2, R3, MODE == COL_INV>(v, buf, t, l, tw, false);

    if constexpr (G::ZL) {
        const int eo = 2 * NT - sc.ke;
        const long long S_POS = RG ? a.s_pos : G::S_POS, S_BATCH = RG ? a.s_batch : G::S_BATCH;
        const int HB = RG ? a.half_b : N;
        const int fy = (int)bt <= HB ? (int)bt : 2 * HB - (int)bt;
        const double *Sy = reinterpret_cast<const double *>(a.S) + (long long)fy * S_BATCH + line;
        float s2 = 0.f, m2 = 0.f;
        int hS = 0;
        StaticFor<0, V / RL>::run([&](auto kc) {
            constexpr int k = decltype(kc)::value;
            StaticFor<0, RL>::run([&](auto rc) {
                constexpr int r = decltype(rc)::value, i = k * RL + r, c = k * TPL + r * (n / RL);
                const int p = t + c, fz = p <= N ? p : n - p;
                fx_bound_mul(v[i], __ldg(Sy + (long long)fz * S_POS), s2, m2, hS);
            });
        });
        int mi = __float_as_int(m2);
        fx_reduce<L, NTH>(s2, hS, mi, red[1]);
        constexpr int R1i = R3 > 1 ? R3 : R2, R2i = R3 > 1 ? R2 : R1, R3i = R3 > 1 ? R1 : 1;
        constexpr int cnt = fx_grow(R1i) + fx_grow(R2i) + fx_grow(R3i);
        const int eS = fx_es(hS);  // else |v| < 2^61 alone
        const bool near = fx_near(eS), bad = sc.bad || eS == 1025;
        const int em = near ? fx_clog2(1.1f * __int_as_float(mi)) + 32 : 61 + eS;  // moduli < 2^em
        const int eL = near ? fx_clog2(1.1f * s2) + 32 : em + cnt;
        const int ke = min(fx_ke<R1i, R2i, R3i, false, 62>(em - 1, eL), 60 - em);
        // the field's odd spectrum (COL_FMO): -i S, negated past the fold in
        // z (odd = 1) or k_y (odd = 2)
        const int flip_b = MODE == COL_FMO && a.odd == 2 && (int)bt > HB ? -1 : 0;
        const int flip_z = MODE == COL_FMO && a.odd == 1 ? -1 : 0;
        StaticFor<0, V / RL>::run([&](auto kc) {
            constexpr int k = decltype(kc)::value;
            StaticFor<0, RL>::run([&](auto rc) {
                constexpr int r = decltype(rc)::value, i = k * RL + r, c = k * TPL + r * (n / RL);
                const int p = t + c, fz = p <= N ? p : n - p;
                const cfx q = fx_mul_s(v[i], __ldg(Sy + (long long)fz * S_POS), ke,
                                       MODE == COL_FMO ? flip_b ^ (p > N ? flip_z : 0) : 0, eS > -900);
                v[i] = MODE == COL_FMI ? q : cfx{q.y, -q.x};
            });
        });
        Fst<+1, n, V, L>::template compute<R1i, 1, false, false>(v, t, tw);
        fx_rest<+1, n, V, L, R1i, R2i, R3i, true>(v, buf, t, l, tw, true);
        const FxOut<true, true> out(eo - ke + 2 * NT, bad);
        constexpr int RF = R1;
        StaticFor<0, V / RF>::run([&](auto kc) {
            constexpr int k = decltype(kc)::value;
            StaticFor<0, RF / 2>::run([&](auto rc) {
                constexpr int r = decltype(rc)::value;
                constexpr long long c = k * TPL + r * (n / RF);
                out_t[c * OUT_POS] = out(v[k * RF + r]);
            });
        });
    } else {
        constexpr bool HO = MODE == COL_INV;
        const FxOut<HO, true> out(2 * NT - sc.ke, sc.bad);
        StaticFor<0, V / RL>::run([&](auto kc) {
            constexpr int k = decltype(kc)::value;
            StaticFor<0, HO ? RL / 2 : RL>::run([&](auto rc) {
                constexpr int r = decltype(rc)::value;
                constexpr long long c = k * TPL + r * (n / RL);
                out_t[c * OUT_POS] = out(v[k * RL + r]);
            });
        });
    }
}

// P1: k_fast_r2c in fixed point.
template <int N, int V, int L, int R1, int R2, int R3>
__global__ void __launch_bounds__(L *(N / V)) k_fx_r2c(const RowArgs a) {
    pdl_wait();
    constexpr int TPL = N / V, LD = L + 1, NTH = L * TPL, H = N / 2;
    constexpr int RL = LastR<R1, R2, R3>::value, NT = R3 > 1 ? 2 : 1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cfx *buf = reinterpret_cast<cfx *>(smem_raw);
    double2 *dbuf = reinterpret_cast<double2 *>(smem_raw);
    __shared__ int4 red[(NTH / 32) * L];
    const int tid = threadIdx.x, l = tid % L, t = tid / L;
    const long long row0 = (long long)blockIdx.x * L;
    const double *x = reinterpret_cast<const double *>(a.x);
    {
        constexpr int PER = (L * H + NTH - 1) / NTH;
        double2 q[PER];
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const int idx = tid + i * NTH, m = idx % H, rr = idx / H;
            q[i] = idx < L * H && row0 + rr < a.nrows
                       ? reinterpret_cast<const double2 *>(x + (row0 + rr) * N)[m]
                       : double2{0.0, 0.0};
        }
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const int idx = tid + i * NTH;
            if (idx < L * H) dbuf[(idx % H) * LD + idx / H] = q[i];
        }
    }
    __syncthreads();
    const fxw *tw = reinterpret_cast<const fxw *>(a.tw);
    cfx v[V];
    float s = 0.f;
    int h = 0;
#pragma unroll
    for (int k = 0; k < V / R1; ++k)
#pragma unroll
        for (int r = 0; r < R1 / 2; ++r) {
            v[k * R1 + r] = buf[(t + k * TPL + r * (N / R1)) * LD + l];
            fx_bound(v[k * R1 + r], s, h);
        }
    fx_reduce<L, NTH>(s, h, red);
    const FxScale sc = fx_scale<R1, R2, R3, true, 61>(s, h);
#pragma unroll
    for (int k = 0; k < V / R1; ++k)
#pragma unroll
        for (int r = 0; r < R1 / 2; ++r) v[k * R1 + r] = fx_conv<true, true>(v[k * R1 + r], sc);
    Fst<-1, N, V, L>::template compute<R1, 1, true, false>(v, t, tw);
    fx_rest<-1, N, V, L, R1, R2, R3, false>(v, buf, t, l, tw, true);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < V / RL; ++k)
#pragma unroll
        for (int r = 0; r < RL; ++r) buf[(t + k * TPL + r * (N / RL)) * LD + l] = v[k * RL + r];
    __syncthreads();
    // X[k] = E + w^k O, X[N-k] = conj(E - w^k O), E = (Z[k] + conj Z[N-k]) / 2,
    // O = -i (Z[k] - conj Z[N-k]) / 2: here times 1/2 (a quarter of the sums)
    const fxw *tw2 = reinterpret_cast<const fxw *>(a.tw2);
    const FxOut<true, false> out(2 * NT - sc.ke + 1, sc.bad);
    for (int k = t; 2 * k <= N; k += TPL) {
        const int kc = k == 0 ? 0 : N - k;
        const cfx zk = buf[k * LD + l], zc = buf[kc * LD + l];
        const cfx e = cfx{fx_quarter(zk.x + zc.x), fx_quarter(zk.y - zc.y)};
        const cfx o = cfx{zk.y + zc.y, zc.x - zk.x};
        if (k == 0) {
            const cfx o4 = cfx{fx_quarter(o.x), fx_quarter(o.y)};
            dbuf[l] = out(cadd(e, o4));
            dbuf[N * LD + l] = out(csub(e, o4));
        } else {
            const int4 q = __ldg(reinterpret_cast<const int4 *>(tw2) + k);
            const cfx wo = fx_twiddle<-1>(o, fxw{q.x, q.y, q.z, q.w});
            dbuf[k * LD + l] = out(cadd(e, wo));
            if (2 * k != N) dbuf[kc * LD + l] = out(cfx{e.x - wo.x, wo.y - e.y});
        }
    }
    __syncthreads();
    double2 *c = reinterpret_cast<double2 *>(a.c);
    const int warp = tid >> 5, lane = tid & 31;
    for (int rr = warp; rr < L; rr += NTH / 32) {
        if (row0 + rr < a.nrows) {
            double2 *crow = c + (row0 + rr) * row_pitch(N);
            for (int k = lane; k <= N; k += 32) crow[k] = dbuf[k * LD + rr];
        }
    }
}

// P5: k_fast_c2r in fixed point.
template <int N, int V, int L, int R1, int R2, int R3>
__global__ void __launch_bounds__(L *(N / V)) k_fx_c2r(const RowArgs a) {
    pdl_wait();
    constexpr int TPL = N / V, LD = L + 1, NTH = L * TPL, H = N / 2;
    constexpr int RL = LastR<R1, R2, R3>::value, NT = R3 > 1 ? 2 : 1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cfx *buf = reinterpret_cast<cfx *>(smem_raw);
    double2 *dbuf = reinterpret_cast<double2 *>(smem_raw);
    __shared__ int4 red[(NTH / 32) * L];
    const int tid = threadIdx.x, l = tid % L, t = tid / L;
    const long long row0 = (long long)blockIdx.x * L;
    const double2 *c = reinterpret_cast<const double2 *>(a.c);
    const int warp = tid >> 5, lane = tid & 31;
    {
        constexpr int NW = NTH / 32, RPW = (L + NW - 1) / NW, KPL = (N + 32) / 32;
        double2 q[RPW * KPL];
#pragma unroll
        for (int i = 0; i < RPW; ++i) {
            const int rr = warp + i * NW;
            const bool okr = rr < L && row0 + rr < a.nrows;
            const double2 *crow = c + (okr ? row0 + rr : 0) * row_pitch(N);
#pragma unroll
            for (int j = 0; j < KPL; ++j) {
                const int k = lane + 32 * j;
                q[i * KPL + j] = okr && k <= N ? crow[k] : double2{0.0, 0.0};
            }
        }
#pragma unroll
        for (int i = 0; i < RPW; ++i) {
            const int rr = warp + i * NW;
#pragma unroll
            for (int j = 0; j < KPL; ++j) {
                const int k = lane + 32 * j;
                if (rr < L && k <= N) dbuf[k * LD + rr] = q[i * KPL + j];
            }
        }
    }
    __syncthreads();
    // Z[k] = A + i conj(w^k) B, Z[N-k] = conj A + i w^k conj B with
    // A, B = X[k] +- conj X[N-k]: here a quarter of them, |Z / 4| <= the mean
    // of |X[k]| and |X[N-k]|, so the inputs' bounds hold for the transform's
    float s = 0.f;
    int h = 0;
    for (int k = t; k <= N; k += TPL) fx_bound(buf[k * LD + l], s, h);
    fx_reduce<L, NTH>(s, h, red);
    const FxScale sc = fx_scale<R1, R2, R3, false, 62>(s, h);
    const fxw *tw2 = reinterpret_cast<const fxw *>(a.tw2);
    for (int k = t; 2 * k <= N; k += TPL) {
        const int kc = N - k;
        const cfx xk = fx_conv<true, false>(buf[k * LD + l], sc), xc = fx_conv<true, false>(buf[kc * LD + l], sc);
        const cfx A = cfx{fx_quarter(xk.x + xc.x), fx_quarter(xk.y - xc.y)};
        const cfx B = cfx{xk.x - xc.x, xk.y + xc.y};
        const int4 q = __ldg(reinterpret_cast<const int4 *>(tw2) + k);
        const cfx wb = fx_twiddle<+1>(B, fxw{q.x, q.y, q.z, q.w});
        // i w^k conj B = conj(-i conj(w^k) B)
        buf[k * LD + l] = cfx{A.x - wb.y, A.y + wb.x};
        if (k != 0 && 2 * k != N) buf[kc * LD + l] = cfx{A.x + wb.y, wb.x - A.y};
    }
    __syncthreads();
    const fxw *tw = reinterpret_cast<const fxw *>(a.tw);
    cfx v[V];
    Stg<fx, +1, N, V, L>::template load_in<R1>(v, buf, t, l);
    Fst<+1, N, V, L>::template compute<R1, 1, false, false>(v, t, tw);
    fx_rest<+1, N, V, L, R1, R2, R3, true>(v, buf, t, l, tw, true);
    __syncthreads();
    const FxOut<true, true> out(2 * NT + 2 - sc.ke + a.exp, sc.bad);
#pragma unroll
    for (int k = 0; k < V / RL; ++k)
#pragma unroll
        for (int r = 0; r < RL / 2; ++r) dbuf[(t + k * TPL + r * (N / RL)) * LD + l] = out(v[k * RL + r]);
    __syncthreads();
    double *x = reinterpret_cast<double *>(const_cast<void *>(a.x));
#pragma unroll 4
    for (int idx = tid; idx < L * H; idx += NTH) {
        const int m = idx % H, rr = idx / H;
        if (row0 + rr < a.nrows) reinterpret_cast<double2 *>(x + (row0 + rr) * N)[m] = dbuf[m * LD + rr];
    }
}

// ----------------------------------------------------- configurations --
// Tile shape and radix schedule per length: V values per thread, L lines.
// Measured at N = 256 (lines of 512), per pass: 8*8*8 with 4 lines (256
// threads) 0.28 ms for P2 and P4 and 1.07 for P3, with 8 lines 0.31 / 0.32 /
// 1.13, 16*16*2 with V = 16 0.30 / 0.30 / 1.10 (before the exchanges of 4 lines
// were free of conflicts).
template <int n> struct CfgX {
    static constexpr bool Ok = false;
    static constexpr int V = 8, L = 8, R1 = 8, R2 = 8, R3 = 1;
};
#define FSP_CFGX(NN, VV, LL, A, B, CC)                                     \
    template <> struct CfgX<NN> {                                          \
        static constexpr bool Ok = true;                                   \
        static constexpr int V = VV, L = LL, R1 = A, R2 = B, R3 = CC;      \
    };
FSP_CFGX(48, 12, 8, 4, 3, 4)
// N = 32: few lines for 152 SMs, so few values per thread (a warp's own
// instruction stream is what a pass waits for)
FSP_CFGX(32, 4, 8, 4, 2, 4)
FSP_CFGX(64, 4, 8, 4, 4, 4)
FSP_CFGX(96, 12, 8, 4, 6, 4)
FSP_CFGX(128, 8, 8, 8, 2, 8)
FSP_CFGX(192, 12, 8, 4, 12, 4)
FSP_CFGX(256, 8, 8, 8, 4, 8)
FSP_CFGX(384, 24, 8, 8, 6, 8)
FSP_CFGX(512, 8, 4, 8, 8, 8)
FSP_CFGX(1024, 16, 4, 16, 8, 8)
#undef FSP_CFGX
// Rows: lengths 64 and 256 run faster in two stages (P1 / P5 at N = 256 0.161 /
// 0.154 ms with 16*16, 0.166 / 0.162 with 8*4*8)
template <int N> struct RowX : CfgX<N> {};
template <> struct RowX<64> {
    static constexpr int V = 8, L = 16, R1 = 8, R2 = 8, R3 = 1;
};
template <> struct RowX<256> {
    static constexpr int V = 16, L = 8, R1 = 16, R2 = 16, R3 = 1;
};
// CTAs per SM the registers must allow.  With 8 values per thread 24 warps for
// P3 (80 registers, a few spilled: 1.051 ms at N = 256, 1.071 with 32 warps,
// 1.149 with 16) and 32 for P2 and P4 (0.267 / 0.256 ms, 0.275 / 0.285 with
// 24); fewer where a thread holds more.
template <int n, int MODE> constexpr int fx_minb() {
    constexpr int th = CfgX<n>::L * (n / CfgX<n>::V), V = CfgX<n>::V;
    if (MODE != COL_FMI && MODE != COL_FMO) return V <= 8 ? 1024 / th : 1;
    return V <= 8 ? 768 / th : V <= 12 ? 640 / th : V <= 16 ? 512 / th : 1;
}

template <int n, int MODE, bool RG> cudaError_t launch_fx_col_n(const ColArgs &a, int nbatch, cudaStream_t s) {
    using K = CfgX<n>;
    if constexpr (!K::Ok) {
        return cudaErrorInvalidValue;
    } else {
        auto kern = k_fx_col<n, K::V, K::L, K::R1, K::R2, K::R3, MODE, RG, fx_minb<n, MODE>()>;
        const size_t sm = Fxc<n, K::V, K::L>::smem;
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        if (e != cudaSuccess) return e;
        ColArgs b = a;
        dim3 grid;
        if constexpr (!RG) {
            constexpr int N = n / 2;
            static_assert(N % K::L == 0, "tiles must cover k_x < N exactly");
            if (nbatch % N != 0) return cudaErrorInvalidValue;
            grid = dim3((unsigned)(N / K::L), (unsigned)(nbatch + nbatch / N));
        } else {
            const int nx = a.nlines - 1;
            if (nx <= 0 || nx % K::L != 0 || nbatch % K::L != 0) return cudaErrorInvalidValue;
            b.nbatch = nbatch;
            b.xrows = (nbatch / K::L + nx / K::L - 1) / (nx / K::L);
            grid = dim3((unsigned)(nx / K::L), (unsigned)(nbatch + b.xrows));
        }
        return launch_pass(kern, grid, K::L * (n / K::V), sm, s, b);
    }
}
template <int MODE> cudaError_t launch_fx_col(int n, const ColArgs &a, int nbatch, cudaStream_t s) {
    switch (n) {
    case 64: return launch_fx_col_n<64, MODE, false>(a, nbatch, s);
    case 96: return launch_fx_col_n<96, MODE, false>(a, nbatch, s);
    case 128: return launch_fx_col_n<128, MODE, false>(a, nbatch, s);
    case 192: return launch_fx_col_n<192, MODE, false>(a, nbatch, s);
    case 256: return launch_fx_col_n<256, MODE, false>(a, nbatch, s);
    case 384: return launch_fx_col_n<384, MODE, false>(a, nbatch, s);
    case 512: return launch_fx_col_n<512, MODE, false>(a, nbatch, s);
    case 1024: return launch_fx_col_n<1024, MODE, false>(a, nbatch, s);
    }
    return cudaErrorInvalidValue;
}
template <int MODE> cudaError_t launch_fx_col_rg(int n, const ColArgs &a, int nbatch, cudaStream_t s) {
    switch (n) {
    case 64: return launch_fx_col_n<64, MODE, true>(a, nbatch, s);
    case 128: return launch_fx_col_n<128, MODE, true>(a, nbatch, s);
    case 256: return launch_fx_col_n<256, MODE, true>(a, nbatch, s);
    case 512: return launch_fx_col_n<512, MODE, true>(a, nbatch, s);
    case 1024: return launch_fx_col_n<1024, MODE, true>(a, nbatch, s);
    }
    return cudaErrorInvalidValue;
}

template <int N, bool R2C> cudaError_t launch_fx_row_n(const RowArgs &a, cudaStream_t s) {
    using K = RowX<N>;
    auto kern = R2C ? k_fx_r2c<N, K::V, K::L, K::R1, K::R2, K::R3> : k_fx_c2r<N, K::V, K::L, K::R1, K::R2, K::R3>;
    const size_t sm = sizeof(cfx) * (N + 1) * (K::L + 1);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    const dim3 grid((unsigned)((a.nrows + K::L - 1) / K::L));
    return launch_pass(kern, grid, K::L * (N / K::V), sm, s, a);
}
template <bool R2C> cudaError_t launch_fx_row(int N, const RowArgs &a, cudaStream_t s) {
    switch (N) {
    case 32: return launch_fx_row_n<32, R2C>(a, s);
    case 48: return launch_fx_row_n<48, R2C>(a, s);
    case 64: return launch_fx_row_n<64, R2C>(a, s);
    case 96: return launch_fx_row_n<96, R2C>(a, s);
    case 128: return launch_fx_row_n<128, R2C>(a, s);
    case 192: return launch_fx_row_n<192, R2C>(a, s);
    case 256: return launch_fx_row_n<256, R2C>(a, s);
    case 512: return launch_fx_row_n<512, R2C>(a, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace fast
}  // namespace fsp
