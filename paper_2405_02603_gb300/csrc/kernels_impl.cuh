// kernels_impl.cuh -- definitions of the line-transform kernels (included once
// per real type by kernels_f32.cu / kernels_f64.cu).
//
// FP64 lines (T = double) are transformed in 64-bit fixed point (fx.cuh): the
// doubles of a tile are loaded into shared memory as they are, tile_scale
// turns them into integers at their line's scale, and the store turns the
// results back.  Where a kernel has the two forms, W is the working type and
// FX says which form it is.
#pragma once
#include "fast.cuh"
#include "fx_line.cuh"
#include "kernels.cuh"
#include "tiles.h"

namespace fsp {

constexpr int kMaxThreads = 512;
// 512-thread CTAs per SM the registers must allow: two in FP32 (64 registers;
// left to itself the compiler takes 72-74 for some passes: N = 225 1.47 ms
// instead of 1.27), one in fixed point
template <typename T> constexpr int lines_minb() { return sizeof(T) == 4 ? 2 : 1; }
constexpr int kMaxLines = 32;  // lines per CTA (lgL <= 5)

template <typename T> struct work_of {
    using t = T;
};
template <> struct work_of<double> {
    using t = fx;
};
template <int D> struct Dft<fx, D> {
    using C = cfx;
    static __device__ __forceinline__ void r2(C *v) { fast::RD<fx, D>::template dft<2, false, false>(v); }
    static __device__ __forceinline__ void r3(C *v) { fast::RD<fx, D>::template dft<3, false, false>(v); }
    static __device__ __forceinline__ void r4(C *v) { fast::RD<fx, D>::template dft<4, false, false>(v); }
    static __device__ __forceinline__ void r5(C *v) { fast::RD<fx, D>::template dft<5, false, false>(v); }
    static __device__ __forceinline__ void r8(C *v) { fast::RD<fx, D>::template dft<8, false, false>(v); }
};

// Per line of a tile: the largest upper word and the 1-norm in units of
// 2^(em - 16) (integers, so that the order of the atomics does not matter),
// the largest modulus of a product with S, and the scale of the results.
struct TileLines {
    int hmax[kMaxLines], mmax[kMaxLines];
    unsigned sum[kMaxLines], sum2[kMaxLines];
    int hS[kMaxLines];
    int eo[kMaxLines];
    bool bad[kMaxLines];
};
__device__ __forceinline__ void tile_clear(TileLines &q) {
    if (threadIdx.x < kMaxLines) {
        q.hmax[threadIdx.x] = q.mmax[threadIdx.x] = q.hS[threadIdx.x] = 0;
        q.sum[threadIdx.x] = q.sum2[threadIdx.x] = 0;
    }
}
// Turns the doubles at positions p < np of line l into integers; every thread
// of the CTA calls it after the barrier that ends the loads, and a barrier
// follows.  The result's scale is that of the integers.
__device__ __forceinline__ FxScale tile_scale(cfx *buf, int ld, int np, const Stages &st, int B, int l, int sub,
                                              int tpl, bool act, TileLines &q) {
    float s = 0.f;
    int h = 0;
    if (act) {
        for (int p = sub; p < np; p += tpl) fx_bound(buf[p * ld + l], s, h);
        atomicMax(&q.hmax[l], h);
    }
    __syncthreads();
    h = q.hmax[l];
    const int em = fx_em(h);
    FxScale sc;
    sc.any = fx_far(em), sc.bad = (h >> 20) == 0x7ff;
    const bool sum = h != 0 && !sc.bad;  // neither a zero line nor an infinite one
    if (act && sum) {
        if (sc.any) {  // the 1-norm in units of 2^em: as it is, no float holds it
            s = 0.f;
            for (int p = sub; p < np; p += tpl) fx_bound(buf[p * ld + l], s, h, em);
        }
        atomicAdd(&q.sum[l], tile_units(s, sc.any ? 0 : em));
    }
    __syncthreads();
    const int eL = sum ? em - 16 + fx_clog2(1.5f * (float)q.sum[l] + 1e-30f) : em + tile_log2(st);
    sc.ke = tile_ke(st, em, eL, B);
    if (act)
        for (int p = sub; p < np; p += tpl) buf[p * ld + l] = fx_conv<true, false>(buf[p * ld + l], sc);
    return sc;
}
// a double or a float as the real part of a working value, still unscaled
__device__ __forceinline__ fx tile_real(double x) { return fx(__double_as_longlong(x), 0); }
__device__ __forceinline__ float tile_real(float x) { return x; }
__device__ __forceinline__ cfx tile_cplx(double2 q) { return fx_raw(q); }
__device__ __forceinline__ float2 tile_cplx(float2 q) { return q; }
// a result of line l for the store
__device__ __forceinline__ double2 tile_out(const cfx &v, const TileLines &q, int l) {
    return FxOut<true, false>(q.eo[l], q.bad[l])(v);
}
__device__ __forceinline__ double tile_out_re(const cfx &v, const TileLines &q, int l) {
    return FxOut<true, true>(q.eo[l], q.bad[l]).template one<true>(v.x.v);
}
__device__ __forceinline__ float2 tile_out(float2 v, const TileLines &, int) { return v; }
__device__ __forceinline__ float tile_out_re(float2 v, const TileLines &, int) { return v.x; }

// Loads of data another CTA of the same launch may have written (the
// persistent batched kernel) bypass L1, which is not coherent across SMs.
template <bool COH, typename V> __device__ __forceinline__ V ldw(const V *p) {
    if constexpr (COH)
        return __ldcg(p);
    else
        return *p;
}

// whether a complex line carries two real ones
__host__ __device__ constexpr bool lines_pair(int in) { return in != IN_CPLX; }

// ---------------------------------------------------------- lines_tile --
// One tile of a batched line transform: (complex) lines [bx*L, bx*L + L) of batch `by`.
// Every thread of the CTA must call it (barriers); threads beyond L*tpl idle.
template <typename T, int IN, int OUT, int MODE, bool COH>
__device__ __forceinline__ void lines_tile(const LinesArgs &a, int bx, long long by, unsigned char *smem_raw) {
    using W = typename work_of<T>::t;
    using C = cx_t<W>;
    using IC = cx_t<T>;
    constexpr bool FX = std::is_same<W, fx>::value;
    constexpr bool PAIR = lines_pair(IN);
    static_assert(!PAIR || OUT == OUT_REAL, "pairs of real lines have real transforms");
    __shared__ TileLines tl;
    if constexpr (FX) tile_clear(tl);
    C *buf = reinterpret_cast<C *>(smem_raw);
    const int L = 1 << a.lgL, lmask = L - 1;
    const int ld = L + 1;
    const int tid = threadIdx.x, nth = blockDim.x;
    const int line0 = bx << a.lgL;
    const long long b = by;
    const int n = a.st.n;

    // ---- load (with zero padding / even extension); U loads of a thread are
    // issued before their shared-memory stores, so that several are in flight
    constexpr int U = 4;
    if (IN == IN_CPLX) {
        const IC *in = reinterpret_cast<const IC *>(a.in) + b * a.in_batch;
        const int cnt = L * a.n_in;
        if (a.in_line == 1) {
            for (int base = tid; base < cnt; base += U * nth) {
                C q[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int idx = base + u * nth, l = idx & lmask, p = idx >> a.lgL;
                    q[u] = C{W(0), W(0)};
                    if (idx < cnt && line0 + l < a.nlines)
                        q[u] = tile_cplx(ldw<COH>(in + ((long long)(line0 + l) + (long long)p * a.in_pos)));
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int idx = base + u * nth;
                    if (idx < cnt) buf[(idx >> a.lgL) * ld + (idx & lmask)] = q[u];
                }
            }
        } else {
            const FastDiv by(a.n_in);
            for (int base = tid; base < cnt; base += U * nth) {
                C q[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int idx = base + u * nth, l = by.quot(idx), p = idx - l * a.n_in;
                    q[u] = C{W(0), W(0)};
                    if (idx < cnt && line0 + l < a.nlines)
                        q[u] = tile_cplx(ldw<COH>(in + ((long long)(line0 + l) * a.in_line + (long long)p * a.in_pos)));
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int idx = base + u * nth;
                    const int l = by.quot(idx);
                    if (idx < cnt) buf[(idx - l * a.n_in) * ld + l] = q[u];
                }
            }
        }
        const int zc = L * (n - a.n_in);
        for (int idx = tid; idx < zc; idx += nth) buf[(a.n_in + (idx >> a.lgL)) * ld + (idx & lmask)] = C{W(0), W(0)};
    } else {
        // DCT-I through the DFT of the even extension: y[j] = x[j] for j <= M,
        // y[2M - j] = x[j] for 0 < j < M.  DST-I through the DFT of
        // y[j] = i x[j], y[2M - j] = -i x[j] for 0 < j < M, y[0] = y[M] = 0,
        // which is 2 sum_j x[j] sin(pi j k / M), real.
        //
        // A complex line holds two real ones (2 c and 2 c + 1, as its real and
        // imaginary part): both transforms are real, so they come out apart.
        const T *in = reinterpret_cast<const T *>(a.in) + b * a.in_batch;
        const int M = n >> 1, np = M + 1, cnt = L * np;
        const bool col = (a.in_line == 1);
        const FastDiv by(np);
        for (int idx = tid; idx < cnt; idx += nth) {
            int l, p;
            if (col) {
                l = idx & lmask;
                p = idx >> a.lgL;
            } else {
                l = by.quot(idx);
                p = idx - l * np;
            }
            const int r0 = 2 * (line0 + l);
            const T *q = in + ((long long)r0 * a.in_line + (long long)p * a.in_pos);
            T x = T(0), y = T(0);
            if (r0 < a.nlines) x = ldw<COH>(q);
            if (r0 + 1 < a.nlines) y = ldw<COH>(q + a.in_line);
            const bool inner = p > 0 && p < M;
            if (IN == IN_REAL_EVEN) {
                buf[p * ld + l] = C{tile_real(x), tile_real(y)};
                if (inner) buf[(n - p) * ld + l] = C{tile_real(x), tile_real(y)};
            } else {  // i (x + i y)
                buf[p * ld + l] = inner ? C{tile_real(-y), tile_real(x)} : C{W(0), W(0)};
                if (inner) buf[(n - p) * ld + l] = C{tile_real(y), tile_real(-x)};
            }
        }
    }
    __syncthreads();

    const int l = tid & lmask, sub = tid >> a.lgL;
    const bool act = (PAIR ? 2 * (line0 + l) : line0 + l) < a.nlines && sub < a.tpl;
    const fx_tw_t<W> *tw = reinterpret_cast<const fx_tw_t<W> *>(a.tw);
    FxScale sc{};
    if constexpr (FX) {
        sc = tile_scale(buf, ld, IN == IN_CPLX ? a.n_in : n, a.st, MODE == M_FWD_MUL_INV ? 61 : 62, l, sub, a.tpl, act,
                        tl);
        if (MODE != M_FWD_MUL_INV && act && sub == 0) tl.eo[l] = tile_div(a.st) - sc.ke, tl.bad[l] = sc.bad;
        __syncthreads();
    }
    if (MODE == M_INV)
        Engine<W, +1>::run(buf, ld, a.st, tw, l, sub, a.tpl, act);
    else
        Engine<W, -1>::run(buf, ld, a.st, tw, l, sub, a.tpl, act);

    if (MODE == M_FWD_MUL_INV) {
        const T *S = reinterpret_cast<const T *>(a.S);
        const int h2 = 2 * a.half;
        const int hb = a.half_b ? a.half_b : a.half;
        const int fy = (int)b <= hb ? (int)b : 2 * hb - (int)b;
        const int cnt = L * n;
        const int odd = a.odd;
        if constexpr (FX) {
            // as k_fx_col: bounds of the products, then the products at the
            // scale of the inverse
            const double *Sl = S + (long long)fy * a.s_batch + line0 + l;
            const int kS = fx_base(S[a.s_pos + a.s_batch + 1]);
            float s2 = 0.f, m2 = 0.f;
            int hS = 0;
            if (act) {
                for (int p = sub; p < n; p += a.tpl)
                    fx_bound_mul(buf[p * ld + l], Sl[(long long)(p <= a.half ? p : h2 - p) * a.s_pos], s2, m2, hS, kS);
                atomicMax(&tl.hS[l], hS);
                atomicMax(&tl.mmax[l], __float_as_int(m2));
            }
            __syncthreads();
            const int eS = fx_es(tl.hS[l]);
            const bool near = fx_near(eS, kS), bad = sc.bad || eS == 1025;
            // products' moduli are below 2^em (near: in units of 2^(32 + kS))
            const int ef = fx_clog2(1.1f * __int_as_float(tl.mmax[l]));
            const int em = near ? ef + 32 + kS : 61 + eS;
            if (act && near) atomicAdd(&tl.sum2[l], tile_units(s2, ef));
            __syncthreads();
            const int eL = near ? em - 16 + fx_clog2(1.1f * (float)tl.sum2[l] + 1e-30f) : em + tile_log2(a.st);
            const int ke = min(tile_ke(a.st, em - 1, eL, 62), 60 - em);
            const int neg_b = odd == 2 && (int)b > hb ? -1 : 0, neg_z = odd == 1 ? -1 : 0;
            if (act) {
                for (int p = sub; p < n; p += a.tpl) {
                    const cfx q = fx_mul_s(buf[p * ld + l], Sl[(long long)(p <= a.half ? p : h2 - p) * a.s_pos], ke,
                                           neg_b ^ (p > a.half ? neg_z : 0), eS > -900);
                    buf[p * ld + l] = odd == 0 ? q : cfx{q.y, -q.x};
                }
                if (sub == 0) tl.eo[l] = 2 * tile_div(a.st) - sc.ke - ke, tl.bad[l] = bad;
            }
        } else {
        const T sb = odd == 2 && (int)b > hb ? T(-1) : T(1);
        for (int idx = tid; idx < cnt; idx += nth) {
            const int ll = idx & lmask, p = idx >> a.lgL;
            if (line0 + ll < a.nlines) {
                const int fz = p <= a.half ? p : h2 - p;
                T s = S[(long long)fz * a.s_pos + (long long)fy * a.s_batch + line0 + ll];
                C v = buf[p * ld + ll];
                if (odd == 0) {
                    v.x *= s;
                    v.y *= s;
                } else {
                    // -i s v; the line index (k_x <= half) never flips the sign
                    if (odd == 1 && p > a.half) s = -s;
                    s *= sb;
                    v = C{s * v.y, -(s * v.x)};
                }
                buf[p * ld + ll] = v;
            }
        }
        }
        __syncthreads();
        Engine<W, +1>::run(buf, ld, a.st, tw, l, sub, a.tpl, act);
    }

    // ---- store (crop to n_out positions)
    const int cnt = L * a.n_out;
    const bool col = (a.out_line == 1);
    const FastDiv by_out(a.n_out);
    if (OUT == OUT_CPLX) {
        IC *out = reinterpret_cast<IC *>(a.out) + b * a.out_batch;
        for (int idx = tid; idx < cnt; idx += nth) {
            int ll, p;
            if (col) {
                ll = idx & lmask;
                p = idx >> a.lgL;
            } else {
                ll = by_out.quot(idx);
                p = idx - ll * a.n_out;
            }
            if (line0 + ll < a.nlines)
                out[(long long)(line0 + ll) * a.out_line + (long long)p * a.out_pos] = tile_out(buf[p * ld + ll], tl, ll);
        }
    } else {
        T *out = reinterpret_cast<T *>(a.out) + b * a.out_batch;
        for (int idx = tid; idx < cnt; idx += nth) {
            int ll, p;
            if (col) {
                ll = idx & lmask;
                p = idx >> a.lgL;
            } else {
                ll = by_out.quot(idx);
                p = idx - ll * a.n_out;
            }
            if constexpr (PAIR) {
                const int r0 = 2 * (line0 + ll);
                if (r0 < a.nlines) {
                    const IC v = tile_out(buf[p * ld + ll], tl, ll);
                    T *q = out + ((long long)r0 * a.out_line + (long long)p * a.out_pos);
                    q[0] = v.x;
                    if (r0 + 1 < a.nlines) q[a.out_line] = v.y;
                }
            } else if (line0 + ll < a.nlines) {
                out[(long long)(line0 + ll) * a.out_line + (long long)p * a.out_pos] = tile_out_re(buf[p * ld + ll], tl, ll);
            }
        }
    }
}

template <typename T, int IN, int OUT, int MODE>
__global__ void __launch_bounds__(kMaxThreads, lines_minb<T>()) k_lines(const LinesArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    pdl_wait();
    lines_tile<T, IN, OUT, MODE, false>(a, blockIdx.x, blockIdx.y, smem_raw);
}

// ------------------------------------------------------------ r2c_tile --
// Sec. 2.2 steps 2 and 4 along x: each row of N reals, zero-padded to 2N, is
// transformed to its N+1 non-redundant coefficients.  With z[m] = x[2m] +
// i x[2m+1] (zero for 2m >= N) and Z = FFT_N(z):
//   E = (Z[k] + conj Z[N-k]) / 2,  O = -i (Z[k] - conj Z[N-k]) / 2,
//   X[k] = E + w^k O,  X[N-k] = conj(E - w^k O),  w = exp(-2 pi i / 2N).
template <typename T, bool COH>
__device__ __forceinline__ void r2c_tile(const RowsArgs &a, int bx, unsigned char *smem_raw) {
    using W = typename work_of<T>::t;
    using C = cx_t<W>;
    using IC = cx_t<T>;
    constexpr bool FX = std::is_same<W, fx>::value;
    __shared__ TileLines tl;
    if constexpr (FX) tile_clear(tl);
    C *buf = reinterpret_cast<C *>(smem_raw);
    const int L = 1 << a.lgL, lmask = L - 1, ld = L + 1;
    const int tid = threadIdx.x, nth = blockDim.x;
    const long long row0 = (long long)bx << a.lgL;
    const int N = a.N, Mh = (N + 1) >> 1;
    const T *x = reinterpret_cast<const T *>(a.x);

    const int cnt = L * Mh;
    const FastDiv by(Mh);
    constexpr int U = 4;  // loads in flight per thread
    for (int base = tid; base < cnt; base += U * nth) {
        C q[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int idx = base + u * nth, l = by.quot(idx), m = idx - l * Mh;
            q[u] = C{W(0), W(0)};
            if (idx < cnt && row0 + l < a.nrows) {
                const T *xr = x + (row0 + l) * a.x_row;
                if ((N & 1) == 0) {
                    q[u] = tile_cplx(ldw<COH>(reinterpret_cast<const IC *>(xr) + m));
                } else {
                    q[u].x = tile_real(ldw<COH>(xr + 2 * m));
                    q[u].y = tile_real((2 * m + 1 < N) ? ldw<COH>(xr + 2 * m + 1) : T(0));
                }
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int idx = base + u * nth;
            const int l = by.quot(idx);
            if (idx < cnt) buf[(idx - l * Mh) * ld + l] = q[u];
        }
    }
    const int zc = L * (N - Mh);
    for (int idx = tid; idx < zc; idx += nth) buf[(Mh + (idx >> a.lgL)) * ld + (idx & lmask)] = C{W(0), W(0)};
    __syncthreads();

    const int l = tid & lmask, sub = tid >> a.lgL;
    const bool act = (row0 + l) < a.nrows && sub < a.tpl;
    if constexpr (FX) {
        const FxScale sc = tile_scale(buf, ld, Mh, a.st, 61, l, sub, a.tpl, act, tl);
        // the coefficients below come out at half their scale
        if (act && sub == 0) tl.eo[l] = tile_div(a.st) - sc.ke + 1, tl.bad[l] = sc.bad;
        __syncthreads();
    }
    Engine<W, -1>::run(buf, ld, a.st, reinterpret_cast<const fx_tw_t<W> *>(a.tw), l, sub, a.tpl, act);

    const fx_tw_t<W> *tw2 = reinterpret_cast<const fx_tw_t<W> *>(a.tw2);
    if (act) {
        for (int k = sub; 2 * k <= N; k += a.tpl) {
            const int kc = (k == 0) ? 0 : N - k;
            const C zk = buf[k * ld + l], zc = buf[kc * ld + l];
            C e, wo;
            if constexpr (FX) {  // a quarter of the sums: X / 2
                e = C{fx_quarter(zk.x + zc.x), fx_quarter(zk.y - zc.y)};
                wo = fx_twiddle<-1>(C{zk.y + zc.y, zc.x - zk.x}, tw2[k]);
            } else {
                e = C{T(0.5) * (zk.x + zc.x), T(0.5) * (zk.y - zc.y)};
                const C o = C{T(0.5) * (zk.y + zc.y), T(-0.5) * (zk.x - zc.x)};
                wo = k == 0 ? o : cmul(tw2[k], o);
            }
            if (k == 0) {
                buf[0 * ld + l] = cadd(e, wo);
                buf[N * ld + l] = csub(e, wo);
            } else {
                buf[k * ld + l] = cadd(e, wo);
                if (2 * k != N) buf[kc * ld + l] = cconj(csub(e, wo));
            }
        }
    }
    __syncthreads();

    IC *c = reinterpret_cast<IC *>(a.c);
    const int np = N + 1, cnt2 = L * np;
    const FastDiv by_np(np);
    for (int idx = tid; idx < cnt2; idx += nth) {
        const int ll = by_np.quot(idx), k = idx - ll * np;
        if (row0 + ll < a.nrows) c[(row0 + ll) * a.c_row + k] = tile_out(buf[k * ld + ll], tl, ll);
    }
}

template <typename T> __global__ void __launch_bounds__(kMaxThreads, lines_minb<T>()) k_r2c_rows(const RowsArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    pdl_wait();
    r2c_tile<T, false>(a, blockIdx.x, smem_raw);
}

// ------------------------------------------------------------ c2r_tile --
// Sec. 2.2 steps 4 and 5 along x: from the N+1 coefficients X[k] of a real
// length-2N signal y, y[j] = sum_k X[k] exp(+2 pi i jk / 2N), keep j < N.
// With A = X[k] + conj X[N-k], B = X[k] - conj X[N-k], w = exp(-2 pi i/2N):
//   Z[k] = A + i conj(w^k) B,  Z[N-k] = conj A + i w^k conj B,
//   z = IFFT_N(Z) (unnormalised),  y[2m] = Re z[m],  y[2m+1] = Im z[m].
template <typename T, bool COH>
__device__ __forceinline__ void c2r_tile(const RowsArgs &a, int bx, unsigned char *smem_raw) {
    using W = typename work_of<T>::t;
    using C = cx_t<W>;
    using IC = cx_t<T>;
    constexpr bool FX = std::is_same<W, fx>::value;
    __shared__ TileLines tl;
    if constexpr (FX) tile_clear(tl);
    C *buf = reinterpret_cast<C *>(smem_raw);
    const int L = 1 << a.lgL, ld = L + 1;
    const int tid = threadIdx.x, nth = blockDim.x;
    const long long row0 = (long long)bx << a.lgL;
    const int N = a.N, np = N + 1;
    const IC *c = reinterpret_cast<const IC *>(a.c);

    const int cnt = L * np;
    const FastDiv by(np);
    constexpr int U = 4;  // loads in flight per thread
    for (int base = tid; base < cnt; base += U * nth) {
        C q[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int idx = base + u * nth, l = by.quot(idx), k = idx - l * np;
            q[u] = C{W(0), W(0)};
            if (idx < cnt && row0 + l < a.nrows) q[u] = tile_cplx(ldw<COH>(c + ((row0 + l) * a.c_row + k)));
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int idx = base + u * nth;
            const int l = by.quot(idx);
            if (idx < cnt) buf[(idx - l * np) * ld + l] = q[u];
        }
    }
    __syncthreads();

    const int l = tid & (L - 1), sub = tid >> a.lgL;
    const bool act = (row0 + l) < a.nrows && sub < a.tpl;
    const fx_tw_t<W> *tw2 = reinterpret_cast<const fx_tw_t<W> *>(a.tw2);
    if constexpr (FX) {
        // the inputs' bounds hold for Z / 4 (|Z| / 4 <= the mean of |X[k]| and |X[N-k]|)
        const FxScale sc = tile_scale(buf, ld, np, a.st, 62, l, sub, a.tpl, act, tl);
        if (act && sub == 0) tl.eo[l] = tile_div(a.st) + 2 - sc.ke + a.exp, tl.bad[l] = sc.bad;
        __syncthreads();
    }
    if (act) {
        for (int k = sub; 2 * k <= N; k += a.tpl) {
            const int kc = N - k;
            const C xk = buf[k * ld + l], xc = buf[kc * ld + l];
            if constexpr (FX) {  // Z / 4; i w^k conj B = conj(-i conj(w^k) B)
                const C A = C{fx_quarter(xk.x + xc.x), fx_quarter(xk.y - xc.y)};
                const C wb = fx_twiddle<+1>(C{xk.x - xc.x, xk.y + xc.y}, tw2[k]);
                buf[k * ld + l] = C{A.x - wb.y, A.y + wb.x};
                if (k != 0 && 2 * k != N) buf[kc * ld + l] = C{A.x + wb.y, wb.x - A.y};
            } else {
                const C A = C{xk.x + xc.x, xk.y - xc.y};
                const C B = C{xk.x - xc.x, xk.y + xc.y};
                const C w = tw2[k];
                buf[k * ld + l] = cadd(A, cmuli(cmul(cconj(w), B)));
                if (k != 0 && 2 * k != N) buf[kc * ld + l] = cadd(cconj(A), cmuli(cmul(w, cconj(B))));
            }
        }
    }
    __syncthreads();
    Engine<W, +1>::run(buf, ld, a.st, reinterpret_cast<const fx_tw_t<W> *>(a.tw), l, sub, a.tpl, act);

    T *x = reinterpret_cast<T *>(const_cast<void *>(a.x));
    const int Mh = (N + 1) >> 1, cnt2 = L * Mh;
    const FastDiv by_m(Mh);
    for (int idx = tid; idx < cnt2; idx += nth) {
        const int ll = by_m.quot(idx), m = idx - ll * Mh;
        if (row0 + ll < a.nrows) {
            T *xr = x + (row0 + ll) * a.x_row;
            const IC v = tile_out(buf[m * ld + ll], tl, ll);
            if ((N & 1) == 0) {
                reinterpret_cast<IC *>(xr)[m] = v;
            } else {
                xr[2 * m] = v.x;
                if (2 * m + 1 < N) xr[2 * m + 1] = v.y;
            }
        }
    }
}

template <typename T> __global__ void __launch_bounds__(kMaxThreads, lines_minb<T>()) k_c2r_rows(const RowsArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    pdl_wait();
    c2r_tile<T, false>(a, blockIdx.x, smem_raw);
}

// -------------------------------------------------------------- k_roots --
template <typename T> __global__ void k_roots(cx_t<T> *tw, int n) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e < n) {
        // angle -2 pi e/n reduced to (-pi, pi]: sincospi of -2e/n
        const int er = (2 * e > n) ? e - n : e;
        double s, c;
        sincospi(-2.0 * (double)er / (double)n, &s, &c);
        tw[e] = cx_t<T>{T(c), T(s)};
    }
}

// ---------------------------------------------------------------- hosts --
template <typename T> size_t lines_smem_bytes(const LinesArgs &a) {
    int np = a.st.n;
    return (size_t)np * smem_pitch(a.lgL) * sizeof(cx_t<T>);
}
template <typename T> size_t rows_smem_bytes(const RowsArgs &a) {
    return (size_t)(a.N + 1) * smem_pitch(a.lgL) * sizeof(cx_t<T>);
}

template <typename K> static cudaError_t set_smem(K kernel) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxTileSmem);
}

template <typename T, int IN, int OUT, int MODE> cudaError_t launch_lines(const LinesArgs &a, cudaStream_t s) {
    const size_t sm = lines_smem_bytes<T>(a);
    auto kern = k_lines<T, IN, OUT, MODE>;
    cudaError_t e = set_smem(kern);
    if (e != cudaSuccess) return e;
    const int nl = lines_pair(IN) ? (a.nlines + 1) / 2 : a.nlines;
    dim3 grid((unsigned)((nl + (1 << a.lgL) - 1) >> a.lgL), (unsigned)a.nbatch);
    return launch_pass(kern, grid, (1 << a.lgL) * a.tpl, sm, s, a);
}

template <typename T> cudaError_t launch_r2c_rows(const RowsArgs &a, cudaStream_t s) {
    const size_t sm = rows_smem_bytes<T>(a);
    cudaError_t e = set_smem(k_r2c_rows<T>);
    if (e != cudaSuccess) return e;
    const dim3 grid((unsigned)((a.nrows + (1 << a.lgL) - 1) >> a.lgL));
    return launch_pass(k_r2c_rows<T>, grid, (1 << a.lgL) * a.tpl, sm, s, a);
}

template <typename T> cudaError_t launch_c2r_rows(const RowsArgs &a, cudaStream_t s) {
    const size_t sm = rows_smem_bytes<T>(a);
    cudaError_t e = set_smem(k_c2r_rows<T>);
    if (e != cudaSuccess) return e;
    const dim3 grid((unsigned)((a.nrows + (1 << a.lgL) - 1) >> a.lgL));
    return launch_pass(k_c2r_rows<T>, grid, (1 << a.lgL) * a.tpl, sm, s, a);
}

template <typename T> cudaError_t launch_roots(void *tw, int n, cudaStream_t s) {
    k_roots<T><<<(n + 255) / 256, 256, 0, s>>>(reinterpret_cast<cx_t<T> *>(tw), n);
    return cudaGetLastError();
}

#define FSP_INSTANTIATE_PASSES(T)                                                                   \
    template cudaError_t launch_lines<T, IN_CPLX, OUT_CPLX, M_FWD>(const LinesArgs &, cudaStream_t); \
    template cudaError_t launch_lines<T, IN_CPLX, OUT_CPLX, M_INV>(const LinesArgs &, cudaStream_t); \
    template cudaError_t launch_lines<T, IN_CPLX, OUT_CPLX, M_FWD_MUL_INV>(const LinesArgs &, cudaStream_t); \
    template cudaError_t launch_r2c_rows<T>(const RowsArgs &, cudaStream_t);                         \
    template cudaError_t launch_c2r_rows<T>(const RowsArgs &, cudaStream_t);                         \
    template size_t lines_smem_bytes<T>(const LinesArgs &);                                          \
    template size_t rows_smem_bytes<T>(const RowsArgs &);
#define FSP_INSTANTIATE(T)                                                                          \
    FSP_INSTANTIATE_PASSES(T)                                                                       \
    template cudaError_t launch_roots<T>(void *, int, cudaStream_t);

}  // namespace fsp
