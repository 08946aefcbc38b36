// Spectral <-> physical transforms of the pseudo-spectral pipe-flow step
// (Keuchel & Avila, Section 2.4): theta synthesis, the z pass with the
// pointwise products of the nonlinear term, theta analysis.  3/2-padded grids,
// hand-written FFTs in shared memory: in FP32 for the mixed precisions, in 64-bit
// fixed point for the FP64 ones, but for the z pass of the continuous adjoint,
// which is in FP64 there.  Batched launches
// carry the batch entry in the grid's z dimension (with the field index for
// the theta kernels) and offset spectral and physical buffers by its slot.
#include "dev_common.cuh"
#include "dev_x64.cuh"
#include "kernels.hpp"

#include <algorithm>
#include <cmath>
#include <type_traits>
#include <utility>

namespace pnop {

// ------------------------------------------------------------------ shared-memory FFT
// Batched Stockham FFT (autosort) over `ncol` columns of length N stored as
// a[n * ld + col].  Radix 4, then 2, then 3 stages; N = 2^p 3^q.  tw holds
// e^{-2 pi i n / N}; sign = -1 forward, +1 inverse (unnormalised).  Returns the
// buffer holding the result.  All threads of the block must call it.
template <class T2>
__device__ __forceinline__ void small_dft(T2* v, const int R, const int sign) {
    using T = typename RealOf<T2>::T;
    if (R == 2) {
        T2 a = v[0], b = v[1];
        v[0] = cadd(a, b);
        v[1] = csub(a, b);
    } else if (R == 4) {
        T2 s02 = cadd(v[0], v[2]), d02 = csub(v[0], v[2]);
        T2 s13 = cadd(v[1], v[3]), d13 = csub(v[1], v[3]);
        T2 id = imul(d13, (T)sign);
        v[0] = cadd(s02, s13);
        v[2] = csub(s02, s13);
        v[1] = cadd(d02, id);
        v[3] = csub(d02, id);
    } else {  // R == 3
        const T h = (T)0.86602540378443864676;  // sqrt(3)/2
        T2 t1 = cadd(v[1], v[2]);
        T2 t2 = mk<T2>(v[0].x - (T)0.5 * t1.x, v[0].y - (T)0.5 * t1.y);
        T2 d = csub(v[1], v[2]);
        T2 t3 = imul(d, (T)sign * h);
        v[0] = cadd(v[0], t1);
        v[1] = cadd(t2, t3);
        v[2] = csub(t2, t3);
    }
}

// One radix-R Stockham stage.  Ns (the size of the sub-transforms already
// done) is a power of two 2^lgNs for every stage but the second and later
// radix-3 stages (radix 3 runs last), so the index split is a shift there.
template <class T2, int R, int NCOL, int LD, int SIGN>
__device__ __forceinline__ void fft_stage(const T2* __restrict__ a, T2* __restrict__ b, int N, int Ns, int lgNs,
                                          const T2* __restrict__ tw) {
    const int stride = N / R;
    const int nb = stride * NCOL;
    const int tstep = N / (Ns * R);
    for (int idx = threadIdx.x; idx < nb; idx += blockDim.x) {
        const int col = idx % NCOL;
        const int jb = idx / NCOL;
        int q, kk;
        if (lgNs >= 0) {
            q = jb >> lgNs;
            kk = jb & (Ns - 1);
        } else {
            q = jb / Ns;
            kk = jb - q * Ns;
        }
        T2 v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = a[(jb + r * stride) * LD + col];
        if (Ns > 1) {  // the first stage has unit twiddles
            const int tb = kk * tstep;  // r * tb < N
#pragma unroll
            for (int r = 1; r < R; ++r) {
                T2 w = tw[r * tb];
                if (SIGN > 0) w.y = -w.y;
                v[r] = cmul(v[r], w);
            }
        }
        small_dft(v, R, SIGN);
        const int idxD = q * Ns * R + kk;
#pragma unroll
        for (int r = 0; r < R; ++r) b[(idxD + r * Ns) * LD + col] = v[r];
    }
}

template <class T2, int NCOL, int LD, int SIGN>
__device__ T2* fft_cols(T2* a, T2* b, int N, const T2* tw) {
    const int n2 = __ffs(N) - 1;  // N = 2^n2 3^n3
    int n3 = 0;
    for (int t = N >> n2; t > 1; t /= 3) ++n3;
    int Ns = 1, lgNs = 0;
    for (int st = 0; st < n2 / 2; ++st) {
        fft_stage<T2, 4, NCOL, LD, SIGN>(a, b, N, Ns, lgNs, tw);
        __syncthreads();
        T2* t = a; a = b; b = t;
        Ns *= 4;
        lgNs += 2;
    }
    if (n2 & 1) {
        fft_stage<T2, 2, NCOL, LD, SIGN>(a, b, N, Ns, lgNs, tw);
        __syncthreads();
        T2* t = a; a = b; b = t;
        Ns *= 2;
        lgNs += 1;
    }
    for (int st = 0; st < n3; ++st) {
        fft_stage<T2, 3, NCOL, LD, SIGN>(a, b, N, Ns, st == 0 ? lgNs : -1, tw);
        __syncthreads();
        T2* t = a; a = b; b = t;
        Ns *= 3;
    }
    return a;
}

// spectral input value of an FP32 synthesis: fields stored in FP32
// (FieldPtrs::inf) are read as they are, FP64 fields converted (with the hardware,
// whose FP64 pipe has room between the loads; the theta analysis converts by
// integer operations, since its FP64 pipe also carries the additions of the
// base-flow terms: each measured fastest that way on the 64x64x256 gradient)
template <class T2>
__device__ __forceinline__ T2 synth_in(const double2* src, const float2* srcf, size_t i) {
    static_assert(std::is_same<T2, float2>::value, "FP64 fields take k_synth_x");
    if (srcf) return srcf[i];
    const double2 v = src[i];
    return make_float2((float)v.x, (float)v.y);
}

// ------------------------------------------------------------------ theta synthesis
// Y[f][j][a][k] = sum_m X_f[j][m][k] e^{i m theta_a}   (zero-padded to nt points)
template <class T2, int KB>
__global__ void k_synth_theta(Geo g, FieldPtrs f, T2* __restrict__ Y, const T2* __restrict__ twg) {
    grid_dep_sync();
    extern __shared__ __align__(16) unsigned char smem[];
    T2* buf0 = reinterpret_cast<T2*>(smem);
    T2* buf1 = buf0 + g.nt * KB;
    T2* tw = buf1 + g.nt * KB;
    const int k0 = blockIdx.x * KB, j = blockIdx.y;
    const int nf = gridDim.z / g.nb, b = blockIdx.z / nf, fi = blockIdx.z - b * nf, slot = g.slot[b];
    Y += (size_t)slot * g.ps;
    const int kw = min(KB, g.nk - k0);
    for (int i = threadIdx.x; i < g.nt; i += blockDim.x) tw[i] = twg[i];
    for (int i = threadIdx.x; i < g.nt * KB; i += blockDim.x) buf0[i] = mk<T2>(0, 0);
    __syncthreads();
    const size_t base = (size_t)slot * g.fs + (size_t)j * g.nm * g.nk;
    const float2* srcf = f.inf[fi] ? f.inf[fi] + base : nullptr;
    const double2* src = srcf ? nullptr : f.in[fi] + base;
    for (int i = threadIdx.x; i < g.nm * KB; i += blockDim.x) {
        const int im = i / KB, kk = i % KB;
        if (kk < kw) {
            const int m = im - g.M;
            const int a = m < 0 ? m + g.nt : m;
            buf0[a * KB + kk] = synth_in<T2>(src, srcf, (size_t)im * g.nk + k0 + kk);
        }
    }
    __syncthreads();
    T2* res = fft_cols<T2, KB, KB, +1>(buf0, buf1, g.nt, tw);
    T2* dst = Y + ((size_t)(fi * g.nr + j) * g.nt) * g.nk;
    for (int i = threadIdx.x; i < g.nt * KB; i += blockDim.x) {
        const int a = i / KB, kk = i % KB;
        if (kk < kw) dst[(size_t)a * g.nk + k0 + kk] = res[i];
    }
}

// Products of the continuous-adjoint forcing at one physical point from the
// packed columns (u_r, u_theta), (u_z, o_r), (o_theta, o_z), (w_r, w_theta),
// (w_z, G_rr), (G_rtheta, G_rz), (G_thetar, G_thetatheta), (G_thetaz, G_zr),
// (G_ztheta, G_zz), o = curl w, G = grad u:
//   P = -u x o - 2 G . w,  (G . w)_i = sum_j G_ij w_j;  out: (P_r, P_theta), (P_z, 0)
template <class T2>
__device__ __forceinline__ void cadj_products(const T2* row, T2* out) {
    using T = typename RealOf<T2>::T;
    const T ur = row[0].x, ut = row[0].y, uz = row[1].x;
    const T orr = row[1].y, ot = row[2].x, oz = row[2].y;
    const T wr = row[3].x, wt = row[3].y, wz = row[4].x;
    const T Grr = row[4].y, Grt = row[5].x, Grz = row[5].y;
    const T Gtr = row[6].x, Gtt = row[6].y, Gtz = row[7].x;
    const T Gzr = row[7].y, Gzt = row[8].x, Gzz = row[8].y;
    const T pr = -(ut * oz - uz * ot) - (T)2 * (Grr * wr + Grt * wt + Grz * wz);
    const T pt = -(uz * orr - ur * oz) - (T)2 * (Gtr * wr + Gtt * wt + Gtz * wz);
    const T pz = -(ur * ot - ut * orr) - (T)2 * (Gzr * wr + Gzt * wt + Gzz * wz);
    out[0] = mk<T2>(pr, pt);
    out[1] = mk<T2>(pz, 0);
}

// ------------------------------------------------------------------ z pass + products
// One block per (j, theta_a) row.  The Hermitian z spectra of two real fields
// are packed into one complex inverse FFT; the pointwise products of the
// physical fields are formed; two real products are packed into one forward
// FFT and separated; the result is truncated to k <= K and scaled.
//   ZFWD: inputs u (3), w (3)          -> outputs u x w (3)
//   ZADJ: inputs u (3), w (3), g (3)   -> outputs w x g (3), g x u (3)
template <class T2, int MODE>
__global__ void k_zpass(Geo g, const T2* __restrict__ Y, T2* __restrict__ Z, ZScales sc, const T2* __restrict__ twg) {
    grid_dep_sync();
    using T = typename RealOf<T2>::T;
    constexpr int NIN = MODE == ZFWD ? 6 : (MODE == ZADJ ? 9 : 18);
    constexpr int NPI = (NIN + 1) / 2;
    constexpr int NOUT = MODE == ZADJ ? 6 : 3;
    constexpr int NPO = (NOUT + 1) / 2;
    constexpr int LD = NPI;  // NPI >= NPO
    extern __shared__ __align__(16) unsigned char smem[];
    const int N = g.nzp, K = g.K, nk = g.nk;
    T2* bufA = reinterpret_cast<T2*>(smem);
    T2* bufB = bufA + N * LD;
    T2* tw = bufB + N * LD;
    const int a = blockIdx.x, j = blockIdx.y;
    const size_t poff = (size_t)g.slot[blockIdx.z] * g.ps;  // batch entry blockIdx.z
    Y += poff;
    Z += poff;
    for (int i = threadIdx.x; i < N; i += blockDim.x) tw[i] = twg[i];
    // Hermitian-extended spectra, two fields per column
    for (int p = 0; p < NPI; ++p)
    for (int n = threadIdx.x; n < N; n += blockDim.x) {
        int k = -1;
        bool neg = false;
        if (n <= K) k = n;
        else if (n >= N - K) { k = N - n; neg = true; }
        T2 q = mk<T2>(0, 0);
        if (k >= 0) {
            const int f1 = 2 * p, f2 = 2 * p + 1;
            T2 y1 = Y[((size_t)(f1 * g.nr + j) * g.nt + a) * nk + k];
            T2 h1 = k == 0 ? mk<T2>(zs<T>(sc.h0, sc.fh0, f1) * y1.x, 0)
                           : mk<T2>(zs<T>(sc.hk, sc.fhk, f1) * y1.x, zs<T>(sc.hk, sc.fhk, f1) * y1.y);
            T2 h2 = mk<T2>(0, 0);
            if (f2 < NIN) {
                T2 y2 = Y[((size_t)(f2 * g.nr + j) * g.nt + a) * nk + k];
                h2 = k == 0 ? mk<T2>(zs<T>(sc.h0, sc.fh0, f2) * y2.x, 0)
                            : mk<T2>(zs<T>(sc.hk, sc.fhk, f2) * y2.x, zs<T>(sc.hk, sc.fhk, f2) * y2.y);
            }
            if (!neg) q = mk<T2>(h1.x - h2.y, h1.y + h2.x);   // H1 + i H2
            else q = mk<T2>(h1.x + h2.y, -h1.y + h2.x);       // conj(H1) + i conj(H2)
        }
        bufA[n * LD + p] = q;
    }
    __syncthreads();
    T2* ph = fft_cols<T2, NPI, LD, +1>(bufA, bufB, N, tw);
    T2* pr = (ph == bufA) ? bufB : bufA;
    for (int n = threadIdx.x; n < N; n += blockDim.x) {
        const T2* row = ph + n * LD;
        const T ur = row[0].x, ut = row[0].y, uz = row[1].x;
        const T wr = row[1].y, wt = row[2].x, wz = row[2].y;
        T2* o = pr + n * LD;
        if (MODE == ZFWD) {
            o[0] = mk<T2>(ut * wz - uz * wt, uz * wr - ur * wz);
            o[1] = mk<T2>(ur * wt - ut * wr, 0);
        } else if (MODE == ZCADJ) {
            cadj_products<T2>(row, o);
        } else {
            const T gr = row[3].x, gt = row[3].y, gz = row[4].x;
            // w x g
            o[0] = mk<T2>(wt * gz - wz * gt, wz * gr - wr * gz);
            // (w x g)_z, (g x u)_r
            o[1] = mk<T2>(wr * gt - wt * gr, gt * uz - gz * ut);
            // (g x u)_theta, (g x u)_z
            o[2] = mk<T2>(gz * ur - gr * uz, gr * ut - gt * ur);
        }
    }
    __syncthreads();
    T2* sp = fft_cols<T2, NPO, LD, -1>(pr, ph, N, tw);
    for (int p = 0; p < NPO; ++p)
    for (int k = threadIdx.x; k < nk; k += blockDim.x) {
        const T2 P = sp[k * LD + p];
        const T2 Pm = sp[((N - k) % N) * LD + p];
        const int o1 = 2 * p, o2 = 2 * p + 1;
        const T s1 = k == 0 ? zs<T>(sc.o0, sc.fo0, o1) : zs<T>(sc.ok, sc.fok, o1);
        T2 z1 = mk<T2>((T)0.5 * (P.x + Pm.x) * s1, (T)0.5 * (P.y - Pm.y) * s1);
        Z[((size_t)(o1 * g.nr + j) * g.nt + a) * nk + k] = z1;
        if (o2 < NOUT) {
            const T s2 = k == 0 ? zs<T>(sc.o0, sc.fo0, o2) : zs<T>(sc.ok, sc.fok, o2);
            T2 z2 = mk<T2>((T)0.5 * (P.y + Pm.y) * s2, (T)-0.5 * (P.x - Pm.x) * s2);
            Z[((size_t)(o2 * g.nr + j) * g.nt + a) * nk + k] = z2;
        }
    }
}

// ------------------------------------------------------------------ fixed-point transforms
// The FP64 transforms run in 64-bit fixed point (dev_x64.cuh): an FP64 addition
// takes 77 cycles of its pipe, a 64-bit integer one about 2, and a product by a
// twiddle factor (62 fractional bits) four IMAD.WIDE of 4.2.  The values of a
// transform share one exponent.  For spectra it is chosen from the sum of the
// magnitudes of the inputs, which bounds every intermediate result: a unit is
// 2^-60 of that sum.  The forward z transform takes its values, products of
// physical fields, at full length (the largest below 2^58, moved there in the
// first stage) and divides them by the power of two that the stages so far can
// have multiplied them by (SCALE).  Nothing can wrap either way.
struct fx2 {
    long long x, y;
};
constexpr int kXT = 62;  // fractional bits of a twiddle factor
__device__ __forceinline__ fx2 fx_add(fx2 a, fx2 b) { return {a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ fx2 fx_sub(fx2 a, fx2 b) { return {a.x - b.x, a.y - b.y}; }
// (a c + b s) 2^-SH with multipliers of kXT fractional bits, |c|, |s| <= 1, |a|, |b| < 2^61
template <int SH> __device__ __forceinline__ long long fx_dot2(xdig a, int2 c, xdig b, int2 s) {
    long long m = x_mad(s.y, b.l, x_mad(s.x, b.h, x_mad(c.y, a.l, x_mad(c.x, a.h, 1ll << (kXT - 33 + SH)))));
    const long long l0 = x_mul(c.x, a.l), l1 = x_mul(s.x, b.l), h = x_mad(s.y, b.h, x_mul(c.y, a.h));
    m += (long long)(int)(l0 >> 32) + (long long)(int)(l1 >> 32);
    if (SH > 64 - kXT) return ((h << (64 - kXT - 1)) + (m >> (kXT - 31))) >> (SH - 1);
    return (h << (64 - kXT - SH > 0 ? 64 - kXT - SH : 0)) + (m >> (kXT - 32 + SH));
}
// v e^{SIGN i phi} 2^-SH, w = (cos, -sin) of phi
template <int SIGN, int SH> __device__ __forceinline__ fx2 fx_rot(fx2 v, int4 w) {
    const xdig x = x_split(v.x), y = x_split(v.y);
    const int2 c = make_int2(w.x, w.y), s = make_int2(w.z, w.w), ns = make_int2(-w.z, -w.w);
    // e^{-i phi} = c + i s: (x c - y s, y c + x s); e^{+i phi} = c - i s
    return SIGN < 0 ? fx2{fx_dot2<SH>(x, c, y, ns), fx_dot2<SH>(y, c, x, s)}
                    : fx2{fx_dot2<SH>(x, c, y, s), fx_dot2<SH>(y, c, x, ns)};
}
constexpr long long kSqrt34 = 3993837246235628775ll;  // sqrt(3)/2 2^62
// v c, c = C 2^-kXT
template <long long C> __device__ __forceinline__ long long fx_mul(long long v) {
    const int2 c = make_int2((int)(unsigned)(C & 0xFFFFFFFFll), (int)((C + (1ll << 31)) >> 32));
    return x_prod<kXT>(c, x_split(v), 1ll << (kXT - 33));
}
template <int SIGN> __device__ __forceinline__ fx2 fx_quarter(fx2 v) {  // SIGN i v
    return SIGN > 0 ? fx2{-v.y, v.x} : fx2{v.y, -v.x};
}
template <int R, int SIGN> __device__ __forceinline__ void fx_dft(fx2* v) {
    if constexpr (R == 2) {
        const fx2 a = v[0], b = v[1];
        v[0] = fx_add(a, b);
        v[1] = fx_sub(a, b);
    } else if constexpr (R == 4) {
        const fx2 s02 = fx_add(v[0], v[2]), d02 = fx_sub(v[0], v[2]), s13 = fx_add(v[1], v[3]);
        const fx2 id = fx_quarter<SIGN>(fx_sub(v[1], v[3]));
        v[0] = fx_add(s02, s13);
        v[2] = fx_sub(s02, s13);
        v[1] = fx_add(d02, id);
        v[3] = fx_sub(d02, id);
    } else if constexpr (R == 6) {  // n = 3 a + 2 b, k = 3 (k mod 2) + 4 (k mod 3) mod 6: no turns in between
        fx2 t[2][3];
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const fx2 p = v[(2 * b) % 6], q = v[(3 + 2 * b) % 6];
            t[0][b] = fx_add(p, q);
            t[1][b] = fx_sub(p, q);
        }
        fx_dft<3, SIGN>(t[0]);
        fx_dft<3, SIGN>(t[1]);
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            v[(4 * b) % 6] = t[0][b];
            v[(3 + 4 * b) % 6] = t[1][b];
        }
    } else {  // R == 3
        const fx2 t1 = fx_add(v[1], v[2]), d = fx_sub(v[1], v[2]);
        const fx2 t2 = {v[0].x - (t1.x >> 1), v[0].y - (t1.y >> 1)};
        const fx2 t3 = fx_quarter<SIGN>(fx2{fx_mul<kSqrt34>(d.x), fx_mul<kSqrt34>(d.y)});
        v[0] = fx_add(v[0], t1);
        v[1] = fx_add(t2, t3);
        v[2] = fx_sub(t2, t3);
    }
}
// bits that n values of a sum can add
__host__ __device__ constexpr int fx_growth(int n) {
    int b = 0;
    while ((1 << b) < n) ++b;
    return b;
}
// Bits by which the first stage moves up the real (i = 0) and imaginary part of
// column col, so that the largest value fills `room` bits.
struct xlift {
    const int* top;  // bits of the largest values of the columns' parts
    int room;
    __device__ __forceinline__ int operator()(int col, int i) const { return max(room - top[2 * col + i], 0); }
};
// the Stockham stages of fft_cols in fixed point, scaled by 2^-SH
template <int R, int NCOL, int LD, int SIGN, int SH>
__device__ __forceinline__ void fx_stage(const fx2* __restrict__ a, fx2* __restrict__ b, int N, int Ns, int lgNs,
                                         const int4* __restrict__ tw, const xlift* lift) {
    const int stride = N / R, nb = stride * NCOL, tstep = N / (Ns * R);
    for (int idx = threadIdx.x; idx < nb; idx += blockDim.x) {
        const int col = idx % NCOL, jb = idx / NCOL;
        int q, kk;
        if (lgNs >= 0) {
            q = jb >> lgNs;
            kk = jb & (Ns - 1);
        } else {
            q = jb / Ns;
            kk = jb - q * Ns;
        }
        fx2 v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = a[(jb + r * stride) * LD + col];
        if (lift) {
            const int lx = (*lift)(col, 0), ly = (*lift)(col, 1);
#pragma unroll
            for (int r = 0; r < R; ++r) v[r] = {v[r].x << lx, v[r].y << ly};
        }
        if (Ns > 1) {
            const int tb = kk * tstep;
#pragma unroll
            for (int r = 1; r < R; ++r) v[r] = fx_rot<SIGN, SH>(v[r], tw[r * tb]);
            if (SH) v[0] = {(v[0].x + (1ll << SH >> 1)) >> SH, (v[0].y + (1ll << SH >> 1)) >> SH};
        }
        fx_dft<R, SIGN>(v);
        const int idxD = q * Ns * R + kk;
#pragma unroll
        for (int r = 0; r < R; ++r) b[(idxD + r * Ns) * LD + col] = v[r];
    }
}
// halvings: what the result is to be multiplied by, as an exponent of 2 (SCALE).
// The first stage is not scaled; after it a value is at most 2^fx_growth(first
// radix) times the largest input, and stays so.
template <int NCOL, int LD, int SIGN, bool SCALE = false>
__device__ fx2* fx_cols(fx2* a, fx2* b, int N, const int4* tw, int* halvings = nullptr, const xlift* lift = nullptr) {
    int n2 = __ffs(N) - 1, n3 = 0;
    for (int t = N >> n2; t > 1; t /= 3) ++n3;
    int Ns = 1, lgNs = 0;
    auto next = [&](int R, int SH) {
        __syncthreads();
        fx2* t = a;
        a = b;
        b = t;
        if (SCALE && Ns > 1) *halvings += SH;
        Ns *= R;
        lift = nullptr;
    };
    // radix 4, a remaining 2 with a 3 as radix 6 (64x64x256 z pass, before its fields
    // had units of their own: 197 and 358 us; with radix 2 and 3 apart 215 and 387,
    // with radix 8 and 6 227 and 350).  Radix 4, 2 and 6 follow powers of four, so that
    // a stage's scale depends on the radix alone; radix 3 takes one or two bits (3, 9, 27, 81, 243 times: 2, 4, 5, 7, 8).
    for (; n2 >= 2; n2 -= 2) {
        fx_stage<4, NCOL, LD, SIGN, SCALE ? 2 : 0>(a, b, N, Ns, lgNs, tw, lift);
        next(4, 2);
        lgNs += 2;
    }
    if (n2 == 1 && n3 > 0) {
        fx_stage<6, NCOL, LD, SIGN, SCALE ? 3 : 0>(a, b, N, Ns, lgNs, tw, lift);
        next(6, 3);
        lgNs = -1;
        --n3;
    } else if (n2 == 1) {
        fx_stage<2, NCOL, LD, SIGN, SCALE ? 1 : 0>(a, b, N, Ns, lgNs, tw, lift);
        next(2, 1);
        lgNs += 1;
    }
    for (; n3 > 0; --n3) {
        const bool two = SCALE && fx_growth(3 * Ns) - fx_growth(Ns) == 2;
        if (two) fx_stage<3, NCOL, LD, SIGN, SCALE ? 2 : 0>(a, b, N, Ns, lgNs, tw, lift);
        else fx_stage<3, NCOL, LD, SIGN, SCALE ? 1 : 0>(a, b, N, Ns, lgNs, tw, lift);
        next(3, two ? 2 : 1);
        lgNs = -1;
    }
    return a;
}
// magnitude of x relative to 2^top as a count of 2^-19, rounded up (0 for zero);
// top: the exponent field of the largest value
__device__ __forceinline__ unsigned fx_count(double x, int top) {
    const int h = __double2hiint(x) & 0x7FFFFFFF, e = h >> 20;
    return e ? ((((unsigned)h & 0xFFFFFu) | 0x100000u) >> min(top - e + 1, 31)) + 1u : 0u;
}
// unit (as an exponent of 2) in which values sum to less than 2^bits, `sum` being
// the sum of their counts in steps of four
__device__ __forceinline__ int fx_unit(unsigned sum, int top, int bits) {
    return top - 1023 - 17 + (32 - __clz((int)sum)) - bits;
}
__device__ __forceinline__ int x_top(long long v) { return 64 - __clzll(v ^ (v >> 63)); }  // |v| <= 2^top

// The z pass in fixed point: contract of k_zpass (FP64), any length.  Bound by
// integer issue and its barriers (35% of the warps' slots in use at 64x64x256);
// 828 -> 208 us forward and 1308 -> 341 us adjoint against the FP64 Stockham
// kernel, 73 and 108 FP64 instructions a point at 77 cycles.  Every field has a
// unit of its own (the components of u and of w differ by orders of magnitude
// in streaky flows), and every output one from the larger of its two products:
// a component's error is 1.0e-16 to 2.3e-16 of its root mean square at 24 to 243
// points (FP64 arithmetic: 2e-16 to 6e-16, and up to 2e-12 where a small
// component shared a packed column with a large one).  At most 80 registers:
// 43.6 -> 41.9 us at 48x32x96, whose blocks are the smaller for it.
// The fields fall into the groups u, w and (mode ZADJ) g; g's input scale is gs
// for k = 0 and gs hs for k > 0, hs a power of two (hsh its exponent), and gs is
// part of the output scales o0, ok.
struct XScales {
    int hsh[3];
    double o0[6], ok[6];
};
constexpr int kXProd = 59;  // a product of two fields, each below 2^60, keeps its bits from here on
__device__ __forceinline__ long long fx_prod(xdig p, xdig q) {
    const long long m = x_mad(p.h, q.l, x_mul(p.l, q.h)) + (long long)(int)(x_mul(p.l, q.l) >> 32);
    return (x_mul(p.h, q.h) << (64 - kXProd)) + (m >> (kXProd - 32));
}
template <int MODE>
__global__ void __launch_bounds__(256, 3)
    k_zpass_x(Geo g, const double2* __restrict__ Y, double2* __restrict__ Z, XScales sc, const int4* __restrict__ twg) {
    grid_dep_sync();
    constexpr int NIN = MODE == ZFWD ? 6 : 9;
    constexpr int NPI = (NIN + 1) / 2;
    constexpr int NOUT = MODE == ZADJ ? 6 : 3;
    constexpr int NPO = (NOUT + 1) / 2;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int top_sh[NIN], max_sh[NIN], out_sh[NOUT][3], omax_sh[2 * NPO];
    __shared__ unsigned sum_sh[NIN];
    const int N = g.nzp, nk = g.nk;
    fx2* bufA = reinterpret_cast<fx2*>(smem);
    fx2* bufB = bufA + N * NPI;
    int4* tw = reinterpret_cast<int4*>(bufB + N * NPI);
    auto at = [](int n, int p) { return n * NPI + p; };
    const int a = blockIdx.x, j = blockIdx.y;
    const size_t poff = (size_t)g.slot[blockIdx.z] * g.ps;
    Y += poff;
    Z += poff;
    if (threadIdx.x < NIN) top_sh[threadIdx.x] = max_sh[threadIdx.x] = sum_sh[threadIdx.x] = 0;
    if (threadIdx.x < 2 * NPO) omax_sh[threadIdx.x] = 0;
    for (int i = threadIdx.x; i < N; i += blockDim.x) tw[i] = twg[i];
    __syncthreads();
    // inputs into bufB as they are, the largest exponent of each field
    double2* raw = reinterpret_cast<double2*>(bufB);  // [NIN][nk]
    {
        int mx[NIN] = {};
        for (int k = threadIdx.x; k < nk; k += blockDim.x) {
            double2 y[NIN];
#pragma unroll
            for (int f = 0; f < NIN; ++f) y[f] = Y[((size_t)(f * g.nr + j) * g.nt + a) * nk + k];
#pragma unroll
            for (int f = 0; f < NIN; ++f) {
                if (k == 0) y[f].y = 0;
                raw[f * nk + k] = y[f];
                mx[f] = max(mx[f], max(__double2hiint(y[f].x) & 0x7FFFFFFF, __double2hiint(y[f].y) & 0x7FFFFFFF));
            }
        }
#pragma unroll
        for (int f = 0; f < NIN; ++f) mx[f] = __reduce_max_sync(0xffffffffu, mx[f]);
        if ((threadIdx.x & 31) == 0)
#pragma unroll
            for (int f = 0; f < NIN; ++f) atomicMax(&top_sh[f], mx[f]);
    }
    __syncthreads();
    bool bad = false;
    {
        unsigned sum[NIN] = {};
        int top[NIN];
#pragma unroll
        for (int f = 0; f < NIN; ++f) {
            bad = bad || top_sh[f] >= 0x7FF00000;
            top[f] = top_sh[f] >> 20;
        }
        for (int k = threadIdx.x; k < nk; k += blockDim.x) {
#pragma unroll
            for (int f = 0; f < NIN; ++f) {
                const double2 y = raw[f * nk + k];
                sum[f] += (fx_count(y.x, top[f]) + fx_count(y.y, top[f]) + 3u) >> 2;  // nk up to 2^12
            }
        }
#pragma unroll
        for (int f = 0; f < NIN; ++f) sum[f] = __reduce_add_sync(0xffffffffu, sum[f]);
        if ((threadIdx.x & 31) == 0)
#pragma unroll
            for (int f = 0; f < NIN; ++f) atomicAdd(&sum_sh[f], sum[f]);
    }
    __syncthreads();
    // |f| <= 2 sum of the magnitudes < 2^60 units; a packed column < 2^61
    auto unit = [&](int f) { return max(fx_unit(sum_sh[f], top_sh[f] >> 20, 59), -kXTop); };
    // Hermitian-extended spectra, two fields per column
    for (int n = threadIdx.x; n < NPI * (N - 2 * nk + 1); n += blockDim.x) bufA[at(nk, n)] = {0, 0};
#pragma unroll
    for (int p = 0; p < NPI; ++p) {
        constexpr int none = NIN;
        const int f1 = 2 * p, f2 = 2 * p + 1 < NIN ? 2 * p + 1 : none, g1 = f1 / 3, g2 = f2 == none ? g1 : f2 / 3;
        const int e1 = unit(f1), e2 = f2 == none ? e1 : unit(f2);
        const xunit u01 = x_unit(e1), u02 = x_unit(e2);  // k = 0
        const xunit u1 = MODE == ZADJ ? x_unit(e1 + sc.hsh[g1]) : u01, u2 = MODE == ZADJ ? x_unit(e2 + sc.hsh[g2]) : u02;
        for (int k = threadIdx.x; k < nk; k += blockDim.x) {
            const double2 y1 = raw[f1 * nk + k], y2 = f2 == none ? make_double2(0, 0) : raw[f2 * nk + k];
            const xunit v1 = k ? u1 : u01, v2 = k ? u2 : u02;
            const fx2 h1 = {x_load(y1.x, v1), x_load(y1.y, v1)};
            fx2 h2 = {0, 0};
            if (f2 != none) h2 = {x_load(y2.x, v2), x_load(y2.y, v2)};
            bufA[at(k, p)] = {h1.x - h2.y, h1.y + h2.x};                    // H1 + i H2
            if (k > 0) bufA[at(N - k, p)] = {h1.x + h2.y, h2.x - h1.y};  // conj(H1) + i conj(H2)
        }
    }
    __syncthreads();
    fx2* ph = fx_cols<NPI, NPI, +1>(bufA, bufB, N, tw);
    fx2* pr = ph == bufA ? bufB : bufA;
    // largest physical values of the fields, for the units of the products (a field
    // that is 0 stays 0, whatever rounding errors its column has)
    {
        long long mx[NIN] = {};
        for (int n = threadIdx.x; n < N; n += blockDim.x) {
#pragma unroll
            for (int f = 0; f < NIN; ++f) {
                const fx2 c = ph[at(n, f / 2)];
                const long long x = f % 2 ? c.y : c.x;
                mx[f] |= x ^ (x >> 63);
            }
        }
        int m[NIN];
#pragma unroll
        for (int f = 0; f < NIN; ++f) m[f] = __reduce_max_sync(0xffffffffu, top_sh[f] ? x_top(mx[f]) : 0);
        if ((threadIdx.x & 31) == 0)
#pragma unroll
            for (int f = 0; f < NIN; ++f) atomicMax(&max_sh[f], m[f]);
    }
    __syncthreads();
    // Output f = p q - r t: (w x g) for the adjoint pass, then u x w or g x u.
    // The fields are moved up to 2^60 first, so that the products take shifts
    // known at compile time, but for the smaller of an output's two, which moves
    // down to the other's unit.  An output stays below 2^room, and what the
    // first stage of the forward transform adds up, four or three packed complex
    // values (six where N is an odd multiple of two), below 2^61.  out_sh: the
    // output's unit and what its two products are moved down by.
    const int room = N % 4 == 2 ? 57 : 58, drop = 121 - room - kXProd;
    auto factors = [](int f, int& p, int& q, int& r, int& t) {
        const int a = MODE == ZFWD ? 0 : (f < 3 ? 3 : 6), b = MODE == ZFWD ? 3 : (f < 3 ? 6 : 0), c = f % 3;
        p = a + (c + 1) % 3;
        q = b + (c + 2) % 3;
        r = a + (c + 2) % 3;
        t = b + (c + 1) % 3;
    };
    if (threadIdx.x < NOUT) {
        int p, q, r, t;
        factors(threadIdx.x, p, q, r, t);
        const int none = -100000;  // of a product that is 0 everywhere
        auto top = [&](int f) { return unit(f) + max_sh[f]; };
        const int t1 = max_sh[p] && max_sh[q] ? top(p) + top(q) : none;
        const int t2 = max_sh[r] && max_sh[t] ? top(r) + top(t) : none, tm = max(t1, t2);
        // an output that is 0 stays 0: a unit below the subnormals for the rounding
        // errors of the one that shares its column
        out_sh[threadIdx.x][0] = tm == none ? -4000 : tm + 1 - room;
        out_sh[threadIdx.x][1] = min(tm - t1, 63);
        out_sh[threadIdx.x][2] = min(tm - t2, 63);
    }
    __syncthreads();
    int up[NIN];
#pragma unroll
    for (int f = 0; f < NIN; ++f) up[f] = max_sh[f] ? max(60 - max_sh[f], 0) : 0;
    long long omx[NOUT] = {};
    for (int n = threadIdx.x; n < N; n += blockDim.x) {
        xdig v[2 * NPI];  // the fields' digits
#pragma unroll
        for (int p = 0; p < NPI; ++p) {
            const fx2 c = ph[at(n, p)];
            v[2 * p] = x_split(c.x << up[2 * p]);
            if (2 * p + 1 < NIN) v[2 * p + 1] = x_split(c.y << up[2 * p + 1]);
        }
        long long o[2 * NPO] = {};
#pragma unroll
        for (int f = 0; f < NOUT; ++f) {
            int p = 0, q = 0, r = 0, t = 0;
            factors(f, p, q, r, t);
            const long long d = (fx_prod(v[p], v[q]) >> out_sh[f][1]) - (fx_prod(v[r], v[t]) >> out_sh[f][2]);
            o[f] = (d + (1ll << drop >> 1)) >> drop;
            omx[f] |= o[f] ^ (o[f] >> 63);
        }
#pragma unroll
        for (int p = 0; p < NPO; ++p) pr[at(n, p)] = {o[2 * p], o[2 * p + 1]};
    }
    {
        int m[NOUT];
#pragma unroll
        for (int f = 0; f < NOUT; ++f) m[f] = __reduce_max_sync(0xffffffffu, x_top(omx[f]));
        if ((threadIdx.x & 31) == 0)
#pragma unroll
            for (int f = 0; f < NOUT; ++f) atomicMax(&omax_sh[f], m[f]);
    }
    __syncthreads();
    // the bits that the bound left unused (factors of two in each factor, and
    // maxima that do not meet at one z), usually two to four
    const xlift lift = {omax_sh, room};
    int halvings = 0;
    fx2* sp = fx_cols<NPO, NPI, -1, true>(pr, ph, N, tw, &halvings, &lift);
    const int nan = bad ? 0x7FF80000 : 0;
    const int Eh = halvings - 1;  // the separation's 1/2
    bool far = false;
#pragma unroll
    for (int f = 0; f < NOUT; ++f) {
        const int e = out_sh[f][0] - lift(f / 2, f % 2) + Eh;
        far = far || e < -1000 || e > 900;
    }
    auto put = [&](int f, int k, long long x, long long y) {
        const int e = out_sh[f][0] - lift(f / 2, f % 2) + Eh;
        const double s = k == 0 ? sc.o0[f] : sc.ok[f];
        double2 z;
        if (far) z = make_double2(x_store_any(x, e, nan) * s, x_store_any(y, e, nan) * s);
        else z = make_double2(x_store(x, e, nan) * s, x_store(y, e, nan) * s);
        Z[((size_t)(f * g.nr + j) * g.nt + a) * nk + k] = z;
    };
#pragma unroll
    for (int p = 0; p < NPO; ++p)
        for (int k = threadIdx.x; k < nk; k += blockDim.x) {
            const fx2 P = sp[at(k, p)], Q = sp[at(k ? N - k : 0, p)];
            put(2 * p, k, P.x + Q.x, P.y - Q.y);
            if (2 * p + 1 < NOUT) put(2 * p + 1, k, P.y + Q.y, Q.x - P.x);
        }
}

// The theta transforms in fixed point, any length: contract of k_synth_theta and
// k_anal_theta (FP64).  206 -> 68 us (synthesis) and 158 -> 69 us (analysis) at
// 64x64x256 against the FP64 two-pass kernels.  A block takes KB columns k of one
// (field, j), all in one unit (the z pass sums over k, so a column far below its
// neighbours does not count there: on spectra falling as e^-k/4 to e^-k the error
// of every k is 5 to 50 times below that of FP64 transforms).  Rows of `in` values from memory into `raw`, and the unit in
// which the magnitudes of every column sum to less than 2^61; bad: infinities or NaN.
template <int KB, class F>
__device__ __forceinline__ int fx_columns(int rows, int kw, double2* raw, F&& load, int* top_sh, unsigned* sum_sh, bool& bad) {
    const int kk = threadIdx.x % KB, r0 = threadIdx.x / KB, dr = blockDim.x / KB;  // a thread keeps to one column
    if (threadIdx.x == 0) *top_sh = 0;
    if (threadIdx.x < KB) sum_sh[threadIdx.x] = 0;
    __syncthreads();
    int mx = 0;
    for (int r = r0; r < rows; r += dr) {
        const double2 y = kk < kw ? load(r, kk) : make_double2(0, 0);
        raw[r * KB + kk] = y;
        mx = max(mx, max(__double2hiint(y.x) & 0x7FFFFFFF, __double2hiint(y.y) & 0x7FFFFFFF));
    }
    mx = __reduce_max_sync(0xffffffffu, mx);
    if ((threadIdx.x & 31) == 0) atomicMax(top_sh, mx);
    __syncthreads();
    mx = *top_sh;
    bad = mx >= 0x7FF00000;
    const int top = mx >> 20;
    unsigned s = 0;
    for (int r = r0; r < rows; r += dr) {
        const double2 y = raw[r * KB + kk];
        s += (fx_count(y.x, top) + fx_count(y.y, top) + 3u) >> 2;
    }
    atomicAdd(&sum_sh[kk], s);
    __syncthreads();
    s = 0;
#pragma unroll
    for (int i = 0; i < KB; ++i) s = max(s, sum_sh[i]);
    return max(fx_unit(s, top, 61), -kXTop);
}
__device__ __forceinline__ double2 fx_out(fx2 v, int E, bool far, int nan) {
    return far ? make_double2(x_store_any(v.x, E, nan), x_store_any(v.y, E, nan))
               : make_double2(x_store(v.x, E, nan), x_store(v.y, E, nan));
}

template <int KB>
__global__ void k_synth_x(Geo g, FieldPtrs f, double2* __restrict__ Y, const int4* __restrict__ twg) {
    grid_dep_sync();
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int top_sh;
    __shared__ unsigned sum_sh[KB];
    fx2* buf0 = reinterpret_cast<fx2*>(smem);
    fx2* buf1 = buf0 + g.nt * KB;
    int4* tw = reinterpret_cast<int4*>(buf1 + g.nt * KB);
    const int k0 = blockIdx.x * KB, j = blockIdx.y;
    const int nf = gridDim.z / g.nb, b = blockIdx.z / nf, fi = blockIdx.z - b * nf, slot = g.slot[b];
    Y += (size_t)slot * g.ps;
    const int kw = min(KB, g.nk - k0);
    for (int i = threadIdx.x; i < g.nt; i += blockDim.x) tw[i] = twg[i];
    const double2* src = f.in[fi] + (size_t)slot * g.fs + (size_t)j * g.nm * g.nk + k0;
    double2* raw = reinterpret_cast<double2*>(buf1);
    bool bad;
    const int E = fx_columns<KB>(g.nm, kw, raw, [&](int r, int kk) { return src[(size_t)r * g.nk + kk]; }, &top_sh, sum_sh, bad);
    const xunit u = x_unit(E);
    for (int i = threadIdx.x; i < g.nt * KB; i += blockDim.x) {
        const int n = i / KB, m = n <= g.M ? n : n - g.nt;  // zero-padded beyond |m| <= M
        fx2 v = {0, 0};
        if (m >= -g.M) {
            const double2 y = raw[(m + g.M) * KB + i % KB];
            v = {x_load(y.x, u), x_load(y.y, u)};
        }
        buf0[i] = v;
    }
    __syncthreads();
    const fx2* res = fx_cols<KB, KB, +1>(buf0, buf1, g.nt, tw);
    const int nan = bad ? 0x7FF80000 : 0;
    const bool far = E < -1000 || E > 900;
    double2* dst = Y + ((size_t)(fi * g.nr + j) * g.nt) * g.nk + k0;
    for (int i = threadIdx.x; i < g.nt * KB; i += blockDim.x) {
        const int a = i / KB, kk = i % KB;
        if (kk < kw) dst[(size_t)a * g.nk + kk] = fx_out(res[i], E, far, nan);
    }
}

template <int KB>
__global__ void k_anal_x(Geo g, FieldPtrs f, const double2* __restrict__ Z, const int4* __restrict__ twg) {
    grid_dep_sync();
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int top_sh;
    __shared__ unsigned sum_sh[KB];
    fx2* buf0 = reinterpret_cast<fx2*>(smem);
    fx2* buf1 = buf0 + g.nt * KB;
    int4* tw = reinterpret_cast<int4*>(buf1 + g.nt * KB);
    const int k0 = blockIdx.x * KB, j = blockIdx.y;
    const int nf = gridDim.z / g.nb, b = blockIdx.z / nf, fi = blockIdx.z - b * nf, slot = g.slot[b];
    Z += (size_t)slot * g.ps;
    const int kw = min(KB, g.nk - k0);
    for (int i = threadIdx.x; i < g.nt; i += blockDim.x) tw[i] = twg[i];
    const double2* src = Z + ((size_t)(fi * g.nr + j) * g.nt) * g.nk + k0;
    double2* raw = reinterpret_cast<double2*>(buf1);
    bool bad;
    const int E = fx_columns<KB>(g.nt, kw, raw, [&](int r, int kk) { return src[(size_t)r * g.nk + kk]; }, &top_sh, sum_sh, bad);
    const xunit u = x_unit(E);
    for (int i = threadIdx.x; i < g.nt * KB; i += blockDim.x) {
        const double2 y = raw[i];
        buf0[i] = {x_load(y.x, u), x_load(y.y, u)};
    }
    __syncthreads();
    const fx2* res = fx_cols<KB, KB, -1>(buf0, buf1, g.nt, tw);
    const int nan = bad ? 0x7FF80000 : 0;
    const bool far = E < -1000 || E > 900;
    const size_t base = (size_t)slot * g.fs + (size_t)j * g.nm * g.nk + k0;
    double2* dst = f.out[fi] + base;
    const double2* add = f.add[fi] ? f.add[fi] + base : nullptr;
    for (int i = threadIdx.x; i < g.nm * KB; i += blockDim.x) {
        const int im = i / KB, kk = i % KB, m = im - g.M;
        if (kk >= kw) continue;
        const size_t o = (size_t)im * g.nk + kk;
        fx2 v = res[(m < 0 ? m + g.nt : m) * KB + kk];
        int e = E;
        if (k0 + kk == 0) {  // Hermitian part
            const fx2 w = res[(m > 0 ? g.nt - m : -m) * KB + kk];
            v = {v.x + w.x, v.y - w.y};
            e = E - 1;
        }
        double2 z = fx_out(v, e, far, nan);
        if (add) {
            const double2 y = add[o];
            z = make_double2(z.x + y.x, z.y + y.y);
        }
        dst[o] = z;
    }
}

// ------------------------------------------------------------------ theta analysis
// X_f[j][m][k] = sum_a Z_f[j][a][k] e^{-i m theta_a}, |m| <= M, with the k = 0
// plane projected onto Hermitian symmetry.
template <class T2, int KB>
__global__ void k_anal_theta(Geo g, FieldPtrs f, const T2* __restrict__ Z, const T2* __restrict__ twg) {
    grid_dep_sync();
    extern __shared__ __align__(16) unsigned char smem[];
    T2* buf0 = reinterpret_cast<T2*>(smem);
    T2* buf1 = buf0 + g.nt * KB;
    T2* tw = buf1 + g.nt * KB;
    const int k0 = blockIdx.x * KB, j = blockIdx.y;
    const int nf = gridDim.z / g.nb, b = blockIdx.z / nf, fi = blockIdx.z - b * nf, slot = g.slot[b];
    const size_t off = (size_t)slot * g.fs;
    Z += (size_t)slot * g.ps;
    const int kw = min(KB, g.nk - k0);
    for (int i = threadIdx.x; i < g.nt; i += blockDim.x) tw[i] = twg[i];
    const T2* src = Z + ((size_t)(fi * g.nr + j) * g.nt) * g.nk;
    for (int i = threadIdx.x; i < g.nt * KB; i += blockDim.x) {
        const int a = i / KB, kk = i % KB;
        buf0[i] = kk < kw ? src[(size_t)a * g.nk + k0 + kk] : mk<T2>(0, 0);
    }
    __syncthreads();
    T2* res = fft_cols<T2, KB, KB, -1>(buf0, buf1, g.nt, tw);
    const size_t base = off + (size_t)j * g.nm * g.nk;
    float2* dstf = f.outf[fi] ? f.outf[fi] + base : nullptr;
    double2* dst = dstf ? nullptr : f.out[fi] + base;
    const double2* add = f.add[fi] ? f.add[fi] + base : nullptr;
    for (int i = threadIdx.x; i < g.nm * KB; i += blockDim.x) {
        const int im = i / KB, kk = i % KB;
        if (kk >= kw) continue;
        const int m = im - g.M;
        const size_t o = (size_t)im * g.nk + k0 + kk;
        if (dstf) {
            using T = typename RealOf<T2>::T;
            T2 v = res[(m < 0 ? m + g.nt : m) * KB + kk];
            if (k0 + kk == 0) {
                const T2 vm = res[(m > 0 ? g.nt - m : -m) * KB + kk];
                v = mk<T2>((T)0.5 * (v.x + vm.x), (T)0.5 * (v.y - vm.y));
            }
            dstf[o] = v;
            continue;
        }
        double2 v = to_d(res[(m < 0 ? m + g.nt : m) * KB + kk]);
        if (k0 + kk == 0) {
            double2 vm = to_d(res[(m > 0 ? g.nt - m : -m) * KB + kk]);
            v = make_double2(0.5 * (v.x + vm.x), 0.5 * (v.y - vm.y));
        }
        if (add) v = make_double2(v.x + add[o].x, v.y + add[o].y);
        dst[o] = v;
    }
}

// ------------------------------------------------------------------ two-pass register FFT
// A length N = N1 N2 transform as N2 DFTs of length N1 on stride-N2
// subsequences, a twiddle W_N^{n2 k1}, and N1 DFTs of length N2 on
// contiguous runs (Cooley-Tukey with one shared-memory exchange).  Each DFT
// runs in the registers of one thread, fully unrolled, with its internal
// twiddles folded to compile-time constants.  The inverse transforms below
// take the spectrum in natural order and leave physical index k1 + N1 k2 in
// slot k2 + N2 k1; the forward transforms take that slot order back to a
// natural-order spectrum.  The physical-space work in between is pointwise,
// so the permutation never has to be undone.

// cos and sin of 2 pi e / L evaluated by the compiler: e is reduced to a
// quadrant with integer arithmetic, the remaining angle x in [0, pi/2) goes
// through the Taylor series of sin and cos (16 terms, below 1e-17 there).
namespace ct {
constexpr double kTwoPi = 6.283185307179586476925286766559;
__host__ __device__ constexpr double tsin(double x) {
    double t = x, s = x;
    for (int i = 1; i < 16; ++i) {
        t *= -x * x / ((2.0 * i) * (2.0 * i + 1.0));
        s += t;
    }
    return s;
}
__host__ __device__ constexpr double tcos(double x) {
    double t = 1.0, s = 1.0;
    for (int i = 1; i < 16; ++i) {
        t *= -x * x / ((2.0 * i - 1.0) * (2.0 * i));
        s += t;
    }
    return s;
}
__host__ __device__ constexpr double cos2pi(long e, long L) {
    const long n = ((e % L) + L) % L, q = 4 * n / L;
    const double x = kTwoPi * (double)(4 * n - q * L) / (4.0 * (double)L);
    return q == 0 ? tcos(x) : q == 1 ? -tsin(x) : q == 2 ? -tcos(x) : tsin(x);
}
__host__ __device__ constexpr double sin2pi(long e, long L) {
    const long n = ((e % L) + L) % L, q = 4 * n / L;
    const double x = kTwoPi * (double)(4 * n - q * L) / (4.0 * (double)L);
    return q == 0 ? tsin(x) : q == 1 ? tcos(x) : q == 2 ? -tsin(x) : -tcos(x);
}
}  // namespace ct

// x e^{SIGN 2 pi i E / L} for a compile-time exponent E
template <class T2, int L, int SIGN, int E>
__device__ __forceinline__ T2 twc(T2 x) {
    using T = typename RealOf<T2>::T;
    constexpr int e = ((E % L) + L) % L;
    if constexpr (e == 0) {
        return x;
    } else if constexpr (2 * e == L) {
        return mk<T2>(-x.x, -x.y);
    } else if constexpr (4 * e == L) {  // SIGN i
        return SIGN > 0 ? mk<T2>(-x.y, x.x) : mk<T2>(x.y, -x.x);
    } else if constexpr (4 * e == 3 * L) {  // -SIGN i
        return SIGN > 0 ? mk<T2>(x.y, -x.x) : mk<T2>(-x.y, x.x);
    } else {
        constexpr T c = (T)ct::cos2pi(e, L);
        constexpr T sn = (T)(SIGN * ct::sin2pi(e, L));
        return mk<T2>(c * x.x - sn * x.y, c * x.y + sn * x.x);
    }
}

// x e^{SIGN 2 pi i e / N} for a run-time exponent 0 <= e < N, from the table
// tw[n] = e^{-2 pi i n / N}
template <class T2, int SIGN>
__device__ __forceinline__ T2 twr(T2 x, const T2* tw, int e) {
    T2 w = tw[e];
    if (SIGN > 0) w.y = -w.y;
    return cmul(x, w);
}

template <class T2, int L, int SIGN, int R, int Q, int... I>
__device__ __forceinline__ void rtwiddle(T2 (&s)[R][Q], std::integer_sequence<int, I...>) {
    ((s[I / Q][I % Q] = twc<T2, L, SIGN, (I / Q) * (I % Q)>(s[I / Q][I % Q])), ...);
}

// In-register DFT X[k] = sum_n v[n] e^{SIGN 2 pi i n k / L}, L = 2^a 3^b:
// radix-2/3/4 butterflies at the leaves, mixed-radix Cooley-Tukey above them
// (n = a + R b, k = kb + Q ka).
template <class T2, int L, int SIGN>
__device__ __forceinline__ void rdft(T2 (&v)[L]) {
    using T = typename RealOf<T2>::T;
    if constexpr (L == 1) {
    } else if constexpr (L == 2) {
        const T2 a = v[0], b = v[1];
        v[0] = cadd(a, b);
        v[1] = csub(a, b);
    } else if constexpr (L == 3) {
        constexpr T h = (T)(SIGN * 0.86602540378443864676);  // SIGN sqrt(3)/2
        const T2 t1 = cadd(v[1], v[2]);
        const T2 t2 = mk<T2>(v[0].x - (T)0.5 * t1.x, v[0].y - (T)0.5 * t1.y);
        const T2 t3 = imul(csub(v[1], v[2]), h);
        v[0] = cadd(v[0], t1);
        v[1] = cadd(t2, t3);
        v[2] = csub(t2, t3);
    } else if constexpr (L == 4) {
        const T2 s02 = cadd(v[0], v[2]), d02 = csub(v[0], v[2]);
        const T2 s13 = cadd(v[1], v[3]), d13 = csub(v[1], v[3]);
        const T2 id = imul(d13, (T)SIGN);
        v[0] = cadd(s02, s13);
        v[2] = csub(s02, s13);
        v[1] = cadd(d02, id);
        v[3] = csub(d02, id);
    } else {
        constexpr int R = (L % 4 == 0) ? 4 : ((L % 2 == 0) ? 2 : 3);
        constexpr int Q = L / R;
        T2 s[R][Q];
#pragma unroll
        for (int a = 0; a < R; ++a)
#pragma unroll
            for (int b = 0; b < Q; ++b) s[a][b] = v[a + R * b];
#pragma unroll
        for (int a = 0; a < R; ++a) rdft<T2, Q, SIGN>(s[a]);
        rtwiddle<T2, L, SIGN, R, Q>(s, std::make_integer_sequence<int, R * Q>{});
#pragma unroll
        for (int b = 0; b < Q; ++b) {
            T2 t[R];
#pragma unroll
            for (int a = 0; a < R; ++a) t[a] = s[a][b];
            rdft<T2, R, SIGN>(t);
#pragma unroll
            for (int a = 0; a < R; ++a) v[b + Q * a] = t[a];
        }
    }
}

// theta synthesis, two-pass: block (k tile of KB, j, field) of kT2 threads,
// KB * N1 or KB * N2 tasks per pass.  Slot s of the output rows holds theta
// index (s / N2) + N1 (s % N2).  The task counts are multiples of the block
// size, so each thread runs a fixed number of tasks; in FP32, where their
// inputs fit in registers (at most 24 values), it loads all of them before the
// first DFT, so that one memory latency is exposed per pass instead of one per
// task, and runs at 64 registers (eight blocks per SM).
constexpr int kT2 = 128;
template <class T2, int KB, int N1, int N2>
__global__ void __launch_bounds__(kT2, sizeof(T2) == 8 ? 8 : 1)
    k_synth2(Geo g, FieldPtrs f, T2* __restrict__ Y, const T2* __restrict__ twg) {
    grid_dep_sync();
    constexpr int N = N1 * N2, IT1 = KB * N2 / kT2, IT2 = KB * N1 / kT2;
    static_assert(KB * N2 % kT2 == 0 && KB * N1 % kT2 == 0, "whole tasks per thread");
    extern __shared__ __align__(16) unsigned char smem[];
    T2* buf = reinterpret_cast<T2*>(smem);  // [N][KB]
    T2* tw = buf + N * KB;                   // [N]
    const int k0 = blockIdx.x * KB, j = blockIdx.y;
    const int nf = gridDim.z / g.nb, b = blockIdx.z / nf, fi = blockIdx.z - b * nf, slot = g.slot[b];
    Y += (size_t)slot * g.ps;
    for (int i = threadIdx.x; i < N; i += kT2) tw[i] = twg[i];
    const size_t base = (size_t)slot * g.fs + (size_t)j * g.nm * g.nk;
    const float2* srcf = f.inf[fi] ? f.inf[fi] + base : nullptr;
    const double2* src = srcf ? nullptr : f.in[fi] + base;
    auto load = [&](int it, T2 (&v)[N1]) {
        const int t = threadIdx.x + it * kT2, kk = t % KB, n2 = t / KB, k = k0 + kk;
#pragma unroll
        for (int n1 = 0; n1 < N1; ++n1) {
            const int n = n2 + N2 * n1;  // m mod N; zero padding for |m| > M
            const int m = n <= g.M ? n : n - N;
            v[n1] = (k < g.nk && m >= -g.M) ? synth_in<T2>(src, srcf, (size_t)(m + g.M) * g.nk + k) : mk<T2>(0, 0);
        }
    };
    auto dft1 = [&](int it, T2 (&v)[N1]) {
        const int t = threadIdx.x + it * kT2, kk = t % KB, n2 = t / KB;
        rdft<T2, N1, +1>(v);
#pragma unroll
        for (int k1 = 0; k1 < N1; ++k1) buf[(n2 + N2 * k1) * KB + kk] = twr<T2, +1>(v[k1], tw, n2 * k1);
    };
    if constexpr (sizeof(T2) == 8 && IT1 * N1 <= 24) {  // FP32 values only: FP64 ones would spill
        T2 v[IT1][N1];
#pragma unroll
        for (int it = 0; it < IT1; ++it) load(it, v[it]);
        __syncthreads();  // twiddles
#pragma unroll
        for (int it = 0; it < IT1; ++it) dft1(it, v[it]);
    } else {
        __syncthreads();  // twiddles
#pragma unroll 1
        for (int it = 0; it < IT1; ++it) {
            T2 v[N1];
            load(it, v);
            dft1(it, v);
        }
    }
    __syncthreads();
    T2* dst = Y + ((size_t)(fi * g.nr + j) * N) * g.nk;
    constexpr int kUnroll2 = sizeof(T2) == 8 ? IT2 : 1;  // FP64 tasks one at a time (registers)
#pragma unroll kUnroll2
    for (int it = 0; it < IT2; ++it) {
        const int t = threadIdx.x + it * kT2, kk = t % KB, k1 = t / KB, k = k0 + kk;
        T2 v[N2];
#pragma unroll
        for (int n2 = 0; n2 < N2; ++n2) v[n2] = buf[(N2 * k1 + n2) * KB + kk];
        rdft<T2, N2, +1>(v);
        if (k < g.nk) {
#pragma unroll
            for (int k2 = 0; k2 < N2; ++k2) dst[(size_t)(N2 * k1 + k2) * g.nk + k] = v[k2];
        }
    }
}

// theta analysis, two-pass (input rows in the slot order of k_synth2), with
// the k = 0 plane projected onto Hermitian symmetry.  Same thread layout as
// k_synth2; the first pass loads all its inputs before its DFTs where they
// fit in registers, and each task of the second pass loads the values to add
// (the base-flow terms) before its DFT.
template <class T2, int KB, int N1, int N2>
__global__ void __launch_bounds__(kT2, sizeof(T2) == 8 ? 6 : 1) k_anal2(Geo g, FieldPtrs f, const T2* __restrict__ Z,
                                               const T2* __restrict__ twg) {
    grid_dep_sync();
    constexpr int N = N1 * N2, IT1 = KB * N1 / kT2, IT2 = KB * N2 / kT2;
    static_assert(KB * N2 % kT2 == 0 && KB * N1 % kT2 == 0, "whole tasks per thread");
    extern __shared__ __align__(16) unsigned char smem[];
    T2* buf = reinterpret_cast<T2*>(smem);  // [N][KB]
    T2* tw = buf + N * KB;                   // [N]
    const int k0 = blockIdx.x * KB, j = blockIdx.y;
    const int nf = gridDim.z / g.nb, b = blockIdx.z / nf, fi = blockIdx.z - b * nf, slot = g.slot[b];
    const size_t off = (size_t)slot * g.fs;
    Z += (size_t)slot * g.ps;
    for (int i = threadIdx.x; i < N; i += kT2) tw[i] = twg[i];
    const T2* src = Z + ((size_t)(fi * g.nr + j) * N) * g.nk;
    auto load = [&](int it, T2 (&v)[N2]) {
        const int t = threadIdx.x + it * kT2, kk = t % KB, k1 = t / KB, k = k0 + kk;
#pragma unroll
        for (int n2 = 0; n2 < N2; ++n2) v[n2] = k < g.nk ? src[(size_t)(N2 * k1 + n2) * g.nk + k] : mk<T2>(0, 0);
    };
    auto dft1 = [&](int it, T2 (&v)[N2]) {
        const int t = threadIdx.x + it * kT2, kk = t % KB, k1 = t / KB;
        rdft<T2, N2, -1>(v);
#pragma unroll
        for (int m2 = 0; m2 < N2; ++m2) buf[(N2 * k1 + m2) * KB + kk] = twr<T2, -1>(v[m2], tw, k1 * m2);
    };
    if constexpr (sizeof(T2) == 8 && IT1 * N2 <= 24) {  // FP32 values only: FP64 ones would spill
        T2 v[IT1][N2];
#pragma unroll
        for (int it = 0; it < IT1; ++it) load(it, v[it]);
        __syncthreads();  // twiddles
#pragma unroll
        for (int it = 0; it < IT1; ++it) dft1(it, v[it]);
    } else {
        __syncthreads();  // twiddles
#pragma unroll 1
        for (int it = 0; it < IT1; ++it) {
            T2 v[N2];
            load(it, v);
            dft1(it, v);
        }
    }
    __syncthreads();
    const size_t base = off + (size_t)j * g.nm * g.nk;
    float2* dstf = f.outf[fi] ? f.outf[fi] + base : nullptr;
    double2* dst = dstf ? nullptr : f.out[fi] + base;
    const double2* add = f.add[fi] ? f.add[fi] + base : nullptr;
#pragma unroll 1
    for (int it = 0; it < IT2; ++it) {
        const int t = threadIdx.x + it * kT2, kk = t % KB, m2 = t / KB, k = k0 + kk;
        constexpr bool kEarly = sizeof(T2) == 8 && N1 <= 8;  // larger or FP64 tasks: no room in registers
        double2 ad[kEarly ? N1 : 1];
        if constexpr (kEarly) {
#pragma unroll
            for (int m1 = 0; m1 < N1; ++m1) {
                const int n = m2 + N2 * m1;
                const int m = n <= g.M ? n : n - N;
                ad[m1] = (add && k > 0 && k < g.nk && m >= -g.M) ? add[(size_t)(m + g.M) * g.nk + k]
                                                                  : make_double2(0, 0);
            }
        }
        T2 v[N1];
#pragma unroll
        for (int k1 = 0; k1 < N1; ++k1) v[k1] = buf[(m2 + N2 * k1) * KB + kk];
        rdft<T2, N1, -1>(v);
#pragma unroll
        for (int m1 = 0; m1 < N1; ++m1) {
            const int n = m2 + N2 * m1;
            const int m = n <= g.M ? n : n - N;
            if (k < g.nk && m >= -g.M) {
                if (k == 0) {
                    buf[n * KB + kk] = v[m1];
                } else if (dstf) {
                    dstf[(size_t)(m + g.M) * g.nk + k] = v[m1];
                } else {
                    const size_t o = (size_t)(m + g.M) * g.nk + k;
                    double2 x = to_d(v[m1]);
                    if (add) {
                        const double2 a = kEarly ? ad[kEarly ? m1 : 0] : add[o];
                        x = make_double2(x.x + a.x, x.y + a.y);
                    }
                    dst[o] = x;
                }
            }
        }
    }
    if (k0 == 0) {  // block-uniform
        __syncthreads();
        for (int im = threadIdx.x; im < g.nm; im += blockDim.x) {
            const int m = im - g.M;
            if (dstf) {
                using T = typename RealOf<T2>::T;
                const T2 v = buf[(m < 0 ? m + N : m) * KB], vm = buf[(m > 0 ? N - m : -m) * KB];
                dstf[(size_t)im * g.nk] = mk<T2>((T)0.5 * (v.x + vm.x), (T)0.5 * (v.y - vm.y));
                continue;
            }
            const double2 v = to_d(buf[(m < 0 ? m + N : m) * KB]);
            const double2 vm = to_d(buf[(m > 0 ? N - m : -m) * KB]);
            double2 x = make_double2(0.5 * (v.x + vm.x), 0.5 * (v.y - vm.y));
            if (add) x = make_double2(x.x + add[(size_t)im * g.nk].x, x.y + add[(size_t)im * g.nk].y);
            dst[(size_t)im * g.nk] = x;
        }
    }
}

// Compile-time loop: f(std::integral_constant<int, 0>()) ... f(<N - 1>).
template <class F, int... I>
__device__ __forceinline__ void static_for_impl(F& f, std::integer_sequence<int, I...>) {
    (f(std::integral_constant<int, I>()), ...);
}
template <int N, class F> __device__ __forceinline__ void static_for(F&& f) {
    static_for_impl(f, std::make_integer_sequence<int, N>());
}

// z pass, two-pass FFTs in place in padded shared-memory columns (one gap
// after every run of N2 slots keeps both access patterns free of bank
// conflicts), RB rows (theta indices a) of one radial index per block.  The
// spectra are 3/2-padded: K = N/3 - 1 is a compile-time constant here (the
// launcher checks it), so the inverse pass knows at compile time which of its
// strided inputs fall in the zero band K < n < N - K and loads none of them,
// and the forward pass stores no output of that band (the separation never
// reads it).  Same contract as k_zpass.
template <class T2, int MODE, int N1, int N2, int RB>
__global__ void __launch_bounds__(96, 6)
    k_zpass2(Geo g, const T2* __restrict__ Y, T2* __restrict__ Z, ZScales sc, const T2* __restrict__ twg) {
    grid_dep_sync();
    using T = typename RealOf<T2>::T;
    constexpr int N = N1 * N2, NP = N + N1, KC = N / 3 - 1, NK = KC + 1;
    constexpr int NIN = MODE == ZFWD ? 6 : (MODE == ZADJ ? 9 : 18);
    constexpr int NPI = (NIN + 1) / 2;
    constexpr int NOUT = MODE == ZADJ ? 6 : 3;
    constexpr int NPO = (NOUT + 1) / 2;
    extern __shared__ __align__(16) unsigned char smem[];
    T2* col = reinterpret_cast<T2*>(smem);  // [RB][NPI][NP]
    T2* tw = col + RB * NPI * NP;            // [N]
    const int a0 = blockIdx.x * RB, j = blockIdx.y;
    const size_t poff = (size_t)g.slot[blockIdx.z] * g.ps;  // batch entry blockIdx.z
    Y += poff;
    Z += poff;
    auto at = [](int s) { return s + s / N2; };
    for (int i = threadIdx.x; i < N; i += blockDim.x) tw[i] = twg[i];
    __syncthreads();
    // inverse, strided pass: Hermitian-extended spectra, two real fields per column
    for (int t = threadIdx.x; t < RB * NPI * N2; t += blockDim.x) {
        const int r = t / (NPI * N2), pn = t - r * (NPI * N2), p = pn / N2, n2 = pn - p * N2;
        const int f1 = 2 * p, f2 = 2 * p + 1;
        const bool has2 = f2 < NIN;
        const T2* y1 = Y + ((size_t)(f1 * g.nr + j) * g.nt + a0 + r) * NK;
        const T2* y2 = Y + ((size_t)((has2 ? f2 : f1) * g.nr + j) * g.nt + a0 + r) * NK;
        const T h01 = zs<T>(sc.h0, sc.fh0, f1), hk1 = zs<T>(sc.hk, sc.fhk, f1);
        const T h02 = has2 ? zs<T>(sc.h0, sc.fh0, f2) : (T)0, hk2 = has2 ? zs<T>(sc.hk, sc.fhk, f2) : (T)0;
        // H1 + i H2 at z-wavenumber k (positive side) or conj(H1) + i conj(H2)
        // (negative side); only k = 0 drops its imaginary parts
        auto entry = [&](int k, bool neg, bool may0) {
            const T2 a1 = y1[k], a2 = has2 ? y2[k] : mk<T2>(0, 0);
            const bool z0 = may0 && k == 0;
            const T2 h1 = z0 ? mk<T2>(h01 * a1.x, 0) : mk<T2>(hk1 * a1.x, hk1 * a1.y);
            const T2 h2 = z0 ? mk<T2>(h02 * a2.x, 0) : mk<T2>(hk2 * a2.x, hk2 * a2.y);
            return !neg ? mk<T2>(h1.x - h2.y, h1.y + h2.x) : mk<T2>(h1.x + h2.y, -h1.y + h2.x);
        };
        T2 v[N1];
        static_for<N1>([&](auto I) {
            constexpr int n1 = decltype(I)::value;
            constexpr int lo = N2 * n1, hi = lo + N2 - 1;
            const int n = n2 + lo;
            if constexpr (hi <= KC) {
                v[n1] = entry(n, false, n1 == 0);
            } else if constexpr (lo >= N - KC) {
                v[n1] = entry(N - n, true, false);
            } else if constexpr (lo > KC && hi < N - KC) {
                v[n1] = mk<T2>(0, 0);
            } else {
                v[n1] = n <= KC ? entry(n, false, n1 == 0) : (n >= N - KC ? entry(N - n, true, false) : mk<T2>(0, 0));
            }
        });
        rdft<T2, N1, +1>(v);
        T2* c = col + (r * NPI + p) * NP;
#pragma unroll
        for (int k1 = 0; k1 < N1; ++k1) c[at(n2 + N2 * k1)] = twr<T2, +1>(v[k1], tw, n2 * k1);
    }
    __syncthreads();
    // inverse, contiguous pass: physical values
    for (int t = threadIdx.x; t < RB * NPI * N1; t += blockDim.x) {
        const int rp = t / N1, k1 = t - rp * N1;
        T2* c = col + rp * NP;
        T2 v[N2];
#pragma unroll
        for (int n2 = 0; n2 < N2; ++n2) v[n2] = c[at(N2 * k1 + n2)];
        rdft<T2, N2, +1>(v);
#pragma unroll
        for (int k2 = 0; k2 < N2; ++k2) c[at(N2 * k1 + k2)] = v[k2];
    }
    __syncthreads();
    // pointwise products, in place (each slot read and written by one thread)
    for (int t = threadIdx.x; t < RB * N; t += blockDim.x) {
        const int r = t / N, s = t - r * N;
        T2* c = col + r * NPI * NP;
        const int o = at(s);
        if constexpr (MODE == ZCADJ) {
            T2 row[NPI], res[2];
#pragma unroll
            for (int p = 0; p < NPI; ++p) row[p] = c[p * NP + o];
            cadj_products<T2>(row, res);
            c[o] = res[0];
            c[NP + o] = res[1];
            continue;
        }
        const T2 c0 = c[o], c1 = c[NP + o], c2 = c[2 * NP + o];
        const T ur = c0.x, ut = c0.y, uz = c1.x;
        const T wr = c1.y, wt = c2.x, wz = c2.y;
        if (MODE == ZFWD) {
            c[o] = mk<T2>(ut * wz - uz * wt, uz * wr - ur * wz);
            c[NP + o] = mk<T2>(ur * wt - ut * wr, 0);
        } else {
            const T2 c3 = c[3 * NP + o], c4 = c[4 * NP + o];
            const T gr = c3.x, gt = c3.y, gz = c4.x;
            c[o] = mk<T2>(wt * gz - wz * gt, wz * gr - wr * gz);           // w x g
            c[NP + o] = mk<T2>(wr * gt - wt * gr, gt * uz - gz * ut);      // (w x g)_z, (g x u)_r
            c[2 * NP + o] = mk<T2>(gz * ur - gr * uz, gr * ut - gt * ur);  // (g x u)_theta, (g x u)_z
        }
    }
    __syncthreads();
    // forward, contiguous pass
    for (int t = threadIdx.x; t < RB * NPO * N1; t += blockDim.x) {
        const int r = t / (NPO * N1), pk = t - r * (NPO * N1), p = pk / N1, k1 = pk - p * N1;
        T2* c = col + (r * NPI + p) * NP;
        T2 v[N2];
#pragma unroll
        for (int k2 = 0; k2 < N2; ++k2) v[k2] = c[at(N2 * k1 + k2)];
        rdft<T2, N2, -1>(v);
#pragma unroll
        for (int m2 = 0; m2 < N2; ++m2) c[at(N2 * k1 + m2)] = twr<T2, -1>(v[m2], tw, k1 * m2);
    }
    __syncthreads();
    // forward, strided pass: natural-order spectra, the zero band left out
    for (int t = threadIdx.x; t < RB * NPO * N2; t += blockDim.x) {
        const int r = t / (NPO * N2), pm = t - r * (NPO * N2), p = pm / N2, m2 = pm - p * N2;
        T2* c = col + (r * NPI + p) * NP;
        T2 v[N1];
#pragma unroll
        for (int k1 = 0; k1 < N1; ++k1) v[k1] = c[at(m2 + N2 * k1)];
        rdft<T2, N1, -1>(v);
        static_for<N1>([&](auto I) {
            constexpr int m1 = decltype(I)::value;
            constexpr int lo = N2 * m1, hi = lo + N2 - 1;
            if constexpr (!(lo > KC && hi < N - KC)) c[at(m2 + lo)] = v[m1];
        });
    }
    __syncthreads();
    // separate the two real products of each column, truncate to k <= K, scale
    for (int t = threadIdx.x; t < RB * NPO * NK; t += blockDim.x) {
        const int r = t / (NPO * NK), pk = t - r * (NPO * NK), p = pk / NK, k = pk - p * NK;
        const T2* c = col + (r * NPI + p) * NP;
        const T2 P = c[at(k)];
        const T2 Pm = c[at((N - k) % N)];
        const int o1 = 2 * p, o2 = 2 * p + 1;
        const size_t row = (size_t)j * g.nt + a0 + r;
        const T s1 = k == 0 ? zs<T>(sc.o0, sc.fo0, o1) : zs<T>(sc.ok, sc.fok, o1);
        Z[((size_t)o1 * g.nr * g.nt + row) * NK + k] = mk<T2>((T)0.5 * (P.x + Pm.x) * s1, (T)0.5 * (P.y - Pm.y) * s1);
        if (o2 < NOUT) {
            const T s2 = k == 0 ? zs<T>(sc.o0, sc.fo0, o2) : zs<T>(sc.ok, sc.fok, o2);
            Z[((size_t)o2 * g.nr * g.nt + row) * NK + k] =
                mk<T2>((T)0.5 * (P.y + Pm.y) * s2, (T)-0.5 * (P.x - Pm.x) * s2);
        }
    }
}

// ------------------------------------------------------------------ launchers
template <class T2> static const T2* tw_z(const Twiddles& t);
template <> const double2* tw_z<double2>(const Twiddles& t) { return t.z_d; }
template <> const float2* tw_z<float2>(const Twiddles& t) { return t.z_f; }

template <class T2> static int theta_kb(const Geo& g) {
    int kb = 32;
    while (kb > 4 && (kb / 2 >= g.nk || (size_t)(2 * g.nt * kb + g.nt) * sizeof(T2) > 100 * 1024)) kb /= 2;
    return kb;
}

template <class T2, int KB>
static void synth_theta_kb(const Geo& g, const FieldPtrs& f, int nfield, T2* Y, const T2* tw, cudaStream_t s) {
    const size_t sm = (size_t)(2 * g.nt * KB + g.nt) * sizeof(T2);
    smem_limit((const void*)k_synth_theta<T2, KB>);
    dim3 grid((g.nk + KB - 1) / KB, g.nr, nfield * g.nb);
    launch_pdl(k_synth_theta<T2, KB>, grid, 256, sm, s, g, f, Y, tw);
}

template <class T2, int KB>
static void anal_theta_kb(const Geo& g, const FieldPtrs& f, int nfield, const T2* Z, const T2* tw, cudaStream_t s) {
    const size_t sm = (size_t)(2 * g.nt * KB + g.nt) * sizeof(T2);
    smem_limit((const void*)k_anal_theta<T2, KB>);
    dim3 grid((g.nk + KB - 1) / KB, g.nr, nfield * g.nb);
    launch_pdl(k_anal_theta<T2, KB>, grid, 256, sm, s, g, f, Z, tw);
}

// Two-pass register kernels serve the lengths with a split N = N1 N2 below;
// the Stockham kernels serve every other 2^a 3^b length.  The theta kernels
// take KB k-columns per block.
template <class T2, int KB, int N1, int N2>
static void synth2(const Geo& g, const FieldPtrs& f, int nfield, T2* Y, const T2* tw, cudaStream_t s) {
    const size_t sm = (size_t)(N1 * N2 * KB + N1 * N2) * sizeof(T2);
    smem_limit((const void*)k_synth2<T2, KB, N1, N2>);
    dim3 grid((g.nk + KB - 1) / KB, g.nr, nfield * g.nb);
    launch_pdl(k_synth2<T2, KB, N1, N2>, grid, kT2, sm, s, g, f, Y, tw);
}
template <class T2, int KB, int N1, int N2>
static void anal2(const Geo& g, const FieldPtrs& f, int nfield, const T2* Z, const T2* tw, cudaStream_t s) {
    const size_t sm = (size_t)(N1 * N2 * KB + N1 * N2) * sizeof(T2);
    smem_limit((const void*)k_anal2<T2, KB, N1, N2>);
    dim3 grid((g.nk + KB - 1) / KB, g.nr, nfield * g.nb);
    launch_pdl(k_anal2<T2, KB, N1, N2>, grid, kT2, sm, s, g, f, Z, tw);
}

// columns per block of the fixed-point theta kernels: about 50 KB of shared
// memory, 128 to 256 contiguous bytes per row
// (64x64x256: synthesis 67 us at 16, 73 at 8, 76 at 4, analysis 57, 59, 54; 48x48x128: 26,
// 28, 29 and 24, 23, 20; 48x32x96: 18, 18, 16 and 14, 14, 12; 64x96x128, 144 points: 67, 67, 78
// and 50, 53, 53; 48x128x64, 192 points: 39, 34, 39 and 29, 29, 27)
static int theta_kx(const Geo& g) { return g.nt <= 96 && g.nk > 8 ? 16 : (g.nt <= 192 ? 8 : 4); }
template <int KB> static size_t theta_sx(const Geo& g) { return (size_t)(2 * g.nt * KB + g.nt) * sizeof(double2); }
static unsigned theta_tx(const Geo& g, int kb) {
    return (unsigned)std::max(64, std::min(256, (g.nt * kb / 4 + 31) / 32 * 32));
}
template <int KB>
static void synth_x(const Geo& g, const FieldPtrs& f, int nfield, double2* Y, const int4* tw, cudaStream_t s) {
    smem_limit((const void*)k_synth_x<KB>);
    launch_pdl(k_synth_x<KB>, dim3((g.nk + KB - 1) / KB, g.nr, nfield * g.nb), theta_tx(g, KB), theta_sx<KB>(g), s, g, f,
               Y, tw);
}
template <int KB>
static void anal_x(const Geo& g, const FieldPtrs& f, int nfield, const double2* Z, const int4* tw, cudaStream_t s) {
    smem_limit((const void*)k_anal_x<KB>);
    launch_pdl(k_anal_x<KB>, dim3((g.nk + KB - 1) / KB, g.nr, nfield * g.nb), theta_tx(g, KB), theta_sx<KB>(g), s, g, f,
               Z, tw);
}

template <class T2>
void launch_synth_theta(const Geo& g, const FieldPtrs& f, int nfield, T2* Y, const Twiddles& tw, cudaStream_t s) {
    if constexpr (std::is_same<T2, double2>::value) {
        switch (theta_kx(g)) {
            case 16: synth_x<16>(g, f, nfield, Y, tw.th_x, s); break;
            case 8: synth_x<8>(g, f, nfield, Y, tw.th_x, s); break;
            default: synth_x<4>(g, f, nfield, Y, tw.th_x, s); break;
        }
        check_launch("synth_theta");
        return;
    } else {
    switch (g.nt) {
        case 96: synth2<T2, 32, 8, 12>(g, f, nfield, Y, tw.th_f, s); check_launch("synth_theta"); return;
        case 192: synth2<T2, 32, 16, 12>(g, f, nfield, Y, tw.th_f, s); check_launch("synth_theta"); return;
        case 384: synth2<T2, 16, 16, 24>(g, f, nfield, Y, tw.th_f, s); check_launch("synth_theta"); return;
        default: break;
    }
    switch (theta_kb<T2>(g)) {
        case 32: synth_theta_kb<T2, 32>(g, f, nfield, Y, tw.th_f, s); break;
        case 16: synth_theta_kb<T2, 16>(g, f, nfield, Y, tw.th_f, s); break;
        case 8: synth_theta_kb<T2, 8>(g, f, nfield, Y, tw.th_f, s); break;
        default: synth_theta_kb<T2, 4>(g, f, nfield, Y, tw.th_f, s); break;
    }
    check_launch("synth_theta");
    }
}

template <class T2>
void launch_anal_theta(const Geo& g, const FieldPtrs& f, int nfield, const T2* Z, const Twiddles& tw, cudaStream_t s) {
    if constexpr (std::is_same<T2, double2>::value) {
        switch (theta_kx(g)) {
            case 16: anal_x<16>(g, f, nfield, Z, tw.th_x, s); break;
            case 8: anal_x<8>(g, f, nfield, Z, tw.th_x, s); break;
            default: anal_x<4>(g, f, nfield, Z, tw.th_x, s); break;
        }
        check_launch("anal_theta");
        return;
    } else {
    switch (g.nt) {
        case 96: anal2<T2, 32, 8, 12>(g, f, nfield, Z, tw.th_f, s); check_launch("anal_theta"); return;
        case 192: anal2<T2, 32, 16, 12>(g, f, nfield, Z, tw.th_f, s); check_launch("anal_theta"); return;
        case 384: anal2<T2, 16, 16, 24>(g, f, nfield, Z, tw.th_f, s); check_launch("anal_theta"); return;
        default: break;
    }
    switch (theta_kb<T2>(g)) {
        case 32: anal_theta_kb<T2, 32>(g, f, nfield, Z, tw.th_f, s); break;
        case 16: anal_theta_kb<T2, 16>(g, f, nfield, Z, tw.th_f, s); break;
        case 8: anal_theta_kb<T2, 8>(g, f, nfield, Z, tw.th_f, s); break;
        default: anal_theta_kb<T2, 4>(g, f, nfield, Z, tw.th_f, s); break;
    }
    check_launch("anal_theta");
    }
}

// N/4 threads divide the radix-4 (and the radix-2, radix-3) stages of a
// length-N column exactly; at least one warp, at most 256.
static unsigned zpass_threads(const Geo& g) {
    const int t = (g.nzp / 4 + 31) / 32 * 32;
    return (unsigned)std::max(32, std::min(256, t));
}

// rows per block of the two-pass z kernel: two for the forward pass (its
// three packed columns then fill the block's threads better, at 22 KB of
// shared memory: 16.6 against 18.4 ms per 64x64x256 gradient), one for the
// adjoint passes, whose five and nine columns fill them already (two rows
// measured slower there: 13.6 against 12.8 ms)
template <int MODE> constexpr int zpass_rows() { return MODE == ZFWD ? 2 : 1; }

template <class T2, int MODE, int N1, int N2, int RB>
static void zpass2(const Geo& g, const T2* Y, T2* Z, const ZScales& sc, const T2* tw, cudaStream_t s) {
    constexpr int NPI = MODE == ZFWD ? 3 : (MODE == ZADJ ? 5 : 9);
    const size_t sm = (size_t)(RB * NPI * (N1 * N2 + N1) + N1 * N2) * sizeof(T2);
    smem_limit((const void*)k_zpass2<T2, MODE, N1, N2, RB>);
    launch_pdl(k_zpass2<T2, MODE, N1, N2, RB>, dim3(g.nt / RB, g.nr, g.nb), zpass_threads(g), sm, s, g, Y, Z, sc,
               tw);
}
template <class T2, int MODE, int N1, int N2>
static void zpass2_rows(const Geo& g, const T2* Y, T2* Z, const ZScales& sc, const T2* tw, cudaStream_t s) {
    constexpr int RB = zpass_rows<MODE>();
    if (g.nt % RB == 0) zpass2<T2, MODE, N1, N2, RB>(g, Y, Z, sc, tw, s);
    else zpass2<T2, MODE, N1, N2, 1>(g, Y, Z, sc, tw, s);
}
// The two-pass kernel serves the 3/2-padded lengths N = 3 (K + 1) below; any
// other length goes to the Stockham kernel.
template <class T2, int MODE>
static bool zpass2_any(const Geo& g, const T2* Y, T2* Z, const ZScales& sc, const T2* tw, cudaStream_t s) {
    if (g.nzp != 3 * g.nk || g.K != g.nk - 1) return false;
    switch (g.nzp) {
        case 96: zpass2_rows<T2, MODE, 8, 12>(g, Y, Z, sc, tw, s); return true;
        case 192: zpass2_rows<T2, MODE, 16, 12>(g, Y, Z, sc, tw, s); return true;
        case 384: zpass2_rows<T2, MODE, 16, 24>(g, Y, Z, sc, tw, s); return true;
        default: return false;
    }
}

// FP64 forward and adjoint passes in fixed point
template <int MODE>
static void zpass_fixed(const Geo& g, const double2* Y, double2* Z, const ZScales& sc, const int4* tw, cudaStream_t s) {
    constexpr int NPI = MODE == ZFWD ? 3 : 5, NG = MODE == ZFWD ? 2 : 3, NOUT = MODE == ZFWD ? 3 : 6;
    // u and w come as they are; the cotangents (ZADJ) may have a scale, smaller by a
    // power of two for k > 0, which every output of theirs is linear in
    XScales x{};
    double gs = 1.0;
    for (int i = 0; i < 3 * NG; ++i) {
        int e = 1;
        bool ok = sc.h0[i] == sc.h0[i / 3 * 3] && sc.hk[i] == sc.hk[i / 3 * 3];
        if (i < 6) ok = ok && sc.h0[i] == 1.0 && sc.hk[i] == 1.0;
        else ok = ok && std::frexp(sc.hk[i] / sc.h0[i], &e) == 0.5 && e <= 1;
        if (!ok) throw std::runtime_error("zpass: unsupported input scales");
        x.hsh[i / 3] = 1 - e;
        if (i == 6) gs = sc.h0[i];
    }
    for (int i = 0; i < NOUT; ++i) {
        x.o0[i] = sc.o0[i] * gs;
        x.ok[i] = sc.ok[i] * gs;
    }
    const size_t sm = (size_t)(2 * g.nzp * NPI + g.nzp) * sizeof(double2);
    smem_limit((const void*)k_zpass_x<MODE>);
    launch_pdl(k_zpass_x<MODE>, dim3(g.nt, g.nr, g.nb), std::max(64u, std::min(256u, (unsigned)(g.nzp / 2 + 31) / 32 * 32)),
               sm, s, g, Y, Z, x, tw);
}

template <class T2, int MODE>
static void zpass_stockham(const Geo& g, const T2* Y, T2* Z, const ZScales& sc, const T2* tw, cudaStream_t s) {
    constexpr int LD = MODE == ZFWD ? 3 : (MODE == ZADJ ? 5 : 9);
    const size_t sm = (size_t)(2 * g.nzp * LD + g.nzp) * sizeof(T2);
    smem_limit((const void*)k_zpass<T2, MODE>);
    launch_pdl(k_zpass<T2, MODE>, dim3(g.nt, g.nr, g.nb), zpass_threads(g), sm, s, g, Y, Z, sc, tw);
}

template <class T2>
void launch_zpass(const Geo& g, int mode, const T2* Y, T2* Z, const ZScales& sc_in, const Twiddles& tw, cudaStream_t s) {
    ZScales sc = sc_in;
    for (int i = 0; i < kMaxIn; ++i) {
        sc.fh0[i] = (float)sc.h0[i];
        sc.fhk[i] = (float)sc.hk[i];
    }
    for (int i = 0; i < 6; ++i) {
        sc.fo0[i] = (float)sc.o0[i];
        sc.fok[i] = (float)sc.ok[i];
    }
    const T2* t = tw_z<T2>(tw);
    if constexpr (std::is_same<T2, double2>::value) {
        if (mode == ZFWD) zpass_fixed<ZFWD>(g, Y, Z, sc, tw.z_x, s);
        else if (mode == ZADJ) zpass_fixed<ZADJ>(g, Y, Z, sc, tw.z_x, s);
        else zpass_stockham<T2, ZCADJ>(g, Y, Z, sc, t, s);
    } else {
        const bool done = mode == ZFWD ? zpass2_any<T2, ZFWD>(g, Y, Z, sc, t, s)
                                       : (mode == ZADJ ? zpass2_any<T2, ZADJ>(g, Y, Z, sc, t, s)
                                                       : zpass2_any<T2, ZCADJ>(g, Y, Z, sc, t, s));
        if (!done) {
            if (mode == ZFWD) zpass_stockham<T2, ZFWD>(g, Y, Z, sc, t, s);
            else if (mode == ZADJ) zpass_stockham<T2, ZADJ>(g, Y, Z, sc, t, s);
            else zpass_stockham<T2, ZCADJ>(g, Y, Z, sc, t, s);
        }
    }
    check_launch("zpass");
}

template void launch_synth_theta<double2>(const Geo&, const FieldPtrs&, int, double2*, const Twiddles&, cudaStream_t);
template void launch_synth_theta<float2>(const Geo&, const FieldPtrs&, int, float2*, const Twiddles&, cudaStream_t);
template void launch_anal_theta<double2>(const Geo&, const FieldPtrs&, int, const double2*, const Twiddles&,
                                         cudaStream_t);
template void launch_anal_theta<float2>(const Geo&, const FieldPtrs&, int, const float2*, const Twiddles&,
                                        cudaStream_t);
template void launch_zpass<double2>(const Geo&, int, const double2*, double2*, const ZScales&, const Twiddles&,
                                    cudaStream_t);
template void launch_zpass<float2>(const Geo&, int, const float2*, float2*, const ZScales&, const Twiddles&,
                                   cudaStream_t);

}  // namespace pnop
