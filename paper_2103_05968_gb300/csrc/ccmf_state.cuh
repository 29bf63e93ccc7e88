// State formats of the passes, vector and pack accesses.
//
// Compact state. After an update, v = P_C(z) and e = (z - v) / rho of one voxel are functions of
// z = v + rho xi (Eq. 30, Eq. 19): v = s z with the one scalar s = min(1, gamma / |z|), and
// e = (z - s z) / rho with the rho of that update. So the FP32 passes keep the seven values (z, s)
// of a voxel and rho_prev (SolveScalars) instead of the twelve components of (e, v), and every
// reader forms v = s z, e = (z - v) / rho_prev with the very operations that the update uses for its
// own sums. The update is bound by HBM: it moves 36 + 28 B/voxel instead of 56 + 48, and the
// divergence pass 28 + 4 instead of 48 + 4. Measured on GB300, 512^3: update 2.37 -> 1.53 ms,
// divergence pass 1.09 -> 0.89 ms. FP64 is bound by its arithmetic (1/64 of the FP32 rate)
// and keeps (e, v): three more operations a component would cost it more than the bytes.
//
// A state that no update wrote (an imported one, or one that an update variant with the (e, v) format
// left) has S.zs_iter != S.iters + 1: it is read in the (e, v) format, and the first update writes (z, s).
//
// Packs. The arithmetic runs on Pk<T>::V: two voxels of FP32 per register pair (the packed
// add / mul / fma of sm_100 and later, half the issue slots), one voxel in FP64. Every product that feeds
// an addition is an explicit fma, so the compiler has nothing to contract and the rounding of a voxel does not
// depend on which variant or read format processes it.
#pragma once

#include "ccmf_types.cuh"

namespace ccmf {

// ---------------------------------------------------------------------------
// 16-byte vectors of the field type (4 floats or 2 doubles).
// ---------------------------------------------------------------------------
template <typename T> struct Vec16;
template <> struct Vec16<float> {
    using type = float4;
    static constexpr int W = 4;
    __device__ __forceinline__ static void ld(const float* __restrict__ p, float (&o)[4]) {
        const float4 t = __ldg(reinterpret_cast<const float4*>(p));
        o[0] = t.x; o[1] = t.y; o[2] = t.z; o[3] = t.w;
    }
    __device__ __forceinline__ static void st(float* p, const float (&o)[4]) {
        *reinterpret_cast<float4*>(p) = make_float4(o[0], o[1], o[2], o[3]);
    }
};
template <> struct Vec16<double> {
    using type = double2;
    static constexpr int W = 2;
    __device__ __forceinline__ static void ld(const double* __restrict__ p, double (&o)[2]) {
        const double2 t = __ldg(reinterpret_cast<const double2*>(p));
        o[0] = t.x; o[1] = t.y;
    }
    __device__ __forceinline__ static void st(double* p, const double (&o)[2]) {
        *reinterpret_cast<double2*>(p) = make_double2(o[0], o[1]);
    }
};

// VW consecutive elements of the field type with one aligned load / store.
template <typename T, int VW> struct VecN;
template <> struct VecN<float, 4> {
    __device__ __forceinline__ static void ld(const float* __restrict__ p, float (&o)[4]) {
        const float4 t = __ldg(reinterpret_cast<const float4*>(p));
        o[0] = t.x; o[1] = t.y; o[2] = t.z; o[3] = t.w;
    }
    __device__ __forceinline__ static void st(float* p, const float (&o)[4]) {
        *reinterpret_cast<float4*>(p) = make_float4(o[0], o[1], o[2], o[3]);
    }
};
template <> struct VecN<float, 2> {
    __device__ __forceinline__ static void ld(const float* __restrict__ p, float (&o)[2]) {
        const float2 t = __ldg(reinterpret_cast<const float2*>(p));
        o[0] = t.x; o[1] = t.y;
    }
    __device__ __forceinline__ static void ldcg(const float* p, float (&o)[2]) {
        const float2 t = __ldcg(reinterpret_cast<const float2*>(p));
        o[0] = t.x; o[1] = t.y;
    }
    __device__ __forceinline__ static void st(float* p, const float (&o)[2]) {
        *reinterpret_cast<float2*>(p) = make_float2(o[0], o[1]);
    }
};
template <> struct VecN<float, 1> {
    __device__ __forceinline__ static void ld(const float* __restrict__ p, float (&o)[1]) { o[0] = __ldg(p); }
    __device__ __forceinline__ static void st(float* p, const float (&o)[1]) { p[0] = o[0]; }
};
template <> struct VecN<double, 2> {
    __device__ __forceinline__ static void ld(const double* __restrict__ p, double (&o)[2]) {
        const double2 t = __ldg(reinterpret_cast<const double2*>(p));
        o[0] = t.x; o[1] = t.y;
    }
    __device__ __forceinline__ static void st(double* p, const double (&o)[2]) {
        *reinterpret_cast<double2*>(p) = make_double2(o[0], o[1]);
    }
};
template <> struct VecN<double, 1> {
    __device__ __forceinline__ static void ld(const double* __restrict__ p, double (&o)[1]) { o[0] = __ldg(p); }
    __device__ __forceinline__ static void st(double* p, const double (&o)[1]) { p[0] = o[0]; }
};

// Neighbour offsets of the row (i, j) of a solve: rows (i+1, j), (i-1, j), (i, j+1), (i, j-1).
struct RowNb {
    long long row, ip, im, jp, jm;  // element offsets of k = 0 of each row
};

__device__ __forceinline__ RowNb row_neighbours(const Geom& g, unsigned row) {
    const unsigned i = fdiv(row, g.div_n2);
    const int j = (int)(row - i * (unsigned)g.n2);
    const int ip = ((int)i + 1 == g.n1) ? 0 : (int)i + 1, im = (i == 0) ? g.n1 - 1 : (int)i - 1;
    const int jp = (j + 1 == g.n2) ? 0 : j + 1, jm = (j == 0) ? g.n2 - 1 : j - 1;
    RowNb r;
    const long long n3 = g.n3;
    r.row = (long long)row * n3;
    r.ip = ((long long)ip * g.n2 + j) * n3;
    r.im = ((long long)im * g.n2 + j) * n3;
    r.jp = ((long long)i * g.n2 + jp) * n3;
    r.jm = ((long long)i * g.n2 + jm) * n3;
    return r;
}

// 1 / x and 1 / sqrt(x) in FP64 from the FP32 reciprocals by one step of Newton (second order) and Halley; the
// start's relative error of 2^-22 leaves 2^-60 and less before rounding. The FP64 unit of GB300 takes a warp's
// instruction every 16 cycles, and the library's division and square root issue about 20 of them each against 4 and 5
// here. x must lie well inside the range of float.
__device__ __forceinline__ double rcp_newton(double x) {
    const double y = (double)(1.0f / (float)x);
    const double e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
}
__device__ __forceinline__ double rsqrt_halley(double x) {
    const double y = (double)rsqrtf((float)x);
    const double e = fma(-x, y * y, 1.0);
    return fma(y * e, fma(0.375, e, 0.5), y);
}
// 2^-100 <= x < 2^100, on the bits (a comparison of doubles occupies the FP64 unit too).
__device__ __forceinline__ bool in_float_range(double x) {
    return (unsigned)(__double2hiint(x) - (923 << 20)) < (200u << 20);
}
// sqrt(x) > g for the correctly rounded square root, without taking it: the root rounds up past g where it exceeds the
// middle of g and its successor g', that is where x > g g' (what (g + g')^2 / 4 adds to that is too little for a double
// x to lie between). The fma rounds g g' - x once, so its sign is exact. x > g^2 would be one ulp of x too sharp: before
// the first update |z| = rho0 = min gamma on a whole phase, and a rounding error there would pass for a clipped voxel.
__device__ __forceinline__ bool root_exceeds(double x, double g) {
    const double next = __longlong_as_double(__double_as_longlong(g) + 1);
    return __double2hiint(fma(g, next, -x)) < 0;
}

// Projection helpers: clips = |z| > gamma, scale = gamma / |z| where it clips, else 1, and norm = |x|, from squared
// norms. The reverse mode differentiates the branch that clips gives: it calls it on the same fma chain. FP64
// decides as the IEEE square root would and uses rsqrt_halley where the square lies inside float's range, the IEEE
// square root and division elsewhere. FP32 compares squares and uses the hardware reciprocal square root (relative error ~1e-7, below FP32 field noise).
template <typename T> struct Proj;
template <> struct Proj<double> {
    __device__ __forceinline__ static bool clips(double nz2, double gm) {
        return in_float_range(nz2) ? root_exceeds(nz2, gm) : sqrt(nz2) > gm;
    }
    __device__ __forceinline__ static double scale(double nz2, double gm) {
        double s = 1.0;
        if (in_float_range(nz2)) {
            if (root_exceeds(nz2, gm)) s = gm * rsqrt_halley(nz2);
        } else {
            const double nz = sqrt(nz2);
            if (nz > gm) s = gm / nz;
        }
        return s;
    }
    __device__ __forceinline__ static double norm(double x2) {
        return in_float_range(x2) ? x2 * rsqrt_halley(x2) : sqrt(x2);
    }
};
template <> struct Proj<float> {
    __device__ __forceinline__ static bool clips(float nz2, float gm) { return nz2 > gm * gm; }
    __device__ __forceinline__ static float scale(float nz2, float gm) {
        return clips(nz2, gm) ? gm * rsqrtf(nz2) : 1.0f;
    }
    __device__ __forceinline__ static float norm(float x2) { return x2 > 0.0f ? x2 * rsqrtf(x2) : 0.0f; }
};

// The factors 1/sqrt2 of div^- A* (pass 1) and of A grad^+ (the update, the only reader of phi). FP64 is bound by
// its arithmetic: its passes leave both out and put their product 1/2 into the Poisson gain, so that d of pass 1
// is sqrt2 times, and phi is 1/sqrt2 times the paper's, and a face of the update costs four operations instead of
// six. FP32 is bound by HBM and keeps the factors where they are.
template <typename T>
__host__ __device__ constexpr bool fold_h() { return sizeof(T) == 8; }
template <typename T>
__host__ __device__ constexpr T div_scale() { return fold_h<T>() ? T(1) : T(0.70710678118654752440084436210485); }
template <typename T>
__host__ __device__ constexpr double poisson_scale() { return fold_h<T>() ? 0.5 : 1.0; }

template <bool B> struct BoolC { static constexpr bool value = B; };

template <typename T> struct Pk;
template <> struct Pk<float> {
    using V = float2;
    static constexpr int N = 2;
    __device__ __forceinline__ static V set(float a) { return make_float2(a, a); }
    __device__ __forceinline__ static V make(float a, float b) { return make_float2(a, b); }
    __device__ __forceinline__ static V add(V a, V b) { return __fadd2_rn(a, b); }
    __device__ __forceinline__ static V sub(V a, V b) { return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a); }
    __device__ __forceinline__ static V mul(V a, V b) { return __fmul2_rn(a, b); }
    __device__ __forceinline__ static V fma(V a, V b, V c) { return __ffma2_rn(a, b, c); }
    __device__ __forceinline__ static float get(V a, int i) { return i ? a.y : a.x; }
    __device__ __forceinline__ static float sum(V a) { return a.x + a.y; }
    // scale of P_C and gamma |x| per voxel (Proj<float>)
    __device__ __forceinline__ static V scale(V n2, V g) {
        return make_float2(Proj<float>::scale(n2.x, g.x), Proj<float>::scale(n2.y, g.y));
    }
    __device__ __forceinline__ static V norm(V x2) {
        return make_float2(Proj<float>::norm(x2.x), Proj<float>::norm(x2.y));
    }
};
template <> struct Pk<double> {
    using V = double;
    static constexpr int N = 1;
    __device__ __forceinline__ static V set(double a) { return a; }
    __device__ __forceinline__ static V make(double a, double) { return a; }
    __device__ __forceinline__ static V add(V a, V b) { return __dadd_rn(a, b); }
    __device__ __forceinline__ static V sub(V a, V b) { return __dsub_rn(a, b); }
    __device__ __forceinline__ static V mul(V a, V b) { return __dmul_rn(a, b); }
    __device__ __forceinline__ static V fma(V a, V b, V c) { return __fma_rn(a, b, c); }
    __device__ __forceinline__ static double get(V a, int) { return a; }
    __device__ __forceinline__ static double sum(V a) { return a; }
    __device__ __forceinline__ static V scale(V n2, V g) { return Proj<double>::scale(n2, g); }
    __device__ __forceinline__ static V norm(V x2) { return Proj<double>::norm(x2); }
};

// The state fields of one solve as a pass reads them: (e, v), or (z, s) in a and the first N values of b.
template <typename T>
struct StateSrc {
    const T* __restrict__ a;
    const T* __restrict__ b;
    long long N;
    typename Pk<T>::V nir;   // -1 / rho
    typename Pk<T>::V irp;   // 1 / rho_prev ((z, s) format)
};

// 1 / rho and 1 / rho_prev: by one thread of a block for all of them, through shared memory (an FP64 division of
// every thread of a block costs the SM as much as the update of some twenty voxels).
template <typename T>
__device__ __forceinline__ void state_recip(const SolveScalars& S, T (&r)[2]) {
    r[0] = T(1) / (T)S.rho;
    r[1] = sizeof(T) == 4 ? T(1) / (T)S.rho_prev : T(1);
}

template <typename T>
__device__ __forceinline__ StateSrc<T> state_src(const Ptrs<T>& p, const SolveScalars& S, int s, long long N,
                                                 const T (&recip)[2]) {
    StateSrc<T> f;
    const long long cur = (long long)(S.iters & 1) * p.sstride + (long long)s * 6 * N;
    f.a = p.e + cur;
    f.b = p.v + cur;
    f.N = N;
    f.nir = Pk<T>::set(-recip[0]);
    f.irp = Pk<T>::set(recip[1]);
    return f;
}

// Whether the current state of a solve is in the (z, s) format.
template <typename T>
__device__ __forceinline__ bool state_is_zs(const SolveScalars& S) {
    return sizeof(T) == 4 && S.zs_iter == S.iters + 1;
}

// (e, v, w = e - v / rho) of a pack from what the format stores: (z, s) or (e, v).
template <typename T, bool ZS>
__device__ __forceinline__ void state_evw(const StateSrc<T>& f, typename Pk<T>::V x, typename Pk<T>::V y,
                                          typename Pk<T>::V& e, typename Pk<T>::V& v, typename Pk<T>::V& w) {
    using P = Pk<T>;
    if constexpr (ZS) {
        v = P::mul(x, y);
        e = P::mul(P::sub(x, v), f.irp);
    } else {
        e = x;
        v = y;
    }
    w = P::fma(v, f.nir, e);
}

// Where the voxels of a group lie. W > 0: W consecutive voxels of a z row (one offset, vector accesses);
// W = 0: the Pk<T>::N voxels of one pack, anywhere (one offset each).
template <typename T, int W>
struct GroupOff {
    static constexpr int M = W > 0 ? 1 : Pk<T>::N;
    long long o[M];
};

template <typename T, int W>
struct Group {
    using P = Pk<T>;
    using V = typename P::V;
    using Off = GroupOff<T, W>;
    static constexpr int VPT = W > 0 ? W : P::N;   // voxels of the group
    static constexpr int NP = VPT / P::N;          // packs of the group
    // CG: through L2 only, for data that the same launch writes
    template <bool CG = false>
    __device__ __forceinline__ static void ld(const T* __restrict__ base, const Off& off, V (&x)[NP]) {
        if constexpr (W > 0) {
            T t[W];
            if constexpr (CG)
                VecN<T, W>::ldcg(base + off.o[0], t);
            else
                VecN<T, W>::ld(base + off.o[0], t);
#pragma unroll
            for (int q = 0; q < NP; ++q) x[q] = P::make(t[q * P::N], t[q * P::N + P::N - 1]);
        } else {
            T t[P::N];
#pragma unroll
            for (int i = 0; i < P::N; ++i) t[i] = CG ? __ldcg(base + off.o[i]) : __ldg(base + off.o[i]);
            x[0] = P::make(t[0], t[P::N - 1]);
        }
    }
    // valid: whether the second voxel of a strided pack exists (W = 0)
    __device__ __forceinline__ static void st(T* base, const Off& off, const V (&x)[NP], bool valid) {
        if constexpr (W > 0) {
            T t[W];
#pragma unroll
            for (int u = 0; u < W; ++u) t[u] = P::get(x[u / P::N], u % P::N);
            VecN<T, W>::st(base + off.o[0], t);
        } else {
            base[off.o[0]] = P::get(x[0], 0);
            if constexpr (P::N > 1) {
                if (valid) base[off.o[P::N - 1]] = P::get(x[0], 1);
            }
        }
    }
    // x moved by one voxel along z inside the group: up (x of the next voxel, `edge` after the last) or down
    __device__ __forceinline__ static void shift_up(const V (&x)[NP], T edge, V (&r)[NP]) {
        T t[VPT + 1];
#pragma unroll
        for (int u = 0; u < VPT; ++u) t[u] = P::get(x[u / P::N], u % P::N);
        t[VPT] = edge;
#pragma unroll
        for (int q = 0; q < NP; ++q) r[q] = P::make(t[q * P::N + 1], t[q * P::N + P::N]);
    }
    __device__ __forceinline__ static void shift_down(const V (&x)[NP], T edge, V (&r)[NP]) {
        T t[VPT + 1];
        t[0] = edge;
#pragma unroll
        for (int u = 0; u < VPT; ++u) t[u + 1] = P::get(x[u / P::N], u % P::N);
#pragma unroll
        for (int q = 0; q < NP; ++q) r[q] = P::make(t[q * P::N], t[q * P::N + P::N - 1]);
    }
};

// Pass 1's divergence d = div^- A* (e - v / rho) (Sec. 2.2, Eq. 17) of kDivW consecutive voxels of a z row, with
// vector loads: d(p) = (1/sqrt2) sum_a [w1_a(p) - w1_a(p - e_a) + w2_a(p + e_a) - w2_a(p)]. kp / km: the voxels
// just after / before the group (periodic). Two voxels per thread: all loads of a group then fit 64 registers
// and are in flight at once in four blocks per SM.
constexpr int kDivW = 2;

template <typename T, bool ZS>
__device__ __forceinline__ void div_group(const StateSrc<T>& f, const RowNb& rn, int k0, int kp, int km,
                                          T (&d)[kDivW]) {
    using P = Pk<T>;
    using V = typename P::V;
    using G = Group<T, kDivW>;
    constexpr int NP = G::NP;
    const long long N = f.N;
    const typename G::Off own = {{rn.row + k0}};
    const typename G::Off om[2] = {{{rn.im + k0}}, {{rn.jm + k0}}}, op[2] = {{{rn.ip + k0}}, {{rn.jp + k0}}};
    // x, y: what the format stores of a component (z_c and s, or e_c and v_c)
    V x0[6][NP], y0[ZS ? 1 : 6][NP], xm[2][NP], ym[2][NP], xp[2][NP], yp[2][NP];
#pragma unroll
    for (int c = 0; c < 6; ++c) G::ld(f.a + c * N, own, x0[c]);
#pragma unroll
    for (int c = 0; c < (ZS ? 1 : 6); ++c) G::ld(f.b + c * N, own, y0[c]);
#pragma unroll
    for (int a = 0; a < 2; ++a) {
        G::ld(f.a + a * N, om[a], xm[a]);
        G::ld(ZS ? f.b : f.b + a * N, om[a], ym[a]);
        G::ld(f.a + (3 + a) * N, op[a], xp[a]);
        G::ld(ZS ? f.b : f.b + (3 + a) * N, op[a], yp[a]);
    }
    const T xa = __ldg(f.a + 5 * N + rn.row + kp), ya = __ldg((ZS ? f.b : f.b + 5 * N) + rn.row + kp);
    const T xb = __ldg(f.a + 2 * N + rn.row + km), yb = __ldg((ZS ? f.b : f.b + 2 * N) + rn.row + km);
    V w[6][NP], acc[NP], e, v;
#pragma unroll
    for (int c = 0; c < 6; ++c)
#pragma unroll
        for (int q = 0; q < NP; ++q) state_evw<T, ZS>(f, x0[c][q], y0[ZS ? 0 : c][q], e, v, w[c][q]);
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int q = 0; q < NP; ++q) {
            V n, t;
            state_evw<T, ZS>(f, xm[a][q], ym[a][q], e, v, n);
            t = P::sub(w[a][q], n);
            state_evw<T, ZS>(f, xp[a][q], yp[a][q], e, v, n);
            t = P::sub(P::add(t, n), w[3 + a][q]);
            acc[q] = a == 0 ? t : P::add(acc[q], t);
        }
    T wa, wb;
    {
        V w_;
        state_evw<T, ZS>(f, P::make(xa, xb), P::make(ya, yb), e, v, w_);
        wa = P::get(w_, 0);
        if constexpr (P::N == 1) state_evw<T, ZS>(f, P::make(xb, xb), P::make(yb, yb), e, v, w_);
        wb = P::get(w_, P::N - 1);
    }
    V lo[NP], hi[NP];
    G::shift_down(w[2], wb, lo);
    G::shift_up(w[5], wa, hi);
#pragma unroll
    for (int q = 0; q < NP; ++q) {
        const V t = P::sub(P::add(P::sub(w[2][q], lo[q]), hi[q]), w[5][q]);
        V r = P::add(acc[q], t);
        if constexpr (!fold_h<T>()) r = P::mul(P::set(div_scale<T>()), r);
#pragma unroll
        for (int i = 0; i < P::N; ++i) d[q * P::N + i] = P::get(r, i);
    }
}

// The same of one voxel with scalar loads (any N3).
template <typename T, bool ZS>
__device__ __forceinline__ T div_voxel(const StateSrc<T>& f, const RowNb& rn, int k, int kp, int km) {
    using P = Pk<T>;
    using V = typename P::V;
    const long long N = f.N;
    // w of two components per pack (FP32) or one after the other (FP64)
    auto w2 = [&](int c0, long long o0, int c1, long long o1, T& r0, T& r1) {
        const T x0 = __ldg(f.a + c0 * N + o0), y0 = __ldg((ZS ? f.b : f.b + c0 * N) + o0);
        const T x1 = __ldg(f.a + c1 * N + o1), y1 = __ldg((ZS ? f.b : f.b + c1 * N) + o1);
        V e, v, w;
        state_evw<T, ZS>(f, P::make(x0, x1), P::make(y0, y1), e, v, w);
        r0 = P::get(w, 0);
        if constexpr (P::N == 1) state_evw<T, ZS>(f, P::make(x1, x1), P::make(y1, y1), e, v, w);
        r1 = P::get(w, P::N - 1);
    };
    const long long o = rn.row + k;
    const long long om[3] = {rn.im + k, rn.jm + k, rn.row + km}, op[3] = {rn.ip + k, rn.jp + k, rn.row + kp};
    T sa[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        T w1, w1m, w2p, w2o;
        w2(a, o, a, om[a], w1, w1m);
        w2(3 + a, op[a], 3 + a, o, w2p, w2o);
        sa[a] = w1 - w1m + w2p - w2o;
    }
    return div_scale<T>() * (sa[0] + sa[1] + sa[2]);
}

}  // namespace ccmf
