// The update pass (pass 6 of the iteration, see ccmf_kernels.cuh) on register packs, and the format changes
// of the FP32 state (ccmf_state.cuh).
#pragma once

#include "ccmf_kernels.cuh"

namespace ccmf {

// Constants of one solve's update in pack form.
template <typename T>
struct UpdConsts {
    using V = typename Pk<T>::V;
    V h, nh, half, alpha, nbeta, rho, irho;
    V xi[3];   // xi_bar, over sqrt2 where the factors are folded (fold_h)
};

template <typename T>
struct UpdIo {
    StateSrc<T> f;
    const T* __restrict__ phi;
    const T* __restrict__ gam;
    T* __restrict__ ao;     // the other copy of the state: e or z
    T* __restrict__ bo;     // v or s
    T* cut;
    T* flow;
    T* zout;                // z = v + rho xi of an (e, v)-format update, may be null
};

template <typename T>
__device__ __forceinline__ UpdConsts<T> upd_consts(const StepConsts<T>& C) {
    using P = Pk<T>;
    UpdConsts<T> K;
    K.h = P::set(C.h);
    K.nh = P::set(-C.h);
    K.half = P::set(T(0.5));
    K.alpha = P::set(C.alpha);
    K.nbeta = P::set(-C.beta);
    K.rho = P::set(C.rho);
    K.irho = P::set(C.irho);
#pragma unroll
    for (int a = 0; a < 3; ++a) K.xi[a] = P::set(fold_h<T>() ? C.hxi[a] : C.xi[a]);
    return K;
}

template <typename T, bool OUT>
__device__ __forceinline__ UpdIo<T> upd_io(const Ptrs<T>& p, const SolveScalars& S, int s, long long N,
                                           const T (&recip)[2]) {
    const long long other = (long long)(1 - (S.iters & 1)) * p.sstride + (long long)s * 6 * N;
    UpdIo<T> io;
    io.f = state_src<T>(p, S, s, N, recip);
    io.phi = p.phi + (size_t)s * N;
    io.gam = gamma_of(p, s);
    io.ao = p.e + other;
    io.bo = p.v + other;
    io.cut = OUT && p.cut ? p.cut + (size_t)s * 6 * N : nullptr;
    io.flow = OUT && p.flow ? p.flow + (size_t)s * 3 * N : nullptr;
    io.zout = !OUT && p.zout ? p.zout + (size_t)s * 6 * N : nullptr;
    return io;
}

// One group of the update. OUT: the final evaluation (cut, flow, sums of the state) instead of an
// update. RZS / WZS: the format read / written. RULE: the penalty sums accumulated: 0 those of the BB and
// residual-balancing rules, 1 none (constant or replayed penalties), 2 the LTD rule's, -1 all. mask: 1 per voxel that counts (a strided pack whose second
// voxel lies beyond the grid repeats the first with mask 0).
template <typename T, int W, bool OUT, int RULE, bool RZS, bool WZS, bool CG = false>
__device__ __forceinline__ void update_group(const Geom& g, const UpdIo<T>& io, const UpdConsts<T>& K, long long lin0,
                                             long long lin1, bool valid, typename Pk<T>::V (&acc)[kNSum]) {
    using P = Pk<T>;
    using V = typename P::V;
    using G = Group<T, W>;
    using Off = typename G::Off;
    constexpr int NP = G::NP;
    const StateSrc<T>& f = io.f;
    const long long N = f.N;
    Off own, ip, im, jp, jm, kp, km;
#pragma unroll
    for (int m = 0; m < Off::M; ++m) {
        const long long lin = m == 0 ? lin0 : lin1;
        const unsigned row = fdiv((unsigned)lin, g.div_n3);
        const int k = (int)(lin - (long long)row * g.n3);
        const RowNb rn = row_neighbours(g, row);
        constexpr int step = W > 0 ? W : 1;
        own.o[m] = lin;
        ip.o[m] = rn.ip + k;
        im.o[m] = rn.im + k;
        jp.o[m] = rn.jp + k;
        jm.o[m] = rn.jm + k;
        kp.o[m] = rn.row + ((k + step == g.n3) ? 0 : k + step);
        km.o[m] = rn.row + ((k == 0) ? g.n3 - 1 : k - 1);
    }
    // the scalar of the (z, s) format, or component c of v
    auto second = [&](int c, const Off& o, V (&y)[NP]) { G::ld(RZS ? f.b : f.b + c * N, o, y); };
    V ec[6][NP], vc[6][NP], w[6][NP];
    {
        V s[NP];
        if constexpr (RZS) second(0, own, s);
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            V x[NP], y[NP];
            G::ld(f.a + c * N, own, x);
            if constexpr (!RZS) second(c, own, y);
#pragma unroll
            for (int q = 0; q < NP; ++q)
                state_evw<T, RZS>(f, x[q], RZS ? s[q] : y[q], ec[c][q], vc[c][q], w[c][q]);
        }
    }
    // w and v of component c of another row
    auto other = [&](int c, const Off& o, V (&wo)[NP], V (&vo)[NP]) {
        V x[NP], y[NP], eo;
        G::ld(f.a + c * N, o, x);
        second(c, o, y);
#pragma unroll
        for (int q = 0; q < NP; ++q) state_evw<T, RZS>(f, x[q], y[q], eo, vo[q], wo[q]);
    };
    V gm[NP], ph[NP], w2p[3][NP], v2p[3][NP], w1m[3][NP], php[3][NP], phm[3][NP], vdump[NP];
    G::ld(io.gam, own, gm);
    G::template ld<CG>(io.phi, own, ph);
    other(3, ip, w2p[0], v2p[0]);
    other(0, im, w1m[0], vdump);
    other(4, jp, w2p[1], v2p[1]);
    other(1, jm, w1m[1], vdump);
    G::template ld<CG>(io.phi, ip, php[0]);
    G::template ld<CG>(io.phi, im, phm[0]);
    G::template ld<CG>(io.phi, jp, php[1]);
    G::template ld<CG>(io.phi, jm, phm[1]);
    if constexpr (W > 0) {
        // z neighbours: inside the group, or one voxel on each side of it
        const T xa = __ldg(f.a + 5 * N + kp.o[0]), ya = __ldg((RZS ? f.b : f.b + 5 * N) + kp.o[0]);
        const T xb = __ldg(f.a + 2 * N + km.o[0]), yb = __ldg((RZS ? f.b : f.b + 2 * N) + km.o[0]);
        const T pa = CG ? __ldcg(io.phi + kp.o[0]) : __ldg(io.phi + kp.o[0]);
        const T pb = CG ? __ldcg(io.phi + km.o[0]) : __ldg(io.phi + km.o[0]);
        T wa, wb, va;
        V e_, v_, w_;
        if constexpr (P::N == 2) {
            state_evw<T, RZS>(f, P::make(xa, xb), P::make(ya, yb), e_, v_, w_);
            wa = P::get(w_, 0);
            va = P::get(v_, 0);
            wb = P::get(w_, 1);
        } else {
            state_evw<T, RZS>(f, P::make(xa, xa), P::make(ya, ya), e_, v_, w_);
            wa = P::get(w_, 0);
            va = P::get(v_, 0);
            state_evw<T, RZS>(f, P::make(xb, xb), P::make(yb, yb), e_, v_, w_);
            wb = P::get(w_, 0);
        }
        G::shift_up(w[5], wa, w2p[2]);
        if constexpr (OUT) G::shift_up(vc[5], va, v2p[2]);
        G::shift_down(w[2], wb, w1m[2]);
        G::shift_up(ph, pa, php[2]);
        G::shift_down(ph, pb, phm[2]);
    } else {
        other(5, kp, w2p[2], v2p[2]);
        other(2, km, w1m[2], vdump);
        G::template ld<CG>(io.phi, kp, php[2]);
        G::template ld<CG>(io.phi, km, phm[2]);
    }
    const V mask = P::make(T(1), valid ? T(1) : T(0));
    auto take = [&](int i, V x) { acc[i] = (W > 0 || P::N == 1) ? P::add(acc[i], x) : P::fma(x, mask, acc[i]); };
    // FP64 sums products straight into the accumulators (one addition less per sum); FP32 sums a voxel's six first
    constexpr bool kDirect = sizeof(T) == 8;
    auto sum_sq = [&](int i, V a, V b, V& local) {
        if constexpr (kDirect)
            acc[i] = P::fma(a, b, acc[i]);
        else
            local = P::fma(a, b, local);
    };
    V oa[6][NP], ob[6][NP], of[3][NP];
#pragma unroll
    for (int q = 0; q < NP; ++q) {
        // xi^{k+1/2} = w - A (A* w - grad phi - xi_bar), by the six faces of the voxel 
        V x[6];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            if constexpr (fold_h<T>()) {
                const V up = P::add(P::sub(php[a][q], ph[q]), K.xi[a]);
                const V um = P::add(P::sub(ph[q], phm[a][q]), K.xi[a]);
                x[a] = P::fma(K.half, P::sub(w[a][q], w2p[a][q]), up);
                x[3 + a] = P::fma(K.half, P::sub(w[3 + a][q], w1m[a][q]), um);
            } else {
                const V yp = P::sub(P::fma(K.h, P::add(w[a][q], w2p[a][q]), P::sub(ph[q], php[a][q])), K.xi[a]);
                const V ym = P::sub(P::fma(K.h, P::add(w1m[a][q], w[3 + a][q]), P::sub(phm[a][q], ph[q])), K.xi[a]);
                x[a] = P::fma(K.nh, yp, w[a][q]);
                x[3 + a] = P::fma(K.nh, ym, w[3 + a][q]);
            }
            if constexpr (OUT) of[a][q] = P::mul(K.h, P::add(vc[a][q], v2p[a][q]));   // A* v
        }
        V r2 = P::set(T(0)), nx2 = P::set(T(0)), nz2 = P::set(T(0)), z[6];
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            const V d = P::sub(x[c], ec[c][q]);
            sum_sq(kSumRes, d, d, r2);
            nx2 = P::fma(x[c], x[c], nx2);
            take(kSumV + c, vc[c][q]);
            if constexpr (OUT) {
                oa[c][q] = x[c];
            } else {
                // over-relaxation alpha x - beta e, alpha = 2 (1 - delta), beta = 1 - 2 delta; alpha - beta = 1
                const V m = fold_h<T>() ? P::fma(K.alpha, d, ec[c][q])
                                        : P::fma(K.alpha, x[c], P::mul(K.nbeta, ec[c][q]));
                z[c] = P::fma(K.rho, m, vc[c][q]);
                nz2 = P::fma(z[c], z[c], nz2);
            }
        }
        if constexpr (!kDirect) take(kSumRes, r2);
        if constexpr (kDirect)
            acc[kSumPrimal] = P::fma(gm[q], P::norm(nx2), acc[kSumPrimal]);
        else
            take(kSumPrimal, P::mul(gm[q], P::norm(nx2)));
        if constexpr (!OUT) {
            const V s = P::scale(nz2, gm[q]);
            const V te = P::mul(P::sub(P::set(T(1)), s), K.irho);
            V dvde = P::set(T(0)), dede = P::set(T(0)), dvdv = P::set(T(0)), vv = P::set(T(0)), ee = P::set(T(0));
#pragma unroll
            for (int c = 0; c < 6; ++c) {
                const V vn = P::mul(z[c], s);
                // e' = (z - v') / rho; FP64 saves an operation a component by z ((1 - s) / rho)
                const V en = fold_h<T>() ? P::mul(z[c], te) : P::mul(P::sub(z[c], vn), K.irho);
                const V dv = P::sub(vn, vc[c][q]), de = P::sub(en, ec[c][q]);
                if constexpr (RULE == 0 || RULE == -1) {
                    sum_sq(kSumDvDe, dv, de, dvde);
                    sum_sq(kSumDeDe, de, de, dede);
                    sum_sq(kSumDvDv, dv, dv, dvdv);
                }
                if constexpr (RULE == 2 || RULE == -1) {
                    sum_sq(kSumVV, vn, vn, vv);
                    sum_sq(kSumEE, en, en, ee);
                }
                if constexpr (WZS) {
                    oa[c][q] = z[c];
                } else {
                    oa[c][q] = en;
                    ob[c][q] = vn;
                }
            }
            if constexpr (WZS) ob[0][q] = s;
            if constexpr (!kDirect && (RULE == 0 || RULE == -1)) {
                take(kSumDvDe, dvde);
                take(kSumDeDe, dede);
                take(kSumDvDv, dvdv);
            }
            if constexpr (!kDirect && (RULE == 2 || RULE == -1)) {
                take(kSumVV, vv);
                take(kSumEE, ee);
            }
            if constexpr (!WZS) {
                if (io.zout) {   // kept for the reverse pass
                    if constexpr (W == 0) {
#pragma unroll
                        for (int c = 0; c < 6; ++c) {
                            V t[1] = {z[c]};
                            Group<T, 0>::st(io.zout + c * N, own, t, valid);
                        }
                    } else {
#pragma unroll
                        for (int c = 0; c < 6; ++c)
#pragma unroll
                            for (int i = 0; i < P::N; ++i) io.zout[c * N + lin0 + q * P::N + i] = P::get(z[c], i);
                    }
                }
            }
        }
    }
    if constexpr (OUT) {
        if (io.cut) {
#pragma unroll
            for (int c = 0; c < 6; ++c) G::st(io.cut + c * N, own, oa[c], valid);
        }
        if (io.flow) {
#pragma unroll
            for (int a = 0; a < 3; ++a) G::st(io.flow + a * N, own, of[a], valid);
        }
    } else {
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            G::st(io.ao + c * N, own, oa[c], valid);
            if constexpr (!WZS) G::st(io.bo + c * N, own, ob[c], valid);
        }
        if constexpr (WZS) G::st(io.bo, own, ob[0], valid);
    }
}

// The update pass (OUT: the final evaluation, which writes the cut xi^{K+1/2} and the flow A* v^K instead
// of advancing the state). W consecutive voxels per thread group with vector accesses (N3 a multiple
// of W, gamma aligned), or W = 0: packs of voxels kThreads apart with scalar accesses (any N3, any alignment;
// neighbouring threads still take neighbouring voxels).
//
// Dynamic schedule: blocks take chunks of vec_chunk_groups x kThreads groups (32 rows at N3 = 512 and W = 4)
// in order from a per-solve ticket counter, the next ticket fetched while the current chunk runs (one chunk per
// block, without the counter, where the blocks are as many).
// The chunks in flight then form one narrow front through the grid, and the x- and y-neighbour rows a chunk
// reads were read as other chunks' own rows moments before, so they come from L2. (With a
// grid-stride loop the blocks drift apart over a long pass; at 512^3, 42 % more than the algorithmic
// reads came from DRAM.) Each chunk stores its own partial sums and the last block reduces them in
// chunk order, so the result does not depend on which block took which chunk.
template <typename T, int W, bool OUT, int RULE, bool WZS, int MINB>
__global__ void __launch_bounds__(kThreads, MINB) k_update(Geom g, Ptrs<T> p, LoopConfig cfg) {
    using P = Pk<T>;
    using V = typename P::V;
    constexpr int VPT = Group<T, W>::VPT;
    const int s = blockIdx.y + p.s0;
    SolveScalars& S = p.sc[s];
    if (!OUT && !S.active) return;
    const long long N = g.N;
    const double rho_d = S.rho;
    __shared__ StepConsts<T> C;
    __shared__ T recip[2];
    __shared__ unsigned ticket[2];
    const long long nchunks = vec_update_chunks<T>(N, VPT);
    if (threadIdx.x == 0) {
        ticket[0] = gridDim.x < nchunks ? atomicAdd(&S.chunk, 1u) : blockIdx.x;
        C = step_consts<T>(S, cfg);
        state_recip<T>(S, recip);
    }
    __syncthreads();
    const UpdConsts<T> K = upd_consts<T>(C);
    const UpdIo<T> io = upd_io<T, OUT>(p, S, s, N, recip);
    const bool rzs = state_is_zs<T>(S);
    const int cgroups = vec_chunk_groups<T>(N, VPT);
    double* part = p.partial + (size_t)s * nchunks * kNSum;
    for (int it = 0;; ++it) {
        const unsigned ck = ticket[it & 1];
        if (ck >= nchunks) break;   // the same value for the whole block
        if (threadIdx.x == 0)
            ticket[(it + 1) & 1] = gridDim.x < nchunks ? atomicAdd(&S.chunk, 1u) : (unsigned)nchunks;
        V acc[kNSum];
#pragma unroll
        for (int q = 0; q < kNSum; ++q) acc[q] = P::set(T(0));
        auto sweep = [&](auto fmt) {
            constexpr bool RZS = decltype(fmt)::value;
#pragma unroll 1
            for (int gi = 0; gi < cgroups; ++gi) {
                const long long gb = ((long long)ck * cgroups + gi) * kThreads;   // first group of the block
                const long long lin0 = W > 0 ? (gb + threadIdx.x) * W : gb * VPT + threadIdx.x;
                if (lin0 < N) {
                    const bool valid = W > 0 || lin0 + kThreads < N;
                    update_group<T, W, OUT, RULE, RZS, WZS>(g, io, K, lin0, valid ? lin0 + kThreads : lin0, valid,
                                                            acc);
                }
            }
        };
        if constexpr (sizeof(T) == 4) {
            if (rzs)
                sweep(BoolC<true>{});
            else
                sweep(BoolC<false>{});
        } else {
            sweep(BoolC<false>{});
        }
        T sums[kNSum];
#pragma unroll
        for (int q = 0; q < kNSum; ++q) sums[q] = P::sum(acc[q]);
        block_store_partial<T, kNSum>(sums, part, ck);
        __syncthreads();   // the next ticket is visible, this one is read by everyone, red[] is free
    }
    if (block_ticket(&S.counter, gridDim.x))
        update_finish<T, OUT, kThreads, false, WZS>(g, p, cfg, S, s, rho_d, part, (int)nchunks);
}

// ---------------------------------------------------------------------------
// Format changes of the FP32 state.
// ---------------------------------------------------------------------------

// (z, s) -> (e, v) of the solves whose current copy is in the (z, s) format: into the other copy
// (to_other = 1, for an export; the next update overwrites that copy) or in place (to_other = 0, before an
// update variant that reads (e, v); k_state_mark_ev records the change afterwards). A thread reads the seven
// values of its voxel before it writes them over.
template <typename T>
__global__ void __launch_bounds__(kThreads) k_state_to_ev(Geom g, Ptrs<T> p, int to_other) {
    using P = Pk<T>;
    const int s = blockIdx.y + p.s0;
    const SolveScalars& S = p.sc[s];
    if (!state_is_zs<T>(S)) return;
    const long long N = g.N;
    const int par = S.iters & 1;
    const long long src = (long long)par * p.sstride + (long long)s * 6 * N;
    const long long dst = (long long)(to_other ? 1 - par : par) * p.sstride + (long long)s * 6 * N;
    T recip[2];
    state_recip<T>(S, recip);
    const StateSrc<T> f = state_src<T>(p, S, s, N, recip);
    const long long stride = (long long)gridDim.x * kThreads;
    for (long long lin = (long long)blockIdx.x * kThreads + threadIdx.x; lin < N; lin += stride) {
        const T sc = p.v[src + lin];
        T z[6];
#pragma unroll
        for (int c = 0; c < 6; ++c) z[c] = p.e[src + c * N + lin];
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            typename P::V e, v, w;
            state_evw<T, true>(f, P::set(z[c]), P::set(sc), e, v, w);
            p.e[dst + c * N + lin] = P::get(e, 0);
            p.v[dst + c * N + lin] = P::get(v, 0);
        }
    }
}

template <typename T>
__global__ void k_state_mark_ev(SolveScalars* sc, int batch) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s < batch) sc[s].zs_iter = 0;
}

}  // namespace ccmf
