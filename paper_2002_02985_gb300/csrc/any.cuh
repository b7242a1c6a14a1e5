// FFT-carrying kernels for any 2^a3^b5^c axis length: the length, the tile width and the
// radices of its passes are read at run time, each butterfly is compiled for its radix
// (2 3 4 5 6 8 9 10 12 15 16, so that lengths up to 256 need two passes and up to 1024
// three, where prime-power radices up to 8 need three and four).
//
// Index arithmetic is what such kernels pay for their generality: every division of the
// inner loops is a shift (tiles are a power of two wide) or a multiplication by a
// precomputed reciprocal, and no 64-bit division is left inside a loop.
#pragma once

#include "recip.cuh"

namespace ofdft {

// ---------------------------------------------------------------- composite butterflies
// R = A B with A, B coprime (Good-Thomas: no twiddles), inverse residues at compile time
constexpr int any_inv(int a, int m) {
    for (int x = 1; x < m; x++)
        if (a * x % m == 1) return x;
    return 1;
}
template <int DIR, int R, typename C> __device__ __forceinline__ void adft(C *v);
template <int DIR, int A, int B, typename C> __device__ __forceinline__ void adft_coprime(C *v) {
    constexpr int R = A * B, ca = B * any_inv(B % A, A), cb = A * any_inv(A % B, B);
    C t[A][B];
#pragma unroll
    for (int b = 0; b < B; b++) {
        C u[A];
#pragma unroll
        for (int i = 0; i < A; i++) u[i] = v[(B * i + A * b) % R];
        adft<DIR, A>(u);
#pragma unroll
        for (int i = 0; i < A; i++) t[i][b] = u[i];
    }
#pragma unroll
    for (int i = 0; i < A; i++) {
        adft<DIR, B>(t[i]);
#pragma unroll
        for (int b = 0; b < B; b++) v[(ca * i + cb * b) % R] = t[i][b];
    }
}
template <int DIR, typename C> __device__ __forceinline__ void adft9(C *v) {
    typedef decltype(C::x) T;
    C t[3][3];
#pragma unroll
    for (int b = 0; b < 3; b++) {
        t[b][0] = v[b];
        t[b][1] = v[b + 3];
        t[b][2] = v[b + 6];
        dft3<DIR>(t[b]);
    }
    const T s = (T)DIR;
    auto rot = [&](C &x, T cr, T si) { x = cmake<C>(x.x * cr - s * x.y * si, x.y * cr + s * x.x * si); };
    rot(t[1][1], (T)0.766044443118978, (T)0.6427876096865394);       // W9^1
    rot(t[1][2], (T)0.17364817766693033, (T)0.984807753012208);      // W9^2
    rot(t[2][1], (T)0.17364817766693033, (T)0.984807753012208);      // W9^2
    rot(t[2][2], (T)-0.9396926207859084, (T)0.3420201433256687);     // W9^4
#pragma unroll
    for (int k = 0; k < 3; k++) {
        C u[3] = {t[0][k], t[1][k], t[2][k]};
        dft3<DIR>(u);
        v[k] = u[0];
        v[k + 3] = u[1];
        v[k + 6] = u[2];
    }
}
template <int DIR, int R, typename C> __device__ __forceinline__ void adft(C *v) {
    if constexpr (R == 6) adft_coprime<DIR, 2, 3>(v);
    else if constexpr (R == 9) adft9<DIR>(v);
    else if constexpr (R == 10) adft_coprime<DIR, 2, 5>(v);
    else if constexpr (R == 12) adft_coprime<DIR, 4, 3>(v);
    else if constexpr (R == 15) adft_coprime<DIR, 3, 5>(v);
    else dft<DIR, R>(v);
}

// ---------------------------------------------------------------- one pass
// Butterflies idx = threadIdx.x, + blockDim.x, ... of a pass.  dec(idx, b, j) gives the sequence
// b and the butterfly j; element e of sequence b sits e `ld` steps from in(b) and out(b) (Src and
// Dst: shared memory or a guarded global column), so an element costs one multiply-add of
// addressing.
template <typename C> struct AnyShared {
    C *s;
    int ld;
    __device__ __forceinline__ C *at(int b) const { return s + b; }
    __device__ __forceinline__ bool ok() const { return true; }
};
template <typename C> struct AnyGlobal {
    C *g;
    int ld;
    bool valid;
    __device__ __forceinline__ C *at(int) const { return g; }
    __device__ __forceinline__ bool ok() const { return valid; }
};
template <int DIR, int R, typename C, class Dec, class Src, class Dst>
__device__ __forceinline__ void any_pass_r(const AnyPass p, int total, int nthr, const C *__restrict__ tw, Dec dec,
                                           Src src, Dst dst) {
    const int ns = p.ns, nb = p.nb, stride = p.stride, magic = p.magic;
    const int istep = nb * src.ld, ostep = ns * dst.ld;
#pragma unroll 1
    for (int idx = threadIdx.x; idx < total; idx += nthr) {
        int b, j;
        dec(idx, b, j);
        C v[R];
        const C *in = src.at(b) + j * src.ld;
#pragma unroll
        for (int r = 0; r < R; r++) v[r] = src.ok() ? in[r * istep] : cmake<C>(0, 0);
        int k = 0;
        if (ns > 1) {
            k = j - ((j * magic) >> 20) * ns;                 // j mod ns
            const int ks = k * stride;
#pragma unroll
            for (int r = 1; r < R; r++) {
                C w = __ldg(tw + r * ks);
                if (DIR > 0) w.y = -w.y;
                v[r] = cmul(v[r], w);
            }
        }
        adft<DIR, R>(v);
        C *out = dst.at(b) + ((j - k) * R + k) * dst.ld;
        if (dst.ok()) {
#pragma unroll
            for (int r = 0; r < R; r++) out[r * ostep] = v[r];
        }
    }
}
template <int DIR, typename C, class Dec, class Src, class Dst>
__device__ __forceinline__ void any_pass(const AnyPass &p, int total, const C *__restrict__ tw, Dec dec, Src src,
                                         Dst dst) {
    const int nthr = blockDim.x;
    switch (p.R) {
        case 16: any_pass_r<DIR, 16>(p, total, nthr, tw, dec, src, dst); break;
        case 15: any_pass_r<DIR, 15>(p, total, nthr, tw, dec, src, dst); break;
        case 12: any_pass_r<DIR, 12>(p, total, nthr, tw, dec, src, dst); break;
        case 10: any_pass_r<DIR, 10>(p, total, nthr, tw, dec, src, dst); break;
        case 9: any_pass_r<DIR, 9>(p, total, nthr, tw, dec, src, dst); break;
        case 8: any_pass_r<DIR, 8>(p, total, nthr, tw, dec, src, dst); break;
        case 6: any_pass_r<DIR, 6>(p, total, nthr, tw, dec, src, dst); break;
        case 5: any_pass_r<DIR, 5>(p, total, nthr, tw, dec, src, dst); break;
        case 4: any_pass_r<DIR, 4>(p, total, nthr, tw, dec, src, dst); break;
        case 3: any_pass_r<DIR, 3>(p, total, nthr, tw, dec, src, dst); break;
        default: any_pass_r<DIR, 2>(p, total, nthr, tw, dec, src, dst); break;
    }
}

// Plans known at compile time: radices R1 R2 R3 (R3 = 1: two passes).  The same pass code with
// every bound, stride and twiddle step folded to a constant.
constexpr AnyPass any_const_pass(int n, int R, int ns) {
    return AnyPass{R, ns, n / R, n / (ns * R), ((1 << 20) + ns - 1) / ns};
}

// arguments of a block: the launch's own (one evaluation) or entry gk of a batch's list
template <typename T>
__device__ __forceinline__ const EvalArgs<T> &any_args(const EvalArgs<T> &a, const EvalArgs<T> *ga, int bps, int &bid) {
    if (!ga) {
        bid = blockIdx.x;
        return a;
    }
    const int gk = blockIdx.x / bps;
    bid = blockIdx.x - gk * bps;
    return ga[gk];
}

// ---------------------------------------------------------------- pencils (C2C along n1)
// block size: a thread per butterfly of the pass with the fewest (at 256 for all lengths half the
// threads of short or unequal plans had none), 85 registers
constexpr int any_max3(int a, int b, int c) { return a > b ? (a > c ? a : c) : (b > c ? b : c); }
constexpr int any_ct_pencil_threads(int n, int rmax, int lg) {
    const int t = ((n / rmax << lg) + 31) / 32 * 32;
    return t < 64 ? 64 : (t > 256 ? 256 : t);
}
// One tile of 2^lg consecutive columns per block.  The first pass takes its inputs straight
// from global memory into registers and the last one stores straight from registers (a warp
// reads and writes whole rows of the tile), so an element crosses shared memory once per
// exchange and nothing else; many small blocks per SM keep the loads in flight.
// (R1 = 0: the launch's plan and tile width; else n1 = R1 R2 R3, R3 = 1 for two passes, and 2^LG columns)
template <typename T, int DIR, int R1 = 0, int R2 = 1, int R3 = 1, int LG = 0>
__device__ __forceinline__ void pencil_any_body(const EvalArgs<T> &a, const int bid) {
    typedef typename Vec2<T>::type C;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr bool CT = R1 > 0;
    constexpr int NC = CT ? R1 * R2 * R3 : 1;
    const AnyPlan &q = a.q1;
    const int n = CT ? NC : q.n, lg = CT ? LG : a.lg1, TW = 1 << lg, n2h = a.n2h, np = CT ? (R3 > 1 ? 3 : 2) : q.np;
    C *const X = (C *)smem_raw, *const Y = X + (np > 2 ? (n << lg) : 0);
    const int ncols = a.n0 * n2h;
    const int ntile = (ncols + TW - 1) >> lg;
    const int ci = bid / ntile;
    const int w = threadIdx.x & (TW - 1);
    const int c = ((bid - ci * ntile) << lg) + w;
    const bool ok = c < ncols;
    const int k0 = ok ? c / n2h : 0, k2 = ok ? c - k0 * n2h : 0;
    const int ch = DIR < 0 ? a.col_ch[ci] : a.col_inv_ch[ci];
    C *const g = a.chan + (size_t)ch * a.NH + (size_t)k0 * n * n2h + k2;
    const C *const tw = a.tw1;
    auto dec = [&](int idx, int &b, int &j) { b = w; j = idx >> lg; };
    const AnyGlobal<C> G{g, n2h, ok};
    const AnyShared<C> SX{X, TW}, SY{Y, TW};
    if constexpr (CT) {
        constexpr int NT = any_ct_pencil_threads(NC, any_max3(R1, R2, R3), LG);
        any_pass_r<DIR, R1>(any_const_pass(NC, R1, 1), NC / R1 << LG, NT, tw, dec, G, SX);
        __syncthreads();
        if constexpr (R3 > 1) {
            any_pass_r<DIR, R2>(any_const_pass(NC, R2, R1), NC / R2 << LG, NT, tw, dec, SX, SY);
            __syncthreads();
            any_pass_r<DIR, R3>(any_const_pass(NC, R3, R1 * R2), NC / R3 << LG, NT, tw, dec, SY, G);
        } else {
            any_pass_r<DIR, R2>(any_const_pass(NC, R2, R1), NC / R2 << LG, NT, tw, dec, SX, G);
        }
        return;
    }
    any_pass<DIR>(q.p[0], q.p[0].nb << lg, tw, dec, G, SX);
    __syncthreads();
    if (np > 2) {
        any_pass<DIR>(q.p[1], q.p[1].nb << lg, tw, dec, SX, SY);
        __syncthreads();
    }
    any_pass<DIR>(q.p[np - 1], q.p[np - 1].nb << lg, tw, dec, SY, G);
}
template <typename T, int DIR>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 3 : 2)
    pencil_any_kernel(const __grid_constant__ EvalArgs<T> a, const EvalArgs<T> *__restrict__ ga, int bps) {
    pdl_begin();
    int bid;
    const EvalArgs<T> &ar = any_args(a, ga, bps, bid);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int f = DIR > 0 ? ar.fin : 0;
    if (f && bid == 0) energies_block(ar, (double *)smem_raw);
    else pencil_any_body<T, DIR>(ar, bid - f);
}

template <typename T, int DIR, int R1, int R2, int R3, int LG>
__global__ void __launch_bounds__(any_ct_pencil_threads(R1 *R2 *R3, any_max3(R1, R2, R3), LG),
                                  768 / any_ct_pencil_threads(R1 *R2 *R3, any_max3(R1, R2, R3), LG))
    pencil_ct_kernel(const __grid_constant__ EvalArgs<T> a, const EvalArgs<T> *__restrict__ ga, int bps) {
    pdl_begin();
    int bid;
    const EvalArgs<T> &ar = any_args(a, ga, bps, bid);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int f = DIR > 0 ? ar.fin : 0;
    if (f && bid == 0) energies_block(ar, (double *)smem_raw);
    else pencil_any_body<T, DIR, R1, R2, R3, LG>(ar, bid - f);
}

// ---------------------------------------------------------------- reciprocal-space pass
// One tile of 2^lg columns (k1, k2) and all k0 per block.  Thread (t, w) owns the RL
// frequencies t + r m (m = n0 / RL) of column w: the forward transform's last pass, radix RL,
// ends there, the products are applied in registers, and the inverse starts with the same RL
// values (radices in reverse order), so the spectra themselves never touch shared memory.
// The next channel's tile arrives by cp.async while the current one is worked on; the last
// inverse pass stores straight to global memory.  rho^beta hat, the term-2 accumulator and
// |G| stay in registers for the whole tile.
//
// A grid of few tiles (32^3: 34 of 16 columns) leaves most SMs idle while one block takes the
// channels in turn, about 2 us each; there up to eight blocks share a tile's channels.
//
// R1 = 0: the plan and the tile width of the launch; R1 > 0: n0 = R1 R2 RL (R2 = 1: two passes)
// and 2^LG columns, fixed at compile time.
template <typename T, int RL, bool MGP, int R1 = 0, int R2 = 1, int LG = 0>
__device__ __forceinline__ void axis0_any_body(const EvalArgs<T> &a, const int bid) {
    constexpr bool CT = R1 > 0;
    constexpr int NC = CT ? R1 * R2 * RL : 1;
    typedef typename Vec2<T>::type C;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double sd[4 * 32];
    __shared__ T sk[OFDFT_MAX_KNOTS];
    __shared__ short order[kMaxChan + 2];
    __shared__ RecipOp ops[kMaxChan + 2];
    __shared__ int s_nload, s_nops;
    const AnyPlan &q = a.q0, &qi = a.q0i;
    const int n = CT ? NC : q.n, lg = CT ? LG : a.lg0, TW = 1 << lg, np = CT ? (R2 > 1 ? 3 : 2) : q.np;
    const int m = n / RL, n2h = a.n2h, nthr = CT ? ((NC / RL << LG) + 31) / 32 * 32 : blockDim.x;
    const int PL = a.n1 * n2h;
    C *const L0 = (C *)smem_raw, *const L1 = L0 + (n << lg), *const X = L1 + (n << lg);
    const C *const tw = a.tw0;
    const bool lwt = a.kernel == 0, exact = a.nlpot == 0, hp = a.terms & (8u | 16u), pp = a.terms & 16u;
    const bool nl = a.terms & 4u;
    const int w = threadIdx.x & (TW - 1), t = threadIdx.x >> lg;
    const bool act = t < m;                                  // (the block is rounded up to whole warps)
    const int S = a.ax0_split, tile = S > 1 ? bid / S : bid, sp = bid - tile * S;
    const int col = (tile << lg) + w;
    const bool ok = col < PL;
    // the channels in load order and the operations of the tile, as in the persistent kernel
    if (threadIdx.x == 0) {
        int nload = 0, no = 0;
        auto op = [&](int kind, int fwd, int store, int k) {
            ops[no].kind = (signed char)kind;
            ops[no].fwd = (signed char)fwd;
            ops[no].store = (short)store;
            ops[no].m = (short)k;
            no++;
            if (fwd) order[nload++] = (short)(kind == OP_RB ? CH_NL : store);
        };
        // (a tile shared by S blocks: the channels go round, every block transforms rho^beta for its
        // knots and leaves its part of term 2 in a slot of its own, summed by the inverse rows)
        int u = 0;
        auto mine = [&]() { return S == 1 || u++ % S == sp; };
        if (hp && mine()) op(OP_HPP, 1, CH_HPP, 0);
        if ((a.terms & 2u) && mine()) op(OP_VW, 1, CH_VW, 0);
        if (nl) {
            op(OP_RB, 1, -1, 0);
            if (!lwt) {
                op(OP_WT, 1, CH_KNOT0, 0);
                op(OP_RR, 0, CH_NL, 0);
            } else {
                for (int k = 0; k < a.M; k++)
                    if (mine()) op(exact ? OP_EX : OP_IP, exact ? 1 : 0, CH_KNOT0 + k, k);
                if (exact) op(OP_A, 0, S > 1 ? a.t2_slot + sp : CH_NL, 0);
            }
        }
        s_nload = nload;
        s_nops = no;
    }
    if (nl && lwt)
        for (int i = threadIdx.x; i < a.M; i += nthr) sk[i] = a.knots_t[i];
    __syncthreads();
    const int nload = s_nload, nops = s_nops;
    const C *const gcol = a.chan + (ok ? col : 0);
    auto prefetch = [&](C *dst, int ch) {
        const C *src = gcol + (size_t)ch * a.NH;
        const int step = nthr >> lg;
        for (int i = t; i < n; i += step) cp_async<sizeof(C)>(dst + (i << lg) + w, src + (size_t)i * PL, ok);
        cp_async_commit();
    };
    int issued = 0;
    C *cur = L1, *nxt = L0;
    if (nload > 0) prefetch(L0, order[0]);
    auto dec = [&](int idx, int &b, int &j) { b = w; j = idx >> lg; };
    auto sh = [&](C *S) { return AnyShared<C>{S, TW}; };
    C v[RL], Rr[RL], A[RL];
    T gn[RL];
    T cw;
    T gmin = (T)3.0e38;
    {
        const int k1 = ok ? col / n2h : 0, k2 = ok ? col - k1 * n2h : 0;
        const double m1 = (k1 <= a.n1 / 2) ? k1 : k1 - a.n1, m2 = k2;
        T cv[3];
#pragma unroll
        for (int d = 0; d < 3; d++) cv[d] = (T)(m1 * a.bvec[3 + d] + m2 * a.bvec[6 + d]);
        cw = (ok && act) ? ((k2 == 0 || (a.n2 % 2 == 0 && k2 == a.n2 / 2)) ? (T)1 : (T)2) : (T)0;
        const T bx = (T)a.bvec[0], by = (T)a.bvec[1], bz = (T)a.bvec[2];
#pragma unroll
        for (int r = 0; r < RL; r++) {
            const int k0 = t + r * m;
            const T m0 = (T)(k0 <= n / 2 ? k0 : k0 - n);
            const T gx = cv[0] + m0 * bx, gy = cv[1] + m0 * by, gz = cv[2] + m0 * bz;
            // (threads past the last frequency carry zeros: any |G| that keeps their kernel finite)
            gn[r] = g_state(act ? gx * gx + gy * gy + gz * gz : (T)1e6);
            gmin = gn[r] < gmin ? gn[r] : gmin;
        }
    }
#pragma unroll
    for (int r = 0; r < RL; r++) v[r] = Rr[r] = A[r] = cmake<C>((T)0, (T)0);
    const T invN = (T)(1.0 / (double)a.N);
    double eH = 0.0, eV = 0.0, eP = 0.0, eN = 0.0;
    for (int o = 0; o < nops; o++) {
        const RecipOp op = ops[o];
        const int kind = op.kind;
        // (the last pass of the previous operation may still read its exchange tile)
        if (op.fwd) cp_async_wait<0>();
        __syncthreads();
        if (op.fwd) {
            // the next channel's tile becomes `cur`, the one after it starts to load
            C *x = cur;
            cur = nxt;
            nxt = x;
            issued++;
            if (issued < nload) prefetch(nxt, order[issued]);
            // forward transform; v[r] ends at frequency t + r m
            if constexpr (CT)
                any_pass_r<-1, R1>(any_const_pass(NC, R1, 1), NC / R1 << LG, nthr, tw, dec, sh(cur), sh(X));
            else any_pass<-1>(q.p[0], q.p[0].nb << lg, tw, dec, sh(cur), sh(X));
            __syncthreads();
            C *S = X;
            if (np > 2) {
                if constexpr (CT && R2 > 1)
                    any_pass_r<-1, R2>(any_const_pass(NC, R2, R1), NC / R2 << LG, nthr, tw, dec, sh(X), sh(cur));
                else if constexpr (!CT) any_pass<-1>(q.p[1], q.p[1].nb << lg, tw, dec, sh(X), sh(cur));
                __syncthreads();
                S = cur;
            }
            if (act) {
#pragma unroll
                for (int r = 0; r < RL; r++) v[r] = S[(t << lg) + w + r * (m << lg)];
#pragma unroll
                for (int r = 1; r < RL; r++) v[r] = cmul(v[r], __ldg(tw + r * t));
                adft<-1, RL>(v);
            }
        }
        if (kind == OP_WT || kind == OP_EX || kind == OP_IP) {
            // the kernel of this knot (WT: of the mean density's kF) at the thread's |G|
            const T hk = kind == OP_WT ? (T)(0.5 / a.scal[S_KF_WT]) : (T)0.5 / sk[op.m];
            const T ihk2 = (T)1 / (hk * hk);
            Part<T, false> fN;
            auto knot = [&](auto large) {
#pragma unroll
                for (int r = 0; r < RL; r++) {
                    T K;
                    if constexpr (decltype(large)::value) K = kernel_value_large(gn[r] * hk);
                    else K = kernel_of_state<T, MGP>(a, gn[r], hk, ihk2);
                    if (kind == OP_EX) {
                        // E_NL += Omega sum_G w Re(conj(FFT[h_k rho^alpha]) K_k FFT[rho^beta])
                        const C Sm = cscale(v[r], invN);
                        fN.add(cw * K * (Sm.x * Rr[r].x + Sm.y * Rr[r].y));
                        A[r] = cadd(A[r], cscale(Sm, K));
                        v[r] = cscale(Rr[r], K);
                    } else if (kind == OP_IP) {
                        v[r] = cscale(Rr[r], K);
                    } else {
                        const C Sa = cscale(v[r], invN);
                        fN.add(cw * K * (Sa.x * Rr[r].x + Sa.y * Rr[r].y));
                        Rr[r] = cscale(Rr[r], K);
                        v[r] = cscale(Sa, K);
                    }
                }
            };
            if (warp_all_large<T, MGP>(gmin, hk)) knot(std::true_type{});
            else knot(std::false_type{});
            eN += fN.value();
        } else if (kind == OP_HPP) {
            Part<T, false> fH, fP;
#pragma unroll
            for (int r = 0; r < RL; r++) {
                const C X0 = cscale(v[r], invN);
                const T g2 = g2_of(gn[r]);
                const size_t e = (size_t)(t + r * m) * PL + col;
                if (a.rhohat_out && ok && act) a.rhohat_out[e] = X0;
                C out = cmake<C>((T)0, (T)0), vx = out;
                if (pp && ok && act) vx = a.vext[e];
                if (g2 > (T)0) {
                    if (a.terms & 8u) {
                        const T f = (T)1 / g2;
                        fH.add(cw * (X0.x * X0.x + X0.y * X0.y) * f);
                        out = cscale(X0, (T)(4.0 * kPi) * f);
                    }
                    if (pp) {
                        fP.add(cw * (X0.x * vx.x + X0.y * vx.y));
                        out = cadd(out, vx);
                    }
                } else if (pp) {
                    out = vx;                                     // G = 0: V_ext(0) only
                }
                v[r] = out;
            }
            eH += fH.value();
            eP += fP.value();
        } else if (kind == OP_VW) {
            Part<T, false> fV;
#pragma unroll
            for (int r = 0; r < RL; r++) {
                const C X0 = cscale(v[r], invN);
                const T g2 = g2_of(gn[r]);
                fV.add(cw * g2 * (X0.x * X0.x + X0.y * X0.y));
                v[r] = cscale(X0, g2);
            }
            eV += fV.value();
        } else if (kind == OP_RB) {
#pragma unroll
            for (int r = 0; r < RL; r++) Rr[r] = cscale(v[r], invN);
        } else {
#pragma unroll
            for (int r = 0; r < RL; r++) v[r] = kind == OP_RR ? Rr[r] : A[r];
        }
        if (op.store < 0) continue;
        // inverse transform, stored into the channel.  The exchange goes through the buffer that
        // no pass still reads (cur after a two-pass forward transform, X after three).
        C *D = np > 2 ? X : cur;
        if (act) {
            adft<+1, RL>(v);
#pragma unroll
            for (int r = 0; r < RL; r++) D[((t * RL) << lg) + w + (r << lg)] = v[r];
        }
        __syncthreads();
        C *S = D;
        if (np > 2) {
            if constexpr (CT && R2 > 1)
                any_pass_r<+1, R2>(any_const_pass(NC, R2, RL), NC / R2 << LG, nthr, tw, dec, sh(D), sh(cur));
            else if constexpr (!CT) any_pass<+1>(qi.p[1], qi.p[1].nb << lg, tw, dec, sh(D), sh(cur));
            __syncthreads();
            S = cur;
        }
        C *dst = a.chan + (size_t)op.store * a.NH + (ok ? col : 0);
        const AnyGlobal<C> G{dst, PL, ok};
        if constexpr (CT)
            any_pass_r<+1, R1>(any_const_pass(NC, R1, R2 * RL), NC / R1 << LG, nthr, tw, dec, sh(S), G);
        else any_pass<+1>(qi.p[np - 1], qi.p[np - 1].nb << lg, tw, dec, sh(S), G);
    }
    double r4[4] = {eH, eV, eP, eN};
    // (a tile shared by several blocks: the block's sum in FP64, its few blocks hide the slow adds; the terms of
    // a thread's RL frequencies are added in FP32 in either case)
    if (sizeof(T) == 4 && S == 1) block_sum_n_f32warp<4>(r4, sd);
    else block_sum_n<4>(r4, sd);
    if (threadIdx.x == 0)
        for (int k = 0; k < 4; k++) a.part_ax0[4 * bid + k] = r4[k];
}
// RL = 12 and more live in up to 255 registers at one block of 256 threads; the smaller ones
// leave room for 512 threads
template <typename T, int RL> constexpr int any_ax0_threads() {
    return sizeof(T) == 4 ? (RL >= 12 ? 256 : 512) : 256;
}
template <typename T, int RL, bool MGP>
__global__ void __launch_bounds__(any_ax0_threads<T, RL>(), 1)
    axis0_any_kernel(const __grid_constant__ EvalArgs<T> a, const EvalArgs<T> *__restrict__ ga, int bps) {
    int bid;
    const EvalArgs<T> &ar = any_args(a, ga, bps, bid);
    axis0_any_body<T, RL, MGP>(ar, bid);
}

// compile-time lengths: as many blocks per SM as 128 registers a thread allow, 168 from RL = 12 on
// (the spectra, the kernel state and term 2 of 12 to 15 frequencies fit without spills) and 255 at 16
constexpr int any_ct_threads(int N, int RL, int lg) { return ((N / RL << lg) + 31) / 32 * 32; }
constexpr int any_ct_blocks(int N, int RL, int lg) {
    const int b = (RL >= 16 ? 256 : (RL >= 12 ? 384 : 512)) / any_ct_threads(N, RL, lg);
    return b > 1 ? b : 1;
}
// Columns per tile (log2) of the compiled pass.  RL >= 12: 8 columns, so that two or three blocks
// of 128 threads share an SM and cover one another's barriers (with 16 columns one block of 8 warps
// issued in 29 % of the cycles; whole evaluations at 180^3 / 192^3 / 240^3 / 256^3: 1.356 / 2.014 /
// 3.167 / 3.606 -> 1.245 / 1.903 / 2.969 / 3.534 ms).  Smaller RL keep the list's width, and from 72
// points on the tuner may take 8 columns where that fills the last wave of blocks better (108^3:
// 0.340 -> 0.299 ms, 100^3: 0.260 -> 0.257, 144^3: 0.689 -> 0.673; 96^3 and 160^3 keep 16).
constexpr int any_ct_lg(int RL, int W) { return RL >= 12 ? 3 : W; }
constexpr bool any_ct_narrow(int N, int RL, int W) { return N >= 72 && RL < 12 && W == 4; }
template <typename T, int R1, int R2, int RL, int LG, bool MGP>
__global__ void __launch_bounds__(any_ct_threads(R1 *R2 *RL, RL, LG), any_ct_blocks(R1 *R2 *RL, RL, LG))
    axis0_ct_kernel(const __grid_constant__ EvalArgs<T> a, const EvalArgs<T> *__restrict__ ga, int bps) {
    int bid;
    const EvalArgs<T> &ar = any_args(a, ga, bps, bid);
    axis0_any_body<T, RL, MGP, R1, R2, LG>(ar, bid);
}

// the compiled pass of n0 = R1 R2 RL at its default width, or (narrow) at 8 columns
template <int R1, int R2, int RL, int W> bool any_ct_axis0_pick(bool narrow, AnyCt &c) {
    constexpr int N = R1 * R2 * RL;
    auto put = [&](auto lg) {
        constexpr int LG = decltype(lg)::value;
        c.k = (const void *)axis0_ct_kernel<float, R1, R2, RL, LG, false>;
        c.k2 = (const void *)axis0_ct_kernel<float, R1, R2, RL, LG, true>;
        c.RL = RL;
        c.lg = LG;
        c.nt = any_ct_threads(N, RL, LG);
        return true;
    };
    if (!narrow) return put(std::integral_constant<int, any_ct_lg(RL, W)>{});
    if constexpr (any_ct_narrow(N, RL, W)) return put(std::integral_constant<int, 3>{});
    return false;
}

// ---------------------------------------------------------------- rows
// Policy of the channel-batched row bodies (kernels.cuh) for any n2: E elements per thread,
// the channel group and the transform's passes read at run time.
template <typename T, int E__, bool INV, int R1 = 0, int R2 = 1, int R3 = 1> struct RowAny {
    static constexpr int NC = R1 * R2 * R3;               // 0: the length of the launch
    typedef typename Vec2<T>::type C;
    static constexpr bool ct = false;
    static constexpr int E = E__, NT_ = E__ == 4 ? 256 : 320;
    __device__ static int n(const EvalArgs<T> &a) { return NC ? NC : a.n2; }
    __device__ static int Gn(const EvalArgs<T> &a) { return a.any_G[INV]; }
    __device__ static int Ld(const EvalArgs<T> &a) { return a.any_G[INV] | 1; }
    __device__ static int Nt() { return blockDim.x; }
    __device__ static int Scr(const EvalArgs<T> &a) {
        const int x = n(a) * Ld(a), y = Gn(a) * (n(a) + 2);
        return x > y ? x : y;
    }
    __device__ static int slot(const EvalArgs<T> &a, int idx) {
        return NC ? idx / (NC / 2 + 1) : (int)__umulhi((unsigned)idx, a.magic_n2h);
    }
    __device__ static int slot2(const EvalArgs<T> &a, int idx) { return (int)__umulhi((unsigned)idx, a.magic_2n2h); }
    template <int DIR> __device__ static C *fft(C *x, C *y, const EvalArgs<T> &a, const C *) {
        const AnyPlan &q = a.q2;
        const C *const tw = a.tw2;
        const int G = Gn(a), ld = Ld(a);
        const unsigned mg = a.magic_G[INV];
        auto dec = [&](int idx, int &b, int &j) {
            j = G > 1 ? (int)__umulhi((unsigned)idx, mg) : idx;
            b = idx - j * G;
        };
        if constexpr (NC > 0) {
            const int nt = blockDim.x;
            const AnyShared<C> X{x, ld}, Y{y, ld};
            any_pass_r<DIR, R1>(any_const_pass(NC, R1, 1), NC / R1 * G, nt, tw, dec, X, Y);
            __syncthreads();
            any_pass_r<DIR, R2>(any_const_pass(NC, R2, R1), NC / R2 * G, nt, tw, dec, Y, X);
            __syncthreads();
            if constexpr (R3 > 1) {
                any_pass_r<DIR, R3>(any_const_pass(NC, R3, R1 * R2), NC / R3 * G, nt, tw, dec, X, Y);
                __syncthreads();
                return y;
            }
            return x;
        } else {
            for (int s = 0; s < q.np; s++) {
                any_pass<DIR>(q.p[s], q.p[s].nb * G, tw, dec, AnyShared<C>{x, ld}, AnyShared<C>{y, ld});
                __syncthreads();
                C *z = x;
                x = y;
                y = z;
            }
            return x;
        }
    }
};
// Elements per thread, largest block and blocks per SM of the compiled rows for length n.  Up to 200
// points one element per thread and 80 registers, so that three to five blocks overlap one another's
// loads, barriers and stores (inverse rows of 18 channels at n2 = 108: 117 us with 320 threads and 96
// registers, 70 us with 160 and 72).  Longer rows keep two elements per thread, which spares the idle
// threads of small channel groups (256^3, forward / inverse: 613 / 870 us against 648 / 900 us).
constexpr int any_ct_E(int n) { return n <= 200 ? 1 : 2; }
// Beyond 256 points a block has one thread per two points and at least six warps, and 24 warps (21 from 385
// to 448 points, three blocks of 7) share an SM at 80 registers (320 threads at two blocks per SM: whole
// evaluations of 256 x 256 x 320 and 256 x 256 x 512 5.00 and 7.77 ms, now 4.60 and 7.22; 512^3 with 15
// channels 28.99 -> 27.70 ms); 129 to 160 points take 192 threads, so that all channels of an ordinary call
// go in one group (144^3: 0.690 -> 0.670 ms).
constexpr int any_ct_row_threads(int n) {
    return n <= 128 ? 160 : (n <= 160 ? 192 : (n <= 200 ? 256 : (n <= 256 ? 320 : (n <= 384 ? 192 : ((n + 63) / 64 * 32)))));
}
constexpr int any_ct_row_blocks(int n) {
    return n <= 128 ? 5 : (n <= 160 ? 4 : (n <= 200 ? 3 : (n <= 256 ? 2 : 768 / any_ct_row_threads(n))));
}
template <typename T, int E>
__global__ void __launch_bounds__(RowAny<T, E, false>::NT_, sizeof(T) == 4 ? 2 : 1)
    row_fwd_any_kernel(const __grid_constant__ EvalArgs<T> a, const EvalArgs<T> *__restrict__ ga, int bps) {
    int bid;
    const EvalArgs<T> &ar = any_args(a, ga, bps, bid);
    row_fwd2_body<T, RowAny<T, E, false>>(ar, bid, 0);
}
template <typename T, int E>
__global__ void __launch_bounds__(RowAny<T, E, true>::NT_, sizeof(T) == 4 ? 2 : 1)
    row_inv_any_kernel(const __grid_constant__ EvalArgs<T> a, const EvalArgs<T> *__restrict__ ga, int bps) {
    int bid;
    const EvalArgs<T> &ar = any_args(a, ga, bps, bid);
    row_inv2_body<T, RowAny<T, E, true>>(ar, bid, 0);
}

template <typename T, int R1, int R2, int R3>
__global__ void __launch_bounds__(any_ct_row_threads(R1 *R2 *R3), any_ct_row_blocks(R1 *R2 *R3))
    row_fwd_ct_kernel(const __grid_constant__ EvalArgs<T> a, const EvalArgs<T> *__restrict__ ga, int bps) {
    int bid;
    const EvalArgs<T> &ar = any_args(a, ga, bps, bid);
    row_fwd2_body<T, RowAny<T, any_ct_E(R1 *R2 *R3), false, R1, R2, R3>>(ar, bid, 0);
}
template <typename T, int R1, int R2, int R3>
__global__ void __launch_bounds__(any_ct_row_threads(R1 *R2 *R3), any_ct_row_blocks(R1 *R2 *R3))
    row_inv_ct_kernel(const __grid_constant__ EvalArgs<T> a, const EvalArgs<T> *__restrict__ ga, int bps) {
    int bid;
    const EvalArgs<T> &ar = any_args(a, ga, bps, bid);
    row_inv2_body<T, RowAny<T, any_ct_E(R1 *R2 *R3), true, R1, R2, R3>>(ar, bid, 0);
}

}  // namespace ofdft
