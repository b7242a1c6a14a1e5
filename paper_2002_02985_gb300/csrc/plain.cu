// Plain one-field transforms for any length (any.cuh): the optimiser's preconditioner, TD-OFDFT's
// Hamiltonian, forces, PME and interpolation transform a single real field at a time.
//
// A filter out = IFFT(f(G) FFT(u)) is five launches: the rows (R2C), the n1 pencils, the n0 pass
// (forward, factor and inverse in one launch, the column never leaving shared memory), the n1
// pencils back, and the rows back with the caller's pointwise epilogue fused into their stores.
// (the chain it replaces -- stats, per-channel rows, n0 transform, factor kernel, n0 transform,
// rows, potential kernel -- took 133 us at 128^3, most of it in launches of 8 to 35 us that move
// 17 MB each)
// One field's launches fill less than a wave (512 blocks at 128^3, and four to eight fit an SM), so
// two fields that take the same filter share each launch (blockIdx.y is the field).
#include "any.cuh"
#include "plain.cuh"
#include "sample.cuh"

namespace ofdft {

// 128 threads: a block's 16 transforms of 128 points are 128 radix-16 butterflies
constexpr int kPlainThreads = 128;

// ---------------------------------------------------------------- mean
// scal[S_RHO_MEAN] = sum of u / N (FP32: runs of 16 summed in FP32, the runs in FP64)
template <typename T>
__global__ void __launch_bounds__(256) plain_mean_kernel(const T *u, long long N, double *part, double *scal,
                                                         unsigned *ticket) {
    pdl_begin();
    __shared__ double sd[32];
    __shared__ bool last;
    double acc = 0.0;
    const long long stride = (long long)gridDim.x * 256;
    long long i = blockIdx.x * 256LL + threadIdx.x;
    while (i < N) {
        T s = 0;
#pragma unroll
        for (int k = 0; k < 16; k++, i += stride) {
            if (sizeof(T) == 8) acc += i < N ? (double)u[i] : 0.0;
            else s += i < N ? u[i] : (T)0;
        }
        if (sizeof(T) == 4) acc += (double)s;
    }
    acc = block_sum(acc, sd);
    if (threadIdx.x == 0) {
        part[blockIdx.x] = acc;
        __threadfence();
        last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    acc = 0.0;
    for (int b = threadIdx.x; b < (int)gridDim.x; b += 256) acc += __ldcg(part + b);
    acc = block_sum(acc, sd);
    if (threadIdx.x == 0) {
        scal[S_SUM_RHO] = acc;
        scal[S_RHO_MEAN] = acc / (double)N;
        *ticket = 0u;
    }
}

// ---------------------------------------------------------------- rows
__device__ __forceinline__ void store4(float *p, const float v[4]) {
    *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void store4(double *p, const double v[4]) {
    reinterpret_cast<double2 *>(p)[0] = make_double2(v[0], v[1]);
    reinterpret_cast<double2 *>(p)[1] = make_double2(v[2], v[3]);
}
// 2^lgB pairs of rows per block, a pair packed as z = x_2p + i x_2p+1 (element e of pair b at
// buf[e (2^lgB + 1) + b]: the odd stride keeps both the transposing copies and the passes free of
// bank conflicts)
template <typename T> __device__ __forceinline__ typename Vec2<T>::type *plain_passes(const PlainArgs<T> &a, int dir,
                                                                                      typename Vec2<T>::type *x,
                                                                                      typename Vec2<T>::type *y) {
    typedef typename Vec2<T>::type C;
    const int lg = a.lgB, ld = (1 << lg) + 1;
    auto dec = [&](int idx, int &b, int &j) {
        b = idx & ((1 << lg) - 1);
        j = idx >> lg;
    };
    for (int s = 0; s < a.q2.np; s++) {
        const AnyShared<C> X{x, ld}, Y{y, ld};
        if (dir < 0) any_pass<-1>(a.q2.p[s], a.q2.p[s].nb << lg, a.tw2, dec, X, Y);
        else any_pass<+1>(a.q2.p[s], a.q2.p[s].nb << lg, a.tw2, dec, X, Y);
        __syncthreads();
        C *z = x;
        x = y;
        y = z;
    }
    return x;
}

// What the rows subtract before the transform.  A transform alone takes the mean.  A filter only
// needs a constant near it, so that the FP32 passes do not carry a large G = 0 term: the mean of
// the field at 1024 points spread evenly over the cell (sample.cuh: within a tenth of the mean for
// a density localised in the cell), which every block takes for itself (the same loads in the
// same order, so the same value) instead of waiting for a pass over the whole field; block 0
// leaves it for the inverse rows.
template <typename T> __device__ __forceinline__ T plain_offset(const PlainArgs<T> &a) {
    const int f = blockIdx.y;
    if (!a.sampled) return (T)a.scal[S_RHO_MEAN];
    const T *const u = a.u[f];
    __shared__ T ws[kPlainThreads / 32];
    T s = 0;
#pragma unroll
    for (int k = 0; k < kPlainSamples / kPlainThreads; k++)
        s += u[plain_sample((int)threadIdx.x + k * kPlainThreads, a.n0, a.n1, a.n2)];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = s;
    __syncthreads();
    s = 0;
#pragma unroll
    for (int k = 0; k < kPlainThreads / 32; k++) s += ws[k];
    s *= (T)(1.0 / kPlainSamples);
    if (blockIdx.x == 0 && threadIdx.x == 0) const_cast<double *>(a.scal)[f ? S_PAIR_MEAN : S_RHO_MEAN] = (double)s;
    return s;
}
template <typename T> __global__ void __launch_bounds__(kPlainThreads, 4) plain_rows_fwd(const __grid_constant__ PlainArgs<T> a) {
    pdl_begin();
    typedef typename Vec2<T>::type C;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int n = a.n2, n2h = a.n2h, lg = a.lgB, ld = (1 << lg) + 1;
    C *const buf = (C *)smem_raw, *const scr = buf + n * ld;
    const int R = a.n0 * a.n1, row0 = blockIdx.x << (lg + 1);
    const T mean = plain_offset(a);
    const T *const u = a.u[blockIdx.y];
    C *const h = a.h + blockIdx.y * a.hs;
    if (a.vec) {
        // four consecutive points of a row per thread and step, several steps in flight
        const int n4 = n >> 2;
#pragma unroll 4
        for (int idx = threadIdx.x; idx < (n4 << (lg + 1)); idx += kPlainThreads) {
            const int rr = (int)__umulhi((unsigned)idx, a.magic_n4), e = 4 * (idx - rr * n4);
            T x[4] = {mean, mean, mean, mean};
            if (row0 + rr < R) load4(u + (size_t)(row0 + rr) * n + e, x);
#pragma unroll
            for (int q = 0; q < 4; q++) ((T *)(buf + (e + q) * ld + (rr >> 1)))[rr & 1] = x[q] - mean;
        }
    } else {
        for (int idx = threadIdx.x; idx < (n << (lg + 1)); idx += kPlainThreads) {
            const int rr = (int)__umulhi((unsigned)idx, a.magic_n), e = idx - rr * n;
            const T x = row0 + rr < R ? u[(size_t)(row0 + rr) * n + e] - mean : (T)0;
            ((T *)(buf + e * ld + (rr >> 1)))[rr & 1] = x;
        }
    }
    __syncthreads();
    const C *Z = plain_passes<T>(a, -1, buf, scr);
    for (int idx = threadIdx.x; idx < n2h << lg; idx += kPlainThreads) {
        const int b = (int)__umulhi((unsigned)idx, a.magic_n2h), k = idx - b * n2h;
        const C A = Z[k * ld + b], Bv = Z[(k ? n - k : 0) * ld + b];
        const int r0 = row0 + 2 * b;
        C *out = h + (size_t)r0 * n2h + k;
        if (r0 < R) out[0] = cmake<C>((T)0.5 * (A.x + Bv.x), (T)0.5 * (A.y - Bv.y));
        if (r0 + 1 < R) out[n2h] = cmake<C>((T)0.5 * (A.y + Bv.y), (T)0.5 * (Bv.x - A.x));
    }
}

// out = c0 base + c1 (y + madd mean + v u), y the inverse transform (null pointers: left out); out
// overlaps none of the inputs
template <typename T> __global__ void __launch_bounds__(kPlainThreads, 4) plain_rows_inv(const __grid_constant__ PlainArgs<T> a) {
    pdl_begin();
    typedef typename Vec2<T>::type C;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int n = a.n2, n2h = a.n2h, lg = a.lgB, ld = (1 << lg) + 1;
    C *const buf = (C *)smem_raw, *const scr = buf + n * ld;
    const int R = a.n0 * a.n1, row0 = blockIdx.x << (lg + 1), f = blockIdx.y;
    const C *const h = a.h + f * a.hs;
#pragma unroll 4
    for (int idx = threadIdx.x; idx < n2h << lg; idx += kPlainThreads) {
        const int b = (int)__umulhi((unsigned)idx, a.magic_n2h), k = idx - b * n2h;
        const int r0 = row0 + 2 * b;
        const C zero = cmake<C>((T)0, (T)0);
        const C *in = h + (size_t)r0 * n2h + k;
        const C X0 = r0 < R ? in[0] : zero, X1 = r0 + 1 < R ? in[n2h] : zero;
        if (k == 0 || 2 * k == n) {
            buf[k * ld + b] = cmake<C>(X0.x, X1.x);
        } else {
            buf[k * ld + b] = cmake<C>(X0.x - X1.y, X0.y + X1.x);
            buf[(n - k) * ld + b] = cmake<C>(X0.x + X1.y, X1.x - X0.y);
        }
    }
    __syncthreads();
    const C *Z = plain_passes<T>(a, +1, buf, scr);
    const T shift = a.madd != (T)0 ? a.madd * (T)a.scal[f ? S_PAIR_MEAN : S_RHO_MEAN] : (T)0;
    if (a.vec) {
        const int n4 = n >> 2;
        const T *const __restrict__ pv = a.v, *const __restrict__ pu = a.vu[f], *const __restrict__ pb = a.base[f];
        T *const __restrict__ po = a.out[f];
#pragma unroll 4
        for (int idx = threadIdx.x; idx < (n4 << (lg + 1)); idx += kPlainThreads) {
            const int rr = (int)__umulhi((unsigned)idx, a.magic_n4), e = 4 * (idx - rr * n4);
            if (row0 + rr < R) {
                const size_t i = (size_t)(row0 + rr) * n + e;
                T v[4] = {0, 0, 0, 0}, u[4] = {0, 0, 0, 0}, b[4] = {0, 0, 0, 0};
                if (pv) {
                    load4(pv + i, v);
                    load4(pu + i, u);
                }
                if (pb) load4(pb + i, b);
#pragma unroll
                for (int q = 0; q < 4; q++) {
                    const T y = ((const T *)(Z + (e + q) * ld + (rr >> 1)))[rr & 1] + shift + v[q] * u[q];
                    v[q] = pb ? a.c0 * b[q] + a.c1 * y : a.c1 * y;
                }
                store4(po + i, v);
            }
        }
        return;
    }
    for (int idx = threadIdx.x; idx < (n << (lg + 1)); idx += kPlainThreads) {
        const int rr = (int)__umulhi((unsigned)idx, a.magic_n), e = idx - rr * n;
        if (row0 + rr >= R) break;
        const size_t i = (size_t)(row0 + rr) * n + e;
        T y = ((const T *)(Z + e * ld + (rr >> 1)))[rr & 1] + shift;
        if (a.v) y += a.v[i] * a.vu[f][i];
        a.out[f][i] = a.base[f] ? a.c0 * a.base[f][i] + a.c1 * y : a.c1 * y;
    }
}

// ---------------------------------------------------------------- n0
template <typename T> __device__ __forceinline__ T plain_factor(const PlainArgs<T> &a, T g2) {
    if (a.mode == PLAIN_KINETIC) return (T)0.5 * g2;
    if (a.mode == PLAIN_CN) {
        const T x = a.p1 * ((T)0.5 * g2 + a.p2);
        return (T)1 / ((T)1 + x * x);
    }
    return g2 > (T)0 ? a.p1 * g2 / (g2 * g2 + a.p1 * g2 + a.p2) : (T)1;       // PLAIN_PRECOND
}
template <typename T> __global__ void __launch_bounds__(kPlainThreads, 4) plain_n0(const __grid_constant__ PlainArgs<T> a) {
    pdl_begin();
    typedef typename Vec2<T>::type C;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const AnyPlan &q = a.q0;
    const int n = q.n, lg = a.lg0, TW = 1 << lg, np = q.np, n2h = a.n2h, PL = a.n1 * n2h;
    C *X = (C *)smem_raw, *Y = X + (n << lg);
    const int w = threadIdx.x & (TW - 1), col = (blockIdx.x << lg) + w;
    const bool ok = col < PL;
    const AnyGlobal<C> G{a.h + blockIdx.y * a.hs + (ok ? col : 0), PL, ok};
    auto dec = [&](int idx, int &b, int &j) {
        b = w;
        j = idx >> lg;
    };
    auto sh = [&](C *S) { return AnyShared<C>{S, TW}; };
    auto swap = [&]() {
        C *z = X;
        X = Y;
        Y = z;
    };
    if (a.mode != PLAIN_INVERSE) {
        any_pass<-1>(q.p[0], q.p[0].nb << lg, a.tw0, dec, G, sh(X));
        __syncthreads();
        for (int s = 1; s < np; s++) {
            any_pass<-1>(q.p[s], q.p[s].nb << lg, a.tw0, dec, sh(X), sh(Y));
            __syncthreads();
            swap();
        }
        const int step = kPlainThreads >> lg;
        if (a.mode == PLAIN_FORWARD) {
            if (ok)
                for (int i = threadIdx.x >> lg; i < n; i += step) G.g[(size_t)i * PL] = cscale(X[(i << lg) + w], a.scale);
            return;
        }
        const int k1 = ok ? col / n2h : 0, k2 = ok ? col - k1 * n2h : 0;
        const T m1 = (T)(k1 <= a.n1 / 2 ? k1 : k1 - a.n1), m2 = (T)k2;
        const T cx = m1 * a.b[3] + m2 * a.b[6], cy = m1 * a.b[4] + m2 * a.b[7], cz = m1 * a.b[5] + m2 * a.b[8];
        for (int i = threadIdx.x >> lg; i < n; i += step) {
            const T m0 = (T)(i <= n / 2 ? i : i - n);
            const T gx = m0 * a.b[0] + cx, gy = m0 * a.b[1] + cy, gz = m0 * a.b[2] + cz;
            C *x = X + (i << lg) + w;
            *x = cscale(*x, a.scale * plain_factor(a, gx * gx + gy * gy + gz * gz));
        }
        __syncthreads();
        for (int s = 0; s + 1 < np; s++) {
            any_pass<+1>(q.p[s], q.p[s].nb << lg, a.tw0, dec, sh(X), sh(Y));
            __syncthreads();
            swap();
        }
    } else {
        any_pass<+1>(q.p[0], q.p[0].nb << lg, a.tw0, dec, G, sh(X));
        __syncthreads();
        for (int s = 1; s + 1 < np; s++) {
            any_pass<+1>(q.p[s], q.p[s].nb << lg, a.tw0, dec, sh(X), sh(Y));
            __syncthreads();
            swap();
        }
    }
    any_pass<+1>(q.p[np - 1], q.p[np - 1].nb << lg, a.tw0, dec, sh(X), G);
}

// ---------------------------------------------------------------- launches
// (for every grid: the attribute belongs to the device that is current)
template <typename T> static cudaError_t prepare_plain() {
    cudaError_t r = allow_max_dynamic_smem(plain_rows_fwd<T>);
    if (r == cudaSuccess) r = allow_max_dynamic_smem(plain_rows_inv<T>);
    if (r == cudaSuccess) r = allow_max_dynamic_smem(plain_n0<T>);
    return r;
}

template <typename T> bool plain_setup(PlainArgs<T> &a, int nsm) {
    a.q0 = any_plan(a.n0);
    a.q2 = any_plan(a.n2);
    if (a.q0.np < 2 || a.q2.np < 1) return false;
    const size_t cb = 2 * sizeof(T);
    // rows: up to 16 pairs per block in at most 72 KB, fewer while the grid has no two blocks per SM
    const long long R = (long long)a.n0 * a.n1;
    for (a.lgB = 4; a.lgB > 1; a.lgB--)
        if (2 * cb * a.n2 * ((1 << a.lgB) + 1) <= 72 * 1024 && (R >> (a.lgB + 1)) >= 2 * nsm) break;
    if (2 * cb * a.n2 * ((1 << a.lgB) + 1) > 200 * 1024) return false;
    // n0: 16 columns in at most 72 KB, fewer while the grid has no tile per SM
    const long long PL = (long long)a.n1 * a.n2h;
    for (a.lg0 = 4; a.lg0 > 2; a.lg0--)
        if (2 * cb * ((size_t)a.n0 << a.lg0) <= 72 * 1024 && (PL >> a.lg0) >= nsm) break;
    if (2 * cb * ((size_t)a.n0 << a.lg0) > 200 * 1024) return false;
    a.magic_n = (unsigned)(((1ull << 32) + a.n2 - 1) / a.n2);
    a.magic_n4 = a.n2 >= 8 ? (unsigned)(((1ull << 32) + a.n2 / 4 - 1) / (a.n2 / 4)) : 0;
    a.magic_n2h = (unsigned)(((1ull << 32) + a.n2h - 1) / a.n2h);
    return prepare_plain<T>() == cudaSuccess;
}
template <typename T>
cudaError_t launch_plain_mean(const T *u, long long N, int nblk, double *part, double *scal, unsigned *ticket,
                              cudaStream_t s) {
    void *args[] = {(void *)&u, (void *)&N, (void *)&part, (void *)&scal, (void *)&ticket};
    return launch_pdl((const void *)plain_mean_kernel<T>, (unsigned)nblk, 256, args, 0, s);
}
template <typename T> cudaError_t launch_plain_rows(const PlainArgs<T> &a_in, bool inverse, cudaStream_t s) {
    // 16-byte (FP32) accesses where every row of every field starts on such a boundary
    PlainArgs<T> a = a_in;
    uintptr_t at = (uintptr_t)a.v;
    for (int f = 0; f < 2; f++)
        at |= (uintptr_t)a.u[f] | (uintptr_t)a.out[f] | (uintptr_t)a.vu[f] | (uintptr_t)a.base[f];
    a.vec = a.n2 % 4 == 0 && a.n2 >= 8 && at % 16 == 0;
    const long long R = (long long)a.n0 * a.n1;
    const unsigned nb = (unsigned)((R + (2 << a.lgB) - 1) >> (a.lgB + 1));
    const size_t sm = 2 * 2 * sizeof(T) * (size_t)a.n2 * ((1 << a.lgB) + 1);
    void *args[] = {(void *)&a};
    return launch_pdl(inverse ? (const void *)plain_rows_inv<T> : (const void *)plain_rows_fwd<T>,
                      dim3(nb, a.nf > 1 ? 2 : 1), kPlainThreads, args,
                      sm, s);
}
template <typename T> cudaError_t launch_plain_n0(const PlainArgs<T> &a, cudaStream_t s) {
    const long long PL = (long long)a.n1 * a.n2h;
    const unsigned nb = (unsigned)((PL + (1 << a.lg0) - 1) >> a.lg0);
    void *args[] = {(void *)&a};
    return launch_pdl((const void *)plain_n0<T>, dim3(nb, a.nf > 1 ? 2 : 1), kPlainThreads, args,
                      2 * 2 * sizeof(T) * ((size_t)a.n0 << a.lg0), s);
}
#define INST(T)                                                                                                     \
    template bool plain_setup<T>(PlainArgs<T> &, int);                                                              \
    template cudaError_t launch_plain_mean<T>(const T *, long long, int, double *, double *, unsigned *, cudaStream_t); \
    template cudaError_t launch_plain_rows<T>(const PlainArgs<T> &, bool, cudaStream_t);                            \
    template cudaError_t launch_plain_n0<T>(const PlainArgs<T> &, cudaStream_t);
INST(float)
INST(double)

}  // namespace ofdft
