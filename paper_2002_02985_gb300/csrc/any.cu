// Plans, candidates and instantiations of the any-length kernels (any.cuh); the
// reciprocal-space kernels are instantiated in any_ax0.cu.
#include <algorithm>
#include <cstdio>

#include "any.cuh"

namespace ofdft {

static const int kRadices[] = {16, 15, 12, 10, 9, 8, 6, 5, 4, 3, 2};

AnyPlan any_plan(int n, int last) {
    AnyPlan q;
    q.n = n;
    q.np = 0;
    if (n < 4 || n > 1024) return q;
    // two passes where the radices allow, else three; of equal pass counts the plan whose
    // largest radix is smallest (most butterflies per pass, fewest registers)
    int best[3] = {0, 0, 0}, np = 0, score = 1 << 30;
    for (int a : kRadices)
        for (int b : kRadices) {
            if (n % (a * b)) continue;
            const int c = n / (a * b);
            if (c == 1) {
                if (last && b != last) continue;
                if (!last && a < b) continue;
                const int s = std::max(a, b) * 32 + a;
                if (np != 2 || s < score) {
                    np = 2;
                    score = s;
                    best[0] = a;
                    best[1] = b;
                }
            } else if (np != 2 && std::find(std::begin(kRadices), std::end(kRadices), c) != std::end(kRadices)) {
                if (last && c != last) continue;
                if (a < b || (!last && b < c)) continue;
                const int s = (std::max(a, std::max(b, c)) * 32 + a) * 32 + b;
                if (s < score) {
                    np = 3;
                    score = s;
                    best[0] = a;
                    best[1] = b;
                    best[2] = c;
                }
            }
        }
    q.np = np;
    int ns = 1;
    for (int i = 0; i < np; i++) {
        AnyPass &p = q.p[i];
        p.R = best[i];
        p.ns = ns;
        p.nb = n / p.R;
        p.stride = n / (ns * p.R);
        p.magic = ((1 << 20) + ns - 1) / ns;
        ns *= p.R;
    }
    return q;
}

// the same radices in reverse order (an inverse transform that starts where the forward ended)
AnyPlan any_reversed(const AnyPlan &q) {
    AnyPlan r = q;
    int ns = 1;
    for (int i = 0; i < q.np; i++) {
        AnyPass &p = r.p[i];
        p.R = q.p[q.np - 1 - i].R;
        p.ns = ns;
        p.nb = q.n / p.R;
        p.stride = q.n / (ns * p.R);
        p.magic = ((1 << 20) + ns - 1) / ns;
        ns *= p.R;
    }
    return r;
}

// the reciprocal-space kernels (any_ax0.cu): null where RL is not compiled for T
template <typename T> const void *any_axis0_kernel(int RL, bool mgp);

// the compile-time plans (any_ct*.cu)
bool any_ct_axis0_1(int, bool, AnyCt &);
bool any_ct_axis0_2(int, bool, AnyCt &);
bool any_ct_axis0_3(int, bool, AnyCt &);
bool any_ct_axis0_4(int, bool, AnyCt &);
bool any_ct_pencil_1(int, AnyCt &);
bool any_ct_pencil_2(int, AnyCt &);
bool any_ct_pencil_3(int, AnyCt &);
bool any_ct_pencil_4(int, AnyCt &);
bool any_ct_rows_1(int, AnyCt &);
bool any_ct_rows_2(int, AnyCt &);
bool any_ct_rows_3(int, AnyCt &);
bool any_ct_rows_4(int, AnyCt &);

template <typename T> const void *any_row_kernel(int E, bool inverse) {
    if (E <= 1) return inverse ? (const void *)row_inv_any_kernel<T, 1> : (const void *)row_fwd_any_kernel<T, 1>;
    if (E <= 2) return inverse ? (const void *)row_inv_any_kernel<T, 2> : (const void *)row_fwd_any_kernel<T, 2>;
    return inverse ? (const void *)row_inv_any_kernel<T, 4> : (const void *)row_fwd_any_kernel<T, 4>;
}

template <typename T> void any_candidates(int role, int n, long long cols, int nsm, std::vector<KernelCand> &out) {
    KernelCand c;
    c.any = 1;
    auto add = [&](const void *k1, const void *k2, int B, int nt, const char *kind) {
        c.k1 = c.g1 = k1;
        c.k2 = c.g2 = k2;
        c.B = B;
        c.nt = nt;
        std::snprintf(c.name, sizeof(c.name), "%s %dx%d", kind, B, nt);
        out.push_back(c);
    };
    const AnyPlan q = any_plan(n);
    if (role == ROLE_PENCIL && q.np >= 2) {
        AnyCt ct;
        if (sizeof(T) == 4 && (any_ct_pencil_1(n, ct) || any_ct_pencil_2(n, ct) || any_ct_pencil_3(n, ct) || any_ct_pencil_4(n, ct))) {
            c.any = 2;
            add(ct.k, ct.k2, 1 << ct.lg, ct.nt, "ctpencil");
            return;
        }
        // 16-column tiles (128-byte rows in FP32) while three blocks fit an SM, else 8
        int rmax = 1;
        for (int i = 0; i < q.np; i++) rmax = std::max(rmax, q.p[i].R);
        for (int lg : {4, 3}) {
            if (any_pencil_smem<T>(q, lg) > 74 * 1024 && lg > 3) continue;
            if (any_pencil_smem<T>(q, lg) > 200 * 1024) continue;
            add((const void *)pencil_any_kernel<T, -1>, (const void *)pencil_any_kernel<T, +1>, 1 << lg,
                any_ct_pencil_threads(n, rmax, lg), "anypencil");
            break;
        }
    }
    if (role == ROLE_ROW2 && q.np >= 1) {
        c.batched = true;
        int last = 0;
        AnyCt ct;
        if (sizeof(T) == 4 && (any_ct_rows_1(n, ct) || any_ct_rows_2(n, ct) || any_ct_rows_3(n, ct) || any_ct_rows_4(n, ct)))
            c.any = 2;
        // the channel group fills a fifth, a quarter or a third of an SM's shared memory per block (512
        // points: nine channels leave room for two blocks, seven for the three that the threads allow)
        for (int kb : {40, 60, 76}) {
            const int G = std::min(34, (int)(kb * 1024 / (2 * (size_t)(n + 2) * 2 * sizeof(T))));
            if (G < 1 || G == last) continue;
            last = G;
            c.batched = true;
            add(c.any == 2 ? ct.k : any_row_kernel<T>(1, false), c.any == 2 ? ct.k2 : any_row_kernel<T>(1, true), G, 320,
                c.any == 2 ? "ctrows" : "anyrows");
        }
    }
    if (role == ROLE_AXIS0) {
        int made = 0;
        AnyCt ct;
        // blocks per tile: 1 where the tiles fill the SMs, else up to two blocks per SM
        auto split = [&](int lg) {
            const long long tiles = (cols + (1 << lg) - 1) >> lg;
            return tiles >= nsm ? 1 : (int)std::max(1LL, std::min<long long>(kMaxSplit, 2 * nsm / tiles));
        };
        auto put = [&](const void *k, const void *km, int RL, int lg, int nt, const char *kind) {
            c.RL = RL;
            c.split = split(lg);
            add(k, km, 1 << lg, nt, kind);
            std::snprintf(out.back().name, sizeof(c.name), "%s r%d %dx%d s%d", kind, RL, 1 << lg, nt, c.split);
            made++;
        };
        auto compiled = [&](bool narrow) {
            return any_ct_axis0_1(n, narrow, ct) || any_ct_axis0_2(n, narrow, ct) || any_ct_axis0_3(n, narrow, ct) ||
                   any_ct_axis0_4(n, narrow, ct);
        };
        if (sizeof(T) == 4 && compiled(false)) {
            c.any = 2;
            put(ct.k, ct.k2, ct.RL, ct.lg, ct.nt, "ctrecip");
            // the run-time kernels only where the compiled tiles leave SMs without one
            const bool enough = c.split == 1;
            if (compiled(true)) put(ct.k, ct.k2, ct.RL, ct.lg, ct.nt, "ctrecip");
            c.any = 1;
            if (enough) return;
        }
        for (int RL : {16, 15, 12, 10, 9, 8, 5, 4}) {
            const void *k = any_axis0_kernel<T>(RL, false), *km = any_axis0_kernel<T>(RL, true);
            if (!k || n % RL || any_plan(n, RL).np < 2 || made >= 4) continue;
            const int tmax = sizeof(T) == 4 ? (RL >= 12 ? 256 : 512) : 256;
            // the widest of 16, 8 or 4 columns that leaves room for two blocks per SM, and the
            // narrowest as well where the grid has fewer tiles than SMs
            int widest = -1;
            for (int lg : {4, 3, 2}) {
                const int nt = ((n / RL << lg) + 31) / 32 * 32;
                if (nt > tmax || any_axis0_smem<T>(n, lg) > (lg == 4 ? 100 : 200) * 1024) continue;
                if (widest >= 0 && !(lg == 2 && (cols >> widest) < nsm)) continue;
                if (widest < 0) widest = lg;
                put(k, km, RL, lg, nt, "anyrecip");
            }
        }
    }
}

#define INST(T)                                                              \
    template const void *any_row_kernel<T>(int, bool);                       \
    template void any_candidates<T>(int, int, long long, int, std::vector<KernelCand> &);
INST(float)
INST(double)

}  // namespace ofdft
