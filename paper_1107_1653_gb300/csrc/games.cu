// Finite games given by explicit transition tables (Sec. 2): validation and
// set-up of the CSR tables, and a persistent kernel in which each thread block
// takes games from a queue and runs the whole policy iteration on one game
// (Algorithm 2 with Algorithm 1 inside) -- improvement, assembly, multigrid
// policy evaluation, stopping tests -- with the game's vectors in shared memory.
//
// Multigrid for the policy-fixed system (I - mu M) w = r of a general game: the
// smoother is Jacobi relaxation; the coarse space is spanned by the constant
// vector, whose Galerkin operator is 1^T A 1 = sum of A's row sums.  For a
// stochastic M the constant vector is the slow mode of I - mu M (eigenvalue
// 1 - mu), which relaxation cannot remove and the coarse correction removes
// exactly; the other modes contract at the rate of M's second eigenvalue.
#include <algorithm>
#include <cfloat>

#include "device_once.h"
#include "games.cuh"
#include "gridsync.cuh"

namespace gs {

namespace {

constexpr int kThreads = 512;

// ------------------------------------------------------------------ validation
__global__ void k_game_validate(GameTables T, int count, const int64_t* __restrict__ st_off,
                                int* __restrict__ bad) {
    const int64_t R = (int64_t)T.m1 * T.m2;
    const int64_t rows = st_off[count] * R;
    for (int64_t row = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; row < rows;
         row += (int64_t)gridDim.x * blockDim.x) {
        // game of this row: binary search over the state offsets
        const int64_t x = row / R;
        int lo = 0, hi = count - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) / 2;
            if (st_off[mid] <= x) lo = mid;
            else hi = mid - 1;
        }
        const int64_t n = st_off[lo + 1] - st_off[lo];
        const int64_t k0 = T.row_ptr[row], k1 = T.row_ptr[row + 1];
        int err = 0;
        if (k1 < k0) err |= 1;
        double sum = 0.0;
        for (int64_t k = k0; k < k1 && !(err & 1); ++k) {
            const int32_t c = T.col[k];
            const double p = T.prob[k];
            if (c < 0 || c >= n) err |= 2;
            if (!(p >= 0.0) || !(p <= 1.0)) err |= 4;
            sum += p;
        }
        if (sum > 1.0 + 1e-12) err |= 8;
        if (!(fabs(T.rew[row]) <= DBL_MAX)) err |= 16;
        if (k1 - k0 != T.row_ptr[1] - T.row_ptr[0]) err |= 32;   // rows of unequal length (allowed)
        if (err) atomicOr(bad, err);
    }
}

// Per row: leakage 1 - mu sum_k p_k (float64) and the float32 or bfloat16 copy of p.
__global__ void k_game_prepare(GameTables T, int count, const int64_t* __restrict__ st_off,
                               const double* __restrict__ mu, double* __restrict__ leak,
                               float* __restrict__ leak32, float* __restrict__ prob32,
                               __nv_bfloat16* __restrict__ prob16) {
    const int64_t R = (int64_t)T.m1 * T.m2;
    const int64_t rows = st_off[count] * R;
    for (int64_t row = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; row < rows;
         row += (int64_t)gridDim.x * blockDim.x) {
        const int64_t x = row / R;
        int lo = 0, hi = count - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) / 2;
            if (st_off[mid] <= x) lo = mid;
            else hi = mid - 1;
        }
        double sum = 0.0;
        for (int64_t k = T.row_ptr[row]; k < T.row_ptr[row + 1]; ++k) {
            sum += T.prob[k];
            if (prob16) prob16[k] = __double2bfloat16(T.prob[k]);
            else prob32[k] = (float)T.prob[k];
        }
        leak[row] = 1.0 - mu[lo] * sum;
        leak32[row] = (float)leak[row];
    }
}

// ------------------------------------------------------------------ block helpers
template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Maximum of 64-bit patterns over a warp by two 32-bit reductions (non-negative
// doubles order like their bits; a float64 compare costs as much as float64
// arithmetic here).
__device__ __forceinline__ unsigned long long warp_max_bits(unsigned long long v) {
    const unsigned hi = (unsigned)(v >> 32);
    const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
    const unsigned ml = __reduce_max_sync(0xffffffffu, hi == mh ? (unsigned)v : 0u);
    return (unsigned long long)mh << 32 | ml;
}

// Shared scratch of the block reductions: two copies used in turn, so that one
// block barrier per reduction is enough (a copy is written again only after
// the barrier of the reduction in between).
struct RedScratch {
    unsigned long long m[2][2][32];
    double d[2][32];
    int i[2][32];
};

// Block-wide reductions over `bufs`; every thread gets the result.
__device__ __forceinline__ void block_max2(unsigned long long a, unsigned long long b, RedScratch& S, int f,
                                           unsigned long long* A, unsigned long long* B) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    a = warp_max_bits(a);
    b = warp_max_bits(b);
    if (lane == 0) {
        S.m[f][0][w] = a;
        S.m[f][1][w] = b;
    }
    __syncthreads();
    *A = warp_max_bits(lane < nw ? S.m[f][0][lane] : 0ull);
    *B = warp_max_bits(lane < nw ? S.m[f][1][lane] : 0ull);
}
__device__ __forceinline__ int block_sum_int(int v, RedScratch& S, int f) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    v = __reduce_add_sync(0xffffffffu, v);
    if (lane == 0) S.i[f][w] = v;
    __syncthreads();
    return __reduce_add_sync(0xffffffffu, lane < nw ? S.i[f][lane] : 0);
}
// Sum in a fixed order: a tree over the lanes, then a tree over the warps.
__device__ __forceinline__ double block_sum_double(double v, RedScratch& S, int f) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    v = warp_sum(v);
    if (lane == 0) S.d[f][w] = v;
    __syncthreads();
    v = lane < nw ? S.d[f][lane] : 0.0;
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return __shfl_sync(0xffffffffu, v, 0);   // at most 16 warps: the tree over lanes 0 .. 15
}

// ------------------------------------------------------------------ one game
// Transition probability k rounded to float32 (the screen's error bound
// assumes float32 rounding: with bfloat16 storage it rounds the float64 value).
__device__ __forceinline__ float prob_at_f(const GameTables& tb, int64_t k) {
    return tb.prob16 ? f64_to_f32(tb.prob[k]) : tb.prob32[k];
}

struct Game {
    GameTables T;
    int64_t x0, n, row0;   // first state, states, first row
    double mu;
    float mu_f;            // mu rounded to float32
    int R;                 // m1 * m2
};

// sum_k p_k v(col_k) over a row, v indexed locally.  Two partial sums: a
// float64 operation's latency is 64 cycles here.
__device__ __forceinline__ double row_sum(const Game& G, int64_t row, const double* v) {
    int64_t k0, k1;
    row_range(G.T, row, &k0, &k1);
    double s0 = 0.0, s1 = 0.0;
    int64_t k = k0;
    for (; k + 1 < k1; k += 2) {
        s0 = fma(G.T.prob[k], v[G.T.col[k]], s0);
        s1 = fma(G.T.prob[k + 1], v[G.T.col[k + 1]], s1);
    }
    if (k < k1) s0 = fma(G.T.prob[k], v[G.T.col[k]], s0);
    return s0 + s1;
}

// F(v; x, a, b) = mu sum_k p_k v(col_k) + r(x, a, b)  (Eq. (ILPI)).
__device__ __forceinline__ double row_value(const Game& G, int64_t row, const double* v) {
    return G.mu * row_sum(G, row, v) + G.T.rew[row];
}

// The same in float32 from the float32 copies (a screen; |error| <= err_of).
__device__ __forceinline__ float row_value_f(const Game& G, int64_t row, const float* v32) {
    int64_t k0, k1;
    row_range(G.T, row, &k0, &k1);
    float s = 0.0f;
    for (int64_t k = k0; k < k1; ++k) s = fmaf(prob_at_f(G.T, k), v32[G.T.col[k]], s);
    return G.mu_f * s + f64_to_f32(G.T.rew[row]);
}

// The exact float64 decisions for one state (near-ties of the float32 screen).
// Not inlined: the compiler must not evaluate these rows for every state.
__device__ __noinline__ int improve_state_exact(const Game& G, const BatchOut& O, int mode, int64_t i,
                                                double tau, const double* v, double* res) {
    const int m1 = G.T.m1, m2 = G.T.m2;
    const int64_t x = G.x0 + i;
    const int64_t rb = G.row0 + i * G.R;
    const int acur = O.alpha[x];
    double Fa[kGameMaxM1];
    int changed = 0;
    for (int a = 0; a < m1; ++a) {
        if (mode == 1 && a != acur) continue;
        uint8_t& bref = O.beta[x * m1 + a];
        const int bcur = bref;
        double best = 0.0, fcur = 0.0;
        int first = 0;
        for (int b = 0; b < m2; ++b) {
            const double F = row_value(G, rb + a * m2 + b, v);
            if (b == 0 || F < best) { best = F; first = b; }
            if (b == bcur) fcur = F;
        }
        const int bnew = (fcur - best > tau) ? first : bcur;
        if (bnew != bcur) {
            bref = (uint8_t)bnew;
            if (mode == 1) changed = 1;
        }
        Fa[a] = best;
    }
    int anew = acur;
    if (mode == 0) {
        double fmax_ = Fa[0];
        int first = 0;
        for (int a = 1; a < m1; ++a)
            if (Fa[a] > fmax_) { fmax_ = Fa[a]; first = a; }
        anew = (fmax_ - Fa[acur] > tau) ? first : acur;
        changed = anew != acur;
        *res = fabs(fmax_ - v[i]);
        O.alpha[x] = (uint8_t)anew;
    }
    const int64_t row = rb + anew * m2 + O.beta[x * m1 + anew];
    O.sel[x] = row;
    O.rhs[x] = G.T.rew[row];
    return changed;
}

// Policy improvement at local state i (modes as for the Isaacs grid), screened
// in float32: every F(v; x, a, b) is first taken from the float32 copies of p
// and v, within err = 2^-18 (mu |v|_inf + |r|) of its float64 value (float32
// rounding of the inputs and of at most 10 operations, with a wide margin).
// A decision whose best candidate beats the second by more than 2 err + tau
// is the float64 one; otherwise the state takes the exact path.  float64 then
// only evaluates |F(v) - v| for the chosen row (outer mode).
// Returns the number of changed policy entries; *res gets |F(v) - v| (outer).
__device__ int improve_state(const Game& G, const BatchOut& O, int mode, int64_t i, double tau,
                             float tauf, float vmaxf, const double* v, double* res) {
    // games with many MAX actions (fine discretisations of continuous action
    // sets) take the float64 decisions directly
    if (G.T.m1 > kScreenMaxM1) return improve_state_exact(G, O, mode, i, tau, v, res);
    const int m1 = G.T.m1, m2 = G.T.m2;
    const int64_t x = G.x0 + i;
    const int64_t rb = G.row0 + i * G.R;
    const int acur = O.alpha[x];
    const float* v32 = O.v32 + G.x0;
    float Fa[kScreenMaxM1];
    int bsel[kScreenMaxM1];
    bool sure = true;
    for (int a = 0; a < m1 && sure; ++a) {
        if (mode == 1 && a != acur) continue;
        float best = INFINITY, second = INFINITY, rmax = 0.0f;
        int first = 0;
        for (int b = 0; b < m2; ++b) {
            const int64_t row = rb + a * m2 + b;
            const float F = row_value_f(G, row, v32);
            rmax = fmaxf(rmax, fabsf(f64_to_f32(G.T.rew[row])));
            if (F < best) {
                second = best;
                best = F;
                first = b;
            } else if (F < second) {
                second = F;
            }
        }
        const float err = 0x1p-18f * (G.mu_f * vmaxf + rmax);
        sure = m2 == 1 || second - best > 2.0f * err + tauf;
        Fa[a] = best;
        bsel[a] = first;
    }
    int anew = acur;
    if (sure && mode == 0) {
        float g1 = -INFINITY, g2 = -INFINITY;
        int first = 0;
        for (int a = 0; a < m1; ++a) {
            if (Fa[a] > g1) {
                g2 = g1;
                g1 = Fa[a];
                first = a;
            } else if (Fa[a] > g2) {
                g2 = Fa[a];
            }
        }
        float rmax = 0.0f;
        for (int r = 0; r < G.R; ++r) rmax = fmaxf(rmax, fabsf(f64_to_f32(G.T.rew[rb + r])));
        const float err = 0x1p-18f * (G.mu_f * vmaxf + rmax);
        sure = m1 == 1 || g1 - g2 > 2.0f * err + tauf;
        anew = first;
    }
    if (!sure) return improve_state_exact(G, O, mode, i, tau, v, res);
    int changed = 0;
    for (int a = 0; a < m1; ++a) {
        if (mode == 1 && a != acur) continue;
        uint8_t& bref = O.beta[x * m1 + a];
        if (bref != bsel[a]) {
            bref = (uint8_t)bsel[a];
            if (mode == 1) changed = 1;
        }
    }
    const int64_t row = rb + anew * m2 + O.beta[x * m1 + anew];
    if (mode == 0) {
        changed = anew != acur;
        *res = fabs(row_value(G, row, v) - v[i]);
        O.alpha[x] = (uint8_t)anew;
    }
    O.sel[x] = row;
    O.rhs[x] = G.T.rew[row];
    return changed;
}

// ------------------------------------------------------------------ improvement, one lane per row
// 32 consecutive aligned bytes by one 256-bit load (the tables do not change
// while a kernel runs).
__device__ __forceinline__ void load_32b(const void* p, unsigned r[8]) {
    unsigned long long q[4];
    asm("ld.global.nc.v4.b64 {%0, %1, %2, %3}, [%4];" : "=l"(q[0]), "=l"(q[1]), "=l"(q[2]), "=l"(q[3]) : "l"(p));
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        r[2 * k] = (unsigned)q[k];
        r[2 * k + 1] = (unsigned)(q[k] >> 32);
    }
}

// One row's entries in registers: columns and probabilities rounded to float32
// (rows of 8 entries; with bfloat16 storage rounded from the float64 values).
struct Row8 {
    unsigned c[8];
    float p[8];
    __device__ __forceinline__ void load(const GameTables& T, int64_t row) {
        load_32b(T.col + row * 8, c);
        unsigned q[8];
        if (T.prob32) {
            load_32b(T.prob32 + row * 8, q);
#pragma unroll
            for (int k = 0; k < 8; ++k) p[k] = __uint_as_float(q[k]);
        } else {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                load_32b(T.prob + row * 8 + 4 * h, q);
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    p[4 * h + k] = f64_to_f32(__hiloint2double((int)q[2 * k + 1], (int)q[2 * k]));
            }
        }
    }
    // F(v; x, a, b) in float32 (row_value_f's order of operations).
    __device__ __forceinline__ float value(const Game& G, const float* v32, float r) const {
        float vc[8], s = 0.0f;
#pragma unroll
        for (int k = 0; k < 8; ++k) vc[k] = v32[c[k]];
#pragma unroll
        for (int k = 0; k < 8; ++k) s = fmaf(p[k], vc[k], s);
        return G.mu_f * s + r;
    }
};

// Whether the improvement below takes a game's action counts: the rows of a
// state, and those of one MAX action, each fill an aligned group of lanes.
__host__ __device__ __forceinline__ bool rows_in_lanes(int m1, int m2) {
    return m1 <= kScreenMaxM1 && m1 * m2 <= 32 && (m1 & (m1 - 1)) == 0 && (m2 & (m2 - 1)) == 0;
}

// Policy improvement of a whole game with one lane per row (x, a, b): the
// decisions and their float32 screen are those of improve_state, but a warp
// reads its rows' entries as consecutive memory (256-bit loads), and the
// minimum over b and the maximum over a are taken by lane exchanges inside the
// state's group of lanes (m1 m2 of them; the m2 of the current action in mode
// 1).  NE states per lane group are in flight at once.  Bound by the shared-
// memory or L2 gathers from v32 and the bytes of the rows (72 per row of 8
// entries); one lane per action walking its m2 rows issues fewer instructions
// but touches a cache line per lane and was slower (212 and 71 us below).
// Measured per improvement, games of 4224 states on average with 4 x 4 actions,
// one block each: all actions 823 -> 200 us, MIN's reply at fixed alpha 258 ->
// 55 us; one game of 5e5 states on the whole GPU: 892 -> 306 and 324 -> 80 us
// (the first figures: one thread per state).  Writes beta, sel, rhs (and alpha
// in mode 0); returns this thread's count of changed policy entries.
template <int KC, int MODE, class Ctx>
__device__ __noinline__ int improve_rows(const Game& G, const BatchOut& O, double tau, float vmaxf, const double* v,
                                         const float* v32, const Ctx& C) {
    constexpr int NE = 2;
    const int m1 = G.T.m1, m2 = G.T.m2;
    const int grp = MODE == 1 ? m2 : G.R;
    const int lane = threadIdx.x & 31, sub = lane & (grp - 1);
    const int gl = __ffs(grp) - 1, bl = __ffs(m2) - 1;   // log2
    const int per = 32 >> gl;                            // states per warp step
    const int b = sub & (m2 - 1);
    const float tauf = f64_to_f32(tau);
    int changed = 0;
    for (int64_t base = (int64_t)C.warp() * per * NE; base < G.n; base += (int64_t)C.warps() * per * NE) {
        int64_t st[NE], row[NE];
        int a[NE], acur[NE], bcurs[NE];
        bool ok[NE];
        double r64[NE];
        float F[NE];
#pragma unroll
        for (int e = 0; e < NE; ++e) {
            const int64_t i = base + e * per + (lane >> gl);
            ok[e] = i < G.n;
            st[e] = ok[e] ? i : G.n - 1;
            acur[e] = O.alpha[G.x0 + st[e]];
        }
#pragma unroll
        for (int e = 0; e < NE; ++e) {
            a[e] = MODE == 1 ? acur[e] : sub >> bl;
            row[e] = G.row0 + st[e] * G.R + a[e] * m2 + b;
            r64[e] = G.T.rew[row[e]];
            bcurs[e] = O.beta[(G.x0 + st[e]) * m1 + a[e]];
        }
        if constexpr (KC == 8) {
            Row8 R8[NE];
#pragma unroll
            for (int e = 0; e < NE; ++e) R8[e].load(G.T, row[e]);
#pragma unroll
            for (int e = 0; e < NE; ++e) F[e] = R8[e].value(G, v32, f64_to_f32(r64[e]));
        } else {
#pragma unroll
            for (int e = 0; e < NE; ++e) {
                int64_t k0, k1;
                row_range(G.T, row[e], &k0, &k1);
                float sum = 0.0f;
                for (int64_t k = k0; k < k1; ++k) sum = fmaf(prob_at_f(G.T, k), v32[G.T.col[k]], sum);
                F[e] = G.mu_f * sum + f64_to_f32(r64[e]);
            }
        }
#pragma unroll
        for (int e = 0; e < NE; ++e) {
            // smallest and second smallest F over b (ties: the lower b), largest |r|
            float best = F[e], second = INFINITY, rmax = fabsf(f64_to_f32(r64[e]));
            int first = b;
            for (int o = 1; o < m2; o <<= 1) {
                const float b2 = __shfl_xor_sync(0xffffffffu, best, o);
                const float s2 = __shfl_xor_sync(0xffffffffu, second, o);
                const int f2 = __shfl_xor_sync(0xffffffffu, first, o);
                rmax = fmaxf(rmax, __shfl_xor_sync(0xffffffffu, rmax, o));
                second = fminf(fminf(second, s2), fmaxf(best, b2));
                if (b2 < best || (b2 == best && f2 < first)) {
                    best = b2;
                    first = f2;
                }
            }
            float err = 0x1p-18f * (G.mu_f * vmaxf + rmax);
            bool sure = m2 == 1 || second - best > 2.0f * err + tauf;
            int anew = acur[e];
            if (MODE != 1) {
                // every reply must be sure; the largest and second largest over a
                float g1 = best, g2 = -INFINITY;
                int ga = a[e];
                for (int o = m2; o < grp; o <<= 1) {
                    const float h1 = __shfl_xor_sync(0xffffffffu, g1, o);
                    const float h2 = __shfl_xor_sync(0xffffffffu, g2, o);
                    const int ha = __shfl_xor_sync(0xffffffffu, ga, o);
                    rmax = fmaxf(rmax, __shfl_xor_sync(0xffffffffu, rmax, o));
                    sure &= __shfl_xor_sync(0xffffffffu, (int)sure, o) != 0;
                    g2 = fmaxf(fmaxf(g2, h2), fminf(g1, h1));
                    if (h1 > g1 || (h1 == g1 && ha < ga)) {
                        g1 = h1;
                        ga = ha;
                    }
                }
                if (MODE == 0) {
                    err = 0x1p-18f * (G.mu_f * vmaxf + rmax);
                    sure = sure && (m1 == 1 || g1 - g2 > 2.0f * err + tauf);
                    anew = ga;
                }
            }
            const int64_t x = G.x0 + st[e];
            const int bcur = bcurs[e];
            int bsel = first;
            if (__any_sync(0xffffffffu, !sure)) {
                // the exact float64 decisions (improve_state_exact's) for the
                // states whose screen was not conclusive, a row per lane: one
                // lane evaluating a state's rows in turn held its warp up for
                // tens of microseconds
                const double F64 = row_value(G, row[e], v);
                double fb = F64;
                int fi = b;
                for (int o = 1; o < m2; o <<= 1) {
                    const double b2 = __shfl_xor_sync(0xffffffffu, fb, o);
                    const int f2 = __shfl_xor_sync(0xffffffffu, fi, o);
                    if (b2 < fb || (b2 == fb && f2 < fi)) {
                        fb = b2;
                        fi = f2;
                    }
                }
                const double fcur = __shfl_sync(0xffffffffu, F64, (lane & ~(m2 - 1)) | (bcur & (m2 - 1)));
                const int bx = fcur - fb > tau ? fi : bcur;
                int ax = acur[e];
                if (MODE == 0) {
                    double h = fb;
                    int ha = a[e];
                    for (int o = m2; o < grp; o <<= 1) {
                        const double h2 = __shfl_xor_sync(0xffffffffu, h, o);
                        const int a2 = __shfl_xor_sync(0xffffffffu, ha, o);
                        if (h2 > h || (h2 == h && a2 < ha)) {
                            h = h2;
                            ha = a2;
                        }
                    }
                    const double hcur = __shfl_sync(0xffffffffu, fb, (lane & ~(grp - 1)) | acur[e] << bl);
                    ax = h - hcur > tau ? ha : acur[e];
                }
                if (!sure) {
                    bsel = bx;
                    anew = ax;
                }
            }
            if (ok[e] && b == bsel) {   // the lane of the chosen b of its action
                if (bcur != b) {
                    O.beta[x * m1 + a[e]] = (uint8_t)b;
                    if (MODE == 1) ++changed;
                }
                if (a[e] == anew) {   // ... of the state's action
                    if (MODE == 0 && anew != acur[e]) {
                        O.alpha[x] = (uint8_t)anew;
                        ++changed;
                    }
                    O.sel[x] = row[e];
                    O.rhs[x] = r64[e];
                }
            }
        }
    }
    return changed;
}

// ------------------------------------------------------------------ policy-fixed rows
// Transition probability k in the relaxation's precision.
template <typename T>
__device__ __forceinline__ T prob_at(const GameTables& tb, int64_t k) {
    if constexpr (sizeof(T) == 8) return tb.prob[k];
    else return tb.prob16 ? __bfloat162float(tb.prob16[k]) : tb.prob32[k];
}

// (A e)_i and the diagonal of A = I - mu M for the selected row, leakage form:
// (A e)_i = s_i e_i + mu sum_k p_k (e_i - e_col), s_i = 1 - mu sum_k p_k.
template <typename T>
__device__ __forceinline__ void apply_row(const Game& G, const BatchOut& O, int64_t i, const T* e,
                                          T* Ae, T* diag) {
    const int64_t row = O.sel[G.x0 + i];
    const T ei = e[i];
    const T mu = sizeof(T) == 4 ? (T)G.mu_f : (T)G.mu;
    const T leak = sizeof(T) == 4 ? (T)G.T.leak32[row] : (T)G.T.leak[row];
    T acc = leak * ei, off = 0;
    int64_t k0, k1;
    row_range(G.T, row, &k0, &k1);
    for (int64_t k = k0; k < k1; ++k) {
        const int32_t c = G.T.col[k];
        const T p = prob_at<T>(G.T, k);
        acc += mu * p * (ei - e[c]);
        if (c != i) off += mu * p;
    }
    *Ae = acc;
    *diag = leak + off;
}

// Diagonal of A for the selected row: s_i + mu sum_{k: col_k != i} p_k.
template <typename T>
__device__ __forceinline__ T diag_row(const Game& G, const BatchOut& O, int64_t i) {
    const int64_t row = O.sel[G.x0 + i];
    const T mu = sizeof(T) == 4 ? (T)G.mu_f : (T)G.mu;
    T off = 0;
    int64_t k0, k1;
    row_range(G.T, row, &k0, &k1);
    for (int64_t k = k0; k < k1; ++k)
        if (G.T.col[k] != i) off += mu * prob_at<T>(G.T, k);
    return (sizeof(T) == 4 ? (T)G.T.leak32[row] : (T)G.T.leak[row]) + off;
}

// Copies state i's selected row into the slot-major arrays, with the inverse
// of its diagonal (the relaxation multiplies by it: the inverse's rounding is one
// of the relaxation's weight, not of the residual the correction answers, which
// every check forms anew in float64).
template <typename T, int KC>
__device__ __forceinline__ void compact_row(const Game& G, const Compact& S, int64_t i, int64_t row) {
    const int K = KC > 0 ? KC : S.K;
    const int64_t k0 = row * K;
    const T mu = sizeof(T) == 4 ? (T)G.mu_f : (T)G.mu;
    T off = 0;
    auto put = [&](int k, int32_t c, double p64) {
        T p;
        if constexpr (sizeof(T) == 8) p = p64;
        else p = prob_at<T>(G.T, k0 + k);
        S.col[k * G.n + i] = c;
        S.p64[k * G.n + i] = p64;
        if constexpr (sizeof(T) == 4) S.p32[k * G.n + i] = mu * p;
        if (c != i) off += mu * p;
    };
    if constexpr (KC == 8) {
        unsigned c[8], lo[8], hi[8];
        load_32b(G.T.col + k0, c);
        load_32b(G.T.prob + k0, lo);
        load_32b(G.T.prob + k0 + 4, hi);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const unsigned* q = k < 4 ? lo : hi;
            put(k, (int32_t)c[k], __hiloint2double((int)q[2 * (k & 3) + 1], (int)q[2 * (k & 3)]));
        }
    } else {
        for (int k = 0; k < K; ++k) put(k, G.T.col[k0 + k], G.T.prob[k0 + k]);
    }
    S.leak64[i] = G.T.leak[row];
    S.leak32[i] = G.T.leak32[row];
    const T leak = sizeof(T) == 4 ? (T)G.T.leak32[row] : (T)G.T.leak[row];
    ((T*)S.dinv)[i] = T(1) / (leak + off);
    S.cur[i] = row;
}

// sum_k p_k v(col_k) and (A e)_i over the slot-major rows, in the order of the
// row's entries (KC > 0: rows of exactly KC entries, known at compile time, so
// that a row's loads are issued together; KC = 0: S.K at run time).
template <int KC>
__device__ __forceinline__ double row_sum_c(const Compact& S, int64_t n, int64_t i, const double* v) {
    const int K = KC > 0 ? KC : S.K;
    double s0 = 0.0, s1 = 0.0;
    int k = 0;
#pragma unroll
    for (; k + 1 < K; k += 2) {
        s0 = fma(S.p64[k * n + i], v[S.col[k * n + i]], s0);
        s1 = fma(S.p64[(k + 1) * n + i], v[S.col[(k + 1) * n + i]], s1);
    }
    if (k < K) s0 = fma(S.p64[k * n + i], v[S.col[k * n + i]], s0);
    return s0 + s1;
}
// (A e)_i in the leakage form, s_i e_i + mu sum_k p_k (e_i - e_col), which is exact
// on the constant mode: e_i - mu sum_k p_k e_col rounds there by 1 / (1 - mu) more
// (float32: mu p_k is stored, float64: 18 operations; one game of 3001 states
// 1.95 ms, with the ten operations of the shorter form 1.90 ms).
template <int KC>
__device__ __forceinline__ float apply_row_c(const Game& G, const Compact& S, int64_t i, const float* e) {
    const int K = KC > 0 ? KC : S.K;
    const float ei = e[i];
    float acc = S.leak32[i] * ei;
#pragma unroll
    for (int k = 0; k < K; ++k) acc = fmaf(S.p32[k * G.n + i], ei - e[S.col[k * G.n + i]], acc);
    return acc;
}
template <int KC>
__device__ __forceinline__ double apply_row_c(const Game& G, const Compact& S, int64_t i, const double* e) {
    const int K = KC > 0 ? KC : S.K;
    const double ei = e[i];
    double s0 = 0.0, s1 = 0.0;
    int k = 0;
#pragma unroll
    for (; k + 1 < K; k += 2) {
        s0 = fma(S.p64[k * G.n + i], ei - e[S.col[k * G.n + i]], s0);
        s1 = fma(S.p64[(k + 1) * G.n + i], ei - e[S.col[(k + 1) * G.n + i]], s1);
    }
    if (k < K) s0 = fma(S.p64[k * G.n + i], ei - e[S.col[k * G.n + i]], s0);
    return fma(G.mu, s0 + s1, S.leak64[i] * ei);
}

// A slot-major row of 8 entries held in registers: the passes below load the
// rows of a thread's next states while they work on the current one, D of them
// at a time, because a pass has too few warps (16 per SM) to cover the latency
// of its loads from L2 otherwise.  Games of 4224 states on average, one block
// each, mixed: residual check 26.1 -> 15.7 us (its float64 operations alone take
// 11), product with the correction 16.6 -> 8.4 us.
template <typename P>
struct SlotRow8 {
    int c[8];
    P p[8];
    __device__ __forceinline__ void load(const int32_t* __restrict__ col, const P* __restrict__ prob, int64_t n, int64_t i) {
#pragma unroll
        for (int k = 0; k < 8; ++k) c[k] = col[k * n + i];
#pragma unroll
        for (int k = 0; k < 8; ++k) p[k] = prob[k * n + i];
    }
};
// sum_k p_k v(col_k), in row_sum_c's order.
__device__ __forceinline__ double row_sum_r(const SlotRow8<double>& R, const double* v) {
    double x[8], s0 = 0.0, s1 = 0.0;
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = v[R.c[k]];
#pragma unroll
    for (int k = 0; k < 8; k += 2) {
        s0 = fma(R.p[k], x[k], s0);
        s1 = fma(R.p[k + 1], x[k + 1], s1);
    }
    return s0 + s1;
}
// (A e)_i from a prefetched row, as apply_row_c.
__device__ __forceinline__ float apply_row_r(const Game&, const SlotRow8<float>& R, float leak, float ei, const float* e) {
    float x[8], acc = leak * ei;
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = e[R.c[k]];
#pragma unroll
    for (int k = 0; k < 8; ++k) acc = fmaf(R.p[k], ei - x[k], acc);
    return acc;
}
__device__ __forceinline__ double apply_row_r(const Game& G, const SlotRow8<double>& R, double leak, double ei,
                                              const double* e) {
    double x[8], s0 = 0.0, s1 = 0.0;
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = e[R.c[k]];
#pragma unroll
    for (int k = 0; k < 8; k += 2) {
        s0 = fma(R.p[k], ei - x[k], s0);
        s1 = fma(R.p[k + 1], ei - x[k + 1], s1);
    }
    return fma(G.mu, s0 + s1, leak * ei);
}
// The relaxation's slot-major weights and leakage in its type.
__device__ __forceinline__ const float* slot_p(const Compact& S, float) { return S.p32; }
__device__ __forceinline__ const double* slot_p(const Compact& S, double) { return S.p64; }
__device__ __forceinline__ const float* slot_leak(const Compact& S, float) { return S.leak32; }
__device__ __forceinline__ const double* slot_leak(const Compact& S, double) { return S.leak64; }

// Execution context of one game's policy iteration: which threads share the
// work, how they synchronise, and where the correction vectors live.  The
// block context runs a game inside one thread block (vectors in shared
// memory); the grid context spreads one game over a cooperative grid (vectors
// in global memory, bounded grid barriers).  Maxima and counts do not depend
// on the order they are combined in; sums are formed in a fixed order.
template <typename T>
struct BlockCtx {
    T *r, *e, *t;      // correction right-hand side, correction, Jacobi work vector
    double* v;         // the iterate in shared memory (null: global)
    RedScratch* red;
    Compact cp{};      // slot-major selected rows (cp.col null: rows read in place)
    int flip = 0;
    __device__ size_t begin() const { return threadIdx.x; }
    __device__ size_t stride() const { return blockDim.x; }
    __device__ unsigned warp() const { return threadIdx.x >> 5; }
    __device__ unsigned warps() const { return blockDim.x >> 5; }
    __device__ bool sync() { __syncthreads(); return true; }
    __device__ int turn() { return flip ^= 1; }
    __device__ void max2(unsigned long long a, unsigned long long b, unsigned long long* A, unsigned long long* B) {
        block_max2(a, b, *red, turn(), A, B);
    }
    // Sum of arr[0 .. n) in its double value, `part` this thread's share.
    template <typename U>
    __device__ double sum(double part, const U*, int64_t) {
        return block_sum_double(part, *red, turn());
    }
    __device__ int sumi(int v) { return block_sum_int(v, *red, turn()); }
    __device__ bool failed() const { return false; }
    __device__ bool leader() const { return threadIdx.x == 0; }
    __device__ bool own_copy() const { return true; }
    // The float32 copy of v that the improvement gathers from: in shared memory.
    __device__ const float* gather_copy(const Game& G, const BatchOut&, const double* vv) {
        float* c = (float*)t;
        for (int64_t i = threadIdx.x; i < G.n; i += blockDim.x) c[i] = f64_to_f32(vv[i]);
        __syncthreads();
        return c;
    }
};

// f64 of a value of the relaxation's type, float32 widened on the integer pipe.
__device__ __forceinline__ double as_f64(float x) { return f32_to_f64(x); }
__device__ __forceinline__ double as_f64(double x) { return x; }

template <typename T>
struct GridCtx {
    T *r, *e, *t;
    double* part;      // [2][gridDim.x] per-block partials (alternating)
    GridScal* gs;      // barrier and the reductions' slots
    Compact cp;        // slot-major selected rows (cp.col null: rows read in place)
    RedScratch* red;
    int flip, slot;
    bool bad;
    // Warp w of every block comes before warp w + 1 of any block: a small
    // game's states are spread over all the blocks' SMs.
    __device__ unsigned warp() const { return (threadIdx.x >> 5) * gridDim.x + blockIdx.x; }
    __device__ unsigned warps() const { return gridDim.x * (blockDim.x >> 5); }
    __device__ size_t begin() const { return (size_t)warp() * 32 + (threadIdx.x & 31); }
    __device__ size_t stride() const { return (size_t)gridDim.x * blockDim.x; }
    __device__ bool sync() {
        if (!bad) bad = !GridSync{&gs->bar, gridDim.x}.sync();
        return !bad;
    }
    __device__ int turn() { return flip ^= 1; }
    // Three slots in turn: reduction t uses slot t mod 3 and clears the next
    // one, whose last readers have passed the barrier before this one's.
    __device__ int take_slot() {
        const int k = slot;
        slot = slot == 2 ? 0 : slot + 1;
        if (leader()) {
            gs->mx[slot][0] = 0ull;
            gs->mx[slot][1] = 0ull;
            gs->cnt[slot] = 0;
        }
        return k;
    }
    __device__ void max2(unsigned long long a, unsigned long long b, unsigned long long* A, unsigned long long* B) {
        const int k = take_slot();
        block_max2(a, b, *red, turn(), A, B);
        if (threadIdx.x == 0) {
            atomicMax(&gs->mx[k][0], *A);
            atomicMax(&gs->mx[k][1], *B);
        }
        if (!sync()) return;
        *A = __ldcg(&gs->mx[k][0]);
        *B = __ldcg(&gs->mx[k][1]);
    }
    __device__ int sumi(int v) {
        const int k = take_slot();
        v = block_sum_int(v, *red, turn());
        if (threadIdx.x == 0 && v) atomicAdd(&gs->cnt[k], v);
        if (!sync()) return 0;
        return __ldcg(&gs->cnt[k]);
    }
    // Games of the size a batch solves by one block: every block sums the whole
    // array itself, in the order one block of this size sums its own game, so
    // that a game solved alone and in a batch gives the same bits.  Larger
    // games: per-block partials combined in block order.
    template <typename U>
    __device__ double sum(double p, const U* arr, int64_t n) {
        if (n < kGameBatchedStates) {
            if (!sync()) return 0.0;
            double acc = 0.0;
            for (int64_t i = threadIdx.x; i < n; i += blockDim.x) acc += as_f64(__ldcg(arr + i));
            return block_sum_double(acc, *red, turn());
        }
        const int f = turn();
        p = block_sum_double(p, *red, f);
        double* P = part + (size_t)f * gridDim.x;
        if (threadIdx.x == 0) P[blockIdx.x] = p;
        if (!sync()) return 0.0;
        double acc = 0.0;
        for (unsigned k = threadIdx.x & 31; k < gridDim.x; k += 32) acc += __ldcg(P + k);
        return warp_sum(acc);
    }
    __device__ bool failed() const { return bad; }
    __device__ bool leader() const { return blockIdx.x == 0 && threadIdx.x == 0; }
    __device__ bool own_copy() const { return false; }
    __device__ const float* gather_copy(const Game& G, const BatchOut& O, const double*) { return O.v32 + G.x0; }
};

// One game over one cluster of kClusterBlocks thread blocks (one launch is one
// cluster): the hardware's cluster barrier instead of the grid barrier and
// reductions through distributed shared memory.  A small game's passes are
// shorter than a grid barrier and its partials' round trip through L2: 3001
// states in float64, per cycle 14.4 us on 94 blocks with the grid barrier.
// Block b holds the chunks of 32 states numbered b modulo 16, so that its partial
// sum is the one warp b of a 512-thread block forms over its own game: the same
// bits alone and in a batch.
constexpr int kClusterBlocks = 16;
struct ClusterScratch {
    unsigned long long m[2][2][kClusterBlocks];   // from every block, two copies in turn
    double d[2][kClusterBlocks];
    int i[2][kClusterBlocks];
    double part[kThreads / 32][32];
};
template <typename T>
struct ClusterCtx {
    T *r, *e, *t;
    Compact cp;
    RedScratch* red;
    ClusterScratch* cs;
    int flip;
    __device__ unsigned warp() const { return (threadIdx.x >> 5) * kClusterBlocks + blockIdx.x; }
    __device__ unsigned warps() const { return kClusterBlocks * (blockDim.x >> 5); }
    __device__ size_t begin() const { return (size_t)warp() * 32 + (threadIdx.x & 31); }
    __device__ size_t stride() const { return (size_t)kClusterBlocks * blockDim.x; }
    __device__ bool sync() {
        asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;" ::: "memory");
        return true;
    }
    __device__ int turn() { return flip ^= 1; }
    // This block's value into slot blockIdx.x of block `rank`'s array.
    template <typename U>
    __device__ void put(U* slots, U v, unsigned rank) const {
        const unsigned local = (unsigned)__cvta_generic_to_shared(slots + blockIdx.x);
        unsigned remote;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local), "r"(rank));
        if constexpr (sizeof(U) == 4)
            asm volatile("st.shared::cluster.b32 [%0], %1;" ::"r"(remote), "r"(__builtin_bit_cast(unsigned, v)) : "memory");
        else
            asm volatile("st.shared::cluster.b64 [%0], %1;" ::"r"(remote), "l"(__builtin_bit_cast(unsigned long long, v))
                         : "memory");
    }
    __device__ void max2(unsigned long long a, unsigned long long b, unsigned long long* A, unsigned long long* B) {
        const int f = turn(), lane = threadIdx.x & 31;
        block_max2(a, b, *red, f, A, B);
        if (threadIdx.x < kClusterBlocks) {
            put(cs->m[f][0], *A, threadIdx.x);
            put(cs->m[f][1], *B, threadIdx.x);
        }
        sync();
        *A = warp_max_bits(lane < kClusterBlocks ? cs->m[f][0][lane] : 0ull);
        *B = warp_max_bits(lane < kClusterBlocks ? cs->m[f][1][lane] : 0ull);
    }
    __device__ int sumi(int v) {
        const int f = turn(), lane = threadIdx.x & 31;
        v = block_sum_int(v, *red, f);
        if (threadIdx.x < kClusterBlocks) put(cs->i[f], v, threadIdx.x);
        sync();
        return __reduce_add_sync(0xffffffffu, lane < kClusterBlocks ? cs->i[f][lane] : 0);
    }
    // At most one state per thread: `part` is its value (n < kGameBatchedStates).
    template <typename U>
    __device__ double sum(double part, const U*, int64_t n) {
        const int f = turn(), lane = threadIdx.x & 31, w = threadIdx.x >> 5;
        cs->part[w][lane] = part;
        __syncthreads();
        if (w == 0) {
            double acc = 0.0;
            for (int k = 0; k < (int)((n + kThreads - 1) / kThreads); ++k) acc += cs->part[k][lane];
            acc = warp_sum(acc);
            if (lane < kClusterBlocks) put(cs->d[f], acc, (unsigned)lane);
        }
        sync();
        double v = lane < kClusterBlocks ? cs->d[f][lane] : 0.0;
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        return __shfl_sync(0xffffffffu, v, 0);
    }
    __device__ bool failed() const { return false; }
    __device__ bool leader() const { return blockIdx.x == 0 && threadIdx.x == 0; }
    __device__ bool own_copy() const { return false; }
    __device__ const float* gather_copy(const Game& G, const BatchOut& O, const double*) { return O.v32 + G.x0; }
};
static_assert(kGameBatchedStates <= kClusterBlocks * kThreads, "one state per thread");
static_assert(kClusterBlocks * 32 == kThreads, "a block's chunks are one warp's of a whole block");

// State of the policy evaluation: the last residual check's |r|_inf and
// |v|_inf and the sum of the system's row sums.
template <typename T>
struct Eval {
    double res, vm;
    T asum;
};

__device__ __forceinline__ unsigned long long abs_bits(double x) { return bits_of(x) & 0x7fffffffffffffffull; }

// One state's part of the residual check: r = rhs - (v - mu M v) (float64, Mv
// given) -> C.r.
template <typename T, class Ctx>
__device__ __forceinline__ double check_tail(const Game& G, const Ctx& C, int64_t i, double Mv, double vi, double rhs) {
    const double r = rhs - (vi - G.mu * Mv);
    T rt;
    if constexpr (sizeof(T) == 4) rt = f64_to_f32(r);
    else rt = r;
    C.r[i] = rt;
    return r;
}

// float64 residual check: fills E.res and E.vm.  fresh: the policies may have
// changed since the last check; changed rows are copied slot-major first and
// E.asum (the Galerkin operator of the constant vector) is formed.
template <typename T, int KC, class Ctx>
__device__ __noinline__ void check_k(const Game& G, const BatchOut& O, const double* v, Ctx& C, bool fresh,
                                     bool jacobi0, Eval<T>& E) {
    unsigned long long rm = 0, vm = 0;
    double part = 0.0;
    if (fresh) {
        for (int64_t i = C.begin(); i < G.n; i += C.stride()) {
            const int64_t row = O.sel[G.x0 + i];
            if constexpr (KC >= 0) {
                if (C.cp.cur[i] != row) compact_row<T, KC>(G, C.cp, i, row);
                part += C.cp.leak64[i];
            } else {
                const double l = G.T.leak[row];
                O.leaksel[G.x0 + i] = l;
                part += l;
            }
        }
    }
    auto take = [&](int64_t i, double Mv, double rhs) {
        const double vi = v[i];
        const unsigned long long rb = abs_bits(check_tail<T>(G, C, i, Mv, vi, rhs));
        const unsigned long long vb = abs_bits(vi);
        rm = rb > rm ? rb : rm;
        vm = vb > vm ? vb : vm;
    };
    if constexpr (KC == 8) {
        constexpr int D = 2;
        SlotRow8<double> R[D];
        double rhs[D];
        T dinv[D];
        const int64_t st = C.stride(), last = G.n - 1;
        auto fetch = [&](int d, int64_t i) {
            i = i < last ? i : last;
            R[d].load(C.cp.col, C.cp.p64, G.n, i);
            rhs[d] = O.rhs[G.x0 + i];
            dinv[d] = ((const T*)C.cp.dinv)[i];
        };
        int64_t i = C.begin();
#pragma unroll
        for (int d = 0; d < D; ++d) fetch(d, i + d * st);
        for (; i < G.n; i += D * st) {
#pragma unroll
            for (int d = 0; d < D; ++d) {
                const int64_t x = i + d * st;
                if (x < G.n) {
                    take(x, row_sum_r(R[d], v), rhs[d]);
                    C.e[x] = C.r[x] * dinv[d];
                }
                fetch(d, x + D * st);
            }
        }
    } else {
        for (int64_t i = C.begin(); i < G.n; i += C.stride()) {
            double Mv;
            if constexpr (KC >= 0) Mv = row_sum_c<KC>(C.cp, G.n, i, v);
            else Mv = row_sum(G, O.sel[G.x0 + i], v);
            take(i, Mv, O.rhs[G.x0 + i]);
            if constexpr (KC >= 0) C.e[i] = C.r[i] * ((const T*)C.cp.dinv)[i];
            else if (jacobi0) C.e[i] = C.r[i] / diag_row<T>(G, O, i);
        }
    }
    unsigned long long R, V;
    C.max2(rm, vm, &R, &V);
    E.res = from_bits(R);
    E.vm = from_bits(V);
    if (fresh && !C.failed())
        E.asum = (T)C.sum(part, KC >= 0 ? (const double*)C.cp.leak64 : (const double*)O.leaksel + G.x0, G.n);
}

template <typename T, class Ctx>
__device__ __forceinline__ void check(const Game& G, const BatchOut& O, const double* v, Ctx& C, bool fresh,
                                      bool jacobi0, Eval<T>& E) {
    if (C.cp.col == nullptr) check_k<T, -1>(G, O, v, C, fresh, jacobi0, E);
    else if (C.cp.K == 8) check_k<T, 8>(G, O, v, C, fresh, jacobi0, E);
    else check_k<T, 0>(G, O, v, C, fresh, jacobi0, E);
}

// One two-level cycle on A e = r from e = 0, then v += e.  Returns false if a
// grid barrier gave up.
template <typename T, class Ctx>
__device__ bool cycle(const Game& G, const BatchOut& O, double* v, Ctx& C, T asum, int nu1, int nu2) {
    // pre-relaxation (Jacobi; the first sweep from zero)
    for (int k = 0; k < nu1; ++k) {
        for (int64_t i = C.begin(); i < G.n; i += C.stride()) {
            if (k == 0) {
                C.t[i] = C.r[i] / diag_row<T>(G, O, i);
            } else {
                T Ae, d;
                apply_row<T>(G, O, i, C.e, &Ae, &d);
                C.t[i] = C.e[i] + (C.r[i] - Ae) / d;
            }
        }
        if (!C.sync()) return false;
        T* sw = C.e; C.e = C.t; C.t = sw;
    }
    if (nu1 == 0) {
        for (int64_t i = C.begin(); i < G.n; i += C.stride()) C.e[i] = 0;
        if (!C.sync()) return false;
    }
    // coarse correction on the constant vector: e += (1^T (r - A e)) / (1^T A 1)
    double part = 0.0;
    for (int64_t i = C.begin(); i < G.n; i += C.stride()) {
        T Ae, d;
        apply_row<T>(G, O, i, C.e, &Ae, &d);
        const T q = C.r[i] - Ae;
        C.t[i] = q;
        part += as_f64(q);
    }
    const double tot = C.sum(part, C.t, G.n);
    if (C.failed()) return false;
    const T c = asum != T(0) ? (T)(tot / (double)asum) : T(0);
    for (int64_t i = C.begin(); i < G.n; i += C.stride()) C.e[i] += c;
    if (!C.sync()) return false;
    // post-relaxation
    for (int k = 0; k < nu2; ++k) {
        for (int64_t i = C.begin(); i < G.n; i += C.stride()) {
            T Ae, d;
            apply_row<T>(G, O, i, C.e, &Ae, &d);
            C.t[i] = C.e[i] + (C.r[i] - Ae) / d;
        }
        if (!C.sync()) return false;
        T* sw = C.e; C.e = C.t; C.t = sw;
    }
    float* v32 = O.v32 + G.x0;
    for (int64_t i = C.begin(); i < G.n; i += C.stride()) {
        const double vi = v[i] + as_f64(C.e[i]);
        v[i] = vi;
        v32[i] = f64_to_f32(vi);
    }
    return C.sync();
}

// The same two-level cycle for one Jacobi sweep before and after the coarse
// correction, in two passes over the rows (the first sweep e1 = r / diag came
// with the residual check): A e1 gives the coarse correction c (e2 = e1 + c)
// and, since A 1 is the leakage s of each row, A e2 = A e1 + c s without
// another product; the post-sweep e = e2 + (r - A e2) / diag and v += e close
// the cycle.  Same iteration as cycle() with nu1 = nu2 = 1.
template <typename T, int KC, class Ctx>
__device__ __noinline__ bool cycle11_k(const Game& G, const BatchOut& O, double* v, Ctx& C, T asum) {
    double part = 0.0;
    const int64_t st = C.stride();
    auto put = [&](int64_t i, T q) {
        part += as_f64(q);
        C.r[i] = q;   // r - A e1 (r itself is not needed again)
    };
    if constexpr (KC == 8) {
        constexpr int D = sizeof(T) == 4 ? 3 : 2;
        SlotRow8<T> R[D];
        T leak[D];
        const int64_t last = G.n - 1;
        auto fetch = [&](int d, int64_t i) {
            i = i < last ? i : last;
            R[d].load(C.cp.col, slot_p(C.cp, T()), G.n, i);
            leak[d] = slot_leak(C.cp, T())[i];
        };
        int64_t i = C.begin();
#pragma unroll
        for (int d = 0; d < D; ++d) fetch(d, i + d * st);
        for (; i < G.n; i += D * st) {
#pragma unroll
            for (int d = 0; d < D; ++d) {
                const int64_t x = i + d * st;
                if (x < G.n) put(x, C.r[x] - apply_row_r(G, R[d], leak[d], C.e[x], C.e));
                fetch(d, x + D * st);
            }
        }
    } else {
        for (int64_t i = C.begin(); i < G.n; i += st) {
            if constexpr (KC >= 0) {
                put(i, C.r[i] - apply_row_c<KC>(G, C.cp, i, C.e));
            } else {
                T Ae, d;
                apply_row<T>(G, O, i, C.e, &Ae, &d);
                C.t[i] = d;
                put(i, C.r[i] - Ae);
            }
        }
    }
    const double tot = C.sum(part, C.r, G.n);
    if (C.failed()) return false;
    const T c = asum != T(0) ? (T)(tot / (double)asum) : T(0);
    // the improvement gathers from the context's own copy of v where it has one
    float* v32 = C.own_copy() && rows_in_lanes(G.T.m1, G.T.m2) ? nullptr : O.v32 + G.x0;
    auto close = [&](int64_t i, T e) {
        const double vi = v[i] + as_f64(e);
        v[i] = vi;
        if (v32) v32[i] = f64_to_f32(vi);
    };
    if constexpr (KC >= 0) {
        constexpr int B = 4;   // states whose loads are issued together
        const T* leak = slot_leak(C.cp, T());
        const T* dinv = (const T*)C.cp.dinv;
        for (int64_t i = C.begin(); i < G.n; i += B * st) {
            T s[B], w[B];
#pragma unroll
            for (int k = 0; k < B; ++k) {
                const int64_t x = i + k * st;
                if (x < G.n) {
                    s[k] = leak[x];
                    w[k] = dinv[x];
                }
            }
#pragma unroll
            for (int k = 0; k < B; ++k) {
                const int64_t x = i + k * st;
                if (x < G.n) close(x, C.e[x] + c + (C.r[x] - c * s[k]) * w[k]);
            }
        }
    } else {
        for (int64_t i = C.begin(); i < G.n; i += st) {
            const int64_t row = O.sel[G.x0 + i];
            const T s = sizeof(T) == 4 ? (T)G.T.leak32[row] : (T)G.T.leak[row];
            close(i, C.e[i] + c + (C.r[i] - c * s) / C.t[i]);
        }
    }
    return C.sync();
}

template <typename T, class Ctx>
__device__ __forceinline__ bool cycle11(const Game& G, const BatchOut& O, double* v, Ctx& C, T asum) {
    if (C.cp.col == nullptr) return cycle11_k<T, -1>(G, O, v, C, asum);
    if (C.cp.K == 8) return cycle11_k<T, 8>(G, O, v, C, asum);
    return cycle11_k<T, 0>(G, O, v, C, asum);
}

// Why a policy evaluation stopped.
enum { kEvalExact = 0, kEvalInexact = 1, kEvalCapped = 2 };

// Policy evaluation: cycles until the float64 floor / tolerance (kEvalExact),
// a residual drop by rel_tol (kEvalInexact) or max_cycles (kEvalCapped).
// checked: E and the correction vectors hold the check of the current v and
// policies already (the last evaluation's, or the outer improvement's).
template <typename T, class Ctx>
__device__ int evaluate(const Game& G, const BatchOut& O, const BatchOpts& P, double* v, Ctx& C, bool checked,
                        double rel_tol, int* cycles, Eval<T>& E) {
    const bool v11 = P.nu1 == 1 && P.nu2 == 1;
    if (!checked) check<T>(G, O, v, C, true, v11, E);
    const double res0 = E.res;
    double prev = E.res;
    int slow = 0;
    for (int cyc = 0;; ++cyc) {
        if (C.failed()) return kEvalExact;   // a barrier gave up: the caller leaves
        if (E.res <= P.lin_tol * fmax(E.vm, 1e-300) || E.res == 0.0) return kEvalExact;
        if (cyc > 0) {
            slow = E.res > 0.5 * prev ? slow + 1 : 0;
            if (slow >= 2 && E.res < 1e-12 * fmax(E.vm, 1e-300)) return kEvalExact;
            if (E.res <= rel_tol * res0) return kEvalInexact;
            prev = fmin(prev, E.res);
        }
        if (cyc >= P.max_cycles) return kEvalCapped;
        if (!(v11 ? cycle11<T>(G, O, v, C, E.asum) : cycle<T>(G, O, v, C, E.asum, P.nu1, P.nu2)))
            return kEvalExact;
        ++*cycles;
        check<T>(G, O, v, C, false, v11, E);
    }
}

// Policy improvement of the whole game; vm is |v|_inf.  Returns the number of
// changed policy entries; every thread of the context has passed a barrier
// after the last write.
template <class Ctx>
__device__ int improve_all(const Game& G, const BatchOut& O, int mode, const double* v, double vm, Ctx& C) {
    const double tau = 1e-13 * fmax(1.0, vm);
    const float vmaxf = f64_to_f32(vm);
    int changed = 0;
    if (rows_in_lanes(G.T.m1, G.T.m2)) {
        const float* v32 = C.gather_copy(G, O, v);
        const bool wide = G.T.k_uniform == 8;
        if (mode == 1) changed = wide ? improve_rows<8, 1>(G, O, tau, vmaxf, v, v32, C)
                                      : improve_rows<0, 1>(G, O, tau, vmaxf, v, v32, C);
        else if (mode == 0) changed = wide ? improve_rows<8, 0>(G, O, tau, vmaxf, v, v32, C)
                                           : improve_rows<0, 0>(G, O, tau, vmaxf, v, v32, C);
        else changed = wide ? improve_rows<8, 2>(G, O, tau, vmaxf, v, v32, C)
                            : improve_rows<0, 2>(G, O, tau, vmaxf, v, v32, C);
    } else {
        const float tauf = f64_to_f32(tau);
        for (int64_t i = C.begin(); i < G.n; i += C.stride()) {
            double r;
            changed += improve_state(G, O, mode, i, tau, tauf, vmaxf, v, &r);
        }
    }
    return C.sumi(changed);
}

// Algorithm 2 with Algorithm 1 inside for game g (see the Isaacs driver for
// the stopping rules and the exact confirmation of inexact evaluations).
// |F(v) - v| of an outer improvement is the residual of the system its
// policies select, so it comes from that system's first residual check.
template <typename T, class Ctx>
__device__ void solve_game(const BatchArgs& B, int g, Ctx& C, double* vs) {
    Game G;
    G.T = B.T;
    G.x0 = B.st_off[g];
    G.n = B.st_off[g + 1] - G.x0;
    G.R = B.T.m1 * B.T.m2;
    G.row0 = G.x0 * G.R;
    G.mu = B.mu[g];
    G.mu_f = f64_to_f32(G.mu);
    const BatchOut& O = B.out;
    const BatchOpts& P = B.opt;
    const bool v11 = P.nu1 == 1 && P.nu2 == 1;
    if (!v11) C.cp.col = nullptr;   // the general cycle reads the rows in place
    double* v = vs ? vs : O.v + G.x0;
    const int a0 = P.default_alpha;
    for (int64_t i = C.begin(); i < G.n; i += C.stride()) {
        v[i] = 0.0;
        O.v32[G.x0 + i] = 0.0f;
        O.alpha[G.x0 + i] = (uint8_t)(a0 < G.T.m1 ? a0 : 0);
        for (int a = 0; a < G.T.m1; ++a) O.beta[(G.x0 + i) * G.T.m1 + a] = 0;
        if (C.cp.col) C.cp.cur[i] = -1;
    }
    if (!C.sync()) return;
    improve_all(G, O, 2, v, 0.0, C);   // MIN's first reply, assembly
    if (C.failed()) return;
    int outer = 0, systems = 0, cycles = 0, converged = 0;
    bool capped = false;   // an evaluation stopped at max_cycles: no decision may rest on it
    bool checked = false;
    Eval<T> E{0.0, 0.0, T(0)};
    while (true) {
        for (int j = 0; j < P.max_inner; ++j) {
            const int why = evaluate<T>(G, O, P, v, C, checked, P.pi_rtol, &cycles, E);
            checked = true;
            ++systems;
            if (C.failed()) return;
            if (why == kEvalCapped) {
                capped = true;
                break;
            }
            const int ch = improve_all(G, O, 1, v, E.vm, C);
            if (C.failed()) return;
            if (ch != 0) {
                checked = false;
                continue;
            }
            if (why == kEvalInexact) {
                if (evaluate<T>(G, O, P, v, C, true, 0.0, &cycles, E) == kEvalCapped) capped = true;
                if (C.failed()) return;
                if (capped) break;
                const int ch2 = improve_all(G, O, 1, v, E.vm, C);
                if (C.failed()) return;
                if (ch2 != 0) {
                    checked = false;
                    continue;
                }
            }
            break;
        }
        ++outer;
        const int ach = improve_all(G, O, 0, v, E.vm, C);
        if (C.failed()) return;
        check<T>(G, O, v, C, true, v11, E);
        if (C.failed()) return;
        checked = true;
        if (capped) break;   // unconverged; v is the best iterate, E.res its residual
        if (E.res <= P.eps || ach == 0) {
            converged = 1;
            break;
        }
        if (outer >= P.max_outer) break;
    }
    if (vs)
        for (int64_t i = C.begin(); i < G.n; i += C.stride()) O.v[G.x0 + i] = v[i];
    if (C.leader()) {
        O.gstats[4 * g + 0] = outer;
        O.gstats[4 * g + 1] = systems;
        O.gstats[4 * g + 2] = cycles;
        O.gstats[4 * g + 3] = converged;
        O.gres[g] = E.res;
    }
    C.sync();
}

// One thread block of NT threads per game; blocks take games from the queue
// in the order B.order gives (512 / NT blocks per SM fit the registers).
template <typename T, int NT>
__global__ void __launch_bounds__(NT, 512 / NT) k_games_pi(const __grid_constant__ BatchArgs B) {
    extern __shared__ __align__(16) char smem[];
    __shared__ int s_game;
    __shared__ RedScratch red;
    while (true) {
        if (threadIdx.x == 0) {
            const int q = atomicAdd(B.queue, 1);
            s_game = q < B.count ? B.order[q] : -1;
        }
        __syncthreads();
        const int g = s_game;
        __syncthreads();
        if (g < 0) break;
        BlockCtx<T> C;
        double* vs = B.v_in_smem ? (double*)smem : nullptr;
        C.r = (T*)(smem + (vs ? sizeof(double) * (size_t)B.max_n : 0));
        C.e = C.r + B.max_n;
        C.t = C.e + B.max_n;
        C.red = &red;
        if (B.cp.col) {   // this game's part of the slot-major rows
            const int64_t x0 = B.st_off[g], K = B.cp.K;
            C.cp = Compact{B.cp.col + x0 * K, B.cp.p32 + x0 * K, B.cp.p64 + x0 * K, B.cp.leak32 + x0,
                           B.cp.leak64 + x0, B.cp.dinv + x0, B.cp.cur + x0, B.cp.K};
        }
        solve_game<T>(B, g, C, vs);
    }
}

// One game over a cooperative grid.
template <typename T>
__global__ void __launch_bounds__(kThreads) k_game_pi_grid(const __grid_constant__ BatchArgs B,
                                                           GridWork W) {
    __shared__ RedScratch red;
    GridCtx<T> C;
    C.r = (T*)W.r;
    C.e = (T*)W.e;
    C.t = (T*)W.t;
    C.part = W.part;
    C.gs = W.gs;
    C.cp = W.cp;
    C.red = &red;
    C.flip = 0;
    C.slot = 0;
    C.bad = false;
    solve_game<T>(B, 0, C, nullptr);
}

// One game over one cluster.
template <typename T>
__global__ void __launch_bounds__(kThreads) k_game_pi_cluster(const __grid_constant__ BatchArgs B, GridWork W) {
    __shared__ RedScratch red;
    __shared__ ClusterScratch cs;
    ClusterCtx<T> C;
    C.r = (T*)W.r;
    C.e = (T*)W.e;
    C.t = (T*)W.t;
    C.cp = W.cp;
    C.red = &red;
    C.cs = &cs;
    C.flip = 0;
    C.sync();   // every block has started: its shared memory may be written
    solve_game<T>(B, 0, C, nullptr);
    C.sync();   // no block leaves while others may still write to it
}

// One policy improvement of game 0 over the whole grid (the algebraic
// multigrid path runs policy iteration from the host): keep-current
// tolerance from |v|_inf (bits at scal + 4), changed entries summed into
// scal[0], |F(v) - v|_inf (outer mode) as bits at scal + 2.
__global__ void k_game_improve_one(const __grid_constant__ BatchArgs B, int mode, int* scal) {
    Game G;
    G.T = B.T;
    G.x0 = 0;
    G.n = B.st_off[1];
    G.R = B.T.m1 * B.T.m2;
    G.row0 = 0;
    G.mu = B.mu[0];
    G.mu_f = f64_to_f32(G.mu);
    const double vm = from_bits(*reinterpret_cast<const unsigned long long*>(scal + 4));
    const double tau = 1e-13 * fmax(1.0, vm);
    const float tauf = f64_to_f32(tau), vmaxf = f64_to_f32(vm);
    int changed = 0;
    unsigned long long rb = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < G.n;
         i += (int64_t)gridDim.x * blockDim.x) {
        double r = 0.0;
        changed += improve_state(G, B.out, mode, i, tau, tauf, vmaxf, B.out.v, &r);
        const unsigned long long b = bits_of(r);
        rb = b > rb ? b : rb;
    }
    changed = warp_sum(changed);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long w = __shfl_xor_sync(0xffffffffu, rb, o);
        rb = w > rb ? w : rb;
    }
    if ((threadIdx.x & 31) == 0) {
        if (changed) atomicAdd(scal, changed);
        atomicMax(reinterpret_cast<unsigned long long*>(scal + 2), rb);
    }
}

}  // namespace

void launch_game_improve_one(const BatchArgs& B, int mode, int64_t n, int* scal, cudaStream_t st) {
    const unsigned g = (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 152 * 8));
    k_game_improve_one<<<g, 256, 0, st>>>(B, mode, scal);
    GS_CHECK_LAUNCH();
}

void launch_game_validate(const GameTables& T, int count, const int64_t* st_off, int64_t rows,
                          int* bad, cudaStream_t st) {
    const unsigned g = (unsigned)std::min<int64_t>((rows + 255) / 256, 152 * 32);
    k_game_validate<<<std::max(1u, g), 256, 0, st>>>(T, count, st_off, bad);
    GS_CHECK_LAUNCH();
}

void launch_game_prepare(const GameTables& T, int count, const int64_t* st_off, int64_t rows,
                         const double* mu, double* leak, float* leak32, float* prob32,
                         __nv_bfloat16* prob16, cudaStream_t st) {
    const unsigned g = (unsigned)std::min<int64_t>((rows + 255) / 256, 152 * 32);
    k_game_prepare<<<std::max(1u, g), 256, 0, st>>>(T, count, st_off, mu, leak, leak32, prob32, prob16);
    GS_CHECK_LAUNCH();
}

int game_grid_blocks(int64_t n, int cap) {
    static PerDevice<int64_t> resident;
    const int dev = current_device();
    const int64_t all = resident.get(dev, [&] {
        int a = 0, b = 0;
        GS_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, k_game_pi_grid<float>, kThreads, 0));
        GS_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_game_pi_grid<double>, kThreads, 0));
        return (int64_t)std::max(1, std::min(a, b)) * sm_count(dev);
    });
    // one warp of states per block until every SM has one
    int blocks = (int)std::min<int64_t>((n + 31) / 32, all);
    if (cap > 0) blocks = std::min(blocks, cap);
    return std::max(1, blocks);
}

// Dynamic shared memory a block of the one-block kernel may take; what an SM has,
// and what each block takes of it besides (its static arrays and the system's).
constexpr size_t kGameSmemMax = 224 * 1024, kSmemPerSM = 228 * 1024, kGameSmemBeside = 3 * 1024;

// Whether one cluster of the cluster kernel fits the current device.
static bool cluster_fits(const void* fn, bool mixed) {
    static PerDevice<bool> fits[2];
    return fits[mixed ? 1 : 0].get(current_device(), [&] {
        cudaLaunchConfig_t cfg{};
        cudaLaunchAttribute at{};
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = kClusterBlocks;
        at.val.clusterDim.y = at.val.clusterDim.z = 1;
        cfg.gridDim = dim3(kClusterBlocks);
        cfg.blockDim = dim3(kThreads);
        cfg.attrs = &at;
        cfg.numAttrs = 1;
        int count = 0;
        const bool ok = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
                        cudaOccupancyMaxActiveClusters(&count, fn, &cfg) == cudaSuccess && count > 0;
        cudaGetLastError();
        return ok;
    });
}

void launch_game_pi_grid(const BatchArgs& B, const GridWork& W, int blocks, bool mixed,
                         cudaStream_t st) {
    // games small enough to be batched: one cluster, unless the caller's cap on
    // the blocks is below it
    const void* cl = mixed ? (const void*)k_game_pi_cluster<float> : (const void*)k_game_pi_cluster<double>;
    if (B.max_n < kGameBatchedStates && blocks >= kClusterBlocks && cluster_fits(cl, mixed)) {
        void* args[] = {(void*)&B, (void*)&W};
        cudaLaunchConfig_t cfg{};
        cudaLaunchAttribute at{};
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = kClusterBlocks;
        at.val.clusterDim.y = at.val.clusterDim.z = 1;
        cfg.gridDim = dim3(kClusterBlocks);
        cfg.blockDim = dim3(kThreads);
        cfg.stream = st;
        cfg.attrs = &at;
        cfg.numAttrs = 1;
        GS_CUDA(cudaLaunchKernelExC(&cfg, cl, args));
        note_launches(1);
        return;
    }
    const void* fn = mixed ? (const void*)k_game_pi_grid<float> : (const void*)k_game_pi_grid<double>;
    void* args[] = {(void*)&B, (void*)&W};
    GS_CUDA(cudaLaunchCooperativeKernel(fn, dim3(blocks), dim3(kThreads), args, 0, st));
    note_launches(1);
}

size_t games_smem_bytes(int max_n, bool mixed, bool v_in_smem) {
    return (size_t)max_n * (3 * (mixed ? sizeof(float) : sizeof(double)) + (v_in_smem ? sizeof(double) : 0));
}

void launch_games_pi(const BatchArgs& Bin, bool mixed, int threads, cudaStream_t st) {
    // the iterate joins the correction vectors in shared memory where all
    // 512 / threads blocks of an SM still fit (304 games of 5700 states, mixed, 256
    // threads: 25.9 ms beside one another with the iterate outside, 33.5 ms one by one)
    BatchArgs B = Bin;
    const size_t with_v = games_smem_bytes(B.max_n, mixed, true);
    B.v_in_smem = with_v <= kGameSmemMax && (with_v + kGameSmemBeside) * (512 / threads) <= kSmemPerSM;
    const size_t smem = games_smem_bytes(B.max_n, mixed, B.v_in_smem);
    const void* fn = threads == 256 ? (mixed ? (const void*)k_games_pi<float, 256>
                                             : (const void*)k_games_pi<double, 256>)
                                    : (mixed ? (const void*)k_games_pi<float, 512>
                                             : (const void*)k_games_pi<double, 512>);
    const int nt = threads == 256 ? 256 : 512;
    static PerDevice<int> sms_of[4];
    const int dev = current_device();
    // (the limit, not this launch's size: another thread's launch may be between the two)
    const int sms = sms_of[(threads == 256) * 2 + mixed].get(dev, [&] {
        GS_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGameSmemMax));
        return sm_count(dev);
    });
    int per_sm = 0;
    GS_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, nt, smem));
    const int blocks = std::max(1, std::min(B.count, std::max(1, per_sm) * sms));
    void* args[] = {(void*)&B};
    GS_CUDA(cudaLaunchKernel(fn, dim3(blocks), dim3(nt), args, smem, st));
    note_launches(1);
}

}  // namespace gs
