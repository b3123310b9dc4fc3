// Phases of the finest level of a mixed V-cycle (5-point rows given by policy
// codes, float32 correction u, right-hand side f) in wide accesses.
//
// u and f have side + 1 = 2^k elements per row between zeros on every side, so
// rows are aligned, a point's neighbours outside the grid read zero, and the
// index arithmetic is shifts.  A thread block owns a run of whole rows in every
// phase.  An item is eight consecutive points of a row: 16-byte loads of the
// rows around it, four points of one colour updated, two 16-byte stores; the
// weights of a policy code come from a table in shared memory.  Bound by the
// latency of one round of loads from L2 and the grid barrier between phases (at
// 1023^2), by HBM and the float64 pipe where the vectors leave the L2 (2047^2).
// Measured at 1023^2 against one scalar access per neighbour, integer division,
// bounds tests and a division per point: a cycle's phases of the finest level
// 89 -> 75 us (prolongation and first colour 14.9 -> 11.0, restriction 12.4 ->
// 9.4, last colour with v += e 13.0 -> 9.9, residual check 17.6 -> 15.9 us); a
// 2047^2 solve 24.7 -> 22.0 ms.
#pragma once

#include "fine_stage.h"
#include "mgsolve.cuh"
#include "stencil.cuh"

namespace gs {

// Weights of one policy code: w = minus the couplings (W, E, S, N), the inverse
// diagonal (rounded once from its float64 value; the residual these corrections
// answer is formed in float64 with the exact rows) and the row sum.
struct FineTab {
    float4 w[kCodes];
    float dinv[kCodes], s[kCodes];
};

// Whether the wide phases take a grid: rows of at least 8 elements.
__host__ __device__ __forceinline__ bool fine_wide(int side) { return side >= 7; }

__device__ __forceinline__ void fine_tab_fill(FineTab& T, const IsaacsConsts* K) {
    for (int c = threadIdx.x; c < kCodes; c += blockDim.x) {
        T.w[c] = make_float4(-K->amf[c][1], -K->amf[c][2], -K->amf[c][3], -K->amf[c][4]);
        T.dinv[c] = (float)K->am0inv[c];
        T.s[c] = c == kStopCode ? 1.0f : K->kappa_f;
    }
}

struct FineView {
    float *u, *f;            // grid point (0, 0)
    const uint8_t* code;
    int side, P, lg;         // P = side + 1 = 2^lg elements per row
    __device__ explicit FineView(const SolveArgs& a)
        : u((float*)a.L[0].u), f((float*)a.L[0].f), code(a.code), side(a.L[0].side), P(a.L[0].side + 1),
          lg(a.lg0) {}
    __device__ __forceinline__ bool last(int q) const { return 8 * q + 8 == P; }   // the row's last octet
};

// Rows [r0, r1) of n of this block.
__device__ __forceinline__ void block_rows(int n, int* r0, int* r1) {
    *r0 = (int)((long long)n * blockIdx.x / gridDim.x);
    *r1 = (int)((long long)n * (blockIdx.x + 1) / gridDim.x);
}

// Eight points of a row with what a colour update or residual needs.
struct Octet {
    float o[10];             // u at -1 .. 8 of the row
    float s[8], n[8], f[8];
    unsigned long long code;
    __device__ __forceinline__ void load(const FineView& V, int j, int q) {
        const size_t x = (size_t)j * V.P + 8 * q;
        const float *u = V.u + x, *g = V.f + x;
        o[0] = u[-1];
        o[9] = u[8];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float4 a = ((const float4*)u)[h], b = ((const float4*)(u - V.P))[h],
                         c = ((const float4*)(u + V.P))[h], d = ((const float4*)g)[h];
            o[1 + 4 * h] = a.x; o[2 + 4 * h] = a.y; o[3 + 4 * h] = a.z; o[4 + 4 * h] = a.w;
            s[4 * h] = b.x; s[1 + 4 * h] = b.y; s[2 + 4 * h] = b.z; s[3 + 4 * h] = b.w;
            n[4 * h] = c.x; n[1 + 4 * h] = c.y; n[2 + 4 * h] = c.z; n[3 + 4 * h] = c.w;
            f[4 * h] = d.x; f[1 + 4 * h] = d.y; f[2 + 4 * h] = d.z; f[3 + 4 * h] = d.w;
        }
        code = *(const unsigned long long*)(V.code + x);
    }
    // The points k = par, par + 2, .. are chosen by selects: one code for both
    // parities (the kernel runs each phase once per cycle, and its instructions
    // must stay in the instruction cache).
    __device__ __forceinline__ void relax(const FineTab& T, bool par) {
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const int c = (int)(code >> (16 * m + (par ? 8 : 0))) & 0xff;
            const float4 w = T.w[c];
            const float W = par ? o[2 * m + 1] : o[2 * m], E = par ? o[2 * m + 3] : o[2 * m + 2];
            const float S = par ? s[2 * m + 1] : s[2 * m], N = par ? n[2 * m + 1] : n[2 * m];
            const float g = par ? f[2 * m + 1] : f[2 * m];
            const float v = (g + w.x * W + w.y * E + w.z * S + w.w * N) * T.dinv[c];
            if (par) o[2 * m + 2] = v;
            else o[2 * m + 1] = v;
        }
    }
    // Residuals of those points in the leakage form: f - s u + sum_d w_d (u_d - u).
    __device__ __forceinline__ float4 resid(const FineTab& T, bool par) const {
        float r[4];
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const int c = (int)(code >> (16 * m + (par ? 8 : 0))) & 0xff;
            const float4 w = T.w[c];
            const float x = par ? o[2 * m + 2] : o[2 * m + 1];
            const float W = par ? o[2 * m + 1] : o[2 * m], E = par ? o[2 * m + 3] : o[2 * m + 2];
            const float S = par ? s[2 * m + 1] : s[2 * m], N = par ? n[2 * m + 1] : n[2 * m];
            const float g = par ? f[2 * m + 1] : f[2 * m];
            r[m] = g - T.s[c] * x + w.x * (W - x) + w.y * (E - x) + w.z * (S - x) + w.w * (N - x);
        }
        return make_float4(r[0], r[1], r[2], r[3]);
    }
    // The eight values of u.  last: the row's last octet, whose eighth element lies
    // outside the grid and stays zero whatever its neighbours hold: an iterate
    // that is not finite must not reach the padding, which no launch clears.
    __device__ __forceinline__ void store(float* p, bool last) const {
        ((float4*)p)[0] = make_float4(o[1], o[2], o[3], o[4]);
        ((float4*)p)[1] = make_float4(o[5], o[6], o[7], last ? 0.0f : o[8]);
    }
};

// Runs f(j, q, octet) for the octets of rows [r0, r1), the next one's loads on
// their way (f updates only points its neighbours' octets do not read).
template <class F>
__device__ __forceinline__ void for_octets(const FineView& V, int r0, int r1, F&& f) {
    const int lq = V.lg - 3, cnt = (r1 - r0) << lq, mask = (1 << lq) - 1;
    int t = threadIdx.x;
    if (t >= cnt) return;
    Octet next;
    next.load(V, r0 + (t >> lq), t & mask);
#pragma unroll 1
    for (; t < cnt; t += blockDim.x) {
        Octet A = next;
        const int t2 = t + blockDim.x < cnt ? t + blockDim.x : t;
        next.load(V, r0 + (t2 >> lq), t2 & mask);
        f(r0 + (t >> lq), t & mask, A);
    }
}

// One colour of the red-black relaxation (colour 0: i + j even).
__device__ __noinline__ void fine_relax_wide(const SolveArgs& a, const FineTab& T, int c) {
    const FineView V(a);
    int r0, r1;
    block_rows(V.side, &r0, &r1);
    for_octets(V, r0, r1, [&](int j, int q, Octet& O) {
        O.relax(T, (j + c) & 1);
        O.store(V.u + (size_t)j * V.P + 8 * q, V.last(q));
    });
}

// The last colour of the last relaxation with the float64 update v += e: the
// rows' corrections pass through shared memory so that v, whose rows are not
// aligned, is updated by consecutive threads.
__device__ __noinline__ void fine_update_wide(const SolveArgs& a, const FineTab& T, int c, float* stage) {
    const FineView V(a);
    double* __restrict__ v = a.v;
    int r0, r1;
    block_rows(V.side, &r0, &r1);
    const int chunk = fine_update_chunk(V.side);
    for (; r0 < r1; r0 += chunk) {
        const int re = min(r1, r0 + chunk);
        for_octets(V, r0, re, [&](int j, int q, Octet& O) {
            O.relax(T, (j + c) & 1);
            O.store(V.u + (size_t)j * V.P + 8 * q, V.last(q));
            O.store(stage + ((j - r0) << V.lg) + 8 * q, V.last(q));
        });
        __syncthreads();
        constexpr int B = 4;
        const int cnt = (re - r0) << V.lg;
#pragma unroll 1
        for (int t = threadIdx.x; t < cnt; t += B * blockDim.x) {
            double w[B];
            double* p[B];
#pragma unroll
            for (int b = 0; b < B; ++b) {
                const int x = t + b * blockDim.x, i = x & (V.P - 1), j = r0 + (x >> V.lg);
                p[b] = x < cnt && i < V.side ? v + (size_t)j * V.side + i : nullptr;
                if (p[b]) w[b] = *p[b];
            }
#pragma unroll
            for (int b = 0; b < B; ++b)
                if (p[b]) *p[b] = w[b] + f32_to_f64(stage[t + b * blockDim.x]);
        }
        __syncthreads();
    }
}

// Four consecutive interpolation weights, widened.
__device__ __forceinline__ float4 wide4(const float* p) { return *(const float4*)p; }
__device__ __forceinline__ float4 wide4(const __nv_bfloat16* p) {
    const uint2 b = *(const uint2*)p;
    return make_float4(__uint_as_float(b.x << 16), __uint_as_float(b.x & 0xffff0000u), __uint_as_float(b.y << 16),
                       __uint_as_float(b.y & 0xffff0000u));
}

// u += P u_c at the colour-1 (edge) points, four cells (eight points of two
// rows) per item; the colour-0 values are overwritten, unread, by the
// relaxation that follows.  uc: the first coarse level's u, side sc, dense.
template <typename W>
__device__ __noinline__ void fine_prolong_wide(const SolveArgs& a, const float* __restrict__ uc) {
    const FineView V(a);
    const W* __restrict__ Pw = (const W*)a.L[0].P;
    const int sc = a.L[0].sc, nc1 = sc + 1, lq = V.lg - 3, mask = (1 << lq) - 1;
    const size_t ncell = (size_t)nc1 * nc1;
    int r0, r1;
    block_rows(nc1, &r0, &r1);
    const int cnt = (r1 - r0) << lq;
    for (int t = threadIdx.x; t < cnt; t += blockDim.x) {
        const int J = r0 + (t >> lq), q = t & mask, I0 = 4 * q;
        const size_t c = (size_t)J * nc1 + I0;
        float lo[4], hi[5];   // u_c at (I0 .. I0 + 3, J - 1) and (I0 - 1 .. I0 + 3, J)
#pragma unroll
        for (int k = 0; k < 4; ++k) lo[k] = J > 0 && I0 + k < sc ? uc[(size_t)(J - 1) * sc + I0 + k] : 0.0f;
#pragma unroll
        for (int k = 0; k < 5; ++k) hi[k] = J < sc && I0 + k > 0 && I0 + k - 1 < sc ? uc[(size_t)J * sc + I0 + k - 1] : 0.0f;
        const float4 s = wide4(Pw + PYS * ncell + c), n = wide4(Pw + PYN * ncell + c);
        float* y = V.u + (size_t)(2 * J) * V.P + 8 * q;   // y-edges: odd i of row 2J
        float4 y0 = ((float4*)y)[0], y1 = ((float4*)y)[1];
        y0.y += s.x * lo[0] + n.x * hi[1];
        y0.w += s.y * lo[1] + n.y * hi[2];
        y1.y += s.z * lo[2] + n.z * hi[3];
        if (I0 + 3 < sc) y1.w += s.w * lo[3] + n.w * hi[4];
        ((float4*)y)[0] = y0;
        ((float4*)y)[1] = y1;
        if (J < sc) {
            const float4 w = wide4(Pw + PXW * ncell + c), e = wide4(Pw + PXE * ncell + c);
            float* x = y + V.P;                           // x-edges: even i of row 2J + 1
            float4 x0 = ((float4*)x)[0], x1 = ((float4*)x)[1];
            x0.x += w.x * hi[0] + e.x * hi[1];
            x0.z += w.y * hi[1] + e.y * hi[2];
            x1.x += w.z * hi[2] + e.z * hi[3];
            x1.z += w.w * hi[3] + e.w * hi[4];
            ((float4*)x)[0] = x0;
            ((float4*)x)[1] = x1;
        }
    }
}

// f_1 = R (f - A u) after at least one pre-smoothing sweep: the sweep ends with
// colour 1, whose residuals it has made zero up to rounding, so only the
// colour-0 points' residuals (C points and corners) are formed, each once, in
// shared memory.  first: also u_1's first colour from zero (f_1 / diagonal at
// its C points, zero elsewhere); otherwise u_1 is cleared where clear is set.
template <typename W>
__device__ __noinline__ void fine_restrict_wide(const SolveArgs& a, const FineTab& T, bool first, bool clear, float* r) {
    const FineView V(a);
    const LevelArgs& C = a.L[1];
    const W* __restrict__ Pw = (const W*)a.L[0].P;
    const int sc = a.L[0].sc, nc1 = sc + 1, lh = V.lg - 1, H = 1 << lh;   // H values per row
    const size_t ncell = (size_t)nc1 * nc1;
    const L9Op<float, W> cop{(const W*)C.A, C.n, C.side};
    float* __restrict__ fc = (float*)C.f;
    float* __restrict__ uc = (float*)C.u;
    int J0, J1;
    block_rows(sc, &J0, &J1);
    const int chunk = fine_restrict_chunk(V.side);
    for (; J0 < J1; J0 += chunk) {
        const int Je = min(J1, J0 + chunk), j0 = 2 * J0, j1 = 2 * Je + 1;
        for_octets(V, j0, j1, [&](int j, int q, Octet& O) {
            *(float4*)(r + ((j - j0) << lh) + 4 * q) = O.resid(T, j & 1);
        });
        __syncthreads();
        const int cnt = (Je - J0) << lh;
        for (int t = threadIdx.x; t < cnt; t += blockDim.x) {
            const int I = t & (H - 1), J = J0 + (t >> lh);
            if (I >= sc) continue;
            const size_t c = (size_t)J * nc1 + I;
            const float* row = r + ((2 * (J - J0)) << lh) + I;   // corner row 2J
            const float acc = row[H] + wval(Pw[PNE * ncell + c]) * row[0] + wval(Pw[PNW * ncell + c + 1]) * row[1] +
                              wval(Pw[PSE * ncell + c + nc1]) * row[2 * H] +
                              wval(Pw[PSW * ncell + c + nc1 + 1]) * row[2 * H + 1];
            const size_t x = (size_t)J * sc + I;
            fc[x] = acc;
            if (first) uc[x] = I & J & 1 ? acc / cop.diag(I, J) : 0.0f;
            else if (clear) uc[x] = 0.0f;
        }
        __syncthreads();
    }
}

// float64 residual r = rhs - A v with |r|_inf and |v|_inf; r rounded to float32
// is the correction's right-hand side, and with first its first relaxation
// colour from zero (e = r / diagonal at the colour-0 points) is formed, else
// the correction is cleared.  K: the constants in shared memory.
__device__ __forceinline__ void fine_check_rows(const SolveArgs& a, const IsaacsConsts& K, const FineTab& T, bool first,
                                                int r0, int r1, unsigned long long* rmax, unsigned long long* vmax) {
    const FineView V(a);
    const double *__restrict__ v = a.v, *__restrict__ rhs = a.rhs;
    const int side = V.side, cnt = (r1 - r0) << V.lg;
    unsigned long long rm = 0, vm = 0;
    constexpr int B = 2;
#pragma unroll 1
    for (int t0 = threadIdx.x; t0 < cnt; t0 += B * blockDim.x) {
        double c[B], w[B], e[B], s[B], n[B], f[B];
        int code[B];
        bool ok[B];
#pragma unroll
        for (int b = 0; b < B; ++b) {
            const int t = t0 + b * blockDim.x, i = t & (V.P - 1), j = r0 + (t >> V.lg);
            ok[b] = t < cnt && i < side;
            const size_t x = ok[b] ? (size_t)j * side + i : 0;
            code[b] = ok[b] ? V.code[((size_t)j << V.lg) + i] : kStopCode;
            c[b] = load_or_zero(v, x, ok[b]);
            w[b] = load_or_zero(v, x - 1, ok[b] && i > 0);
            e[b] = load_or_zero(v, x + 1, ok[b] && i + 1 < side);
            s[b] = load_or_zero(v, x - side, ok[b] && j > 0);
            n[b] = load_or_zero(v, x + side, ok[b] && j + 1 < side);
            f[b] = load_or_zero(rhs, x, ok[b]);
        }
#pragma unroll
        for (int b = 0; b < B; ++b) {
            const double* am = K.am[code[b]];
            double r = fma(-am[0], c[b], f[b]);
            r = fma(-am[1], w[b], r);
            r = fma(-am[2], e[b], r);
            r = fma(-am[3], s[b], r);
            r = fma(-am[4], n[b], r);
            if (!ok[b]) continue;
            const int t = t0 + b * blockDim.x, i = t & (V.P - 1), j = r0 + (t >> V.lg);
            const size_t at = ((size_t)j << V.lg) + i;
            const float rf = f64_to_f32(r);
            V.f[at] = rf;
            if (first) {
                if (((i + j) & 1) == 0) V.u[at] = rf * T.dinv[code[b]];
            } else {
                V.u[at] = 0.0f;
            }
            rm = max(rm, bits_of(r) & 0x7fffffffffffffffull);
            vm = max(vm, bits_of(c[b]) & 0x7fffffffffffffffull);
        }
    }
    *rmax = rm;
    *vmax = vm;
}

}  // namespace gs
