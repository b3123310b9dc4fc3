// The small coarse levels of a V-cycle (Algorithm 3, gamma = 1) by one thread
// block out of shared memory.
//
// A level of side s = 2 M - 1 is a grid of M x M cells; cell (I, J) holds the C
// point (2I+1, 2J+1), the corner (2I, 2J), the x-edge (2I, 2J+1) and the y-edge
// point (2I+1, 2J), the four relaxation colours in this order.  Every array is
// kept by colour and cell:
//  - u: planes of (M + 2)^2 with a border of zeros, so that a colour's eight
//    neighbours are eight fixed offsets into the other planes and no point
//    needs a bounds test;
//  - the operator: per colour the eight couplings, the inverse diagonal (its
//    rounding is one of the relaxation's weight: the tail computes a correction,
//    whose residual the finest level forms anew), and the row sum (float32) or the
//    diagonal (float64);
//    points outside the grid (the last row and column of cells) have zero
//    couplings and a zero inverse, and stay zero.
// A cell's operator, weights, f and residuals are one record (57 numbers, an odd
// stride: no bank conflicts) and the u planes have one pitch on every level, so
// that a colour phase is 18 shared loads at immediate offsets, nine operations
// and a store per thread, without divisions or index arithmetic, by one code for
// all the levels (each phase runs once per cycle: a copy per level size did not
// stay in the instruction cache).  Levels of at most 16 cells are run by one
// warp, without block barriers.
//
// Bound by the latency of its chain of phases (39 per cycle at V(1,2) from
// 31^2) and, in float64, by the float64 pipe (64 cycles per warp instruction).
// Measured from 31^2, barrier included: 16.5 us in float32 at V(1,2), 27.6 us in
// float64 at V(1,1).  Walking point-ordered arrays with a division and bounds
// tests per point took 35.5 us in float32; planes addressed through generic
// pointers with strides from memory took 18.2 and 31.3 us.
#pragma once

#include "mgsolve.cuh"
#include "stencil.cuh"

namespace gs {

constexpr int kTailMaxM = 16;                    // largest top level: side 31
constexpr int kTailW = kTailMaxM + 2;            // pitch of a u plane
constexpr int kTailPlane = kTailW * kTailW;
// A cell's record: per colour eight couplings, the inverse diagonal and the row
// sum / diagonal; then f and the residual per colour, and the weights.
constexpr int kTailF = 40, kTailR = 44, kTailP = 48, kTailRec = 57;

__host__ __device__ constexpr int tail_level_elems(int M) { return kTailRec * M * M + 4 * kTailPlane; }
// Offset of the level of M x M cells: the smaller levels come first.
__host__ __device__ inline int tail_level_at(int M) {
    int off = 0;
    for (int k = 1; k < M; k *= 2) off += tail_level_elems(k);
    return off;
}

// Shared memory of the tail levels `from` .. nlev - 1: coarsest inverse and
// right-hand side (float64), then the levels.
__host__ __device__ inline size_t tail_set_bytes(const SolveArgs& a, int from, size_t elem) {
    const size_t n = a.L[a.nlev - 1].n;
    const int M = (a.L[from].side + 1) / 2;
    if (M > kTailMaxM) return (size_t)1 << 40;   // not taken
    return ((n * n + n) * sizeof(double) + 15) / 16 * 16 + (size_t)tail_level_at(2 * M) * elem;
}

// Plane (colour) and parities of the colours: C, corner, x-edge, y-edge.
__host__ __device__ constexpr int tail_px(int c) { return c == 0 || c == 3 ? 1 : 0; }
__host__ __device__ constexpr int tail_py(int c) { return c == 0 || c == 2 ? 1 : 0; }
__host__ __device__ constexpr int tail_colour(int px, int py) {
    return px && py ? 0 : !px && !py ? 1 : py ? 2 : 3;
}
// Cell offset of the neighbour at d = -1, 0, 1 along one direction of a point of parity p.
__host__ __device__ constexpr int tail_shift(int p, int d) { return d == 0 ? 0 : p ? (d > 0 ? 1 : 0) : (d > 0 ? 0 : -1); }

// The levels of one launch in the dynamic shared memory.
struct TailBase {
    int lev;             // element offset of the levels
    int top, coarse;     // M of the first level and of the coarsest
    int n;               // unknowns of the coarsest level
};

template <typename T>
__device__ __forceinline__ T* tail_smem() {
    extern __shared__ __align__(16) char smem_t[];
    return (T*)smem_t;
}

// One level: its records and its u planes.
template <typename T>
struct TailLevel {
    T *rec, *u;
    int M, lg;
    __device__ __forceinline__ TailLevel(const TailBase& B, int M_) : M(M_), lg((M_ >= 2) + (M_ >= 4) + (M_ >= 8) + (M_ >= 16)) {
        rec = tail_smem<T>() + B.lev + tail_level_at(M);
        u = rec + kTailRec * M * M;
    }
    // f(record, pointer into plane 0 of u, I, J) for every cell; `one`: by warp 0
    // alone, else by the block.  Ends with the barrier of that group.
    template <class F>
    __device__ __forceinline__ void cells(bool one, F&& f) const {
        const int step = one ? 32 : blockDim.x;
        for (int cell = threadIdx.x; cell < M * M; cell += step) {
            const int J = cell >> lg, I = cell & (M - 1);
            f(rec + kTailRec * cell, u + (J + 1) * kTailW + I + 1, I, J);
        }
        if (one) __syncwarp();
        else __syncthreads();
    }
};

// Carves the levels out of shared memory and fills the fixed parts from the
// global operators (one block, all threads).
template <typename T, typename W>
__device__ __noinline__ TailBase tail_stage(const SolveArgs& a, int from) {
    TailBase B;
    B.n = (int)a.L[a.nlev - 1].n;
    B.top = (a.L[from].side + 1) / 2;
    B.coarse = (a.L[a.nlev - 1].side + 1) / 2;
    B.lev = (int)((((size_t)B.n * B.n + B.n) * sizeof(double) + 15) / 16 * 16 / sizeof(T));
    double* inv = tail_smem<double>();
    for (int k = threadIdx.x; k < B.n * B.n; k += blockDim.x) inv[k] = a.inv[k];
    for (int l = from; l < a.nlev; ++l) {
        const LevelArgs& G = a.L[l];
        const int m = (G.side + 1) / 2, c = m * m;
        const TailLevel<T> L(B, m);
        const bool solved = l + 1 == a.nlev;   // by the inverse: no operator needed
        for (int k = threadIdx.x; k < 4 * kTailPlane; k += blockDim.x) L.u[k] = T(0);
        for (int k = threadIdx.x; k < 4 * c; k += blockDim.x) {
            const int col = k / c, cell = k - col * c;
            T* R = L.rec + kTailRec * cell;
            R[kTailF + col] = T(0);
            if (solved) continue;
            const int i = 2 * (cell % m) + tail_px(col), j = 2 * (cell / m) + tail_py(col);
            const bool in = i < G.side && j < G.side;
            const size_t x = (size_t)j * G.side + i;
            const W* gA = (const W*)G.A;
            const T s = in ? (T)wval(gA[x]) : T(0);
            T diag = s;
#pragma unroll
            for (int d = 1; d < 9; ++d) {
                const T v = in ? (T)wval(gA[d * G.n + x]) : T(0);
                R[10 * col + d - 1] = v;
                if constexpr (sizeof(T) == 4) diag -= v;
            }
            R[10 * col + 8] = in ? T(1) / diag : T(0);
            R[10 * col + 9] = s;
        }
        if (!solved) {
            const W* gP = (const W*)G.P;   // (sc + 1)^2 = m^2 cells
            for (int k = threadIdx.x; k < 8 * c; k += blockDim.x)
                L.rec[kTailRec * (k % c) + kTailP + k / c] = (T)wval(gP[k]);
        }
    }
    __syncthreads();
    return B;
}

// x - sum_d a_d u_d (relaxation, float64 residual) or x - sum_d a_d (u_d - ux)
// (float32 residual) over the eight couplings of colour COL's point of a cell:
// one chain of fused operations (float64: the pipe, not the chain, is the bound).
template <typename T, int COL, bool leak>
__device__ __forceinline__ T tail_couple(T x, const T* R, const T* u, T ux) {
#pragma unroll
    for (int d = 1; d < 9; ++d) {
        const int qx = (tail_px(COL) + dir_di(d)) & 1, qy = (tail_py(COL) + dir_dj(d)) & 1;
        const int ox = tail_shift(tail_px(COL), dir_di(d)), oy = tail_shift(tail_py(COL), dir_dj(d));
        const T un = u[tail_colour(qx, qy) * kTailPlane + oy * kTailW + ox];
        x -= R[10 * COL + d - 1] * (leak ? un - ux : un);
    }
    return x;
}

template <typename T, int COL>
__device__ __forceinline__ void tail_relax(const TailLevel<T>& L, bool one) {
    L.cells(one, [&](const T* R, T* u, int, int) {
        u[COL * kTailPlane] = tail_couple<T, COL, false>(R[kTailF + COL], R, u, T(0)) * R[10 * COL + 8];
    });
}
template <typename T>
__device__ __noinline__ void tail_sweep(const TailLevel<T> L, bool one, bool first) {
    if (first) tail_relax<T, 0>(L, one);
    tail_relax<T, 1>(L, one);
    tail_relax<T, 2>(L, one);
    tail_relax<T, 3>(L, one);
}

template <typename T, int COL>
__device__ __forceinline__ void tail_resid(T* R, const T* u) {
    const T ux = u[COL * kTailPlane];
    R[kTailR + COL] = tail_couple<T, COL, sizeof(T) == 4>(R[kTailF + COL] - R[10 * COL + 9] * ux, R, u, ux);
}

// Pre-smoothing from u = 0, residual, restriction into the next level.  A sweep
// ends with the y-edges, whose residuals it has made zero up to rounding: after
// at least one sweep they are taken as zero.
template <typename T>
__device__ __noinline__ void tail_down(const TailLevel<T> L, const TailLevel<T> C, bool one, int nu1) {
    // u = 0 but, with pre-smoothing, the first colour: f / diag
    L.cells(one, [&](const T* R, T* u, int, int) {
        u[0] = nu1 > 0 ? R[kTailF] * R[8] : T(0);
        u[kTailPlane] = u[2 * kTailPlane] = u[3 * kTailPlane] = T(0);
    });
    for (int s = 0; s < nu1; ++s) tail_sweep<T>(L, one, s > 0);
    L.cells(one, [&](T* R, const T* u, int, int) {
        tail_resid<T, 0>(R, u);
        tail_resid<T, 1>(R, u);
        tail_resid<T, 2>(R, u);
        if (nu1 == 0) tail_resid<T, 3>(R, u);
    });
    L.cells(one, [&](const T* R, const T*, int I, int J) {
        if (I == L.M - 1 || J == L.M - 1) return;   // (M - 1)^2 coarse points
        const T *E = R + kTailRec, *N = R + kTailRec * L.M, *NE = N + kTailRec;
        constexpr int C0 = kTailR, K = kTailR + 1, X = kTailR + 2, Y = kTailR + 3, P = kTailP;
        T acc = R[C0];
        acc += R[P + PXE] * R[X] + E[P + PXW] * E[X];
        if (nu1 == 0) acc += R[P + PYN] * R[Y] + N[P + PYS] * N[Y];
        acc += R[P + PNE] * R[K] + E[P + PNW] * E[K];
        acc += N[P + PSE] * N[K] + NE[P + PSW] * NE[K];
        C.rec[kTailRec * ((J >> 1) * C.M + (I >> 1)) + kTailF + tail_colour(I & 1, J & 1)] = acc;
    });
}

// Prolongation from the next level, post-smoothing.
template <typename T>
__device__ __noinline__ void tail_up(const TailLevel<T> L, const TailLevel<T> C, bool one, int nu2) {
    auto U = [&](int I, int J) {   // -1 .. M - 1; the border planes hold zeros
        return C.u[tail_colour(I & 1, J & 1) * kTailPlane + ((J >> 1) + 1) * kTailW + (I >> 1) + 1];
    };
    L.cells(one, [&](const T* R, T* u, int I, int J) {
        const T* P = R + kTailP;
        const T uSW = U(I - 1, J - 1), uSE = U(I, J - 1), uNW = U(I - 1, J), uNE = U(I, J);
        const bool e = I < L.M - 1, n = J < L.M - 1;
        if (nu2 == 0 && e && n) u[0] += uNE;   // else overwritten, unread, by the first colour
        u[kTailPlane] += P[PSW] * uSW + P[PSE] * uSE + P[PNW] * uNW + P[PNE] * uNE;
        if (n) u[2 * kTailPlane] += P[PXW] * uNW + P[PXE] * uNE;
        if (e) u[3 * kTailPlane] += P[PYS] * uSE + P[PYN] * uNE;
    });
    for (int s = 0; s < nu2; ++s) tail_sweep<T>(L, one, true);
}

// The coarsest level by its explicit inverse, in float64 (warp 0).
template <typename T>
__device__ __noinline__ void tail_coarsest(const TailBase& B) {
    const TailLevel<T> L(B, B.coarse);
    const int side = 2 * L.M - 1, n = B.n;
    const double* inv = tail_smem<double>();
    double* fs = tail_smem<double>() + n * n;
    for (int x = threadIdx.x; x < n; x += 32) {
        const int j = x / side, i = x - j * side;
        fs[x] = (double)L.rec[kTailRec * ((j >> 1) * L.M + (i >> 1)) + kTailF + tail_colour(i & 1, j & 1)];
    }
    __syncwarp();
    for (int x = threadIdx.x; x < n; x += 32) {
        const int j = x / side, i = x - j * side;
        double acc = 0.0;
        for (int k = 0; k < n; ++k) acc += inv[x * n + k] * fs[k];
        L.u[tail_colour(i & 1, j & 1) * kTailPlane + ((j >> 1) + 1) * kTailW + (i >> 1) + 1] = (T)acc;
    }
    __syncwarp();
}

// One V-cycle visit of the tail: right-hand side from, correction to, its top
// level's global vectors f and u.
template <typename T>
__device__ __noinline__ void tail_cycle(const TailBase& B, const T* f, T* u, int nu1, int nu2) {
    const TailLevel<T> L(B, B.top);
    const int side = 2 * L.M - 1, n = side * side;
    for (int x = threadIdx.x; x < n; x += blockDim.x) {
        const int j = x / side, i = x - j * side;
        L.rec[kTailRec * ((j >> 1) * L.M + (i >> 1)) + kTailF + tail_colour(i & 1, j & 1)] = __ldcg(f + x);
    }
    __syncthreads();
    int M = B.top;
    for (; M > B.coarse && M > 4; M /= 2) tail_down<T>(TailLevel<T>(B, M), TailLevel<T>(B, M / 2), false, nu1);
    if (threadIdx.x < 32) {
        int q = M;
        for (; q > B.coarse; q /= 2) tail_down<T>(TailLevel<T>(B, q), TailLevel<T>(B, q / 2), true, nu1);
        tail_coarsest<T>(B);
        for (q *= 2; q <= M; q *= 2) tail_up<T>(TailLevel<T>(B, q), TailLevel<T>(B, q / 2), true, nu2);
    }
    __syncthreads();
    for (M *= 2; M <= B.top; M *= 2) tail_up<T>(TailLevel<T>(B, M), TailLevel<T>(B, M / 2), false, nu2);
    for (int x = threadIdx.x; x < n; x += blockDim.x) {
        const int j = x / side, i = x - j * side;
        u[x] = L.u[tail_colour(i & 1, j & 1) * kTailPlane + ((j >> 1) + 1) * kTailW + (i >> 1) + 1];
    }
}

}  // namespace gs
