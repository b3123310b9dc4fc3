// Fine-level kernels of the finite-difference Isaacs game (Sec. 3.3, Sec. 6.1):
// reward set-up, policy improvement (Eq. (eq1)/(ILPI)) fused with the
// policy-fixed assembly (Eq. (LSPI)), and the
// FAMGpi interpolations (Sec. 5.2).
#include <algorithm>

#include "kernels.cuh"
#include "stencil.cuh"

namespace gs {

namespace {

constexpr int kBlock = 256;

// SplitMix64 (Steele, Lea & Flood 2014): output i of the stream `seed`.
__device__ __forceinline__ uint64_t splitmix64(uint64_t seed, uint64_t i) {
    uint64_t z = seed + (i + 1ull) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// sin(pi x) of the grid lines: the rewards' product sin(pi x1) sin(pi x2) needs
// 2 side sines, not two per point (89 -> 12 us at 1023^2).
__global__ void k_line_sines(int side, double h, double* __restrict__ line) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < side) line[i] = sin(M_PI * ((i + 1) * h));
}

__global__ void k_isaacs_r0(int side, double kappa, NoiseSrc ns, const double* __restrict__ line,
                            double* __restrict__ r0) {
    const size_t n = (size_t)side * side;
    size_t x = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= n) return;
    unsigned iu;
    const int j = (int)FastDiv((unsigned)side).divmod((unsigned)x, &iu), i = (int)iu;
    const size_t ii = (size_t)(i + 1) * ns.step - 1, jj = (size_t)(j + 1) * ns.step - 1;
    const size_t fx = jj * ns.fine_side + ii;
    double xi;
    if (ns.xi_fine) {
        xi = ns.xi_fine[fx];
    } else {
        const double u = (double)(splitmix64(ns.seed, fx) >> 11) * 0x1.0p-53;
        xi = __dsub_rn(__dmul_rn(u, 0.1), 0.05);   // 0.1 u - 0.05, no contraction
    }
    r0[x] = kappa * (line[i] * line[j] + xi);
}

__device__ __forceinline__ double obstacle_psi(int i, int j, double h) {
    const double x1 = (i + 1) * h - 0.5, x2 = (j + 1) * h - 0.5;
    return 0.2 - (x1 * x1 + x2 * x2);
}

// Maximum of non-negative doubles through their bit patterns (integer ops).
__device__ __forceinline__ unsigned long long warp_max_bits(double v) {
    unsigned long long b = bits_of(v);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long w = __shfl_xor_sync(0xffffffffu, b, o);
        b = w > b ? w : b;
    }
    return b;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
// Shapley rows of the Isaacs game, factored.  With S the sum of the four
// neighbour values, w0 = 1/(2 c0) the weight of a direction without drift and
// delta = h/(2 c0) the extra weight of half a unit of drift, the drift
// (e_a - e_b)/2 puts delta on direction a and on the direction opposite to b
// (both on a when b is opposite to a), and a == b puts 2 delta on x itself:
//   F(v; x, a, b) = base + A_a + T_b            (a != b)
//   F(v; x, a, a) = base + 2 g v(x)
// with g = mu delta, base = mu w0 S + r0(x), A_a = g v(x + e_a) + c a,
// T_b = g v(x - e_b) - c b and c = 0.1 (1 - mu).  For fixed a, F(v; x, a, .)
// is base + A_a + u_b with u_b = T_b (b != a) and u_a = 2 g v(x) - A_a, so the
// argmin over b and the keep-current test compare the u_b.
struct Nbr {
    double vE, vW, vN, vS, vx;
};

// MIN's reply at fixed a with the keep-current rule: returns the new b and
// sets *fmin to min_b F(v; x, a, b).
__device__ __forceinline__ int reply_b(const double T[4], double A, double D, double base, int a,
                                       int bcur, double tau, double* fmin) {
    double u[4];
#pragma unroll
    for (int b = 0; b < 4; ++b) u[b] = (b == a) ? D - A : T[b];
    double m = u[0];
    int first = 0;
#pragma unroll
    for (int b = 1; b < 4; ++b)
        if (u[b] < m) { m = u[b]; first = b; }
    *fmin = base + A + m;
    return (u[bcur] - m > tau) ? first : bcur;
}

// MIN's reply at fixed a screened in float32: the float32 copies of the u_b
// are within err of the float64 values the exact path compares (err bounds
// the float32 rounding of the inputs and of every operation, with a wide
// margin), so when the smallest float32 u_b beats every other by more than
// 2 err + tau, the float64 comparisons pick the same index, and with the
// keep-current rule the reply is that index.  Returns false (undecided)
// otherwise.  *phi = A_a + min_b u_b in float32.
__device__ __forceinline__ bool screen_reply(const float Tf[4], float Af, float Df, int a, float err,
                                             float tauf, int* b_out, float* phi) {
    float u[4];
#pragma unroll
    for (int b = 0; b < 4; ++b) u[b] = (b == a) ? Df - Af : Tf[b];
    float m1 = u[0], m2 = INFINITY;
    int first = 0;
#pragma unroll
    for (int b = 1; b < 4; ++b) {
        if (u[b] < m1) {
            m2 = m1;
            m1 = u[b];
            first = b;
        } else if (u[b] < m2) {
            m2 = u[b];
        }
    }
    *b_out = first;
    *phi = Af + m1;
    return m2 - m1 > 2.0f * err + tauf;
}

// k = 0 .. 3 as a double, from its encoding (a conversion takes the float64 pipe).
__device__ __forceinline__ double small_double(int k) {
    return __hiloint2double(k == 0 ? 0 : k == 1 ? 0x3ff00000 : k == 2 ? 0x40000000 : 0x40080000, 0);
}

// Keep-current tolerance 1e-13 max(1, |v|_inf) from the reduced |v|_inf.
__device__ __noinline__ double tau_of_vmax(const DevScalars* sc) {
    return 1e-13 * fmax(1.0, __longlong_as_double((long long)sc->vmax));
}

// The exact float64 decisions of one state, for the states whose float32
// screen was not conclusive (near-ties).  Not inlined: the compiler must not
// evaluate these float64 rows speculatively for every state.
template <int MODE>
__device__ __noinline__ void improve_exact(const IsaacsConsts* __restrict__ K, const Nbr nb,
                                           double rx, int i, int j, int m1, int acur, uint32_t bw,
                                           double tau, uint32_t* bnew_out, int* anew_out,
                                           double* fmax_out) {
    const double g = K->gmu, c = K->c01;
    const double base = K->w0mu * (nb.vE + nb.vW + nb.vN + nb.vS) + rx;
    const double D = 2.0 * g * nb.vx;
    // T_b = g v(x - e_b) - c b for b = +x1, -x1, +x2, -x2
    const double T[4] = {g * nb.vW, g * nb.vE - c, g * nb.vS - 2.0 * c, g * nb.vN - 3.0 * c};
    // A_a = g v(x + e_a) + c a
    const double A[4] = {g * nb.vE, g * nb.vW + c, g * nb.vN + 2.0 * c, g * nb.vS + 3.0 * c};
    uint32_t bnew = bw;
    int anew = acur;
    if (MODE == IMP_INNER) {
        if (acur < 4) {
            const int bc = (bw >> (8 * acur)) & 0xff;
            double fmin;
            const int b = reply_b(T, A[acur], D, base, acur, bc, tau, &fmin);
            bnew = (bw & ~(0xffu << (8 * acur))) | ((uint32_t)b << (8 * acur));
        }
    } else {
        double Fa[5];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const int bc = (bw >> (8 * a)) & 0xff;
            const int b = reply_b(T, A[a], D, base, a, bc, tau, &Fa[a]);
            bnew = (bnew & ~(0xffu << (8 * a))) | ((uint32_t)b << (8 * a));
        }
        if (m1 == 5) Fa[4] = obstacle_psi(i, j, K->h);
        if (MODE == IMP_OUTER) {
            double fmax_ = Fa[0];
            int first = 0;
            for (int a = 1; a < m1; ++a)
                if (Fa[a] > fmax_) { fmax_ = Fa[a]; first = a; }
            anew = (fmax_ - Fa[acur] > tau) ? first : acur;
            *fmax_out = fmax_;
        }
    }
    *bnew_out = bnew;
    *anew_out = anew;
}

// What the improvement reads at one point.
struct ImprovePoint {
    Nbr nb;
    double rx;
    int i, j, acur, old_code;
    uint32_t bw;
    __device__ __forceinline__ void load(const ImproveArgs& A, const FastDiv& dv, unsigned x) {
        const int side = A.side;
        const double* __restrict__ v = A.v;
        unsigned iu;
        j = (int)dv.divmod(x, &iu);
        i = (int)iu;
        nb.vx = v[x];
        nb.vE = load_or_zero(v, (size_t)x + 1, i + 1 < side);
        nb.vW = load_or_zero(v, (size_t)x - 1, i > 0);
        nb.vN = load_or_zero(v, (size_t)x + side, j + 1 < side);
        nb.vS = load_or_zero(v, (size_t)x - side, j > 0);
        rx = A.r0[x];
        acur = A.alpha[x];
        bw = A.beta[x];
        old_code = A.code ? A.code[code_at(side, i, j)] : 0;
    }
};

// Every thread walks points a grid apart and loads the next one while it works
// on the current; counts and maxima are combined per block at its end.  Bound by
// the float64 operations in the outer mode (17 for the stored values and 4
// differences per point: 36 us at 1023^2), by memory latency in the others.  One point per thread with
// a few atomics per warp on the scalars, and the screen below on the values, took
// 117 us for the obstacle game at 1023^2 (48 us now).
template <int MODE>
__global__ void __launch_bounds__(kBlock) k_isaacs_improve(const __grid_constant__ ImproveArgs A, double tau_host,
                                                           float tau_host_f, int tau_from_vmax) {
    if (A.solved) {
        const int gave_up = A.solve_bar->error, reason = A.solved->reason;   // (one round trip for both)
        if (gave_up || (reason != kLinExact && reason != kLinInexact)) return;
    }
    const IsaacsConsts* __restrict__ K = A.K;
    const int side = A.side, variant = A.variant;
    const double tau = tau_from_vmax ? tau_of_vmax(A.sc) : tau_host;
    const float tauf = tau_from_vmax ? f64_to_f32(tau) : tau_host_f;
    const unsigned n = (unsigned)side * side, stride = gridDim.x * blockDim.x;
    const FastDiv dv((unsigned)side);
    double wsq = 0.0;
    unsigned long long wres = 0;
    int wch = 0, wcc = 0;
    unsigned x = blockIdx.x * blockDim.x + threadIdx.x;
    ImprovePoint next;
    if (x < n) next.load(A, dv, x);
#pragma unroll 1
    for (; x < n; x += stride) {
        const ImprovePoint pt = next;
        next.load(A, dv, x + stride < n ? x + stride : x);
        const Nbr& nb = pt.nb;
        const double rx = pt.rx;
        const int i = pt.i, j = pt.j, acur = pt.acur;
        const uint32_t bw = pt.bw;
        double res = 0.0;
        int changed = 0;
        const int m1 = variant == 1 ? 5 : 4;

        // ---- float32 screen of every decision this mode takes.  The rows share
        // base + 2 g v(x); the outer and reply modes subtract v(x) in float64
        // first, so that the terms carry the differences between neighbours, not
        // the values: the error bound shrinks by |dv| / |v| (about 1e-2 at 1023^2),
        // and with it the share of warps that have to take the exact path (from
        // four in five to a few in a hundred).  The inner mode takes one decision
        // instead of five: there the four subtractions would cost what they save.
        const float gf = K->gmu_f, cf = K->c01_f;
        float fx, fE, fW, fN, fS, err;
        if (MODE == IMP_INNER) {
            fx = f64_to_f32(nb.vx);
            fE = f64_to_f32(nb.vE);
            fW = f64_to_f32(nb.vW);
            fN = f64_to_f32(nb.vN);
            fS = f64_to_f32(nb.vS);
        } else {
            fx = 0.0f;
            fE = f64_to_f32(nb.vE - nb.vx);
            fW = f64_to_f32(nb.vW - nb.vx);
            fN = f64_to_f32(nb.vN - nb.vx);
            fS = f64_to_f32(nb.vS - nb.vx);
        }
        const float Vm = fmaxf(fmaxf(fabsf(fx), fmaxf(fabsf(fE), fabsf(fW))), fmaxf(fabsf(fN), fabsf(fS)));
        err = 0x1p-18f * (3.0f * gf * Vm + 6.0f * cf);
        float vabs = 0.0f;   // |v(x)|, an upper bound to float32 rounding
        if (MODE != IMP_INNER) {
            // the float64 comparisons' own rounding, in terms of the values
            vabs = fabsf(f64_to_f32(nb.vx)) + Vm;
            err += 0x1p-46f * gf * vabs;
        }
        const float Tf[4] = {gf * fW, gf * fE - cf, gf * fS - 2.0f * cf, gf * fN - 3.0f * cf};
        const float Af[4] = {gf * fE, gf * fW + cf, gf * fN + 2.0f * cf, gf * fS + 3.0f * cf};
        const float Df = 2.0f * gf * fx;
        bool sure = true;
        uint32_t bnew = bw;
        int anew = acur, amax = acur;
        float gbest = 0.0f;
        int bfirst[4] = {0, 0, 0, 0};
        if (MODE == IMP_INNER) {
            if (acur < 4) {
                float phi;
                // select, not index: a runtime index would put Af in local memory
                const float Aa = acur == 0 ? Af[0] : acur == 1 ? Af[1] : acur == 2 ? Af[2] : Af[3];
                sure = screen_reply(Tf, Aa, Df, acur, err, tauf, &bfirst[0], &phi);
                bnew = (bw & ~(0xffu << (8 * acur))) | ((uint32_t)bfirst[0] << (8 * acur));
            }
        } else {
            float G[4];
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                sure &= screen_reply(Tf, Af[a], Df, a, err, tauf, &bfirst[a], &G[a]);
                bnew = (bnew & ~(0xffu << (8 * a))) | ((uint32_t)bfirst[a] << (8 * a));
            }
            if (MODE == IMP_OUTER && sure) {
                // the best move (base and 2 g v(x) cancel between the four)
                float g1 = G[0], g2 = -INFINITY;
                int first = 0;
#pragma unroll
                for (int a = 1; a < 4; ++a) {
                    if (G[a] > g1) {
                        g2 = g1;
                        g1 = G[a];
                        first = a;
                    } else if (G[a] > g2) {
                        g2 = G[a];
                    }
                }
                sure = g1 - g2 > 4.0f * err + tauf;
                amax = first;
                gbest = g1;
            }
        }

        double fmax_ = 0.0, psi = 0.0;
        if (sure) {
            // float64 only where a value is stored
            if (MODE == IMP_OUTER) {
                // against the stop value psi: float32 where the two are well
                // apart, else the float64 values (the move's is needed anyway)
                bool move = true, stop = false;
                if (m1 == 5) {
                    const float fv = f64_to_f32(nb.vx);
                    const float mf = K->w0mu_f * (4.0f * fv + ((fE + fW) + (fN + fS))) + 2.0f * gf * fv + f64_to_f32(rx) + gbest;
                    const float x1 = (i + 1) * K->h_f - 0.5f, x2 = (j + 1) * K->h_f - 0.5f;
                    const float psif = 0.2f - (x1 * x1 + x2 * x2);
                    const float margin = 4.0f * err + tauf + 0x1p-17f * (K->w0mu_f * 8.0f * vabs + fabsf(mf) + fabsf(psif) + 1.0f);
                    stop = !(mf - psif > margin);
                    move = !(psif - mf > margin);
                }
                if (move) {
                    const double g = K->gmu, c = K->c01;
                    const double base = K->w0mu * (nb.vE + nb.vW + nb.vN + nb.vS) + rx;
                    const int b = amax == 0 ? bfirst[0] : amax == 1 ? bfirst[1] : amax == 2 ? bfirst[2] : bfirst[3];
                    const double vb = b == 0 ? nb.vW : b == 1 ? nb.vE : b == 2 ? nb.vS : nb.vN;
                    const double va = amax == 0 ? nb.vE : amax == 1 ? nb.vW : amax == 2 ? nb.vN : nb.vS;
                    const double Aa = g * va + c * small_double(amax);
                    // u_b = g v(x - e_b) - c b, or 2 g v(x) - A_a when b == a (as reply_b forms them)
                    const double u = (b == amax) ? 2.0 * g * nb.vx - Aa : g * vb - c * small_double(b);
                    fmax_ = base + Aa + u;
                }
                if (stop) psi = obstacle_psi(i, j, K->h);
                anew = amax;
                if (stop && (!move || psi > fmax_)) anew = 4;
                if (stop && move) {
                    // near-tie: keep the current action unless beaten by more than
                    // tau (a current move other than the best one is: by its margin)
                    const double fcur = acur == 4 ? psi : fmax_, top = anew == 4 ? psi : fmax_;
                    if ((acur == 4 || acur == amax) && !(top - fcur > tau)) anew = acur;
                    fmax_ = top;
                } else if (stop) {
                    fmax_ = psi;
                }
            }
        } else {
            improve_exact<MODE>(K, nb, rx, i, j, m1, acur, bw, tau, &bnew, &anew, &fmax_);
        }
        if (MODE == IMP_OUTER) {
            changed = anew != acur;
            res = fabs(fmax_ - nb.vx);
            if (A.fv) A.fv[x] = fmax_;
            if (A.alpha_out) A.alpha_out[x] = (uint8_t)anew;
            wsq = fma(res, res, wsq);
            const unsigned long long rb = bits_of(res);
            wres = rb > wres ? rb : wres;
        } else if (MODE == IMP_INNER) {
            changed = bnew != bw;
        }
        wch += changed;
        if (A.beta_out) A.beta_out[x] = bnew;
        if (A.beta5) {
            uint8_t* d = A.beta5 + 5 * x;
#pragma unroll
            for (int a = 0; a < 4; ++a) d[a] = (uint8_t)(bnew >> (8 * a));
            d[4] = A.beta4[x];
        }
        if (A.code) {
            // policy-fixed assembly for (alpha, beta(., alpha))
            const size_t cx = code_at(side, i, j);
            int new_code;
            if (anew == 4) {
                new_code = kStopCode;
                A.rhs[x] = obstacle_psi(i, j, K->h);
            } else {
                new_code = 4 * anew + (int)((bnew >> (8 * anew)) & 0xff);
                A.rhs[x] = rx + K->dr[anew][new_code & 3];
            }
            wcc += new_code != pt.old_code;
            A.code[cx] = (uint8_t)new_code;
        }
    }
    __shared__ double red_sq[kBlock / 32];
    __shared__ unsigned long long red_res[kBlock / 32];
    __shared__ int red_ch[kBlock / 32], red_cc[kBlock / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    wch = __reduce_add_sync(0xffffffffu, wch);
    wcc = __reduce_add_sync(0xffffffffu, wcc);
    if (MODE == IMP_OUTER) {
        wres = warp_max_bits(from_bits(wres));
        wsq = warp_sum(wsq);
    }
    if (lane == 0) {
        red_ch[w] = wch;
        red_cc[w] = wcc;
        red_res[w] = wres;
        red_sq[w] = wsq;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < kBlock / 32; ++k) {
            wch += red_ch[k];
            wcc += red_cc[k];
            if (MODE == IMP_OUTER) {
                wres = red_res[k] > wres ? red_res[k] : wres;
                wsq += red_sq[k];
            }
        }
        if (wch) atomicAdd(&A.sc->changed, wch);
        if (wcc) atomicAdd(&A.sc->code_changed, wcc);
        if (MODE == IMP_OUTER) {
            atomicMax(&A.sc->res, wres);
            atomicAdd(&A.sc->res_sq, wsq);
        }
    }
}

__global__ void k_isaacs_assemble(const IsaacsConsts* __restrict__ K, int side,
                                  const uint8_t* __restrict__ alpha, const uint32_t* __restrict__ beta,
                                  const double* __restrict__ r0, uint8_t* __restrict__ code,
                                  double* __restrict__ rhs) {
    const size_t n = (size_t)side * side;
    const size_t x = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= n) return;
    const int a = alpha[x];
    const int i = (int)(x % side), j = (int)(x / side);
    const size_t cx = code_at(side, i, j);
    if (a == 4) {
        code[cx] = kStopCode;
        rhs[x] = obstacle_psi(i, j, K->h);
    } else {
        const int b = (beta[x] >> (8 * a)) & 0xff;
        code[cx] = (uint8_t)(4 * a + b);
        rhs[x] = r0[x] + K->dr[a][b];
    }
}

__global__ void __launch_bounds__(kBlock) k_absmax(const double* __restrict__ v, size_t n, unsigned long long* out) {
    unsigned long long m = 0;
    for (size_t x = (size_t)blockIdx.x * blockDim.x + threadIdx.x; x < n;
         x += (size_t)gridDim.x * blockDim.x) {
        const unsigned long long b = bits_of(v[x]) & 0x7fffffffffffffffull;
        m = b > m ? b : m;
    }
    __shared__ unsigned long long red[kBlock / 32];
    m = warp_max_bits(from_bits(m));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < kBlock / 32; ++k) m = red[k] > m ? red[k] : m;
        atomicMax(out, m);
    }
}


// FAMGpi interpolation from side sc to sf = 2 sc + 1 (1-based fine (p, q),
// coarse (P, Q) at fine (2P, 2Q); P or Q in {0, sc+1} is the boundary).
__global__ void k_fmg_interp(int sc, const double* __restrict__ vc, const uint8_t* __restrict__ ac,
                             const uint32_t* __restrict__ bc, const uint8_t* __restrict__ b4c,
                             double* __restrict__ vf, uint8_t* __restrict__ af,
                             uint32_t* __restrict__ bf, uint8_t* __restrict__ b4f) {
    const int sf = 2 * sc + 1;
    const size_t x = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= (size_t)sf * sf) return;
    const int p = (int)(x % sf) + 1, q = (int)(x / sf) + 1;
    auto V = [&](int P, int Q) -> double {
        return (P < 1 || Q < 1 || P > sc || Q > sc) ? 0.0 : vc[(size_t)(Q - 1) * sc + (P - 1)];
    };
    double val;
    int P, Q;   // source of the policies: lowest-index interior member of N(x)
    if (!(p & 1) && !(q & 1)) {
        P = p / 2; Q = q / 2;
        val = V(P, Q);
    } else if ((p & 1) && !(q & 1)) {
        Q = q / 2;
        val = (V((p - 1) / 2, Q) + V((p + 1) / 2, Q)) / 2.0;
        P = (p - 1) / 2 >= 1 ? (p - 1) / 2 : (p + 1) / 2;
    } else if (!(p & 1) && (q & 1)) {
        P = p / 2;
        val = (V(P, (q - 1) / 2) + V(P, (q + 1) / 2)) / 2.0;
        Q = (q - 1) / 2 >= 1 ? (q - 1) / 2 : (q + 1) / 2;
    } else {
        const int P0 = (p - 1) / 2, P1 = (p + 1) / 2, Q0 = (q - 1) / 2, Q1 = (q + 1) / 2;
        val = (V(P0, Q0) + V(P1, Q0) + V(P0, Q1) + V(P1, Q1)) / 4.0;
        Q = Q0 >= 1 ? Q0 : Q1;
        P = P0 >= 1 ? P0 : P1;
        if (P > sc) P = P0;
        if (Q > sc) Q = Q0;
    }
    if (P > sc) P = sc;
    if (Q > sc) Q = sc;
    const size_t src = (size_t)(Q - 1) * sc + (P - 1);
    vf[x] = val;
    af[x] = ac[src];
    bf[x] = bc[src];
    if (b4f) b4f[x] = b4c[src];
}

}  // namespace

void launch_isaacs_r0(int side, double kappa, NoiseSrc ns, double* scratch, double* r0, cudaStream_t st) {
    const size_t n = (size_t)side * side;
    k_line_sines<<<div_up(side, kBlock), kBlock, 0, st>>>(side, 1.0 / (side + 1), scratch);
    k_isaacs_r0<<<div_up(n, kBlock), kBlock, 0, st>>>(side, kappa, ns, scratch, r0);
    GS_CHECK_LAUNCH_N(2);
}

void launch_isaacs_improve(ImproveMode mode, const ImproveArgs& a, cudaStream_t st) {
    const size_t n = (size_t)a.side * a.side;
    const double tau = a.tau < 0.0 ? 0.0 : a.tau;
    const int from_vmax = a.tau < 0.0 ? 1 : 0;
    auto run = [&](auto kernel) {
        // as many blocks as fit the GPU at once
        int per_sm = 0, dev = 0, sms = 0;
        GS_CUDA(cudaGetDevice(&dev));
        GS_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        GS_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kBlock, 0));
        const unsigned g = std::min(div_up(n, kBlock), (unsigned)(std::max(1, per_sm) * sms));
        kernel<<<g, kBlock, 0, st>>>(a, tau, (float)tau, from_vmax);
    };
    if (mode == IMP_OUTER) run(k_isaacs_improve<IMP_OUTER>);
    else if (mode == IMP_INNER) run(k_isaacs_improve<IMP_INNER>);
    else run(k_isaacs_improve<IMP_REPLY>);
    GS_CHECK_LAUNCH();
}

void launch_isaacs_assemble(const IsaacsConsts* K, int side, const uint8_t* alpha,
                            const uint32_t* beta, const double* r0, uint8_t* code, double* rhs,
                            cudaStream_t st) {
    const size_t n = (size_t)side * side;
    k_isaacs_assemble<<<div_up(n, kBlock), kBlock, 0, st>>>(K, side, alpha, beta, r0, code, rhs);
    GS_CHECK_LAUNCH();
}

void launch_absmax(const double* v, size_t n, unsigned long long* out, cudaStream_t st) {
    unsigned g = div_up(n, kBlock);
    if (g > 152 * 8) g = 152 * 8;
    k_absmax<<<g, kBlock, 0, st>>>(v, n, out);
    GS_CHECK_LAUNCH();
}


void launch_fmg_interp(int sc, const double* v_c, const uint8_t* alpha_c, const uint32_t* beta_c,
                       const uint8_t* beta4_c, double* v_f, uint8_t* alpha_f, uint32_t* beta_f,
                       uint8_t* beta4_f, cudaStream_t st) {
    const int sf = 2 * sc + 1;
    k_fmg_interp<<<div_up((size_t)sf * sf, kBlock), kBlock, 0, st>>>(sc, v_c, alpha_c, beta_c,
                                                                     beta4_c, v_f, alpha_f, beta_f,
                                                                     beta4_f);
    GS_CHECK_LAUNCH();
}

}  // namespace gs
