// mg.cu -- the multigrid field solve of the timestep (Sec. 2.5, Algorithm 1),
// arranged for one launch and little FP64 work on GB300.
//
// Same method as the oracle and as the reference GPU multigrid in field.cu:
// finite-volume operator, z-only coarsening, V(0,1) cycles with a red-black
// r-line sweep per level on the way up, [1/2 1 1/2] restriction of
// volume-integrated residuals, linear prolongation in z.  What changes is the
// arrangement:
//  - every r-line of every level is factored once per solve (the line
//    matrices do not change between cycles) for a warp-level solver: Thomas
//    on a chunk of the line per lane, the chunks' interface unknowns by
//    parallel cyclic reduction over the lanes;
//  - the whole solve is one cooperative launch: the residual and the
//    restriction chain run over tiles of columns, convergence is decided on
//    the device, and a block sweeps one black line with the two red lines
//    beside it as soon as the coarse rows above it are there;
//  - prolongation is folded into the red sweep: red (odd) rows are
//    recomputed whole by their line solve, so only the injection of the
//    coarse correction into the black (even) neighbour rows is ever used;
//  - the cycle works on the correction of phi; the mixed path keeps the
//    correction, the coarse right-hand sides and the line factors in FP32
//    and the residual in FP64 (iterative refinement).
#include <math.h>
#include <string.h>

#include <algorithm>

#include "mg.cuh"

namespace pic {

namespace {

// bit pattern of |x|: ordered like |x| for numbers, above them for a NaN
__device__ __forceinline__ unsigned long long abs_bits(double x) {
    return (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
}

// ---- set-up ----

// Set-up, first launch: rho and chi from the particles' deposit (a timestep;
// else chi is given), and nodal chi of every coarse level: full weighting in z,
// injection on the boundary rows.  A block takes 2^lc columns: rows loaded side
// by side, a warp per column down the levels in shared memory, levels stored
// by rows.  Bound by launch latency and one trip to L2 each way.
__global__ void __launch_bounds__(256) k_setup_levels(const MGFast *__restrict__ mp, int nr, int lc, FieldSource f,
                                                      const StepCtl *ctl) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const MGFast &m = *mp;
    if (ctl && ctl->halt) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nz0 = m.nz[0], nlev = m.nlev;
    const int cols = 1 << lc, j0 = blockIdx.x << lc, st = 2 * nz0 + kMaxLevels;
    double *s = reinterpret_cast<double *>(smem_raw);
    for (int e = threadIdx.x; e < nz0 << lc; e += blockDim.x) {
        const int c = e & (cols - 1), i = e >> lc, j = j0 + c;
        if (j >= nr) continue;
        const size_t k = (size_t)i * nr + j;
        double x;
        if (f.Ne) {
            double rho;
            node_field(f.Ne[k], f.Ni[k], f.iV[k], f.q0, f.q1, f.c0, f.c1, rho, x);
            f.rho[k] = rho;
            f.chi[k] = x;
        } else {
            x = f.chi[k];
        }
        s[(size_t)c * st + i] = x;
    }
    if (nlev == 1) return;
    __syncthreads();
    for (int c = warp; c < cols; c += blockDim.x >> 5) {
        const double *src = s + (size_t)c * st;
        double *dst = s + (size_t)c * st + nz0;
        for (int l = 1; l < nlev; ++l) {
            const int nzc = m.nz[l];
            for (int I = lane; I < nzc; I += 32)
                dst[I] = (I == 0 || I == nzc - 1)
                             ? src[2 * I]
                             : 0.25 * src[2 * I - 1] + 0.5 * src[2 * I] + 0.25 * src[2 * I + 1];
            __syncwarp();
            src = dst;
            dst += nzc;
        }
    }
    __syncthreads();
    int at = nz0;
    for (int l = 1; l < nlev; ++l) {
        const int nzc = m.nz[l];
        double *chi = m.chi[l];
        for (int e = threadIdx.x; e < nzc << lc; e += blockDim.x) {
            const int c = e & (cols - 1), I = e >> lc, j = j0 + c;
            if (j < nr) chi[(size_t)I * nr + j] = s[(size_t)c * st + at + I];
        }
        at += nzc;
    }
}

// 1/x: IEEE division in FP32; in FP64 a float reciprocal refined by two
// Newton-Raphson steps r <- r (2 - x r) (relative error ~1e-16 from ~6e-8)
__device__ __forceinline__ float recip(float x) { return 1.0f / x; }
__device__ __forceinline__ double recip(double x) {
    double r = (double)(1.0f / (float)x);
    r = fma(r, fma(-x, r, 1.0), r);
    r = fma(r, fma(-x, r, 1.0), r);
    return r;
}

// ---- r-line factors for the warp line solve ----
//
// Line system of row i: lo_j x_{j-1} + dg_j x_j + up_j x_{j+1} = b_j with
// lo_j = -cr[i][j-1] (0 on the axis), dg_j = a + c + d + e, up_j = -cr[i][j]
// (0 on the last unknown).  One warp solves a line: lane p owns the chunk
// j = pM .. pM + M - 1 (unknowns past n are x = 0 rows).  The chunk's last
// unknown is its interface I_p; the M - 1 interior unknowns are
//     y = z + I_{p-1} v + I_p w,
// z the interior solution with zero neighbours (Thomas), v and w the
// responses to the two neighbouring interfaces.  Substituting into the
// interface equations leaves a tridiagonal system in I_0..I_31, which the
// warp reduces by parallel cyclic reduction over lanes (shuffles).  Only the
// right-hand side changes between cycles, so all of this except the
// right-hand-side sweeps is computed once per solve.  Per line the factors
// are, lane-minor ([arr][k][32]):
//   ell (forward multipliers), invd (1/pivot), cp (up * invd), v, w
//   (5 arrays of M), then loI, upI (interface couplings), the five PCR
//   steps' alpha and gamma, and 1/diagonal of the reduced system.
//
// FP64 lines of 65 to 512 unknowns take 128 lanes (four warps) instead: a warp's
// FP64 instruction occupies its SM partition's pipe for ~60 cycles, so one warp
// per line left three of the four pipes idle (7700 cycles a line at M = 16).
// The chunks are a quarter as long, the interface system has seven reduction
// steps, and lanes exchange through shared memory.  Longer lines' factors
// would not fit shared memory that way; shorter ones have under two unknowns a
// lane, gain nothing, and their factors take four times the space, so that
// tall meshes reload them every cycle (whole solves, 32 / 128 lanes: 1025 x 65
// 682 / 818 us, 33 x 65 202 / 224; 65 x 129 310 / 291).
constexpr int kLine = 32;  // lanes per line

constexpr bool grouped(int M, bool f64) { return f64 && M >= 4 && M <= 16; }

// how a line of up to 32 M unknowns is laid out
template <typename Ts, int M>
struct Shape {
    static constexpr bool group = grouped(M, sizeof(Ts) == 8);
    static constexpr int lanes = group ? 128 : kLine;
    static constexpr int chunk = group ? M / 4 : M;
    static constexpr int steps = group ? 7 : 5;
    static constexpr int row = lanes + 1;          // a line buffer's row of one unknown of every chunk, padded
    static constexpr int unknowns = lanes * chunk;  // with padding
    static constexpr int elems = 5 * chunk * lanes + (3 + 2 * steps) * lanes;
    // position of unknown j in a line buffer
    static __device__ __forceinline__ int at(int j) { return (j % chunk) * row + j / chunk; }
};
int line_elems(int M, bool f64) {
    if (!grouped(M, f64)) return 5 * M * kLine + 13 * kLine;
    return 5 * (M / 4) * 128 + 17 * 128;
}
int line_buffer(int M, bool f64) {
    return grouped(M, f64) ? (M / 4) * 129 : M * 33;
}

// FP64 lines of more than 128 unknowns: four lines' factors (110 KB and more)
// leave an SM room for one block, however few registers it takes.  A batch's
// solves of such lines have an SM per block too, then: all its registers (128
// made them spill, 2 KB a thread above 512 unknowns), up to as many blocks as a
// reactor alone, and wider residual tiles the fewer they get (fit_tiles).
// Steps of batches, against 128 registers, a block per two rows and tiles of 4
// columns: six 33 x 1025 reactors 2130 -> 1375 us, forty 17 x 700 4340 -> 2360,
// sixteen 33 x 513 1620 -> 1260, forty 33 x 257 2510 -> 2020.
constexpr bool one_block(int M, bool f64) { return f64 && M >= 8; }

// chunk per lane: the least power of two M with 32 M >= n
inline int line_chunk(int n) {
    int M = 1;
    while (kLine * M < n) M <<= 1;
    return M;
}

// The solve's control block starts cleared, with the one decision all of the
// solve's blocks take whether it runs (one thread of the set-up calls it).
// They do not look at `halt` themselves: the cell sort beside the solve may
// set it, and blocks that went on without the others would leave words behind
// under tags that the next solve uses again.
__device__ __forceinline__ void begin_solve(const MGFast &m, const StepCtl *ctl) {
    MGCtl c{};
    c.skip = ctl && *(const volatile int32_t *)&ctl->halt;
    *m.ctl = c;
}

// what a node of the fine level starts from: the right-hand side
// rho A_j dz / eps0, the operator's diagonal and the Dirichlet data of phi;
// with phi_prev (a warm solve) the interior starts from 2 phi - phi_prev, the
// linear extrapolation in time of the last two steps' potentials, and
// phi_prev takes the last step's
struct RhsArgs {
    const double *rho;
    double *phi;
    const double *phi_zL;
    double V;
    int cold, v_from_ctl;
    double *phi_prev;
};
__device__ __forceinline__ void rhs_node(const MGFast &m, const RhsArgs &a, double V, int nz, int nr, int i, int j,
                                         double diag) {
    const size_t k = (size_t)i * nr + j;
    const bool inner = i > 0 && i < nz - 1 && j < nr - 1;
    m.f0[k] = inner ? a.rho[k] * m.ga[j] : 0.0;
    m.dg0[k] = inner ? diag : 0.0;
    double p;
    if (i == 0)
        p = (j == nr - 1) ? 0.0 : V;
    else if (i == nz - 1)
        p = a.phi_zL ? a.phi_zL[j] : 0.0;
    else if (j == nr - 1)
        p = 0.0;
    else if (a.cold)
        p = 0.0;
    else if (a.phi_prev) {
        const double t = a.phi[k];
        p = 2.0 * t - a.phi_prev[k];
        a.phi_prev[k] = t;
    } else
        p = a.phi[k];
    a.phi[k] = p;
}

// Set-up, second launch: per row of every level (a block each) the face
// coefficients, stored for the solve and kept in shared memory for the row's
// line factors (its first warp); on the fine level also what its nodes start
// from.  One launch for what were three (coefficients, factors, right-hand
// side), where the factors made a trip to L2 between each and the next (11 us
// on c2, 32 us on c3 and in FP64).  Bound by the FP64 pipe: ~8 operations a
// node, so a row's nodes are spread over the four SM partitions; a warp per
// row was slower than the three launches.
constexpr int kSetupThreads = 128;
template <typename Ts, int M>
__global__ void __launch_bounds__(kSetupThreads)
    k_setup_lines(const MGFast *__restrict__ mp, const double *__restrict__ chi0, int nr, int face_mean, RhsArgs a,
                  const StepCtl *ctl) {
    using Sh = Shape<Ts, M>;
    constexpr int MC = Sh::chunk, NL = Sh::lanes;
    __shared__ Ts sd[MC * Sh::row], se[MC * Sh::row];  // cz below + above the row, cr
    __shared__ Ts sx[2][6][Sh::group ? NL : 1];         // exchange between the lanes' warps
    const MGFast &m = *mp;
    if (blockIdx.x == 0 && threadIdx.x == 0) begin_solve(m, ctl);
    if (ctl && ctl->halt) return;
    const int n = nr - 1, p = threadIdx.x & (NL - 1);
    int i = blockIdx.x, l = 0;
    while (i >= m.nz[l]) i -= m.nz[l++];
    const int nz = m.nz[l];
    const double *chi = (l == 0 ? chi0 : m.chi[l]) + (size_t)i * nr;
    const bool inner = i > 0 && i < nz - 1, mixed = m.cz32[l] != nullptr;
    const double V = (ctl && a.v_from_ctl) ? ctl->V : a.V;  // in a timestep the source voltage comes with the step
    // (1 + chi of the face) g; the maximum of two values that are not negative
    // (nor NaN) by their bit patterns, off the FP64 pipe
    auto face = [&](double x, double y, double g) {
        double f;
        if (face_mean) {
            f = 0.5 * (x + y);
        } else {
            const unsigned long long bx = (unsigned long long)__double_as_longlong(x),
                                     by = (unsigned long long)__double_as_longlong(y);
            f = (bx | by) < 0x7ff0000000000000ull ? __longlong_as_double((long long)max(bx, by)) : fmax(x, y);
        }
        return fma(f, g, g);
    };
    for (int j = threadIdx.x; j < nr; j += kSetupThreads) {
        double lo = 0.0, hi = 0.0, right = 0.0;  // cz below and above the row, cr
        const double c = chi[j], gz = m.gz[l][j];
        if (i > 0) lo = face(chi[j - nr], c, gz);
        if (i + 1 < nz) hi = face(c, chi[j + nr], gz);
        if (j + 1 < nr) right = face(c, chi[j + 1], m.gr[l][j]);
        const size_t k = (size_t)i * nr + j;
        if (mixed) m.cz32[l][k] = (float)hi;
        if (!mixed || l == 0) m.cz[l][k] = hi;  // (the mixed path's coarse levels are FP32)
        if (l == 0) {
            m.cr[k] = right;
            const double left = j > 0 ? face(chi[j - 1], c, m.gr[0][j - 1]) : 0.0;
            rhs_node(m, a, V, nz, nr, i, j, lo + hi + left + right);
        }
        if (inner && j < n) {
            sd[Sh::at(j)] = (Ts)lo + (Ts)hi;
            se[Sh::at(j)] = (Ts)right;
        }
    }
    __syncthreads();
    if (!inner || threadIdx.x >= NL) return;
    const bool f64 = sizeof(Ts) == 8;
    Ts *fac = (l == m.nlev - 1) ? (f64 ? (Ts *)m.facc : (Ts *)m.facc32)
                                : (f64 ? (Ts *)m.fac64[l] : (Ts *)m.fac32[l]);
    Ts *F = fac + (size_t)(i - 1) * Sh::elems;
    auto coef = [&](int k, Ts &lo, Ts &dg, Ts &up) {
        const int j = p * MC + k;
        if (j >= n) {
            lo = 0;
            dg = 1;
            up = 0;
            return;
        }
        lo = j > 0 ? -se[Sh::at(j - 1)] : (Ts)0;
        dg = sd[Sh::at(j)] - lo + se[Sh::at(j)];
        up = j < n - 1 ? -se[Sh::at(j)] : (Ts)0;
    };
    constexpr int MI = MC - 1;
    // values of the lanes s to the left and right (undefined past the ends)
    int turn = 0;
    auto swap = [&](auto &...x) {
        if constexpr (Sh::group) {
            int w = 0;
            ((sx[turn][w++][p] = x), ...);
            __syncthreads();
        }
    };
    auto left = [&](Ts x, int w, int s) -> Ts {
        if constexpr (Sh::group)
            return sx[turn][w][(p - s) & (NL - 1)];
        else
            return __shfl_up_sync(0xffffffffu, x, s);
    };
    auto right = [&](Ts x, int w, int s) -> Ts {
        if constexpr (Sh::group)
            return sx[turn][w][(p + s) & (NL - 1)];
        else
            return __shfl_down_sync(0xffffffffu, x, s);
    };
    Ts A, B, C;  // reduced (interface) equation of this lane
    Ts loI, dgI, upI;
    coef(MC - 1, loI, dgI, upI);
    if constexpr (MI > 0) {
        // interior Thomas factors
        Ts ell[MI], invd[MI], cp[MI], v[MI], w[MI];
        Ts upm = 0, iv = 0, lo0 = 0, upL = 0;
#pragma unroll
        for (int k = 0; k < MI; ++k) {
            Ts lo, dg, up;
            coef(k, lo, dg, up);
            Ts el = 0, d = dg;
            if (k > 0) {
                el = lo * iv;
                d = dg - el * upm;
            } else {
                lo0 = lo;
            }
            iv = recip(d);
            ell[k] = el;
            invd[k] = iv;
            cp[k] = up * iv;
            upm = up;
            upL = up;
        }
        // spikes: v answers -lo_0 at the first interior unknown, w answers
        // -up_{MI-1} at the last (forward sweep, then backward)
        v[0] = -lo0;
#pragma unroll
        for (int k = 1; k < MI; ++k) v[k] = -ell[k] * v[k - 1];
        v[MI - 1] = v[MI - 1] * invd[MI - 1];
        w[MI - 1] = -upL * invd[MI - 1];
#pragma unroll
        for (int k = MI - 2; k >= 0; --k) {
            v[k] = v[k] * invd[k] - cp[k] * v[k + 1];
            w[k] = -cp[k] * w[k + 1];
        }
#pragma unroll
        for (int k = 0; k < MI; ++k) {
            F[(size_t)k * NL + p] = ell[k];
            F[(size_t)(MC + k) * NL + p] = invd[k];
            F[(size_t)(2 * MC + k) * NL + p] = cp[k];
            F[(size_t)(3 * MC + k) * NL + p] = v[k];
            F[(size_t)(4 * MC + k) * NL + p] = w[k];
        }
        swap(v[0], w[0]);
        const Ts v0n = right(v[0], 0, 1), w0n = right(w[0], 1, 1);
        turn ^= 1;
        A = loI * v[MI - 1];
        B = dgI + loI * w[MI - 1] + (p < NL - 1 ? upI * v0n : (Ts)0);
        C = p < NL - 1 ? upI * w0n : (Ts)0;
    } else {
        A = loI;
        B = dgI;
        C = upI;
    }
    Ts *Gf = F + (size_t)5 * MC * NL;
    Gf[p] = loI;
    Gf[NL + p] = upI;
    // parallel cyclic reduction of the interface system over the lanes
#pragma unroll
    for (int st = 0; st < Sh::steps; ++st) {
        const int s = 1 << st;
        swap(A, B, C);
        const Ts Am = left(A, 0, s), Bm = left(B, 1, s), Cm = left(C, 2, s);
        const Ts Ap = right(A, 0, s), Bp = right(B, 1, s), Cp = right(C, 2, s);
        turn ^= 1;
        Ts al = 0, ga = 0;
        if (p >= s) al = -A * recip(Bm);
        if (p + s < NL) ga = -C * recip(Bp);
        Gf[(2 + st) * NL + p] = al;
        Gf[(2 + Sh::steps + st) * NL + p] = ga;
        const Ts nB = B + (p >= s ? al * Cm : (Ts)0) + (p + s < NL ? ga * Ap : (Ts)0);
        A = p >= s ? al * Am : (Ts)0;
        C = p + s < NL ? ga * Cp : (Ts)0;
        B = nB;
    }
    Gf[(2 + 2 * Sh::steps) * NL + p] = recip(B);
}

// Warp solve of one line: right-hand side in Bs and solution out to the same
// place, both [k * 33 + p] (lane-minor with a pad against bank conflicts).
// All 32 lanes take part.  A line is one chain of dependent operations, so the
// chain is kept to one fused multiply-add per unknown and sweep (the products
// that do not depend on it are taken out of it) and the factors come in
// registers where they fit (LineFactors::load, before the right-hand side is
// there): FP32, M = 16, 635 -> 474 cycles, M = 8, 443 -> 363; the five
// shuffled reduction steps are ~170 of them.  In FP64 a line is bound by
// GB300's narrow FP64 pipe (~70 cycles per warp instruction) instead.
constexpr int kRow = 33;

__device__ __forceinline__ float fma_(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fma_(double a, double b, double c) { return fma(a, b, c); }

// a line's factors, lane p's share: in registers (REG), or read from shared
// memory as they are used
template <typename Ts, int M, bool REG>
struct LineFactors;
template <typename Ts, int M>
struct LineFactors<Ts, M, false> {
    const Ts *F;
    int p;
    __device__ __forceinline__ void load(const Ts *f, int lane) {
        F = f;
        p = lane;
    }
    template <int ARR>
    __device__ __forceinline__ Ts at(int k) const {
        return F[(ARR * M + k) * kLine + p];
    }
    __device__ __forceinline__ Ts tail(int k) const { return F[(5 * M + k) * kLine + p]; }
};
template <typename Ts, int M>
struct LineFactors<Ts, M, true> {
    Ts a[5][M > 1 ? M - 1 : 1], t[13];
    __device__ __forceinline__ void load(const Ts *F, int p) {
#pragma unroll
        for (int r = 0; r < 5; ++r)
#pragma unroll
            for (int k = 0; k < M - 1; ++k) a[r][k] = F[(r * M + k) * kLine + p];
#pragma unroll
        for (int k = 0; k < 13; ++k) t[k] = F[(5 * M + k) * kLine + p];
    }
    template <int ARR>
    __device__ __forceinline__ Ts at(int k) const {
        return a[ARR][k];
    }
    __device__ __forceinline__ Ts tail(int k) const { return t[k]; }
};

template <typename Ts, int M, bool REG>
__device__ __forceinline__ void warp_line_solve(const LineFactors<Ts, M, REG> &q, Ts *Bs, int p) {
    constexpr int MI = M - 1;
    Ts z[M];
#pragma unroll
    for (int k = 0; k < M; ++k) z[k] = Bs[k * kRow + p];
    Ts r = z[M - 1];
    if constexpr (MI > 0) {
#pragma unroll
        for (int k = 1; k < MI; ++k) z[k] = fma_(-q.template at<0>(k), z[k - 1], z[k]);
#pragma unroll
        for (int k = 0; k < MI; ++k) z[k] *= q.template at<1>(k);
#pragma unroll
        for (int k = MI - 2; k >= 0; --k) z[k] = fma_(-q.template at<2>(k), z[k + 1], z[k]);
        const Ts z0n = __shfl_down_sync(0xffffffffu, z[0], 1);
        r = fma_(-q.tail(0), z[MI - 1], r);
        if (p < kLine - 1) r = fma_(-q.tail(1), z0n, r);
    }
#pragma unroll
    for (int st = 0; st < 5; ++st) {
        const int s = 1 << st;
        const Ts rm = __shfl_up_sync(0xffffffffu, r, s), rp = __shfl_down_sync(0xffffffffu, r, s);
        r = fma_(q.tail(7 + st), rp, fma_(q.tail(2 + st), rm, r));
    }
    const Ts I = r * q.tail(12);
    if constexpr (MI > 0) {
        const Ts Ip = __shfl_up_sync(0xffffffffu, I, 1);  // lane 0: v is zero there
#pragma unroll
        for (int k = 0; k < MI; ++k)
            Bs[k * kRow + p] = fma_(q.template at<4>(k), I, fma_(q.template at<3>(k), Ip, z[k]));
    }
    Bs[(M - 1) * kRow + p] = I;
}

// The same by 128 threads (p: the thread's lane; X: 2 x 128 values of shared
// memory of their own; bar: a named barrier of their own)
template <typename Ts, int M>
__device__ __forceinline__ void group_line_solve(const Ts *__restrict__ F, Ts *Bs, Ts *X, int p, int bar) {
    using Sh = Shape<Ts, M>;
    constexpr int MC = Sh::chunk, MI = MC - 1, NL = Sh::lanes;
    const Ts *G = F + 5 * MC * NL;
    Ts z[MC];
#pragma unroll
    for (int k = 0; k < MC; ++k) z[k] = Bs[k * Sh::row + p];
    int turn = 0;
    auto share = [&](Ts x) {
        turn ^= NL;
        X[turn + p] = x;
        asm volatile("bar.sync %0, 128;" ::"r"(bar) : "memory");
    };
    Ts r = z[MC - 1];
    if constexpr (MI > 0) {
#pragma unroll
        for (int k = 1; k < MI; ++k) z[k] = fma_(-F[k * NL + p], z[k - 1], z[k]);
#pragma unroll
        for (int k = 0; k < MI; ++k) z[k] *= F[(MC + k) * NL + p];
#pragma unroll
        for (int k = MI - 2; k >= 0; --k) z[k] = fma_(-F[(2 * MC + k) * NL + p], z[k + 1], z[k]);
        share(z[0]);
        r = fma_(-G[p], z[MI - 1], r);
        if (p < NL - 1) r = fma_(-G[NL + p], X[turn + p + 1], r);
    }
#pragma unroll
    for (int st = 0; st < Sh::steps; ++st) {
        const int s = 1 << st;
        share(r);
        const Ts rm = X[turn + ((p - s) & (NL - 1))], rp = X[turn + ((p + s) & (NL - 1))];
        r = fma_(G[(2 + Sh::steps + st) * NL + p], rp, fma_(G[(2 + st) * NL + p], rm, r));
    }
    const Ts I = r * G[(2 + 2 * Sh::steps) * NL + p];
    if constexpr (MI > 0) {
        share(I);
        const Ts Ip = X[turn + ((p - 1) & (NL - 1))];  // lane 0: v is zero there
#pragma unroll
        for (int k = 0; k < MI; ++k)
            Bs[k * Sh::row + p] = fma_(F[(4 * MC + k) * NL + p], I, fma_(F[(3 * MC + k) * NL + p], Ip, z[k]));
    }
    Bs[(MC - 1) * Sh::row + p] = I;
}

template <typename Ts, int M>
__device__ __forceinline__ void warp_line_solve(const Ts *F, Ts *Bs, int p) {
    LineFactors<Ts, M, false> q;
    q.load(F, p);
    warp_line_solve<Ts, M, false>(q, Bs, p);
}

// a further solve with the operator of the one before: its right-hand side and
// boundary data alone
__global__ void k_rhs_bc(const MGFast *__restrict__ mp, RhsArgs a, int nz, int nr, const StepCtl *ctl) {
    const MGFast &m = *mp;
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nz * nr) return;
    if (k == 0) begin_solve(m, ctl);
    rhs_node(m, a, (ctl && a.v_from_ctl) ? ctl->V : a.V, nz, nr, k / nr, k % nr, m.dg0[k]);
}

// ---------------------------------------------------------------------------
// The whole solve in one cooperative launch (its blocks are co-resident).
// The V-cycle works on the correction delta of phi in both precisions (FP32
// delta and residual for the mixed path).  Per cycle:
//   1. one tile of columns per block: the residual (FP64 path: of phi + delta;
//      mixed path: by the GCR step), its norm, and the restriction chain down
//      to the coarsest level;
//   2. convergence decision: every block reads the same norms;
//   3. up the levels: the unit of a black line i = 2q + 2 solves the red lines
//      2q + 1 and 2q + 3 beside it (two warps at once), keeps them in shared
//      memory and solves the black line.  A red line shared by two units is
//      computed by both from the same data, bit for bit, and stored by one.
// The solve is bound by latency: a c2 cycle is a chain of one tile phase, two
// all-to-all exchanges and seven levels of line solves, each under a
// microsecond of arithmetic.  So no barrier separates the phases: what one
// block hands to another (rows of the correction, the restricted right-hand
// sides, norms, dot products) travels in flagged words that the reader polls
// (Flag in pic_internal.cuh), and a unit starts when its three coarse rows
// are there.  Units are dealt coarse to fine, block b taking units b, b + P,
// ...; a unit waits only for units before it, so the chain cannot lock.  Each
// unit's line factors stay in shared memory for the whole solve where they
// fit; operator, Krylov vectors and phi are read and written by the block
// that owns them, and nothing drops them from L1.
// Words are reused every cycle under a new tag.  That is safe: a tile phase
// starts with every row of the cycle's level-0 correction, each of which comes
// after all its unit's reads and after those of all units above it; rows of
// the next correction start with the coarsest, for which all tile phases of
// that cycle must be through; and no block is more than a cycle ahead of
// another's look at the norms, which are kept in two sets.  A solve's tags
// start where the one before ended (block 0 moves `epoch` on), so either all
// of its blocks run or none does (MGCtl::skip).
// What is exchanged all-to-all is kept in kCopies copies (with one, 128 blocks
// polling the same few lines of L2 take 3 us for the norms, so 1.8), sums and
// maxima take few FP64 and 64-bit operations, a tile's restricted levels are
// stored by rows, and FP32 lines' factors wait in registers.
// Measured, a whole stand-alone solve with its set-up, against one whose phases
// meet at grid barriers (~1 us each, and each costs every phase its L1): 33 x 65
// mixed 218 -> 117 us, 65 x 300 mixed 327 -> 178, 257 x 1025 mixed 627 -> 460,
// 129 x 513 FP64 887 -> 527 (there the line solves take the rest of the time).
// ---------------------------------------------------------------------------

// ---- factor lines into shared memory ----
// Bulk copies that complete on an mbarrier (thread 0 issues them).  All
// threads of the block keep the same state: per region the parity of the next
// completion and whether a copy is pending.
struct Loader {
    unsigned mbar;     // the first region's mbarrier (8 bytes each)
    unsigned phase, pending;  // bit per region
};

__device__ __forceinline__ void ld_begin(Loader &q, int r, unsigned bytes) {
    if (threadIdx.x == 0) {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(q.mbar + 8 * r), "r"(bytes)
                     : "memory");
    }
    q.pending |= 1u << r;
}

// sizes and addresses are multiples of 16 bytes
__device__ __forceinline__ void ld_copy(const Loader &q, int r, void *dst, const void *src, unsigned bytes) {
    if (threadIdx.x == 0)
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                     ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src), "r"(bytes), "r"(q.mbar + 8 * r)
                     : "memory");
}

// wait for region r's copy (every thread of the block calls it); false where
// the bounded wait gave up
__device__ __forceinline__ bool ld_wait(Loader &q, int r) {
    if (!(q.pending >> r & 1u)) return true;
    bool ok = false;
    for (long long it = 0; it < kSpinLimit && !ok; ++it) {
        unsigned done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
            : "=r"(done)
            : "r"(q.mbar + 8 * r), "r"(q.phase >> r & 1u)
            : "memory");
        ok = done != 0;
    }
    q.pending &= ~(1u << r);
    q.phase ^= 1u << r;
    return ok;
}

constexpr int kSolveThreads = 256;

// the warp's largest of 64-bit words: high halves first, then the low halves
// of those that have it (two integer reductions)
__device__ __forceinline__ unsigned long long warp_max(unsigned long long x) {
    const unsigned hi = __reduce_max_sync(0xffffffffu, (unsigned)(x >> 32));
    const unsigned lo = __reduce_max_sync(0xffffffffu, (unsigned)(x >> 32) == hi ? (unsigned)x : 0u);
    return ((unsigned long long)hi << 32) | lo;
}

// the largest of a over the block's threads (bit patterns), and of b
__device__ __forceinline__ void block_max2(unsigned long long &a, unsigned long long &b,
                                           unsigned long long (*s)[kSolveThreads / 32]) {
    a = warp_max(a);
    b = warp_max(b);
    const int lane = threadIdx.x & 31;
    if (lane == 0) {
        s[0][threadIdx.x >> 5] = a;
        s[1][threadIdx.x >> 5] = b;
    }
    __syncthreads();
    a = warp_max(lane < kSolveThreads / 32 ? s[0][lane] : 0ull);
    b = warp_max(lane < kSolveThreads / 32 ? s[1][lane] : 0ull);
}

// nz = 3: one interior row, phi's own, solved exactly in FP64 by one block
template <int M>
__device__ __noinline__ void solve_row(const MGFast &m, double *phi, int nr, double tol, int max_cycles,
                                          double *B, double *F) {
    using Sh = Shape<double, M>;
    __shared__ unsigned long long s_max[2][kSolveThreads / 32];
    __shared__ double s_x[256];
    const int tid = threadIdx.x, n = nr - 1;
    const double *cz = m.cz[0], *cr = m.cr;
    for (int k = tid; k < Sh::elems; k += kSolveThreads) F[k] = m.facc[k];
    double bn = 0.0;
    for (int cyc = 0;; ++cyc) {
        unsigned long long rmax = 0ull, bmax = 0ull;
        for (int j = tid; j < n; j += kSolveThreads) {
            const size_t k = (size_t)nr + j;
            const double below = cz[k - nr] * phi[k - nr], above = cz[k] * phi[k + nr], right = cr[k] * phi[k + 1];
            const double left = j > 0 ? cr[k - 1] * phi[k - 1] : 0.0;
            rmax = max(rmax, abs_bits(m.f0[k] - (m.dg0[k] * phi[k] - below - above - right - left)));
            bmax = max(bmax, abs_bits(m.f0[k] + below + above + (j == n - 1 ? right : 0.0)));
        }
        block_max2(rmax, bmax, s_max);
        const double rn = __longlong_as_double((long long)rmax);
        if (cyc == 0) bn = __longlong_as_double((long long)bmax);
        int d = 0;
        if (bn == 0.0)
            d = 3;
        else if (tol > 0.0 && rn <= tol * bn)
            d = 1;
        else if (cyc >= max_cycles)
            d = tol > 0.0 ? 2 : 1;
        if (tid == 0) {
            m.ctl->last_res = rn;
            m.ctl->bnorm = bn;
            m.ctl->cycles = cyc;
            if (d == 1) m.ctl->converged = 1;
            if (d == 3) m.ctl->zero_rhs = 1;
        }
        if (d == 3)
            for (int j = tid; j < n; j += kSolveThreads) phi[nr + j] = 0.0;
        if (d) return;
        for (int j = tid; j < Sh::unknowns; j += kSolveThreads) {
            double rhs = 0.0;
            if (j < n) {
                const size_t k = (size_t)nr + j;
                rhs = m.f0[k] + cz[k - nr] * phi[k - nr] + cz[k] * phi[k + nr];
                if (j == n - 1) rhs += cr[k] * phi[k + 1];
            }
            B[Sh::at(j)] = rhs;
        }
        __syncthreads();
        if constexpr (Sh::group) {
            if (tid < 128) group_line_solve<double, M>(F, B, s_x, tid, 1);
        } else {
            if (tid < 32) warp_line_solve<double, M>(F, B, tid);
        }
        __syncthreads();
        for (int j = tid; j < n; j += kSolveThreads) phi[nr + j] = B[Sh::at(j)];
        __syncthreads();
    }
}

// One reactor's solve on P blocks (bid: this block's index among them).
// WIDE: a block per SM; else two, with half the registers.
template <typename Tv, int M, bool WIDE>
__device__ __forceinline__ void solve_body(const MGFast *__restrict__ mp, double *phi, int nr,
                                           const SolveLayout &lay, double tol, int max_cycles,
                                           const int bid, const int P) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int nt = kSolveThreads;
    constexpr int kU = WIDE ? 4 : 2;  // elements per thread and batch in the residual phase
    // the level table in shared memory (read in front of every phase's loads)
    __shared__ __align__(16) MGFast s_m;
    {
        static_assert(sizeof(MGFast) % 8 == 0, "the level table is copied in 8-byte words");
        const unsigned long long *src = reinterpret_cast<const unsigned long long *>(mp);
        unsigned long long *dst = reinterpret_cast<unsigned long long *>(&s_m);
        for (int k = tid; k < (int)(sizeof(MGFast) / 8); k += nt) dst[k] = src[k];
        __syncthreads();
    }
    const MGFast &m = s_m;
    MGCtl *ctl = m.ctl;
    const unsigned ep = *(volatile unsigned *)m.epoch;  // tags of this solve: ep + 1 + cycle
    if (ctl->skip) return;  // an earlier failure of this step
    const int n = nr - 1, nz0 = m.nz[0], L = m.nlev - 1;
    using Sh = Shape<Tv, M>;
    constexpr int NW = Sh::unknowns, LFE = Sh::elems;
    if (L == 0) {
        if (bid == 0)
            solve_row<M>(m, phi, nr, tol, max_cycles, reinterpret_cast<double *>(smem_raw),
                         reinterpret_cast<double *>(smem_raw + lay.offC));
        return;
    }
    using Fv = Flag<Tv>;
    using Wv = typename Fv::W;
    constexpr bool mixed = sizeof(Tv) == 4;  // flexible GCR(1) around the V-cycle; else the plain V(0,1) iteration
    __shared__ unsigned long long s_max[2][2][nt / 32];
    __shared__ double s_dot[2][4][nt / 32];
    __shared__ double s_ab[4];  // the GCR step's beta, alpha, |q|^2 and the inverse of that
    __shared__ __align__(8) unsigned long long s_mbar[kMaxSlots + 1];
    double bn = 0.0;  // max |b|
    if (tid == 0) {
        s_ab[3] = 0.0;
        for (int b = 0; b <= kMaxSlots; ++b)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"((unsigned)__cvta_generic_to_shared(&s_mbar[b]))
                         : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    Loader ld{(unsigned)__cvta_generic_to_shared(&s_mbar[0]), 0u, 0u};
    // ---- this block's units: levels L-1 (one unit) .. 0, coarse to fine ----
    const int units = (2 << L) - 2 - L, nun = units > bid ? (units - bid + P - 1) / P : 0;
    const int S = lay.slots;
    auto unit_at = [&](int u, int &l, int &q) {
        l = L - 1;
        for (int w = 1; u >= w; w = 2 * w + 1) {  // units of level l
            u -= w;
            --l;
        }
        q = u;
    };
    Tv *slots = reinterpret_cast<Tv *>(smem_raw + lay.offF);
    constexpr unsigned FB = (unsigned)(LFE * sizeof(Tv));
    // request the factors of this block's k-th unit (its k-th modulo nun) into slot r
    auto request = [&](int k, int r) {
        int l, q;
        unit_at(bid + (k % nun) * P, l, q);
        const Tv *fac = mixed ? (const Tv *)m.fac32[l] : (const Tv *)m.fac64[l];
        Tv *dst = slots + (size_t)r * 3 * LFE;
        ld_begin(ld, r, 3 * FB);
        // lines 2q + 1, 2q + 2, 2q + 3 lie one after another
        ld_copy(ld, r, dst, fac + (size_t)(2 * q) * LFE, 3 * FB);
    };
    for (int k = 0; k < min(nun, S); ++k) request(k, k);
    Tv *FC = reinterpret_cast<Tv *>(smem_raw + lay.offC);
    if (bid == 0) {  // the coarsest row
        ld_begin(ld, kMaxSlots, FB);
        ld_copy(ld, kMaxSlots, FC, mixed ? (const Tv *)m.facc32 : (const Tv *)m.facc, FB);
    }
    // line buffers: the two reds, the black line
    Tv *const Bf = reinterpret_cast<Tv *>(smem_raw);
    constexpr int BL = Sh::chunk * Sh::row;
    __shared__ Tv s_x[Sh::group ? 512 : 1];  // a group's exchange: 2 x 128 values each
    double *St = reinterpret_cast<double *>(smem_raw);
    const int tw = lay.tw, ltw = __ffs(tw) - 1, sw = tw + 2, ntile = (n + tw - 1) >> ltw, tn = tw * (nz0 - 2);
    // e / sw for e < sw * nz0 (< 2^17): e * ceil(2^32 / sw) >> 32
    const unsigned sw_inv = 0xffffffffu / (unsigned)sw + 1u;
    auto div_sw = [&](int e) { return (int)__umulhi((unsigned)e, sw_inv); };
    Tv *T0 = reinterpret_cast<Tv *>(smem_raw + lay.offT), *T1 = T0 + (size_t)tw * nz0;
    Wv *lu0 = (Wv *)m.lu[0], *lf0 = (Wv *)m.lf[0];
    bool fail = false;
    int g = 0;  // units done
    int cyc = 0;
    for (;; ++cyc) {
        const unsigned tag = ep + 1u + (unsigned)cyc;
        __syncthreads();  // the line buffers are read; the tile takes their place
        // maxima as bit patterns of |x| (ordered like the values; a NaN
        // compares above every number), so the reductions are integer work
        unsigned long long rmax = 0ull, bmax = 0ull;
        const double *cz = m.cz[0], *cr = m.cr;
        // the level-0 correction of the cycle before at the tile's nodes and
        // its neighbour columns' (zero on the boundary), a batch per thread
        auto delta_batch = [&](int e0, int j0, Tv (&dv)[kU]) {
            const Wv *p[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const int e = e0 + u * nt, i = div_sw(e), c = e - i * sw - 1, j = j0 + c;
                p[u] = (e < sw * nz0 && j >= 0 && j < n && i > 0 && i < nz0 - 1) ? lu0 + (size_t)i * nr + j : nullptr;
            }
            flag_wait<Tv, kU>(p, dv, tag - 1u, &ctl->timeout, fail);
        };
        // the restriction chain of the residual tile T0 (columns j0 ..) down
        // to the coarsest level, in the V-cycle's type: a warp per column, the
        // levels one after another in T1; then all of it stored by rows (a
        // warp's words in few sectors), the coarsest level first, which the
        // line phases start with
        auto chain = [&](int j0) {
            for (int c = warp; c < tw; c += nt / 32) {
                const Tv *src = T0 + (size_t)c * nz0;
                Tv *dst = T1 + (size_t)c * (nz0 + kMaxLevels);
                for (int l = 1; l <= L; ++l) {
                    const int nzc = m.nz[l];
                    for (int I = 1 + lane; I < nzc - 1; I += 32)
                        dst[I] = (Tv)0.5 * src[2 * I - 1] + src[2 * I] + (Tv)0.5 * src[2 * I + 1];
                    __syncwarp();
                    src = dst;
                    dst += nzc;
                }
            }
            __syncthreads();
            int at_l = 0;  // level l's place in a column
            for (int l = 1; l < L; ++l) at_l += m.nz[l];
            for (int l = L; l > 0; --l) {
                const int nzc = m.nz[l];
                Wv *fl = (Wv *)m.lf[l];
                for (int e = tid; e < (nzc - 2) << ltw; e += nt) {
                    const int c = e & (tw - 1), I = 1 + (e >> ltw), j = j0 + c;
                    if (j < n) Fv::store(fl + (size_t)I * nr + j, T1[(size_t)c * (nz0 + kMaxLevels) + at_l + I], tag);
                }
                if (l > 1) at_l -= m.nz[l - 1];
            }
        };
        if (mixed && cyc > 0) {
            // ---- flexible GCR(1) step (mixed path) ----
            // z: the V-cycle's correction of the last cycle; w = A z; the
            // direction is z less its projection on the previous one (in the
            // A-image), the step length minimises |r|_2
            double a[4] = {0.0, 0.0, 0.0, 0.0};  // r.w, w.w, w.wp, r.wp
            for (int t = bid; t < ntile; t += P) {
                const int j0 = t * tw;
                for (int e0 = tid; e0 < sw * nz0; e0 += kU * nt) {
                    Tv dv[kU];
                    delta_batch(e0, j0, dv);
#pragma unroll
                    for (int u = 0; u < kU; ++u) {
                        const int e = e0 + u * nt, i = div_sw(e), c = e - i * sw - 1;
                        if (e < sw * nz0) St[(size_t)(c + 1) * nz0 + i] = (double)dv[u];
                    }
                }
                __syncthreads();
                const size_t q0 = (size_t)t * tn;
                // batches of kU nodes per thread, loads first
                for (int e0 = tid; e0 < tn; e0 += kU * nt) {
                    double ca[kU], cb[kU], ce[kU], cd[kU], dgv[kU], rv[kU], wpv[kU];
#pragma unroll
                    for (int u = 0; u < kU; ++u) {
                        const int e = e0 + u * nt, c = e & (tw - 1), i = 1 + (e >> ltw), j = j0 + c;
                        ca[u] = cb[u] = ce[u] = cd[u] = dgv[u] = rv[u] = wpv[u] = 0.0;
                        if (e < tn && j < n) {
                            const size_t k = (size_t)i * nr + j;
                            ca[u] = cz[k - nr];
                            cb[u] = cz[k];
                            ce[u] = cr[k];
                            cd[u] = j > 0 ? cr[k - 1] : 0.0;
                            dgv[u] = m.dg0[k];
                            rv[u] = m.kr[q0 + e];
                            wpv[u] = m.kwp[q0 + e];
                        }
                    }
#pragma unroll
                    for (int u = 0; u < kU; ++u) {
                        const int e = e0 + u * nt, c = e & (tw - 1), i = 1 + (e >> ltw), j = j0 + c;
                        if (e >= tn || j >= n) continue;
                        const double *Sc = St + (size_t)(c + 1) * nz0 + i;
                        const double w = dgv[u] * Sc[0] - ca[u] * Sc[-1] - cb[u] * Sc[1] - ce[u] * Sc[nz0] -
                                         cd[u] * Sc[-nz0];
                        m.kw[q0 + e] = w;
                        a[0] += rv[u] * w;
                        a[1] += w * w;
                        a[2] += w * wpv[u];
                        a[3] += rv[u] * wpv[u];
                    }
                }
                if (t + P < ntile) __syncthreads();  // the tile is rewritten by the next
            }
            // the warp's four sums with few FP64 additions (the pipe is
            // narrow): halves of the warp trade the products they do not
            // keep (16 apart: 0, 1 stay low, 2, 3 high; 8 apart: one
            // product per quarter), then each quarter sums its own;
            // product 2 (lane >> 4) + ((lane >> 3) & 1) ends in the
            // quarter's lanes
            {
                const bool hi = lane >= 16, q1 = (lane & 8) != 0;
                const double s0 = __shfl_xor_sync(0xffffffffu, hi ? a[0] : a[2], 16);
                const double s1 = __shfl_xor_sync(0xffffffffu, hi ? a[1] : a[3], 16);
                const double b0 = (hi ? a[2] : a[0]) + s0, b1 = (hi ? a[3] : a[1]) + s1;
                double c = (q1 ? b1 : b0) + __shfl_xor_sync(0xffffffffu, q1 ? b0 : b1, 8);
                for (int o = 4; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
                if ((lane & 7) == 0) s_dot[0][2 * (lane >> 4) + ((lane >> 3) & 1)][warp] = c;
            }
            if (__syncthreads_or(fail)) break;
            // (lane 4 w + k of a warp takes product k of warp w: three additions)
            auto over_warps = [&](int set) {
                double v = s_dot[set][lane & 3][lane >> 2];
                for (int o = 4; o < 32; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                return v;
            };
            static_assert(nt / 32 == 8, "a lane for each product of each warp");
            if (warp == 0) {
                const double v = over_warps(0);
                // one copy for each kCopies-th reader: lane 4 c + k the copy c of product k
                Flag<double>::store(m.xd + ((size_t)(lane >> 2) * kMaxSolveBlocks + bid) * 4 + (lane & 3), v, tag);
            }
            // every block sums the partial products in the same fixed order
            // (the same step length everywhere): thread t takes entries t,
            // t + nt, ... of product t % 4 (nt is a multiple of 32)
            {
                const ulonglong2 *xd = m.xd + (size_t)(bid % kCopies) * kMaxSolveBlocks * 4;
                double v = 0.0;
                for (int e0 = tid; e0 < 4 * P; e0 += 2 * nt) {
                    const ulonglong2 *p[2] = {xd + e0, e0 + nt < 4 * P ? xd + e0 + nt : nullptr};
                    double x[2];
                    flag_wait<double, 2>(p, x, tag, &ctl->timeout, fail);
                    v += x[0];
                    if (p[1]) v += x[1];
                }
                for (int o = 4; o < 32; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                if (lane < 4) s_dot[1][lane][warp] = v;
                if (__syncthreads_or(fail)) break;
                // the step's scalars by one thread: GB300's FP64 pipe is
                // narrow, and every thread dividing cost microseconds
                if (warp == 0) {
                    const double t = over_warps(1);
                    const double rw = __shfl_sync(0xffffffffu, t, 0), ww = __shfl_sync(0xffffffffu, t, 1);
                    double wwp = __shfl_sync(0xffffffffu, t, 2), rwp = __shfl_sync(0xffffffffu, t, 3);
                    if (lane == 0) {
                        // no previous direction (a solve's first step): what lies
                        // there is an earlier solve's, perhaps not finite
                        if (!(s_ab[3] > 0.0)) wwp = rwp = 0.0;
                        const double beta = wwp * s_ab[3];
                        const double den = ww - beta * wwp;
                        s_ab[0] = beta;
                        s_ab[1] = den > 0.0 ? (rw - beta * rwp) / den : 1.0;
                        s_ab[2] = den > 0.0 ? den : 0.0;
                    }
                }
                __syncthreads();
            }
            const double beta = s_ab[0], alpha = s_ab[1];
            // 1 / |q|^2 for the next step's beta, off this one's path (none where
            // the inverse would not be finite: the next step starts anew)
            if (tid == nt - 1) s_ab[3] = s_ab[2] >= 2.2250738585072014e-308 ? 1.0 / s_ab[2] : 0.0;
            const bool one = bid + P >= ntile;  // the block's only tile: z is still in St
            for (int t = bid; t < ntile; t += P) {
                const int j0 = t * tw;
                const size_t q0 = (size_t)t * tn;
                for (int e0 = tid; e0 < tn; e0 += kU * nt) {
                    double pz[kU], qw[kU], zp[kU], wpv[kU], xv[kU], rv[kU];
#pragma unroll
                    for (int u = 0; u < kU; ++u) {
                        const int e = e0 + u * nt, c = e & (tw - 1), i = 1 + (e >> ltw), j = j0 + c;
                        pz[u] = qw[u] = zp[u] = wpv[u] = xv[u] = rv[u] = 0.0;
                        if (e < tn && j < n) {
                            const size_t k = (size_t)i * nr + j;
                            pz[u] = one ? St[(size_t)(c + 1) * nz0 + i] : (double)Fv::value(Fv::load(lu0 + k));
                            qw[u] = m.kw[q0 + e];
                            if (beta != 0.0) {
                                zp[u] = m.kzp[q0 + e];
                                wpv[u] = m.kwp[q0 + e];
                            }
                            xv[u] = phi[k];
                            rv[u] = m.kr[q0 + e];
                        }
                    }
#pragma unroll
                    for (int u = 0; u < kU; ++u) {
                        const int e = e0 + u * nt, c = e & (tw - 1), i = 1 + (e >> ltw), j = j0 + c;
                        if (e >= tn) break;
                        double rn = 0.0;
                        if (j < n) {
                            const size_t k = (size_t)i * nr + j;
                            const double p = pz[u] - beta * zp[u], q = qw[u] - beta * wpv[u];
                            phi[k] = xv[u] + alpha * p;
                            rn = rv[u] - alpha * q;
                            m.kr[q0 + e] = rn;
                            m.kzp[q0 + e] = p;
                            m.kwp[q0 + e] = q;
                            rmax = max(rmax, abs_bits(rn));
                            Fv::store(lf0 + k, (Tv)rn, tag);
                        }
                        T0[(size_t)c * nz0 + i] = (Tv)rn;
                    }
                }
                __syncthreads();
                chain(j0);
                if (t + P < ntile) __syncthreads();
            }
        } else {
            for (int t = bid; t < ntile; t += P) {
                const int j0 = t * tw;
                // phi of the tile and its two neighbour columns, all rows: the
                // iterate at first, then (FP64 path) the tile's own copy plus
                // the correction; batches of kU elements per thread, loads first
                double *own = m.ps + (size_t)t * sw * nz0;
                for (int e0 = tid; e0 < sw * nz0; e0 += kU * nt) {
                    double pv[kU];
                    Tv dv[kU];
#pragma unroll
                    for (int u = 0; u < kU; ++u) {
                        const int e = e0 + u * nt, i = div_sw(e), c = e - i * sw - 1, j = j0 + c;
                        pv[u] = 0.0;
                        dv[u] = 0;
                        if (e < sw * nz0 && j >= 0 && j < nr) pv[u] = !mixed && cyc > 0 ? own[e] : phi[(size_t)i * nr + j];
                    }
                    if (!mixed && cyc > 0) delta_batch(e0, j0, dv);
#pragma unroll
                    for (int u = 0; u < kU; ++u) {
                        const int e = e0 + u * nt, i = div_sw(e), c = e - i * sw - 1, j = j0 + c;
                        if (e >= sw * nz0) break;
                        const double v = pv[u] + (double)dv[u];
                        if (!mixed) own[e] = v;
                        // the iterate, stored by the tile that owns the node
                        if (!mixed && cyc > 0 && c >= 0 && c < tw && j < n && i > 0 && i < nz0 - 1)
                            phi[(size_t)i * nr + j] = v;
                        St[(size_t)(c + 1) * nz0 + i] = v;
                    }
                }
                __syncthreads();
                const size_t q0 = (size_t)t * tn;
                // interior rows only: the chain never reads a level's boundary rows
                for (int e0 = tid; e0 < tn; e0 += kU * nt) {
                    double ca[kU], cb[kU], ce[kU], cd[kU], dgv[kU], fv[kU];
#pragma unroll
                    for (int u = 0; u < kU; ++u) {
                        const int e = e0 + u * nt, c = e & (tw - 1), i = 1 + (e >> ltw), j = j0 + c;
                        ca[u] = cb[u] = ce[u] = cd[u] = dgv[u] = fv[u] = 0.0;
                        if (e < tn && j < n) {
                            const size_t k = (size_t)i * nr + j;
                            ca[u] = cz[k - nr];
                            cb[u] = cz[k];
                            ce[u] = cr[k];
                            cd[u] = j > 0 ? cr[k - 1] : 0.0;
                            dgv[u] = m.dg0[k];
                            fv[u] = m.f0[k];
                        }
                    }
#pragma unroll
                    for (int u = 0; u < kU; ++u) {
                        const int e = e0 + u * nt, c = e & (tw - 1), i = 1 + (e >> ltw), j = j0 + c;
                        if (e >= tn) break;
                        double r = 0.0;
                        if (j < n) {
                            const size_t k = (size_t)i * nr + j;
                            const double *Sc = St + (size_t)(c + 1) * nz0 + i;
                            const double a = ca[u], cc = cb[u], ee = ce[u], d = cd[u];
                            const double Au = dgv[u] * Sc[0] - a * Sc[-1] - cc * Sc[1] - ee * Sc[nz0] - d * Sc[-nz0];
                            const double f = fv[u];
                            r = f - Au;
                            rmax = max(rmax, abs_bits(r));
                            if (cyc == 0) {
                                double bb = f;
                                if (i == 1) bb += a * Sc[-1];
                                if (i == nz0 - 2) bb += cc * Sc[1];
                                if (j == nr - 2) bb += ee * Sc[nz0];
                                bmax = max(bmax, abs_bits(bb));
                            }
                            Fv::store(lf0 + k, (Tv)r, tag);
                            if (mixed) m.kr[q0 + e] = r;
                        }
                        T0[(size_t)c * nz0 + i] = (Tv)r;
                    }
                }
                __syncthreads();
                chain(j0);
                if (t + P < ntile) __syncthreads();
            }
        }
        block_max2(rmax, bmax, s_max[0]);
        // (two sets in turn: a block that owns no unit may still be reading the
        // norms of the cycle before)
        ulonglong2 *xr = m.xr + (size_t)(cyc & 1) * kCopies * 2 * kMaxSolveBlocks;
        if (tid < kCopies) {
            ulonglong2 *to = xr + (size_t)tid * 2 * kMaxSolveBlocks + 2 * bid;
            Flag<double>::store(to, __longlong_as_double((long long)rmax), tag);
            if (cyc == 0) Flag<double>::store(to + 1, __longlong_as_double((long long)bmax), tag);
        }
        xr += (size_t)(bid % kCopies) * 2 * kMaxSolveBlocks;
        // ---- decision: every block reads every block's maxima, and comes to
        // the same: 0 continue, 1 converged, 2 out of cycles, 3 zero right-hand
        // side, 4 a wait gave up.  phi holds the iterate of this residual.  The
        // line phases start without it (they do not change phi): a block looks
        // while it waits for its coarse rows, the one with the coarsest row,
        // which all others wait for, when it has handed that on.
        auto check = [&]() -> int {
            unsigned long long rm = 0ull, bm = 0ull;
            for (int e = tid; e < P; e += nt) {
                const ulonglong2 *p[2] = {xr + 2 * e, cyc == 0 ? xr + 2 * e + 1 : nullptr};
                double x[2];
                flag_wait<double, 2>(p, x, tag, &ctl->timeout, fail);
                rm = max(rm, (unsigned long long)__double_as_longlong(x[0]));
                bm = max(bm, (unsigned long long)__double_as_longlong(x[1]));
            }
            block_max2(rm, bm, s_max[1]);
            if (__syncthreads_or(fail)) {
                fail = true;
                return 4;
            }
            const double rn = __longlong_as_double((long long)rm);
            if (cyc == 0) bn = __longlong_as_double((long long)bm);
            int d = 0;
            if (bn == 0.0)
                d = 3;
            else if (tol > 0.0 && rn <= tol * bn)
                d = 1;
            else if (cyc >= max_cycles)
                d = tol > 0.0 ? 2 : 1;
            if (bid == 0 && tid == 0) {
                ctl->last_res = rn;
                ctl->bnorm = bn;
                ctl->cycles = cyc;
                if (d == 1) ctl->converged = 1;
                if (d == 3) ctl->zero_rhs = 1;
            }
            return d;
        };
        int decide = -1;  // not looked yet
        // ---- up: per unit, a black line with the two red lines beside it ----
        constexpr int kE = (NW + nt - 1) / nt;  // unknowns of a line per thread
        for (int k = 0; k < nun; ++k, ++g) {
            int l, q;
            unit_at(bid + k * P, l, q);
            const int nzc = m.nz[l + 1], slot = nun <= S ? k : g % S;
            const bool deep = l == L - 1;  // the coarsest row is solved here first
            const int ra = 2 * q + 1;      // rows ra and ra + 2 red, ra + 1 black
            Wv *u = (Wv *)m.lu[l] + (size_t)ra * nr;
            const Tv *czl = (mixed ? (const Tv *)m.cz32[l] : (const Tv *)m.cz[l]) + (size_t)2 * q * nr;
            // warps 0 and 1 solve the reds, warp 2 the black line: their factors
            // come into registers while the coarse rows are on their way
            if (!ld_wait(ld, slot) || (deep && !ld_wait(ld, kMaxSlots))) fail = true;
            constexpr bool kReg = WIDE && sizeof(Tv) == 4 && M <= 16;
            const Tv *F = slots + (size_t)slot * 3 * LFE;
            LineFactors<Tv, M, kReg> lf;
            if (!Sh::group && warp < 3) lf.load(F + (size_t)(warp == 0 ? 0 : 3 - warp) * LFE, lane);
            Tv um0[kE];  // deep: the coarsest row
            if (deep) {
                const Wv *p[kE];
                Tv x[kE];
#pragma unroll
                for (int s = 0; s < kE; ++s) p[s] = tid + s * nt < n ? (const Wv *)m.lf[L] + nr + tid + s * nt : nullptr;
                flag_wait<Tv, kE>(p, x, tag, &ctl->timeout, fail);
#pragma unroll
                for (int s = 0; s < kE; ++s)
                    if (tid + s * nt < NW) Bf[Sh::at(tid + s * nt)] = x[s];
                if (__syncthreads_or(fail)) {
                    fail = true;
                    break;
                }
                if constexpr (Sh::group) {
                    if (tid < 128) group_line_solve<Tv, M>(FC, Bf, s_x, tid, 1);
                } else {
                    if (warp == 0) warp_line_solve<Tv, M>(FC, Bf, lane);
                }
                __syncthreads();
#pragma unroll
                for (int s = 0; s < kE; ++s) um0[s] = tid + s * nt < NW ? Bf[Sh::at(tid + s * nt)] : (Tv)0;
            }
            Tv z[4][kE], fx[3 * kE], ux[3 * kE];  // z: cz below ra, ra + 1, ra + 2 and above it
            {
                const Wv *p[3 * kE];
                const Wv *f = (const Wv *)m.lf[l] + (size_t)ra * nr, *uc = (const Wv *)m.lu[l + 1] + (size_t)q * nr;
#pragma unroll
                for (int s = 0; s < kE; ++s) {
                    const int j = tid + s * nt;
#pragma unroll
                    for (int w = 0; w < 4; ++w) z[w][s] = j < n ? czl[(size_t)w * nr + j] : (Tv)0;
#pragma unroll
                    for (int w = 0; w < 3; ++w) p[3 * s + w] = j < n ? f + (size_t)w * nr + j : nullptr;
                }
                flag_wait<Tv, 3 * kE>(p, fx, tag, &ctl->timeout, fail);
                if (!deep && decide < 0 && (decide = check()) != 0) break;
                if (!deep) {
                    // coarse rows below ra, between (row ra + 1) and above
                    // ra + 2: q, q + 1, q + 2, zero at the level's ends
                    const bool lo = q > 0, hi = q + 2 < nzc - 1;
#pragma unroll
                    for (int s = 0; s < kE; ++s) {
                        const int j = tid + s * nt;
                        p[3 * s] = j < n && lo ? uc + j : nullptr;
                        p[3 * s + 1] = j < n ? uc + nr + j : nullptr;
                        p[3 * s + 2] = j < n && hi ? uc + (size_t)2 * nr + j : nullptr;
                    }
                    flag_wait<Tv, 3 * kE>(p, ux, tag, &ctl->timeout, fail);
                } else {
#pragma unroll
                    for (int s = 0; s < kE; ++s) {
                        ux[3 * s] = ux[3 * s + 2] = 0;
                        ux[3 * s + 1] = um0[s];
                    }
                }
            }
            // right-hand sides: the reds get f plus the coarse correction
            // injected at the rows beside them; the black line its own f
#pragma unroll
            for (int s = 0; s < kE; ++s) {
                const int j = tid + s * nt;
                if (j >= NW) break;
                Tv *B = Bf + Sh::at(j);
                B[0] = fx[3 * s] + z[0][s] * ux[3 * s] + z[1][s] * ux[3 * s + 1];
                B[BL] = fx[3 * s + 2] + z[2][s] * ux[3 * s + 1] + z[3][s] * ux[3 * s + 2];
            }
            if (__syncthreads_or(fail)) {
                fail = true;
                break;
            }
            if constexpr (Sh::group) {  // a red line each half of the block
                const int w = tid >> 7;
                group_line_solve<Tv, M>(F + (size_t)2 * w * LFE, Bf + w * BL, s_x + 256 * w, tid & 127, 1 + w);
            } else {
                if (warp < 2) warp_line_solve<Tv, M, kReg>(lf, Bf + warp * BL, lane);
            }
            __syncthreads();
#pragma unroll
            for (int s = 0; s < kE; ++s) {
                const int j = tid + s * nt;
                if (j >= NW) break;
                Tv *B = Bf + Sh::at(j);
                const Tv x0 = B[0], x1 = B[BL];
                B[2 * BL] = fx[3 * s + 1] + z[1][s] * x0 + z[2][s] * x1;
                if (j < n) {
                    Fv::store(u + j, x0, tag);
                    // red ra + 2 is also the next unit's ra: one stores it
                    if (ra + 2 == m.nz[l] - 2) Fv::store(u + (size_t)2 * nr + j, x1, tag);
                }
            }
            __syncthreads();
            if constexpr (Sh::group) {
                if (tid < 128) group_line_solve<Tv, M>(F + LFE, Bf + 2 * BL, s_x, tid, 1);
            } else {
                if (warp == 2) warp_line_solve<Tv, M, kReg>(lf, Bf + 2 * BL, lane);
            }
            __syncthreads();
            if (nun > S) request(g + S, slot);
#pragma unroll
            for (int s = 0; s < kE; ++s) {
                const int j = tid + s * nt;
                if (j < n) Fv::store(u + nr + j, Bf[2 * BL + Sh::at(j)], tag);
            }
        }
        if (!fail && decide < 0) decide = check();
        if (decide == 3)
            for (int t = bid; t < ntile; t += P)
                for (int e = tid; e < tn; e += nt) {
                    const int j = t * tw + (e & (tw - 1));
                    if (j < n) phi[(size_t)(1 + (e >> ltw)) * nr + j] = 0.0;
                }
        if (fail || decide != 0) break;
    }
    // leave with no copy in flight (bounded waits), the tags used up
    if (fail && tid == 0) atomicExch(&ctl->timeout, 1);
#pragma unroll 1
    for (int r = 0; r <= kMaxSlots; ++r) ld_wait(ld, r);
    if (bid == 0 && tid == 0) *m.epoch = ep + (unsigned)cyc + 4u;
}

// MINB: blocks per SM the registers must allow: one for a reactor's solve
// alone, two for the solves of a batch of reactors, which share SMs (one where
// one_block says so).
template <typename Tv, int M, int MINB>
__global__ void __launch_bounds__(kSolveThreads, one_block(M, sizeof(Tv) == 8) ? 1 : MINB)
    k_solve_persistent(const MGFast *__restrict__ mp, double *phi, int nr, SolveLayout lay, double tol,
                       int max_cycles) {
    solve_body<Tv, M, MINB == 1>(mp, phi, nr, lay, tol, max_cycles, blockIdx.x, gridDim.x);
}

// The solves of several reactors (one line chunk M, one precision) in one
// cooperative launch: job k takes blocks [block0, block0 + nblocks) and hands
// its words to its own blocks only, so the reactors proceed side by side.
template <typename Tv, int M>
__global__ void __launch_bounds__(kSolveThreads, one_block(M, sizeof(Tv) == 8) ? 1 : 2)
    k_solve_multi(const SolveJob *__restrict__ jobs, int njobs) {
    int lo = 0, hi = njobs - 1;  // the job whose block range holds this block
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (jobs[mid].block0 <= (int)blockIdx.x)
            lo = mid;
        else
            hi = mid - 1;
    }
    const SolveJob &j = jobs[lo];
    const int bid = (int)blockIdx.x - j.block0;
    if (bid >= j.nblocks) return;
    solve_body<Tv, M, false>(j.mp, j.phi, j.nr, j.lay, j.tol, j.max_cycles, bid, j.nblocks);
}

}  // namespace

size_t mg_line_factor_elems(int nr, bool f64) { return (size_t)line_elems(line_chunk(nr - 1), f64); }

// tiles of one to eight columns (FP64: to kWideTile), the last one whole, FP64
// with two neighbour columns each
constexpr int kWideTile = 32;
size_t mg_tile_elems(int nz, int nr, bool with_neighbours) {
    return with_neighbours ? (size_t)nz * (nr + kWideTile) * 3 : (size_t)nz * (nr + 8);
}

namespace {

template <typename Tv, int M>
void *solve_fn(int minb) {
    return minb == 2 ? (void *)k_solve_persistent<Tv, M, 2> : (void *)k_solve_persistent<Tv, M, 1>;
}

template <typename Tv>
void *multi_kernel(int M) {
    switch (M) {
        case 1: return (void *)k_solve_multi<Tv, 1>;
        case 2: return (void *)k_solve_multi<Tv, 2>;
        case 4: return (void *)k_solve_multi<Tv, 4>;
        case 8: return (void *)k_solve_multi<Tv, 8>;
        case 16: return (void *)k_solve_multi<Tv, 16>;
        default: return (void *)k_solve_multi<Tv, 32>;
    }
}

template <typename Tv>
void *solve_kernel(int M, int minb) {
    switch (M) {
        case 1: return solve_fn<Tv, 1>(minb);
        case 2: return solve_fn<Tv, 2>(minb);
        case 4: return solve_fn<Tv, 4>(minb);
        case 8: return solve_fn<Tv, 8>(minb);
        case 16: return solve_fn<Tv, 16>(minb);
        default: return solve_fn<Tv, 32>(minb);
    }
}

// kernels whose dynamic shared memory can pass 48 KB on the largest meshes
constexpr size_t kSolveSmemLimit = 220 * 1024;

void raise_smem_limits() {
    static bool done = false;
    if (done) return;
    // (what the kernel's static shared memory leaves of a block's 227 KB)
    auto raise = [](void *fn) {
        cudaFuncAttributes a;
        if (cudaFuncGetAttributes(&a, fn) == cudaSuccess)
            cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)std::min(kSolveSmemLimit, 227 * 1024 - a.sharedSizeBytes));
    };
    raise((void *)k_setup_levels);
    for (int M = 1; M <= 32; M <<= 1) {
        for (int minb = 1; minb <= 2; ++minb) {
            raise(solve_kernel<float>(M, minb));
            raise(solve_kernel<double>(M, minb));
        }
        raise(multi_kernel<float>(M));
        raise(multi_kernel<double>(M));
    }
    done = true;
}

}  // namespace

namespace {

__global__ void k_solve_done(const MGCtl *c, StepCtl *s, int cont) { solve_report(c, s, cont); }

}  // namespace

void mg_fast_geometry(const MGFast &m, int nr, double dr, std::vector<double> &out) {
    // FV face areas of the annuli (z faces) and cylinder sides (r faces)
    // over the node distances, Sec. 2.4: the set-up kernels only scale them
    // by 1 + chi of the face
    out.assign((size_t)(2 * m.nlev + 1) * nr, 0.0);
    for (int l = 0; l < m.nlev; ++l) {
        const double dz = m.dz[l];
        double *gz = out.data() + (size_t)2 * l * nr, *gr = gz + nr;
        for (int j = 0; j < nr; ++j) {
            const double rp = (j + 0.5) * dr, rm = j > 0 ? (j - 0.5) * dr : 0.0;
            gz[j] = (kPi * (rp * rp - rm * rm)) / dz;
            gr[j] = 2.0 * kPi * rp * dz / dr;
        }
    }
    double *ga = out.data() + (size_t)2 * m.nlev * nr;
    for (int j = 0; j < nr; ++j) {
        const double rp = (j + 0.5) * dr, rm = j > 0 ? (j - 0.5) * dr : 0.0;
        ga[j] = (kPi * (rp * rp - rm * rm)) * m.dz[0] / kEps0;
    }
}

void mg_fast_upload(MGFast &m, cudaStream_t st) {
    cudaMemcpyAsync(m.self, &m, sizeof(MGFast), cudaMemcpyHostToDevice, st);
    cudaStreamSynchronize(st);
}

size_t tile_bytes(int tw, int nz) { return ((size_t)(tw + 2) * nz * sizeof(double) + 127) & ~(size_t)127; }

// Residual tiles for the job's number of blocks, no wider than the layout has
// room for: the widest, but for those that would leave a block without one.  A
// tile of a short mesh fills half a block's threads at 4 columns and costs a
// fixed chain of trips to L2.
void fit_tiles(SolveJob &j) {
    if (!j.lay.tw_max) return;
    j.lay.tw = j.lay.tw_max;
    while (j.lay.tw > 4 && (j.nr - 1 + j.lay.tw / 2 - 1) / (j.lay.tw / 2) <= j.nblocks) j.lay.tw /= 2;
    j.lay.offT = (int)tile_bytes(j.lay.tw, j.nz);
}

// The launch shape of one reactor's one-launch solve (shared-memory layout,
// blocks, kernel); false when it cannot be launched.
bool solve_job(const FieldDims &fd, MGFast &m, double *phi, bool mixed, double tol, int max_cycles, bool wide,
               SolveJob &job) {
    const int nz = fd.nz, nr = fd.nr, n = nr - 1;
    const int M = line_chunk(n);
    raise_smem_limits();
    int dev = 0, nsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const size_t es = mixed ? sizeof(float) : sizeof(double);
    const size_t LFE = (size_t)line_elems(M, !mixed || m.nlev == 1);
    SolveLayout lay{};
    const int L = m.nlev - 1;
    size_t off = 0;
    auto take = [&](size_t b) {
        const size_t o = off;
        off += (b + 127) & ~(size_t)127;
        return (int)o;
    };
    int grid = 1, most = 1;
    const int minb = wide ? 1 : 2;
    if (L == 0) {
        take((size_t)line_buffer(M, true) * sizeof(double));
        lay.offC = take(LFE * sizeof(double));
        lay.tw = 4;
    } else {
        // residual tiles of 4 columns (a 32-byte sector of flagged words per
        // row) while there are as many SMs, and on the FP64 path alone, whose
        // factor lines leave no room for more; else 8, or what fit_tiles takes
        const bool one = one_block(M, !mixed), fit = one && !wide;
        lay.tw = fit ? kWideTile : mixed && (!wide || n > 4 * nsm) ? 8 : 4;
        // the line buffers of the line phases share their space with the residual phase's tile (with its two neighbour columns) and
        // restriction buffers (very tall meshes: narrower tiles)
        const size_t line = (size_t)3 * line_buffer(M, !mixed) * es;
        const size_t fac = LFE * es + (size_t)3 * LFE * es + 512;
        size_t tile = 0, both = 0;
        for (;; lay.tw /= 2) {
            tile = tile_bytes(lay.tw, nz);
            both = std::max(line, tile + (size_t)lay.tw * (2 * nz + kMaxLevels) * es);
            // (FP64: room for the static exchange buffers too)
            if (lay.tw == 1 || both + fac + (mixed ? 0 : 8192) <= kSolveSmemLimit) break;
        }
        lay.offT = (int)tile;
        if (fit && lay.tw > 4) lay.tw_max = lay.tw;
        take(both);
        lay.offC = take(LFE * es);
        // a block per tile and per unit of the line phases
        const int units = (2 << L) - 2 - L, tw = std::min(lay.tw, fit ? 4 : 8), ntile = (n + tw - 1) / tw;
        most = std::min(nsm, std::max(units, ntile));
        grid = wide ? most : std::max(1, (nz - 1) / 2);
        // factor slots: all of a block's units, as far as they fit (a batch's
        // blocks: two to an SM)
        const size_t room = wide ? kSolveSmemLimit : kSolveSmemLimit / 2;
        const int want = std::min(kMaxSlots, (units + grid - 1) / grid);
        lay.slots = 1;
        while (lay.slots < want && off + (size_t)(lay.slots + 1) * 3 * LFE * es <= room) ++lay.slots;
        lay.offF = take((size_t)lay.slots * 3 * LFE * es);
    }
    const size_t sp = off;
    void *fn = mixed ? solve_kernel<float>(M, minb) : solve_kernel<double>(M, minb);
    int per_sm = 0;
    if (sp <= kSolveSmemLimit) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kSolveThreads, sp);
    if (per_sm < 1) return false;
    grid = std::min(std::min(grid, nsm * per_sm), kMaxSolveBlocks);
    job.mp = m.self;
    job.phi = phi;
    job.nz = nz;
    job.nr = nr;
    job.lay = lay;
    job.tol = tol;
    job.max_cycles = max_cycles;
    job.block0 = 0;
    job.nblocks = grid;
    job.most = lay.tw_max ? std::max(most, grid) : grid;
    job.M = M;
    job.mixed = mixed ? 1 : 0;
    job.smem = sp;
    job.fn = fn;
    fit_tiles(job);
    return true;
}

template <typename Ts>
static void launch_setup_lines(int M, int grid, cudaStream_t st, const MGFast *mp, const double *chi, int nr, int mean,
                               const RhsArgs &a, const StepCtl *ctl) {
    constexpr int nt = kSetupThreads;
    switch (M) {
        case 1: k_setup_lines<Ts, 1><<<grid, nt, 0, st>>>(mp, chi, nr, mean, a, ctl); break;
        case 2: k_setup_lines<Ts, 2><<<grid, nt, 0, st>>>(mp, chi, nr, mean, a, ctl); break;
        case 4: k_setup_lines<Ts, 4><<<grid, nt, 0, st>>>(mp, chi, nr, mean, a, ctl); break;
        case 8: k_setup_lines<Ts, 8><<<grid, nt, 0, st>>>(mp, chi, nr, mean, a, ctl); break;
        case 16: k_setup_lines<Ts, 16><<<grid, nt, 0, st>>>(mp, chi, nr, mean, a, ctl); break;
        default: k_setup_lines<Ts, 32><<<grid, nt, 0, st>>>(mp, chi, nr, mean, a, ctl); break;
    }
}

int mg_fast_solve(const FieldDims &fd, MGFast &m, const FieldSource &src, double V,
                  const double *phi_zL, double *phi, bool warm, bool mixed, double tol,
                  int max_cycles, double *rel_res, int *launches, StepCtl *sctl, cudaStream_t st,
                  bool v_from_ctl, bool setup, cudaEvent_t at_solve, bool wide, SolveJob *defer,
                  double *phi_prev, bool report, cudaEvent_t after, MGCtl *pinned) {
    const int nz = fd.nz, nr = fd.nr, n = nr - 1, ng = nz * nr;
    const int M = line_chunk(n);
    const int nlev = m.nlev;
    int L = 0;
    raise_smem_limits();
    MGFast *mp = m.self;  // uploaded once (mg_fast_upload)
    const RhsArgs ra{src.rho, phi, phi_zL, V, warm ? 0 : 1, v_from_ctl ? 1 : 0, warm ? phi_prev : nullptr};
    if (setup) {
        int lc = 2;  // four columns: a 32-byte sector a row, and blocks for most SMs
        size_t smem = 0;
        while ((smem = (((size_t)2 * nz + kMaxLevels) * sizeof(double)) << lc) > kSolveSmemLimit && lc > 0) --lc;
        if (src.Ne || nlev > 1) {
            k_setup_levels<<<(nr + (1 << lc) - 1) >> lc, 256, smem, st>>>(mp, nr, lc, src, sctl);
            ++L;
        }
        if (after) cudaStreamWaitEvent(st, after, 0);
        // line factors in the V-cycle's type (nz = 3: the single row is phi's
        // own, solved in FP64)
        int rows = 0;
        for (int l = 0; l < nlev; ++l) rows += m.nz[l];
        const int mean = fd.chi_face == PIC_CHI_MEAN;
        if (mixed && nlev > 1)
            launch_setup_lines<float>(M, rows, st, mp, src.chi, nr, mean, ra, sctl);
        else
            launch_setup_lines<double>(M, rows, st, mp, src.chi, nr, mean, ra, sctl);
        ++L;
    } else {
        // the operator is the one of the previous solve
        if (after) cudaStreamWaitEvent(st, after, 0);
        k_rhs_bc<<<(ng + 255) / 256, 256, 0, st>>>(mp, ra, nz, nr, sctl);
        ++L;
    }
    // all cycles in one cooperative launch
    SolveJob job;
    if (!solve_job(fd, m, phi, mixed, tol, max_cycles, wide, job)) {
        if (at_solve) cudaEventRecord(at_solve, st);
        if (launches) *launches += L;
        return kSolveNoLaunch;
    }
    if (defer) {
        // the caller launches it with other reactors' solves (mg_multi_launch)
        *defer = job;
        if (launches) *launches += L;
        return 0;
    }
    const SolveLayout lay = job.lay;
    const size_t sp = job.smem;
    void *fn = job.fn;
    const int grid = job.nblocks;
    int nrv = nr, mc = max_cycles;
    double tv = tol;
    void *args[] = {(void *)&mp, (void *)&phi, (void *)&nrv, (void *)&lay, (void *)&tv, (void *)&mc};
    // the highest stream priority: when a step sorts beside the solve, the
    // solve's blocks take SMs as soon as the sort's short blocks retire
    static int prio = 1;
    if (prio > 0) {
        int least = 0, greatest = 0;
        cudaDeviceGetStreamPriorityRange(&least, &greatest);
        prio = greatest;
    }
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(grid);
    lc.blockDim = dim3(kSolveThreads);
    lc.dynamicSmemBytes = sp;
    lc.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    at[1].id = cudaLaunchAttributePriority;
    at[1].val.priority = prio;
    lc.attrs = at;
    lc.numAttrs = 2;
    if (at_solve) cudaEventRecord(at_solve, st);
    const cudaError_t e = cudaLaunchKernelExC(&lc, fn, args);
    ++L;
    if (e != cudaSuccess) {
        if (launches) *launches += L;
        return kSolveNoLaunch;
    }
    if (sctl) {
        // inside a timestep: the result stays on the device
        if (report) {
            k_solve_done<<<1, 1, 0, st>>>(m.ctl, sctl, setup ? 0 : 1);
            ++L;
        }
        if (launches) *launches += L;
        return 0;
    }
    if (launches) *launches += L;
    MGCtl local;
    MGCtl *cp = pinned ? pinned : &local;
    cudaMemcpyAsync(cp, m.ctl, sizeof(MGCtl), cudaMemcpyDeviceToHost, st);
    cudaStreamSynchronize(st);
    const MGCtl ch = *cp;
    if (ch.timeout) {
        if (rel_res) *rel_res = 0.0;
        return kSolveTimeout;
    }
    if (ch.zero_rhs) {
        if (rel_res) *rel_res = 0.0;
        return 0;
    }
    if (rel_res) *rel_res = ch.bnorm > 0 ? ch.last_res / ch.bnorm : 0.0;
    return ch.converged ? ch.cycles : -ch.cycles - 1;
}

std::vector<std::pair<int, int>> mg_multi_plan(std::vector<SolveJob> &jobs, bool &concurrent) {
    std::stable_sort(jobs.begin(), jobs.end(), [](const SolveJob &a, const SolveJob &b) {
        return a.mixed != b.mixed ? a.mixed < b.mixed : a.M < b.M;
    });
    std::vector<std::pair<int, int>> out;
    int dev = 0, nsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    // the kinds' ranges, their kernels and their share of the GPU: every
    // kind's launch gets SMs in proportion to the blocks its jobs would take
    // alone, so that the launches of all kinds fit the GPU together
    struct Kind {
        size_t a, b;
        void *fn;
        size_t smem;
        int want;
    };
    std::vector<Kind> kinds;
    int want_all = 0;
    for (size_t a = 0; a < jobs.size();) {
        size_t b = a;
        size_t smem = 0;
        int want = 0;
        while (b < jobs.size() && jobs[b].mixed == jobs[a].mixed && jobs[b].M == jobs[a].M) {
            smem = std::max(smem, jobs[b].smem);
            want += jobs[b].nblocks;
            ++b;
        }
        void *fn = jobs[a].mixed ? multi_kernel<float>(jobs[a].M) : multi_kernel<double>(jobs[a].M);
        kinds.push_back({a, b, fn, smem, want});
        want_all += want;
        a = b;
    }
    // side by side only while that leaves the jobs a fair part of their
    // blocks: with more than six times the GPU's co-resident blocks wanted
    // (64 c4 reactors), the kinds take the whole GPU one after another
    // (measured: 16 and 32 reactors 1.08 -> 1.35 and 1.21 -> 1.35e10
    // particle-steps/s side by side, 64 reactors 1.48 -> 1.32e10)
    int per_min = 1 << 30;
    for (const Kind &k : kinds) {
        int per_sm = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k.fn, kSolveThreads, k.smem);
        per_min = std::min(per_min, std::max(per_sm, 1));
    }
    const bool side_by_side = want_all <= 6 * per_min * nsm;
    concurrent = side_by_side;
    for (const Kind &k : kinds) {
        int per_sm = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k.fn, kSolveThreads, k.smem);
        const int share = side_by_side ? std::max(1, (int)((double)nsm * k.want / std::max(want_all, 1))) : nsm;
        const int cap = std::max(1, per_sm * share);
        // launches of at most `cap` blocks and one block per job at least
        for (size_t a = k.a; a < k.b;) {
            const size_t e = std::min(k.b, a + (size_t)cap);
            int want = 0;
            for (size_t j = a; j < e; ++j) want += jobs[j].nblocks;
            const double scale = (double)cap / want;
            int used = 0;
            for (size_t j = a; j < e; ++j) {
                jobs[j].nblocks = std::max(1, std::min(jobs[j].most, (int)(jobs[j].nblocks * scale)));
                used += jobs[j].nblocks;
            }
            while (used > cap) {  // the one-block floors overshot: trim the largest
                size_t big = a;
                for (size_t j = a; j < e; ++j)
                    if (jobs[j].nblocks > jobs[big].nblocks) big = j;
                if (jobs[big].nblocks <= 1) break;
                --jobs[big].nblocks;
                --used;
            }
            used = 0;
            for (size_t j = a; j < e; ++j) {
                fit_tiles(jobs[j]);
                jobs[j].block0 = used;
                jobs[j].fn = k.fn;
                jobs[j].smem = k.smem;
                used += jobs[j].nblocks;
            }
            out.push_back({(int)a, (int)e});
            a = e;
        }
    }
    return out;
}

int mg_multi_launch(const std::vector<SolveJob> &jobs, int j0, int j1, const SolveJob *jobs_dev,
                    cudaStream_t st) {
    if (j1 <= j0) return 0;
    int blocks = 0;
    for (int k = j0; k < j1; ++k) blocks = std::max(blocks, jobs[k].block0 + jobs[k].nblocks);
    const SolveJob *tab = jobs_dev + j0;
    int nj = j1 - j0;
    void *args[] = {(void *)&tab, (void *)&nj};
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(blocks);
    lc.blockDim = dim3(kSolveThreads);
    lc.dynamicSmemBytes = jobs[j0].smem;
    lc.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    lc.attrs = at;
    lc.numAttrs = 1;
    return cudaLaunchKernelExC(&lc, jobs[j0].fn, args) == cudaSuccess ? 0 : kSolveNoLaunch;
}

}  // namespace pic
