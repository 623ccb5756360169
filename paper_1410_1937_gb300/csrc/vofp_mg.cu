// Coarse-grid correction of the red-black preconditioner (templated on the precision of the iteration).
//
// CG on the red Schur complement (vofp_rbc.cuh, vofp_rb.cuh) has a residual r on the black unknowns
// and no preconditioner of its own; its iteration count grows with the grid (2500 at 512x256x128 to
// a residual of 1e-8) because one iteration moves information by two cells.  Here the search
// direction comes from z = r + B r, where B solves approximately for the smooth part of the error:
//   restriction    b_1 = sum over the 2x2x2 cells of an aggregate of sq r   (sq = 1/s: the residual
//                  of the unscaled equation; red entries are 0 after the elimination)
//   hierarchy      level l + 1 is the Galerkin operator of piecewise constants on 2x2x2 aggregates of
//                  level l: its face coefficients are sums of the fine ones across the aggregate's
//                  faces, so every level is again a 7-point operator with positive face coefficients
//   V-cycle        one red-black Gauss-Seidel sweep before (red, black) and one after (black, red) the
//                  next level's correction, so that B is symmetric and positive
//   prolongation   z = r + sq e_1 of the aggregate
// B is additive (z = r + B r, no second fine-grid sweep), so the fine grid costs one pass more over r
// and the weights sq, and r.z = r.r + e_1.b_1 comes from the coarse vectors.  Measured (solves to
// 1e-12, the plain iteration and with the correction): 512x256x128 5120 iterations in 574 ms, 432 in
// 106 ms; 256x128x64 2368 in 86 ms, 336 in 25.6 ms; 64x48x40 832 in 18.7 ms, 272 in 12 ms.  FP64 mode
// (hierarchy and vectors in FP64): 512x256x128 3248 iterations in 2178 ms, 416 in 411 ms; 128x64x64 872 in
// 43.7 ms, 216 in 20 ms; 125x61x47 792 in 34.7 ms, 232 in 20.7 ms.
//
// Merge groups: the group's unknown is present at every member cell of the expanded vectors.  Its
// master represents it in the restriction (weight sq); the other members, small cells whose own
// aggregate may have next to no coupling, carry weight -1 like the red cells of the full-grid vectors:
// left out of the sums, and given the master's z.  On the compact vectors an even-parity master sits after the N/2 pairs; a mask byte per
// aggregate says which of its four even cells are such masters.
//
// Everything is gathered (no floating-point atomics), so a solve is bitwise reproducible.
#include <algorithm>
#include <cmath>
#include <cstdlib>

#include "vofp_kernels.cuh"

namespace vofp {
namespace {

constexpr int kNT = 256;
// levels of at most kBottomCells cells are taken by one block, a thread per cell
constexpr int kBottomCells = 512;
constexpr int kBottomThreads = 512;
constexpr int kMaxBottom = 10;                    // levels from kBottomCells down to one cell
// six values per cell; every chain of levels from at most 512 cells down has at most 1023 in all
constexpr int kBottomValues = 6 * 2 * kBottomCells;
static_assert(kBottomValues * sizeof(double) <= 48 * 1024, "static shared memory");

int grid_n(long long n) {
    return (int)std::max(1LL, std::min((n + kNT - 1) / kNT, (long long)num_sms() * 8));
}
// one wave of the update and direction kernels (three 256-thread blocks per SM)
int grid_fine(long long items) {
    return (int)std::max(1LL, std::min((items + kNT - 1) / kNT, (long long)num_sms() * 3));
}

// ---- hierarchy ---------------------------------------------------------------------------------

__global__ void k_mg_max(long long n, const double* __restrict__ diag, unsigned long long* out) {
    double m = 0.0;
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n; c += (long long)gridDim.x * blockDim.x)
        m = fmax(m, diag[c]);
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(out, (unsigned long long)__double_as_longlong(m));
}

// The hierarchy is kept in FP32 relative to the largest diagonal: coefficients times 4^-h, weights
// times 2^-h with 4^h about the largest diagonal (powers of two: no rounding; the correction
// sq A^-1 sq does not change).
__device__ __forceinline__ int mg_exponent(const unsigned long long* dmax) {
    const double m = __longlong_as_double((long long)*dmax);
    return (m > 0.0 && isfinite(m)) ? (ilogb(m) >> 1) : 0;
}

template <typename T>
struct MgCoef {
    const T *tx, *ty, *tz, *di;
};

// level 1 from the FP64 operator
template <typename T>
__global__ void k_mg_coarsen_fine(Dims d, int nx1, int ny1, int nz1, const double* __restrict__ Tx,
                                  const double* __restrict__ Ty, const double* __restrict__ Tz,
                                  const double* __restrict__ diag, const unsigned long long* dmax,
                                  T* __restrict__ tx, T* __restrict__ ty, T* __restrict__ tz, T* __restrict__ ex) {
    const long long n1 = (long long)nx1 * ny1 * nz1;
    const double g = scalbn(1.0, -2 * mg_exponent(dmax));
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n1; q += (long long)gridDim.x * blockDim.x) {
        const int I = int(q % nx1), J = int((q / nx1) % ny1), K = int(q / ((long long)nx1 * ny1));
        double sx = 0.0, sy = 0.0, sz = 0.0, se = 0.0;
        for (int k = 2 * K; k < min(2 * K + 2, d.nz); ++k)
            for (int j = 2 * J; j < min(2 * J + 2, d.ny); ++j)
                for (int i = 2 * I; i < min(2 * I + 2, d.nx); ++i) {
                    const long long c = i + (long long)d.nx * j + d.plane * k;
                    const double x = Tx[c], y = Ty[c], z = Tz[c];
                    // the six face coefficients in the order the assembly sums them: what the
                    // diagonal has beyond is the p = 0 domain faces', exactly 0 elsewhere
                    double s = x + y + z;
                    if (i > 0) s += Tx[c - 1];
                    if (j > 0) s += Ty[c - d.nx];
                    if (k > 0) s += Tz[c - d.plane];
                    se += fmax(diag[c] - s, 0.0);
                    if (i & 1) sx += x;
                    if (j & 1) sy += y;
                    if (k & 1) sz += z;
                }
        tx[q] = (T)(sx * g);
        ty[q] = (T)(sy * g);
        tz[q] = (T)(sz * g);
        ex[q] = (T)(se * g);
    }
}

template <typename T>
__global__ void k_mg_coarsen(int nx, int ny, int nz, const T* __restrict__ tx, const T* __restrict__ ty,
                             const T* __restrict__ tz, const T* __restrict__ ex, int nx1, int ny1, int nz1,
                             T* __restrict__ ctx, T* __restrict__ cty, T* __restrict__ ctz,
                             T* __restrict__ cex) {
    const long long n1 = (long long)nx1 * ny1 * nz1;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n1; q += (long long)gridDim.x * blockDim.x) {
        const int I = int(q % nx1), J = int((q / nx1) % ny1), K = int(q / ((long long)nx1 * ny1));
        double sx = 0.0, sy = 0.0, sz = 0.0, se = 0.0;
        for (int k = 2 * K; k < min(2 * K + 2, nz); ++k)
            for (int j = 2 * J; j < min(2 * J + 2, ny); ++j)
                for (int i = 2 * I; i < min(2 * I + 2, nx); ++i) {
                    const long long c = i + (long long)nx * (j + (long long)ny * k);
                    se += (double)ex[c];
                    if (i & 1) sx += (double)tx[c];
                    if (j & 1) sy += (double)ty[c];
                    if (k & 1) sz += (double)tz[c];
                }
        ctx[q] = (T)sx;
        cty[q] = (T)sy;
        ctz[q] = (T)sz;
        cex[q] = (T)se;
    }
}

// inverse diagonals of a level from its stored coefficients (0 where a cell has no coupling)
template <typename T>
__global__ void k_mg_dinv(int nx, int ny, int nz, const T* __restrict__ tx, const T* __restrict__ ty,
                          const T* __restrict__ tz, const T* __restrict__ ex, T* __restrict__ di) {
    const long long n = (long long)nx * ny * nz, pl = (long long)nx * ny;
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n; c += (long long)gridDim.x * blockDim.x) {
        const int i = int(c % nx), j = int((c / nx) % ny), k = int(c / pl);
        double s = (double)tx[c] + (double)ty[c] + (double)tz[c] + (double)ex[c];
        if (i > 0) s += (double)tx[c - 1];
        if (j > 0) s += (double)ty[c - nx];
        if (k > 0) s += (double)tz[c - pl];
        di[c] = s > 1e-30 ? (T)(1.0 / s) : T(0);
    }
}

// weights of the vector entries (before the merge groups): sq of a non-red cell with an unknown, 0 of one
// without, -1 (in no sum; z stays 0) of a red one: the iteration kernel writes no row there, so q holds
// whatever the passes before the loop left, and with a starting pressure those are rounding errors that r
// gathers in every iteration.  On the compact vectors entries past N/2 belong to group members (-1)
template <bool COMPACT, typename T>
__global__ void k_mg_weights(Dims d, long long n, long long nh, const double* __restrict__ sq,
                             const int32_t* __restrict__ root, const uint32_t* __restrict__ red,
                             const unsigned long long* dmax, T* __restrict__ w) {
    const double g = scalbn(1.0, -mg_exponent(dmax));
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
        if (COMPACT) {
            if (t >= nh) {
                w[t] = T(-1);
                continue;
            }
            const long long row = t / (d.nx >> 1);
            const int j = int(row % d.ny), k = int(row / d.ny);
            const long long c = 2 * t + 1 - ((j + k) & 1);   // black cell of pair t
            w[t] = root[c] < 0 ? T(0) : (T)(sq[c] * g);
        } else {
            w[t] = is_slave(red, t) ? T(-1) : root[t] < 0 ? T(0) : (T)(sq[t] * g);
        }
    }
}

// Most that w^2 D^-1 of a master's aggregate may be: the part of its own r that one level adds to its z.  (Cells without a
// group have about a quarter; see k_mg_groups.  At 0.5 the operators named there take a tenth fewer iterations still, but
// ordinary ones other bits as well; at 1 nearly all of those keep theirs.)
constexpr double kMaxSelf = 1.0;

// merge groups: the master's entry and aggregate (rep) and its weight, -1 for the other members.  The master stands
// for couplings of all of the group's cells, and its aggregate has only those of the cells that lie in it: where they
// are few the aggregate seems as good as free and answers with a multiple of what it should.  So the weight is at most
// what keeps w^2 D^-1 at kMaxSelf.  Without that, with cells of less than half their volume merged: 232x32x206 hull with
// every tenth face closed, to 1e-9, mixed 4160 iterations (1984 without the correction) -> 528; 132x80x102 sphere 608
// (832) -> 208, FP64 328 (696) -> 184.  On the compact vectors also the aggregates' mask bits of even-parity masters
// and their entries, four per aggregate (read, and written, only where the bit is set).  Member entries: gref
// (compact) or the cells
template <bool COMPACT, typename T>
__global__ void k_mg_groups(Dims d, int ng, int nx1, int ny1, const int* __restrict__ gptr,
                            const int* __restrict__ gcells, const int* __restrict__ gref,
                            const double* __restrict__ sq, const unsigned long long* dmax, const T* __restrict__ di,
                            T* __restrict__ w, int2* __restrict__ rep, uint32_t* __restrict__ mask, int* __restrict__ even) {
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= ng) return;
    const double sg = scalbn(1.0, -mg_exponent(dmax));
    const int u0 = gptr[g], u1 = gptr[g + 1];
    int i, j, k;
    cell_ijk(d, gcells[u0], i, j, k);
    const int t = (i >> 1) + nx1 * ((j >> 1) + ny1 * (k >> 1)), u = 2 * (k & 1) + (j & 1);
    double ws = sq[gcells[u0]] * sg;
    if (ws * ws * (double)di[t] > kMaxSelf) ws = sqrt(kMaxSelf / (double)di[t]);
    for (int u = u0; u < u1; ++u)
        w[COMPACT ? gref[u] : gcells[u]] = u == u0 ? (T)ws : T(-1);
    rep[g] = make_int2(COMPACT ? gref[u0] : gcells[u0], t);
    if (!COMPACT || ((i + j + k) & 1)) return;
    atomicOr(&mask[t >> 2], (1u << u) << (8 * (t & 3)));
    even[4LL * t + u] = gref[u0];
}

// per block the sums of the scaled couplings along x, y and z
__global__ void __launch_bounds__(kNT) k_mg_couplings(long long n, const float* __restrict__ tx, const float* __restrict__ ty,
                                                      const float* __restrict__ tz, double* __restrict__ part) {
    __shared__ double sh[3][kNT / 32];
    AccF2 a[3];
    for (long long c = blockIdx.x * (long long)kNT + threadIdx.x; c < n; c += (long long)gridDim.x * kNT) {
        a[0].add(tx[c], 1.0f);
        a[1].add(ty[c], 1.0f);
        a[2].add(tz[c], 1.0f);
    }
#pragma unroll
    for (int e = 0; e < 3; ++e) {
        const double v = warp_sum(a[e].value());
        if ((threadIdx.x & 31) == 0) sh[e][threadIdx.x >> 5] = v;
    }
    __syncthreads();
    if (threadIdx.x < 3) part[3 * blockIdx.x + threadIdx.x] = sum_warps(sh[threadIdx.x], kNT / 32);
}

// ---- fine grid: update with restriction, and z --------------------------------------------------

// The entries of A neighbouring aggregates (I .. I + A - 1, J, K) of a vector, E words per aggregate row:
// on the compact vectors the pairs I, I + 1 of rows 2J, 2J+1 in planes 2K, 2K+1 (four 8-byte words; the
// pairs of a row and the aggregates along x are a multiple of four there); on full-grid vectors the
// eight cells of one aggregate.
template <bool COMPACT>
struct MgEntries {
    static constexpr int A = COMPACT ? 2 : 1;
    static constexpr int W = COMPACT ? 4 : 8;       // words of a thread
    long long at[W];
    bool in[W];
    __device__ __forceinline__ void set(const Dims& d, int I, int J, int K) {
#pragma unroll
        for (int e = 0; e < W; ++e) {
            const int dj = COMPACT ? e & 1 : (e >> 1) & 1, dk = COMPACT ? e >> 1 : e >> 2, di = COMPACT ? 0 : e & 1;
            const int j = 2 * J + dj, k = 2 * K + dk;
            in[e] = j < d.ny && k < d.nz && (COMPACT || 2 * I + di < d.nx);
            const long long row = j + (long long)d.ny * k;
            at[e] = COMPACT ? I + (long long)(d.nx >> 1) * row : 2LL * I + di + d.nx * row;
        }
    }
};
// one word of A values (two floats: an 8-byte word)
__device__ __forceinline__ void mg_get(float (&v)[2], const float* a, long long at) {
    const float2 x = *reinterpret_cast<const float2*>(a + at);
    v[0] = x.x;
    v[1] = x.y;
}
template <typename T>
__device__ __forceinline__ void mg_get(T (&v)[1], const T* a, long long at) { v[0] = a[at]; }
__device__ __forceinline__ void mg_put(const float (&v)[2], float* a, long long at) {
    *reinterpret_cast<float2*>(a + at) = make_float2(v[0], v[1]);
}
template <typename T>
__device__ __forceinline__ void mg_put(const T (&v)[1], T* a, long long at) { a[at] = v[0]; }

// alpha = r.z / p.Ap;  r -= alpha q;  r.r;  b_1 = restriction of the new r.  With UPD = false only the
// restriction (the start of an inner solve, whose r and r.r are there).  Memory-bound (8.6 bytes per
// cell on the compact vectors: 31 us at 512x256x128 under ncu, 43 with 4-byte words): a thread takes two
// aggregates along x at a time there (12 independent 8-byte loads), the first ones before it sums p.Ap
// and divides.
template <bool COMPACT, bool UPD, typename T>
__global__ void __launch_bounds__(kNT, 3)
k_mg_update(const Dims d, const int nx1, const int ny1, const int n1, const long long nh, const long long nvec,
            T* __restrict__ r, const T* __restrict__ q, const T* __restrict__ w,
            const uint8_t* __restrict__ mask, const int* __restrict__ even, T* __restrict__ b1, CgScalars* sc,
            double* __restrict__ partials, unsigned int* __restrict__ counter,
            cudaGraphConditionalHandle handle, int use_handle, const double* __restrict__ pq_part, int npq) {
    using En = MgEntries<COMPACT>;
    constexpr int A = En::A, W = En::W;
    __shared__ double sh[32];
    __shared__ double s_alpha;
    __shared__ int s_flags;
    grid_dep_wait();
    const int stride = gridDim.x * kNT, items = n1 / A, nxa = nx1 / A;
    int t = blockIdx.x * kNT + threadIdx.x;
    En en;
    T rv[W][A], qv[W][A], wv[W][A];
    uint32_t mk = 0;
    auto load = [&]() {
        const int tj = t / nxa, K = tj / ny1;
        en.set(d, (t - tj * nxa) * A, tj - K * ny1, K);
#pragma unroll
        for (int e = 0; e < W; ++e) {
#pragma unroll
            for (int a = 0; a < A; ++a) {
                rv[e][a] = qv[e][a] = T(0);
                wv[e][a] = T(-1);
            }
            if (!en.in[e]) continue;
            mg_get(rv[e], r, en.at[e]);
            if (UPD) mg_get(qv[e], q, en.at[e]);
            mg_get(wv[e], w, en.at[e]);
        }
        if (COMPACT) mk = *reinterpret_cast<const uint16_t*>(mask + (long long)A * t);
    };
    if (t < items) load();
    if (UPD) {
        double pq_sum = 0.0, v = 0.0;
        for (int i = threadIdx.x; i < npq; i += kNT) v += __ldcg(&pq_part[i]);
        v = warp_sum(v);
        if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
        __syncthreads();
        if (threadIdx.x == 0) pq_sum = sum_warps<true>(sh, kNT / 32);
        if (threadIdx.x == 0) {
            const double rr = sc->rr, rz = sc->rz, pq = pq_sum;
            // rr == 0: the residual vanished exactly (later unrolled iterations are no-ops)
            const bool ok = sc->status == VOFP_OK && pq > 0.0 && isfinite(pq) && isfinite(rr) && rr > 0.0 && rz > 0.0;
            const bool broke = !ok && !(rr == 0.0 && sc->status == VOFP_OK);
            s_alpha = ok ? rz / pq : 0.0;
            s_flags = broke ? 1 : 0;
        }
        __syncthreads();
    }
    const T na = UPD ? -(T)s_alpha : T(0);
    typename AccFor<T>::type acc;
    while (t < items) {
        T b[A];
#pragma unroll
        for (int a = 0; a < A; ++a) b[a] = T(0);
#pragma unroll
        for (int e = 0; e < W; ++e) {
#pragma unroll
            for (int a = 0; a < A; ++a) {
                if (UPD) rv[e][a] = fmav(na, qv[e][a], rv[e][a]);
                if (wv[e][a] >= T(0)) {
                    if (UPD) acc.add(rv[e][a], rv[e][a]);
                    b[a] = fmav(wv[e][a], rv[e][a], b[a]);
                }
            }
            if (UPD && en.in[e]) mg_put(rv[e], r, en.at[e]);
        }
        if (COMPACT) {
            // even-parity masters of these aggregates (rare)
            for (; mk; mk &= mk - 1) {
                const int f = __ffs(mk) - 1, a = f >> 3, at = even[4 * ((long long)A * t + a) + (f & 7)];
                T v = r[at];
                if (UPD) {
                    v = fmav(na, q[at], v);
                    r[at] = v;
                    acc.add(v, v);
                }
                const T s = w[at] * v;
                b[0] += a == 0 ? s : T(0);
                b[A - 1] += a == A - 1 && A > 1 ? s : T(0);
            }
        }
        mg_put(b, b1, (long long)A * t);
        t += stride;
        if (t < items) load();
    }
    if (!UPD) return;
    // the other even-parity members of merge groups (copies: not in the sums)
    if (COMPACT)
        for (long long c = nh + blockIdx.x * kNT + threadIdx.x; c < nvec; c += stride)
            if (w[c] < T(0)) r[c] = fmav(na, q[c], r[c]);
    double tot;
    if (grid_reduce<true>(acc.value(), partials, counter, sh, &tot)) {
        const bool broke = s_flags != 0;
        sc->rr_prev = sc->rr;
        sc->rr = tot;
        sc->rz_prev = sc->rz;
        sc->alpha = s_alpha;
        sc->iter += 1;
        sc->iter_total += 1;
        if ((broke || !isfinite(tot)) && sc->status == VOFP_OK && !sc->timing) {
            sc->status = VOFP_ERR_BREAKDOWN;
            sc->alpha = 0.0;
        }
        const bool stop = broke || !isfinite(tot) || tot <= sc->inner_target * sc->inner_target * sc->rr0 ||
                          sc->iter >= sc->max_iter || sc->iter_total >= sc->max_iter;
        if (stop) sc->inner_done = 1;
        if (use_handle && stop) cudaGraphSetConditional(handle, 0);
    }
}

// z = r + sq e_1 and r.z = r.r + e_1.b_1; beta of the next direction.  Merge groups: every member
// takes the master's z (formed here from r: no order between the two loops).
template <bool COMPACT, typename T>
__global__ void __launch_bounds__(kNT, 3)
k_mg_direction(const Dims d, const int nx1, const int ny1, const int n1, const T* __restrict__ r,
               const T* __restrict__ w, const T* __restrict__ e1, const T* __restrict__ b1,
               T* __restrict__ z, const int ng, const int2* __restrict__ rep, const int* __restrict__ gptr,
               const int* __restrict__ gidx, CgScalars* sc, double* __restrict__ partials,
               unsigned int* __restrict__ counter, int start) {
    using En = MgEntries<COMPACT>;
    constexpr int A = En::A, W = En::W;
    __shared__ double sh[32];
    grid_dep_wait();
    typename AccFor<T>::type acc;
    const int stride = gridDim.x * kNT, items = n1 / A, nxa = nx1 / A;
    // the groups first, from the last blocks: their chain of loads overlaps the stream
    for (int g = (gridDim.x - 1 - blockIdx.x) * kNT + threadIdx.x; g < ng; g += stride) {
        const int2 m = rep[g];
        const int u0 = gptr[g], u1 = gptr[g + 1];
        const T v = fmav(w[m.x], e1[m.y], r[m.x]);
        for (int u = u0; u < u1; ++u) z[gidx[u]] = v;
    }
    for (int t = blockIdx.x * kNT + threadIdx.x; t < items; t += stride) {
        const int tj = t / nxa, K = tj / ny1;
        En en;
        en.set(d, (t - tj * nxa) * A, tj - K * ny1, K);
        T ev[A], bv[A], rv[W][A], wv[W][A];
        mg_get(ev, e1, (long long)A * t);
        mg_get(bv, b1, (long long)A * t);
#pragma unroll
        for (int e = 0; e < W; ++e)
            if (en.in[e]) {
                mg_get(rv[e], r, en.at[e]);
                mg_get(wv[e], w, en.at[e]);
            }
#pragma unroll
        for (int a = 0; a < A; ++a) acc.add(ev[a], bv[a]);
#pragma unroll
        for (int e = 0; e < W; ++e) {
            if (!en.in[e]) continue;
            bool all = true;
            T v[A];
#pragma unroll
            for (int a = 0; a < A; ++a) {
                all &= wv[e][a] >= T(0);
                v[a] = fmav(wv[e][a], ev[a], rv[e][a]);
            }
            if (all) {
                mg_put(v, z, en.at[e]);
            } else {   // a group member beside it: written below
#pragma unroll
                for (int a = 0; a < A; ++a)
                    if (wv[e][a] >= T(0)) z[en.at[e] + a] = v[a];
            }
        }
    }
    double tot;
    if (grid_reduce<true>(acc.value(), partials, counter, sh, &tot)) {
        const double rz = sc->rr + tot;
        sc->rz = rz;
        double beta = sc->rz_prev > 0.0 ? rz / sc->rz_prev : 0.0;
        if (start) beta *= sc->bscale;
        if (!isfinite(beta) || !(rz > 0.0) || sc->status != VOFP_OK) beta = 0.0;
        sc->beta = beta;
    }
}

// ---- V-cycle -----------------------------------------------------------------------------------

// A block takes 8 x 4 x 2 aggregates of the next level, 16 x 8 x 4 cells of its own, with a two-cell
// halo of values in shared memory, so that one kernel does the level's whole sweep: the red cells
// (two-cell halo), the black ones (one-cell halo), the red ones again.  The levels are small and a
// sweep is a chain of three dependent steps, so the time is latency: a thread has at most one cell
// of each step (two of the first), and every coefficient it will need is loaded before the first
// barrier, so that a kernel waits for memory once.  (Tiles of 32 x 8 x 8 cells with 256 threads that
// loaded in each step: 13 us for the small levels, 29-33 us at 2.1 M cells.)
constexpr int kTX = 16, kTY = 8, kTZ = 4;
constexpr int kPX = kTX + 4, kPY = kTY + 4, kPZ = kTZ + 4;
constexpr int kReds = kPX / 2 * kPY * kPZ;                          // 960
constexpr int kBlacks = (kTX + 2) / 2 * (kTY + 2) * (kTZ + 2);      // 540
constexpr int kCore = kTX / 2 * kTY * kTZ;                          // 256 red cells, as many black
constexpr int kTileThreads = 576;
static_assert(kReds <= 2 * kTileThreads && kBlacks <= kTileThreads && kCore <= kTileThreads, "one cell per thread and step");

struct MgGeom {
    int nx, ny, nz;      // the level
    int mx, my, mz;      // the next level
    int tiles_x, tiles_y;
};

// One cell of a step: its place in the tile, and what its sum over the faces takes.
template <typename T>
struct MgCell {
    int at;              // index in the tile; -1: none
    long long c;         // cell; -1 outside the grid
    T xp, xm, yp, ym, zp, zm;
    __device__ __forceinline__ void load(const MgGeom& g, const MgCoef<T>& m, int i, int j, int k) {
        const long long pl = (long long)g.nx * g.ny;
        c = -1;
        xp = xm = yp = ym = zp = zm = T(0);
        if (i < 0 || i >= g.nx || j < 0 || j >= g.ny || k < 0 || k >= g.nz) return;
        c = i + g.nx * (long long)j + pl * k;
        xp = m.tx[c];                            // 0 for the last cell of a row
        yp = m.ty[c];
        zp = m.tz[c];
        if (i > 0) xm = m.tx[c - 1];
        if (j > 0) ym = m.ty[c - g.nx];
        if (k > 0) zm = m.tz[c - pl];
    }
    __device__ __forceinline__ T sum(const T* xs) const {
        const T* p = xs + at;
        T s = xp * p[1];
        s = fmav(xm, p[-1], s);
        s = fmav(yp, p[kPX], s);
        s = fmav(ym, p[-kPX], s);
        s = fmav(zp, p[kPX * kPY], s);
        return fmav(zm, p[-kPX * kPY], s);
    }
};

// DOWN (before the next level): red cells from b alone (the first guess is 0), black cells, and the
// red cells' residual, summed over each aggregate into the next level's b (the black cells' residual
// is 0).  Else (after it): red cells from b and the next level's x, black cells, red cells; x.
template <bool DOWN, typename T>
__global__ void __launch_bounds__(kTileThreads, 2)
k_mg_level(const MgGeom g, const MgCoef<T> m, const T* __restrict__ b, const T* __restrict__ en,
           T* __restrict__ out) {
    __shared__ T xs[kPX * kPY * kPZ];
    const int t = threadIdx.x;
    const int tb = blockIdx.x, bx = tb % g.tiles_x, by = (tb / g.tiles_x) % g.tiles_y, bz = tb / (g.tiles_x * g.tiles_y);
    const int i0 = bx * kTX, j0 = by * kTY, k0 = bz * kTZ;
    // black cell of the pair (i0 - 1 + 2a, + 1): the sum of its coordinates is odd
    MgCell<T> bc, rc;
    bc.at = rc.at = -1;
    T bd = T(0), bb = T(0), rd = T(0), rb = T(0);
    if (t < kBlacks) {
        const int a = t % (kTX / 2 + 1), y = (t / (kTX / 2 + 1)) % (kTY + 2), z = t / ((kTX / 2 + 1) * (kTY + 2));
        const int j = j0 - 1 + y, k = k0 - 1 + z, x = 2 * a + ((j + k) & 1);
        bc.at = (x + 1) + kPX * ((y + 1) + kPY * (z + 1));
        bc.load(g, m, i0 - 1 + x, j, k);
        if (bc.c >= 0) bd = m.di[bc.c];
    }
    // red cell: the four of an aggregate in neighbouring lanes
    const int dj = t & 1, dk = (t >> 1) & 1, ca = (t >> 2) % (kTX / 2), cy = (t >> 2) / (kTX / 2) % (kTY / 2),
              cz = (t >> 2) / (kTX / 2 * (kTY / 2));
    const int rx = 2 * ca + ((dj + dk) & 1);
    if (t < kCore) {
        rc.at = (rx + 2) + kPX * ((2 * cy + dj + 2) + kPY * (2 * cz + dk + 2));
        rc.load(g, m, i0 + rx, j0 + 2 * cy + dj, k0 + 2 * cz + dk);
        if (!DOWN && rc.c >= 0) rd = m.di[rc.c];
    }
    int at[2];
    long long hc[2], he[2];
    T hd[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int u = t + q * kTileThreads;
        at[q] = -1;
        hc[q] = -1;
        hd[q] = T(0);
        if (u >= kReds) continue;
        const int a = u % (kPX / 2), y = (u / (kPX / 2)) % kPY, z = u / (kPX / 2 * kPY);
        const int j = j0 - 2 + y, k = k0 - 2 + z, x = 2 * a + ((j + k) & 1), i = i0 - 2 + x;
        at[q] = x + kPX * (y + kPY * z);
        if (i < 0 || i >= g.nx || j < 0 || j >= g.ny || k < 0 || k >= g.nz) continue;
        hc[q] = i + g.nx * ((long long)j + (long long)g.ny * k);
        hd[q] = m.di[hc[q]];
        if (!DOWN) he[q] = (i >> 1) + g.mx * ((long long)(j >> 1) + (long long)g.my * (k >> 1));
    }
    // the operator does not change inside a solve; b and en come from the kernels before
    grid_dep_wait();
    grid_dep_trigger();
    if (bc.c >= 0 && bc.at >= 0) bb = b[bc.c];
    if (!DOWN && rc.at >= 0 && rc.c >= 0) rb = b[rc.c];
#pragma unroll
    for (int q = 0; q < 2; ++q)
        if (at[q] >= 0) {
            T v = T(0);
            if (hc[q] >= 0) v = DOWN ? hd[q] * b[hc[q]] : fmav(hd[q], b[hc[q]], en[he[q]]);
            xs[at[q]] = v;
        }
    __syncthreads();
    if (bc.at >= 0) xs[bc.at] = bc.c >= 0 ? bd * (bb + bc.sum(xs)) : T(0);
    __syncthreads();
    if (t >= kCore) return;
    T s = rc.c >= 0 ? rc.sum(xs) : T(0);
    if (DOWN) {
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        s += __shfl_xor_sync(0xffffffffu, s, 2);
        const int I = bx * (kTX / 2) + ca, J = by * (kTY / 2) + cy, K = bz * (kTZ / 2) + cz;
        if ((t & 3) == 0 && I < g.mx && J < g.my && K < g.mz) out[I + g.mx * ((long long)J + (long long)g.my * K)] = s;
    } else {
        // this red cell and the black one of its pair
        const int j = j0 + 2 * cy + dj, k = k0 + 2 * cz + dk, ib = i0 + (rx ^ 1);
        if (rc.c >= 0) out[rc.c] = rd * (rb + s);
        if (ib < g.nx && j < g.ny && k < g.nz)
            out[ib + g.nx * ((long long)j + (long long)g.ny * k)] = xs[rc.at + ((rx & 1) ? -1 : 1)];
    }
}

// The same sweeps for levels large enough to fill the chip: 32 x 8 x 8 cells per block, a thread takes
// a column of pairs along z, so that its indices are formed once per column (the one-cell-per-thread
// form above spends most of its issue slots on them: 41 us a sweep at 2.1 M cells).  Blocks whose halo
// lies inside the grid skip the bounds checks.
constexpr int kLX = 32, kLY = 8, kLZ = 8;
constexpr int kRX = kLX + 4, kRY = kLY + 4, kRZ = kLZ + 4;
constexpr int kLargeThreads = 256;
constexpr long long kLargeCells = 600 * 1000;
static_assert(kRX / 2 * kRY <= kLargeThreads && kLX / 2 * kLY * 2 == kLargeThreads, "columns per block");

template <bool DOWN, bool INNER, typename T>
__device__ __forceinline__ void large_sweep(const MgGeom& g, const MgCoef<T>& m, const T* __restrict__ b,
                                            const T* __restrict__ en, T* __restrict__ out, T* xs, int i0,
                                            int j0, int k0) {
    const int t = threadIdx.x, nx = g.nx, pl = g.nx * g.ny;
    auto face_sum = [&](int c, int i, int j, int k, const T* p) {
        T s = m.tx[c] * p[1];
        if (INNER || i > 0) s = fmav(m.tx[c - 1], p[-1], s);
        s = fmav(m.ty[c], p[kRX], s);
        if (INNER || j > 0) s = fmav(m.ty[c - nx], p[-kRX], s);
        s = fmav(m.tz[c], p[kRX * kRY], s);
        if (INNER || k > 0) s = fmav(m.tz[c - pl], p[-kRX * kRY], s);
        return s;
    };
    if (t < kRX / 2 * kRY) {
        const int a = t % (kRX / 2), y = t / (kRX / 2), i2 = i0 - 2 + 2 * a, j = j0 - 2 + y;
        const bool row = INNER || (j >= 0 && j < g.ny);
#pragma unroll
        for (int z = 0; z < kRZ; ++z) {
            const int k = k0 - 2 + z, par = (j + k) & 1, i = i2 + par;
            T v = T(0);
            if (INNER || (row && k >= 0 && k < g.nz && i >= 0 && i < nx)) {
                const int c = i + nx * j + pl * k;
                v = m.di[c] * b[c];
                if (!DOWN) v = fmav(m.di[c], b[c], en[(i >> 1) + g.mx * ((j >> 1) + g.my * (k >> 1))]);
            }
            xs[2 * a + par + kRX * (y + kRY * z)] = v;
        }
    }
    __syncthreads();
    if (t < (kLX / 2 + 1) * (kLY + 2)) {
        const int a = t % (kLX / 2 + 1), y = t / (kLX / 2 + 1), i2 = i0 - 1 + 2 * a, j = j0 - 1 + y;
        const bool row = INNER || (j >= 0 && j < g.ny);
#pragma unroll 5
        for (int z = 0; z < kLZ + 2; ++z) {
            const int k = k0 - 1 + z, par = (j + k) & 1, i = i2 + par;
            T* p = xs + (2 * a + par + 1) + kRX * ((y + 1) + kRY * (z + 1));
            T v = T(0);
            if (INNER || (row && k >= 0 && k < g.nz && i >= 0 && i < nx)) {
                const int c = i + nx * j + pl * k;
                v = m.di[c] * (b[c] + face_sum(c, i, j, k, p));
            }
            *p = v;
        }
    }
    __syncthreads();
    // pair a of row y, four planes from z0
    const int a = t % (kLX / 2), y = (t / (kLX / 2)) % kLY, z0 = 4 * (t / (kLX / 2 * kLY));
    const int ip = i0 + 2 * a, j = j0 + y;
#pragma unroll
    for (int z = z0; z < z0 + 4; z += 2) {
        T s2 = T(0);
#pragma unroll
        for (int dk = 0; dk < 2; ++dk) {
            const int k = k0 + z + dk, par = (j + k) & 1, i = ip + par;
            const T* p = xs + (2 * a + par + 2) + kRX * ((y + 2) + kRY * (z + dk + 2));
            if (!(INNER || (j < g.ny && k < g.nz && ip < nx))) continue;
            const int c = i + nx * j + pl * k;
            if (DOWN) {
                if (INNER || i < nx) s2 += face_sum(c, i, j, k, p);
            } else {
                if (INNER || i < nx) out[c] = m.di[c] * (b[c] + face_sum(c, i, j, k, p));
                if (INNER || ip + (par ^ 1) < nx) out[c + 1 - 2 * par] = p[1 - 2 * par];
            }
        }
        if (DOWN) {
            s2 += __shfl_xor_sync(0xffffffffu, s2, kLX / 2);
            const int I = ip >> 1, J = j >> 1, K = (k0 + z) >> 1;
            if (!(y & 1) && I < g.mx && J < g.my && K < g.mz) out[I + g.mx * (J + g.my * K)] = s2;
        }
    }
}

template <bool DOWN, typename T>
__global__ void __launch_bounds__(kLargeThreads, 4)
k_mg_level_large(const MgGeom g, const MgCoef<T> m, const T* __restrict__ b, const T* __restrict__ en,
                 T* __restrict__ out) {
    __shared__ T xs[kRX * kRY * kRZ];
    const int tb = blockIdx.x, bx = tb % g.tiles_x, by = (tb / g.tiles_x) % g.tiles_y, bz = tb / (g.tiles_x * g.tiles_y);
    const int i0 = bx * kLX, j0 = by * kLY, k0 = bz * kLZ;
    grid_dep_wait();
    const bool inner = i0 > 2 && i0 + kLX + 2 <= g.nx && j0 > 2 && j0 + kLY + 2 <= g.ny && k0 > 2 && k0 + kLZ + 2 <= g.nz;
    if (inner)
        large_sweep<DOWN, true, T>(g, m, b, en, out, xs, i0, j0, k0);
    else
        large_sweep<DOWN, false, T>(g, m, b, en, out, xs, i0, j0, k0);
}

// The levels of at most kBottomCells cells in one block, a thread per cell, down to a single cell
// (which is solved) and back.  Level l keeps tx, ty, tz, D^-1, b, x, each of n[l] values.
template <typename T>
struct MgBottom {
    int levels;
    int nx[kMaxBottom], ny[kMaxBottom], nz[kMaxBottom];
    int off[kMaxBottom];                 // first T of the level in shared memory
    MgCoef<T> m[kMaxBottom];
    const T* b;
    T* x;
};

template <typename T>
__global__ void __launch_bounds__(kBottomThreads) k_mg_bottom(const MgBottom<T> a) {
    __shared__ T sm[kBottomValues];
    const int t = threadIdx.x;
    for (int l = 0; l < a.levels; ++l) {
        const int n = a.nx[l] * a.ny[l] * a.nz[l];
        T* p = sm + a.off[l];
        if (t < n) {
            p[t] = a.m[l].tx[t];
            p[n + t] = a.m[l].ty[t];
            p[2 * n + t] = a.m[l].tz[t];
            p[3 * n + t] = a.m[l].di[t];
        }
    }
    grid_dep_wait();
    grid_dep_trigger();
    {
        const int n = a.nx[0] * a.ny[0] * a.nz[0];
        if (t < n) sm[a.off[0] + 4 * n + t] = a.b[t];
    }
    __syncthreads();
    // sum of coefficient times neighbour's x over the faces of cell c
    auto sum = [&](const T* p, int n, int nx, int ny, int nz, int c, int i, int j, int k) {
        const int pl = nx * ny;
        const T* x = p + 5 * n;
        T s = T(0);
        if (i < nx - 1) s = fmav(p[c], x[c + 1], s);
        if (i > 0) s = fmav(p[c - 1], x[c - 1], s);
        if (j < ny - 1) s = fmav(p[n + c], x[c + nx], s);
        if (j > 0) s = fmav(p[n + c - nx], x[c - nx], s);
        if (k < nz - 1) s = fmav(p[2 * n + c], x[c + pl], s);
        if (k > 0) s = fmav(p[2 * n + c - pl], x[c - pl], s);
        return s;
    };
    for (int l = 0; l < a.levels; ++l) {
        const int nx = a.nx[l], ny = a.ny[l], nz = a.nz[l], n = nx * ny * nz;
        T* p = sm + a.off[l];
        const int r = t / nx, i = t - r * nx, k = r / ny, j = r - k * ny;
        const bool on = t < n, black = ((i + j + k) & 1) != 0;
        T* x = p + 5 * n;
        const T d = on ? p[3 * n + t] : T(0), b = on ? p[4 * n + t] : T(0);
        if (on) x[t] = black ? T(0) : d * b;
        __syncthreads();
        if (l == a.levels - 1) break;
        if (on && black) x[t] = d * (b + sum(p, n, nx, ny, nz, t, i, j, k));
        __syncthreads();
        const int mx = a.nx[l + 1], my = a.ny[l + 1], mz = a.nz[l + 1], mn = mx * my * mz;
        if (t < mn) {
            const int R = t / mx, I = t - R * mx, K = R / my, J = R - K * my;
            T s = T(0);
            for (int u = 0; u < 4; ++u) {
                const int dj = u & 1, dk = u >> 1, ii = 2 * I + ((dj + dk) & 1), jj = 2 * J + dj, kk = 2 * K + dk;
                if (ii < nx && jj < ny && kk < nz) s += sum(p, n, nx, ny, nz, ii + nx * (jj + ny * kk), ii, jj, kk);
            }
            sm[a.off[l + 1] + 4 * mn + t] = s;
        }
        __syncthreads();
    }
    for (int l = a.levels - 2; l >= 0; --l) {
        const int nx = a.nx[l], ny = a.ny[l], nz = a.nz[l], n = nx * ny * nz;
        T* p = sm + a.off[l];
        const int r = t / nx, i = t - r * nx, k = r / ny, j = r - k * ny;
        const bool on = t < n, black = ((i + j + k) & 1) != 0;
        T* x = p + 5 * n;
        const T d = on ? p[3 * n + t] : T(0), b = on ? p[4 * n + t] : T(0);
        const int mx = a.nx[l + 1], my = a.ny[l + 1], mn = mx * my * a.nz[l + 1];
        if (on && !black) x[t] = fmav(d, b, sm[a.off[l + 1] + 5 * mn + (i >> 1) + mx * ((j >> 1) + my * (k >> 1))]);
        __syncthreads();
        if (on && black) x[t] = d * (b + sum(p, n, nx, ny, nz, t, i, j, k));
        __syncthreads();
        if (on && !black) x[t] = d * (b + sum(p, n, nx, ny, nz, t, i, j, k));
        __syncthreads();
    }
    const int n = a.nx[0] * a.ny[0] * a.nz[0];
    if (t < n) a.x[t] = sm[a.off[0] + 5 * n + t];
}

// ---- host --------------------------------------------------------------------------------------

template <typename T, bool DOWN>
void launch_level(vofp_ctx* c, cudaStream_t st, bool pdl, const MgLevel<T>& l, const MgLevel<T>& n) {
    const bool large = l.n >= kLargeCells;
    const int tx = large ? kLX : kTX, ty = large ? kLY : kTY, tz = large ? kLZ : kTZ;
    const MgGeom g{l.nx, l.ny, l.nz, n.nx, n.ny, n.nz, ceil_div(l.nx, tx), ceil_div(l.ny, ty)};
    const dim3 grid((unsigned)(g.tiles_x * g.tiles_y * ceil_div(l.nz, tz)));
    const MgCoef<T> m{l.tx, l.ty, l.tz, l.di};
    const T *b = l.b, *en = n.x;
    T* out = DOWN ? n.b : l.x;
    if (large)
        launch_dep(c, pdl, k_mg_level_large<DOWN, T>, grid, dim3(kLargeThreads), 0, st, g, m, b, en, out);
    else
        launch_dep(c, pdl, k_mg_level<DOWN, T>, grid, dim3(kTileThreads), 0, st, g, m, b, en, out);
}

template <typename T>
int bottom_level(const MgSet<T>& m) {
    int l = 0;
    while (m.lv[l].n > kBottomCells) ++l;
    return l;
}

template <typename T>
void vcycle(vofp_ctx* c, cudaStream_t st, bool pdl, const MgSet<T>& m) {
    const int lb = bottom_level(m), nl = (int)m.lv.size();
    for (int l = 0; l < lb; ++l) launch_level<T, true>(c, st, pdl, m.lv[l], m.lv[l + 1]);
    MgBottom<T> a{};
    a.levels = nl - lb;
    int off = 0;
    for (int l = lb; l < nl; ++l) {
        const MgLevel<T>& v = m.lv[l];
        a.nx[l - lb] = v.nx;
        a.ny[l - lb] = v.ny;
        a.nz[l - lb] = v.nz;
        a.off[l - lb] = off;
        off += 6 * (int)v.n;
        a.m[l - lb] = MgCoef<T>{v.tx, v.ty, v.tz, v.di};
    }
    a.b = m.lv[lb].b;
    a.x = m.lv[lb].x;
    launch_dep(c, pdl, k_mg_bottom<T>, dim3(1), dim3(kBottomThreads), 0, st, a);
    for (int l = lb - 1; l >= 0; --l) launch_level<T, false>(c, st, pdl, m.lv[l], m.lv[l + 1]);
}

template <typename T>
MgSet<T>& set_of(vofp_ctx* c) {
    if constexpr (sizeof(T) == 4)
        return c->mgf;
    else
        return c->mgd;
}
// the vectors of the iteration: compact or full-grid FP32 ones, full-grid FP64 ones
template <bool COMPACT, typename T>
T* vec_r(vofp_ctx* c) {
    if constexpr (COMPACT)
        return c->rbc_r;
    else if constexpr (sizeof(T) == 4)
        return c->rf;
    else
        return c->r;
}
template <bool COMPACT, typename T>
const T* vec_q(vofp_ctx* c) {
    if constexpr (COMPACT)
        return c->rbc_q;
    else if constexpr (sizeof(T) == 4)
        return c->qf;
    else
        return c->q;
}

template <bool COMPACT, typename T>
void launch_direction(vofp_ctx* c, cudaStream_t st, bool pdl, int start) {
    MgSet<T>& m = set_of<T>(c);
    const MgLevel<T>& l = m.lv[0];
    launch_dep(c, pdl, k_mg_direction<COMPACT, T>, dim3(grid_fine(l.n / MgEntries<COMPACT>::A)), dim3(kNT), 0, st, c->d,
               l.nx, l.ny, (int)l.n, (const T*)vec_r<COMPACT, T>(c), (const T*)m.w, (const T*)l.x, (const T*)l.b, m.z,
               c->ngroups, reinterpret_cast<const int2*>(m.rep), (const int*)c->gptr,
               (const int*)(COMPACT ? c->rbc_gref : c->gcells), c->sc, c->partials, c->counters, start);
}
template <bool COMPACT, bool UPD, typename T>
void launch_update(vofp_ctx* c, cudaStream_t st, bool pdl, cudaGraphConditionalHandle h, int use_h, int npq) {
    MgSet<T>& m = set_of<T>(c);
    const MgLevel<T>& l = m.lv[0];
    const long long nh = COMPACT ? c->rbc_nh : c->d.n, nv = COMPACT ? c->rbc_nh + c->rbc_ne : c->d.n;
    launch_dep(c, pdl, k_mg_update<COMPACT, UPD, T>, dim3(grid_fine(l.n / MgEntries<COMPACT>::A)), dim3(kNT), 0, st, c->d,
               l.nx, l.ny, (int)l.n, nh, nv, vec_r<COMPACT, T>(c), vec_q<COMPACT, T>(c), (const T*)m.w,
               (const uint8_t*)c->mg_mask, (const int*)c->mg_even, l.b, c->sc, c->partials, c->counters, h, use_h,
               (const double*)(c->partials + kPqBase), npq);
}

// give back a hierarchy's memory
template <typename T>
void drop(vofp_ctx* c, MgSet<T>& m) {
    for (MgLevel<T>& l : m.lv)
        for (T** p : {&l.tx, &l.ty, &l.tz, &l.di, &l.ex, &l.b, &l.x}) c->release(p, l.n);
    if (sizeof(T) == 4 && !m.lv.empty()) {
        c->release(&c->mg_mask, (m.lv[0].n + 3) / 4);
        c->release(&c->mg_even, 4 * m.lv[0].n);
    }
    c->release(&m.w, m.cap);
    c->release(&m.z, m.cap);
    c->release(&m.rep, 2 * m.rep_cap);
    m = MgSet<T>();
}

// The hierarchy and the weights of the current operator (once per operator and precision).
template <bool COMPACT, typename T>
vofp_status build(vofp_ctx* c) {
    MgSet<T>& m = set_of<T>(c);
    const Dims d = c->d;
    cudaStream_t st = c->stream;
    vofp_status s;
    if (m.lv.empty()) {
        int nx = d.nx, ny = d.ny, nz = d.nz;
        do {
            MgLevel<T> l{};
            l.nx = nx = (nx + 1) / 2;
            l.ny = ny = (ny + 1) / 2;
            l.nz = nz = (nz + 1) / 2;
            l.n = (long long)nx * ny * nz;
            m.lv.push_back(l);
        } while (m.lv.back().n > 1);
        for (MgLevel<T>& l : m.lv)
            for (T** p : {&l.tx, &l.ty, &l.tz, &l.di, &l.ex, &l.b, &l.x})
                if ((s = c->alloc(p, l.n))) return s;
        if (!c->mg_dmax && (s = c->alloc(&c->mg_dmax, 1))) return s;
    }
    const MgLevel<T>& l1 = m.lv[0];
    if (COMPACT) {
        if (!c->mg_even &&
            ((s = c->alloc(&c->mg_mask, (l1.n + 3) / 4)) || (s = c->alloc(&c->mg_even, 4 * l1.n))))
            return s;
        VOFP_CUDA_TRY(c, cudaMemsetAsync(c->mg_mask, 0, sizeof(uint32_t) * ((l1.n + 3) / 4), st));
    }
    const long long nv = COMPACT ? c->rbc_cap : d.n;
    if (nv > m.cap) {
        // entries past the vectors in use stay 0 (the tensor copies read whole boxes)
        c->release(&m.w, m.cap);
        c->release(&m.z, m.cap);
        m.cap = nv;
        if ((s = c->alloc(&m.w, nv)) || (s = c->alloc(&m.z, nv))) return s;
    }
    VOFP_CUDA_TRY(c, cudaMemsetAsync(m.z, 0, sizeof(T) * m.cap, st));
    if (c->ngroups > m.rep_cap) {
        c->release(&m.rep, 2 * m.rep_cap);
        m.rep_cap = c->ngroups + c->ngroups / 2 + 64;
        if ((s = c->alloc(&m.rep, 2 * m.rep_cap))) return s;
    }
    VOFP_CUDA_TRY(c, cudaMemsetAsync(c->mg_dmax, 0, sizeof(unsigned long long), st));
    launch(c, k_mg_max, grid_n(d.n), kNT, st, d.n, (const double*)c->diag, c->mg_dmax);
    const unsigned long long* dmax = c->mg_dmax;
    launch(c, k_mg_coarsen_fine<T>, ceil_div(l1.n, kNT), kNT, st, d, l1.nx, l1.ny, l1.nz, (const double*)c->Tx,
           (const double*)c->Ty, (const double*)c->Tz, (const double*)c->diag, dmax, l1.tx, l1.ty, l1.tz, l1.ex);
    for (size_t q = 0; q < m.lv.size(); ++q) {
        const MgLevel<T>& l = m.lv[q];
        if (q > 0) {
            const MgLevel<T>& f = m.lv[q - 1];
            launch(c, k_mg_coarsen<T>, ceil_div(l.n, kNT), kNT, st, f.nx, f.ny, f.nz, (const T*)f.tx, (const T*)f.ty,
                   (const T*)f.tz, (const T*)f.ex, l.nx, l.ny, l.nz, l.tx, l.ty, l.tz, l.ex);
        }
        launch(c, k_mg_dinv<T>, ceil_div(l.n, kNT), kNT, st, l.nx, l.ny, l.nz, (const T*)l.tx, (const T*)l.ty,
               (const T*)l.tz, (const T*)l.ex, l.di);
    }
    const long long n = COMPACT ? c->rbc_nh + c->rbc_ne : d.n;
    launch(c, k_mg_weights<COMPACT, T>, grid_n(n), kNT, st, d, n, COMPACT ? c->rbc_nh : d.n, (const double*)c->sq,
           (const int32_t*)c->root, (const uint32_t*)c->red_bits, dmax, m.w);
    if (c->ngroups > 0)
        launch(c, k_mg_groups<COMPACT, T>, ceil_div(c->ngroups, kNT), kNT, st, d, c->ngroups, l1.nx, l1.ny,
               (const int*)c->gptr, (const int*)c->gcells, (const int*)c->rbc_gref, (const double*)c->sq, dmax, (const T*)l1.di,
               m.w, reinterpret_cast<int2*>(m.rep), c->mg_mask, c->mg_even);
    VOFP_CUDA_TRY(c, cudaGetLastError());
    m.ok = true;
    return VOFP_OK;
}

template <bool COMPACT, typename T>
void precondition(vofp_ctx* c, cudaStream_t st, bool pdl, int start) {
    if (start) launch_update<COMPACT, false, T>(c, st, false, (cudaGraphConditionalHandle)0, 0, 0);
    vcycle<T>(c, st, pdl, set_of<T>(c));
    launch_direction<COMPACT, T>(c, st, pdl, start);
}

}  // namespace

// Whether the correction is likely to pay for this operator (an iteration with it takes about twice the time), from the
// mean scaled couplings m_x, m_y, m_z of a cell to its + neighbours: together half of the unit diagonal, less what closed
// faces, walls and unequal neighbours leave out.  With c = m / sum m:
//   sum m        at least kMgMinCoupling: where many faces are closed aggregates do not follow the open ones
//   anisotropy   largest c over smallest, at most kMgMaxAnisotropy: 2 x 2 x 2 aggregates join weakly coupled cells
//   condition    1 / lambda of the smoothest error of a uniform operator with these couplings, which is what the plain
//                iteration's count grows with: lambda = sum over the axes with p = 0 walls of c (pi / L)^2, L the cells
//                between two of them or twice those from one to the opposite wall; without any the least c (pi / cells)^2
//   sqrt(cells) condition / anisotropy  at least kMgMinScore
// 1225 solves of 246 random operators (65,536 to 5 M cells, aspect ratios of cells to 30 and of grids to 300, density
// ratios to 1e5, walls of every kind, open, with a tenth and with a third of the faces closed, tolerances 1e-7 to 1e-12;
// time without the correction over time with it, geometric mean): 1.56 with it everywhere, 209 solves slower by more than
// 5 %, the worst 0.33; 1.60 by this rule, which takes it for 871, with 35 slower, the worst 0.69.
static bool pays(const Dims& d, const int bc[6], const double m[3]) {
    const int n[3] = {d.nx, d.ny, d.nz};
    const double sum = m[0] + m[1] + m[2];
    if (!(sum >= kMgMinCoupling)) return false;
    double lambda = 0.0, closed = INFINITY, most = 0.0, least = INFINITY;
    for (int a = 0; a < 3; ++a) {
        if (n[a] == 1) continue;
        const double c = m[a] / sum, q = M_PI / n[a];
        const int ends = (bc[2 * a] == VOFP_BC_DIRICHLET) + (bc[2 * a + 1] == VOFP_BC_DIRICHLET);
        if (ends) lambda += c * q * q / (ends == 1 ? 4.0 : 1.0);
        closed = std::min(closed, c * q * q);
        most = std::max(most, c);
        least = std::min(least, c);
    }
    if (lambda == 0.0) lambda = closed;
    return most <= kMgMaxAnisotropy * least && std::sqrt((double)d.n) * least / (most * lambda) >= kMgMinScore;
}

// Grids below kMgMinCells, tolerances above kMgMaxRtol and operators for which it does not pay keep the plain
// iteration (VOFP_MG=0: every solve does, 2: none).
vofp_status mg_wanted(vofp_ctx* c, double rtol, bool* wanted) {
    const char* env = std::getenv("VOFP_MG");
    const int use = env ? std::atoi(env) : 1;
    *wanted = use == 2;
    if (use == 0 || use == 2 || c->d.n < kMgMinCells || !(rtol <= kMgMaxRtol)) return VOFP_OK;
    if (c->mg_pays < 0) {
        const int nb = grid_n(c->d.n);
        std::vector<double> part(3 * nb);
        launch(c, k_mg_couplings, nb, kNT, c->stream, c->d.n, (const float*)c->Txf, (const float*)c->Tyf, (const float*)c->Tzf,
               c->partials);
        VOFP_CUDA_TRY(c, cudaMemcpyAsync(part.data(), c->partials, sizeof(double) * part.size(), cudaMemcpyDeviceToHost,
                                         c->stream));
        VOFP_CUDA_TRY(c, cudaStreamSynchronize(c->stream));
        double m[3] = {0.0, 0.0, 0.0};
        for (size_t i = 0; i < part.size(); ++i) m[i % 3] += part[i];
        for (double& v : m) v /= (double)std::max(1LL, c->d.n - c->n_inactive);
        c->mg_pays = pays(c->d, c->bc, m);
    }
    *wanted = c->mg_pays != 0;
    return VOFP_OK;
}

// Where there is no memory for the hierarchy the solves of this operator are plain ones (ok stays false), and
// what was allocated is given back.
vofp_status mg_ensure(vofp_ctx* c, bool fp64) {
    bool& built = fp64 ? c->mgd.built : c->mgf.built;
    if (built) return VOFP_OK;
    (fp64 ? c->mgd.ok : c->mgf.ok) = false;
    const vofp_status s = fp64 ? build<false, double>(c) : c->rbc_ok ? build<true, float>(c) : build<false, float>(c);
    if (s == VOFP_ERR_OOM) {
        cudaGetLastError();   // (the refused allocation's)
        c->err.clear();
        if (fp64)
            drop(c, c->mgd);
        else
            drop(c, c->mgf);
    } else if (s) {
        return s;
    }
    built = true;
    return VOFP_OK;
}

// b_1 (at the start of a loop: from the new residual), the V-cycle, z, r.z and beta
void mg_precondition(vofp_ctx* c, cudaStream_t st, bool fp64, bool pdl, int start) {
    if (fp64)
        precondition<false, double>(c, st, pdl, start);
    else if (c->rbc_ok)
        precondition<true, float>(c, st, pdl, start);
    else
        precondition<false, float>(c, st, pdl, start);
}

// r -= alpha q, r.r, the inner loop's stop test and b_1; npq: block partials of p.Ap
void mg_update(vofp_ctx* c, cudaStream_t st, bool fp64, bool pdl, cudaGraphConditionalHandle h, int use_h, int npq) {
    if (fp64)
        launch_update<false, true, double>(c, st, pdl, h, use_h, npq);
    else if (c->rbc_ok)
        launch_update<true, true, float>(c, st, pdl, h, use_h, npq);
    else
        launch_update<false, true, float>(c, st, pdl, h, use_h, npq);
}

int mg_precondition_kernels(const vofp_ctx* c, bool fp64) {
    return 2 * (fp64 ? bottom_level(c->mgd) : bottom_level(c->mgf)) + 2;
}

}  // namespace vofp
