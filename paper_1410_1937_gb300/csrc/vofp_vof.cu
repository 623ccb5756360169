// VOF operator of Sec. 2.4: flux-error correction and operator-split advection of the volume
// fraction with a dilation term (FP64).
//
// Correction (one pass over the cells): face fluxes F = A (u - v) with A the open face area
// (aperture x face area) and u - v the relative velocity given on the faces; the cell's
// conservation error E = sum_i (F+_i - F-_i) (Eq. diverge) is removed along z,
//   F~+_z = F+_z - E A+_z / (A+_z + A-_z),   F~-_z = F-_z + E A-_z / (A+_z + A-_z),
// and the stage velocities are u^_i = dx_i F~_i / V = F~_i / (uncut face area): shared on x and y
// faces, per cell on z faces (the two cells of a z face may disagree).
//
// Stage along axis d (two passes): the piecewise-linear interface of every cell with 0 < phi < 1
// (normal m = -grad phi by central differences weighted (1, 2, 1) x (1, 2, 1) across the other
// axes; plane constant alpha with the fluid volume {m.x <= alpha} equal to phi V, by Newton steps),
// then per cell the fluid carried through its two d faces in slabs of thickness |u^| dt of the
// donor cell (the cell itself on outflow, the neighbour on inflow; the boundary cell on inflow
// through a domain face), and
//   implicit stage:  phi_new = (phi - (F+ - F-) / V) / (1 - dt (u^+ - u^-) / dx_d)
//   explicit stage:  phi_new =  phi - (F+ - F-) / V + dt phi (u^+ - u^-) / dx_d.
// The first two stages are implicit, the third explicit; the axes run x, y, z (order 0) or
// z, y, x (order 1).  Neighbours inside the body (no open volume) and outside the domain take the
// cell's own value in the normal; a slab is at most the donor cell; phi is not clipped.
//
// The FP64 rate (1.05 TFLOP/s) bounds this operator as soon as every cell does arithmetic: 100 FP64
// operations a cell take 1.6 ms at 512x256x128, its 392 bytes 1 ms.  So the work is kept to the cells
// that need it:
//   - the cells with 0 < phi < 1 (about one in a hundred) are listed by the pass that writes phi (the
//     correction for the first stage, each stage for the next), and the planes are formed one thread per
//     listed cell: a warp's FP64 instruction takes as long for one active lane as for 32, so full warps
//     matter, and no plane is written or read elsewhere;
//   - the plane constant starts from Newton steps in FP32 (75 times the FP64 rate), so that two FP64
//     steps finish it instead of nine;
//   - a stage copies phi where the cell and both neighbours are all full, or all empty, and the slabs stay
//     within half a cell: the advection and dilation terms cancel there.  The test is on the words' bits;
//     the other cells are listed and take the stage in full warps;
//   - the reciprocals of widths come from tables, and a slab's fluid is a fraction of its own unit cube (one
//     or two divisions);
//   - the correction multiplies by apertures only where they are not 1 and divides only where the two
//     z apertures differ from 1.
// One step of the 512x256x128 hull in waves at Courant number 0.4 on a projected field: 1.7 ms (32.7 ms
// with every cell's plane formed and stored and every cell's stage in full).
#include <algorithm>
#include <type_traits>

#include "vofp_internal.cuh"

namespace vofp {
namespace {

constexpr int kNT = 256;

int grid_cells(long long n) {
    return (int)std::max(1LL, std::min((n + kNT - 1) / kNT, (long long)num_sms() * 64));
}

// ---- fluid volume below a plane in a box -------------------------------------------------------

__device__ __forceinline__ uint32_t high_abs(double v) { return (uint32_t)__double2hiint(v) & 0x7fffffffu; }

__device__ __forceinline__ void sort3(double& a, double& b, double& c) {
    if (a > b) { const double t = a; a = b; b = t; }
    if (b > c) { const double t = b; b = c; c = t; }
    if (a > b) { const double t = a; a = b; b = t; }
}

// Fraction of the unit cube in {c.y <= b} for 0 <= c1 <= c2 <= c3 and 0 < b <= (c1 + c2 + c3) / 2 as a quotient,
// region by region in forms that divide by the smallest component only where the region's width is that component.
__device__ __forceinline__ double region_fraction(double c1, double c2, double c3, double b, double& den) {
    den = c2 * c3;
    if (b < c1) return (b * (b / c1)) * (b / 6.0);
    if (b < c2) return 0.5 * fma(b, b - c1, c1 * c1 * (1.0 / 3.0));
    const double c12 = c1 + c2, p1 = fma(3.0 * b, b - c1, c1 * c1), e2 = b - c2;
    if (b < fmin(c12, c3)) return fma(-e2 * (e2 / c1), e2, p1) * (1.0 / 6.0);
    if (c3 < c12) {
        const double e3 = b - c3;
        return fma(-e3 * (e3 / c1), e3, fma(-e2 * (e2 / c1), e2, p1)) * (1.0 / 6.0);
    }
    den = 2.0 * c3;
    return 2.0 * b - c12;
}
// the same where the denominator would leave the range of FP64: scaled by a power of two, which changes nothing else
__device__ __noinline__ double scaled_fraction(double c1, double c2, double c3, double b) {
    const int e = isfinite(c3) ? -ilogb(c3) : 0;
    double den;
    const double num = region_fraction(scalbn(c1, e), scalbn(c2, e), scalbn(c3, e), scalbn(b, e), den);
    return num / den;
}

// fraction of the unit cube in {a.y <= alpha} (any signs).  a is of the size of the gradient of phi, which is
// 1e-162 and less where all fractions around are.
__device__ double cube_fraction(double a1, double a2, double a3, double alpha) {
    // reflect negative components (y -> 1 - y)
    if (a1 < 0.0) alpha -= a1;
    if (a2 < 0.0) alpha -= a2;
    if (a3 < 0.0) alpha -= a3;
    double c1 = fabs(a1), c2 = fabs(a2), c3 = fabs(a3);
    const double s = (c1 + c2) + c3;
    if (alpha <= 0.0) return 0.0;
    if (alpha >= s) return 1.0;
    sort3(c1, c2, c3);
    const bool flip = alpha > 0.5 * s;
    const double b = flip ? s - alpha : alpha;
    double den;
    const double num = region_fraction(c1, c2, c3, b, den);
    // outside 2^-900 .. 2^900
    const double f = (high_abs(den) >> 20) - 123u >= 1800u ? scaled_fraction(c1, c2, c3, b) : num / den;
    return flip ? 1.0 - f : f;
}

// the unit-cube fraction of one cell's normal with its divisions done once (for the root search)
template <typename T>
struct CubeFrac {
    T c1, c2, c3, ic1, k6, k2, k5;
    __device__ CubeFrac(T a1, T a2, T a3) {
        if (a1 > a2) { const T t = a1; a1 = a2; a2 = t; }
        if (a2 > a3) { const T t = a2; a2 = a3; a3 = t; }
        if (a1 > a2) { const T t = a1; a1 = a2; a2 = t; }
        c1 = a1;
        c2 = a2;
        c3 = a3;
        ic1 = c1 > T(0) ? T(1) / c1 : T(0);
        k2 = T(1) / (T(2) * c2 * c3);
        k6 = k2 * T(1.0 / 3.0);
        k5 = T(1) / (T(2) * c3);
    }
    // the fraction at b and its derivative, the area of the cut, region by region (f(b) = 1 - f(1 - b),
    // so the derivative at b is the one at 1 - b)
    __device__ T operator()(T b, T* dv) const {
        const bool flip = b > T(0.5);
        if (flip) b = T(1) - b;
        T f = T(0), g = T(0);
        if (b > T(0)) {
            const T c12 = c1 + c2;
            if (b < c1) {
                f = b * (b * ic1) * b * k6;
                g = b * (b * ic1) * (T(3) * k6);
            } else if (b < c2) {
                f = (b * (b - c1) + c1 * c1 / T(3)) * k2;
                g = (T(2) * b - c1) * k2;
            } else {
                const T p1 = T(3) * b * b - T(3) * b * c1 + c1 * c1, e2 = b - c2, q2 = e2 * (e2 * ic1);
                if (b < (c12 < c3 ? c12 : c3)) {
                    f = (p1 - q2 * e2) * k6;
                    g = (T(2) * b - c1 - q2) * k2;
                } else if (c3 < c12) {
                    const T e3 = b - c3, q3 = e3 * (e3 * ic1);
                    f = (p1 - q2 * e2 - q3 * e3) * k6;
                    g = (T(2) * b - c1 - q2 - q3) * k2;
                } else {
                    f = (T(2) * b - c12) * k5;
                    g = T(2) * k5;
                }
            }
        }
        *dv = g;
        return flip ? T(1) - f : f;
    }
};

// The root b of volume(b) = pc for a fraction pc below rounding, a_i and their sum unscaled: in FP64 and from
// below, as the volume is at most that of each region's formula with the other faces left out and, for a small
// fraction, near one of the three.  (In line it cost k_vof_plic 8 of 159 us at 512x256x128, as a call 3.)
__device__ __noinline__ double vanishing_root(double a1, double a2, double a3, double sum, double pc) {
    if (sum < 0x1p-1000) {   // its reciprocal would overflow
        a1 *= 0x1p200;
        a2 *= 0x1p200;
        a3 *= 0x1p200;
        sum *= 0x1p200;
    }
    const double is = 1.0 / sum;
    const CubeFrac<double> f(a1 * is, a2 * is, a3 * is);
    double lo = 0.0, hi = 1.0, dv;
    double b = fmax(cbrt(6.0 * f.c1 * f.c2 * f.c3 * pc), fmax(sqrt(2.0 * f.c2 * f.c3 * pc), f.c3 * pc));
    for (int it = 0; it < 100; ++it) {
        const double res = f(b, &dv) - pc;
        if (res == 0.0) break;
        if (res < 0.0) lo = b;
        else hi = b;
        const double nb = dv > 0.0 ? b - res / dv : 2.0;
        if (fabs(nb - b) <= 1e-9 * b) return nb;
        b = nb > lo && nb < hi ? nb : 0.5 * (lo + hi);
    }
    return b;
}

// ---- per-call tables and the interface list -----------------------------------------------------

__device__ __forceinline__ double span(const double* __restrict__ w, int i, int n) {
    const double wp = i > 0 ? w[i - 1] : w[i], wn = i < n - 1 ? w[i + 1] : w[i];
    return 0.5 * wp + w[i] + 0.5 * wn;
}

// Per axis: 1 / width, -1/16 over the distance of a cell's two neighbours' centres, and the high word of 0.49 width / dt, the least of a cell and its two neighbours: a
// velocity whose high word is below it moves less than half a donor cell (false for NaN)
__global__ void k_vof_tables(Dims d, double dt, const double* __restrict__ dx, const double* __restrict__ dy,
                             const double* __restrict__ dz, double* __restrict__ rec, double* __restrict__ rsp,
                             uint32_t* __restrict__ lim, unsigned int* __restrict__ counts) {
    const int n = d.nx + d.ny + d.nz;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) {
        const double* h = t < d.nx ? dx : t < d.nx + d.ny ? dy : dz;
        const int i = t < d.nx ? t : t < d.nx + d.ny ? t - d.nx : t - d.nx - d.ny;
        const int len = t < d.nx ? d.nx : t < d.nx + d.ny ? d.ny : d.nz;
        rec[t] = 1.0 / h[i];
        rsp[t] = -0.0625 / span(h, i, len);
        // the donor of a slab may be either neighbour
        lim[t] = high_abs(0.49 * fmin(h[i], fmin(h[max(i - 1, 0)], h[min(i + 1, len - 1)])) / dt);
    }
    if (blockIdx.x == 0 && threadIdx.x < 6) counts[threadIdx.x] = 0u;
}

// 0 < ph < 1, on the words (comparisons of doubles take the FP64 pipe): positive bit patterns are ordered
__device__ __forceinline__ bool cut(double ph) {
    return (unsigned long long)__double_as_longlong(ph) - 1ULL < 0x3ff0000000000000ULL - 1ULL;
}

// append cell c to the list where `on` (every thread of the warp calls); one counter update per warp
__device__ __forceinline__ void append(bool on, int c, int* __restrict__ list, unsigned int* __restrict__ count) {
    const unsigned int m = __ballot_sync(0xffffffffu, on);
    if (!m) return;
    const int lane = threadIdx.x & 31;
    unsigned int at = 0;
    if (lane == __ffs(m) - 1) at = atomicAdd(count, (unsigned int)__popc(m));
    at = __shfl_sync(0xffffffffu, at, __ffs(m) - 1);
    if (on) list[at + __popc(m & ((1u << lane) - 1u))] = c;
}

// ---- correction --------------------------------------------------------------------------------

// aperture times velocity, without the product where the aperture is 1
__device__ __forceinline__ double open_flux(double a, double u) {
    return __double_as_longlong(a) == 0x3ff0000000000000LL ? u : a * u;
}

// In units of the velocities: F / S = aperture x velocity, E / S_z and the z faces' shares of it.
// With phi: also lists its cut cells for the first stage.
__global__ void __launch_bounds__(kNT)
k_vof_correct(Dims d, const double* __restrict__ dz, const double* __restrict__ rec, const double* __restrict__ ax,
              const double* __restrict__ ay, const double* __restrict__ az, const double* __restrict__ u,
              const double* __restrict__ v, const double* __restrict__ w, double* __restrict__ uxh,
              double* __restrict__ uyh, double* __restrict__ wmh, double* __restrict__ wph,
              const double* __restrict__ phi, int* __restrict__ list, unsigned int* __restrict__ count) {
    const int n = (int)d.n, stride = gridDim.x * kNT;
    for (long long base = (long long)blockIdx.x * kNT; base < n; base += stride) {
        const long long c = base + threadIdx.x;
        const bool in = c < n;
        if (in) {
            int i, j, k;
            cell_ijk(d, c, i, j, k);
            const long long fxm = fx_idx(d, i, j, k), fym = fy_idx(d, i, j, k), fzm = fz_idx(d, i, j, k);
            const long long fxp = fxm + 1, fyp = fym + d.nx, fzp = fzm + d.plane;
            const double am = az[fzm], ap = az[fzp];
            const double xm = open_flux(ax[fxm], u[fxm]), xp = open_flux(ax[fxp], u[fxp]);
            const double ym = open_flux(ay[fym], v[fym]), yp = open_flux(ay[fyp], v[fyp]);
            const double zm = open_flux(am, w[fzm]), zp = open_flux(ap, w[fzp]);
            // E / S_z: S_x / S_z = dz / dx, S_y / S_z = dz / dy
            const double e = fma(dz[k], fma(xp - xm, rec[i], (yp - ym) * rec[d.nx + j]), zp - zm);
            if (__double_as_longlong(am) == 0x3ff0000000000000LL && __double_as_longlong(ap) == 0x3ff0000000000000LL) {
                wph[c] = fma(-0.5, e, zp);
                wmh[c] = fma(0.5, e, zm);
            } else {
                const double tot = ap + am, share = tot > 0.0 ? e / tot : 0.0;
                wph[c] = zp - share * ap;
                wmh[c] = zm + share * am;
            }
            uxh[fxm] = xm;
            if (i == d.nx - 1) uxh[fxp] = xp;
            uyh[fym] = ym;
            if (j == d.ny - 1) uyh[fyp] = yp;
        }
        if (phi) append(in && cut(phi[in ? c : 0]), (int)c, list, count);
    }
}

// ---- reconstruction ----------------------------------------------------------------------------

// Planes of the listed cells (0 < phi < 1) in the cell's unit cube: the normal times the cell's widths, and
// alpha (0, 0, 0, 0 where the gradient vanishes).
__global__ void __launch_bounds__(128)
k_vof_plic(Dims d, const double* __restrict__ dx, const double* __restrict__ dy, const double* __restrict__ dz,
           const double* __restrict__ rsp, const double* __restrict__ vf, const double* __restrict__ phi,
           const int* __restrict__ list, const unsigned int* __restrict__ count, double4* __restrict__ plic) {
    const unsigned int n = *count;
    for (unsigned int q = blockIdx.x * 128u + threadIdx.x; q < n; q += gridDim.x * 128u) {
        const int c = list[q];
        const double pc = phi[c];
        int i, j, k;
        cell_ijk(d, c, i, j, k);
        double val[3][3][3];
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int b = 0; b < 3; ++b)
#pragma unroll
                for (int e = 0; e < 3; ++e) {
                    const int kk = k + a - 1, jj = j + b - 1, ii = i + e - 1;
                    val[a][b][e] = pc;
                    if (kk < 0 || kk >= d.nz || jj < 0 || jj >= d.ny || ii < 0 || ii >= d.nx) continue;
                    const int m = ii + d.nx * (jj + d.ny * kk);
                    if (vf[m] > 0.0) val[a][b][e] = phi[m];
                }
        // differences first: a uniform neighbourhood has a gradient of exactly 0
        double gx = 0.0, gy = 0.0, gz = 0.0;
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                const double wt = (a == 1 ? 2.0 : 1.0) * (b == 1 ? 2.0 : 1.0);
                gx = fma(wt, val[a][b][2] - val[a][b][0], gx);
                gy = fma(wt, val[a][2][b] - val[a][0][b], gy);
                gz = fma(wt, val[2][a][b] - val[0][a][b], gz);
            }
        const double wx = gx * rsp[i] * dx[i], wy = gy * rsp[d.nx + j] * dy[j], wz = gz * rsp[d.nx + d.ny + k] * dz[k];
        // with y_i -> 1 - y_i for negative components the fluid is {a.y <= beta} in the unit cube,
        // a_i = |w_i| / s, beta = (alpha - lo) / s, s = sum |w_i|: Newton steps on beta with the cut area
        // as derivative, kept inside a bracket that bisects when a step leaves it
        const double lo0 = fmin(wx, 0.0) + fmin(wy, 0.0) + fmin(wz, 0.0);
        double a1 = fabs(wx), a2 = fabs(wy), a3 = fabs(wz);
        const double sum = (a1 + a2) + a3;
        double alpha = 0.0;
        if (sum > 0.0) {
            double b;
            if (high_abs(pc) < 0x3a200000u) {   // 2^-93: the FP32 quotient below would lose its residual
                b = vanishing_root(a1, a2, a3, sum, pc);
            } else {
                const double is = 1.0 / sum;
                a1 *= is;
                a2 *= is;
                a3 *= is;
                // FP32 first (its result only starts the FP64 search)
                b = pc;
                {
                    const CubeFrac<float> f((float)a1, (float)a2, (float)a3);
                    const float p = (float)pc;
                    float lo = 0.0f, hi = 1.0f, x = p;
                    for (int it = 0; it < 24; ++it) {
                        float dv;
                        const float res = f(x, &dv) - p;
                        if (res == 0.0f) break;
                        if (res < 0.0f) lo = x;
                        else hi = x;
                        float nx = dv > 0.0f ? x - res / dv : 0.5f * (lo + hi);
                        if (!(nx > lo && nx < hi)) nx = 0.5f * (lo + hi);
                        const float step = fabsf(nx - x);
                        x = nx;
                        if (step <= 2e-7f * x) break;
                    }
                    if (x > 0.0f && x < 1.0f) b = (double)x;
                }
                const CubeFrac<double> f(a1, a2, a3);
                double lo = 0.0, hi = 1.0;
                for (int it = 0; it < 100; ++it) {
                    double dv;
                    const double res = f(b, &dv) - pc;
                    if (res == 0.0) break;
                    if (res < 0.0) lo = b;
                    else hi = b;
                    // the quotient in FP32: a Newton step is right to 1e-7 of itself, and as an error of e becomes
                    // one of about e^2 / min(b, 1 - b), one of at most 1e-9 of that leaves an error below its
                    // rounding and ends the search; a step that leaves the bracket becomes a bisection
                    const double step = dv > 0.0 ? (double)((float)res / (float)dv) : 2.0;
                    const double nb = b - step;
                    if (fabs(step) <= 1e-9 * fmin(b, 1.0 - b)) {
                        b = nb;
                        break;
                    }
                    b = nb > lo && nb < hi ? nb : 0.5 * (lo + hi);
                }
            }
            alpha = lo0 + b * sum;
        }
        plic[c] = make_double4(wx, wy, wz, alpha);
    }
}

// ---- one stage ---------------------------------------------------------------------------------

// Fluid in the slab of thickness t at the + or - face of cell q along AXIS, per cross-section area; h and
// rh: the cell's width and its reciprocal.
template <int AXIS>
__device__ double slab(double ph, const double4* __restrict__ plic, long long q, double h, double rh, bool plus, double t) {
    t = fmin(t, h);
    if (!(t > 0.0)) return 0.0;
    if (cut(ph)) {
        const double4 pl = plic[q];
        if (fabs(pl.x) + fabs(pl.y) + fabs(pl.z) > 0.0) {
            // the slab as a unit cube: its width scales the normal's component along AXIS
            const double w = AXIS == 0 ? pl.x : AXIS == 1 ? pl.y : pl.z, ws = w * (t * rh);
            return t * cube_fraction(AXIS == 0 ? ws : pl.x, AXIS == 1 ? ws : pl.y, AXIS == 2 ? ws : pl.z,
                                     plus ? pl.w - (w - ws) : pl.w);
        }
    }
    return ph * t;
}

// A stage, first part: phi where the cell and both neighbours are all full or all empty and the slabs stay
// within half a cell (the advection and dilation terms cancel); the other cells are listed.
template <int AXIS>
__global__ void __launch_bounds__(kNT)
k_vof_uniform(Dims d, const uint32_t* __restrict__ lim, const double* __restrict__ phi, const double* __restrict__ vm,
              const double* __restrict__ vp, double* __restrict__ out, int* __restrict__ todo,
              unsigned int* __restrict__ ntodo) {
    const int n = (int)d.n, stride = gridDim.x * kNT;
    for (long long base = (long long)blockIdx.x * kNT; base < n; base += stride) {
        const long long c = base + threadIdx.x;
        bool work = false;
        if (c < n) {
            int i, j, k;
            cell_ijk(d, c, i, j, k);
            const int pos = AXIS == 0 ? i : AXIS == 1 ? j : k, len = AXIS == 0 ? d.nx : AXIS == 1 ? d.ny : d.nz;
            const long long step = AXIS == 0 ? 1 : AXIS == 1 ? (long long)d.nx : d.plane;
            const long long f = AXIS == 0 ? fx_idx(d, i, j, k) : AXIS == 1 ? fy_idx(d, i, j, k) : c;
            const double um = vm[f], up = vp[f], pc = phi[c];
            const double pn = phi[pos < len - 1 ? c + step : c], pp = phi[pos > 0 ? c - step : c];
            const long long bits = __double_as_longlong(pc);
            const uint32_t lm = lim[pos];
            work = !((bits == 0 || bits == 0x3ff0000000000000LL) && __double_as_longlong(pn) == bits &&
                     __double_as_longlong(pp) == bits && high_abs(um) < lm && high_abs(up) < lm);
            if (!work) out[c] = pc;
        }
        append(work, (int)c, todo, ntodo);
    }
}

// Second part, the listed cells.  um, up: the corrected velocities of the cell's - and + face along AXIS.
// Lists the cut cells of the new phi for the next stage (list null in the last one).
template <int AXIS>
__global__ void __launch_bounds__(128)
k_vof_stage(Dims d, int implicit, double dt, const double* __restrict__ h, const double* __restrict__ rec,
            const double* __restrict__ phi, const double4* __restrict__ plic, const double* __restrict__ vm,
            const double* __restrict__ vp, double* __restrict__ out, const int* __restrict__ todo,
            const unsigned int* __restrict__ ntodo, int* __restrict__ list, unsigned int* __restrict__ count) {
    const unsigned int n = *ntodo;
    for (unsigned int base = blockIdx.x * 128u; base < n; base += gridDim.x * 128u) {
        const unsigned int q = base + threadIdx.x;
        double res = 0.0;
        int c = 0;
        if (q < n) {
            c = todo[q];
            int i, j, k;
            cell_ijk(d, c, i, j, k);
            const int pos = AXIS == 0 ? i : AXIS == 1 ? j : k, len = AXIS == 0 ? d.nx : AXIS == 1 ? d.ny : d.nz;
            const long long step = AXIS == 0 ? 1 : AXIS == 1 ? (long long)d.nx : d.plane;
            const long long f = AXIS == 0 ? fx_idx(d, i, j, k) : AXIS == 1 ? fy_idx(d, i, j, k) : c;
            const double um = vm[f], up = vp[f], pc = phi[c], hc = h[pos], rc = rec[pos];
            // donors: the cell itself on outflow, the neighbour (the cell at the boundary) on inflow
            double Fp, Fm;
            if (up > 0.0) {
                Fp = slab<AXIS>(pc, plic, c, hc, rc, true, up * dt);
            } else {
                const int p = pos < len - 1 ? pos + 1 : pos;
                const long long q2 = c + (p - pos) * step;
                Fp = -slab<AXIS>(phi[q2], plic, q2, h[p], rec[p], false, -up * dt);
            }
            if (um > 0.0) {
                const int p = pos > 0 ? pos - 1 : pos;
                const long long q2 = c + (p - pos) * step;
                Fm = slab<AXIS>(phi[q2], plic, q2, h[p], rec[p], true, um * dt);
            } else {
                Fm = -slab<AXIS>(pc, plic, c, hc, rc, false, -um * dt);
            }
            const double adv = fma(Fm - Fp, rc, pc), div = dt * (up - um) * rc;
            res = implicit ? adv / (1.0 - div) : fma(pc, div, adv);
            out[c] = res;
        }
        if (list) append(q < n && cut(res), c, list, count);
    }
}

// scratch of both entry points: tables (8 + 4 bytes per cell width), list counters
vofp_status ensure_tables(vofp_ctx* c) {
    if (c->vof_rec) return VOFP_OK;
    const long long n = (long long)c->d.nx + c->d.ny + c->d.nz;
    vofp_status s;
    if ((s = c->alloc(&c->vof_lim, n)) || (s = c->alloc(&c->vof_count, 8)) || (s = c->alloc(&c->vof_rec, 2 * n))) return s;
    return VOFP_OK;
}
void launch_correct(vofp_ctx* c, double dt, const double* ax, const double* ay, const double* az, const double* u,
                    const double* v, const double* w, double* uxh, double* uyh, double* wmh, double* wph,
                    const double* phi) {
    const Dims d = c->d;
    launch(c, k_vof_tables, std::min(16, ceil_div(d.nx + d.ny + d.nz, kNT)), kNT, c->stream, d, dt, (const double*)c->dx,
           (const double*)c->dy, (const double*)c->dz, c->vof_rec, c->vof_rec + d.nx + d.ny + d.nz, c->vof_lim, c->vof_count);
    launch(c, k_vof_correct, grid_cells(d.n), kNT, c->stream, d, (const double*)c->dz, (const double*)c->vof_rec, ax, ay,
           az, u, v, w, uxh, uyh, wmh, wph, phi, c->vof_list, c->vof_count);
}

}  // namespace

vofp_status vof_flux_correct(vofp_ctx* c, const double* ax, const double* ay, const double* az, const double* u,
                             const double* v, const double* w, double* uxh, double* uyh, double* wmh, double* wph) {
    vofp_status s = ensure_tables(c);
    if (s) return s;
    launch_correct(c, 1.0, ax, ay, az, u, v, w, uxh, uyh, wmh, wph, nullptr);
    return VOFP_OK;
}

vofp_status vof_advect(vofp_ctx* c, const double* F, const double* ax, const double* ay, const double* az,
                       const double* vf, const double* u, const double* v, const double* w, double dt, int order,
                       double* F_out) {
    const Dims d = c->d;
    const long long N = d.n;
    vofp_status s = ensure_tables(c);
    if (s) return s;
    if (!c->vof_uxh) {
        if ((s = c->alloc(&c->vof_uxh, (long long)(d.nx + 1) * d.ny * d.nz)) ||
            (s = c->alloc(&c->vof_uyh, (long long)d.nx * (d.ny + 1) * d.nz)) || (s = c->alloc(&c->vof_wmh, N)) ||
            (s = c->alloc(&c->vof_wph, N)) || (s = c->alloc(&c->vof_phi, 2 * N)) ||
            (s = c->alloc(&c->vof_plic, 4 * N)) || (s = c->alloc(&c->vof_list, 2 * N)))
            return s;
    }
    cudaStream_t st = c->stream;
    launch_correct(c, dt, ax, ay, az, u, v, w, c->vof_uxh, c->vof_uyh, c->vof_wmh, c->vof_wph, F);
    const int axes[2][3] = {{0, 1, 2}, {2, 1, 0}};
    const double* in = F;
    double4* plic = reinterpret_cast<double4*>(c->vof_plic);
    const double *dx = c->dx, *dy = c->dy, *dz = c->dz;
    const int gc = grid_cells(N);
    const int gl = (int)std::max(1LL, std::min((N + 127) / 128, (long long)num_sms() * 8));
    // list lengths: cut cells of the coming stage (0 .. 2), cells of its second part (3 .. 5)
    unsigned int* n = c->vof_count;
    int *list = c->vof_list, *todo = c->vof_list + N;
    const double *rec = c->vof_rec, *rsp = c->vof_rec + d.nx + d.ny + d.nz;
    auto stage_on = [&](auto axis_c, const double* h, int first, const double* vm, const double* vp, int stage, double* out) {
        constexpr int AXIS = decltype(axis_c)::value;
        launch(c, k_vof_uniform<AXIS>, gc, kNT, st, d, (const uint32_t*)(c->vof_lim + first), in, vm, vp, out, todo,
               n + 3 + stage);
        launch(c, k_vof_stage<AXIS>, gl, 128, st, d, stage < 2 ? 1 : 0, dt, h, rec + first, in, (const double4*)plic, vm, vp,
               out, (const int*)todo, (const unsigned int*)(n + 3 + stage), stage < 2 ? list : (int*)nullptr,
               n + (stage < 2 ? stage + 1 : 2));
    };
    for (int stage = 0; stage < 3; ++stage) {
        double* out = stage == 2 ? F_out : c->vof_phi + (stage % 2) * N;
        // the list is read here and rewritten by the stage after
        launch(c, k_vof_plic, gl, 128, st, d, dx, dy, dz, rsp, vf, in, (const int*)list, (const unsigned int*)(n + stage),
               plic);
        const int axis = axes[order ? 1 : 0][stage];
        if (axis == 0)
            stage_on(std::integral_constant<int, 0>{}, dx, 0, c->vof_uxh, c->vof_uxh + 1, stage, out);
        else if (axis == 1)
            stage_on(std::integral_constant<int, 1>{}, dy, d.nx, c->vof_uyh, c->vof_uyh + d.nx, stage, out);
        else
            stage_on(std::integral_constant<int, 2>{}, dz, d.nx + d.ny, c->vof_wmh, c->vof_wph, stage, out);
        in = out;
    }
    return VOFP_OK;
}

}  // namespace vofp
