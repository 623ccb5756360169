// Operator assembly of the pressure Poisson equation (Sec. 2 Eq. density; Sec. 2.3 Eqs.
// integral1-integral2 and cell merging; Sec. 2.10 density smoothing) and the divergence
// right-hand side (Sec. 2.1 Eq. poisson1; Sec. 2.4 F_i = A_i u_i).
//
// Cell-centred kernels: each thread owns one cell and writes the coefficient of its +x, +y and
// +z face, so every face coefficient is computed once and stored once (structure of arrays).
#include <algorithm>
#include <cmath>

#include "vofp_fp.cuh"
#include "vofp_internal.cuh"

namespace vofp {
namespace {

constexpr int kNT = 256;


// How the passes below are laid out. FP64 arithmetic bounds them on this part: one FP64 instruction per cell of
// 512 x 256 x 128 takes 32 us, as long as moving 13 bytes per cell. So a thread takes one (x, y) column over a
// range of planes (what belongs to a face between two planes is formed once, and row and column indices are
// formed once), values are compared as integers, an open aperture's factor 1.0 is not multiplied by, and what
// a density of pure liquid or pure gas gives is looked up. Every value that is formed is formed by the same
// operations in the same order as by the plain formula.
struct March {
    int kc, nch;   // planes per range, ranges
};
// ranges of at most 16 planes, fewer where that leaves fewer than two threads per resident one
March march_of(const Dims& d) {
    const long long per = d.n / ((long long)num_sms() * 4096);
    March m;
    m.kc = (int)std::max(1LL, std::min(16LL, per));
    m.nch = ceil_div(d.nz, m.kc);
    return m;
}
struct Column {
    int i, j, k0, k1;
    long long c;    // first cell
    bool on;
};
__device__ __forceinline__ Column column_of(const Dims& d, const March m) {
    const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    Column q;
    q.on = t < d.plane * m.nch;
    const unsigned int tt = q.on ? (unsigned int)t : 0u, plane = (unsigned int)d.plane, nx = (unsigned int)d.nx;
    const unsigned int ch = tt / plane, p = tt - ch * plane;
    q.j = int(p / nx);
    q.i = int(p - (unsigned int)q.j * nx);
    q.k0 = (int)ch * m.kc;
    q.k1 = q.on ? min(q.k0 + m.kc, d.nz) : q.k0;
    q.c = p + (long long)q.k0 * d.plane;
    return q;
}
// a > 0.0 (false for NaN)
__device__ __forceinline__ bool positive(double a) {
    return (unsigned long long)(bits_of(a) - 1) < 0x7ff0000000000000ull;
}
// Whether it holds for every thread of the warp that is here.  The passes branch on this around whole blocks:
// around one operation the compiler forms a predicated one, which takes its time on the FP64 pipe all the same.
__device__ __forceinline__ bool whole_warp(bool a) { return __all_sync(__activemask(), a); }
__device__ __forceinline__ bool is_one(double a) { return bits_of(a) == 0x3ff0000000000000ll; }

__device__ __forceinline__ double density(double F, double rl, double rg) { return rg + (rl - rg) * F; }
__device__ __forceinline__ double smooth3(double lo, double in, double hi) { return 0.25 * lo + 0.5 * in + 0.25 * hi; }
// inverse resistance of the face between two cells; the x faces of odd cells in rows of even length take their
// neighbours the other way round, which decides the last bit of some (operators have always been built so)
__device__ __forceinline__ double face_inv(double h0, double r0, double h1, double r1) {
    return 1.0 / (0.5 * __fma_rn(h0, r0, __dmul_rn(h1, r1)));
}
__device__ __forceinline__ double face_inv_x(const Dims& d, int i, const double* __restrict__ dx, double r0, double r1) {
    return (i & 1) && !(d.nx & 1) ? face_inv(dx[i + 1], r1, dx[i], r0) : face_inv(dx[i], r0, dx[i + 1], r1);
}

// Tables of one operator: the density of F = 0 and F = 1 before and after each smoothing pass (pure[phase][pass],
// 2 x 4), and 1 / ((d_L rho + d_R rho) / 2) of every face between two cells of that final density along each
// axis ([phase][axis cell], from tab + 8).
__global__ void k_tables(Dims d, double rl, double rg, int smoothing, const double* __restrict__ dx,
                         const double* __restrict__ dy, const double* __restrict__ dz, double* __restrict__ tab) {
    const int len = d.nx + d.ny + d.nz;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < 2 * len; t += gridDim.x * blockDim.x) {
        const int ph = t >= len, at = t - ph * len;
        double r[4];
        r[0] = density(ph ? 1.0 : 0.0, rl, rg);
        for (int q = 1; q < 4; ++q) r[q] = smoothing ? smooth3(r[q - 1], r[q - 1], r[q - 1]) : r[q - 1];
        if (at == 0)
            for (int q = 0; q < 4; ++q) tab[4 * ph + q] = r[q];
        const double* h = at < d.nx ? dx : at < d.nx + d.ny ? dy : dz;
        const int o = at < d.nx ? at : at < d.nx + d.ny ? at - d.nx : at - d.nx - d.ny;
        const int n = at < d.nx ? d.nx : at < d.nx + d.ny ? d.ny : d.nz;
        tab[8 + t] = o == n - 1 ? 0.0 : at < d.nx ? face_inv_x(d, o, dx, r[3], r[3]) : face_inv(h[o], r[3], h[o + 1], r[3]);
    }
}

// rho = rho_g + (rho_l - rho_g) F   (Eq. density with H(phi) = phi)
__device__ __forceinline__ bool is_pure(double F) { return bits_of(F) == 0 || is_one(F); }
__device__ __forceinline__ double density_of(double F, double rl, double rg, double r0, double r1) {
    const double r = is_one(F) ? r1 : r0;
    return whole_warp(is_pure(F)) ? r : density(F, rl, rg);
}
__global__ void k_density(Dims d, const double* __restrict__ F, double rl, double rg, const double* __restrict__ tab,
                          double* __restrict__ rho) {
    const double r0 = tab[0], r1 = tab[4];
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < d.n;
         c += (long long)gridDim.x * blockDim.x)
        rho[c] = density_of(F[c], rl, rg, r0, r1);
}

// The (1/4, 1/2, 1/4) filter (Sec. 2.10); a missing neighbour at a domain wall is replaced by the cell itself.
// `pure`: the densities of the pure phases before this pass (stride 4) and after it (one further).
__device__ __forceinline__ double smooth_of(double lo, double in, double hi, const double* p) {
    const long long b = bits_of(in);
    if (bits_of(lo) == b && bits_of(hi) == b) {
        if (b == bits_of(p[0])) return p[1];
        if (b == bits_of(p[4])) return p[5];
    }
    return smooth3(lo, in, hi);
}
// Density and its x pass, then the y and z passes: two sweeps over memory for what four kernels and a copy did
// (512 x 256 x 128: 390 us -> 127).
__global__ void k_density_x(Dims d, const double* __restrict__ F, double rl, double rg, const double* __restrict__ tab,
                            double* __restrict__ out) {
    const double p0 = tab[1], p1 = tab[5];
    const unsigned int nx = (unsigned int)d.nx;
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < d.n;
         c += (long long)gridDim.x * blockDim.x) {
        const int i = int((unsigned int)c % nx);
        const double f = F[c], fl = i > 0 ? F[c - 1] : f, fh = i < d.nx - 1 ? F[c + 1] : f;
        // one pure phase in all three cells, in every thread of the warp
        if (whole_warp(is_pure(f) && bits_of(fl) == bits_of(f) && bits_of(fh) == bits_of(f))) {
            out[c] = is_one(f) ? p1 : p0;
        } else {
            out[c] = smooth3(density(fl, rl, rg), density(f, rl, rg), density(fh, rl, rg));
        }
    }
}
__global__ void k_smooth_yz(Dims d, March m, const double* __restrict__ in, const double* __restrict__ tab,
                            double* __restrict__ out) {
    const Column q = column_of(d, m);
    if (!q.on) return;
    const double py[6] = {tab[1], tab[2], 0.0, 0.0, tab[5], tab[6]}, pz[6] = {tab[2], tab[3], 0.0, 0.0, tab[6], tab[7]};
    auto row = [&](long long c) {
        const double v = in[c];
        return smooth_of(q.j > 0 ? in[c - d.nx] : v, v, q.j < d.ny - 1 ? in[c + d.nx] : v, py);
    };
    long long c = q.c;
    double cur = row(c), lo = q.k0 > 0 ? row(c - d.plane) : cur;
    for (int k = q.k0; k < q.k1; ++k, c += d.plane) {
        const double hi = k < d.nz - 1 ? row(c + d.plane) : cur;
        out[c] = smooth_of(lo, cur, hi, pz);
        lo = cur;
        cur = hi;
    }
}

__global__ void k_activity_init(Dims d, const double* __restrict__ vf, uint8_t* __restrict__ ina) {
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < d.n;
         c += (long long)gridDim.x * blockDim.x)
        ina[c] = vf ? (uint8_t)!(vf[c] > 0.0) : (uint8_t)0;
}

struct Bc6 {
    int k[6];
};

// A cell loses its unknown when none of its flux-carrying faces (interior faces towards a cell
// that still has one, or p = 0 domain faces) is open.
__global__ void k_activity_step(Dims d, Bc6 bc, const double* __restrict__ ax,
                                const double* __restrict__ ay, const double* __restrict__ az,
                                const uint8_t* __restrict__ in, uint8_t* __restrict__ out,
                                unsigned int* changed) {
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < d.n;
         c += (long long)gridDim.x * blockDim.x) {
        if (in[c]) {
            out[c] = 1;
            continue;
        }
        int i, j, k;
        cell_ijk(d, c, i, j, k);
        bool open = false;
        open |= ax[fx_idx(d, i, j, k)] > 0.0 && (i > 0 ? !in[c - 1] : bc.k[0] == VOFP_BC_DIRICHLET);
        open |= ax[fx_idx(d, i + 1, j, k)] > 0.0 && (i < d.nx - 1 ? !in[c + 1] : bc.k[1] == VOFP_BC_DIRICHLET);
        open |= ay[fy_idx(d, i, j, k)] > 0.0 && (j > 0 ? !in[c - d.nx] : bc.k[2] == VOFP_BC_DIRICHLET);
        open |= ay[fy_idx(d, i, j + 1, k)] > 0.0 && (j < d.ny - 1 ? !in[c + d.nx] : bc.k[3] == VOFP_BC_DIRICHLET);
        open |= az[fz_idx(d, i, j, k)] > 0.0 && (k > 0 ? !in[c - d.plane] : bc.k[4] == VOFP_BC_DIRICHLET);
        open |= az[fz_idx(d, i, j, k + 1)] > 0.0 && (k < d.nz - 1 ? !in[c + d.plane] : bc.k[5] == VOFP_BC_DIRICHLET);
        out[c] = open ? 0 : 1;
        if (!open) atomicAdd(changed, 1u);
    }
}

// One pass over the cells: whether each has an unknown (from its open volume, or from `ina_in` where that has
// been settled before), the first step of the activity iteration (k_activity_step: `cnt[0]` counts the cells
// that it would take out; if there are any, the caller settles the activity and runs the pass again), the
// effective apertures (faces touching a cell without an unknown are closed), the roots, the number of cells
// without an unknown (cnt[2]) and the list of the small cells.  Those are cells with an unknown and open volume
// below the threshold; their merge target is the neighbour across the interior face of largest open area
// (first of -x,+x,-y,+y,-z,+z on ties).  The list's slots come in arrival order (the order is not significant);
// cnt[1] counts them, and the caller grows the lists and runs again if they overflow.
// Seven passes of 700 us together before, 300 here (512 x 256 x 128: 1.0 GB, 150 us at copy bandwidth).
template <int FROM>   // activity from the open volume (0), from `ina_in` (1), every cell active (2)
__global__ void __launch_bounds__(kNT, 6)
k_cells(Dims d, March m, Bc6 bc, double thr, const double* __restrict__ vf,
                        const uint8_t* __restrict__ ina_in, const double* __restrict__ ax,
                        const double* __restrict__ ay, const double* __restrict__ az, const double* __restrict__ dx,
                        const double* __restrict__ dy, const double* __restrict__ dz, uint8_t* __restrict__ ina,
                        int32_t* __restrict__ root, double* __restrict__ axe, double* __restrict__ aye,
                        double* __restrict__ aze, unsigned int* __restrict__ cnt, long long cap,
                        long long* __restrict__ cells, long long* __restrict__ targets, double* __restrict__ vfs) {
    const Column q = column_of(d, m);
    const int i = q.i, j = q.j;
    auto active = [&](long long c) { return FROM == 0 ? positive(vf[c]) : FROM == 1 ? !ina_in[c] : true; };
    const long long tb = positive(thr) ? bits_of(thr) : 0;
    const bool xl = i == 0, xr = i == d.nx - 1, yl = j == 0, yr = j == d.ny - 1;
    long long c = q.c;
    bool am = true, ac = true;
    double zlo = 0.0;
    if (q.on) {
        am = q.k0 == 0 || active(c - d.plane);
        ac = active(c);
        zlo = az[c];
    }
    unsigned int lost = 0, none = 0;
    long long fx = fx_idx(d, i, j, q.k0), fy = fy_idx(d, i, j, q.k0);
    const long long fxs = (long long)(d.nx + 1) * d.ny, fys = (long long)d.nx * (d.ny + 1);
    for (int k = q.k0; k < q.k1; ++k, c += d.plane, fx += fxs, fy += fys) {
        const bool zl = k == 0, zr = k == d.nz - 1;
        const bool axm = xl || active(c - 1), axp = xr || active(c + 1);
        const bool aym = yl || active(c - d.nx), ayp = yr || active(c + d.nx), azp = zr || active(c + d.plane);
        const double x0 = ax[fx], x1 = ax[fx + 1], y0 = ay[fy], y1 = ay[fy + d.nx], z0 = zlo, z1 = az[c + d.plane];
        ina[c] = ac ? 0 : 1;
        root[c] = ac ? (int32_t)c : -1;
        axe[fx] = ac && axm ? x0 : 0.0;
        if (xr) axe[fx + 1] = ac ? x1 : 0.0;
        aye[fy] = ac && aym ? y0 : 0.0;
        if (yr) aye[fy + d.nx] = ac ? y1 : 0.0;
        aze[c] = ac && am ? z0 : 0.0;
        if (zr) aze[c + d.plane] = ac ? z1 : 0.0;
        if (ac) {
            bool open = false;
            open |= positive(x0) && (xl ? bc.k[0] == VOFP_BC_DIRICHLET : axm);
            open |= positive(x1) && (xr ? bc.k[1] == VOFP_BC_DIRICHLET : axp);
            open |= positive(y0) && (yl ? bc.k[2] == VOFP_BC_DIRICHLET : aym);
            open |= positive(y1) && (yr ? bc.k[3] == VOFP_BC_DIRICHLET : ayp);
            open |= positive(z0) && (zl ? bc.k[4] == VOFP_BC_DIRICHLET : am);
            open |= positive(z1) && (zr ? bc.k[5] == VOFP_BC_DIRICHLET : azp);
            lost += open ? 0u : 1u;
            if (tb > 0 && bits_of(vf[c]) < tb) {   // both positive
                double a[6];
                a[0] = !xl && axm ? x0 * (dz[k] * dy[j]) : 0.0;
                a[1] = !xr && axp ? x1 * (dz[k] * dy[j]) : 0.0;
                a[2] = !yl && aym ? y0 * (dz[k] * dx[i]) : 0.0;
                a[3] = !yr && ayp ? y1 * (dz[k] * dx[i]) : 0.0;
                a[4] = !zl && am ? z0 * (dy[j] * dx[i]) : 0.0;
                a[5] = !zr && azp ? z1 * (dy[j] * dx[i]) : 0.0;
                int best = 0;
                for (int f = 1; f < 6; ++f)
                    if (a[f] > a[best]) best = f;
                if (a[best] > 0.0) {
                    const long long off[6] = {-1, 1, -(long long)d.nx, (long long)d.nx, -d.plane, d.plane};
                    const unsigned int slot = atomicAdd(&cnt[1], 1u);
                    if ((long long)slot < cap) {
                        cells[slot] = c;
                        targets[slot] = c + off[best];
                        vfs[slot] = vf[c];
                    }
                }
            }
        } else {
            ++none;
        }
        am = ac;
        ac = azp;
        zlo = z1;
    }
    __syncwarp();
    lost = __reduce_add_sync(0xffffffffu, lost);
    none = __reduce_add_sync(0xffffffffu, none);
    if ((threadIdx.x & 31) == 0) {
        if (lost) atomicAdd(&cnt[0], lost);
        if (none) atomicAdd(&cnt[2], none);
    }
}

// T of each cell's +x, +y, +z interior face: A_f S_f / ((d_L rho_L + d_R rho_R) / 2), 0 on domain faces, and the
// face's inverse resistance kappa = 1 / ((d_L rho_L + d_R rho_R) / 2) where the face is open (0 where it is
// closed or on the domain boundary), which the projection of the face velocities uses.
// 512 x 256 x 128: 1075 us with three divisions in every cell, 330 with the pure phases' looked up (1.3 GB,
// 200 us at copy bandwidth).
__global__ void __launch_bounds__(kNT, 5)
k_face_coeffs(Dims d, March m, const double* __restrict__ dx, const double* __restrict__ dy,
                              const double* __restrict__ dz, const double* __restrict__ rho,
                              const double* __restrict__ axe, const double* __restrict__ aye,
                              const double* __restrict__ aze, const double* __restrict__ tab, double* __restrict__ Tx,
                              double* __restrict__ Ty, double* __restrict__ Tz, double* __restrict__ kx,
                              double* __restrict__ ky, double* __restrict__ kz) {
    const Column q = column_of(d, m);
    if (!q.on) return;
    const int i = q.i, j = q.j;
    const long long p0 = bits_of(tab[3]), p1 = bits_of(tab[7]);
    const int len = d.nx + d.ny + d.nz;
    const double* ti = tab + 8;
    const double Sz = dy[j] * dx[i];
    long long c = q.c;
    double rc = rho[c];
    const bool fx = i < d.nx - 1, fy = j < d.ny - 1;
    long long ox = fx_idx(d, i + 1, j, q.k0), oy = fy_idx(d, i, j + 1, q.k0);
    const long long oxs = (long long)(d.nx + 1) * d.ny, oys = (long long)d.nx * (d.ny + 1);
    for (int k = q.k0; k < q.k1; ++k, c += d.plane, ox += oxs, oy += oys) {
        const bool fz = k < d.nz - 1;
        const double rx = fx ? rho[c + 1] : 0.0, ry = fy ? rho[c + d.nx] : 0.0, rz = fz ? rho[c + d.plane] : 0.0;
        const double axv = fx ? axe[ox] : 0.0, ayv = fy ? aye[oy] : 0.0,
                     azv = fz ? aze[c + d.plane] : 0.0;
        const long long rb = bits_of(rc);
        const int ph = rb == p0 ? 0 : rb == p1 ? len : -1;   // offset of the phase's tables
        double tx = 0.0, ty = 0.0, tz = 0.0, qx = 0.0, qy = 0.0, qz = 0.0;
        const double dzk = dz[k];
        // one pure phase across all three faces, open entirely (or on the domain boundary)
        if (whole_warp(ph >= 0 && (!fx || (bits_of(rx) == rb && is_one(axv))) && (!fy || (bits_of(ry) == rb && is_one(ayv))) &&
                       (!fz || (bits_of(rz) == rb && is_one(azv))))) {
            qx = fx ? ti[ph + i] : 0.0;
            qy = fy ? ti[ph + d.nx + j] : 0.0;
            qz = fz ? ti[ph + d.nx + d.ny + k] : 0.0;
            tx = (dzk * dy[j]) * qx;
            ty = (dzk * dx[i]) * qy;
            tz = Sz * qz;
        } else {
            if (fx) {
                const double inv = face_inv_x(d, i, dx, rc, rx);
                tx = (axv * (dzk * dy[j])) * inv;
                qx = positive(axv) ? inv : 0.0;
            }
            if (fy) {
                const double inv = face_inv(dy[j], rc, dy[j + 1], ry);
                ty = (ayv * (dzk * dx[i])) * inv;
                qy = positive(ayv) ? inv : 0.0;
            }
            if (fz) {
                const double inv = face_inv(dzk, rc, dz[k + 1], rz);
                tz = (azv * Sz) * inv;
                qz = positive(azv) ? inv : 0.0;
            }
        }
        Tx[c] = tx;
        Ty[c] = ty;
        Tz[c] = tz;
        kx[c] = qx;
        ky[c] = qy;
        kz[c] = qz;
        rc = rz;
    }
}

// Diagonal of the unmerged operator (sum of the six face coefficients plus p = 0 faces) and the symmetric
// scaling s = diag^-1/2, sq = diag^1/2 (0 without an unknown; the groups' follow in k_scale_groups).
// FP64 arithmetic bounds it: 650 us as two kernels with sqrt and a division, 355 here (512 x 256 x 128).
__global__ void __launch_bounds__(kNT, 5)
k_diag_scale(Dims d, March m, Bc6 bc, const double* __restrict__ dx, const double* __restrict__ dy,
                             const double* __restrict__ dz, const double* __restrict__ rho,
                             const double* __restrict__ axe, const double* __restrict__ aye,
                             const double* __restrict__ aze, const double* __restrict__ Tx,
                             const double* __restrict__ Ty, const double* __restrict__ Tz,
                             const uint8_t* __restrict__ ina, double* __restrict__ diag, double* __restrict__ s,
                             double* __restrict__ sq) {
    const Column q = column_of(d, m);
    if (!q.on) return;
    const int i = q.i, j = q.j;
    const bool edge = (i == 0 && bc.k[0] == VOFP_BC_DIRICHLET) || (i == d.nx - 1 && bc.k[1] == VOFP_BC_DIRICHLET) ||
                      (j == 0 && bc.k[2] == VOFP_BC_DIRICHLET) || (j == d.ny - 1 && bc.k[3] == VOFP_BC_DIRICHLET);
    long long c = q.c;
    double tzm = q.k0 > 0 ? Tz[c - d.plane] : 0.0;
    double last = __longlong_as_double(-1ll), r = 0.0, inv = 0.0;   // of the plane before: r and inv of `last`
    for (int k = q.k0; k < q.k1; ++k, c += d.plane) {
        const double tx = Tx[c], ty = Ty[c], tz = Tz[c];
        const double txm = i > 0 ? Tx[c - 1] : 0.0, tym = j > 0 ? Ty[c - d.nx] : 0.0;
        const bool off = ina[c] != 0;
        double v = tx + ty + tz;
        if (i > 0) v += txm;
        if (j > 0) v += tym;
        if (k > 0) v += tzm;
        if (edge || k == 0 || k == d.nz - 1) {
            const double rc = rho[c];
            if (i == 0 && bc.k[0] == VOFP_BC_DIRICHLET) v += (axe[fx_idx(d, 0, j, k)] * (dz[k] * dy[j])) / (0.5 * dx[0] * rc);
            if (i == d.nx - 1 && bc.k[1] == VOFP_BC_DIRICHLET) v += (axe[fx_idx(d, d.nx, j, k)] * (dz[k] * dy[j])) / (0.5 * dx[i] * rc);
            if (j == 0 && bc.k[2] == VOFP_BC_DIRICHLET) v += (aye[fy_idx(d, i, 0, k)] * (dz[k] * dx[i])) / (0.5 * dy[0] * rc);
            if (j == d.ny - 1 && bc.k[3] == VOFP_BC_DIRICHLET) v += (aye[fy_idx(d, i, d.ny, k)] * (dz[k] * dx[i])) / (0.5 * dy[j] * rc);
            if (k == 0 && bc.k[4] == VOFP_BC_DIRICHLET) v += (aze[fz_idx(d, i, j, 0)] * (dy[j] * dx[i])) / (0.5 * dz[0] * rc);
            if (k == d.nz - 1 && bc.k[5] == VOFP_BC_DIRICHLET) v += (aze[fz_idx(d, i, j, d.nz)] * (dy[j] * dx[i])) / (0.5 * dz[k] * rc);
        }
        diag[c] = v;
        if (!off && bits_of(v) != bits_of(last)) {
            sqrt_and_inverse(v, r, inv);
            last = v;
        }
        s[c] = off ? 0.0 : inv;
        sq[c] = off ? 0.0 : r;
        tzm = tz;
    }
}

// slot_of[cell] = slot of every listed small cell (the other entries were set to -1 before)
__global__ void k_small_slots(int m, const long long* __restrict__ cells, int32_t* __restrict__ slot_of) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < m) slot_of[cells[t]] = t;
}

// slot of each small cell's target among the small cells, -1 if the target is not one of them
__global__ void k_small_target_slots(int m, const long long* __restrict__ targets,
                                     const int32_t* __restrict__ slot_of, int32_t* __restrict__ tslot) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < m) tslot[t] = slot_of[targets[t]];
}

__global__ void k_root_scatter(int m, const long long* __restrict__ cells,
                               const long long* __restrict__ roots, int32_t* __restrict__ root) {
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < m) root[cells[t]] = (int32_t)roots[t];
}

// diag(A_hat) of a merge group = sum over its cells of the diagonal minus the couplings between
// its own cells (both directions); all cells of the group get the group's scale.
__global__ void k_scale_groups(Dims d, int ng, const int* __restrict__ gptr,
                               const int* __restrict__ gcells, const int32_t* __restrict__ root,
                               const double* __restrict__ diag, const double* __restrict__ Tx,
                               const double* __restrict__ Ty, const double* __restrict__ Tz,
                               double* __restrict__ s, double* __restrict__ sq,
                               double* __restrict__ gcorr) {
    int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= ng) return;
    const int b = gptr[g], e = gptr[g + 1];
    const int32_t m = gcells[b];
    double dsum = 0.0, intra = 0.0;
    for (int t = b; t < e; ++t) {
        long long c = gcells[t];
        int i, j, k;
        cell_ijk(d, c, i, j, k);
        dsum += diag[c];
        if (i > 0 && root[c - 1] == m) intra += Tx[c - 1];
        if (i < d.nx - 1 && root[c + 1] == m) intra += Tx[c];
        if (j > 0 && root[c - d.nx] == m) intra += Ty[c - d.nx];
        if (j < d.ny - 1 && root[c + d.nx] == m) intra += Ty[c];
        if (k > 0 && root[c - d.plane] == m) intra += Tz[c - d.plane];
        if (k < d.nz - 1 && root[c + d.plane] == m) intra += Tz[c];
    }
    const double dhat = dsum - intra;
    const double r = sqrt(dhat);
    const double sm = 1.0 / r;
    for (int t = b; t < e; ++t) {
        s[gcells[t]] = sm;
        sq[gcells[t]] = r;
    }
    gcorr[g] = sm * sm * dsum - double(e - b);
}

// The scaled operator in FP64 and FP32, and Tzr = Tzf with the sign bit set on red cells (coefficients are >= 0,
// so the sign carries the red flag through the same tensor copy as the coefficient; -0.0 marks a red cell with a
// closed face).  512 x 256 x 128: 315 us as two kernels with converting instructions, 215 here.
__global__ void k_scaled_coeffs(Dims d, March m, const double* __restrict__ s, const double* __restrict__ Tx,
                                const double* __restrict__ Ty, const double* __restrict__ Tz,
                                const uint32_t* __restrict__ red, double* __restrict__ Txs, double* __restrict__ Tys,
                                double* __restrict__ Tzs, float* __restrict__ Txf, float* __restrict__ Tyf,
                                float* __restrict__ Tzf, float* __restrict__ Tzr) {
    const Column q = column_of(d, m);
    if (!q.on) return;
    const bool fx = q.i < d.nx - 1, fy = q.j < d.ny - 1;
    long long c = q.c;
    double sc = s[c];
    for (int k = q.k0; k < q.k1; ++k, c += d.plane) {
        const bool fz = k < d.nz - 1;
        const double sx = fx ? s[c + 1] : 0.0, sy = fy ? s[c + d.nx] : 0.0, sz = fz ? s[c + d.plane] : 0.0;
        const double tx = Tx[c], ty = Ty[c], tz = Tz[c];
        const uint32_t w = red[c >> 5] >> (c & 31);
        const double a = fx ? sc * tx * sx : 0.0;
        const double b = fy ? sc * ty * sy : 0.0;
        const double e = fz ? sc * tz * sz : 0.0;
        const float ef = to_float(e);
        Txs[c] = a;
        Tys[c] = b;
        Tzs[c] = e;
        Txf[c] = to_float(a);
        Tyf[c] = to_float(b);
        Tzf[c] = ef;
        Tzr[c] = (w & 1u) ? -fabsf(ef) : ef;
        sc = sz;
    }
}

// Merged cells and red cells as bits.  A red cell has (i+j+k) even, an unknown of its own and no merge group (the
// groups' cells are taken out by k_group_flags; a count of the red cells goes with both).
__global__ void k_cell_bits(Dims d, const uint8_t* __restrict__ ina, uint32_t* __restrict__ slave,
                            uint32_t* __restrict__ red, unsigned int* __restrict__ count) {
    const long long nw = (d.n + 31) / 32;
    unsigned int mine = 0;
    for (long long w = blockIdx.x * (long long)blockDim.x + threadIdx.x; w < nw;
         w += (long long)gridDim.x * blockDim.x) {
        const long long c0 = w * 32;
        const int n = (int)min(32LL, d.n - c0);
        int i, j, k;
        cell_ijk(d, c0, i, j, k);
        uint32_t par = 0u;   // bit b: cell c0 + b has i+j+k even
        for (int b = 0; b < n;) {
            const int run = min(n - b, d.nx - i);   // cells left in this row
            const uint32_t pat = ((i + j + k + b) & 1) == 0 ? 0x55555555u : 0xaaaaaaaau;
            const uint32_t part = run == 32 ? 0xffffffffu : ((1u << run) - 1u) << b;
            par |= pat & part;
            b += run;
            i = 0;
            if (++j == d.ny) {
                j = 0;
                ++k;
            }
        }
        uint32_t v = 0u;
        if (n == 32) {
            const uint4* p = reinterpret_cast<const uint4*>(ina + c0);
            const uint4 a = p[0], b = p[1];
            const uint32_t x[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
            // bytes of 0 or 1: their low bits to four neighbouring bits
#pragma unroll
            for (int t = 0; t < 8; ++t) v |= (((x[t] & 0x01010101u) * 0x10204080u) >> 28) << (4 * t);
            v = ~v;
        } else {
            for (int b = 0; b < n; ++b) v |= (ina[c0 + b] ? 0u : 1u) << b;
        }
        v &= par;
        slave[w] = 0u;
        red[w] = v;
        mine += __popc(v);
    }
    __syncwarp();
    mine = __reduce_add_sync(0xffffffffu, mine);
    if ((threadIdx.x & 31) == 0 && mine) atomicAdd(count, mine);
}
__global__ void k_group_flags(int ng, const int* __restrict__ gptr, const int* __restrict__ gcells,
                              uint32_t* __restrict__ slave, uint32_t* __restrict__ red, unsigned int* __restrict__ count) {
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= ng) return;
    for (int t = gptr[g]; t < gptr[g + 1]; ++t) {
        const int c = gcells[t];
        const uint32_t bit = 1u << (c & 31);
        if (t > gptr[g]) atomicOr(&slave[c >> 5], bit);
        if (atomicAnd(&red[c >> 5], ~bit) & bit) atomicSub(count, 1u);
    }
}
__global__ void k_excl_bits(long long nw, const uint32_t* __restrict__ slave, const uint32_t* __restrict__ red,
                            uint32_t* __restrict__ excl) {
    for (long long w = blockIdx.x * (long long)blockDim.x + threadIdx.x; w < nw; w += (long long)gridDim.x * blockDim.x)
        excl[w] = slave[w] | red[w];
}

struct Flux6 {
    const double* g[6];
};

// b_c = -(1/dt) (sum of outward open-face fluxes + body flux) + prescribed Neumann fluxes
// Fluxes through partly open faces.  Not inlined: the compiler would predicate the products in every cell.
struct Flux5 {
    double xm, xp, ym, yp, zp;
};
__device__ __noinline__ Flux5 cut_fluxes(double x0, double x1, double y0, double y1, double z1, double Sx, double Sy,
                                         double Sz, double u0, double u1, double v0, double v1, double w1) {
    Flux5 f;
    f.xm = __dmul_rn(x0 * Sx, u0);
    f.xp = __dmul_rn(x1 * Sx, u1);
    f.ym = __dmul_rn(y0 * Sy, v0);
    f.yp = __dmul_rn(y1 * Sy, v1);
    f.zp = __dmul_rn(z1 * Sz, w1);
    return f;
}
// FP64 arithmetic bounds it (512 x 256 x 128; 0.94 GB, 140 us at copy bandwidth): 1057 us with both faces of every
// direction formed from three factors and a division in every cell; 757 here (23.7 FP64 instructions a cell), as a time
// step's dt takes it, and 505 (15.4) where dt is a power of two and the division a multiplication by its exact reciprocal,
// given as dt.  1 is one of them: without the multiplication it took 505 as well.
template <bool RECIPROCAL>
__global__ void __launch_bounds__(kNT, 5)
k_rhs(Dims d, March m, Bc6 bc, Flux6 nf, double dt, const double* __restrict__ dx,
                      const double* __restrict__ dy, const double* __restrict__ dz,
                      const double* __restrict__ axe, const double* __restrict__ aye,
                      const double* __restrict__ aze, const uint8_t* __restrict__ ina,
                      const double* __restrict__ u, const double* __restrict__ v,
                      const double* __restrict__ w, const double* __restrict__ body,
                      double* __restrict__ b) {
    const Column q = column_of(d, m);
    if (!q.on) return;
    const int i = q.i, j = q.j;
    const bool wall[6] = {i == 0 && bc.k[0] != VOFP_BC_DIRICHLET, i == d.nx - 1 && bc.k[1] != VOFP_BC_DIRICHLET,
                          j == 0 && bc.k[2] != VOFP_BC_DIRICHLET, j == d.ny - 1 && bc.k[3] != VOFP_BC_DIRICHLET,
                          bc.k[4] != VOFP_BC_DIRICHLET, bc.k[5] != VOFP_BC_DIRICHLET};
    const bool edge = (i == 0 && nf.g[0]) || (i == d.nx - 1 && nf.g[1]) || (j == 0 && nf.g[2]) || (j == d.ny - 1 && nf.g[3]);
    const double Sz = dy[j] * dx[i];
    long long c = q.c;
    double fzm = q.k0 == 0 && wall[4] ? 0.0 : aze[c] * Sz * w[c];
    long long fx = fx_idx(d, i, j, q.k0), fy = fy_idx(d, i, j, q.k0);
    const long long fxs = (long long)(d.nx + 1) * d.ny, fys = (long long)d.nx * (d.ny + 1);
    for (int k = q.k0; k < q.k1; ++k, c += d.plane, fx += fxs, fy += fys) {
        const long long fz = c + d.plane;
        const double x0 = axe[fx], x1 = axe[fx + 1], y0 = aye[fy], y1 = aye[fy + d.nx], z1 = aze[fz];
        const double u0 = u[fx], u1 = u[fx + 1], v0 = v[fy], v1 = v[fy + d.nx], w1 = w[fz];
        const bool off = ina[c] != 0;
        const double Sx = dz[k] * dy[j], Sy = dz[k] * dx[i];
        Flux5 f;
        if (whole_warp(is_one(x0) && is_one(x1) && is_one(y0) && is_one(y1) && is_one(z1))) {
            f.xm = __dmul_rn(Sx, u0);
            f.xp = __dmul_rn(Sx, u1);
            f.ym = __dmul_rn(Sy, v0);
            f.yp = __dmul_rn(Sy, v1);
            f.zp = __dmul_rn(Sz, w1);
        } else {
            f = cut_fluxes(x0, x1, y0, y1, z1, Sx, Sy, Sz, u0, u1, v0, v1, w1);
        }
        if (wall[0]) f.xm = 0.0;
        if (wall[1]) f.xp = 0.0;
        if (wall[2]) f.ym = 0.0;
        if (wall[3]) f.yp = 0.0;
        if (k == d.nz - 1 && wall[5]) f.zp = 0.0;
        double div = __dadd_rn(__dadd_rn(__dsub_rn(f.xp, f.xm), __dsub_rn(f.yp, f.ym)), __dsub_rn(f.zp, fzm));
        if (body) div += body[c];
        double bb = RECIPROCAL ? -div * dt : -div / dt;
        if (edge || (k == 0 && nf.g[4]) || (k == d.nz - 1 && nf.g[5])) {
            if (i == 0 && bc.k[0] == VOFP_BC_NEUMANN && nf.g[0]) bb += axe[fx_idx(d, 0, j, k)] * Sx * nf.g[0][j + (long long)d.ny * k];
            if (i == d.nx - 1 && bc.k[1] == VOFP_BC_NEUMANN && nf.g[1]) bb += axe[fx_idx(d, d.nx, j, k)] * Sx * nf.g[1][j + (long long)d.ny * k];
            if (j == 0 && bc.k[2] == VOFP_BC_NEUMANN && nf.g[2]) bb += aye[fy_idx(d, i, 0, k)] * Sy * nf.g[2][i + (long long)d.nx * k];
            if (j == d.ny - 1 && bc.k[3] == VOFP_BC_NEUMANN && nf.g[3]) bb += aye[fy_idx(d, i, d.ny, k)] * Sy * nf.g[3][i + (long long)d.nx * k];
            if (k == 0 && bc.k[4] == VOFP_BC_NEUMANN && nf.g[4]) bb += aze[fz_idx(d, i, j, 0)] * Sz * nf.g[4][i + (long long)d.nx * j];
            if (k == d.nz - 1 && bc.k[5] == VOFP_BC_NEUMANN && nf.g[5]) bb += aze[fz_idx(d, i, j, d.nz)] * Sz * nf.g[5][i + (long long)d.nx * j];
        }
        b[c] = off ? 0.0 : bb;
        fzm = f.zp;
    }
}

__global__ void k_group_fold(int ng, const int* __restrict__ gptr, const int* __restrict__ gcells,
                             double* __restrict__ v, int zero_slaves) {
    int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= ng) return;
    double s = 0.0;
    for (int t = gptr[g]; t < gptr[g + 1]; ++t) s += v[gcells[t]];
    v[gcells[gptr[g]]] = s;
    for (int t = gptr[g] + 1; t < gptr[g + 1]; ++t) v[gcells[t]] = zero_slaves ? 0.0 : s;
}

int grid_for(long long n) {
    long long b = (n + kNT - 1) / kNT;
    long long cap = (long long)num_sms() * 16;
    return int(std::max(1LL, std::min(b, cap)));
}

}  // namespace

void launch_group_fold(vofp_ctx* c, double* v, bool zero_slaves) {
    if (c->ngroups == 0) return;
    launch(c, k_group_fold, ceil_div(c->ngroups, kNT), kNT, c->stream, c->ngroups, c->gptr, c->gcells, v,
                                                                    zero_slaves ? 1 : 0);
}

// Resolve merge chains on the host: the root of a small cell is the end of its target chain;
// a cycle of small cells is rooted at its member of largest open volume (lowest index on ties).
// Small cells are addressed by their slot in the lists (any order): tslot[t] is the slot of the
// target of slot t, -1 when the target does not merge. The roots do not depend on the order.
static void resolve_roots(const std::vector<long long>& cells, const std::vector<long long>& targets,
                          const std::vector<double>& vfs, const std::vector<int32_t>& tslot,
                          std::vector<long long>& roots) {
    const long long m = (long long)cells.size();
    std::vector<long long> root(m, -1);      // resolved root cell per slot
    std::vector<long long> stamp(m, -1);     // first slot of the walk that last visited it
    std::vector<long long> where(m, 0);      // its index on that walk's path
    std::vector<long long> path;
    for (long long t0 = 0; t0 < m; ++t0) {
        if (root[t0] >= 0) continue;
        path.clear();
        long long q = t0, r;
        while (true) {
            if (root[q] >= 0) {
                r = root[q];
                break;
            }
            if (stamp[q] == t0) {
                // a cycle: path[where[q]] .. the end
                long long best = -1;
                double bv = -1.0;
                for (size_t k = (size_t)where[q]; k < path.size(); ++k) {
                    const long long cm = cells[path[k]];
                    const double vm = vfs[path[k]];
                    if (vm > bv || (vm == bv && cm < best)) {
                        bv = vm;
                        best = cm;
                    }
                }
                for (size_t k = (size_t)where[q]; k < path.size(); ++k) root[path[k]] = best;
                r = best;
                break;
            }
            stamp[q] = t0;
            where[q] = (long long)path.size();
            path.push_back(q);
            if (tslot[q] < 0) {
                r = targets[q];   // the chain ends at a cell that does not merge
                break;
            }
            q = tslot[q];
        }
        for (long long k : path)
            if (root[k] < 0) root[k] = r;
    }
    roots.assign(root.begin(), root.end());
}

// Device lists of the small cells, kept across operator builds and grown when they overflow.
static vofp_status grow_small(vofp_ctx* c, long long cap) {
    void* old[4] = {c->small_cells, c->small_targets, c->small_vf, c->small_tslot};
    for (void* p : old)
        if (p) {
            cudaFree(p);
            c->allocs.erase(std::remove(c->allocs.begin(), c->allocs.end(), p), c->allocs.end());
        }
    c->bytes -= c->small_cap * (long long)(2 * sizeof(long long) + sizeof(double) + sizeof(int32_t));
    c->small_cells = c->small_targets = nullptr;
    c->small_vf = nullptr;
    c->small_tslot = nullptr;
    c->small_cap = 0;
    vofp_status s;
    if ((s = c->alloc(&c->small_cells, cap)) || (s = c->alloc(&c->small_targets, cap)) ||
        (s = c->alloc(&c->small_vf, cap)) || (s = c->alloc(&c->small_tslot, cap)))
        return s;
    c->small_cap = cap;
    return VOFP_OK;
}

// Group arrays (offsets, cells, corrections), kept across builds and grown when too small.
static vofp_status grow_groups(vofp_ctx* c, long long ng, long long ncells) {
    if (ng + 1 <= c->gptr_cap && ncells <= c->gcells_cap) return VOFP_OK;
    void* old[3] = {c->gptr, c->gcells, c->gcorr};
    for (void* p : old)
        if (p) {
            cudaFree(p);
            c->allocs.erase(std::remove(c->allocs.begin(), c->allocs.end(), p), c->allocs.end());
        }
    c->bytes -= c->gptr_cap * (long long)(sizeof(int) + sizeof(double)) + c->gcells_cap * (long long)sizeof(int);
    c->gptr = c->gcells = nullptr;
    c->gcorr = nullptr;
    c->gptr_cap = c->gcells_cap = 0;
    const long long pc = (ng + 1) * 3 / 2 + 16, cc = ncells * 3 / 2 + 16;
    vofp_status s;
    if ((s = c->alloc(&c->gptr, pc)) || (s = c->alloc(&c->gcells, cc)) || (s = c->alloc(&c->gcorr, pc))) return s;
    c->gptr_cap = pc;
    c->gcells_cap = cc;
    return VOFP_OK;
}

vofp_status build_operator(vofp_ctx* c, const double* F, const double* ax, const double* ay,
                           const double* az, const double* vf, const vofp_bc* bc,
                           const vofp_phys* phys) {
    const Dims d = c->d;
    const long long N = d.n;
    const long long nfx = (long long)(d.nx + 1) * d.ny * d.nz;
    const long long nfy = (long long)d.nx * (d.ny + 1) * d.nz;
    const long long nfz = (long long)d.nx * d.ny * (d.nz + 1);
    cudaStream_t st = c->stream;
    vofp_status s;
    if (!c->Tx) {
        if ((s = c->alloc(&c->Tx, N)) || (s = c->alloc(&c->Ty, N)) || (s = c->alloc(&c->Tz, N)) ||
            (s = c->alloc(&c->diag, N)) || (s = c->alloc(&c->axe, nfx)) || (s = c->alloc(&c->aye, nfy)) ||
            (s = c->alloc(&c->aze, nfz)) || (s = c->alloc(&c->s, N)) || (s = c->alloc(&c->sq, N)) ||
            (s = c->alloc(&c->Txs, N)) || (s = c->alloc(&c->Tys, N)) || (s = c->alloc(&c->Tzs, N)) ||
            (s = c->alloc(&c->Txf, N)) || (s = c->alloc(&c->Tyf, N)) || (s = c->alloc(&c->Tzf, N)) ||
            (s = c->alloc(&c->Tzr, N)) || (s = c->alloc(&c->rho, N)) || (s = c->alloc(&c->kx, N)) ||
            (s = c->alloc(&c->ky, N)) || (s = c->alloc(&c->kz, N)) ||
            (s = c->alloc(&c->slave_bits, (N + 31) / 32)) || (s = c->alloc(&c->root, N)) ||
            (s = c->alloc(&c->red_bits, (N + 31) / 32)) || (s = c->alloc(&c->excl_bits, (N + 31) / 32)) ||
            (s = c->alloc(&c->inactive, N)) ||
            (s = c->alloc(&c->tab, 8 + 2 * ((long long)d.nx + d.ny + d.nz))) || (s = c->alloc(&c->work, N)) ||
            (s = c->alloc(&c->partials, kMaxPartials)) || (s = c->alloc(&c->counters, 64)) ||
            (s = c->alloc(&c->sc, 4)))
            return s;
        VOFP_CUDA_TRY(c, cudaMemsetAsync(c->counters, 0, 64 * sizeof(unsigned int), st));
    }
    c->built = false;
    c->rbc_built = false;
    c->rbc_ok = false;
    c->grp_built = false;
    c->mgf.built = c->mgf.ok = false;
    c->mgd.built = c->mgd.ok = false;
    c->mg_pays = -1;
    for (int f = 0; f < 6; ++f) c->bc[f] = bc->kind[f];
    c->phys = *phys;
    c->dirichlet = false;
    Bc6 b6;
    for (int f = 0; f < 6; ++f) {
        b6.k[f] = bc->kind[f];
        c->dirichlet |= bc->kind[f] == VOFP_BC_DIRICHLET;
    }
    const int gN = grid_for(N);
    const March m3 = march_of(d);
    const int gM = (int)ceil_div(d.plane * m3.nch, kNT);

    // density (Eq. density), optional smoothing (Sec. 2.10, through Txs)
    launch(c, k_tables, ceil_div(2 * (d.nx + d.ny + d.nz), kNT), kNT, st, d, phys->rho_liquid, phys->rho_gas,
           phys->density_smoothing ? 1 : 0, (const double*)c->dx, (const double*)c->dy, (const double*)c->dz, c->tab);
    if (phys->density_smoothing) {
        launch(c, k_density_x, gN, kNT, st, d, F, phys->rho_liquid, phys->rho_gas, (const double*)c->tab, c->Txs);
        launch(c, k_smooth_yz, gM, kNT, st, d, m3, (const double*)c->Txs, (const double*)c->tab, c->rho);
    } else {
        launch(c, k_density, gN, kNT, st, d, F, phys->rho_liquid, phys->rho_gas, (const double*)c->tab, c->rho);
    }
    // activity, effective apertures and small cells; the activity is iterated to a fixed point, which it
    // nearly always is at the start
    unsigned int* cnt = c->counters + 32;
    unsigned int hc[3] = {0, 0, 0};   // cells that lose their unknown, small cells, cells without one
    const double thr = vf ? phys->merge_threshold : 0.0;
    const uint8_t* settled = nullptr;
    for (int attempt = 0; attempt < 3; ++attempt) {
        VOFP_CUDA_TRY(c, cudaMemsetAsync(cnt, 0, sizeof(hc), st));
        launch(c, settled ? k_cells<1> : vf ? k_cells<0> : k_cells<2>, gM, kNT, st, d, m3, b6, thr, vf, settled, ax, ay, az,
               c->dx, c->dy, c->dz, c->inactive, c->root, c->axe, c->aye, c->aze, cnt, c->small_cap, c->small_cells,
               c->small_targets, c->small_vf);
        VOFP_CUDA_TRY(c, cudaMemcpyAsync(hc, cnt, sizeof(hc), cudaMemcpyDeviceToHost, st));
        VOFP_CUDA_TRY(c, cudaStreamSynchronize(st));
        const bool settle = !settled && hc[0] > 0, grow = (long long)hc[1] > c->small_cap;
        if (!settle && !grow) break;
        if (settle) {
            uint8_t* ina_a = reinterpret_cast<uint8_t*>(c->work);
            uint8_t* ina_b = ina_a + N;
            launch(c, k_activity_init, gN, kNT, st, d, vf, ina_a);
            for (int pass = 0; pass < 100000; ++pass) {
                VOFP_CUDA_TRY(c, cudaMemsetAsync(cnt, 0, sizeof(unsigned int), st));
                launch(c, k_activity_step, gN, kNT, st, d, b6, ax, ay, az, ina_a, ina_b, cnt);
                unsigned int h = 0;
                VOFP_CUDA_TRY(c, cudaMemcpyAsync(&h, cnt, sizeof(h), cudaMemcpyDeviceToHost, st));
                VOFP_CUDA_TRY(c, cudaStreamSynchronize(st));
                std::swap(ina_a, ina_b);
                if (h == 0) break;
            }
            settled = ina_a;
        }
        if (grow && attempt < 2 && (s = grow_small(c, (long long)hc[1] + hc[1] / 2 + 1024))) return s;
    }
    const unsigned int m = hc[1];
    if ((long long)m > c->small_cap) {
        c->set_error("small-cell count changed between two passes over the same input");
        return VOFP_ERR_CUDA;
    }
    c->n_inactive = hc[2];
    // prescribed Neumann fluxes are copied so the caller's arrays need not outlive this call
    for (int f = 0; f < 6; ++f) {
        const long long nb = f < 2 ? (long long)d.ny * d.nz : f < 4 ? (long long)d.nx * d.nz : (long long)d.nx * d.ny;
        if (bc->neumann_flux[f] && bc->kind[f] == VOFP_BC_NEUMANN) {
            if (!c->nflux[f] && (s = c->alloc(&c->nflux[f], nb))) return s;
            VOFP_CUDA_TRY(c, cudaMemcpyAsync(c->nflux[f], bc->neumann_flux[f], sizeof(double) * nb,
                                             cudaMemcpyDeviceToDevice, st));
            c->has_nflux[f] = true;
        } else {
            c->has_nflux[f] = false;
        }
    }
    // merge map (Sec. 2.3): small cells listed on the device, chains resolved on the host
    std::vector<long long> cells, targets, roots;
    std::vector<double> vfs;
    std::vector<int32_t> tslot;
    if (m > 0) {
        // the slots are mapped through Txs, which is not in use here
        int32_t* slot_of = reinterpret_cast<int32_t*>(c->Txs);
        VOFP_CUDA_TRY(c, cudaMemsetAsync(slot_of, 0xff, sizeof(int32_t) * N, st));
        launch(c, k_small_slots, ceil_div(m, kNT), kNT, st, (int)m, (const long long*)c->small_cells, slot_of);
        launch(c, k_small_target_slots, ceil_div(m, kNT), kNT, st, (int)m, (const long long*)c->small_targets,
               (const int32_t*)slot_of, c->small_tslot);
        cells.resize(m);
        targets.resize(m);
        vfs.resize(m);
        tslot.resize(m);
        VOFP_CUDA_TRY(c, cudaMemcpyAsync(cells.data(), c->small_cells, sizeof(long long) * m,
                                         cudaMemcpyDeviceToHost, st));
        VOFP_CUDA_TRY(c, cudaMemcpyAsync(targets.data(), c->small_targets, sizeof(long long) * m,
                                         cudaMemcpyDeviceToHost, st));
        VOFP_CUDA_TRY(c, cudaMemcpyAsync(vfs.data(), c->small_vf, sizeof(double) * m, cudaMemcpyDeviceToHost, st));
        VOFP_CUDA_TRY(c, cudaMemcpyAsync(tslot.data(), c->small_tslot, sizeof(int32_t) * m,
                                         cudaMemcpyDeviceToHost, st));
        VOFP_CUDA_TRY(c, cudaStreamSynchronize(st));
    }
    // the coefficients, the diagonal and its scaling do not need the merge map: the device forms them while the
    // host resolves it
    unsigned int* nred = c->counters + 35;
    VOFP_CUDA_TRY(c, cudaMemsetAsync(nred, 0, sizeof(unsigned int), st));
    launch(c, k_face_coeffs, gM, kNT, st, d, m3, c->dx, c->dy, c->dz, c->rho, c->axe, c->aye, c->aze, c->tab, c->Tx, c->Ty,
           c->Tz, c->kx, c->ky, c->kz);
    launch(c, k_diag_scale, gM, kNT, st, d, m3, b6, c->dx, c->dy, c->dz, c->rho, c->axe, c->aye, c->aze, c->Tx, c->Ty,
           c->Tz, c->inactive, c->diag, c->s, c->sq);
    launch(c, k_cell_bits, grid_for((N + 31) / 32), kNT, st, d, (const uint8_t*)c->inactive, c->slave_bits, c->red_bits,
           nred);
    resolve_roots(cells, targets, vfs, tslot, roots);
    // groups: cells whose root differs from themselves, plus the roots
    std::vector<std::pair<long long, long long>> members;   // (root, cell)
    for (size_t t = 0; t < cells.size(); ++t)
        if (roots[t] != cells[t]) members.push_back({roots[t], cells[t]});
    std::sort(members.begin(), members.end());
    std::vector<int> gptr(1, 0), gcells;
    for (size_t t = 0; t < members.size();) {
        long long r = members[t].first;
        gcells.push_back((int)r);
        while (t < members.size() && members[t].first == r) gcells.push_back((int)members[t++].second);
        gptr.push_back((int)gcells.size());
    }
    c->ngroups = (int)gptr.size() - 1;
    c->n_merged = (long long)members.size();
    c->n_unknowns = N - c->n_inactive - c->n_merged;
    if (c->ngroups > 0) {
        if ((s = grow_groups(c, c->ngroups, (long long)gcells.size()))) return s;
        VOFP_CUDA_TRY(c, cudaMemcpyAsync(c->gptr, gptr.data(), sizeof(int) * gptr.size(), cudaMemcpyHostToDevice, st));
        VOFP_CUDA_TRY(c, cudaMemcpyAsync(c->gcells, gcells.data(), sizeof(int) * gcells.size(), cudaMemcpyHostToDevice, st));
        // (cell, root) of every merged cell, through the small-cell lists (there are no more
        // merged cells than small cells); copies from pageable host memory are staged before
        // cudaMemcpyAsync returns, so the vectors may go out of scope
        std::vector<long long> mc, mr;
        mc.reserve(members.size());
        mr.reserve(members.size());
        for (auto& pr : members) {
            mc.push_back(pr.second);
            mr.push_back(pr.first);
        }
        VOFP_CUDA_TRY(c, cudaMemcpyAsync(c->small_cells, mc.data(), sizeof(long long) * mc.size(),
                                         cudaMemcpyHostToDevice, st));
        VOFP_CUDA_TRY(c, cudaMemcpyAsync(c->small_targets, mr.data(), sizeof(long long) * mr.size(),
                                         cudaMemcpyHostToDevice, st));
        launch(c, k_root_scatter, ceil_div((long long)mc.size(), kNT), kNT, st, (int)mc.size(),
               (const long long*)c->small_cells, (const long long*)c->small_targets, c->root);
    }
    // the groups' scale s = diag(A_hat)^-1/2 and flags
    if (c->ngroups > 0) {
        launch(c, k_scale_groups, ceil_div(c->ngroups, kNT), kNT, st, d, c->ngroups, c->gptr, c->gcells, c->root, c->diag,
                                                                  c->Tx, c->Ty, c->Tz, c->s, c->sq, c->gcorr);
        launch(c, k_group_flags, ceil_div(c->ngroups, kNT), kNT, st, c->ngroups, (const int*)c->gptr,
               (const int*)c->gcells, c->slave_bits, c->red_bits, nred);
    }
    launch(c, k_excl_bits, grid_for((N + 31) / 32), kNT, st, (N + 31) / 32, (const uint32_t*)c->slave_bits,
           (const uint32_t*)c->red_bits, c->excl_bits);
    launch(c, k_scaled_coeffs, gM, kNT, st, d, m3, (const double*)c->s, (const double*)c->Tx, (const double*)c->Ty,
           (const double*)c->Tz, (const uint32_t*)c->red_bits, c->Txs, c->Tys, c->Tzs, c->Txf, c->Tyf, c->Tzf, c->Tzr);
    unsigned int hred = 0;
    VOFP_CUDA_TRY(c, cudaMemcpyAsync(&hred, nred, sizeof(hred), cudaMemcpyDeviceToHost, st));
    VOFP_CUDA_TRY(c, cudaGetLastError());
    VOFP_CUDA_TRY(c, cudaStreamSynchronize(st));
    c->n_red = hred;
    c->built = true;
    return VOFP_OK;
}

vofp_status rhs(vofp_ctx* c, const double* u, const double* v, const double* w, const double* body,
                double* b) {
    const Dims d = c->d;
    Bc6 b6;
    for (int f = 0; f < 6; ++f) b6.k[f] = c->bc[f];
    Flux6 nf{};
    for (int f = 0; f < 6; ++f) nf.g[f] = c->has_nflux[f] ? c->nflux[f] : nullptr;
    const March m = march_of(d);
    const double dt = c->phys.dt;
    int e = 0;
    const bool pow2 = std::isnormal(dt) && std::fabs(std::frexp(dt, &e)) == 0.5 && std::isnormal(1.0 / dt);
    launch(c, pow2 ? k_rhs<true> : k_rhs<false>, ceil_div(d.plane * m.nch, kNT), kNT, c->stream, d, m, b6, nf,
           pow2 ? 1.0 / dt : dt, c->dx, c->dy, c->dz, c->axe, c->aye, c->aze, c->inactive, u, v, w, body, b);
    VOFP_CUDA_TRY(c, cudaGetLastError());
    return VOFP_OK;
}

}  // namespace vofp
