// FP64 particle cycle (Sec. III): CIC gather of the finite-difference field
// (Eqs. 3-4), leapfrog push (Eqs. 1-2), MD subcycling with the PPPM
// correction near grains (Eqs. 5-6), grain and electrode absorption,
// null-collision MCC with the argon background (Table I) and the fixed-point
// CIC deposit.
//
// This translation unit is compiled with --fmad=false: every product and sum
// rounds on its own, in the order written, so an FP64 step on the GPU is
// bit-identical to a plain FP64 CPU evaluation of the same formulas.
#include <algorithm>
#include <cmath>

#include "pic_internal.cuh"

namespace pic {
namespace {

struct Geo {
    int nx, ny, nz;
    double dx, Lx, Ly, Lz;
    double rdx;                  // 1 / dx rounded to nearest, or 0: divide
    unsigned long long fix_c;    // 1 / dx = fix_c 2^(-63 - fix_e), fix_c rounded down (0: not used, see fix_cell)
    int fix_e;
};

struct P64 {
    Geo g;
    double Lx, Ly;
    double dt, dtm;
    int M;
    int sp;
    double qmdt, qmdtm, hm, nu_max, de;
    unsigned long long null_below;   // a particle collides if its 32-bit draw is below this
    unsigned int* mcc_list;      // slots of this step's collision candidates
    unsigned int* mcc_n;
    double n_gas, sig_n, eps_exc, eps_ion, mr2, kc;
    int n_xs;
    const double* xs;
    uint2 key;
    const uint32_t* step;        // device step counter (Philox counter word 2)
    int flags;
    int ng;
    const double* gpos;
    const double* grad;
    const int* gcell;
    const double* gq;
    const double* gtab;
    unsigned long long* gabs;
    const int* cell_ng;
    const int* cell_g;
    const double* ex;
    const double* ey;
    const double* ez;
    unsigned long long* rq;
    double4* pos;
    double4* vel;
    const unsigned long long* nslot;
    unsigned long long* cnt;
    int* err;
    ChildRec* child;
    unsigned long long child_cap;
    unsigned long long* nch;
};

// x / dx, correctly rounded, from the rounded reciprocal: two residual
// corrections by fused multiply-adds (Markstein, IBM J. Res. Dev. 34, 1990: with
// y = RN(1 / b) and q within an ulp of a / b, RN(q + y RN(a - b q)) is the
// correctly rounded quotient; the first correction brings q there).  5 FP64
// instructions, where the pipe issues one every 16 cycles per warp and a
// particle divides six times.
__device__ __forceinline__ double over_dx(const Geo& g, double x)
{
    if (g.rdx == 0.0) return x / g.dx;
    double q = x * g.rdx;
    q = fma(fma(-q, g.dx, x), g.rdx, q);
    return fma(fma(-q, g.dx, x), g.rdx, q);
}

__device__ __forceinline__ void locate(const Geo& g, const double x[3], int c[3], double f[3])
{
    const int nn[3] = {g.nx, g.ny, g.nz};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const double q = over_dx(g, x[a]);
        int i = __double2int_rd(q);
        if (i > nn[a] - 1) i = nn[a] - 1;
        if (i < 0) i = 0;
        c[a] = i;
        f[a] = q - (double)i;
    }
}

// Fixed-point CIC weights: per axis a = round_half_even(f 2^14) in [0, 2^14] as an
// integer (deposit) and the pair (1 - a 2^-14, a 2^-14) in FP64 (gather; the
// products of three are exact).  The rounding is the sum with 1.5 2^52, whose
// last place is 1 and whose low word then holds the integer: no conversion.
struct Cic {
    int a[3];
    double w[3][2];
    __device__ __forceinline__ explicit Cic(const double f[3])
    {
        const double big = 6755399441055744.0;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const double t = f[d] * (double)kWQ + big;
            int q = __double2loint(t);
            double u = t - big;
            if (!(u >= 0.0)) { q = 0; u = 0.0; }
            if (u > (double)kWQ) { q = kWQ; u = (double)kWQ; }
            a[d] = q;
            w[d][1] = u * (1.0 / (double)kWQ);
            w[d][0] = 1.0 - w[d][1];
        }
    }
};

// Cell i and weight a of one coordinate in integer arithmetic: the FP64 pipe
// issues a warp instruction every 16 cycles and SM, the integer pipes two a
// cycle, so 30 integer instructions are cheaper than the 14 FP64 ones of
// locate and Cic.  With q = RN(x / dx), i = floor(q) and
// a = round_half_even((q - i) 2^14) (q - i is exact).  Here Y = x / dx 2^46 as an
// integer, off by at most 3 (the reciprocal and the product are each cut once),
// and q 2^46 itself is within 2^-53 x / dx 2^46 <= 2^9 of the exact quotient for
// x / dx < 2^16: unless Y lies within 2^12 of a cell boundary or of a tie, both
// results are those of any number within that distance, q among them.  Returns
// false there (one coordinate in 5e5, and coordinates on nodes), at x = 0, and
// for x / dx >= 2^16.
__device__ __forceinline__ bool fix_cell(const Geo& g, double x, int& i, int& a)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int E = (int)(b >> 52);                                // x >= 0: the biased exponent
    const unsigned long long m = ((b << 11) | (1ull << 63));     // significand, leading one made explicit
    const int sh = 1039 + g.fix_e - E;
    if (sh < 1 || sh > 63) return false;
    const unsigned long long Y = __umul64hi(m, g.fix_c) >> sh;
    const unsigned int hi = (unsigned int)(Y >> 32), lo = (unsigned int)Y;
    const unsigned long long t = Y + 4096ull;
    if (lo - 0x80000000u + 4096u < 8192u || ((((unsigned int)(t >> 32)) & 0x3fffu) == 0u && (unsigned int)t < 8192u))
        return false;
    i = (int)(hi >> 14);
    a = (int)((hi + (lo >> 31)) - ((unsigned int)i << 14));
    return true;
}

__device__ __noinline__ void exact_cell(const Geo& g, const double x[3], int c[3], int a[3])
{
    double f[3];
    locate(g, x, c, f);
    const Cic w(f);
#pragma unroll
    for (int d = 0; d < 3; ++d) a[d] = w.a[d];
}

// cell and integer weights of a position
__device__ __forceinline__ void cell_weights(const Geo& g, const double x[3], int c[3], int a[3])
{
    bool ok = g.fix_c != 0ull;
    if (ok)
#pragma unroll
        for (int d = 0; d < 3; ++d) ok = fix_cell(g, x[d], c[d], a[d]) && ok;
    if (!ok) exact_cell(g, x, c, a);
}

// n as a double, 0 <= n < 2^53, by integer instructions
__device__ __forceinline__ double exact_double(unsigned long long n)
{
    const int e = 63 - __clzll((long long)n);
    return n ? __longlong_as_double((long long)(((unsigned long long)(1022 + e) << 52) + (n << (52 - e)))) : 0.0;
}
// a whole number 0 <= v < 2^32
__device__ __forceinline__ unsigned int exact_uint(double v)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const int e = (int)(b >> 52) - 1023;
    return e < 0 ? 0u : (unsigned int)(((b & ((1ull << 52) - 1ull)) | (1ull << 52)) >> (52 - e));
}

// node index of the cell's corner (di, dy, dz), periodic in x and y
__device__ __forceinline__ unsigned int corner(const Geo& g, const int c[3], int di, int dy, int dz)
{
    const int i = c[0] + di == g.nx ? 0 : c[0] + di, j = c[1] + dy == g.ny ? 0 : c[1] + dy;
    return ((unsigned int)(c[2] + dz) * g.ny + j) * g.nx + i;
}

__device__ __forceinline__ int cell_of(const Geo& g, const int c[3]) { return (c[2] * g.ny + c[1]) * g.nx + c[0]; }

__device__ __forceinline__ void deposit(const Geo& g, unsigned long long* rq, const int c[3], const int a[3], int charge)
{
    const int x[2] = {charge * (kWQ - a[0]), charge * a[0]};
#pragma unroll
    for (int dz = 0; dz < 2; ++dz)
#pragma unroll
        for (int dy = 0; dy < 2; ++dy) {
            const int yz = (dy ? a[1] : kWQ - a[1]) * (dz ? a[2] : kWQ - a[2]);
#pragma unroll
            for (int di = 0; di < 2; ++di) {
                const long long v = (long long)x[di] * yz;
                if (v != 0) atomicAdd(rq + corner(g, c, di, dy, dz), (unsigned long long)v);
            }
        }
}

__device__ __forceinline__ void gather(const Geo& g, const double* fx, const double* fy, const double* fz,
                                       const int c[3], const Cic& w, double E[3])
{
    E[0] = 0.0; E[1] = 0.0; E[2] = 0.0;
#pragma unroll
    for (int dz = 0; dz < 2; ++dz)
#pragma unroll
        for (int dy = 0; dy < 2; ++dy) {
            const double yz = w.w[1][dy] * w.w[2][dz];
#pragma unroll
            for (int di = 0; di < 2; ++di) {
                const double wt = w.w[0][di] * yz;
                const unsigned int n = corner(g, c, di, dy, dz);
                E[0] = E[0] + wt * fx[n];
                E[1] = E[1] + wt * fy[n];
                E[2] = E[2] + wt * fz[n];
            }
        }
}

// The same gather times 2^42, from the integer weights: the products of three are
// whole numbers, exact in FP64, and the scale is a power of two, so every sum
// rounds as in `gather`.
__device__ __forceinline__ void gather_scaled(const Geo& g, const double* fx, const double* fy, const double* fz,
                                              const int c[3], const int a[3], double E[3])
{
    E[0] = 0.0; E[1] = 0.0; E[2] = 0.0;
#pragma unroll
    for (int dz = 0; dz < 2; ++dz)
#pragma unroll
        for (int dy = 0; dy < 2; ++dy) {
            const unsigned int yz = (unsigned int)((dy ? a[1] : kWQ - a[1]) * (dz ? a[2] : kWQ - a[2]));
#pragma unroll
            for (int di = 0; di < 2; ++di) {
                const double wt = exact_double((unsigned long long)(unsigned int)(di ? a[0] : kWQ - a[0]) * yz);
                const unsigned int n = corner(g, c, di, dy, dz);
                E[0] = E[0] + wt * fx[n];
                E[1] = E[1] + wt * fy[n];
                E[2] = E[2] + wt * fz[n];
            }
        }
}

__device__ __forceinline__ void grain_sep(const P64& p, int gi, const double x[3], double d[3])
{
    const double L[2] = {p.Lx, p.Ly};
#pragma unroll
    for (int a = 0; a < 2; ++a) {
        double q = x[a] - p.gpos[3 * gi + a];
        if (q > 0.5 * L[a]) q = q - L[a];
        else if (q < -0.5 * L[a]) q = q + L[a];
        d[a] = q;
    }
    d[2] = x[2] - p.gpos[3 * gi + 2];
}

// E = E_PIC - Q g(x) + Q (x - x_g) / (4 pi eps0 |x - x_g|^3) for the grains whose
// MD region holds the particle's cell (Eqs. 5-6)
__device__ void md_correct(const P64& p, const Geo& g, const double x[3], const int c[3], const Cic& w, double E[3])
{
    const int cell = cell_of(g, c);
    const int n = p.cell_ng[cell];
    for (int t = 0; t < n; ++t) {
        const int gi = p.cell_g[cell * kMaxG + t];
        const int gc0 = p.gcell[3 * gi], gc1 = p.gcell[3 * gi + 1], gc2 = p.gcell[3 * gi + 2];
        double Ed[3] = {0.0, 0.0, 0.0};
        for (int dz = 0; dz < 2; ++dz)
            for (int dy = 0; dy < 2; ++dy)
                for (int di = 0; di < 2; ++di) {
                    const double wt = w.w[0][di] * (w.w[1][dy] * w.w[2][dz]);
                    const int li = ((c[0] + di - gc0 + 1) % g.nx + g.nx) % g.nx;
                    const int lj = ((c[1] + dy - gc1 + 1) % g.ny + g.ny) % g.ny;
                    const int lk = c[2] + dz - gc2 + 1;
                    const double* tv = p.gtab + ((size_t)gi * 64 + (lk * 4 + lj) * 4 + li) * 3;
                    Ed[0] = Ed[0] + wt * tv[0];
                    Ed[1] = Ed[1] + wt * tv[1];
                    Ed[2] = Ed[2] + wt * tv[2];
                }
        double d[3];
        grain_sep(p, gi, x, d);
        const double r2 = (d[0] * d[0] + d[1] * d[1]) + d[2] * d[2];
        const double Q = p.gq[gi];
        double coef = 0.0;
        if (r2 > 0.0) {
            const double r = sqrt(r2);
            coef = (Q * p.kc) / (r2 * r);
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) E[a] = (E[a] - Q * Ed[a]) + coef * d[a];
    }
}

// 0 alive, 1 lost at z = 0, 2 lost at z = Lz, 3 invalid; the comparisons on the
// bits (ordered as the values from +0 up)
__device__ __forceinline__ int boundary(const Geo& g, double x[3])
{
    const long long inf = 0x7ff0000000000000ll, minus0 = (long long)0x8000000000000000ull;
    const long long z = __double_as_longlong(x[2]);
    if ((z & 0x7fffffffffffffffll) > inf) return 3;
    if (z < 0 && z != minus0) return 1;
    if (z > __double_as_longlong(g.Lz)) return 2;
    const double L[2] = {g.Lx, g.Ly};
#pragma unroll
    for (int a = 0; a < 2; ++a) {
        const long long b = __double_as_longlong(x[a]);
        const bool below = b < 0 && b != minus0;
        if (!below && b < __double_as_longlong(L[a])) continue;
        x[a] = below ? x[a] + L[a] : x[a] - L[a];
        if (!(x[a] >= 0.0 && x[a] <= L[a])) return 3;
    }
    return 0;
}

__device__ int absorbed_by(const P64& p, const Geo& g, const double x[3])
{
    int c[3];
    double f[3];
    locate(g, x, c, f);
    const int cell = cell_of(g, c);
    const int n = p.cell_ng[cell];
    for (int t = 0; t < n; ++t) {
        const int gi = p.cell_g[cell * kMaxG + t];
        double d[3];
        grain_sep(p, gi, x, d);
        const double r2 = (d[0] * d[0] + d[1] * d[1]) + d[2] * d[2];
        if (r2 <= p.grad[gi] * p.grad[gi]) return gi;
    }
    return -1;
}

__device__ __forceinline__ double xs_at(const double* tab, int n, double de, double eps)
{
    const double t = eps / de;
    if (t >= (double)(n - 1)) return tab[n - 1];
    const int i = (int)t;
    const double fr = t - (double)i;
    return tab[i] + fr * (tab[i + 1] - tab[i]);
}

__device__ __forceinline__ void pair(RStream& r, double& a, double& b)
{
    const uint32_t ua = r.next(), ub = r.next();
    a = 2.0 * u01d(ua) - 1.0;
    b = 2.0 * u01d(ub) - 1.0;
}

// isotropic direction (Marsaglia 1972)
__device__ void iso(RStream& r, double o[3])
{
    for (int t = 0; t < 128; ++t) {
        double a, b;
        pair(r, a, b);
        const double s = a * a + b * b;
        if (s < 1.0) {
            const double q = 2.0 * sqrt(1.0 - s);
            o[0] = a * q; o[1] = b * q; o[2] = 1.0 - 2.0 * s;
            return;
        }
    }
    o[0] = 0.0; o[1] = 0.0; o[2] = 1.0;
}

// two standard normals (Marsaglia polar method)
__device__ void gauss2(RStream& r, double& n1, double& n2)
{
    for (int t = 0; t < 128; ++t) {
        double a, b;
        pair(r, a, b);
        const double s = a * a + b * b;
        if (s < 1.0) {
            const double f = sqrt((-2.0 * ln_series(s)) / s);
            n1 = a * f; n2 = b * f;
            return;
        }
    }
    n1 = 0.0; n2 = 0.0;
}

__device__ void gauss3(RStream& r, double o[3])
{
    double d;
    gauss2(r, o[0], o[1]);
    gauss2(r, o[2], d);
}

__device__ __forceinline__ void latch(int* err, int code) { atomicCAS(err, 0, code); }

// process choice and kinematics of a collision candidate (Table I); u = its
// Philox draw; may record an ionization product
__device__ void mcc(const P64& p, uint32_t step, uint4 u, const double x[3], double v[3], uint32_t id, int cell)
{
    const double ng = p.n_gas;
    const int nx = p.n_xs;
    if (p.sp == 0) {
        const double v2 = (v[0] * v[0] + v[1] * v[1]) + v[2] * v[2];
        const double eps = v2 * p.hm;
        const double vm = sqrt(v2);
        const double nu_el = (ng * xs_at(p.xs + 0 * nx, nx, p.de, eps)) * vm;
        const double nu_ex = (ng * xs_at(p.xs + 1 * nx, nx, p.de, eps)) * vm;
        const double nu_io = (ng * xs_at(p.xs + 2 * nx, nx, p.de, eps)) * vm;
        const double R = u01d(u.y) * p.nu_max;
        double acc = nu_el;
        RStream rd(id, step, kPurDir, p.key);
        double dir[3];
        if (R < acc) {
            iso(rd, dir);
            const double cosx = ((dir[0] * v[0] + dir[1] * v[1]) + dir[2] * v[2]) / vm;
            const double fac = 1.0 - p.mr2 * (1.0 - cosx);
            const double vn = vm * sqrt(fac);
#pragma unroll
            for (int a = 0; a < 3; ++a) v[a] = vn * dir[a];
            atomicAdd(p.cnt + PIC_C_E_EL, 1ull);
            return;
        }
        acc = acc + nu_ex;
        if (R < acc) {
            double e2 = eps - p.eps_exc;
            if (e2 < 0.0) e2 = 0.0;
            iso(rd, dir);
            const double vn = sqrt(e2 / p.hm);
#pragma unroll
            for (int a = 0; a < 3; ++a) v[a] = vn * dir[a];
            atomicAdd(p.cnt + PIC_C_E_EXC, 1ull);
            return;
        }
        acc = acc + nu_io;
        if (R < acc) {
            double e2 = eps - p.eps_ion;
            if (e2 < 0.0) e2 = 0.0;
            const double vn = sqrt((0.5 * e2) / p.hm);
            iso(rd, dir);
            ChildRec cr;
            cr.parent = id;
            cr.cell = cell;
#pragma unroll
            for (int a = 0; a < 3; ++a) { v[a] = vn * dir[a]; cr.x[a] = x[a]; }
            double d2[3], gn[3];
            RStream rc(id, step, kPurChildDir, p.key);
            iso(rc, d2);
            RStream rn(id, step, kPurChildNeutral, p.key);
            gauss3(rn, gn);
#pragma unroll
            for (int a = 0; a < 3; ++a) { cr.ve[a] = vn * d2[a]; cr.vi[a] = p.sig_n * gn[a]; }
            const unsigned long long slot = atomicAdd(p.nch, 1ull);
            if (slot < p.child_cap) p.child[slot] = cr;
            else latch(p.err, kErrCapacity);
            atomicAdd(p.cnt + PIC_C_E_ION, 1ull);
        }
        return;
    }
    double gn[3];
    RStream rn(id, step, kPurNeutral, p.key);
    gauss3(rn, gn);
    const double vn[3] = {p.sig_n * gn[0], p.sig_n * gn[1], p.sig_n * gn[2]};
    const double gv[3] = {v[0] - vn[0], v[1] - vn[1], v[2] - vn[2]};
    const double g2 = (gv[0] * gv[0] + gv[1] * gv[1]) + gv[2] * gv[2];
    const double eps = g2 * p.hm;
    const double gm = sqrt(g2);
    const double nu_el = (ng * xs_at(p.xs + 3 * nx, nx, p.de, eps)) * gm;
    const double nu_cx = (ng * xs_at(p.xs + 4 * nx, nx, p.de, eps)) * gm;
    const double R = u01d(u.y) * p.nu_max;
    double acc = nu_el;
    if (R < acc) {
        double dir[3];
        RStream rd(id, step, kPurDir, p.key);
        iso(rd, dir);
#pragma unroll
        for (int a = 0; a < 3; ++a) v[a] = (v[a] + vn[a]) * 0.5 + (0.5 * gm) * dir[a];
        atomicAdd(p.cnt + PIC_C_I_EL, 1ull);
        return;
    }
    acc = acc + nu_cx;
    if (R < acc) {
#pragma unroll
        for (int a = 0; a < 3; ++a) v[a] = vn[a];
        atomicAdd(p.cnt + PIC_C_I_CX, 1ull);
    }
}

// One step of every particle of both species (blockIdx.y): gather, push (MD
// particles with their substeps), absorption, the null-collision test and the
// deposit.  The few per cent that pass the test are listed for k_mcc64: their
// collision, a long chain of FP64 divisions and roots, would otherwise run in
// almost every warp with one or two lanes active.
// FP64 bound: the pipe issues one warp instruction per 16 cycles and SM, so what
// counts is FP64 instructions per particle: 75, of which the gather's products
// and sums are 48 (each rounds on its own) and the push 12; cells, weights,
// comparisons and the null test are integer work (fix_cell, exact_double,
// boundary).  5e6 particles per species, one launch for both: 2 x 2.42 -> 1.98 ms
// (with the collisions listed and divisions as products only, 163 FP64
// instructions, 3.99 ms), the pipe 73% active.  5 blocks per SM: 1.98 ms, 3 (all
// registers) 2.00, 8 2.06.
constexpr int kPush64Threads = 128;
constexpr int kCand64 = 512;   // candidates a block stages before they go to the list one by one

__global__ void __launch_bounds__(kPush64Threads, 5) k_push64(const P64 pe, const P64 pi)
{
    __shared__ unsigned int s_n, s_base, s_cand[kCand64];
    const P64& p = blockIdx.y == 0 ? pe : pi;
    const Geo& g = p.g;
    const unsigned long long n = p.nslot[p.sp];
    const uint32_t step = *p.step;
    const bool frozen = (p.sp == 1) && (p.flags & PIC_F_IONS_FROZEN);
    const int charge = p.sp == 0 ? -1 : 1;
    unsigned int live = 0;
    if (threadIdx.x == 0) s_n = 0u;
    __syncthreads();
    for (unsigned long long q = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; q < n;
         q += (unsigned long long)gridDim.x * blockDim.x) {
        double4 P = p.pos[q];
        if (__double2hiint(P.w) < 0) continue;   // dead: -1
        ++live;
        double x[3] = {P.x, P.y, P.z};
        int c[3], ci[3];
        cell_weights(g, x, c, ci);
        if (frozen) {
            deposit(g, p.rq, c, ci, charge);
            continue;
        }
        const double4 V = p.vel[q];
        double v[3] = {V.x, V.y, V.z};
        int fate = 0, grain = -1;
        if (p.cell_ng[cell_of(g, c)] == 0) {
            double E[3];
            gather_scaled(g, p.ex, p.ey, p.ez, c, ci, E);
#pragma unroll
            for (int a = 0; a < 3; ++a) v[a] = v[a] + p.qmdt * E[a];   // (qmdt carries the 2^-42)
#pragma unroll
            for (int a = 0; a < 3; ++a) x[a] = x[a] + v[a] * p.dt;
            fate = boundary(g, x);
        } else {
            for (int m = 0; m < p.M; ++m) {
                double E[3], f[3];
                locate(g, x, c, f);
                const Cic w(f);
                gather(g, p.ex, p.ey, p.ez, c, w, E);
                md_correct(p, g, x, c, w, E);
#pragma unroll
                for (int a = 0; a < 3; ++a) v[a] = v[a] + p.qmdtm * E[a];
#pragma unroll
                for (int a = 0; a < 3; ++a) x[a] = x[a] + v[a] * p.dtm;
                fate = boundary(g, x);
                if (fate) break;
                grain = absorbed_by(p, g, x);
                if (grain >= 0) break;
            }
        }
        if (fate != 0 || grain >= 0) {
            p.pos[q].w = -1.0;
            if (fate == 1) atomicAdd(p.cnt + (p.sp == 0 ? PIC_C_LOST_BOT_E : PIC_C_LOST_BOT_I), 1ull);
            else if (fate == 2) atomicAdd(p.cnt + (p.sp == 0 ? PIC_C_LOST_TOP_E : PIC_C_LOST_TOP_I), 1ull);
            else if (fate == 3) {
                atomicAdd(p.cnt + PIC_C_ERR, 1ull);
                latch(p.err, kErrNonFinite);
            } else {
                atomicAdd(p.gabs + 2 * grain + p.sp, 1ull);
                atomicAdd(p.cnt + (p.sp == 0 ? PIC_C_ABS_E : PIC_C_ABS_I), 1ull);
            }
            continue;
        }
        cell_weights(g, x, c, ci);
        if (!(p.flags & PIC_F_NO_MCC)) {
            const uint4 u = philox4x32_10(make_uint4(exact_uint(V.w), step, kPurMCC, 0u), p.key);
            // (u + 1/2) 2^-32 < pnull, both sides exact
            if ((unsigned long long)u.x < p.null_below) {
                const unsigned int at = atomicAdd(&s_n, 1u);
                if (at < kCand64) s_cand[at] = (unsigned int)q;
                else p.mcc_list[atomicAdd(p.mcc_n, 1u)] = (unsigned int)q;
            }
        }
        p.pos[q] = make_double4(x[0], x[1], x[2], exact_double((unsigned long long)(unsigned int)cell_of(g, c)));
        p.vel[q] = make_double4(v[0], v[1], v[2], V.w);
        deposit(g, p.rq, c, ci, charge);
    }
    live = __reduce_add_sync(0xffffffffu, live);
    if ((threadIdx.x & 31) == 0 && live) atomicAdd(p.cnt + PIC_C_PUSHED, (unsigned long long)live);
    __syncthreads();
    const unsigned int k = min(s_n, (unsigned int)kCand64);
    if (threadIdx.x == 0 && k) s_base = atomicAdd(p.mcc_n, k);
    __syncthreads();
    for (unsigned int t = threadIdx.x; t < k; t += blockDim.x) p.mcc_list[s_base + t] = s_cand[t];
}

// the listed collision candidates of both species (blockIdx.y), after the push
__global__ void __launch_bounds__(kPush64Threads) k_mcc64(const P64 pe, const P64 pi)
{
    const P64& p = blockIdx.y == 0 ? pe : pi;
    const unsigned int n = *p.mcc_n;
    const uint32_t step = *p.step;
    for (unsigned int t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) {
        const unsigned int q = p.mcc_list[t];
        const double4 P = p.pos[q], V = p.vel[q];
        const uint32_t id = (uint32_t)V.w;
        const uint4 u = philox4x32_10(make_uint4(id, step, kPurMCC, 0u), p.key);
        const double x[3] = {P.x, P.y, P.z};
        double v[3] = {V.x, V.y, V.z};
        mcc(p, step, u, x, v, id, (int)P.w);
        p.vel[q] = make_double4(v[0], v[1], v[2], V.w);
    }
}

// deposit every live particle (initial rho and re-deposits)
__global__ void k_deposit64(Geo g, const double4* pos, const unsigned long long* nslot, int sp,
                            unsigned long long* rq)
{
    const unsigned long long n = nslot[sp];
    const int charge = sp == 0 ? -1 : 1;
    for (unsigned long long q = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; q < n;
         q += (unsigned long long)gridDim.x * blockDim.x) {
        const double4 P = pos[q];
        if (P.w < 0.0) continue;
        const double x[3] = {P.x, P.y, P.z};
        int c[3];
        double f[3];
        locate(g, x, c, f);
        deposit(g, rq, c, Cic(f).a, charge);
    }
}

// E = -grad phi at the nodes (Eq. 4): central differences, one-sided second
// order on the electrode planes
__global__ void k_efield64(int nx, int ny, int nz, double dx, const double* __restrict__ phi, double* __restrict__ ex,
                           double* __restrict__ ey, double* __restrict__ ez)
{
    const size_t P = (size_t)nx * ny;
    const size_t N = P * (nz + 1);
    const double h2 = 2.0 * dx;
    for (size_t n = blockIdx.x * (size_t)blockDim.x + threadIdx.x; n < N; n += (size_t)gridDim.x * blockDim.x) {
        const int i = (int)(n % nx);
        const int j = (int)((n / nx) % ny);
        const int k = (int)(n / P);
        const size_t row = ((size_t)k * ny + j) * nx;
        const int ip = (i + 1) % nx, im = (i + nx - 1) % nx;
        const int jp = (j + 1) % ny, jm = (j + ny - 1) % ny;
        ex[n] = (phi[row + im] - phi[row + ip]) / h2;
        ey[n] = (phi[((size_t)k * ny + jm) * nx + i] - phi[((size_t)k * ny + jp) * nx + i]) / h2;
        if (k == 0)
            ez[n] = ((3.0 * phi[n] - 4.0 * phi[n + P]) + phi[n + 2 * P]) / h2;
        else if (k == nz)
            ez[n] = ((4.0 * phi[n - P] - 3.0 * phi[n]) - phi[n - 2 * P]) / h2;
        else
            ez[n] = (phi[n - P] - phi[n + P]) / h2;
    }
}

// Number the ionization products by their parents' ids (rank among this
// step's parents), append electron/ion pairs after the live slots, deposit.
__global__ void k_children64(Geo g, ChildRec* rec, const unsigned long long* nch, unsigned long long child_cap,
                             const unsigned long long* nslot, const unsigned int* next_id, double4* pos_e,
                             double4* vel_e, double4* pos_i, double4* vel_i, long long cap_e, long long cap_i,
                             unsigned long long* rq, int* err)
{
    __shared__ uint32_t tile[256];
    const unsigned long long n = min(*nch, child_cap);   // records past the buffer were never written
    const unsigned long long base_e = nslot[0], base_i = nslot[1];
    const unsigned int nid = *next_id;
    for (unsigned long long r0 = blockIdx.x * (unsigned long long)blockDim.x; r0 < n;
         r0 += (unsigned long long)gridDim.x * blockDim.x) {
        const unsigned long long r = r0 + threadIdx.x;
        const uint32_t mine = r < n ? rec[r].parent : 0xFFFFFFFFu;
        unsigned long long rank = 0;
        for (unsigned long long t0 = 0; t0 < n; t0 += blockDim.x) {
            __syncthreads();
            tile[threadIdx.x] = (t0 + threadIdx.x < n) ? rec[t0 + threadIdx.x].parent : 0xFFFFFFFFu;
            __syncthreads();
            const int lim = (int)min((unsigned long long)blockDim.x, n - t0);
            for (int t = 0; t < lim; ++t) rank += tile[t] < mine;
        }
        if (r >= n) continue;
        const ChildRec cr = rec[r];
        const unsigned long long se = base_e + rank, si = base_i + rank;
        if (se >= (unsigned long long)cap_e || si >= (unsigned long long)cap_i) {
            atomicCAS(err, 0, (int)kErrCapacity);
            continue;
        }
        const double x[3] = {cr.x[0], cr.x[1], cr.x[2]};
        int c[3];
        double f[3];
        locate(g, x, c, f);
        const Cic w(f);
        const double cell = (double)cell_of(g, c);
        pos_e[se] = make_double4(x[0], x[1], x[2], cell);
        vel_e[se] = make_double4(cr.ve[0], cr.ve[1], cr.ve[2], (double)(nid + (unsigned)(2 * rank)));
        pos_i[si] = make_double4(x[0], x[1], x[2], cell);
        vel_i[si] = make_double4(cr.vi[0], cr.vi[1], cr.vi[2], (double)(nid + (unsigned)(2 * rank + 1)));
        deposit(g, rq, c, w.a, -1);
        deposit(g, rq, c, w.a, 1);
    }
}

__global__ void k_children_finish(unsigned long long* nch, unsigned long long child_cap, unsigned long long* nslot,
                                  unsigned int* next_id, long long cap_e, long long cap_i, uint32_t* step)
{
    *step += 1u;   // the step is complete on the particle side
    const unsigned long long n = min(*nch, child_cap);
    nslot[0] = min(nslot[0] + n, (unsigned long long)cap_e);
    nslot[1] = min(nslot[1] + n, (unsigned long long)cap_i);
    *next_id += (unsigned int)(2 * n);
    *nch = 0;
}

// grain charges from the exact counts (Q = e W (N_ion - N_e)) and their CIC deposit
__global__ void k_grains(Geo g, int ng, double qw, const unsigned long long* gabs, const double* gpos, double* gq,
                         float* gq32, unsigned long long* rq)
{
    const int gi = blockIdx.x * blockDim.x + threadIdx.x;
    if (gi >= ng) return;
    const long long net = (long long)gabs[2 * gi + 1] - (long long)gabs[2 * gi];
    const double Q = qw * (double)net;
    gq[gi] = Q;
    gq32[gi] = (float)Q;
    const double x[3] = {gpos[3 * gi], gpos[3 * gi + 1], gpos[3 * gi + 2]};
    int c[3];
    double f[3];
    locate(g, x, c, f);
    const Cic w(f);
#pragma unroll
    for (int d = 0; d < 8; ++d) {
        const int di = d & 1, dy = (d >> 1) & 1, dz = d >> 2;
        const long long v = net * ((long long)(di ? w.a[0] : kWQ - w.a[0]) * ((dy ? w.a[1] : kWQ - w.a[1]) *
                                                                            (dz ? w.a[2] : kWQ - w.a[2])));
        if (v != 0) atomicAdd(rq + corner(g, c, di, dy, dz), (unsigned long long)v);
    }
}

// The grains of each MD cell (the 3 x 3 x 3 cells around a grain's own, periodic in x
// and y), in grain order; at most kMaxG, as the caller has checked.  A thread per
// grain and cell claims the cell's next entry; the first to come leaves its grain's
// complement, by which the second kernel knows the one thread that sorts the cell's
// entries.  On the host the tables of 64 x 64 x 128 cells took 0.4 ms to fill and
// 0.2 ms to copy.
__device__ __forceinline__ size_t list_cell(int nx, int ny, const int* gcell, int g, int o)
{
    const int i = (gcell[3 * g] + o % 3 - 1 + nx) % nx, j = (gcell[3 * g + 1] + (o / 3) % 3 - 1 + ny) % ny;
    return ((size_t)(gcell[3 * g + 2] + o / 9 - 1) * ny + j) * nx + i;
}

__global__ void k_cell_claim(int ng, int nx, int ny, const int* gcell, int* cell_ng, int* cell_g)
{
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= 27LL * ng) return;
    const int g = (int)(t / 27);
    const size_t c = list_cell(nx, ny, gcell, g, (int)(t % 27));
    const int at = atomicAdd(cell_ng + c, 1);
    if (at < kMaxG) cell_g[c * kMaxG + at] = at == 0 ? ~g : g;
}

__global__ void k_cell_order(int ng, int nx, int ny, const int* gcell, const int* cell_ng, int* cell_g)
{
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= 27LL * ng) return;
    const int g = (int)(t / 27);
    const size_t c = list_cell(nx, ny, gcell, g, (int)(t % 27));
    int* l = cell_g + c * kMaxG;
    if (l[0] != ~g) return;
    const int n = min(cell_ng[c], kMaxG);
    int v[kMaxG];
    v[0] = g;
    for (int a = 1; a < n; ++a) {
        const int x = l[a];
        int b = a;
        for (; b > 0 && v[b - 1] > x; --b) v[b] = v[b - 1];
        v[b] = x;
    }
    for (int a = 0; a < n; ++a) l[a] = v[a];
}

// The unit-charge tables by superposition: the mesh is periodic in x and y,
// so the potential of a unit charge on node (i, j, k) is that of a unit charge
// on node (0, 0, k) moved by (i, j).  k_green_block gives that potential for
// every node plane k that some grain's cell corners lie on, at offsets -3..3 in
// x, y and z around the node.  A grain's unit charge is its CIC deposit on the 8
// corners of its cell (the weights of k_grains, summing to 2^42), so its
// potential near the grain is the weighted sum of the 8 corners' moved blocks,
// and k_grain_table_sup takes its table from that sum with central
// differences (one-sided second-order ones on the electrodes).
constexpr int kGreenR = 3, kGreenW = 2 * kGreenR + 1;
constexpr int kGreenThreads = 512;

// The discrete potential of a unit charge on node (0, 0, k) in closed form: a
// cosine sum over the Fourier modes in x and y of the tridiagonal operator's
// inverse in z,
//     G(k', k) = sinh(theta k_<) sinh(theta (nz - k_>)) / (sinh theta sinh theta nz),
// 4 sinh^2(theta / 2) the mode's eigenvalue (k_< (nz - k_>) / nz for the constant
// mode).  Block (plane, z offset): the modes with 0 <= 2 mx <= nx, 0 <= 2 my <= ny
// (the others repeat them) over its threads, 4 x 4 sums for the offsets 0..3 in
// x and y, added in thread order.  It replaces an iterative solve of the whole
// mesh to 1e-12 per plane: FP64 bound, about 300 instructions per mode; the start
// of a run of 64 x 64 x 128 cells with 2e6 particles and 7 grains went from 13.0 to
// 5.4 ms with it (and to 3.2 ms with fewer allocations).
__global__ void __launch_bounds__(kGreenThreads) k_green_block(int nx, int ny, int nz, double c0, const int* planes,
                                                              double* blk)
{
    constexpr int D = kGreenR + 1, NW = kGreenThreads / 32;
    __shared__ double red[NW][D * D];
    const int k = planes[blockIdx.x], kk = k + (int)blockIdx.y - kGreenR;
    const int lo = min(k, kk), hi = max(k, kk);
    double s[D * D];
#pragma unroll
    for (int q = 0; q < D * D; ++q) s[q] = 0.0;
    const int hx = nx / 2 + 1, hy = ny / 2 + 1;
    if (lo > 0 && hi < nz)
        for (int m = threadIdx.x; m < hx * hy; m += kGreenThreads) {
            const int mx = m % hx, my = m / hx;
            const double sx = sinpi((double)mx / nx), sy = sinpi((double)my / ny);
            double g;
            if (m == 0) {
                g = ((double)lo * (double)(nz - hi)) / (double)nz;
            } else {
                const double th = 2.0 * asinh(sqrt(sx * sx + sy * sy));
                g = exp(-th * (double)(hi - lo + 1)) * (expm1(-2.0 * th * lo) * expm1(-2.0 * th * (nz - hi))) /
                    (expm1(-2.0 * th) * expm1(-2.0 * th * nz));
            }
            // modes that occur twice
            if (mx > 0 && 2 * mx < nx) g *= 2.0;
            if (my > 0 && 2 * my < ny) g *= 2.0;
            double cx[D], cy[D];   // cos(2 pi m d / n), d = 0..3
            cx[0] = cy[0] = 1.0;
            cx[1] = 1.0 - 2.0 * sx * sx;
            cy[1] = 1.0 - 2.0 * sy * sy;
#pragma unroll
            for (int d = 2; d < D; ++d) {
                cx[d] = 2.0 * cx[1] * cx[d - 1] - cx[d - 2];
                cy[d] = 2.0 * cy[1] * cy[d - 1] - cy[d - 2];
            }
#pragma unroll
            for (int q = 0; q < D * D; ++q) s[q] += g * (cy[q / D] * cx[q % D]);
        }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int q = 0; q < D * D; ++q) {
        double v = s[q];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (lane == 0) red[w][q] = v;
    }
    __syncthreads();
    const int t = threadIdx.x;
    if (t >= kGreenW * kGreenW) return;
    const int dx = abs(t % kGreenW - kGreenR), dy = abs(t / kGreenW - kGreenR);
    double v = 0.0;
    for (int q = 0; q < NW; ++q) v += red[q][dy * D + dx];
    // (c0: the charge on the node over eps0 dx, over the nx ny modes)
    blk[((size_t)blockIdx.x * kGreenW + blockIdx.y) * (kGreenW * kGreenW) + t] = v * c0;
}

__device__ __forceinline__ int wrap_off(int d, int n)
{
    if (2 * d > n) d -= n;
    if (2 * d < -n) d += n;
    return d;
}

// potential of grain gi's unit charge at node (i, j, k) (i, j already wrapped)
__device__ double sup_phi(const Geo& g, const double* blk, const int* plane, const int c[3], const long long w[3][2],
                          int i, int j, int k)
{
    double s = 0.0;
#pragma unroll
    for (int dz = 0; dz < 2; ++dz)
#pragma unroll
        for (int dy = 0; dy < 2; ++dy)
#pragma unroll
            for (int di = 0; di < 2; ++di) {
                const int ci = (c[0] + di) % g.nx, cj = (c[1] + dy) % g.ny, ck = c[2] + dz;
                const int ox = wrap_off(i - ci, g.nx), oy = wrap_off(j - cj, g.ny), oz = k - ck;
                const double wt = (double)(w[0][di] * w[1][dy] * w[2][dz]) * 0x1p-42;
                const double* b = blk + (size_t)plane[ck] * (kGreenW * kGreenW * kGreenW);
                s = s + wt * b[((oz + kGreenR) * kGreenW + (oy + kGreenR)) * kGreenW + (ox + kGreenR)];
            }
    return s;
}

__global__ void k_grain_table_sup(Geo g, const double* gpos, const int* gcell, const double* blk, const int* plane,
                                  double* tab)
{
    const int gi = blockIdx.x, t = threadIdx.x;
    if (t >= 64) return;
    const double x[3] = {gpos[3 * gi], gpos[3 * gi + 1], gpos[3 * gi + 2]};
    int c[3];
    double f[3];
    locate(g, x, c, f);
    const Cic cic(f);
    const long long w[3][2] = {{kWQ - cic.a[0], cic.a[0]}, {kWQ - cic.a[1], cic.a[1]}, {kWQ - cic.a[2], cic.a[2]}};
    const int nx = g.nx, ny = g.ny, nz = g.nz;
    const int li = t % 4, lj = (t / 4) % 4, lk = t / 16;
    const int i = ((gcell[3 * gi] - 1 + li) % nx + nx) % nx;
    const int j = ((gcell[3 * gi + 1] - 1 + lj) % ny + ny) % ny;
    const int k = gcell[3 * gi + 2] - 1 + lk;
    const double h2 = 2.0 * g.dx;
    auto ph = [&](int a, int b, int z) { return sup_phi(g, blk, plane, c, w, a, b, z); };
    double* o = tab + ((size_t)gi * 64 + t) * 3;
    o[0] = (ph((i + nx - 1) % nx, j, k) - ph((i + 1) % nx, j, k)) / h2;
    o[1] = (ph(i, (j + ny - 1) % ny, k) - ph(i, (j + 1) % ny, k)) / h2;
    if (k == 0)
        o[2] = ((3.0 * ph(i, j, k) - 4.0 * ph(i, j, k + 1)) + ph(i, j, k + 2)) / h2;
    else if (k == nz)
        o[2] = ((4.0 * ph(i, j, k - 1) - 3.0 * ph(i, j, k)) - ph(i, j, k - 2)) / h2;
    else
        o[2] = (ph(i, j, k - 1) - ph(i, j, k + 1)) / h2;
}

// node moments: CIC sums of 1 and v per species (double atomics), into the
// slice of the sample's rf phase bin
__global__ void k_moments64(Geo g, const double4* pos, const double4* vel, const unsigned long long* nslot, int sp,
                            double* mom, double* mke, const int* bin, size_t nodes)
{
    const unsigned long long n = nslot[sp];
    mom += (size_t)*bin * 4 * nodes;
    mke += (size_t)*bin * nodes;
    for (unsigned long long q = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; q < n;
         q += (unsigned long long)gridDim.x * blockDim.x) {
        const double4 P = pos[q];
        if (P.w < 0.0) continue;
        const double4 V = vel[q];
        const double v2 = (V.x * V.x + V.y * V.y) + V.z * V.z;
        const double x[3] = {P.x, P.y, P.z};
        int c[3];
        double f[3];
        locate(g, x, c, f);
        const Cic w(f);
        for (int dz = 0; dz < 2; ++dz)
            for (int dy = 0; dy < 2; ++dy)
                for (int di = 0; di < 2; ++di) {
                    const double wt = w.w[0][di] * (w.w[1][dy] * w.w[2][dz]);
                    if (wt == 0.0) continue;
                    const size_t node = corner(g, c, di, dy, dz);
                    double* m = mom + 4 * node;
                    atomicAdd(m, wt);
                    atomicAdd(m + 1, wt * V.x);
                    atomicAdd(m + 2, wt * V.y);
                    atomicAdd(m + 3, wt * V.z);
                    atomicAdd(mke + node, wt * v2);
                }
    }
}

// (the reciprocal's corrections keep clear of under- and overflow in this range of dx)
Geo geo(const pic_ctx* c)
{
    Geo g{c->nx, c->ny, c->nz, c->dx, c->Lx, c->Ly, c->Lz, 0.0, 0ull, 0};
    if (c->dx > 1e-100 && c->dx < 1e100) {
        g.rdx = 1.0 / c->dx;
        // dx = D 2^(e - 53), 2^52 <= D < 2^53: 1 / dx = (2^116 / D) 2^(-63 - e)
        int e = 0;
        const unsigned long long D = (unsigned long long)std::ldexp(std::frexp(c->dx, &e), 53);
        if (D == 1ull << 52) --e;
        g.fix_c = D == 1ull << 52 ? 1ull << 63 : (unsigned long long)((((unsigned __int128)1) << 116) / D);
        g.fix_e = e;
        if (c->nx >= 65536 || c->ny >= 65536 || c->nz >= 65536) g.fix_c = 0ull;
    }
    return g;
}


// Initial plasma drawn from the run's seed, the same definition the oracle
// states: particle id p takes three uniforms at a time from its stream (p,
// step 0, kPurInitPos) for a point u L until it lies farther than 1.5 radii
// from every grain (minimum image in x and y; at most 64 tries, else the last
// point), and three normals from (p, 0, kPurInitVel) times sqrt(T e / m).
// Only the grains listed for the point's cell are tested: a point within
// 1.5 r < dx of a grain lies in the grain's 3x3x3 region, whose cells list it.
// The FP64 result is converted to the mixed layout exactly as the host upload
// converts host arrays.
struct InitP {
    Geo g;
    uint2 key;
    int64_t n;
    uint32_t id0;
    double vth, vs;              // thermal speed (m/s); dt/dx (mixed velocities in cells/step)
    const int* cell_ng;
    const int* cell_g;
    const double* gpos;
    const double* grad;
    double4* pos64;
    double4* vel64;
    float4* pos32;
    float4* vel32;
};

__device__ bool near_grain(const InitP& p, const double x[3])
{
    int c[3];
    double f[3];
    locate(p.g, x, c, f);
    const int cell = cell_of(p.g, c);
    const int ng = p.cell_ng[cell];
    const double L[3] = {p.g.Lx, p.g.Ly, p.g.Lz};
    for (int t = 0; t < ng; ++t) {
        const int gi = p.cell_g[cell * kMaxG + t];
        double d[3];
        for (int a = 0; a < 3; ++a) {
            d[a] = x[a] - p.gpos[3 * gi + a];
            if (a < 2 && d[a] > 0.5 * L[a]) d[a] = d[a] - L[a];
            else if (a < 2 && d[a] < -0.5 * L[a]) d[a] = d[a] + L[a];
        }
        const double rx = 1.5 * p.grad[gi];
        if (((d[0] * d[0] + d[1] * d[1]) + d[2] * d[2]) <= rx * rx) return true;
    }
    return false;
}

__global__ void k_init_plasma(const InitP p)
{
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < p.n; q += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t id = p.id0 + (uint32_t)q;
        const double L[3] = {p.g.Lx, p.g.Ly, p.g.Lz};
        double x[3];
        RStream rp(id, 0u, kPurInitPos, p.key);
        for (int t = 0; t < 64; ++t) {
            for (int a = 0; a < 3; ++a) x[a] = u01d(rp.next()) * L[a];
            if (!near_grain(p, x)) break;
        }
        double nv[3], v[3];
        RStream rv(id, 0u, kPurInitVel, p.key);
        gauss3(rv, nv);
        for (int a = 0; a < 3; ++a) v[a] = p.vth * nv[a];
        int c[3];
        double f[3];
        locate(p.g, x, c, f);
        if (p.pos64) {
            p.pos64[q] = make_double4(x[0], x[1], x[2], (double)cell_of(p.g, c));
            p.vel64[q] = make_double4(v[0], v[1], v[2], (double)id);
        } else {
            float o[3];
            for (int a = 0; a < 3; ++a) o[a] = fminf((float)f[a], 0.99999994f);
            const int cell = c[0] | (c[1] << 10) | (c[2] << 20);
            p.pos32[q] = make_float4(o[0], o[1], o[2], __int_as_float(cell));
            p.vel32[q] = make_float4((float)(v[0] * p.vs), (float)(v[1] * p.vs), (float)(v[2] * p.vs),
                                     __uint_as_float(id));
        }
    }
}

// Caller-supplied particles (x, v in SI as 3 doubles each, uint32 ids) into the
// run's records, particle q of the arrays to slot q0 + q: the same conversion
// as k_init_plasma's (cell and in-cell offset by `locate`; mixed velocities in
// cells per step), checked as pic_init requires (finite, 0 <= x < Lx,
// 0 <= y < Ly, 0 <= z <= Lz); a bad particle sets *bad.  *max_id takes the
// largest id.  The arrays may be host memory the device reads directly.
struct StageP {
    Geo g;
    double vs;
    const double* x;
    const double* v;
    const uint32_t* id;
    int64_t n, q0;
    double4* pos64;
    double4* vel64;
    float4* pos32;
    float4* vel32;
    unsigned int* bad;
    unsigned int* max_id;
};

__global__ void k_stage_particles(const StageP p)
{
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < p.n; q += (int64_t)gridDim.x * blockDim.x) {
        const double x[3] = {p.x[3 * q], p.x[3 * q + 1], p.x[3 * q + 2]};
        const double v[3] = {p.v[3 * q], p.v[3 * q + 1], p.v[3 * q + 2]};
        const uint32_t id = p.id[q];
        atomicMax(p.max_id, id);
        bool ok = true;
        for (int a = 0; a < 3; ++a) ok = ok && isfinite(x[a]) && isfinite(v[a]);
        ok = ok && x[0] >= 0.0 && x[0] < p.g.Lx && x[1] >= 0.0 && x[1] < p.g.Ly && x[2] >= 0.0 && x[2] <= p.g.Lz;
        if (!ok) {
            atomicOr(p.bad, 1u);
            continue;
        }
        int c[3];
        double f[3];
        locate(p.g, x, c, f);
        const int64_t d = p.q0 + q;
        if (p.pos64) {
            p.pos64[d] = make_double4(x[0], x[1], x[2], (double)cell_of(p.g, c));
            p.vel64[d] = make_double4(v[0], v[1], v[2], (double)id);
        } else {
            float o[3];
            for (int a = 0; a < 3; ++a) o[a] = fminf((float)f[a], 0.99999994f);
            const int cell = c[0] | (c[1] << 10) | (c[2] << 20);
            p.pos32[d] = make_float4(o[0], o[1], o[2], __int_as_float(cell));
            p.vel32[d] = make_float4((float)(v[0] * p.vs), (float)(v[1] * p.vs), (float)(v[2] * p.vs),
                                     __uint_as_float(id));
        }
    }
}
}  // namespace

void launch_stage_particles(pic_ctx* c, int sp, const double* x, const double* v, const uint32_t* id, int64_t n,
                            int64_t q0, unsigned int* bad, unsigned int* max_id)
{
    if (n <= 0) return;
    StageP p;
    p.g = geo(c);
    p.vs = c->dt / c->dx;
    p.x = x;
    p.v = v;
    p.id = id;
    p.n = n;
    p.q0 = q0;
    const bool mixed = c->prec == PIC_MIXED;
    p.pos64 = mixed ? nullptr : (double4*)c->pos[sp];
    p.vel64 = mixed ? nullptr : (double4*)c->vel[sp];
    p.pos32 = mixed ? (float4*)c->pos[sp] : nullptr;
    p.vel32 = mixed ? (float4*)c->vel[sp] : nullptr;
    p.bad = bad;
    p.max_id = max_id;
    k_stage_particles<<<grid_for(n, 256, 152 * 16), 256, 0, c->stream>>>(p);
    c->launches += 1;
}

void launch_push64(pic_ctx* c)
{
    P64 ps[2];
    for (int sp = 0; sp < 2; ++sp) {
        P64& p = ps[sp];
        p.g = geo(c);
        p.Lx = c->Lx; p.Ly = c->Ly;
        p.M = c->md_sub > 0 ? c->md_sub : 1;
        p.dt = c->dt;
        p.dtm = c->dt / (double)p.M;
        p.sp = sp;
        p.qmdt = (c->qm[sp] * c->dt) * 0x1p-42;   // for gather_scaled
        p.qmdtm = c->qm[sp] * p.dtm;
        p.hm = c->hm[sp];
        const double below = std::ceil(c->pnull[sp] * 0x1p32 - 0.5);   // u + 1/2 < pnull 2^32
        p.null_below = below > 0.0 ? (unsigned long long)below : 0ull;
        p.mcc_list = (unsigned int*)c->pos_alt[sp];   // (the sort's other buffers are free between sorts)
        p.mcc_n = c->d_lists + 2 * sp + 1;
        p.nu_max = c->nu_max[sp];
        p.de = c->de[sp];
        p.n_gas = c->n_gas;
        p.sig_n = c->sig_n;
        p.eps_exc = c->eps_exc;
        p.eps_ion = c->eps_ion;
        p.mr2 = (2.0 * kME) / kMAR;
        p.kc = 1.0 / (4.0 * kPI * kEPS0);
        p.n_xs = c->n_xs;
        p.xs = c->xs64;
        p.key = c->key;
        p.step = c->d_step;
        p.flags = c->flags;
        p.ng = c->ng;
        p.gpos = c->gpos; p.grad = c->grad; p.gcell = c->gcell; p.gq = c->gq; p.gtab = c->gtab; p.gabs = c->gabs;
        p.cell_ng = c->cell_ng; p.cell_g = c->cell_g;
        p.ex = c->e64; p.ey = c->e64 + c->nodes; p.ez = c->e64 + 2 * c->nodes;
        p.rq = c->rq;
        p.pos = (double4*)c->pos[sp];
        p.vel = (double4*)c->vel[sp];
        p.nslot = c->d_nslot;
        p.cnt = c->d_cnt;
        p.err = c->d_err;
        p.child = c->d_child;
        p.child_cap = (unsigned long long)c->child_cap;
        p.nch = c->d_nch;
    }
    cudaMemsetAsync(c->d_lists, 0, 4 * sizeof(unsigned int), c->stream);
    const int64_t most = std::max(c->cap[0], c->cap[1]);
    k_push64<<<dim3((unsigned)grid_for(most, kPush64Threads, 152 * 16), 2), kPush64Threads, 0, c->stream>>>(ps[0], ps[1]);
    c->launches += 1;
    if (!(c->flags & PIC_F_NO_MCC)) {
        k_mcc64<<<dim3(152 * 4, 2), kPush64Threads, 0, c->stream>>>(ps[0], ps[1]);
        c->launches += 1;
    }
}

void launch_children64(pic_ctx* c)
{
    k_children64<<<64, 256, 0, c->stream>>>(geo(c), c->d_child, c->d_nch, (unsigned long long)c->child_cap,
                                              c->d_nslot, c->d_next_id,
                                              (double4*)c->pos[0], (double4*)c->vel[0], (double4*)c->pos[1],
                                              (double4*)c->vel[1], c->cap[0], c->cap[1], c->rq, c->d_err);
    k_children_finish<<<1, 1, 0, c->stream>>>(c->d_nch, (unsigned long long)c->child_cap, c->d_nslot, c->d_next_id,
                                              c->cap[0], c->cap[1], c->d_step);
    c->launches += 2;
}

void launch_deposit64(pic_ctx* c)
{
    for (int sp = 0; sp < 2; ++sp)
        k_deposit64<<<grid_for(c->cap[sp], 256, 152 * 8), 256, 0, c->stream>>>(geo(c), (const double4*)c->pos[sp],
                                                                               c->d_nslot, sp, c->rq);
    c->launches += 2;
}

void launch_efield64(pic_ctx* c)
{
    k_efield64<<<grid_for((int64_t)c->nodes, 256, 152 * 8), 256, 0, c->stream>>>(c->nx, c->ny, c->nz, c->dx, c->phi,
                                                                                c->e64, c->e64 + c->nodes,
                                                                                c->e64 + 2 * c->nodes);
    c->launches += 1;
}

void launch_moments64(pic_ctx* c)
{
    for (int sp = 0; sp < 2; ++sp)
        k_moments64<<<grid_for(c->cap[sp], 256, 152 * 8), 256, 0, c->stream>>>(
            geo(c), (const double4*)c->pos[sp], (const double4*)c->vel[sp], c->d_nslot, sp, c->mom[sp], c->mke[sp],
            c->d_bin, c->nodes);
    c->launches += 2;
}

void launch_grains(pic_ctx* c)
{
    if (c->ng == 0) return;
    k_grains<<<(c->ng + 63) / 64, 64, 0, c->stream>>>(geo(c), c->ng, kQE * c->W, c->gabs, c->gpos, c->gq, c->gq32,
                                                     c->rq);
    c->launches += 1;
}

cudaError_t launch_cell_lists(pic_ctx* c)
{
    cudaError_t e = cudaMemsetAsync(c->cell_ng, 0, sizeof(int) * c->cells, c->stream);
    if (e != cudaSuccess || c->ng == 0) return e;
    const unsigned grid = (unsigned)((27 * (int64_t)c->ng + 127) / 128);
    k_cell_claim<<<grid, 128, 0, c->stream>>>(c->ng, c->nx, c->ny, c->gcell, c->cell_ng, c->cell_g);
    k_cell_order<<<grid, 128, 0, c->stream>>>(c->ng, c->nx, c->ny, c->gcell, c->cell_ng, c->cell_g);
    c->launches += 2;
    return cudaGetLastError();
}

void launch_green_blocks(pic_ctx* c, const int* planes, int n, double* blk)
{
    if (n == 0) return;
    k_green_block<<<dim3((unsigned)n, kGreenW), kGreenThreads, 0, c->stream>>>(
        c->nx, c->ny, c->nz, 1.0 / (kEPS0 * c->dx) / ((double)c->nx * (double)c->ny), planes, blk);
    c->launches += 1;
}

void launch_grain_tables_sup(pic_ctx* c, const double* blk, const int* plane)
{
    if (c->ng == 0) return;
    k_grain_table_sup<<<c->ng, 64, 0, c->stream>>>(geo(c), c->gpos, c->gcell, blk, plane, c->gtab);
    c->launches += 1;
}

void launch_init_plasma(pic_ctx* c, int sp, int64_t n, uint32_t id0, double t_ev)
{
    if (n <= 0) return;
    InitP p;
    p.g = geo(c);
    p.key = c->key;
    p.n = n;
    p.id0 = id0;
    p.vth = sqrt((t_ev * kQE) / (sp == 0 ? kME : kMAR));
    p.vs = c->dt / c->dx;
    p.cell_ng = c->cell_ng;
    p.cell_g = c->cell_g;
    p.gpos = c->gpos;
    p.grad = c->grad;
    const bool mixed = c->prec == PIC_MIXED;
    p.pos64 = mixed ? nullptr : (double4*)c->pos[sp];
    p.vel64 = mixed ? nullptr : (double4*)c->vel[sp];
    p.pos32 = mixed ? (float4*)c->pos[sp] : nullptr;
    p.vel32 = mixed ? (float4*)c->vel[sp] : nullptr;
    k_init_plasma<<<grid_for(n, 256, 152 * 16), 256, 0, c->stream>>>(p);
    c->launches += 1;
}

}  // namespace pic
