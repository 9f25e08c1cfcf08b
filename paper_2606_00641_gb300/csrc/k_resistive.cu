// k_resistive.cu -- resistive incompressible MHD channel: D3Q19 flow lattice
// plus three D3Q7 magnetic lattices, FP32, one fused kernel per step.
//
// Model (sec. 2.3 "Incompressible resistive MHD", read with a standard
// second-order flow equilibrium; sec. 2.4 "Static boundaries"):
//   rho = sum f_i,  m = sum f_i c_i + F/2,  u = m / rho,  B_b = sum_i g_bi
//   f_eq_i = w_i [rho + c_i.m/cs2 + (c_i c_i - cs2 I):(rho u u + |B|^2/2 I - B B)/(2 cs2^2)]
//   f*_i   = f_i + omega_f (f_eq_i - f_i)
//            + (1 - omega_f/2) w_i [(c_i - u)/cs2 + (c_i.u) c_i/cs2^2] . F    (Guo)
//   g_eq_bi = w_i (B_b + c_i . Phi_b / cs2_7),  Phi_{b,a} = u_a B_b - B_a u_b  (Eq. 3, 12)
//   g*_bi  = g_bi + omega_m (g_eq_bi - g_bi)
// Walls (rows y = 0 and ny - 1 when walls_y): halfway bounce-back for f;
// wall cells emit g*_bi = w_i b_wall_b (equilibrium of the applied field at
// rest) for the magnetic lattices.
//
// Slots: flow directions j = 0..18, then magnetic lattice b direction i at
// j = 19 + 7 b + i.  AA in-place pattern as in vlbm_internal.cuh; with walls,
// a flow population whose source (odd parity read) or destination (odd
// parity write) is a wall cell is taken from / put into the cell's own slot
// of the same direction -- the halfway bounce-back in AA form.
#include "vlbm_internal.cuh"

#include "split_f32.cuh"

namespace vlbm {
namespace {

constexpr int kQf = 19;
constexpr int kSlots = 19 + 21;

// D3Q19 velocities in the ABI order: i = 2 p - 1 and 2 p are opposite (opp_axis).
__host__ __device__ constexpr int cx19(int i)
{
    return (i == 1 || i == 7 || i == 9 || i == 11 || i == 13) ? 1
           : (i == 2 || i == 8 || i == 10 || i == 12 || i == 14) ? -1
                                                                  : 0;
}
__host__ __device__ constexpr int cy19(int i)
{
    return (i == 3 || i == 7 || i == 10 || i == 15 || i == 17) ? 1
           : (i == 4 || i == 8 || i == 9 || i == 16 || i == 18) ? -1
                                                                 : 0;
}
__host__ __device__ constexpr int cz19(int i)
{
    return (i == 5 || i == 11 || i == 14 || i == 15 || i == 18) ? 1
           : (i == 6 || i == 12 || i == 13 || i == 16 || i == 17) ? -1
                                                                   : 0;
}
__host__ __device__ constexpr float w19(int i) { return i == 0 ? 1.0f / 3.0f : (i <= 6 ? 1.0f / 18.0f : 1.0f / 36.0f); }

struct Args {
    float *pop;
    int nx, ny, nz;
    int64_t stride;
    float omega_f, omega_m;
    float F[3];
    float guo;             // 1 - omega_f / 2
    float bw[3];           // wall field
    int walls_y;
    unsigned *flags;
    FastDiv by_nx;
    bool next_early;       // the chained step after this one is let in at once
};

// Offsets of x + c (periodic) from x along each axis, for c = -1, 0, +1.
struct Offsets {
    int64_t ox[3], oy[3], oz[3];
};

__device__ __forceinline__ Offsets offsets(int x, int y, int z, int nx, int ny, int nz)
{
    Offsets o;
    const int64_t row = nx, plane = (int64_t)nx * ny, vol = plane * nz;
    o.ox[0] = x > 0 ? -1 : nx - 1;
    o.ox[1] = 0;
    o.ox[2] = x + 1 < nx ? 1 : 1 - nx;
    o.oy[0] = y > 0 ? -row : plane - row;
    o.oy[1] = 0;
    o.oy[2] = y + 1 < ny ? row : row - plane;
    o.oz[0] = z > 0 ? -plane : vol - plane;
    o.oz[1] = 0;
    o.oz[2] = z + 1 < nz ? plane : plane - vol;
    return o;
}

__device__ __forceinline__ int64_t nbr(const Offsets &o, int64_t cell, int cx, int cy, int cz)
{
    return cell + o.ox[cx + 1] + o.oy[cy + 1] + o.oz[cz + 1];
}

__device__ __forceinline__ bool wall_row(int y, int ny, int walls) { return walls && (y == 0 || y == ny - 1); }

template <bool ODD, bool PLANES>
__global__ void __launch_bounds__(kBlockX, 5) k_res_step(const Args a)
{
    int x, y, z;
    if (!step_cell<PLANES>(a.nx, a.ny, a.by_nx, x, y, z)) return;
    chain_wait();
    if (a.next_early) chain_next();
    const int64_t cell = x + (int64_t)a.nx * (y + (int64_t)a.ny * z);
    const Offsets o = offsets(x, y, z, a.nx, a.ny, a.nz);
    float *pop = a.pop;
    const int64_t S = a.stride;

    if (wall_row(y, a.ny, a.walls_y)) {
        // magnetic wall: emit the equilibrium of b_wall at rest
#pragma unroll
        for (int b = 0; b < 3; ++b)
#pragma unroll
            for (int i = 0; i < 7; ++i) {
                const float v = (i == 0 ? 0.25f : 0.125f) * a.bw[b];
                const int j = ODD ? i : opp_axis(i);
                const int64_t at = ODD ? nbr(o, cell, cx19(i), cy19(i), cz19(i)) : cell;
                pop[(int64_t)(19 + 7 * b + j) * S + at] = v;
            }
        return;
    }
    const bool wall_lo = a.walls_y && y == 1;            // y - 1 is a wall row
    const bool wall_hi = a.walls_y && y == a.ny - 2;     // y + 1 is a wall row

    // ---- load ----
    float f[kQf], g[3][7];
#pragma unroll
    for (int i = 0; i < kQf; ++i) {
        int64_t at;
        int j;
        if (!ODD) {
            j = i;
            at = cell;
        } else {
            // source x - c_i; a wall source means the population bounced back
            const bool from_wall = (cy19(i) > 0 && wall_lo) || (cy19(i) < 0 && wall_hi);
            j = from_wall ? i : opp_axis(i);
            at = from_wall ? cell : nbr(o, cell, -cx19(i), -cy19(i), -cz19(i));
        }
        f[i] = pop[(int64_t)j * S + at];
    }
#pragma unroll
    for (int b = 0; b < 3; ++b)
#pragma unroll
        for (int i = 0; i < 7; ++i) {
            const int j = ODD ? opp_axis(i) : i;
            const int64_t at = ODD ? nbr(o, cell, -cx19(i), -cy19(i), -cz19(i)) : cell;
            g[b][i] = pop[(int64_t)(19 + 7 * b + j) * S + at];
        }

    // ---- moments ----
    float rho = 0.f, jx = 0.f, jy = 0.f, jz = 0.f;
#pragma unroll
    for (int i = 0; i < kQf; ++i) {
        rho += f[i];
        if (cx19(i)) jx += cx19(i) * f[i];
        if (cy19(i)) jy += cy19(i) * f[i];
        if (cz19(i)) jz += cz19(i) * f[i];
    }
    const float m[3] = {jx + 0.5f * a.F[0], jy + 0.5f * a.F[1], jz + 0.5f * a.F[2]};
    const float ir = 1.0f / rho;
    const float u[3] = {m[0] * ir, m[1] * ir, m[2] * ir};
    float B[3];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        float s = g[b][0];
#pragma unroll
        for (int i = 1; i < 7; ++i) s += g[b][i];
        B[b] = s;
    }
    if (!(rho > 0.f)) atomicOr(a.flags, kFlagNonPhysical);
    const float B2 = B[0] * B[0] + B[1] * B[1] + B[2] * B[2];
    const float u2 = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
    const float uF = u[0] * a.F[0] + u[1] * a.F[1] + u[2] * a.F[2];

    // ---- flow collision (cs2 = 1/3) ----
    const float om = a.omega_f, omc = 1.f - om;
#pragma unroll
    for (int i = 0; i < kQf; ++i) {
        const float cu = cx19(i) * u[0] + cy19(i) * u[1] + cz19(i) * u[2];
        const float cm = cx19(i) * m[0] + cy19(i) * m[1] + cz19(i) * m[2];
        const float cB = cx19(i) * B[0] + cy19(i) * B[1] + cz19(i) * B[2];
        const float cF = cx19(i) * a.F[0] + cy19(i) * a.F[1] + cz19(i) * a.F[2];
        const float c2 = float(cx19(i) * cx19(i) + cy19(i) * cy19(i) + cz19(i) * cz19(i));
        // (c c - cs2 I) : (rho u u + B^2/2 I - B B)
        const float second = rho * (cu * cu - u2 * (1.f / 3.f)) + 0.5f * B2 * (c2 - 1.f) - (cB * cB - B2 * (1.f / 3.f));
        const float feq = w19(i) * (rho + 3.f * cm + 4.5f * second);
        const float force = a.guo * w19(i) * (3.f * (cF - uF) + 9.f * cu * cF);
        f[i] = omc * f[i] + om * feq + force;
    }
    // ---- magnetic collision (D3Q7, cs2 = 1/4, w_moving/cs2 = 1/2) ----
    const float omm = a.omega_m, ommc = 1.f - omm;
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        const float A0 = omm * 0.25f * B[b];
        const float A1 = omm * 0.125f * B[b];
        g[b][0] = ommc * g[b][0] + A0;
#pragma unroll
        for (int ax = 0; ax < 3; ++ax) {
            const float phi = (ax == b) ? 0.f : u[ax] * B[b] - B[ax] * u[b];
            const float bv = 0.5f * omm * phi;
            g[b][2 * ax + 1] = ommc * g[b][2 * ax + 1] + A1 + bv;
            g[b][2 * ax + 2] = ommc * g[b][2 * ax + 2] + A1 - bv;
        }
    }

    // ---- store ---- (addresses recomputed from an opaque stride, not held)
    const int64_t Ss = opaque(S);
#pragma unroll
    for (int i = 0; i < kQf; ++i) {
        int64_t at;
        int j;
        if (!ODD) {
            j = opp_axis(i);
            at = cell;
        } else {
            // destination x + c_i; a wall destination bounces back into the own slot
            const bool to_wall = (cy19(i) > 0 && wall_hi) || (cy19(i) < 0 && wall_lo);
            j = to_wall ? opp_axis(i) : i;
            at = to_wall ? cell : nbr(o, cell, cx19(i), cy19(i), cz19(i));
        }
        pop[(int64_t)j * Ss + at] = f[i];
    }
#pragma unroll
    for (int b = 0; b < 3; ++b)
#pragma unroll
        for (int i = 0; i < 7; ++i) {
            const int j = ODD ? i : opp_axis(i);
            const int64_t at = ODD ? nbr(o, cell, cx19(i), cy19(i), cz19(i)) : cell;
            pop[(int64_t)(19 + 7 * b + j) * Ss + at] = g[b][i];
        }
    chain_next();
}

// f = f_eq(rho, m - F/2, B), g = g_eq(B, u = m/rho) at parity 0: the FP64 expressions' values
// rounded to FP32 once.  Carried in split floats (split_f32.cuh): in FP64, with the velocities in
// a table, the pass took 4.22 ms at 128 x 128 x 256 for 0.13 ms worth of memory traffic; 0.53-0.54 ms
// so.  Opposite directions share the part even in c, w (rho + 4.5 (c c - cs2 I):(rho v v + ...)),
// and differ in the sign of the odd one, 3 w c.j.  Split floats keep some 42 bits of the largest
// term, so where a value lies that close to the middle of two floats (in one cell of some
// two thousand) the population is formed again in FP64, and each is the FP64 form's.
struct InitArgs {
    float *pop;
    int64_t stride, c0, count, qstride;
    double F[3];
};

// In FP64, the populations whose bits are set (flow, magnetic): all for states beyond the range in
// which split floats keep their digits, else the one or two next to a rounding boundary, for
// which nothing is formed that they do not need (the whole cell: 0.65 against 0.54 ms at
// 128 x 128 x 256, and 41 against 36 us at 46 x 19 x 24, where a pass is a wave or two).
__device__ __noinline__ void res_init_wide(const InitArgs &a, const double *__restrict__ Qin, int64_t t, float *out,
                                           uint32_t flow, uint32_t magnetic)
{
    const double rho = Qin[t];
    const double *m = Qin + a.qstride + t, *B = Qin + 4 * a.qstride + t;
    if (flow) {
        double j[3], v[3], b[3];
#pragma unroll
        for (int ax = 0; ax < 3; ++ax) {
            j[ax] = m[ax * a.qstride] - 0.5 * a.F[ax];
            v[ax] = j[ax] / rho;
            b[ax] = B[ax * a.qstride];
        }
        const double v2 = (v[0] * v[0] + v[1] * v[1] + v[2] * v[2]) / 3.0;
        const double B2 = b[0] * b[0] + b[1] * b[1] + b[2] * b[2];
        for (; flow; flow &= flow - 1u) {
            const int i = __ffs((int)flow) - 1;
            const int c[3] = {cx19(i), cy19(i), cz19(i)};
            double cv = 0.0, cj = 0.0, cB = 0.0;
#pragma unroll
            for (int ax = 0; ax < 3; ++ax)
                if (c[ax] != 0) {
                    cv += c[ax] > 0 ? v[ax] : -v[ax];
                    cj += c[ax] > 0 ? j[ax] : -j[ax];
                    cB += c[ax] > 0 ? b[ax] : -b[ax];
                }
            // B^2 (c^2 - 1) / 2 + B^2 / 3 for c^2 = 0, 1, 2
            const double even = i == 0 ? -1.0 / 6.0 : (i <= 6 ? 1.0 / 3.0 : 5.0 / 6.0);
            const double second = rho * (cv * cv - v2) + (even * B2 - cB * cB);
            const double w = i == 0 ? 1.0 / 3.0 : (i <= 6 ? 1.0 / 18.0 : 1.0 / 36.0);
            out[(int64_t)i * a.stride] = (float)(w * (rho + 3.0 * cj + 4.5 * second));
        }
    }
    for (; magnetic; magnetic &= magnetic - 1u) {
        const int i = __ffs((int)magnetic) - 1, k = i / 7, d = i % 7, ax = (d - 1) / 2;
        const double Bk = B[k * a.qstride];
        double cphi = 0.0;
        if (d > 0 && ax != k) {
            cphi = m[ax * a.qstride] / rho * Bk - B[ax * a.qstride] * (m[k * a.qstride] / rho);
            if (!(d & 1)) cphi = -cphi;
        }
        out[(int64_t)(kQf + i) * a.stride] = (float)((d == 0 ? 0.25 : 0.125) * (Bk + 4.0 * cphi));
    }
}

__global__ void __launch_bounds__(128) k_res_init(const InitArgs a, const double *__restrict__ Qin)
{
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= a.count) return;
    float *out = a.pop + a.c0 + t;
    {
        // rho in 2^-19 .. 2^19, components zero or 2^-99 .. 2^19 in size: on the upper words, as
        // each comparison in FP64 takes 16 cycles of an SM
        auto word = [](double x) { return (uint32_t)__double2hiint(x); };
        auto exponent = [](int e) { return (uint32_t)(1023 + e) << 20; };
        bool usual = word(Qin[t]) >= exponent(-19) && word(Qin[t]) < exponent(19);
#pragma unroll
        for (int k = 1; k < 7; ++k) {
            const uint32_t v = word(Qin[k * a.qstride + t]) & 0x7FFFFFFFu;
            usual = usual && v < exponent(19) && (v >= exponent(-99) || v == 0u);
        }
        if (!usual) {
            res_init_wide(a, Qin, t, out, (1u << kQf) - 1u, (1u << 21) - 1u);
            return;
        }
    }
    const Split rho = split(Qin[t]);
    Split j[3], B[3], u[3], v[3];
    const Split ir = reciprocal(rho);
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        const double m = Qin[(1 + ax) * a.qstride + t];
        B[ax] = split(Qin[(4 + ax) * a.qstride + t]);
        j[ax] = split(m - 0.5 * a.F[ax]);
        u[ax] = split(m) * ir;
        v[ax] = j[ax] * ir;
    }
    // Bounds of the errors below, u = 2^-24: a split input is off by u^2 of itself, a product by
    // 6 u^2, a sum by 3 u^2, the reciprocal by 6 u^2 (its Newton step leaves (2 u)^2); so rho (c.v)^2 by
    // 2^-42.9 of rho |v|_1^2, and a flow population by 2^-41.9 of w `most`; a magnetic one by 2^-43 of
    // its terms.  Taken as 2^-41 and 2^-42, which covers the FP64 form's own 2^-50 and these
    // sums' roundings too, and 2^-125 for what is lost below the normal floats (2^-149 a product,
    // times a component below 2^19).
    auto one_norm = [](const Split (&x)[3]) { return fabsf(x[0].hi) + fabsf(x[1].hi) + fabsf(x[2].hi); };
    const float sv = one_norm(v), sB = one_norm(B);
    const float most = rho.hi + 3.f * one_norm(j) + 6.1f * rho.hi * sv * sv + 8.3f * sB * sB;
    uint32_t flow = 0u, magnetic = 0u;  // populations to form again
    const Split third = {1.f / 3.f, (float)(1.0 / 3.0 - (double)(1.f / 3.f))};
    const Split B2 = B[0] * B[0] + B[1] * B[1] + B[2] * B[2];
    const Split v2 = v[0] * v[0] + v[1] * v[1] + v[2] * v[2];
    // (c c - cs2 I) : (rho v v + B^2/2 I - B B) = rho (c.v)^2 - (c.B)^2 + (c^2 - 1) B^2/2 + base
    const Split base = (B2 - rho * v2) * third;
    const Split four_half = {4.5f, 0.f}, three = {3.f, 0.f}, halfs = {0.5f, 0.f};
    const Split hB2 = halfs * B2;
#pragma unroll
    for (int p = 0; p < 10; ++p) {  // the rest population, then the nine opposite pairs
        const int i = p == 0 ? 0 : 2 * p - 1;
        const double wd = i == 0 ? 1.0 / 3.0 : (i <= 6 ? 1.0 / 18.0 : 1.0 / 36.0);
        const Split w = {(float)wd, (float)(wd - (double)(float)wd)};
        auto along = [&](const Split (&x)[3]) {  // c_i . x, i a compile-time constant
            Split s = {0.f, 0.f};
            bool first = true;
            const int c[3] = {cx19(i), cy19(i), cz19(i)};
#pragma unroll
            for (int ax = 0; ax < 3; ++ax)
                if (c[ax] != 0) {
                    const Split y = c[ax] > 0 ? x[ax] : -x[ax];
                    s = first ? y : s + y;
                    first = false;
                }
            return s;
        };
        const float off = 0x1p-41f * w.hi * most;
        if (p == 0) {
            const Split f = w * (rho + four_half * (base - hB2));
            out[0] = f.hi;
            if (!rounds_surely(f, off)) flow |= 1u;
            continue;
        }
        const Split cv = along(v), cB = along(B);
        Split second = base + rho * (cv * cv) - cB * cB;
        if (i > 6) second = second + hB2;
        const Split even = w * (rho + four_half * second), odd = w * (three * along(j));
        const Split plus = even + odd, minus = even - odd;
        out[(int64_t)i * a.stride] = plus.hi;
        out[(int64_t)(i + 1) * a.stride] = minus.hi;
        if (!rounds_surely(plus, off)) flow |= 1u << i;
        if (!rounds_surely(minus, off)) flow |= 2u << i;
    }
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        float *g = out + (int64_t)(kQf + 7 * b) * a.stride;
        g[0] = 0.25f * B[b].hi;
        const Split w = {0.125f, 0.f}, B8 = w * B[b];
#pragma unroll
        for (int ax = 0; ax < 3; ++ax) {  // w (B +- 4 (u_a B_b - B_a u_b)), zero for a = b
            Split s = {0.f, 0.f};
            if (ax != b) s = halfs * (u[ax] * B[b] - B[ax] * u[b]);
            const Split plus = B8 + s, minus = B8 - s;
            g[(int64_t)(2 * ax + 1) * a.stride] = plus.hi;
            g[(int64_t)(2 * ax + 2) * a.stride] = minus.hi;
            if (ax == b) continue;  // B / 8 itself, rounded once by the split
            const float terms = fabsf(B8.hi) + 0.5f * (fabsf(u[ax].hi * B[b].hi) + fabsf(B[ax].hi * u[b].hi));
            const float off = terms > 0.f ? fmaf(0x1p-42f, terms, 0x1p-125f) : 0.f;
            if (!rounds_surely(plus, off)) magnetic |= 1u << (7 * b + 2 * ax + 1);
            if (!rounds_surely(minus, off)) magnetic |= 2u << (7 * b + 2 * ax + 1);
        }
    }
    if ((flow | magnetic) != 0u) res_init_wide(a, Qin, t, out, flow, magnetic);
}

struct ReadArgs {
    const float *pop;
    int nx, ny, nz;
    int64_t stride;
    int parity;
    int walls_y;
    double F[3], bw[3];
};

__device__ __forceinline__ void cell_xyz(int64_t cell, int nx, int ny, int &x, int &y, int &z)
{
    x = (int)(cell % nx);
    const int64_t r = cell / nx;
    y = (int)(r % ny);
    z = (int)(r / ny);
}

// logical pre-collision population of slot j (0..39) at a fluid cell
__device__ double res_logical(const ReadArgs &a, int64_t cell, int x, int y, int z, int jslot)
{
    const Offsets o = offsets(x, y, z, a.nx, a.ny, a.nz);
    const bool wall_lo = a.walls_y && y == 1, wall_hi = a.walls_y && y == a.ny - 2;
    if (jslot < kQf) {
        const int i = jslot;
        if (!a.parity) return a.pop[(int64_t)i * a.stride + cell];
        const bool from_wall = (cy19(i) > 0 && wall_lo) || (cy19(i) < 0 && wall_hi);
        if (from_wall) return a.pop[(int64_t)i * a.stride + cell];
        return a.pop[(int64_t)opp_axis(i) * a.stride + nbr(o, cell, -cx19(i), -cy19(i), -cz19(i))];
    }
    const int b = (jslot - kQf) / 7, i = (jslot - kQf) % 7;
    if (!a.parity) return a.pop[(int64_t)(19 + 7 * b + i) * a.stride + cell];
    return a.pop[(int64_t)(19 + 7 * b + opp_axis(i)) * a.stride + nbr(o, cell, -cx19(i), -cy19(i), -cz19(i))];
}

// Moments of one cell in FP64 from its FP32 populations: sums carried in three floats
// (split_f32.cuh), the 40 conversions and 110 additions of the FP64 form on the slow
// FP64 pipe replaced (1.55 -> 0.29 ms a pass at 128 x 128 x 256, 0.13 ms of it memory
// traffic).  A sum that leaves the finite numbers is formed again in FP64.
template <bool ODD>
__device__ __forceinline__ void res_cell_moments(const ReadArgs &a, int64_t cell, double (&q)[7])
{
    int x, y, z;
    cell_xyz(cell, a.nx, a.ny, x, y, z);
    if (wall_row(y, a.ny, a.walls_y)) {
        q[0] = 1.0;
#pragma unroll
        for (int ax = 0; ax < 3; ++ax) {
            q[1 + ax] = 0.0;
            q[4 + ax] = a.bw[ax];
        }
        return;
    }
    const Offsets o = offsets(x, y, z, a.nx, a.ny, a.nz);
    const bool wall_lo = a.walls_y && y == 1, wall_hi = a.walls_y && y == a.ny - 2;
    auto flow = [&](int i) -> float {
        if (!ODD) return a.pop[(int64_t)i * a.stride + cell];
        const bool from_wall = (cy19(i) > 0 && wall_lo) || (cy19(i) < 0 && wall_hi);
        const int64_t at = from_wall ? cell : nbr(o, cell, -cx19(i), -cy19(i), -cz19(i));
        return a.pop[(int64_t)(from_wall ? i : opp_axis(i)) * a.stride + at];
    };
    auto magnetic = [&](int b, int i) -> float {
        if (!ODD) return a.pop[(int64_t)(kQf + 7 * b + i) * a.stride + cell];
        return a.pop[(int64_t)(kQf + 7 * b + opp_axis(i)) * a.stride + nbr(o, cell, -cx19(i), -cy19(i), -cz19(i))];
    };
    Sum3 s[7];
    float f[kQf];
#pragma unroll
    for (int i = 0; i < kQf; ++i) f[i] = flow(i);
#pragma unroll
    for (int i = 0; i < kQf; ++i) {
        s[0].add(f[i]);
        const int c[3] = {cx19(i), cy19(i), cz19(i)};
#pragma unroll
        for (int ax = 0; ax < 3; ++ax)
            if (c[ax] != 0) s[1 + ax].add(c[ax] > 0 ? f[i] : -f[i]);
    }
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        float g[7];
#pragma unroll
        for (int i = 0; i < 7; ++i) g[i] = magnetic(b, i);
#pragma unroll
        for (int i = 0; i < 7; ++i) s[4 + b].add(g[i]);
    }
    bool finite = true;
#pragma unroll
    for (int v = 0; v < 7; ++v) {
        finite = finite && s[v].finite();
        q[v] = s[v].value();
    }
    if (!finite) {
        double d[7] = {0, 0, 0, 0, 0, 0, 0};
#pragma unroll 1
        for (int i = 0; i < kQf; ++i) {
            const double v = res_logical(a, cell, x, y, z, i);
            d[0] += v;
            d[1] += cx19(i) * v;
            d[2] += cy19(i) * v;
            d[3] += cz19(i) * v;
        }
#pragma unroll 1
        for (int i = 0; i < 21; ++i) {
            const double v = res_logical(a, cell, x, y, z, kQf + i);
            if (i < 7) d[4] += v;
            else if (i < 14) d[5] += v;
            else d[6] += v;
        }
#pragma unroll
        for (int v = 0; v < 7; ++v) q[v] = d[v];
    }
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) q[1 + ax] += 0.5 * a.F[ax];
}

template <bool ODD>
__global__ void __launch_bounds__(128) k_res_moments(const ReadArgs a, int64_t c0, int64_t count, int64_t ostride,
                                                     double *__restrict__ out)
{
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= count) return;
    double q[7];
    res_cell_moments<ODD>(a, c0 + t, q);
#pragma unroll
    for (int v = 0; v < 7; ++v) out[v * ostride + t] = q[v];
}

__global__ void k_res_gather(const ReadArgs a, const int64_t *__restrict__ cells, int n, double *__restrict__ out)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    const int64_t cell = cells[t];
    int x, y, z;
    cell_xyz(cell, a.nx, a.ny, x, y, z);
    for (int j = 0; j < kSlots; ++j) out[(int64_t)t * kSlots + j] = res_logical(a, cell, x, y, z, j);
}

template <bool ODD>
__global__ void __launch_bounds__(kReduceThreads) k_res_partials(const ReadArgs a, int64_t ncell,
                                                                 double *partials, unsigned *ticket,
                                                                 double *__restrict__ sums)
{
    double acc[7] = {0, 0, 0, 0, 0, 0, 0};
    for (int64_t cell = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; cell < ncell;
         cell += (int64_t)gridDim.x * blockDim.x) {
        double q[7];
        res_cell_moments<ODD>(a, cell, q);
#pragma unroll
        for (int v = 0; v < 7; ++v) acc[v] += q[v];
    }
    domain_sums(acc, partials, ticket, sums);
}

Args make_args(vlbm_ctx *c)
{
    const Domain &d = c->dom[0];
    Args a{};
    a.pop = static_cast<float *>(c->pop);
    a.nx = d.nx;
    a.ny = d.ny;
    a.nz = d.nz;
    a.stride = d.stride;
    a.omega_f = (float)(1.0 / d.tau[0]);
    a.omega_m = (float)(1.0 / d.tau[1]);
    for (int ax = 0; ax < 3; ++ax) {
        a.F[ax] = (float)d.force[ax];
        a.bw[ax] = (float)d.b_wall[ax];
    }
    a.guo = (float)(1.0 - 0.5 / d.tau[0]);
    a.walls_y = d.walls_y;
    a.flags = c->d_flags;
    return a;
}

ReadArgs make_read(vlbm_ctx *c, int di)
{
    const Domain &d = c->dom[di];
    ReadArgs a{};
    a.pop = static_cast<const float *>(c->pop) + d.offset;
    a.nx = d.nx;
    a.ny = d.ny;
    a.nz = d.nz;
    a.stride = d.stride;
    a.parity = (int)(c->step & 1);
    a.walls_y = d.walls_y;
    for (int ax = 0; ax < 3; ++ax) {
        a.F[ax] = d.force[ax];
        a.bw[ax] = d.b_wall[ax];
    }
    return a;
}

}  // namespace

vlbm_status resistive_step(vlbm_ctx *c, int parity)
{
    const Domain &d = c->dom[0];
    Args a = make_args(c);
    const StepGrid g = step_grid(d.nx, d.ny, d.nz);
    a.by_nx = g.nx;
    // with at most one CTA per SM nothing can pile up, and the next step's set-up is hidden
    // behind all of this one: 32 CTAs 2.50 -> 2.18 us a step in a graph, 96: 2.72 -> 2.50, 128 the same
    a.next_early = (int64_t)g.grid.x * g.grid.y * g.grid.z <= c->sms;
    with_flags(parity != 0, g.planes, [&](auto odd, auto planes) {
        // chained: 2.81 -> 2.15 us a step in a graph at 32 CTAs, 3.96 -> 3.51 at 400, 7.00 -> 6.53 at 1024
        launch_step_kernel(c->chain, k_res_step<decltype(odd)::value, decltype(planes)::value>, g.grid, kBlockX,
                           c->stream, a);
    });
    c->launches++;
    return cuda_check(c, cudaGetLastError(), "resistive step launch");
}

vlbm_status resistive_init_range(vlbm_ctx *c, int di, const double *Q, int64_t c0, int64_t n, int64_t qstride)
{
    const Domain &d = c->dom[di];
    InitArgs a{};
    a.pop = static_cast<float *>(c->pop) + d.offset;
    a.stride = d.stride;
    a.c0 = c0;
    a.count = n;
    a.qstride = qstride;
    for (int ax = 0; ax < 3; ++ax) a.F[ax] = d.force[ax];
    k_res_init<<<(unsigned)((n + 127) / 128), 128, 0, c->stream>>>(a, Q);
    c->launches++;
    return cuda_check(c, cudaGetLastError(), "resistive init launch");
}

vlbm_status resistive_init(vlbm_ctx *c, int d, const double *Q_dev)
{
    const int64_t N = c->dom[d].ncell;
    return resistive_init_range(c, d, Q_dev, 0, N, N);
}

vlbm_status resistive_moments_range(vlbm_ctx *c, int di, double *out, int64_t c0, int64_t n, int64_t ostride)
{
    const ReadArgs a = make_read(c, di);
    const unsigned blocks = (unsigned)((n + 127) / 128);
    if (a.parity) k_res_moments<true><<<blocks, 128, 0, c->stream>>>(a, c0, n, ostride, out);
    else k_res_moments<false><<<blocks, 128, 0, c->stream>>>(a, c0, n, ostride, out);
    c->launches++;
    return cuda_check(c, cudaGetLastError(), "resistive moments launch");
}

vlbm_status resistive_moments(vlbm_ctx *c, int d, double *Q_dev)
{
    const int64_t N = c->dom[d].ncell;
    return resistive_moments_range(c, d, Q_dev, 0, N, N);
}

vlbm_status resistive_gather(vlbm_ctx *c, int di, const int64_t *cells_dev, int n, double *out_dev)
{
    k_res_gather<<<(unsigned)((n + 127) / 128), 128, 0, c->stream>>>(make_read(c, di), cells_dev, n, out_dev);
    c->launches++;
    return cuda_check(c, cudaGetLastError(), "resistive gather launch");
}

vlbm_status resistive_sums(vlbm_ctx *c, int di, double *sums_dev)
{
    const ReadArgs a = make_read(c, di);
    const int64_t ncell = c->dom[di].ncell;
    const int blocks = reduce_blocks(ncell);
    if (a.parity)
        k_res_partials<true><<<blocks, kReduceThreads, 0, c->stream>>>(a, ncell, c->d_partials, c->d_flags + 1, sums_dev);
    else
        k_res_partials<false><<<blocks, kReduceThreads, 0, c->stream>>>(a, ncell, c->d_partials, c->d_flags + 1, sums_dev);
    c->launches++;
    return cuda_check(c, cudaGetLastError(), "resistive sums launch");
}

}  // namespace vlbm
