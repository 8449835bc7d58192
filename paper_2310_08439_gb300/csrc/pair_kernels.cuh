// Pair kernels of the TensorMD evaluation (Sec. "The Tensor Formalism"):
//   k_desc          setup (D, R, Dhat), H_abck = f_k f_c, M_abcd,
//                   P_abkd = sum_c H M, G_abkm = sigma(T_dm P^2)
//                                        -- Eqs. tensor_formalism, sigma_function
//   k_force(_merged) P' = 2 T sigma' P G'; V = P' H and W = P' H' (so that
//                   F1 = U H' R' = W . M and F2 = V M' with M' formed on the
//                   fly); ScatterSum into forces, virial
//                                        -- Eqs. dP_abkd, U_abck, F1_abcx, F2_abcx
//
// The moments are kept in 16 components, not the 20 monomials of Eq. T_dm.  On
// the unit sphere the monomials of rank 2 and 3 repeat those of rank 0 and 1
// (xx + yy + zz = 1, xxx + xyy + xzz = x, ...), so the rank-m sum
// sum_d T_dm P_d^2, which is the double sum of (u_j . u_k)^m, splits into
// harmonics: (u.v)^2 = 1/3 + (5 terms of degree 2), (u.v)^3 = 3/5 u.v + (7
// terms of degree 3).  harmonics16 lists the polynomials, c_W their weights:
//   G_0 = |A_0|                     G_1 = sum_{1..3} A_c^2
//   G_2 = A_0^2 / 3 + sum_{4..8} w_c A_c^2
//   G_3 = 3/5 G_1 + sum_{9..15} w_c A_c^2
// (1/3, 3/5 and, in dE/dA, 2/3 as hi + lo: an error of such a constant is the
// same in every atom and adds up in the virial.)
// The sums are the same numbers with 16 instead of 20 multiply-adds per
// channel, pair and pass, and every term is a square with a positive weight.
//
// One warp owns one centre atom.  The in-cutoff pairs of each atom come from
// the pair cache (filled by k_screen in screen.cu, read by both passes) or,
// without a cache, from screening the table in the pass itself, compacted
// through a per-warp shared-memory queue; either way every lane works on an
// in-cutoff pair.  k_desc: the pairs' geometry is staged in shared memory and
// the sums run on the tensor cores.  k_force: a lane owns one or two pairs and
// reads the atom's P' from shared memory with broadcast loads.
//
// Templates over the radial channel count K and the species count S; each
// pair_k<K>.cu translation unit instantiates one K (compiled in parallel).
#pragma once

#include <algorithm>

#include "tmd_internal.cuh"

namespace tmd {

namespace {

constexpr int PW = PAIR_WARPS;   // warps per block in the pair kernels
constexpr float PI_F = 3.14159265358979323846f;

// weights w_c of the squared sums A_c, in the order of harmonics16
__constant__ float c_W[NHAR] = {1.f, 1.f, 1.f, 1.f, 2.f, 2.f, 2.f, 0.5f, 1.5f, 0.1f, 0.15f, 0.15f, 1.5f, 6.f, 0.25f, 0.25f};

// a x + b for a constant a of which FP32 holds a_hi and a_lo is the rest
#define FMA_HILO(a, x, b) fmaf((float)(a), x, fmaf((float)((a) - (double)(float)(a)), x, b))

__device__ __forceinline__ float2 bc2(float x) { return make_float2(x, x); }

// 1 | x y z | xy yz xz x^2-y^2 | z^2-1/3, z(5z^2-3) x(5z^2-1) y(5z^2-1) | z(x^2-y^2) xyz x(x^2-3y^2) y(3x^2-y^2)
// of two unit vectors (degrees 0; 1; 2; 3; packed FP32x2)
__device__ __forceinline__ void harmonics16(float2 x, float2 y, float2 z, float2 *Y) {
    const float2 xx = __fmul2_rn(x, x), yy = __fmul2_rn(y, y), zz = __fmul2_rn(z, z);
    const float2 d = __ffma2_rn(yy, bc2(-1.f), xx), q = __ffma2_rn(zz, bc2(5.f), bc2(-1.f));
    Y[0] = bc2(1.f);
    Y[1] = x; Y[2] = y; Y[3] = z;
    Y[4] = __fmul2_rn(x, y); Y[5] = __fmul2_rn(y, z); Y[6] = __fmul2_rn(x, z); Y[7] = d;
    Y[8] = __fadd2_rn(zz, bc2(-1.f / 3.f));
    Y[9] = __fmul2_rn(z, __fadd2_rn(q, bc2(-2.f))); Y[10] = __fmul2_rn(x, q); Y[11] = __fmul2_rn(y, q);
    Y[12] = __fmul2_rn(z, d); Y[13] = __fmul2_rn(Y[4], z);
    Y[14] = __fmul2_rn(x, __ffma2_rn(yy, bc2(-3.f), xx));
    Y[15] = __fmul2_rn(y, __ffma2_rn(xx, bc2(3.f), __fmul2_rn(yy, bc2(-1.f))));
}

// 2^x and 1/sqrt(x) from the special-function unit (PTX ex2.approx /
// rsqrt.approx, relative error about 2^-22; flush-to-zero: a result below
// 2^-126 becomes 0, and no argument here is subnormal)
__device__ __forceinline__ float ex2_ftz(float x) {
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float rsqrt_ftz(float x) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// sin(pi t) and cos(pi t) for |t| <= 1/2 from their Taylor series in
// y = pi t (|y| <= pi/2): the sine through y^13 and the cosine through y^12
// leave truncation errors of at most 7e-10 and 7e-9.
__device__ __forceinline__ void sincospi_half(float t, float &sn, float &cs) {
    const float y = PI_F * t, u = y * y;
    float p = 1.f / 6227020800.f;
    p = fmaf(p, u, -1.f / 39916800.f);
    p = fmaf(p, u, 1.f / 362880.f);
    p = fmaf(p, u, -1.f / 5040.f);
    p = fmaf(p, u, 1.f / 120.f);
    p = fmaf(p, u, -1.f / 6.f);
    sn = fmaf(y * u, p, y);
    float q = 1.f / 479001600.f;
    q = fmaf(q, u, -1.f / 3628800.f);
    q = fmaf(q, u, 1.f / 40320.f);
    q = fmaf(q, u, -1.f / 720.f);
    q = fmaf(q, u, 1.f / 24.f);
    q = fmaf(q, u, -0.5f);
    cs = fmaf(u, q, 1.f);
}

// f_c = (cos(pi r / rc) + 1) / 2 and df_c/dr for r < rc, through t = r / rc - 1/2:
// cos(pi r / rc) = -sin(pi t), sin(pi r / rc) = cos(pi t).
__device__ __forceinline__ void cutoff_fn(float r, float inv_rc, float &fc, float &dfc) {
    float sn, cs;
    sincospi_half(fmaf(r, inv_rc, -0.5f), sn, cs);
    fc = 0.5f - 0.5f * sn;
    dfc = -0.5f * PI_F * inv_rc * cs;
}

// H_k = f_k f_c (and dH_k/dr when DERIV) for r < rc, two channels at a time
// on packed FP32x2 arithmetic (fma/add/mul .f32x2 issue two FP32 operations as
// one instruction, each rounded as its scalar form).  The model's table holds
// (mu_hi, mu_lo, eta log2 e, 2 eta) per channel; r = r_hi + r_lo so that
// t = r - mu keeps ~FP64 accuracy (the Gaussians are steep: dlnH/dr = -2 eta t
// amplifies any rounding of r).  rad2 = the channel pairs of one species pair,
// two float4 per pair (k, k+1): (-mu_hi, -mu_hi', -mu_lo, -mu_lo') and
// (-eta log2 e, -eta' log2 e, -2 eta, -2 eta'), written by stage_rad2.
__device__ __forceinline__ void stage_rad2(float4 *dst, const float4 *src, int n) {
    for (int t = threadIdx.x; t < n / 2; t += blockDim.x) {
        const float4 a = src[2 * t], b = src[2 * t + 1];
        dst[2 * t] = make_float4(-a.x, -b.x, -a.y, -b.y);
        dst[2 * t + 1] = make_float4(-a.z, -b.z, -a.w, -b.w);
    }
}

struct Radial2 {
    float2 H, dH;
};

template <bool DERIV>
__device__ __forceinline__ Radial2 radial2(const float4 *rad2, int k, float2 rh2, float2 rl2, float2 fc2, float2 dfc2) {
    const float4 A = rad2[k], B = rad2[k + 1];   // channel pair k / 2
    const float2 t = __fadd2_rn(__fadd2_rn(rh2, make_float2(A.x, A.y)), __fadd2_rn(rl2, make_float2(A.z, A.w)));
    const float2 a = __fmul2_rn(__fmul2_rn(make_float2(B.x, B.y), t), t);
    const float2 f = make_float2(ex2_ftz(a.x), ex2_ftz(a.y));
    Radial2 o;
    o.H = __fmul2_rn(f, fc2);
    if (DERIV) o.dH = __fmul2_rn(f, __ffma2_rn(__fmul2_rn(make_float2(B.z, B.w), t), fc2, dfc2));
    return o;
}

// Tabulated radial basis (Sec. "The H_abck tensor and Batch Rational 1D
// Interpolation": H and H' read from a table with the cutoff folded in).
// Interval g = [g/scale, (g+1)/scale) holds, per k, the coefficients
// (c0, c1, c2, c3) of the cubic Hermite polynomial in t = r scale - g through
// H and H' at both ends; H = c0 + t (c1 + t (c2 + t c3)) and
// H' = scale (c1 + t (2 c2 + 3 t c3)).  scale is a power of two, so r_hi scale
// and its integer part are exact and t carries r_lo.  tab = the intervals of
// this species pair, [interval][k] float4.
struct TabCell {
    const float4 *c;   // this pair's interval: K float4
    float t, t3;       // t and 3 t
};

// interval number from its floating value (exact for 0 <= gf < 2^22); inside
// the table also where r is not a number (two atoms at one place)
__device__ __forceinline__ int tab_interval(float gf, int n) {
    return (int)min((unsigned)(__float_as_int(gf + 12582912.0f) - 0x4B400000), (unsigned)(n - 1));
}

__device__ __forceinline__ TabCell tab_cell(const float *tab, int K, int n, float scale, float r_hi, float r_lo) {
    const float x = r_hi * scale;
    const float gf = floorf(x);
    const int g = tab_interval(gf, n);
    TabCell c;
    c.c = reinterpret_cast<const float4 *>(tab) + (size_t)g * K;
    c.t = (x - gf) + r_lo * scale;
    c.t3 = 3.f * c.t;
    return c;
}

__device__ __forceinline__ void tab_eval(const TabCell &tc, int k, float scale, float &H, float &dH) {
    const float4 q = __ldg(tc.c + k);
    H = fmaf(tc.t, fmaf(tc.t, fmaf(tc.t, q.w, q.z), q.y), q.x);
    dH = scale * fmaf(tc.t, fmaf(tc.t3, q.w, 2.f * q.z), q.y);
}

// r = |D| as an unevaluated sum r_hi + r_lo from r^2 = r2_hi + r2_lo, and 1/r.
// r_hi = r2 y with y ~ 1/sqrt(r2_hi) (pairs never coincide, r2_hi >= ~1); r_lo is the Newton correction (exact
// residual by FMA), so r_hi + r_lo is accurate to ~1e-13 whatever the error of
// y; 1/r is y refined by one Newton step against r_hi + r_lo.
__device__ __forceinline__ void split_sqrt(float r2_hi, float r2_lo, float &r_hi, float &r_lo, float &ir) {
    const float y = rsqrt_ftz(r2_hi);
    r_hi = r2_hi * y;
    r_lo = (fmaf(-r_hi, r_hi, r2_hi) + r2_lo) * 0.5f * y;
    const float e = fmaf(-r_hi, y, 1.f) - r_lo * y;
    ir = fmaf(y, e, y);
}

// split_sqrt and f_c (cutoff_fn) of two pairs (packed FP32x2)
__device__ __forceinline__ void split_sqrt2(float2 r2h, float2 r2l, float2 &r_hi, float2 &r_lo, float2 &ir) {
    const float2 y = make_float2(rsqrt_ftz(r2h.x), rsqrt_ftz(r2h.y));
    r_hi = __fmul2_rn(r2h, y);
    const float2 nr = __fmul2_rn(r_hi, bc2(-1.f));
    r_lo = __fmul2_rn(__fadd2_rn(__ffma2_rn(nr, r_hi, r2h), r2l), __fmul2_rn(y, bc2(0.5f)));
    const float2 e = __ffma2_rn(__fmul2_rn(r_lo, bc2(-1.f)), y, __ffma2_rn(nr, y, bc2(1.f)));
    ir = __ffma2_rn(y, e, y);
}
__device__ __forceinline__ float2 cutoff2(float2 r, float inv_rc) {
    const float2 y = __fmul2_rn(bc2(PI_F), __ffma2_rn(r, bc2(inv_rc), bc2(-0.5f))), u = __fmul2_rn(y, y);
    float2 p = bc2(1.f / 6227020800.f);
    p = __ffma2_rn(p, u, bc2(-1.f / 39916800.f));
    p = __ffma2_rn(p, u, bc2(1.f / 362880.f));
    p = __ffma2_rn(p, u, bc2(-1.f / 5040.f));
    p = __ffma2_rn(p, u, bc2(1.f / 120.f));
    p = __ffma2_rn(p, u, bc2(-1.f / 6.f));
    return __ffma2_rn(__ffma2_rn(__fmul2_rn(y, u), p, y), bc2(-0.5f), bc2(0.5f));
}

// Double-float helpers: a value is carried as an unevaluated sum hi + lo of two
// floats.  two_sum is Knuth's error-free addition.
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e) {
    s = a + b;
    const float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}

// The box on the 2^-10 grid split: of the atom's system when batched
__device__ __forceinline__ void pair_box(const DevNlist &nl, int a, float (&Lh)[3], float (&Ll)[3]) {
    if (nl.sys_of) {
        const SysParams &q = nl.sp[nl.sys_of[a]];
#pragma unroll
        for (int x = 0; x < 3; ++x) { Lh[x] = q.Gh[x]; Ll[x] = q.Gl[x]; }
    } else {
#pragma unroll
        for (int x = 0; x < 3; ++x) { Lh[x] = nl.Lh[x]; Ll[x] = nl.Ll[x]; }
    }
}

// Pair geometry on the 2^-10 grid split (grid_split): every position and box
// length is hi + lo with hi a multiple of 2^-10 A and |lo| <= 2^-11 A.  Then
// D_hi = (x_j,hi - x_i,hi) + s L_hi is exact in FP32 (a multiple of 2^-10
// below 2^13 A in magnitude needs at most 23 significand bits; the box
// checks keep |s| L below 2^13), and D_lo = (x_j,lo - x_i,lo) + s L_lo is a
// small correction carried to ~1e-10 A.  |D|^2 is formed as an FP32 hi + lo
// pair from the exact squares of D_hi (FMA residuals, error-free sums) and the
// cross terms (2 D_hi + D_lo) D_lo, so r^2 keeps ~FP64 accuracy with no FP64
// instruction.  D itself is returned rounded to FP32.
__device__ __forceinline__ void pair_geom(const float4 jh, const float4 jl, const float4 ih, const float4 il,
                                          const char4 sh, const float (&Lh)[3], const float (&Ll)[3], float &dx,
                                          float &dy, float &dz, float &r2h, float &r2l) {
    // (float)s from the signed byte with one add and one subtract (|s| < 2^22)
    const float sx = __int_as_float(0x4B400000 + (int)sh.x) - 12582912.0f;
    const float sy = __int_as_float(0x4B400000 + (int)sh.y) - 12582912.0f;
    const float sz = __int_as_float(0x4B400000 + (int)sh.z) - 12582912.0f;
    const float hx = fmaf(sx, Lh[0], jh.x - ih.x), lx = fmaf(sx, Ll[0], jl.x - il.x);
    const float hy = fmaf(sy, Lh[1], jh.y - ih.y), ly = fmaf(sy, Ll[1], jl.y - il.y);
    const float hz = fmaf(sz, Lh[2], jh.z - ih.z), lz = fmaf(sz, Ll[2], jl.z - il.z);
    const float px = hx * hx, ex = fmaf(hx, hx, -px);
    const float py = hy * hy, ey = fmaf(hy, hy, -py);
    const float pz = hz * hz, ez = fmaf(hz, hz, -pz);
    float s1, e1, s2, e2;
    two_sum(px, py, s1, e1);
    two_sum(s1, pz, s2, e2);
    const float cross = fmaf(fmaf(2.f, hx, lx), lx, fmaf(fmaf(2.f, hy, ly), ly, fmaf(2.f, hz, lz) * lz));
    const float lo = ((ex + ey) + ez) + (e1 + e2) + cross;
    r2h = s2 + lo;
    r2l = lo - (r2h - s2);
    dx = hx + lx;
    dy = hy + ly;
    dz = hz + lz;
}

// Walk the entries [beg, end) of atom a, keep pairs with r^2 < rc^2 and hand
// them to f in batches of up to 32 (one per lane).  D = x_j + s L - x_i and r^2
// are formed in double-float FP32 arithmetic from hi/lo positions (no FP64
// instructions: on this GPU FP64 runs at a small fraction of the FP32 rate).
// The queue holds (Dx, Dy, Dz, j | b<<28) rounded to FP32 and r^2 as hi/lo.
// Used when there is no pair cache (k_screen in screen.cu fills the cache
// with the same pairs, in the same order, by the same arithmetic).
//
// f(q, q2, nb) takes the first nb pairs of the queue (nb = NB but for the
// atom's last batch).
template <int NB, typename F>
__device__ __forceinline__ void queue_pairs(const DevNlist &nl, int a, int64_t beg, int64_t end, float rc2h, float rc2l,
                                            float4 *q, float2 *q2, int lane, F &&f) {
    int qn = 0;
    const unsigned lt = (1u << lane) - 1u;
    const float4 ih = nl.ph[a], il = nl.pl[a];
    float Lh[3], Ll[3];
    pair_box(nl, a, Lh, Ll);
    int64_t base = beg;
    while (true) {
        while (qn < NB && base < end) {
            const int64_t c = base + lane;
            bool v = false;
            float4 e = make_float4(0.f, 0.f, 0.f, 0.f);
            float2 e2 = make_float2(0.f, 0.f);
            if (c < end) {
                const int j = nl.nbr[c];
                const char4 s = nl.shift[c];
                const float4 jh = nl.ph[j], jl = nl.pl[j];
                float dx, dy, dz, r2h, r2l;
                pair_geom(jh, jl, ih, il, s, Lh, Ll, dx, dy, dz, r2h, r2l);
                v = (r2h < rc2h) || (r2h == rc2h && r2l < rc2l);
                e = make_float4(dx, dy, dz, __uint_as_float((uint32_t)j | ((uint32_t)s.w << 28)));
                e2 = make_float2(r2h, r2l);
            }
            const unsigned m = __ballot_sync(0xffffffffu, v);
            if (v) {
                const int slot = qn + __popc(m & lt);
                q[slot] = e;
                q2[slot] = e2;
            }
            qn += __popc(m);
            base += 32;
        }
        if (qn == 0) break;
        // one call site: full batches while entries remain, then the tail
        const int nb = min(qn, NB);
        __syncwarp();
        f(q, q2, nb);
        __syncwarp();
        if (lane < qn - nb) {
            q[lane] = q[lane + NB];
            q2[lane] = q2[lane + NB];
        }
        __syncwarp();
        qn -= nb;
    }
}

// Two neighbouring pairs of a lane (pairs 2 lane and 2 lane + 1 of a batch of 64).
struct PairTwo {
    float4 e0, e1;
    float2 q0, q1;
};
// pairs i and i + 1 of the n >= 1 at p, p2 (the last pair again past the end)
__device__ __forceinline__ PairTwo load_two(const float4 *p, const float2 *p2, int i, int n) {
    const int i0 = min(i, n - 1), i1 = min(i + 1, n - 1);
    PairTwo t;
    t.e0 = p[i0];
    t.e1 = p[i1];
    t.q0 = p2[i0];
    t.q1 = p2[i1];
    return t;
}

// A warp's stream of pair-cache batches (64 pairs, two per lane) over its atoms
// p, p + total, ... (perm order), read one batch ahead.
struct PairStream {
    int a = -1, np = 0;          // current atom and its in-cutoff pair count
    int64_t pb = 0;
    int an = -1, npn = 0;        // next atom (segment start and count read one atom ahead)
    int64_t pbn = 0;
    int an2 = -1;                // the atom after next (perm entry read two atoms ahead)
    int ty = 0, tyn = 0;         // species of the current and the next atom (0 unless asked for)
    PairTwo pf;                  // the batch that is taken next

    __device__ __forceinline__ void load(const DevNlist &nl, int64_t at, int n, int lane) {
        if (n > 0) pf = load_two(nl.pq + at, nl.pq2 + at, 2 * lane, n);
    }
    __device__ __forceinline__ void start(const DevNlist &nl, const int32_t *types, int64_t p, int64_t total, int lane) {
        pf.e0 = pf.e1 = make_float4(1.f, 0.f, 0.f, 0.f);
        pf.q0 = pf.q1 = make_float2(1.f, 0.f);
        if (p < nl.n) {
            a = nl.perm[p];
            if (types) ty = types[a];
            pb = nl.beg[a];
            np = nl.npair[a];
            load(nl, pb, np, lane);
        }
        an = p + total < nl.n ? nl.perm[p + total] : -1;
    }
    // at the start of atom p: the next atom's segment, the perm entry after it
    __device__ __forceinline__ void atom_begins(const DevNlist &nl, const int32_t *types, int64_t p, int64_t total) {
        npn = 0;
        if (an >= 0) {
            if (types) tyn = types[an];
            pbn = nl.beg[an];
            npn = nl.npair[an];
        }
        an2 = p + 2 * total < nl.n ? nl.perm[p + 2 * total] : -1;
    }
    // the batch after the one starting at base: the atom's next batch, or the
    // next atom's first
    __device__ __forceinline__ void advance(const DevNlist &nl, int base, int lane) {
        if (base + 64 < np)
            load(nl, pb + base + 64, np - base - 64, lane);
        else
            load(nl, pbn, npn, lane);
    }
    __device__ __forceinline__ void atom_ends() {
        a = an;
        ty = tyn;
        pb = pbn;
        np = npn;
        an = an2;
    }
};

// G_m of one channel, m = g, from the sums A of the four lanes g = 0..3 that
// hold components 4g .. 4g + 3 of it (lane 0: degrees 0 and 1; lane 1: four of
// degree 2; lane 2: the fifth of degree 2 and three of degree 3; lane 3: four
// of degree 3).  m = 0 is |A_0| and not the root of its square, so that a
// channel's tiny sum (|A_0| < 1e-19, whose square underflows in FP32) is not
// read as 0.
__device__ __forceinline__ float desc_value(const float (&A)[4], const float (&Wg)[4], int g) {
    const float s0 = Wg[0] * A[0] * A[0];
    const float s13 = Wg[1] * A[1] * A[1] + Wg[2] * A[2] * A[2] + Wg[3] * A[3] * A[3];
    const int quad = (threadIdx.x & 31) & ~3;
    const float a00 = __shfl_sync(0xffffffffu, s0, quad);     // A_0^2
    const float one = __shfl_sync(0xffffffffu, s13, quad);    // G_1
    const float up = __shfl_up_sync(0xffffffffu, g == 1 ? s0 + s13 : s13, 1);
    const float val2 = FMA_HILO(1.0 / 3.0, a00, up + s0), val3 = FMA_HILO(0.6, one, up + (s0 + s13));
    return g == 0 ? fabsf(A[0]) : (g == 1 ? one : (g == 2 ? val2 : val3));
}

// ---------------------------------------------------------------------------
// descriptor forward: A and G per atom
// ---------------------------------------------------------------------------
__device__ __forceinline__ void split_tf32(float x, uint32_t &hi, uint32_t &lo) {
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(hi) : "f"(x));
    const float rest = x - __uint_as_float(hi);   // exact
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(lo) : "f"(rest));
}

// c += a b for one m16n8k8 tile (a: 16 x 8 row-major, b: 8 x 8, c: 16 x 8)
__device__ __forceinline__ void mma_tf32(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// c = a b for one m16n8k8 tile
__device__ __forceinline__ void mma_tf32_first(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%10, %10, %10, %10};"
        : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
}

// Two values as operands of a split product: x_h = x rounded to TF32 (11
// significant bits, ties away) and x_l = x - x_h (exact, 12 bits or fewer), of
// which the tensor cores read the TF32 part: half a unit of that is added, so
// that the last bit of x is rounded where it does not fit, not dropped.  Integer
// operations: the conversion cvt.rna.tf32 issues at the rate of the special
// functions and made it the bound of the descriptor pass.
struct Split2 {
    uint32_t h0, h1, l0, l1;
};

__device__ __forceinline__ Split2 split2(const float2 x) {
    Split2 o;
    o.h0 = (__float_as_uint(x.x) + 0x1000u) & 0xffffe000u;
    o.h1 = (__float_as_uint(x.y) + 0x1000u) & 0xffffe000u;
    const float2 r = __ffma2_rn(make_float2(__uint_as_float(o.h0), __uint_as_float(o.h1)), make_float2(-1.f, -1.f), x);
    o.l0 = __float_as_uint(r.x) + 0x1000u;
    o.l1 = __float_as_uint(r.y) + 0x1000u;
    return o;
}

// The contraction A[k][c] = sum_j H_jk Y_jc of one atom is a K x 16 product
// over its pairs, run on the tensor cores (mma.sync) 8 pairs at a time: rows =
// 16 channels, columns = the 16 components in two tiles of 8.  Every lane forms
// the H of its own operand elements (two channels, two pairs of the 8), so H
// is never staged; r, f_c and the 16 harmonics of a pair are formed once, by
// the lane that holds the pair, and staged in shared memory, one row per
// quantity and one column per pair.
//
// FP32 accuracy from split operands: x = x_h + x_l + O(2^-24 x), both parts
// TF32, and x y = x_l y_l + x_l y_h + x_h y_l + x_h y_h (the products are exact in
// FP32).  The tensor cores cut the sum to 24 bits where an FP32 add would round
// it: the sums of 8 pairs therefore start from zero, small terms first, and are
// added to the totals in FP32.  What the cut takes from each of them is known on
// average, half a unit in the last place of a number whose leading digits are as
// those of numbers are: 2^-24 (1/2) / ln 2 of it, and is put back once, at the end
// (UNCUT).  Component 0, the sum of H over the pairs, to which all terms add with
// one sign, is not left to them: every lane adds the H that it forms, in FP32.
// Errors against FP64 over 543 evaluations of the workloads and of random models,
// lattices and sizes, as multiples of those with FP32 multiply-adds in sequence
// and k_mlp (rms, K up to 64): G 0.95 to 1.00, forces 0.85 to 1.00.  Without x_l y_l
// and the rounding of x_l the forces of a 32-atom fcc and an 8,160-atom bcc cell are
// 1.04 and 1.05 (now 0.99 and 1.00).
// K = 128 (FINE false): three products and no separate sum, whose registers and
// additions would cost 0.07 of 0.32 ms (39,366 atoms): G 1.03, forces 0.94.
//
// A lane stages two pairs (2 l, 2 l + 1 of a batch of 64) on packed FP32x2
// arithmetic, so that most atoms need one batch.
//
// What bounds it: instruction issue (59 % of the slots; 880 warp instructions per
// atom at 54 pairs and K = 16; FMA pipe 36 %, ALU 34 %, tensor 30 %; waits on results
// of the steps before it).  The pass before it (packed FP32
// multiply-adds on a (K/8 x 4) block per lane) staged H as well, read 6 shared
// float4 per 16 multiply-add instructions and waited on shared memory.  1,048,576
// atoms, K = 16: 1.60 -> 1.20 ms; 148,176 atoms, K = 32: 0.356 -> 0.330; 39,366
// atoms, K = 128: 0.487 -> 0.322 ms.  (Three products, no separate sum of H: 1.03,
// 0.286, 0.338 ms, with the errors above.)
//
// CACHED: the atom's in-cutoff pairs come from the pair cache filled by
// k_screen; otherwise the pass screens the table itself (queue_pairs).
// Blocks per SM asked for (registers): measured 7 of 5 .. 8 at K = 16, S = 1
// (1.20 ms for 1M atoms, 6 and 8 the same, 5 1.21; for few atoms 7 is ahead: 37,044
// atoms 106 us, 6 blocks 115), 4 at K = 32, S = 1 (0.330 ms for 148,176 atoms; 5
// spill, 0.357, 3 0.383) and 5 at K = 16, S = 2 and 3 (S = 3: 0.432 ms for the batch
// of 128 systems, 4 blocks 0.445); the totals of larger S K leave no choice.
constexpr int desc_min_blocks(int s, int k) { return s * k <= 16 ? 7 : (s == 1 && k == 32 ? 4 : (s * k <= 48 ? 5 : 1)); }

constexpr float UNCUT = 4.3e-8f;

template <int K, int S, bool TAB, bool CACHED>
__global__ void __launch_bounds__(PW * 32, desc_min_blocks(S, K)) k_desc(DevModel m, DevNlist nl, const double *__restrict__ pos,
                                                  const int32_t *__restrict__ types, float *__restrict__ G,
                                                  float *__restrict__ Pout) {
    constexpr int MT = (K + 15) / 16;     // tiles of 16 channels
    constexpr int NC = K < 16 ? 1 : 2;    // channels of a lane per tile (rows g and g + 8)
    // slots of a batch of 64 pairs: groups of the neighbour species, each a
    // multiple of 8; row stride 8 mod 32 so that the float2 operand reads are
    // conflict-free
    constexpr int RS = S <= 2 ? 72 : 104;
    constexpr int Dd = S * K * 4;
    constexpr bool FINE = K <= 64;        // the product x_l y_l and a separate sum of H
    constexpr bool HOIST = MT <= 2;       // channel parameters in registers (per species group)
    constexpr bool RSH = S * S * K <= 512;   // the channel parameters fit beside the staging
    __shared__ float4 s_rad[RSH ? S * S * K : 1];   // (-mu_hi, -mu_lo, -eta log2 e, 0)
    __shared__ float4 s_q[CACHED ? 1 : PW][CACHED ? 1 : 96];
    __shared__ float2 s_q2[CACHED ? 1 : PW][CACHED ? 1 : 96];
    // rows: r_hi, r_lo, f_c (TAB: t, interval, 1), then component c in row
    // 3 + 8 ((c >> 1) & 1) + 2 (c >> 2) + (c & 1): operand column n of tile i
    // is component 4 (n >> 1) + 2 i + (n & 1), which leaves the lane t of a
    // quad with components 4t .. 4t + 3 of its channels
    __shared__ __align__(16) float s_st[PW][(3 + NHAR) * RS];
    if constexpr (RSH)
        for (int i = threadIdx.x; i < S * S * K; i += blockDim.x) {
            const float4 a = m.radial[i];
            s_rad[i] = make_float4(-a.x, -a.y, -a.z, 0.f);
        }
    auto channel = [&](int i) {
        if constexpr (RSH) return s_rad[i];
        const float4 a = __ldg(m.radial + i);
        return make_float4(-a.x, -a.y, -a.z, 0.f);
    };
    if (nl.err_clear && blockIdx.x == 0 && threadIdx.x == 0) *nl.err_clear = 0;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 2, t = lane & 3;   // operand row (channel) / column (pairs 2t, 2t + 1)
    const unsigned lt = (1u << lane) - 1u;
    float *const st = s_st[warp];
    // unused slots hold f_c = 0 and finite values; component 0 is 1
    auto clear_staging = [&]() {
        for (int i = lane; i < (3 + NHAR) * RS; i += 32) st[i] = (i / RS == 3) ? 1.f : 0.f;
    };
    clear_staging();
    __syncthreads();
    float Wt[4];
#pragma unroll
    for (int dd = 0; dd < 4; ++dd) Wt[dd] = c_W[4 * t + dd];
    const int64_t total = (int64_t)gridDim.x * PW;
    // CACHED: the pair-cache batches are read one batch ahead, across atom
    // boundaries (the next atom's segment one atom ahead, its perm entry two
    // atoms ahead), so that the pass waits on no load of its own stream.
    PairStream ps;
    const int32_t *const tys = S > 1 ? types : nullptr;
    if constexpr (CACHED) ps.start(nl, tys, (int64_t)blockIdx.x * PW + warp, total, lane);
    for (int64_t p = (int64_t)blockIdx.x * PW + warp; p < nl.n; p += total) {
        const int a = CACHED ? ps.a : nl.perm[p];
        const int ti = S == 1 ? 0 : (CACHED ? ps.ty : types[a]);
        if constexpr (CACHED) ps.atom_begins(nl, tys, p, total);
        // totals: tile i, channel g (x, y of [i]) and g + 8 ([2 + i])
        float2 acc[S][MT][4];
#pragma unroll
        for (int s = 0; s < S; ++s)
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                for (int i = 0; i < 4; ++i) acc[s][mt][i] = make_float2(0.f, 0.f);
        float sum0[S][MT][NC];   // component 0: this lane's pairs
#pragma unroll
        for (int s = 0; s < S; ++s)
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                for (int h = 0; h < NC; ++h) sum0[s][mt][h] = 0.f;
        auto pair_fn = [&](const PairTwo &w, int nb) {   // pairs 2 lane, 2 lane + 1 of nb
            const bool v0 = 2 * lane < nb, v1 = 2 * lane + 1 < nb;
            int slot0 = 2 * lane, slot1 = 2 * lane + 1, cnt[S];
            if constexpr (S == 1) {
                cnt[0] = nb;
            } else {
                const int b0 = v0 ? (int)(__float_as_uint(w.e0.w) >> 28) : S;
                const int b1 = v1 ? (int)(__float_as_uint(w.e1.w) >> 28) : S;
                int start = 0;
#pragma unroll
                for (int s = 0; s < S; ++s) {
                    const unsigned m0 = __ballot_sync(0xffffffffu, b0 == s), m1 = __ballot_sync(0xffffffffu, b1 == s);
                    const int before = start + __popc(m0 & lt) + __popc(m1 & lt);
                    if (b0 == s) slot0 = before;
                    if (b1 == s) slot1 = before + (b0 == s);
                    cnt[s] = __popc(m0) + __popc(m1);
                    start += (cnt[s] + 7) & ~7;
                }
                // f_c of every slot: the groups' padding contributes nothing
#pragma unroll
                for (int i = 0; i < RS; i += 32)
                    if (i + lane < RS) st[2 * RS + i + lane] = 0.f;
                __syncwarp();
            }
            auto put = [&](int row, const float2 v) {
                if constexpr (S == 1) {
                    *reinterpret_cast<float2 *>(st + row * RS + 2 * lane) = v;
                } else {
                    if (v0) st[row * RS + slot0] = v.x;
                    if (v1) st[row * RS + slot1] = v.y;
                }
            };
            float2 r_hi, r_lo, ir;
            split_sqrt2(make_float2(w.q0.x, w.q1.x), make_float2(w.q0.y, w.q1.y), r_hi, r_lo, ir);
            // Two atoms at one place have no direction and r is not a number.
            // What such a pair stages must not be there when its slots pad a
            // group of a later atom (0 x NaN is NaN): the staging is cleared
            // after this batch.  (One species: every slot is written each time.)
            const bool broken = S > 1 && __any_sync(0xffffffffu, !(r_hi.x + r_hi.y < INFINITY));
            if constexpr (TAB) {
                const float2 x = __fmul2_rn(r_hi, bc2(m.rtab_scale)), gf = make_float2(floorf(x.x), floorf(x.y));
                put(0, __ffma2_rn(r_lo, bc2(m.rtab_scale), __ffma2_rn(gf, bc2(-1.f), x)));
                // as tab_cell; a place without a pair reads interval 0
                put(1, make_float2(__int_as_float(v0 ? tab_interval(gf.x, m.rtab_n) : 0),
                                   __int_as_float(v1 ? tab_interval(gf.y, m.rtab_n) : 0)));
                put(2, make_float2(v0 ? 1.f : 0.f, v1 ? 1.f : 0.f));
            } else {
                const float2 fc = cutoff2(r_hi, m.inv_rc);
                put(0, r_hi);
                put(1, r_lo);
                put(2, make_float2(v0 ? fc.x : 0.f, v1 ? fc.y : 0.f));
            }
            float2 Y[NHAR];
            harmonics16(__fmul2_rn(make_float2(w.e0.x, w.e1.x), ir), __fmul2_rn(make_float2(w.e0.y, w.e1.y), ir),
                          __fmul2_rn(make_float2(w.e0.z, w.e1.z), ir), Y);
#pragma unroll
            for (int c = 1; c < NHAR; ++c) put(3 + 8 * ((c >> 1) & 1) + 2 * (c >> 2) + (c & 1), Y[c]);
            __syncwarp();
            int start = 0;
#pragma unroll
            for (int s = 0; s < S; ++s) {
                const int stop = start + cnt[s];
                const int rad = (ti * S + s) * K;
                const float *tab = TAB ? m.rtab + (size_t)(ti * S + s) * m.rtab_n * 4 * K : nullptr;
                float2 mh[HOIST ? MT : 1][NC], ml[HOIST ? MT : 1][NC], et[HOIST ? MT : 1][NC];
                if constexpr (HOIST && !TAB) {
#pragma unroll
                    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                        for (int h = 0; h < NC; ++h) {
                            const float4 q = channel(rad + 16 * mt + 8 * h + g);
                            mh[mt][h] = make_float2(q.x, q.x);
                            ml[mt][h] = make_float2(q.y, q.y);
                            et[mt][h] = make_float2(q.z, q.z);
                        }
                }
#pragma unroll 1
                for (int q0 = start; q0 < stop; q0 += 8) {
                    const int q = q0 + 2 * t;   // this lane's pairs q, q + 1
                    const float2 r0 = *reinterpret_cast<const float2 *>(st + q);
                    const float2 r1 = *reinterpret_cast<const float2 *>(st + RS + q);
                    const float2 fc = *reinterpret_cast<const float2 *>(st + 2 * RS + q);
                    Split2 y[2];
#pragma unroll
                    for (int i = 0; i < 2; ++i)
                        y[i] = split2(*reinterpret_cast<const float2 *>(st + (3 + 8 * i + g) * RS + q));
#pragma unroll
                    for (int mt = 0; mt < MT; ++mt) {
                        Split2 x[2];
                        x[1] = Split2{0u, 0u, 0u, 0u};
#pragma unroll
                        for (int h = 0; h < NC; ++h) {
                            float2 H;
                            if constexpr (TAB) {
                                const int k = 16 * mt + 8 * h + g;
                                const float4 *c = reinterpret_cast<const float4 *>(tab);
                                const float4 u = __ldg(c + (size_t)__float_as_int(r1.x) * K + k);
                                const float4 v = __ldg(c + (size_t)__float_as_int(r1.y) * K + k);
                                H.x = fmaf(r0.x, fmaf(r0.x, fmaf(r0.x, u.w, u.z), u.y), u.x);
                                H.y = fmaf(r0.y, fmaf(r0.y, fmaf(r0.y, v.w, v.z), v.y), v.x);
                                H = __fmul2_rn(H, fc);
                            } else {
                                float2 qh, ql, qe;
                                if constexpr (HOIST) {
                                    qh = mh[mt][h]; ql = ml[mt][h]; qe = et[mt][h];
                                } else {
                                    const float4 u = channel(rad + 16 * mt + 8 * h + g);
                                    qh = bc2(u.x); ql = bc2(u.y); qe = bc2(u.z);
                                }
                                const float2 d = __fadd2_rn(__fadd2_rn(r0, qh), __fadd2_rn(r1, ql));
                                const float2 ex = __fmul2_rn(__fmul2_rn(qe, d), d);
                                H = __fmul2_rn(make_float2(ex2_ftz(ex.x), ex2_ftz(ex.y)), fc);
                            }
                            if constexpr (FINE) sum0[s][mt][h] += H.x + H.y;
                            x[h] = split2(H);
                        }
#pragma unroll
                        for (int i = 0; i < 2; ++i) {
                            float c[4];
                            const uint32_t xl[4] = {x[0].l0, x[1].l0, x[0].l1, x[1].l1};
                            const uint32_t xh[4] = {x[0].h0, x[1].h0, x[0].h1, x[1].h1};
                            if constexpr (FINE) {
                                mma_tf32_first(c, xl, y[i].l0, y[i].l1);
                                mma_tf32(c, xl, y[i].h0, y[i].h1);
                            } else {
                                mma_tf32_first(c, xl, y[i].h0, y[i].h1);
                            }
                            mma_tf32(c, xh, y[i].l0, y[i].l1);
                            mma_tf32(c, xh, y[i].h0, y[i].h1);
                            acc[s][mt][i] = __fadd2_rn(make_float2(c[0], c[1]), acc[s][mt][i]);
                            if (NC == 2) acc[s][mt][2 + i] = __fadd2_rn(make_float2(c[2], c[3]), acc[s][mt][2 + i]);
                        }
                    }
                }
                start += (cnt[s] + 7) & ~7;
            }
            __syncwarp();
            if (broken) {
                clear_staging();
                __syncwarp();
            }
        };
        if constexpr (CACHED) {
            for (int base = 0; base < ps.np; base += 64) {
                const PairTwo w = ps.pf;
                ps.advance(nl, base, lane);
                pair_fn(w, min(64, ps.np - base));
            }
            if (ps.np == 0) ps.advance(nl, 0, lane);
        } else {
            queue_pairs<64>(nl, a, nl.beg[a], nl.end[a], m.rc2h, m.rc2l, s_q[warp], s_q2[warp], lane,
                           [&](const float4 *p, const float2 *p2, int nb) {
                               pair_fn(load_two(p, p2, 2 * lane, nb), nb);
                           });
        }
        // A[b][k][c] for the backward pass, and G
        float *Pa = Pout + (size_t)p * (S * K * NHAR);   // workspaces are indexed by perm position
        float *Ga = G + (size_t)p * Dd;
#pragma unroll
        for (int s = 0; s < S; ++s)
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                for (int h = 0; h < NC; ++h) {
                    const int row = s * K + 16 * mt + 8 * h + g;
                    float A[4] = {acc[s][mt][2 * h].x, acc[s][mt][2 * h].y, acc[s][mt][2 * h + 1].x,
                                  acc[s][mt][2 * h + 1].y};
#pragma unroll
                    for (int i = 0; i < 4; ++i) A[i] = fmaf(A[i], UNCUT, A[i]);
                    if constexpr (FINE) {
                        float a0 = sum0[s][mt][h];
                        a0 += __shfl_xor_sync(0xffffffffu, a0, 1);
                        a0 += __shfl_xor_sync(0xffffffffu, a0, 2);
                        if (t == 0) A[0] = a0;
                    }
                    *reinterpret_cast<float4 *>(Pa + row * NHAR + 4 * t) = make_float4(A[0], A[1], A[2], A[3]);
                    Ga[row * 4 + t] = desc_value(A, Wt, t);
                }
        if constexpr (CACHED) ps.atom_ends();
    }
}

// ---------------------------------------------------------------------------
// backward: P', pair gradients, ScatterSum, virial
// ---------------------------------------------------------------------------
// round(g * 2^32) as int64 (the 2^-32 fixed point of the ScatterSum) from
// 32-bit conversions only (on this GPU float <-> int64 conversions issue on
// the slow FP64 pipe); valid for |g| < 2^21.
__device__ __forceinline__ long long to_fixed(float g) {
    // two 32-bit stages: x = g 2^10 = r + v with r = rint(x) (|r| < 2^31 for
    // |g| < 2^21) and |v| <= 1/2 exact; then round(v 2^22) (exact scaling,
    // |.| <= 2^21): round(g 2^32) = r 2^22 + round(v 2^22), both roundings to
    // nearest even as a single rounding of g 2^32 would be
    const float x = g * 1024.0f;
    const float r = rintf(x);
    const int h1 = __float2int_rz(r);              // exact: r is an integer
    const int h2 = __float2int_rn((x - r) * 4194304.0f);
    return (long long)h1 * 4194304LL + (long long)h2;
}

// Sum of a fixed-point value over the 32 lanes of a warp, exact modulo 2^64
// (two's complement): each lane's value is cut into 21-, 21- and 22-bit
// chunks, whose lane sums (< 2^27) fit the 32-bit warp reduction, and the
// three sums are put back together.  Every lane receives the total.
__device__ __forceinline__ long long warp_sum_fixed(long long v) {
    const unsigned long long u = (unsigned long long)v;
    const unsigned c0 = __reduce_add_sync(0xffffffffu, (unsigned)(u & 0x1FFFFFull));
    const unsigned c1 = __reduce_add_sync(0xffffffffu, (unsigned)((u >> 21) & 0x1FFFFFull));
    const unsigned c2 = __reduce_add_sync(0xffffffffu, (unsigned)(u >> 42));
    return (long long)((unsigned long long)c0 + ((unsigned long long)c1 << 21) + ((unsigned long long)c2 << 42));
}

__device__ __forceinline__ void kahan_add(float &sum, float &comp, float x) {
    const float y = x - comp;
    const float t = sum + y;
    comp = (t - sum) - y;
    sum = t;
}

// The rest of g_ij once V_c and W_c of the pair are known, as packed pairs
// (c, c + 1).  The harmonics are formed in the same pairs, so that
// dE/dr = sum_c W_c Y_c runs on FP32x2 multiply-adds.
__device__ __forceinline__ void pair_grad_tail(const float2 (&V2)[NHAR / 2], const float2 (&W2)[NHAR / 2], float x,
                                               float y, float z, float ir, float &gxs, float &gys, float &gzs) {
    const float xx = x * x, yy = y * y, zz = z * z, d = xx - yy, q = fmaf(5.f, zz, -1.f);
    const float xy = x * y, yz = y * z, xz = x * z;
    const float p14 = fmaf(-3.f, yy, xx), p15 = fmaf(3.f, xx, -yy);
    const float2 Y2[NHAR / 2] = {make_float2(1.f, x),
                                 make_float2(y, z),
                                 make_float2(xy, yz),
                                 make_float2(xz, d),
                                 make_float2(zz - (1.f / 3.f), z * fmaf(5.f, zz, -3.f)),
                                 make_float2(x * q, y * q),
                                 make_float2(z * d, xy * z),
                                 make_float2(x * p14, y * p15)};
    float2 s0 = make_float2(0.f, 0.f), s1 = make_float2(0.f, 0.f);
#pragma unroll
    for (int t = 0; t < NHAR / 2; t += 2) {
        s0 = __ffma2_rn(W2[t], Y2[t], s0);
        s1 = __ffma2_rn(W2[t + 1], Y2[t + 1], s1);
    }
    const float dEdr = (s0.x + s0.y) + (s1.x + s1.y);
    // F2 = V M': dE/du = sum_c V_c grad Y_c.  Only its part tangent to the
    // sphere is used below, on which the gradients of the polynomials agree
    // with those of any other form of the same functions on the sphere.
    auto V = [&](int c) { return (c & 1) ? V2[c >> 1].y : V2[c >> 1].x; };
    const float b = 3.f * d;
    float gx = V(1) + y * V(4) + z * V(6) + q * V(10) + yz * V(13);
    float gy = V(2) + x * V(4) + z * V(5) + q * V(11) + xz * V(13);
    float gz = V(3) + y * V(5) + x * V(6) + 2.f * z * V(8) + fmaf(15.f, zz, -3.f) * V(9) + 10.f * xz * V(10) +
               10.f * yz * V(11) + d * V(12) + xy * V(13);
    gx += 2.f * x * (V(7) + z * V(12)) + b * V(14) + 6.f * xy * V(15);
    gy += -2.f * y * (V(7) + z * V(12)) - 6.f * xy * V(14) + b * V(15);
    const float ug = x * gx + y * gy + z * gz;
    // g_ij = dE/dD_ij = dE/dr u + (I - u u^T) dE/du / r
    gxs = fmaf(dEdr, x, (gx - x * ug) * ir);
    gys = fmaf(dEdr, y, (gy - y * ug) * ir);
    gzs = fmaf(dEdr, z, (gz - z * ug) * ir);
}

// g_ij = dE/dD_ij of one in-cutoff pair (Eqs. dP_abkd, U_abck, F1_abcx,
// F2_abcx): Pb = the centre atom's P' for the neighbour's species, rad = the
// radial parameters of the (centre, neighbour) species pair in the packed
// layout of stage_rad2.
template <int K, bool TAB>
__device__ __forceinline__ void pair_grad(const DevModel &m, const float4 e, const float2 e2, const float *Pb,
                                          const float4 *rad, const float *tab, float &gxs, float &gys, float &gzs) {
    float r_hi, r_lo, ir;
    split_sqrt(e2.x, e2.y, r_hi, r_lo, ir);
    const float ux = e.x * ir, uy = e.y * ir, uz = e.z * ir;
    // V_d = sum_k P'_kd H_k and W_d = sum_k P'_kd H'_k, so that
    // F1 = U H' R' = sum_d W_d M_d and F2 = V M'
    // V and W as packed pairs (d, d + 1): every multiply-add of the channel
    // loop is one FP32x2 instruction (each half rounded as fmaf)
    float2 V2[NHAR / 2], W2[NHAR / 2];
#pragma unroll
    for (int d = 0; d < NHAR / 2; ++d) V2[d] = W2[d] = make_float2(0.f, 0.f);
    float fc = 0.f, dfc = 0.f;
    TabCell tc;
    if (TAB)
        tc = tab_cell(tab, K, m.rtab_n, m.rtab_scale, r_hi, r_lo);
    else
        cutoff_fn(r_hi, m.inv_rc, fc, dfc);
    const float2 rh2 = make_float2(r_hi, r_hi), rl2 = make_float2(r_lo, r_lo);
    const float2 fc2 = make_float2(fc, fc), dfc2 = make_float2(dfc, dfc);
    constexpr int KU = K > 32 ? 16 : K;   // channels per unrolled block
#pragma unroll 1
    for (int kb = 0; kb < K; kb += KU)
#pragma unroll
    for (int ku = 0; ku < KU; ku += 2) {
        const int k = kb + ku;
        // H and H' of channels k, k + 1 formed inside the loop (no per-pair arrays)
        float Hk[2], dHk[2];
        if (TAB) {
            tab_eval(tc, k, m.rtab_scale, Hk[0], dHk[0]);
            tab_eval(tc, k + 1, m.rtab_scale, Hk[1], dHk[1]);
        } else {
            const Radial2 o = radial2<true>(rad, k, rh2, rl2, fc2, dfc2);
            Hk[0] = o.H.x; Hk[1] = o.H.y;
            dHk[0] = o.dH.x; dHk[1] = o.dH.y;
        }
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const float2 h2 = make_float2(Hk[c], Hk[c]), d2 = make_float2(dHk[c], dHk[c]);
#pragma unroll
            for (int q4 = 0; q4 < NHAR / 4; ++q4) {
                const float4 pd = *reinterpret_cast<const float4 *>(Pb + (k + c) * NHAR + 4 * q4);
                const float2 plo = make_float2(pd.x, pd.y), phi = make_float2(pd.z, pd.w);
                V2[2 * q4] = __ffma2_rn(plo, h2, V2[2 * q4]);
                V2[2 * q4 + 1] = __ffma2_rn(phi, h2, V2[2 * q4 + 1]);
                W2[2 * q4] = __ffma2_rn(plo, d2, W2[2 * q4]);
                W2[2 * q4 + 1] = __ffma2_rn(phi, d2, W2[2 * q4 + 1]);
            }
        }
    }
    pair_grad_tail(V2, W2, ux, uy, uz, ir, gxs, gys, gzs);
}

// V_c = sum_k A'_kc H_k and W_c = sum_k A'_kc H'_k of two in-cutoff pairs
// of one atom with neighbours of one species (Eqs. dP_abkd, U_abck, F1_abcx,
// F2_abcx), as packed pairs (c, c + 1): every multiply-add of the channel loop
// is one FP32x2 instruction (each half rounded as fmaf).  Pb = the atom's A' for
// the neighbours' species, rad = the channels of the (centre, neighbour) species
// pair in the packed layout of stage_rad2.
template <int K, bool TAB>
__device__ __forceinline__ void pair_sums2(const DevModel &m, const float (&rh)[2], const float (&rl)[2], const float *Pb,
                                            const float4 *rad, const float *tab, float2 (&V)[2][NHAR / 2],
                                           float2 (&W)[2][NHAR / 2]) {
    TabCell tc[2];
    float2 fc[2], dfc[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
#pragma unroll
        for (int d = 0; d < NHAR / 2; ++d) V[i][d] = W[i][d] = make_float2(0.f, 0.f);
        if (TAB) {
            tc[i] = tab_cell(tab, K, m.rtab_n, m.rtab_scale, rh[i], rl[i]);
        } else {
            float c, d;
            cutoff_fn(rh[i], m.inv_rc, c, d);
            fc[i] = bc2(c);
            dfc[i] = bc2(d);
        }
    }
    constexpr int KU = K > 32 ? 16 : K;   // channels per unrolled block
#pragma unroll 1
    for (int kb = 0; kb < K; kb += KU)
#pragma unroll
    for (int ku = 0; ku < KU; ku += 2) {
        const int k = kb + ku;
        // H and H' of channels k, k + 1 formed inside the loop (no per-pair arrays)
        float2 H[2], dH[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            if (TAB) {
                tab_eval(tc[i], k, m.rtab_scale, H[i].x, dH[i].x);
                tab_eval(tc[i], k + 1, m.rtab_scale, H[i].y, dH[i].y);
            } else {
                const Radial2 o = radial2<true>(rad, k, bc2(rh[i]), bc2(rl[i]), fc[i], dfc[i]);
                H[i] = o.H;
                dH[i] = o.dH;
            }
        }
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
            for (int q4 = 0; q4 < NHAR / 4; ++q4) {
                const float4 pd = *reinterpret_cast<const float4 *>(Pb + (k + c) * NHAR + 4 * q4);
                const float2 plo = make_float2(pd.x, pd.y), phi = make_float2(pd.z, pd.w);
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const float2 h2 = bc2(c ? H[i].y : H[i].x), d2 = bc2(c ? dH[i].y : dH[i].x);
                    V[i][2 * q4] = __ffma2_rn(plo, h2, V[i][2 * q4]);
                    V[i][2 * q4 + 1] = __ffma2_rn(phi, h2, V[i][2 * q4 + 1]);
                    W[i][2 * q4] = __ffma2_rn(plo, d2, W[i][2 * q4]);
                    W[i][2 * q4 + 1] = __ffma2_rn(phi, d2, W[i][2 * q4 + 1]);
                }
            }
    }
}

// A'_bkc = dE/dA_bkc (Eq. dP_abkd) of the atom at perm position p (A and G'
// are indexed by perm position) into a shared slot, each lane its (K/8 x 4)
// block: 2 w_c A_c G'_m(c) with, from the parts that ranks 2 and 3 hold of the
// lower degrees, G'_0 sign(A_0) + 2/3 G'_2 A_0 (c = 0) and G'_1 + 3/5 G'_3 in
// the place of G'_1 (c = 1..3).
__device__ __forceinline__ float4 aprime(const float4 A, const float4 gm, const float (&Wg)[4], int g) {
    const float h0 = g == 1 || g == 2 ? gm.z : gm.w;                      // c = 4g
    const float h = g == 0 ? FMA_HILO(0.6, gm.w, gm.y) : (g == 1 ? gm.z : gm.w);
    float4 o = make_float4(2.f * Wg[0] * A.x * h0, 2.f * Wg[1] * A.y * h, 2.f * Wg[2] * A.z * h, 2.f * Wg[3] * A.w * h);
    if (g == 0) o.x = fmaf(FMA_HILO(2.0 / 3.0, gm.z, 0.f), A.x, (A.x > 0.f) ? gm.x : ((A.x < 0.f) ? -gm.x : 0.f));
    return o;
}

template <int K, int S>
__device__ __forceinline__ void pprime_setup(const float *__restrict__ Pin, const float *__restrict__ dG, int64_t p,
                                             float *slot, int kg, int g, const float (&Wg)[4]) {
    constexpr int KPL = K / 8;
    constexpr int PSTR = K * NHAR + 4;
    constexpr int Dd = S * K * 4;
    const float *Pa = Pin + (size_t)p * (S * K * NHAR);
    const float *dGa = dG + (size_t)p * Dd;
#pragma unroll
    for (int s = 0; s < S; ++s)
#pragma unroll
        for (int kk = 0; kk < KPL; ++kk) {
            const int k = kg * KPL + kk;
            const float4 gm = *reinterpret_cast<const float4 *>(dGa + (s * K + k) * 4);
            const float4 A = *reinterpret_cast<const float4 *>(Pa + (s * K + k) * NHAR + 4 * g);
            *reinterpret_cast<float4 *>(slot + s * PSTR + k * NHAR + 4 * g) = aprime(A, gm, Wg, g);
        }
}

// Lane sums of the virial -> warp total (FP32, fixed order) added to the warp's
// FP64 accumulator; the lane sums restart from zero.  A lane sums the pairs of about
// VFLUSH / 32 of the warp's atoms between flushes, so the FP32 rounding stays at
// the level of one atom's virial.  The lanes halve eight of the values among
// themselves as they add, and eight lanes add them to the accumulator (nine
// butterflies and nine FP64 additions by one lane: k_force at 1,048,576 atoms 2.07 ms,
// at 16,384 atoms of two species 66.5 us; this 2.03 ms and 63.5 us).
constexpr int VFLUSH = 8;
__device__ __forceinline__ void virial_flush(float (&wacc)[9], double *acc, int lane) {
#pragma unroll
    for (int n = 4; n >= 1; n >>= 1) {
        const bool up = lane & (4 * n);
#pragma unroll
        for (int i = 0; i < n; ++i) {
            const float send = up ? wacc[i] : wacc[i + n], keep = up ? wacc[i + n] : wacc[i];
            wacc[i] = keep + __shfl_xor_sync(0xffffffffu, send, 4 * n);
        }
    }
    float v = wacc[0], w = wacc[8];
#pragma unroll
    for (int o = 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
    if (!(lane & 3)) acc[((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1)] += (double)v;
    if (lane == 1) acc[8] += (double)w;
#pragma unroll
    for (int t = 0; t < 9; ++t) wacc[t] = 0.f;
}

// Force pass over the pair cache with full lane batches: each warp walks a
// contiguous run of atoms (perm order) and fills every batch of 32 lanes with
// the rest of the current atom's pairs followed by the first pairs of the
// next atom (two P' slots per warp, two self-force accumulators).
// For one species: there it is the faster one on the whole (1,048,576 atoms, K = 16,
// 54 pairs: 2.04 ms, k_force 2.10; 128,000 atoms of the dense bcc lattice, 82 pairs:
// 0.34 and 0.39; 39,366 atoms, K = 128: 0.63 and 0.70; K = 32 and 64 are 2 % the other
// way: 0.530 and 0.517, 0.447 and 0.437), for its batches are full.  Two pairs per
// lane in this form: 2.37 ms.
template <int K, int S, bool TAB>
__global__ void __launch_bounds__(PW * 32, 4) k_force_merged(DevModel m, DevNlist nl, const int32_t *__restrict__ types,
                                                          const float *__restrict__ Pin, const float *__restrict__ dG,
                                                          unsigned long long *__restrict__ Fq,
                                                          double *__restrict__ part_w) {
    constexpr int PSTR = K * NHAR + 4;
    __shared__ float4 s_rad[S * S * K];
    __shared__ __align__(16) float s_Pd[PW][2][S * PSTR];
    __shared__ double s_w[PW][9];
    stage_rad2(s_rad, m.radial, S * S * K);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane < 9) s_w[warp][lane] = 0.0;
    __syncthreads();
    const int kg = lane >> 2, g = lane & 3;
    float Wg[4];
#pragma unroll
    for (int dd = 0; dd < 4; ++dd) Wg[dd] = c_W[4 * g + dd];
    // virial: each lane's pairs summed in FP32 over VFLUSH atoms, then the
    // warp's total added to an FP64 accumulator in shared memory
    float wacc[9];
#pragma unroll
    for (int t = 0; t < 9; ++t) wacc[t] = 0.f;
    int since = 0;
    const int64_t nw = (int64_t)gridDim.x * PW, wid = (int64_t)blockIdx.x * PW + warp;
    const int64_t chunk = (nl.n + nw - 1) / nw;
    int64_t p = wid * chunk;
    const int64_t pend = min(nl.n, p + chunk);
    if (p < pend) {
        int slot = 0;
        int a = nl.perm[p], ta = types[a];
        pprime_setup<K, S>(Pin, dG, p, s_Pd[warp][0], kg, g, Wg);
        int64_t cb = nl.beg[a];
        int cr = nl.npair[a];
        long long fcx = 0, fcy = 0, fcz = 0;
        while (p < pend) {
            const int take_c = min(cr, 32);
            const bool has_n = cr < 32 && p + 1 < pend;
            int take_n = 0, an = 0, tn = 0, nr = 0;
            int64_t nb = 0;
            if (has_n) {   // bring in the next atom
                an = nl.perm[p + 1];
                tn = types[an];
                pprime_setup<K, S>(Pin, dG, p + 1, s_Pd[warp][slot ^ 1], kg, g, Wg);
                nb = nl.beg[an];
                nr = nl.npair[an];
                take_n = min(nr, 32 - cr);
            }
            __syncwarp();
            long long fnx = 0, fny = 0, fnz = 0;
            const bool isc = lane < take_c, isn = !isc && lane < take_c + take_n;
            if (isc || isn) {
                const int64_t c = isc ? cb + lane : nb + (lane - take_c);
                const float4 e = nl.pq[c];
                const float2 e2 = nl.pq2[c];
                const uint32_t jb = __float_as_uint(e.w);
                const int b = (int)(jb >> 28);
                const int j = (int)(jb & 0x0FFFFFFFu);
                const float *Pb = s_Pd[warp][isc ? slot : slot ^ 1] + b * PSTR;
                const int tp = (isc ? ta : tn) * S + b;
                float gxs, gys, gzs;
                pair_grad<K, TAB>(m, e, e2, Pb, &s_rad[tp * K], TAB ? m.rtab + (size_t)tp * m.rtab_n * 4 * K : nullptr,
                                  gxs, gys, gzs);
                // ScatterSum in 2^-32 fixed point (exact, order independent)
                const long long qx = to_fixed(gxs);
                const long long qy = to_fixed(gys);
                const long long qz = to_fixed(gzs);
                if (isc) { fcx += qx; fcy += qy; fcz += qz; }
                else { fnx = qx; fny = qy; fnz = qz; }
                atomicAdd(&Fq[3 * (int64_t)j], (unsigned long long)(-qx));
                atomicAdd(&Fq[3 * (int64_t)j + 1], (unsigned long long)(-qy));
                atomicAdd(&Fq[3 * (int64_t)j + 2], (unsigned long long)(-qz));
                const float D[3] = {e.x, e.y, e.z};
                const float gv[3] = {gxs, gys, gzs};
#pragma unroll
                for (int al = 0; al < 3; ++al)
#pragma unroll
                    for (int be = 0; be < 3; ++be) wacc[al * 3 + be] = fmaf(-D[al], gv[be], wacc[al * 3 + be]);
            }
            cb += take_c;
            cr -= take_c;
            if (cr == 0) {   // the current atom is complete: its own force
                fcx = warp_sum_fixed(fcx);
                fcy = warp_sum_fixed(fcy);
                fcz = warp_sum_fixed(fcz);
                if (lane == 0) {
                    atomicAdd(&Fq[3 * (int64_t)a], (unsigned long long)fcx);
                    atomicAdd(&Fq[3 * (int64_t)a + 1], (unsigned long long)fcy);
                    atomicAdd(&Fq[3 * (int64_t)a + 2], (unsigned long long)fcz);
                }
                if (++since == VFLUSH) {
                    virial_flush(wacc, s_w[warp], lane);
                    since = 0;
                }
                ++p;
                if (p < pend) {
                    if (has_n) {   // the next atom (already set up) becomes the current one
                        a = an;
                        ta = tn;
                        slot ^= 1;
                        cb = nb + take_n;
                        cr = nr - take_n;
                        fcx = fnx; fcy = fny; fcz = fnz;
                    } else {
                        __syncwarp();
                        a = nl.perm[p];
                        ta = types[a];
                        pprime_setup<K, S>(Pin, dG, p, s_Pd[warp][slot], kg, g, Wg);
                        cb = nl.beg[a];
                        cr = nl.npair[a];
                        fcx = fcy = fcz = 0;
                    }
                }
            }
            __syncwarp();
        }
    }
    virial_flush(wacc, s_w[warp], lane);
    __syncthreads();
    if (threadIdx.x < 9) {
        double v = 0.0;
        for (int w = 0; w < PW; ++w) v += s_w[w][threadIdx.x];
        part_w[(size_t)blockIdx.x * 9 + threadIdx.x] = v;
    }
}

// ---------------------------------------------------------------------------
// force pass with the per-atom contractions on tensor cores
// ---------------------------------------------------------------------------
// For one atom the pair sums V_jd = sum_k H_jk P'_kd and W_jd = sum_k H'_jk P'_kd
// (Eqs. U_abck, F1_abcx, F2_abcx) are one matrix product: [H; H'] (rows =
// pairs, columns = k) times P' (k x d).  Each warp takes its atom's cached
// pairs 32 at a time: every lane forms H and H' of its pair into a shared
// 64 x K tile (rows 0-31 H, rows 32-63 H'), the warp multiplies the tile by P'
// with mma.sync m16n8k8 on TF32 operands, and
// every lane reads back the V and W rows of its pair for the rest of g_ij.
// FP32 accuracy from TF32 products: each operand x is split into
// x_hi = tf32(x) and x_lo = tf32(x - x_hi), and a product is accumulated as
// a_lo b_hi + a_hi b_lo + a_hi b_hi in FP32 (the dropped a_lo b_lo and the
// split remainders are about 2^-22 of |a b|).
// One species, direct radial basis, pair cache present.
template <int K>
__global__ void __launch_bounds__(PW * 32, 4) k_force_tc(DevModel m, DevNlist nl, const float *__restrict__ Pin,
                                                      const float *__restrict__ dG,
                                                      unsigned long long *__restrict__ Fq,
                                                      double *__restrict__ part_w) {
    static_assert(K % 8 == 0 && K <= 32, "k steps of 8, one pass");
    constexpr int KS = K / 8;        // k steps of the product
    constexpr int AS = K + 4;        // row stride of the H / H' tile (conflict-free fragment loads)
    constexpr int CS = 20;           // row stride of the V / W tile (16 columns, 16-byte rows)
    constexpr int PSTR = K * NHAR + 4;
    // the V / W tile is written over the H / H' tile, one m tile at a time,
    // in descending order when its rows are longer (CS > AS) and ascending
    // otherwise: the words a tile's results land on then hold only H / H'
    // rows of this tile (already in registers) or of tiles already multiplied
    constexpr int TILE = (64 * CS > 64 * AS) ? 64 * CS : 64 * AS;
    constexpr bool ASCENDING = AS >= CS;
    __shared__ float4 s_rad[K];
    __shared__ __align__(16) float s_Pd[PW][PSTR];
    __shared__ __align__(16) float s_T[PW][TILE];
    __shared__ double s_w[PW][9];
    for (int t = threadIdx.x; t < K; t += blockDim.x) s_rad[t] = m.radial[t];
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int kg = lane >> 2, g = lane & 3;   // P' setup block; also the fragment row / column group
    float Wg[4];
#pragma unroll
    for (int dd = 0; dd < 4; ++dd) Wg[dd] = c_W[4 * g + dd];
    float wsum[9], wcmp[9];
#pragma unroll
    for (int t = 0; t < 9; ++t) { wsum[t] = 0.f; wcmp[t] = 0.f; }
    float *sPd = s_Pd[warp];
    float *sT = s_T[warp];
    const int64_t total = (int64_t)gridDim.x * PW;
    for (int64_t p = (int64_t)blockIdx.x * PW + warp; p < nl.n; p += total) {
        const int a = nl.perm[p];
        pprime_setup<K, 1>(Pin, dG, p, sPd, kg, g, Wg);
        __syncwarp();
        // B fragments of P' (k x 16), hi and lo parts: b0 = (k = t, n = g), b1 = (k = t + 4, n = g)
        uint32_t bh[KS][2][2], bl[KS][2][2];
#pragma unroll
        for (int ks = 0; ks < KS; ++ks)
#pragma unroll
            for (int nt = 0; nt < 2; ++nt)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int k = ks * 8 + g + 4 * h, d = nt * 8 + kg;
                    split_tf32(sPd[k * NHAR + d], bh[ks][nt][h], bl[ks][nt][h]);
                }
        const int np = nl.npair[a];
        const int64_t pb = nl.beg[a];
        long long fx = 0, fy = 0, fz = 0;
        float wa[9];
#pragma unroll
        for (int t = 0; t < 9; ++t) wa[t] = 0.f;
        for (int base = 0; base < np; base += 32) {
            const int nb = min(32, np - base);
            const bool valid = lane < nb;
            float4 e = make_float4(0.f, 0.f, 0.f, 0.f);
            float2 e2 = make_float2(1.f, 0.f);
            if (valid) {
                e = nl.pq[pb + base + lane];
                e2 = nl.pq2[pb + base + lane];
            }
            float r_hi, r_lo, ir;
            split_sqrt(e2.x, e2.y, r_hi, r_lo, ir);
            {   // H and H' of this lane's pair into rows lane and 32 + lane (zeros for idle lanes)
                float fc, dfc;
                cutoff_fn(r_hi, m.inv_rc, fc, dfc);
                if (!valid) fc = dfc = 0.f;
                float *hrow = sT + lane * AS, *drow = sT + (32 + lane) * AS;
#pragma unroll
                for (int k4 = 0; k4 < K; k4 += 4) {
                    float hv[4], dv[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const float4 rp = s_rad[k4 + u];
                        const float t = (r_hi - rp.x) + (r_lo - rp.y);
                        const float f = ex2_ftz(-rp.z * t * t);
                        hv[u] = f * fc;
                        dv[u] = f * fmaf(-rp.w * t, fc, dfc);
                    }
                    *reinterpret_cast<float4 *>(hrow + k4) = make_float4(hv[0], hv[1], hv[2], hv[3]);
                    *reinterpret_cast<float4 *>(drow + k4) = make_float4(dv[0], dv[1], dv[2], dv[3]);
                }
            }
            __syncwarp();
            // [H; H'] P' -> V / W rows (m tiles 0, 1: H; 2, 3: H'); tiles past
            // the last pair are skipped
            const int mt_used = (nb + 15) >> 4;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int mt = ASCENDING ? i : 3 - i;
                if ((mt & 1) >= mt_used) continue;
                float c[2][4];
#pragma unroll
                for (int nt = 0; nt < 2; ++nt)
#pragma unroll
                    for (int q = 0; q < 4; ++q) c[nt][q] = 0.f;
#pragma unroll
                for (int ks = 0; ks < KS; ++ks) {
                    const float *r0 = sT + (mt * 16 + kg) * AS + ks * 8 + g;
                    const float *r1 = r0 + 8 * AS;
                    uint32_t ah[4], al[4];
                    split_tf32(r0[0], ah[0], al[0]);
                    split_tf32(r1[0], ah[1], al[1]);
                    split_tf32(r0[4], ah[2], al[2]);
                    split_tf32(r1[4], ah[3], al[3]);
#pragma unroll
                    for (int nt = 0; nt < 2; ++nt) {
                        mma_tf32(c[nt], al, bh[ks][nt][0], bh[ks][nt][1]);
                        mma_tf32(c[nt], ah, bl[ks][nt][0], bl[ks][nt][1]);
                        mma_tf32(c[nt], ah, bh[ks][nt][0], bh[ks][nt][1]);
                    }
                }
                __syncwarp();   // every lane's fragment loads of this tile precede the stores below
#pragma unroll
                for (int nt = 0; nt < 2; ++nt) {
                    float *c0 = sT + (mt * 16 + kg) * CS + nt * 8 + 2 * g;
                    *reinterpret_cast<float2 *>(c0) = make_float2(c[nt][0], c[nt][1]);
                    *reinterpret_cast<float2 *>(c0 + 8 * CS) = make_float2(c[nt][2], c[nt][3]);
                }
                __syncwarp();
            }
            if (valid) {
                float2 V2[NHAR / 2], W2[NHAR / 2];
                const float *vr = sT + lane * CS, *wr = sT + (32 + lane) * CS;
#pragma unroll
                for (int q4 = 0; q4 < NHAR / 4; ++q4) {
                    const float4 v = *reinterpret_cast<const float4 *>(vr + 4 * q4);
                    const float4 w = *reinterpret_cast<const float4 *>(wr + 4 * q4);
                    V2[2 * q4] = make_float2(v.x, v.y); V2[2 * q4 + 1] = make_float2(v.z, v.w);
                    W2[2 * q4] = make_float2(w.x, w.y); W2[2 * q4 + 1] = make_float2(w.z, w.w);
                }
                float gxs, gys, gzs;
                pair_grad_tail(V2, W2, e.x * ir, e.y * ir, e.z * ir, ir, gxs, gys, gzs);
                const int j = (int)(__float_as_uint(e.w) & 0x0FFFFFFFu);
                // ScatterSum in 2^-32 fixed point (exact, order independent)
                const long long qx = to_fixed(gxs);
                const long long qy = to_fixed(gys);
                const long long qz = to_fixed(gzs);
                fx += qx; fy += qy; fz += qz;
                atomicAdd(&Fq[3 * (int64_t)j], (unsigned long long)(-qx));
                atomicAdd(&Fq[3 * (int64_t)j + 1], (unsigned long long)(-qy));
                atomicAdd(&Fq[3 * (int64_t)j + 2], (unsigned long long)(-qz));
                const float D[3] = {e.x, e.y, e.z};
                const float gv[3] = {gxs, gys, gzs};
#pragma unroll
                for (int al = 0; al < 3; ++al)
#pragma unroll
                    for (int be = 0; be < 3; ++be) wa[al * 3 + be] = fmaf(-D[al], gv[be], wa[al * 3 + be]);
            }
            __syncwarp();   // the tile is rewritten by the next batch
        }
        fx = warp_sum_fixed(fx);
        fy = warp_sum_fixed(fy);
        fz = warp_sum_fixed(fz);
        if (lane == 0) {
            atomicAdd(&Fq[3 * (int64_t)a], (unsigned long long)fx);
            atomicAdd(&Fq[3 * (int64_t)a + 1], (unsigned long long)fy);
            atomicAdd(&Fq[3 * (int64_t)a + 2], (unsigned long long)fz);
        }
#pragma unroll
        for (int t = 0; t < 9; ++t) kahan_add(wsum[t], wcmp[t], wa[t]);
        __syncwarp();   // sPd is rewritten by the next atom
    }
    // virial: per-lane compensated sums -> warp total as an FP32 double-float -> FP64 block total
#pragma unroll
    for (int t = 0; t < 9; ++t) {
        float hi = wsum[t], lo = -wcmp[t];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float oh = __shfl_xor_sync(0xffffffffu, hi, o), ol = __shfl_xor_sync(0xffffffffu, lo, o);
            float sh, se;
            two_sum(hi, oh, sh, se);
            lo = (lo + ol) + se;
            two_sum(sh, lo, hi, lo);
        }
        if (lane == 0) s_w[warp][t] = (double)hi + (double)lo;
    }
    __syncthreads();
    if (threadIdx.x < 9) {
        double v = 0.0;
        for (int w = 0; w < PW; ++w) v += s_w[w][threadIdx.x];
        part_w[(size_t)blockIdx.x * 9 + threadIdx.x] = v;
    }
}

// Force pass: A' = dE/dA of every atom, g_ij = dE/dD_ij of its pairs, the
// ScatterSum of g_ij and the virial.  One warp per atom.  Batches of up to BF
// pairs, two neighbouring places per lane: pairs of one species, so that a lane
// reads each A' value once for both (more than one species: the batch is put in
// shared memory in groups of the neighbour species, padded to even length); up
// to 32 remaining pairs go one per lane.
//
// What bounds it: the A' values of the channel loop.  16 floats a channel and
// lane take the data path of shared memory 4 cycles for each 16 bytes a lane,
// for one pair per lane more than their multiply-adds take the FP32 pipes
// (without these loads the pass runs in 1.29 ms instead of 2.1 at 1,048,576
// atoms, K = 16).  A batch passes through shared memory also with one species:
// pairs read from global memory stay in registers over the channel loop, which
// then spills (2.99 ms against 2.10).  Measured, one pair per lane -> two:
// 16,384 atoms, 2 species, K = 16, 78 pairs: 87 -> 64 us; 225,008 atoms in 128
// systems, 3 species, 54 pairs: 0.76 -> 0.69 ms; 93,802 atoms in 24 systems, 2
// species: 0.40 -> 0.33 ms; table screened in the pass, 8,160 atoms: 46 -> 39 us.
//
// CACHED: the pairs are those of the pair cache, else the table is screened
// here.  PAW (batched): each atom's virial is summed over its own pairs and
// written to w_atom [atoms][9] for per-system reductions; otherwise each block
// writes one FP64 partial: without a cache every atom's virial goes to FP64 by
// itself, with one those of VFLUSH atoms together.
template <int K, int S, bool PAW, bool CACHED, bool TAB>
__global__ void __launch_bounds__(PW * 32, 4) k_force(DevModel m, DevNlist nl, const int32_t *__restrict__ types,
                                                   const float *__restrict__ Pin, const float *__restrict__ dG,
                                                   unsigned long long *__restrict__ Fq,
                                                   double *__restrict__ part_w, float *__restrict__ w_atom) {
    constexpr int PSTR = K * NHAR + 4;   // per-species stride of A' (bank offset between species)
    constexpr int BF = S == 1 ? 64 : (64 - S) & ~1;
    constexpr bool QUEUE = !CACHED;
    constexpr int FLUSH = CACHED ? VFLUSH : 1;   // atoms whose virial is summed in FP32
    __shared__ float4 s_rad[S * S * K];
    __shared__ float4 s_q[QUEUE ? PW : 1][QUEUE ? 96 : 1];
    __shared__ float2 s_q2[QUEUE ? PW : 1][QUEUE ? 96 : 1];
    constexpr bool STAGE = S > 1 || CACHED;
    __shared__ float4 s_g[STAGE ? PW : 1][STAGE ? 64 : 1];   // a batch in species groups
    __shared__ float2 s_g2[STAGE ? PW : 1][STAGE ? 64 : 1];
    __shared__ __align__(16) float s_Pd[PW][S * PSTR];
    __shared__ double s_w[PW][9];
    stage_rad2(s_rad, m.radial, S * S * K);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane < 9) s_w[warp][lane] = 0.0;
    __syncthreads();
    const int kg = lane >> 2, g = lane & 3;
    const unsigned lt = (1u << lane) - 1u;
    float Wg[4];
#pragma unroll
    for (int dd = 0; dd < 4; ++dd) Wg[dd] = c_W[4 * g + dd];
    float wacc[9];   // virial: this lane's pairs of the atom (PAW) or of up to FLUSH atoms
#pragma unroll
    for (int t = 0; t < 9; ++t) wacc[t] = 0.f;
    int since = 0;
    float *const sPd = s_Pd[warp];
    const int nw = (int)gridDim.x * PW;
    int p = (int)blockIdx.x * PW + warp;
    const int n = (int)nl.n;
    int a = p < n ? nl.perm[p] : -1;
    while (a >= 0) {
        const int an = p + nw < n ? nl.perm[p + nw] : -1;
        const int ti = S > 1 ? types[a] : 0;
        const int64_t pb = nl.beg[a];
        const int np = CACHED ? nl.npair[a] : 0;
        pprime_setup<K, S>(Pin, dG, p, sPd, kg, g, Wg);
        __syncwarp();
        long long fx = 0, fy = 0, fz = 0;
        auto scatter = [&](float gx, float gy, float gz, const float4 e) {
            // ScatterSum in 2^-32 fixed point: integer adds are exact and
            // order independent, so forces are bitwise reproducible.
            const long long qx = to_fixed(gx), qy = to_fixed(gy), qz = to_fixed(gz);
            fx += qx; fy += qy; fz += qz;
            unsigned long long *const Fj = Fq + 3 * (int64_t)(__float_as_uint(e.w) & 0x0FFFFFFFu);
            atomicAdd(Fj, (unsigned long long)(-qx));
            atomicAdd(Fj + 1, (unsigned long long)(-qy));
            atomicAdd(Fj + 2, (unsigned long long)(-qz));
            const float D[3] = {e.x, e.y, e.z};
            const float gv[3] = {gx, gy, gz};
#pragma unroll
            for (int al = 0; al < 3; ++al)
#pragma unroll
                for (int be = 0; be < 3; ++be) wacc[al * 3 + be] = fmaf(-D[al], gv[be], wacc[al * 3 + be]);
        };
        // the nb pairs at q, q2: in shared memory or in the cache
        auto batch = [&](const float4 *q, const float2 *q2, int nb) {
            if (nb <= 32) {   // one pair per lane
                if (lane < nb) {
                    const float4 e = q[lane];
                    const int b = S > 1 ? (int)(__float_as_uint(e.w) >> 28) : 0;
                    float gx, gy, gz;
                    pair_grad<K, TAB>(m, e, q2[lane], sPd + b * PSTR, &s_rad[(ti * S + b) * K],
                                      TAB ? m.rtab + (size_t)(ti * S + b) * m.rtab_n * 4 * K : nullptr, gx, gy, gz);
                    scatter(gx, gy, gz, e);
                }
                return;
            }
            int b = 0, n0 = nb;   // this lane's species group, the end of its pairs
            if constexpr (S == 1 && STAGE) {
                s_g[warp][lane] = q[lane];
                s_g2[warp][lane] = q2[lane];
                if (lane + 32 < nb) {
                    s_g[warp][lane + 32] = q[lane + 32];
                    s_g2[warp][lane + 32] = q2[lane + 32];
                }
                q = s_g[warp];
                q2 = s_g2[warp];
                __syncwarp();
            } else if constexpr (S > 1) {
                const bool two = lane + 32 < nb;
                const float4 e0 = q[lane], e1 = q[two ? lane + 32 : lane];
                const float2 f0 = q2[lane], f1 = q2[two ? lane + 32 : lane];
                const int b0 = (int)(__float_as_uint(e0.w) >> 28), b1 = two ? (int)(__float_as_uint(e1.w) >> 28) : S;
                int start = 0;
                n0 = 0;
#pragma unroll
                for (int s = 0; s < S; ++s) {
                    const unsigned m0 = __ballot_sync(0xffffffffu, b0 == s), m1 = __ballot_sync(0xffffffffu, b1 == s);
                    const int c0 = start + __popc(m0 & lt), c1 = start + __popc(m0) + __popc(m1 & lt);
                    if (b0 == s) { s_g[warp][c0] = e0; s_g2[warp][c0] = f0; }
                    if (b1 == s) { s_g[warp][c1] = e1; s_g2[warp][c1] = f1; }
                    const int cnt = __popc(m0) + __popc(m1);
                    if (2 * lane >= start && 2 * lane < start + cnt) { b = s; n0 = start + cnt; }
                    start += (cnt + 1) & ~1;
                }
                q = s_g[warp];
                q2 = s_g2[warp];
                __syncwarp();
            }
            const int i0 = 2 * lane;
            if (i0 < n0) {
                const bool two = i0 + 1 < n0;
                const float2 ra = q2[i0], rb = q2[two ? i0 + 1 : i0];
                float2 rh, rl, ir;
                split_sqrt2(make_float2(ra.x, rb.x), make_float2(ra.y, rb.y), rh, rl, ir);
                float2 V[2][NHAR / 2], W[2][NHAR / 2];
                const float rhx[2] = {rh.x, rh.y}, rlx[2] = {rl.x, rl.y};
                pair_sums2<K, TAB>(m, rhx, rlx, sPd + b * PSTR, &s_rad[(ti * S + b) * K],
                                     TAB ? m.rtab + (size_t)(ti * S + b) * m.rtab_n * 4 * K : nullptr, V, W);
#pragma unroll
                for (int i = 0; i < 2; ++i)
                    if (i == 0 || two) {
                        const float4 e = q[i0 + i];
                        const float r1 = i ? ir.y : ir.x;
                        float gx, gy, gz;
                        pair_grad_tail(V[i], W[i], e.x * r1, e.y * r1, e.z * r1, r1, gx, gy, gz);
                        scatter(gx, gy, gz, e);
                    }
            }
            if (STAGE) __syncwarp();   // the groups are rewritten by the next batch
        };
        if constexpr (CACHED) {
            for (int base = 0; base < np; base += BF) batch(nl.pq + pb + base, nl.pq2 + pb + base, min(BF, np - base));
        } else {
            queue_pairs<BF>(nl, a, pb, nl.end[a], m.rc2h, m.rc2l, s_q[warp], s_q2[warp], lane, batch);
        }
        fx = warp_sum_fixed(fx);
        fy = warp_sum_fixed(fy);
        fz = warp_sum_fixed(fz);
        if (lane < 3) atomicAdd(&Fq[3 * (int64_t)a + lane], (unsigned long long)(lane == 0 ? fx : (lane == 1 ? fy : fz)));
        if constexpr (PAW) {
#pragma unroll
            for (int t = 0; t < 9; ++t) {
                float v = wacc[t];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                if (lane == 0) w_atom[(size_t)a * 9 + t] = v;
                wacc[t] = 0.f;
            }
        } else if (++since == FLUSH) {
            virial_flush(wacc, s_w[warp], lane);
            since = 0;
        }
        __syncwarp();   // A' is rewritten by the next atom
        p += nw;
        a = an;
    }
    if (!PAW) {
        virial_flush(wacc, s_w[warp], lane);
        __syncthreads();
        if (threadIdx.x < 9) {
            double v = 0.0;
            for (int w = 0; w < PW; ++w) v += s_w[w][threadIdx.x];
            part_w[(size_t)blockIdx.x * 9 + threadIdx.x] = v;
        }
    }
}

// Blocks of the descriptor pass: what the GPU holds at once, and more once every
// warp would run over 512 channels (atoms x S x K), so that blocks that finish early
// are replaced (1M atoms, K = 16, when the pass took 1.02 ms: 1.12 ms with the
// resident 7 blocks per SM, 1.04 with 4 times, 1.02 with 8 times and 1.05 with 64
// times as many; 39,366 atoms, K = 128: 0.51 ms with the resident blocks, 0.34 with 4
// atoms per warp; 16,384 atoms, K = 16: 0.041 ms with the resident blocks, 0.045 with
// 8 times as many).  In tuned models, too: their pair_bps, 4 to 32 blocks per SM, is
// the force pass's (here 4 to 16 took 1.27 to 1.49 ms at 1M atoms instead of 1.20).
constexpr int CHANNELS_PER_WARP = 512;
template <auto KERNEL>
int desc_blocks(const DevModel &dm, int64_t n) {
    static const int resident = [] {
        int dev = 0, nsm = 0, per_sm = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, KERNEL, PW * 32, 0);
        return std::max(1, nsm) * std::max(1, per_sm);
    }();
    const int64_t most = (n + PW - 1) / PW;
    return (int)std::max<int64_t>(1, std::min<int64_t>(most, std::max<int64_t>(resident, n * dm.S * dm.K / (PW * CHANNELS_PER_WARP))));
}

template <int K, int S, bool TAB, bool CACHED>
void launch_desc(const DevModel &dm, const DevNlist &dn, const double *pos, const int32_t *types, tmd_nlist *nl,
                 cudaStream_t s) {
    const int nb = desc_blocks<k_desc<K, S, TAB, CACHED>>(dm, dn.n);
    TMD_LAUNCH("k_desc", s, k_desc<K, S, TAB, CACHED><<<nb, PW * 32, 0, s>>>(dm, dn, pos, types, nl->G, nl->P));
}

template <int K, int S, bool PAW, bool CACHED, bool TAB>
void launch_force(const DevModel &dm, const DevNlist &dn, const double *pos, const int32_t *types, tmd_nlist *nl,
                  double *part_w, int nblk, cudaStream_t s, float *w_atom) {
    TMD_LAUNCH("k_force", s, k_force<K, S, PAW, CACHED, TAB><<<nblk, PW * 32, 0, s>>>(dm, dn, types, nl->P, nl->dG,
                                                                                   nl->Fq, part_w, w_atom));
}

template <int K, int S>
tmd_status launch_pair_kernels(const DevModel &dm, const DevNlist &dn, const double *pos, const int32_t *types,
                               tmd_nlist *nl, double *part_w, int nblk, cudaStream_t s, bool forward,
                               float *w_atom) {
    if (forward && dn.pq) {   // screen into the pair cache, then stream it
        const tmd_status st = launch_screen(dm, dn, s);
        if (st != TMD_OK) return st;
        if (dm.rtab) launch_desc<K, S, true, true>(dm, dn, pos, types, nl, s);
        else launch_desc<K, S, false, true>(dm, dn, pos, types, nl, s);
    } else if (forward && dm.rtab)
        launch_desc<K, S, true, false>(dm, dn, pos, types, nl, s);
    else if (forward)
        launch_desc<K, S, false, false>(dm, dn, pos, types, nl, s);
    else if (w_atom && dm.rtab)   // batched evaluations always run with the pair cache
        launch_force<K, S, true, true, true>(dm, dn, pos, types, nl, part_w, nblk, s, w_atom);
    else if (w_atom)
        launch_force<K, S, true, true, false>(dm, dn, pos, types, nl, part_w, nblk, s, w_atom);
    // the tensor-core pass reads the pair cache; an evaluation without one
    // (the allocation-free call) runs the SIMT pass whatever the setting
    else if (force_kernel() == TMD_FORCE_TENSOR && dn.pq && !(!dm.rtab && S == 1 && K <= 32)) {
        set_error("the tensor-core force pass needs one species, K <= 32 and the direct radial basis");
        return TMD_ERR_UNIMPLEMENTED;
    } else if (force_kernel() == TMD_FORCE_TENSOR && dn.pq) {
        if constexpr (S == 1 && K <= 32)
            TMD_LAUNCH("k_force", s, k_force_tc<K><<<nblk, PW * 32, 0, s>>>(dm, dn, nl->P, nl->dG, nl->Fq, part_w));
    } else if (dn.pq && dm.rtab) {
        if constexpr (S == 1)
            TMD_LAUNCH("k_force", s, k_force_merged<K, S, true><<<nblk, PW * 32, 0, s>>>(dm, dn, types, nl->P, nl->dG,
                                                                                       nl->Fq, part_w));
        else
            launch_force<K, S, false, true, true>(dm, dn, pos, types, nl, part_w, nblk, s, nullptr);
    } else if (dn.pq) {
        if constexpr (S == 1)
            TMD_LAUNCH("k_force", s, k_force_merged<K, S, false><<<nblk, PW * 32, 0, s>>>(dm, dn, types, nl->P, nl->dG,
                                                                                        nl->Fq, part_w));
        else
            launch_force<K, S, false, true, false>(dm, dn, pos, types, nl, part_w, nblk, s, nullptr);
    }
    else if (dm.rtab)
        launch_force<K, S, false, false, true>(dm, dn, pos, types, nl, part_w, nblk, s, nullptr);
    else
        launch_force<K, S, false, false, false>(dm, dn, pos, types, nl, part_w, nblk, s, nullptr);
    TMD_CUDA(cudaGetLastError());
    return TMD_OK;
}

}  // namespace

}  // namespace tmd
