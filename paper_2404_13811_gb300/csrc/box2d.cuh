// Device building blocks of the 2D local solves, shared by the forward
// kernels (local2d.cu) and their adjoints (adjoint2d.cu): the box and its
// cell-centred RT0 operator (Sec. 2.2), the block LDL^T factorisation over
// grid lines, warp-level solves (FP64, or FP32 sweeps with FP64 residual
// refinement), right-hand-side generators and the bulk-copy helpers.
#pragma once
#include "mrcm_internal.cuh"
#include <type_traits>

namespace {

constexpr int NWARP = 4;

// FP32 normal range of an FP64 value, from its exponent bits (integer pipe).
__device__ __forceinline__ bool in_f32_range(double x) {
    const unsigned e11 = ((unsigned)__double2hiint(x) >> 20) & 0x7ffu;
    return e11 >= 1023u - 126u && e11 <= 1023u + 126u;   // 2^-126 <= |x| < 2^127
}

// 1/x in FP64 by Newton-Raphson iteration for the reciprocal, r <- r (2 - x r),
// from the correctly rounded FP32 reciprocal of x: each step squares the
// relative error (about 2^-23 for the seed, below the FP64 rounding after two
// steps), without the FP64 division.  Outside the FP32 normal range the seed
// would be 0 or infinite, and the FP64 division is used.
__device__ __forceinline__ double rcp64(double x) {
    if (!in_f32_range(x)) return 1.0 / x;
    double r = (double)__frcp_rn((float)x);
    r = r * (2.0 - x * r);
    r = r * (2.0 - x * r);
    return r;
}

// Box description shared by all threads of a CTA.
struct Box {
    int lo[2], hi[2];
    int nx, ny, n;
    int kind[4];      // 0 Neumann, 1 Dirichlet, 2 Robin
    double val[4];    // physical data (g or z)
    double alpha;
    double rlen[4];   // 1 / (faces on the side)
};

// side offsets into the per-side boundary arrays: x sides have ny faces,
// y sides have nx faces.
__device__ __forceinline__ int side_off(const Box& B, int sid) {
    return sid == 0 ? 0 : sid == 1 ? B.ny : sid == 2 ? 2 * B.ny : 2 * B.ny + B.nx;
}

// P0: 1; P1: affine coordinate of the face centre along the side, in [-1, 1].
__device__ __forceinline__ double psi_val(int m, int pos, int len, double rlen) {
    return m == 0 ? 1.0 : (double)(2 * pos + 1 - len) * rlen;
}

// Shared-memory copy of the box operator.
struct Ops {
    double* cd;   // diagonal
    double* cx;   // coupling of cell (i, j) with (i + 1, j)
    double* cy;   // coupling of cell (i, j) with (i, j + 1)
    double* hk;   // h / (2K) per cell, x and y interleaved [2n]
    double* bT;   // boundary-face transmissibility per side
    double* bB;   // Robin beta per side
    double* dsc;  // Jacobi scale (1 in the FP64 form)
};

// Loads the face coefficients of the box and forms the boundary faces.
__device__ void build_ops(const Box& B, const MemberDev& md, const DevPtrs& P, Ops& O) {
    const double* Tf = P.Tf + md.cell_off * 3;
    const double* hkg = P.hk + md.cell_off * 3;
    const double* wh = P.wh + md.cell_off * 3;
    const int nxg = md.n[0];
    for (int c = threadIdx.x; c < B.n; c += blockDim.x) {
        const int i = c % B.nx, j = c / B.nx;
        const long long g = (B.lo[0] + i) + (long long)nxg * (B.lo[1] + j);
        O.cx[c] = i < B.nx - 1 ? Tf[g * 3 + 0] : 0.0;
        O.cy[c] = j < B.ny - 1 ? Tf[g * 3 + 1] : 0.0;
        if (O.hk) {   // null where the kernel reads h / 2K from global memory
            O.hk[2 * c] = hkg[g * 3 + 0];
            O.hk[2 * c + 1] = hkg[g * 3 + 1];
        }
    }
    const double ax = md.h[1], ay = md.h[0];  // face areas (normal to x, normal to y)
    for (int sid = 0; sid < 4; ++sid) {
        const int a = sid >> 1;
        const int len = a == 0 ? B.ny : B.nx;
        const double area = a == 0 ? ax : ay;
        const int off = side_off(B, sid);
        for (int pos = threadIdx.x; pos < len; pos += blockDim.x) {
            int i, j;
            if (a == 0) { j = pos; i = (sid == 0) ? 0 : B.nx - 1; }
            else        { i = pos; j = (sid == 2) ? 0 : B.ny - 1; }
            const long long g = (B.lo[0] + i) + (long long)nxg * (B.lo[1] + j);
            const double hin = hkg[g * 3 + a];
            double T = 0.0, beta = 0.0;
            if (B.kind[sid] == 2) {
                // the face to the outside cell: owned by the lower of the two cells
                const long long gf = (sid & 1) ? g : g - (a == 0 ? 1 : nxg);
                beta = B.alpha * wh[gf * 3 + a];
                T = area * rcp64(hin + beta);
            } else if (B.kind[sid] == 1) {
                T = area * rcp64(hin);
            }
            O.bT[off + pos] = T;
            O.bB[off + pos] = beta;
        }
    }
    __syncthreads();
    for (int c = threadIdx.x; c < B.n; c += blockDim.x) {
        const int i = c % B.nx, j = c / B.nx;
        double d = O.cx[c] + O.cy[c];
        if (i > 0) d += O.cx[c - 1];
        if (j > 0) d += O.cy[c - B.nx];
        if (i == 0) d += O.bT[side_off(B, 0) + j];
        if (i == B.nx - 1) d += O.bT[side_off(B, 1) + j];
        if (j == 0) d += O.bT[side_off(B, 2) + i];
        if (j == B.ny - 1) d += O.bT[side_off(B, 3) + i];
        O.cd[c] = d;
    }
    __syncthreads();
}

// --- FP32 <-> FP64 conversions on the integer pipe ---------------------------
// On GB300 every FP64-pipe warp instruction, conversions included, occupies
// the sub-partition's FP64 unit for 64 cycles, and the refinement of the
// mixed form converts twice per cell and step; these do it with integer
// operations instead.  FP32 -> FP64 is exact for normal numbers and zero
// (FP32 subnormals are flushed to zero; infinities and NaN keep their class).
// FP64 -> FP32 truncates the mantissa -- it serves only the right-hand side
// of a correction solve, where an error below one FP32 ulp is immaterial --
// flushes results below the FP32 normal range to zero and takes larger ones
// to infinity (NaN stays NaN).  ex: the FP32 value stands for f 2^-ex.
__device__ __forceinline__ double f2d_bits(float f, int ex = 0) {
    const unsigned u = __float_as_uint(f);
    const unsigned e = (u >> 23) & 0xffu;
    const unsigned hs = u & 0x80000000u;
    const unsigned e11 = e == 0xffu ? 0x7ffu : e + (unsigned)(896 - ex);
    const unsigned hi = e == 0u ? hs : (hs | (e11 << 20) | ((u & 0x7fffffu) >> 3));
    const unsigned lo = e == 0u ? 0u : (u << 29);
    return __hiloint2double((int)hi, (int)lo);
}
__device__ __forceinline__ float d2f_bits(double d, int ex = 0) {
    const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
    const unsigned s = hi & 0x80000000u;
    const int e11 = (int)((hi >> 20) & 0x7ffu);
    const int e = e11 - 896 + ex;
    const unsigned m = ((hi & 0xfffffu) << 3) | (lo >> 29);
    unsigned r = s | ((unsigned)e << 23) | m;
    if (e <= 0) r = s;
    if (e >= 255) r = s | 0x7f800000u | ((e11 == 0x7ff && ((hi & 0xfffffu) | lo)) ? 0x400000u : 0u);
    return __uint_as_float(r);
}

// The exponent ex that takes a vector of FP64 values to FP32 values of at most
// 2 in magnitude, from the largest high word of the values (without signs).  A
// refinement follows its right-hand side down by twelve or more digits, and
// residuals below the FP32 normal range, flushed to zero, would count as
// converged: with right-hand sides of 1e-30 the result is off by 1e-7.
__device__ __forceinline__ unsigned abs_hi(double d) { return (unsigned)__double2hiint(d) & 0x7fffffffu; }
__device__ __forceinline__ int norm_shift(unsigned hmax) { return max(-896, min(896, 1023 - (int)(hmax >> 20))); }

// d2f_bits rounded to nearest (ties away from zero): for values that stay in the
// factor, where truncation would shift every pivot the same way.
__device__ __forceinline__ float d2f_near(double d, int ex = 0) {
    const unsigned t = __float_as_uint(d2f_bits(d, ex));
    const unsigned e = (t >> 23) & 0xffu;
    return __uint_as_float(e - 1u < 254u ? t + (((unsigned)__double2loint(d) >> 28) & 1u) : t);
}

// The mixed form refines in Jacobi-scaled variables: O holds D A D (D =
// diag(dsc)) after scale_ops, the iterate is x~ = D^-1 x and the right-hand
// side b~ = D b, so that a residual b~ - (D A D) x~ is five FP64 FMAs per cell
// and an update one FP64 add.  The FP64 form keeps D = I and A.
__device__ void scale_ops(const Box& B, Ops& O) {
    for (int c = threadIdx.x; c < B.n; c += blockDim.x) {
        const int i = c % B.nx, j = c / B.nx;
        const double d = O.dsc[c];
        O.cx[c] = i < B.nx - 1 ? O.cx[c] * d * O.dsc[c + 1] : 0.0;
        O.cy[c] = j < B.ny - 1 ? O.cy[c] * d * O.dsc[c + B.nx] : 0.0;
        O.cd[c] = O.cd[c] * d * d;
    }
    __syncthreads();
}

// b~_c - ((D A D) x~)_c with O scaled.
__device__ __forceinline__ double resid_sc(const Box& B, const Ops& O, const double* x, double bt, int c, int i,
                                           int j) {
    double s = fma(-O.cd[c], x[c], bt);
    if (i > 0) s = fma(O.cx[c - 1], x[c - 1], s);
    if (i < B.nx - 1) s = fma(O.cx[c], x[c + 1], s);
    if (j > 0) s = fma(O.cy[c - B.nx], x[c - B.nx], s);
    if (j < B.ny - 1) s = fma(O.cy[c], x[c + B.nx], s);
    return s;
}

// ---------------------------------------------------------------------------
// Twisted block LDL^T over the grid lines of a box.
//
// The Jacobi-scaled operator is block tridiagonal over its nb lines of b
// cells: diagonal blocks T_j (the couplings inside line j) and off-diagonal
// blocks -C_j, C_j = diag(cys_j), between lines j and j + 1.  It is factored
// from both ends towards the middle line m = nb / 2 (a twisted, or
// burn-at-both-ends, block factorisation):
//   top     S_j = T_j - C_{j-1} S_{j-1}^-1 C_{j-1},                j = 0 .. m - 1
//   bottom  R_j = T_j - C_j R_{j+1}^-1 C_j,                        j = nb - 1 .. m + 1
//   middle  M   = T_m - C_{m-1} S_{m-1}^-1 C_{m-1} - C_m R_{m+1}^-1 C_m
// and S_j^-1 (j < m), M^-1 (j = m), R_j^-1 (j > m) are kept in line order.
// A solve runs two half-length sweeps from the ends, meeting at line m:
//   forward  y_j = S_j^-1 (b_j + C_{j-1} y_{j-1}),  y_j = R_j^-1 (b_j + C_j y_{j+1})
//   middle   x_m = M^-1 (b_m + C_{m-1} y_{m-1} + C_m y_{m+1})
//   back     x_j = y_j + S_j^-1 C_j x_{j+1},        x_j = y_j + R_j^-1 C_{j-1} x_{j-1}
// The blocks are those of a one-sided block LDL^T in another elimination
// order.  The two chains of a solve run interleaved on one warp (a step
// issues both chains' line products, which costs little more than one), so
// a solve is nb / 2 + 1 dependent steps instead of 2 nb - 1; the two chains
// of the factorisation run on two warps (nb / 2 + 1 line inversions in a
// chain instead of nb).
//
// Storage: block j of lines of b cells at j b ld, row-major with row stride
// ld = sld(bp), bp the line width.  FP32 lines are widened to bp, the next
// multiple of 4 (entries beyond b are zero, and so are the entries of a line's
// input there), so that every row is read as float4 by one lane, at any b;
// rows of bp floats with bp / 4 even would put the rows of lanes i and i + 4
// (or closer) of an 8-lane phase in one bank group, so they are padded by four
// floats (then ld / 4 is odd and the eight rows start in distinct groups).
// The line couplings cys are kept with bp entries a line.  FP64 blocks are
// read by column (no widening, no padding), as are FP32 ones of a handle whose
// boxes would not fit shared memory with widened lines (pad = 0): one warp by
// column takes about twice as long per sweep as two by row.
// ---------------------------------------------------------------------------
__host__ __device__ constexpr int sld_of(int bp, int tsz) {
    return (tsz == 4 && bp % 4 == 0 && (bp / 4) % 2 == 0) ? bp + 4 : bp;
}
template <typename T>
__host__ __device__ constexpr int sld(int bp) { return sld_of(bp, (int)sizeof(T)); }
// line width of lines of b cells
__host__ __device__ constexpr int line_width(int b, int tsz, int pad) { return tsz == 4 && pad ? (b + 3) & ~3 : b; }
__host__ __device__ inline size_t sinv_len(int nx, int ny, int tsz, int pad) {
    return (size_t)ny * nx * sld_of(line_width(nx, tsz, pad), tsz);
}

// In-register Gauss-Jordan inverse of an SPD b x b block (row i in lane i),
// SPD so no pivoting.  The pivot row reaches every lane by shuffles from lane
// k; the pivot lane and the other lanes update with selects (no divergent
// paths), so a step is one chain of b shuffles and b FMAs.  Pivot
// reciprocals: the correctly rounded FP32 reciprocal in the FP32 form, FP64
// otherwise.  EX: BW is the line width (lanes and entries beyond b hold the
// identity); else b <= BW.
template <typename T, int BW, bool EX>
__device__ __forceinline__ void gj_regs(T (&a)[BW], int b, int* bad) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int k = 0; k < BW; ++k) {
        if (EX || k < b) {
            T rv[BW];
#pragma unroll
            for (int c = 0; c < BW; ++c) rv[c] = __shfl_sync(0xffffffffu, a[c], k);
            T piv = rv[k];
            if (!(piv > T(0))) {
                if (lane == 0) *bad = 1;
                piv = T(1);
            }
            T ip;
            if constexpr (std::is_same<T, float>::value) ip = __frcp_rn(piv);
            else ip = rcp64(piv);
            const bool isk = lane == k;
            const T f = a[k] * ip;
            const T ck = isk ? ip : -f;
            if constexpr (std::is_same<T, float>::value) {
                // FP32 form (Jacobi-scaled, so 0 < piv <= 1 and |1 - ip| <= ip):
                // one FMA per entry and no select -- the other lanes compute
                // a - f rv, the pivot lane, whose row is rv, rv - (1 - ip) rv = ip rv
                const T fl = isk ? T(1) - ip : f;
#pragma unroll
                for (int c = 0; c < BW; ++c) a[c] = (c == k) ? ck : a[c] - fl * rv[c];
            } else {
                // FP64 form (unscaled pivots of any size): the pivot lane computes
                // 0 - (-ip) rv = ip rv, the others a - f rv
                const T fl = isk ? -ip : f;
#pragma unroll
                for (int c = 0; c < BW; ++c) {
                    const T base = isk ? T(0) : a[c];
                    a[c] = (c == k) ? ck : base - fl * rv[c];
                }
            }
        }
    }
}

// Line block j of the twisted factorisation in registers (lane i holds row
// i): T_j minus C S^-1 C for each kept neighbour inverse given (up: the
// inverse of line j - 1, coupled through cys_{j-1}; dn: the inverse of line
// j + 1, coupled through cys_j).  Off-diagonal entries in T, the diagonal
// d_i - sum c_i^2 (S^-1)_ii -- where the cancellation is -- in FP64.  With
// the width known at compile time (EX, FP32) lane i reads row i of the
// (symmetric) neighbour inverse and the coupling vector as float4 and the
// FP64 diagonal converts on the integer pipe (FP32 -> FP64 exact, the FP64
// result truncated to FP32 within one ulp, or rounded to nearest in widened
// lines); otherwise lane i reads column i.
template <typename T, int BW, bool EX, bool SC>
__device__ __forceinline__ void form_line(T (&a)[BW], const Ops& O, const T* cys, const T* cxs, int b, int ld,
                                          int j, const T* up, const T* dn) {
    if constexpr (EX) ld = sld<T>(BW);
    const int cs = EX ? BW : b;   // line stride of cys
    const int i = threadIdx.x & 31;
    const bool act = i < b;
    const int ii = act ? i : 0;
    const int ci = j * b + ii;
    const T cu = up ? cys[(j - 1) * cs + ii] : T(0);
    const T cn = dn ? cys[j * cs + ii] : T(0);
    // in-line couplings of cell i: to i + 1 and to i - 1
    const T xr = (act && ii < b - 1) ? cxs[ci] : T(0);
    const T xl = (act && ii > 0) ? cxs[ci - 1] : T(0);
    constexpr bool VEC = EX && std::is_same<T, float>::value && (BW % 4 == 0);
    double d = SC ? O.cd[ci] : O.cd[ci] * O.dsc[ci] * O.dsc[ci];
    if constexpr (VEC) {
        const double cu2 = up ? f2d_bits(cu) * f2d_bits(cu) : 0.0;   // exact in FP64
        const double cn2 = dn ? f2d_bits(cn) * f2d_bits(cn) : 0.0;
        if (up) d = fma(-cu2, f2d_bits(up[ii * ld + ii]), d);
        if (dn) d = fma(-cn2, f2d_bits(dn[ii * ld + ii]), d);
    } else {
        // c (c S_ii), not c^2 S_ii: c^2 leaves the FP64 range for couplings
        // below ~1e-154 (permeabilities scaled that far), c S_ii does not
        if (up) d -= (double)cu * ((double)cu * (double)up[ii * ld + ii]);
        if (dn) d -= (double)cn * ((double)cn * (double)dn[ii * ld + ii]);
    }
    T dT;
    if constexpr (VEC) dT = b < BW ? d2f_near(d) : d2f_bits(d);
    else dT = (T)d;
    if constexpr (VEC) {
        constexpr int NQ = BW / 4;
        float4 ru[NQ], rd[NQ], ku[NQ], kd[NQ];
        if (up) {
            const float4* r = reinterpret_cast<const float4*>(up + ii * ld);
            const float4* k = reinterpret_cast<const float4*>(cys + (j - 1) * BW);
#pragma unroll
            for (int q = 0; q < NQ; ++q) { ru[q] = r[q]; ku[q] = k[q]; }
        }
        if (dn) {
            const float4* r = reinterpret_cast<const float4*>(dn + ii * ld);
            const float4* k = reinterpret_cast<const float4*>(cys + j * BW);
#pragma unroll
            for (int q = 0; q < NQ; ++q) { rd[q] = r[q]; kd[q] = k[q]; }
        }
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            float su[4] = {0.f, 0.f, 0.f, 0.f}, sd[4] = {0.f, 0.f, 0.f, 0.f};
            if (up) {
                su[0] = cu * ru[q].x * ku[q].x; su[1] = cu * ru[q].y * ku[q].y;
                su[2] = cu * ru[q].z * ku[q].z; su[3] = cu * ru[q].w * ku[q].w;
            }
            if (dn) {
                sd[0] = cn * rd[q].x * kd[q].x; sd[1] = cn * rd[q].y * kd[q].y;
                sd[2] = cn * rd[q].z * kd[q].z; sd[3] = cn * rd[q].w * kd[q].w;
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int c = 4 * q + e;
                const float off = (c == i + 1 ? xr : c == i - 1 ? xl : 0.f) - su[e] - sd[e];
                a[c] = act ? (c == i ? dT : off) : T(i == c ? 1 : 0);
            }
        }
    } else {
#pragma unroll
        for (int c = 0; c < BW; ++c) {
            T s = T(0);
            if (act && (EX || c < b)) {
                s = c == i + 1 ? xr : c == i - 1 ? xl : T(0);
                // by column (consecutive lanes, consecutive words) where rows are not read as float4
                if (up) s -= cu * up[c * ld + ii] * cys[(j - 1) * cs + c];
                if (dn) s -= cn * dn[c * ld + ii] * cys[j * cs + c];
            }
            a[c] = (act && (EX || c < b)) ? (c == i ? dT : s) : T(i == c ? 1 : 0);
        }
    }
}

// Stores the inverse held in registers (lane i, entry c) as entry (c, i) of
// the row-major block (consecutive lanes, consecutive words); the inverse of
// an SPD block is symmetric, so this is the block up to rounding.  Widened
// FP32 lines (b < BW): by rows, as float4.  There the sweeps then apply the
// inverse as computed, and the diagonal is rounded to nearest, as where lines
// of such widths are read by column: transposed and truncated, the fluxes of a
// 225 x 192 field in boxes of 18 and 21 cells came out two to four times
// further from the exact ones at the same ir_tol (1.2e-11 and 2.8e-11 with
// only the rows, 1.2e-11 with both).  Lines of full width keep theirs: with both
// changed the 512x512 step took 3403 instead of 3374 us, at 6.8e-11 from the
// exact fluxes instead of 4.0e-11.
template <typename T, int BW, bool EX>
__device__ __forceinline__ void store_line(const T (&a)[BW], T* S, int b, int ld) {
    if constexpr (EX) ld = sld<T>(BW);
    const int i = threadIdx.x & 31;
    if constexpr (EX && std::is_same<T, float>::value && BW % 4 == 0) {
        if (b < BW) {
            if (i >= b) return;
            float4* r = reinterpret_cast<float4*>(S + i * ld);
#pragma unroll
            for (int q = 0; q < BW / 4; ++q) r[q] = make_float4(a[4 * q], a[4 * q + 1], a[4 * q + 2], a[4 * q + 3]);
            return;
        }
    }
    if (i < b) {
#pragma unroll
        for (int c = 0; c < BW; ++c)
            if (c < b) S[c * ld + i] = a[c];
    }
}

// 1 / v for the pivots.  FP32: correctly rounded.  FP64: from the FP32 seed r one third-order step,
// r + r (e + e^2) with e = 1 - v r (e is about 2^-22, the error left e^3); the
// conversions on the integer pipe.  The division outside the FP32 normal range,
// and from 2^126 on, where the seed would be subnormal and flushed to zero.
__device__ __forceinline__ float rcp_piv(float v) { return __frcp_rn(v); }
__device__ __forceinline__ double rcp_piv(double v) {
    const unsigned e11 = ((unsigned)__double2hiint(v) >> 20) & 0x7ffu;
    if (e11 < 1023u - 126u || e11 > 1023u + 125u) return 1.0 / v;
    const double r = f2d_bits(__frcp_rn(d2f_bits(v)));
    const double e = fma(-v, r, 1.0);
    return fma(r, fma(e, e, e), r);
}

// The FP64 form of the twisted factorisation for lines of 12 to 28 cells
// (four warps).  Two warps run each chain: a line block is held as the 4 x 4
// tiles (I, J), I <= J, of its upper triangle -- in-place Gauss-Jordan keeps
// M_IJ = +-M_JI^T, minus when exactly one of I, J has been eliminated -- tile t
// in lane t, rows 0-1 of it in the chain's first warp and rows 2-3 in the
// second.  Pivots go by blocks K of 4: the panel M_K. and its product with the
// inverse pivot block P = M_KK^-1 pass through shared memory (in the block's
// own storage, which is written only once the line is done), each warp
// inverts the next pivot block with an entry per lane while its tiles are
// updated.  The inverse of the last line stays in the registers, where the
// next one is formed from it.
// Bound by the FP64 pipe (a warp instruction takes 64 cycles of its quarter of
// the SM).  With one warp per chain, whole rows, a shuffle per entry and the
// full square a line of 24 cells took 70k cycles.
constexpr int F64_MIN = 12, F64_MAX = 28;

__device__ __forceinline__ void bar_pair(int id) { asm volatile("bar.sync %0, 64;" ::"r"(id) : "memory"); }

__device__ void factor_box64(const Box& B, const Ops& O, double* Sinv, const double* cys, const double* cxs, int* bad) {
    const int b = B.nx, nb = B.ny, nb4 = (b + 3) >> 2, bp = 4 * nb4, m = nb >> 1;
    const int bl = b * b;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int h = warp >> 1, y0 = 2 * (warp & 1);   // chain; first tile row of this warp
    const bool act = lane < nb4 * (nb4 + 1) / 2;
    int I = 0, J = lane;
    if (act) {
        while (J >= nb4 - I) {
            J -= nb4 - I;
            ++I;
        }
        J += I;
    } else {
        I = J = -4;
    }
    const int py = (lane >> 2) & 3, px = lane & 3;   // entry of a pivot block held by this lane
    double V[2][4];
#pragma unroll
    for (int y = 0; y < 2; ++y)
#pragma unroll
        for (int x = 0; x < 4; ++x) V[y][x] = 0.0;
    auto invert = [&](double v) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            double piv = __shfl_sync(0xffffffffu, v, 5 * q);
            if (!(piv > 0.0)) {
                if (lane == 0) *bad = 1;
                piv = 1.0;
            }
            const double ip = rcp_piv(piv);
            const double r = __shfl_sync(0xffffffffu, v, 4 * q + px), c = __shfl_sync(0xffffffffu, v, 4 * py + q);
            const double rp = px == q ? ip : r * ip;
            v = py == q ? rp : (px == q ? 0.0 : v) - c * rp;
        }
        return v;
    };
    // line block j in V (from the last inverse in V when up, minus the kept inverse dn of line j + 1 for the middle
    // line), its inverse in V and in Sinv
    auto line = [&](int j, bool chained, int jc, const double* dn) {
        double* S = Sinv + (size_t)j * bl;
        double* R = S;             // [4][bp]
        double* Rn = S + 4 * bp;   // [4][bp]
        double* D = S + 8 * bp;    // [16] the next pivot block before this block's update
        if (act) {
#pragma unroll
            for (int y = 0; y < 2; ++y) {
                const int i = 4 * I + y0 + y;
                const double ci = (chained && i < b) ? cys[jc * b + i] : 0.0;
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    const int k = 4 * J + x;
                    double s;
                    if (i >= b || k >= b) {
                        s = i == k ? 1.0 : 0.0;   // padding: the identity
                    } else {
                        const double vs = V[y][x];
                        if (i == k) {
                            // c (c S_ii), not c^2 S_ii (range at tiny couplings)
                            s = O.cd[j * b + i] * O.dsc[j * b + i] * O.dsc[j * b + i];
                            if (chained) s -= ci * (ci * vs);
                        } else {
                            s = chained ? -(ci * vs * cys[jc * b + k]) : 0.0;
                            if (k == i + 1) s += cxs[j * b + i];
                            if (k == i - 1) s += cxs[j * b + k];
                        }
                        if (dn) s -= cys[j * b + i] * dn[i * b + k] * cys[j * b + k];
                    }
                    V[y][x] = s;
                }
            }
        }
        double p = 0.0;
#pragma unroll 1
        for (int k = 0; k < nb4; ++k) {
            if (I == k) {
#pragma unroll
                for (int y = 0; y < 2; ++y)
#pragma unroll
                    for (int x = 0; x < 4; ++x) R[(y0 + y) * bp + 4 * J + x] = V[y][x];
            } else if (J == k) {
                // I < k has been eliminated: M_kI = -M_Ik^T
#pragma unroll
                for (int y = 0; y < 2; ++y)
#pragma unroll
                    for (int x = 0; x < 4; ++x) R[x * bp + 4 * I + y0 + y] = -V[y][x];
            }
            if (I == k + 1 && J == k + 1) {
#pragma unroll
                for (int y = 0; y < 2; ++y)
#pragma unroll
                    for (int x = 0; x < 4; ++x) D[4 * (y0 + y) + x] = V[y][x];
            }
            bar_pair(2 + h);
            if (k == 0) p = invert(R[py * bp + px]);
            {
                // rows y0, y0 + 1 of P M_k., column `lane`
                const int c = lane < bp ? lane : 0;
                const double r0 = R[c], r1 = R[bp + c], r2 = R[2 * bp + c], r3 = R[3 * bp + c];
#pragma unroll
                for (int y = 0; y < 2; ++y) {
                    const int s = 4 * (y0 + y);
                    const double q0 = __shfl_sync(0xffffffffu, p, s), q1 = __shfl_sync(0xffffffffu, p, s + 1);
                    const double q2 = __shfl_sync(0xffffffffu, p, s + 2), q3 = __shfl_sync(0xffffffffu, p, s + 3);
                    const double own = __shfl_sync(0xffffffffu, p, s + (c & 3));
                    const double v = (q0 * r0 + q1 * r1) + (q2 * r2 + q3 * r3);
                    if (lane < bp) Rn[(y0 + y) * bp + c] = (c >> 2) == k ? own : v;
                }
            }
            bar_pair(2 + h);
            if (k + 1 < nb4) {
                // the next pivot block, updated here and inverted
                const int c = 4 * (k + 1);
                double v = D[lane & 15];
#pragma unroll
                for (int q = 0; q < 4; ++q) v -= R[q * bp + c + py] * Rn[q * bp + c + px];
                p = invert(v);
            }
            if (I == k) {
#pragma unroll
                for (int y = 0; y < 2; ++y)
#pragma unroll
                    for (int x = 0; x < 4; ++x) V[y][x] = Rn[(y0 + y) * bp + 4 * J + x];
            } else if (J == k) {
#pragma unroll
                for (int y = 0; y < 2; ++y)
#pragma unroll
                    for (int x = 0; x < 4; ++x) V[y][x] = Rn[x * bp + 4 * I + y0 + y];
            } else if (act) {
                // V -= M_IK (P M_KJ), M_IK = R^T where I is not eliminated yet, else -R^T
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    double a[2];
#pragma unroll
                    for (int y = 0; y < 2; ++y) {
                        a[y] = R[q * bp + 4 * I + y0 + y];
                        a[y] = I > k ? -a[y] : a[y];
                    }
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        const double r = Rn[q * bp + 4 * J + x];
#pragma unroll
                        for (int y = 0; y < 2; ++y) V[y][x] = fma(a[y], r, V[y][x]);
                    }
                }
            }
            bar_pair(2 + h);
        }
        if (act) {
#pragma unroll
            for (int y = 0; y < 2; ++y)
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    const int i = 4 * I + y0 + y, k = 4 * J + x;
                    if (i < b && k < b) {
                        S[i * b + k] = V[y][x];
                        if (I != J) S[k * b + i] = V[y][x];
                    }
                }
        }
    };
    const int cnt = h == 0 ? m : nb - 1 - m;
    for (int s = 0; s < cnt; ++s) {
        const int j = h == 0 ? s : nb - 1 - s;
        line(j, s > 0, h == 0 ? j - 1 : j, nullptr);
    }
    __syncthreads();
    if (h == 0) line(m, m > 0, m - 1, m < nb - 1 ? Sinv + (size_t)(m + 1) * bl : nullptr);
    __syncthreads();
}

// Twisted block LDL^T factorisation: Sinv[j] as above.  cys / cxs: the scaled
// line / in-line couplings (type T, formed once by all threads).  Warp 0
// runs the top chain and then the middle line, warp 1 the bottom chain.
// EX: the line width is BW.
template <typename T, int BW, bool EX, bool SC = false>
__device__ void factor_box(const Box& B, const Ops& O, T* Sinv, T* cys, T* cxs, int* bad) {
    const int b = B.nx, nb = B.ny;
    const int ld = sld<T>(EX ? BW : b);
    const size_t bl = (size_t)b * ld;
    const int tid = threadIdx.x, nt = blockDim.x;
    const int cs = EX ? BW : b;   // line stride of cys
    for (int c = tid; c < B.n; c += nt) {
        const int cj = c / b, ci = c - cj * b;
        if (SC) {   // the operator is scaled already (scale_ops)
            cys[cj * cs + ci] = (T)O.cy[c];
            cxs[c] = (T)(-O.cx[c]);
        } else {
            cys[cj * cs + ci] = (T)(O.cy[c] * O.dsc[c] * ((c + b < B.n) ? O.dsc[c + b] : 0.0));
            cxs[c] = (T)(-O.cx[c] * O.dsc[c] * (ci < b - 1 ? O.dsc[c + 1] : 0.0));
        }
    }
    if (EX && b < BW)
        for (int t = tid; t < nb * (BW - b); t += nt) cys[(t / (BW - b)) * BW + b + t % (BW - b)] = T(0);
    __syncthreads();
    if constexpr (std::is_same<T, double>::value && BW >= 16) {
        if (b >= F64_MIN && b <= F64_MAX && blockDim.x == 128) {
            factor_box64(B, O, Sinv, cys, cxs, bad);
            return;
        }
    }
    const int warp = tid >> 5;
    const int m = nb >> 1;
    if (warp < 2) {
        const bool top = warp == 0;
        const int cnt = top ? m : nb - 1 - m;
        for (int s = 0; s < cnt; ++s) {
            const int j = top ? s : nb - 1 - s;
            T a[BW];
            form_line<T, BW, EX, SC>(a, O, cys, cxs, b, ld, j, (top && j > 0) ? Sinv + (j - 1) * bl : nullptr,
                                 (!top && j < nb - 1) ? Sinv + (j + 1) * bl : nullptr);
            gj_regs<T, BW, EX>(a, b, bad);
            store_line<T, BW, EX>(a, Sinv + j * bl, b, ld);
            __syncwarp();
        }
    }
    __syncthreads();
    if (warp == 0) {
        T a[BW];
        form_line<T, BW, EX, SC>(a, O, cys, cxs, b, ld, m, m > 0 ? Sinv + (m - 1) * bl : nullptr,
                             m < nb - 1 ? Sinv + (m + 1) * bl : nullptr);
        gj_regs<T, BW, EX>(a, b, bad);
        store_line<T, BW, EX>(a, Sinv + m * bl, b, ld);
    }
    __syncthreads();
}

// --- line products of the sweeps --------------------------------------------
// FP32, line width BB known at compile time (a multiple of 4): lane i holds
// row i of a block as BB / 4 float4, loaded before the line's input is ready;
// the line input is read back as float4 broadcasts; four accumulators.
template <int BB>
struct RowF {
    static constexpr int LD = sld<float>(BB), NQ = BB / 4;
    float4 s[NQ];
    // a row of a narrower line width (nq < NQ groups of 4, row stride ld)
    __device__ __forceinline__ void load(const float* __restrict__ S, int lane, int nq, int ld) {
        const float4* r = reinterpret_cast<const float4*>(S + lane * ld);
#pragma unroll
        for (int q = 0; q < NQ; ++q) s[q] = q < nq ? r[q] : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __device__ __forceinline__ void load(const float* __restrict__ S, int lane) {
        const float4* r = reinterpret_cast<const float4*>(S + (lane < BB ? lane : 0) * LD);
#pragma unroll
        for (int q = 0; q < NQ; ++q) s[q] = r[q];
    }
    // row . z, entry k of z in lane k
    __device__ __forceinline__ float dot(float z) const {
        float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            a0 += s[q].x * __shfl_sync(0xffffffffu, z, 4 * q);
            a1 += s[q].y * __shfl_sync(0xffffffffu, z, 4 * q + 1);
            a2 += s[q].z * __shfl_sync(0xffffffffu, z, 4 * q + 2);
            a3 += s[q].w * __shfl_sync(0xffffffffu, z, 4 * q + 3);
        }
        return (a0 + a1) + (a2 + a3);
    }
};

// Any width and type: lane i reads column i by scalar loads (the block is
// symmetric up to rounding), two accumulators.
template <typename T>
__device__ __forceinline__ T dot_col(const T* __restrict__ S, const T* z, int b, int ld, int lane) {
    T a0 = T(0), a1 = T(0);
    if (lane < b) {
        int k = 0;
        for (; k + 1 < b; k += 2) {
            a0 += S[k * ld + lane] * z[k];
            a1 += S[(k + 1) * ld + lane] * z[k + 1];
        }
        if (k < b) a0 += S[k * ld + lane] * z[k];
    }
    return a0 + a1;
}

// Both twisted sweeps by one warp, the two chains interleaved step by step.
// w: the scaled right-hand side in, the scaled solution out (line-major, b
// per line); z: 64 entries (two line inputs), 16-byte aligned.  BB > 0: the
// FP32 row path for lines of width BB; BB = 0: the column path for any b.
// Steps where both chains have a line run as one unit (both products in one
// loop, so the loads and FMAs of the two chains overlap); the top chain has
// at most one line more than the bottom one, run alone at the end.
template <typename T, int BB>
__device__ void tw_warp(const T* __restrict__ Sinv, const T* __restrict__ cys, T* w, T* z, int b, int nb) {
    const int cs = BB > 0 ? BB : b;   // line stride of cys
    using Row = RowF<(BB > 0 ? BB : 4)>;
    const int ld = BB > 0 ? Row::LD : sld<T>(b);
    const int lane = threadIdx.x & 31;
    const bool act = lane < b;
    const size_t bl = (size_t)b * ld;
    const int m = nb >> 1, ntop = m, nbot = nb - 1 - m;   // ntop - nbot is 0 or 1
    T* zt = z;
    T* zb = z + 32;
    Row Lt, Lb;
    // one line product of each chain (or of the top chain alone)
    auto prod2 = [&](const Row& Rt, const Row& Rb, const T* St, const T* Sb, T& rt, T& rb, bool two) {
        if constexpr (BB > 0) {
            const float4* z4t = reinterpret_cast<const float4*>(zt);
            const float4* z4b = reinterpret_cast<const float4*>(zb);
            float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f, c0 = 0.f, c1 = 0.f, c2 = 0.f, c3 = 0.f;
            if (two) {
#pragma unroll
                for (int q = 0; q < Row::NQ; ++q) {
                    const float4 u = z4t[q], v = z4b[q];
                    a0 += Rt.s[q].x * u.x; a1 += Rt.s[q].y * u.y; a2 += Rt.s[q].z * u.z; a3 += Rt.s[q].w * u.w;
                    c0 += Rb.s[q].x * v.x; c1 += Rb.s[q].y * v.y; c2 += Rb.s[q].z * v.z; c3 += Rb.s[q].w * v.w;
                }
                rb = (c0 + c1) + (c2 + c3);
            } else {
#pragma unroll
                for (int q = 0; q < Row::NQ; ++q) {
                    const float4 u = z4t[q];
                    a0 += Rt.s[q].x * u.x; a1 += Rt.s[q].y * u.y; a2 += Rt.s[q].z * u.z; a3 += Rt.s[q].w * u.w;
                }
            }
            rt = (a0 + a1) + (a2 + a3);
        } else {
            rt = dot_col<T>(St, zt, b, ld, lane);
            if (two) rb = dot_col<T>(Sb, zb, b, ld, lane);
        }
    };
    T ct = T(0), cb = T(0);   // this lane's entries of the last finished top / bottom line
    // forward: top j = s, bottom j = nb - 1 - s.  The rows of step s + 1 are
    // loaded at the end of step s (into the other register set), so that
    // their latency overlaps the exchange of the line inputs.
    Row Nt, Nb;
    auto fwd = [&](int s, Row& Ct, Row& Cb, Row& Xt, Row& Xb) {
        const int jt = s, jb = nb - 1 - s;
        zt[lane] = act ? w[jt * b + lane] + (jt > 0 ? cys[(jt - 1) * cs + lane] * ct : T(0)) : T(0);
        zb[lane] = act ? w[jb * b + lane] + (s > 0 ? cys[jb * cs + lane] * cb : T(0)) : T(0);
        __syncwarp();
        prod2(Ct, Cb, Sinv + jt * bl, Sinv + jb * bl, ct, cb, true);
        if constexpr (BB > 0) {
            if (s + 1 < nbot) {
                Xt.load((const float*)(Sinv + (jt + 1) * bl), lane);
                Xb.load((const float*)(Sinv + (jb - 1) * bl), lane);
            }
        }
        if (act) {
            w[jt * b + lane] = ct;
            w[jb * b + lane] = cb;
        }
        __syncwarp();
    };
    if constexpr (BB > 0) {
        if (nbot > 0) {
            Nt.load((const float*)Sinv, lane);
            Nb.load((const float*)(Sinv + (nb - 1) * bl), lane);
        }
    }
    {
        Row Pt, Pb;
        int s = 0;
        for (; s + 1 < nbot; s += 2) {
            fwd(s, Nt, Nb, Pt, Pb);
            fwd(s + 1, Pt, Pb, Nt, Nb);
        }
        if (s < nbot) fwd(s, Nt, Nb, Pt, Pb);
    }
    if (ntop > nbot) {   // the last top line, j = ntop - 1
        const int jt = ntop - 1;
        if constexpr (BB > 0) Lt.load((const float*)(Sinv + jt * bl), lane);
        zt[lane] = act ? w[jt * b + lane] + (jt > 0 ? cys[(jt - 1) * cs + lane] * ct : T(0)) : T(0);
        __syncwarp();
        T dummy = T(0);
        prod2(Lt, Lb, Sinv + jt * bl, Sinv, ct, dummy, false);
        if (act) w[jt * b + lane] = ct;
        __syncwarp();
    }
    // middle line
    {
        if constexpr (BB > 0) Lt.load((const float*)(Sinv + m * bl), lane);
        T zm = T(0);
        if (act) {
            zm = w[m * b + lane];
            if (m > 0) zm += cys[(m - 1) * cs + lane] * ct;
            if (m < nb - 1) zm += cys[m * cs + lane] * cb;
        }
        zt[lane] = zm;
        __syncwarp();
        T dummy = T(0);
        prod2(Lt, Lb, Sinv + m * bl, Sinv, ct, dummy, false);
        cb = ct;
        if (act) w[m * b + lane] = ct;
        __syncwarp();
    }
    // back: top j = m - 1 - s, bottom j = m + 1 + s (rows of the next step
    // prefetched as in the forward sweep)
    auto bwd = [&](int s, Row& Ct, Row& Cb, Row& Xt, Row& Xb) {
        const int jt = m - 1 - s, jb = m + 1 + s;
        T wt = T(0), wb = T(0);
        zt[lane] = act ? cys[jt * cs + lane] * ct : T(0);
        zb[lane] = act ? cys[(jb - 1) * cs + lane] * cb : T(0);
        if (act) {
            wt = w[jt * b + lane];
            wb = w[jb * b + lane];
        }
        __syncwarp();
        T pt, pb;
        prod2(Ct, Cb, Sinv + jt * bl, Sinv + jb * bl, pt, pb, true);
        if constexpr (BB > 0) {
            if (s + 1 < nbot) {
                Xt.load((const float*)(Sinv + (jt - 1) * bl), lane);
                Xb.load((const float*)(Sinv + (jb + 1) * bl), lane);
            }
        }
        ct = wt + pt;
        cb = wb + pb;
        if (act) {
            w[jt * b + lane] = ct;
            w[jb * b + lane] = cb;
        }
        __syncwarp();
    };
    {
        Row Pt, Pb;
        if constexpr (BB > 0) {
            if (nbot > 0) {
                Nt.load((const float*)(Sinv + (m - 1) * bl), lane);
                Nb.load((const float*)(Sinv + (m + 1) * bl), lane);
            }
        }
        int s = 0;
        for (; s + 1 < nbot; s += 2) {
            bwd(s, Nt, Nb, Pt, Pb);
            bwd(s + 1, Pt, Pb, Nt, Nb);
        }
        if (s < nbot) bwd(s, Nt, Nb, Pt, Pb);
    }
    if (ntop > nbot) {   // the last top line, j = 0
        if constexpr (BB > 0) Lt.load((const float*)Sinv, lane);
        T wt = T(0);
        zt[lane] = act ? cys[lane] * ct : T(0);
        if (act) wt = w[lane];
        __syncwarp();
        T pt, dummy = T(0);
        prod2(Lt, Lb, Sinv, Sinv, pt, dummy, false);
        ct = wt + pt;
        if (act) w[lane] = ct;
        __syncwarp();
    }
}

// Out-of-line entry of one row-path width, for kernels that serve boxes of
// several widths: each width's sweeps get their own register allocation
// (inlined together they would share one and spill).  Called once per
// refinement step.
template <int BB>
__device__ __noinline__ void tw_warp_f32(const float* __restrict__ Sinv, const float* __restrict__ cys, float* w,
                                         float* z, int b, int nb) {
    tw_warp<float, BB>(Sinv, cys, w, z, b, nb);
}

// Both twisted sweeps on two warps (FP32 row path, lines of width bp <= BB): warp
// 0 runs the top chain (lines 0 .. m - 1) and warp 1 the bottom chain (lines
// nb - 1 .. m + 1); after a barrier of the two warps (named barrier 1) warp 0
// solves the middle line m from both chains' last lines, and after another
// the two chains run back out from it.  A line's input stays in registers, an
// entry a lane, and reaches the others by shuffles; the next line's row and
// entries are loaded a line ahead: a step is the chain of its BB shuffles and
// multiply-adds.  (Through shared memory, with the line products of tw_warp,
// a step took 370 cycles for 24 cells.)  Called by threads 0 .. 63.
template <int BB>
__device__ __forceinline__ void tw_2warp(const float* __restrict__ Sinv, const float* __restrict__ cys, float* w, int b,
                                         int nb, int bp) {
    using Row = RowF<BB>;
    const int lane = threadIdx.x & 31, h = (threadIdx.x >> 5) & 1;
    const bool act = lane < b;
    const int row = act ? lane : 0, nq = bp >> 2, ld = sld<float>(bp);
    const int bl = b * ld;
    const int m = nb >> 1;
    const int cnt = h == 0 ? m : nb - 1 - m;   // lines of this warp's chain
    const int d = h == 0 ? 1 : -1;             // the next line, towards the middle
    const int j0 = h == 0 ? 0 : nb - 1;
    // the couplings of step s of a chain: between its lines j - d and j, line min(j - d, j)
    const float* cyl = cys + (h == 0 ? -bp : 0) + lane;
    float c = 0.f;   // this lane's entry of the chain's last finished line
    Row N, P;
    float wn = 0.f, cn = 0.f;   // w and coupling of the next line
    auto pre_f = [&](int s, Row& X) {
        const int j = j0 + d * s;
        X.load(Sinv + j * bl, row, nq, ld);
        if (act) {
            wn = w[j * b + lane];
            cn = s > 0 ? cyl[j * bp] : 0.f;
        }
    };
    auto fwd = [&](int s, Row& C, Row& X) {
        const float z = act ? fmaf(cn, c, wn) : 0.f;
        if (s + 1 < cnt) pre_f(s + 1, X);
        c = C.dot(z);
        if (act) w[(j0 + d * s) * b + lane] = c;
    };
    if (cnt > 0) pre_f(0, N);
    {
        int s = 0;
#pragma unroll 1
        for (; s + 1 < cnt; s += 2) {
            fwd(s, N, P);
            fwd(s + 1, P, N);
        }
        if (s < cnt) fwd(s, N, P);
    }
    asm volatile("bar.sync 1, 64;" ::: "memory");
    if (h == 0) {
        N.load(Sinv + m * bl, row, nq, ld);
        float z = 0.f;
        if (act) {
            z = w[m * b + lane];
            if (m > 0) z += cys[(m - 1) * bp + lane] * w[(m - 1) * b + lane];
            if (m < nb - 1) z += cys[m * bp + lane] * w[(m + 1) * b + lane];
        }
        const float r = N.dot(z);
        if (act) w[m * b + lane] = r;
    }
    asm volatile("bar.sync 1, 64;" ::: "memory");
    c = act ? w[m * b + lane] : 0.f;
    // back: lines m - d (s = 0) .. j0, coupled to the line finished before
    auto pre_b = [&](int s, Row& X) {
        const int j = m - d * (s + 1);
        X.load(Sinv + j * bl, row, nq, ld);
        if (act) {
            wn = w[j * b + lane];
            cn = cyl[(j + d) * bp];
        }
    };
    auto bwd = [&](int s, Row& C, Row& X) {
        const float z = act ? cn * c : 0.f, wj = wn;
        if (s + 1 < cnt) pre_b(s + 1, X);
        c = wj + C.dot(z);
        if (act) w[(m - d * (s + 1)) * b + lane] = c;
    };
    wn = cn = 0.f;
    if (cnt > 0) pre_b(0, N);
    {
        int s = 0;
#pragma unroll 1
        for (; s + 1 < cnt; s += 2) {
            bwd(s, N, P);
            bwd(s + 1, P, N);
        }
        if (s < cnt) bwd(s, N, P);
    }
}

template <int BB>
__device__ __noinline__ void tw_2warp_f32(const float* __restrict__ Sinv, const float* __restrict__ cys, float* w,
                                          int b, int nb) {
    tw_2warp<BB>(Sinv, cys, w, b, nb, BB);
}

// The FP32 sweeps of one right-hand side by threads 0 .. 63: two warps on the
// row path of the line width bp where there is one, else warp 0 alone by
// column (zbuf: 64 entries, for that).  The caller synchronises the block afterwards.
__device__ void warp2_sweeps(const float* __restrict__ Sinv, const float* __restrict__ cys, float* w, float* zbuf,
                             int b, int nb, int bp) {
    switch (bp) {
        case 4: tw_2warp_f32<4>(Sinv, cys, w, b, nb); return;
        case 8: tw_2warp_f32<8>(Sinv, cys, w, b, nb); return;
        case 12: tw_2warp_f32<12>(Sinv, cys, w, b, nb); return;
        case 16: tw_2warp_f32<16>(Sinv, cys, w, b, nb); return;
        case 20: tw_2warp_f32<20>(Sinv, cys, w, b, nb); return;
        case 24: tw_2warp_f32<24>(Sinv, cys, w, b, nb); return;
        case 28: tw_2warp_f32<28>(Sinv, cys, w, b, nb); return;
        case 32: tw_2warp_f32<32>(Sinv, cys, w, b, nb); return;
        default: break;
    }
    if (threadIdx.x < 32) tw_warp<float, 0>(Sinv, cys, w, zbuf, b, nb);
}

// One warp solves in place (one right-hand side): the twisted sweeps, on the
// FP32 row path of the line width bp where there is one, else by column.
// zbuf: 64 entries of this warp.
template <typename T>
__device__ void warp_sweeps(const T* __restrict__ Sinv, const T* __restrict__ cys, T* w, T* zbuf, int b, int nb,
                            int bp) {
    if constexpr (std::is_same<T, float>::value) {
        switch (bp) {
            case 4: tw_warp_f32<4>(Sinv, cys, w, zbuf, b, nb); return;
            case 8: tw_warp_f32<8>(Sinv, cys, w, zbuf, b, nb); return;
            case 12: tw_warp_f32<12>(Sinv, cys, w, zbuf, b, nb); return;
            case 16: tw_warp_f32<16>(Sinv, cys, w, zbuf, b, nb); return;
            case 20: tw_warp_f32<20>(Sinv, cys, w, zbuf, b, nb); return;
            case 24: tw_warp_f32<24>(Sinv, cys, w, zbuf, b, nb); return;
            case 28: tw_warp_f32<28>(Sinv, cys, w, zbuf, b, nb); return;
            case 32: tw_warp_f32<32>(Sinv, cys, w, zbuf, b, nb); return;
            default: break;
        }
    }
    tw_warp<T, 0>(Sinv, cys, w, zbuf, b, nb);
}

// Right-hand side generators -------------------------------------------------

// Basis problem: Robin data psi_m on side sk of the box, homogeneous elsewhere.
struct RhsBasis {
    int sk, m;
    __device__ double operator()(const Box& B, const Ops& O, int i, int j) const {
        const int a = sk >> 1;
        const bool on = (sk == 0 && i == 0) || (sk == 1 && i == B.nx - 1) || (sk == 2 && j == 0) ||
                        (sk == 3 && j == B.ny - 1);
        if (!on) return 0.0;
        const int pos = a == 0 ? j : i;
        const int len = a == 0 ? B.ny : B.nx;
        return O.bT[side_off(B, sk) + pos] * psi_val(m, pos, len, B.rlen[sk]);
    }
};

// Fixed right-hand side kept in shared memory (sources + boundary data).
struct RhsStored {
    const double* b;
    __device__ double operator()(const Box& B, const Ops&, int i, int j) const { return b[j * B.nx + i]; }
};

// f |c| + Dirichlet / Neumann data + Robin data lam (lam may be null).
__device__ double source_rhs(const Box& B, const Ops& O, const double* fm, int nxg, double vol, double ax,
                             double ay, const double* lam, int i, int j) {
    double r = fm[(B.lo[0] + i) + (long long)nxg * (B.lo[1] + j)] * vol;
    const int sides[4] = {i == 0 ? 0 : -1, i == B.nx - 1 ? 1 : -1, j == 0 ? 2 : -1, j == B.ny - 1 ? 3 : -1};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int sid = sides[q];
        if (sid < 0) continue;
        const int pos = (sid >> 1) == 0 ? j : i;
        const double area = (sid >> 1) == 0 ? ax : ay;
        if (B.kind[sid] == 1) r += O.bT[side_off(B, sid) + pos] * B.val[sid];
        else if (B.kind[sid] == 0) r -= area * B.val[sid];
        else if (lam) r += O.bT[side_off(B, sid) + pos] * lam[side_off(B, sid) + pos];
    }
    return r;
}

// Solves A x = b for one right-hand side with one warp in the FP64 form: one
// solve, in w.
template <typename Rhs>
__device__ int warp_solve64(const Box& B, const Ops& O, const double* Sinv, const double* cys, double* w, double* zbuf,
                            const Rhs& rhs) {
    const int lane = threadIdx.x & 31;
    for (int j = 0; j < B.ny; ++j)
        for (int i = lane; i < B.nx; i += 32) w[j * B.nx + i] = rhs(B, O, i, j);
    __syncwarp();
    warp_sweeps<double>(Sinv, cys, w, zbuf, B.nx, B.ny, B.nx);
    return 1;
}

// The twisted sweeps of an FP64 solve by four warps: two per chain, each with
// half of a line product's columns (the narrow FP64 pipe is fed by all four
// quarters of the SM), the line input passed by shuffles, the halves' sums met
// in red (double-buffered by line parity: one barrier of the pair per line).
// w: the right-hand side in, the solution out; red: 8 x 32 entries.  (The four
// warps on one chain after the other took 1.7k cycles a line of 24 cells: twice
// as many steps, and a chain of six multiply-adds and four sums in each.)
__device__ void tw_4warp64(const double* __restrict__ Sinv, const double* __restrict__ cys, double* w, double* red,
                           int b, int nb) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int h = warp >> 1, q = warp & 1;
    const bool act = lane < b;
    const int row = act ? lane : 0;
    const size_t bl = (size_t)b * b;
    const int m = nb >> 1, cnt = h == 0 ? m : nb - 1 - m, d = h == 0 ? 1 : -1, j0 = h == 0 ? 0 : nb - 1;
    const int kq = (b + 1) >> 1, ka = q * kq, kb = min(b, ka + kq);
    const double* cyl = cys + (h == 0 ? -b : 0) + row;   // coupling towards the line before, as in tw_2warp
    int par = 0;
    auto prod = [&](const double* S, double z) {
        double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
        const double* s = S + (size_t)ka * b + row;
        int k = ka;
        for (; k + 3 < kb; k += 4, s += 4 * b) {
            a0 = fma(s[0], __shfl_sync(0xffffffffu, z, k), a0);
            a1 = fma(s[b], __shfl_sync(0xffffffffu, z, k + 1), a1);
            a2 = fma(s[2 * b], __shfl_sync(0xffffffffu, z, k + 2), a2);
            a3 = fma(s[3 * b], __shfl_sync(0xffffffffu, z, k + 3), a3);
        }
        for (; k < kb; ++k, s += b) a0 = fma(s[0], __shfl_sync(0xffffffffu, z, k), a0);
        const double mine = (a0 + a1) + (a2 + a3);
        red[(par * 4 + warp) * 32 + lane] = mine;
        bar_pair(2 + h);
        const double other = red[(par * 4 + (warp ^ 1)) * 32 + lane];
        par ^= 1;
        return mine + other;
    };
    double c = 0.0;
    for (int s = 0; s < cnt; ++s) {
        const int j = j0 + d * s;
        double z = 0.0;
        if (act) z = s > 0 ? fma(cyl[j * b], c, w[j * b + lane]) : w[j * b + lane];
        c = prod(Sinv + j * bl, z);
        if (q == 0 && act) w[j * b + lane] = c;
    }
    __syncthreads();
    if (h == 0) {
        double z = 0.0;
        if (act) {
            z = w[m * b + lane];
            if (m > 0) z += cys[(m - 1) * b + lane] * c;
            if (m < nb - 1) z += cys[m * b + lane] * w[(m + 1) * b + lane];
        }
        const double r = prod(Sinv + m * bl, z);
        if (q == 0 && act) w[m * b + lane] = r;
    }
    __syncthreads();
    c = act ? w[m * b + lane] : 0.0;
    for (int s = 0; s < cnt; ++s) {
        const int j = m - d * (s + 1);
        const double z = act ? cyl[(j + d) * b] * c : 0.0;
        const double wj = act ? w[j * b + lane] : 0.0;
        c = wj + prod(Sinv + j * bl, z);
        if (q == 0 && act) w[j * b + lane] = c;
    }
    __syncthreads();
}

// One right-hand side by the whole CTA in the FP64 form: one solve.
template <typename Rhs>
__device__ int cta_solve64(const Box& B, const Ops& O, const double* Sinv, const double* cys, double* w, double* red,
                           const Rhs& rhs) {
    const int b = B.nx, nb = B.ny;
    for (int c = threadIdx.x; c < B.n; c += blockDim.x) w[c] = rhs(B, O, c % b, c / b);
    __syncthreads();
    tw_4warp64(Sinv, cys, w, red, b, nb);
    return 1;
}

// --- the mixed form's refinement in scaled variables -------------------------
// Right-hand sides b~ for the scaled solves.  Basis problem: nonzero only on
// the Robin side sk, where lane pos holds b~ of the side's face pos (a
// register, fetched by shuffle: every lane of the warp calls it); the faces
// beyond the 32 lanes (x sides of boxes higher than 32 cells) are formed anew
// at each use; stored: an array of b~.
struct RhsScSide {
    int sk, m;
    const double *dsc, *bT;   // of Ops
    double mine;              // b~ of face `lane` of side sk (0 beyond the side)
    __device__ static double face(const Box& B, const double* dsc, const double* bT, int sk, int m, int pos) {
        const int len = (sk >> 1) == 0 ? B.ny : B.nx;
        const int ci = (sk >> 1) == 0 ? pos * B.nx + (sk == 0 ? 0 : B.nx - 1)
                                      : (sk == 2 ? 0 : (B.ny - 1) * B.nx) + pos;
        return dsc[ci] * bT[side_off(B, sk) + pos] * psi_val(m, pos, len, B.rlen[sk]);
    }
    __device__ double operator()(const Box& B, int i, int j) const {
        const bool on = (sk == 0 && i == 0) || (sk == 1 && i == B.nx - 1) || (sk == 2 && j == 0) ||
                        (sk == 3 && j == B.ny - 1);
        const int pos = (sk >> 1) == 0 ? j : i;
        const double v = __shfl_sync(0xffffffffu, mine, pos & 31);
        if (on && pos >= 32) return face(B, dsc, bT, sk, m, pos);
        return on ? v : 0.0;
    }
    // this lane's part of the largest high word of b~
    __device__ unsigned top(const Box& B) const {
        unsigned h = abs_hi(mine);
        for (int pos = (threadIdx.x & 31) + 32; pos < ((sk >> 1) == 0 ? B.ny : B.nx); pos += 32)
            h = max(h, abs_hi(face(B, dsc, bT, sk, m, pos)));
        return h;
    }
};
struct RhsScStored {
    const double* b;
    __device__ double operator()(const Box& B, int i, int j) const { return b[j * B.nx + i]; }
    __device__ unsigned top(const Box& B) const {
        unsigned h = 0u;
        for (int c = threadIdx.x & 31; c < B.n; c += 32) h = max(h, abs_hi(b[c]));
        return h;
    }
};

// (i, j) of cell c of lines of b <= 32 cells, rb = 1.f / b: (c + 0.5) / b is
// at least 1 / 64 away from an integer, far above the FP32 error for c < 2^16.
__device__ __forceinline__ void cell_ij(int c, int b, float rb, int& i, int& j) {
    j = (int)(((float)c + 0.5f) * rb);
    i = c - j * b;
}

// One right-hand side by one warp in the mixed form: FP32 twisted sweeps of
// the kept factor, FP64 residuals of the scaled operator, until
// |r~|_inf <= tol |b~|_inf.  Cells are visited 32 at a time by all lanes.  On exit x
// holds x~ (the caller scales back with dsc).  Returns the number of sweeps.
// SW: the line width where it is a template's (0: by column; -1: the row path
// of the width b where there is one, chosen at run time).  The FP32 vectors
// are scaled by the right-hand side's exponent (norm_shift).
template <typename Rhs, int SW = 0>
__device__ int warp_solve_sc(const Box& B, const Ops& O, const float* Sinv, const float* cys, double* x, float* w,
                             float* zbuf, const Rhs& rhs, double tol, int max_ir, int* noconv) {
    const int lane = threadIdx.x & 31;
    const int b = B.nx, nb = B.ny;
    const float rb = 1.f / (float)b;
    const int nit = (B.n + 31) >> 5;
    float bn = 0.f;
    const int ex = norm_shift(__reduce_max_sync(0xffffffffu, rhs.top(B)));
    for (int k = 0; k < nit; ++k) {
        const int c = k * 32 + lane;
        const bool ok = c < B.n;
        int i, j;
        cell_ij(ok ? c : 0, b, rb, i, j);
        const double bt = rhs(B, i, j);
        if (ok) {
            const float wc = d2f_bits(bt, ex);
            x[c] = 0.0;
            w[c] = wc;
            bn = fmaxf(bn, fabsf(wc));
        }
    }
    for (int o = 16; o; o >>= 1) bn = fmaxf(bn, __shfl_xor_sync(0xffffffffu, bn, o));
    __syncwarp();
    int it = 0;
    for (; it < max_ir; ++it) {
        if constexpr (SW > 0) tw_warp<float, SW>(Sinv, cys, w, zbuf, b, nb);
        else if constexpr (SW < 0) warp_sweeps<float>(Sinv, cys, w, zbuf, b, nb, b);
        else tw_warp<float, 0>(Sinv, cys, w, zbuf, b, nb);
        for (int c = lane; c < B.n; c += 32) x[c] += f2d_bits(w[c], ex);
        __syncwarp();
        float rn = 0.f;
        for (int k = 0; k < nit; ++k) {
            const int c = k * 32 + lane;
            const bool ok = c < B.n;
            int i, j;
            cell_ij(ok ? c : 0, b, rb, i, j);
            const double bt = rhs(B, i, j);
            if (ok) {
                const float wc = d2f_bits(resid_sc(B, O, x, bt, c, i, j), ex);
                w[c] = wc;
                rn = fmaxf(rn, fabsf(wc));
            }
        }
        for (int o = 16; o; o >>= 1) rn = fmaxf(rn, __shfl_xor_sync(0xffffffffu, rn, o));
        __syncwarp();
        if ((double)rn <= tol * (double)bn || bn == 0.f) { ++it; break; }
        if (it == max_ir - 1 && lane == 0) *noconv = 1;
    }
    return it;
}

// The same by the whole CTA (the smoothing solves): sweeps by two warps (a
// chain each), FP64 updates and residuals over all threads.  warm: x holds a
// starting x~ and the refinement starts from its residual (stopping rule
// still relative to b~; no sweep when the start meets it).  b~ is stored.
// BB > 0: lines of width at most BB; BB = 0: any width by a switch (bp).
// nrm: 3 entries.
template <int BB = 0>
__device__ int cta_solve_sc(const Box& B, const Ops& O, const float* Sinv, const float* cys, double* x, float* w,
                            float* zw, unsigned int* nrm, const double* bt, double tol, int max_ir, int* noconv,
                            bool warm, int bp) {
    const int tid = threadIdx.x, nt = blockDim.x;
    const int b = B.nx, nb = B.ny;
    const float rb = 1.f / (float)b;
    if (tid < 3) nrm[tid] = 0u;
    __syncthreads();
    unsigned hm = 0u;
    for (int c = tid; c < B.n; c += nt) hm = max(hm, abs_hi(bt[c]));
    hm = __reduce_max_sync(0xffffffffu, hm);
    if ((tid & 31) == 0) atomicMax(&nrm[2], hm);
    __syncthreads();
    const int ex = norm_shift(nrm[2]);
    float bn = 0.f, r0 = 0.f;
    for (int c = tid; c < B.n; c += nt) {
        int i, j;
        cell_ij(c, b, rb, i, j);
        const float wb = d2f_bits(bt[c], ex);
        const float wc = warm ? d2f_bits(resid_sc(B, O, x, bt[c], c, i, j), ex) : wb;
        w[c] = wc;
        bn = fmaxf(bn, fabsf(wb));
        r0 = fmaxf(r0, fabsf(wc));
    }
    if (!warm)
        for (int c = tid; c < B.n; c += nt) x[c] = 0.0;
    for (int o = 16; o; o >>= 1) {
        bn = fmaxf(bn, __shfl_xor_sync(0xffffffffu, bn, o));
        r0 = fmaxf(r0, __shfl_xor_sync(0xffffffffu, r0, o));
    }
    if ((tid & 31) == 0) {
        atomicMax(&nrm[0], __float_as_uint(bn));
        atomicMax(&nrm[1], __float_as_uint(r0));
    }
    __syncthreads();
    bn = __uint_as_float(nrm[0]);
    r0 = __uint_as_float(nrm[1]);
    __syncthreads();   // nrm[1] is reset at the top of the first step
    int it = 0;
    if (warm && ((double)r0 <= tol * (double)bn || bn == 0.f)) return 0;
    for (; it < max_ir; ++it) {
        if constexpr (BB > 0) {
            if (tid < 64) tw_2warp<BB>(Sinv, cys, w, b, nb, bp);
        } else {
            if (tid < 64) warp2_sweeps(Sinv, cys, w, zw, b, nb, bp);
        }
        __syncthreads();
        for (int c = tid; c < B.n; c += nt) x[c] += f2d_bits(w[c], ex);
        if (tid == 0) nrm[1] = 0u;
        __syncthreads();
        float rn = 0.f;
        for (int c = tid; c < B.n; c += nt) {
            int i, j;
            cell_ij(c, b, rb, i, j);
            const float wc = d2f_bits(resid_sc(B, O, x, bt[c], c, i, j), ex);
            w[c] = wc;
            rn = fmaxf(rn, fabsf(wc));
        }
        for (int o = 16; o; o >>= 1) rn = fmaxf(rn, __shfl_xor_sync(0xffffffffu, rn, o));
        if ((tid & 31) == 0) atomicMax(&nrm[1], __float_as_uint(rn));
        __syncthreads();
        rn = __uint_as_float(nrm[1]);
        if ((double)rn <= tol * (double)bn || bn == 0.f) { ++it; break; }
        if (it == max_ir - 1 && tid == 0) *noconv = 1;
        __syncthreads();   // nrm[1] is reset at the top of the next step
    }
    __syncthreads();
    return it;
}

__host__ __device__ inline size_t align16(size_t v) { return (v + 15) & ~size_t(15); }

// The smoothing pack of one 2D subdomain: everything the smoothing solves
// need that does not change between smoothing steps, written once after the
// factorisation in the byte layout the smoothing kernel's shared memory
// starts with, so that one bulk copy stages it.  S^-1 blocks first (the
// factor slot other kernels read), then the FP64 operator (diagonal, x / y
// couplings, Jacobi scaling), the box-side transmissibilities and Robin
// beta, the fixed part of the right-hand side (sources and physical
// boundary data) and the scaled y couplings of the sweeps.  Every field
// starts on 16 bytes; the total is a multiple of 16.
struct SPack {
    size_t cd, cx, cy, dsc, bT, bB, bst, cys, bytes;
};

__host__ __device__ inline SPack spack_layout(int nx, int ny, size_t tsz, int pad) {
    SPack L;
    const size_t n = (size_t)nx * ny, m = 2 * (size_t)(nx + ny);
    size_t o = align16(tsz * sinv_len(nx, ny, (int)tsz, pad));
    L.cd = o;  o += align16(sizeof(double) * n);
    L.cx = o;  o += align16(sizeof(double) * n);
    L.cy = o;  o += align16(sizeof(double) * n);
    L.dsc = o; o += align16(sizeof(double) * n);
    L.bT = o;  o += align16(sizeof(double) * m);
    L.bB = o;  o += align16(sizeof(double) * m);
    L.bst = o; o += align16(sizeof(double) * n);
    L.cys = o; o += align16(tsz * (size_t)line_width(nx, (int)tsz, pad) * ny);
    L.bytes = o;
    return L;
}

// Shared-memory carve-up ----------------------------------------------------
template <typename T>
struct Carve {
    Ops O;
    T* Sinv;
    T* cys;
    T* cxs;
    T* zbuf;   // NWARP * 64: two line inputs per warp
    double* bsrc; // n: fixed right-hand side of the particular problem
    double* X; // nrhs * n
    T* W;      // nrhs * n
    int* flags;
    size_t end;   // bytes of shared memory the layout takes
};

template <typename T>
// (the basis / particular kernel keeps no h / 2K array -- it reads the few
// values it needs at the Gamma faces from global memory -- and a stored
// right-hand side only for the particular problem, so that two CTAs of the
// 24 x 24 basis boxes fit on one SM)
__host__ __device__ inline size_t carve_bytes(int nx, int ny, int nrhs, bool part, int pad) {
    const size_t n = (size_t)nx * ny;
    size_t s = align16(sizeof(double) * n) * 4;                                      // cd cx cy dsc
    s += align16(sizeof(double) * 2 * (nx + ny)) * 2;                                 // bT bB
    s += align16(sizeof(T) * sinv_len(nx, ny, sizeof(T), pad)) +
         align16(sizeof(T) * line_width(nx, sizeof(T), pad) * ny);                     // Sinv, cys (cxs lives in W)
    s += align16(sizeof(T) * 64 * NWARP) + (part ? align16(sizeof(double) * n) : 0);
    if (std::is_same<T, float>::value) s += align16(sizeof(double) * n * nrhs);
    s += align16(sizeof(T) * n * nrhs);
    return s + 64;
}

template <typename T>
__device__ Carve<T> carve(unsigned char* base, int nx, int ny, int nrhs, bool part, int pad) {
    Carve<T> C;
    const size_t n = (size_t)nx * ny;
    size_t o = 0;
    auto take = [&](size_t bytes) { unsigned char* p = base + o; o += align16(bytes); return p; };
    C.O.cd = (double*)take(sizeof(double) * n);
    C.O.cx = (double*)take(sizeof(double) * n);
    C.O.cy = (double*)take(sizeof(double) * n);
    C.O.dsc = (double*)take(sizeof(double) * n);
    C.O.hk = nullptr;
    C.O.bT = (double*)take(sizeof(double) * 2 * (nx + ny));
    C.O.bB = (double*)take(sizeof(double) * 2 * (nx + ny));
    C.Sinv = (T*)take(sizeof(T) * sinv_len(nx, ny, sizeof(T), pad));
    C.cys = (T*)take(sizeof(T) * line_width(nx, sizeof(T), pad) * ny);
    C.zbuf = (T*)take(sizeof(T) * 64 * NWARP);
    C.bsrc = part ? (double*)take(sizeof(double) * n) : nullptr;
    if (std::is_same<T, float>::value) C.X = (double*)take(sizeof(double) * n * nrhs);
    C.W = (T*)take(sizeof(T) * n * nrhs);
    if (std::is_same<T, double>::value) C.X = (double*)C.W;
    C.cxs = C.W;   // the in-line couplings are needed only while factoring, before any solve
    C.flags = (int*)take(64);
    C.end = o;
    return C;
}

__device__ void setup_box(Box& B, const MemberDev& md, const int* lo, const int* hi, double alpha) {
    for (int a = 0; a < 2; ++a) {
        B.lo[a] = lo[a];
        B.hi[a] = hi[a];
    }
    B.nx = hi[0] - lo[0];
    B.ny = hi[1] - lo[1];
    B.n = B.nx * B.ny;
    B.alpha = alpha;
    for (int sid = 0; sid < 4; ++sid) {
        const int a = sid >> 1;
        const bool phys = (sid & 1) ? (hi[a] == md.n[a]) : (lo[a] == 0);
        if (phys) {
            B.kind[sid] = md.bc_kind[sid] == 1 ? 1 : 0;
            B.val[sid] = md.bc_val[sid];
        } else {
            B.kind[sid] = 2;
            B.val[sid] = 0.0;
        }
        B.rlen[sid] = 1.0 / (double)(a == 0 ? B.ny : B.nx);
    }
}

__device__ void fill_scale(const Box& B, Ops& O, bool mixed) {
    for (int c = threadIdx.x; c < B.n; c += blockDim.x)
        O.dsc[c] = !mixed ? 1.0 : in_f32_range(O.cd[c]) ? (double)rsqrtf((float)O.cd[c]) : 1.0 / sqrt(O.cd[c]);
    __syncthreads();
}

// --- bulk (TMA engine) copy global -> shared with an mbarrier -------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}
// Waits for phase `parity` of the barrier for at most `limit` cycles (2^31,
// about a second, by default); false on timeout.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, long long limit = 1LL << 31) {
    const long long t0 = clock64();
    while (true) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(smem_u32(bar)), "r"(parity)
            : "memory");
        if (ok) return true;
        if (clock64() - t0 > limit) return false;
    }
}

}  // namespace
