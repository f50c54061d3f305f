// 3D local Robin/Darcy solves of MRCM-OS on sm_103a.
//
// One CTA (17 warps) per job (a subdomain box).  The cell-centred RT0
// operator of the box (Sec. 2.2; the face laws of Eq. (genRobin)) is block
// tridiagonal over the planes normal to the box's longest axis a2; a plane
// has b = n_a0 n_a1 cells (a0 fastest) and planes couple through diagonal
// blocks D_j (the a2-face transmissibilities).  The factorisation
// (Algorithm 1, Steps 1 and 6) keeps the inverses of the plane Schur
// complements S_j = A_jj - D_{j-1} S_{j-1}^{-1} D_{j-1}: S_j is formed in
// registers from S_{j-1}^{-1} in place (D is diagonal) and inverted there by
// the whole CTA (Gauss-Jordan, SPD so no pivoting); the inverses go to global
// memory (a box's factor, n_a2 b^2 entries, does not fit on chip).
// A solve is two sweeps of dense b x b products, all right-hand sides of a
// round at once, so each plane inverse is read once per sweep.
//
// Precision: T = double is the FP64 form.  T = float is the mixed form:
// Jacobi-scaled factor, Schur diagonals from FP64, FP32 sweeps on scaled
// residuals, FP64 residuals of the unscaled operator, refined to ir_tol.
#include "box2d.cuh"

namespace {

constexpr int NW3 = 16;             // warps that compute in the sweeps
constexpr int T3 = 32 * (NW3 + 1);  // threads per CTA: one more warp issues the sweeps' copies
constexpr int NR3 = 4;              // right-hand sides per round, at most
constexpr int GT3 = 4;              // side of a register tile of the plane inverses
constexpr int GB3 = 128;            // widest plane inverted in registers
constexpr int ST3 = 4;              // most stages of the sweeps' copies

// row stride of a plane inverse: b entries padded to 4 (16 bytes in FP32, 32 in FP64)
__host__ __device__ constexpr int plane_ld(int b) { return (b + 3) & ~3; }
__host__ __device__ __forceinline__ size_t plane_stride(int b) { return (size_t)b * plane_ld(b); }
// rows of a plane inverse per copy (32 KB in FP32, 16 KB in FP64 for planes of
// 128 cells): a wait and its bookkeeping cost a few hundred cycles, as much as
// the products of 32 FP32 rows
__host__ __device__ constexpr int stage_rows(int tsz) { return tsz == 4 ? 64 : 16; }

struct Box3 {
    int lo[3], hi[3], n[3];
    int nc;
    int a0, a1, a2;   // in-plane axes (a0 fastest) and the plane axis
    int b, np;        // plane size, number of planes
    int kind[6];      // 0 Neumann, 1 Dirichlet, 2 Robin
    double val[6];
    double alpha;
    int ts[6], tt[6]; // tangential axes (ascending) of each side
    int soff[7];      // offsets of the sides in the boundary-face arrays
    // index strides, so that no coordinate array is indexed at run time
    long long g0;     // first cell of the box in the member's grid
    int gs[3], gb[3]; // grid strides by natural axis and by block axis (a0, a1, a2)
    int bs[3];        // block-order strides by natural axis
    int es[6][3], eb[6][3];   // face-index strides of each side by natural and by block axis (0 along its normal)
    int bit[6];       // the neighbour bit that cells on the side lack
    float rb, r0;     // 1 / b, 1 / n[a0]
};

__device__ void setup_box3(Box3& B, const MemberDev& md, const int* lo, const int* hi, double alpha) {
    for (int a = 0; a < 3; ++a) {
        B.lo[a] = lo[a];
        B.hi[a] = hi[a];
        B.n[a] = hi[a] - lo[a];
    }
    B.nc = B.n[0] * B.n[1] * B.n[2];
    int a2 = 2;
    for (int a = 1; a >= 0; --a)
        if (B.n[a] > B.n[a2]) a2 = a;
    B.a2 = a2;
    B.a0 = a2 == 0 ? 1 : 0;
    B.a1 = a2 == 2 ? 1 : 2;
    B.b = B.n[B.a0] * B.n[B.a1];
    B.np = B.n[a2];
    B.alpha = alpha;
    B.soff[0] = 0;
    for (int sid = 0; sid < 6; ++sid) {
        const int a = sid >> 1;
        const bool phys = (sid & 1) ? (hi[a] == md.n[a]) : (lo[a] == 0);
        if (phys) {
            B.kind[sid] = md.bc_kind[sid] == 1 ? 1 : 0;
            B.val[sid] = md.bc_val[sid];
        } else {
            B.kind[sid] = 2;
            B.val[sid] = 0.0;
        }
        B.ts[sid] = a == 0 ? 1 : 0;
        B.tt[sid] = a == 2 ? 1 : 2;
        B.soff[sid + 1] = B.soff[sid] + B.n[B.ts[sid]] * B.n[B.tt[sid]];
    }
    const int ax[3] = {B.a0, B.a1, B.a2};
    B.gs[0] = 1;
    B.gs[1] = md.n[0];
    B.gs[2] = md.n[0] * md.n[1];
    B.g0 = lo[0] + (long long)B.gs[1] * lo[1] + (long long)B.gs[2] * lo[2];
    B.bs[B.a0] = 1;
    B.bs[B.a1] = B.n[B.a0];
    B.bs[B.a2] = B.b;
    for (int sid = 0; sid < 6; ++sid)
        for (int a = 0; a < 3; ++a) B.es[sid][a] = a == B.ts[sid] ? 1 : a == B.tt[sid] ? B.n[B.ts[sid]] : 0;
    for (int p = 0; p < 3; ++p) {
        B.gb[p] = B.gs[ax[p]];
        for (int sid = 0; sid < 6; ++sid) B.eb[sid][p] = B.es[sid][ax[p]];
        B.bit[2 * ax[p]] = 1 << (2 * p);
        B.bit[2 * ax[p] + 1] = 2 << (2 * p);
    }
    B.rb = 1.f / (float)B.b;
    B.r0 = 1.f / (float)B.n[B.a0];
}

// block coordinates (along a0, a1, a2) of the cell at block index t: by FP32
// reciprocals, (t + 0.5) / b is at least 1 / 512 away from an integer, far above
// the rounding for the t < 2^14 of a box
struct Ijk {
    int i, j, k;
};
__device__ __forceinline__ Ijk bcoord(const Box3& B, int t) {
    Ijk c;
    c.k = (int)(((float)t + 0.5f) * B.rb);
    const int pos = t - c.k * B.b;
    c.j = (int)(((float)pos + 0.5f) * B.r0);
    c.i = pos - c.j * B.n[B.a0];
    return c;
}
__device__ __forceinline__ long long gidx(const Box3& B, const Ijk& c) {
    return B.g0 + c.i * B.gb[0] + c.j * B.gb[1] + (long long)c.k * B.gb[2];
}
// face index of a cell on side sid (first tangential axis fastest)
__device__ __forceinline__ int side_e(const Box3& B, int sid, const Ijk& c) {
    return c.i * B.eb[sid][0] + c.j * B.eb[sid][1] + c.k * B.eb[sid][2];
}
// P0 / P1 function m on a side face with tangential coordinates (cs, ct)
// relative to a side of extents (ls, lt): 1, s, t in [-1, 1]
__device__ __forceinline__ double psi3(int m, int cs, int ls, int ct, int lt) {
    return m == 0 ? 1.0 : m == 1 ? (double)(2 * cs + 1 - ls) / ls : (double)(2 * ct + 1 - lt) / lt;
}

struct Ops3 {
    double *cd, *c0, *c1, *c2, *dsc;  // diagonal, couplings to +a0, +a1, +a2, Jacobi scale (block order)
    double *bT, *bB;                   // boundary-face transmissibility and Robin beta per side face
    unsigned char* nb;                 // neighbour bits: 1 -a0, 2 +a0, 4 -a1, 8 +a1, 16 -a2, 32 +a2
};

// side of face f of the boundary-face arrays
__device__ __forceinline__ int side_of(const Box3& B, int f) {
    int sid = 0;
#pragma unroll
    for (int s = 1; s < 6; ++s) sid += f >= B.soff[s];
    return sid;
}
// grid index of the cell at face f of the boundary-face arrays (side sid)
__device__ __forceinline__ long long face_cell(const Box3& B, int sid, int f) {
    const int a = sid >> 1, e = f - B.soff[sid], ls = B.n[B.ts[sid]], q = e / ls;
    return B.g0 + ((sid & 1) ? (long long)(B.n[a] - 1) * B.gs[a] : 0) + (e - q * ls) * B.gs[B.ts[sid]] +
           (long long)q * B.gs[B.tt[sid]];
}

// The box operator from the face coefficients.  The faces of all sides are
// one list, so that their loads are in flight together.
__device__ void build_ops3(const Box3& B, const MemberDev& md, const DevPtrs& P, Ops3& O, bool mixed) {
    const double* Tf = P.Tf + md.cell_off * 3;
    const double* hkg = P.hk + md.cell_off * 3;
    const double* wh = P.wh + md.cell_off * 3;
    const double vol = md.h[0] * md.h[1] * md.h[2];
    const int a0 = B.a0, a1 = B.a1, a2 = B.a2, e0 = B.n[a0], e1 = B.n[a1], e2 = B.np, b = B.b, nc = B.nc;
    for (int t = threadIdx.x; t < nc; t += blockDim.x) {
        const Ijk c = bcoord(B, t);
        const double* T = Tf + gidx(B, c) * 3;
        const double t0 = T[a0], t1 = T[a1], t2 = T[a2];
        const int i = c.i, j = c.j, k = c.k;
        O.c0[t] = i < e0 - 1 ? t0 : 0.0;
        O.c1[t] = j < e1 - 1 ? t1 : 0.0;
        O.c2[t] = k < e2 - 1 ? t2 : 0.0;
        O.nb[t] = (unsigned char)((i > 0) | (i < e0 - 1) << 1 | (j > 0) << 2 | (j < e1 - 1) << 3 | (k > 0) << 4 |
                                  (k < e2 - 1) << 5);
    }
    for (int f = threadIdx.x; f < B.soff[6]; f += blockDim.x) {
        const int sid = side_of(B, f), a = sid >> 1;
        const long long g = face_cell(B, sid, f);
        const double area = vol / md.h[a];
        const double hin = hkg[g * 3 + a];
        double T = 0.0, beta = 0.0;
        if (B.kind[sid] == 2) {
            const long long gf = (sid & 1) ? g : g - B.gs[a];
            beta = B.alpha * wh[gf * 3 + a];
            T = area * rcp64(hin + beta);
        } else if (B.kind[sid] == 1) {
            T = area * rcp64(hin);
        }
        O.bT[f] = T;
        O.bB[f] = beta;
    }
    __syncthreads();
    for (int t = threadIdx.x; t < nc; t += blockDim.x) {
        const unsigned char m = O.nb[t];
        double d = O.c0[t] + O.c1[t] + O.c2[t];
        if (m & 1) d += O.c0[t - 1];
        if (m & 4) d += O.c1[t - e0];
        if (m & 16) d += O.c2[t - b];
        if ((m & 63) != 63) {
            const Ijk c = bcoord(B, t);
            for (int sid = 0; sid < 6; ++sid)
                if (!(m & B.bit[sid])) d += O.bT[B.soff[sid] + side_e(B, sid, c)];
        }
        O.cd[t] = d;
        if (mixed) O.dsc[t] = in_f32_range(d) ? (double)rsqrtf((float)d) : 1.0 / sqrt(d);
    }
    __syncthreads();
}

// Mixed form: the couplings of the scaled operator D A D in FP32, for the factor
// and the sweeps (the operator itself stays unscaled).
__device__ __forceinline__ float scaled3(const Ops3& O, const double* c, unsigned bit, int step, int t) {
    return (O.nb[t] & bit) ? (float)(c[t] * O.dsc[t] * O.dsc[t + step]) : 0.f;
}

// Mixed form, after the factorisation: the diagonal's place takes its box-side
// part, the rest of a row being differences (resid3).
__device__ void side_diag3(const Box3& B, Ops3& O) {
    for (int t = threadIdx.x; t < B.nc; t += blockDim.x) {
        const unsigned char m = O.nb[t];
        double d = 0.0;
        if ((m & 63) != 63) {
            const Ijk c = bcoord(B, t);
            for (int sid = 0; sid < 6; ++sid)
                if (!(m & B.bit[sid])) d += O.bT[B.soff[sid] + side_e(B, sid, c)];
        }
        O.cd[t] = d;
    }
    __syncthreads();
}

// b_t - (A x)_t in FP64.  DIFF (mixed form): in differences of neighbouring
// values, so that its rounding is that of the fluxes and not of the pressures.
// With entries of D A D, each rounded once more, the fluxes of 60 layered fields
// of 60 x 110 x 40 cells came out 1.7 times further from the exact ones; with rows
// summed up by the unscaled diagonal they did not, but 5 of 200 layered fields of
// 60 x 220 x 85 cells missed ir_tol (a box's rounding floor above it) against 1
// with DIFF.  It costs six FP64 instructions a cell: 45.2 against 42.8 ms a step.
template <bool DIFF>
__device__ __forceinline__ double resid3(const Ops3& O, int s1, int s2, const double* x, double bt, int t) {
    const unsigned char m = O.nb[t];
    const double xt = x[t], x0 = DIFF ? xt : 0.0;
    double s = fma(-O.cd[t], xt, bt);
    if (m & 1) s = fma(O.c0[t - 1], DIFF ? x[t - 1] - x0 : x[t - 1], s);
    if (m & 2) s = fma(O.c0[t], DIFF ? x[t + 1] - x0 : x[t + 1], s);
    if (m & 4) s = fma(O.c1[t - s1], DIFF ? x[t - s1] - x0 : x[t - s1], s);
    if (m & 8) s = fma(O.c1[t], DIFF ? x[t + s1] - x0 : x[t + s1], s);
    if (m & 16) s = fma(O.c2[t - s2], DIFF ? x[t - s2] - x0 : x[t - s2], s);
    if (m & 32) s = fma(O.c2[t], DIFF ? x[t + s2] - x0 : x[t + s2], s);
    return s;
}

// N consecutive values of shared memory, 16 bytes a load where N allows it
template <typename T, int N>
__device__ __forceinline__ void ldv(const T* __restrict__ p, T (&v)[N]) {
    constexpr int W = 16 / (int)sizeof(T);
    if constexpr (N % W == 0) {
        using V = std::conditional_t<sizeof(T) == 4, float4, double2>;
#pragma unroll
        for (int q = 0; q < N / W; ++q) {
            const V t = reinterpret_cast<const V*>(p)[q];
            v[W * q] = t.x;
            v[W * q + 1] = t.y;
            if constexpr (W == 4) {
                v[W * q + 2] = t.z;
                v[W * q + 3] = t.w;
            }
        }
    } else if constexpr (N == 2) {
        const float2 t = *reinterpret_cast<const float2*>(p);
        v[0] = t.x;
        v[1] = t.y;
    } else {
#pragma unroll
        for (int q = 0; q < N; ++q) v[q] = p[q];
    }
}
template <typename T>
__device__ __forceinline__ void stv4(T* p, T a, T b, T c, T d) {
    if constexpr (sizeof(T) == 4) {
        *reinterpret_cast<float4*>(p) = make_float4(a, b, c, d);
    } else {
        reinterpret_cast<double2*>(p)[0] = make_double2(a, b);
        reinterpret_cast<double2*>(p)[1] = make_double2(c, d);
    }
}

// Workspace of the register inverses (entries): two panels of GT3 rows, the
// scaled panel, two inverse pivot blocks, two diagonal tiles, the diagonal of
// the last inverse and of the next Schur block.
constexpr int GLD3 = GB3 + 4;
constexpr int GJW3 = 3 * GT3 * GLD3 + 4 * GT3 * GT3 + 2 * GLD3;

// Block LDL^T over planes of at most GB3 cells, each plane's Schur block
// inverted in registers: the block is symmetric, and the in-place
// Gauss-Jordan elimination of a symmetric block keeps M_IJ = +-M_JI^T (minus
// when exactly one of I, J has been eliminated), so only the GT3 x GT3 tiles
// (I, J), I <= J, are held, one per thread (528 for 128 cells).  Pivots go by
// blocks K of GT3 rows, two barriers per block:
//   - the threads holding row or column block K have published the panel
//     M_K., the last warp the inverse pivot block P = M_KK^-1; every thread
//     forms one entry of P M_K.;
//   - every thread updates its tile, M_IJ -= M_IK (P M_KJ), and publishes it
//     if it belongs to the next panel.  Meanwhile the last warp updates the
//     next pivot block by itself, from the copy its holder left in dt, and
//     inverts it with one entry per lane, so that the pivots' reciprocals are
//     off the chain.
// Bound by the update's FP64 FMAs in the FP64 form, by the latency of the
// per-block chain in the mixed form.  c0s, c1s: the in-plane couplings in T.
template <typename T>
__device__ void factor3_reg(const Box3& B, const Ops3& O, const T* c0s, const T* c1s, const T* c2s, T* F, T* ws,
                            int* bad) {
    constexpr int G = GT3;
    const int b = B.b, ld = plane_ld(b), nb4 = ld / G, n0 = B.n[B.a0], np = B.np;
    T* R = ws;                        // [2][G][GLD3]
    T* Rn = R + 2 * G * GLD3;         // [G][GLD3]
    T* pinv = Rn + G * GLD3;          // [2][G * G]
    T* dt = pinv + 2 * G * G;         // [2][G * G] tile (k, k) before the update by block k - 1
    T* dg = dt + 2 * G * G;           // [GLD3] diagonal of the last inverse
    T* dn = dg + GLD3;                // [GLD3] diagonal of the Schur block
    const int tid = threadIdx.x, lane = tid & 31;
    const bool act = tid < nb4 * (nb4 + 1) / 2;
    const bool pivot_warp = tid >= 32 * NW3;
    int I = 0, J = tid;               // tile of this thread, row-major over I <= J
    if (act) {
        while (J >= nb4 - I) {
            J -= nb4 - I;
            ++I;
        }
        J += I;
    } else {
        I = J = -4;
    }
    const int dd = G * (J - I), o1 = n0 - dd;   // the plane's couplings of stride n0 are at x - y == o1
    T V[G][G];
#pragma unroll
    for (int y = 0; y < G; ++y)
#pragma unroll
        for (int x = 0; x < G; ++x) V[y][x] = T(0);
    // the panel of block k from the tiles that hold it, and the next pivot block
    auto publish = [&](int k) {
        T* Rk = R + (k & 1) * G * GLD3;
        if (I == k) {
#pragma unroll
            for (int y = 0; y < G; ++y) stv4(Rk + y * GLD3 + G * J, V[y][0], V[y][1], V[y][2], V[y][3]);
        } else if (J == k) {
            // I < k has been eliminated: M_kI = -M_Ik^T
#pragma unroll
            for (int x = 0; x < G; ++x) stv4(Rk + x * GLD3 + G * I, -V[0][x], -V[1][x], -V[2][x], -V[3][x]);
        }
        if (I == k + 1 && J == k + 1) {
            T* d = dt + ((k + 1) & 1) * G * G;
#pragma unroll
            for (int y = 0; y < G; ++y) stv4(d + G * y, V[y][0], V[y][1], V[y][2], V[y][3]);
        }
    };
    // (last warp) inverse of the pivot block whose entry (lane / 4 mod 4, lane mod 4) is v
    auto invert = [&](T v, int k) {
        const int y = (lane >> 2) & 3, x = lane & 3;
#pragma unroll
        for (int q = 0; q < G; ++q) {
            T piv = __shfl_sync(0xffffffffu, v, 5 * q);
            if (!(piv > T(0))) {
                if (lane == 0) *bad = 1;
                piv = T(1);
            }
            const T ip = rcp_piv(piv);
            const T r = __shfl_sync(0xffffffffu, v, G * q + x), c = __shfl_sync(0xffffffffu, v, G * y + q);
            const T rp = x == q ? ip : r * ip;
            v = y == q ? rp : (x == q ? T(0) : v) - c * rp;
        }
        if (lane < G * G) pinv[(k & 1) * G * G + lane] = v;
    };
    const int rc = tid & (GB3 - 1), ry = tid >> 7;   // the entry of P M_K. this thread forms
    for (int j = 0; j < np; ++j) {
        const int p0 = j * b;
        // diagonal of S_j in FP64 (where the cancellation is)
        if (tid < b) {
            double s = O.cd[p0 + tid];
            if constexpr (std::is_same<T, float>::value) s *= O.dsc[p0 + tid] * O.dsc[p0 + tid];
            if (j > 0) {
                const double cc = (double)c2s[p0 - b + tid];
                s -= cc * (cc * (double)dg[tid]);   // not cc^2 (range at tiny couplings)
            }
            dn[tid] = (T)s;
        }
        __syncthreads();
        if (act) {
            T ci[G], ck[G];
#pragma unroll
            for (int y = 0; y < G; ++y) {
                ci[y] = (j > 0 && G * I + y < b) ? c2s[p0 - b + G * I + y] : T(0);
                ck[y] = (j > 0 && G * J + y < b) ? c2s[p0 - b + G * J + y] : T(0);
            }
#pragma unroll
            for (int y = 0; y < G; ++y)
#pragma unroll
                for (int x = 0; x < G; ++x) V[y][x] = -(ci[y] * V[y][x] * ck[x]);
            if (dd <= G) {
                // couplings of stride 1, the diagonal; padding: the identity
                T e[G];
#pragma unroll
                for (int y = 0; y < G; ++y) e[y] = G * I + y + 1 < b ? c0s[p0 + G * I + y] : T(0);
                if (dd == G) {
                    V[G - 1][0] -= e[G - 1];
                } else {
#pragma unroll
                    for (int y = 0; y < G; ++y) {
                        V[y][y] = G * I + y < b ? dn[G * I + y] : T(1);
                        if (y + 1 < G) {
                            V[y][y + 1] -= e[y];
                            V[y + 1][y] -= e[y];
                        }
                    }
                }
            }
            if (o1 > -G && o1 < G) {
                T e[G];
#pragma unroll
                for (int y = 0; y < G; ++y) e[y] = G * I + y + n0 < b ? c1s[p0 + G * I + y] : T(0);
#pragma unroll
                for (int y = 0; y < G; ++y)
#pragma unroll
                    for (int x = 0; x < G; ++x) {
                        if (x - y == o1) V[y][x] -= e[y];
                        if (dd == 0 && y - x == o1) V[y][x] -= e[x];
                    }
            }
        }
        publish(0);
        if (I == 0 && J == 0) {
#pragma unroll
            for (int y = 0; y < G; ++y) stv4(dt + G * y, V[y][0], V[y][1], V[y][2], V[y][3]);
        }
        __syncthreads();
        if (pivot_warp) invert(dt[lane & (G * G - 1)], 0);
        __syncthreads();
        for (int k = 0; k < nb4; ++k) {
            const T* Rk = R + (k & 1) * G * GLD3;
            if (!pivot_warp && rc < ld) {
                const bool own = (rc / G) == k;
                T r[G], p[G];
#pragma unroll
                for (int m = 0; m < G; ++m) r[m] = Rk[m * GLD3 + rc];
                ldv<T, G>(pinv + (k & 1) * G * G + G * ry, p);
                const T v = (p[0] * r[0] + p[1] * r[1]) + (p[2] * r[2] + p[3] * r[3]);
                Rn[ry * GLD3 + rc] = own ? pinv[(k & 1) * G * G + G * ry + (rc & (G - 1))] : v;
            }
            __syncthreads();
            if (pivot_warp && k + 1 < nb4) {
                const int y = (lane >> 2) & 3, x = lane & 3, c = G * (k + 1);
                T v = dt[((k + 1) & 1) * G * G + (lane & (G * G - 1))];
#pragma unroll
                for (int m = 0; m < G; ++m) v -= Rk[m * GLD3 + c + y] * Rn[m * GLD3 + c + x];
                invert(v, k + 1);
            }
            if (act) {
                if (I == k) {
#pragma unroll
                    for (int y = 0; y < G; ++y) {
                        T r[G];
                        ldv<T, G>(Rn + y * GLD3 + G * J, r);
#pragma unroll
                        for (int x = 0; x < G; ++x) V[y][x] = r[x];
                    }
                } else if (J == k) {
#pragma unroll
                    for (int x = 0; x < G; ++x) {
                        T r[G];
                        ldv<T, G>(Rn + x * GLD3 + G * I, r);
#pragma unroll
                        for (int y = 0; y < G; ++y) V[y][x] = r[y];
                    }
                } else if (I > k) {
                    // V -= M_IK (P M_KJ), M_IK = R^T where I is not eliminated yet, else -R^T
#pragma unroll
                    for (int m = 0; m < G; ++m) {
                        T a[G], r[G];
                        ldv<T, G>(Rk + m * GLD3 + G * I, a);
                        ldv<T, G>(Rn + m * GLD3 + G * J, r);
#pragma unroll
                        for (int y = 0; y < G; ++y)
#pragma unroll
                            for (int x = 0; x < G; ++x) V[y][x] -= a[y] * r[x];
                    }
                } else {
#pragma unroll
                    for (int m = 0; m < G; ++m) {
                        T a[G], r[G];
                        ldv<T, G>(Rk + m * GLD3 + G * I, a);
                        ldv<T, G>(Rn + m * GLD3 + G * J, r);
#pragma unroll
                        for (int y = 0; y < G; ++y)
#pragma unroll
                            for (int x = 0; x < G; ++x) V[y][x] += a[y] * r[x];
                    }
                }
                if (k + 1 < nb4) publish(k + 1);
            }
            __syncthreads();
        }
        // the inverse to global memory (both triangles) and its diagonal to dg
        if (act) {
            T* Fj = F + (size_t)j * plane_stride(b);
#pragma unroll
            for (int y = 0; y < G; ++y)
                if (G * I + y < b) stv4(Fj + (size_t)(G * I + y) * ld + G * J, V[y][0], V[y][1], V[y][2], V[y][3]);
            if (I != J) {
#pragma unroll
                for (int x = 0; x < G; ++x)
                    if (G * J + x < b) stv4(Fj + (size_t)(G * J + x) * ld + G * I, V[0][x], V[1][x], V[2][x], V[3][x]);
            } else {
#pragma unroll
                for (int y = 0; y < G; ++y) dg[G * I + y] = V[y][y];
            }
        }
        __syncthreads();
    }
    // the solves read the factor through the bulk-copy (async) proxy, into
    // shared memory this phase used
    asm volatile("fence.proxy.async;" ::: "memory");
    __syncthreads();
}

// 16-byte vectors of the shared-memory path
template <typename T> struct V16;
template <> struct V16<float> {
    using V = float4;
    static constexpr int W = 4;
};
template <> struct V16<double> {
    using V = double2;
    static constexpr int W = 2;
};
template <typename T>
union VU {
    typename V16<T>::V v;
    T a[V16<T>::W];
};

// In-place Gauss-Jordan inverse of an SPD b x b matrix in shared memory by
// the whole CTA (row-major, leading dimension ld = plane_ld(b), padding
// columns zero), for planes wider than GB3.  Each thread updates 16-byte
// groups of a row.
template <typename T>
__device__ void gj_cta(T* S, int b, int ld, T* rowbuf, T* colbuf, T* ipb, int* bad) {
    constexpr int W = V16<T>::W;
    using V = typename V16<T>::V;
    const int tid = threadIdx.x, nt = blockDim.x;
    const int ng = ld / W;                 // groups per row
    const int tot = b * ng;
    const int i0 = tid / ng, g0 = tid - i0 * ng;
    const int di = nt / ng, dg = nt - di * ng;
    for (int k = 0; k < b; ++k) {
        if (tid == 0) {
            double piv = (double)S[k * ld + k];
            if (!(piv > 0.0)) {
                *bad = 1;
                piv = 1.0;
            }
            *ipb = std::is_same<T, float>::value ? (T)__frcp_rn((float)piv) : (T)rcp64(piv);
        }
        for (int t = tid; t < ld; t += nt) {
            rowbuf[t] = S[k * ld + t];
            if (t < b) colbuf[t] = S[t * ld + k];
        }
        __syncthreads();
        const T ip = *ipb;
        const int gk = k / W, ek = k - gk * W;
        int i = i0, g = g0;
        for (int t = tid; t < tot; t += nt) {
            VU<T> x, r;
            x.v = *reinterpret_cast<const V*>(&S[i * ld + g * W]);
            r.v = *reinterpret_cast<const V*>(&rowbuf[g * W]);
            const bool colk = g == gk;
            if (i == k) {
#pragma unroll
                for (int e = 0; e < W; ++e) x.a[e] = (colk && e == ek) ? ip : r.a[e] * ip;
            } else {
                const T f = colbuf[i] * ip;
#pragma unroll
                for (int e = 0; e < W; ++e) x.a[e] = (colk && e == ek) ? -f : x.a[e] - f * r.a[e];
            }
            *reinterpret_cast<V*>(&S[i * ld + g * W]) = x.v;
            g += dg;
            i += di;
            if (g >= ng) {
                g -= ng;
                ++i;
            }
        }
        __syncthreads();
    }
}

// The same factorisation for planes wider than GB3, the Schur block in shared
// memory.  Sb: b x plane_ld(b).
template <typename T>
__device__ void factor3_smem(const Box3& B, const Ops3& O, const T* c2s, T* F, T* Sb, T* rowbuf, T* colbuf, T* ipb,
                             int* bad) {
    constexpr bool mixed = std::is_same<T, float>::value;
    const int b = B.b, ld = plane_ld(b), bb = b * b;
    const int tid = threadIdx.x, nt = blockDim.x;
    const int n0 = B.n[B.a0];
    for (int t = tid; t < b * ld; t += nt) Sb[t] = T(0);   // padding columns stay zero
    __syncthreads();
    for (int j = 0; j < B.np; ++j) {
        for (int t = tid; t < bb; t += nt) {
            const int i = t / b, k = t - i * b;
            const int ci = j * b + i, ck = j * b + k;
            const int sidx = i * ld + k;
            if (i == k) {
                double s = O.cd[ci];
                if constexpr (mixed) s *= O.dsc[ci] * O.dsc[ci];
                if (j > 0) {
                    const double cc = (double)c2s[ci - b];
                    s -= cc * (cc * (double)Sb[sidx]);   // not cc^2 (range at tiny couplings)
                }
                Sb[sidx] = (T)s;
            } else {
                T s = T(0);
                const int dk = k > i ? k - i : i - k, cl = k > i ? ci : ck;   // the coupling of the lower cell
                if (dk == 1) s -= mixed ? (T)scaled3(O, O.c0, 2u, 1, cl) : (T)O.c0[cl];
                if (dk == n0) s -= mixed ? (T)scaled3(O, O.c1, 8u, n0, cl) : (T)O.c1[cl];
                if (j > 0) s -= c2s[ci - b] * Sb[sidx] * c2s[ck - b];
                Sb[sidx] = s;
            }
        }
        __syncthreads();
        gj_cta<T>(Sb, b, ld, rowbuf, colbuf, ipb, bad);
        T* Fj = F + (size_t)j * plane_stride(b);
        for (int t = tid; t < b * ld; t += nt) Fj[t] = Sb[t];
        __syncthreads();
    }
    asm volatile("fence.proxy.async;" ::: "memory");
    __syncthreads();
}

// The sweeps' copies: stages of `cap` entries filled by bulk copies (full) and
// handed back by the computing warps (empty).  Every thread tracks its own
// position; waits are bounded.
template <typename T>
struct Pipe3 {
    uint64_t *full, *empty;
    T* buf;
    size_t cap;
    int st;            // stages
    int slot;          // position of this thread
    uint32_t ph;
    uint32_t issued;   // copies issued (the issuing thread)
    bool ok;           // no wait of this thread ran out
    __device__ __forceinline__ void next() {
        if (++slot == st) {
            slot = 0;
            ph ^= 1u;
        }
    }
};

// One poll, then the bounded wait.
__device__ __forceinline__ bool wait3(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok || mbar_wait(bar, parity);
}
__device__ __forceinline__ void bar_consumers() { asm volatile("bar.sync 1, %0;" ::"n"(32 * NW3) : "memory"); }
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// Two sweeps over the planes for NR right-hand sides in W ([NR][nc], block
// order): on entry the scaled right-hand sides, on exit the scaled solutions.
// The plane inverses (symmetric, rows padded to 16 bytes) stream from global
// memory through the bulk-copy (TMA) engine in chunks of stage_rows rows;
// the last warp issues the copies, up to Pipe3::st chunks ahead of their use
// and across planes, so that only the dependence of a plane on the one
// before it is waited for.  The other NW3 warps form S v: a lane takes RW
// consecutive rows (read as columns: consecutive lanes, consecutive words),
// nrw warps cover the rows of a plane, and G groups of them take every G-th
// column; the groups' partial sums meet in red, and the thread that adds
// them writes the plane's result and its part of the next plane's input
// (vb[c][q]).  Two barriers of the computing warps per plane.
// RW: 4, 2 or 1 in FP32, so that a plane of up to 128, 64 or 32 cells is one
// warp wide (one row per lane took 18 instructions per column and 5400 cycles
// per plane of 126 cells, four rows a quarter of the instructions); 1 in FP64,
// where the FMAs bind.
// GC: the groups, where they are known at compile time (planes of up to 32 RW
// cells), else 0.
template <typename T, int NR, int RW, int GC>
__device__ __forceinline__ void sweeps3_rw(const Box3& B, const T* c2s, T* W, T* vb, T* red, Pipe3<T>& pref, int* bad) {
    Pipe3<T> pp = pref;   // in registers
    constexpr int VS = NR == 3 ? 4 : NR;   // stride of vb
    const int b = B.b, nc = B.nc, ld = plane_ld(b), np = B.np;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    constexpr int CR = stage_rows(sizeof(T));
    const int nplane = 2 * np - 1;                    // forward planes, then backward planes np-2 .. 0
    const int nrw = GC > 0 ? NW3 / GC : (b + 32 * RW - 1) / (32 * RW), G = GC > 0 ? GC : NW3 / nrw;
    const int RP = nrw * 32 * RW;
    const int g = warp / nrw, r0 = ((warp - g * nrw) * 32 + lane) * RW;
    const bool act = g < G && r0 < b;
    // the thread's result rows: row rs of right-hand sides qs, qs + qd, ...
    const int rs = tid % RP, qs = tid / RP, qd = (32 * NW3) / RP;
    const bool sum = rs < b && qs < qd;
    if (sum)
        for (int q = qs; q < NR; q += qd) vb[rs * VS + q] = W[q * nc + rs];
    bar_consumers();
    for (int p = 0; p < nplane; ++p) {
        const int j = p < np ? p : 2 * np - 2 - p;
        T acc[NR][RW];
#pragma unroll
        for (int q = 0; q < NR; ++q)
#pragma unroll
            for (int e = 0; e < RW; ++e) acc[q][e] = T(0);
        for (int c0 = 0; c0 < b; c0 += CR) {
            if (pp.ok && !wait3(&pp.full[pp.slot], pp.ph)) {
                pp.ok = false;
                *bad = 1;
            }
            if (act) {
                const int cr = min(CR, b - c0);
                const T* S = pp.buf + pp.slot * pp.cap + g * ld + r0;
                const T* v0 = vb + (c0 + g) * VS;
                const int sS = G * ld;
                if (GC > 0 && cr == CR) {
#pragma unroll
                    for (int i = 0; i < (GC > 0 ? CR / GC : 1); ++i) {
                        T sr[RW], v[VS];
                        ldv<T, RW>(S + i * sS, sr);
                        ldv<T, VS>(v0 + i * GC * VS, v);
#pragma unroll
                        for (int q = 0; q < NR; ++q)
#pragma unroll
                            for (int e = 0; e < RW; ++e) acc[q][e] += sr[e] * v[q];
                    }
                } else {
                    const int sv = G * VS;
#pragma unroll 4
                    for (int c = g; c < cr; c += G) {
                        T sr[RW], v[VS];
                        ldv<T, RW>(S, sr);
                        ldv<T, VS>(v0, v);
                        S += sS;
                        v0 += sv;
#pragma unroll
                        for (int q = 0; q < NR; ++q)
#pragma unroll
                            for (int e = 0; e < RW; ++e) acc[q][e] += sr[e] * v[q];
                    }
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&pp.empty[pp.slot]);
            pp.next();
        }
        if (act) {
#pragma unroll
            for (int q = 0; q < NR; ++q) {
                T* d = red + (q * G + g) * RP + r0;
                if constexpr (RW == 4) stv4(d, acc[q][0], acc[q][1], acc[q][2], acc[q][3]);
                else {
#pragma unroll
                    for (int e = 0; e < RW; ++e) d[e] = acc[q][e];
                }
            }
        }
        bar_consumers();
        if (sum)
            for (int q = qs; q < NR; q += qd) {
                const T* d = red + q * G * RP + rs;
                T y0 = T(0), y1 = T(0);
                int k = 0;
#pragma unroll 4
                for (; k + 1 < G; k += 2) {
                    y0 += d[k * RP];
                    y1 += d[(k + 1) * RP];
                }
                if (k < G) y0 += d[k * RP];
                T y = y0 + y1;
                T* w = W + q * nc + j * b + rs;
                T v = T(0);
                if (p < np) {
                    w[0] = y;
                    if (p + 1 < np) v = w[b] + c2s[j * b + rs] * y;
                } else {
                    y += w[0];
                    w[0] = y;
                }
                if (p + 1 >= np && j > 0) v = c2s[(j - 1) * b + rs] * y;
                vb[rs * VS + q] = v;
            }
        bar_consumers();
    }
    pref.slot = pp.slot;
    pref.ph = pp.ph;
    pref.ok = pp.ok;
}

// issues the sweeps' copies (one lane of the last warp)
template <typename T>
__device__ void sweeps3_copies(const Box3& B, const T* __restrict__ F, Pipe3<T>& pref, int* bad) {
    Pipe3<T> pp = pref;   // in registers
    const int b = B.b, ld = plane_ld(b), np = B.np;
    constexpr int CR = stage_rows(sizeof(T));
    const size_t ps = plane_stride(b);
    for (int p = 0; p < 2 * np - 1 && pp.ok; ++p) {
        const T* Fj = F + (size_t)(p < np ? p : 2 * np - 2 - p) * ps;
        for (int c0 = 0; c0 < b; c0 += CR) {
            if (!wait3(&pp.empty[pp.slot], pp.ph ^ 1u)) {
                pp.ok = false;
                *bad = 1;
                break;
            }
            const uint32_t bytes = (uint32_t)(sizeof(T) * (size_t)min(CR, b - c0) * ld);
            mbar_expect_tx(&pp.full[pp.slot], bytes);
            bulk_g2s(pp.buf + pp.slot * pp.cap, Fj + (size_t)c0 * ld, bytes, &pp.full[pp.slot]);
            ++pp.issued;
            pp.next();
        }
    }
    pref = pp;
}

template <typename T, int NR>
__device__ void sweeps3(const Box3& B, const T* __restrict__ F, const T* c2s, T* W, T* vb, T* red, Pipe3<T>& pp,
                        int* bad) {
    if (threadIdx.x >= 32 * NW3) {
        if (threadIdx.x == 32 * NW3) sweeps3_copies<T>(B, F, pp, bad);
        __syncwarp();
    } else if constexpr (sizeof(T) == 8) {
        sweeps3_rw<T, NR, 1, 0>(B, c2s, W, vb, red, pp, bad);
    } else {
        if (B.b <= 32) sweeps3_rw<T, NR, 1, NW3>(B, c2s, W, vb, red, pp, bad);
        else if (B.b <= 64) sweeps3_rw<T, NR, 2, NW3>(B, c2s, W, vb, red, pp, bad);
        else if (B.b <= 128) sweeps3_rw<T, NR, 4, NW3>(B, c2s, W, vb, red, pp, bad);
        else sweeps3_rw<T, NR, 4, NW3 / 2>(B, c2s, W, vb, red, pp, bad);
    }
}

// Maximum norms by the bits of |v|, whose order is that of the values, with NaN
// above infinity: fmaxf would drop a NaN, and a solve whose every entry is one
// would count as converged.
__device__ __forceinline__ unsigned abs_bits(float v) { return __float_as_uint(v) & 0x7fffffffu; }
__device__ __forceinline__ void warp_max_to(unsigned int* a, unsigned v) {
    v = __reduce_max_sync(0xffffffffu, v);
    if ((threadIdx.x & 31) == 0) atomicMax(a, v);
}

// Solves A x_q = rhs_q for NR right-hand sides with the whole CTA: sweeps
// with the kept factor (FP32 in the mixed form, FP64 in the FP64 form) and
// refinement with FP64 residuals from X = 0, the iterate X in FP64; in the mixed
// form the sweeps take the scaled residual D r and X gets D times their result.
// High-contrast boxes reach a residual floor above what a fixed tolerance can ask
// for, so the refinement runs to that floor: it stops
// when every right-hand side has |r| <= 1e-3 ir_tol |b| (scaled max norms),
// or has |r| <= ir_tol |b| and no longer halves its residual per step.  The
// FP64 form (a direct solve, then refinement with the same rule, at most 4
// sweep pairs) never reports non-convergence.  Returns the number of sweep
// pairs.
template <typename T, int NR, typename Rhs>
__device__ int solve3_n(const Box3& B, const Ops3& O, const T* F, const T* c2s, double* X, T* W, T* vb, T* red,
                        Pipe3<T>& pp, unsigned int* nrm, const Rhs& rhs, double tol, int max_ir, int* noconv, int* bad) {
    constexpr bool mixed = std::is_same<T, float>::value;
    const int nc = B.nc, tid = threadIdx.x, nt = blockDim.x;
    const int s1 = B.n[B.a0], s2 = B.b;
    const int mit = mixed ? max_ir : 4;
    if (*bad) return 0;   // a staged copy failed earlier: the buffers are not usable
    // |b|, |r|, |r| of the previous step (inf), and (mixed form) the largest high word of b, or a bound of it
    if (tid < 4 * NR3) nrm[tid] = tid < 2 * NR3 || tid >= 3 * NR3 ? 0u : 0x7f800000u;
    __syncthreads();
    // mixed form: the FP32 vectors of right-hand side q stand for their values times 2^-shift(q)
    auto shift = [&](int q) { return norm_shift(nrm[3 * NR3 + q]); };
    if constexpr (mixed) {
#pragma unroll
        for (int q = 0; q < NR; ++q) {
            warp_max_to(&nrm[3 * NR3 + q], rhs.top(q, tid, nt));
        }
        __syncthreads();
    }
#pragma unroll
    for (int q = 0; q < NR; ++q) {
        unsigned bn = 0u;
        const int ex = mixed ? shift(q) : 0;
        for (int t = tid; t < nc; t += nt) {
            const double v = rhs(q, t);
            X[q * nc + t] = 0.0;
            if constexpr (mixed) {
                const float w = d2f_near(O.dsc[t] * v, ex);
                W[q * nc + t] = w;
                bn = max(bn, abs_bits(w));
            } else {
                W[q * nc + t] = v;
                bn = max(bn, abs_bits((float)v));
            }
        }
        warp_max_to(&nrm[q], bn);
    }
    __syncthreads();
    // done: every residual at its floor; reached: every residual within tol
    auto test = [&](bool& reached) {
        bool done = true;
        reached = true;
        for (int q = 0; q < NR; ++q) {
            const double bn = (double)__uint_as_float(nrm[q]), rn = (double)__uint_as_float(nrm[NR3 + q]);
            const double rp = (double)__uint_as_float(nrm[2 * NR3 + q]);
            if (!(bn == 0.0 || rn <= 1e-3 * tol * bn || (rn <= tol * bn && rn > 0.5 * rp))) done = false;
            if (!(bn == 0.0 || rn <= tol * bn)) reached = false;
        }
        return done;
    };
    bool reached = false, done = false;
    int it = 0;
    for (; !done && it < mit; ++it) {
        sweeps3<T, NR>(B, F, c2s, W, vb, red, pp, bad);
        __syncthreads();
        if (*bad) break;
#pragma unroll
        for (int q = 0; q < NR; ++q) {
            const int ex = mixed ? shift(q) : 0;
            for (int t = tid; t < nc; t += nt) {
                if constexpr (mixed) X[q * nc + t] += O.dsc[t] * f2d_bits(W[q * nc + t], ex);
                else X[q * nc + t] += W[q * nc + t];
            }
        }
        if (tid < NR3) {
            nrm[2 * NR3 + tid] = it == 0 ? 0x7f800000u : nrm[NR3 + tid];
            nrm[NR3 + tid] = 0u;
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < NR; ++q) {
            unsigned rn = 0u;
            const int ex = mixed ? shift(q) : 0;
            for (int t = tid; t < nc; t += nt) {
                const double v = resid3<mixed>(O, s1, s2, X + q * nc, rhs(q, t), t);
                if constexpr (mixed) {
                    const float w = d2f_near(O.dsc[t] * v, ex);
                    W[q * nc + t] = w;
                    rn = max(rn, abs_bits(w));
                } else {
                    W[q * nc + t] = v;
                    rn = max(rn, abs_bits((float)v));
                }
            }
            warp_max_to(&nrm[NR3 + q], rn);
        }
        __syncthreads();
        done = test(reached);
        if (!done && it == mit - 1 && !reached && tid == 0 && mixed) *noconv = 1;
        __syncthreads();
    }
    __syncthreads();
    return it;
}

template <typename T, typename Rhs>
__device__ int solve3(int nr, const Box3& B, const Ops3& O, const T* F, const T* c2s, double* X, T* W, T* vb, T* red,
                      Pipe3<T>& pp, unsigned int* nrm, const Rhs& rhs, double tol, int max_ir, int* noconv, int* bad) {
    switch (nr) {   // the sweeps' work is that of the right-hand sides there are
        case 1: return solve3_n<T, 1>(B, O, F, c2s, X, W, vb, red, pp, nrm, rhs, tol, max_ir, noconv, bad);
        case 2: return solve3_n<T, 2>(B, O, F, c2s, X, W, vb, red, pp, nrm, rhs, tol, max_ir, noconv, bad);
        case 3: return solve3_n<T, 3>(B, O, F, c2s, X, W, vb, red, pp, nrm, rhs, tol, max_ir, noconv, bad);
        default: return solve3_n<T, 4>(B, O, F, c2s, X, W, vb, red, pp, nrm, rhs, tol, max_ir, noconv, bad);
    }
}

// f |c| + Dirichlet / Neumann data + Robin data lam (may be null) of cell t
__device__ double source_rhs3(const Box3& B, const Ops3& O, const MemberDev& md, const double* fm, const double* lam,
                              int t) {
    const Ijk c = bcoord(B, t);
    const double vol = md.h[0] * md.h[1] * md.h[2];
    double r = fm[gidx(B, c)] * vol;
    const unsigned char m = O.nb[t];
    if ((m & 63) != 63) {
        for (int sid = 0; sid < 6; ++sid) {
            const int a = sid >> 1;
            if (m & B.bit[sid]) continue;
            const int e = B.soff[sid] + side_e(B, sid, c);
            if (B.kind[sid] == 1) r += O.bT[e] * B.val[sid];
            else if (B.kind[sid] == 0) r -= vol / md.h[a] * B.val[sid];
            else if (lam) r += O.bT[e] * lam[e];
        }
    }
    return r;
}

// Right-hand sides of a group of basis solves; sk[q] < 0 marks the particular
// problem on hat-Omega_i (a variant of Step 4), whose vector bs is stored.
struct RhsBasis3 {
    const Box3* B;
    const Ops3* O;
    const double* bs;
    int sk[NR3], mk[NR3], bit[NR3];   // side, function, and the neighbour bit that cells of the side lack
    __device__ double operator()(int q, int t) const {
        if (sk[q] < 0) return bs[t];
        if (O->nb[t] & bit[q]) return 0.0;
        const int sid = sk[q];
        const int ls = B->n[B->ts[sid]], lt = B->n[B->tt[sid]];
        const int e = side_e(*B, sid, bcoord(*B, t)), ct = e / ls;
        return O->bT[B->soff[sid] + e] * psi3(mk[q], e - ct * ls, ls, ct, lt);
    }
    // this thread's part of the largest high word of D b: at most that of its side's face coefficients (|psi| <= 1)
    __device__ unsigned top(int q, int tid, int nt) const {
        unsigned h = 0u;
        if (sk[q] < 0) {
            for (int t = tid; t < B->nc; t += nt) h = max(h, abs_hi(O->dsc[t] * bs[t]));
            return h;
        }
        const int sid = sk[q], a = sid >> 1, ls = B->n[B->ts[sid]];
        for (int f = B->soff[sid] + tid; f < B->soff[sid + 1]; f += nt) {
            const int e = f - B->soff[sid], ct = e / ls;
            const int t = (e - ct * ls) * B->bs[B->ts[sid]] + ct * B->bs[B->tt[sid]] + ((sid & 1) ? (B->n[a] - 1) * B->bs[a] : 0);
            h = max(h, abs_hi(O->dsc[t] * O->bT[f]));
        }
        return h;
    }
};

struct RhsStored3 {
    const double* b;
    const double* dsc;   // (mixed form)
    int nc;
    __device__ double operator()(int, int t) const { return b[t]; }
    __device__ unsigned top(int, int tid, int nt) const {
        unsigned h = 0u;
        for (int t = tid; t < nc; t += nt) h = max(h, abs_hi(dsc[t] * b[t]));
        return h;
    }
};

// Shared-memory layout.  Persistent: the operator, neighbour bits, scaled
// plane coupling, boundary faces, and (smoothing) Robin data and (one right-
// hand side) the stored right-hand side.  Overlaid: the factor phase (the
// panels of the register inverses, or the plane Schur block where it is too
// wide for them) and the solve phase (work vectors, sweep input, partial
// sums and the stages of the streamed plane inverses, as many as fit, two at
// least).  The FP64 iterates live in global scratch (one slot per CTA).
__host__ __device__ inline void box3_dims(int nx, int ny, int nz, int* b, int* npl) {
    int n[3] = {nx, ny, nz};
    int a2 = 2;
    for (int a = 1; a >= 0; --a)
        if (n[a] > n[a2]) a2 = a;
    *b = nx * ny * nz / n[a2];
    *npl = n[a2];
}

// partial sums of the sweeps per right-hand side: G RP of sweeps3_rw
__host__ __device__ inline size_t red3(int tsz, int b) {
    const int rw = tsz == 8 || b <= 32 ? 1 : b <= 64 ? 2 : 4;
    return (size_t)32 * NW3 * rw;
}

struct Lay3 {
    size_t fixed;    // persistent bytes
    size_t fac;      // factor phase
    size_t work;     // solve phase without the stages
    size_t stage;    // bytes of one stage
    int st;          // stages
    size_t total;
};

__host__ __device__ inline Lay3 lay3(int tsz, int nx, int ny, int nz, int nr, bool stored_rhs, bool robin) {
    int b, npl;
    box3_dims(nx, ny, nz, &b, &npl);
    const bool mixed = tsz == 4;
    const size_t nc = (size_t)nx * ny * nz, ld = (size_t)plane_ld(b);
    const size_t per = 2 * ((size_t)nx * ny + (size_t)ny * nz + (size_t)nx * nz);
    Lay3 L;
    L.fixed = align16(sizeof(double) * nc) * 4;                               // cd c0 c1 c2
    if (mixed) L.fixed += align16(sizeof(double) * nc) + align16(tsz * nc);   // dsc c2s
    L.fixed += align16(nc);                                                    // nb
    L.fixed += align16(sizeof(double) * per) * (robin ? 3 : 2);                // bT bB (lam)
    if (stored_rhs) L.fixed += align16(sizeof(double) * nc);                   // bsrc
    L.fac = b <= GB3 ? align16((size_t)tsz * (GJW3 + (mixed ? 2 * nc : 0)))
                     : align16(tsz * b * ld) + align16(tsz * ld) + align16((size_t)tsz * b) + 16;
    L.work = align16(tsz * nr * nc) + align16((size_t)tsz * NR3 * b) + align16((size_t)tsz * nr * red3(tsz, b));
    const int rows = b < stage_rows(tsz) ? b : stage_rows(tsz);
    L.stage = tsz * rows * ld;
    const size_t tail = 64 + 32 + 2 * sizeof(uint64_t) * ST3;
    L.st = ST3;
    while (L.st > 2 && L.fixed + L.work + L.st * L.stage + tail > 226 * 1024) --L.st;
    const size_t sol = L.work + L.st * L.stage;
    L.total = L.fixed + (L.fac > sol ? L.fac : sol) + tail;
    return L;
}

// Right-hand sides of a basis round: NR3, fewer where the work vectors of so
// many do not fit (mixed form, boxes that nearly fill shared memory with their
// operator: 3 x 22 x 34 cells take three, 7 x 15 x 22 two).
__host__ __device__ inline int round3(int tsz, int nx, int ny, int nz) {
    int nr = NR3;
    while (nr > 1 && lay3(tsz, nx, ny, nz, nr, false, false).total > SMEM_LOCAL3D) --nr;
    return nr;
}

template <typename T>
struct Carve3 {
    Ops3 O;
    T* c2s;
    double* lam;
    double* bsrc;
    T* fac;                          // factor phase
    double* X;                       // solve phase (global scratch)
    T *W, *vb, *red;
    Pipe3<T> pp;
    int* flags;
    unsigned int* nrm;
    size_t end;   // bytes of shared memory the layout takes
};

template <typename T>
__device__ Carve3<T> carve3(unsigned char* base, const Box3& B, int nr, bool stored_rhs, bool robin, double* xglobal) {
    constexpr bool mixed = std::is_same<T, float>::value;
    Carve3<T> C;
    const size_t nc = B.nc, b = B.b;
    const size_t per = B.soff[6];
    const Lay3 L = lay3((int)sizeof(T), B.n[0], B.n[1], B.n[2], nr, stored_rhs, robin);
    size_t o = 0;
    auto take = [&](size_t bytes) { unsigned char* p = base + o; o += align16(bytes); return p; };
    C.O.cd = (double*)take(sizeof(double) * nc);
    C.O.c0 = (double*)take(sizeof(double) * nc);
    C.O.c1 = (double*)take(sizeof(double) * nc);
    C.O.c2 = (double*)take(sizeof(double) * nc);
    if (mixed) {
        C.O.dsc = (double*)take(sizeof(double) * nc);
        C.c2s = (T*)take(sizeof(T) * nc);
    } else {
        C.O.dsc = nullptr;
        C.c2s = (T*)C.O.c2;
    }
    C.O.nb = (unsigned char*)take(nc);
    C.O.bT = (double*)take(sizeof(double) * per);
    C.O.bB = (double*)take(sizeof(double) * per);
    C.lam = robin ? (double*)take(sizeof(double) * per) : nullptr;
    C.bsrc = stored_rhs ? (double*)take(sizeof(double) * nc) : nullptr;
    C.X = xglobal;
    const size_t u0 = o;
    C.fac = (T*)(base + u0);
    C.W = (T*)take(sizeof(T) * nr * nc);
    C.vb = (T*)take(sizeof(T) * NR3 * b);
    C.red = (T*)take(sizeof(T) * nr * red3((int)sizeof(T), (int)b));
    C.pp.buf = (T*)(base + o);
    C.pp.cap = L.stage / sizeof(T);
    C.pp.st = L.st;
    C.pp.slot = 0;
    C.pp.ph = 0u;
    C.pp.issued = 0u;
    C.pp.ok = true;
    o += L.st * L.stage;
    if (o < u0 + L.fac) o = u0 + L.fac;
    C.flags = (int*)take(32);
    C.nrm = (unsigned int*)take(64);
    C.pp.full = (uint64_t*)take(sizeof(uint64_t) * ST3);
    C.pp.empty = (uint64_t*)take(sizeof(uint64_t) * ST3);
    C.end = o;
    if (threadIdx.x == 0) {
        C.flags[0] = 0;
        C.flags[1] = 0;
        C.flags[2] = 0;
        for (int s = 0; s < ST3; ++s) {
            mbar_init(&C.pp.full[s], 1);
            mbar_init(&C.pp.empty[s], NW3);
        }
    }
    return C;
}

// After a wait that ran out: no copy may target the shared memory of a CTA
// that has left, so the issuing thread waits (bounded) for its last copy into
// each stage.
template <typename T>
__device__ void drain3(Pipe3<T>& pp) {
    if (threadIdx.x != 32 * NW3) return;
    for (int s = 0; s < pp.st && s < (int)pp.issued; ++s) {
        const uint32_t k = (pp.issued - 1 - s) / pp.st;   // rounds before the stage's last copy
        mbar_wait(&pp.full[s], k & 1u);
    }
}

}  // namespace

// ---------------------------------------------------------------------------
// Steps 1, 2, 4 and 6 of Algorithm 1 for 3D subdomains (one CTA per job).
// The factor goes to the job's slot: the kept smoothing factor (basis job
// with alpha_basis == alpha_smooth, or the Step 6 job), or scratch.
// ---------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(T3, 1) k_local3d(DevPtrs P, MethodDev Mth, const Job* jobs) {
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr bool mixed = std::is_same<T, float>::value;
    const Job job = jobs[blockIdx.x];
    const SubDev sd = P.sub[job.item];
    const MemberDev& md = P.mem[sd.member];
    const bool part = job.type == JOB_PART;
    __shared__ Box3 B;
    __shared__ int round;   // right-hand sides per round
    if (threadIdx.x == 0) {
        if (part) setup_box3(B, md, sd.lo, sd.hi, Mth.alpha_b);
        else setup_box3(B, md, sd.loh, sd.hih, job.type == JOB_SFACT ? Mth.alpha_s : Mth.alpha_b);
        round = part ? 1 : round3((int)sizeof(T), B.n[0], B.n[1], B.n[2]);
    }
    __syncthreads();
    if (!mrcm_check(P.status,
                    lay3((int)sizeof(T), B.n[0], B.n[1], B.n[2], round, part, false).total <= mrcm_dyn_smem_bytes(),
                    6, 0))
        return;   // uniform
    Carve3<T> C = carve3<T>(smem, B, round, part, false, P.xs + (size_t)blockIdx.x * P.xs_stride);
    build_ops3(B, md, P, C.O, mixed);
    if constexpr (mixed) {
        for (int t = threadIdx.x; t < B.nc; t += blockDim.x) C.c2s[t] = scaled3(C.O, C.O.c2, 32u, B.b, t);
        __syncthreads();
    }
    T* F;
    if (part) F = (T*)P.fac_part + (size_t)job.item * P.part_stride;
    else if (job.type == JOB_SFACT || Mth.same_alpha) F = (T*)P.fac + (size_t)job.item * P.fac_stride;
    else F = (T*)P.fac_aux + (size_t)job.item * P.fac_stride;
    if (B.b <= GB3) {
        const T *c0s, *c1s;
        if constexpr (mixed) {
            T* cs = C.fac + GJW3;   // in-plane couplings in T, in the factor phase's overlay
            for (int t = threadIdx.x; t < B.nc; t += blockDim.x) {
                cs[t] = scaled3(C.O, C.O.c0, 2u, 1, t);
                cs[B.nc + t] = scaled3(C.O, C.O.c1, 8u, B.n[B.a0], t);
            }
            c0s = cs;
            c1s = cs + B.nc;
        } else {
            c0s = C.O.c0;
            c1s = C.O.c1;
        }
        factor3_reg<T>(B, C.O, c0s, c1s, C.c2s, F, C.fac, &C.flags[0]);
    } else {
        const size_t ld = plane_ld(B.b);
        T* Sb = C.fac;
        T* rowbuf = (T*)((unsigned char*)Sb + align16(sizeof(T) * B.b * ld));
        T* colbuf = (T*)((unsigned char*)rowbuf + align16(sizeof(T) * ld));
        T* ipb = (T*)((unsigned char*)colbuf + align16(sizeof(T) * B.b));
        factor3_smem<T>(B, C.O, C.c2s, F, Sb, rowbuf, colbuf, ipb, &C.flags[0]);
    }
    if constexpr (mixed) side_diag3(B, C.O);
    if (C.flags[0] && threadIdx.x == 0) {
        atomicOr(&P.status[0], ST_NOT_SPD);
        atomicExch(&P.status[2], job.item);
    }
    // with the particular problem on hat-Omega_i (a variant) it is the basis
    // job's last right-hand side, k = nbasis, its vector kept in global memory
    const bool hat_part = job.type == JOB_BASIS && Mth.part_hat;
    const int nrhs = job.type == JOB_BASIS ? sd.nbasis + (hat_part ? 1 : 0) : (part ? 1 : 0);
    if (nrhs == 0) return;

    const int npsi = Mth.npsi;
    const double vol = md.h[0] * md.h[1] * md.h[2];
    const double* fm = P.f + md.cell_off;
    double* bsg = hat_part ? P.bsrc + (size_t)job.item * P.box_stride : nullptr;
    if (part || hat_part) {
        double* bs = part ? C.bsrc : bsg;
        for (int t = threadIdx.x; t < B.nc; t += blockDim.x) bs[t] = source_rhs3(B, C.O, md, fm, nullptr, t);
        __syncthreads();
    }
    // Omega_i in the box (in shared memory: indexed by the axis at run time)
    __shared__ int nI[3], off[3];
    if (threadIdx.x == 0)
        for (int a = 0; a < 3; ++a) {
            nI[a] = sd.hi[a] - sd.lo[a];
            off[a] = sd.lo[a] - B.lo[a];
        }
    __syncthreads();
    const int nI0 = nI[0], nI1 = nI[1], nIc = nI0 * nI1 * nI[2];
    const float r0i = 1.f / (float)nI0, r01 = 1.f / (float)(nI0 * nI1);
    const int tO = off[0] * B.bs[0] + off[1] * B.bs[1] + off[2] * B.bs[2];   // its first cell
    const long long gO = B.g0 + off[0] * B.gs[0] + off[1] * (long long)B.gs[1] + off[2] * (long long)B.gs[2];
    int maxit = 0, nsolve = 0;
    for (int k0 = 0; k0 < nrhs; k0 += round) {
        const int nr = min(round, nrhs - k0);
        int it;
        RhsBasis3 rb;
        rb.B = &B;
        rb.O = &C.O;
        rb.bs = bsg;
        if (!part) {
#pragma unroll
            for (int q = 0; q < NR3; ++q) {
                const int k = k0 + q;
                int qq = k / npsi;
                rb.mk[q] = k % npsi;
                rb.sk[q] = k >= sd.nbasis ? -1 : 0;
                if (k < sd.nbasis)
                    for (int sid = 0; sid < 6; ++sid)
                        if (sd.side_mask & (1 << sid)) {
                            if (qq == 0) { rb.sk[q] = sid; break; }
                            --qq;
                        }
                rb.bit[q] = rb.sk[q] >= 0 ? B.bit[rb.sk[q]] : 0;
            }
            it = solve3<T>(nr, B, C.O, F, C.c2s, C.X, C.W, C.vb, C.red, C.pp, C.nrm, rb, Mth.ir_tol, Mth.max_ir,
                           &C.flags[1], &C.flags[2]);
        } else {
            RhsStored3 rs{C.bsrc, C.O.dsc, B.nc};
            it = solve3_n<T, 1>(B, C.O, F, C.c2s, C.X, C.W, C.vb, C.red, C.pp, C.nrm, rs, Mth.ir_tol, Mth.max_ir,
                                &C.flags[1], &C.flags[2]);
        }
        maxit = max(maxit, it);
        nsolve += it * nr;
        __syncthreads();
        // ---- outputs: restriction to Omega_i, Gamma_i velocities and moments ----
        for (int q = 0; q < nr; ++q) {
            const double* x = C.X + (size_t)q * B.nc;
            const bool pq = part || k0 + q >= sd.nbasis;   // the particular problem
            double* psi_out = pq ? P.pbar + (size_t)job.item * P.ncell_i_max
                                 : P.Psi + ((size_t)job.item * P.nbasis_max + k0 + q) * P.ncell_i_max;
            for (int ci = threadIdx.x; ci < nIc; ci += blockDim.x) {
                const int z = (int)(((float)ci + 0.5f) * r01), xy = ci - z * nI0 * nI1;
                const int y = (int)(((float)xy + 0.5f) * r0i);
                psi_out[ci] = x[tO + (xy - y * nI0) * B.bs[0] + y * B.bs[1] + z * B.bs[2]];
            }
        }
        __syncthreads();
        // one warp per right-hand side and side: velocities, and their moments by a warp reduction
        for (int w = threadIdx.x >> 5; w < nr * 6; w += T3 / 32) {
            const int q = w / 6, sid = w - 6 * (w / 6), lane = threadIdx.x & 31;
            if (!(sd.side_mask & (1 << sid))) continue;
            const double* x = C.X + (size_t)q * B.nc;
            const int k = k0 + q;
            const bool pq = part || k >= sd.nbasis;
            int skq = -1, mkq = 0;
            if (!pq) {
#pragma unroll
                for (int e = 0; e < NR3; ++e)
                    if (e == q) {
                        skq = rb.sk[e];
                        mkq = rb.mk[e];
                    }
            }
            const int a = sid >> 1;
            const int ts = B.ts[sid], tt = B.tt[sid];
            const int ls = nI[ts], lt = nI[tt];
            const double area = vol / md.h[a];
            const double rarea = 1.0 / area;
            double* ug = pq ? P.ubg + ((size_t)job.item * MRCM_MAXSIDE + sid) * P.side_max
                            : P.Ug + (((size_t)job.item * P.nbasis_max + k) * MRCM_MAXSIDE + sid) * P.side_max;
            double fmv[3] = {0.0, 0.0, 0.0}, pmv[3] = {0.0, 0.0, 0.0};
            const int cn = off[a] + ((sid & 1) ? nI[a] - 1 : 0);   // the side's cells along its normal
            const bool inner = (sid & 1) ? cn + 1 < B.n[a] : cn > 0;
            const int t0 = tO + (cn - off[a]) * B.bs[a];
            const long long g0 = gO + (cn - off[a]) * (long long)B.gs[a];
            for (int e = lane; e < ls * lt; e += 32) {
                const int ct = e / ls, cs = e - ct * ls;
                const int tL = t0 + cs * B.bs[ts] + ct * B.bs[tt];
                const double pL = x[tL];
                const long long gL = g0 + cs * (long long)B.gs[ts] + ct * (long long)B.gs[tt];
                const double hkL = P.hk[(md.cell_off + gL) * 3 + a];
                double uo, pi;
                if (inner) {
                    const long long gf = (sid & 1) ? gL : gL - B.gs[a];
                    const double Tf = P.Tf[(md.cell_off + gf) * 3 + a];
                    uo = Tf * (pL - x[(sid & 1) ? tL + B.bs[a] : tL - B.bs[a]]) * rarea;
                    pi = pL - uo * hkL;
                } else {
                    const int bcs = off[ts] + cs, bct = off[tt] + ct;
                    const int eb = B.soff[sid] + bcs + B.n[ts] * bct;
                    const double lam = sid == skq ? psi3(mkq, bcs, B.n[ts], bct, B.n[tt]) : 0.0;
                    uo = C.O.bT[eb] * (pL - lam) * rarea;
                    pi = part ? C.O.bB[eb] * uo : pL - uo * hkL;
                }
                ug[e] = uo;
#pragma unroll
                for (int m = 0; m < 3; ++m)
                    if (m < npsi) {
                        const double ps = psi3(m, cs, ls, ct, lt);
                        fmv[m] += ps * uo * area;
                        pmv[m] += area * ps * pi;
                    }
            }
            const int slot = pq ? P.nbasis_max : k;
            double* mom = P.mom + (((size_t)job.item * (P.nbasis_max + 1) + slot) * MRCM_MAXSIDE + sid) * npsi * 2;
#pragma unroll
            for (int m = 0; m < 3; ++m)
                if (m < npsi) {
                    for (int o = 16; o; o >>= 1) {
                        fmv[m] += __shfl_xor_sync(0xffffffffu, fmv[m], o);
                        pmv[m] += __shfl_xor_sync(0xffffffffu, pmv[m], o);
                    }
                    if (lane == 0) {
                        mom[m * 2] = fmv[m];
                        mom[m * 2 + 1] = pmv[m];
                    }
                }
        }
        __syncthreads();
    }
    if (C.flags[2]) drain3(C.pp);
    if (threadIdx.x == 0) {
        atomicMax(&P.status[1], maxit);
        atomicAdd(&P.status[3], nsolve);
        if (C.flags[1]) atomicOr(&P.status[0], ST_NO_CONV);
        if (C.flags[2]) atomicOr(&P.status[0], ST_BAD);
    }
}

// ---------------------------------------------------------------------------
// Step 7 in 3D: one colour phase of a smoothing step (Sec. 3, Eqs.
// (sm_1)-(sm_2)), one CTA per subdomain of the colour, kept factor read from
// global memory.
// ---------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(T3, 1) k_smooth3d(DevPtrs P, MethodDev Mth, const int* items) {
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr bool mixed = std::is_same<T, float>::value;
    const int item = items[blockIdx.x];
    const SubDev sd = P.sub[item];
    const MemberDev& md = P.mem[sd.member];
    __shared__ Box3 B;
    if (threadIdx.x == 0) setup_box3(B, md, sd.loh, sd.hih, Mth.alpha_s);
    __syncthreads();
    if (!mrcm_check(P.status,
                    lay3((int)sizeof(T), B.n[0], B.n[1], B.n[2], 1, true, true).total <= mrcm_dyn_smem_bytes(), 6, 0))
        return;   // uniform
    Carve3<T> C = carve3<T>(smem, B, 1, true, true, P.xs + (size_t)blockIdx.x * P.xs_stride);
    // (the Jacobi scale comes out as in the factorisation: the same faces, the same arithmetic)
    build_ops3(B, md, P, C.O, mixed);
    if constexpr (mixed) {
        for (int t = threadIdx.x; t < B.nc; t += blockDim.x) C.c2s[t] = scaled3(C.O, C.O.c2, 32u, B.b, t);
        side_diag3(B, C.O);
    }
    // Robin data from the current solution: lambda = -beta u.n + pi (n outward of hat-Omega_i)
    const double* pst = P.p + md.cell_off;
    const double* ust = P.u + md.cell_off * 6;
    for (int f = threadIdx.x; f < B.soff[6]; f += blockDim.x) {
        const int sid = side_of(B, f), a = sid >> 1;
        if (B.kind[sid] != 2) continue;
        const long long g = face_cell(B, sid, f);
        const double un = ust[g * 6 + sid];
        C.lam[f] = -C.O.bB[f] * un + (pst[g] - un * P.hk[(md.cell_off + g) * 3 + a]);
    }
    __syncthreads();
    const double* fm = P.f + md.cell_off;
    for (int t = threadIdx.x; t < B.nc; t += blockDim.x) C.bsrc[t] = source_rhs3(B, C.O, md, fm, C.lam, t);
    __syncthreads();
    const T* F = (const T*)P.fac + (size_t)item * P.fac_stride;
    RhsStored3 rs{C.bsrc, C.O.dsc, B.nc};
    const int it = solve3_n<T, 1>(B, C.O, F, C.c2s, C.X, C.W, C.vb, C.red, C.pp, C.nrm, rs, Mth.ir_tol, Mth.max_ir,
                                  &C.flags[0], &C.flags[2]);
    if (C.flags[2]) drain3(C.pp);
    __syncthreads();
    // overwrite (u, p) on Omega_i with the restriction
    const int nI0 = sd.hi[0] - sd.lo[0], nI1 = sd.hi[1] - sd.lo[1], nI2 = sd.hi[2] - sd.lo[2];
    const int o0 = sd.lo[0] - B.lo[0], o1 = sd.lo[1] - B.lo[1], o2 = sd.lo[2] - B.lo[2];
    const int nIc = nI0 * nI1 * nI2;
    const float r0i = 1.f / (float)nI0, r01 = 1.f / (float)(nI0 * nI1);
    double* pw = P.p + md.cell_off;
    double* uw = P.u + md.cell_off * 6;
    const double* Tfm = P.Tf + md.cell_off * 3;
    const double vol = md.h[0] * md.h[1] * md.h[2];
    const double* x = C.X;
    for (int ci = threadIdx.x; ci < nIc; ci += blockDim.x) {
        const int z = (int)(((float)ci + 0.5f) * r01), xy = ci - z * nI0 * nI1;
        const int y = (int)(((float)xy + 0.5f) * r0i);
        const int c0 = xy - y * nI0 + o0, c1 = y + o1, c2 = z + o2;
        const int t = c0 * B.bs[0] + c1 * B.bs[1] + c2 * B.bs[2];
        const long long g = B.g0 + c0 + c1 * (long long)B.gs[1] + c2 * (long long)B.gs[2];
        if (!mrcm_check(P.status, g >= 0 && g < (long long)md.n[0] * md.n[1] * md.n[2], 7, g)) continue;
        const double pc = x[t];
        const unsigned char m = C.O.nb[t];
        pw[g] = pc;
        double uo[6];
#pragma unroll
        for (int sid = 0; sid < 6; ++sid) {
            const int a = sid >> 1;
            const double rarea = md.h[a] / vol;
            if (m & B.bit[sid]) {
                const long long gf = (sid & 1) ? g : g - B.gs[a];
                uo[sid] = Tfm[gf * 3 + a] * (pc - x[(sid & 1) ? t + B.bs[a] : t - B.bs[a]]) * rarea;
            } else {
                const int eb = B.soff[sid] + c0 * B.es[sid][0] + c1 * B.es[sid][1] + c2 * B.es[sid][2];
                if (B.kind[sid] == 2) uo[sid] = C.O.bT[eb] * (pc - C.lam[eb]) * rarea;
                else if (B.kind[sid] == 1) uo[sid] = C.O.bT[eb] * (pc - B.val[sid]) * rarea;
                else uo[sid] = B.val[sid];
            }
        }
#pragma unroll
        for (int sid = 0; sid < 6; ++sid) uw[g * 6 + sid] = uo[sid];
    }
    if (threadIdx.x == 0) {
        atomicMax(&P.status[1], it);
        atomicAdd(&P.status[3], it);
        if (C.flags[0]) atomicOr(&P.status[0], ST_NO_CONV);
        if (C.flags[2]) atomicOr(&P.status[0], ST_BAD);
    }
}

// ---------------------------------------------------------------------------
// Superposition in 3D (Eqs. (addu), (addp), (uhatphat)): p = pbar + sum_k
// X_k Psi_k on Omega_i; Gamma_i velocities ubar + sum_k X_k U_k; interior
// faces from the assembled pressure; physical faces from the data.
// ---------------------------------------------------------------------------
__global__ void k_assemble3d(DevPtrs P, const double* __restrict__ X) {
    extern __shared__ double ps3[];
    const int item = blockIdx.x;
    const SubDev sd = P.sub[item];
    const MemberDev& md = P.mem[sd.member];
    int nI[3];
    for (int a = 0; a < 3; ++a) nI[a] = sd.hi[a] - sd.lo[a];
    const int n = nI[0] * nI[1] * nI[2];
    const double* xs = X + sd.col0;
    const double* Psi = P.Psi + (size_t)item * P.nbasis_max * P.ncell_i_max;
    const double* pb = P.pbar + (size_t)item * P.ncell_i_max;
    for (int c = threadIdx.x; c < n; c += blockDim.x) {
        double v = pb[c];
        for (int k = 0; k < sd.nbasis; ++k) v += xs[k] * Psi[(size_t)k * P.ncell_i_max + c];
        ps3[c] = v;
    }
    __syncthreads();
    const double* Tf = P.Tf + md.cell_off * 3;
    const double* hk = P.hk + md.cell_off * 3;
    double* pw = P.p + md.cell_off;
    double* uw = P.u + md.cell_off * 6;
    const double vol = md.h[0] * md.h[1] * md.h[2];
    const int cst[3] = {1, nI[0], nI[0] * nI[1]};
    for (int ci = threadIdx.x; ci < n; ci += blockDim.x) {
        int c[3];
        c[0] = ci % nI[0];
        c[1] = (ci / nI[0]) % nI[1];
        c[2] = ci / (nI[0] * nI[1]);
        const long long g = (sd.lo[0] + c[0]) + (long long)md.n[0] * ((sd.lo[1] + c[1]) + (long long)md.n[1] * (sd.lo[2] + c[2]));
        if (!mrcm_check(P.status, g >= 0 && g < (long long)md.n[0] * md.n[1] * md.n[2], 7, g)) continue;
        const double pc = ps3[ci];
        pw[g] = pc;
        for (int sid = 0; sid < 6; ++sid) {
            const int a = sid >> 1;
            const bool hi = sid & 1;
            const bool edge = hi ? (c[a] == nI[a] - 1) : (c[a] == 0);
            const double rarea = md.h[a] / vol;
            const long long gs = a == 0 ? 1LL : a == 1 ? (long long)md.n[0] : (long long)md.n[0] * md.n[1];
            double uo;
            if (!edge) {
                const int cn = ci + (hi ? cst[a] : -cst[a]);
                const long long gf = hi ? g : g - gs;
                uo = Tf[gf * 3 + a] * (pc - ps3[cn]) * rarea;
            } else if (sd.side_mask & (1 << sid)) {
                const int ts = a == 0 ? 1 : 0, tt = a == 2 ? 1 : 2;
                const int e = c[ts] + nI[ts] * c[tt];
                double v = P.ubg[((size_t)item * MRCM_MAXSIDE + sid) * P.side_max + e];
                for (int k = 0; k < sd.nbasis; ++k)
                    v += xs[k] * P.Ug[(((size_t)item * P.nbasis_max + k) * MRCM_MAXSIDE + sid) * P.side_max + e];
                uo = v;
            } else if (md.bc_kind[sid] == 1) {
                uo = (pc - md.bc_val[sid]) / (hk[g * 3 + a]) ;   // T / a = 1 / hk
            } else {
                uo = md.bc_val[sid];
            }
            uw[g * 6 + sid] = uo;
        }
    }
}

// ---------------------------------------------------------------------------
// host-side launch helpers
// ---------------------------------------------------------------------------
size_t local3d_smem(int prec, int nx, int ny, int nz, bool part) {
    const int tsz = prec == 0 ? 8 : 4;
    return lay3(tsz, nx, ny, nz, part ? 1 : round3(tsz, nx, ny, nz), part, false).total;
}

size_t smooth3d_smem(int prec, int nx, int ny, int nz) { return lay3(prec == 0 ? 8 : 4, nx, ny, nz, 1, true, true).total; }

// entries of one box factor (n_a2 planes of b rows)
size_t factor3_entries(int nx, int ny, int nz) {
    int b, npl;
    box3_dims(nx, ny, nz, &b, &npl);
    return plane_stride(b) * npl;
}

template <typename T>
static cudaError_t launch_local3d_t(const DevPtrs& P, const MethodDev& M, const Job* jobs, int njobs, size_t smem,
                                    cudaStream_t s) {
    static size_t cur = 0;
    if (smem > cur) {
        cudaError_t e = cudaFuncSetAttribute(k_local3d<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        cur = smem;
    }
    k_local3d<T><<<njobs, T3, smem, s>>>(P, M, jobs);
    return cudaGetLastError();
}

cudaError_t launch_local3d(const DevPtrs& P, const MethodDev& M, const Job* jobs, int njobs, size_t smem,
                           cudaStream_t s) {
    if (njobs == 0) return cudaSuccess;
    return M.prec == 0 ? launch_local3d_t<double>(P, M, jobs, njobs, smem, s)
                       : launch_local3d_t<float>(P, M, jobs, njobs, smem, s);
}

template <typename T>
static cudaError_t launch_smooth3d_t(const DevPtrs& P, const MethodDev& M, const int* items, int nitems, size_t smem,
                                     cudaStream_t s) {
    static size_t cur = 0;
    if (smem > cur) {
        cudaError_t e = cudaFuncSetAttribute(k_smooth3d<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        cur = smem;
    }
    k_smooth3d<T><<<nitems, T3, smem, s>>>(P, M, items);
    return cudaGetLastError();
}

cudaError_t launch_smooth3d(const DevPtrs& P, const MethodDev& M, const int* items, int nitems, size_t smem,
                            cudaStream_t s) {
    if (nitems == 0) return cudaSuccess;
    return M.prec == 0 ? launch_smooth3d_t<double>(P, M, items, nitems, smem, s)
                       : launch_smooth3d_t<float>(P, M, items, nitems, smem, s);
}

cudaError_t launch_assemble3d(const DevPtrs& P, const double* X, int nitems, int ncell_i_max, cudaStream_t s) {
    k_assemble3d<<<nitems, 256, sizeof(double) * ncell_i_max, s>>>(P, X);
    return cudaGetLastError();
}
