// Assembly of the MRCM-O solution from the interface coefficients and the
// kept basis data (Eqs. (addu), (addp), (uhatphat); Algorithm 1, Step 5), and
// output of the current solution.
#include "mrcm_internal.cuh"
#include <algorithm>


// One CTA per subdomain: p = pbar + sum_k X_k Psi_k on Omega_i, Gamma_i
// velocities ubar + sum_k X_k U_k, interior faces from the assembled
// pressure (the same face law holds for every term of the superposition),
// physical faces from the boundary data.  The transmissibilities are those of
// k_faces (forming them here took three FP64 divisions per face: 79 us on
// 512x512 cells).
__global__ void k_assemble2d(DevPtrs P, const double* __restrict__ X) {
    extern __shared__ double ps[];
    const int item = blockIdx.x;
    const SubDev sd = P.sub[item];
    const MemberDev& md = P.mem[sd.member];
    const int nIx = sd.hi[0] - sd.lo[0], nIy = sd.hi[1] - sd.lo[1];
    const int n = nIx * nIy;
    const double* xs = X + sd.col0;
    const double* Psi = P.Psi + (size_t)item * P.nbasis_max * P.ncell_i_max;
    const double* pb = P.pbar + (size_t)item * P.ncell_i_max;
    for (int c = threadIdx.x; c < n; c += blockDim.x) {
        double v = pb[c];
        for (int k = 0; k < sd.nbasis; ++k) v += xs[k] * Psi[(size_t)k * P.ncell_i_max + c];
        ps[c] = v;
    }
    __syncthreads();
    const double* Tf = P.Tf + md.cell_off * 3;
    const double* hk = P.hk + md.cell_off * 3;
    double* pw = P.p + md.cell_off;
    double* uw = P.u + md.cell_off * 4;
    const double rax = 1.0 / md.h[1], ray = 1.0 / md.h[0];
    for (int c = threadIdx.x; c < n; c += blockDim.x) {
        const int i = c % nIx, j = c / nIx;
        const int gx = sd.lo[0] + i, gy = sd.lo[1] + j;
        const long long g = gx + (long long)md.n[0] * gy;
        if (!mrcm_check(P.status, g >= 0 && g < (long long)md.n[0] * md.n[1], 5, g)) continue;
        const double pc = ps[c];
        // transmissibilities of the faces x-, x+, y-, y+ (0 where there is none)
        const double tf[4] = {i > 0 ? Tf[(g - 1) * 3] : 0.0, Tf[g * 3], j > 0 ? Tf[(g - md.n[0]) * 3 + 1] : 0.0,
                              Tf[g * 3 + 1]};
        double uo[4];
#pragma unroll
        for (int sid = 0; sid < 4; ++sid) {
            const int a = sid >> 1;
            const bool hi = sid & 1;
            const int li = a == 0 ? i : j;
            const int lext = a == 0 ? nIx : nIy;
            const bool edge = hi ? (li == lext - 1) : (li == 0);
            if (!edge) {
                const int cn = c + (a == 0 ? (hi ? 1 : -1) : (hi ? nIx : -nIx));
                uo[sid] = tf[sid] * (pc - ps[cn]) * (a == 0 ? rax : ray);
            } else if (sd.side_mask & (1 << sid)) {
                const int e = a == 0 ? j : i;
                double v = P.ubg[((size_t)item * MRCM_MAXSIDE + sid) * P.side_max + e];
                for (int k = 0; k < sd.nbasis; ++k)
                    v += xs[k] * P.Ug[(((size_t)item * P.nbasis_max + k) * MRCM_MAXSIDE + sid) * P.side_max + e];
                uo[sid] = v;
            } else if (md.bc_kind[sid] == 1) {
                uo[sid] = (pc - md.bc_val[sid]) / hk[g * 3 + a];   // T / a = 1 / hk
            } else {
                uo[sid] = md.bc_val[sid];
            }
        }
        pw[g] = pc;
#pragma unroll
        for (int sid = 0; sid < 4; ++sid) uw[g * 4 + sid] = uo[sid];
    }
}

// Partial sums of a member's pressure in a fixed order (pure-Neumann members
// are reported with zero mean): block b sums cells [b * per, (b + 1) * per).
// One block per member took 179 us for 262,144 cells (one SM's loads, each
// waited for); with a block per 2048 cells (256 blocks at most) the sum is a
// few microseconds, and members with a Dirichlet side skip it.
constexpr int GAUGE_BLOCKS = 256;   // most partial sums (the handle's scratch)
constexpr int GAUGE_CELLS = 2048;   // cells per block below that

__global__ void __launch_bounds__(256) k_gauge_partials(const double* __restrict__ p, long long nc, long long per,
                                                        double* part) {
    __shared__ double red[8];
    const long long c0 = blockIdx.x * per, c1 = min(nc, c0 + per);
    double s = 0.0;
#pragma unroll 4
    for (long long c = c0 + threadIdx.x; c < c1; c += 256) s += p[c];
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < 8; ++w) t += red[w];
        part[blockIdx.x] = t;
    }
}

// Copies a member's pressure (less the mean given by npart partial sums, 0: no
// gauge) and velocities, both as flat arrays: consecutive threads, consecutive
// values.
__global__ void __launch_bounds__(256) k_output(const double* __restrict__ p, const double* __restrict__ u,
                                                long long nc, int nside, const double* __restrict__ part, int npart,
                                                double* __restrict__ pout, double* __restrict__ uout) {
    double mean = 0.0;
    if (npart > 0) {
        __shared__ double sm;
        if (threadIdx.x < 32) {
            double s = 0.0;
            for (int b = threadIdx.x; b < npart; b += 32) s += part[b];
            for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (threadIdx.x == 0) sm = s / (double)nc;
        }
        __syncthreads();
        mean = sm;
    }
    const long long t0 = blockIdx.x * 256LL + threadIdx.x, step = gridDim.x * 256LL;
    if (pout)
        for (long long c = t0; c < nc; c += step) pout[c] = p[c] - mean;
    if (uout) {
        const long long n = nc * nside;
#pragma unroll 4
        for (long long c = t0; c < n; c += step) uout[c] = u[c];
    }
}

cudaError_t launch_assemble2d(const DevPtrs& P, const double* X, int nitems, int ncell_i_max,
                              cudaStream_t s) {
    k_assemble2d<<<nitems, 256, sizeof(double) * ncell_i_max, s>>>(P, X);
    return cudaGetLastError();
}

// part: scratch of at least output_scratch() doubles; gauge: report zero mean.
int output_scratch() { return GAUGE_BLOCKS; }

cudaError_t launch_output(const double* p, const double* u, long long nc, int nside, bool gauge, double* part,
                          double* pout, double* uout, cudaStream_t s) {
    int npart = 0;
    if (gauge && pout) {
        const long long per = std::max<long long>(GAUGE_CELLS, (nc + GAUGE_BLOCKS - 1) / GAUGE_BLOCKS);
        npart = (int)((nc + per - 1) / per);
        k_gauge_partials<<<npart, 256, 0, s>>>(p, nc, per, part);
    }
    const int blocks = (int)std::min<long long>((nc + 255) / 256, 152 * 8);
    k_output<<<blocks, 256, 0, s>>>(p, u, nc, nside, part, npart, pout, uout);
    return cudaGetLastError();
}

// Face coefficients of the cell-centred RT0 operator, once per problem:
// T = a 2 K_L K_R / (h (K_L + K_R)) to the +axis neighbour, h / (2K) per
// cell and H / K_H per face (so that a Robin face has T = a / (h/2K + alpha H/K_H)).
__global__ void k_faces(const MemberDev* mem, int nmem, const double* K, double* Tf, double* hk, double* wh) {
    const int m = blockIdx.y;
    if (m >= nmem) return;
    const MemberDev& md = mem[m];
    const long long nc = (long long)md.n[0] * md.n[1] * md.n[2];
    const long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (c >= nc) return;
    const long long g = md.cell_off + c;
    const int ix = (int)(c % md.n[0]);
    const int iy = (int)((c / md.n[0]) % md.n[1]);
    const int iz = (int)(c / ((long long)md.n[0] * md.n[1]));
    const int idx[3] = {ix, iy, iz};
    const long long st[3] = {1, md.n[0], (long long)md.n[0] * md.n[1]};
    const double kc = K[g];
    double vol = md.h[0] * md.h[1] * (md.dim == 3 ? md.h[2] : 1.0);
    for (int a = 0; a < 3; ++a) {
        double T = 0.0, w = 0.0, hh = 0.0;
        if (a < md.dim) {
            const double area = vol / md.h[a];
            hh = md.h[a] / (2.0 * kc);
            if (idx[a] < md.n[a] - 1) {
                const double kn = K[g + st[a]];
                // harmonic-mean laws written without the product K_L K_R, which
                // leaves the FP64 range for permeabilities beyond ~1e+-154
                T = area * 2.0 * kc * (kn / (kc + kn)) / md.h[a];
                w = md.Hw[a] * 0.5 * (1.0 / kc + 1.0 / kn);
            }
        }
        Tf[g * 3 + a] = T;
        hk[g * 3 + a] = hh;
        wh[g * 3 + a] = w;
    }
}

cudaError_t launch_faces(const MemberDev* dmem, int nmem, long long maxcells, const double* K, double* Tf,
                         double* hk, double* wh, cudaStream_t s) {
    dim3 grid((unsigned)((maxcells + 255) / 256), nmem);
    k_faces<<<grid, 256, 0, s>>>(dmem, nmem, K, Tf, hk, wh);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// mrcm_fluxes_static: the output path without any device allocation.
//
// mrcm_fluxes allocates a device staging buffer whenever it writes to host
// memory, and reduces the pure-Neumann pressure gauge into scratch owned by
// the handle.  Some callers cannot allocate device memory at the point where
// they read results -- an application whose device memory is already held
// by another framework's caching allocator, or a real-time loop in which no
// allocation may happen.  This variant writes into caller device buffers and
// does its multi-block gauge reduction in the fixed static array below
// (8 KB, held by every device that loads the library until the process
// exits).  It allocates nothing.
// ---------------------------------------------------------------------------
#include "../../include/mrcm.h"

#define MRCM_STATIC_PARTIALS 1024             // partial sums, one per block
#define MRCM_STATIC_CELLS_PER_BLOCK 4096      // cells summed by one block
#define MRCM_STATIC_MAX_CELLS ((long long)MRCM_STATIC_PARTIALS * MRCM_STATIC_CELLS_PER_BLOCK)
#define MRCM_STATIC_MAX_DEVICES 64

static __device__ __align__(256) double g_gauge_partials[MRCM_STATIC_PARTIALS];

// Block b sums the pressure of cells [b * CELLS_PER_BLOCK, (b + 1) * CELLS_PER_BLOCK)
// in a fixed order and writes (not accumulates) partials[b].
__global__ void k_gauge_partials_static(const double* __restrict__ p, long long nc, double* partials) {
    __shared__ double red[256];
    const long long c0 = (long long)blockIdx.x * MRCM_STATIC_CELLS_PER_BLOCK;
    const long long c1 = min(nc, c0 + MRCM_STATIC_CELLS_PER_BLOCK);
    double s = 0.0;
    for (long long c = c0 + threadIdx.x; c < c1; c += blockDim.x) s += p[c];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int o = blockDim.x / 2; o; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) partials[blockIdx.x] = red[0];
}

__global__ void k_output_static(const double* __restrict__ p, const double* __restrict__ u, long long nc, int nside,
                                const double* partials, int nblk, int gauge, double* pout, double* uout) {
    __shared__ double mean;
    if (threadIdx.x == 0) {
        double s = 0.0;
        if (gauge)
            for (int b = 0; b < nblk; ++b) s += partials[b];
        mean = gauge ? s / (double)nc : 0.0;
    }
    __syncthreads();
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < nc;
         c += (long long)gridDim.x * blockDim.x) {
        if (pout) pout[c] = p[c] - mean;
        if (uout)
            for (int s = 0; s < nside; ++s) uout[c * nside + s] = u[c * nside + s];
    }
}

// internal accessors defined with the handle (api.cu)
int mrcm_internal_member_state(mrcm_handle* h, int member, cudaStream_t* st, const double** p, const double** u,
                               long long* nc, int* nside, int* gauge, int* device);
int mrcm_internal_fail(mrcm_handle* h, int code, const char* msg);

static double* g_partials_addr[MRCM_STATIC_MAX_DEVICES] = {nullptr};

extern "C" int mrcm_fluxes_static(mrcm_handle* h, int member, double* u_cellfaces, double* p_cells) {
    if (!h) return MRCM_ERR_BAD_INPUT;
    cudaStream_t st;
    const double *p, *u;
    long long nc;
    int nside, gauge, hdev;
    int rc = mrcm_internal_member_state(h, member, &st, &p, &u, &nc, &nside, &gauge, &hdev);
    if (rc) return rc;
    if (nc > MRCM_STATIC_MAX_CELLS)
        return mrcm_internal_fail(h, MRCM_ERR_UNSUPPORTED,
                                  "mrcm_fluxes_static: member larger than its static scratch (4194304 cells)");
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess || dev < 0 || dev >= MRCM_STATIC_MAX_DEVICES)
        return mrcm_internal_fail(h, MRCM_ERR_CUDA, "mrcm_fluxes_static: no usable current device");
    // the address below belongs to the current device, the kernels run on the
    // handle's stream: both must be the handle's device
    if (dev != hdev)
        return mrcm_internal_fail(h, MRCM_ERR_BAD_INPUT,
                                  "mrcm_fluxes_static: the handle's device must be the current device");
    if (!g_partials_addr[dev]) {
        // once per device, with that device current: the device address of the
        // static array (every thread that races here stores the same value)
        void* addr = nullptr;
        e = cudaGetSymbolAddress(&addr, g_gauge_partials);
        if (e != cudaSuccess) return mrcm_internal_fail(h, MRCM_ERR_CUDA, cudaGetErrorString(e));
        g_partials_addr[dev] = (double*)addr;
    }
    double* partials = g_partials_addr[dev];
    const int nblk = (int)((nc + MRCM_STATIC_CELLS_PER_BLOCK - 1) / MRCM_STATIC_CELLS_PER_BLOCK);
    if (gauge) k_gauge_partials_static<<<nblk, 256, 0, st>>>(p, nc, partials);
    const int nout = (int)std::min<long long>((nc + 255) / 256, 4096);
    k_output_static<<<nout, 256, 0, st>>>(p, u, nc, nside, partials, nblk, gauge, p_cells, u_cellfaces);
    e = cudaGetLastError();
    if (e != cudaSuccess) return mrcm_internal_fail(h, MRCM_ERR_CUDA, cudaGetErrorString(e));
    return MRCM_OK;
}
