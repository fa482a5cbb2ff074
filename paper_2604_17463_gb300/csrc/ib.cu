// ib.cu -- immersed-boundary kernels of libiblb: nodal forces (A1), force
// spreading with band marking (A2 + A3), velocity interpolation with forward
// Euler advection (A5 + A6), and the FP64 observables (A7).
//
// Paper, Sec. 2:
//   Eq. 7  qdot_j = sum_x u(x) Delta(q_j - x)           (interpolation)
//   Eq. 8  F(x)   = sum_j phi_j Delta(q_j - x)           (spreading)
//   Eq. 9  interface force = surface tension + wetting term along n
//   Eq. 10 Pi(d)  = A [(xi/d)^n - (xi/d)^m]
//   nodal wetting force phi_Pi,j = -chi_j Pi(d_j) n_j / 3 (3D), / 2 for the
//   2D ring (each segment is shared by two nodes); n_j is the normalised mean
//   of the unit normals of the faces sharing node j, chi_j their total area.
//   The surface-tension force is -sigma times the gradient of the interface
//   area (3D) / length (2D) with linear elements; an elastic interface adds
//   minus the gradient of Skalak's strain energy (ib_core.cuh).
// Delta is the tensor product of Peskin's 4-point kernel; stencil points on a
// solid layer (or outside the lattice along the wall axis) take no force and
// give zero velocity.
#include "ib_core.cuh"

namespace iblb {

// Threads per block of the node kernels: one warp per block up to 8 warps per
// SM, so that the warps spread over the SMs (an SM's FP64 pipe serves one warp
// instruction in 16 clocks), else two.
// A 2D binary16 run keeps blocks of 128: the order in which neighbouring
// warps' additions reach a cell is part of its trajectory.
static int node_block(int storage, int dim, int n)
{
    if (dim == 2 && storage == ST_FP16) return 128;
    return n <= 152 * 256 ? 32 : 64;
}

// ------------------------------------------------------------------ A1 forces
// 2D ring: one thread per node.
template <bool KEEP>
__global__ void k_forces_ring(const double* __restrict__ q, int N, ForceParams fp,
                              double* __restrict__ phi, double* __restrict__ nrm,
                              double* __restrict__ chi, int* err)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= N) return;
    ring_node_force<KEEP>(q, N, j, fp, phi, nrm, chi, err);
}

// 3D mesh, pass 1: one thread per face writes its three corner records.
__global__ void k_face_geometry(const double* __restrict__ q, const int* __restrict__ tri, int M,
                                const int* __restrict__ entry_pos, ForceParams fp,
                                double* __restrict__ rec)
{
    const int f = blockIdx.x * blockDim.x + threadIdx.x;
    if (f >= M) return;
    face_records(q, tri, f, entry_pos, fp, rec);
}

// Elastic reference of the interface as it is now: per face (3D) the inverse
// reference edge matrix and area, per segment (2D) the length.
__global__ void k_elastic_reference(int dim, const double* __restrict__ q, int N, int M,
                                    const int* __restrict__ tri, double* __restrict__ eref)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (dim == 3) {
        if (t < M) face_elastic_reference(q, tri, t, eref + 5 * (long long)t);
    } else if (t < N) {
        const int tn = (t + 1 == N) ? 0 : t + 1;
        const double sx = q[2 * tn] - q[2 * t], sy = q[2 * tn + 1] - q[2 * t + 1];
        eref[t] = sqrt(sx * sx + sy * sy);
    }
}

void launch_elastic_reference(int dim, const double* q, int N, int M, const int* tri, double* eref,
                              cudaStream_t s)
{
    const int n = dim == 3 ? M : N;
    if (n > 0) k_elastic_reference<<<(n + 127) / 128, 128, 0, s>>>(dim, q, N, M, tri, eref);
}

// 3D mesh, pass 2: one thread per node sums its records (no atomics).
__global__ void k_node_forces(const double* __restrict__ q, int N, const double* __restrict__ rec,
                              const int* __restrict__ csr_ptr, ForceParams fp,
                              double* __restrict__ phi, double* __restrict__ nrm,
                              double* __restrict__ chi, int* err)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= N) return;
    mesh_node_force(q, j, rec, csr_ptr, fp, phi, nrm, chi, err);
}

void launch_forces(int storage, int dim, const double* q, int N, int M, const int* tri, const int* csr_ptr,
                   const int* entry_pos, double* entry_rec, const ForceParams& fp, double* phi,
                   double* normal, double* chi, int* err, cudaStream_t s)
{
    if (dim == 2) {
        const int b = node_block(storage, dim, N), g = (N + b - 1) / b;
        if (storage == ST_FP16) k_forces_ring<true><<<g, b, 0, s>>>(q, N, fp, phi, normal, chi, err);
        else k_forces_ring<false><<<g, b, 0, s>>>(q, N, fp, phi, normal, chi, err);
    } else {
        const int b = 64;
        k_face_geometry<<<(M + b - 1) / b, b, 0, s>>>(q, tri, M, entry_pos, fp, entry_rec);
        k_node_forces<<<(N + b - 1) / b, b, 0, s>>>(q, N, entry_rec, csr_ptr, fp, phi, normal,
                                                    chi, err);
    }
}

// ------------------------------------------------------------------ A2 + A3 spread
// One thread per node (spread_node in ib_core.cuh): one vector atomic per
// stencil point, the touched 32-cell row segments marked.  Measured against
// one warp per node (lanes sharing the stencil points) on the 59 292-node
// paper-scale mesh: 45 us against 44 us per step, so the simpler form stays.
template <int D, typename R>
__global__ void __launch_bounds__(128)
k_spread_t(const double* __restrict__ q, const double* __restrict__ phi, int N,
           R* __restrict__ F, uint8_t* __restrict__ flags, uint8_t* __restrict__ fine,
           GridParams g)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < N) spread_node<D, R>(g, q, phi, j, F, flags, fine);
}

void launch_spread(int storage, int dim, const double* q, const double* phi, int N, void* F,
                   uint8_t* flags, uint8_t* fine, const GridParams& g, cudaStream_t s)
{
    if (N <= 0) return;
    const int b = node_block(storage, dim, N), grid = (N + b - 1) / b;
    if (storage == ST_FP64) {
        if (dim == 2) k_spread_t<2, double><<<grid, b, 0, s>>>(q, phi, N, (double*)F, flags, fine, g);
        else k_spread_t<3, double><<<grid, b, 0, s>>>(q, phi, N, (double*)F, flags, fine, g);
    } else {
        if (dim == 2) k_spread_t<2, float><<<grid, b, 0, s>>>(q, phi, N, (float*)F, flags, fine, g);
        else k_spread_t<3, float><<<grid, b, 0, s>>>(q, phi, N, (float*)F, flags, fine, g);
    }
}

// ------------------------------------------------------------------ fused IB kernels
// 2D ring between two stream-collides: advection with the last step's
// velocity, forces, spread (ring_warp in ib_core.cuh), one warp per block.
template <typename R, bool FIRST>
__global__ void __launch_bounds__(32)
k_ring(const double* __restrict__ q, double* __restrict__ q_out, int N, ForceParams fp,
       const R* __restrict__ mom, R* __restrict__ F, uint8_t* __restrict__ flags, GridParams g,
       int* err)
{
    ring_warp<R, FIRST>(g, q, q_out, N, blockIdx.x * RING_OWN, fp, mom, F, flags, err);
}

void launch_ring(int storage, bool first, const double* q, double* q_out, int N,
                 const ForceParams& fp, const void* moments, void* F, uint8_t* flags,
                 const GridParams& g, int* err, cudaStream_t s)
{
    const int grid = (N + RING_OWN - 1) / RING_OWN;
#define IBLB_RING(RR, FF) \
    k_ring<RR, FF><<<grid, 32, 0, s>>>(q, q_out, N, fp, (const RR*)moments, (RR*)F, flags, g, err)
    if (storage == ST_FP64) {
        if (first) IBLB_RING(double, true);
        else IBLB_RING(double, false);
    } else {
        if (first) IBLB_RING(float, true);
        else IBLB_RING(float, false);
    }
#undef IBLB_RING
}

// 3D mesh, pass 2 with the spread: one thread per node sums its face records
// and spreads the force it holds.
template <typename R>
__global__ void __launch_bounds__(64)
k_node_spread(const double* __restrict__ q, int N, const double* __restrict__ rec,
              const int* __restrict__ csr_ptr, ForceParams fp, R* __restrict__ F,
              uint8_t* __restrict__ flags, uint8_t* __restrict__ fine, GridParams g, int* err)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < N) mesh_node_spread<R>(g, q, j, rec, csr_ptr, fp, F, flags, fine, err);
}

void launch_mesh_spread(int storage, const double* q, int N, int M, const int* tri,
                        const int* csr_ptr, const int* entry_pos, double* entry_rec,
                        const ForceParams& fp, void* F, uint8_t* flags, uint8_t* fine,
                        const GridParams& g, int* err, cudaStream_t s)
{
    k_face_geometry<<<(M + 63) / 64, 64, 0, s>>>(q, tri, M, entry_pos, fp, entry_rec);
    const int b = node_block(storage, 3, N), grid = (N + b - 1) / b;
    if (storage == ST_FP64)
        k_node_spread<double><<<grid, b, 0, s>>>(q, N, entry_rec, csr_ptr, fp, (double*)F, flags, fine, g, err);
    else
        k_node_spread<float><<<grid, b, 0, s>>>(q, N, entry_rec, csr_ptr, fp, (float*)F, flags, fine, g, err);
}

// ------------------------------------------------------------------ A5 + A6 interpolate, advect
// One thread per node (interp_node in ib_core.cuh): 16 velocity reads in
// flight per thread; on the 59 292-node mesh 16 us per step against 35 us
// for one warp per node with two reads per lane and a shuffle reduction.
template <int D, typename R, bool KEEP = keep_weights<D, R>>
__global__ void __launch_bounds__(128)
k_interp_t(double* __restrict__ q, const R* __restrict__ mom, int N, double* __restrict__ qdot,
           int advect, GridParams g)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= N) return;
    R acc[3];
    interp_node<D, R, KEEP>(g, q, mom, j, acc);
    for (int k = 0; k < D; k++) {
        if (qdot) qdot[D * j + k] = (double)acc[k];
        if (advect) q[D * j + k] += (double)acc[k];
    }
}

void launch_interp(int storage, int dim, double* q, const void* moments, int N, double* qdot,
                   bool advect, bool ordered, const GridParams& g, cudaStream_t s)
{
    if (N <= 0) return;
    const int b = node_block(storage, dim, N), grid = (N + b - 1) / b;
    if (storage == ST_FP64) {
        if (dim == 2) k_interp_t<2, double><<<grid, b, 0, s>>>(q, (const double*)moments, N, qdot, advect, g);
        else k_interp_t<3, double><<<grid, b, 0, s>>>(q, (const double*)moments, N, qdot, advect, g);
    } else {
        if (dim == 2) k_interp_t<2, float><<<grid, b, 0, s>>>(q, (const float*)moments, N, qdot, advect, g);
        else if (keep_weights_3d(storage, ordered)) k_interp_t<3, float, true><<<grid, b, 0, s>>>(q, (const float*)moments, N, qdot, advect, g);
        else k_interp_t<3, float><<<grid, b, 0, s>>>(q, (const float*)moments, N, qdot, advect, g);
    }
}

// ------------------------------------------------------------------ A7 observables
// Fixed thread -> item assignment and reduction trees, so the results are
// deterministic.  Contact-angle estimator: algebraic least-squares circle
// (2D) / sphere (3D) through the nodes with d > 3 xi, centred on their mean,
// intersected with the plane d = min_j d_j.

// Reduce nv values per thread to thread 0 (sum), in a fixed order.
template <int B>
__device__ void block_sum(double* v, int nv, double (*sh)[B / 32])
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int k = 0; k < nv; k++) {
        double x = v[k];
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (lane == 0) sh[k][wid] = x;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 0; k < nv; k++) {
            double t = 0.0;
            for (int w = 0; w < B / 32; w++) t += sh[k][w];
            v[k] = t;
        }
    }
    __syncthreads();
}

template <int B>
__device__ void block_minmax(double& mn, double& mx, double (*sh)[B / 32])
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int o = 16; o > 0; o >>= 1) {
        mn = fmin(mn, __shfl_xor_sync(0xffffffffu, mn, o));
        mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    if (lane == 0) {
        sh[0][wid] = mn;
        sh[1][wid] = mx;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 0; w < B / 32; w++) {
            mn = fmin(mn, sh[0][w]);
            mx = fmax(mx, sh[1][w]);
        }
    }
    __syncthreads();
}

__device__ bool solve_small(int n, double* A, double* b)
{
    for (int col = 0; col < n; col++) {
        int piv = col;
        for (int r = col + 1; r < n; r++)
            if (fabs(A[r * n + col]) > fabs(A[piv * n + col])) piv = r;
        if (A[piv * n + col] == 0.0) return false;
        if (piv != col) {
            for (int k = 0; k < n; k++) {
                const double t = A[col * n + k];
                A[col * n + k] = A[piv * n + k];
                A[piv * n + k] = t;
            }
            const double t = b[col];
            b[col] = b[piv];
            b[piv] = t;
        }
        for (int r = col + 1; r < n; r++) {
            const double f = A[r * n + col] / A[col * n + col];
            for (int k = col; k < n; k++) A[r * n + k] -= f * A[col * n + k];
            b[r] -= f * b[col];
        }
    }
    for (int r = n - 1; r >= 0; r--) {
        double acc = b[r];
        for (int k = r + 1; k < n; k++) acc -= A[r * n + k] * b[k];
        b[r] = acc / A[r * n + r];
    }
    return true;
}

// The three passes of the observables (sums and extremes; normal equations of
// the fit; film under the drop) and the last sum, one kernel each over up to
// OBS_GRID blocks: a pass's blocks each add up the previous pass's partial
// sums for themselves.  FP64 arithmetic bounds them: in one block, on one SM's
// pipe, the call (with the mass sum and its synchronisations) took 0.16 ms on
// the 128 x 64 ring, 0.41 ms with 10 242 nodes on 101 x 101 x 77 and 1.63 ms with
// 40 962 on 256 x 256 x 128; with these passes and the mass sum of lbm.cu 0.10,
// 0.14 and 0.26 ms.
constexpr int OBS_THREADS = 256;
constexpr int OBS_P1 = 8, OBS_P2 = 20, OBS_P3 = 2;  // doubles per block and pass

struct ObsArgs {
    int dim;
    const double* q;
    int N;
    const int* tri;
    int M;
    const double* mass_partial;
    int n_partial;
    double xi, wp;
    double* out;           // 12 results
    double *p1, *p2, *p3;  // partial sums [block][...]
};

// Sums over the blocks of column k of a partial array, by the first warp
// (ascending rows per lane, then a fixed tree).
__device__ __forceinline__ double column_sum(const double* p, int stride, int k, int grid)
{
    double s = 0.0;
    for (int r = threadIdx.x; r < grid; r += 32) s += p[r * stride + k];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

__global__ void __launch_bounds__(OBS_THREADS) k_obs_sums(ObsArgs a)
{
    __shared__ double sh[6][OBS_THREADS / 32];
    const int t0 = blockIdx.x * OBS_THREADS + threadIdx.x, nt = gridDim.x * OBS_THREADS;
    const int dim = a.dim, wax = dim - 1;
    const double* q = a.q;
    double v[6] = {0, 0, 0, 0, 0, 0};  // mass, volume, sum of the fit set (3), its count
    for (int b = t0; b < a.n_partial; b += nt) v[0] += a.mass_partial[b];
    if (dim == 2) {
        for (int j = t0; j < a.N; j += nt) {
            const int jn = (j + 1 == a.N) ? 0 : j + 1;
            v[1] += q[2 * j] * q[2 * jn + 1] - q[2 * jn] * q[2 * j + 1];
        }
    } else {
        for (int f = t0; f < a.M; f += nt) {
            const double* x = q + 3 * a.tri[3 * f];
            const double* y = q + 3 * a.tri[3 * f + 1];
            const double* z = q + 3 * a.tri[3 * f + 2];
            v[1] += x[0] * (y[1] * z[2] - y[2] * z[1]) + x[1] * (y[2] * z[0] - y[0] * z[2]) +
                    x[2] * (y[0] * z[1] - y[1] * z[0]);
        }
    }
    double hmin = 1e300, hmax = -1e300;
    for (int j = t0; j < a.N; j += nt) {
        const double h = q[dim * j + wax];
        hmin = fmin(hmin, h);
        hmax = fmax(hmax, h);
        if (h - a.wp > 3.0 * a.xi) {
            for (int k = 0; k < dim; k++) v[2 + k] += q[dim * j + k];
            v[5] += 1.0;
        }
    }
    block_sum<OBS_THREADS>(v, 6, sh);
    block_minmax<OBS_THREADS>(hmin, hmax, sh);
    if (threadIdx.x == 0) {
        double* r = a.p1 + OBS_P1 * blockIdx.x;
        for (int k = 0; k < 6; k++) r[k] = v[k];
        r[6] = hmin;
        r[7] = hmax;
    }
}

__global__ void __launch_bounds__(OBS_THREADS) k_obs_fit(ObsArgs a)
{
    __shared__ double sh[OBS_P2][OBS_THREADS / 32];
    __shared__ double tot[6];
    const int dim = a.dim, wax = dim - 1, np = dim + 1;
    if (threadIdx.x < 32)
        for (int k = 0; k < 6; k++) {
            const double s = column_sum(a.p1, OBS_P1, k, gridDim.x);
            if (threadIdx.x == 0) tot[k] = s;
        }
    __syncthreads();
    const double cnt = tot[5];
    double mean[3] = {0, 0, 0};
    for (int k = 0; k < dim; k++) mean[k] = cnt > 0 ? tot[2 + k] / cnt : 0.0;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        double hmin = 1e300, hmax = -1e300;
        for (int r = 0; r < (int)gridDim.x; r++) {
            hmin = fmin(hmin, a.p1[OBS_P1 * r + 6]);
            hmax = fmax(hmax, a.p1[OBS_P1 * r + 7]);
        }
        a.out[0] = tot[0];
        a.out[1] = (dim == 2) ? 0.5 * tot[1] : tot[1] / 6.0;
        a.out[2] = hmax - hmin;
        a.out[6] = hmin - a.wp;
    }
    double v[OBS_P2];
    for (int k = 0; k < OBS_P2; k++) v[k] = 0.0;
    const double* q = a.q;
    for (int j = blockIdx.x * OBS_THREADS + threadIdx.x; j < a.N; j += gridDim.x * OBS_THREADS) {
        if (!(q[dim * j + wax] - a.wp > 3.0 * a.xi)) continue;
        double vv[4], r2 = 0.0;
        for (int k = 0; k < dim; k++) {
            vv[k] = q[dim * j + k] - mean[k];
            r2 += vv[k] * vv[k];
        }
        vv[dim] = 1.0;
        for (int x = 0; x < np; x++) {
            for (int y = 0; y < np; y++) v[x * np + y] += vv[x] * vv[y];
            v[16 + x] -= vv[x] * r2;
        }
    }
    block_sum<OBS_THREADS>(v, OBS_P2, sh);
    if (threadIdx.x == 0)
        for (int k = 0; k < OBS_P2; k++) a.p2[OBS_P2 * blockIdx.x + k] = v[k];
}

__global__ void __launch_bounds__(OBS_THREADS) k_obs_film(ObsArgs a)
{
    __shared__ double sh[OBS_P3][OBS_THREADS / 32];
    __shared__ double sums[OBS_P2], tot[6], bc[3];
    const int dim = a.dim, np = dim + 1;
    if (threadIdx.x < 32) {
        for (int k = 2; k < 6; k++) {
            const double s = column_sum(a.p1, OBS_P1, k, gridDim.x);
            if (threadIdx.x == 0) tot[k] = s;
        }
        for (int k = 0; k < OBS_P2; k++) {
            const double s = column_sum(a.p2, OBS_P2, k, gridDim.x);
            if (threadIdx.x == 0) sums[k] = s;
        }
    }
    __syncthreads();
    double* out = a.out;
    const bool writer = blockIdx.x == 0;
    if (threadIdx.x == 0) {
        const double cnt = tot[5];
        bool ok = cnt >= dim + 1;
        double Am[16], rhs[4];
        for (int k = 0; k < np * np; k++) Am[k] = sums[k];
        for (int k = 0; k < np; k++) rhs[k] = sums[16 + k];
        if (ok) ok = solve_small(np, Am, rhs);
        if (!ok) {
            if (writer) {
                out[3] = out[4] = out[5] = out[11] = nan("");
                out[7] = out[8] = out[9] = 0.0;
            }
            bc[0] = -1.0;
        } else {
            double cen[3] = {0, 0, 0}, R2 = 0.0;
            for (int k = 0; k < dim; k++) {
                cen[k] = -0.5 * rhs[k];
                R2 += cen[k] * cen[k];
            }
            R2 -= rhs[dim];
            const double R = sqrt(R2);
            for (int k = 0; k < dim; k++) cen[k] += cnt > 0 ? tot[2 + k] / cnt : 0.0;
            double hmin = 1e300;
            for (int r = 0; r < (int)gridDim.x; r++) hmin = fmin(hmin, a.p1[OBS_P1 * r + 6]);
            const double dz = a.wp + (hmin - a.wp) - cen[dim - 1];
            const double rc2 = R * R - dz * dz;
            const double rc = rc2 > 0.0 ? sqrt(rc2) : 0.0;
            if (writer) {
                const double cth = fmin(1.0, fmax(-1.0, dz / R));
                out[3] = acos(cth) * (180.0 / 3.141592653589793);
                out[4] = rc;
                out[7] = cen[0];
                out[8] = cen[1];
                out[9] = cen[2];
                out[10] = R;
            }
            bc[0] = rc;
            bc[1] = cen[0];
            bc[2] = cen[1];
        }
    }
    __syncthreads();
    const double rcl = bc[0], c0 = bc[1], c1 = bc[2];
    double v[OBS_P3] = {0, 0};
    if (rcl >= 0.0) {
        const double* q = a.q;
        for (int j = blockIdx.x * OBS_THREADS + threadIdx.x; j < a.N; j += gridDim.x * OBS_THREADS) {
            const double d = q[dim * j + dim - 1] - a.wp;
            double rr = 0.0;
            const double t0 = q[dim * j] - c0;
            rr += t0 * t0;
            if (dim == 3) {
                const double t1 = q[dim * j + 1] - c1;
                rr += t1 * t1;
            }
            if (sqrt(rr) < 0.5 * rcl && d <= 3.0 * a.xi) {
                v[0] += d;
                v[1] += 1.0;
            }
        }
    }
    block_sum<OBS_THREADS>(v, OBS_P3, sh);
    if (threadIdx.x == 0) {
        a.p3[OBS_P3 * blockIdx.x] = v[0];
        a.p3[OBS_P3 * blockIdx.x + 1] = rcl >= 0.0 ? v[1] : -1.0;  // no fit: no film
    }
}

__global__ void __launch_bounds__(32) k_obs_last(ObsArgs a, int grid)
{
    const double d = column_sum(a.p3, OBS_P3, 0, grid), n = column_sum(a.p3, OBS_P3, 1, grid);
    if (threadIdx.x != 0) return;
    if (n >= 0.0) a.out[5] = n > 0 ? d / n : nan("");
    if (a.N == 0)
        for (int k = 1; k < 12; k++) a.out[k] = 0.0;
}

// Deformation index (Sec. 4, Eq. 15): the enclosed region is split into
// simplices from the node mean p0 (triangles of the ring in 2D, tetrahedra of
// the mesh in 3D).  Over a simplex with vertices v_k relative to p0 and
// signed measure |K|: int x = |K| sum(v_k) / (d + 1) and
// int x x^T = |K| (sum v_k v_k^T + s s^T) / ((d + 1)(d + 2)), s = sum v_k.
// The central second moments in the shear plane (x and the wall axis) give
// the semi-axes sqrt(4 lambda / area) (2D) or sqrt(5 lambda / volume) (3D).
// Three kernels: node sums, simplex sums about their mean, results; up to
// OBS_GRID blocks (the call with 20 480 faces took 0.49 ms in one block, with 81 920 now 0.07).
__global__ void __launch_bounds__(OBS_THREADS) k_def_mean(int dim, const double* __restrict__ q, int N, double* part)
{
    __shared__ double sh[3][OBS_THREADS / 32];
    double v[3] = {0, 0, 0};
    for (int j = blockIdx.x * OBS_THREADS + threadIdx.x; j < N; j += gridDim.x * OBS_THREADS)
        for (int k = 0; k < dim; k++) v[k] += q[dim * j + k];
    block_sum<OBS_THREADS>(v, 3, sh);
    if (threadIdx.x == 0)
        for (int k = 0; k < 3; k++) part[3 * blockIdx.x + k] = v[k];
}

__global__ void __launch_bounds__(OBS_THREADS)
k_def_moments(int dim, const double* __restrict__ q, int N, const int* __restrict__ tri, int M,
              const double* __restrict__ mean_part, double* part)
{
    __shared__ double sh[6][OBS_THREADS / 32];
    __shared__ double p0s[3];
    if (threadIdx.x < 32)
        for (int k = 0; k < 3; k++) {
            const double s = column_sum(mean_part, 3, k, gridDim.x);
            if (threadIdx.x == 0) p0s[k] = k < dim ? s / N : 0.0;
        }
    __syncthreads();
    const double p0[3] = {p0s[0], p0s[1], p0s[2]};
    const int w = dim - 1;
    double v[6] = {0, 0, 0, 0, 0, 0};
    const int nsimp = dim == 2 ? N : M;
    for (int e = blockIdx.x * OBS_THREADS + threadIdx.x; e < nsimp; e += gridDim.x * OBS_THREADS) {
        double a[3] = {0, 0, 0}, b[3] = {0, 0, 0}, c[3] = {0, 0, 0};
        double meas;
        if (dim == 2) {
            const int jn = (e + 1 == N) ? 0 : e + 1;
            for (int k = 0; k < 2; k++) {
                a[k] = q[2 * e + k] - p0[k];
                b[k] = q[2 * jn + k] - p0[k];
            }
            meas = 0.5 * (a[0] * b[1] - a[1] * b[0]);
        } else {
            const double* A = q + 3 * tri[3 * e];
            const double* B = q + 3 * tri[3 * e + 1];
            const double* C = q + 3 * tri[3 * e + 2];
            for (int k = 0; k < 3; k++) {
                a[k] = A[k] - p0[k];
                b[k] = B[k] - p0[k];
                c[k] = C[k] - p0[k];
            }
            meas = (a[0] * (b[1] * c[2] - b[2] * c[1]) + a[1] * (b[2] * c[0] - b[0] * c[2]) +
                    a[2] * (b[0] * c[1] - b[1] * c[0])) / 6.0;
        }
        const double sx = a[0] + b[0] + c[0], sw = a[w] + b[w] + c[w];
        const double f2 = meas / ((dim + 1) * (dim + 2));
        v[0] += meas;
        v[1] += meas * sx / (dim + 1);
        v[2] += meas * sw / (dim + 1);
        v[3] += f2 * (a[0] * a[0] + b[0] * b[0] + c[0] * c[0] + sx * sx);
        v[4] += f2 * (a[w] * a[w] + b[w] * b[w] + c[w] * c[w] + sw * sw);
        v[5] += f2 * (a[0] * a[w] + b[0] * b[w] + c[0] * c[w] + sx * sw);
    }
    block_sum<OBS_THREADS>(v, 6, sh);
    if (threadIdx.x == 0)
        for (int k = 0; k < 6; k++) part[6 * blockIdx.x + k] = v[k];
}

__global__ void __launch_bounds__(32) k_def_last(int dim, const double* __restrict__ part, int grid, double* out)
{
    double v[6];
    for (int k = 0; k < 6; k++) v[k] = column_sum(part, 6, k, grid);
    if (threadIdx.x == 0) {
        const double vol = v[0];
        const double gx = v[1] / vol, gw = v[2] / vol;
        const double sxx = v[3] - vol * gx * gx;
        const double sww = v[4] - vol * gw * gw;
        const double sxw = v[5] - vol * gx * gw;
        const double mean = 0.5 * (sxx + sww);
        const double rad = sqrt(0.25 * (sxx - sww) * (sxx - sww) + sxw * sxw);
        const double kk = dim == 2 ? 4.0 : 5.0;
        const double r1 = sqrt(kk * (mean + rad) / vol), r3 = sqrt(kk * (mean - rad) / vol);
        out[0] = (r1 - r3) / (r1 + r3);
        out[1] = r1;
        out[2] = r3;
        out[3] = 0.5 * atan2(2.0 * sxw, sxx - sww) * (180.0 / 3.141592653589793);
        out[4] = vol;
    }
}

void launch_deformation(int dim, const double* q, int N, const int* tri, int M, double* out,
                        double* ws, int blocks, cudaStream_t s)
{
    const int n = dim == 2 ? N : (M > N ? M : N);
    int grid = (n + OBS_THREADS - 1) / OBS_THREADS;
    grid = grid < 1 ? 1 : (grid > blocks ? blocks : grid);
    double* mean_part = ws;
    double* part = mean_part + 3 * grid;
    static_assert(9 <= OBS_WS, "deformation workspace");
    k_def_mean<<<grid, OBS_THREADS, 0, s>>>(dim, q, N, mean_part);
    k_def_moments<<<grid, OBS_THREADS, 0, s>>>(dim, q, N, tri, M, mean_part, part);
    k_def_last<<<1, 32, 0, s>>>(dim, part, grid, out);
}

void launch_observables(int dim, const double* q, int N, const int* tri, int M,
                        const double* mass_partial, int n_partial, double xi, double wall_plane,
                        double* out, double* ws, int blocks, cudaStream_t s)
{
    ObsArgs a{dim, q, N, tri, M, mass_partial, n_partial, xi, wall_plane, out, nullptr, nullptr, nullptr};
    int grid = ((N > n_partial ? N : n_partial) + OBS_THREADS - 1) / OBS_THREADS;
    grid = grid < 1 ? 1 : (grid > blocks ? blocks : grid);
    a.p1 = ws;
    a.p2 = a.p1 + OBS_P1 * grid;
    a.p3 = a.p2 + OBS_P2 * grid;
    static_assert(OBS_P1 + OBS_P2 + OBS_P3 <= OBS_WS, "observables workspace");
    k_obs_sums<<<grid, OBS_THREADS, 0, s>>>(a);
    k_obs_fit<<<grid, OBS_THREADS, 0, s>>>(a);
    k_obs_film<<<grid, OBS_THREADS, 0, s>>>(a);
    k_obs_last<<<1, 32, 0, s>>>(a, grid);
}

}  // namespace iblb
