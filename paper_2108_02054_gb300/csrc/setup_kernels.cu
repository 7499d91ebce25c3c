// setup_kernels.cu -- full-setup kernels (Alg. 1 of arXiv 2108.02054) of the
// smoothed-aggregation hierarchy, all on the GPU: pattern checks, strength of
// connection, distance-2 maximal-independent-set aggregation, smoothed
// prolongation, R = P^T, the symbolic Galerkin product and the gather
// metadata that lets every later numeric product skip the symbolic phase
// (Sec. 5).  Also the synthetic pressure-Poisson assembly used as workload.
//
// Floating point that decides structure (strength test, aggregation ties, P
// values feeding coarser levels) is written as separately rounded IEEE
// operations in a fixed order; the library is built with --fmad=false so no
// multiply-add is contracted behind our back.
#include <climits>

#include "common.cuh"
#include "fdiv.cuh"

namespace amgpr {

namespace {

constexpr int kThreads = 256;

inline int nblocks(int64_t n, int t = kThreads) {
    int64_t b = (n + t - 1) / t;
    return (int)(b < 1 ? 1 : b);
}

__device__ __forceinline__ uint32_t node_priority(uint32_t h) {
    // murmur3 32-bit finaliser: a bijection of the 32-bit integers
    h ^= h >> 16;
    h *= 0x85ebca6bu;
    h ^= h >> 13;
    h *= 0xc2b2ae35u;
    h ^= h >> 16;
    return h;
}

__device__ __forceinline__ int32_t find_in_row(const int32_t *__restrict__ col, int32_t lo, int32_t hi, int32_t c) {
    while (lo < hi) {
        int32_t mid = lo + ((hi - lo) >> 1);
        if (col[mid] < c) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// ------------------------------------------------------------------ scan
constexpr int kScanThreads = 1024;
constexpr int kScanItems = 4;
constexpr int kScanTile = kScanThreads * kScanItems;

__device__ int64_t block_exclusive_scan(int64_t v, int64_t *warp_tot, int64_t *total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int64_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int64_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_tot[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int nw = blockDim.x >> 5;
        int64_t w = lane < nw ? warp_tot[lane] : 0;
        int64_t z = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int64_t y = __shfl_up_sync(0xffffffffu, z, o);
            if (lane >= o) z += y;
        }
        if (lane < nw) warp_tot[lane] = z - w;
        if (lane == 31) *total = z;
    }
    __syncthreads();
    int64_t r = warp_tot[warp] + x - v;
    __syncthreads();
    return r;
}

__global__ void k_scan_reduce(const int32_t *__restrict__ in, int64_t n, int64_t *__restrict__ bsum) {
    __shared__ int64_t wt[32];
    __shared__ int64_t tot;
    int64_t base = (int64_t)blockIdx.x * kScanTile;
    int64_t s = 0;
    for (int k = 0; k < kScanItems; ++k) {
        int64_t i = base + (int64_t)threadIdx.x * kScanItems + k;
        if (i < n) s += in[i];
    }
    block_exclusive_scan(s, wt, &tot);
    if (threadIdx.x == 0) bsum[blockIdx.x] = tot;
}

__global__ void k_scan_blocks(int64_t *__restrict__ bsum, int64_t nb) {
    __shared__ int64_t wt[32];
    __shared__ int64_t tot;
    int64_t carry = 0;
    for (int64_t b0 = 0; b0 < nb; b0 += blockDim.x) {
        int64_t i = b0 + threadIdx.x;
        int64_t v = i < nb ? bsum[i] : 0;
        int64_t e = block_exclusive_scan(v, wt, &tot);
        if (i < nb) bsum[i] = carry + e;
        carry += tot;
        __syncthreads();
    }
    if (threadIdx.x == 0) bsum[nb] = carry;
}

// a scan of at most one tile in one launch
__global__ void k_scan_one(const int32_t *__restrict__ in, int32_t *__restrict__ out, int64_t n, int *st) {
    __shared__ int64_t wt[32];
    __shared__ int64_t tot;
    const int64_t base = (int64_t)threadIdx.x * kScanItems;
    int64_t v[kScanItems], s = 0;
    for (int k = 0; k < kScanItems; ++k) {
        v[k] = base + k < n ? in[base + k] : 0;
        s += v[k];
    }
    int64_t e = block_exclusive_scan(s, wt, &tot);
    for (int k = 0; k < kScanItems; ++k) {
        if (base + k < n) {
            if (e > INT32_MAX) atomicOr(st, DEV_ERR_OVERFLOW);
            out[base + k] = (int32_t)e;
        }
        e += v[k];
    }
    if (threadIdx.x == 0) {
        if (tot > INT32_MAX) atomicOr(st, DEV_ERR_OVERFLOW);
        out[n] = (int32_t)tot;
    }
}

__global__ void k_scan_final(const int32_t *__restrict__ in, int32_t *__restrict__ out, int64_t n,
                             const int64_t *__restrict__ bsum, int64_t nb, int *st) {
    __shared__ int64_t wt[32];
    __shared__ int64_t tot;
    int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;
    int64_t v[kScanItems];
    int64_t s = 0;
    for (int k = 0; k < kScanItems; ++k) {
        v[k] = (base + k < n) ? in[base + k] : 0;
        s += v[k];
    }
    int64_t e = block_exclusive_scan(s, wt, &tot) + bsum[blockIdx.x];
    for (int k = 0; k < kScanItems; ++k) {
        if (base + k < n) {
            if (e > INT32_MAX) atomicOr(st, DEV_ERR_OVERFLOW);
            out[base + k] = (int32_t)e;
        }
        e += v[k];
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        int64_t t = bsum[nb];
        if (t > INT32_MAX) atomicOr(st, DEV_ERR_OVERFLOW);
        out[n] = (int32_t)t;
    }
}

// ------------------------------------------------------------------ assembly
__device__ __forceinline__ void cell_coords(int dim, int N, int64_t c, int64_t &x, int64_t &y, int64_t &z) {
    x = c % N;
    y = (c / N) % N;
    z = dim == 3 ? c / ((int64_t)N * N) : 0;
}

__global__ void k_poisson_rowlen(int dim, int N, int64_t n, int32_t *__restrict__ len) {
    int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= n) return;
    int64_t x, y, z;
    cell_coords(dim, N, c, x, y, z);
    int l = 1 + (x > 0) + (x < N - 1) + (y > 0) + (y < N - 1);
    if (dim == 3) l += (z > 0) + (z < N - 1);
    len[c] = l;
}

__global__ void k_poisson_cols(int dim, int N, int64_t n, const int32_t *__restrict__ ptr, int32_t *__restrict__ col) {
    int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= n) return;
    int64_t x, y, z;
    cell_coords(dim, N, c, x, y, z);
    const int64_t s2 = N, s3 = (int64_t)N * N;
    int32_t p = ptr[c];
    if (dim == 3 && z > 0) col[p++] = (int32_t)(c - s3);
    if (y > 0) col[p++] = (int32_t)(c - s2);
    if (x > 0) col[p++] = (int32_t)(c - 1);
    col[p++] = (int32_t)c;
    if (x < N - 1) col[p++] = (int32_t)(c + 1);
    if (y < N - 1) col[p++] = (int32_t)(c + s2);
    if (dim == 3 && z < N - 1) col[p++] = (int32_t)(c + s3);
}

// per-cell density: the input itself, or exp of it when the input is the
// log-density theta = log rho
__device__ __forceinline__ double cell_rho(const double *__restrict__ in, int64_t c, int logd) {
    const double x = in[c];
    return logd ? exp(x) : x;
}

// 2 / s, correctly rounded, in integer arithmetic (the FP64 division bounds the
// assembly on this part), formed once while s stays the same: in a two-fluid
// field all faces of a cell away from the interface have one sum
struct TwoOver {
    unsigned long long bits = 0ull;  // s = +0: an infinite quotient
    double q = __builtin_huge_val();
    __device__ __forceinline__ double operator()(double s) {
        const unsigned long long b = (unsigned long long)__double_as_longlong(s);
        if (b != bits) {
            bits = b;
            q = div_rn(2.0, div_recip(s));
        }
        return q;
    }
};

// A cell's faces in ascending neighbour order: z-, y-, x-, x+, y+, z+
struct CellFaces {
    bool has[6];
    __device__ __forceinline__ CellFaces(int dim, int N, int32_t x, int32_t y, int32_t z)
        : has{dim == 3 && z > 0, y > 0, x > 0, x < N - 1, y < N - 1, dim == 3 && z < N - 1} {}
    __device__ __forceinline__ int count() const { return has[0] + has[1] + has[2] + has[3] + has[4] + has[5]; }
};

// Row c: neighbours in ascending index order, off-diagonal -2/(rho_c + rho_nb),
// diagonal = running sum of the face coefficients in that order, then the
// ghost-cell Dirichlet term 2/rho_c on the top face.
template <class R>
__device__ __forceinline__ void poisson_row(const CellFaces &F, bool top, double rc, R rho_nb, double *out) {
    TwoOver two;
    double diag = 0.0;
    int p = 0, dpos = 0;
#pragma unroll
    for (int q = 0; q < 6; ++q) {
        if (q == 3) dpos = p++;
        if (F.has[q]) {
            const double k = two(rc + rho_nb(q));
            diag = diag + k;
            out[p++] = -k;
        }
    }
    if (top) diag = diag + two(rc);
    out[dpos] = diag;
}

// A warp's 32 consecutive rows are one contiguous range of values, written
// through shared memory with whole-line stores (one row per thread stored 8
// bytes of each line at a time).  192^3: 885 us with FP64 divisions and those
// stores, 290 now; 64^3: 47 -> 18.
constexpr int kAsmWarps = 8;
template <class R>
__device__ __forceinline__ void store_poisson_rows(const int32_t *__restrict__ ptr, double *__restrict__ val,
                                                   double *buf, int64_t c, bool in, const CellFaces &F, bool top,
                                                   double rc, R rho_nb) {
    const int lane = threadIdx.x & 31;
    const int len = in ? F.count() + 1 : 0;
    int off = len;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, off, o);
        if (lane >= o) off += v;
    }
    const int total = __shfl_sync(0xffffffffu, off, 31);
    off -= len;
    if (in) poisson_row(F, top, rc, rho_nb, buf + off);
    __syncwarp();
    const int32_t p = in ? ptr[c] : 0, p0 = __shfl_sync(0xffffffffu, p, 0);
    if (__all_sync(0xffffffffu, !in || p == p0 + off)) {
        for (int e = lane; e < total; e += 32) val[p0 + e] = buf[e];
    } else {  // rows with gaps between them
        for (int e = 0; e < len; ++e) val[p + e] = buf[off + e];
    }
    __syncwarp();
}

__global__ void __launch_bounds__(kAsmWarps * 32)
k_poisson_vals(int dim, int N, int64_t n, int top, const double *__restrict__ rho, int logd,
               const int32_t *__restrict__ ptr, double *__restrict__ val) {
    __shared__ double s_row[kAsmWarps][32 * 7];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, c0 = c - lane;
    if (c0 >= n) return;  // warp-uniform
    const bool in = c < n;
    const int64_t cc = in ? c : c0;
    int64_t x, y, z;
    cell_coords(dim, N, cc, x, y, z);
    const int64_t s3 = (int64_t)N * N;
    const int64_t nb[6] = {cc - s3, cc - N, cc - 1, cc + 1, cc + N, cc + s3};
    store_poisson_rows(ptr, val, s_row[w], cc, in, CellFaces(dim, N, (int32_t)x, (int32_t)y, (int32_t)z),
                       top && (dim == 2 ? y : z) == N - 1, cell_rho(rho, cc, logd),
                       [&](int q) { return cell_rho(rho, nb[q], logd); });
}

// The log-density forms march in z: a block takes 256 consecutive cells of a
// plane through kLogPlanes planes, a cell's density exp(theta) kept in
// registers for its own plane and the next, the plane's tile (with N cells on
// either side for the y neighbours) in shared memory.  An FP64 exponential is
// some 25 instructions of the slow pipe and a cell's seven densities bound the
// direct kernels above and below; this forms about 1 + 2 N / 256 + 1/4 per cell.
// It is used where it is the faster form (and a tile fits, kLogTile cells):
// - 2D below 384 cells a side, where the halo leaves fewer than four
//   exponentials a cell of the direct form's five.  Values, marching against
//   direct: 256^2 13.4 / 16.5 us, 320^2 19.4 / 22.2, 384^2 30.1 / 29.3, 512^2
//   50.7 / 48.5, 1,024^2 298 / 177, 1,900^2 1,719 / 601.
// - 3D from three quarters of the SMs' number of blocks on: a block's chain of
//   eight planes takes 55 us however few there are.  16^3 49.6 / 14.4 us, 32^3
//   55.2 / 14.3, 48^3 56.5 / 30.4, 58^3 57.3 / 55.3, 60^3 57.5 / 57.9, 64^3 57.7 /
//   67.7, 128^3 274 / 493.
// (The gradient's times cross at the same sizes.)
constexpr int kLogPlanes = 8, kLogTile = 4096, kLogWide2d = 384, kLogBlocks3d = 114;
template <class Cell>
__device__ __forceinline__ void march_log(int dim, int N, const double *__restrict__ theta, Cell cell) {
    extern __shared__ double s_tile[];  // 256 + 2 N densities: cell t of the tile at t + N
    const int64_t P = (int64_t)N * N;
    const int64_t t0 = (int64_t)blockIdx.x * 256, t = t0 + threadIdx.x;  // in-plane index
    const int nz = dim == 3 ? N : 1, z0 = blockIdx.y * kLogPlanes, z1 = min(nz, z0 + kLogPlanes);
    const bool in = t < P;
    const int32_t x = (int32_t)(t % N), y = (int32_t)(t / N);
    double prev = in && z0 > 0 ? exp(theta[(z0 - 1) * P + t]) : 0.0;
    double cur = in ? exp(theta[z0 * P + t]) : 0.0;
    for (int z = z0; z < z1; ++z) {
        const double *plane = theta + (int64_t)z * P;
        const double next = in && z + 1 < nz ? exp(plane[P + t]) : 0.0;
        s_tile[N + threadIdx.x] = cur;
        for (int h = threadIdx.x; h < 2 * N; h += 256) {
            const int64_t k = h < N ? t0 - N + h : t0 + 256 + (h - N);
            s_tile[h < N ? h : 256 + h] = k >= 0 && k < P ? exp(plane[k]) : 0.0;
        }
        __syncthreads();
        const double *me = s_tile + N + threadIdx.x;
        const double nb[6] = {prev, me[-N], me[-1], me[1], me[N], next};
        cell(in, (int64_t)z * P + t, CellFaces(dim, N, x, y, z), (dim == 2 ? y : z) == N - 1, cur, nb);
        __syncthreads();
        prev = cur;
        cur = next;
    }
}

__global__ void __launch_bounds__(256)
k_poisson_vals_log(int dim, int N, int64_t n, int top, const double *__restrict__ theta,
                   const int32_t *__restrict__ ptr, double *__restrict__ val) {
    __shared__ double s_row[kAsmWarps][32 * 7];
    march_log(dim, N, theta, [&](bool in, int64_t c, const CellFaces &F, bool is_top, double rc, const double(&nb)[6]) {
        if (!__any_sync(0xffffffffu, in)) return;  // (a warp's cells in the plane are its first lanes)
        store_poisson_rows(ptr, val, s_row[threadIdx.x >> 5], c, in, F, top && is_top, rc,
                           [&](int q) { return nb[q]; });
    });
}

// Level-set transport stand-in (Sec. 4, eq. 5): implicit upwind
// convection-diffusion on the Poisson pattern.  With w_f the outward face
// flux of cell c (the face velocity, sign-flipped on the low faces):
// off-diagonal min(w_f, 0) - 0.1, diagonal 1 + sum over faces, in the
// neighbour order, of (max(w_f, 0) + 0.1).  Face arrays, x fastest:
// fx[(z N + y)(N + 1) + x_face], fy[(z (N + 1) + y_face) N + x],
// fz[(z_face N + y) N + x].
__global__ void k_levelset_vals(int dim, int N, int64_t n, const double *__restrict__ fx,
                                const double *__restrict__ fy, const double *__restrict__ fz,
                                const int32_t *__restrict__ ptr, double *__restrict__ val) {
    int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= n) return;
    int64_t x, y, z;
    cell_coords(dim, N, c, x, y, z);
    const int64_t N1 = N + 1;
    double w[7];
    int nnb = 0, dslot = 0;
    if (dim == 3 && z > 0) w[nnb++] = -fz[(z * N + y) * N + x];
    if (y > 0) w[nnb++] = -fy[(z * N1 + y) * N + x];
    if (x > 0) w[nnb++] = -fx[(z * N + y) * N1 + x];
    dslot = nnb;
    w[nnb++] = 0.0;
    if (x < N - 1) w[nnb++] = fx[(z * N + y) * N1 + x + 1];
    if (y < N - 1) w[nnb++] = fy[(z * N1 + y + 1) * N + x];
    if (dim == 3 && z < N - 1) w[nnb++] = fz[((z + 1) * N + y) * N + x];
    double diag = 1.0;
    const int32_t p0 = ptr[c];
    for (int t = 0; t < nnb; ++t) {
        if (t == dslot) continue;
        const double wf = w[t];
        diag = diag + ((wf > 0.0 ? wf : 0.0) + 0.1);
        val[p0 + t] = (wf < 0.0 ? wf : 0.0) - 0.1;
    }
    val[p0 + dslot] = diag;
}

// dL/dtheta for theta = log rho, gathered per cell (no atomics): every face
// of cell c contributes dL/dk_f * dk_f/dtheta_c with
// dL/dk_f = -(lam_c - lam_j)(u_c - u_j), dk_f/dtheta_c = -2 rho_c/(rho_c + rho_j)^2;
// the Dirichlet term contributes (-lam_c u_c) * (-2/rho_c).
// (Faces in ascending neighbour order; rho_c / s^2 through the IEEE division.)
template <class R>
__device__ __forceinline__ double poisson_grad_cell(const CellFaces &F, bool top, int64_t c, const int64_t (&nb)[6],
                                                    double rc, R rho_nb, const double *__restrict__ u,
                                                    const double *__restrict__ lam) {
    const double lc = lam[c], uc = u[c];
    double g = 0.0;
    // the last face's sum and its factor: formed again only when it changes
    unsigned long long bits = 0ull;
    double fac = 0.0;
    bool have = false;
#pragma unroll
    for (int q = 0; q < 6; ++q) {
        if (!F.has[q]) continue;
        const double dLdk = -(lc - lam[nb[q]]) * (uc - u[nb[q]]);
        const double s = rc + rho_nb(q);
        const unsigned long long b = (unsigned long long)__double_as_longlong(s);
        if (!have || b != bits) {
            have = true;
            bits = b;
            fac = div_rn(-2.0 * rc, div_recip(s * s));
        }
        g += dLdk * fac;
    }
    if (top) g += (-lc * uc) * div_rn(-2.0, div_recip(rc));
    return g;
}
__global__ void k_poisson_grad(int dim, int N, int64_t n, int top, const double *__restrict__ rho, int logd,
                               const double *__restrict__ u, const double *__restrict__ lam,
                               double *__restrict__ grad) {
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= n) return;
    int64_t x, y, z;
    cell_coords(dim, N, c, x, y, z);
    const int64_t s3 = (int64_t)N * N;
    const int64_t nb[6] = {c - s3, c - N, c - 1, c + 1, c + N, c + s3};
    grad[c] = poisson_grad_cell(CellFaces(dim, N, (int32_t)x, (int32_t)y, (int32_t)z),
                                top && (dim == 2 ? y : z) == N - 1, c, nb, cell_rho(rho, c, logd),
                                [&](int q) { return cell_rho(rho, nb[q], logd); }, u, lam);
}
__global__ void __launch_bounds__(256)
k_poisson_grad_log(int dim, int N, int64_t n, int top, const double *__restrict__ theta,
                   const double *__restrict__ u, const double *__restrict__ lam, double *__restrict__ grad) {
    const int64_t s3 = (int64_t)N * N;
    march_log(dim, N, theta, [&](bool in, int64_t c, const CellFaces &F, bool is_top, double rc, const double(&r)[6]) {
        if (!in) return;
        const int64_t nb[6] = {c - s3, c - N, c - 1, c + 1, c + N, c + s3};
        grad[c] = poisson_grad_cell(F, top && is_top, c, nb, rc, [&](int q) { return r[q]; }, u, lam);
    });
}

// ------------------------------------------------------------------ checks
// a caller's row pointers: ptr[0] = 0, non-decreasing, ptr[n] = nnz, checked
// before any kernel reads the columns they delimit
__global__ void k_check_rowptr(int32_t n, int32_t nnz, const int32_t *__restrict__ ptr, int *st) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i <= n; i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t v = ptr[i];
        bool bad = v < 0 || v > nnz;
        if (i == 0) bad = bad || v != 0;
        if (i == n) bad = bad || v != nnz;
        else bad = bad || ptr[i + 1] < v;
        if (bad) atomicOr(st, DEV_ERR_PATTERN);
    }
}

// The setup's row kernels take G lanes per row: one on grids' finest levels
// (5 to 7 entries a row), a warp where rows hold more than eight on average
// (the launchers' row_lanes), since a coarse level of a thousand rows of 50 to
// 100 entries leaves one thread per row with a long serial chain on an idle
// chip.  What a row's lanes find is combined without regard to their order, or
// in the row's column order where that decides the result, so both forms give
// the same bits.  At 64^3 (levels of 24,028 and 1,289 rows) with one thread per
// row: P's pattern 125 + 333 us, its values 129 + 218, the slots of A P 142 +
// 267, A P 128 + 225, strength 95 + 144, a round of the independent set 42 + 59;
// the step with a full setup went from 9.18 to 6.01 ms.
template <int G>
__device__ __forceinline__ int32_t row_of_thread(int &sub) {
    const int64_t gt = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    sub = (int)(gt % G);
    return (int32_t)(gt / G);
}
template <int G>
__device__ __forceinline__ bool row_any(bool x) {
    return G == 1 ? x : __any_sync(0xffffffffu, x) != 0;
}

template <int G>
__global__ void k_check_pattern(int32_t n, const int32_t *__restrict__ ptr, const int32_t *__restrict__ col,
                                int32_t *__restrict__ dia, int *st) {
    int sub;
    const int32_t i = row_of_thread<G>(sub);
    if (i == 0 && sub == 0 && ptr[0] != 0) atomicOr(st, DEV_ERR_PATTERN);
    if (i >= n) return;  // (a warp's lanes share the row)
    const int32_t b = ptr[i], e = ptr[i + 1];
    int32_t d = -1;
    bool bad = e < b;
    for (int32_t p = b + sub; p < e && !bad; p += G) {
        const int32_t c = col[p];
        if (c < 0 || c >= n || (p > b && c <= col[p - 1])) bad = true;
        if (c == i) d = p;
    }
    if (G > 1) {
        bad = row_any<G>(bad);
        d = __reduce_max_sync(0xffffffffu, d);
    }
    if (sub != 0) return;
    if (bad || d < 0) atomicOr(st, DEV_ERR_PATTERN);
    dia[i] = d < 0 ? b : d;
}

__global__ void k_check_finite(int64_t n, const double *__restrict__ v, int *st) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        if (!isfinite(v[i])) { atomicOr(st, DEV_ERR_NONFINITE); return; }
}

// ------------------------------------------------------------------ strength
// (i,j), j != i, is strong iff a_ij^2 > eps^2 |a_ii a_jj| holds in row i's
// direction or in row j's; each product separately rounded.
template <int G>
__global__ void k_strength(int32_t n, const int32_t *__restrict__ ptr, const int32_t *__restrict__ col,
                           const double *__restrict__ val, const int32_t *__restrict__ dia, double eps2,
                           uint8_t *__restrict__ strong, int32_t *__restrict__ deg) {
    int sub;
    const int32_t i = row_of_thread<G>(sub);
    if (i >= n) return;
    const double aii = val[dia[i]];
    int32_t cnt = 0;
    for (int32_t p = ptr[i] + sub; p < ptr[i + 1]; p += G) {
        int32_t j = col[p];
        uint8_t s = 0;
        if (j != i) {
            const double ajj = val[dia[j]];
            const double a = val[p];
            s = __dmul_rn(a, a) > __dmul_rn(eps2, fabs(__dmul_rn(aii, ajj)));
            if (!s) {
                int32_t b = ptr[j], e = ptr[j + 1];
                int32_t t = find_in_row(col, b, e, i);
                if (t < e && col[t] == i) {
                    const double at = val[t];
                    s = __dmul_rn(at, at) > __dmul_rn(eps2, fabs(__dmul_rn(ajj, aii)));
                }
            }
        }
        strong[p] = s;
        cnt += s;
    }
    if (G > 1) cnt = __reduce_add_sync(0xffffffffu, cnt);
    if (sub == 0) deg[i] = cnt;
}

// ------------------------------------------------------------------ aggregation
// state: 0 undecided, 1 root, 2 excluded (within distance 2 of a root), 3 isolated
__global__ void k_mis_init(int32_t n, const int32_t *__restrict__ deg, int8_t *__restrict__ state) {
    int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) state[i] = deg[i] > 0 ? 0 : 3;
}

// m1[i] = largest priority among undecided nodes of {i} + strong(i), -1 if none
template <int G>
__global__ void k_mis_m1(int32_t n, const int32_t *__restrict__ ptr, const int32_t *__restrict__ col,
                         const uint8_t *__restrict__ strong, const int8_t *__restrict__ state,
                         int64_t *__restrict__ m1) {
    int sub;
    const int32_t i = row_of_thread<G>(sub);
    if (i >= n) return;
    const int8_t si = state[i];
    if (si == 3) {
        if (sub == 0) m1[i] = -1;
        return;
    }
    bool has = si == 0;
    uint32_t m = has ? node_priority((uint32_t)i) : 0u;
    for (int32_t p = ptr[i] + sub; p < ptr[i + 1]; p += G) {
        if (!strong[p]) continue;
        const int32_t j = col[p];
        if (state[j] == 0) {
            m = max(m, node_priority((uint32_t)j));
            has = true;
        }
    }
    if (G > 1) {
        m = __reduce_max_sync(0xffffffffu, m);
        has = row_any<G>(has);
    }
    if (sub == 0) m1[i] = has ? (int64_t)m : -1;
}

// an undecided node whose priority is the largest among undecided nodes
// within strong distance 2 becomes a root
template <int G>
__global__ void k_mis_select(int32_t n, const int32_t *__restrict__ ptr, const int32_t *__restrict__ col,
                             const uint8_t *__restrict__ strong, int8_t *__restrict__ state,
                             const int64_t *__restrict__ m1) {
    int sub;
    const int32_t i = row_of_thread<G>(sub);
    if (i >= n || state[i] != 0) return;
    const int64_t own = (int64_t)node_priority((uint32_t)i);
    bool larger = m1[i] > own;
    for (int32_t p = ptr[i] + sub; p < ptr[i + 1]; p += G)
        if (strong[p]) larger = larger || m1[col[p]] > own;
    larger = row_any<G>(larger);
    // (m1[i] is at least the node's own priority)
    if (sub == 0 && !larger) state[i] = 1;
}

template <int G>
__global__ void k_mis_r1(int32_t n, const int32_t *__restrict__ ptr, const int32_t *__restrict__ col,
                         const uint8_t *__restrict__ strong, const int8_t *__restrict__ state,
                         uint8_t *__restrict__ r1) {
    int sub;
    const int32_t i = row_of_thread<G>(sub);
    if (i >= n) return;
    bool r = state[i] == 1;
    for (int32_t p = ptr[i] + sub; p < ptr[i + 1] && !r; p += G)
        if (strong[p] && state[col[p]] == 1) r = true;
    r = row_any<G>(r);
    if (sub == 0) r1[i] = r;
}

template <int G>
__global__ void k_mis_exclude(int32_t n, const int32_t *__restrict__ ptr, const int32_t *__restrict__ col,
                              const uint8_t *__restrict__ strong, int8_t *__restrict__ state,
                              const uint8_t *__restrict__ r1, int *__restrict__ undecided) {
    int sub;
    const int32_t i = row_of_thread<G>(sub);
    if (i >= n || state[i] != 0) return;
    bool ex = r1[i];
    for (int32_t p = ptr[i] + sub; p < ptr[i + 1] && !ex; p += G)
        if (strong[p] && r1[col[p]]) ex = true;
    ex = row_any<G>(ex);
    if (sub != 0) return;
    if (ex) state[i] = 2;
    else atomicAdd(undecided, 1);
}

__global__ void k_root_flags(int32_t n, const int8_t *__restrict__ state, int32_t *__restrict__ flag) {
    int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) flag[i] = state[i] == 1;
}

// phase 1: a root and its strong neighbours form aggregate root_id[root] (the
// first root in column order, should a one-sided pattern offer several)
template <int G>
__global__ void k_agg_phase1(int32_t n, const int32_t *__restrict__ ptr, const int32_t *__restrict__ col,
                             const uint8_t *__restrict__ strong, const int8_t *__restrict__ state,
                             const int32_t *__restrict__ root_id, int32_t *__restrict__ agg1,
                             int32_t *__restrict__ root_of) {
    int sub;
    const int32_t i = row_of_thread<G>(sub);
    if (i >= n) return;
    const int8_t si = state[i];
    int32_t a = -1;
    if (si == 1) {
        a = root_id[i];
        if (sub == 0) root_of[a] = i;
    } else if (si != 3) {
        int32_t first = INT_MAX;
        for (int32_t p = ptr[i] + sub; p < ptr[i + 1]; p += G)
            if (strong[p] && state[col[p]] == 1) {
                first = p;
                break;
            }
        if (G > 1) first = __reduce_min_sync(0xffffffffu, first);
        if (first != INT_MAX) a = root_id[col[first]];
    }
    if (sub == 0) agg1[i] = a;
}

// phase 2: a remaining non-isolated node joins the phase-1 aggregate of its
// strong neighbour with the largest |a_ij| (ties: larger root priority; equal
// priorities are one root)
template <int G>
__global__ void k_agg_phase2(int32_t n, const int32_t *__restrict__ ptr, const int32_t *__restrict__ col,
                             const double *__restrict__ val, const uint8_t *__restrict__ strong,
                             const int8_t *__restrict__ state, const int32_t *__restrict__ agg1,
                             const int32_t *__restrict__ root_of, int32_t *__restrict__ agg, int *st) {
    int sub;
    const int32_t i = row_of_thread<G>(sub);
    if (i >= n) return;
    int32_t a = agg1[i];
    if (state[i] != 3 && a < 0) {
        double bestv = -1.0;
        uint32_t bestk = 0;
        for (int32_t p = ptr[i] + sub; p < ptr[i + 1]; p += G) {
            if (!strong[p]) continue;
            const int32_t aj = agg1[col[p]];
            if (aj < 0) continue;
            const double v = fabs(val[p]);
            const uint32_t k = node_priority((uint32_t)root_of[aj]);
            if (a < 0 || v > bestv || (v == bestv && k > bestk)) { a = aj; bestv = v; bestk = k; }
        }
        if (G > 1) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const int32_t ao = __shfl_xor_sync(0xffffffffu, a, o);
                const double vo = __shfl_xor_sync(0xffffffffu, bestv, o);
                const uint32_t ko = __shfl_xor_sync(0xffffffffu, bestk, o);
                if (ao >= 0 && (a < 0 || vo > bestv || (vo == bestv && ko > bestk))) { a = ao; bestv = vo; bestk = ko; }
            }
        }
        if (a < 0 && sub == 0) atomicOr(st, DEV_ERR_STATE);
    }
    if (sub == 0) agg[i] = a;
}

// ------------------------------------------------------------------ prolongation
// row i of smoothed P has one column per distinct aggregate among {i} + strong(i)
__device__ __forceinline__ int32_t p_row_count(int32_t i, int32_t b, int32_t e, const int32_t *__restrict__ col,
                                               const uint8_t *__restrict__ strong, const int32_t *__restrict__ agg) {
    int32_t cnt = 0;
    for (int32_t p = b; p < e; ++p) {
        int32_t j = col[p];
        if (j != i && !strong[p]) continue;
        int32_t c = agg[j];
        if (c < 0) continue;
        bool dup = false;
        for (int32_t q = b; q < p && !dup; ++q) {
            int32_t jq = col[q];
            if (jq != i && !strong[q]) continue;
            dup = agg[jq] == c;
        }
        cnt += !dup;
    }
    return cnt;
}
__global__ void k_p_count(int32_t n, const int32_t *__restrict__ ptr, const int32_t *__restrict__ col,
                          const uint8_t *__restrict__ strong, const int32_t *__restrict__ agg, int smoothed,
                          int32_t *__restrict__ plen) {
    int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (agg[i] < 0) { plen[i] = 0; return; }
    if (!smoothed) { plen[i] = 1; return; }
    plen[i] = p_row_count(i, ptr[i], ptr[i + 1], col, strong, agg);
}

// P = (I - w D_F^-1 A_F) P_tent: d_i = a_ii + weak off-diagonals (column order);
// P[i,c] = [c == agg(i)] - sum_{j in {i}+strong(i), agg(j) = c} (w * A_F[i,j]) / d_i
// in column order, A_F[i,i] = d_i.
__device__ __forceinline__ void p_row_fill(int32_t i, int32_t b, int32_t e, int32_t ai, int32_t base,
                                           const int32_t *__restrict__ col, const double *__restrict__ val,
                                           const uint8_t *__restrict__ strong, const int32_t *__restrict__ dia,
                                           const int32_t *__restrict__ agg, double omega,
                                           int32_t *__restrict__ P_col, double *__restrict__ P_val) {
    int32_t nc = 0;
    for (int32_t p = b; p < e; ++p) {
        int32_t j = col[p];
        if (j != i && !strong[p]) continue;
        int32_t c = agg[j];
        if (c < 0) continue;
        bool dup = false;
        for (int32_t s = 0; s < nc && !dup; ++s) dup = P_col[base + s] == c;
        if (dup) continue;
        int32_t t = nc;
        while (t > 0 && P_col[base + t - 1] > c) { P_col[base + t] = P_col[base + t - 1]; --t; }
        P_col[base + t] = c;
        ++nc;
    }
    double d = val[dia[i]];
    for (int32_t p = b; p < e; ++p)
        if (col[p] != i && !strong[p]) d = __dadd_rn(d, val[p]);
    // every term divides by d: its reciprocal once, then correctly rounded
    // quotients in integer arithmetic (the FP64 division bounds this kernel)
    const DivRecip rd = div_recip(d);
    for (int32_t s = 0; s < nc; ++s) {
        const int32_t c = P_col[base + s];
        double v = (c == ai) ? 1.0 : 0.0;
        for (int32_t p = b; p < e; ++p) {
            int32_t j = col[p];
            if (j != i && !strong[p]) continue;
            if (agg[j] != c) continue;
            double w = (j == i) ? d : val[p];
            v = __dsub_rn(v, div_rn(__dmul_rn(omega, w), rd));
        }
        P_val[base + s] = v;
    }
}
__global__ void k_p_fill(int32_t n, const int32_t *__restrict__ ptr, const int32_t *__restrict__ col,
                         const double *__restrict__ val, const uint8_t *__restrict__ strong,
                         const int32_t *__restrict__ dia, const int32_t *__restrict__ agg, double omega,
                         int smoothed, const int32_t *__restrict__ P_ptr, int32_t *__restrict__ P_col,
                         double *__restrict__ P_val) {
    int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int32_t ai = agg[i];
    if (ai < 0) return;
    const int32_t base = P_ptr[i];
    if (!smoothed) {
        P_col[base] = ai;
        P_val[base] = 1.0;
        return;
    }
    p_row_fill(i, ptr[i], ptr[i + 1], ai, base, col, val, strong, dia, agg, omega, P_col, P_val);
}

// The same two passes with a warp per row: the row's aggregates (-1: none, -2:
// a weak off-diagonal) and its quotients staged in shared memory, the lanes
// over the entries.  The diagonal sum and each entry's sum over its terms run in
// column order as above.  Rows longer than kPRow are taken by one lane as above.
constexpr int kPWarps = 4, kPRow = 512;
__device__ __forceinline__ int32_t stage_row_aggs(int32_t i, int32_t b, int32_t len, int lane,
                                                  const int32_t *__restrict__ col,
                                                  const uint8_t *__restrict__ strong,
                                                  const int32_t *__restrict__ agg, int32_t *c) {
    for (int32_t e = lane; e < len; e += 32) {
        const int32_t j = col[b + e];
        c[e] = j == i || strong[b + e] ? max(agg[j], -1) : -2;
    }
    __syncwarp();
    return len;
}
__device__ __forceinline__ bool first_of_its_agg(const int32_t *c, int32_t e) {
    if (c[e] < 0) return false;
    for (int32_t q = 0; q < e; ++q)
        if (c[q] == c[e]) return false;
    return true;
}
__global__ void __launch_bounds__(kPWarps * 32)
k_p_count_warp(int32_t n, const int32_t *__restrict__ ptr, const int32_t *__restrict__ col,
               const uint8_t *__restrict__ strong, const int32_t *__restrict__ agg, int32_t *__restrict__ plen) {
    __shared__ int32_t s_c[kPWarps][kPRow];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int32_t i = blockIdx.x * kPWarps + w;
    if (i >= n) return;  // warp-uniform
    if (agg[i] < 0) {
        if (lane == 0) plen[i] = 0;
        return;
    }
    const int32_t b = ptr[i], len = ptr[i + 1] - b;
    if (len > kPRow) {
        if (lane == 0) plen[i] = p_row_count(i, b, b + len, col, strong, agg);
        return;
    }
    stage_row_aggs(i, b, len, lane, col, strong, agg, s_c[w]);
    int32_t cnt = 0;
    for (int32_t e = lane; e < len; e += 32) cnt += first_of_its_agg(s_c[w], e);
    cnt = __reduce_add_sync(0xffffffffu, cnt);
    if (lane == 0) plen[i] = cnt;
}
__global__ void __launch_bounds__(kPWarps * 32)
k_p_fill_warp(int32_t n, const int32_t *__restrict__ ptr, const int32_t *__restrict__ col,
              const double *__restrict__ val, const uint8_t *__restrict__ strong, const int32_t *__restrict__ dia,
              const int32_t *__restrict__ agg, double omega, const int32_t *__restrict__ P_ptr,
              int32_t *__restrict__ P_col, double *__restrict__ P_val) {
    __shared__ int32_t s_c[kPWarps][kPRow], s_list[kPWarps][kPRow];
    __shared__ double s_t[kPWarps][kPRow];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int32_t i = blockIdx.x * kPWarps + w;
    if (i >= n) return;  // warp-uniform
    const int32_t ai = agg[i];
    if (ai < 0) return;
    const int32_t b = ptr[i], len = ptr[i + 1] - b, base = P_ptr[i];
    if (len > kPRow) {
        if (lane == 0) p_row_fill(i, b, b + len, ai, base, col, val, strong, dia, agg, omega, P_col, P_val);
        return;
    }
    int32_t *c = s_c[w], *list = s_list[w];
    double *t = s_t[w];
    for (int32_t e = lane; e < len; e += 32) t[e] = val[b + e];
    stage_row_aggs(i, b, len, lane, col, strong, agg, c);
    const int32_t ed = dia[i] - b;
    double d = t[ed];
    for (int32_t e = 0; e < len; ++e)
        if (c[e] == -2) d = __dadd_rn(d, t[e]);  // every lane forms the same sum
    __syncwarp();
    const DivRecip rd = div_recip(d);
    int32_t nd = 0;
    for (int32_t e0 = 0; e0 < len; e0 += 32) {
        const int32_t e = e0 + lane;
        bool first = false;
        if (e < len) {
            first = first_of_its_agg(c, e);
            if (c[e] >= 0) t[e] = div_rn(__dmul_rn(omega, e == ed ? d : t[e]), rd);
        }
        const unsigned m = __ballot_sync(0xffffffffu, first);
        if (first) list[nd + __popc(m & ((1u << lane) - 1u))] = e;
        nd += __popc(m);
    }
    __syncwarp();
    for (int32_t k = lane; k < nd; k += 32) {
        const int32_t e0 = list[k], ck = c[e0];
        int32_t rank = 0;
        for (int32_t q = 0; q < nd; ++q) rank += c[list[q]] < ck;
        double v = ck == ai ? 1.0 : 0.0;
        for (int32_t e = e0; e < len; ++e)
            if (c[e] == ck) v = __dsub_rn(v, t[e]);
        P_col[base + rank] = ck;
        P_val[base + rank] = v;
    }
}

__global__ void k_count_cols(int64_t nnz, const int32_t *__restrict__ col, int32_t *__restrict__ cnt) {
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < nnz; p += (int64_t)gridDim.x * blockDim.x)
        atomicAdd(&cnt[col[p]], 1);
}

__global__ void k_transpose_scatter(int32_t n, const int32_t *__restrict__ P_ptr, const int32_t *__restrict__ P_col,
                                    const double *__restrict__ P_val, const int32_t *__restrict__ R_ptr,
                                    int32_t *__restrict__ cursor, int32_t *__restrict__ R_col,
                                    double *__restrict__ R_val) {
    int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    for (int32_t p = P_ptr[i]; p < P_ptr[i + 1]; ++p) {
        int32_t c = P_col[p];
        int32_t pos = R_ptr[c] + atomicAdd(&cursor[c], 1);
        R_col[pos] = i;
        R_val[pos] = P_val[p];
    }
}

// Sort each row of a CSR matrix by column (columns distinct within a row),
// one warp per row.  Rows of up to 512 entries are sorted in registers by a
// bitonic network over the warp (entry e = 32 j + lane in slot j; padding
// sorts last); longer rows by an insertion sort in place.  (With the network up
// to 128 entries only, the few longer rows of a coarse R took 567 us at 64^3.)
template <int E>
__device__ __forceinline__ void warp_bitonic(int32_t (&key)[E], double (&val)[E], int lane) {
#pragma unroll
    for (int k = 2; k <= 32 * E; k <<= 1) {
#pragma unroll
        for (int s = k >> 1; s > 0; s >>= 1) {
            if (s >= 32) {
#pragma unroll
                for (int j = 0; j < E; ++j) {
                    const int jp = j ^ (s >> 5);
                    if (jp > j) {
                        const bool up = ((j * 32 + lane) & k) == 0;
                        if ((key[j] > key[jp]) == up) {
                            const int32_t tk = key[j];
                            key[j] = key[jp];
                            key[jp] = tk;
                            const double tv = val[j];
                            val[j] = val[jp];
                            val[jp] = tv;
                        }
                    }
                }
            } else {
#pragma unroll
                for (int j = 0; j < E; ++j) {
                    const int e = j * 32 + lane;
                    const int32_t pk = __shfl_xor_sync(0xffffffffu, key[j], s);
                    const double pv = __shfl_xor_sync(0xffffffffu, val[j], s);
                    const bool up = (e & k) == 0, lower = (e & s) == 0;
                    if (lower == up ? pk < key[j] : pk > key[j]) {
                        key[j] = pk;
                        val[j] = pv;
                    }
                }
            }
        }
    }
}
template <int E>
__device__ __forceinline__ void warp_sort_row(int32_t b, int32_t len, int32_t *__restrict__ col,
                                              double *__restrict__ val, int lane) {
    int32_t key[E];
    double v[E];
#pragma unroll
    for (int j = 0; j < E; ++j) {
        const int e = j * 32 + lane;
        key[j] = e < len ? col[b + e] : INT_MAX;
        v[j] = e < len ? val[b + e] : 0.0;
    }
    warp_bitonic<E>(key, v, lane);
#pragma unroll
    for (int j = 0; j < E; ++j) {
        const int e = j * 32 + lane;
        if (e < len) {
            col[b + e] = key[j];
            val[b + e] = v[j];
        }
    }
}
constexpr int kSortWarps = 4;
// rows of more than `above` entries (the others are left to another launch)
template <int EMAX>
__global__ void __launch_bounds__(kSortWarps * 32)
k_sort_rows(int32_t nrows, int32_t above, const int32_t *__restrict__ ptr, int32_t *__restrict__ col,
            double *__restrict__ val) {
    const int lane = threadIdx.x & 31;
    const int32_t r = blockIdx.x * kSortWarps + (threadIdx.x >> 5);
    if (r >= nrows) return;  // warp-uniform
    const int32_t b = ptr[r], e = ptr[r + 1], len = e - b;
    if (len <= 1 || len <= above || (EMAX == 4 && len > 128)) return;
    if (len <= 64) warp_sort_row<2>(b, len, col, val, lane);
    else if (len <= 128) warp_sort_row<4>(b, len, col, val, lane);
    else if (EMAX > 4 && len <= 256) warp_sort_row<8>(b, len, col, val, lane);
    else if (EMAX > 4 && len <= 512) warp_sort_row<16>(b, len, col, val, lane);
    else if (lane == 0)
        for (int32_t a = b + 1; a < e; ++a) {
            int32_t c = col[a];
            double v = val[a];
            int32_t t = a;
            while (t > b && col[t - 1] > c) { col[t] = col[t - 1]; val[t] = val[t - 1]; --t; }
            col[t] = c;
            val[t] = v;
        }
}

// ------------------------------------------------------------------ symbolic product
// Each row's distinct columns go through a shared-memory hash table of `cap`
// slots (a power of two, at least twice the product's longest row of terms,
// so that a row's distinct columns always fit and probes stay short; at most
// kHashCap), then are ranked into sorted order.
constexpr int kSymSmemMax = 112 * 1024;

__device__ __forceinline__ bool hash_insert(int32_t *keys, int32_t *count, int32_t c, int cap, int shift) {
    uint32_t h = ((uint32_t)c * 2654435761u) >> shift;
    for (int probe = 0; probe < cap; ++probe) {
        int32_t old = atomicCAS(&keys[h], -1, c);
        if (old == -1) { atomicAdd(count, 1); return true; }
        if (old == c) return true;
        h = (h + 1) & (uint32_t)(cap - 1);
    }
    return false;
}

// the most terms (entries of the selected Y rows, plus the diagonal) of any
// row of C = X * Y: a bound on its distinct columns
__global__ void k_row_terms_max(int32_t nrows, const int32_t *__restrict__ X_ptr, const int32_t *__restrict__ X_col,
                                const int32_t *__restrict__ Y_ptr, int add_diag, int *out) {
    const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    int32_t c = 0;
    if (i < nrows) {
        c = add_diag ? 1 : 0;
        for (int32_t p = X_ptr[i]; p < X_ptr[i + 1]; ++p) {
            const int32_t k = X_col[p];
            c += Y_ptr[k + 1] - Y_ptr[k];
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c = max(c, __shfl_xor_sync(0xffffffffu, c, o));
    if ((threadIdx.x & 31) == 0) atomicMax(out, c);
}

// G lanes per row of C = X * Y (32 / G rows per warp, each with its own hash
// table): the union of the Y-rows selected by X's row.  The warp's rows run
// the same code with warp-wide syncs; a row past the end takes part with no
// entries.
template <int G>
__global__ void k_spgemm_symbolic(int32_t nrows, int32_t ncols, const int32_t *__restrict__ X_ptr,
                                  const int32_t *__restrict__ X_col, const int32_t *__restrict__ Y_ptr,
                                  const int32_t *__restrict__ Y_col, int add_diag, int cap, int shift,
                                  int32_t *__restrict__ len, const int32_t *__restrict__ C_ptr,
                                  int32_t *__restrict__ C_col, int *st) {
    extern __shared__ int32_t smem[];
    const int lane = threadIdx.x & 31, sub = lane % G;
    const int g = threadIdx.x / G;  // the row's group within the block
    const int lcap = cap / 2;       // distinct columns a row may hold
    int32_t *keys = smem + g * (cap + lcap + 2);
    int32_t *list = keys + cap;
    int32_t *cnt = list + lcap;
    const int32_t row = blockIdx.x * (blockDim.x / G) + g;
    const bool live = row < nrows;
    for (int h = sub; h < cap; h += G) keys[h] = -1;
    if (sub == 0) { cnt[0] = 0; cnt[1] = 0; }
    __syncwarp();
    bool ok = true;
    if (live && add_diag && row < ncols && sub == 0) ok = hash_insert(keys, &cnt[0], row, cap, shift);
    if (live)
        for (int32_t p = X_ptr[row] + sub; p < X_ptr[row + 1]; p += G) {
            int32_t k = X_col[p];
            for (int32_t q = Y_ptr[k]; q < Y_ptr[k + 1] && ok; ++q) ok = hash_insert(keys, &cnt[0], Y_col[q], cap, shift);
        }
    __syncwarp();
    const int32_t L = cnt[0];
    const bool bad = !__all_sync(0xffffffffu, ok) || __any_sync(0xffffffffu, live && L > lcap);
    if (bad) {
        if (lane == 0) atomicOr(st, DEV_ERR_CAPACITY);
        return;
    }
    if (C_ptr == nullptr) {
        if (live && sub == 0) len[row] = L;
        return;
    }
    for (int h = sub; h < cap; h += G) {
        int32_t c = keys[h];
        if (c >= 0) list[atomicAdd(&cnt[1], 1)] = c;
    }
    __syncwarp();
    if (!live) return;
    const int32_t base = C_ptr[row];
    if (C_ptr[row + 1] - base != L) {
        if (sub == 0) atomicOr(st, DEV_ERR_STATE);
        return;
    }
    for (int32_t e = sub; e < L; e += G) {
        int32_t v = list[e], rank = 0;
        for (int32_t x = 0; x < L; ++x) rank += list[x] < v;
        C_col[base + rank] = v;
    }
}

// ------------------------------------------------------------------ gather metadata
__global__ void k_t1_count(int32_t n, const int32_t *__restrict__ A_ptr, const int32_t *__restrict__ A_col,
                           const int32_t *__restrict__ P_ptr, int32_t *__restrict__ cnt) {
    int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int32_t c = 0;
    for (int32_t p = A_ptr[i]; p < A_ptr[i + 1]; ++p) {
        int32_t k = A_col[p];
        c += P_ptr[k + 1] - P_ptr[k];
    }
    cnt[i] = c;
}

// slot1[t]: position within row i of A*P of the column of the t-th term
// (A entry (i,k) in column order, then P row k in column order)
__global__ void k_t1_fill(int32_t n, const int32_t *__restrict__ A_ptr, const int32_t *__restrict__ A_col,
                          const int32_t *__restrict__ P_ptr, const int32_t *__restrict__ P_col,
                          const int32_t *__restrict__ AP_ptr, const int32_t *__restrict__ AP_col,
                          const int32_t *__restrict__ t1ptr, uint16_t *__restrict__ slot1, int *st) {
    int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int64_t t = t1ptr[i];
    const int32_t b = AP_ptr[i], e = AP_ptr[i + 1];
    for (int32_t p = A_ptr[i]; p < A_ptr[i + 1]; ++p) {
        int32_t k = A_col[p];
        for (int32_t q = P_ptr[k]; q < P_ptr[k + 1]; ++q) {
            int32_t c = P_col[q];
            int32_t pos = find_in_row(AP_col, b, e, c);
            if (pos >= e || AP_col[pos] != c) { atomicOr(st, DEV_ERR_STATE); pos = b; }
            slot1[t++] = (uint16_t)(pos - b);
        }
    }
}

__global__ void k_t2_count(int32_t nc, const int32_t *__restrict__ R_ptr, const int32_t *__restrict__ R_col,
                           const int32_t *__restrict__ AP_ptr, int32_t *__restrict__ cnt) {
    int32_t I = blockIdx.x * blockDim.x + threadIdx.x;
    if (I >= nc) return;
    int32_t c = 0;
    for (int32_t r = R_ptr[I]; r < R_ptr[I + 1]; ++r) {
        int32_t i = R_col[r];
        c += AP_ptr[i + 1] - AP_ptr[i];
    }
    cnt[I] = c;
}

// slot2[t]: position within coarse row I of the column of the t-th term
// (R entry (I,i) in column order, then row i of A*P in column order).  One
// warp per coarse row: the row's columns of A_c staged in shared memory (rows
// of up to kT2Cols entries; longer ones are searched in place), the lanes over
// the R entries, the prefix of their A P row lengths giving each term's index
constexpr int kT2Warps = 4;
constexpr int kT2Cols = 1024;
__global__ void __launch_bounds__(kT2Warps * 32)
k_t2_fill(int32_t nc, const int32_t *__restrict__ R_ptr, const int32_t *__restrict__ R_col,
               const int32_t *__restrict__ AP_ptr, const int32_t *__restrict__ AP_col,
               const int32_t *__restrict__ Ac_ptr, const int32_t *__restrict__ Ac_col,
               const int32_t *__restrict__ t2ptr, uint16_t *__restrict__ slot2, int *st) {
    __shared__ int32_t s_cols[kT2Warps][kT2Cols];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int32_t I = blockIdx.x * kT2Warps + w;
    if (I >= nc) return;  // warp-uniform
    const int32_t b = Ac_ptr[I], L = Ac_ptr[I + 1] - b;
    const int32_t *cols = Ac_col + b;
    if (L <= kT2Cols) {
        for (int32_t x = lane; x < L; x += 32) s_cols[w][x] = cols[x];
        __syncwarp();
        cols = s_cols[w];
    }
    const int64_t t0 = t2ptr[I];
    const int32_t r1 = R_ptr[I + 1];
    int64_t carry = 0;
    for (int32_t rc = R_ptr[I]; rc < r1; rc += 32) {
        const int32_t r = rc + lane;
        int32_t q0 = 0, len = 0;
        if (r < r1) {
            const int32_t i = R_col[r];
            q0 = AP_ptr[i];
            len = AP_ptr[i + 1] - q0;
        }
        int32_t inc = len;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        const int64_t t = t0 + carry + (inc - len);
        for (int32_t q = 0; q < len; ++q) {
            const int32_t c = AP_col[q0 + q];
            int32_t pos = find_in_row(cols, 0, L, c);
            if (pos >= L || cols[pos] != c) { atomicOr(st, DEV_ERR_STATE); pos = 0; }
            slot2[t + q] = (uint16_t)pos;
        }
        carry += __shfl_sync(0xffffffffu, inc, 31);
    }
}

// ------------------------------------------------------------------ gather operators
// With P and R fixed, the numeric Galerkin product is linear in the values:
// AP = N a and A_c = M AP, with fixed sparse N (coefficients P_kJ) and M
// (coefficients R_Ii).  These kernels build N and M from the slot metadata:
// each output entry's terms are grouped, keeping their sequential order.

constexpr int kGroupWarps = 4;
constexpr int kGroupSlots = 2048;

// One warp per output row: a stable counting sort of the row's terms by slot.
// eptr[out_ptr[row] + s] = first sorted position of slot s; perm[pos] = term.
__global__ void __launch_bounds__(kGroupWarps * 32)
k_group_terms(int32_t nrows, const int32_t *__restrict__ tptr, const uint16_t *__restrict__ slot,
              const int32_t *__restrict__ out_ptr, int32_t *__restrict__ eptr, int32_t *__restrict__ perm,
              int *st) {
    __shared__ int32_t cnt[kGroupWarps][kGroupSlots];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int32_t row = blockIdx.x * kGroupWarps + w;
    if (row >= nrows) return;  // warp-uniform
    const int32_t t0 = tptr[row], t1 = tptr[row + 1];
    const int32_t ob = out_ptr[row], L = out_ptr[row + 1] - ob;
    if (L > kGroupSlots) {
        if (lane == 0) atomicOr(st, DEV_ERR_CAPACITY);
        return;
    }
    int32_t *c = cnt[w];
    for (int s = lane; s < L; s += 32) c[s] = 0;
    __syncwarp();
    for (int32_t t = t0 + lane; t < t1; t += 32) atomicAdd(&c[slot[t]], 1);
    __syncwarp();
    int32_t carry = 0;
    for (int32_t s0 = 0; s0 < L; s0 += 32) {
        const int32_t s = s0 + lane;
        const int32_t v = s < L ? c[s] : 0;
        int32_t inc = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        if (s < L) {
            const int32_t start = carry + inc - v;
            c[s] = start;
            eptr[ob + s] = t0 + start;
        }
        carry += __shfl_sync(0xffffffffu, inc, 31);
    }
    __syncwarp();
    for (int32_t base = t0; base < t1; base += 32) {
        const int32_t t = base + lane;
        const bool valid = t < t1;
        const unsigned active = __ballot_sync(0xffffffffu, valid);
        if (valid) {
            const int sl = slot[t];
            const unsigned peers = __match_any_sync(active, sl);
            const int rank = __popc(peers & ((1u << lane) - 1u));
            perm[t0 + c[sl] + rank] = t;
            __syncwarp(active);
            if (rank == 0) c[sl] += __popc(peers);
        }
        __syncwarp();
    }
}

// term attributes in the sequential order, stage 1: A entry and P value
__global__ void k_stage1_terms(int32_t n, const int32_t *__restrict__ A_ptr, const int32_t *__restrict__ A_col,
                               const int32_t *__restrict__ P_ptr, const double *__restrict__ P_val,
                               const int32_t *__restrict__ t1ptr, int32_t *__restrict__ idx,
                               double *__restrict__ wgt) {
    const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int64_t t = t1ptr[i];
    for (int32_t p = A_ptr[i]; p < A_ptr[i + 1]; ++p) {
        const int32_t k = A_col[p];
        for (int32_t q = P_ptr[k]; q < P_ptr[k + 1]; ++q) {
            idx[t] = p;
            wgt[t] = P_val[q];
            ++t;
        }
    }
}

// stage 2: AP entry and R value
__global__ void k_stage2_terms(int32_t nc, const int32_t *__restrict__ R_ptr, const int32_t *__restrict__ R_col,
                               const double *__restrict__ R_val, const int32_t *__restrict__ AP_ptr,
                               const int32_t *__restrict__ t2ptr, int32_t *__restrict__ idx,
                               double *__restrict__ wgt) {
    const int32_t I = blockIdx.x * blockDim.x + threadIdx.x;
    if (I >= nc) return;
    int64_t t = t2ptr[I];
    for (int32_t r = R_ptr[I]; r < R_ptr[I + 1]; ++r) {
        const int32_t i = R_col[r];
        const double x = R_val[r];
        for (int32_t e = AP_ptr[i]; e < AP_ptr[i + 1]; ++e) {
            idx[t] = e;
            wgt[t] = x;
            ++t;
        }
    }
}

// sorted operator: idx_out[pos] = idx_in[perm[pos]], weights likewise (FP64 or FP32)
__global__ void k_permute_terms(int64_t nt, const int32_t *__restrict__ perm, const int32_t *__restrict__ idx_in,
                                const double *__restrict__ w_in, int32_t *__restrict__ idx_out,
                                double *__restrict__ w_out, float *__restrict__ wf_out) {
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < nt; p += (int64_t)gridDim.x * blockDim.x) {
        const int32_t t = perm[p];
        idx_out[p] = idx_in[t];
        const double w = w_in[t];
        if (w_out) w_out[p] = w;
        if (wf_out) wf_out[p] = (float)w;
    }
}

// last[i]: the last column of row i (rows sorted), -1 for an empty row
__global__ void k_row_last(int32_t n, const int32_t *__restrict__ ptr, const int32_t *__restrict__ col,
                           int32_t *__restrict__ last) {
    const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int32_t e = ptr[i + 1];
    last[i] = e > ptr[i] ? col[e - 1] : -1;
}

__global__ void k_row_maxlen(int32_t n, const int32_t *__restrict__ ptr, int *out) {
    int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    int l = i < n ? ptr[i + 1] - ptr[i] : 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) l = max(l, __shfl_xor_sync(0xffffffffu, l, o));
    if ((threadIdx.x & 31) == 0) atomicMax(out, l);
}

}  // namespace

// ======================================================================= launchers
int64_t scan_tmp_elems(int64_t n) { return (n + kScanTile - 1) / kScanTile + 2; }

void scan_counts(const int32_t *in, int32_t *out, int64_t n, int *st, int64_t *tmp, cudaStream_t s) {
    if (n <= 0) {
        cudaMemsetAsync(out, 0, sizeof(int32_t), s);
        return;
    }
    int64_t nb = (n + kScanTile - 1) / kScanTile;
    if (nb == 1) {
        count_launch();
        k_scan_one<<<1, kScanThreads, 0, s>>>(in, out, n, st);
        return;
    }
    count_launch();
    k_scan_reduce<<<(unsigned)nb, kScanThreads, 0, s>>>(in, n, tmp);
    count_launch();
    k_scan_blocks<<<1, kScanThreads, 0, s>>>(tmp, nb);
    count_launch();
    k_scan_final<<<(unsigned)nb, kScanThreads, 0, s>>>(in, out, n, tmp, nb, st);
}

void launch_poisson_rowlen(int dim, int N, int32_t *len, cudaStream_t s) {
    int64_t n = dim == 2 ? (int64_t)N * N : (int64_t)N * N * N;
    count_launch();
    k_poisson_rowlen<<<nblocks(n), kThreads, 0, s>>>(dim, N, n, len);
}
void launch_poisson_cols(int dim, int N, const int32_t *ptr, int32_t *col, cudaStream_t s) {
    int64_t n = dim == 2 ? (int64_t)N * N : (int64_t)N * N * N;
    count_launch();
    k_poisson_cols<<<nblocks(n), kThreads, 0, s>>>(dim, N, n, ptr, col);
}
namespace {
// the marching kernels' grid (tiles of a plane, chunks of planes), where they
// are the faster form and a tile fits
bool log_grid(int dim, int N, dim3 &g, size_t &smem) {
    if (256 + 2 * N > kLogTile) return false;
    const int64_t tiles = ((int64_t)N * N + 255) / 256, chunks = dim == 3 ? (N + kLogPlanes - 1) / kLogPlanes : 1;
    if (dim == 2 ? N >= kLogWide2d : tiles * chunks < kLogBlocks3d) return false;
    g = dim3((unsigned)tiles, (unsigned)chunks);
    smem = sizeof(double) * (size_t)(256 + 2 * N);
    return g.y <= 65535;
}
}  // namespace
void launch_poisson_vals(int dim, int N, int top, const double *rho, int logd, const int32_t *ptr, double *val,
                         cudaStream_t s) {
    int64_t n = dim == 2 ? (int64_t)N * N : (int64_t)N * N * N;
    count_launch();
    dim3 g;
    size_t smem = 0;
    if (logd && log_grid(dim, N, g, smem)) k_poisson_vals_log<<<g, 256, smem, s>>>(dim, N, n, top, rho, ptr, val);
    else k_poisson_vals<<<nblocks(n, kAsmWarps * 32), kAsmWarps * 32, 0, s>>>(dim, N, n, top, rho, logd, ptr, val);
}
void launch_poisson_grad(int dim, int N, int top, const double *rho, int logd, const double *u, const double *lam,
                         double *grad, cudaStream_t s) {
    int64_t n = dim == 2 ? (int64_t)N * N : (int64_t)N * N * N;
    count_launch();
    dim3 g;
    size_t smem = 0;
    if (logd && log_grid(dim, N, g, smem)) k_poisson_grad_log<<<g, 256, smem, s>>>(dim, N, n, top, rho, u, lam, grad);
    else k_poisson_grad<<<nblocks(n), kThreads, 0, s>>>(dim, N, n, top, rho, logd, u, lam, grad);
}

void launch_levelset_vals(int dim, int N, const double *fx, const double *fy, const double *fz, const int32_t *ptr,
                          double *val, cudaStream_t s) {
    int64_t n = dim == 2 ? (int64_t)N * N : (int64_t)N * N * N;
    count_launch();
    k_levelset_vals<<<nblocks(n), kThreads, 0, s>>>(dim, N, n, fx, fy, fz, ptr, val);
}

void launch_check_rowptr(int32_t n, int32_t nnz, const int32_t *ptr, int *st, cudaStream_t s) {
    const int64_t b = nblocks((int64_t)n + 1);
    count_launch();
    k_check_rowptr<<<(unsigned)(b > 4096 ? 4096 : b), kThreads, 0, s>>>(n, nnz, ptr, st);
}
namespace {
// lanes per row of the setup's row kernels: a warp above eight entries a row
// on average (grids' finest levels have 5 to 7, coarse levels 30 and more)
bool warp_rows(int32_t n, int32_t nnz) { return (int64_t)nnz > 8 * (int64_t)n; }
}  // namespace
#define ROW_LANES(KERNEL, ...)                                                                     \
    do {                                                                                           \
        count_launch();                                                                            \
        if (warp_rows(n, nnz)) KERNEL<32><<<nblocks((int64_t)n * 32), kThreads, 0, s>>>(__VA_ARGS__); \
        else KERNEL<1><<<nblocks(n), kThreads, 0, s>>>(__VA_ARGS__);                               \
    } while (0)
void launch_check_pattern(int32_t n, int32_t nnz, const int32_t *ptr, const int32_t *col, int32_t *dia, int *st,
                          cudaStream_t s) {
    ROW_LANES(k_check_pattern, n, ptr, col, dia, st);
}
void launch_check_finite(int64_t nnz, const double *val, int *st, cudaStream_t s) {
    int64_t b = nblocks(nnz);
    count_launch();
    k_check_finite<<<(unsigned)(b > 4096 ? 4096 : b), kThreads, 0, s>>>(nnz, val, st);
}
void launch_strength(int32_t n, int32_t nnz, const int32_t *ptr, const int32_t *col, const double *val,
                     const int32_t *dia, double eps2, uint8_t *strong, int32_t *deg, cudaStream_t s) {
    ROW_LANES(k_strength, n, ptr, col, val, dia, eps2, strong, deg);
}
int32_t run_aggregation(int32_t n, int32_t nnz, const int32_t *ptr, const int32_t *col, const double *val,
                        const uint8_t *strong, const int32_t *deg, int32_t *agg, int8_t *state, int64_t *m1,
                        uint8_t *r1, int32_t *root_id, int32_t *agg1, int32_t *root_of, int *counter, int *st,
                        int64_t *scan_tmp, int32_t *h_pin, cudaStream_t s) {
    const int nb = nblocks(n);
    count_launch();
    k_mis_init<<<nb, kThreads, 0, s>>>(n, deg, state);
    // every round turns at least the undecided node of largest priority into
    // a root, so at most n rounds; in practice a few dozen
    for (int32_t round = 0; round <= n; ++round) {
        ROW_LANES(k_mis_m1, n, ptr, col, strong, state, m1);
        ROW_LANES(k_mis_select, n, ptr, col, strong, state, m1);
        ROW_LANES(k_mis_r1, n, ptr, col, strong, state, r1);
        cudaMemsetAsync(counter, 0, sizeof(int), s);
        ROW_LANES(k_mis_exclude, n, ptr, col, strong, state, r1, counter);
        if (cudaMemcpyAsync(h_pin, counter, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess) return -1;
        if (cudaStreamSynchronize(s) != cudaSuccess) return -1;
        if (*h_pin == 0) break;
        if (round == n) return -1;
    }
    count_launch();
    k_root_flags<<<nb, kThreads, 0, s>>>(n, state, agg);
    scan_counts(agg, root_id, n, st, scan_tmp, s);
    if (cudaMemcpyAsync(h_pin, root_id + n, sizeof(int32_t), cudaMemcpyDeviceToHost, s) != cudaSuccess) return -1;
    if (cudaStreamSynchronize(s) != cudaSuccess) return -1;
    const int32_t nagg = *h_pin;
    ROW_LANES(k_agg_phase1, n, ptr, col, strong, state, root_id, agg1, root_of);
    ROW_LANES(k_agg_phase2, n, ptr, col, val, strong, state, agg1, root_of, agg, st);
    return nagg;
}

void launch_p_count(int32_t n, int32_t nnz, const int32_t *ptr, const int32_t *col, const uint8_t *strong,
                    const int32_t *agg, int smoothed, int32_t *plen, cudaStream_t s) {
    count_launch();
    if (smoothed && warp_rows(n, nnz))
        k_p_count_warp<<<nblocks(n, kPWarps), kPWarps * 32, 0, s>>>(n, ptr, col, strong, agg, plen);
    else
        k_p_count<<<nblocks(n), kThreads, 0, s>>>(n, ptr, col, strong, agg, smoothed, plen);
}
void launch_p_fill(int32_t n, int32_t nnz, const int32_t *ptr, const int32_t *col, const double *val,
                   const uint8_t *strong, const int32_t *dia, const int32_t *agg, double omega, int smoothed,
                   const int32_t *P_ptr, int32_t *P_col, double *P_val, cudaStream_t s) {
    count_launch();
    if (smoothed && warp_rows(n, nnz))
        k_p_fill_warp<<<nblocks(n, kPWarps), kPWarps * 32, 0, s>>>(n, ptr, col, val, strong, dia, agg, omega, P_ptr,
                                                                   P_col, P_val);
    else
        k_p_fill<<<nblocks(n), kThreads, 0, s>>>(n, ptr, col, val, strong, dia, agg, omega, smoothed, P_ptr, P_col,
                                                 P_val);
}
void launch_count_cols(int64_t nnz, const int32_t *col, int32_t *cnt, cudaStream_t s) {
    int64_t b = nblocks(nnz);
    count_launch();
    k_count_cols<<<(unsigned)(b > 8192 ? 8192 : b), kThreads, 0, s>>>(nnz, col, cnt);
}
void launch_transpose_scatter(int32_t n, const int32_t *P_ptr, const int32_t *P_col, const double *P_val,
                              const int32_t *R_ptr, int32_t *cursor, int32_t *R_col, double *R_val,
                              cudaStream_t s) {
    count_launch();
    k_transpose_scatter<<<nblocks(n), kThreads, 0, s>>>(n, P_ptr, P_col, P_val, R_ptr, cursor, R_col, R_val);
}
void launch_sort_rows(int32_t nrows, const int32_t *ptr, int32_t *col, double *val, cudaStream_t s) {
    if (nrows <= 0) return;
    // many rows: the short ones by the kernel with fewer registers, then the
    // few long ones; a small level in one launch
    const unsigned g = (unsigned)((nrows + kSortWarps - 1) / kSortWarps);
    const bool split = nrows > 152 * 64;
    if (split) {
        count_launch();
        k_sort_rows<4><<<g, kSortWarps * 32, 0, s>>>(nrows, 0, ptr, col, val);
    }
    count_launch();
    k_sort_rows<16><<<g, kSortWarps * 32, 0, s>>>(nrows, split ? 128 : 0, ptr, col, val);
}

void launch_row_terms_max(int32_t nrows, const int32_t *X_ptr, const int32_t *X_col, const int32_t *Y_ptr,
                          int add_diag, int *out, cudaStream_t s) {
    if (nrows <= 0) return;
    count_launch();
    k_row_terms_max<<<nblocks(nrows), kThreads, 0, s>>>(nrows, X_ptr, X_col, Y_ptr, add_diag, out);
}
int spgemm_symbolic_cap(int32_t max_terms) {
    int cap = 64;
    while (cap < kHashCap && cap < 2 * max_terms) cap *= 2;
    return cap;
}
namespace {
template <int G>
void launch_symbolic_g(int32_t nrows, int32_t ncols, const int32_t *X_ptr, const int32_t *X_col,
                       const int32_t *Y_ptr, const int32_t *Y_col, int add_diag, int cap, int shift, int32_t *len,
                       const int32_t *C_ptr, int32_t *C_col, int *st, cudaStream_t s) {
    static bool attr_set = false;
    if (!attr_set) {
        cudaFuncSetAttribute(k_spgemm_symbolic<G>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSymSmemMax);
        attr_set = true;
    }
    const size_t per_row = (size_t)(cap + cap / 2 + 2) * sizeof(int32_t);
    int warps = 8;
    while (warps > 1 && per_row * (size_t)(warps * 32 / G) > (size_t)kSymSmemMax) warps >>= 1;
    const int rows = warps * 32 / G;
    const unsigned grid = (unsigned)((nrows + rows - 1) / rows);
    count_launch();
    k_spgemm_symbolic<G><<<grid, warps * 32, per_row * (size_t)rows, s>>>(nrows, ncols, X_ptr, X_col, Y_ptr, Y_col,
                                                                         add_diag, cap, shift, len, C_ptr, C_col, st);
}
}  // namespace

void launch_spgemm_symbolic(int32_t nrows, int32_t ncols, const int32_t *X_ptr, const int32_t *X_col,
                            const int32_t *Y_ptr, const int32_t *Y_col, int add_diag, int cap, int lanes,
                            int32_t *len, const int32_t *C_ptr, int32_t *C_col, int *st, cudaStream_t s) {
    if (nrows <= 0) return;
    int shift = 32;
    for (int c = cap; c > 1; c >>= 1) --shift;  // cap = 2^(32 - shift)
    if (lanes <= 8)
        launch_symbolic_g<8>(nrows, ncols, X_ptr, X_col, Y_ptr, Y_col, add_diag, cap, shift, len, C_ptr, C_col, st, s);
    else if (lanes <= 16)
        launch_symbolic_g<16>(nrows, ncols, X_ptr, X_col, Y_ptr, Y_col, add_diag, cap, shift, len, C_ptr, C_col, st,
                              s);
    else
        launch_symbolic_g<32>(nrows, ncols, X_ptr, X_col, Y_ptr, Y_col, add_diag, cap, shift, len, C_ptr, C_col, st,
                              s);
}

void launch_t1_count(int32_t n, const int32_t *A_ptr, const int32_t *A_col, const int32_t *P_ptr, int32_t *cnt,
                     cudaStream_t s) {
    count_launch();
    k_t1_count<<<nblocks(n), kThreads, 0, s>>>(n, A_ptr, A_col, P_ptr, cnt);
}
void launch_t1_fill(int32_t n, int32_t nnz, const int32_t *A_ptr, const int32_t *A_col, const int32_t *P_ptr,
                    const int32_t *P_col, const int32_t *AP_ptr, const int32_t *AP_col, const int32_t *t1ptr,
                    uint16_t *slot1, int *st, cudaStream_t s) {
    // long rows: the warp-per-row fill of stage 2 (the same positions)
    if (warp_rows(n, nnz)) {
        launch_t2_fill(n, A_ptr, A_col, P_ptr, P_col, AP_ptr, AP_col, t1ptr, slot1, st, s);
        return;
    }
    count_launch();
    k_t1_fill<<<nblocks(n), kThreads, 0, s>>>(n, A_ptr, A_col, P_ptr, P_col, AP_ptr, AP_col, t1ptr, slot1, st);
}
void launch_t2_count(int32_t nc, const int32_t *R_ptr, const int32_t *R_col, const int32_t *AP_ptr, int32_t *cnt,
                     cudaStream_t s) {
    count_launch();
    k_t2_count<<<nblocks(nc), kThreads, 0, s>>>(nc, R_ptr, R_col, AP_ptr, cnt);
}
void launch_t2_fill(int32_t nc, const int32_t *R_ptr, const int32_t *R_col, const int32_t *AP_ptr,
                    const int32_t *AP_col, const int32_t *Ac_ptr, const int32_t *Ac_col, const int32_t *t2ptr,
                    uint16_t *slot2, int *st, cudaStream_t s) {
    count_launch();
    if (nc <= 0) return;
    k_t2_fill<<<(unsigned)((nc + kT2Warps - 1) / kT2Warps), kT2Warps * 32, 0, s>>>(nc, R_ptr, R_col, AP_ptr,
                                                                                     AP_col, Ac_ptr, Ac_col, t2ptr,
                                                                                     slot2, st);
}
void launch_group_terms(int32_t nrows, const int32_t *tptr, const uint16_t *slot, const int32_t *out_ptr,
                        int32_t *eptr, int32_t *perm, int *st, cudaStream_t s) {
    if (nrows <= 0) return;
    count_launch();
    k_group_terms<<<(unsigned)((nrows + kGroupWarps - 1) / kGroupWarps), kGroupWarps * 32, 0, s>>>(
        nrows, tptr, slot, out_ptr, eptr, perm, st);
}
void launch_stage1_terms(int32_t n, const int32_t *A_ptr, const int32_t *A_col, const int32_t *P_ptr,
                         const double *P_val, const int32_t *t1ptr, int32_t *idx, double *wgt, cudaStream_t s) {
    count_launch();
    k_stage1_terms<<<nblocks(n), kThreads, 0, s>>>(n, A_ptr, A_col, P_ptr, P_val, t1ptr, idx, wgt);
}
void launch_stage2_terms(int32_t nc, const int32_t *R_ptr, const int32_t *R_col, const double *R_val,
                         const int32_t *AP_ptr, const int32_t *t2ptr, int32_t *idx, double *wgt, cudaStream_t s) {
    count_launch();
    k_stage2_terms<<<nblocks(nc, 128), 128, 0, s>>>(nc, R_ptr, R_col, R_val, AP_ptr, t2ptr, idx, wgt);
}
void launch_permute_terms(int64_t nt, const int32_t *perm, const int32_t *idx_in, const double *w_in,
                          int32_t *idx_out, double *w_out, float *wf_out, cudaStream_t s) {
    if (nt <= 0) return;
    int64_t b = nblocks(nt);
    count_launch();
    k_permute_terms<<<(unsigned)(b > 8192 ? 8192 : b), kThreads, 0, s>>>(nt, perm, idx_in, w_in, idx_out, w_out,
                                                                         wf_out);
}
void launch_row_last(int32_t n, const int32_t *ptr, const int32_t *col, int32_t *last, cudaStream_t s) {
    if (n <= 0) return;
    count_launch();
    k_row_last<<<nblocks(n), kThreads, 0, s>>>(n, ptr, col, last);
}
void launch_row_maxlen(int32_t n, const int32_t *ptr, int *out, cudaStream_t s) {
    count_launch();
    k_row_maxlen<<<nblocks(n), kThreads, 0, s>>>(n, ptr, out);
}

}  // namespace amgpr
