// Allocation-free variant of the non-bonded pair energy + gradient.
//
// Some callers cannot let a library allocate device memory: an application
// that runs inside another framework's memory pool with a hard cap, or a
// real-time loop that cannot afford cudaMalloc's implicit device
// synchronisation.  ffmin_pair_energy_grad_noalloc serves them: the caller
// passes device buffers for the inputs and outputs, and the only scratch it
// needs (partial row sums, block energies, a ticket counter) lives in the
// file-scope device array `g_noalloc_scratch` below, which every GPU that
// loads this library holds until the process exits.
//
// Computation: an FP64 row sweep over all pairs of one system, Coulomb +
// Lennard-Jones, no bonded terms: every pair in both of its rows, since the
// fixed scratch has no room for the opposite forces.  Bound: the FP64 pipe;
// differences, terms and their sums are formed on the integer pipes
// (pair64.cuh), which leaves 4 FP64 instructions an evaluated pair of about 28.  Blocks of 32 i-atoms against a
// j-chunk, the chunk's atoms dealt to the four warps, give about 1,000 equal
// blocks at 4,000 atoms (128 i-atoms per block: 256, 1.7 per SM).  4,000 atoms:
// 1.10 -> 0.37 ms a call with the terms added in FP64 (9 instructions), 0.34 ms now.  Partial rows go to the scratch, then one thread per atom
// sums its chunks in a fixed order and the last block sums the block
// energies and flags a non-finite energy or gradient (two coincident atoms),
// which the call reports after synchronising its stream.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <mutex>
#include <type_traits>

#include "ffmin.h"
#include "pair64.cuh"

namespace {

using namespace ffm;

constexpr int NA_TI = 32;       // i atoms per block (one per lane, the same for every warp)
constexpr int NA_TJ = 128;      // j atoms staged per shared-memory tile
constexpr int NA_NT = 128;      // threads per block
constexpr int NA_CHUNKS = 16;   // j chunks per row, at most
constexpr int NA_MAX_ATOMS = 8192;
constexpr int NA_FT = 64;       // atoms per block of the final sum
constexpr int NA_MAX_BLOCKS = (NA_MAX_ATOMS + NA_FT - 1) / NA_FT;
// doubles: the atoms' parameters [3][n], partial rows [chunk][n][4] (as many
// chunks as fit), block energies, one 8-byte word holding the last-block
// ticket and the non-finite flag (two uint32)
constexpr size_t NA_ROWS = (size_t)8 * NA_MAX_ATOMS * 4;
constexpr size_t NA_SCRATCH = NA_ROWS + NA_MAX_BLOCKS + 1;

__device__ __align__(256) double g_noalloc_scratch[NA_SCRATCH];

constexpr int NA_MAX_DEVICES = 64;
// device address of the array per device ordinal, looked up once in the
// device's primary context (a cudaDeviceReset or another context would need
// a new lookup); the lock guards the first lookup against concurrent callers
double *g_scratch_ptr[NA_MAX_DEVICES];
std::mutex g_scratch_lock;

struct NaArgs {
    const double *x, *q, *sigma, *eps;
    int n, chunks;
    double sqrt_c;
    double *g, *e;
    double *par;       // [3][n] q sqrt(C), a sigma^3, a sigma^6 (a = sqrt(24 eps))
    double *part;      // [chunks][n][4]
    double *eblock;    // [NA_MAX_BLOCKS]
    unsigned int *ticket;  // [0] last-block ticket, [1] non-finite flag
};

// per-atom parameters once per call; the ticket and the flag start at zero
// (the array keeps the last call's contents)
__global__ void __launch_bounds__(NA_NT) k_na_prepare(NaArgs a) {
    const int i = blockIdx.x * NA_NT + threadIdx.x;
    if (i == 0) a.ticket[0] = a.ticket[1] = 0u;
    if (i >= a.n) return;
    const double s3 = a.sigma[i] * a.sigma[i] * a.sigma[i];
    const double w = sqrt(24.0 * a.eps[i]);
    a.par[i] = a.q[i] * a.sqrt_c;
    a.par[a.n + i] = w * s3;
    a.par[2 * a.n + i] = w * s3 * s3;
}

__device__ __forceinline__ void na_atom(const NaArgs &a, int j, double far, double (&x)[3], double (&p)[3]) {
    if (j < a.n) {
        for (int k = 0; k < 3; k++) {
            x[k] = a.x[3 * j + k];
            p[k] = a.par[k * a.n + j];
        }
    } else {  // padding atom: far away, no charge, no Lennard-Jones
        x[0] = x[1] = x[2] = far;
        p[0] = p[1] = p[2] = 0.0;
    }
}

__global__ void __launch_bounds__(NA_NT, 5) k_na_rows(NaArgs a) {
    __shared__ ulonglong2 s_xy[NA_TJ], s_zq[NA_TJ], s_c[NA_TJ];
    __shared__ int2 s_e[NA_TJ];
    __shared__ double s_p[3][NA_TJ];  // the parameters as they are (the plain formula)
    __shared__ double4_32a s_sum[NA_NT / 32][32];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int i = blockIdx.x * NA_TI + lane;
    double xi[3], pi[3];
    na_atom(a, i, -1e6, xi, pi);
    u64 m1, m6, m12;
    int e1, e6, e12;
    bool in_range = split64(pi[0], m1, e1);
    in_range = split64(pi[1], m6, e6) && in_range && !(pi[1] < 0.0);  // the forms keep no sign of C6, C12
    in_range = split64(pi[2], m12, e12) && in_range && !(pi[2] < 0.0);
    const int ce = (e6 << 16) | e12;
    const uint32_t qs = (uint32_t)(bits64(pi[0]) >> 32) & 0x80000000u;
    long long fi[3];
    bool i_fix = in_range;
    for (int k = 0; k < 3; k++) i_fix = fix64(xi[k], fi[k]) && i_fix;
    if (i >= a.n) {
        fi[0] = fi[1] = fi[2] = -FIX_FAR;
        i_fix = true;
    }
    const int len = (a.n + a.chunks - 1) / a.chunks;
    const int j0 = blockIdx.y * len, j1 = min(a.n, j0 + len);
    double gx = 0.0, gy = 0.0, gz = 0.0, es6 = 0.0;  // es6: six times the energy
    for (int jt = j0; jt < j1; jt += NA_TJ) {
        double xj[3], pj[3];
        const bool real = jt + tid < j1;
        na_atom(a, real ? jt + tid : a.n, 1e6, xj, pj);
        u64 u1, u6, u12;
        int f1, f6, f12;
        bool range = split64(pj[0], u1, f1) && in_range;
        range = split64(pj[1], u6, f6) && range && !(pj[1] < 0.0);
        range = split64(pj[2], u12, f12) && range && !(pj[2] < 0.0);
        long long fj[3] = {FIX_FAR, FIX_FAR, FIX_FAR};
        bool j_fix = i_fix;
        if (real)
            for (int k = 0; k < 3; k++) j_fix = fix64(xj[k], fj[k]) && j_fix;
        // fixed-point coordinates for the tile when all of them fit (the
        // barrier also ends the reads of the last tile)
        const bool fix = __syncthreads_and(j_fix && range);
        const bool plain = fix ? false : __syncthreads_or(!range);
        s_xy[tid] = fix ? make_ulonglong2((u64)fj[0], (u64)fj[1]) : make_ulonglong2(bits64(xj[0]), bits64(xj[1]));
        s_zq[tid] = make_ulonglong2(fix ? (u64)fj[2] : bits64(xj[2]), u1);
        s_c[tid] = make_ulonglong2(u6, u12);
        s_e[tid] = make_int2((int)((uint32_t)f1 | ((uint32_t)(bits64(pj[0]) >> 32) & 0x80000000u)), (f6 << 16) | f12);
        for (int k = 0; k < 3; k++) s_p[k][tid] = pj[k];
        __syncthreads();
        const int kend = min(w * 32 + 32, j1 - jt);
        auto rows = [&](auto FIX) {
            for (int k = w * 32; k < kend; k++) {  // the same j for every lane
                const ulonglong2 xy = s_xy[k], zq = s_zq[k], cj = s_c[k];
                const int2 ej = s_e[k];
                const bool on = jt + k != i;
                Inv64 v;
                bool ok;
                double dx = 1.0, dy = 0.0, dz = 0.0;
                if constexpr (decltype(FIX)::value) {
                    const long long gx_ = (long long)xy.x - fi[0], gy_ = (long long)xy.y - fi[1],
                                    gz_ = (long long)zq.x - fi[2];
                    u64 ax, ay, az;
                    int n;
                    ok = inv64_fix(gx_, gy_, gz_, v, ax, ay, az, n) || !on;
                    dx = fix_to_double(ax, n, gx_);
                    dy = fix_to_double(ay, n, gy_);
                    dz = fix_to_double(az, n, gz_);
                } else {
                    if (on) {
                        dx = from_bits64(xy.x) - xi[0];
                        dy = from_bits64(xy.y) - xi[1];
                        dz = from_bits64(zq.x) - xi[2];
                    }
                    ok = inv64(dx, dy, dz, v);
                }
                const int es = ce + ej.y;
                double f, y;
                inv64_force(v, m1, zq.y, e1 + (ej.x & 0xffff), ((uint32_t)ej.x ^ qs) & 0x80000000u, m6, cj.x,
                            (int)((uint32_t)es >> 16), m12, cj.y, es & 0xffff, f, y);
                if (__any_sync(0xffffffffu, !ok) || plain) {
                    if (decltype(FIX)::value) {
                        dx = 1.0; dy = dz = 0.0;
                        if (on) {
                            dx = a.x[3 * (jt + k)] - xi[0];
                            dy = a.x[3 * (jt + k) + 1] - xi[1];
                            dz = a.x[3 * (jt + k) + 2] - xi[2];
                        }
                    }
                    const double ri = rsqrt(dx * dx + dy * dy + dz * dz);
                    const double ri2 = ri * ri, ri6 = ri2 * ri2 * ri2;
                    const double p12 = pi[2] * s_p[2][k] * ri6 * ri6, u = p12 - pi[1] * s_p[1][k] * ri6,
                                 e = pi[0] * s_p[0][k] * ri;
                    f = ((u + p12) + e) * ri2;
                    y = fma(6.0, e, u);
                }
                if (!on) f = y = 0.0;
                es6 += y;
                gx = fma(f, dx, gx);
                gy = fma(f, dy, gy);
                gz = fma(f, dz, gz);
            }
        };
        if (fix) rows(std::true_type{});
        else rows(std::false_type{});
    }
    __syncthreads();
    s_sum[w][lane] = make_double4_32a(gx, gy, gz, es6 * (1.0 / 6.0));
    __syncthreads();
    // component w of atom `lane`, the warps in order
    const double *col = reinterpret_cast<const double *>(&s_sum[0][0]) + 4 * lane + w;
    double sum = col[0];
    for (int v = 1; v < NA_NT / 32; v++) sum += col[4 * 32 * v];
    if (i < a.n) a.part[((size_t)blockIdx.y * a.n + i) * 4 + w] = sum;
}

// four threads per atom (gradient components and energy)
__global__ void __launch_bounds__(4 * NA_FT) k_na_final(NaArgs a) {
    __shared__ double se[NA_FT];
    const int i = blockIdx.x * NA_FT + threadIdx.x / 4, k = threadIdx.x % 4;
    bool bad = false;
    double s = 0.0;
    if (i < a.n) {
#pragma unroll 4
        for (int ch = 0; ch < a.chunks; ch++) s += a.part[((size_t)ch * a.n + i) * 4 + k];
        if (k < 3) {
            a.g[3 * i + k] = s;
            bad = !isfinite(s);
        } else {
            s *= 0.5;  // each pair appears in two rows
        }
    }
    if (k == 3) se[threadIdx.x / 4] = s;
    if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(a.ticket + 1, 1u);
    if (threadIdx.x >= 32) return;
    const int lane = threadIdx.x;
    double t = se[lane] + se[lane + 32];
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    unsigned last = 0u;
    if (lane == 0) {
        a.eblock[blockIdx.x] = t;
        __threadfence();
        last = atomicAdd(a.ticket, 1u) == gridDim.x - 1 ? 1u : 0u;
    }
    if (!__shfl_sync(0xffffffffu, last, 0)) return;
    __threadfence();  // last block: total over the blocks in a fixed order
    double tot = 0.0;
    for (int b = lane; b < (int)gridDim.x; b += 32) tot += __ldcg(&a.eblock[b]);
    for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
    if (lane == 0) {
        *a.e = tot;
        if (!isfinite(tot)) atomicOr(a.ticket + 1, 1u);
    }
}

}  // namespace

extern "C" ffmin_status ffmin_pair_energy_grad_noalloc(const double *x_dev, const double *charge_dev,
                                                      const double *sigma_dev, const double *epsilon_dev,
                                                      int32_t n_atoms, double coulomb_c, double *g_dev,
                                                      double *e_dev, void *cuda_stream) {
    if (n_atoms < 1 || n_atoms > NA_MAX_ATOMS || !x_dev || !charge_dev || !sigma_dev || !epsilon_dev ||
        !g_dev || !e_dev)
        return FFMIN_ERR_INVALID_ARG;  // sizes beyond the fixed scratch are refused
    if (!(coulomb_c >= 0.0) || !std::isfinite(coulomb_c)) return FFMIN_ERR_INVALID_ARG;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= NA_MAX_DEVICES) return FFMIN_ERR_CUDA;
    double *scr;
    {
        std::lock_guard<std::mutex> lock(g_scratch_lock);
        if (!g_scratch_ptr[dev]) {  // first call on this device: look up the array's device address
            void *p = nullptr;
            if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) return FFMIN_ERR_CUDA;
            g_scratch_ptr[dev] = (double *)p;
        }
        scr = g_scratch_ptr[dev];
    }
    cudaStream_t s = (cudaStream_t)cuda_stream;
    NaArgs a;
    a.x = x_dev; a.q = charge_dev; a.sigma = sigma_dev; a.eps = epsilon_dev;
    a.n = n_atoms;
    a.sqrt_c = std::sqrt(coulomb_c == 0.0 ? 1389.38757 / 4.184 : coulomb_c);
    a.g = g_dev;
    a.e = e_dev;
    a.par = scr;
    a.part = scr + (size_t)3 * n_atoms;
    a.chunks = (int)std::min<size_t>(NA_CHUNKS, (NA_ROWS - (size_t)3 * n_atoms) / ((size_t)4 * n_atoms));
    a.eblock = scr + NA_ROWS;
    a.ticket = (unsigned int *)(a.eblock + NA_MAX_BLOCKS);
    k_na_prepare<<<(n_atoms + NA_NT - 1) / NA_NT, NA_NT, 0, s>>>(a);
    k_na_rows<<<dim3((n_atoms + NA_TI - 1) / NA_TI, a.chunks), NA_NT, 0, s>>>(a);
    k_na_final<<<(n_atoms + NA_FT - 1) / NA_FT, 4 * NA_FT, 0, s>>>(a);
    if (cudaGetLastError() != cudaSuccess) return FFMIN_ERR_CUDA;
    // the status needs the flag: read it back (pageable host word) and wait
    unsigned int flag = 0u;
    if (cudaMemcpyAsync(&flag, a.ticket + 1, sizeof(flag), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return FFMIN_ERR_CUDA;
    return flag ? FFMIN_ERR_NONFINITE : FFMIN_OK;
}
