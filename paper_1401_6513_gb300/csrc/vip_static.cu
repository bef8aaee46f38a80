// vip_bicgstab_static: a BiCGSTAB solve that allocates no device memory.
//
// For callers that cannot call cudaMalloc while they run -- for example a host
// process whose device memory is owned by another framework's pooling allocator,
// a real-time loop that must not allocate, or code that runs with a fixed device
// memory budget.  The caller passes the matrix (CSR), the right-hand side and the
// solution vector in its own device memory; every other buffer the solver needs
// (Krylov vectors, reduction partials, the grid-barrier words, the result record)
// lives in file-scope static device arrays of fixed size (about 6.3 MB), which a
// device holds from the moment the library's code is loaded on it until the
// process exits.
//
// The solver is plain FP64 BiCGSTAB in one cooperative launch of a block per SM: each block
// keeps its rows' vectors in shared memory for the whole call, and their part of the matrix
// where that fits too (rows of about 15 entries at the largest size), read once and
// coalesced; only p and s, which other blocks gather from, go to the workspace.  An
// iteration is five phases between grid barriers (0.9 us each, every wait bounded: 2 s, then
// VIP_ERR_TIMEOUT), three of them with a reduction (about 2 us, a chain of dependent FP64
// additions), and is bound by those and by the FP64 unit.  131,072 rows of 5 entries: 57 ->
// 23 us per iteration (25 with 256 or 1,024 threads a block; before:
// four blocks per SM meeting at a barrier that slept, CSR rows read by one thread each from
// memory, six phases).
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>

#include "../../include/vip.h"

namespace {

constexpr int64_t MAX_ROWS = VIP_STATIC_MAX_ROWS;
constexpr int NVEC = 6;                      // r, rhat, p, v, s, t
constexpr int MAX_BLOCKS = 1024;
constexpr int NQ = 3;                        // reduced quantities per phase, at most
constexpr int THREADS = 512, WARPS = THREADS / 32;
// At least MIN_ROWS rows per block.  Up to ONE_BLOCK rows the first block solves alone if its
// shared memory holds the matrix (its barrier is a __syncthreads: 204 rows of 5 entries take
// 11.5 us per iteration, 15.2 in four blocks); 500 rows of 500 entries take 546 us in one block
// and 157 in eight.  The host does not know the entry count, so the kernel decides.
constexpr int ONE_BLOCK = 512, MIN_ROWS = 64;
// Shared memory asked for the matrix up to ONE_BLOCK rows: 32 entries a row, SMALL_MATRIX at
// least (a dense one of 120 rows in two blocks); a solve of 250 rows leaves half of its SM to
// others.  Beyond, where every SM has a block, all there is.
constexpr int64_t SMALL_MATRIX = 96 << 10;
constexpr int64_t OFF_PART = NVEC * MAX_ROWS;
// two sets of block partials, used by alternate reductions: a block that runs
// ahead into the next reduction never overwrites a partial another block is
// still reading
constexpr int64_t OFF_RES = OFF_PART + 2LL * NQ * MAX_BLOCKS;
constexpr int64_t SCRATCH = OFF_RES + 8;     // doubles (about 6.3 MB); the last 8: results, barrier word

// The shared workspace.  In host code this name is only a stand-in for the
// device object; its device address comes from cudaGetSymbolAddress.
static __device__ __align__(256) double g_scratch[SCRATCH];

struct Args {
    int64_t n;
    const int64_t* ptr;
    const int32_t* col;
    const double* val;
    const double* b;
    double* x;
    double rtol;
    int max_iters;
    double* ws;          // device address of g_scratch
    unsigned int* bar;   // the barrier word, in its result record
    int vec_smem;        // a block's vectors are in shared memory (else in the workspace)
    int64_t mat_smem;    // bytes of shared memory for a block's part of the matrix
};

__device__ __forceinline__ unsigned ld_acq(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ unsigned long long now_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Grid barrier with a bounded wait; returns false (and flags the timeout) after 2 s.  Block 0
// adds 2^31 - (blocks - 1), the others 1: the word's top bit flips when the last arrives.
__device__ __noinline__ bool barrier(unsigned* bar, unsigned nb, double* res) {
    __shared__ int ok;
    __syncthreads();
    if (nb == 1) return true;
    if (threadIdx.x == 0) {
        ok = 1;
        const unsigned add = blockIdx.x == 0 ? 0x80000000u - (nb - 1u) : 1u;
        unsigned old;
        asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], %2;" : "=r"(old) : "l"(bar), "r"(add) : "memory");
        const unsigned long long t0 = now_ns();
        for (unsigned k = 1; ((ld_acq(bar) ^ old) & 0x80000000u) == 0; ++k) {
            if ((k & 63u) == 0 && now_ns() - t0 > 2000000000ull) {
                res[3] = 1.0;  // timeout flag
                ok = 0;
                break;
            }
        }
    }
    __syncthreads();
    return ok != 0;
}

struct Scalars {
    double bnorm, tol, rho, alpha, omega, beta;
    int it, status, stop, half;
};

__global__ void __launch_bounds__(THREADS, 1) k_bicgstab_static(Args a) {
    extern __shared__ __align__(16) double sm[];
    __shared__ double red[NQ][THREADS];
    __shared__ double tot[NQ];
    __shared__ Scalars S;
    const int64_t n = a.n;
    unsigned nb = gridDim.x;
    if (nb > 1 && n <= ONE_BLOCK && (a.ptr[n] - a.ptr[0]) * 12 + (n + 1) * 8 <= a.mat_smem) {
        if (blockIdx.x > 0) return;
        nb = 1;
    }
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t row0 = n * blockIdx.x / nb;
    const int rows = (int)(n * (blockIdx.x + 1) / nb - row0);
    double* gp = a.ws + 2 * MAX_ROWS;   // p and s of every row
    double* gs = a.ws + 4 * MAX_ROWS;
    double* part = a.ws + OFF_PART;
    double* res = a.ws + OFF_RES;
    // the block's vectors: shared memory, or its rows of the workspace (and of x)
    auto vec = [&](int k) -> double* { return a.vec_smem ? sm + (int64_t)k * rows : a.ws + k * MAX_ROWS + row0; };
    double *r = vec(0), *rh = vec(1), *p = vec(2), *v = vec(3), *s = vec(4), *t = vec(5);
    double* x = a.vec_smem ? sm + (int64_t)NVEC * rows : a.x + row0;
    const int64_t e0 = a.ptr[row0];
    const double* val = a.val + e0;
    const int32_t* col = a.col + e0;
    const int64_t ne = a.ptr[row0 + rows] - e0;
    // the rows' first entries, then their columns and values
    int64_t* first = reinterpret_cast<int64_t*>(sm) + (a.vec_smem ? (int64_t)(NVEC + 1) * rows : 0);
    const bool row_smem = a.mat_smem >= (rows + 1) * 8;
    if (row_smem)
        for (int i = tid; i <= rows; i += THREADS) first[i] = a.ptr[row0 + i] - e0;
    if (ne * 12 + (rows + 1) * 8 <= a.mat_smem) {
        double* sv = reinterpret_cast<double*>(first + rows + 1);
        int32_t* sc = reinterpret_cast<int32_t*>(sv + ne);
        for (int64_t k = tid; k < ne; k += THREADS) {
            sv[k] = val[k];
            sc[k] = col[k];
        }
        val = sv;
        col = sc;
    }
    if (a.vec_smem)
        for (int i = tid; i < rows; i += THREADS) x[i] = a.x[row0 + i];
    __syncthreads();
    // (A in)_row in entry order; four entries' gathers at a time
    auto row_sum = [&](int i, const double* in) -> double {
        const int64_t k1 = row_smem ? first[i + 1] : a.ptr[row0 + i + 1] - e0;
        double sum = 0.0;
        for (int64_t k = row_smem ? first[i] : a.ptr[row0 + i] - e0; k < k1; k += 4) {
            double av[4], g[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                av[u] = g[u] = 0.0;
                if (k + u < k1) {
                    av[u] = val[k + u];
                    g[u] = in[col[k + u]];
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (k + u < k1) sum += av[u] * g[u];
        }
        return sum;
    };
    int set = 0;  // partial set of the next reduction
    // totals of q[0..nq) in a fixed order: a warp per quantity adds the threads' values, then
    // the blocks' partials
    auto reduce = [&](const double (&q)[NQ], int nq) -> bool {
#pragma unroll
        for (int k = 0; k < NQ; ++k)
            if (k < nq) red[k][tid] = q[k];
        __syncthreads();
        double* ps = part + (int64_t)set * NQ * MAX_BLOCKS;
        set ^= 1;
        if (warp < nq) {
            const double* src = red[warp] + lane;
            double w = 0.0;
#pragma unroll
            for (int k = 0; k < WARPS; k += 4)
                w += (src[32 * k] + src[32 * k + 32]) + (src[32 * k + 64] + src[32 * k + 96]);
            for (int o = 16; o > 0; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
            if (lane == 0) __stcg(ps + (int64_t)warp * MAX_BLOCKS + blockIdx.x, w);
        }
        if (!barrier(a.bar, nb, res)) return false;
        if (warp < nq) {
            double w = 0.0;
            for (unsigned bb = lane; bb < nb; bb += 5 * 32) {
                double g[5];
#pragma unroll
                for (int u = 0; u < 5; ++u)
                    g[u] = bb + 32 * u < nb ? __ldcg(ps + (int64_t)warp * MAX_BLOCKS + bb + 32 * u) : 0.0;
                w += ((g[0] + g[1]) + (g[2] + g[3])) + g[4];
            }
            for (int o = 16; o > 0; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
            if (lane == 0) tot[warp] = w;
        }
        __syncthreads();
        return true;
    };

    // r = b - A x, rhat = r; ||b||, ||r||
    {
        double q[NQ] = {0.0, 0.0, 0.0};
        for (int i = tid; i < rows; i += THREADS) {
            const double bi = a.b[row0 + i];
            const double ri = bi - row_sum(i, a.x);
            r[i] = ri;
            rh[i] = ri;
            p[i] = 0.0;
            v[i] = 0.0;
            q[0] += bi * bi;
            q[1] += ri * ri;
        }
        if (!reduce(q, 2)) return;
    }
    // The scalars are one thread's: a quotient or a root by all threads of the block would
    // cost its FP64 unit (two lanes per clock) about 2 us each.
    if (tid == 0) {
        S = Scalars{};
        S.bnorm = sqrt(tot[0]);
        S.tol = a.rtol * S.bnorm;
        S.rho = tot[1];
        S.alpha = S.omega = 1.0;
        S.beta = S.rho;  // (rho / 1) (1 / 1); p = v = 0
        S.stop = S.bnorm == 0.0 || sqrt(tot[1]) <= S.tol;
    }
    __syncthreads();
    if (S.bnorm == 0.0)
        for (int i = tid; i < rows; i += THREADS) x[i] = 0.0;
    while (!S.stop) {
        if (S.it >= a.max_iters) {
            if (tid == 0) S.status = VIP_ERR_NOT_CONVERGED;
            break;
        }
        for (int i = tid; i < rows; i += THREADS) {
            const double pi = r[i] + S.beta * (p[i] - S.omega * v[i]);
            p[i] = pi;
            gp[row0 + i] = pi;
        }
        if (!barrier(a.bar, nb, res)) return;
        {
            double q[NQ] = {0.0, 0.0, 0.0};
            for (int i = tid; i < rows; i += THREADS) {
                const double vi = row_sum(i, gp);
                v[i] = vi;
                q[0] += rh[i] * vi;
            }
            if (!reduce(q, 1)) return;
        }
        if (tid == 0) {
            if (tot[0] == 0.0) { S.status = VIP_ERR_BREAKDOWN; S.stop = 1; }
            else S.alpha = S.rho / tot[0];
        }
        __syncthreads();
        if (S.stop) break;
        for (int i = tid; i < rows; i += THREADS) {
            const double si = r[i] - S.alpha * v[i];
            s[i] = si;
            gs[row0 + i] = si;
        }
        if (!barrier(a.bar, nb, res)) return;
        {   // s . s is tested with t's products: a converged s wastes the last application,
            // and every iteration saves a reduction
            double q[NQ] = {0.0, 0.0, 0.0};
            for (int i = tid; i < rows; i += THREADS) {
                const double ti = row_sum(i, gs);
                t[i] = ti;
                const double si = s[i];
                q[0] += ti * si;
                q[1] += ti * ti;
                q[2] += si * si;
            }
            if (!reduce(q, 3)) return;
        }
        if (tid == 0) {
            ++S.it;
            if (sqrt(tot[2]) <= S.tol) S.stop = S.half = 1;
            else if (tot[1] == 0.0) { S.status = VIP_ERR_BREAKDOWN; S.stop = 1; }
            else S.omega = tot[0] / tot[1];
        }
        __syncthreads();
        if (S.stop) break;
        {
            double q[NQ] = {0.0, 0.0, 0.0};
            for (int i = tid; i < rows; i += THREADS) {
                const double si = s[i];
                x[i] += S.alpha * p[i] + S.omega * si;
                const double ri = si - S.omega * t[i];
                r[i] = ri;
                q[0] += ri * ri;
                q[1] += rh[i] * ri;
            }
            if (!reduce(q, 2)) return;
        }
        if (tid == 0) {
            const double rho = tot[1];
            if (sqrt(tot[0]) <= S.tol) {
                S.stop = 1;
            } else if (rho == 0.0 || S.omega == 0.0) {
                S.status = VIP_ERR_BREAKDOWN;
                S.stop = 1;
            } else {
                S.beta = (rho / S.rho) * (S.alpha / S.omega);
                S.rho = rho;
            }
        }
        __syncthreads();
    }
    if (S.half)  // s converged: x stops half way through its iteration
        for (int i = tid; i < rows; i += THREADS) x[i] += S.alpha * p[i];
    // x back, and the true residual of the returned x
    if (a.vec_smem)
        for (int i = tid; i < rows; i += THREADS) a.x[row0 + i] = x[i];
    if (!barrier(a.bar, nb, res)) return;
    double q[NQ] = {0.0, 0.0, 0.0};
    for (int i = tid; i < rows; i += THREADS) {
        const double ri = a.b[row0 + i] - row_sum(i, a.x);
        q[0] += ri * ri;
    }
    if (!reduce(q, 1)) return;
    if (blockIdx.x == 0 && tid == 0) {
        res[0] = (double)S.it;
        res[1] = S.bnorm > 0.0 ? sqrt(tot[0]) / S.bnorm : 0.0;
        res[2] = (double)S.status;
    }
}

// Device addresses of the workspace, looked up once per device (the first call
// on a device also loads this module's kernels there).
std::mutex g_mu;
constexpr int MAX_DEVICES = 64;
double* g_ws_addr[MAX_DEVICES] = {};
int g_sms[MAX_DEVICES] = {}, g_smem[MAX_DEVICES] = {};  // multiprocessors; shared memory a block may have

// makes `device` current for the call and puts the caller's device back
struct DeviceGuard {
    int prev = -1;
    bool ok = false;
    explicit DeviceGuard(int device) {
        if (cudaGetDevice(&prev) != cudaSuccess) return;
        ok = cudaSetDevice(device) == cudaSuccess;
    }
    ~DeviceGuard() {
        if (prev >= 0) cudaSetDevice(prev);
    }
};

vip_status setup(int device, double** ws, int* sms, int* smem) {
    std::lock_guard<std::mutex> lock(g_mu);
    if (!g_ws_addr[device]) {
        void* p1 = nullptr;
        cudaFuncAttributes fa{};
        int optin = 0;
        if (cudaGetSymbolAddress(&p1, g_scratch) != cudaSuccess) return VIP_ERR_CUDA;
        if (cudaDeviceGetAttribute(&g_sms[device], cudaDevAttrMultiProcessorCount, device) != cudaSuccess ||
            cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device) != cudaSuccess ||
            cudaFuncGetAttributes(&fa, k_bicgstab_static) != cudaSuccess)
            return VIP_ERR_CUDA;
        const int dyn = std::max(0, optin - (int)fa.sharedSizeBytes - 1024);
        if (cudaFuncSetAttribute(k_bicgstab_static, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn) != cudaSuccess)
            return VIP_ERR_CUDA;
        g_smem[device] = dyn;
        g_ws_addr[device] = static_cast<double*>(p1);
    }
    *ws = g_ws_addr[device];
    *sms = g_sms[device];
    *smem = g_smem[device];
    return VIP_OK;
}

// q is managed memory, or device memory of `device` (memory of another GPU would be
// read as a peer address, which faults without peer access)
bool on_device(const void* q, int device) {
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, q) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeManaged || (at.type == cudaMemoryTypeDevice && at.device == device);
}

}  // namespace

extern "C" vip_status vip_bicgstab_static(int device, void* cuda_stream, int64_t n, const int64_t* row_ptr,
                                          const int32_t* col, const double* val, const double* b, double* x,
                                          double rtol, int32_t max_iters, int32_t* iters, double* relres) {
    if (n < 1 || n > MAX_ROWS) return VIP_ERR_ARG;  // beyond the static workspace
    if (!row_ptr || !col || !val || !b || !x || !(rtol > 0.0) || max_iters < 1) return VIP_ERR_ARG;
    if (device < 0 || device >= MAX_DEVICES) return VIP_ERR_ARG;
    DeviceGuard guard(device);
    if (!guard.ok) return VIP_ERR_CUDA;
    if (!on_device(row_ptr, device) || !on_device(col, device) || !on_device(val, device) ||
        !on_device(b, device) || !on_device(x, device))
        return VIP_ERR_ARG;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    {   // the call synchronises its stream and reads results back: it cannot be captured
        cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(st, &cs) != cudaSuccess) return VIP_ERR_CUDA;
        if (cs != cudaStreamCaptureStatusNone) return VIP_ERR_ARG;
    }
    double* ws = nullptr;
    int sms = 0, smem = 0;
    vip_status st0 = setup(device, &ws, &sms, &smem);
    if (st0 != VIP_OK) return st0;
    const int grid = (int)std::min<int64_t>({(n + MIN_ROWS - 1) / MIN_ROWS, (int64_t)sms, (int64_t)MAX_BLOCKS});
    Args a{n, row_ptr, col, val, b, x, rtol, max_iters, ws, reinterpret_cast<unsigned int*>(ws + OFF_RES + 4), 0, 0};
    const int64_t rows = n <= ONE_BLOCK ? n : (n + grid - 1) / grid;   // of a block, at most
    const int64_t vb = (NVEC + 1) * rows * 8;
    a.vec_smem = vb <= smem;
    const int64_t dyn = n <= ONE_BLOCK ? std::min<int64_t>(smem, vb + std::max(SMALL_MATRIX, n * 32 * 12)) : smem;
    a.mat_smem = dyn - (a.vec_smem ? vb : 0);
    // the barrier word and the result record start at zero on every call; the
    // Krylov vectors and partials need no clearing (each is written before it is read)
    if (cudaMemsetAsync(ws + OFF_RES, 0, 8 * sizeof(double), st) != cudaSuccess) return VIP_ERR_CUDA;
    void* args[] = {&a};
    if (cudaLaunchCooperativeKernel((const void*)k_bicgstab_static, dim3(grid), dim3(THREADS), args, (size_t)dyn, st) !=
        cudaSuccess)
        return VIP_ERR_CUDA;
    double h[4] = {0, 0, 0, 0};
    if (cudaMemcpyAsync(h, ws + OFF_RES, 4 * sizeof(double), cudaMemcpyDeviceToHost, st) != cudaSuccess)
        return VIP_ERR_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return VIP_ERR_CUDA;
    if (iters) *iters = (int32_t)h[0];
    if (relres) *relres = h[1];
    if (h[3] != 0.0) return VIP_ERR_TIMEOUT;
    if (h[2] != 0.0) return (vip_status)(int)h[2];
    return VIP_OK;
}
