// Krylov solves of Eqs. (12) and (13): one persistent cooperative launch solves a
// batch of independent sparse systems (block-diagonal SELL-32 operator, each
// system a contiguous range of slices) with BiCGSTAB (van der Vorst, 1992),
// right-preconditioned by one V-cycle of the aggregation multigrid for Eq. (13),
// inside an FP64 iterative-refinement loop:
//
//   repeat:  r = b - A x   (FP64 operator, FP64 vectors);  stop if ||r|| <= rtol ||b||
//            solve A d = r by BiCGSTAB in precision T from d = 0 with r_hat = r,
//            until ||r_d|| <= tol_in, or until |r_hat.r| or |r_hat.v| falls below
//            a small fraction of its norms (restart);   x += d
//
// Two precisions: T for the Krylov vectors, operator applications and vector
// updates, TM for the V-cycle (its vectors, operators and arithmetic).
//   <double, double>  the plain FP64 form (tol_in = rtol ||b|| / 2: one pass);
//   <float, float>    the mixed form: FP32 arithmetic on FP32 copies of the
//                     operators and FP32 vectors inside, tol_in =
//                     max(inner_rtol ||r||, rtol ||b|| / 2), the correction d
//                     accumulated as an FP32 (hi, lo) pair by error-free
//                     transformations (no FP64 operation per row inside);
//   <double, float>   FP64 Krylov iteration with an FP32 V-cycle.
// FP32 applications of the fine operator use the differenced row form
// sum_k a_ik (x_k - x_i) + rowsum_i x_i with the FP64 row sum rounded to FP32: on
// the smooth vectors of a Poisson solve x_k - x_i is small and exact, so the
// large, nearly cancelling products a_ik x_k of the plain form never appear.
//
// Every system keeps its own scalars; all systems advance in lock step, and the
// slices of the systems still iterating are re-spread over all blocks whenever a
// system finishes.  Dot products are reduced deterministically: per-thread sums in
// registers, a fixed tree over the block, per-block partials summed in block order by
// every block, so all blocks hold identical scalars.  Blocks meet at a grid barrier
// whose wait is bounded (2 s, then VIP_ERR_TIMEOUT).
//
// What bounds it (GB300): an iteration is 19-29 phases between grid barriers of 0.9 us,
// each a chain of dependent trips to memory, FP64 scalar steps (a dependent FP64
// operation takes about 0.1 us on this part) and instruction fetches: the launch's code
// is larger than the instruction caches, so what every iteration executes is kept in one
// copy (one V-cycle and one operator application for both half steps, reductions and
// barriers as calls: 220 KB of instructions, 400 in two copies).  512 threads with 128
// registers beat 384, 640 and 768 (2.1M rows in FP32: 0.39 ms per iteration against 0.44,
// 0.43 and 0.49) and, but for the sets of LARGE_STREAM, 1,024.  A row's entries come a warp's
// item ahead into L2 by two bulk prefetches, which hold no registers.  The FP64 unit (two
// lanes per clock) bounds the coarse tiles and half of a fine pass, so FP64 sums hold no
// operation but their products.  Microseconds per Poisson iteration (in brackets: 1,024 threads
// of 64 registers for every set, one row per lane, no work items): 4,096 rows FP64 70 (96), 65,536 rows FP64
// 110 (136), 525,065 rows FP32 132 (198), 2.1M rows FP32 314 (477); triangular cavities in FP64,
// all active: 16 of 217,425 rows 226 (246), 20 of 671,018 477 (498), 64 of 2.7M 1398 (1461); the
// last with an FP32 V-cycle 1076 (1124).
#include <cstdio>
#include <cstring>
#include <type_traits>
#include <vector>

#include "vip_internal.cuh"

namespace vip {

constexpr int NT64 = 512, NT32 = 512;  // threads of the launch's CTAs (one per SM): FP64 and FP32 iteration
// A preconditioned FP64 iteration takes twice the threads where it streams LARGE_STREAM operator
// entries or more (those of slices without a shared stencil): the entries then come from memory
// beyond L2 in every pass, and twice the warps hide more of that than the wider batches of fewer
// warps.  The form has 64 registers a thread, so it keeps the plain row loop only (no four-slice
// items, no rows shared by lanes), loads a tile's coefficients when it needs them and sums b_1
// in a phase of its own.  Microseconds per iteration with 512 and 1,024 threads, all FP64: 0.67M
// rows of triangular cavities (9.2M entries) 477 and 480, 1.9M rows (27M) 1072 and 1004, 2.7M
// rows (39M) 1507 and 1398; with an FP32 V-cycle 367 and 380, 865 and 762, 1208 and 1076.
// Without a preconditioner (Helmholtz, a fifth of the passes) 512 threads stay ahead: 253
// and 260, 383 and 404.
constexpr int NT64_LARGE = 1024;
#ifndef VIP_LARGE_STREAM   // (set by the tests)
#define VIP_LARGE_STREAM 16000000
#endif
constexpr int64_t LARGE_STREAM = VIP_LARGE_STREAM;
constexpr int MAXSYS = 128;
constexpr int KSMEM_TILE = (36 * 36 + 32 * 32) * (int)sizeof(double);  // a coarse tile and its halo, its own cells
// per-thread dot-product sums: RED_SLOTS systems x RED_Q quantities x NT values of T,
// or, for a block that holds more systems, per-warp sums [MAXSYS_PB][NQ][KWARPS] in FP64
constexpr int RED_SLOTS = 2, RED_Q = 3;
// entries of the shared stencils kept in shared memory for the whole launch (a launch
// with more of them reads them from global memory)
constexpr int UCAP = 2560;
template <class TM>
constexpr int ust_bytes() {
    return UCAP * (int)(sizeof(TM) + sizeof(int32_t));
}
template <class T, int NT>
constexpr int red_bytes() {
    const int a = RED_SLOTS * RED_Q * NT * (int)sizeof(T), b = MAXSYS_PB * NQ * (NT / 32) * (int)sizeof(double);
    return a > b ? a : b;
}

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ int ld_volatile_i(const int* p) {
    return *(const volatile int*)p;
}
__device__ __forceinline__ uint64_t gtimer() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ unsigned atom_add_acq_rel(unsigned* p, unsigned v) {
    unsigned old;
    asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
    return old;
}

// Grid barrier for a cooperative launch; returns false after a timeout.
// bar[0] is an arrival counter whose top bit flips once per barrier: thread 0 of
// CTA 0 adds 2^31 - (nblocks - 1), every other CTA adds 1, so the counter moves by
// exactly 2^31 per barrier and its top bit changes precisely when the last CTA has
// arrived (partial sums stay below the next multiple of 2^31).  Each CTA polls the
// same word until its top bit differs from the value it saw when arriving, so no
// separate release store has to travel after the last arrival.  The arrival is an
// acquire-release add and the poll an acquire load: every write before the barrier
// happens before every read after it, for weak loads too.  The counter must start
// at 0.  A wait gives up after 2 s (VIP_ERR_TIMEOUT), or early when another CTA has
// already reported a timeout.
__device__ __noinline__ bool grid_sync(uint32_t* bar, unsigned nblocks, int32_t* status) {
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        int ok = 1;
        const unsigned add = blockIdx.x == 0 ? 0x80000000u - (nblocks - 1u) : 1u;
        const unsigned old = atom_add_acq_rel(bar, add);
        const uint64_t t0 = gtimer();
        for (unsigned k = 1; ((ld_acquire(bar) ^ old) & 0x80000000u) == 0; ++k) {
            if ((k & 63u) == 0 && (ld_volatile_i(status) == VIP_ERR_TIMEOUT || gtimer() - t0 > 2000000000ull)) {
                set_status(status, VIP_ERR_TIMEOUT);
                ok = 0;
                break;
            }
        }
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

template <class T, class TM>
struct KArgs {
    const int4* sinfo;      // packed slice records (Sell::sinfo)
    const int32_t* col;
    const double* a64;      // FP64 operator (refinement residual)
    const T* aT;            // the operator in T (Krylov applications)
    const TM* aM;           // the operator in TM (the V-cycle's fine level)
    const int32_t* ucode;   // shared stencils of the uniform slices
    int nust;               // their entries, if kept in shared memory (else 0)
    const double* u64;
    const T* uT;
    const TM* uM;
    const float* rs32;      // FP64 row sums rounded to FP32 (FP32 differenced rows)
    const int32_t* slice_sys;
    const int32_t* blk_s0;
    const int32_t* blk_s1;
    const int32_t* blk_g0;
    const int32_t* blk_ng;
    const int32_t* sys_b0;
    const int32_t* sys_b1;
    const int32_t* sys_s0;   // [nsys] first slice of each system
    const int32_t* sys_s1;   // [nsys] one past its last slice
    double* partial;     // [2][nsys][NQ][nblocks], zero where a block has no rows of a system
    uint32_t* bar;
    int nsys;
    const double* b;
    double* x;
    double* dx;          // the pass's correction: FP64, or an FP32 (hi, lo) pair per row in the
                         // FP32 iteration (the same 8 bytes), accumulated without rounding loss
    T *r, *rhat, *p, *v, *s, *t;
    double rtol, inner_rtol;
    int max_iters, max_outer, max_pass;
    int32_t* out_iters;
    int32_t* out_outer;
    double* out_relres;
    int32_t* out_status;
    int32_t* status;
    int use_mg;          // right preconditioning by one multigrid V-cycle
    int prefetch;        // the iteration's vectors exceed L2: phases prefetch their streamed rows
    MgDev<TM> mg;
    T *phat, *shat;      // M^{-1} p and M^{-1} s (alias p and s without a preconditioner)
};

struct SysState {
    double bnorm, rnorm, tol, rho, alpha, omega, beta, rhat_norm, relres;
    int outer_active;  // still solving
    int inner_active;  // inside a BiCGSTAB pass
    int s_conv;        // ||s|| met the inner tolerance this iteration
    int zero_x;        // b == 0: set x = 0
    int pass_bad;      // the pass produced a non-finite or diverging correction: discard it
    int bad_passes;    // consecutive discarded passes
    double r0_in;      // ||r|| at the start of the pass
    int pass_cap;      // iteration cap of the current pass (halved after a discarded pass)
    int iters, outer, pass_iters, status;
    float alpha_f, omega_f, beta_f;  // the scalars rounded to FP32 (FP32 vector updates)
};

// the scalar of precision T: the FP64 value, or its FP32 rounding
template <class T>
__device__ __forceinline__ T sc(double d, float f);
template <>
__device__ __forceinline__ double sc<double>(double d, float) { return d; }
template <>
__device__ __forceinline__ float sc<float>(double, float f) { return f; }

// A reduced value is usable if finite.
__device__ __forceinline__ bool fin(double v) { return isfinite(v); }

// Loads of vectors that the launch itself writes: plain (weak) global loads, which
// may hit in L1.  They are ordered after the writes of the previous phase by the
// grid barrier (a GPU-scope acquire in thread 0, then a CTA barrier), which the
// memory model requires to make those writes visible to weak loads; the
// non-coherent read-only path (__ldg) is used only for data no phase writes.
template <class T>
__device__ __forceinline__ T ldv(const T* p) { return *p; }

// Operator entries are streamed once per pass: evict-first, so they do not push the
// gathered vectors out of the caches.
template <class T>
__device__ __forceinline__ T ldm(const T* p) { return __ldcs(p); }

// warp sum (fixed butterfly order)
template <class V>
__device__ __forceinline__ V wsum(V v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Entries sub, sub + L, sub + 2L, ... of one SELL row (lane of the slice's warp, or
// the row's share of an L-lane group): sum_k A[row, k] f(col[row, k]) in precision TA.
// DIFF: the differenced form's sum_k A[row, k] (f(col) - xi), xi the row's own value.
// ROW_U entries are loaded before their gathers and every batch is predicated, so a row
// of up to ROW_U L entries costs three dependent trips to memory (record, entries,
// gathers) instead of the eight of a four-entry loop with a one-entry tail.  A uniform
// slice (at >= 0, warp-uniform) reads its shared stencil instead of its own
// entries: the same values and columns, so the same sum.  at >= 0: the shared stencil;
// else ~at: the row's first entry.  One chain in ascending column order: two chains,
// shorter by half, cost a batch of closed cavities 6 % more iterations (the border
// column's term has to meet a row sum that has cancelled already).
template <int ROW_U, bool DIFF, class TA, class F>
__device__ __forceinline__ TA sell_part(const int32_t* __restrict__ col, const TA* __restrict__ A,
                                        const int32_t* __restrict__ ucode, const TA* __restrict__ uA,
                                        int64_t at, int w, int32_t row, int rl, int sub, int L, TA xi, F&& f) {
    TA sum = (TA)0;
    const int64_t base = ~at + rl;
    const bool shared = at >= 0;
#pragma unroll 1
    for (int k0 = sub; k0 < w; k0 += ROW_U * L) {
        int c[ROW_U];
        TA av[ROW_U], xv[ROW_U];
        if (shared) {
#pragma unroll
            for (int u = 0; u < ROW_U; ++u) {
                const int k = k0 + u * L;
                c[u] = row;
                av[u] = (TA)0;
                if (k < w) {
                    const int32_t code = __ldg(ucode + at + k);
                    c[u] = (code & 1) ? (code >> 1) : row + (code >> 1);
                    av[u] = __ldg(uA + at + k);
                }
            }
        } else {
#pragma unroll
            for (int u = 0; u < ROW_U; ++u) {
                const int k = k0 + u * L;
                c[u] = row;
                av[u] = (TA)0;
                if (k < w) {
                    const int64_t e = base + (int64_t)k * SLICE;
                    c[u] = ldm(col + e);
                    av[u] = ldm(A + e);
                }
            }
        }
#pragma unroll
        for (int u = 0; u < ROW_U; ++u) {
            xv[u] = (TA)0;
            if (k0 + u * L < w) {
                xv[u] = f(c[u]);
                if (DIFF) xv[u] -= xi;
            }
        }
#pragma unroll
        for (int u = 0; u < ROW_U; ++u)
            if (k0 + u * L < w) sum += av[u] * xv[u];
    }
    return sum;
}

// Bulk prefetch of [p, p + bytes) into L2 (TMA; p 16-byte aligned, bytes a multiple
// of 16).  A hint: no register receives data and nothing waits for it.
__device__ __forceinline__ void l2_prefetch(const void* p, uint32_t bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// Error-free FP32 transformations (Knuth's TwoSum; the product's rounding error
// by one fused multiply-add).  The _rn intrinsics are never contracted into a
// fused multiply-add, which would change the rounding these formulas rely on.
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// (hi, lo) += al * ph + om * sh with FP32 operations only: the two products are
// split exactly into rounded value and error, the rounded values are added to hi
// by TwoSum, and every error term goes into lo; the pair is then renormalised.
// The pair carries the sum to about 2^-44 of its size, so the correction of a
// refinement pass keeps the digits an FP64 accumulator would.
__device__ __forceinline__ float2 dd_axpy2(float2 d, float al, float ph, float om, float sh) {
    const float p1 = __fmul_rn(al, ph), e1 = fmaf(al, ph, -p1);
    const float p2 = __fmul_rn(om, sh), e2 = fmaf(om, sh, -p2);
    float s1, t1, s2, t2;
    two_sum(d.x, p1, s1, t1);
    two_sum(s1, p2, s2, t2);
    const float lo = __fadd_rn(d.y, __fadd_rn(__fadd_rn(t1, t2), __fadd_rn(e1, e2)));
    const float hi = __fadd_rn(s2, lo);
    return make_float2(hi, __fsub_rn(lo, __fsub_rn(hi, s2)));
}

// N consecutive values moved by one 16-byte (or narrower) access
template <class T, int N>
struct alignas(sizeof(T) * N > 16 ? 16 : sizeof(T) * N) Pack {
    T v[N];
};
template <int N, class T>
__device__ __forceinline__ Pack<T, N> ldp(const T* p) {
    return *reinterpret_cast<const Pack<T, N>*>(p);
}
template <int N, class T>
__device__ __forceinline__ void stp(T* p, const Pack<T, N>& q) {
    *reinterpret_cast<Pack<T, N>*>(p) = q;
}

// Work items of a block's fine passes, made once per partition: up to four consecutive
// slices of one segment that share a stencil of relative columns, or one slice.  x = slice,
// y = slices | width << 3 | system << 20; two or more slices: z = their shared stencil; one:
// z, w = low and high word of sell_part's `at`.
// A block's items are dealt
// to its warps in turn.  (Slices dealt in turn instead put every boundary slice of a
// lattice whose rows are a multiple of the warps' stride long on the same warp: 38 us per
// pass on the h = 1/64 bumpy channel, whose row is 64 slices, against 13 with items.)
#ifndef VIP_ITEM_CAP   // (set by the tests)
#define VIP_ITEM_CAP 768
#endif
constexpr int ITEM_CAP = VIP_ITEM_CAP;
__device__ __forceinline__ int64_t entries_at(const int4 si) {  // sell_part's `at` of a slice record
    return si.z >= 0 ? (int64_t)si.z : ~((int64_t)si.y << 32 | (uint32_t)si.x);
}
__device__ __forceinline__ int4 make_item(int sl, int count, int g, const int4 si) {
    const int64_t at = entries_at(si);
    return make_int4(sl, count | (si.w & SINFO_WIDTH) << 3 | g << 20, (int)(uint32_t)at, (int)(at >> 32));
}

// Work partition of one block of the Krylov launch (see k_bicgstab): this block's
// slices are nv "virtual" slices in nseg segments, segment k being the slices
// segs[k] + [0, segv[k+1] - segv[k]); its dot-product slots j < ng belong to systems
// sys[j] (j[g] = slot of system g, -1 if none); the partials of system g come from
// blocks [b0[g], b1[g]).
struct Partition {
    int nv, nseg, ng, valid;
    int mixed;                     // 1: the static partition (a segment may span systems)
    int segv[MAXSYS_PB + 1], segs[MAXSYS_PB];
    int b0[MAXSYS], b1[MAXSYS], j[MAXSYS], sys[MAXSYS_PB];
    int ss0[MAXSYS], ss1[MAXSYS];  // slices [ss0[g], ss1[g]) of system g
    uint32_t mask[MAXSYS / 32];    // the set the partition was made for
    int item0[MAXSYS_PB + 1];      // items of segment k: [item0[k], item0[k + 1]) (-1: no list)
};

// Recomputes block bid's partition for the systems flagged in S (inner: inside a
// BiCGSTAB pass; else solving or to be zeroed) if that set changed.  The slices of
// those systems are spread evenly over all nb blocks; every block computes the
// whole partition from the same states, so all blocks agree without communicating.
// A block holds one segment per active system in its range (finished systems in
// between are passed over) and reduces only for those systems.  A partition in
// which some block would hold more than MAXSYS_PB active systems is replaced by
// the launch's static one (one segment of all the block's slices).  Run by one
// thread; kept out of line, as it runs only when a system finishes.
__device__ __noinline__ void partition_update(Partition& P, const SysState* S, int nsys, int inner,
                                              int nb, int bid, const int32_t* blk_s0,
                                              const int32_t* blk_s1, const int32_t* blk_g0,
                                              const int32_t* blk_ng, const int32_t* sys_b0,
                                              const int32_t* sys_b1) {
    uint32_t m[MAXSYS / 32];
    for (int w = 0; w < MAXSYS / 32; ++w) m[w] = 0;
    for (int g = 0; g < nsys; ++g) {
        const bool on = inner ? S[g].inner_active : (S[g].outer_active || S[g].zero_x);
        if (on) m[g >> 5] |= 1u << (g & 31);
    }
    bool same = P.valid != 0;
    for (int w = 0; w < MAXSYS / 32; ++w) same = same && m[w] == P.mask[w];
    if (!same) {
        auto on = [&](int g) { return ((m[g >> 5] >> (g & 31)) & 1u) != 0; };
        auto len = [&](int g) -> int64_t { return on(g) ? (int64_t)(P.ss1[g] - P.ss0[g]) : 0; };
        int64_t W = 0;
        for (int g = 0; g < nsys; ++g) W += len(g);
        for (int g = 0; g < nsys; ++g) { P.b0[g] = 0; P.b1[g] = 0; P.j[g] = -1; }
        P.nv = P.nseg = P.ng = 0;
        P.segv[0] = 0;
        bool ok = true;
        int gl = 0, gh = 0;
        int64_t cl = 0, ch = 0;  // active slices of the systems before gl, gh
        // block b takes the active slices [W b / nb, W (b + 1) / nb); a block
        // with none (fewer active slices than blocks) holds an empty range
        // of the active system at its position, for which it reduces a zero,
        // so that the blocks listed for a system are exactly those that
        // write its partials
        for (int b = 0; b < nb && ok && W > 0; ++b) {
            const int64_t lo = W * b / nb, hi = W * (b + 1) / nb;
            while (lo >= cl + len(gl)) { cl += len(gl); ++gl; }
            int last = gl;
            if (hi > lo) {
                while (hi - 1 >= ch + len(gh)) { ch += len(gh); ++gh; }
                last = gh;
            }
            int cnt = 0;
            for (int g = gl; g <= last; ++g) cnt += on(g) ? 1 : 0;
            if (cnt > MAXSYS_PB) { ok = false; break; }
            if (b == bid) {
                int64_t cg = cl;  // active slices before system g
                for (int g = gl; g <= last; ++g) {
                    if (!on(g)) continue;
                    P.j[g] = P.ng;
                    P.sys[P.ng] = g;
                    ++P.ng;
                    const int64_t v0 = lo > cg ? lo : cg;
                    const int64_t v1 = hi < cg + len(g) ? hi : cg + len(g);
                    if (v1 > v0) {
                        P.segs[P.nseg] = P.ss0[g] + (int)(v0 - cg);
                        P.segv[P.nseg + 1] = P.segv[P.nseg] + (int)(v1 - v0);
                        ++P.nseg;
                    }
                    cg += len(g);
                }
                P.nv = P.segv[P.nseg];
            }
            for (int g = gl; g <= last; ++g) {
                if (!on(g)) continue;
                if (P.b1[g] == 0) P.b0[g] = b;
                P.b1[g] = b + 1;
            }
        }
        P.mixed = 0;
        if (!ok) {  // the static partition: every system of the block's range
            const int g0 = blk_g0[bid];
            P.mixed = 1;
            P.nseg = 1;
            P.segs[0] = blk_s0[bid];
            P.segv[0] = 0;
            P.segv[1] = blk_s1[bid] - blk_s0[bid];
            P.nv = P.segv[1];
            P.ng = blk_ng[bid];
            for (int g = 0; g < nsys; ++g) {
                P.b0[g] = sys_b0[g];
                P.b1[g] = sys_b1[g];
                P.j[g] = (g >= g0 && g < g0 + P.ng) ? g - g0 : -1;
            }
            for (int j = 0; j < P.ng; ++j) P.sys[j] = g0 + j;
        }
        for (int w = 0; w < MAXSYS / 32; ++w) P.mask[w] = m[w];
        P.valid = 1;
    }
}

__device__ __noinline__ void warp_add(double v, double* to) {
    v = wsum(v);
    if ((threadIdx.x & 31) == 0) *to += v;
}

// The work items of P's segments (all threads of the block; item0[0] = -1 if there are too
// many).  Each run of 32 slices is cut by one warp: a slice starts an item where its stencil
// differs from its predecessor's, is not shared or holds an absolute column, and every
// fourth slice of a run.
template <int NT>
__device__ __noinline__ void make_items(Partition& P, int4* items, const int4* sinfo, const int32_t* slice_sys) {
    constexpr int KWARPS = NT / 32;
    __shared__ int s_cnt[KWARPS], s_base;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) s_base = 0;
    for (int k = 0; k < P.nseg; ++k) {
        const int s0 = P.segs[k], n = P.segv[k + 1] - P.segv[k];
        if (threadIdx.x == 0) P.item0[k] = s_base;
        for (int c0 = 0; c0 < n; c0 += 32 * KWARPS) {
            const int v = c0 + 32 * warp + lane;
            const bool in = v < n;
            const int4 si = in ? __ldg(sinfo + s0 + v) : make_int4(0, 0, -1, 0);
            const int zp = __shfl_up_sync(0xffffffffu, si.z, 1);
            const bool single = si.z < 0 || (si.w & SINFO_ABS);
            const bool sp = __shfl_up_sync(0xffffffffu, (int)single, 1) != 0;
            const bool start = lane == 0 || si.z != zp || single || sp;
            const unsigned runs = __ballot_sync(0xffffffffu, start);
            const int pos = lane - (31 - __clz(runs & (0xffffffffu >> (31 - lane))));
            const unsigned heads = __ballot_sync(0xffffffffu, in && (pos & 3) == 0);
            if (lane == 0) s_cnt[warp] = __popc(heads);
            __syncthreads();
            int at = s_base, tot = 0;
            for (int w = 0; w < KWARPS; ++w) {
                if (w < warp) at += s_cnt[w];
                tot += s_cnt[w];
            }
            at += __popc(heads & ((1u << lane) - 1u));
            if (in && (pos & 3) == 0 && at < ITEM_CAP) {
                // up to the next head, but not past the segment's end
                const unsigned later = lane == 31 ? 0u : heads >> (lane + 1);
                const int cnt = later ? __ffs(later) : min(32 - lane, n - v);
                items[at] = make_item(s0 + v, cnt, __ldg(slice_sys + s0), si);
            }
            __syncthreads();
            if (threadIdx.x == 0) s_base += tot;
            __syncthreads();
        }
    }
    if (threadIdx.x == 0) {
        P.item0[P.nseg] = s_base;
        if (s_base > ITEM_CAP || P.mixed) P.item0[0] = -1;
    }
    __syncthreads();
}

// Block partials -> global, barrier, totals of every system -> stot.  Layout
// part[(g * NQ + k) * nb + block]: the blocks of one system are a contiguous run,
// summed by one warp (lanes stride over blocks, then a fixed butterfly), so the order is
// fixed and the loads are independent.  The caller alternates between two partial sets:
// a block that has read one reduction's totals and runs ahead into the next one writes
// the other set, so it never overwrites a partial that a slower block is still reading.
template <class T, int NT>
__device__ __noinline__ bool block_reduce(bool fast, const double* s_dyn, const Partition& P, double* part, int nq,
                                          int nb, int nsys, uint32_t* bar, int32_t* status, double (*stot)[NQ]) {
    constexpr int KTHREADS = NT, KWARPS = NT / 32;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int ni = P.ng * nq;
    if (fast) {
        // a quarter of the warps' values per warp, then the four quarters
        __shared__ double s_quart[4 * RED_SLOTS * RED_Q][32];
        constexpr int QW = KWARPS / 4;
        static_assert(KWARPS % 4 == 0 && QW % 2 == 0, "a quarter's values are added in pairs");
        // warps that may hold rows: a segment of n slices is worked by at most 4 n warps
        const int wact = min(4 * P.nv, KWARPS);
#pragma unroll 1
        for (int t = warp; t < 4 * ni; t += KWARPS) {
            const T* src = reinterpret_cast<const T*>(s_dyn) + (t >> 2) * KTHREADS + (t & 3) * QW * 32 + lane;
            double s0 = 0.0, s1 = 0.0;
            if ((t & 3) * QW < wact) {
#pragma unroll
                for (int w = 0; w < QW; w += 2) {
                    s0 += (double)src[w * 32];
                    s1 += (double)src[w * 32 + 32];
                }
            }
            s_quart[t][lane] = s0 + s1;
        }
        __syncthreads();
        for (int i = warp; i < ni; i += KWARPS) {
            const double s = wsum((s_quart[4 * i][lane] + s_quart[4 * i + 1][lane]) +
                                  (s_quart[4 * i + 2][lane] + s_quart[4 * i + 3][lane]));
            if (lane == 0) __stcg(&part[((int64_t)P.sys[i / nq] * NQ + i % nq) * nb + blockIdx.x], s);
        }
    } else {
#pragma unroll 1
        for (int i = warp; i < ni; i += KWARPS) {
            const int j = i / nq, k = i - j * nq;
            const double s = wsum(lane < KWARPS ? s_dyn[(j * NQ + k) * KWARPS + lane] : 0.0);
            if (lane == 0) __stcg(&part[((int64_t)P.sys[j] * NQ + k) * nb + blockIdx.x], s);
        }
    }
    if (!grid_sync(bar, (unsigned)nb, status)) return false;
#pragma unroll 1
    for (int i = warp; i < nsys * nq; i += KWARPS) {
        const int g = i / nq, k = i - g * nq;
        const double* src = part + ((int64_t)g * NQ + k) * nb;
        const int b1 = P.b1[g];
        double sum = 0.0;
#pragma unroll 1
        for (int bb = P.b0[g] + lane; bb < b1; bb += 5 * 32) {
            double v[5];
#pragma unroll
            for (int u = 0; u < 5; ++u) v[u] = bb + 32 * u < b1 ? __ldcg(src + bb + 32 * u) : 0.0;
            sum += ((v[0] + v[1]) + (v[2] + v[3])) + v[4];
        }
        sum = wsum(sum);
        if (lane == 0) stot[g][k] = sum;
    }
    __syncthreads();
    return true;
}

// L2 prefetch of this block's rows of a row-indexed vector (elem bytes per row) by bulk
// copies of at most 64 KB, issued by the lanes of one warp.  Slices start on 128-byte
// boundaries, so every copy is 16-byte aligned with a size that is a multiple of 16, as
// the bulk copy requires.
__device__ __noinline__ void prefetch_rows(const Partition& P, const void* vec, int elem) {
    for (int k = threadIdx.x & 31; k < P.nseg; k += 32) {
        const char* p0 = static_cast<const char*>(vec) + (int64_t)P.segs[k] * SLICE * elem;
        uint64_t left = (uint64_t)(P.segv[k + 1] - P.segv[k]) * SLICE * elem;
#pragma unroll 1
        while (left > 0) {
            const uint32_t n = left > 65536u ? 65536u : (uint32_t)left;
            l2_prefetch(p0, n);
            p0 += n;
            left -= n;
        }
    }
}

// Descriptor of tile t of level l: its corner, its geometry's lattice on the level and, from
// poff on, on the next level
constexpr int TILE_CAP = 4;
struct TileMeta {
    int64_t off, poff;
    int g, x0, y0, nx, ny, sx, px, py, pnx, pny, psx, pad;
};
template <class TM>
__device__ __noinline__ TileMeta tile_meta(const MgDev<TM>& M, int l, int64_t t) {
    const MgTile tile = M.tiles[l][t];
    const MgLevGeom q = M.lg[l][tile.g], p = M.lg[l + 1][tile.g];
    return TileMeta{q.off, p.off, tile.g, tile.x0, tile.y0, q.nx, q.ny, q.sx, q.px, q.py, p.nx, p.ny, p.sx, 0};
}

template <class T, class TM, int NT>
__global__ void __launch_bounds__(NT, 1) k_bicgstab(KArgs<T, TM> a) {
    constexpr int KTHREADS = NT, KWARPS = NT / 32;
    constexpr bool LARGE = NT > NT64;  // the streaming form: 64 registers a thread, so the plain row loop only
    constexpr int TROWS = (32 + KWARPS - 1) / KWARPS;  // rows of a 32-row coarse tile per warp
    // |r_hat . r| below this fraction of ||r_hat|| ||r|| is rounding noise in T
    // (FP32 vectors of ~1e6 rows: ~6e-8 / sqrt(n) relative noise in a dot product)
    const double bd_tol = sizeof(T) == 8 ? 1e-14 : 1e-9;
    constexpr bool K32 = std::is_same_v<T, float>;   // FP32 Krylov iteration
    constexpr bool M32 = std::is_same_v<TM, float>;  // FP32 V-cycle
    constexpr bool fold = M32 && !LARGE;             // level 1 goes down straight from the fine residual

    constexpr int V = 16 / (int)sizeof(T);  // rows per thread of the streaming phases

    __shared__ double stot[MAXSYS][NQ];
    __shared__ SysState S[MAXSYS];
    extern __shared__ __align__(16) double s_dyn[];
    T* red = reinterpret_cast<T*>(s_dyn);
    double* sacc = s_dyn;
    // multigrid: a coarse tile and its halo, 36 x 36
    TM* s_tile = reinterpret_cast<TM*>(reinterpret_cast<char*>(s_dyn) + red_bytes<T, NT>());
    TM* s_tile2 = s_tile + 36 * 36;  // level 1, down: the tile's own b_1
    // shared stencils of the uniform slices in TM
    TM* s_uval = reinterpret_cast<TM*>(reinterpret_cast<char*>(s_tile) + KSMEM_TILE);
    int32_t* s_ucode = reinterpret_cast<int32_t*>(s_uval + UCAP);
    __shared__ int4 s_items[ITEM_CAP];
    __shared__ TileMeta s_tiles[MG_MAXLEV][TILE_CAP];
    __shared__ int s_changed;  // a system left its pass since the last partition
    __shared__ Partition P;    // this block's share of the work
    const int bid = blockIdx.x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned nb = gridDim.x;
    const int nsys = a.nsys;
    for (int g = threadIdx.x; g < nsys; g += KTHREADS) {
        P.ss0[g] = a.sys_s0[g];
        P.ss1[g] = a.sys_s1[g];
    }
    if (a.use_mg)
        for (int i = threadIdx.x; i < (a.mg.nlev - 1) * TILE_CAP; i += KTHREADS) {
            const int l = 1 + i / TILE_CAP, k = i % TILE_CAP;
            const int64_t t = bid + (int64_t)k * gridDim.x;
            if (t < a.mg.ntiles[l]) s_tiles[l][k] = tile_meta(a.mg, l, t);
        }
    for (int i = threadIdx.x; i < a.nust; i += KTHREADS) {
        s_uval[i] = a.uM[i];
        s_ucode[i] = a.ucode[i];
    }
    if (threadIdx.x == 0) P.valid = 0;
    int nv = 0, ng_blk = 0, seg0 = 0;
    bool one_seg = true, p_valid_r = false;
    // slice of virtual index v; sg (the segment of the previous call) only advances,
    // as each warp's v increases; a block of one segment needs no lookup
    auto vslice = [&](int v, int& sg) {
        if (one_seg) return seg0 + v;
        while (v >= P.segv[sg + 1]) ++sg;
        return P.segs[sg] + (v - P.segv[sg]);
    };
    // The slices of the systems still being solved (outer set: solving or to be
    // zeroed; inner set: inside a BiCGSTAB pass) are spread evenly over all blocks,
    // recomputed whenever that set changes, so that blocks whose systems have
    // finished take over the work of the others.  Every block computes the whole
    // partition from the same system states, so all blocks agree without
    // communicating.  A block holds one segment of slices per active system in its
    // range (finished systems in between are passed over) and reduces only for
    // those systems.  A partition in which some block would hold more than
    // MAXSYS_PB active systems is replaced by the launch's static one (one segment
    // of all slices, finished systems' rows skipped).
    auto repartition = [&](int inner) {
        if (nsys == 1 && p_valid_r) return;  // one system: the partition never changes
        p_valid_r = true;
        __syncthreads();  // every thread has read s_changed
        if (threadIdx.x == 0) {
            partition_update(P, S, nsys, inner, (int)nb, bid, a.blk_s0, a.blk_s1, a.blk_g0, a.blk_ng,
                             a.sys_b0, a.sys_b1);
            s_changed = 0;
        }
        __syncthreads();
        make_items<NT>(P, s_items, a.sinfo, a.slice_sys);
        nv = P.nv;
        ng_blk = P.ng;
        one_seg = P.nseg <= 1;
        seg0 = P.nseg >= 1 ? P.segs[0] : 0;
    };

    // Dot products.  Contributions are summed per thread over all its rows of one
    // system.  In a block of at most RED_SLOTS systems (fast) every thread then puts its
    // sums into shared memory and the block adds the NT values of each quantity in FP64,
    // about one warp-wide addition per warp, where a butterfly in every warp takes five
    // on an FP64 unit of two lanes per clock (h = 1/32 cylinder, two quantities: 5.1 ->
    // 2.0 us per phase).  A block of more systems reduces across each warp at every change
    // of system.  The order is fixed either way, so sums are deterministic.  T-valued
    // contributions are summed in T (qacck), FP64 ones beside a FP32 iteration in FP64
    // (qacc).
    double qacc[RED_Q];
    T qacck[RED_Q];
    int qj = -1, qg = -1;
    bool fast = false, dot_t = true;
    auto begin_dots = [&](int nq, bool in_t) {
        dot_t = in_t;
        qj = qg = -1;
#pragma unroll
        for (int k = 0; k < RED_Q; ++k) { qacc[k] = 0.0; qacck[k] = (T)0; }
        fast = in_t && !P.mixed && ng_blk <= RED_SLOTS;
        if (fast) {
            for (int i = 0; i < ng_blk * nq; ++i) red[i * KTHREADS + threadIdx.x] = (T)0;
        } else {
#pragma unroll 1
            for (int i = threadIdx.x; i < KWARPS * MAXSYS_PB * NQ; i += KTHREADS) sacc[i] = 0.0;
            __syncthreads();
        }
    };
    auto flush_acc = [&](int nq) {  // warp-uniform unless fast
        if (qj >= 0) {
            if (fast) {
#pragma unroll
                for (int k = 0; k < RED_Q; ++k)
                    if (k < nq) red[(qj * nq + k) * KTHREADS + threadIdx.x] = qacck[k];
            } else {
#pragma unroll
                for (int k = 0; k < RED_Q; ++k)
                    warp_add(!K32 || dot_t ? (double)qacck[k] : qacc[k], sacc + (qj * NQ + k) * KWARPS + warp);
            }
        }
        qj = -1;
        qg = -1;
    };
    // the rows that follow belong to system g (warp-uniform)
    auto enter = [&](int g, int nq) {
        if (g == qg) return;
        flush_acc(nq);
        qg = g;
        qj = P.j[g];
#pragma unroll
        for (int k = 0; k < RED_Q; ++k) { qacc[k] = 0.0; qacck[k] = (T)0; }
    };
    // add a row's contributions q[0..nq)
    auto acc = [&](int nq, const auto* q) {
        using Q = std::remove_cv_t<std::remove_pointer_t<decltype(q)>>;
        if constexpr (std::is_same_v<Q, T>) {
#pragma unroll
            for (int k = 0; k < RED_Q; ++k)
                if (k < nq) qacck[k] += q[k];
        } else {
#pragma unroll
            for (int k = 0; k < RED_Q; ++k)
                if (k < nq) qacc[k] += q[k];
        }
    };
    int pset = 0;  // partial set of the next reduction
    auto reduce = [&](int nq) -> bool {
        flush_acc(nq);
        __syncthreads();
        double* part = a.partial + (int64_t)pset * nsys * NQ * nb;
        pset ^= 1;
        return block_reduce<T, NT>(fast, s_dyn, P, part, nq, (int)nb, nsys, a.bar, a.status, stot);
    };
    // system of a slice (a launch of one system needs no lookup)
    auto sysof = [&](int sl) -> int { return nsys == 1 ? 0 : __ldg(a.slice_sys + sl); };
    // The streaming phases take V consecutive rows per thread with 16-byte accesses
    // (consecutive threads, consecutive rows), so one round trip to memory serves V
    // rows.  body(row0, g) for row0 a multiple of V in a slice of system g still in its
    // pass.  Threads of a warp may have rows or not (a segment's last rows), so a phase
    // with dot products first makes every thread register the segment's system
    // (begin(g), all threads together): a warp-wide flush of the per-lane sums then only
    // ever runs with the whole warp.  In the static partition (P.mixed) a segment may
    // span systems, so it is walked slice by slice.
    auto rows_of = [&](auto&& begin, auto&& body) {
#pragma unroll 1
        for (int k = 0; k < P.nseg; ++k) {
            const int n = P.segv[k + 1] - P.segv[k], step = P.mixed ? 1 : n;
#pragma unroll 1
            for (int v = 0; v < n; v += step) {
                const int64_t r0 = (int64_t)(P.segs[k] + v) * SLICE;
                const int g = sysof(P.segs[k] + v);
                if (!S[g].inner_active) continue;
                begin(g);
#pragma unroll 1
                for (int q = threadIdx.x; q < step * (SLICE / V); q += KTHREADS) body(r0 + (int64_t)V * q, g);
            }
        }
    };
    auto no_enter = [](int) {};
    // A phase's streamed inputs are prefetched into L2, so that they are on their way from
    // DRAM while its warps start; vector i of a phase is issued by warp i (one thread
    // issuing six vectors took 1.2 us, 4.2 us at 2.1M rows).  Skipped where the
    // iteration's vectors stay in L2 (a.prefetch).
    auto prefetch = [&](int i, const void* vec, int elem) {
        if (a.prefetch && warp == i) prefetch_rows(P, vec, elem);
    };
    // The fine operator applied to vec over this block's rows of the systems for which
    // on(g): epi(row, own, (A vec)_row, vec_row, pre(row)), pre's loads issued before
    // the gathers.  Entries in vec's type; diff: the differenced FP32 form; nq: dot products
    // that epi adds to (0: none).
    //
    // A block with enough slices is worked by items (make_items).  In an item of four
    // slices each entry of their shared stencil is read once for 128 rows and its four
    // gathers are independent.  Where a block has few slices, two or four lanes share a
    // row, so that all warps have work and a row's dependent trips shrink; FP64 keeps one
    // lane per row sooner, since the lanes' extra additions cost its narrow unit more.
    // own: the lane that holds the row; every lane calls epi, so that warp-wide
    // operations in it see the whole warp.
    auto fine = [&](const auto* vec, const auto* A, const auto* uA, auto diff, auto&& on, int nq, auto&& pre, auto&& epi) {
        using TA = std::remove_cv_t<std::remove_pointer_t<decltype(vec)>>;
        constexpr bool D = decltype(diff)::value;
        constexpr int ROW_U = sizeof(TA) == 8 ? (LARGE ? 5 : 7) : (LARGE ? 8 : 14);  // entries of a row in flight
        constexpr int LANES4 = sizeof(TA) == 8 ? KWARPS / 4 : KWARPS / 2, LANES2 = sizeof(TA) == 8 ? KWARPS / 2 : 2 * KWARPS;
        auto ld = [&](int j) -> TA { return ldv(vec + j); };
        auto rs = [&](int64_t row) -> TA {
            if constexpr (D) return (TA)__ldg(a.rs32 + row);
            else return (TA)0;
        };
        const bool listed = P.item0[0] >= 0;
        if (LARGE || P.nv > LANES2 || P.mixed) {
            const int i1 = listed ? P.item0[P.nseg] : P.nv;
            int gon = -1;  // system of the item before
            bool is_on = false;
            int sgk = 0;
#pragma unroll 1
            for (int i = warp; i < i1; i += KWARPS) {
                int4 it;
                if (listed) {
                    it = s_items[i];
                } else {
                    const int sl = vslice(i, sgk);
                    it = make_item(sl, 1, sysof(sl), __ldg(a.sinfo + sl));
                }
                const int c = it.y & 7, w0 = (it.y >> 3) & SINFO_WIDTH, g = it.y >> 20;
                if (g != gon) {
                    gon = g;
                    is_on = on(g);
                    if (nq && is_on) enter(g, nq);
                }
                if (!is_on) continue;
                // the warp's next item on its way to L2 (no register waits for it)
                if (listed && i + KWARPS < i1) {
                    const int4 nx = s_items[i + KWARPS];
                    const uint32_t n = (uint32_t)((nx.y >> 3) & SINFO_WIDTH) * SLICE;
                    if (nx.w < 0 && n && lane < 2) {
                        const int64_t e = ~((int64_t)nx.w << 32 | (uint32_t)nx.z);
                        if (lane == 0) l2_prefetch(a.col + e, n * (uint32_t)sizeof(int32_t));
                        else l2_prefetch(A + e, n * (uint32_t)sizeof(TA));
                    }
                }
                if (!LARGE && c == 4) {
                    const int64_t r0 = (int64_t)it.x * SLICE + lane;
                    TA sum[4], xi[4];
                    decltype(pre((int64_t)0)) pr[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        xi[j] = ldv(vec + r0 + 32 * j);
                        pr[j] = pre(r0 + 32 * j);
                        sum[j] = (TA)0;
                    }
                    // generic pointers: the copies in shared memory, or global memory
                    const bool in_smem = a.nust > 0 && std::is_same_v<TA, TM>;
                    const int32_t* uc = (in_smem ? s_ucode : a.ucode) + it.z;
                    const TA* ua = (in_smem ? reinterpret_cast<const TA*>(s_uval) : uA) + it.z;
                    const TA* v0 = vec + r0;
#pragma unroll 4
                    for (int e = 0; e < w0; ++e) {
                        const TA* pv = v0 + (uc[e] >> 1);
                        const TA av = ua[e];
#pragma unroll
                        for (int j = 0; j < 4; ++j) sum[j] += av * (D ? ldv(pv + 32 * j) - xi[j] : ldv(pv + 32 * j));
                    }
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        epi(r0 + 32 * j, true, D ? sum[j] + rs(r0 + 32 * j) * xi[j] : sum[j], xi[j], pr[j]);
                } else {
                    const int64_t at = (int64_t)it.w << 32 | (uint32_t)it.z;
#pragma unroll 1
                    for (int j = 0; j < c; ++j) {
                        const int64_t row = (int64_t)(it.x + j) * SLICE + lane;
                        const TA xi = ldv(vec + row);
                        const auto pr = pre(row);
                        const TA r = rs(row);
                        TA sum = sell_part<ROW_U, D, TA>(a.col, A, a.ucode, uA, at, w0, (int32_t)row, lane, 0, 1, xi, ld);
                        if (D) sum += r * xi;
                        epi(row, true, sum, xi, pr);
                    }
                }
            }
            return;
        }
#pragma unroll 1
        for (int k = 0; k < P.nseg; ++k) {
            const int s0 = P.segs[k], n = P.segv[k + 1] - P.segv[k];
            const int g = sysof(s0);
            if (!on(g)) continue;
            if (nq) enter(g, nq);
            const int lg = n > LANES4 ? 1 : 2, L = 1 << lg, rows = 32 >> lg;  // L lanes per row
            const int sub = lane >> (5 - lg), rl = lane & (rows - 1);
#pragma unroll 1
            for (int i = warp; i < n << lg; i += KWARPS) {
                const int sl = s0 + (i >> lg), rr = (i & (L - 1)) * rows + rl;
                const int4 si = __ldg(a.sinfo + sl);
                const int64_t row = (int64_t)sl * SLICE + rr;
                const TA xi = ldv(vec + row);
                const auto pr = pre(row);
                const TA r = rs(row);
                TA sum = sell_part<7, D, TA>(a.col, A, a.ucode, uA, entries_at(si), si.w & SINFO_WIDTH, (int32_t)row, rr, sub,
                                              L, xi, ld);
#pragma unroll 1
                for (int o = rows; o < 32; o <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
                if (D) sum += r * xi;
                epi(row, sub == 0, sum, xi, pr);
            }
        }
    };
    auto in_pass = [&](int g) { return S[g].inner_active != 0; };
    auto solving = [&](int g) { return S[g].outer_active != 0; };
    using Plain = std::integral_constant<bool, false>;
    using DiffK = std::integral_constant<bool, K32>;   // applications in T
    using DiffM = std::integral_constant<bool, M32>;   // applications in TM

    // One V-cycle z = M^{-1} v of the aggregation multigrid: a V(1,1)-cycle with
    // l1-Jacobi smoothing from zero (D = sign(a_ii) sum_j |a_ij|, which stays a
    // convergent smoother on boundary rows that are not diagonally dominant),
    // summed restriction, piecewise-constant prolongation and a scaled coarse
    // correction:
    //   fine, down:   f = w Df^{-1} v (written by the Krylov update that produces v),
    //                 fr = v - A f,  b_1 = sum of fr over the rows of each cell
    //   level l+1:    b_{l+1}(C) = sum over the children c of C of (b_l - A_l x_l)(c),
    //                 x_l = w D_l^{-1} b_l
    //   coarsest:     x_L = A_L^{-1} b_L (dense FP64 inverse of each geometry)
    //   level l, up:  y_l = x_l + w D_l^{-1} (b_l - A_l x_l),
    //                 x_l = w D_l^{-1} b_l + corr s_{l+1}(parent),  s = x_L or y_{l+1}
    //   fine, up:     f += corr s_1(agg),  z = f + w Df^{-1} (v - A f)
    // A coarse level is processed in 32 x th tiles of its cell lattice (th = 32 on
    // large levels, down to 2 on small ones so that every SM gets a share of the
    // FP64 stencil work), one CTA per tile: the smoothing iterate x_l of the tile and
    // a two-cell halo is formed once in shared memory, then each warp applies the 5 x 5
    // stencils of its lattice rows (coefficients read as one contiguous slice per warp; of
    // the outer ring only the offsets that the slice holds).  A tile is a few dependent trips to
    // memory and little work, so everything that does not depend on the staged iterate
    // (3 x 3 coefficients, right-hand side, step, the fine rows of level 1) is loaded
    // with it, and the tiles' descriptors are kept in shared memory for the launch.
    // Going down in FP32 (fold), level 1 forms b_1 from the fine residual itself; in FP64 the
    // halo's sums would cost the narrow unit more than the phase saves, and at the 1,024-thread
    // form's sizes more memory trips (64 cavities: 61 us against 13 + 38).  A tile's
    // residuals are summed over 2 x 2 children straight into b_{l+1}; going up, level 1 adds
    // corr y_1 to the fine rows of each cell directly (y_1 is not stored).  The smoothing
    // steps w D^{-1} are precomputed per omega.  Only rows of systems still in their
    // inner pass are touched on the fine level.
    const TM mcorr = (TM)a.mg.corr;
    auto tile_of = [&](int l, int k) -> TileMeta {
        if (k < TILE_CAP) return s_tiles[l][k];
        return tile_meta(a.mg, l, blockIdx.x + (int64_t)k * nb);
    };
    // sum of fr over a level-1 cell's rows, in ascending order
    auto cell_sum = [&](int64_t c) -> TM {
        const int4 r4 = __ldg(a.mg.crow4 + c);
        TM sum = (TM)0;
        if (r4.w >= -1) {
            TM f[4];
            f[0] = r4.x >= 0 ? ldv(a.mg.fr + r4.x) : (TM)0;
            f[1] = r4.y >= 0 ? ldv(a.mg.fr + r4.y) : (TM)0;
            f[2] = r4.z >= 0 ? ldv(a.mg.fr + r4.z) : (TM)0;
            f[3] = r4.w >= 0 ? ldv(a.mg.fr + r4.w) : (TM)0;
            sum = ((f[0] + f[1]) + f[2]) + f[3];
        } else {  // more than four rows
            const int64_t q1 = __ldg(a.mg.cptr + c + 1);
            for (int64_t q = __ldg(a.mg.cptr + c); q < q1; ++q) sum += ldv(a.mg.fr + __ldg(a.mg.crow + q));
        }
        return sum;
    };
    // one tile of level l: down (residual restricted to level l + 1) or up (sol: the
    // coarser level's solution)
    auto tile_pass = [&](int l, const TileMeta& m, bool down, const TM* sol) {
        const MgDev<TM>& M = a.mg;
        const TM* bl = M.b[l];
        const TM* wdl = M.wdinv[l];
        const int th = M.th[l];
        constexpr int NST = (36 * 36 + KTHREADS - 1) / KTHREADS;
        TM v[NST], bc[TROWS], wd[TROWS], co[TROWS][9];
        bool in[TROWS];
        uint32_t rg[TROWS];  // outer offsets that the cell's slice holds
#pragma unroll
        for (int k = 0; k < TROWS; ++k) {
            const int r = warp + k * KWARPS, x = m.x0 + lane, y = m.y0 + r;
            in[k] = r < th && x < m.nx && y < m.ny;
            rg[k] = 0;
            bc[k] = wd[k] = (TM)0;
            if (in[k]) {
                const int64_t c = m.off + (int64_t)y * m.sx + x;
                const TM* cp = M.coefs[l] + (c >> 5) * 800 + (c & 31);
                rg[k] = __ldg(M.ring[l] + (c >> 5));
#pragma unroll
                for (int o = 0; o < (LARGE ? 0 : 9); ++o) co[k][o] = ldm(cp + ((1 + o / 3) * 5 + 1 + o % 3) * 32);
                wd[k] = __ldg(wdl + c);
                if (!down || l > 1 || !fold) bc[k] = ldv(bl + c);
            }
        }
        const int nst = 36 * (th + 4);
#pragma unroll
        for (int h = 0; h < NST; ++h) {
            const int k = threadIdx.x + h * KTHREADS;
            v[h] = (TM)0;
            if (k < nst) {
                const int yy0 = k / 36, xx0 = k - 36 * yy0;
                int xx = m.x0 - 2 + xx0, yy = m.y0 - 2 + yy0;
                bool ok = true;
                if (m.px) { xx %= m.nx; if (xx < 0) xx += m.nx; } else ok = xx >= 0 && xx < m.nx;
                if (m.py) { yy %= m.ny; if (yy < 0) yy += m.ny; } else ok = ok && yy >= 0 && yy < m.ny;
                if (ok) {
                    const int64_t j = m.off + (int64_t)yy * m.sx + xx;
                    if (!down) {
                        v[h] = __ldg(wdl + j) * ldv(bl + j) +
                               mcorr * ldv(sol + m.poff + (int64_t)(yy >> 1) * m.psx + (xx >> 1));
                    } else if (l > 1 || !fold) {
                        v[h] = __ldg(wdl + j) * ldv(bl + j);
                    } else {
                        const TM b = cell_sum(j);
                        v[h] = __ldg(wdl + j) * b;
                        const int tx = xx0 - 2, ty = yy0 - 2;
                        if (tx >= 0 && tx < 32 && ty >= 0 && ty < th) {  // the tile's own cells
                            M.b[1][j] = b;
                            s_tile2[ty * 32 + tx] = b;
                        }
                    }
                }
            }
        }
        __syncthreads();  // the previous tile's reads of s_tile are done
#pragma unroll
        for (int h = 0; h < NST; ++h) {
            const int k = threadIdx.x + h * KTHREADS;
            if (k < nst) s_tile[k] = v[h];
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < TROWS; ++k) {
            const int r = warp + k * KWARPS;
            const uint32_t outer = __reduce_or_sync(0xffffffffu, rg[k]);
            if (in[k]) {
                const int x = m.x0 + lane, y = m.y0 + r;
                const int64_t c = m.off + (int64_t)y * m.sx + x;
                const TM* cp = M.coefs[l] + (c >> 5) * 800 + (c & 31);
                if constexpr (LARGE) {
#pragma unroll
                    for (int o = 0; o < 9; ++o) co[k][o] = ldm(cp + ((1 + o / 3) * 5 + 1 + o % 3) * 32);
                }
                if (fold && down && l == 1) bc[k] = s_tile2[r * 32 + lane];
                TM res = bc[k];
                if constexpr (M32) {
                    TM acc[3];  // one chain per stencil row
#pragma unroll
                    for (int dy = 0; dy < 3; ++dy) {
                        const TM* t = s_tile + (r + 1 + dy) * 36 + lane + 1;
                        acc[dy] = co[k][3 * dy] * t[0] + co[k][3 * dy + 1] * t[1] + co[k][3 * dy + 2] * t[2];
                    }
                    TM e[2] = {(TM)0, (TM)0};
#pragma unroll 1
                    for (uint32_t m2 = outer; m2;) {  // two offsets at a time
                        const int o0 = __ffs(m2) - 1;
                        m2 &= m2 - 1;
                        const int o1 = m2 ? __ffs(m2) - 1 : -1;
                        m2 &= m2 - 1;
                        const TM c0 = ldm(cp + o0 * 32), c1 = o1 >= 0 ? ldm(cp + o1 * 32) : (TM)0;
                        e[0] += c0 * s_tile[(r + o0 / 5) * 36 + lane + o0 % 5];
                        if (o1 >= 0) e[1] += c1 * s_tile[(r + o1 / 5) * 36 + lane + o1 % 5];
                    }
                    if (outer) {
                        acc[0] += e[0];
                        acc[2] += e[1];
                    }
                    res -= (acc[0] + acc[1]) + acc[2];
                } else {  // the narrow FP64 unit: no operation but the products
#pragma unroll
                    for (int o = 0; o < 9; ++o) res -= co[k][o] * s_tile[(r + 1 + o / 3) * 36 + lane + 1 + o % 3];
#pragma unroll 1
                    for (uint32_t m2 = outer; m2;) {  // four offsets at a time
                        int o[4];
                        TM q[4];
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            o[u] = m2 ? __ffs(m2) - 1 : -1;
                            m2 &= m2 - 1;
                        }
#pragma unroll
                        for (int u = 0; u < 4; ++u) q[u] = o[u] >= 0 ? ldm(cp + o[u] * 32) : (TM)0;
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            if (o[u] >= 0) res -= q[u] * s_tile[(r + o[u] / 5) * 36 + lane + o[u] % 5];
                    }
                }
                if (down) {
                    bc[k] = res;
                } else {
                    const TM ynew = s_tile[(r + 2) * 36 + lane + 2] + wd[k] * res;
                    if (l > 1) {
                        M.y[l][c] = ynew;
                    } else {  // fine prolongation f += corr y_1 over the cell's rows
                        const int4 r4 = __ldg(M.crow4 + c);
                        if (r4.w >= -1) {
                            TM f[4];
                            if (r4.x >= 0) f[0] = ldv(M.fx + r4.x);
                            if (r4.y >= 0) f[1] = ldv(M.fx + r4.y);
                            if (r4.z >= 0) f[2] = ldv(M.fx + r4.z);
                            if (r4.w >= 0) f[3] = ldv(M.fx + r4.w);
                            if (r4.x >= 0) M.fx[r4.x] = f[0] + mcorr * ynew;
                            if (r4.y >= 0) M.fx[r4.y] = f[1] + mcorr * ynew;
                            if (r4.z >= 0) M.fx[r4.z] = f[2] + mcorr * ynew;
                            if (r4.w >= 0) M.fx[r4.w] = f[3] + mcorr * ynew;
                        } else {
                            const int64_t q1 = __ldg(M.cptr + c + 1);
                            for (int64_t qq = __ldg(M.cptr + c); qq < q1; ++qq) {
                                const int32_t row = __ldg(M.crow + qq);
                                M.fx[row] = ldv(M.fx + row) + mcorr * ynew;
                            }
                        }
                    }
                }
            } else {
                bc[k] = (TM)0;
            }
        }
        if (!down) return;
        // residuals of the tile, summed over 2 x 2 children (s_tile2: own cells' b_1, read above)
        __syncthreads();
#pragma unroll
        for (int k = 0; k < TROWS; ++k)
            if (warp + k * KWARPS < th) s_tile[(warp + k * KWARPS) * 32 + lane] = bc[k];
        __syncthreads();
        if (threadIdx.x < th * 8) {  // 16 x th/2 cells of level l+1
            const int px = threadIdx.x & 15, py = threadIdx.x >> 4;
            const int X = (m.x0 >> 1) + px, Y = (m.y0 >> 1) + py;
            if (X < m.pnx && Y < m.pny) {
                const int k0 = (2 * py) * 32 + 2 * px;
                M.b[l + 1][m.poff + (int64_t)Y * m.psx + X] =
                    (s_tile[k0] + s_tile[k0 + 1]) + (s_tile[k0 + 32] + s_tile[k0 + 33]);
            }
        }
    };
    auto level_pass = [&](int l, bool down, const TM* sol) -> bool {
#pragma unroll 1
        for (int k = 0; blockIdx.x + (int64_t)k * nb < a.mg.ntiles[l]; ++k) {
            const TileMeta m = tile_of(l, k);
            if (S[m.g].inner_active) tile_pass(l, m, down, sol);  // else that geometry's solve is done
        }
        return grid_sync(a.bar, nb, a.status);
    };
    // z = M^{-1} v, given v and f = w Df^{-1} v on the rows of active systems
    auto vcycle = [&](const T* v, T* z) -> bool {
        const MgDev<TM>& M = a.mg;
        const int L = M.nlev;
        prefetch(0, v, sizeof(T));
        prefetch(1, M.fx, sizeof(TM));
        if constexpr (M32) prefetch(2, a.rs32, 4);
        fine((const TM*)M.fx, a.aM, a.uM, DiffM{}, in_pass, 0, [&](int64_t row) { return (TM)ldv(v + row); },
             [&](int64_t row, bool own, TM sum, TM, TM vr) {
                 if (own) M.fr[row] = vr - sum;
             });
        if (!grid_sync(a.bar, nb, a.status)) return false;
        if (!fold || L == 1) {  // level 1's downward pass does not form b_1
            for (int64_t c = (int64_t)blockIdx.x * KTHREADS + threadIdx.x; c < M.n[1]; c += (int64_t)nb * KTHREADS)
                M.b[1][c] = cell_sum(c);
            if (!grid_sync(a.bar, nb, a.status)) return false;
        }
        // levels 1 .. L - 1 down, the coarsest solve, levels L - 1 .. 1 up
#pragma unroll 1
        for (int step = 1; step < 2 * L; ++step) {
            if (step != L) {
                const bool down = step < L;
                const int l = down ? step : 2 * L - step;
                if (!level_pass(l, down, down || l + 1 == L ? M.x[L] : M.y[l + 1])) return false;
                continue;
            }
            // coarsest level: x_L = A_L^{-1} b_L with each geometry's dense FP64 inverse;
            // one warp per coarsest cell of any geometry (cells numbered densely per
            // geometry on this level, geometry found by bisection on the offsets), lanes
            // over the row, then a fixed-order warp sum
#pragma unroll 1
            for (int64_t c = (int64_t)blockIdx.x * KWARPS + warp; c < M.n[L]; c += (int64_t)nb * KWARPS) {
                int lo = 0, hi = M.ngeom - 1;
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (M.lg[L][mid].off <= c) lo = mid;
                    else hi = mid - 1;
                }
                const MgLevGeom q = M.lg[L][lo];
                const int64_t m = (int64_t)q.nx * q.ny;
                const int64_t i = c - q.off;
                if (i >= m || !S[lo].inner_active) continue;  // padding, or a finished geometry (warp-uniform)
                const TM* Ai = M.cinv + __ldg(M.cinv_off + lo) + i * m;
                const TM* bL = M.b[L] + q.off;
                TM sum = (TM)0;
                for (int64_t j = lane; j < m; j += 32) sum += __ldg(Ai + j) * ldv(bL + j);
                sum = wsum(sum);
                if (lane == 0) M.x[L][c] = sum;
            }
            if (!grid_sync(a.bar, nb, a.status)) return false;
        }
        // fine prolongation f += corr s_1(agg) when level 1 is the coarsest; otherwise
        // the level-1 pass above did it
        if (L == 1) {
            const TM* sol1 = M.x[1];
#pragma unroll 1
            for (int iv = warp, sg = 0; iv < nv; iv += KWARPS) {
                const int sl = vslice(iv, sg);
                if (!S[sysof(sl)].inner_active) continue;
                const int64_t rw = (int64_t)sl * 32 + lane;
                const int32_t cc = __ldg(M.agg + rw);
                if (cc >= 0) M.fx[rw] = ldv(M.fx + rw) + mcorr * ldv(sol1 + cc);
            }
            if (!grid_sync(a.bar, nb, a.status)) return false;
        }
        prefetch(0, v, sizeof(T));
        prefetch(1, M.fx, sizeof(TM));
        prefetch(2, M.fwdinv, sizeof(TM));
        if constexpr (M32) prefetch(3, a.rs32, 4);
        struct VW { TM v, w; };
        fine((const TM*)M.fx, a.aM, a.uM, DiffM{}, in_pass, 0,
             [&](int64_t row) { return VW{(TM)ldv(v + row), __ldg(M.fwdinv + row)}; },
             [&](int64_t row, bool own, TM sum, TM fi, VW p) {
                 if (own) z[row] = (T)(fi + p.w * (p.v - sum));
             });
        return grid_sync(a.bar, nb, a.status);
    };

    // Scalars of an iteration.  Thread g tests system g's convergence and breakdown
    // (square roots) while another warp's threads form the iteration's quotients, so the
    // two serial FP64 chains overlap; a CTA barrier that also votes on "any system still
    // active" ends the step.
    const int tg = threadIdx.x;                         // tests of system tg
    const int dg = (int)threadIdx.x - MAXSYS;           // quotient of system dg
    const int bg = ((int)threadIdx.x - MAXSYS) >> 1;    // beta's two quotients (lane pairs)
    if (tg < nsys) {
        SysState& st = S[tg];
        st.bnorm = -1.0; st.rnorm = 0; st.tol = 0; st.rho = st.alpha = st.omega = 1.0;
        st.beta = 0; st.rhat_norm = 0; st.relres = 0;
        st.outer_active = 1; st.inner_active = 0; st.s_conv = 0; st.zero_x = 0;
        st.pass_bad = 0; st.bad_passes = 0; st.r0_in = 0; st.pass_cap = a.max_pass;
        st.iters = 0; st.outer = 0; st.pass_iters = 0; st.status = 0;
        st.alpha_f = st.omega_f = 1.0f; st.beta_f = 0.0f;
    }
    if (threadIdx.x == 0) s_changed = 0;
    __syncthreads();

    bool alive = true;
    for (int outer = 0; alive; ++outer) {
        repartition(0);
        // ---- X: apply the correction of the previous pass
        if (outer > 0) {
#pragma unroll 1
            for (int iv = warp, sg = 0; iv < nv; iv += KWARPS) {
                const int sl = vslice(iv, sg);
                int g = sysof(sl);
                int64_t row = (int64_t)sl * 32 + lane;
                if (S[g].zero_x) a.x[row] = 0.0;
                else if (S[g].outer_active && !S[g].pass_bad) {
                    if constexpr (K32) {
                        const float2 d = ldv(reinterpret_cast<const float2*>(a.dx) + row);
                        a.x[row] = __ldcg(a.x + row) + ((double)d.x + (double)d.y);
                    } else {
                        a.x[row] = __ldcg(a.x + row) + ldv(a.dx + row);
                    }
                }
            }
            if (!grid_sync(a.bar, nb, a.status)) { alive = false; break; }
        }
        // ---- R: FP64 residual, inner initialisation
        begin_dots(3, !K32);
        fine((const double*)a.x, a.a64, a.u64, Plain{}, solving, 3, [&](int64_t row) { return __ldg(a.b + row); },
             [&](int64_t row, bool own, double sum, double, double bi) {
                 const double ri = bi - sum;
                 const T rt = (T)ri;
                 if (own) {
                     a.r[row] = rt;
                     a.rhat[row] = rt;
                     a.p[row] = (T)0;
                     a.v[row] = (T)0;
                     a.dx[row] = 0.0;  // also the pair (0, 0)
                 }
                 const double q[3] = {own ? ri * ri : 0.0, own ? bi * bi : 0.0, own ? (double)rt * (double)rt : 0.0};
                 acc(3, q);
             });
        if (!reduce(3)) { alive = false; break; }
        if (tg < nsys) {
            SysState& st = S[tg];
            if (st.outer_active) {
                if (st.bnorm < 0) st.bnorm = sqrt(stot[tg][1]);
                st.rnorm = sqrt(stot[tg][0]);
                st.zero_x = 0;
                st.inner_active = 0;
                if (st.bnorm == 0.0) {
                    st.relres = 0.0;
                    st.zero_x = 1;            // x = 0 solves A x = 0
                    st.outer_active = 0;
                } else {
                    st.relres = st.rnorm / st.bnorm;
                    if (!(st.relres == st.relres) || isinf(st.relres)) {
                        st.status = VIP_ERR_NONFINITE; st.outer_active = 0;
                    } else if (st.relres <= a.rtol) {
                        st.outer_active = 0;
                    } else if (st.iters >= a.max_iters || st.outer >= a.max_outer) {
                        st.status = VIP_ERR_NOT_CONVERGED; st.outer_active = 0;
                    } else if (st.outer > 0 && st.pass_iters == 0 && !st.pass_bad) {
                        st.status = VIP_ERR_BREAKDOWN; st.outer_active = 0;
                    } else if (st.bad_passes >= 3) {
                        st.status = VIP_ERR_NONFINITE; st.outer_active = 0;
                    } else {
                        st.inner_active = 1;
                        st.outer += 1;
                        double t_abs = 0.5 * a.rtol * st.bnorm;
                        st.tol = (sizeof(T) == 8) ? t_abs : fmax(a.inner_rtol * st.rnorm, t_abs);
                        st.rho = stot[tg][2];
                        st.rhat_norm = sqrt(st.rho);
                        st.r0_in = st.rhat_norm;
                        st.alpha = st.omega = 1.0;
                        st.alpha_f = st.omega_f = 1.0f;
                        st.beta = 0.0;  // p = v = 0: the first direction is r
                        st.beta_f = 0.0f;
                        st.bad_passes = st.pass_bad ? st.bad_passes + 1 : 0;
                        st.pass_cap = st.pass_bad ? max(st.pass_iters / 2, 20)
                                                  : min(2 * st.pass_cap, a.max_pass);
                        st.pass_bad = 0;
                        st.pass_iters = 0;
                    }
                }
            }
        }
        const bool any_zero = __syncthreads_or(tg < nsys && S[tg].zero_x) != 0;
        bool any_inner = __syncthreads_or(tg < nsys && S[tg].inner_active) != 0;
        if (!__syncthreads_or(tg < nsys && S[tg].outer_active)) {
            if (any_zero) {  // final zeroing pass
    #pragma unroll 1
            for (int iv = warp, sg = 0; iv < nv; iv += KWARPS) {
                    const int sl = vslice(iv, sg);
                    int g = sysof(sl);
                    if (S[g].zero_x) a.x[(int64_t)sl * 32 + lane] = 0.0;
                }
            }
            break;
        }

        // ---- inner BiCGSTAB pass
        bool entered = false;
        while (any_inner) {
            if (!entered || s_changed) repartition(1);  // s_changed: uniform, set before a CTA barrier
            entered = true;
            // Two half steps of the same shape, one copy of the code for both (the launch's
            // instructions are fetched anew in every phase):
            //   A: p = r + beta (p - omega v), phat = M^{-1} p;  B: v = A phat, rhat . v
            //   C: s = r - alpha v,            shat = M^{-1} s;  D: t = A shat, t . s, t . t, s . s
#pragma unroll 1
            for (int half = 0; half < 2; ++half) {
                T* const dir = half ? a.s : a.p;
                T* const hat = half ? a.shat : a.phat;
                T* const img = half ? a.t : a.v;
                const T* const dot = half ? a.s : a.rhat;
                const int nq = 2 + half;
                prefetch(0, a.r, sizeof(T));
                prefetch(1, a.v, sizeof(T));
                if (a.use_mg) prefetch(2, a.mg.fwdinv, sizeof(TM));
                if (!half) prefetch(3, a.p, sizeof(T));
                rows_of(no_enter, [&](int64_t r0, int g) {
                    const T c1 = half ? -sc<T>(S[g].alpha, S[g].alpha_f) : sc<T>(S[g].beta, S[g].beta_f);
                    const T om = sc<T>(S[g].omega, S[g].omega_f);
                    const Pack<T, V> rr = ldp<V>(a.r + r0);
                    Pack<T, V> vv = ldp<V>(a.v + r0);
                    Pack<TM, V> wd = {};
                    if (a.use_mg) wd = ldp<V>(a.mg.fwdinv + r0);
                    if (!half) {
                        const Pack<T, V> pp = ldp<V>(a.p + r0);
#pragma unroll
                        for (int u = 0; u < V; ++u) vv.v[u] = pp.v[u] - om * vv.v[u];
                    }
#pragma unroll
                    for (int u = 0; u < V; ++u) vv.v[u] = rr.v[u] + c1 * vv.v[u];
                    stp<V>(dir + r0, vv);
                    if (a.use_mg) {
#pragma unroll
                        for (int u = 0; u < V; ++u) wd.v[u] *= (TM)vv.v[u];
                        stp<V>(a.mg.fx + r0, wd);
                    }
                });
                if (!grid_sync(a.bar, nb, a.status)) { alive = false; break; }
                if (a.use_mg && !vcycle(dir, hat)) { alive = false; break; }
                begin_dots(nq, true);
                prefetch(0, hat, sizeof(T));
                prefetch(1, dot, sizeof(T));
                if constexpr (K32) prefetch(2, a.rs32, 4);
                fine((const T*)hat, a.aT, a.uT, DiffK{}, in_pass, nq, [&](int64_t row) { return ldv(dot + row); },
                     [&](int64_t row, bool own, T y, T, T x) {
                         if (own) img[row] = y;
                         const T q[3] = {own ? x * y : (T)0, own ? y * y : (T)0, own && half ? x * x : (T)0};
                         acc(nq, q);
                     });
                if (!reduce(nq)) { alive = false; break; }
                if (tg < nsys) {
                    SysState& st = S[tg];
                    const double d0 = stot[tg][0], d1 = stot[tg][1];
                    if (half) st.s_conv = 0;
                    if (st.inner_active && !half) {
                        if (!fin(d0) || !fin(d1)) {
                            st.inner_active = 0;
                            st.pass_bad = 1;
                            s_changed = 1;
                        } else if (!(fabs(d0) > bd_tol * st.rhat_norm * sqrt(d1))) {
                            st.inner_active = 0;  // restart from the current x
                            s_changed = 1;
                        }
                    } else if (st.inner_active) {
                        st.iters += 1;
                        st.pass_iters += 1;
                        const double ss = stot[tg][2];
                        if (!fin(d0) || !fin(d1) || !fin(ss)) {
                            st.s_conv = 1;  // stop the pass after E (omega = 0) and discard it
                            st.pass_bad = 1;
                        } else if (sqrt(ss) <= st.tol || d1 == 0.0) {
                            st.s_conv = 1;
                        }
                    }
                } else if (dg >= 0 && dg < nsys) {  // alpha = rho / (rhat . v); omega = (t . s) / (t . t)
                    SysState& st = S[dg];
                    const double q = (half ? stot[dg][0] : st.rho) / stot[dg][half];
                    if (half) {  // unused where s_conv is set
                        st.omega = q;
                        st.omega_f = (float)q;
                    } else {
                        st.alpha = q;
                        st.alpha_f = (float)q;
                    }
                }
                __syncthreads();
            }
            if (!alive) break;
            // E: d += alpha p + omega s; r = s - omega t; rhat.r, r.r
            begin_dots(2, true);
            prefetch(0, a.dx, 8);
            prefetch(1, a.phat, sizeof(T));
            prefetch(2, a.shat, sizeof(T));
            prefetch(3, a.s, sizeof(T));
            prefetch(4, a.t, sizeof(T));
            prefetch(5, a.rhat, sizeof(T));
            rows_of([&](int g) { enter(g, 2); }, [&](int64_t r0, int g) {
                const SysState& st = S[g];
                const T al = sc<T>(st.alpha, st.alpha_f);
                const T om = st.s_conv ? (T)0 : sc<T>(st.omega, st.omega_f);
                const Pack<T, V> ph = ldp<V>(a.phat + r0), sh = ldp<V>(a.shat + r0), ss = ldp<V>(a.s + r0),
                                 tt = ldp<V>(a.t + r0), rh = ldp<V>(a.rhat + r0);
                if constexpr (K32) {
                    float4* dx4 = reinterpret_cast<float4*>(a.dx + r0);  // rows r0, r0 + 1 | r0 + 2, r0 + 3
                    float4 d01 = dx4[0], d23 = dx4[1];
                    float2 d;
                    d = dd_axpy2(make_float2(d01.x, d01.y), al, ph.v[0], om, sh.v[0]); d01.x = d.x; d01.y = d.y;
                    d = dd_axpy2(make_float2(d01.z, d01.w), al, ph.v[1], om, sh.v[1]); d01.z = d.x; d01.w = d.y;
                    d = dd_axpy2(make_float2(d23.x, d23.y), al, ph.v[2], om, sh.v[2]); d23.x = d.x; d23.y = d.y;
                    d = dd_axpy2(make_float2(d23.z, d23.w), al, ph.v[3], om, sh.v[3]); d23.z = d.x; d23.w = d.y;
                    dx4[0] = d01;
                    dx4[1] = d23;
                } else {
                    Pack<double, V> d = ldp<V>(a.dx + r0);
#pragma unroll
                    for (int u = 0; u < V; ++u) d.v[u] = d.v[u] + al * ph.v[u] + om * sh.v[u];
                    stp<V>(a.dx + r0, d);
                }
                Pack<T, V> rn;
                T q0 = (T)0, q1 = (T)0;
#pragma unroll
                for (int u = 0; u < V; ++u) {
                    rn.v[u] = st.s_conv ? ss.v[u] : ss.v[u] - om * tt.v[u];
                    q0 += rh.v[u] * rn.v[u];
                    q1 += rn.v[u] * rn.v[u];
                }
                stp<V>(a.r + r0, rn);
                const T qq[3] = {q0, q1, (T)0};
                acc(2, qq);
            });
            if (!reduce(2)) { alive = false; break; }
            if (tg < nsys) {
                SysState& st = S[tg];
                if (st.inner_active) {
                    const double rho = stot[tg][0], rr = sqrt(stot[tg][1]);
                    if (!fin(rho) || !fin(rr) || rr > 1e8 * st.r0_in) {
                        st.inner_active = 0;  // diverging in precision T: discard the pass
                        st.pass_bad = 1;
                    } else if (st.s_conv || rr <= st.tol || st.omega == 0.0 || st.iters >= a.max_iters ||
                               st.pass_iters >= st.pass_cap) {
                        st.inner_active = 0;
                    } else if (!(fabs(rho) > bd_tol * st.rhat_norm * rr)) {
                        st.inner_active = 0;  // restart
                    }
                    if (!st.inner_active) s_changed = 1;
                }
            } else if (bg >= 0 && bg < nsys) {  // beta = (rho / rho_old) (alpha / omega), one quotient per lane
                SysState& st = S[bg];
                const bool second = threadIdx.x & 1;
                const double rho = stot[bg][0];
                const double q = (second ? st.alpha : rho) / (second ? st.omega : st.rho);
                const int left = 2 * nsys - (((int)threadIdx.x - MAXSYS) & ~31);  // lanes of this branch
                const unsigned lanes = left >= 32 ? 0xffffffffu : (1u << left) - 1u;
                const double beta = q * __shfl_xor_sync(lanes, q, 1);
                if (!second) {
                    st.beta = beta;
                    st.beta_f = (float)beta;
                    st.rho = rho;
                }
            }
            any_inner = __syncthreads_or(tg < nsys && S[tg].inner_active) != 0;
        }
        if (!alive) break;
    }
    if (bid == 0 && threadIdx.x < nsys) {
        SysState& st = S[threadIdx.x];
        a.out_iters[threadIdx.x] = st.iters;
        a.out_outer[threadIdx.x] = st.outer;
        a.out_relres[threadIdx.x] = st.relres;
        a.out_status[threadIdx.x] = st.status;
        if (st.status) set_status(a.status, st.status);
    }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
template <class T, class TM, int NT>
constexpr int dyn_bytes() {
    return red_bytes<T, NT>() + KSMEM_TILE + ust_bytes<TM>();
}

vip_status krylov_plan(vip_ctx* c, KrylovPlan& P, const Sell& A, const std::vector<int64_t>& row0,
                       const std::vector<int64_t>& rows) {
    const int nsys = (int)row0.size();
    if (nsys > MAXSYS) {
        c->err = "too many systems in one Krylov batch (limit 128)";
        return VIP_ERR_ARG;
    }
    // dot-product sums, the coarse tile and the shared stencils live in dynamic shared
    // memory (set here, outside any graph capture); as much L1 as possible for the vector
    // gathers: the smallest shared-memory configuration that holds the block
    {
        struct { const void* k; int nt, dyn; } kern[] = {
            {(const void*)k_bicgstab<double, double, NT64>, NT64, dyn_bytes<double, double, NT64>()},
            {(const void*)k_bicgstab<double, double, NT64_LARGE>, NT64_LARGE, dyn_bytes<double, double, NT64_LARGE>()},
            {(const void*)k_bicgstab<float, float, NT32>, NT32, dyn_bytes<float, float, NT32>()},
            {(const void*)k_bicgstab<double, float, NT64>, NT64, dyn_bytes<double, float, NT64>()},
            {(const void*)k_bicgstab<double, float, NT64_LARGE>, NT64_LARGE, dyn_bytes<double, float, NT64_LARGE>()}};
        for (const auto& k : kern) {
            VIP_CUDA(cudaFuncSetAttribute(k.k, cudaFuncAttributeMaxDynamicSharedMemorySize, k.dyn));
            VIP_CUDA(cudaFuncSetAttribute(k.k, cudaFuncAttributePreferredSharedMemoryCarveout,
                                          cudaSharedmemCarveoutMaxL1));
            int o = 0;
            VIP_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, k.k, k.nt, k.dyn));
            if (o < 1) { c->err = "the Krylov kernel does not fit on an SM"; return VIP_ERR_CUDA; }
        }
    }
    const int64_t nsl = A.nslices;
    std::vector<int32_t> slice_sys(nsl, -1);
    for (int g = 0; g < nsys; ++g) {
        if (row0[g] % SLICE || rows[g] % SLICE) { c->err = "unaligned system"; return VIP_ERR_ARG; }
        for (int64_t s = row0[g] / SLICE; s < (row0[g] + rows[g]) / SLICE; ++s) slice_sys[s] = g;
    }
    for (int64_t s = 0; s < nsl; ++s)
        if (slice_sys[s] < 0) { c->err = "slice without system"; return VIP_ERR_ARG; }
    // contiguous slice chunks, one per block (one per SM); a block may touch MAXSYS_PB systems
    const int nb = (int)std::min<int64_t>(std::max(1, c->num_sms), nsl);
    std::vector<int32_t> bs0(nb), bs1(nb), bg0(nb), bng(nb);
    std::vector<int32_t> sb0(nsys, 1 << 30), sb1(nsys, -1);
    for (int b = 0; b < nb; ++b) {
        bs0[b] = (int32_t)(nsl * b / nb);
        bs1[b] = (int32_t)(nsl * (b + 1) / nb);
        int ga = slice_sys[bs0[b]], gb = slice_sys[bs1[b] - 1];
        bg0[b] = ga;
        bng[b] = gb - ga + 1;
        if (bng[b] > MAXSYS_PB) { c->err = "a block spans too many systems"; return VIP_ERR_ARG; }
        for (int g = ga; g <= gb; ++g) {
            sb0[g] = std::min(sb0[g], b);
            sb1[g] = std::max(sb1[g], b + 1);
        }
    }
    P.nblocks = nb;
    P.nsys = nsys;
    P.nslices = nsl;
    VIP_CUDA(dalloc(c, &P.slice_sys, nsl));
    VIP_CUDA(dalloc(c, &P.blk_s0, nb)); VIP_CUDA(dalloc(c, &P.blk_s1, nb));
    VIP_CUDA(dalloc(c, &P.blk_g0, nb)); VIP_CUDA(dalloc(c, &P.blk_ng, nb));
    VIP_CUDA(dalloc(c, &P.sys_b0, nsys)); VIP_CUDA(dalloc(c, &P.sys_b1, nsys));
    VIP_CUDA(dalloc(c, &P.sys_s0, nsys)); VIP_CUDA(dalloc(c, &P.sys_s1, nsys));
    VIP_CUDA(dalloc(c, &P.partial, (size_t)2 * nb * nsys * NQ));
    VIP_CUDA(cudaMemsetAsync(P.partial, 0, (size_t)2 * nb * nsys * NQ * sizeof(double), c->stream));
    VIP_CUDA(dalloc(c, &P.bar, 2));
    VIP_CUDA(dalloc(c, &P.out_iters, nsys)); VIP_CUDA(dalloc(c, &P.out_outer, nsys));
    VIP_CUDA(dalloc(c, &P.out_relres, nsys)); VIP_CUDA(dalloc(c, &P.out_status, nsys));
    cudaStream_t st = c->stream;
    VIP_CUDA(cudaMemcpyAsync(P.slice_sys, slice_sys.data(), nsl * 4, cudaMemcpyHostToDevice, st));
    VIP_CUDA(cudaMemcpyAsync(P.blk_s0, bs0.data(), nb * 4, cudaMemcpyHostToDevice, st));
    VIP_CUDA(cudaMemcpyAsync(P.blk_s1, bs1.data(), nb * 4, cudaMemcpyHostToDevice, st));
    VIP_CUDA(cudaMemcpyAsync(P.blk_g0, bg0.data(), nb * 4, cudaMemcpyHostToDevice, st));
    VIP_CUDA(cudaMemcpyAsync(P.blk_ng, bng.data(), nb * 4, cudaMemcpyHostToDevice, st));
    VIP_CUDA(cudaMemcpyAsync(P.sys_b0, sb0.data(), nsys * 4, cudaMemcpyHostToDevice, st));
    VIP_CUDA(cudaMemcpyAsync(P.sys_b1, sb1.data(), nsys * 4, cudaMemcpyHostToDevice, st));
    {
        std::vector<int32_t> ss0(nsys), ss1(nsys);
        for (int g = 0; g < nsys; ++g) {
            ss0[g] = (int32_t)(row0[g] / SLICE);
            ss1[g] = (int32_t)((row0[g] + rows[g]) / SLICE);
        }
        VIP_CUDA(cudaMemcpyAsync(P.sys_s0, ss0.data(), nsys * 4, cudaMemcpyHostToDevice, st));
        VIP_CUDA(cudaMemcpyAsync(P.sys_s1, ss1.data(), nsys * 4, cudaMemcpyHostToDevice, st));
        VIP_CUDA(cudaStreamSynchronize(st));
    }
    VIP_CUDA(cudaStreamSynchronize(st));
    return VIP_OK;
}

// the array of precision T: the FP64 one or its FP32 copy
template <class T>
static const T* pick(const double* d, const float* f) {
    if constexpr (std::is_same_v<T, double>) return d;
    else return f;
}

template <class T>
static MgDev<T> mg_view(const Multigrid& M) {
    MgDev<T> d;
    memset(&d, 0, sizeof(d));
    d.nlev = M.nlev;
    d.ngeom = M.ngeom;
    d.agg = M.agg; d.cptr = M.cptr; d.crow = M.crow; d.crow4 = M.crow4;
    d.fwdinv = pick<T>(M.fwdinv, M.fwdinv32);
    d.fr = (T*)M.fr; d.fx = (T*)M.fx;
    for (int l = 1; l <= M.nlev; ++l) {
        const MgLevel& v = M.lev[l];
        d.n[l] = v.n;
        d.ntiles[l] = v.ntiles;
        d.lg[l] = v.lg;
        d.tiles[l] = v.tiles;
        d.coefs[l] = pick<T>(v.coefs, v.coefs32);
        d.ring[l] = v.ring;
        d.th[l] = v.th;
        d.wdinv[l] = pick<T>(v.wdinv, v.wdinv32);
        d.x[l] = (T*)v.x; d.b[l] = (T*)v.b; d.y[l] = (T*)v.y;
    }
    d.corr = M.corr;
    d.cinv = pick<T>(M.cinv, M.cinv32);
    d.cinv_off = M.cinv_off;
    return d;
}

template <class T, class TM, int NT>
static vip_status launch(vip_ctx* c, const KrylovPlan& P, const Sell& A, const double* b, double* x,
                         double rtol, int32_t max_iters, double inner_rtol, const Multigrid* mg) {
    KrylovWork& W = sizeof(T) == 8 ? c->work64 : c->work32;
    if (W.n < A.nrows || c->work64.n < A.nrows) { c->err = "Krylov workspace too small"; return VIP_ERR_ARG; }
    if ((sizeof(T) == 4 || sizeof(TM) == 4) && (!A.v32 || !A.rs32)) {
        c->err = "operator has no FP32 copy";
        return VIP_ERR_ARG;
    }
    KArgs<T, TM> a;
    a.sinfo = A.sinfo; a.col = A.col; a.a64 = A.v64;
    a.aT = pick<T>(A.v64, A.v32);
    a.aM = pick<TM>(A.v64, A.v32);
    a.ucode = A.ucode; a.u64 = A.uv64;
    a.uT = pick<T>(A.uv64, A.uv32);
    a.uM = pick<TM>(A.uv64, A.uv32);
    a.rs32 = A.rs32;
    a.nust = A.nuentries <= UCAP ? (int)A.nuentries : 0;
    a.slice_sys = P.slice_sys; a.blk_s0 = P.blk_s0; a.blk_s1 = P.blk_s1; a.blk_g0 = P.blk_g0;
    a.blk_ng = P.blk_ng;
    a.sys_b0 = P.sys_b0; a.sys_b1 = P.sys_b1; a.partial = P.partial; a.bar = P.bar;
    a.sys_s0 = P.sys_s0; a.sys_s1 = P.sys_s1;
    a.nsys = P.nsys; a.b = b; a.x = x;
    a.r = (T*)W.r; a.rhat = (T*)W.rhat; a.p = (T*)W.p; a.v = (T*)W.v; a.s = (T*)W.s;
    a.t = (T*)W.t;
    a.dx = (double*)c->work64.dx;  // the correction is accumulated in FP64 in every form
    a.rtol = rtol; a.inner_rtol = inner_rtol; a.max_iters = max_iters;
    // FP32 passes are re-anchored on the FP64 residual at least every 4000 iterations
    a.max_outer = 1000;
    a.max_pass = sizeof(T) == 8 ? max_iters : 4000;
    a.out_iters = P.out_iters; a.out_outer = P.out_outer; a.out_relres = P.out_relres;
    a.out_status = P.out_status; a.status = c->d_status;
    a.use_mg = (mg && mg->built) ? 1 : 0;
    if (a.use_mg) {
        a.mg = mg_view<TM>(*mg);
        a.phat = (T*)c->phat;
        a.shat = (T*)c->shat;
    } else {
        memset(&a.mg, 0, sizeof(a.mg));
        a.phat = a.p;
        a.shat = a.s;
    }
    // about 11 vectors of T, the operator's scalings and (MG) the coarse levels per row;
    // prefetches pay once that outgrows the 129 MB L2
    a.prefetch = A.nrows * (int64_t)(16 * sizeof(T)) > (int64_t)96 << 20;
    VIP_CUDA(cudaMemsetAsync(P.bar, 0, 2 * sizeof(uint32_t), c->stream));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(P.nblocks);
    cfg.blockDim = dim3(NT);
    cfg.dynamicSmemBytes = dyn_bytes<T, TM, NT>() - (a.nust ? 0 : ust_bytes<TM>());
    cfg.stream = c->stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    VIP_CUDA(cudaLaunchKernelEx(&cfg, k_bicgstab<T, TM, NT>, a));
    return VIP_OK;
}

vip_status krylov_solve(vip_ctx* c, const KrylovPlan& P, const Sell& A, const double* b, double* x,
                        int precision, double rtol, int32_t max_iters, double inner_rtol,
                        const Multigrid* mg) {
    const bool use_mg = mg && mg->built;
    const bool large = use_mg && A.nstored_other >= LARGE_STREAM;
    if (precision == VIP_PREC_MIXED)
        return launch<float, float, NT32>(c, P, A, b, x, rtol, max_iters, inner_rtol, mg);
    if (precision == VIP_PREC_MG32 && use_mg)
        return large ? launch<double, float, NT64_LARGE>(c, P, A, b, x, rtol, max_iters, inner_rtol, mg)
                     : launch<double, float, NT64>(c, P, A, b, x, rtol, max_iters, inner_rtol, mg);
    return large ? launch<double, double, NT64_LARGE>(c, P, A, b, x, rtol, max_iters, inner_rtol, mg)
                 : launch<double, double, NT64>(c, P, A, b, x, rtol, max_iters, inner_rtol, mg);
}

}  // namespace vip
