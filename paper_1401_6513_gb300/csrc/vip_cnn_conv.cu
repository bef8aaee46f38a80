// 3x3 convolution of the warm-start network as an implicit GEMM on the 5th-generation
// tensor cores (tcgen05, kind::f16: BF16 x BF16 -> FP32 accumulators in TMEM).
//
// A tile is 128 consecutive pixels of one lattice row.  A CTA walks down a strip of 128 columns
// (a contiguous range of the tiles in strip order), so that of the three input rows of a tile
// two are already there: rows live in a ring in shared memory, channel-chunk planar --
// slot[row][c][col] holds channels 8c..8c+7 (16 bytes) of one of 130 pixels.  In that layout the
// 8-pixel x 8-channel core matrices of the MMA operand A are 128 contiguous bytes, so every one
// of the nine taps is the same operand seen from a shifted start address -- no im2col copy.  The
// weights sit in shared memory for the whole launch in the same core-matrix layout
// ([tap][chunk][cout][8 ci]).  One thread issues 9 * Cin/16 MMAs (K = 16 each) and commits them
// to an mbarrier; the four warps then read their 32 TMEM lanes with tcgen05.ld and run the
// epilogue.
//
// Pipeline: a ring of RING rows and two TMEM accumulators.  Rows are fetched with cp.async
// (16-byte copies, neighbouring threads the chunks of one pixel; zero-filled outside the image)
// up to three rows ahead.  In iteration k the CTA waits for the MMAs of tile k, issues those of
// tile k+1, starts the copies of the rows that fit into what tile k has released, and then runs
// tile k's epilogue.  Every mbarrier wait is bounded (2 s, then VIP_ERR_TIMEOUT); TMEM is always
// freed.
//
// A layer of 32 channels moves 67 MB at 513 x 1025 (10 us) and its MMAs read 4 KB of A each from
// shared memory (9 us).  It takes 33 us, bound by the instructions and waits of 12 warps per
// SM (35 to 41 with the channel counts as run-time numbers; 98 when every tile fetched its three
// rows with copies that touched one chunk of 32 pixels at a time, wrote 16 bytes at a time and
// read the ReLU mask element by element).
#include <algorithm>
#include <cstdio>

#include "vip_cnn.cuh"

namespace vip {

constexpr int PLANE_COLS = CNN_TILE + 2;               // 130
constexpr int PLANE_BYTES = PLANE_COLS * 16;           // 2080: one row of one chunk
constexpr int MAX_CHUNKS = CNN_CH / 8;                 // 4
constexpr int SLOT_BYTES = MAX_CHUNKS * PLANE_BYTES;   // 8320: one row
constexpr int RING = 6;   // rows: a tile's three and, where the next tile starts a new strip, its three
constexpr int SMEM_W = 9 * MAX_CHUNKS * CNN_CH * 16;   // 18432
// The ring, the weights, the bias, two mbarriers and the TMEM address word: three CTAs (3 x 64
// TMEM columns) per SM.
constexpr int SMEM_CONV = RING * SLOT_BYTES + SMEM_W + CNN_CH * 4 + 64;
constexpr int CONV_CTAS_PER_SM = 3;

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

// Shared-memory matrix descriptor, no swizzle, K-major operand: start address,
// leading-dimension (K direction) and stride-dimension (M/N direction) byte
// offsets between 8x16-byte core matrices, all >> 4, and the descriptor version 1.
__device__ __forceinline__ uint64_t umma_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1u << 46;
    return d;
}

// Instruction descriptor of kind::f16: FP32 accumulator (bits 4-5 = 1), BF16 A and
// B (bits 7-9 = 1, 10-12 = 1), both K-major, N/8 at bit 17, M/16 at bit 24.
__host__ __device__ constexpr uint32_t umma_idesc(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) |
           ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ uint64_t gtime() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, int count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait for the phase with the given parity; false after 2 s.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity) {
    if (mbar_try_wait(bar, parity)) return true;
    uint64_t t0 = gtime();
    while (!mbar_try_wait(bar, parity)) {
        if (gtime() - t0 > 2000000000ull) return false;
    }
    return true;
}

__device__ __forceinline__ void umma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc,
                                          uint32_t idesc, uint32_t accum) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accum));
}

__device__ __forceinline__ void umma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                 ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ void tc_fence_before() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

__device__ __forceinline__ void tmem_ld_x32(uint32_t taddr, float* v) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
          "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]),
          "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void tmem_ld_x16(uint32_t taddr, float* v) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// 16-byte asynchronous copy global -> shared; src_bytes 0 writes zeros (the source
// address is then not read, but is still a valid one).
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, uint32_t src_bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(src_bytes)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_but_last() {
    asm volatile("cp.async.wait_group 1;" ::: "memory");
}

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
    __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<uint32_t*>(&h);
}

// A walk over tiles in strip order: image by image, 128-column strip by strip, row by row.
struct Walk {
    const CnnImage* img;
    int nimg, im, tpr;   // tpr: strips of the image
    CnnImage I;
    int strip, y;
    __device__ __forceinline__ void seek(const CnnImage* images, int n, int64_t tile) {
        img = images;
        nimg = n;
        im = 0;
        while (im + 1 < nimg && img[im + 1].tile0 <= tile) ++im;
        I = img[im];
        tpr = (I.W + CNN_TILE - 1) / CNN_TILE;
        const int64_t t = tile - I.tile0;
        strip = (int)(t / I.H);
        y = (int)(t - (int64_t)strip * I.H);
    }
    // To the next tile; true if it starts a new strip (nothing of its rows is there yet).
    __device__ __forceinline__ bool next() {
        if (++y < I.H) return false;
        y = 0;
        if (++strip == tpr) {
            strip = 0;
            if (im + 1 < nimg) {
                I = img[++im];
                tpr = (I.W + CNN_TILE - 1) / CNN_TILE;
            }
        }
        return true;
    }
};

// The rows that a range of tiles needs, in order: three for the first tile of a strip, one for
// each further tile.  Row number n of this sequence lives in ring slot n % RING.
struct RowStream {
    Walk w;              // the tile whose rows come next
    int64_t tiles;       // tiles left
    int pend;            // rows left to fetch for it (the last is y + 1)
    int count;           // rows fetched
    int slot;            // count % RING
    __device__ __forceinline__ void init(const CnnImage* img, int nimg, int64_t t0, int64_t t1) {
        tiles = t1 - t0;
        if (tiles > 0) w.seek(img, nimg, t0);
        pend = 3;
        count = 0;
        slot = 0;
    }
    // Start the copies of the next row; with mirror, rows in the ring's first two slots are also
    // written behind its end, so that three rows from any slot on lie in a line.
    template <int CIN, bool MIRROR>
    __device__ __forceinline__ void fetch(const __nv_bfloat16* x, uint32_t ring, int tid) {
        constexpr int NCH = CIN / 8, PIX = 128 / NCH;   // chunks of a pixel; pixels per pass of 128 threads
        const int yy = w.y + 2 - pend;
        const bool row_in = yy >= 0 && yy < w.I.H;
        const int c = tid % NCH, col0 = tid / NCH, xx = w.strip * CNN_TILE - 1 + col0;
        const __nv_bfloat16* src = x + (w.I.off + (int64_t)(row_in ? yy : 0) * w.I.W) * CIN;
        const uint32_t d = ring + slot * SLOT_BYTES + c * PLANE_BYTES + col0 * 16;
#pragma unroll
        for (int j = 0; j < (PLANE_COLS + PIX - 1) / PIX; ++j) {
            if (j * PIX + PIX > PLANE_COLS && j * PIX + col0 >= PLANE_COLS) break;
            const int xj = xx + j * PIX;
            const bool in = row_in && xj >= 0 && xj < w.I.W;
            const __nv_bfloat16* q = in ? src + (int64_t)xj * CIN + c * 8 : x;
            cp_async16(d + j * PIX * 16, q, in ? 16u : 0u);
            if (MIRROR && slot < 2) cp_async16(d + RING * SLOT_BYTES + j * PIX * 16, q, in ? 16u : 0u);
        }
        slot = slot == RING - 1 ? 0 : slot + 1;
        ++count;
        if (--pend == 0) {
            --tiles;
            pend = tiles > 0 && w.next() ? 3 : 1;
        }
    }
};

// The 9 * Cin/16 MMAs of one tile whose first row lies in slot `slot`.  Descriptors differ in
// their start address only (bits 0 to 13, in units of 16 bytes).
template <int CIN, int COUT>
__device__ __forceinline__ void conv_mma(uint32_t ring, int slot, uint32_t w_base, uint32_t tmem_d) {
    constexpr int NCH = CIN / 8;
    constexpr uint32_t idesc = umma_idesc(CNN_TILE, COUT);
    const uint64_t bd = umma_desc(w_base, COUT * 16, 128);
#pragma unroll
    for (int dy = 0; dy < 3; ++dy) {
        const uint64_t ad = umma_desc(ring + slot * SLOT_BYTES, PLANE_BYTES, 128);
        slot = slot == RING - 1 ? 0 : slot + 1;
#pragma unroll
        for (int dx = 0; dx < 3; ++dx)
#pragma unroll
            for (int kc = 0; kc < NCH / 2; ++kc)
                umma_bf16(tmem_d, ad + (2 * kc * PLANE_BYTES + dx * 16) / 16,
                          bd + ((dy * 3 + dx) * NCH + 2 * kc) * COUT, idesc, dy + dx + kc > 0 ? 1u : 0u);
    }
}

__device__ __forceinline__ void st_global_32(void* p, const uint32_t* v) {
    asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "r"(v[0]), "r"(v[1]), "r"(v[2]),
                 "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
                 : "memory");
}

template <int CIN, int COUT, int EPI>
__global__ void __launch_bounds__(128) k_conv_tc(CnnConvArgs a) {
    extern __shared__ __align__(1024) uint8_t smem[];
    uint8_t* s_w = smem + RING * SLOT_BYTES;
    float* s_bias = reinterpret_cast<float*>(s_w + SMEM_W);
    uint64_t* s_bar = reinterpret_cast<uint64_t*>(s_w + SMEM_W + CNN_CH * 4);  // [2]
    uint32_t* s_tmem = reinterpret_cast<uint32_t*>(s_bar + 2);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int ncol = 64;  // TMEM columns: two accumulators of 32 (>= cout) columns

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(s_tmem)), "r"(ncol));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        mbar_init(s_bar, 1);
        mbar_init(s_bar + 1, 1);
    }
    // this CTA's tiles, a contiguous range
    const int64_t t0 = a.ntiles * blockIdx.x / gridDim.x, t1 = a.ntiles * (blockIdx.x + 1) / gridDim.x;
    const int64_t nt = t1 - t0;
    const uint32_t ring = smem_u32(smem);
    RowStream rows;
    rows.init(a.img, a.nimg, t0, t1);
    int c_prev = 0;  // rows fetched before the latest commit group
    for (int h = 0; h < 2; ++h) {
        c_prev = rows.count;
        while (rows.tiles > 0 && rows.count < 3 * (h + 1)) rows.fetch<CIN, false>(a.x, ring, tid);
        cp_async_commit();
    }
    // weights, already in [tap][chunk][cout][8] order: one 16-byte copy per thread step
    for (int i = tid; i < 9 * CIN / 8 * COUT; i += 128)
        reinterpret_cast<uint4*>(s_w)[i] = reinterpret_cast<const uint4*>(a.wpack)[i];
    if (tid < COUT) s_bias[tid] = a.bias ? a.bias[tid] : 0.0f;
    cp_async_wait_but_last();  // the first tile's rows
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *s_tmem;
    const uint32_t w_base = smem_u32(s_w);
    uint32_t phase = 0u;  // bit b: parity of accumulator b's next completion
    int issued = 0;       // bit b: a committed MMA group on accumulator b not yet waited for
    int row = 0, slot = 0;  // first row (number in the sequence) of the tile whose MMAs come next, its slot
    Walk t;               // tile k
    if (nt > 0) {
        t.seek(a.img, a.nimg, t0);
        if (tid == 0) {
            conv_mma<CIN, COUT>(ring, 0, w_base, tmem);
            umma_commit(s_bar);
        }
        issued = 1;
    }

    for (int64_t k = 0; k < nt; ++k) {
        const int b = (int)(k & 1);
        Walk tn = t;
        const int step = tn.next() ? 3 : 1;
        row += step;  // tile k + 1
        slot = slot + step >= RING ? slot + step - RING : slot + step;
        const int x = t.strip * CNN_TILE + warp * 32 + lane;
        const bool in = x < t.I.W;
        const int64_t cell = t.I.off + (int64_t)t.y * t.I.W + x;
        uint4 m[COUT / 8];  // ReLU mask of tile k, on its way while the MMAs finish
        if (EPI == EPI_MASK_BF16 && in) {
            const uint4* src = reinterpret_cast<const uint4*>(a.mask + cell * COUT);
#pragma unroll
            for (int q = 0; q < COUT / 8; ++q) m[q] = __ldg(src + q);
        }
        // the MMAs of tile k
        const bool ok = mbar_wait_bounded(s_bar + b, (phase >> b) & 1u);
        if (ok) {
            phase ^= 1u << b;
            issued &= ~(1 << b);
        } else {  // still in flight: the cleanup below waits for it again
            set_status(a.status, VIP_ERR_TIMEOUT);
        }
        // the rows of tile k + 1
        if (row + 3 <= c_prev) cp_async_wait_but_last();
        else cp_async_wait_all();
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        tc_fence_before();
        // (also: every warp has read accumulator 1 - b of tile k - 1)
        const int failed = __syncthreads_or(!ok);
        tc_fence_after();
        if (failed) break;
        if (k + 1 < nt) {
            if (tid == 0) {
                conv_mma<CIN, COUT>(ring, slot, w_base, tmem + (uint32_t)((1 - b) * 32));
                umma_commit(s_bar + (1 - b));
            }
            issued |= 1 << (1 - b);
        }
        // rows into the slots that tile k has released
        c_prev = rows.count;
        while (rows.tiles > 0 && rows.count < row + RING) rows.fetch<CIN, false>(a.x, ring, tid);
        cp_async_commit();
        // epilogue of tile k: warp w reads TMEM lanes 32w..32w+31 = pixels x0 + 32w + lane
        float v[COUT];
        const uint32_t taddr = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(b * 32);
        if constexpr (COUT == 32) tmem_ld_x32(taddr, v);
        else tmem_ld_x16(taddr, v);
        if (in) {
            if constexpr (EPI == EPI_F32_CH0) {
                a.y32[cell] = v[0] + s_bias[0];
            } else {
                uint32_t packed[COUT / 2];
#pragma unroll
                for (int q = 0; q < COUT / 4; ++q) {
                    float* p = v + 4 * q;
                    if constexpr (EPI == EPI_RELU_BF16) {
                        const float4 bq = reinterpret_cast<const float4*>(s_bias)[q];
                        p[0] = fmaxf(p[0] + bq.x, 0.0f);
                        p[1] = fmaxf(p[1] + bq.y, 0.0f);
                        p[2] = fmaxf(p[2] + bq.z, 0.0f);
                        p[3] = fmaxf(p[3] + bq.w, 0.0f);
                    } else {  // gradient through the ReLU of the layer below
                        const uint32_t m0 = q & 1 ? m[q / 2].z : m[q / 2].x, m1 = q & 1 ? m[q / 2].w : m[q / 2].y;
                        p[0] = __uint_as_float(m0 << 16) > 0.0f ? p[0] : 0.0f;
                        p[1] = __uint_as_float(m0 & 0xffff0000u) > 0.0f ? p[1] : 0.0f;
                        p[2] = __uint_as_float(m1 << 16) > 0.0f ? p[2] : 0.0f;
                        p[3] = __uint_as_float(m1 & 0xffff0000u) > 0.0f ? p[3] : 0.0f;
                    }
                    packed[2 * q] = pack_bf16(p[0], p[1]);
                    packed[2 * q + 1] = pack_bf16(p[2], p[3]);
                }
#pragma unroll
                for (int q = 0; q < COUT / 16; ++q) st_global_32(a.y + cell * COUT + 16 * q, packed + 8 * q);
            }
        }
        t = tn;
    }
    // after a failed wait MMAs may still be in flight: wait for every committed group
    // once more (bounded) before freeing TMEM; no copy is left in flight either
    cp_async_wait_all();
    if (tid == 0)
        for (int bb = 0; bb < 2; ++bb)
            if (issued & (1 << bb)) mbar_wait_bounded(s_bar + bb, (phase >> bb) & 1u);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncol));
}

// Weight gradients dW[tap][ci][co] = sum_p x[p + off(tap)][ci] gy[p][co] as MMAs on the
// tensor cores, K = pixels.  The input rows are staged as for the convolution, in a ring walked
// down the strips.  Read with the pixel as K, an 8-pixel x 8-channel block (128 contiguous bytes)
// is a core matrix of an MN-major operand, so A (M = 4 rows x 32 channels, a tile's three rows and
// whatever lies in the slot behind them: its products are discarded) and B (N = cout channels of
// gy, staged [chunk][pixel] x 16 bytes) need no transpose, and the three column offsets of the
// taps are start addresses 16 bytes apart.  M runs over rows at one stride, so rows in the ring's
// first two slots are written twice, the second time behind its end.  Each block accumulates all
// its tiles in TMEM (three 32-column accumulators, one per column offset) and writes one FP32
// partial.  The bias gradients are summed on the side: warp w takes gy's channels 8w..8w+7, each
// lane four pixels of a tile, and the lanes add up once at the end.
//
// In iteration k the CTA issues tile k's MMAs, sums its biases, waits for the MMAs of tile k-1
// and starts the copies of the rows and of gy (three buffers) that its release makes room for.
// 32 channels at 513 x 1025: 40 us (the MMAs' reads of A alone 12; 93 when each tile waited
// for the copies of four rows and for its MMAs in turn, and one thread per channel summed the
// bias over 128 pixels).
constexpr int WG_SLOTS = RING + 3;
constexpr int WG_SMEM_X = WG_SLOTS * SLOT_BYTES;              // 74880
constexpr int WG_SMEM_G = MAX_CHUNKS * CNN_TILE * 16;         // 8192
constexpr int WG_GBUF = 3;
constexpr int SMEM_WGRAD = WG_SMEM_X + WG_GBUF * WG_SMEM_G + 64;   // two CTAs per SM
// MN-major core matrices, no swizzle: the descriptor's leading-dimension offset is
// the byte distance between core matrices adjacent along K (8 more pixels: 128 bytes
// in both staged layouts), the stride-dimension offset the distance along M/N (8 more
// channels: one plane row of the halo, one chunk plane of gy).  (Checked against the
// FP64 reference of the gradients; the other assignment gives wrong sums.)
constexpr uint32_t WG_K_STRIDE = 128;

__host__ __device__ constexpr uint32_t umma_idesc_mn(int M, int N) {
    return umma_idesc(M, N) | (1u << 15) | (1u << 16);  // A and B MN-major
}

// gy of a tile's 128 pixels, zero beyond the row
template <int COUT>
__device__ __forceinline__ void wgrad_fetch_gy(const __nv_bfloat16* gy, const Walk& t, uint32_t buf, int tid) {
    constexpr int NCH = COUT / 8, PIX = 128 / NCH;
    const int c = tid % NCH, p0 = tid / NCH, x0 = t.strip * CNN_TILE + p0;
    const __nv_bfloat16* src = gy + (t.I.off + (int64_t)t.y * t.I.W + x0) * COUT + c * 8;
    const uint32_t d = buf + (c * CNN_TILE + p0) * 16;
#pragma unroll
    for (int j = 0; j < CNN_TILE / PIX; ++j) {
        const bool in = x0 + j * PIX < t.I.W;
        cp_async16(d + j * PIX * 16, in ? src + j * PIX * COUT : gy, in ? 16u : 0u);
    }
}

template <int CIN, int COUT>
__global__ void __launch_bounds__(128) k_wgrad_tc(CnnWgradArgs a) {
    extern __shared__ __align__(1024) uint8_t smem[];
    uint8_t* s_g = smem + WG_SMEM_X;
    uint64_t* s_bar = reinterpret_cast<uint64_t*>(s_g + WG_GBUF * WG_SMEM_G);   // [2]
    uint32_t* s_tmem = reinterpret_cast<uint32_t*>(s_bar + 2);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int ncol = 128;  // three accumulators of 32 columns

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(s_tmem)), "r"(ncol));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        mbar_init(s_bar, 1);
        mbar_init(s_bar + 1, 1);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *s_tmem;
    const uint32_t idesc = umma_idesc_mn(128, COUT);
    const uint32_t xb = smem_u32(smem), gb = smem_u32(s_g);
    const uint32_t lbo = WG_K_STRIDE, sbo_a = PLANE_BYTES, sbo_b = CNN_TILE * 16;
    const int64_t t0 = a.ntiles * blockIdx.x / gridDim.x, t1 = a.ntiles * (blockIdx.x + 1) / gridDim.x;
    const int64_t nt = t1 - t0;
    RowStream rows;
    rows.init(a.img, a.nimg, t0, t1);
    Walk t, tg;              // tile k; the tile whose gy comes next
    int64_t gleft = nt;      // tiles whose gy is still to fetch
    if (nt > 0) {
        t.seek(a.img, a.nimg, t0);
        tg = t;
    }
    int c_prev = 0;
    for (int h = 0; h < 2; ++h) {
        c_prev = rows.count;
        while (rows.tiles > 0 && rows.count < 3 * (h + 1)) rows.fetch<CIN, true>(a.x, xb, tid);
        if (gleft > 0) {
            wgrad_fetch_gy<COUT>(a.gy, tg, gb + h * WG_SMEM_G, tid);
            if (--gleft > 0) tg.next();
        }
        cp_async_commit();
    }
    float bacc[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) bacc[j] = 0.0f;
    int64_t issued = 0, waited = 0;   // tiles whose MMAs were committed, and waited for
    bool ok = true;
    int failed = 0;
    int row = 0, slot = 0, gbuf = 0;
    for (int64_t k = 0; k < nt; ++k) {
        if (row + 3 <= c_prev) cp_async_wait_but_last();
        else cp_async_wait_all();
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        tc_fence_before();
        failed = __syncthreads_or(!ok);
        tc_fence_after();
        if (failed) break;
        if (tid == 0) {
            const uint64_t ad = umma_desc(xb + slot * SLOT_BYTES, lbo, sbo_a);
            const uint64_t bd = umma_desc(gb + gbuf * WG_SMEM_G, lbo, sbo_b);
#pragma unroll
            for (int dx = 0; dx < 3; ++dx)
#pragma unroll
                for (int kc = 0; kc < CNN_TILE / 16; ++kc)
                    umma_bf16(tmem + (uint32_t)(dx * 32), ad + dx + kc * 2 * WG_K_STRIDE / 16,
                              bd + kc * 2 * WG_K_STRIDE / 16, idesc, (k > 0 || kc > 0) ? 1u : 0u);
            umma_commit(s_bar + (k & 1));
        }
        ++issued;
        if (warp < COUT / 8) {  // bias gradient
            const uint4* g = reinterpret_cast<const uint4*>(s_g + gbuf * WG_SMEM_G) + warp * CNN_TILE + lane;
#pragma unroll
            for (int q = 0; q < CNN_TILE / 32; ++q) {
                const uint4 v = g[q * 32];
                const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    bacc[2 * j] += __uint_as_float(u[j] << 16);
                    bacc[2 * j + 1] += __uint_as_float(u[j] & 0xffff0000u);
                }
            }
        }
        if (k > 0) {  // the MMAs of tile k - 1
            ok = mbar_wait_bounded(s_bar + ((k - 1) & 1), (uint32_t)((k - 1) >> 1) & 1u);
            if (ok) ++waited;
            else set_status(a.status, VIP_ERR_TIMEOUT);
        }
        c_prev = rows.count;
        if (ok) {
            while (rows.tiles > 0 && rows.count < row + RING) rows.fetch<CIN, true>(a.x, xb, tid);
            if (gleft > 0) {
                wgrad_fetch_gy<COUT>(a.gy, tg, gb + (gbuf == 0 ? 2 : gbuf - 1) * WG_SMEM_G, tid);  // tile k + 2
                if (--gleft > 0) tg.next();
            }
        }
        cp_async_commit();
        const int step = t.next() ? 3 : 1;
        row += step;
        slot = slot + step >= RING ? slot + step - RING : slot + step;
        gbuf = gbuf == WG_GBUF - 1 ? 0 : gbuf + 1;
    }
    // the last tile's MMAs (after a failed wait, all that may still be in flight)
    for (; waited < issued; ++waited)
        if (!mbar_wait_bounded(s_bar + (waited & 1), (uint32_t)(waited >> 1) & 1u)) {
            set_status(a.status, VIP_ERR_TIMEOUT);
            ok = false;
        }
    cp_async_wait_all();
    tc_fence_before();
    failed |= __syncthreads_or(!ok);
    tc_fence_after();
    constexpr int nent = 9 * CIN * COUT;
    float* dst = a.part + (int64_t)blockIdx.x * (nent + COUT);
    if (nt > 0 && !failed) {
        // warp w holds TMEM lanes 32w..32w+31 = row w of the window (tap row dy = w), channel = lane
        for (int dx = 0; dx < 3; ++dx) {
            float v[COUT];
            const uint32_t taddr = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(dx * 32);
            if constexpr (COUT == 32) tmem_ld_x32(taddr, v);
            else tmem_ld_x16(taddr, v);
            if (warp < 3 && lane < CIN) {
                float4* o = reinterpret_cast<float4*>(dst + ((warp * 3 + dx) * CIN + lane) * COUT);
#pragma unroll
                for (int q = 0; q < COUT / 4; ++q) o[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
            }
        }
    } else {
        for (int e = tid; e < nent; e += blockDim.x) dst[e] = 0.0f;
    }
    if (warp < COUT / 8)
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            float v = bacc[j];
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (lane == 0) dst[nent + warp * 8 + j] = v;
        }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncol));
}

// The instance for a layer's channel counts (16 or 32 each) and epilogue.
static auto wgrad_kernel(int cin, int cout) {
    return cin == 16 ? (cout == 16 ? k_wgrad_tc<16, 16> : k_wgrad_tc<16, 32>)
                     : (cout == 16 ? k_wgrad_tc<32, 16> : k_wgrad_tc<32, 32>);
}
template <int EPI>
static auto conv_kernel_of(int cin, int cout) {
    return cin == 16 ? (cout == 16 ? k_conv_tc<16, 16, EPI> : k_conv_tc<16, 32, EPI>)
                     : (cout == 16 ? k_conv_tc<32, 16, EPI> : k_conv_tc<32, 32, EPI>);
}
static auto conv_kernel(int cin, int cout, int epi) {
    return epi == EPI_RELU_BF16 ? conv_kernel_of<EPI_RELU_BF16>(cin, cout)
         : epi == EPI_F32_CH0   ? conv_kernel_of<EPI_F32_CH0>(cin, cout)
                                : conv_kernel_of<EPI_MASK_BF16>(cin, cout);
}

cudaError_t cnn_wgrad_tc(const CnnWgradArgs& a, int nblocks, cudaStream_t s, const char** why) {
    *why = "";
    if (a.ntiles <= 0 || nblocks <= 0) return cudaSuccess;
    if (a.cin % 16 || a.cin > CNN_CH || (a.cout != 16 && a.cout != 32)) {
        *why = "unsupported channel counts";
        return cudaErrorInvalidValue;
    }
    wgrad_kernel(a.cin, a.cout)<<<nblocks, 128, SMEM_WGRAD, s>>>(a);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) *why = "weight-gradient launch";
    return e;
}

cudaError_t cnn_conv_init() {
    for (int cin : {16, 32})
        for (int cout : {16, 32}) {
            for (int epi : {EPI_RELU_BF16, EPI_F32_CH0, EPI_MASK_BF16}) {
                const cudaError_t e = cudaFuncSetAttribute(conv_kernel(cin, cout, epi),
                                                           cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_CONV);
                if (e != cudaSuccess) return e;
            }
            const cudaError_t e = cudaFuncSetAttribute(wgrad_kernel(cin, cout),
                                                       cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_WGRAD);
            if (e != cudaSuccess) return e;
        }
    return cudaSuccess;
}

cudaError_t cnn_conv_fwd(const CnnConvArgs& a, int nsm, cudaStream_t s, const char** why) {
    *why = "";
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        *why = "an earlier CUDA call left an error";
        return e;
    }
    if (a.ntiles <= 0) return cudaSuccess;
    if (a.cin % 16 || a.cin > CNN_CH || (a.cout != 16 && a.cout != 32)) {
        *why = "unsupported channel counts";
        return cudaErrorInvalidValue;
    }
    const int grid = (int)std::min<int64_t>(a.ntiles, (int64_t)std::max(nsm, 1) * CONV_CTAS_PER_SM);
    conv_kernel(a.cin, a.cout, a.epi)<<<grid, 128, SMEM_CONV, s>>>(a);
    e = cudaGetLastError();
    if (e != cudaSuccess) *why = "kernel launch";
    return e;
}

}  // namespace vip
