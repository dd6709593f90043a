// A whole solve of a matrix that fits one 128 x 128 tile, in one launch of two CTAs whose
// shared memory holds every iterate (Proposition 1 in the factored form
// A_tau = 1/2 (A - tau P)(I + S); a wide input is the tall problem of A^T).
//
// What bounds it: a solve is a chain of about 64 dependent products per polar factor, each of
// a few MMAs, so the time is the latency of one product's round trip. Through global memory
// (the general kernel: TMA operand loads, TMA stores, a GPU-scope release and acquire of the
// completion counter) that is about 6300 cycles; here the operands stay in shared memory in
// the layout the MMAs read, and a product costs its MMAs, one tensor-memory read, the
// shared-memory stores of the result and one CTA barrier: about 1900 cycles at 64 x 64, of
// which the MMAs' own latency is 500 to 900. 64 x 64, FP32 tier, 30 cubic steps: 415 -> 96 us;
// 97 x 61, BF16 tier, 20 steps: 431 -> 90 us; 128 x 128, BF16 tier: 131 us. Launch, ingest and
// combine take 14 us of these.
//
// Split: a cluster of two CTAs. CTA 0 runs the P chain (X, X^T, Y/Z), CTA 1 the Gram and the
// S chain (S, Y/Z); both ingest A. At the end CTA 0 fetches S' from CTA 1's shared memory and
// runs the combine. Each product is issued by one thread; 16 epilogue warps share the
// accumulator: four per tensor-memory lane quadrant, 16 columns at a time.
//
// Layout: three 64 KiB regions per CTA, each a matrix of up to 128 x 128 as a BF16 hi part and
// (at +32 KiB) a lo part, each part two 64-column groups of 128 rows x 128 bytes with the
// 128-byte swizzle, K-major for the MMA descriptors. Everything outside the matrix is zero, so
// that padded rows, columns and K stay zero through every product. An iterate is overwritten
// in place by the product that reads it (its MMAs have completed before the epilogue starts),
// and Z takes Y's place: an epilogue thread reads C only at the upper-triangle positions that
// it alone writes; mirrored values go to the lower triangle, which is never read as C.
//
// Arithmetic: segment order, K order, scaling, roundings, the mirrored upper triangle and the
// grouping of the norms' sums are those of the general kernel, so results agree with it.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "small_solve.h"
#include "solve_scalars.cuh"
#include "tc_ptx.cuh"

namespace svt {

namespace {

constexpr int kWarps = 16;
constexpr int kCtaThreads = 32 * kWarps;
constexpr uint32_t kPart = 32 << 10;    // one part (hi or lo) of a region
constexpr uint32_t kRegion = 2 * kPart;
constexpr uint32_t kGroup = 16 << 10;   // 64 columns of a part
constexpr int kTmemCols = 128;

// Scalars of one CTA, after the three regions.
struct Shared {
    double colnorm[128];   // squared column norms of the tall matrix
    double nrm_w[kWarps];  // per-warp partial sums of squares
    double inv_alpha2, tau2s, nrm_x0, nrm_s0;
    uint64_t bar;          // completion of a product's MMAs
    alignas(16) uint8_t dummy[128];  // stores of blocks that are not part of a result
    float scale[3];        // alpha, beta, gamma of the first step
    float inv_alpha;
    int status;
    int abort;
    uint32_t tmem;
};

constexpr int kSmemBytes = 3 * (int)kRegion + (int)sizeof(Shared) + kWarps * 129 * 8 + 1024;
static_assert(kSmemBytes <= 232448, "shared memory per CTA");

// Byte offset of element (row, col) within a part.
__device__ __forceinline__ uint32_t at(int row, int col)
{
    return (uint32_t)(col >> 6) * kGroup + (uint32_t)(row * 128 + ((((col >> 3) & 7) ^ (row & 7)) << 4) +
                                                      (col & 7) * 2);
}

// Sixteen values of a row as packed BF16 pairs: hi parts, and lo parts (the rounding
// remainders) where asked for.
struct Row16 {
    uint32_t h[8], l[8];
};

__device__ __forceinline__ void pack16(Row16 &w, const float *v, bool pair)
{
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const __nv_bfloat162 h2 = __floats2bfloat162_rn(v[2 * j], v[2 * j + 1]);
        w.h[j] = *reinterpret_cast<const uint32_t *>(&h2);
        if (pair) {
            const __nv_bfloat162 l2 =
                __floats2bfloat162_rn(v[2 * j] - __low2float(h2), v[2 * j + 1] - __high2float(h2));
            w.l[j] = *reinterpret_cast<const uint32_t *>(&l2);
        }
    }
}

// Row `row`, columns c0 .. c0 + 15 (c0 a multiple of 16): two 16-byte stores per part.
__device__ __forceinline__ void put_row(uint8_t *reg, int row, int c0, const Row16 &w, bool pair)
{
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const uint32_t o = at(row, c0 + 8 * q);
        *reinterpret_cast<uint4 *>(reg + o) =
            make_uint4(w.h[4 * q], w.h[4 * q + 1], w.h[4 * q + 2], w.h[4 * q + 3]);
        if (pair)
            *reinterpret_cast<uint4 *>(reg + kPart + o) =
                make_uint4(w.l[4 * q], w.l[4 * q + 1], w.l[4 * q + 2], w.l[4 * q + 3]);
    }
}

// The transposed place: rows c0 .. c0 + 15 from `from` on, column `col`. A warp's lanes hold
// 32 neighbouring columns, so each store fills 64 bytes of a row.
__device__ __forceinline__ void put_col(uint8_t *reg, int c0, int col, const Row16 &w, bool pair,
                                        int from)
{
    uint8_t *p = reg + (uint32_t)(col >> 6) * kGroup + c0 * 128 + (col & 7) * 2;
    const uint32_t k = (uint32_t)((col >> 3) & 7) << 4;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        if (c0 + i < from)
            continue;
        const uint32_t o = i * 128 + (k ^ ((i & 7) << 4));
        const int sh = 16 * (i & 1);
        *reinterpret_cast<uint16_t *>(p + o) = (uint16_t)(w.h[i >> 1] >> sh);
        if (pair)
            *reinterpret_cast<uint16_t *>(p + kPart + o) = (uint16_t)(w.l[i >> 1] >> sh);
    }
}

// v[i] += beta * C(row, c0 + i), C a part or a hi/lo pair. The general kernel adds the two
// parts one after the other where a row's 32-column chunk is whole, and their sum where the
// matrix ends inside the chunk (edge).
__device__ __forceinline__ void add_c16(const uint8_t *reg, int row, int c0, float beta, float *v,
                                        bool pair, bool edge)
{
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const uint32_t o = at(row, c0 + 8 * q);
        const uint4 wh = *reinterpret_cast<const uint4 *>(reg + o);
        uint4 wl = make_uint4(0, 0, 0, 0);
        if (pair)
            wl = *reinterpret_cast<const uint4 *>(reg + kPart + o);
        const __nv_bfloat162 *h = reinterpret_cast<const __nv_bfloat162 *>(&wh);
        const __nv_bfloat162 *l = reinterpret_cast<const __nv_bfloat162 *>(&wl);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            float2 x = __bfloat1622float2(h[j]);
            const float2 y = __bfloat1622float2(l[j]);
            float &a = v[8 * q + 2 * j], &b = v[8 * q + 2 * j + 1];
            if (pair && edge) {
                x.x += y.x;
                x.y += y.y;
            }
            a = fmaf(beta, x.x, a);
            b = fmaf(beta, x.y, b);
            if (pair && !edge) {
                a = fmaf(beta, y.x, a);
                b = fmaf(beta, y.y, b);
            }
        }
    }
}

// 32 lanes x 16 consecutive FP32 columns of tensor memory into registers.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float *v)
{
    uint32_t r[16];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 "
                 "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                   "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]),
                   "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                 : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i)
        v[i] = __uint_as_float(r[i]);
}

// One CTA's view of the solve.
struct Cta {
    Shared *sh;
    uint32_t parity;
    bool ok;  // false once a bounded wait has given up: no further products
};

// D = sum over the hi/lo segments of L R^T into tensor memory: L's 128 rows against R's
// first rows, K = 64 kblocks. All threads call it; their earlier shared-memory stores are
// made visible to the MMAs, and D is complete for all of them on return.
__device__ __forceinline__ void product(Cta &c, const uint8_t *L, bool lpair, const uint8_t *R,
                                        bool rpair, int kblocks, uint32_t idesc)
{
    fence_async_smem();
    tc_fence_before();
    if (__syncthreads_or(c.ok ? 0 : 1)) {
        c.ok = false;
        return;
    }
    if (threadIdx.x < 32 && elect_one()) {
        tc_fence_after();
        // Descriptor addresses count 16-byte units: 2 per K step, kGroup and kPart in bytes.
        const uint64_t dl = sw128_desc(smem_u32(L)), dr = sw128_desc(smem_u32(R));
        const uint32_t d = c.sh->tmem;
        uint32_t acc = 0;
        const int segs = 1 + (rpair ? 1 : 0) + (lpair ? 1 : 0);
        for (int sg = 0; sg < segs; ++sg) {
            const bool rlo = sg == 1 && rpair, llo = sg > 0 && !rlo;
            uint64_t a = dl + (llo ? kPart >> 4 : 0u), b = dr + (rlo ? kPart >> 4 : 0u);
            for (int kb = 0; kb < kblocks; ++kb, a += kGroup >> 4, b += kGroup >> 4) {
#pragma unroll
                for (int kk = 0; kk < kBK / 16; ++kk) {
                    mma_bf16(d, a + 2 * kk, b + 2 * kk, idesc, acc);
                    acc = 1;
                }
            }
        }
        mma_commit(&c.sh->bar);
    }
    c.ok = mbar_wait(&c.sh->bar, c.parity, &c.sh->abort, &c.sh->status, kWaitTimeoutNs);
    c.parity ^= 1u;
    tc_fence_after();
}

// ---- fragment epilogue: every product but the few that need a row per thread (below)
//
// Tensor memory is read in the matrix-fragment shape: thread t holds, of each 8 x 8 block, row
// t / 4 and columns 2 (t % 4), + 1, which is what ldmatrix and stmatrix move. Per 32 x 16
// chunk a result then takes 2 stmatrix for its place and 2 transposing ones for its mirror, and
// C 2 ldmatrix, instead of 16 two-byte stores with their address arithmetic: the four warps of
// a scheduler (one tensor-memory quadrant, so at 64 x 64 two of the four schedulers do all the
// work) issued 2500 instructions a product that way, and a product took 3300 cycles.

// 16 tensor-memory lanes x 16 columns: v[4 k + 0, 1] row t / 4, columns 8 k + 2 (t % 4), + 1;
// v[4 k + 2, 3] row t / 4 + 8.
__device__ __forceinline__ void tmem_ld_frag(uint32_t taddr, float *v)
{
    uint32_t r[8];
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                   "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
#pragma unroll
    for (int i = 0; i < 8; ++i)
        v[i] = __uint_as_float(r[i]);
}

// A thread's shared-memory offsets for its warp's first chunk (rows 32 (warp % 4), columns
// 16 (warp / 4)), the same for every product. stmatrix and ldmatrix move the four 8 x 8 blocks
// g (rows + 8 g) of one column group k (columns + 8 k); lane l gives the address of row l % 8 of
// block l / 8.
struct Lanes {
    uint32_t a[2];   // k = 0, 1 in place
    uint32_t q[2];   // and mirrored
    uint32_t dummy;  // where blocks that are not part of a result go
};

__device__ __forceinline__ Lanes lane_offsets(const Shared *sh)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int r0 = 32 * (warp & 3), c0 = 16 * (warp >> 2);
    Lanes o;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        o.a[k] = at(r0 + lane, c0 + 8 * k);
        o.q[k] = at(c0 + 8 * k + (lane & 7), r0 + 8 * (lane >> 3));
    }
    o.dummy = smem_u32(sh->dummy) + 16u * (lane & 7);
    return o;
}

// One 32 x 16 chunk of epi_frag. GD: the diagonal crosses column group k in block g = GD + k
// (0 or 2; 8: not at all).
template <bool HASC, int GD>
__device__ __forceinline__ void frag_chunk(uint32_t taddr, const Lanes &o, uint32_t dst,
                                           uint32_t dst_t, uint32_t shift, uint32_t shift_t,
                                           bool opair, bool cpair, bool edge, int diag_rows,
                                           float alpha, float beta, float gamma)
{
    const int lane = threadIdx.x & 31;
    const int row = lane >> 2, col = 2 * (lane & 3);
    float v[2][8];  // [tensor-memory lanes 0-15, 16-31][column group, row half, column]
    tmem_ld_frag(taddr, v[0]);
    tmem_ld_frag(taddr + (16u << 16), v[1]);
    uint32_t ch[2][4], cl[2][4];
    if (HASC) {
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            ldmatrix4(ch[k], dst + o.a[k] + shift);
            if (cpair)
                ldmatrix4(cl[k], dst + kPart + o.a[k] + shift);
        }
    }
    tmem_ld_wait();
    float x[2][4][2];
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int g = 0; g < 4; ++g)
#pragma unroll
            for (int e = 0; e < 2; ++e)
                x[k][g][e] = __fmul_rn(v[g >> 1][4 * k + 2 * (g & 1) + e], alpha);
    if (HASC) {
        if (cpair && edge) {
#pragma unroll
            for (int k = 0; k < 2; ++k)
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                    const float2 f = bf16x2(ch[k][g]), l = bf16x2(cl[k][g]);
                    x[k][g][0] = fmaf(beta, f.x + l.x, x[k][g][0]);
                    x[k][g][1] = fmaf(beta, f.y + l.y, x[k][g][1]);
                }
        } else {
#pragma unroll
            for (int k = 0; k < 2; ++k)
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                    const float2 f = bf16x2(ch[k][g]);
                    x[k][g][0] = fmaf(beta, f.x, x[k][g][0]);
                    x[k][g][1] = fmaf(beta, f.y, x[k][g][1]);
                }
            if (cpair) {
#pragma unroll
                for (int k = 0; k < 2; ++k)
#pragma unroll
                    for (int g = 0; g < 4; ++g) {
                        const float2 l = bf16x2(cl[k][g]);
                        x[k][g][0] = fmaf(beta, l.x, x[k][g][0]);
                        x[k][g][1] = fmaf(beta, l.y, x[k][g][1]);
                    }
            }
        }
    }
    if (GD < 4) {
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const bool in = 8 * (GD + k) + row < diag_rows;
            float *d = x[k][GD + k < 4 ? GD + k : 0];
            if (in && row == col)
                d[0] += gamma;
            if (in && row == col + 1)
                d[1] += gamma;
        }
    }
    uint32_t w[2][4];
    auto store = [&](uint32_t part) {
        if (GD < 4) {
#pragma unroll
            for (int k = 0; k < 2; ++k)
                w[k][GD + k < 4 ? GD + k : 0] = mirror_diag(w[k][GD + k < 4 ? GD + k : 0], lane);
        }
        const int g = lane >> 3;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            stmatrix4<false>(GD < 4 && g > GD + k ? o.dummy : dst + part + o.a[k] + shift, w[k]);
            stmatrix4<true>(GD < 4 && g >= GD + k ? o.dummy : dst_t + part + o.q[k] + shift_t, w[k]);
        }
    };
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            const __nv_bfloat162 h2 = __floats2bfloat162_rn(x[k][g][0], x[k][g][1]);
            w[k][g] = *reinterpret_cast<const uint32_t *>(&h2);
            x[k][g][0] -= __low2float(h2);
            x[k][g][1] -= __high2float(h2);
        }
    store(0);
    if (opair) {
#pragma unroll
        for (int k = 0; k < 2; ++k)
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                const __nv_bfloat162 l2 = __floats2bfloat162_rn(x[k][g][0], x[k][g][1]);
                w[k][g] = *reinterpret_cast<const uint32_t *>(&l2);
            }
        store(kPart);
    }
}

// v = alpha D + beta C + gamma I over the warp's chunks, rounded to BF16 parts. SYM: N x N,
// upper triangle and mirror; else rows x N, stored at dst and transposed at dst_t. C is dst's
// previous contents (at upper-triangle places only its own thread writes).
template <bool HASC, bool SYM>
__device__ __forceinline__ void epi_frag(const Cta &c, const Lanes &o, uint8_t *dst, uint8_t *dst_t,
                                         bool opair, bool cpair, int rows, int N, float alpha,
                                         float beta, float gamma)
{
    const int warp = threadIdx.x >> 5;
    const int r0 = 32 * (warp & 3);
    const uint32_t d = smem_u32(dst), dt = smem_u32(dst_t);
#pragma unroll 1
    for (int j = 0; j < 2; ++j) {
        const int c0 = 16 * (warp >> 2) + 64 * j;
        if (r0 >= rows || c0 >= N || (SYM && c0 + 15 < r0))
            continue;
        const uint32_t ta = c.sh->tmem + ((uint32_t)r0 << 16) + (uint32_t)c0;
        const bool edge = N - (c0 & ~31) < 32;  // see add_c16
        const uint32_t sh = j * kGroup, sht = j * 64 * 128;
        if (SYM && c0 == r0)
            frag_chunk<HASC, 0>(ta, o, d, dt, sh, sht, opair, cpair, edge, N - r0, alpha, beta, gamma);
        else if (SYM && c0 == r0 + 16)
            frag_chunk<HASC, 2>(ta, o, d, dt, sh, sht, opair, cpair, edge, N - r0, alpha, beta, gamma);
        else
            frag_chunk<HASC, 8>(ta, o, d, dt, sh, sht, opair, cpair, edge, N - r0, alpha, beta, gamma);
    }
}

// ---- row epilogues (one row per thread), for the products that run once a solve

// Symmetric result with its sum of squares (nrm_w): the shifted Gram (FP64 diagonal) and the
// first step's Y. Norms sum 32 columns of a row in FP32, so one thread takes 32 columns.
__device__ __noinline__ void epi_norm(Shared *sh, uint32_t tmem, uint8_t *dst, bool opair, bool gram,
                                      int N)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int r0 = (warp & 3) * 32, r = r0 + lane;
    float acc = 0.f, d = 0.f;
    if (gram && r < N && (warp >> 2) == (warp & 3))  // the warp that holds the diagonal block
        d = (float)(sh->colnorm[r] * sh->inv_alpha2 - sh->tau2s);
#pragma unroll 1
    for (int j = 0; j < 2; ++j) {
        const int c0 = 16 * (2 * (warp >> 2) + j);
        if (r0 >= N || c0 >= N || c0 + 15 < r0)
            continue;
        float v[16];
        tmem_ld16(tmem + ((uint32_t)r0 << 16) + (uint32_t)c0, v);
        const bool straddle = c0 < r0 + 32;
        if (straddle && gram) {
#pragma unroll
            for (int i = 0; i < 16; ++i)
                if (c0 + i == r)
                    v[i] = d;
        }
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const int cc = c0 + i;
            const float w = (r < N && cc < N) ? (r < cc ? 2.f : (r == cc ? 1.f : 0.f)) : 0.f;
            acc = fmaf(w * v[i], v[i], acc);
        }
        // Rows below the chunk's diagonal block are left out; those within it are stored first
        // and then overwritten by the mirror.
        Row16 w;
        pack16(w, v, opair);
        if (r <= c0 + 15)
            put_row(dst, r, c0, w, opair);
        if (straddle)
            __syncwarp();
        put_col(dst, c0, r, w, opair, straddle ? r + 1 : 0);
    }
    double nrm = (double)acc;
    for (int o = 16; o > 0; o >>= 1)
        nrm += __shfl_xor_sync(0xffffffffu, nrm, o);
    if (lane == 0)
        sh->nrm_w[warp] = nrm;
}

// B = A - tau P' (a hi/lo pair), P' the product.
__device__ __forceinline__ void epi_b(const Cta &c, uint8_t *dst, const SmallSolve &p, int M, int N)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int r0 = (warp & 3) * 32, r = r0 + lane;
    const bool wide = p.n > p.m;
#pragma unroll 1
    for (int c0 = 16 * (warp >> 2); c0 < N; c0 += 64) {
        if (r0 >= M)
            break;
        float v[16];
        tmem_ld16(c.sh->tmem + ((uint32_t)r0 << 16) + (uint32_t)c0, v);
        const float *a = wide ? p.A + c0 * p.lda + r : p.A + r * p.lda + c0;
        const int64_t step = wide ? p.lda : 1;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const float x = (r < M && c0 + i < N) ? a[i * step] : 0.f;
            v[i] = __fadd_rn(__fmul_rn(v[i], -p.tau), x);
        }
        Row16 w;
        pack16(w, v, true);
        put_row(dst, r, c0, w, true);
    }
}

struct Scales {
    float alpha, beta, gamma;
};

// The scales a first step takes from its chain's norm: theta = src^(1/4) (or src^(1/2)), then
// alpha theta^-ea, beta theta^-eb, gamma / theta. One warp (lane k computes scale k).
__device__ __forceinline__ void first_scales(Shared *sh, double src, bool quarter, double alpha,
                                             double beta, double gamma, int ea, int eb)
{
    const int lane = threadIdx.x & 31;
    const double s = lane == 0 ? alpha : (lane == 1 ? beta : gamma);
    const int e = lane == 0 ? ea : (lane == 1 ? eb : 1);
    const double theta = root_theta(src, quarter);
    float out = (float)s;
    if (theta > 0.0 && isfinite(theta))
        out = (float)(s / int_pow(theta, e));
    else if (!isfinite(theta) && lane == 0)
        atomicCAS(&sh->status, 0, (int)SVT_ERR_DIVERGED);
    if (lane < 3)
        sh->scale[lane] = out;  // theta == 0: the chain's matrix is zero; nothing to scale
}

__device__ __forceinline__ double sum_nrm(const Shared *sh)
{
    double t = 0.0;
    for (int w = 0; w < kWarps; ++w)
        t += sh->nrm_w[w];
    return t;
}

// A's elements held by one thread between the two passes of the ingest: row it's rows
// row_of(warp, k), columns 4 lane .. 4 lane + 3.
struct InRegs {
    float v[8][4];
};

__device__ __forceinline__ int row_of(int warp, int k)
{
    return (warp & 7) + 64 * (warp >> 3) + 8 * k;
}

__device__ __forceinline__ void load_input(InRegs &x, const SmallSolve &p)
{
    const int warp = threadIdx.x >> 5, c0 = 4 * (threadIdx.x & 31);
    const bool vec = (reinterpret_cast<uintptr_t>(p.A) & 15u) == 0 && (p.lda & 3) == 0 && c0 + 3 < p.n;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const int r = row_of(warp, k);
        const float *a = p.A + r * p.lda + c0;
        float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
        if (r < p.m) {
            if (vec) {
                q = *reinterpret_cast<const float4 *>(a);
            } else {
                if (c0 < p.n)
                    q.x = a[0];
                if (c0 + 1 < p.n)
                    q.y = a[1];
                if (c0 + 2 < p.n)
                    q.z = a[2];
                if (c0 + 3 < p.n)
                    q.w = a[3];
            }
        }
        x.v[k][0] = q.x;
        x.v[k][1] = q.y;
        x.v[k][2] = q.z;
        x.v[k][3] = q.w;
    }
}

// Squared column norms of the tall matrix, ||A||_F^2 and the finiteness check, with the
// general ingest's grouping: squares in FP32 over four values (rows r, r + 8, r + 16, r + 24
// of a column, or four neighbours of a row of a wide input), FP64 beyond.
__device__ __forceinline__ void ingest_norms(Shared *sh, double *part, const InRegs &x,
                                             const SmallSolve &p)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    bool finite = true;
#pragma unroll
    for (int k = 0; k < 8; ++k)
#pragma unroll
        for (int e = 0; e < 4; ++e)
            finite &= isfinite(x.v[k][e]);
    if (p.m >= p.n) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            float q[2] = {0.f, 0.f};
#pragma unroll
            for (int u = 0; u < 8; ++u)
                q[u >> 2] = fmaf(x.v[u][e], x.v[u][e], q[u >> 2]);
            double s = 0.0;
            if (row_of(warp, 0) < p.m)
                s = (double)q[0] + (double)q[1];
            part[warp * 129 + 4 * lane + e] = s;
        }
        __syncthreads();
        if (threadIdx.x < 128) {
            double t = 0.0;
#pragma unroll
            for (int i = 0; i < kWarps; ++i)
                t += part[i * 129 + threadIdx.x];
            sh->colnorm[threadIdx.x] = t;
        }
    } else {
        const int n4 = p.n >> 2;
        // FP64 adds are the cost (16 cycles a warp): the eight rows' sums over the lanes share
        // their first steps, each lane keeping half of the rows it still carries.
        double s[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
        if (row_of(warp, 0) < p.m) {
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const float *v = x.v[k];
                if (lane < n4)
                    s[k] = (double)fmaf(v[0], v[0], fmaf(v[1], v[1], fmaf(v[2], v[2], v[3] * v[3])));
                if (p.n & 3) {  // the columns past the last four: lane l < 3 takes column 4 n4 + l
                    const float t0 = __shfl_sync(0xffffffffu, v[0], n4),
                                t1 = __shfl_sync(0xffffffffu, v[1], n4),
                                t2 = __shfl_sync(0xffffffffu, v[2], n4);
                    const double t = lane == 0 ? t0 : (lane == 1 ? t1 : (lane == 2 ? t2 : 0.f));
                    s[k] += t * t;
                }
            }
#pragma unroll
            for (int h = 4; h > 0; h >>= 1) {
                const bool up = (lane & (4 * h)) != 0;  // exchange with lane ^ 16, 8, 4
#pragma unroll
                for (int k = 0; k < h; ++k) {
                    const double keep = up ? s[k + h] : s[k], send = up ? s[k] : s[k + h];
                    s[k] = keep + __shfl_xor_sync(0xffffffffu, send, 4 * h);
                }
            }
            s[0] += __shfl_xor_sync(0xffffffffu, s[0], 2);
            s[0] += __shfl_xor_sync(0xffffffffu, s[0], 1);
        }
        if ((lane & 3) == 0)
            sh->colnorm[row_of(warp, lane >> 2)] = s[0];  // rows past m: zero
    }
    if (!finite)
        atomicCAS(&sh->status, 0, (int)SVT_ERR_NONFINITE);
    __syncthreads();
    if (warp == 0) {
        double t = (sh->colnorm[lane] + sh->colnorm[lane + 32]) +
                   (sh->colnorm[lane + 64] + sh->colnorm[lane + 96]);
        for (int o = 16; o > 0; o >>= 1)
            t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane == 0) {
            const double ia = 1.0 / pow2_alpha(t), ia2 = ia * ia;  // powers of two
            sh->inv_alpha = (float)ia;
            sh->inv_alpha2 = ia2;
            sh->tau2s = ((double)p.tau * (double)p.tau) * ia2;
            sh->nrm_x0 = t * ia2;
        }
    }
    __syncthreads();
}

__device__ __forceinline__ void zero_smem(uint8_t *b, uint32_t bytes)
{
    for (uint32_t i = threadIdx.x * 16; i < bytes; i += kCtaThreads * 16)
        *reinterpret_cast<uint4 *>(b + i) = make_uint4(0, 0, 0, 0);
}

__global__ void __launch_bounds__(kCtaThreads, 1) small_solve_kernel(const __grid_constant__ SmallSolve p)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *r0 = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                              ~static_cast<uintptr_t>(1023));
    uint8_t *r1 = r0 + kRegion, *r2 = r1 + kRegion;
    Shared *sh = reinterpret_cast<Shared *>(r2 + kRegion);
    double *part = reinterpret_cast<double *>(sh + 1);  // kWarps x 129, for the column norms
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool is_p = cluster_rank() == 0;
    const bool wide = p.n > p.m;
    const int M = wide ? p.n : p.m, N = wide ? p.m : p.n;
    const int kbM = (M + kBK - 1) / kBK, kbN = (N + kBK - 1) / kBK;
    const uint32_t idesc = idesc_bf16(kBM, (N + 15) / 16 * 16);
    const bool pp = p.pairs != 0;

    if (threadIdx.x == 0) {
        mbar_init(&sh->bar, 1);
        sh->status = 0;
        sh->abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        tmem_alloc<false>(&sh->tmem, kTmemCols);
        tmem_relinquish<false>();
    }
    tc_fence_before();
    InRegs in;
    load_input(in, p);
    zero_smem(r0, 3 * kRegion);
    __syncthreads();
    tc_fence_after();

    // ---- ingest: norms, then X0 = A / alpha in both orientations
    ingest_norms(sh, part, in, p);
    {
        // A's rows are rows of X (tall) or of X^T (wide); the other orientation is transposed
        // from them block by block. CTA 1 needs X^T only, as a pair (for a tall input by way of
        // r2); rank-r mode puts B = A in X's place.
        const bool pair = pp || !is_p || p.rank_r;
        const float sc = is_p && p.rank_r ? 1.0f : sh->inv_alpha;
        uint8_t *src = wide ? r1 : (is_p ? r0 : r2), *dst = wide ? r0 : r1;
        const bool both = is_p ? (wide || !p.rank_r) : !wide;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int i = row_of(warp, k);
            if (i >= p.m || 4 * lane >= p.n)
                continue;
            uint32_t h[2], l[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const float x = in.v[k][2 * e] * sc, y = in.v[k][2 * e + 1] * sc;
                const __nv_bfloat162 h2 = __floats2bfloat162_rn(x, y);
                const __nv_bfloat162 l2 = __floats2bfloat162_rn(x - __low2float(h2), y - __high2float(h2));
                h[e] = *reinterpret_cast<const uint32_t *>(&h2);
                l[e] = *reinterpret_cast<const uint32_t *>(&l2);
            }
            const uint32_t o = at(i, 4 * lane);
            *reinterpret_cast<uint2 *>(src + o) = make_uint2(h[0], h[1]);
            if (pair)
                *reinterpret_cast<uint2 *>(src + kPart + o) = make_uint2(l[0], l[1]);
        }
        __syncthreads();
        if (both) {
            const int units = ((p.m + 31) / 32) * ((p.n + 7) / 8);  // 32 rows x 8 columns each
            for (int u = warp; u < units; u += kWarps) {
                const int rr = 32 * (u % ((p.m + 31) / 32)), cc = 8 * (u / ((p.m + 31) / 32));
                const uint32_t from = at(rr + lane, cc), to = at(cc + (lane & 7), rr + 8 * (lane >> 3));
                for (uint32_t part_off = 0; part_off <= (pair ? kPart : 0u); part_off += kPart) {
                    uint32_t w[4];
                    ldmatrix4(w, smem_u32(src) + part_off + from);
                    stmatrix4<true>(smem_u32(dst) + part_off + to, w);
                }
            }
        }
        // What the chain does not read goes back to zero: the scratch, or X^T in rank-r mode.
        if (src == r2) {
            __syncthreads();
            zero_smem(r2, kRegion);
        }
    }

    // ---- chains (the product's entry barrier orders the shared-memory stores)
    Cta c{sh, 0u, true};
    const Lanes lo = lane_offsets(sh);
    const bool gram_norm = !p.norm_fro;
    auto s_pair = [&](int t) { return pp || t < p.hp_steps; };
    if (!is_p) {  // shifted Gram S0
        product(c, r1, true, r1, true, kbM, idesc);
        epi_norm(sh, sh->tmem, r0, s_pair(0), true, N);
        if (!gram_norm) {
            __syncthreads();
            if (threadIdx.x == 0)
                sh->nrm_s0 = sum_nrm(sh);
        }
    }
    // Iterate of X^T X: X^T for the P chain, S itself for the S chain.
    uint8_t *it = is_p ? r1 : r0;
    const int kb_it = is_p ? kbM : kbN;
    for (int t = 0; t <= p.iters && !(is_p && p.rank_r); ++t) {
        const bool polish = t == p.iters, first = t == 0 && !polish;
        const bool quintic = !polish && (!p.cubic || (first && gram_norm));
        const bool xp = is_p ? pp : s_pair(t);  // the iterate (and so Y and Z) is a pair
        const bool zp = xp || polish;
        // In FP32: FP64 instructions run at 2 lanes a cycle and SM, 16 cycles for each warp.
        Scales z = polish ? Scales{-0.5f, 0.f, 1.5f}
                          : (quintic ? Scales{p.coef[3 * t + 2], p.coef[3 * t + 1], p.coef[3 * t]}
                                     : Scales{p.coef[3 * t + 1], 0.f, p.coef[3 * t]});
        product(c, it, xp, it, xp, kb_it, idesc);  // X^T X
        if (quintic) {
            if (first && gram_norm)
                epi_norm(sh, sh->tmem, r2, xp, false, N);
            else
                epi_frag<false, true>(c, lo, r2, r2, xp, false, N, N, 1.f, 0.f, 0.f);
            product(c, r2, xp, r2, xp, kbN, idesc);  // Y^2
        }
        if (first) {
            if (warp == kWarps - 1)
                first_scales(sh, gram_norm ? sum_nrm(sh) : (is_p ? sh->nrm_x0 : sh->nrm_s0),
                             gram_norm, quintic ? p.first[2] : p.first[1],
                             quintic ? p.first[1] : 0.0, p.first[0], quintic ? 5 : 3,
                             quintic ? 3 : 0);
            __syncthreads();
            z = Scales{sh->scale[0], sh->scale[1], sh->scale[2]};
        }
        if (quintic)  // Z = c Y^2 + b Y + a I in Y's place
            epi_frag<true, true>(c, lo, r2, r2, zp, xp, N, N, z.alpha, z.beta, z.gamma);
        else  // Z = b X^T X + a I
            epi_frag<false, true>(c, lo, r2, r2, zp, false, N, N, z.alpha, 0.f, z.gamma);
        product(c, r0, xp, r2, zp, kbN, idesc);  // X Z
        if (!is_p)
            epi_frag<false, true>(c, lo, r0, r0, polish || s_pair(t + 1), false, N, N, 1.f, 0.f, 0.f);
        else if (!polish)
            epi_frag<false, false>(c, lo, r0, r1, pp, false, M, N, 1.f, 0.f, 0.f);
        else
            epi_b(c, r0, p, M, N);
    }

    // ---- combine in CTA 0: S' from CTA 1's first region into r1
    cluster_sync_all();
    if (is_p) {
        const uint32_t src = peer_addr(r0, 1);
        for (int part = 0; part < 2; ++part)
            for (uint32_t i = threadIdx.x * 16; i < (uint32_t)kbN * kGroup; i += kCtaThreads * 16) {
                const uint32_t o = part * kPart + i;
                uint4 w;
                asm volatile("ld.shared::cluster.v4.u32 {%0, %1, %2, %3}, [%4];"
                             : "=r"(w.x), "=r"(w.y), "=r"(w.z), "=r"(w.w)
                             : "r"(src + o)
                             : "memory");
                *reinterpret_cast<uint4 *>(r1 + o) = w;
            }
        if (threadIdx.x == 0) {
            int st;
            asm volatile("ld.shared::cluster.u32 %0, [%1];"
                         : "=r"(st)
                         : "r"(peer_addr(&sh->status, 1))
                         : "memory");
            if (st)
                atomicCAS(&sh->status, 0, st);
        }
    }
    cluster_sync_all();
    if (is_p) {
        product(c, r0, true, r1, true, kbN, idesc);  // Y = 1/2 (B S' + B)
        const int quad = warp & 3, sub = warp >> 2, row0 = quad * 32, r = row0 + lane;
        float acc = 0.f;
#pragma unroll 1
        for (int j = 0; j < 2; ++j) {
            const int c0 = 16 * (2 * sub + j);
            if (row0 >= M || c0 >= N)
                break;
            float v[16];
            tmem_ld16(sh->tmem + ((uint32_t)row0 << 16) + (uint32_t)c0, v);
#pragma unroll
            for (int i = 0; i < 16; ++i)
                v[i] *= 0.5f;
            add_c16(r0, r, c0, 0.5f, v, true, N - (c0 & ~31) < 32);
            if (r >= M)
                continue;
#pragma unroll
            for (int i = 0; i < 16; ++i)
                if (c0 + i < N)
                    acc = fmaf(v[i], v[i], acc);
            if (wide) {
#pragma unroll
                for (int i = 0; i < 16; ++i)
                    if (c0 + i < N)
                        p.Y[(c0 + i) * p.ldy + r] = v[i];
            } else {
                float *y = p.Y + r * p.ldy + c0;
                if (c0 + 16 <= N && (reinterpret_cast<uintptr_t>(y) & 15u) == 0) {
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        reinterpret_cast<float4 *>(y)[q] =
                            make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
                } else {
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        if (c0 + i < N)
                            y[i] = v[i];
                }
            }
        }
        const int bad = __syncthreads_or(isfinite(acc) ? 0 : 1);
        if (threadIdx.x == 0) {
            int st = *reinterpret_cast<volatile int *>(&sh->status);
            if (st == 0 && bad)
                st = (int)SVT_ERR_DIVERGED;
            if (p.d_status)
                *reinterpret_cast<int *>(p.d_status) = st;
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc<false>(sh->tmem, kTmemCols);
    }
}

} // namespace

cudaError_t small_solve_launch(const SmallSolve &p, cudaStream_t s)
{
    cudaError_t e = cudaFuncSetAttribute(small_solve_kernel,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
    if (e != cudaSuccess)
        return e;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cfg.gridDim = dim3(2, 1, 1);
    cfg.blockDim = dim3(kCtaThreads, 1, 1);
    cfg.dynamicSmemBytes = kSmemBytes;
    cfg.stream = s;
    return cudaLaunchKernelEx(&cfg, small_solve_kernel, p);
}

void small_solve_flops(const SmallSolve &p, double *alg, double *executed)
{
    const double M = p.m > p.n ? p.m : p.n, N = p.m > p.n ? p.n : p.m;
    const double npad = (double)(((int)N + 15) / 16 * 16);
    const double kM = (double)(((int)M + kBK - 1) / kBK * kBK), kN = (double)(((int)N + kBK - 1) / kBK * kBK);
    double a = 0.0, x = 0.0;
    auto add = [&](bool sym, double rows, double k, double kpad, int segs) {
        a += (sym ? 1.0 : 2.0) * rows * N * k;
        x += 2.0 * segs * kBM * npad * kpad;
    };
    auto s_pair = [&](int t) { return p.pairs || t < p.hp_steps; };
    const int ps = p.pairs ? 3 : 1;
    add(true, N, M, kM, 3);
    for (int t = 0; t < p.iters; ++t) {
        const bool quintic = !p.cubic || (t == 0 && !p.norm_fro);
        const int ss = s_pair(t) ? 3 : 1;
        if (!p.rank_r) {
            add(true, N, M, kM, ps);
            if (quintic)
                add(true, N, N, kN, ps);
            add(false, M, N, kN, ps);
        }
        for (int k = 0; k < (quintic ? 3 : 2); ++k)
            add(true, N, N, kN, ss);
    }
    const bool fp = s_pair(p.iters);
    if (!p.rank_r) {
        add(true, N, M, kM, ps);
        add(false, M, N, kN, p.pairs ? 3 : 2);
    }
    add(true, N, N, kN, fp ? 3 : 1);
    add(true, N, N, kN, fp ? 3 : 2);
    add(false, M, N, kN, 3);
    *alg = a;
    *executed = x;
}

} // namespace svt
