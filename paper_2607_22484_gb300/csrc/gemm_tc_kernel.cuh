// Tensor-core product kernel for sm_103a: D = sum_s L_s R_s^T with BF16
// operands staged by TMA into 128-byte-swizzled shared memory, tcgen05.mma
// (kind::f16, BF16 x BF16 -> FP32) accumulating in tensor memory, and a fused
// epilogue that reads the accumulator back with tcgen05.ld. Problems flagged fp8
// (the FP8 experiment) take e4m3 operands through kind::f8f6f4 instead; the operand
// kind, like the epilogue's chunk loop (one copy per product kind), is chosen once
// per tile.
//
// This one kernel carries every dense product of the method (Section 2): the
// shifted Gram A^T A - tau^2 I, the polynomial steps X (a I + b X^T X +
// c (X^T X)^2) of both polar chains, the polish step and the final combine
// 1/2 (A - tau P)(I + S) of Proposition 1.
//
// Structure (persistent, one CTA per SM, 384 threads):
//   warp 0    : TMA producer (an elected lane), STAGES-deep shared-memory ring.
//   warp 1    : tensor-memory allocator and MMA issuer (an elected lane).
//   warps 2-9 : epilogue; warp w reads TMEM lanes 32 (w % 4) .. 32 (w % 4) + 31, and
//               the two warps of a lane quadrant take alternate 64-column units.
//   warp 10   : tile scheduler of fused launches: takes and decodes the next tile and checks
//               its dependencies while the producer loads the current one.
//   warp 11   : publisher of fused launches (one thread): releases finished tiles.
// Two accumulator buffers of BN FP32 columns each let the epilogue of one tile
// overlap the MMAs of the next.
//
// CTA-pair mode (PAIR): a cluster of two CTAs computes one 256 x 256 (or 256 x 128)
// tile with tcgen05.mma.cta_group::2. Each CTA stages its own 128 rows of L and one half
// (128 or 64 rows) of the tile's R, so a pipeline stage is 32 KiB instead of 48 KiB (24
// instead of 32) and every operand byte crosses L2 -> SM once per pair instead of once per CTA.
// The even CTA (leader) issues the MMAs for both, its barriers collect both
// CTAs' TMA bytes and both CTAs' epilogue releases; MMA completion is multicast
// to both CTAs, whose epilogues each drain their own 128 x 256 accumulator.
//
// Every wait on an mbarrier is bounded (kWaitTimeoutNs of global time); on
// expiry the kernel records SVT_ERR_TIMEOUT in the solve's status word (launches that
// several solves share leave that to their finalize kernel, which finds the solves with
// unfinished products), the other roles stop at their next wait, in-flight copies and MMAs
// are drained (again with a bound) and tensor memory is released before the kernel returns.
#pragma once

#include <algorithm>
#include <cstddef>

#include <cuda_bf16.h>
#include <cuda_fp8.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "solve_scalars.cuh"
#include "tc_ptx.cuh"

namespace svt {

namespace {

// Warp roles: producer, MMA issuer, 8 epilogue warps, tile scheduler, publisher.
constexpr int kEpiWarps = 8;
constexpr int kSchedWarp = 2 + kEpiWarps;
constexpr int kPubWarp = kSchedWarp + 1;
constexpr int kThreads = 32 * (kPubWarp + 1);

// Limit of the waits on other tiles' results (the launch's debug setting, else 2 s).
__device__ __forceinline__ uint64_t dep_limit(const TcLaunch &L)
{
    return L.dep_wait_ns ? (uint64_t)L.dep_wait_ns : kWaitTimeoutNs;
}

// Wait for strip `idx` of dependency k of problem P (see TcProblem::sdep_*), unless the
// producing problem is already known (src_done) or found to be complete as a whole,
// which covers every strip; a role then stops checking that source.
__device__ __forceinline__ bool wait_strip(const TcLaunch &L, const TcProblem &P, int k, int idx,
                                           bool &src_done, volatile int *abort_flag, int *status)
{
    if (src_done)
        return true;
    if (ld_acquire_gpu(&L.done[P.sdep_src[k]]) >= P.sdep_whole[k]) {
        src_done = true;
        return true;
    }
    return wait_counter(&L.strips[P.sdep_base[k] + idx], P.sdep_target[k], abort_flag, status,
                        dep_limit(L));
}

// ---------------------------------------------------------------- tiles

struct TileCoord {
    int prob, tm, tn;
    bool valid;
};

__device__ __forceinline__ const TcProblem &prob_at(const TcLaunch &L, int p)
{
    return L.gtab ? L.gtab[p] : L.p[p];
}

// The tile of index `local` within problem p, for tiles of TM x BN.
// Dense problems: column-major over the tile grid. Symmetric problems: only
// tiles holding some element with row <= col; column tn holds r (tn + 1) row
// tiles (r = BN / TM), so the first tile of column tn is r tn (tn + 1) / 2
// (tiles taller than wide, and ROWMAJOR_SYM with square tiles: see below).
template <int BN, int TM, bool ROWMAJOR_SYM>
__device__ TileCoord tile_coord(const TcProblem &P, int p, int local)
{
    TileCoord tc{p, 0, 0, false};
    if (!P.sym) {
        tc.tm = local % P.tiles_m;
        tc.tn = local / P.tiles_m;
        tc.valid = true;
        return tc;
    }
    constexpr int r = BN / TM;
    if (r == 0) {
        // Tiles twice as tall as wide (256 x 128, 128 x 64): columns 2 j and 2 j + 1 hold j + 1
        // row tiles each, the first of them from index j (j + 1) on.
        int j = (int)((sqrtf(4.0f * (float)local + 1.0f) - 1.0f) * 0.5f);
        while (j > 0 && j * (j + 1) > local)
            --j;
        while ((j + 1) * (j + 2) <= local)
            ++j;
        const int rem = local - j * (j + 1);
        tc.tn = 2 * j + (rem > j ? 1 : 0);
        tc.tm = rem > j ? rem - (j + 1) : rem;
        tc.valid = (tc.tm < P.tiles_m) && (tc.tn < P.tiles_n);
        return tc;
    }
    if (ROWMAJOR_SYM && r == 1) {
        // Square tiles: row-major over the upper triangle (row tm holds columns
        // tm .. T - 1, first index tm T - tm (tm - 1) / 2), so that the strips of a
        // symmetric product complete in order.
        const int T = P.tiles_n;
        auto first = [T](int i) { return i * T - i * (i - 1) / 2; };
        const float b = 2.0f * (float)T + 1.0f;
        int tm = (int)((b - sqrtf(fmaxf(b * b - 8.0f * (float)local, 0.0f))) * 0.5f);
        tm = tm < 0 ? 0 : (tm > T - 1 ? T - 1 : tm);
        while (tm > 0 && first(tm) > local)
            --tm;
        while (tm + 1 < T && first(tm + 1) <= local)
            ++tm;
        tc.tm = tm;
        tc.tn = tm + (local - first(tm));
        tc.valid = (tm < P.tiles_m) && (tc.tn < P.tiles_n);
        return tc;
    }
    int tn = (int)((sqrtf(8.0f * (float)local / (float)r + 1.0f) - 1.0f) * 0.5f);
    while (tn > 0 && r * tn * (tn + 1) / 2 > local)
        --tn;
    while (r * (tn + 1) * (tn + 2) / 2 <= local)
        ++tn;
    int tm = local - r * tn * (tn + 1) / 2;
    tc.tm = tm;
    tc.tn = tn;
    tc.valid = (tm < P.tiles_m) && (tn < P.tiles_n);
    return tc;
}

// Tile t of a launch with its problems by value (not fused).
template <int BN, int TM, bool ROWMAJOR_SYM>
__device__ TileCoord decode_tile(const TcLaunch &L, int t)
{
    int p = 0;
    while (p + 1 < L.nprob && t >= L.tile_start[p + 1])
        ++p;
    return tile_coord<BN, TM, ROWMAJOR_SYM>(L.p[p], p, t - L.tile_start[p]);
}

// Problem of tile t in a fused launch's table, by a whole warp. Its tiles' indices only increase,
// so the search goes on from the previous answer (`p`, first tile `start`), 32 problems a load: in
// a batch a CTA's next tile is some twenty problems on, which took one thread nine dependent loads.
__device__ __forceinline__ void find_problem(const TcLaunch &L, int t, int lane, int &p, int &start)
{
    for (;;) {
        const int q = p + 1 + lane;
        const int first = q < L.gcount ? L.gstart[q] : 0x7fffffff;
        const int n = __popc(__ballot_sync(0xffffffffu, first <= t));  // starts increase: a prefix
        if (n > 0)
            start = __shfl_sync(0xffffffffu, first, n - 1);
        p += n;
        if (n < 32)
            return;
    }
}

// ------------------------------------------------------------- epilogue

struct EpiScales {
    float alpha, beta, gamma;
};

// The FP32 scales of a problem's epilogue. Problems scaled by a norm take theta =
// norm^theta_pow (1/2 or 1/4) from the finished sum; their FP64 roots and products run in one
// thread per tile (FP64 is 2 lanes a cycle and SM: the eight epilogue warps computing pow each
// held the first Z products of a solve for 23,500 cycles).
__device__ __forceinline__ EpiScales epi_scales(const TcProblem &P, const CallRec *calls)
{
    const Epi &e = P.ep;
    EpiScales s{e.falpha, e.fbeta, e.fgamma};
    if (P.patch & PT_ALPHA_NEG_TAU)
        s.alpha = -calls[P.call_idx].tau;
    if (e.theta_src) {
        const double theta = root_theta(*e.theta_src, e.theta_pow == 0.25);
        if (theta > 0.0 && isfinite(theta)) {
            s.alpha = (float)(e.alpha / int_pow(theta, (int)e.ea));
            s.beta = (float)(e.beta / int_pow(theta, (int)e.eb));
            s.gamma = (float)(e.gamma / int_pow(theta, (int)e.eg));
        } else if (!isfinite(theta) && e.status) {
            atomicCAS(e.status, 0, (int)SVT_ERR_DIVERGED);
        }  // theta == 0: the chain's matrix is zero; nothing to scale
    }
    return s;
}

__device__ __forceinline__ bool aligned16(const void *p)
{
    return (reinterpret_cast<uintptr_t>(p) & 15u) == 0;
}

// The fields of the current problem that the epilogue reads for every 32 x 32
// block, loaded once per change of problem into registers: the problem table
// lives in global memory, and every memory-clobbering TMA or fence instruction
// of the epilogue would otherwise force these loads to be repeated.
struct EpiHot {
    const void *c0, *c1;
    void *o0, *o1, *t0, *t1;
    const CUtensorMap *maps;  // mapO[0..1], mapT[0..1] of the problem
    double *norm_acc;
    const double *diag, *dss;
    int64_t ldc, ldo, ldt;
    float alpha, beta, gamma;
    int M, N, sym, otma, ttma, wide_tma, c_kind, c_trans, o_kind, o_trans, t_kind;
    void *f0;          // e4m3 copy (FP8 experiment), null: none
    int64_t ldf;
    float fscale;
};

// Raw C values of one lane, loaded ahead. Generic loop: its 32-column row segment in BF16 in
// q[0..3]. Specialised loops: its fragment of the 32 x 32 block, BF16 pairs of block (g, k) in
// word 4 k + g (lo parts 16 further on), or FP32 values in words 2 (4 k + g) + e.
struct CRaw {
    uint4 q[8];
    __device__ __forceinline__ uint32_t &word(int i)
    {
        uint4 &x = q[i >> 2];
        return (i & 3) == 0 ? x.x : ((i & 3) == 1 ? x.y : ((i & 3) == 2 ? x.z : x.w));
    }
};

// Issue the loads of C(r, c0 .. c0 + 31) into registers. Returns false where the vector form does
// not apply (no BF16 C, row outside, a ragged right edge, or a row address that is not 16-byte
// aligned); c_apply then reads C directly. (The products with a C that the generic loop serves,
// those with an e4m3 copy, have a BF16 one.)
__device__ __forceinline__ bool c_load(const EpiHot &h, int64_t r, int64_t c0, bool full_row,
                                       CRaw &cr)
{
    if (h.c_kind != C_BF16 || h.c_trans || !full_row)
        return false;
    const __nv_bfloat16 *ph = static_cast<const __nv_bfloat16 *>(h.c0) + r * h.ldc + c0;
    if (!aligned16(ph))
        return false;
#pragma unroll
    for (int q = 0; q < 4; ++q)
        cr.q[q] = __ldg(reinterpret_cast<const uint4 *>(ph) + q);
    return true;
}

// v[i] += beta * C(r, c0 + i) for i < ncol, from registers loaded by c_load (vec)
// or read directly (any layout, alignment or edge).
__device__ __forceinline__ void c_apply(const EpiHot &h, const CRaw &cr, bool vec, int64_t r,
                                        int64_t c0, int ncol, bool row_ok, float *v)
{
    if (h.c_kind == C_NONE || !row_ok)
        return;
    const float beta = h.beta;
    if (vec) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const __nv_bfloat162 *b = reinterpret_cast<const __nv_bfloat162 *>(&cr.q[q]);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float2 f = __bfloat1622float2(b[j]);
                v[q * 8 + 2 * j] += beta * f.x;
                v[q * 8 + 2 * j + 1] += beta * f.y;
            }
        }
        return;
    }
#pragma unroll
    for (int i = 0; i < 32; ++i) {
        if (i >= ncol)
            continue;
        const int64_t c = c0 + i;
        const int64_t off = h.c_trans ? c * h.ldc + r : r * h.ldc + c;
        float x;
        if (h.c_kind == C_F32)
            x = static_cast<const float *>(h.c0)[off];
        else {
            x = __bfloat162float(static_cast<const __nv_bfloat16 *>(h.c0)[off]);
            if (h.c_kind == C_PAIR)
                x += __bfloat162float(static_cast<const __nv_bfloat16 *>(h.c1)[off]);
        }
        v[i] += beta * x;
    }
}

// Fallback staging: 32 x 32 floats, element (a, b) at a * 32 + (b ^ a); rows and
// columns are both free of bank conflicts.
__device__ __forceinline__ int xs_idx(int a, int b) { return a * 32 + (b ^ a); }

// e4m3 bytes of scale * v, saturated (the FP8 experiment's operand copies), in the
// layout store_block uses: 16 rows x 32 bytes per instruction. Kept out of line so
// that the BF16 epilogue's code is what it is without it.
__device__ __noinline__ void store_block_e4m3(const float *st, void *p0, int64_t ld, int64_t r0,
                                              int64_t c0, int64_t M, int64_t N, bool trans,
                                              bool symdiag, int lane, float scale)
{
    const int64_t orow0 = trans ? c0 : r0, ocol0 = trans ? r0 : c0;
    const int64_t orows = trans ? N : M, ocols = trans ? M : N;
    // e4m3 bytes of scale * v, saturated: 16 rows x 32 bytes per instruction
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int a = k * 16 + (lane >> 1);
        const int q = lane & 1;  // columns 16 q .. 16 q + 15
        const int64_t R = orow0 + a;
        float x[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            const int b = q * 16 + j;
            int sa, sb;
            if (trans) { sa = b; sb = a; }
            else if (symdiag && a > b) { sa = b; sb = a; }
            else { sa = a; sb = b; }
            x[j] = scale * st[xs_idx(sa, sb)];
        }
        if (R >= orows)
            continue;
        const int64_t C = ocol0 + q * 16;
        uint8_t *p = static_cast<uint8_t *>(p0) + R * ld + C;
        if (C + 16 <= ocols && aligned16(p)) {
            uint32_t w[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const uint32_t lo = __nv_cvt_float2_to_fp8x2(make_float2(x[4 * j], x[4 * j + 1]),
                                                             __NV_SATFINITE, __NV_E4M3);
                const uint32_t hi = __nv_cvt_float2_to_fp8x2(make_float2(x[4 * j + 2], x[4 * j + 3]),
                                                             __NV_SATFINITE, __NV_E4M3);
                w[j] = lo | (hi << 16);
            }
            *reinterpret_cast<uint4 *>(p) = make_uint4(w[0], w[1], w[2], w[3]);
        } else {
#pragma unroll
            for (int j = 0; j < 16; ++j)
                if (C + j < ocols)
                    p[j] = __nv_cvt_float_to_fp8(x[j], __NV_SATFINITE, __NV_E4M3);
        }
    }
}

// Store a 32 x 32 block held in shared memory `st` (st[a][b] = value of tile
// element (r0 + a, c0 + b)) to global memory, coalesced: warp lanes cover whole
// row segments (8 rows x 64 B for BF16, 4 rows x 128 B for FP32 per instruction).
//   trans = 0: element (r0 + a, c0 + b) -> p[(r0 + a) * ld + c0 + b];
//              symdiag: the block sits on the diagonal and (a > b) takes st[b][a].
//   trans = 1: element (r0 + b, c0 + a) -> p[(c0 + a) * ld + r0 + b].
// Only elements with row < M and col < N (tile coordinates) are written.
__device__ __forceinline__ void store_block(const float *st, int kind, void *p0, void *p1,
                                            int64_t ld, int64_t r0, int64_t c0, int64_t M,
                                            int64_t N, bool trans, bool symdiag, int lane)
{
    // output rows: tile rows (trans = 0) or tile columns (trans = 1)
    const int64_t orow0 = trans ? c0 : r0, ocol0 = trans ? r0 : c0;
    const int64_t orows = trans ? N : M, ocols = trans ? M : N;
    if (kind == O_BF16 || kind == O_PAIR) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int a = k * 8 + (lane >> 2);  // output row within the block
            const int q = lane & 3;             // 16-byte chunk: columns 8q .. 8q + 7
            const int64_t R = orow0 + a;
            float x[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int b = q * 8 + j;
                int sa, sb;  // staging coordinates
                if (trans) { sa = b; sb = a; }
                else if (symdiag && a > b) { sa = b; sb = a; }
                else { sa = a; sb = b; }
                x[j] = st[xs_idx(sa, sb)];
            }
            if (R >= orows)
                continue;
            const int64_t C = ocol0 + q * 8;
            const int64_t off = R * ld + C;
            if (C + 8 <= ocols && aligned16(static_cast<__nv_bfloat16 *>(p0) + off) &&
                (kind != O_PAIR || aligned16(static_cast<__nv_bfloat16 *>(p1) + off))) {
                uint32_t hw[4], lw[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    __nv_bfloat162 h2 = __floats2bfloat162_rn(x[2 * j], x[2 * j + 1]);
                    hw[j] = *reinterpret_cast<uint32_t *>(&h2);
                    __nv_bfloat162 l2 = __floats2bfloat162_rn(x[2 * j] - __low2float(h2),
                                                              x[2 * j + 1] - __high2float(h2));
                    lw[j] = *reinterpret_cast<uint32_t *>(&l2);
                }
                *reinterpret_cast<uint4 *>(static_cast<__nv_bfloat16 *>(p0) + off) =
                    make_uint4(hw[0], hw[1], hw[2], hw[3]);
                if (kind == O_PAIR)
                    *reinterpret_cast<uint4 *>(static_cast<__nv_bfloat16 *>(p1) + off) =
                        make_uint4(lw[0], lw[1], lw[2], lw[3]);
            } else {
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    if (C + j < ocols) {
                        __nv_bfloat16 h = __float2bfloat16_rn(x[j]);
                        static_cast<__nv_bfloat16 *>(p0)[off + j] = h;
                        if (kind == O_PAIR)
                            static_cast<__nv_bfloat16 *>(p1)[off + j] =
                                __float2bfloat16_rn(x[j] - __bfloat162float(h));
                    }
                }
            }
        }
    } else if (kind == O_F32) {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int a = k * 4 + (lane >> 3);
            const int q = lane & 7;  // columns 4q .. 4q + 3
            const int64_t R = orow0 + a;
            float x[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int b = q * 4 + j;
                int sa, sb;
                if (trans) { sa = b; sb = a; }
                else if (symdiag && a > b) { sa = b; sb = a; }
                else { sa = a; sb = b; }
                x[j] = st[xs_idx(sa, sb)];
            }
            if (R >= orows)
                continue;
            const int64_t C = ocol0 + q * 4;
            const int64_t off = R * ld + C;
            if (C + 4 <= ocols && aligned16(static_cast<float *>(p0) + off)) {
                *reinterpret_cast<float4 *>(static_cast<float *>(p0) + off) =
                    make_float4(x[0], x[1], x[2], x[3]);
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (C + j < ocols)
                        static_cast<float *>(p0)[off + j] = x[j];
            }
        }
    }
}

// Byte offset of element (row, col) of a 32 x 32 staging block laid out the way
// the TMA unit reads it: FP32 rows of 128 B with the 128-byte swizzle (16-byte
// chunk index XOR row % 8), BF16 rows of 64 B with the 64-byte swizzle (chunk
// index XOR (row / 2) % 4). Both orders of writing -- a lane per row with 16-byte
// vectors, or a lane per column with scalars -- are free of bank conflicts.
__device__ __forceinline__ uint32_t stg_off_f32(int row, int col)
{
    return (uint32_t)(row * 128 + ((((col >> 2) ^ (row & 7))) << 4) + (col & 3) * 4);
}
__device__ __forceinline__ uint32_t stg_off_b16(int row, int col)
{
    return (uint32_t)(row * 64 + ((((col >> 3) ^ ((row >> 1) & 3))) << 4) + (col & 7) * 2);
}

// Stage the warp's 32 x 32 block (lane = block row, x[] = its 32 columns) and
// store it with one or two TMA stores (one bulk group): at tile coordinates
// (x = c0, y = r0), or transposed at (x = r0, y = c0). `kind` is O_F32, O_BF16 or
// O_PAIR (hi through m0, lo through m1). The warp owns NSTG 4 KiB staging slots
// (1024-byte aligned) used in turn, so a store's shared-memory read overlaps the
// staging of the next NSTG - 1 blocks; an FP32 block fills a slot, BF16 hi and lo
// take its two halves.
template <int NSTG>
__device__ __forceinline__ void tma_store_block(const float *x, int kind, bool trans,
                                                const CUtensorMap *m0, const CUtensorMap *m1,
                                                int r0, int c0, uint8_t *stg_base, int &slot,
                                                int lane)
{
    uint8_t *stg0 = stg_base + slot * 4096, *stg1 = stg0 + 2048;
    if (++slot == NSTG)
        slot = 0;
    if (elect_one())
        bulk_wait_read<NSTG - 1>();  // the store that last used this slot has read it
    __syncwarp();
    if (kind == O_F32) {
        if (!trans) {
#pragma unroll
            for (int q = 0; q < 8; ++q)
                *reinterpret_cast<float4 *>(stg0 + stg_off_f32(lane, 4 * q)) =
                    make_float4(x[4 * q], x[4 * q + 1], x[4 * q + 2], x[4 * q + 3]);
        } else {
#pragma unroll
            for (int c = 0; c < 32; ++c)
                *reinterpret_cast<float *>(stg0 + stg_off_f32(c, lane)) = x[c];
        }
    } else {
        const bool pair = (kind == O_PAIR);
        if (!trans) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                uint32_t hw[4], lw[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    __nv_bfloat162 h2 = __floats2bfloat162_rn(x[8 * q + 2 * j], x[8 * q + 2 * j + 1]);
                    hw[j] = *reinterpret_cast<uint32_t *>(&h2);
                    __nv_bfloat162 l2 = __floats2bfloat162_rn(x[8 * q + 2 * j] - __low2float(h2),
                                                              x[8 * q + 2 * j + 1] - __high2float(h2));
                    lw[j] = *reinterpret_cast<uint32_t *>(&l2);
                }
                *reinterpret_cast<uint4 *>(stg0 + stg_off_b16(lane, 8 * q)) =
                    make_uint4(hw[0], hw[1], hw[2], hw[3]);
                if (pair)
                    *reinterpret_cast<uint4 *>(stg1 + stg_off_b16(lane, 8 * q)) =
                        make_uint4(lw[0], lw[1], lw[2], lw[3]);
            }
        } else {
#pragma unroll
            for (int c = 0; c < 32; ++c) {
                __nv_bfloat16 h = __float2bfloat16_rn(x[c]);
                *reinterpret_cast<__nv_bfloat16 *>(stg0 + stg_off_b16(c, lane)) = h;
                if (pair)
                    *reinterpret_cast<__nv_bfloat16 *>(stg1 + stg_off_b16(c, lane)) =
                        __float2bfloat16_rn(x[c] - __bfloat162float(h));
            }
        }
    }
    fence_async_smem();
    __syncwarp();
    if (elect_one()) {
        const int sx = trans ? r0 : c0, sy = trans ? c0 : r0;
        tma_store_2d(m0, sx, sy, stg0);
        if (kind == O_PAIR)
            tma_store_2d(m1, sx, sy, stg1);
        bulk_commit();
    }
}

// Rest of the epilogue of one 32 x 32 block after alpha D + beta C: the identity
// term (or the FP64 shifted-Gram diagonal) on the diagonal, the squared-norm
// contribution, then the stores. lane = tile row r0 + lane, columns c0 .. c0 + 31.
// Values are staged in shared memory and stored coalesced to every requested
// destination: the output (row-major or transposed), the extra transposed copy
// and, for symmetric products, the mirror.
template <int NSTG>
__device__ __forceinline__ void epilogue_finish(const EpiHot &h, int64_t r0, int64_t c0, float *v,
                                                double &nrm, uint8_t *stg, int &slot, int lane)
{
    const int64_t r = r0 + lane;
    const bool row_ok = r < h.M;
    const int64_t rem = (int64_t)h.N - c0;
    const int ncol = rem < 32 ? (int)rem : 32;
    const bool diag_block = (r0 == c0);
    if (diag_block) {  // this lane's diagonal element is column i == lane
        const bool dg = h.diag != nullptr;
        const float dval = (dg && row_ok) ? (float)(h.diag[r] * h.dss[0] - h.dss[1]) : 0.f;
        const float g = h.gamma;
#pragma unroll
        for (int i = 0; i < 32; ++i)
            if (i == lane)
                v[i] = dg ? dval : v[i] + g;
    }
    if (h.norm_acc && row_ok) {
        // FP32 within the row's 32 values (relative error <= 32 * 2^-24), FP64 across.
        float acc = 0.f;
#pragma unroll
        for (int i = 0; i < 32; ++i) {
            float w = (i < ncol) ? 1.f : 0.f;
            if (h.sym) {
                const int64_t c = c0 + i;
                w = (r < c) ? 2.f * w : (r == c ? w : 0.f);
            }
            acc = fmaf(w * v[i], v[i], acc);
        }
        nrm += (double)acc;
    }
    const bool symdiag = h.sym && diag_block;
    // Outputs through TMA stores (all but diagonal blocks of symmetric products).
    const bool o_tma = h.otma && h.o_kind != O_NONE && !symdiag;
    if (o_tma)
        tma_store_block<NSTG>(v, h.o_kind, h.o_trans != 0, &h.maps[0], &h.maps[1], (int)r0,
                              (int)c0, stg, slot, lane);
    if (h.sym && !diag_block && h.otma)  // mirror of a block strictly above the diagonal
        tma_store_block<NSTG>(v, h.o_kind, true, &h.maps[0], &h.maps[1], (int)r0, (int)c0, stg,
                              slot, lane);
    if (h.ttma && h.t_kind != O_NONE)
        tma_store_block<NSTG>(v, h.t_kind, true, &h.maps[2], &h.maps[3], (int)r0, (int)c0, stg,
                              slot, lane);
    const bool need_plain = (h.o_kind != O_NONE && !o_tma) || (h.sym && !diag_block && !h.otma) ||
                            (h.t_kind != O_NONE && !h.ttma) || h.f0 != nullptr;
    if (!need_plain)
        return;
    // Coalesced plain-store path: stage with a swizzled pitch, then whole row segments.
    if (elect_one())
        bulk_wait_read0();
    __syncwarp();
    float *st = reinterpret_cast<float *>(stg);
#pragma unroll
    for (int i = 0; i < 32; ++i)
        st[xs_idx(lane, i)] = v[i];
    __syncwarp();
    if (h.o_kind != O_NONE && !o_tma)
        store_block(st, h.o_kind, h.o0, h.o1, h.ldo, r0, c0, h.M, h.N, h.o_trans != 0, symdiag, lane);
    if (h.sym && !diag_block && !h.otma)
        store_block(st, h.o_kind, h.o0, h.o1, h.ldo, r0, c0, h.M, h.N, true, false, lane);
    if (h.t_kind != O_NONE && !h.ttma)
        store_block(st, h.t_kind, h.t0, h.t1, h.ldt, r0, c0, h.M, h.N, true, false, lane);
    if (h.f0) {  // the e4m3 copy, mirrored like the output for symmetric products
        store_block_e4m3(st, h.f0, h.ldf, r0, c0, h.M, h.N, false, symdiag, lane, h.fscale);
        if (h.sym && !diag_block)
            store_block_e4m3(st, h.f0, h.ldf, r0, c0, h.M, h.N, true, false, lane, h.fscale);
    }
    __syncwarp();
}

// Product kinds whose epilogue runs a specialised chunk loop (chosen once per tile), codes:
//   0, 3  symmetric, BF16 / pair output, no C             (Y = X^T X, Y = S^2, S Z)
//   1, 4  symmetric, C of the output kind                 (Z = a I + b Y + c Y^2)
//   2, 5  general, no C, transposed copy of that kind     (X Z and its X^T)
//   6, 7  symmetric, no C, sum of squares, perhaps the FP64 diagonal  (shifted Gram, first Y)
//   8     general, pair output, FP32 C                    (B = A - tau P)
//   9     general, FP32 output by plain stores, pair C, sum of squares  (the combine)
// BF16 and pair outputs go through TMA stores, untransposed. Everything else (e4m3 copies,
// other outputs) runs the generic loop (code -1), which carries every test and takes 17,000 to
// 21,000 cycles for the first tile that fetches its code.
template <int S>
struct EpiSpec {
    static constexpr int code = S;
    static constexpr bool generic = S < 0;
    static constexpr bool pair = S == 3 || S == 4 || S == 5 || S == 7 || S == 8;  // output
    static constexpr bool sym = S == 0 || S == 1 || S == 3 || S == 4 || S == 6 || S == 7;
    static constexpr bool cpair = S == 4 || S == 9;
    static constexpr bool has_c = S == 1 || cpair;  // BF16 C
    static constexpr bool c_f32 = S == 8;
    static constexpr bool norm = S == 6 || S == 7 || S == 9;
    static constexpr bool f32_out = S == 9;
    static constexpr bool mirror = !(S == 8 || S == 9);  // mirrored, or a transposed copy
};

__device__ __forceinline__ int epi_spec(const EpiHot &h)
{
    if (h.f0)
        return -1;
    if (h.o_kind == O_F32)
        return !h.sym && h.c_kind == C_PAIR && !h.c_trans && h.norm_acc && !h.diag &&
                       h.t_kind == O_NONE && h.gamma == 0.f
                   ? 9
                   : -1;
    if ((h.o_kind != O_BF16 && h.o_kind != O_PAIR) || !h.otma || h.o_trans || !h.wide_tma)
        return -1;
    const bool pair = h.o_kind == O_PAIR;
    const int base = pair ? 3 : 0;
    if (h.sym) {
        if (h.t_kind != O_NONE)
            return -1;
        if (h.norm_acc)
            return h.c_kind == C_NONE ? (pair ? 7 : 6) : -1;
        if (h.diag)
            return -1;
        if (h.c_kind == C_NONE)
            return base;
        return h.c_kind == (pair ? C_PAIR : C_BF16) && !h.c_trans ? base + 1 : -1;
    }
    if (h.norm_acc || h.diag || h.gamma != 0.f)
        return -1;
    if (h.c_kind == C_F32)
        return pair && h.t_kind == O_NONE ? 8 : -1;
    return h.t_kind == h.o_kind && h.ttma && h.c_kind == C_NONE ? base + 2 : -1;
}

// Issue the loads of this lane's fragment of C's 32 x 32 block at (r0, c0). Columns past the
// matrix lie in the row padding of the workspace buffers (rows padded to 64 elements).
template <bool PAIRED>
__device__ __forceinline__ void c_load_frag(const EpiHot &h, int64_t r0, int64_t c0, int lane, CRaw &cr)
{
#pragma unroll
    for (int g = 0; g < 4; ++g) {
        const int64_t r = r0 + 8 * g + (lane >> 2);
        const bool ok = r < h.M;
        const int64_t off = r * h.ldc + c0 + 2 * (lane & 3);
        const __nv_bfloat16 *ph = static_cast<const __nv_bfloat16 *>(h.c0) + off;
        const __nv_bfloat16 *pl = static_cast<const __nv_bfloat16 *>(h.c1) + off;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            cr.word(4 * k + g) = ok ? *reinterpret_cast<const uint32_t *>(ph + 8 * k) : 0u;
            if (PAIRED)
                cr.word(16 + 4 * k + g) = ok ? *reinterpret_cast<const uint32_t *>(pl + 8 * k) : 0u;
        }
    }
}

// The same for an FP32 C (the caller's A: any stride and alignment, perhaps transposed): values
// (e = 0, 1) of block (g, k) in words 2 (4 k + g) + e.
__device__ __forceinline__ void c_load_frag_f32(const EpiHot &h, int64_t r0, int64_t c0, int lane,
                                                CRaw &cr)
{
    const float *base = static_cast<const float *>(h.c0);
    const int64_t sr = h.c_trans ? 1 : h.ldc, sc = h.c_trans ? h.ldc : 1;
#pragma unroll
    for (int g = 0; g < 4; ++g) {
        const int64_t r = r0 + 8 * g + (lane >> 2);
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int64_t c = c0 + 8 * k + 2 * (lane & 3) + e;
                cr.word(2 * (4 * k + g) + e) =
                    r < h.M && c < h.N ? __float_as_uint(base[r * sr + c * sc]) : 0u;
            }
    }
}

// Sum of squares of a block's rows, each row's 32 columns in order in one FP32 chain (as the
// row-per-thread loop sums them) that passes through the four lanes of the row; the row sums are
// added in FP64, row 8 g + lane / 4 by the lane with lane % 4 == g. sym: twice the elements right
// of the diagonal, once those on it.
template <bool SYM>
__device__ __forceinline__ void norm_block(const EpiHot &h, const float (&x)[4][4][2], int64_t r0,
                                           int64_t c0, int lane, double &nrm)
{
    const int row = lane >> 2, q = lane & 3;
    const bool diag = SYM && c0 == r0;
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int o = 0; o < 4; ++o) {
            const int col = 8 * k + 2 * o;
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                float a = acc[g];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    float w = 1.f;
                    if (SYM)
                        w = !diag || col + e > 8 * g + row ? 2.f : (col + e == 8 * g + row ? 1.f : 0.f);
                    // columns past the matrix are left out: their C is whatever the padding holds
                    if (c0 + col + e < h.N)
                        a = fmaf(w * x[k][g][e], x[k][g][e], a);
                }
                acc[g] = __shfl_sync(0xffffffffu, a, (lane & ~3) | o);
            }
        }
    const float mine = q == 0 ? acc[0] : (q == 1 ? acc[1] : (q == 2 ? acc[2] : acc[3]));
    if (r0 + 8 * q + row < h.M)
        nrm += (double)mine;
}

// FP32 output of a block by plain stores: a row's four lanes fill 32 bytes of it (or, transposed,
// eight rows' lanes 32 bytes of a column).
__device__ __forceinline__ void store_frag_f32(const EpiHot &h, const float (&x)[4][4][2], int64_t r0,
                                               int64_t c0, int lane)
{
    float *y = static_cast<float *>(h.o0);
    const bool vec = !h.o_trans && (h.ldo & 1) == 0 && (reinterpret_cast<uintptr_t>(y) & 7u) == 0;
#pragma unroll
    for (int g = 0; g < 4; ++g) {
        const int64_t r = r0 + 8 * g + (lane >> 2);
        if (r >= h.M)
            continue;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int64_t c = c0 + 8 * k + 2 * (lane & 3);
            if (vec && c + 1 < h.N) {
                *reinterpret_cast<float2 *>(y + r * h.ldo + c) = make_float2(x[k][g][0], x[k][g][1]);
            } else {
#pragma unroll
                for (int e = 0; e < 2; ++e)
                    if (c + e < h.N)
                        y[h.o_trans ? (c + e) * h.ldo + r : r * h.ldo + c + e] = x[k][g][e];
            }
        }
    }
}

// How a specialised epilogue stages a 32 x 32 block for its TMA stores: as half of a 64-column
// unit (BF16 only: one 64 x 32 box in place, one 32 x 64 box mirrored), by itself, by itself
// on the diagonal of a symmetric product (one box holding both triangles), or in place only.
// A warp's TMA stores and the waits for them run in one elected lane (the same for a given mask:
// bulk groups belong to the thread that commits them).
constexpr int kStgSlots = 2;                  // 4 KiB staging slots of an epilogue warp
constexpr int kStgBytes = kStgSlots * 4096;

enum StageMode { STAGE_UNIT, STAGE_BLOCK, STAGE_DIAG, STAGE_PLAIN };

// Offsets in the warp's 8 KiB of staging. STAGE_UNIT: the 64-column rows (128-byte swizzle) at 0,
// the mirrored rows at kStgMirror64. Else: in place at 0, mirrored at kStgMirror, the lo parts
// kStgLo further on (64-byte swizzle).
constexpr uint32_t kStgMirror = 2048, kStgLo = 4096, kStgMirror64 = 4096;

// Stage one part (hi or lo) of a block: w[k][g] holds this lane's pair of 8 x 8 block (g, k).
// Four blocks g of one k per stmatrix; the transposing form writes their mirror. half: which 32
// columns of the unit.
template <int MODE>
__device__ __forceinline__ void stage_part(uint32_t (&w)[4][4], uint32_t stg, int half, int lane)
{
    const int g = lane >> 3, j = lane & 7;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        uint32_t da, ma;
        if (MODE == STAGE_UNIT) {
            const int row = 32 * half + 8 * k + j;
            da = stg + lane * 128 + (((4 * half + k) ^ j) << 4);
            ma = stg + kStgMirror64 + row * 64 + ((g ^ ((row >> 1) & 3)) << 4);
        } else {
            const int row = 8 * k + j;
            da = stg + lane * 64 + ((k ^ ((lane >> 1) & 3)) << 4);
            ma = stg + (MODE == STAGE_DIAG ? 0u : kStgMirror) + row * 64 + ((g ^ ((row >> 1) & 3)) << 4);
        }
        if (MODE == STAGE_DIAG) {
            // The block's own lower triangle is not part of the result: its 8 x 8 blocks are
            // the mirrors of those above the diagonal, and the ones on it mirror themselves.
            w[k][k] = mirror_diag(w[k][k], lane);
            const uint32_t dummy = stg + kStgMirror + 16 * j;
            if (g > k)
                da = dummy;
            if (g >= k)
                ma = dummy;
        }
        stmatrix4<false>(da, w[k]);
        if (MODE != STAGE_PLAIN)
            stmatrix4<true>(ma, w[k]);
    }
}

// Value arithmetic and staging of one 32 x 32 block of a specialised product: v = alpha D +
// beta C + gamma I from the accumulator at taddr, rounded to BF16 (and lo parts) in the staging.
//
// The accumulator is read as matrix fragments, so the staging takes 8 stmatrix a part where the
// row-per-thread form took 4 16-byte and 32 two-byte stores and converted every value twice.
template <int S, int MODE>
__device__ __forceinline__ void spec_block(const EpiHot &h, CRaw &cr, uint32_t taddr, int64_t r0,
                                           int64_t c0, uint32_t stg, int half, int lane, double &nrm)
{
    using Spec = EpiSpec<S>;
    float v[2][16];
    tmem_ld_frag32(taddr, v[0]);
    tmem_ld_frag32(taddr + (16u << 16), v[1]);
    tmem_ld_wait();
    const bool edge = h.N - c0 < 32;
    float x[4][4][2];
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            float a = __fmul_rn(v[g >> 1][4 * k + 2 * (g & 1)], h.alpha);
            float b = __fmul_rn(v[g >> 1][4 * k + 2 * (g & 1) + 1], h.alpha);
            if (Spec::has_c) {
                float2 c = bf16x2(cr.word(4 * k + g));
                if (Spec::cpair) {
                    const float2 l = bf16x2(cr.word(16 + 4 * k + g));
                    if (edge) {  // a row that ends in this chunk adds the parts' sum
                        c.x += l.x;
                        c.y += l.y;
                    }
                    a = fmaf(h.beta, c.x, a);
                    b = fmaf(h.beta, c.y, b);
                    if (!edge) {
                        a = fmaf(h.beta, l.x, a);
                        b = fmaf(h.beta, l.y, b);
                    }
                } else {
                    a = fmaf(h.beta, c.x, a);
                    b = fmaf(h.beta, c.y, b);
                }
            }
            if (Spec::c_f32) {
                a = fmaf(h.beta, __uint_as_float(cr.word(2 * (4 * k + g))), a);
                b = fmaf(h.beta, __uint_as_float(cr.word(2 * (4 * k + g) + 1)), b);
            }
            if (MODE == STAGE_DIAG && g == k) {
                const int row = lane >> 2, col = 2 * (lane & 3);
                if (Spec::norm && h.diag) {
                    const int64_t r = r0 + 8 * g + row;
                    if ((row >> 1) == (col >> 1) && r < h.M) {  // this lane holds (r, r)
                        const float d = (float)(h.diag[r] * h.dss[0] - h.dss[1]);
                        if (row == col)
                            a = d;
                        else
                            b = d;
                    }
                } else {
                    if (row == col)
                        a += h.gamma;
                    if (row == col + 1)
                        b += h.gamma;
                }
            }
            x[k][g][0] = a;
            x[k][g][1] = b;
        }
    if (Spec::norm)
        norm_block<Spec::sym>(h, x, r0, c0, lane, nrm);
    if constexpr (Spec::f32_out) {
        store_frag_f32(h, x, r0, c0, lane);
    } else {
        uint32_t w[4][4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                const __nv_bfloat162 h2 = __floats2bfloat162_rn(x[k][g][0], x[k][g][1]);
                w[k][g] = *reinterpret_cast<const uint32_t *>(&h2);
                if (Spec::pair) {
                    x[k][g][0] -= __low2float(h2);
                    x[k][g][1] -= __high2float(h2);
                }
            }
        stage_part<MODE>(w, stg, half, lane);
        if (Spec::pair) {
#pragma unroll
            for (int k = 0; k < 4; ++k)
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                    const __nv_bfloat162 l2 = __floats2bfloat162_rn(x[k][g][0], x[k][g][1]);
                    w[k][g] = *reinterpret_cast<const uint32_t *>(&l2);
                }
            stage_part<MODE>(w, stg + kStgLo, half, lane);
        }
    }
}

// The C fragments of a specialised product's block.
template <int S>
__device__ __forceinline__ void spec_c_load(const EpiHot &h, int64_t r0, int64_t c0, int lane, CRaw &cr)
{
    if (EpiSpec<S>::has_c)
        c_load_frag<EpiSpec<S>::cpair>(h, r0, c0, lane, cr);
    else if (EpiSpec<S>::c_f32)
        c_load_frag_f32(h, r0, c0, lane, cr);
}

// Load the epilogue fields of problem P (with the per-call fields of a grouped or
// fused launch) into registers.
__device__ __forceinline__ void load_hot(EpiHot &h, const TcProblem &P, const CallRec *calls,
                                         const EpiScales &sc)
{
    const Epi &e = P.ep;
    h.c0 = e.c0;
    h.c1 = e.c1;
    h.ldc = e.ldc;
    h.o0 = e.o0;
    h.o1 = e.o1;
    h.ldo = e.ldo;
    h.t0 = e.t0;
    h.t1 = e.t1;
    h.ldt = e.ldt;
    h.maps = &P.mapO[0];
    h.norm_acc = e.norm_acc;
    h.diag = e.diag;
    h.dss = e.dss;
    h.M = P.M;
    h.N = P.N;
    h.sym = P.sym;
    h.otma = P.o_tma;
    h.ttma = P.t_tma;
    h.wide_tma = P.u_tma;
    h.c_kind = e.c_kind;
    h.c_trans = e.c_trans;
    h.o_kind = e.o_kind;
    h.o_trans = e.o_trans;
    h.t_kind = e.t_kind;
    h.f0 = e.f0;
    h.ldf = e.ldf;
    h.fscale = e.fscale;
    if (P.patch) {  // grouped / fused launch: per-call fields
        const CallRec &cr = calls[P.call_idx];
        if (P.patch & PT_C_IS_A) {
            h.c0 = cr.A;
            h.ldc = cr.lda;
        }
        if (P.patch & PT_O_IS_Y) {
            h.o0 = cr.Y;
            h.ldo = cr.ldy;
            h.otma = 0;
        }
    }
    h.alpha = sc.alpha;
    h.beta = sc.beta;
    h.gamma = sc.gamma;
}

// --------------------------------------------------------------- kernel

constexpr int kRingTiles = 4;  // fused launches: tiles in flight between the roles

// A tile handed from the scheduler to the other roles (and to the peer CTA of a pair), with its
// epilogue's scales and what the producer and the MMA issuer would otherwise load from the
// problem table between two tiles.
struct RingTile {
    int kblocks;  // of a segment (-1: no more tiles)
    int prob;     // -1: nothing to compute
    int tm, tn;
    float alpha, beta, gamma;
    int geom;  // see pack_geom
};

constexpr int kMaxMaps = 2;  // tensor maps of an operand: hi and lo part

// k-blocks of a segment: one is a 128-byte swizzle row, 64 BF16 or 128 e4m3 elements. (K up to
// 2^30: no field of a packed word.)
__device__ __forceinline__ int seg_kblocks(const TcProblem &P)
{
    const int kshift = P.fp8 ? 7 : 6;
    return (P.K + (1 << kshift) - 1) >> kshift;
}

// Segments in bits 0..1, their L and R parts in 2..4 and 5..7, e4m3 operands in 8, "the operands'
// dependencies are met" in 9.
constexpr int kGeomReady = 1 << 9;
__device__ __forceinline__ int pack_geom(const TcProblem &P)
{
    int g = P.nseg | (P.fp8 ? 1 << 8 : 0);
#pragma unroll
    for (int k = 0; k < 3; ++k)
        g |= P.segL[k] << (2 + k) | P.segR[k] << (5 + k);
    return g;
}
__device__ __forceinline__ int geom_segs(int g) { return g & 3; }
__device__ __forceinline__ int geom_l(int g, int sg) { return (g >> (2 + sg)) & 1; }
__device__ __forceinline__ int geom_r(int g, int sg) { return (g >> (5 + sg)) & 1; }
__device__ __forceinline__ bool geom_fp8(int g) { return (g >> 8) & 1; }

// k-blocks per pipeline slot (one pair of barriers). With 128 x 64 tiles a k-block's four MMAs take
// 134 cycles, while the waits, the vote and the branches of one round of the producer's and of the
// issuer's loop took some 350 and 400 cycles, whatever the tile: slots of two k-blocks halve that
// (420 -> 311 cycles a k-block with the inlined waits of wait_warp; 1000 x 1001 709 -> 689 us). The
// larger tiles have 269 cycles or more of MMAs a k-block, and lose more by waiting for the first two
// k-blocks than they gain (2048 x 1024 FP32 on 256 x 128: 1218 us with one, 1245 with two).
template <int BN, int STAGES>
constexpr int kGroup = BN == 64 && STAGES % 2 == 0 ? 2 : 1;

// k-blocks in the next slot when `left` remain: an odd one comes first, alone, so that the first
// MMAs wait for less.
template <int GROUP>
__device__ __forceinline__ int slot_blocks(int left)
{
    return GROUP == 1 ? 1 : 2 - (left & 1);
}

template <int BN, int STAGES, bool CHAIN, bool PAIR, bool STRIPS>
__global__ void __launch_bounds__(kThreads, 1) tc_gemm_kernel(const __grid_constant__ TcLaunch L)
{
    static_assert(!STRIPS || CHAIN, "strip dependencies exist in fused launches only");
    static_assert(!PAIR || BN == 256 || BN == 128, "CTA pairs compute 256 x 256 or 256 x 128 tiles");
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                ~static_cast<uintptr_t>(1023));
    constexpr int A_BYTES = kBM * kBK * 2;
    constexpr int B_ROWS = PAIR ? BN / 2 : BN;  // rows of R this CTA stages per k-block
    constexpr int B_BYTES = B_ROWS * kBK * 2;
    constexpr int TILE_ROWS = PAIR ? 2 * kBM : kBM;
    constexpr int GROUP = kGroup<BN, STAGES>, SLOTS = STAGES / GROUP;
    static_assert(STAGES % GROUP == 0, "whole slots");
    uint8_t *sA = smem;
    uint8_t *sB = smem + STAGES * A_BYTES;
    uint8_t *stage_all = sB + STAGES * B_BYTES;  // 1024-aligned
    uint64_t *full = reinterpret_cast<uint64_t *>(stage_all + kEpiWarps * kStgBytes);
    uint64_t *empty = full + SLOTS;
    uint64_t *tfull = empty + SLOTS;
    uint64_t *tempty = tfull + 2;
    uint64_t *drain = tempty + 2;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(drain + 1);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
    int *skip_flag = reinterpret_cast<int *>(tmem_slot + 2);
    // Fused launches: the ring of tiles from the scheduler to the other roles; pdone[i]: the
    // epilogue warps' parts of the tile in entry i are in global memory; ptaken: the producer's
    // latest tile can start.
    uint64_t *rfull = reinterpret_cast<uint64_t *>(
        (reinterpret_cast<uintptr_t>(tmem_slot + 3) + 7) & ~static_cast<uintptr_t>(7));
    uint64_t *rempty = rfull + kRingTiles;
    uint64_t *pdone = rempty + kRingTiles;
    uint64_t *ptaken = pdone + kRingTiles;
    volatile RingTile *ring = reinterpret_cast<volatile RingTile *>(
        (reinterpret_cast<uintptr_t>(ptaken + 1) + 15) & ~static_cast<uintptr_t>(15));
    const CallRec *calls = L.calls ? L.calls : &L.call_inline;

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    int *status0 = L.shared ? nullptr : prob_at(L, 0).ep.status;  // of the solve (shared: of none)
    // CTA pairs: rank 0 (leader) issues the MMAs and hands out tile ids.
    const uint32_t rank = PAIR ? cluster_rank() : 0u;
    const bool leader = rank == 0;

    if (threadIdx.x == 0) {
        for (int s = 0; s < SLOTS; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&tfull[b], 1);
            // Pairs: one release per epilogue warp of both CTAs, on the leader's barrier.
            mbar_init(&tempty[b], PAIR ? 2 * kEpiWarps : 32 * kEpiWarps);
        }
        mbar_init(drain, 1);
        for (int i = 0; i < kRingTiles; ++i) {
            mbar_init(&rfull[i], 1);
            // Consumers of a ring entry: producer, MMA issuer, epilogue warps and publisher;
            // for pairs also the peer's (which issues no MMAs).
            mbar_init(&rempty[i], PAIR ? 2 * (2 + kEpiWarps) + 1 : 3 + kEpiWarps);
            mbar_init(&pdone[i], kEpiWarps);
        }
        mbar_init(ptaken, 1);
        *abort_flag = 0;
        // A solve whose earlier launch already timed out does no further work.
        *skip_flag = (status0 && *reinterpret_cast<volatile int *>(status0) == (int)SVT_ERR_TIMEOUT);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (PAIR) {
        // The peer's barriers exist before either CTA signals them.
        __syncthreads();
        cluster_sync_all();
    }
    if (warp == 1) {
        tmem_alloc<PAIR>(tmem_slot, 2 * BN);
        tmem_relinquish<PAIR>();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    const int total = *skip_flag ? 0
                                 : (L.gtab ? (L.tile_hi > 0 ? L.tile_hi : L.gstart[L.gcount])
                                           : L.tile_start[L.nprob]);
    // Static schedule (non-fused launches): CTA (pair) i takes tiles i, i + grid, ...
    const int t_first = PAIR ? (int)(blockIdx.x >> 1) : (int)blockIdx.x;
    const int t_step = PAIR ? (int)(gridDim.x >> 1) : (int)gridDim.x;

    // Take over ring entry ri: wait for it, read it, and release it at once (`keep`: the
    // caller releases it later).
    auto ring_release = [&](int ri) {
        if (PAIR && !leader)
            mbar_arrive_remote(peer_addr(&rempty[ri], 0));
        else
            mbar_arrive(&rempty[ri]);
    };
    if (warp == kSchedWarp) {
        // ------------------------------------------------ tile scheduler (fused launches)
        // Takes tiles in table order, one ahead of the one the producer is loading, so that the
        // counter's round trip, the decoding, the tensor maps' and problem fields' fetches and
        // the dependency check of a tile run beside the copies of the tile before it (in the
        // producer they cost 2200 cycles between tiles). With the publisher: 256-matrix batch
        // 10.03 -> 8.68 ms, single solves 1 to 2 % faster. The whole warp works on one tile.
        if (CHAIN && (!PAIR || leader)) {
            int ri = 0, prob = 0, start = 0;
            uint32_t rphase = 0, taken = 0;
            int dep_prob = -1;  // problem whose whole dependencies have been waited for
            bool src_done[2] = {false, false};  // lane 0: its strip dependencies that are complete
            for (bool first = true;; first = false) {
                if (!first) {
                    if (!wait_warp<false>(ptaken, taken, abort_flag, status0, kWaitTimeoutNs))
                        break;
                    taken ^= 1u;
                }
                if (!wait_warp<PAIR>(&rempty[ri], rphase ^ 1u, abort_flag, status0, kWaitTimeoutNs))
                    break;
                int t = 0;
                if (lane == 0)
                    t = L.tile_lo + atomicAdd(L.tile_counter, 1);
                t = __shfl_sync(0xffffffffu, t, 0);
                if (t >= total)
                    t = -1;
                TileCoord tc{-1, 0, 0, false};
                if (t >= 0) {
                    find_problem(L, t, lane, prob, start);
                    tc = tile_coord<BN, TILE_ROWS, STRIPS>(L.gtab[prob], prob, t - start);
                }
                EpiScales sc{1.f, 0.f, 0.f};
                int geom = 0, kblocks = 0;
                bool ok = true;
                if (tc.valid) {
                    const TcProblem &P = L.gtab[tc.prob];
                    // The fields that the other roles read, into L1, and the tensor maps into the
                    // descriptor cache.
                    const char *pb = reinterpret_cast<const char *>(&P.o_tma);
                    constexpr int nlines =
                        (int)((sizeof(TcProblem) - offsetof(TcProblem, o_tma) + 127) / 128) + 1;
                    static_assert(nlines <= 32 && kMaxMaps <= 32, "one prefetch a lane");
                    if (lane < nlines)
                        asm volatile("prefetch.L1 [%0];" ::"l"(pb + 128 * lane));
                    if (lane < (P.nseg > 1 ? kMaxMaps : 1)) {  // hi, then lo parts
                        prefetch_tensormap(&P.mapL[lane]);
                        prefetch_tensormap(&P.mapR[lane]);
                    }
                    geom = pack_geom(P);
                    kblocks = seg_kblocks(P);
                    // Operands are results of earlier problems. Strip launches wait here until
                    // the strips this tile reads are complete (L: the strip of this tile's row,
                    // R: of its column), and so do tiles whose scales come from a norm. Other
                    // tiles are handed on; where their dependencies are not met yet the producer
                    // waits itself, which leaves no hand-over between the last counter and the
                    // first copy.
                    bool ready = true;
                    if (STRIPS || P.ep.theta_src) {
                        if (lane == 0) {
                            if (!STRIPS || tc.prob != dep_prob)  // strips: once per problem, counts only grow
                                for (int d = 0; d < 2 && ok; ++d)
                                    if (P.dep[d] >= 0)
                                        ok = wait_counter(&L.done[P.dep[d]], P.dep_target[d],
                                                          abort_flag, status0, dep_limit(L));
                            if (STRIPS) {
                                if (tc.prob != dep_prob) {
                                    src_done[0] = !P.sdep_mode[0];
                                    src_done[1] = !P.sdep_mode[1];
                                }
                                for (int q = 0; q < 2 && ok; ++q)
                                    if (!src_done[q])
                                        ok = wait_strip(L, P, q, q ? tc.tn : tc.tm, src_done[q],
                                                        abort_flag, status0);
                                if (P.ep.theta_src)  // the norm its scales come from is complete
                                    for (int d = 0; d < P.nwdep && ok; ++d)
                                        ok = wait_counter(&L.done[P.wdep[d]], P.wdep_target[d],
                                                          abort_flag, status0, dep_limit(L));
                            }
                        }
                        dep_prob = tc.prob;
                        ok = __shfl_sync(0xffffffffu, (int)ok, 0);
                    } else if (tc.prob != dep_prob) {  // met once, met for every later tile
                        const int d = lane < 2 ? P.dep[lane] : -1;
                        ready = __all_sync(0xffffffffu,
                                           d < 0 || ld_acquire_gpu(&L.done[d]) >= P.dep_target[lane & 1]);
                        if (ready)
                            dep_prob = tc.prob;
                    }
                    __syncwarp();  // the lanes' acquires come before what follows in the others
                    if (ready)
                        geom |= kGeomReady;
                    if (ok) {
                        sc = epi_scales(P, calls);
                        fence_async_global();  // the TMA reads of the tile come after the acquire
                    }
                }
                if (!ok) {  // the wait gave up: end the ring, also for the peer CTA
                    t = -1;
                    tc.valid = false;
                }
                const int ent[8] = {t < 0 ? -1 : kblocks, tc.valid ? tc.prob : -1, tc.tm, tc.tn,
                                    __float_as_int(sc.alpha), __float_as_int(sc.beta),
                                    __float_as_int(sc.gamma), geom};
                int word = ent[0];  // lane k < 8 writes word k
#pragma unroll
                for (int q = 1; q < 8; ++q)
                    word = lane == q ? ent[q] : word;
                if (lane < 8) {
                    reinterpret_cast<volatile int *>(&ring[ri])[lane] = word;
                    if (PAIR)
                        st_remote_u32(peer_addr((const void *)&ring[ri], 1) + 4 * lane, word);
                }
                __syncwarp();
                if (elect_one()) {
                    if (PAIR)
                        mbar_arrive_remote(peer_addr(&rfull[ri], 1));
                    mbar_arrive(&rfull[ri]);
                }
                __syncwarp();
                if (++ri == kRingTiles) {
                    ri = 0;
                    rphase ^= 1u;
                }
                if (t < 0)
                    break;
            }
        }
    } else if (warp == kPubWarp && lane == 0) {
        // ------------------------------------------------ publisher (fused launches)
        // Releases a tile's results to the tiles that read them: once every epilogue warp's
        // stores are complete, one GPU-scope fence (cumulative over what the warps released to
        // this thread) and the increment of the problem's counter. The fence takes 1700 to 2200
        // cycles, which the epilogue warps, each fencing for itself, spent between tiles.
        if (CHAIN) {
            int ri = 0;
            uint32_t rphase = 0, par = 0;  // bit i: parity of pdone[i]'s next use
            for (;;) {
                if (!wait_bar<PAIR>(&rfull[ri], rphase, abort_flag, status0, kWaitTimeoutNs))
                    break;
                const int kblocks = ring[ri].kblocks, prob = ring[ri].prob, tm = ring[ri].tm, tn = ring[ri].tn;
                if (prob >= 0) {
                    const TcProblem &P = prob_at(L, prob);
                    const int pid = P.pid;
                    if (!mbar_wait(&pdone[ri], (par >> ri) & 1u, abort_flag, status0, kWaitTimeoutNs))
                        break;
                    par ^= 1u << ri;
                    fence_async_global();
                    asm volatile("fence.acq_rel.gpu;" ::: "memory");
                    red_add_relaxed(&L.done[pid], kEpiWarps);
                    if (STRIPS && P.strip_base >= 0) {  // the strips this tile completes a part of
                        int *sp = L.strips + P.strip_base;
                        red_add_relaxed(sp + tm, kEpiWarps);
                        if (!P.sym)
                            red_add_relaxed(sp + P.tiles_m + tn, kEpiWarps);
                        else if (tn != tm)
                            red_add_relaxed(sp + tn, kEpiWarps);
                    }
                }
                // Released only now: entry ri, and with it pdone[ri], comes round again after this.
                ring_release(ri);
                if (++ri == kRingTiles) {
                    ri = 0;
                    rphase ^= 1u;
                }
                if (kblocks < 0)
                    break;
            }
        }
    } else if (warp == 0) {
        // ------------------------------------------------ TMA producer
        int stage = 0;
        uint32_t phase = 0;
        uint32_t issued = 0, issued_parity = 0;  // bit s: stage s loaded / parity of its last load
        bool ok = true;
        int ri = 0;
        uint32_t rphase = 0;
        for (int t = t_first; ok; t += t_step) {
            TileCoord tc;
            int geom = 0, kblocks = 0;
            if (CHAIN) {
                if (!wait_warp<PAIR>(&rfull[ri], rphase, abort_flag, status0, kWaitTimeoutNs))
                    break;
                kblocks = warp_uniform(ring[ri].kblocks);
                tc.prob = warp_uniform(ring[ri].prob);
                tc.tm = warp_uniform(ring[ri].tm);
                tc.tn = warp_uniform(ring[ri].tn);
                tc.valid = tc.prob >= 0;
                geom = warp_uniform(ring[ri].geom);
                __syncwarp();
                if (elect_one())
                    ring_release(ri);
                if (++ri == kRingTiles) {
                    ri = 0;
                    rphase ^= 1u;
                }
                // The scheduler takes the next tile once this one can start: a CTA holding two
                // tiles that wait would keep work from CTAs that are idle.
                if (kblocks < 0)
                    break;
                if (!tc.valid && (!PAIR || leader) && elect_one())
                    mbar_arrive(ptaken);
            } else {
                if (t >= total)
                    break;
                tc = decode_tile<BN, TILE_ROWS, STRIPS>(L, t);
            }
            if (!tc.valid)
                continue;
            const TcProblem &P = prob_at(L, tc.prob);
            if (!CHAIN) {
                geom = pack_geom(P);
                kblocks = seg_kblocks(P);
            }
            const int kshift = geom_fp8(geom) ? 7 : 6;
            const int row0 = (PAIR ? 2 * tc.tm + (int)rank : tc.tm) * kBM;
            const int col0 = tc.tn * BN + (int)rank * B_ROWS;
            if (CHAIN) {
                if (!(geom & kGeomReady)) {
                    if (lane == 0)
                        for (int d = 0; d < 2 && ok; ++d)
                            if (P.dep[d] >= 0)
                                ok = wait_counter(&L.done[P.dep[d]], P.dep_target[d], abort_flag,
                                                  status0, dep_limit(L));
                    ok = __shfl_sync(0xffffffffu, (int)ok, 0);
                    // Lane 0's acquire comes before the copies of whichever lane is elected: a
                    // shuffle does not order memory.
                    __syncwarp();
                }
                if (!ok)
                    break;
                if ((!PAIR || leader) && elect_one())
                    mbar_arrive(ptaken);
                fence_async_global();  // the TMA reads below come after the acquire
            }
            for (int sg = 0; sg < geom_segs(geom) && ok; ++sg) {
                const CUtensorMap *mL = &P.mapL[geom_l(geom, sg)];
                const CUtensorMap *mR = &P.mapR[geom_r(geom, sg)];
                for (int kb = 0, count; kb < kblocks; kb += count) {
                    if (!wait_warp<PAIR>(&empty[stage], phase ^ 1u, abort_flag, status0, kWaitTimeoutNs)) {
                        ok = false;
                        break;
                    }
                    count = slot_blocks<GROUP>(kblocks - kb);
                    if (elect_one()) {
                        // Both CTAs' bytes of a pair complete on the leader's barrier.
                        const uint32_t fb = PAIR ? peer_addr(&full[stage], 0) : 0u;
                        if (!PAIR || leader)
                            mbar_expect_tx(&full[stage], (uint32_t)((PAIR ? 2 : 1) * (A_BYTES + B_BYTES) * count));
#pragma unroll
                        for (int j = 0; j < GROUP; ++j) {
                            if (j >= count)
                                break;
                            const int x = (kb + j) << kshift;
                            uint8_t *a = sA + (stage * GROUP + j) * A_BYTES;
                            uint8_t *b = sB + (stage * GROUP + j) * B_BYTES;
                            if (PAIR) {
                                tma_load_2d_pair(a, mL, x, row0, fb);
                                tma_load_2d_pair(b, mR, x, col0, fb);
                            } else {
                                tma_load_2d(a, mL, x, row0, &full[stage]);
                                tma_load_2d(b, mR, x, col0, &full[stage]);
                            }
                        }
                    }
                    issued |= 1u << stage;
                    issued_parity = (issued_parity & ~(1u << stage)) | (phase << stage);
                    if (++stage == SLOTS) {
                        stage = 0;
                        phase ^= 1u;
                    }
                }
            }
        }
        // Drain: the last copy into every stage must have landed before exit. The
        // peer of a pair sees its copies land through the leader's MMA consuming them.
        for (int s = 0; s < SLOTS; ++s)
            if ((issued >> s) & 1u) {
                volatile int no_abort = 0;
                if (!PAIR || leader)
                    mbar_wait(&full[s], (issued_parity >> s) & 1u, &no_abort, nullptr, kWaitTimeoutNs / 4);
                else
                    mbar_wait_cluster(&empty[s], (issued_parity >> s) & 1u, &no_abort, nullptr,
                                      kWaitTimeoutNs / 4);
            }
    } else if (warp == 1 && (!PAIR || leader)) {
        // ------------------------------------------------ MMA issuer
        // The whole warp runs the loop and one elected lane issues: its operands then live in
        // uniform registers. A loop that only lane 0 ran took 132 cycles an MMA whatever its
        // shape, twice what a 128 x 128 x 16 needs.
        const uint64_t desc_a = sw128_desc(smem_u32(sA)), desc_b = sw128_desc(smem_u32(sB));
        int stage = 0;
        uint32_t phase = 0;
        int buf = 0;
        uint32_t tphase = 0;
        bool ok = true;
        int ri = 0;
        uint32_t rphase = 0;
        for (int t = t_first; ok; t += t_step) {
            TileCoord tc;
            int geom = 0, kblocks = 0;
            if (CHAIN) {
                if (!wait_warp<false>(&rfull[ri], rphase, abort_flag, status0, kWaitTimeoutNs))
                    break;
                kblocks = warp_uniform(ring[ri].kblocks);
                tc.prob = warp_uniform(ring[ri].prob);
                tc.tm = warp_uniform(ring[ri].tm);
                tc.tn = warp_uniform(ring[ri].tn);
                tc.valid = tc.prob >= 0;
                geom = warp_uniform(ring[ri].geom);
                __syncwarp();
                if (elect_one())
                    ring_release(ri);
                if (++ri == kRingTiles) {
                    ri = 0;
                    rphase ^= 1u;
                }
                if (kblocks < 0)
                    break;
            } else {
                if (t >= total)
                    break;
                tc = decode_tile<BN, TILE_ROWS, STRIPS>(L, t);
                if (tc.valid) {
                    geom = pack_geom(prob_at(L, tc.prob));
                    kblocks = seg_kblocks(prob_at(L, tc.prob));
                }
            }
            if (!tc.valid)
                continue;
            if (!wait_warp<PAIR>(&tempty[buf], tphase ^ 1u, abort_flag, status0, kWaitTimeoutNs))
                break;
            tc_fence_after();
            const uint32_t d_tmem = tmem_base + (uint32_t)(buf * BN);
            // The tile's k-loop, one copy per operand kind chosen once per tile, so that
            // the BF16 loop carries no test of the kind: for each segment and slot of
            // GROUP k-blocks, wait for its copies, issue four MMAs over the 128 bytes of
            // each k-block's rows (K = 16 BF16 or 32 e4m3 elements each) and release the slot.
            auto k_loop = [&](auto f8_tag) -> bool {
                constexpr bool F8 = decltype(f8_tag)::value;
                constexpr uint32_t id = F8 ? idesc_e4m3(TILE_ROWS, BN) : idesc_bf16(TILE_ROWS, BN);
                const int segs = geom_segs(geom);
                uint32_t acc = 0;
                for (int sg = 0; sg < segs; ++sg) {
                    for (int left = kblocks, count; left > 0; left -= count) {
                        count = slot_blocks<GROUP>(left);
                        if (!wait_warp<false>(&full[stage], phase, abort_flag, status0, kWaitTimeoutNs))
                            return false;
                        tc_fence_after();
                        if (elect_one()) {
#pragma unroll
                            for (int j = 0; j < GROUP; ++j) {
                                if (j >= count)
                                    break;
                                // Descriptor addresses count 16-byte units; a K step is 32 bytes.
                                const uint64_t a0 = desc_a + (uint32_t)((stage * GROUP + j) * (A_BYTES >> 4));
                                const uint64_t b0 = desc_b + (uint32_t)((stage * GROUP + j) * (B_BYTES >> 4));
#pragma unroll
                                for (int kk = 0; kk < kBK / 16; ++kk) {
                                    const uint64_t ad = a0 + 2 * kk, bd = b0 + 2 * kk;
                                    const uint32_t on = j + kk == 0 ? acc : 1u;
                                    if (F8) {
                                        if (PAIR)
                                            mma_e4m3_pair(d_tmem, ad, bd, id, on);
                                        else
                                            mma_e4m3(d_tmem, ad, bd, id, on);
                                    } else {
                                        if (PAIR)
                                            mma_bf16_pair(d_tmem, ad, bd, id, on);
                                        else
                                            mma_bf16(d_tmem, ad, bd, id, on);
                                    }
                                }
                            }
                            if (PAIR)
                                mma_commit_both(&empty[stage]);
                            else
                                mma_commit(&empty[stage]);
                        }
                        __syncwarp();
                        acc = 1;
                        if (++stage == SLOTS) {
                            stage = 0;
                            phase ^= 1u;
                        }
                    }
                }
                return true;
            };
            ok = geom_fp8(geom) ? k_loop(BoolTag<true>{}) : k_loop(BoolTag<false>{});
            if (!ok)
                break;
            if (elect_one()) {
                if (PAIR)
                    mma_commit_both(&tfull[buf]);
                else
                    mma_commit(&tfull[buf]);
            }
            __syncwarp();
            if (++buf == 2) {
                buf = 0;
                tphase ^= 1u;
            }
        }
        // Drain: every MMA issued so far completes before tensor memory is freed.
        if (elect_one()) {
            if (PAIR)
                mma_commit_pair_local(drain);
            else
                mma_commit(drain);
        }
        __syncwarp();
        volatile int no_abort = 0;
        mbar_wait(drain, 0, &no_abort, nullptr, kWaitTimeoutNs / 4);
    } else if (warp >= 2 && warp < kSchedWarp) {
        // ------------------------------------------------ epilogue
        const int quad = warp & 3;  // TMEM lane quadrant this warp may access
        const int half = (warp - 2) >> 2;  // two warps per quadrant split the column chunks
        uint8_t *stage_buf = stage_all + (warp - 2) * kStgBytes;
        int slot = 0;  // next staging slot of this warp
        int buf = 0;
        uint32_t tphase = 0;
        int last_prob = -1;
        bool c_done = true;
        int ri = 0;
        uint32_t rphase = 0;
        for (int t = t_first;; t += t_step) {
            TileCoord tc;
            EpiScales sc;
            int entry = 0;  // the tile's ring entry
            if (CHAIN) {
                if (!wait_bar<PAIR>(&rfull[ri], rphase, abort_flag, status0, kWaitTimeoutNs))
                    break;
                const bool end = ring[ri].kblocks < 0;
                tc.prob = ring[ri].prob;
                tc.tm = ring[ri].tm;
                tc.tn = ring[ri].tn;
                tc.valid = tc.prob >= 0;
                sc = EpiScales{ring[ri].alpha, ring[ri].beta, ring[ri].gamma};
                entry = ri;
                __syncwarp();
                if (lane == 0)
                    ring_release(ri);
                if (++ri == kRingTiles) {
                    ri = 0;
                    rphase ^= 1u;
                }
                if (end)
                    break;
            } else {
                if (t >= total)
                    break;
                tc = decode_tile<BN, TILE_ROWS, STRIPS>(L, t);
            }
            if (!tc.valid)
                continue;
            const TcProblem &P = prob_at(L, tc.prob);
            if (CHAIN && !STRIPS && P.ep.c_kind != C_NONE) {
                // C is an earlier result: make it visible to these loads.
                for (int d = 0; d < 2; ++d)
                    if (P.dep[d] >= 0 && lane == 0)
                        wait_counter(&L.done[P.dep[d]], P.dep_target[d], abort_flag, status0,
                                     dep_limit(L));
                __syncwarp();
            }
            if (STRIPS) {
                // C is an earlier result: make it visible to these loads; earlier readers of the
                // buffers this tile overwrites must be done.
                if (lane == 0) {
                    if (tc.prob != last_prob) {  // once per problem: counts only grow
                        if (P.ep.c_kind != C_NONE)
                            for (int d = 0; d < 2; ++d)
                                if (P.dep[d] >= 0)
                                    wait_counter(&L.done[P.dep[d]], P.dep_target[d], abort_flag,
                                                 status0, dep_limit(L));
                        for (int d = 0; d < P.nwdep; ++d)
                            wait_counter(&L.done[P.wdep[d]], P.wdep_target[d], abort_flag,
                                         status0, dep_limit(L));
                        c_done = !P.sdep_mode[2];
                    }
                    if (!c_done)
                        wait_strip(L, P, 2, tc.tm, c_done, abort_flag, status0);
                }
                __syncwarp();
            }
            if (PAIR)
                tc.tm = 2 * tc.tm + (int)rank;  // this CTA's 128-row half of the tile
            EpiHot h;  // per tile: its registers are free outside the tile's loops
            if (!CHAIN)
                sc = epi_scales(P, calls);
            load_hot(h, P, calls, sc);
            const int spec = epi_spec(h);
            last_prob = tc.prob;
            const int64_t warp_row0 = (int64_t)tc.tm * kBM + quad * 32;
            const int64_t row = warp_row0 + lane;
            const bool row_ok = row < h.M;
            // This warp's 32-column chunks: both of every other 64-column unit (of a single unit,
            // one), skipping chunks right of N or wholly below the diagonal (warp-uniform).
            auto step = [](int ch) { return BN == 64 ? 2 : ((ch & 1) ? 3 : 1); };
            auto next_chunk = [&](int ch) {
                for (; ch < BN / 32; ch += step(ch)) {
                    const int64_t c0 = (int64_t)tc.tn * BN + ch * 32;
                    if (c0 < h.N && warp_row0 < h.M && !(h.sym && warp_row0 > c0 + 31))
                        break;
                }
                return ch;
            };
            auto after = [&](int ch) { return next_chunk(ch + step(ch)); };
            auto full_row = [&](int ch) {
                return row_ok && (int64_t)h.N - ((int64_t)tc.tn * BN + ch * 32) >= 32;
            };
            int ch = next_chunk(BN == 64 ? half : 2 * half);
            // The first chunk's C is loaded while the accumulator is still being computed.
            CRaw cr;
            bool cvec = false;
            if (ch < BN / 32) {
                if (spec == 1)
                    spec_c_load<1>(h, warp_row0, (int64_t)tc.tn * BN + ch * 32, lane, cr);
                else if (spec == 4 || spec == 9)
                    spec_c_load<4>(h, warp_row0, (int64_t)tc.tn * BN + ch * 32, lane, cr);
                else if (spec == 8)
                    spec_c_load<8>(h, warp_row0, (int64_t)tc.tn * BN + ch * 32, lane, cr);
                else if (spec < 0)
                    cvec = c_load(h, row, (int64_t)tc.tn * BN + ch * 32, full_row(ch), cr);
            }
            if (!wait_bar<PAIR>(&tfull[buf], tphase, abort_flag, status0, kWaitTimeoutNs))
                break;
            tc_fence_after();
            double nrm = 0.0;
            const uint32_t acc0 = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(buf * BN);
            // The chunk loop, one copy per product kind (epi_spec, chosen once per tile):
            // the specialised copies carry no tests of output, C, norm and copy kinds.
            auto chunk_loop = [&](auto spec_tag) {
                using Spec = decltype(spec_tag);
#pragma unroll 1
                while (ch < BN / 32) {
                    const int nx = after(ch);
                    const int64_t c0 = (int64_t)tc.tn * BN + ch * 32;
                    if constexpr (Spec::generic) {
                        const int64_t rem = (int64_t)h.N - c0;
                        float v[32];
                        tmem_ld32(acc0 + (uint32_t)(ch * 32), v);
#pragma unroll
                        for (int i = 0; i < 32; ++i)
                            v[i] *= h.alpha;
                        c_apply(h, cr, cvec, row, c0, rem < 32 ? (int)rem : 32, row_ok, v);
                        // The next chunk's C is in flight while this chunk is stored.
                        if (nx < BN / 32)
                            cvec = c_load(h, row, (int64_t)tc.tn * BN + nx * 32, full_row(nx), cr);
                        epilogue_finish<kStgSlots>(h, warp_row0, c0, v, nrm, stage_buf, slot, lane);
                    } else {
                        constexpr int S = Spec::code;
                        const uint32_t stg = smem_u32(stage_buf);
                        const bool meets = Spec::sym && (c0 & ~(int64_t)63) < warp_row0 + 32;
                        // staged with its neighbour
                        const bool unit = BN > 64 && !Spec::pair && Spec::mirror && !meets;
                        if (!Spec::f32_out && (!unit || !(ch & 1))) {
                            if (elect_one())  // the staging's last stores have been read
                                bulk_wait_read0();
                            __syncwarp();
                        }
                        const bool diag = Spec::sym && c0 == warp_row0;
                        const uint32_t ta = acc0 + (uint32_t)(ch * 32);
                        if constexpr (!Spec::mirror) {
                            spec_block<S, STAGE_PLAIN>(h, cr, ta, warp_row0, c0, stg, 0, lane, nrm);
                        } else if (unit) {
                            if constexpr (BN > 64 && !Spec::pair)
                                spec_block<S, STAGE_UNIT>(h, cr, ta, warp_row0, c0, stg, ch & 1, lane, nrm);
                        } else if (diag) {
                            if constexpr (Spec::sym)
                                spec_block<S, STAGE_DIAG>(h, cr, ta, warp_row0, c0, stg, 0, lane, nrm);
                        } else {
                            spec_block<S, STAGE_BLOCK>(h, cr, ta, warp_row0, c0, stg, 0, lane, nrm);
                        }
                        // The next chunk's C is in flight while this chunk is stored.
                        if (nx < BN / 32)
                            spec_c_load<S>(h, warp_row0, (int64_t)tc.tn * BN + nx * 32, lane, cr);
                        if (!Spec::f32_out && (!unit || (nx >> 1) != (ch >> 1))) {
                            // a block, or a unit's last chunk
                            fence_async_smem();
                            __syncwarp();
                            if (elect_one()) {
                                const int x = unit ? (int)(c0 & ~(int64_t)63) : (int)c0, y = (int)warp_row0;
                                const CUtensorMap *m = h.maps;
                                const bool both = Spec::mirror && !diag;
                                if (unit) {
                                    tma_store_2d(&m[1], x, y, stage_buf);  // (u_tma's maps)
                                    tma_store_2d(&m[3], y, x, stage_buf + kStgMirror64);
                                } else {
                                    const CUtensorMap *mm = Spec::sym ? m : m + 2;
                                    tma_store_2d(&m[0], x, y, stage_buf);
                                    if (both)
                                        tma_store_2d(&mm[0], y, x, stage_buf + kStgMirror);
                                    if (Spec::pair) {
                                        tma_store_2d(&m[1], x, y, stage_buf + kStgLo);
                                        if (both)
                                            tma_store_2d(&mm[1], y, x, stage_buf + kStgLo + kStgMirror);
                                    }
                                }
                                bulk_commit();
                            }
                        }
                    }
                    ch = nx;
                }
            };
            if (!CHAIN) {  // the previous tile's stores have read the staging
                if (elect_one())
                    bulk_wait_read0();
                __syncwarp();
            }
            switch (spec) {
            case 0: chunk_loop(EpiSpec<0>{}); break;
            case 1: chunk_loop(EpiSpec<1>{}); break;
            case 2: chunk_loop(EpiSpec<2>{}); break;
            case 3: chunk_loop(EpiSpec<3>{}); break;
            case 4: chunk_loop(EpiSpec<4>{}); break;
            case 5: chunk_loop(EpiSpec<5>{}); break;
            case 6: chunk_loop(EpiSpec<6>{}); break;
            case 7: chunk_loop(EpiSpec<7>{}); break;
            case 8: chunk_loop(EpiSpec<8>{}); break;
            case 9: chunk_loop(EpiSpec<9>{}); break;
            default: chunk_loop(EpiSpec<-1>{}); break;
            }
            if (h.norm_acc) {
#pragma unroll
                for (int o = 16; o > 0; o >>= 1)
                    nrm += __shfl_xor_sync(0xffffffffu, nrm, o);
                if (lane == 0 && nrm != 0.0)
                    atomicAdd(h.norm_acc, nrm);
            }
            tc_fence_before();
            if (PAIR) {
                // One release per warp, on the leader's barrier (it issues the next MMAs).
                __syncwarp();
                if (lane == 0)
                    mbar_arrive_remote(peer_addr(&tempty[buf], 0));
            } else {
                mbar_arrive(&tempty[buf]);
            }
            if (++buf == 2) {
                buf = 0;
                tphase ^= 1u;
            }
            if (CHAIN) {
                // This warp's part of the tile is in global memory: tell the publisher. The
                // lanes' plain stores (diagonal blocks of symmetric products, ragged edges) are
                // ordered before lane 0's arrival by __syncwarp, its TMA stores by their
                // completion.
                __syncwarp();
                if (elect_one()) {
                    bulk_wait_all0();
                    fence_async_global();
                    mbar_arrive(&pdone[entry]);
                }
                __syncwarp();
            }
        }
        // All TMA stores of this warp complete before the CTA may exit.
        if (elect_one())
            bulk_wait_all0();
        __syncwarp();
    }

    tc_fence_before();
    __syncthreads();
    if (PAIR)
        cluster_sync_all();  // neither CTA leaves while its peer may still signal it
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc<PAIR>(tmem_base, 2 * BN);
    }
}

static_assert(offsetof(TcProblem, mapT) == offsetof(TcProblem, mapO) + 2 * sizeof(CUtensorMap),
              "the epilogue addresses mapO and mapT as one array");

template <int BN, int STAGES, bool PAIR>
constexpr int smem_bytes()
{
    return STAGES * (kBM + (PAIR ? BN / 2 : BN)) * kBK * 2 +
           kEpiWarps * kStgBytes /* epilogue staging */ + 1024 /* alignment slack */ +
           512 /* barriers, tile ring */;
}

// One launch of the product kernel over total_tiles tiles (tile-width code's
// tiles: CTA pairs for kBnPair). Persistent: at most one CTA (pair) per SM (pair).
template <int BN, int STAGES, bool CHAIN, bool PAIR, bool STRIPS = false>
cudaError_t launch_kernel(const TcLaunch &l, int total_tiles, int num_sms, cudaStream_t s)
{
    constexpr int smem = smem_bytes<BN, STAGES, PAIR>();
    static_assert(smem <= 232448, "shared memory per CTA");
    auto kern = tc_gemm_kernel<BN, STAGES, CHAIN, PAIR, STRIPS>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess)
        return e;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    int grid = total_tiles < num_sms ? total_tiles : num_sms;
    static int max_pairs = -1;  // pairs that can be resident at once (SMs pair up within a GPC)
    if (PAIR) {
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 2;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        if (max_pairs < 0) {
            cfg.gridDim = dim3((unsigned)(num_sms & ~1), 1, 1);
            int nc = 0;
            if (cudaOccupancyMaxActiveClusters(&nc, kern, &cfg) != cudaSuccess || nc <= 0) {
                cudaGetLastError();
                nc = num_sms / 2;
            }
            max_pairs = nc;
        }
    }
    if (total_tiles <= 0)  // only the attributes and the pair count (before a capture)
        return cudaSuccess;
    if (PAIR) {
        const int cap = std::min(max_pairs, num_sms / 2);  // a caller's SM budget caps it too
        const int pairs = std::max(1, std::min(total_tiles, cap));
        grid = 2 * pairs;
    }
    cfg.gridDim = dim3((unsigned)grid, 1, 1);
    return cudaLaunchKernelEx(&cfg, kern, l);
}

} // namespace

} // namespace svt
