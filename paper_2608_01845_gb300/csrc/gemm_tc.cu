// Dense bf16 GEMM on the 5th-generation tensor cores (tcgen05, sm_103a) with
// the DiT's fused epilogues: C = epilogue(A W^T), A [M, K], W [N, K] bf16,
// fp32 accumulation in tensor memory.
//
// Persistent kernel, one CTA per SM, 6 warps:
//   warp 0      TMA producer: A (128 x 64) and W (256 x 64) tiles into a
//               4-stage shared-memory ring (128-byte swizzle), one mbarrier
//               pair per stage;
//   warp 1      MMA issuer: one thread issues tcgen05.mma 128x256x16 into one
//               of two TMEM accumulators (2 x 256 columns), commits the smem
//               stage back to the producer and the accumulator to the
//               epilogue;
//   warps 2-5   epilogue (epilogue_tile): each warp owns its 32-lane TMEM
//               quarter = 32 rows and works through the tile 64 columns at a
//               time: tcgen05.ld, bias / GELU / gated residual, bf16 into a
//               swizzled shared-memory slab, one TMA store per slab; then
//               release the accumulator so the next tile's MMAs overlap.
// Tiles are visited N-fastest inside groups of N tiles sized so a group's
// slab of W stays in L2 (about 40 MB), so W is read from DRAM about once and
// A once per group.
// Tails: TMA zero-fills rows past M / N and columns past K; the epilogue
// masks rows >= M.  Every mbarrier wait is bounded.
#include "dit_kernels.cuh"
#include "ptx.cuh"

#include <cudaTypedefs.h>

#include <mutex>

namespace wdc {

namespace {

constexpr int BM = 128, BN = 256, BK = 64;
constexpr int kGemmThreads = 192;
constexpr uint32_t A_BYTES = BM * BK * 2;
// Epilogue staging: two slabs of 32 rows x 64 bf16 columns (128-byte rows,
// 128-byte swizzle) per epilogue warp.
constexpr uint32_t SLAB_BYTES = 32 * 128;
constexpr uint32_t STAGING_BYTES = 4 * 2 * SLAB_BYTES;

// One-CTA kernel, tiles of 128 x BNT: as deep a ring as the tile leaves room for.
template <int BNT>
struct GemmCfg {
    static constexpr uint32_t B_BYTES = BNT * BK * 2;
    static constexpr uint32_t STAGE_BYTES = A_BYTES + B_BYTES;
    static constexpr int STAGES = BNT == 256 ? 4 : (BNT == 128 ? 6 : 8);
    static constexpr uint32_t TMEM_COLS = 2 * BNT;
    static constexpr uint32_t IDESC = idesc_bf16(BM, BNT);
    static constexpr size_t SMEM = STAGES * STAGE_BYTES + STAGING_BYTES + 1024 + 256;
    static_assert(SMEM <= 227 * 1024, "shared memory per CTA");
};

// Tensor maps of one problem's epilogue: `out` (kEpiStore, kEpiResid) and
// `res` (kEpiResid) in boxes of 32 rows x 64 columns; for kEpiQKV `out` = Q,
// `res` = K ([heads, L, d], boxes of 32 tokens x 64) and `vt` = V^T
// ([heads, d, L], boxes of 64 x 32 tokens).
struct EpiMaps {
    CUtensorMap out, res, vt;
};

struct GemmArgs {
    int M, N, K;
    int m_tiles, n_tiles, k_blocks;
    int group_n;            // pair kernel: N tiles per raster group
    Epi e;
    unsigned* err;
    // pair kernel, grouped launch: a second problem with the same N and K
    // (its own A, W, M and epilogue) whose tiles follow the first problem's
    int nprob;              // 1 or 2
    int M1, m_pairs1;
    Epi e1;
    // whether each problem's epilogue has its tensor maps (else every row goes
    // through the direct stores of epilogue_chunk)
    int staged, staged1;
};

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
    __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<uint32_t*>(&h);
}
__device__ __forceinline__ float2 unpack_bf16(uint32_t u) {
    __nv_bfloat162 h = *reinterpret_cast<__nv_bfloat162*>(&u);
    return __bfloat1622float2(h);
}

// Epilogue forms; each is its own instantiation of the kernels, so that the
// epilogue's code stays small and without branches on the form.
enum Form { kFormStore = 0, kFormGelu = 1, kFormResid = 2, kFormQKV = 3, kFormUnpatch = 4, kForms = 5 };

// Direct epilogue of 32 consecutive columns col0..col0+31 of one row: the
// unpatchify form, and the rows whose slab cannot be moved by one TMA copy.
template <int FORM>
__device__ __forceinline__ void epilogue_chunk(const Epi& e, int m, int col0, const uint32_t (&r)[32]) {
    float v[32];
    if (e.bias) {
        const float4* b4 = reinterpret_cast<const float4*>(e.bias + col0);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const float4 b = __ldg(b4 + j);
            v[4 * j + 0] = __uint_as_float(r[4 * j + 0]) + b.x;
            v[4 * j + 1] = __uint_as_float(r[4 * j + 1]) + b.y;
            v[4 * j + 2] = __uint_as_float(r[4 * j + 2]) + b.z;
            v[4 * j + 3] = __uint_as_float(r[4 * j + 3]) + b.w;
        }
    } else {
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
    }
    if constexpr (FORM == kFormResid) {
        __nv_bfloat16* out = reinterpret_cast<__nv_bfloat16*>(e.out) + (size_t)m * e.ldo + col0;
        uint4* o4 = reinterpret_cast<uint4*>(out);
        {
            const int rm = e.res_rows > 0 ? m % e.res_rows : m;
            const uint4* r4 = reinterpret_cast<const uint4*>(reinterpret_cast<const __nv_bfloat16*>(e.res) +
                                                             (size_t)rm * e.ldo + col0);
            float g[32];
            if (e.gate) {
                const float4* g4 = reinterpret_cast<const float4*>(e.gate + col0);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const float4 t = __ldg(g4 + j);
                    g[4 * j] = t.x; g[4 * j + 1] = t.y; g[4 * j + 2] = t.z; g[4 * j + 3] = t.w;
                }
            } else {
#pragma unroll
                for (int j = 0; j < 32; ++j) g[j] = 1.0f;
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint4 rr = r4[q];
                const uint32_t w[4] = {rr.x, rr.y, rr.z, rr.w};
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const float2 f = unpack_bf16(w[t]);
                    const int j = 8 * q + 2 * t;
                    v[j] = fmaf(g[j], v[j], f.x);
                    v[j + 1] = fmaf(g[j + 1], v[j + 1], f.y);
                }
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            uint4 w;
            w.x = pack_bf16(v[8 * q + 0], v[8 * q + 1]);
            w.y = pack_bf16(v[8 * q + 2], v[8 * q + 3]);
            w.z = pack_bf16(v[8 * q + 4], v[8 * q + 5]);
            w.w = pack_bf16(v[8 * q + 6], v[8 * q + 7]);
            o4[q] = w;
        }
    } else if constexpr (FORM == kFormQKV) {
        const int which = col0 / e.D, c = col0 % e.D, dd0 = c % e.d;
        int b, tok;
        batch_token(e.row_off + m, e.nb, e.Lc, e.L, b, tok);
        const size_t h = (size_t)b * e.H + c / e.d;
        if (which < 2) {
            __nv_bfloat16* base = reinterpret_cast<__nv_bfloat16*>(which == 0 ? e.q : e.k) +
                                  (h * e.L + tok) * e.d + dd0;
            uint4* o4 = reinterpret_cast<uint4*>(base);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                uint4 w;
                w.x = pack_bf16(v[8 * q + 0], v[8 * q + 1]);
                w.y = pack_bf16(v[8 * q + 2], v[8 * q + 3]);
                w.z = pack_bf16(v[8 * q + 4], v[8 * q + 5]);
                w.w = pack_bf16(v[8 * q + 6], v[8 * q + 7]);
                o4[q] = w;
            }
        } else {
            __half* base = reinterpret_cast<__half*>(e.vt) + (h * e.d + dd0) * e.ldv + tok;
            bool sat = false;
#pragma unroll
            for (int j = 0; j < 32; ++j) base[(size_t)j * e.ldv] = to_vt_half(v[j], sat);
            if (sat && e.err) atomicOr(e.err, kErrVSaturated);
        }
    } else {
        // kEpiUnpatch: fp32 scatter into the latent.  The row's place is worked
        // out once, the column's (c, ph, pw) counts up: element by element both
        // were chains of integer divisions (a 272 x 64 tile took 42 us).
        const int hp = e.Hh / e.p, wp = e.Ww / e.p, Lv = e.F * hp * wp;
        const int b = m / Lv, mm = m - b * Lv;
        const int f = mm / (hp * wp), rem = mm - f * (hp * wp), h2 = rem / wp, w2 = rem - h2 * wp;
        const size_t plane = (size_t)e.F * e.Hh * e.Ww;
        float* row = e.v + (size_t)b * e.C * plane + ((size_t)f * e.Hh + (size_t)h2 * e.p) * e.Ww + (size_t)w2 * e.p;
        if (e.p == 2 && !((uintptr_t)e.v & 7)) {       // pw = 0, 1 side by side
            float* o = row + (size_t)(col0 / 4) * plane;
#pragma unroll
            for (int j = 0; j < 32; j += 2)
                *reinterpret_cast<float2*>(o + (size_t)(j / 4) * plane + (size_t)((j / 2) & 1) * e.Ww) =
                    make_float2(v[j], v[j + 1]);
            return;
        }
        const int pp = e.p * e.p;
        int c = col0 / pp, ph = (col0 - c * pp) / e.p, pw = col0 - c * pp - ph * e.p;
#pragma unroll
        for (int j = 0; j < 32; ++j) {
            row[(size_t)c * plane + (size_t)ph * e.Ww + pw] = v[j];
            if (++pw == e.p) {
                pw = 0;
                if (++ph == e.p) { ph = 0; ++c; }
            }
        }
    }
}

// ---------------------------------------------------------------------------
// Staged epilogue of one warp's 32 rows of a tile, 64 columns at a time.
//
// Written straight from the accumulator with one row per lane, a 16-byte store
// or residual load touches 32 different 128-byte lines, which the load/store
// unit works through one by one, and every chunk waits for its bias and gate
// from L2: 11-16k cycles (clock stamps) a 128 x 256 tile for a plain store,
// 20k with GELU, 20-35k with a gated residual, where the tile's MMAs take 9k
// (K = 1024) to 26k (K = 3072).  Now 3.7k, 8.1k and 8.0k, behind the MMAs from
// K = 1024 on:
//  * the accumulator is read in the 16x256b shape: lane t holds columns
//    2 (t % 4), + 1 of every 8 in rows t / 4 + 8 i, so a lane needs 16 bias
//    and gate values per chunk instead of 64, and they are fetched a chunk (for
//    the first chunk a tile) ahead of their use;
//  * packed to 16 bits those are the 8 x 8 fragments of stmatrix / ldmatrix,
//    which move them to and from a slab of shared memory (32 rows x 64 columns,
//    swizzled like the tensor map's box: no bank conflicts; transposed on the
//    way for V^T);
//  * one TMA store moves the slab; a residual slab comes in by a TMA load,
//    the tile's first two while the tile's MMAs run, and is updated in place;
//  * each form is a kernel of its own: with the forms as branches of one kernel
//    the same epilogue took 14-25k cycles.
// 17776 x 3072 x 3072 with the gated residual: 241 -> 193 us; 6400 x 4096 x
// 1024 with GELU: 83 -> 46 us; 272 x 256 x 256 with the residual: 17 -> 13 us.
// Rows past M and columns past N are clipped by the tensor map.  Slabs
// alternate; one is written again once its store has read it
// (cp.async.bulk.wait_group.read).
struct WarpStage {
    uint8_t* slab;        // [2][SLAB_BYTES]
    uint64_t* rbar;       // [2] residual slab landed
    uint32_t cnt;         // slabs used so far: the next one is cnt & 1, its residual's parity (cnt >> 1) & 1
    uint32_t pending;     // residual slabs requested and not yet awaited (cnt, cnt + 1, ...)
    float2 bias[8], gate[8];   // the next chunk's, columns 8 i + 2 (lane % 4), + 1
};

// Requests the residual of columns col0.. of rows m0.. into slab `cnt`.
__device__ __forceinline__ void request_residual(WarpStage& ws, uint32_t cnt, const CUtensorMap* res, int m0, int col0,
                                                 int lane) {
    if (lane == 0) {
        bulk_wait_read<0>();               // the slab's last store has read it
        mbar_arrive_expect_tx(&ws.rbar[cnt & 1], SLAB_BYTES);
        tma_load_2d(ws.slab + (cnt & 1) * SLAB_BYTES, res, &ws.rbar[cnt & 1], col0, m0);
    }
    ++ws.pending;
}

// Fetches the bias and gate of the chunk at col0.  Columns past `end` (whose
// results are clipped) read the last valid ones: a clamped address, since a
// select on the loaded value would wait for it here.
template <int FORM>
__device__ __forceinline__ void fetch_columns(const float* bias, const float* gate, int col0, int end, WarpStage& ws,
                                              int lane) {
    const int c = col0 + 2 * (lane & 3);
    if (bias) {
#pragma unroll
        for (int i = 0; i < 8; ++i) ws.bias[i] = __ldg(reinterpret_cast<const float2*>(bias + min(c + 8 * i, end - 2)));
    }
    if (FORM == kFormResid && gate) {
#pragma unroll
        for (int i = 0; i < 8; ++i) ws.gate[i] = __ldg(reinterpret_cast<const float2*>(gate + min(c + 8 * i, end - 2)));
    }
}

// Before the tile's accumulator is awaited: its first chunk's columns and its
// first two residual slabs.
template <int FORM>
__device__ __forceinline__ void epilogue_prefetch(const float* bias, const float* gate, int staged,
                                                  const CUtensorMap* res, int M, int n0, int end, int m0, WarpStage& ws,
                                                  int lane) {
    if (FORM == kFormUnpatch || !staged || m0 >= M) return;
    fetch_columns<FORM>(bias, gate, n0, end, ws, lane);
    if (FORM != kFormResid) return;
    request_residual(ws, ws.cnt, res, m0, n0, lane);
    if (n0 + 64 < end) request_residual(ws, ws.cnt + 1, res, m0, n0 + 64, lane);
}

// After a wait has given up: no residual copy is left in flight at exit.
__device__ __forceinline__ void epilogue_drain(WarpStage& ws) {
    for (; ws.pending > 0; --ws.pending, ++ws.cnt) {
        const unsigned long long t0 = globaltimer();
        while (!mbar_try_wait(&ws.rbar[ws.cnt & 1], (ws.cnt >> 1) & 1) && globaltimer() - t0 < kWaitLimitNs) {
        }
    }
}

// The tile's columns [n0, end) of rows [m0, m0 + 32), accumulator at taddr;
// `release` runs once the accumulator has been read.  Returns false when a
// residual slab did not arrive in time.
template <int FORM, class Release>
__device__ __forceinline__ bool epilogue_tile(const Epi& e, int staged, const EpiMaps* maps, int M, int m0, int n0, int end,
                                              uint32_t taddr, WarpStage& ws, volatile int* abort_flag,
                                              unsigned* err, int lane, Release release) {
    if (m0 >= M) {
        release();
        return true;
    }
    // QKV: the slab's rows are consecutive tokens of one sample, and rows past
    // M (if any) fall off the end of the tensor
    int b0 = 0, tok0 = 0;
    if (FORM == kFormQKV && staged) {
        const int last = min(m0 + 31, M - 1);
        int b1, tok1;
        batch_token(e.row_off + m0, e.nb, e.Lc, e.L, b0, tok0);
        batch_token(e.row_off + last, e.nb, e.Lc, e.L, b1, tok1);
        staged = b0 == b1 && tok1 - tok0 == last - m0 && (last == m0 + 31 || tok1 == e.L - 1);
    }
    // this lane's row address in an x4 matrix store: row lane % 8 of matrix
    // lane / 8; matrices 0, 1 are row groups 2 hb, 2 hb + 1 of column group i,
    // matrices 2, 3 the same of column group i + 1
    const int mrow = lane & 7, mrg = (lane >> 3) & 1, mcg = lane >> 4;
    for (int col0 = n0; col0 < end; col0 += 64) {
        const uint32_t sl = ws.cnt & 1;
        const uint32_t slab = smem_u32(ws.slab) + sl * SLAB_BYTES;
        const bool vt = FORM == kFormQKV && col0 >= 2 * e.D;
        if (FORM != kFormStore && FORM != kFormGelu && (FORM == kFormUnpatch || !staged || (vt && (tok0 & 7)))) {
            // (a V^T slab must start on a 16-byte boundary of its token row)
#pragma unroll 1
            for (int c32 = col0; c32 < min(col0 + 64, end); c32 += 32) {
                uint32_t r[32];
                tmem_ld32(taddr + (c32 - n0), r);
                tmem_ld_wait();
                if (c32 + 32 >= end) release();
                if (m0 + lane < M) epilogue_chunk<FORM>(e, m0 + lane, c32, r);
            }
            if (FORM == kFormQKV && col0 + 64 < end) fetch_columns<FORM>(e.bias, e.gate, col0 + 64, end, ws, lane);
            continue;
        }
        if constexpr (FORM != kFormUnpatch) {
            float v[2][8][4];                  // [rows 16 hb ..][column group][row t/4: 2, row t/4 + 8: 2]
            tmem_ld16x256(taddr + (col0 - n0), *reinterpret_cast<float(*)[32]>(&v[0]));
            tmem_ld16x256(taddr + (16u << 16) + (col0 - n0), *reinterpret_cast<float(*)[32]>(&v[1]));
            if constexpr (FORM == kFormResid) {
                const bool landed = mbar_wait(&ws.rbar[sl], (ws.cnt >> 1) & 1, abort_flag, err);
                if (!__all_sync(0xffffffffu, landed)) {
                    release();                     // every other wait of the CTA gives up too
                    return false;
                }
                --ws.pending;
            } else {
                if (lane == 0) bulk_wait_read<1>();
            }
            __syncwarp();
            tmem_ld_wait();
            if (col0 + 64 >= end) release();
            if (e.bias) {
#pragma unroll
                for (int i = 0; i < 8; ++i)
#pragma unroll
                    for (int hb = 0; hb < 2; ++hb) {
                        v[hb][i][0] += ws.bias[i].x; v[hb][i][1] += ws.bias[i].y;
                        v[hb][i][2] += ws.bias[i].x; v[hb][i][3] += ws.bias[i].y;
                    }
            }
            if constexpr (FORM == kFormGelu) {
#pragma unroll
                for (int i = 0; i < 8; ++i)
#pragma unroll
                    for (int hb = 0; hb < 2; ++hb)
#pragma unroll
                        for (int j = 0; j < 4; ++j) v[hb][i][j] = gelu_tanh_f(v[hb][i][j]);
            }
            if (vt) {
                // rows = d, 32 tokens (64 bytes) each, 64-byte swizzle
                bool sat[4] = {false, false, false, false};
#pragma unroll
                for (int hb = 0; hb < 2; ++hb)
#pragma unroll
                    for (int i = 0; i < 8; i += 2) {
                        uint32_t w[4];
#pragma unroll
                        for (int q = 0; q < 4; ++q) {          // matrix q: column group i + q / 2, rows of 2 hb + q % 2
                            const float* x = &v[hb][i + (q >> 1)][2 * (q & 1)];
                            const __half2 h = __halves2half2(to_vt_half(x[0], sat[2 * hb + (q & 1)]),
                                                             to_vt_half(x[1], sat[2 * hb + (q & 1)]));
                            w[q] = *reinterpret_cast<const uint32_t*>(&h);
                        }
                        const int dd = 8 * (i + mcg) + mrow;
                        stmatrix_x4_trans(slab + dd * 64 + (((2 * hb + mrg) ^ ((dd >> 1) & 3)) << 4), w);
                    }
                bool any = false;
#pragma unroll
                for (int g = 0; g < 4; ++g) any |= sat[g] && m0 + 8 * g + (lane >> 2) < M;
                if (any && e.err) atomicOr(e.err, kErrVSaturated);
            } else {
#pragma unroll
                for (int hb = 0; hb < 2; ++hb)
#pragma unroll
                    for (int i = 0; i < 8; i += 2) {
                        const uint32_t at = slab + (16 * hb + 8 * mrg + mrow) * 128 + (((i + mcg) ^ mrow) << 4);
                        if constexpr (FORM == kFormResid) {
                            uint32_t rr[4];
                            ldmatrix_x4(at, rr);
#pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                float* x = &v[hb][i + (q >> 1)][2 * (q & 1)];
                                const float2 f = unpack_bf16(rr[q]);
                                const float2 g = e.gate ? ws.gate[i + (q >> 1)] : make_float2(1.f, 1.f);
                                x[0] = fmaf(g.x, x[0], f.x);
                                x[1] = fmaf(g.y, x[1], f.y);
                            }
                        }
                        uint32_t w[4];
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const float* x = &v[hb][i + (q >> 1)][2 * (q & 1)];
                            w[q] = pack_bf16(x[0], x[1]);
                        }
                        stmatrix_x4(at, w);
                    }
            }
            if (col0 + 64 < end) fetch_columns<FORM>(e.bias, e.gate, col0 + 64, end, ws, lane);
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) {
                const uint8_t* src = ws.slab + sl * SLAB_BYTES;
                if constexpr (FORM != kFormQKV) {
                    tma_store_2d(&maps->out, src, col0, m0);
                } else {
                    const int c = col0 % e.D, head = b0 * e.H + c / e.d, dd = c % e.d;
                    if (vt) tma_store_3d(&maps->vt, src, tok0, dd, head);
                    else tma_store_3d(col0 < e.D ? &maps->out : &maps->res, src, dd, tok0, head);
                }
                bulk_commit();
            }
            if (FORM == kFormResid && col0 + 128 < end) request_residual(ws, ws.cnt, &maps->res, m0, col0 + 128, lane);
            ++ws.cnt;
        }
    }
    return true;
}

template <int BNT, int FORM>
__global__ void __launch_bounds__(kGemmThreads, 1)
    gemm_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                   const __grid_constant__ EpiMaps maps, const __grid_constant__ GemmArgs g) {
    using C = GemmCfg<BNT>;
    constexpr int STAGES = C::STAGES;
    constexpr uint32_t STAGE_BYTES = C::STAGE_BYTES;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* staging = smem + STAGES * STAGE_BYTES;
    uint64_t* full = reinterpret_cast<uint64_t*>(staging + STAGING_BYTES);
    uint64_t* empty = full + STAGES;
    uint64_t* tfull = empty + STAGES;
    uint64_t* tempty = tfull + 2;
    uint64_t* mma_done = tempty + 2;
    uint64_t* rbars = mma_done + 1;            // [4 warps][2] residual slabs
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(rbars + 8);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(&tfull[a], 1);
            mbar_init(&tempty[a], 4);
        }
        mbar_init(mma_done, 1);
        for (int i = 0; i < 8; ++i) mbar_init(&rbars[i], 1);
        *abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 0 && lane == 0) {
        prefetch_tmap(&tmA);
        prefetch_tmap(&tmB);
    }
    if (warp == 1) {
        tmem_alloc(tmem_slot, C::TMEM_COLS);
        tmem_relinquish();
    }
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    const int num_tiles = g.m_tiles * g.n_tiles;

    if (warp == 0) {
        if (lane == 0) {
            int stage = 0;
            uint32_t phase = 0;
            uint32_t armed_phase[STAGES];
            bool armed[STAGES];
            for (int s = 0; s < STAGES; ++s) armed[s] = false;
            bool ok = true;
            for (int tile = blockIdx.x; tile < num_tiles && ok; tile += gridDim.x) {
                const int m_blk = tile / g.n_tiles, n_blk = tile % g.n_tiles;
                for (int kb = 0; kb < g.k_blocks; ++kb) {
                    if (!mbar_wait(&empty[stage], phase ^ 1u, abort_flag, g.err)) { ok = false; break; }
                    mbar_arrive_expect_tx(&full[stage], STAGE_BYTES);
                    uint8_t* sa = smem + stage * STAGE_BYTES;
                    tma_load_2d(sa, &tmA, &full[stage], kb * BK, m_blk * BM);
                    tma_load_2d(sa + A_BYTES, &tmB, &full[stage], kb * BK, n_blk * BNT);
                    armed[stage] = true;
                    armed_phase[stage] = phase;
                    if (++stage == STAGES) { stage = 0; phase ^= 1u; }
                }
            }
            // drain: every issued copy has landed before the CTA may exit
            for (int s = 0; s < STAGES; ++s) {
                if (!armed[s]) continue;
                const unsigned long long t0 = globaltimer();
                while (!mbar_try_wait(&full[s], armed_phase[s]) && globaltimer() - t0 < kWaitLimitNs) {
                }
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            int stage = 0;
            uint32_t phase = 0;
            int acc = 0;
            uint32_t acc_phase = 0;
            bool ok = true;
            for (int tile = blockIdx.x; tile < num_tiles && ok; tile += gridDim.x) {
                if (!mbar_wait(&tempty[acc], acc_phase ^ 1u, abort_flag, g.err)) break;
                tc_fence_after();
                const uint32_t d = tmem_base + (uint32_t)(acc * BNT);
                for (int kb = 0; kb < g.k_blocks; ++kb) {
                    if (!mbar_wait(&full[stage], phase, abort_flag, g.err)) { ok = false; break; }
                    tc_fence_after();
                    const uint32_t a0 = smem_u32(smem + stage * STAGE_BYTES);
                    const uint32_t b0 = a0 + A_BYTES;
#pragma unroll
                    for (int k = 0; k < BK / 16; ++k)
                        tc_mma(d, sdesc_sw128(a0 + k * 32), sdesc_sw128(b0 + k * 32), C::IDESC, (kb | k) != 0);
                    tc_commit(&empty[stage]);
                    if (++stage == STAGES) { stage = 0; phase ^= 1u; }
                }
                tc_commit(&tfull[acc]);
                acc ^= 1;
                if (acc == 0) acc_phase ^= 1u;
            }
            // all MMAs issued by this thread have completed before TMEM is freed
            tc_commit(mma_done);
            const unsigned long long t0 = globaltimer();
            while (!mbar_try_wait(mma_done, 0) && globaltimer() - t0 < kWaitLimitNs) {
            }
        }
    } else {
        const int lg = warp & 3;   // TMEM lane quarter this warp may access
        int acc = 0;
        uint32_t acc_phase = 0;
        WarpStage ws{staging + lg * 2 * SLAB_BYTES, rbars + lg * 2, 0, 0, {}, {}};
        for (int tile = blockIdx.x; tile < num_tiles; tile += gridDim.x) {
            const int m_blk = tile / g.n_tiles, n_blk = tile % g.n_tiles;
            const int m0 = m_blk * BM + lg * 32, n0 = n_blk * BNT, end = min(n0 + BNT, g.N);
            epilogue_prefetch<FORM>(g.e.bias, g.e.gate, g.staged, &maps.res, g.M, n0, end, m0, ws, lane);
            if (!mbar_wait(&tfull[acc], acc_phase, abort_flag, g.err)) break;
            tc_fence_after();
            const uint32_t taddr = tmem_base + ((uint32_t)(lg * 32) << 16) + (uint32_t)(acc * BNT);
            const bool ok = epilogue_tile<FORM>(g.e, g.staged, &maps, g.M, m0, n0, end, taddr, ws, abort_flag, g.err, lane, [&] {
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&tempty[acc]);
            });
            if (!ok) break;
            acc ^= 1;
            if (acc == 0) acc_phase ^= 1u;
        }
        if (lane == 0) bulk_wait_read<0>();    // the slabs stay until their stores have read them
        epilogue_drain(ws);
    }
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, C::TMEM_COLS);
    }
}

// ---------------------------------------------------------------------------
// CTA-pair variant (clusters of 2, tcgen05 .cta_group::2): each pair computes a
// 256 x 256 tile with 256 x 256 x 16 MMAs issued by the even CTA; each CTA
// holds its 128 rows of A and its 128-row half of the W tile (32 KB per stage,
// 6 stages beside the 32 KB of epilogue slabs), so twice the MMA work is
// buffered per shared-memory byte.  Both CTAs' tile copies complete on the
// even CTA's mbarrier (the pair form of the tensor copy), which the even CTA
// arms with both CTAs' bytes; the even CTA's commits release both CTAs'
// stages and accumulators.  The pair allocation is collective (both CTAs receive the same TMEM base; the
// leader's base is used for every access and a mismatch is reported), and two
// 256-column accumulators let a tile's epilogue overlap the next tile's MMAs.
constexpr int STAGES2 = 6;
constexpr uint32_t A2_BYTES = 128 * BK * 2;
constexpr uint32_t B2_BYTES = 128 * BK * 2;                  // half of the 256-row W tile
constexpr uint32_t STAGE2_BYTES = A2_BYTES + B2_BYTES;
constexpr uint32_t TMEM2_COLS = 512;
constexpr uint32_t IDESC2 = idesc_bf16(256, 256);
constexpr size_t SMEM2_BYTES = STAGES2 * STAGE2_BYTES + STAGING_BYTES + 1024 + 512;
static_assert(SMEM2_BYTES <= 227 * 1024, "shared memory per CTA");

// Pair-kernel raster: the N tiles are split into groups of group_n; inside a
// group the tiles run N-fastest over every 256-row M block.  A group's slab
// of W (group_n * 256 rows * K) stays in L2 while A streams through once per
// group, so W is read from DRAM about once and A once per group.
__device__ __forceinline__ void pair_tile(const GemmArgs& g, int m_pairs, int tile, int& m_blk, int& n_blk) {
    const int per_group = m_pairs * g.group_n;
    const int grp = tile / per_group, r = tile - grp * per_group;
    const int n_first = grp * g.group_n;
    const int width = min(g.group_n, g.n_tiles - n_first);
    m_blk = r / width;
    n_blk = n_first + (r - m_blk * width);
}

// Tile `tile` of a (possibly grouped) pair launch: problem index, 256-row M
// block and N block.  The first problem's tiles use the raster groups, the
// second problem's follow in plain N-fastest order, so they fill the pairs
// the first problem leaves idle in its last wave.
__device__ __forceinline__ int grouped_tile(const GemmArgs& g, int m_pairs0, int tiles0, int tile, int& m_blk,
                                            int& n_blk) {
    if (tile < tiles0) {
        pair_tile(g, m_pairs0, tile, m_blk, n_blk);
        return 0;
    }
    const int r = tile - tiles0;
    m_blk = r / g.n_tiles;
    n_blk = r - m_blk * g.n_tiles;
    return 1;
}

template <int FORM>
__global__ void __launch_bounds__(kGemmThreads, 1)
    gemm_tc2_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                    const __grid_constant__ CUtensorMap tmA1, const __grid_constant__ CUtensorMap tmB1,
                    const __grid_constant__ EpiMaps maps, const __grid_constant__ EpiMaps maps1,
                    const __grid_constant__ GemmArgs g) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* staging = smem + STAGES2 * STAGE2_BYTES;
    uint64_t* full = reinterpret_cast<uint64_t*>(staging + STAGING_BYTES);   // even CTA: both halves landed
    uint64_t* empty = full + STAGES2;
    uint64_t* tfull = empty + STAGES2;         // [2]
    uint64_t* tempty = tfull + 2;              // [2] even CTA: both CTAs' epilogues are done
    uint64_t* mma_done = tempty + 2;
    uint64_t* rbars = mma_done + 1;            // [4 warps][2] residual slabs
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(rbars + 8);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();
    const int cluster_id = blockIdx.x >> 1, n_clusters = gridDim.x >> 1;
    const int m_pairs = (g.m_tiles + 1) >> 1;  // 256-row tiles (m_tiles counts 128-row tiles)
    const int tiles0 = m_pairs * g.n_tiles;
    const int num_tiles = tiles0 + (g.nprob > 1 ? g.m_pairs1 * g.n_tiles : 0);
    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES2; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(&tfull[a], 1);
            mbar_init(&tempty[a], 8);          // 4 epilogue warps in each CTA
        }
        mbar_init(mma_done, 1);
        for (int i = 0; i < 8; ++i) mbar_init(&rbars[i], 1);
        *abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 0 && lane == 0) {
        prefetch_tmap(&tmA);
        prefetch_tmap(&tmB);
        if (g.nprob > 1) {
            prefetch_tmap(&tmA1);
            prefetch_tmap(&tmB1);
        }
    }
    if (warp == 1) {
        tmem_alloc2(tmem_slot, TMEM2_COLS);
        tmem_relinquish2();
    }
    __syncthreads();
    cluster_sync_all();
    tc_fence_after();
    const uint32_t own_base = *tmem_slot;
    const uint32_t tmem = rank == 0 ? own_base : ld_shared_cluster_u32(mapa_shared(smem_u32(tmem_slot), 0));
    if (threadIdx.x == 0 && tmem != own_base) atomicOr(g.err, kErrTmem);
    const uint32_t leader_tempty0 = mapa_shared(smem_u32(&tempty[0]), 0);
    const uint32_t leader_tempty1 = mapa_shared(smem_u32(&tempty[1]), 0);

    if (warp == 0) {
        if (lane == 0) {
            int stage = 0;
            uint32_t phase = 0;
            uint32_t armed_phase[STAGES2];
            bool armed[STAGES2];
            for (int s = 0; s < STAGES2; ++s) armed[s] = false;
            bool ok = true;
            for (int tile = cluster_id; tile < num_tiles && ok; tile += n_clusters) {
                int mb, nb;
                const int prob = grouped_tile(g, m_pairs, tiles0, tile, mb, nb);
                const CUtensorMap* mA = prob ? &tmA1 : &tmA;
                const CUtensorMap* mB = prob ? &tmB1 : &tmB;
                const int m0 = mb * 256 + (int)rank * 128;
                const int n0 = nb * BN + (int)rank * 128;
                for (int kb = 0; kb < g.k_blocks; ++kb) {
                    if (!mbar_wait(&empty[stage], phase ^ 1u, abort_flag, g.err)) { ok = false; break; }
                    if (rank == 0) mbar_arrive_expect_tx(&full[stage], 2 * STAGE2_BYTES);
                    const uint32_t fb = mapa_shared(smem_u32(&full[stage]), 0);
                    uint8_t* sa = smem + stage * STAGE2_BYTES;
                    tma_load_2d_pair(sa, mA, fb, kb * BK, m0);
                    tma_load_2d_pair(sa + A2_BYTES, mB, fb, kb * BK, n0);
                    armed[stage] = true;
                    armed_phase[stage] = phase;
                    if (++stage == STAGES2) { stage = 0; phase ^= 1u; }
                }
            }
            // drain: every copy of the pair has landed (even CTA's full) and the
            // MMAs have released every stage (both CTAs' empty)
            for (int s = 0; s < STAGES2; ++s) {
                if (!armed[s]) continue;
                if (rank == 0) {
                    const unsigned long long t0 = globaltimer();
                    while (!mbar_try_wait(&full[s], armed_phase[s]) && globaltimer() - t0 < kWaitLimitNs) {
                    }
                }
                const unsigned long long t1 = globaltimer();
                while (!mbar_try_wait(&empty[s], armed_phase[s]) && globaltimer() - t1 < kWaitLimitNs) {
                }
            }
        }
    } else if (warp == 1) {
        if (lane == 0 && rank == 0) {
            // MMA issuer for the pair
            int stage = 0;
            uint32_t phase = 0;
            int acc = 0;
            uint32_t acc_phase = 0;
            bool ok = true;
            for (int tile = cluster_id; tile < num_tiles && ok; tile += n_clusters) {
                if (!mbar_wait(&tempty[acc], acc_phase ^ 1u, abort_flag, g.err)) break;
                tc_fence_after();
                const uint32_t d = tmem + (uint32_t)(acc * BN);
                for (int kb = 0; kb < g.k_blocks; ++kb) {
                    if (!mbar_wait(&full[stage], phase, abort_flag, g.err)) { ok = false; break; }
                    tc_fence_after();
                    const uint32_t a0 = smem_u32(smem + stage * STAGE2_BYTES);
                    const uint32_t b0 = a0 + A2_BYTES;
#pragma unroll
                    for (int k = 0; k < BK / 16; ++k)
                        tc_mma2(d, sdesc_sw128(a0 + k * 32), sdesc_sw128(b0 + k * 32), IDESC2, (kb | k) != 0);
                    tc_commit2_mc(&empty[stage], (uint16_t)0x3);
                    if (++stage == STAGES2) { stage = 0; phase ^= 1u; }
                }
                tc_commit2_mc(&tfull[acc], (uint16_t)0x3);
                acc ^= 1;
                if (acc == 0) acc_phase ^= 1u;
            }
            tc_commit2_mc(mma_done, (uint16_t)0x1);
            const unsigned long long t0 = globaltimer();
            while (!mbar_try_wait(mma_done, 0) && globaltimer() - t0 < kWaitLimitNs) {
            }
        }
    } else {
        const int lg = warp & 3;
        int acc = 0;
        uint32_t acc_phase = 0;
        WarpStage ws{staging + lg * 2 * SLAB_BYTES, rbars + lg * 2, 0, 0, {}, {}};
        for (int tile = cluster_id; tile < num_tiles; tile += n_clusters) {
            int mb, n_blk;
            const int prob = grouped_tile(g, m_pairs, tiles0, tile, mb, n_blk);
            const int m0 = mb * 256 + (int)rank * 128 + lg * 32, n0 = n_blk * BN, end = min(n0 + BN, g.N);
            // the second problem differs in its pointers, rows and maps only
            const int Mp = prob ? g.M1 : g.M, staged = prob ? g.staged1 : g.staged;
            const EpiMaps* mp = prob ? &maps1 : &maps;
            Epi e = g.e;
            if (prob) {
                e.bias = g.e1.bias;
                e.gate = g.e1.gate;
                e.out = g.e1.out;
                e.res = g.e1.res;
                e.row_off = g.e1.row_off;
            }
            epilogue_prefetch<FORM>(e.bias, e.gate, staged, &mp->res, Mp, n0, end, m0, ws, lane);
            if (!mbar_wait(&tfull[acc], acc_phase, abort_flag, g.err)) break;
            tc_fence_after();
            const uint32_t taddr = tmem + ((uint32_t)(lg * 32) << 16) + (uint32_t)(acc * BN);
            auto release = [&] {
                tc_fence_before();
                __syncwarp();
                if (lane == 0) {
                    if (rank == 0) mbar_arrive(&tempty[acc]);
                    else mbar_arrive_remote(acc == 0 ? leader_tempty0 : leader_tempty1);
                }
            };
            const bool ok = epilogue_tile<FORM>(e, staged, mp, Mp, m0, n0, end, taddr, ws, abort_flag, g.err, lane, release);
            if (!ok) break;
            acc ^= 1;
            if (acc == 0) acc_phase ^= 1u;
        }
        if (lane == 0) bulk_wait_read<0>();    // the slabs stay until their stores have read them
        epilogue_drain(ws);
    }
    __syncthreads();
    cluster_sync_all();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc2(own_base, TMEM2_COLS);
    }
}

PFN_cuTensorMapEncodeTiled_v12000 get_encode() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
        else
            cudaGetLastError();
    });
    return fn;
}

}  // namespace

bool encode_tmap_2d(CUtensorMap* map, const void* base, uint64_t inner, uint64_t outer, uint64_t row_bytes,
                    uint32_t box_inner, uint32_t box_outer, std::string* why) {
    auto fn = get_encode();
    if (!fn) { if (why) *why = "cuTensorMapEncodeTiled unavailable"; return false; }
    cuuint64_t dims[2] = {inner, outer};
    cuuint64_t strides[1] = {row_bytes};
    cuuint32_t box[2] = {box_inner, box_outer};
    cuuint32_t es[2] = {1, 1};
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, es,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) { if (why) *why = "cuTensorMapEncodeTiled failed: " + std::to_string((int)r); return false; }
    return true;
}

bool encode_tmap_3d(CUtensorMap* map, const void* base, uint64_t d0, uint64_t d1, uint64_t d2, uint64_t s1_bytes,
                    uint64_t s2_bytes, uint32_t b0, uint32_t b1, uint32_t b2, std::string* why, bool f16,
                    CUtensorMapSwizzle swizzle) {
    auto fn = get_encode();
    if (!fn) { if (why) *why = "cuTensorMapEncodeTiled unavailable"; return false; }
    cuuint64_t dims[3] = {d0, d1, d2};
    cuuint64_t strides[2] = {s1_bytes, s2_bytes};
    cuuint32_t box[3] = {b0, b1, b2};
    cuuint32_t es[3] = {1, 1, 1};
    CUresult r = fn(map, f16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3,
                    const_cast<void*>(base), dims, strides, box, es,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) { if (why) *why = "cuTensorMapEncodeTiled failed: " + std::to_string((int)r); return false; }
    return true;
}

bool tc_gemm_supported(int M, int N, int K) { return M > 0 && N > 0 && K > 0 && N % 32 == 0 && K % 8 == 0; }

namespace {

wdc_status check_operands(Ctx* c, const void* A, const void* W, const Epi& e) {
    if (((uintptr_t)A & 15) || ((uintptr_t)W & 15)) return fail(c, WDC_ERR_INVALID_ARG, "GEMM operands must be 16-byte aligned");
    if ((e.mode == kEpiStore || e.mode == kEpiResid) &&
        (e.ldo % 8 || ((uintptr_t)e.out & 15) || (e.res && ((uintptr_t)e.res & 15))))
        return fail(c, WDC_ERR_INVALID_ARG, "GEMM output must be 16-byte aligned with ldo % 8 == 0");
    if (e.bias && ((uintptr_t)e.bias & 15)) return fail(c, WDC_ERR_INVALID_ARG, "bias must be 16-byte aligned");
    if (e.gate && ((uintptr_t)e.gate & 15)) return fail(c, WDC_ERR_INVALID_ARG, "gate must be 16-byte aligned");
    if (e.mode == kEpiQKV && (e.D % 32 || e.d % 32)) return fail(c, WDC_ERR_UNSUPPORTED, "QKV epilogue needs d % 32 == 0");
    return WDC_OK;
}

using Kernel1 = void (*)(const CUtensorMap, const CUtensorMap, const EpiMaps, const GemmArgs);
using Kernel2 = void (*)(const CUtensorMap, const CUtensorMap, const CUtensorMap, const CUtensorMap, const EpiMaps,
                         const EpiMaps, const GemmArgs);
constexpr Kernel1 kKernel1[kForms] = {gemm_tc_kernel<256, 0>, gemm_tc_kernel<256, 1>, gemm_tc_kernel<256, 2>,
                                      gemm_tc_kernel<256, 3>, gemm_tc_kernel<256, 4>};
constexpr Kernel2 kKernel2[kForms] = {gemm_tc2_kernel<0>, gemm_tc2_kernel<1>, gemm_tc2_kernel<2>, gemm_tc2_kernel<3>,
                                      gemm_tc2_kernel<4>};

int form_of(const Epi& e) {
    switch (e.mode) {
        case kEpiResid: return kFormResid;
        case kEpiQKV: return kFormQKV;
        case kEpiUnpatch: return kFormUnpatch;
        default: return e.gelu ? kFormGelu : kFormStore;
    }
}

void set_attrs() {
    static bool attr_set = false;
    if (!attr_set) {
        for (int f = 0; f < kForms; ++f) {
            cudaFuncSetAttribute(kKernel1[f], cudaFuncAttributeMaxDynamicSharedMemorySize, (int)GemmCfg<256>::SMEM);
            cudaFuncSetAttribute(kKernel2[f], cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM2_BYTES);
        }
        attr_set = true;
    }
}

GemmArgs make_args(Ctx* c, int M, int N, int K, const Epi& e) {
    GemmArgs g{};
    g.M = M;
    g.N = N;
    g.K = K;
    g.m_tiles = (M + BM - 1) / BM;
    g.n_tiles = (N + BN - 1) / BN;
    g.k_blocks = (K + BK - 1) / BK;
    // raster groups: a W slab of at most ~40 MB per group (L2 is 126 MB,
    // shared with the streamed A and the output), as few groups as that
    // allows.  For deep K (> 4096) a 256-row slab of A is itself large
    // and re-reading A per group costs more than it saves (measured on the
    // 17776 x 3072 x 12288 MLP-down GEMM): plain N-fastest order there.
    g.group_n = g.n_tiles;
    if (K <= 4096) {
        const double slab_per_tile = 256.0 * K * 2.0;
        int gn = (int)(40.0e6 / slab_per_tile);
        gn = gn < 1 ? 1 : (gn > g.n_tiles ? g.n_tiles : gn);
        const int groups = (g.n_tiles + gn - 1) / gn;
        g.group_n = (g.n_tiles + groups - 1) / groups;  // balance the groups
    }
    g.e = e;
    g.err = c->err;
    g.nprob = 1;
    return g;
}

// Tensor maps of an epilogue's staged stores and residual loads; 0 when its
// form takes none (unpatchify; a residual whose rows repeat; a residual row
// that is not the output's).
bool encode_epilogue(const Epi& e, int M, int N, EpiMaps* m, int* staged, std::string* why) {
    *staged = 0;
    if (e.mode == kEpiUnpatch || (e.mode == kEpiResid && e.res_rows > 0 && M > e.res_rows)) return true;
    if (e.mode == kEpiQKV) {
        const uint64_t d = e.d, L = e.L, heads = (uint64_t)e.nb * e.H;
        if (!encode_tmap_3d(&m->out, e.q, d, L, heads, d * 2, L * d * 2, 64, 32, 1, why) ||
            !encode_tmap_3d(&m->res, e.k, d, L, heads, d * 2, L * d * 2, 64, 32, 1, why) ||
            !encode_tmap_3d(&m->vt, e.vt, L, d, heads, (uint64_t)e.ldv * 2, (uint64_t)e.ldv * d * 2, 32, 64, 1, why,
                            true, CU_TENSOR_MAP_SWIZZLE_64B))
            return false;
    } else {
        if (!encode_tmap_2d(&m->out, e.out, (uint64_t)N, (uint64_t)M, (uint64_t)e.ldo * 2, 64, 32, why)) return false;
        if (e.mode == kEpiResid &&
            !encode_tmap_2d(&m->res, e.res, (uint64_t)N, (uint64_t)M, (uint64_t)e.ldo * 2, 64, 32, why))
            return false;
    }
    *staged = 1;
    return true;
}

// Pair-kernel launch: a persistent grid of as many CTA pairs as can be
// resident, capped by the tile count.
wdc_status launch_pair(Ctx* c, const CUtensorMap& ta, const CUtensorMap& tb, const CUtensorMap& ta1,
                       const CUtensorMap& tb1, const EpiMaps& maps, const EpiMaps& maps1, const GemmArgs& g,
                       cudaStream_t s) {
    const int tiles = ((g.m_tiles + 1) / 2) * g.n_tiles + (g.nprob > 1 ? g.m_pairs1 * g.n_tiles : 0);
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(kGemmThreads, 1, 1);
    cfg.dynamicSmemBytes = SMEM2_BYTES;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    static int max_clusters = 0;
    if (max_clusters == 0) {
        cfg.gridDim = dim3(c->num_sms, 1, 1);
        if (cudaOccupancyMaxActiveClusters(&max_clusters, kKernel2[0], &cfg) != cudaSuccess || max_clusters < 1) {
            cudaGetLastError();
            max_clusters = c->num_sms / 2;
        }
    }
    int clusters = max_clusters < c->num_sms / 2 ? max_clusters : c->num_sms / 2;
    if (tiles < clusters) clusters = tiles;
    cfg.gridDim = dim3(2 * clusters, 1, 1);
    cudaLaunchKernelEx(&cfg, kKernel2[form_of(g.e)], ta, tb, ta1, tb1, maps, maps1, g);
    cudaError_t err = cudaGetLastError();
    if (err != cudaSuccess) return fail(c, WDC_ERR_CUDA, std::string("tcgen05 GEMM launch: ") + cudaGetErrorString(err));
    return WDC_OK;
}

}  // namespace

wdc_status tc_gemm(Ctx* c, const void* A, const void* W, int M, int N, int K, const Epi& e, cudaStream_t s) {
    wdc_status st = check_operands(c, A, W, e);
    if (st) return st;
    set_attrs();
    const bool pair = M >= 256 && c->num_sms >= 2;
    CUtensorMap ta, tb;
    std::string why;
    if (!encode_tmap_2d(&ta, A, (uint64_t)K, (uint64_t)M, (uint64_t)K * 2, BK, BM, &why) ||
        !encode_tmap_2d(&tb, W, (uint64_t)K, (uint64_t)N, (uint64_t)K * 2, BK, pair ? BN / 2 : BN, &why))
        return fail(c, WDC_ERR_CUDA, why);
    GemmArgs g = make_args(c, M, N, K, e);
    EpiMaps maps{};
    if (!encode_epilogue(e, M, N, &maps, &g.staged, &why)) return fail(c, WDC_ERR_CUDA, why);
    if (pair) return launch_pair(c, ta, tb, ta, tb, maps, maps, g, s);
    const int tiles = g.m_tiles * g.n_tiles;
    const int grid = tiles < c->num_sms ? tiles : c->num_sms;
    kKernel1[form_of(e)]<<<grid, kGemmThreads, GemmCfg<256>::SMEM, s>>>(ta, tb, maps, g);
    cudaError_t err = cudaGetLastError();
    if (err != cudaSuccess) return fail(c, WDC_ERR_CUDA, std::string("tcgen05 GEMM launch: ") + cudaGetErrorString(err));
    return WDC_OK;
}

// Two GEMMs with the same N and K in one launch of the pair kernel (the
// dual-stream blocks' video rows and condition rows): problem 1's tiles
// follow problem 0's, filling the pairs problem 0 leaves idle in its last
// wave.  When problem 0 is too short for the pair kernel the two run as two
// launches on the stream.
wdc_status tc_gemm_grouped(Ctx* c, const void* A0, const void* W0, int M0, const Epi& e0, const void* A1,
                           const void* W1, int M1, const Epi& e1, int N, int K, cudaStream_t s) {
    if (M1 <= 0) return tc_gemm(c, A0, W0, M0, N, K, e0, s);
    if (M0 <= 0) return tc_gemm(c, A1, W1, M1, N, K, e1, s);
    if (M0 < 256 || c->num_sms < 2) {
        wdc_status st = tc_gemm(c, A0, W0, M0, N, K, e0, s);
        return st ? st : tc_gemm(c, A1, W1, M1, N, K, e1, s);
    }
    wdc_status st = check_operands(c, A0, W0, e0);
    if (!st) st = check_operands(c, A1, W1, e1);
    if (st) return st;
    set_attrs();
    CUtensorMap ta, tb, ta1, tb1;
    std::string why;
    if (!encode_tmap_2d(&ta, A0, (uint64_t)K, (uint64_t)M0, (uint64_t)K * 2, BK, BM, &why) ||
        !encode_tmap_2d(&tb, W0, (uint64_t)K, (uint64_t)N, (uint64_t)K * 2, BK, BN / 2, &why) ||
        !encode_tmap_2d(&ta1, A1, (uint64_t)K, (uint64_t)M1, (uint64_t)K * 2, BK, BM, &why) ||
        !encode_tmap_2d(&tb1, W1, (uint64_t)K, (uint64_t)N, (uint64_t)K * 2, BK, BN / 2, &why))
        return fail(c, WDC_ERR_CUDA, why);
    GemmArgs g = make_args(c, M0, N, K, e0);
    g.nprob = 2;
    g.M1 = M1;
    g.m_pairs1 = (M1 + 255) / 256;
    g.e1 = e1;
    EpiMaps maps{}, maps1{};
    if (!encode_epilogue(e0, M0, N, &maps, &g.staged, &why) || !encode_epilogue(e1, M1, N, &maps1, &g.staged1, &why))
        return fail(c, WDC_ERR_CUDA, why);
    return launch_pair(c, ta, tb, ta1, tb1, maps, maps1, g, s);
}

}  // namespace wdc
