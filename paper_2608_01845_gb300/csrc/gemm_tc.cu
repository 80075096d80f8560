// Dense bf16 GEMM on the 5th-generation tensor cores (tcgen05, sm_103a) with
// the DiT's fused epilogues: C = epilogue(A W^T), A [M, K], W [N, K] bf16,
// fp32 accumulation in tensor memory.
//
// Three kernels, 6 warps a CTA (TMA producer, MMA issuer, 4 epilogue warps):
//   gemm_tc2_kernel   persistent, CTA pairs, 256 x 256, 192 or 128 tiles: shapes with
//                     tiles for (nearly) every pair;
//   gemm_tc_kernel    persistent, one CTA a tile of 128 x 128 or 128 x 64:
//                     shapes that would leave most pairs without a tile;
//   gemm_split_kernel one 128 x 128 tile a cluster, its CTAs each summing a
//                     part of K and reducing through distributed shared memory:
//                     shapes with too few tiles for the SMs and a K to split.
// choose_gemm picks one by the estimated cycles of each.
//   warp 0      TMA producer: A and W tiles of 64 columns of K into a
//               shared-memory ring (128-byte swizzle), one mbarrier pair per
//               stage;
//   warp 1      MMA issuer: one elected lane issues the tcgen05.mma of each stage
//               into one of two TMEM accumulators, commits the stage back to
//               the producer and the accumulator to the epilogue;
//   warps 2-5   epilogue (epilogue_tile): each warp owns its 32-lane TMEM
//               quarter = 32 rows and works through the tile 64 columns at a
//               time: tcgen05.ld, bias / GELU / gated residual, bf16 into a
//               swizzled shared-memory slab, one TMA store per slab; then
//               release the accumulator so the next tile's MMAs overlap.
// The pair kernel's tiles are visited N-fastest inside groups of N tiles sized
// so a group's slab of W stays in L2 (about 40 MB), so W is read from DRAM
// about once and A once per group.
// Tails: TMA zero-fills rows past M / N and columns past K; the epilogue
// masks rows >= M.  Every mbarrier wait is bounded.
// Each output element is accumulated over K in the same order by the pair and
// the one-CTA kernels, and whether K is split depends on one sample's rows
// only, so a sample's results are the same bits in any batch.
#include "dit_kernels.cuh"
#include "ptx.cuh"

#include <cudaTypedefs.h>

#include <mutex>

namespace wdc {

namespace {

constexpr int BM = 128, BK = 64;
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
    static constexpr int STAGES = BNT == 128 ? 6 : 8;
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
    int m_tiles, n_tiles, k_blocks;   // 128-row tiles; N tiles of the kernel's width; 64-column K blocks
    int group_n;            // pair kernel: N tiles per raster group
    Epi e;
    unsigned* err;
    // grouped launch: a second problem with the same N and K
    // (its own A, W, M and epilogue) whose tiles follow the first problem's
    int nprob;              // 1 or 2
    int M1, m_tiles1;       // m_tiles1 counts 128-row tiles, as m_tiles
    Epi e1;
    // whether each problem's epilogue has its tensor maps (else every row goes
    // through the direct stores of epilogue_chunk)
    int staged, staged1;
};

// Epilogue of problem `prob`: the second problem differs from the first in
// these fields only.
__device__ __forceinline__ Epi problem_epilogue(const GemmArgs& g, int prob) {
    Epi e = g.e;
    if (prob) {
        e.bias = g.e1.bias;
        e.gate = g.e1.gate;
        e.out = g.e1.out;
        e.res = g.e1.res;
        e.row_off = g.e1.row_off;
    }
    return e;
}

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
enum Form {
    kFormStore = WDC_GEMM_STORE, kFormGelu = WDC_GEMM_GELU, kFormResid = WDC_GEMM_RESID, kFormQKV = WDC_GEMM_QKV,
    kFormUnpatch = WDC_GEMM_UNPATCH, kFormResidGelu = WDC_GEMM_RESID_GELU, kFormResidRepeat = WDC_GEMM_RESID_REPEAT,
    kForms = WDC_GEMM_FORMS
};
// kFormResidGelu: a residual over GELU's result, an operator call's only (the
// blocks apply GELU before another GEMM).
// kFormResidRepeat: a residual whose rows repeat every e.res_rows (a batch's
// position embedding).  Its index arithmetic in kFormResid cost the small
// launches 0.1 us each.
constexpr bool is_resid(int form) { return form == kFormResid || form == kFormResidGelu || form == kFormResidRepeat; }
constexpr bool has_gelu(int form) { return form == kFormGelu || form == kFormResidGelu; }

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
    if constexpr (has_gelu(FORM)) {
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] = gelu_tanh_f(v[j]);
    }
    if constexpr (is_resid(FORM)) {
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
                    const float4 t = ld_chain(g4 + j);
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

// The residual row of a slab's first row, and whether the slab's rows are
// consecutive there (if not it goes the direct way).  6144 x 1024 x 64 with
// four repeats: 18.0 -> 12.3 us against the direct way for all rows.
template <int FORM>
__device__ __forceinline__ int residual_row(const Epi& e, int m0) {
    return FORM == kFormResidRepeat ? m0 % e.res_rows : m0;
}
template <int FORM>
__device__ __forceinline__ bool one_repeat(const Epi& e, int M, int m0) {
    return FORM != kFormResidRepeat || m0 % e.res_rows + min(32, M - m0) <= e.res_rows;
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
    if (is_resid(FORM) && gate) {
#pragma unroll
        for (int i = 0; i < 8; ++i) ws.gate[i] = ld_chain(reinterpret_cast<const float2*>(gate + min(c + 8 * i, end - 2)));
    }
}

// Before the tile's accumulator is awaited: its first chunk's columns and its
// first two residual slabs.
template <int FORM>
__device__ __forceinline__ void epilogue_prefetch(const Epi& e, int staged, const CUtensorMap* res, int M, int n0, int end,
                                                  int m0, WarpStage& ws, int lane) {
    if (FORM == kFormUnpatch || !staged || m0 >= M) return;
    if (!one_repeat<FORM>(e, M, m0)) return;
    fetch_columns<FORM>(e.bias, e.gate, n0, end, ws, lane);
    if (!is_resid(FORM)) return;
    const int rm = residual_row<FORM>(e, m0);
    request_residual(ws, ws.cnt, res, rm, n0, lane);
    if (n0 + 64 < end) request_residual(ws, ws.cnt + 1, res, rm, n0 + 64, lane);
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
    const int rm0 = residual_row<FORM>(e, m0);
    if (!one_repeat<FORM>(e, M, m0)) staged = 0;
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
            if constexpr (is_resid(FORM)) {
                if (!mbar_wait_warp(&ws.rbar[sl], (ws.cnt >> 1) & 1, abort_flag, err)) {
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
            if constexpr (has_gelu(FORM)) {
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
                        if constexpr (is_resid(FORM)) {
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
            if (is_resid(FORM) && col0 + 128 < end) request_residual(ws, ws.cnt, &maps->res, rm0, col0 + 128, lane);
            ++ws.cnt;
        }
    }
    return true;
}

template <int BNT, int FORM>
__global__ void __launch_bounds__(kGemmThreads, 1)
    gemm_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                   const __grid_constant__ CUtensorMap tmA1, const __grid_constant__ CUtensorMap tmB1,
                   const __grid_constant__ EpiMaps maps, const __grid_constant__ EpiMaps maps1,
                   const __grid_constant__ GemmArgs g) {
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
        if (g.nprob > 1) {
            prefetch_tmap(&tmA1);
            prefetch_tmap(&tmB1);
        }
    }
    if (warp == 1) {
        tmem_alloc(tmem_slot, C::TMEM_COLS);
        tmem_relinquish();
    }
    __syncthreads();
    tc_fence_after();
    chain_release();
    chain_wait();
    const uint32_t tmem_base = *tmem_slot;
    // tiles of the first problem, then of the second, N-fastest
    const int tiles0 = g.m_tiles * g.n_tiles;
    const int num_tiles = tiles0 + (g.nprob > 1 ? g.m_tiles1 * g.n_tiles : 0);

    if (warp == 0) {
        {
            int stage = 0;
            uint32_t phase = 0;
            uint32_t armed = 0, parity = 0;        // per stage: a copy was issued; its phase
            bool ok = true;
            for (int tile = blockIdx.x; tile < num_tiles && ok; tile += gridDim.x) {
                const int prob = tile >= tiles0, r = tile - prob * tiles0;
                const int m_blk = r / g.n_tiles, n_blk = r % g.n_tiles;
                const CUtensorMap* mA = prob ? &tmA1 : &tmA;
                const CUtensorMap* mB = prob ? &tmB1 : &tmB;
                for (int kb = 0; kb < g.k_blocks; ++kb) {
                    if (!mbar_wait_warp(&empty[stage], phase ^ 1u, abort_flag, g.err)) { ok = false; break; }
                    if (elect_one()) {
                        mbar_arrive_expect_tx(&full[stage], STAGE_BYTES);
                        uint8_t* sa = smem + stage * STAGE_BYTES;
                        tma_load_2d(sa, mA, &full[stage], kb * BK, m_blk * BM);
                        tma_load_2d(sa + A_BYTES, mB, &full[stage], kb * BK, n_blk * BNT);
                    }
                    __syncwarp();
                    armed |= 1u << stage;
                    parity = (parity & ~(1u << stage)) | (phase << stage);
                    if (++stage == STAGES) { stage = 0; phase ^= 1u; }
                }
            }
            // drain: every issued copy has landed before the CTA may exit
            for (int s = 0; s < STAGES; ++s) {
                if (!((armed >> s) & 1)) continue;
                const unsigned long long t0 = globaltimer();
                while (!mbar_try_wait(&full[s], (parity >> s) & 1) && globaltimer() - t0 < kWaitLimitNs) {
                }
            }
        }
    } else if (warp == 1) {
        // one lane for the whole loop: less code than the other kernels' warp,
        // and code that a short launch runs once costs it its fetch (a forward
        // of 2 layers, 272 tokens: 97.5 -> 95 us)
        if (elect_one()) {
            const uint64_t da = sdesc_sw128(smem_u32(smem)), db = sdesc_sw128(smem_u32(smem) + A_BYTES);
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
#pragma unroll
                    for (int k = 0; k < BK / 16; ++k)
                        tc_mma(d, sdesc_at(da, stage * STAGE_BYTES + k * 32), sdesc_at(db, stage * STAGE_BYTES + k * 32),
                               C::IDESC, (kb | k) != 0);
                    tc_commit(&empty[stage]);
                    if (kb + 1 == g.k_blocks) tc_commit(&tfull[acc]);
                    if (++stage == STAGES) { stage = 0; phase ^= 1u; }
                }
                acc ^= 1;
                if (acc == 0) acc_phase ^= 1u;
            }
            // all MMAs issued by this lane have completed before TMEM is freed
            tc_commit(mma_done);
            const unsigned long long t0 = globaltimer();
            while (!mbar_try_wait(mma_done, 0) && globaltimer() - t0 < kWaitLimitNs) {
            }
        }
        __syncwarp();
    } else {
        const int lg = warp & 3;   // TMEM lane quarter this warp may access
        int acc = 0;
        uint32_t acc_phase = 0;
        WarpStage ws{staging + lg * 2 * SLAB_BYTES, rbars + lg * 2, 0, 0, {}, {}};
        for (int tile = blockIdx.x; tile < num_tiles; tile += gridDim.x) {
            const int prob = tile >= tiles0, r = tile - prob * tiles0;
            const int m0 = (r / g.n_tiles) * BM + lg * 32, n0 = (r % g.n_tiles) * BNT, end = min(n0 + BNT, g.N);
            const int Mp = prob ? g.M1 : g.M, staged = prob ? g.staged1 : g.staged;
            const EpiMaps* mp = prob ? &maps1 : &maps;
            const Epi e = problem_epilogue(g, prob);
            epilogue_prefetch<FORM>(e, staged, &mp->res, Mp, n0, end, m0, ws, lane);
            if (!mbar_wait_warp(&tfull[acc], acc_phase, abort_flag, g.err)) break;
            tc_fence_after();
            const uint32_t taddr = tmem_base + ((uint32_t)(lg * 32) << 16) + (uint32_t)(acc * BNT);
            const bool ok = epilogue_tile<FORM>(e, staged, mp, Mp, m0, n0, end, taddr, ws, abort_flag, g.err, lane, [&] {
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
// The tile's width BNP may also be 192 or 128: a round of narrower tiles is
// shorter, which pays where whole rounds of 256 leave many pairs idle.
constexpr uint32_t A2_BYTES = 128 * BK * 2;
constexpr uint32_t TMEM2_COLS = 512;
template <int BNP>
struct PairCfg {
    static constexpr int STAGES = BNP == 128 ? 8 : 6;
    static constexpr uint32_t B_BYTES = BNP / 2 * BK * 2;    // half of the W tile's rows
    static constexpr uint32_t STAGE_BYTES = A2_BYTES + B_BYTES;
    static constexpr uint32_t IDESC = idesc_bf16(256, BNP);
    static constexpr size_t SMEM = STAGES * STAGE_BYTES + STAGING_BYTES + 1024 + 512;
    static_assert(SMEM <= 227 * 1024, "shared memory per CTA");
    static_assert(B_BYTES % 1024 == 0 && BNP % 64 == 0, "swizzled tiles of whole 64-column chunks");
};

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

template <int BNP, int FORM>
__global__ void __launch_bounds__(kGemmThreads, 1)
    gemm_tc2_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                    const __grid_constant__ CUtensorMap tmA1, const __grid_constant__ CUtensorMap tmB1,
                    const __grid_constant__ EpiMaps maps, const __grid_constant__ EpiMaps maps1,
                    const __grid_constant__ GemmArgs g) {
    using C = PairCfg<BNP>;
    constexpr int STAGES = C::STAGES;
    constexpr uint32_t STAGE_BYTES = C::STAGE_BYTES;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* staging = smem + STAGES * STAGE_BYTES;
    uint64_t* full = reinterpret_cast<uint64_t*>(staging + STAGING_BYTES);   // even CTA: both halves landed
    uint64_t* empty = full + STAGES;
    uint64_t* tfull = empty + STAGES;         // [2]
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
    const int num_tiles = tiles0 + (g.nprob > 1 ? ((g.m_tiles1 + 1) >> 1) * g.n_tiles : 0);
    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
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
    chain_release();
    chain_wait();
    const uint32_t own_base = *tmem_slot;
    const uint32_t tmem = rank == 0 ? own_base : ld_shared_cluster_u32(mapa_shared(smem_u32(tmem_slot), 0));
    if (threadIdx.x == 0 && tmem != own_base) atomicOr(g.err, kErrTmem);
    const uint32_t leader_tempty0 = mapa_shared(smem_u32(&tempty[0]), 0);
    const uint32_t leader_tempty1 = mapa_shared(smem_u32(&tempty[1]), 0);

    if (warp == 0) {
        {
            int stage = 0;
            uint32_t phase = 0;
            uint32_t armed = 0, parity = 0;        // per stage: a copy was issued; its phase
            bool ok = true;
            for (int tile = cluster_id; tile < num_tiles && ok; tile += n_clusters) {
                int mb, nb;
                const int prob = grouped_tile(g, m_pairs, tiles0, tile, mb, nb);
                const CUtensorMap* mA = prob ? &tmA1 : &tmA;
                const CUtensorMap* mB = prob ? &tmB1 : &tmB;
                const int m0 = mb * 256 + (int)rank * 128;
                const int n0 = nb * BNP + (int)rank * (BNP / 2);
                for (int kb = 0; kb < g.k_blocks; ++kb) {
                    if (!mbar_wait_warp(&empty[stage], phase ^ 1u, abort_flag, g.err)) { ok = false; break; }
                    if (elect_one()) {
                        if (rank == 0) mbar_arrive_expect_tx(&full[stage], 2 * STAGE_BYTES);
                        const uint32_t fb = mapa_shared(smem_u32(&full[stage]), 0);
                        uint8_t* sa = smem + stage * STAGE_BYTES;
                        tma_load_2d_pair(sa, mA, fb, kb * BK, m0);
                        tma_load_2d_pair(sa + A2_BYTES, mB, fb, kb * BK, n0);
                    }
                    __syncwarp();
                    armed |= 1u << stage;
                    parity = (parity & ~(1u << stage)) | (phase << stage);
                    if (++stage == STAGES) { stage = 0; phase ^= 1u; }
                }
            }
            // drain: every copy of the pair has landed (even CTA's full) and the
            // MMAs have released every stage (both CTAs' empty)
            for (int s = 0; s < STAGES; ++s) {
                if (!((armed >> s) & 1)) continue;
                if (rank == 0) {
                    const unsigned long long t0 = globaltimer();
                    while (!mbar_try_wait(&full[s], (parity >> s) & 1) && globaltimer() - t0 < kWaitLimitNs) {
                    }
                }
                const unsigned long long t1 = globaltimer();
                while (!mbar_try_wait(&empty[s], (parity >> s) & 1) && globaltimer() - t1 < kWaitLimitNs) {
                }
            }
        }
    } else if (warp == 1) {
        if (rank == 0) {
            // MMA issuer for the pair
            const uint64_t da = sdesc_sw128(smem_u32(smem)), db = sdesc_sw128(smem_u32(smem) + A2_BYTES);
            int stage = 0;
            uint32_t phase = 0;
            int acc = 0;
            uint32_t acc_phase = 0;
            bool ok = true;                        // this lane's waits (elect_one)
            for (int tile = cluster_id; tile < num_tiles; tile += n_clusters) {
                ok = ok && mbar_wait(&tempty[acc], acc_phase ^ 1u, abort_flag, g.err);
                tc_fence_after();
                const uint32_t d = tmem + (uint32_t)(acc * 256);
                for (int kb = 0; kb < g.k_blocks; ++kb) {
                    ok = ok && mbar_wait(&full[stage], phase, abort_flag, g.err);
                    tc_fence_after();
                    if (elect_one() && ok) {
#pragma unroll
                        for (int k = 0; k < BK / 16; ++k)
                            tc_mma2(d, sdesc_at(da, stage * STAGE_BYTES + k * 32), sdesc_at(db, stage * STAGE_BYTES + k * 32),
                                    C::IDESC, (kb | k) != 0);
                        tc_commit2_mc(&empty[stage], (uint16_t)0x3);
                        if (kb + 1 == g.k_blocks) tc_commit2_mc(&tfull[acc], (uint16_t)0x3);
                    }
                    __syncwarp();
                    if (++stage == STAGES) { stage = 0; phase ^= 1u; }
                }
                acc ^= 1;
                if (acc == 0) acc_phase ^= 1u;
            }
            if (elect_one()) tc_commit2_mc(mma_done, (uint16_t)0x1);
            __syncwarp();
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
            const int m0 = mb * 256 + (int)rank * 128 + lg * 32, n0 = n_blk * BNP, end = min(n0 + BNP, g.N);
            const int Mp = prob ? g.M1 : g.M, staged = prob ? g.staged1 : g.staged;
            const EpiMaps* mp = prob ? &maps1 : &maps;
            const Epi e = problem_epilogue(g, prob);
            epilogue_prefetch<FORM>(e, staged, &mp->res, Mp, n0, end, m0, ws, lane);
            if (!mbar_wait_warp(&tfull[acc], acc_phase, abort_flag, g.err)) break;
            tc_fence_after();
            const uint32_t taddr = tmem + ((uint32_t)(lg * 32) << 16) + (uint32_t)(acc * 256);
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

// ---------------------------------------------------------------------------
// Split-K variant: one 128 x 128 tile a cluster of S = 2, 4 or 8 CTAs.  CTA r
// sums K blocks [r kb / S, (r + 1) kb / S) into its tensor memory.  Once every
// CTA is done with its ring, each sends the others their share of its columns
// (128 / S) into their shared memory, and after a cluster barrier each adds the
// S partial sums of its columns in rank order and runs the epilogue on them, 8
// columns a thread at a time.
// A CTA's main loop is bound by its shared memory: a 64-column block of K puts
// 32 KB into it and the MMAs read as much, 430-480 cycles whatever the tile's
// width (482 at 128, 450 at 64), so a small M with a deep K waits for few SMs.
// Partial sums lie as [source][4 columns][row]: a warp sends one 512-byte run.
// (Row by row, 16 bytes a packet, sending took 4-8k cycles; fetching instead of
// sending, one round trip after another, more.)
constexpr int SPLIT_BN = 128, SPLIT_STAGES = 6, SPLIT_MAX = 8;
constexpr uint32_t SPLIT_STAGE_BYTES = A_BYTES + SPLIT_BN * BK * 2;
constexpr size_t SPLIT_SMEM = SPLIT_STAGES * SPLIT_STAGE_BYTES + 1024 + 256;
static_assert(SPLIT_SMEM <= 227 * 1024, "shared memory per CTA");
static_assert(BM * SPLIT_BN * 4 <= SPLIT_STAGES * SPLIT_STAGE_BYTES, "partial sums fit the ring");
// Byte offset of row `row`'s columns 4 c4 .. 4 c4 + 3 of the share of S in
// source p's partial sums: rows are permuted by the column group, so that
// lanes on one row and successive 8-column groups meet different banks.
template <int S>
__device__ __forceinline__ uint32_t split_at(int p, int c4, int row) {
    return (uint32_t)((p * (SPLIT_BN / S / 4) + c4) * BM + (row ^ ((c4 >> 1) & 7))) * 16u;
}

__device__ __forceinline__ uint4 residual8(const Epi& e, int m, int col) {
    const int rm = e.res_rows > 0 ? m % e.res_rows : m;
    return *reinterpret_cast<const uint4*>(reinterpret_cast<const __nv_bfloat16*>(e.res) + (size_t)rm * e.ldo + col);
}

// Bias and gate (0 and 1 where there is none) of 8 columns.
template <int FORM>
__device__ __forceinline__ void columns8(const Epi& e, int col, float (&bias)[8], float (&gate)[8]) {
    auto load = [&](const float* src, float none, float (&x)[8]) {
        float4 a = make_float4(none, none, none, none), b = a;
        if (src) {
            a = ld_chain(reinterpret_cast<const float4*>(src + col));
            b = ld_chain(reinterpret_cast<const float4*>(src + col) + 1);
        }
        x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w;
        x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
    };
    load(e.bias, 0.f, bias);
    if (is_resid(FORM)) load(e.gate, 1.f, gate);
}

// Epilogue of 8 consecutive columns (one 16-byte store) of row m.
template <int FORM>
__device__ __forceinline__ void epilogue8(const Epi& e, int m, int col, float (&v)[8], const float (&bias)[8],
                                          const float (&gate)[8], const uint4& rr) {
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] += bias[j];
    if constexpr (FORM == kFormUnpatch) {
        Epi plain = e;
        plain.bias = nullptr;
#pragma unroll
        for (int j = 0; j < 8; ++j) epi_apply<__nv_bfloat16>(plain, m, col + j, v[j]);
        return;
    }
    if constexpr (has_gelu(FORM)) {
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = gelu_tanh_f(v[j]);
    }
    __nv_bfloat16* dst;
    if constexpr (FORM == kFormQKV) {
        const int which = col / e.D, c = col % e.D, dd = c % e.d;
        int b, tok;
        batch_token(e.row_off + m, e.nb, e.Lc, e.L, b, tok);
        const size_t h = (size_t)b * e.H + c / e.d;
        if (which == 2) {
            __half* base = reinterpret_cast<__half*>(e.vt) + (h * e.d + dd) * e.ldv + tok;
            bool sat = false;
#pragma unroll
            for (int j = 0; j < 8; ++j) base[(size_t)j * e.ldv] = to_vt_half(v[j], sat);
            if (sat && e.err) atomicOr(e.err, kErrVSaturated);
            return;
        }
        dst = reinterpret_cast<__nv_bfloat16*>(which == 0 ? e.q : e.k) + (h * e.L + tok) * e.d + dd;
    } else {
        dst = reinterpret_cast<__nv_bfloat16*>(e.out) + (size_t)m * e.ldo + col;
    }
    if constexpr (is_resid(FORM)) {
        const uint32_t w[4] = {rr.x, rr.y, rr.z, rr.w};
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const float2 f = unpack_bf16(w[t]);
            v[2 * t] = fmaf(gate[2 * t], v[2 * t], f.x);
            v[2 * t + 1] = fmaf(gate[2 * t + 1], v[2 * t + 1], f.y);
        }
    }
    *reinterpret_cast<uint4*>(dst) =
        make_uint4(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]), pack_bf16(v[6], v[7]));
}

template <int FORM, int S>
__global__ void __launch_bounds__(kGemmThreads, 1)
    gemm_split_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                      const __grid_constant__ CUtensorMap tmA1, const __grid_constant__ CUtensorMap tmB1,
                      const __grid_constant__ GemmArgs g) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + SPLIT_STAGES * SPLIT_STAGE_BYTES);
    uint64_t* empty = full + SPLIT_STAGES;
    uint64_t* tfull = empty + SPLIT_STAGES;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tfull + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = (int)cluster_ctarank();
    const int tile = blockIdx.x / S, tiles0 = g.m_tiles * g.n_tiles;
    const int prob = tile >= tiles0, r = tile - prob * tiles0;
    const int m_blk = r / g.n_tiles, n_blk = r % g.n_tiles;
    const int kb0 = rank * g.k_blocks / S, kb1 = (rank + 1) * g.k_blocks / S;
    if (threadIdx.x == 0) {
        for (int s = 0; s < SPLIT_STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(tfull, 1);
        *abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 1) {
        tmem_alloc(tmem_slot, SPLIT_BN);
        tmem_relinquish();
    }
    __syncthreads();
    tc_fence_after();
    chain_release();
    chain_wait();
    const uint32_t tmem_base = *tmem_slot;
    if (warp == 0) {
        {
            const CUtensorMap* mA = prob ? &tmA1 : &tmA;
            const CUtensorMap* mB = prob ? &tmB1 : &tmB;
            uint32_t armed = 0, parity = 0;        // per stage: a copy was issued; its phase
            int stage = 0;
            uint32_t phase = 0;
            for (int kb = kb0; kb < kb1; ++kb) {
                if (!mbar_wait_warp(&empty[stage], phase ^ 1u, abort_flag, g.err)) break;
                if (elect_one()) {
                    mbar_arrive_expect_tx(&full[stage], SPLIT_STAGE_BYTES);
                    uint8_t* sa = smem + stage * SPLIT_STAGE_BYTES;
                    tma_load_2d(sa, mA, &full[stage], kb * BK, m_blk * BM);
                    tma_load_2d(sa + A_BYTES, mB, &full[stage], kb * BK, n_blk * SPLIT_BN);
                }
                __syncwarp();
                armed |= 1u << stage;
                parity = (parity & ~(1u << stage)) | (phase << stage);
                if (++stage == SPLIT_STAGES) { stage = 0; phase ^= 1u; }
            }
            // every issued copy has landed before the ring is reused or the CTA exits
            for (int s = 0; s < SPLIT_STAGES; ++s) {
                if (!((armed >> s) & 1)) continue;
                const unsigned long long t0 = globaltimer();
                while (!mbar_try_wait(&full[s], (parity >> s) & 1) && globaltimer() - t0 < kWaitLimitNs) {
                }
            }
        }
    } else if (warp == 1) {
        {
            const uint64_t da = sdesc_sw128(smem_u32(smem)), db = sdesc_sw128(smem_u32(smem) + A_BYTES);
            int stage = 0;
            uint32_t phase = 0;
            bool ok = true;                        // this lane's waits (elect_one)
            for (int kb = kb0; kb < kb1; ++kb) {
                ok = ok && mbar_wait(&full[stage], phase, abort_flag, g.err);
                tc_fence_after();
                if (elect_one() && ok) {
#pragma unroll
                    for (int k = 0; k < BK / 16; ++k)
                        tc_mma(tmem_base, sdesc_at(da, stage * SPLIT_STAGE_BYTES + k * 32),
                               sdesc_at(db, stage * SPLIT_STAGE_BYTES + k * 32), idesc_bf16(BM, SPLIT_BN),
                               (kb > kb0) || k != 0);
                    tc_commit(&empty[stage]);
                }
                __syncwarp();
                if (++stage == SPLIT_STAGES) { stage = 0; phase ^= 1u; }
            }
            if (elect_one()) tc_commit(tfull);
            __syncwarp();
            const unsigned long long t0 = globaltimer();
            while (!mbar_try_wait(tfull, 0) && globaltimer() - t0 < kWaitLimitNs) {
            }
        }
    }
    __syncthreads();          // this CTA's copies have landed and its MMAs are done
    tc_fence_after();
    const int Mp = prob ? g.M1 : g.M;
    const Epi e = problem_epilogue(g, prob);
    // this thread's items: 8-column groups of this CTA's share.  QKV takes one
    // row (V^T's rows are tokens: consecutive lanes store consecutively), the
    // other forms one group.
    constexpr int NG = SPLIT_BN / 8 / S;                      // groups in the share, = items a thread
    constexpr bool kByRow = FORM == kFormQKV;
    const int tid = threadIdx.x - 64;
    const int col_share = n_blk * SPLIT_BN + rank * (SPLIT_BN / S);
    auto item = [&](int i, int& row, int& grp) {
        row = kByRow ? tid : i * (BM / NG) + tid / NG;
        grp = kByRow ? i : tid % NG;
    };
    // residual rows, bias and gate are fetched before the barriers
    uint4 resid[is_resid(FORM) ? NG : 1];
    if (is_resid(FORM) && warp >= 2) {
#pragma unroll
        for (int i = 0; i < NG; ++i) {
            int row, grp;
            item(i, row, grp);
            const int m = m_blk * BM + row, col = col_share + grp * 8;
            if (m < Mp && col < g.N) resid[i] = residual8(e, m, col);
        }
    }
    float bias[8], gate[8];
    int col_of;
    {
        int row, grp;
        item(0, row, grp);
        col_of = min(col_share + grp * 8, g.N - 8);           // (clamped: a share may lie past N)
    }
    if (!kByRow && warp >= 2) columns8<FORM>(e, col_of, bias, gate);
    cluster_sync_all();       // so are the others': every ring is free
    if (warp >= 2) {
        const int lg = warp & 3, row = lg * 32 + lane;
        const uint32_t taddr = tmem_base + ((uint32_t)(lg * 32) << 16);
        constexpr int C4 = SPLIT_BN / S / 4;                  // 4-column groups in a share
#pragma unroll
        for (int c0 = 0; c0 < SPLIT_BN; c0 += 32) {
            uint32_t v[32];
            tmem_ld32(taddr + c0, v);
            tmem_ld_wait();
#pragma unroll
            for (int j = 0; j < 32; j += 4) {
                const int c4 = (c0 + j) / 4;
                st_shared_cluster_v4(mapa_shared(smem_u32(smem) + split_at<S>(rank, c4 % C4, row), c4 / C4), v[j],
                                     v[j + 1], v[j + 2], v[j + 3]);
            }
        }
        tc_fence_before();
    }
    cluster_sync_all();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, SPLIT_BN);
    }
    if (warp >= 2) {
#pragma unroll
        for (int i = 0; i < NG; ++i) {
            int row, grp;
            item(i, row, grp);
            const int m = m_blk * BM + row, col = col_share + grp * 8;
            float v[8];
#pragma unroll
            for (int p = 0; p < S; ++p) {
                const float4 x = *reinterpret_cast<const float4*>(smem + split_at<S>(p, 2 * grp, row));
                const float4 y = *reinterpret_cast<const float4*>(smem + split_at<S>(p, 2 * grp + 1, row));
                if (p == 0) {
                    v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
                    v[4] = y.x; v[5] = y.y; v[6] = y.z; v[7] = y.w;
                } else {
                    v[0] += x.x; v[1] += x.y; v[2] += x.z; v[3] += x.w;
                    v[4] += y.x; v[5] += y.y; v[6] += y.z; v[7] += y.w;
                }
            }
            if (kByRow) columns8<FORM>(e, min(col, g.N - 8), bias, gate);
            if (m < Mp && col < g.N) epilogue8<FORM>(e, m, col, v, bias, gate, resid[is_resid(FORM) ? i : 0]);
        }
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

using TileKernel = void (*)(const CUtensorMap, const CUtensorMap, const CUtensorMap, const CUtensorMap, const EpiMaps,
                            const EpiMaps, const GemmArgs);
using SplitKernel = void (*)(const CUtensorMap, const CUtensorMap, const CUtensorMap, const CUtensorMap, const GemmArgs);
template <int... F>
struct TileKernels {
    static constexpr TileKernel pair256[] = {gemm_tc2_kernel<256, F>...};
    static constexpr TileKernel pair192[] = {gemm_tc2_kernel<192, F>...};
    static constexpr TileKernel pair128[] = {gemm_tc2_kernel<128, F>...};
    static constexpr TileKernel one128[] = {gemm_tc_kernel<128, F>...};
    static constexpr TileKernel one64[] = {gemm_tc_kernel<64, F>...};
};
template <int... F>
struct SplitKernels {
    static constexpr SplitKernel split2[] = {gemm_split_kernel<F, 2>...};
    static constexpr SplitKernel split4[] = {gemm_split_kernel<F, 4>...};
    static constexpr SplitKernel split8[] = {gemm_split_kernel<F, 8>...};
};
struct Kernels : TileKernels<kFormStore, kFormGelu, kFormResid, kFormQKV, kFormUnpatch, kFormResidGelu, kFormResidRepeat>,
                 SplitKernels<kFormStore, kFormGelu, kFormResid, kFormQKV, kFormUnpatch, kFormResidGelu> {
    static TileKernel pair(int bn, int f) { return bn == 256 ? pair256[f] : (bn == 192 ? pair192[f] : pair128[f]); }
    static SplitKernel split(int S, int f) {
        if (f == kFormResidRepeat) f = kFormResid;         // reads its residual row by row, repeating or not
        return S == 2 ? split2[f] : (S == 4 ? split4[f] : split8[f]);
    }
};

int form_of(const Epi& e, int M) {
    switch (e.mode) {
        case kEpiResid:       // (repeating rows come from the patch embedding alone, without GELU)
            if (e.gelu) return kFormResidGelu;
            return e.res_rows > 0 && M > e.res_rows ? kFormResidRepeat : kFormResid;
        case kEpiQKV: return kFormQKV;
        case kEpiUnpatch: return kFormUnpatch;
        default: return e.gelu ? kFormGelu : kFormStore;
    }
}

size_t pair_smem(int bn) {
    return bn == 256 ? PairCfg<256>::SMEM : (bn == 192 ? PairCfg<192>::SMEM : PairCfg<128>::SMEM);
}

void set_attrs(const Ctx* c) {
    static PerDevice<bool> attr;
    attr.get(c->device, [](bool& ok) {
        ok = true;
        for (int f = 0; f < kForms; ++f) {
            for (int bn : {256, 192, 128}) ok &= allow_smem(Kernels::pair(bn, f), pair_smem(bn));
            ok &= allow_smem(Kernels::one128[f], GemmCfg<128>::SMEM);
            ok &= allow_smem(Kernels::one64[f], GemmCfg<64>::SMEM);
            for (int S = 2; S <= SPLIT_MAX; S *= 2) ok &= allow_smem(Kernels::split(S, f), SPLIT_SMEM);
        }
        return ok;
    });
}

// One launch: the kernel, its N tile and (split kernel) the CTAs a tile.
struct Choice {
    enum Kind { kPair, kOne128, kOne64, kSplit } kind;
    int bn = 256;
    int split = 1;
    wdc_gemm_kernel id() const {
        switch (kind) {
            case kPair: return bn == 256 ? WDC_GEMM_PAIR256 : (bn == 192 ? WDC_GEMM_PAIR192 : WDC_GEMM_PAIR128);
            case kSplit: return split == 2 ? WDC_GEMM_SPLIT2 : (split == 4 ? WDC_GEMM_SPLIT4 : WDC_GEMM_SPLIT8);
            default: return bn == 64 ? WDC_GEMM_ONE64 : WDC_GEMM_ONE128;
        }
    }
};

// Estimated cycles of a launch with `tiles` tiles on `units` SMs or pairs:
// `main` cycles of MMAs a tile, `epi` of epilogue behind them.
double launch_cycles(long long tiles, int units, double main, double epi) {
    const double waves = (double)((tiles + units - 1) / units);
    return main + epi + (waves - 1.0) * (main > epi ? main : epi);
}

// The kernel for a shape is the one with the least estimated cycles; the
// constants are fits to a sweep (us, store unless said; kb = 64-column blocks):
//                          pair 256   192   128  one128  one64  split 2 / 4
//   272 x 768 x 256             7.1   6.5   5.9     4.7    4.1    5.3 / 6.1
//   272 x 256 x 1024 resid     12.1                 8.3    7.1    7.4 / 7.2
//   226 x 3072 x 3072                              15.1   14.2   10.3 / 16.2
//   64 x 3072 x 8192                               33.7   31.3   17.6 / 12.3
//   700 x 1024 x 1024 resid    12.2  10.2   8.7     8.4    7.3    7.6 / 13.5
//   1600 x 1024 x 4096 resid   25.1  20.4  17.2    20.3   32.3   23.2 / 28.3
//   1600 x 3072 x 1024         14.6  12.9  13.8    16.1   21.8   28.6
//   6400 x 1024 x 4096 resid   44.0  37.0  40.9    51.5   90.4   70.3
//   3000 x 3072 x 3072         33.0  35.8  38.8    51.0   89.7   71.9
//   13568 x 3072 x 12288 res    591   613   715     852   1445    889
// A block of K takes a pair 560, 460 or 400 cycles (256 x 256, 192 or 128; the
// narrower, the less of it are MMAs), one CTA 470 (128 x 128) or 450 (128 x
// 64): the widest tile is the most efficient, a narrower one wins where its
// rounds fit the tiles better (6400 x 1024: 100 tiles of 256 on 76 pairs are
// two rounds, of which the second is a third full; 150 of 192 fill both), and
// a launch of few tiles takes as long in a narrow one.  The pair's cluster
// launch and wider tile cost 1900 more to start; the split kernel's two cluster
// barriers, exchange and epilogue 4300-6200, and it runs as many clusters at a
// time as the GPCs hold (76, 36 and 15 of 2, 4 and 8 on this part).
constexpr double kCyclesPair = 560.0, kCyclesPair192 = 460.0, kCyclesPair128 = 400.0, kPairStart = 1900.0;
constexpr double kCycles128 = 470.0, kCycles64 = 450.0, kCyclesSplit = 440.0;

// Fills in the clusters of `size` CTAs of a GEMM kernel resident at a time;
// false where that could not be asked and n is as many as the SMs would hold.
bool resident_clusters(const Ctx* c, const void* kernel, int size, size_t smem, int& n) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(c->num_sms / size * size, 1, 1);
    cfg.blockDim = dim3(kGemmThreads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = size;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) == cudaSuccess && n >= 1) return true;
    cudaGetLastError();
    n = c->num_sms / size > 0 ? c->num_sms / size : 1;
    return false;
}
int split_clusters(const Ctx* c, int S) {
    static PerDevice<int> cap[SPLIT_MAX + 1];
    return cap[S].get(c->device, [&](int& n) {
        return resident_clusters(c, (const void*)Kernels::split(S, 0), S, SPLIT_SMEM, n);
    });
}
int pair_clusters(const Ctx* c) {
    static PerDevice<int> cap;
    const int n = cap.get(c->device, [&](int& v) {
        return resident_clusters(c, (const void*)Kernels::pair(256, 0), 2, pair_smem(256), v);
    });
    return n < c->num_sms / 2 ? n : c->num_sms / 2;
}

// M, M1: the launch's rows (M1: a second problem's, or 0); sample, sample1:
// one sample's rows.  Whether and how K is split, which orders the sums,
// depends on one sample alone; the whole-K kernels sum alike.
Choice choose_gemm(Ctx* c, int form, int M, int M1, int sample, int sample1, int N, int K) {
    const int kb = (K + BK - 1) / BK, sms = c->num_sms;
    const bool plain = form == kFormStore || form == kFormQKV;
    const double chunk = plain ? 900.0 : 2000.0;              // epilogue of 64 columns
    auto tiles = [&](int rows, int rows1, int bm, int bn) {
        return (long long)((rows + bm - 1) / bm + (rows1 + bm - 1) / bm) * ((N + bn - 1) / bn);
    };
    auto whole = [&](int rows, int rows1, Choice* ch) {
        double best = 0;
        auto offer = [&](Choice::Kind kind, int bn, double est) {
            if (best > 0 && est >= best) return;
            best = est;
            ch->kind = kind;
            ch->bn = bn;
        };
        offer(Choice::kOne64, 64, launch_cycles(tiles(rows, rows1, BM, 64), sms, kb * kCycles64, chunk));
        offer(Choice::kOne128, 128, launch_cycles(tiles(rows, rows1, BM, 128), sms, kb * kCycles128, 2 * chunk));
        if (rows >= 256 && sms >= 2) {
            const double cycles[3] = {kCyclesPair, kCyclesPair192, kCyclesPair128};
            for (int i = 0; i < 3; ++i) {
                const int bn = 256 - 64 * i;
                offer(Choice::kPair, bn,
                      kPairStart + launch_cycles(tiles(rows, rows1, 256, bn), sms / 2, kb * cycles[i], bn / 64 * chunk));
            }
        }
        return best;
    };
    Choice ch{Choice::kPair};
    double least = 0.9 * whole(sample, sample1, &ch);         // (a split that gains less is not worth its risk)
    const long long t = tiles(sample, sample1, BM, SPLIT_BN);
    for (int S = 2; S <= SPLIT_MAX && 2 * S <= kb; S *= 2) {
        const int cap = split_clusters(c, S);
        const double reduce = (S == 8 ? 6200.0 : (S == 4 ? 4550.0 : 4300.0)) + (plain || form == kFormGelu ? 0.0 : 2000.0);
        const double est = (double)((t + cap - 1) / cap) * (((kb + S - 1) / S) * kCyclesSplit + reduce);
        if (est < least) {
            least = est;
            ch.kind = Choice::kSplit;
            ch.bn = SPLIT_BN;
            ch.split = S;
        }
    }
    if (ch.kind != Choice::kSplit) whole(M, M1, &ch);
    return ch;
}

// Tensor maps of an epilogue's staged stores and residual loads; staged = 0 when
// its form takes none (unpatchify).
bool encode_epilogue(const Epi& e, int M, int N, EpiMaps* m, int* staged, std::string* why) {
    *staged = 0;
    if (e.mode == kEpiUnpatch) return true;
    if (e.mode == kEpiQKV) {
        const uint64_t d = e.d, L = e.L, heads = (uint64_t)e.nb * e.H;
        if (!encode_tmap_3d(&m->out, e.q, d, L, heads, d * 2, L * d * 2, 64, 32, 1, why) ||
            !encode_tmap_3d(&m->res, e.k, d, L, heads, d * 2, L * d * 2, 64, 32, 1, why) ||
            !encode_tmap_3d(&m->vt, e.vt, L, d, heads, (uint64_t)e.ldv * 2, (uint64_t)e.ldv * d * 2, 32, 64, 1, why,
                            true, CU_TENSOR_MAP_SWIZZLE_64B))
            return false;
    } else {
        if (!encode_tmap_2d(&m->out, e.out, (uint64_t)N, (uint64_t)M, (uint64_t)e.ldo * 2, 64, 32, why)) return false;
        const int res_rows = e.res_rows > 0 && e.res_rows < M ? e.res_rows : M;
        if (e.mode == kEpiResid &&
            !encode_tmap_2d(&m->res, e.res, (uint64_t)N, (uint64_t)res_rows, (uint64_t)e.ldo * 2, 64, 32, why))
            return false;
    }
    *staged = 1;
    return true;
}

// A launch's two problems: operands, rows and epilogues (rows1 == 0: one).
struct Problem {
    const void *A, *W;
    int M, sample;
    const Epi* e;
};

wdc_status launch_gemm(Ctx* c, const Problem& p0, const Problem* p1, int N, int K, cudaStream_t s) {
    wdc_status st = check_operands(c, p0.A, p0.W, *p0.e);
    if (!st && p1) st = check_operands(c, p1->A, p1->W, *p1->e);
    if (st) return st;
    set_attrs(c);
    const int form = form_of(*p0.e, p0.M);
    const Choice ch = choose_gemm(c, form, p0.M, p1 ? p1->M : 0, p0.sample, p1 ? p1->sample : 0, N, K);
    const int bn = ch.bn;
    // W's box: the tile's width, or each CTA's half of it in a pair
    const uint32_t w_rows = ch.kind == Choice::kPair ? bn / 2 : bn;
    GemmArgs g{};
    g.M = p0.M;
    g.N = N;
    g.K = K;
    g.m_tiles = (p0.M + BM - 1) / BM;
    g.n_tiles = (N + bn - 1) / bn;
    g.k_blocks = (K + BK - 1) / BK;
    // raster groups: a W slab of at most ~40 MB per group (L2 is 126 MB,
    // shared with the streamed A and the output), as few groups as that
    // allows.  For deep K (> 4096) a 256-row slab of A is itself large
    // and re-reading A per group costs more than it saves (measured on the
    // 17776 x 3072 x 12288 MLP-down GEMM): plain N-fastest order there.
    g.group_n = g.n_tiles;
    if (K <= 4096) {
        const double slab_per_tile = (double)bn * K * 2.0;
        int gn = (int)(40.0e6 / slab_per_tile);
        gn = gn < 1 ? 1 : (gn > g.n_tiles ? g.n_tiles : gn);
        const int groups = (g.n_tiles + gn - 1) / gn;
        g.group_n = (g.n_tiles + groups - 1) / groups;  // balance the groups
    }
    g.e = *p0.e;
    g.err = c->err;
    g.nprob = p1 ? 2 : 1;
    std::string why;
    CUtensorMap ta, tb, ta1, tb1;
    EpiMaps maps{}, maps1{};
    auto encode = [&](const Problem& p, CUtensorMap* a, CUtensorMap* b, EpiMaps* m, int* staged) {
        return encode_tmap_2d(a, p.A, (uint64_t)K, (uint64_t)p.M, (uint64_t)K * 2, BK, BM, &why) &&
               encode_tmap_2d(b, p.W, (uint64_t)K, (uint64_t)N, (uint64_t)K * 2, BK, w_rows, &why) &&
               (ch.kind == Choice::kSplit || encode_epilogue(*p.e, p.M, N, m, staged, &why));
    };
    if (!encode(p0, &ta, &tb, &maps, &g.staged)) return fail(c, WDC_ERR_CUDA, why);
    if (p1) {
        g.M1 = p1->M;
        g.m_tiles1 = (p1->M + BM - 1) / BM;
        g.e1 = *p1->e;
        if (!encode(*p1, &ta1, &tb1, &maps1, &g.staged1)) return fail(c, WDC_ERR_CUDA, why);
    } else {
        ta1 = ta;
        tb1 = tb;
    }
    const int tiles128 = (g.m_tiles + g.m_tiles1) * g.n_tiles;
    switch (ch.kind) {
        case Choice::kPair: {
            // a persistent grid of as many CTA pairs as can be resident,
            // capped by the tile count
            const int resident = pair_clusters(c), tiles = ((g.m_tiles + 1) / 2 + (g.m_tiles1 + 1) / 2) * g.n_tiles;
            launch_kernel(Kernels::pair(bn, form), dim3(2 * (tiles < resident ? tiles : resident)), kGemmThreads,
                          pair_smem(bn), s, 2, ta, tb, ta1, tb1, maps, maps1, g);
            break;
        }
        case Choice::kSplit:
            launch_kernel(Kernels::split(ch.split, form), dim3(tiles128 * ch.split), kGemmThreads, SPLIT_SMEM, s,
                          ch.split, ta, tb, ta1, tb1, g);
            break;
        default:
            launch_kernel(bn == 64 ? Kernels::one64[form] : Kernels::one128[form],
                          dim3(tiles128 < c->num_sms ? tiles128 : c->num_sms), kGemmThreads,
                          bn == 64 ? GemmCfg<64>::SMEM : GemmCfg<128>::SMEM, s, 1, ta, tb, ta1, tb1, maps, maps1, g);
    }
    cudaError_t err = cudaGetLastError();
    if (err != cudaSuccess) return fail(c, WDC_ERR_CUDA, std::string("tcgen05 GEMM launch: ") + cudaGetErrorString(err));
    c->gemm_launches[ch.id() * kForms + form] += p1 ? 1ull << 32 : 1ull;
    return WDC_OK;
}

}  // namespace

// `sample`: the rows of one sample of a batch (M alone), see choose_gemm.
wdc_status tc_gemm(Ctx* c, const void* A, const void* W, int M, int N, int K, const Epi& e, int sample, cudaStream_t s) {
    return launch_gemm(c, Problem{A, W, M, sample, &e}, nullptr, N, K, s);
}

// Two GEMMs with the same N and K in one launch (the dual-stream blocks' video
// rows and condition rows): problem 1's tiles follow problem 0's, filling the
// SMs problem 0 leaves idle in its last wave.
wdc_status tc_gemm_grouped(Ctx* c, const void* A0, const void* W0, int M0, int sample0, const Epi& e0, const void* A1,
                           const void* W1, int M1, int sample1, const Epi& e1, int N, int K, cudaStream_t s) {
    if (M1 <= 0) return tc_gemm(c, A0, W0, M0, N, K, e0, sample0, s);
    if (M0 <= 0) return tc_gemm(c, A1, W1, M1, N, K, e1, sample1, s);
    const Problem p1{A1, W1, M1, sample1, &e1};
    return launch_gemm(c, Problem{A0, W0, M0, sample0, &e0}, &p1, N, K, s);
}

}  // namespace wdc
