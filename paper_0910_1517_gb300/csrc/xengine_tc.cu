// xengine_tc.cu -- X-engine on the tcgen05 tensor cores (sm_103a).
//
// Per channel k the visibilities are one dense contraction.  With the 2 n_in
// real rows A[r][t], r = 2i + c (c = 0 real, 1 imaginary part of Y_i[t]),
// the real Gram G = A A^T (K = n_int frames) holds every product:
//   Re V_ij = G[2i][2j] + G[2i+1][2j+1],  Im V_ij = G[2i+1][2j] - G[2i][2j+1].
// A is the F-engine's K-block layout, which already is the no-swizzle K-major
// canonical operand layout (core matrices of 8 rows x 16 bytes), so one
// TMA-engine bulk copy per stage lands a ready operand tile and the same shared
// memory tile serves as both A and B.
//
// Work items are (sub-array, channel, row block): 128 Gram rows a0..a0+127 against
// columns b0..b0+N-1.  Up to 128 rows need one item (N <= 128, the rest of the 128
// rows is ignored); 256 rows need two (rows 0-127 x columns 0-255, rows 128-255 x
// columns 128-255; gathered by TMA, the second's stages hold its rows alone).  A persistent CTA walks a cost-ordered item list; several
// sub-arrays of different sizes share one launch.
//
// Roles: warp 0 streams stages in (and owns the TMEM allocation), warp 1 issues
// tcgen05.mma from one elected lane.  One-plane forms (10 warps): warps 2-9 drain the
// accumulators (warp w reads TMEM lanes 32 (w % 4) .. + 31, i.e. Gram rows, and
// the column half (w - 2) / 4 of them; running sums in registers).  Converted forms
// (FP32 split, int8 bytes; 16 warps): the warpgroup of warps 4-7 drains (208 registers a
// thread hold a whole Gram row's running sums), warps 2, 3 and 8-15 convert the input
// stages (96 registers).
// What bounds the converted forms: at the GMRT shape (64 inputs, 1024 channels, 8192 spectra)
// the FP32 form takes 0.80 ms, where its 4.3 GB alone stream in 0.60 ms, its MMAs take 0.31 ms
// and its converters 0.57 ms, each role timed with the others idle; together they share the
// shared-memory pipe (per 64-frame stage: 32 KB landed, 32 read, 32 written, 48 of operands, and
// the drain's TMEM reads).  It was 0.93 ms with a second MMA a step (now T + T^T, write_pair),
// MMAs issued from a lane == 0 branch, one-lane waits and the running sums in shared memory.
// The int8 form takes 0.31 ms (0.45 before) and is paced by its TMA gather of 16-byte pieces, 0.31 ms
// alone (MMAs 0.21, converters 0.22).
// Accumulation is chunked: every `chunk` frames the FP32 accumulator is drained
// and added into a running sum.  Items with N <= 128 rotate over four 128-column
// accumulators (the MMAs run up to three chunks ahead of the drain) and keep the
// running sums in the draining threads' registers (one Gram row per thread);
// wider items use one accumulator of N columns and a running sum in TMEM
// (columns 256-511).  For int8-valued operands (chunk 1024) every product is an
// integer of magnitude at most 127^2 = 16129 and a chunk sum at most 1024 * 16129 =
// 16,516,096 < 2^24, so the FP32 accumulator is exact and the running sum is kept
// as int32: the result equals the integer MAC.
//
// int8 form with byte operands (in8): the F-engine wrote the int8 values as bytes, so each stage
// lands in an input slot at half the fp16 size and the converter warps of the FP32 form widen it
// to the fp16 operand tile (exact: the fp16 bits 0x6400 | (b ^ 0x80) hold 1152 + b, one packed
// subtraction leaves b); one MMA per 16-frame step, chunks of 1024 frames over four rotating
// accumulators, int32 running sums in registers (wider items: in TMEM).
//
// FP32 form: the stages hold FP32 spectra in the CUDA-core engine's layout; ten
// converter warps split each FP32 value v (scaled by a power of two) into fp16
// hi (v rounded to 11 significant bits) and lo = v - hi rounded to fp16, so
// |v - hi - lo| <= 2^-22 |v|, and write both planes as canonical operand tiles;
// each 16-frame step then issues three MMAs, H H^T + H L^T + L H^T (the dropped
// L L^T is below 2^-22 of the product).  The F-engine thus writes FP32 once and
// the X-engine reads it once.  fp16 x fp16 products are exact in FP32, but the
// tensor core's FP32 accumulation drops low bits of every partial sum, a
// loss that grows with the accumulator's size and the number of steps.  So the
// dominant H H^T term is accumulated in 128-frame chunks that the CUDA cores add
// in FP32.  Items of 128 rows (64 inputs, the usual shape) are "paired": the
// converters lay each K-block out as its 128 hi rows followed by its 128 lo rows, so
// that one N = 256 MMA a step forms [H H^T | H L^T] = H [H; L]^T.  L H^T is the
// transpose of H L^T, so the drain keeps T = H H^T / 2 + H L^T (FP32 running sums in
// registers, two 256-column chunk accumulators of 512 frames) and the finished item is
// G = T + T^T.  Other narrow items keep three MMAs: the cross terms,
// 2^-11 of H H^T, go to a separate accumulator over the whole integration (columns
// 256-383), two chunk accumulators alternate in columns 0-255 and the running sums sit
// in columns 384-511.
#include <cudaTypedefs.h>

#include "common.cuh"
#include "fengine.cuh"
#include "xengine.cuh"

namespace gbx {
namespace {

constexpr int kWarps1 = 10;                   // one-plane forms
constexpr int kWarps2 = 16;                   // FP32 form
constexpr int kEpiWarps1 = 8;                 // drain warps, one-plane forms (warps 2 .. 9)
constexpr int kEpiWarps2 = 4;                 // drain warps, converted forms (warps 4 .. 7, one warpgroup)
constexpr int kEpiThreads2 = kEpiWarps2 * 32;
constexpr int kConvWarps = 10;                // converter warps 2, 3 and 8 .. 15
constexpr int kConvThreads = kConvWarps * 32;
// Converted forms, registers a thread after setmaxnreg: a drain thread keeps its Gram row's 128
// running sums in registers, the other warps need few
constexpr int kRegsLaunch = 128, kRegsDrain = 208, kRegsOther = 96;
static_assert(kEpiThreads2 * kRegsDrain + (kWarps2 * 32 - kEpiThreads2) * kRegsOther <= kWarps2 * 32 * kRegsLaunch,
              "the split fits the launch's registers");
constexpr int kStages = 5;                    // fp16 operand slots (one-plane forms)
constexpr int kSlot = kStageMaxBytes + 2048;  // rows past R stay in bounds
constexpr int kTailSlack = 32768;
// FP32 form: stages of kStage2Bytes of FP32 each, three in flight.  An operand slot takes ks * 2 n_in * 4 bytes plus the rows the
// 128-row MMA reads past R; ks * rows_fp32(n_in) * 4 <= kStage2Bytes bounds that by
// kStage2Bytes + (128 - 64) * 16 (R < 64 leaves more room).
constexpr int kOpStages2 = 3;                 // operand slots ...
constexpr int kF32Stages = 3;                 // ... the FP32 slots after them ...
constexpr int kXchPitch = 129;                // ... and 16 rows of a paired item's sums (write_pair)
constexpr int kXchBytes = 16 * kXchPitch * 4;
// int8 form: four operand slots, then five input slots of kStage2Bytes / 2 (an int8 stage is half
// the size of its fp16 operand tile)
constexpr int kOpStagesI8 = 4;
constexpr int kRawI8 = 5;
constexpr int kRawPitch = kStage2Bytes / 2;
constexpr int kInSlots = kRawI8 > kF32Stages ? kRawI8 : kF32Stages;
constexpr int kSlot2 = kStage2Bytes + 1024;
constexpr int kXchOff = kOpStages2 * kSlot2 + kF32Stages * kStage2Bytes;
constexpr int smem_bytes(int form) {
    return form == XT_FORM_F16 ? kStages * kSlot + kTailSlack
         : form == XT_FORM_I8  ? kOpStagesI8 * kSlot2 + kRawI8 * kRawPitch
                               : kXchOff + kXchBytes;
}
static_assert(kOpStagesI8 <= kStages && kOpStages2 <= kStages, "barriers");
static_assert(smem_bytes(0) <= 226 * 1024 && smem_bytes(1) <= 226 * 1024 && smem_bytes(2) <= 226 * 1024, "shared memory");
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kColRun = 256;             // running-sum columns of wide items
constexpr int kAccBufs = 4;                   // 128-column accumulators of narrow items
constexpr uint32_t kColX = 256;               // FP32-form narrow items: the cross-term accumulator
constexpr uint32_t kColRun2 = 384;            // FP32-form narrow items: the running sums
constexpr int kXBit = 4;                      // the cross-term accumulator's parity bit in the phase words

struct Shared {
    uint64_t full[kStages];       // operand slot ready (bulk copy landed, or converted)
    uint64_t empty[kStages];      // operand slot consumed by the MMAs
    uint64_t f32full[kInSlots];     // input slot (FP32 or int8) landed
    uint64_t f32empty[kInSlots];    // input slot converted
    uint64_t accf[kAccBufs];
    uint64_t acce[kAccBufs];
    uint64_t xf;                  // cross-term accumulator complete (MMA -> epilogue)
    uint64_t xe;                  // cross-term accumulator drained (epilogue -> MMA)
    uint32_t taddr;
    int abort_flag;
    int consumed;                 // stages whose bulk copies the consumer has seen land
};

struct ItemGeo {
    int base;      // Gram row and column of the stage's first (a second item gathered by TMA has its own rows only)
    int sub, k, a0, b0, N, R, ntb, n_stage, n_chunk, nkb_stage;
    int Rp, tb32, ntb32;   // FP32 form: padded rows, frames per FP32 K-block, FP32 K-blocks per channel
    bool dbl;      // N <= 128: rotating 128-column accumulators
    bool sep;      // dbl and a converted form
    bool pair;     // sep, FP32 form, 128 rows: hi and lo rows of a K-block side by side, one N = 256 MMA
                   // H [H; L]^T per step into a 256-column chunk accumulator
    bool cross;    // sep and FP32 form otherwise: the cross terms in their own accumulator
    int nbuf;      // accumulators the item rotates over
};

__device__ __forceinline__ ItemGeo item_geo(const XtBatch& t, int it) {
    ItemGeo g;
    const int4 e = t.items[it];
    g.sub = e.x;
    g.k = e.y;
    const XtSub& s = t.sub[g.sub];
    g.R = 2 * s.n_in;
    const bool paired = g.R == 128;
    g.base = 0;
    g.a0 = 128 * e.z;
    if (e.z && (s.quad || s.in8)) {   // the stage holds these rows alone
        g.base = 128;
        g.R -= 128;
        g.a0 = 0;
    }
    g.b0 = (g.R > 128) ? g.a0 : 0;
    g.N = ((g.R - g.b0 + 15) / 16) * 16;
    g.Rp = rows_fp32(s.n_in);
    g.tb32 = tb_fp32(s.n_chan);
    g.ntb32 = s.n_int / g.tb32;
    g.dbl = g.N <= 128;
    g.sep = g.dbl && (s.spec32 != nullptr || s.in8);
    g.pair = g.sep && s.spec32 != nullptr && paired;
    g.cross = g.sep && s.spec32 != nullptr && !g.pair;
    g.nbuf = !g.dbl ? 1 : (g.sep && s.spec32 != nullptr ? 2 : kAccBufs);
    g.ntb = s.n_int / kTbHalf;
    g.nkb_stage = s.ks / kTbHalf;
    g.n_stage = (s.n_int + s.ks - 1) / s.ks;
    g.n_chunk = (s.n_int + s.chunk - 1) / s.chunk;
    return g;
}

// running sum + chunk sum: int32 for int8-valued operands (the FP32 chunk sum is an exact
// integer), FP32 otherwise
__device__ __forceinline__ uint32_t chunk_add(int exact, bool have, uint32_t run, uint32_t v) {
    if (exact) {
        const int x = __float2int_rn(__uint_as_float(v));
        return have ? static_cast<uint32_t>(static_cast<int>(run) + x) : static_cast<uint32_t>(x);
    }
    const float x = __uint_as_float(v);
    return __float_as_uint(have ? __uint_as_float(run) + x : x);
}

// Final sums of Gram row `row`, columns b0 + j0 .. b0 + j0 + W - 1 (every lane of the warp calls
// it): rows 2i and 2i+1 sit in adjacent lanes.  The even lane writes input pairs (i, j) for the
// first W/4 column pairs of the piece and the odd lane for the last W/4; per column pair each lane
// sends its partner the two sums the partner lacks.  With two polarisations and all products the
// entries of (j, j + 1), the two products of one baseline, go out as one 16-byte store.
template <int W>
__device__ __forceinline__ void write_piece(const XtSub& s, const ItemGeo& ig, int row, int j0,
                                            const uint32_t (&run)[W]) {
    constexpr int H = W / 2;                       // columns of the odd lane's half
    const int n_ant = s.n_ant, n_in = s.n_in, sh = s.n_pol - 1;        // n_pol is 1 or 2
    const int npp = s.self ? s.n_pol : s.n_pol * s.n_pol;
    const bool odd = row & 1, exact = s.exact, f32 = s.spec32 != nullptr, pair = sh && !s.self;
    const int i = row >> 1, a = i >> sh, pp = i & sh;
    const int64_t chan = static_cast<int64_t>(ig.k) * (n_ant * (n_ant + 1) / 2) * npp;
    float2* vis = s.vis + chan;
    int2* vis_int = exact && s.vis_int ? s.vis_int + chan : nullptr;
    const int row0 = a * n_ant - a * (a - 1) / 2 - a;                  // baseline (a, a2) is row0 + a2
    // requantisation scales through the read-only path: the loads of every column pair can then
    // issue together instead of one L2 round trip per output behind the previous stores
    const float* sc = s.scale + ig.k;
    const float si = (!f32 && i < n_in) ? __ldg(sc + static_cast<int64_t>(i) * s.n_chan) : 1.0f;
    float2 v[2];
    int2 vi[2];
#pragma unroll
    for (int jh = 0; jh < W / 4; ++jh) {
        const uint32_t r0 = __shfl_xor_sync(0xffffffffu, odd ? run[2 * jh] : run[2 * jh + H], 1);
        const uint32_t r1 = __shfl_xor_sync(0xffffffffu, odd ? run[2 * jh + 1] : run[2 * jh + H + 1], 1);
        const int j = ((ig.base + ig.b0 + j0) >> 1) + jh + (odd ? W / 4 : 0);
        // G[2i][2j], G[2i][2j+1], G[2i+1][2j], G[2i+1][2j+1]
        const uint32_t g_r0c0 = odd ? r0 : run[2 * jh];
        const uint32_t g_r0c1 = odd ? r1 : run[2 * jh + 1];
        const uint32_t g_r1c0 = odd ? run[2 * jh + H] : r0;
        const uint32_t g_r1c1 = odd ? run[2 * jh + H + 1] : r1;
        const int a2 = j >> sh, qq = j & sh, e = jh & 1;
        if (exact) {
            vi[e] = make_int2(static_cast<int>(g_r0c0) + static_cast<int>(g_r1c1),
                              static_cast<int>(g_r1c0) - static_cast<int>(g_r0c1));
            v[e] = make_float2(static_cast<float>(vi[e].x), static_cast<float>(vi[e].y));
        } else {
            v[e] = make_float2(__uint_as_float(g_r0c0) + __uint_as_float(g_r1c1),
                               __uint_as_float(g_r1c0) - __uint_as_float(g_r0c1));
        }
        if (i >= n_in || j >= n_in || a > a2) continue;
        if (f32) {
            v[e] = make_float2(v[e].x * s.descale, v[e].y * s.descale);
        } else {
            const float d = si * __ldg(sc + static_cast<int64_t>(j) * s.n_chan);
            v[e] = make_float2(v[e].x / d, v[e].y / d);
        }
        if (pair) {                                // j0 is a multiple of 16: j is even when e is 0
            if (e == 0) continue;
            const int o = (row0 + a2) * 4 + 2 * pp;
            *reinterpret_cast<float4*>(vis + o) = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
            if (vis_int) *reinterpret_cast<int4*>(vis_int + o) = make_int4(vi[0].x, vi[0].y, vi[1].x, vi[1].y);
        } else if (!s.self || pp == qq) {
            const int o = (row0 + a2) * npp + (s.self ? pp : 0);
            vis[o] = v[e];
            if (vis_int) vis_int[o] = vi[e];
        }
    }
}

// One chunk of a wide item (N > 128, one accumulator at column 0): add this thread's W-column
// pieces (j_first, j_first + j_step, ...) into the running sums at kColRun, or write the final
// sums after the last chunk.
template <int W>
__device__ __forceinline__ void drain_wide(const XtSub& s, const ItemGeo ig, uint32_t tm, int row, int j_first,
                                           int j_step, int chunk) {
    const bool last = chunk == ig.n_chunk - 1;
    for (int j0 = j_first; j0 < ig.N; j0 += j_step) {   // this warp's pieces
        uint32_t v[W], rs[W];
        if constexpr (W == 32) {
            tmem_ld32(tm + j0, v);
            if (chunk > 0) tmem_ld32(tm + kColRun + j0, rs);
        } else {
            tmem_ld16(tm + j0, v);
            if (chunk > 0) tmem_ld16(tm + kColRun + j0, rs);
        }
        tmem_wait_ld();
#pragma unroll
        for (int e = 0; e < W; ++e) rs[e] = chunk_add(s.exact, chunk > 0, rs[e], v[e]);
        if (!last) {
            if constexpr (W == 32) tmem_st32(tm + kColRun + j0, rs);
            else tmem_st16(tm + kColRun + j0, rs);
        } else {
            write_piece<W>(s, ig, row, j0, rs);
        }
    }
    if (!last) tmem_wait_st();
}

// One chunk of a three-product FP32 item (chunk accumulator b, running sums at kColRun2, cross terms
// at kColX): running sums += chunk, or after the last chunk + cross terms -> written.  (With the
// sums in registers, as in the other converted forms, small integrations ran up to 4 % slower.)
__device__ __forceinline__ void drain_split(const XtSub& s, const ItemGeo& ig, uint32_t tm, int row, int b, int chunk) {
    const bool last = chunk == ig.n_chunk - 1;
#pragma unroll 1
    for (int j0 = 0; j0 < ig.N; j0 += 16) {
        uint32_t v[16], rs[16];
        tmem_ld16(tm + b * 128 + j0, v);
        if (chunk > 0) tmem_ld16(tm + kColRun2 + j0, rs);
        tmem_wait_ld();
#pragma unroll
        for (int e = 0; e < 16; ++e) rs[e] = chunk_add(0, chunk > 0, rs[e], v[e]);
        if (!last) {
            tmem_st16(tm + kColRun2 + j0, rs);
        } else {
            tmem_ld16(tm + kColX + j0, v);
            tmem_wait_ld();
#pragma unroll
            for (int e = 0; e < 16; ++e) rs[e] = chunk_add(0, true, rs[e], v[e]);
            write_piece<16>(s, ig, row, j0, rs);
        }
    }
    if (!last) tmem_wait_st();
}

// One chunk of a paired or an int8 narrow item: the running sums of this thread's Gram row (+)= the
// N columns of the accumulator at TMEM address `acc`.  Paired items (PAIR): columns 0 .. 127 hold
// H H^T, 128 .. 255 hold H L^T, and T += H H^T / 2 + H L^T.
template <bool PAIR, int EXACT>
__device__ __forceinline__ void drain_row(uint32_t (&run)[128], uint32_t acc, int N, bool have) {
#pragma unroll
    for (int j0 = 0; j0 < 128; j0 += 16) {
        if (!PAIR && j0 >= N) break;
        uint32_t v[16];
        tmem_ld16(acc + j0, v);
        if constexpr (PAIR) {
            uint32_t x[16];
            tmem_ld16(acc + 128 + j0, x);
            tmem_wait_ld();
#pragma unroll
            for (int e = 0; e < 16; ++e)
                v[e] = __float_as_uint(fmaf(0.5f, __uint_as_float(v[e]), __uint_as_float(x[e])));
        } else {
            tmem_wait_ld();
        }
#pragma unroll
        for (int e = 0; e < 16; ++e) run[j0 + e] = chunk_add(EXACT, have, run[j0 + e], v[e]);
    }
}

// The finished item's sums back into the drained accumulator at TMEM address `acc`, from where the
// write loops take 16 columns at a time.  (Written from the registers the loops would have to be
// unrolled, and their instructions, used once an item, fetched from L2: 34 us an item.)
__device__ __forceinline__ void park_row(uint32_t acc, const uint32_t (&run)[128]) {
#pragma unroll
    for (int j0 = 0; j0 < 128; j0 += 16) {
        uint32_t v[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) v[e] = run[j0 + e];
        tmem_st16(acc + j0, v);
    }
    tmem_wait_st();
}

__device__ __forceinline__ void write_row(const XtSub& s, const ItemGeo& ig, int row, uint32_t acc) {
#pragma unroll 1
    for (int j0 = 0; j0 < ig.N; j0 += 16) {
        uint32_t rs[16];
        tmem_ld16(acc + j0, rs);
        tmem_wait_ld();
        write_piece<16>(s, ig, row, j0, rs);
    }
}

// The finished paired item's Gram G = T + T^T: every drain thread calls it with the sums of row lr,
// also parked at `acc`.  Sixteen rows at a time go through shared memory ([row][column], an odd
// pitch: conflict-free both ways), so that each thread reads its own column of them.
__device__ __forceinline__ void write_pair(const XtSub& s, const ItemGeo& ig, int lr, const uint32_t (&run)[128],
                                           uint32_t acc, uint32_t* xch) {
#pragma unroll 1
    for (int j0 = 0; j0 < 128; j0 += 16) {
        if ((lr & ~15) == j0) {
#pragma unroll
            for (int c = 0; c < 128; ++c) xch[(lr & 15) * kXchPitch + c] = run[c];
        }
        named_bar_sync(1, kEpiThreads2);
        uint32_t rs[16];
        tmem_ld16(acc + j0, rs);
        tmem_wait_ld();
#pragma unroll
        for (int e = 0; e < 16; ++e)
            rs[e] = __float_as_uint(__uint_as_float(rs[e]) + __uint_as_float(xch[e * kXchPitch + lr]));
        named_bar_sync(1, kEpiThreads2);
        write_piece<16>(s, ig, ig.a0 + lr, j0, rs);
    }
}

// run[0..63] (+)= this thread's 64 columns of the accumulator at TMEM address `col`
__device__ __forceinline__ void drain64(uint32_t (&run)[64], uint32_t col, bool have, int exact) {
#pragma unroll
    for (int h = 0; h < 4; ++h) {           // four 16-column loads
        uint32_t v[16];
        tmem_ld16(col + 16 * h, v);
        tmem_wait_ld();
        if (!have) {
#pragma unroll
            for (int e = 0; e < 16; ++e) run[16 * h + e] = chunk_add(exact, false, 0u, v[e]);
        } else if (exact) {
#pragma unroll
            for (int e = 0; e < 16; ++e) run[16 * h + e] = chunk_add(1, true, run[16 * h + e], v[e]);
        } else {
#pragma unroll
            for (int e = 0; e < 16; ++e) run[16 * h + e] = chunk_add(0, true, run[16 * h + e], v[e]);
        }
    }
}

// A drain warp has read an accumulator: it goes back to the MMA issuer (one arrival a warp)
__device__ __forceinline__ void release_acc(uint64_t* bar) {
    tc_fence_before();
    __syncwarp();
    if ((threadIdx.x & 31) == 0) mbar_arrive(bar);
}

// All chunks of a one-plane narrow item (N <= 128): chunk c (global chunk count cc + c) sits in
// accumulator (cc + c) % nbuf; the running sums of this thread's row and 64-column half stay in
// registers and are written after the last chunk.  `par`
// holds the accumulators' phase bits and is updated; false if a wait ran out.
__device__ __forceinline__ bool drain_narrow(Shared& sh, const XtSub& s, const ItemGeo ig, uint32_t tm, int row,
                                             int half, int cc, uint32_t& par, unsigned* err) {
    const int c0 = 64 * half;
    uint32_t run[64];
#pragma unroll
    for (int e = 0; e < 64; ++e) run[e] = 0u;
    for (int chunk = 0; chunk < ig.n_chunk; ++chunk) {
        const int b = (cc + chunk) % ig.nbuf;
        if (!mbar_wait_warp(&sh.accf[b], (par >> b) & 1, err, ERR_WAIT_MMA)) return false;
        par ^= 1u << b;
        tc_fence_after();
        if (c0 < ig.N) drain64(run, tm + b * 128 + c0, chunk > 0, s.exact);
        release_acc(&sh.acce[b]);
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        if (c0 + 32 * j < ig.N) {
            uint32_t piece[32];
#pragma unroll
            for (int e = 0; e < 32; ++e) piece[e] = run[32 * j + e];
            write_piece<32>(s, ig, row, c0 + 32 * j, piece);
        }
    }
    return true;
}

// Veltkamp's split of the pair v = w sc (both lanes at once; each packed operation rounds as its
// scalar counterpart): hi = v rounded to 11 significant bits (2^13 + 1), lo = v - hi exactly; both
// as fp16 pairs.  The power-of-two scale rides on the operations: k8193 = 8193 sc.
__device__ __forceinline__ void split_pair(float2 w, float2 sc, float2 nsc, float2 k8193, uint32_t& hw, uint32_t& lw) {
    const float2 m1 = make_float2(-1.0f, -1.0f);
    const float2 tt = __fmul2_rn(w, k8193);
    const float2 d = __ffma2_rn(w, nsc, tt);                        // tt - v
    const float2 nh = __ffma2_rn(tt, m1, d);                        // -hi = (tt - v) - tt
    const float2 lv = __ffma2_rn(w, sc, nh);                        // v - hi
    const __half2 hh = __floats2half2_rn(-nh.x, -nh.y);
    const __half2 ll = __floats2half2_rn(lv.x, lv.y);
    hw = *reinterpret_cast<const uint32_t*>(&hh);
    lw = *reinterpret_cast<const uint32_t*>(&ll);
}

// The converter warps: input slot g % nin becomes operand slot g % nop.  Work units, strided over
// the converter threads (a stage has at most kUnits per thread, so that a thread first loads all
// its units, while the operand slot may still be read by the tensor core, then converts and stores
// them: their latencies overlap, and none is left of a remainder loop):
//   int8 bytes [kb][R rows][8 frames]: unit u = j R + r, 8 bytes, becomes the 16-byte row r of K-block
//     j of the fp16 operand tile
//   FP32, channel-quad stage [kb][R rows][8 frames]: unit u = (j R + r) 2 + h, frames 4h .. 4h + 3 of
//     row r in K-block j (one 16-byte load; consecutive units, consecutive bytes), whose hi and lo
//     halves (8 bytes each) go into row r of K-block j of the two operand tiles
//   FP32, CUDA-core layout: unit u = j R + r, frames 8j .. 8j + 7 of row r (two 16-byte granules).
// FP32 values are scaled by the power of two split_scale, hi rounded to fp16 and lo the remainder
// rounded to fp16 (split_pair); the lo tile follows the hi tile, or in paired items (128 rows)
// K-block j holds 128 hi rows then 128 lo rows (4096 bytes).
// Each converter warp works on its own units and signals on its own: the whole warp waits for the
// slots by vote, converts, fences its shared stores for the tensor core's (async) proxy, and
// lane 0 arrives on both slots' barriers, which complete after all kConvWarps warps.  No barrier spans warps.  The body is inlined: called as a function, its
// shared-memory accesses cost about twice the time.
template <bool kIn8, bool kPairs>
__device__ __forceinline__ void convert_stages(const XtBatch& t, Shared& sh, unsigned char* smem, int ct) {
    constexpr int nop = kIn8 ? kOpStagesI8 : kOpStages2;      // operand slots
    constexpr int nin = kIn8 ? kRawI8 : kF32Stages, pin = kIn8 ? kRawPitch : kStage2Bytes;   // input slots
    constexpr int kUnits = (kStage2Bytes / 16 + kConvThreads - 1) / kConvThreads;
    constexpr int kUnits8 = (kStage2Bytes / 32 + kConvThreads - 1) / kConvThreads;   // two-granule units
    volatile int* abort_flag = &sh.abort_flag;
    const int lane = ct & 31;
    int g = 0;
    for (int it = blockIdx.x; it < t.n_items; it += gridDim.x) {
        const ItemGeo ig = item_geo(t, it);
        const XtSub& s = t.sub[ig.sub];
        const int R = ig.R, Rp = ig.Rp, tb = ig.tb32;
        const float2 sc = make_float2(s.split_scale, s.split_scale), nsc = make_float2(-sc.x, -sc.x);
        const float2 k8 = make_float2(8193.0f * sc.x, 8193.0f * sc.x);
        const int lo_off = kPairs ? 2048 : ig.nkb_stage * R * 16;
        const bool quad = s.quad;
        const int n_int = s.n_int, ks = s.ks;
        // unit ct of a stage as (K-block j0, row r0), and the step of kConvThreads units
        const int r0 = ct % R, j0 = ct / R, dr = kConvThreads % R, dj = kConvThreads / R;
        for (int st = 0; st < ig.n_stage; ++st, ++g) {
            const int fs = g % nin, os = g % nop;
            auto wait = [&](uint64_t* bar, uint32_t parity, unsigned bit) {
                if (mbar_wait_warp(bar, parity, t.err, bit)) return true;
                *abort_flag = 1;
                return false;
            };
            auto wait_in = [&]() { return wait(&sh.f32full[fs], (g / nin) & 1, ERR_WAIT_STAGE); };
            auto wait_op = [&]() { return wait(&sh.empty[os], ((g / nop) & 1) ^ 1, ERR_WAIT_MMA); };
            if (!wait_in()) return;
            const int kbs = min(ks, n_int - st * ks) / 8;        // K-blocks of this stage
            const unsigned char* src = smem + nop * kSlot2 + fs * pin;
            unsigned char* dst = smem + os * kSlot2;
            if constexpr (kIn8) {
                uint2 q[kUnits];
                const int units = kbs * R;
#pragma unroll
                for (int i = 0; i < kUnits; ++i) {
                    const int u = ct + i * kConvThreads;
                    q[i] = u < units ? *reinterpret_cast<const uint2*>(src + 8 * u) : make_uint2(0u, 0u);
                }
                if (!wait_op()) return;
                const __half2 bias = __float2half2_rn(1152.0f);
#pragma unroll
                for (int i = 0; i < kUnits; ++i) {
                    const uint32_t x[2] = {q[i].x ^ 0x80808080u, q[i].y ^ 0x80808080u};
                    uint32_t w[4];
#pragma unroll
                    for (int m = 0; m < 4; ++m) {   // bytes 2m, 2m + 1 -> fp16 1152 + b -> b
                        const uint32_t hb = __byte_perm(x[m >> 1], 0x64646464u, (m & 1) ? 0x4342 : 0x4140);
                        const __half2 v = __hsub2(*reinterpret_cast<const __half2*>(&hb), bias);
                        w[m] = *reinterpret_cast<const uint32_t*>(&v);
                    }
                    const int u = ct + i * kConvThreads;
                    if (u < units) *reinterpret_cast<uint4*>(dst + 16 * u) = make_uint4(w[0], w[1], w[2], w[3]);
                }
            } else if (quad) {
                float4 q[kUnits];
                const int units = kbs * R * 2;
#pragma unroll
                for (int i = 0; i < kUnits; ++i) {
                    const int u = ct + i * kConvThreads;
                    q[i] = u < units ? *reinterpret_cast<const float4*>(src + 16 * u) : make_float4(0.f, 0.f, 0.f, 0.f);
                }
                if (!wait_op()) return;
#pragma unroll
                for (int i = 0; i < kUnits; ++i) {
                    const int u = ct + i * kConvThreads;
                    uint32_t hw[2], lw[2];
                    split_pair(make_float2(q[i].x, q[i].y), sc, nsc, k8, hw[0], lw[0]);
                    split_pair(make_float2(q[i].z, q[i].w), sc, nsc, k8, hw[1], lw[1]);
                    unsigned char* d = dst + u * 8 + (kPairs ? (u >> 8) * 2048 : 0);
                    if (u < units) {
                        *reinterpret_cast<uint2*>(d) = make_uint2(hw[0], hw[1]);
                        *reinterpret_cast<uint2*>(d + lo_off) = make_uint2(lw[0], lw[1]);
                    }
                }
            } else {
                // (TB 8: rows r and r + 4 of a row group read opposite halves first, so that the 8 rows of a
                // quarter warp hit 8 distinct bank groups)
                float4 q[kUnits8][2];
                const int units = kbs * R;
                {
                    int r = r0, j = j0;
#pragma unroll
                    for (int i = 0; i < kUnits8; ++i) {
                        const bool sw = tb == 8 && ((r >> 2) & 1);
                        const int oa = fp32_off(r, sw ? 4 : 0, tb);
                        const int ob = tb == 8 ? fp32_off(r, sw ? 0 : 4, 8) : Rp * 4 + oa;
                        const float* p = reinterpret_cast<const float*>(src) + j * 8 * Rp;
                        if (ct + i * kConvThreads < units) {
                            const float4 qa = *reinterpret_cast<const float4*>(p + oa);
                            const float4 qb = *reinterpret_cast<const float4*>(p + ob);
                            q[i][0] = sw ? qb : qa;
                            q[i][1] = sw ? qa : qb;
                        } else {
                            q[i][0] = q[i][1] = make_float4(0.f, 0.f, 0.f, 0.f);
                        }
                        r += dr;
                        j += dj;
                        if (r >= R) {
                            r -= R;
                            ++j;
                        }
                    }
                }
                if (!wait_op()) return;
#pragma unroll
                for (int i = 0; i < kUnits8; ++i) {
                    const int u = ct + i * kConvThreads;
                    uint32_t hw[4], lw[4];
                    split_pair(make_float2(q[i][0].x, q[i][0].y), sc, nsc, k8, hw[0], lw[0]);
                    split_pair(make_float2(q[i][0].z, q[i][0].w), sc, nsc, k8, hw[1], lw[1]);
                    split_pair(make_float2(q[i][1].x, q[i][1].y), sc, nsc, k8, hw[2], lw[2]);
                    split_pair(make_float2(q[i][1].z, q[i][1].w), sc, nsc, k8, hw[3], lw[3]);
                    unsigned char* d = dst + u * 16 + (kPairs ? (u >> 7) * 2048 : 0);
                    if (u < units) {
                        *reinterpret_cast<uint4*>(d) = make_uint4(hw[0], hw[1], hw[2], hw[3]);
                        *reinterpret_cast<uint4*>(d + lo_off) = make_uint4(lw[0], lw[1], lw[2], lw[3]);
                    }
                }
            }
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) {
                if (ct == 0) sh.consumed = g + 1;                // this input copy has landed
                mbar_arrive(&sh.f32empty[fs]);
                mbar_arrive(&sh.full[os]);
            }
        }
    }
}

// kForm: XT_FORM_F16 (one plane, copied straight into the operand slots), XT_FORM_F32 (FP32 split),
// XT_FORM_F32P (the same, paired items: 64 inputs), XT_FORM_I8 (int8 bytes widened); one instantiation per form keeps every role's branches static
template <int kForm>
__global__ void __launch_bounds__((kForm != XT_FORM_F16 ? kWarps2 : kWarps1) * 32, 1)
    xengine_tc_kernel(const XtBatch* __restrict__ tab) {
    constexpr bool kF32 = kForm != XT_FORM_F16;   // a converted form
    constexpr bool kIn8 = kForm == XT_FORM_I8;
    constexpr bool kPairs = kForm == XT_FORM_F32P;   // every item is paired
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ Shared sh;
    const XtBatch& t = *tab;
    const int warp = __shfl_sync(0xffffffffu, static_cast<int>(threadIdx.x) / 32, 0), lane = threadIdx.x % 32;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&sh.full[s], kF32 ? kConvWarps : 1);   // converted by every converter warp, or one copy
            mbar_init(&sh.empty[s], 1);
        }
        for (int s = 0; s < kInSlots; ++s) {
            mbar_init(&sh.f32full[s], 1);
            mbar_init(&sh.f32empty[s], kConvWarps);
        }
        for (int b = 0; b < kAccBufs; ++b) {
            mbar_init(&sh.accf[b], 1);
            mbar_init(&sh.acce[b], kF32 ? kEpiWarps2 : kEpiWarps1);
        }
        mbar_init(&sh.xf, 1);
        mbar_init(&sh.xe, kEpiWarps2);
        fence_mbar_init();
        sh.abort_flag = 0;
        sh.consumed = 0;
    }
    if (warp == 0) {
        tmem_alloc(&sh.taddr, kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, sh.taddr, 0);
    volatile int* abort_flag = &sh.abort_flag;

    // ---------------------------------------------------------------- drain (warps 2..9, or 4..7)
    const bool drains = kF32 ? (warp >> 2) == 1 : warp >= 2;
    if (drains) {
        if constexpr (kF32) reg_alloc<kRegsDrain>();
        const int q = warp & 3;                   // TMEM lane quarter this warp may access
        const int lrow = 32 * q + lane;           // row within the item's 128 rows = TMEM lane
        const uint32_t tm = tmem + (static_cast<uint32_t>(32 * q) << 16);
        int cc = 0;
        uint32_t par = 0;                         // bit b: parity of accumulator b's uses so far
        bool go = true;                           // (a warp's waits, and a paired table's drain warps, agree)
        for (int it = blockIdx.x; it < t.n_items && go; it += gridDim.x) {
            const ItemGeo ig = item_geo(t, it);
            const XtSub& s = t.sub[ig.sub];
            const int row = ig.base + ig.a0 + lrow;
            if (kForm == XT_FORM_F32 && ig.sep) {   // three products
                for (int chunk = 0; chunk < ig.n_chunk; ++chunk, ++cc) {
                    const int b = cc % ig.nbuf;
                    const bool last = chunk == ig.n_chunk - 1;
                    go = mbar_wait_warp(&sh.accf[b], (par >> b) & 1, t.err, ERR_WAIT_MMA) &&
                         (!last || mbar_wait_warp(&sh.xf, (par >> kXBit) & 1, t.err, ERR_WAIT_MMA));
                    if (!go) break;
                    par ^= 1u << b;
                    if (last) par ^= 1u << kXBit;
                    tc_fence_after();
                    drain_split(s, ig, tm, row, b, chunk);
                    release_acc(&sh.acce[b]);
                    if (last) release_acc(&sh.xe);
                }
            } else if (kPairs || (kIn8 && ig.sep)) {   // running sums in registers
                uint32_t run[128];
                int b = 0;
                for (int chunk = 0; chunk < ig.n_chunk; ++chunk, ++cc) {
                    if (chunk > 0) release_acc(&sh.acce[b]);
                    b = cc % ig.nbuf;
                    go = mbar_wait_warp(&sh.accf[b], (par >> b) & 1, t.err, ERR_WAIT_MMA);
                    if (kPairs)   // its drain threads trade their sums: they stop together
                        go = !named_bar_or(1, kEpiThreads2, !go);
                    if (!go) break;
                    par ^= 1u << b;
                    tc_fence_after();
                    if (kPairs)
                        drain_row<true, 0>(run, tm + b * 256, 128, chunk > 0);
                    else
                        drain_row<false, kIn8 ? 1 : 0>(run, tm + b * 128, ig.N, chunk > 0);
                }
                if (!go) break;
                const uint32_t acc = tm + b * (kPairs ? 256 : 128);   // the last chunk's, still held
                park_row(acc, run);
                if (kPairs)
                    write_pair(s, ig, lrow, run, acc, reinterpret_cast<uint32_t*>(smem + kXchOff));
                else
                    write_row(s, ig, row, acc);
                release_acc(&sh.acce[b]);
            } else if (!kF32 && ig.dbl) {
                go = drain_narrow(sh, s, ig, tm, row, (warp - 2) >> 2, cc, par, t.err);
                cc += ig.n_chunk;
            } else if constexpr (!kPairs) {
                for (int chunk = 0; chunk < ig.n_chunk; ++chunk, ++cc) {
                    go = mbar_wait_warp(&sh.accf[0], par & 1, t.err, ERR_WAIT_MMA);
                    if (!go) break;
                    par ^= 1u;
                    tc_fence_after();
                    if constexpr (kF32) drain_wide<16>(s, ig, tm, row, 0, 16, chunk);
                    else drain_wide<32>(s, ig, tm, row, 32 * ((warp - 2) >> 2), 64, chunk);
                    release_acc(&sh.acce[0]);
                }
            }
        }
        if (!go) *abort_flag = 1;
    } else {
    if constexpr (kF32) reg_dealloc<kRegsOther>();
    if (warp == 0) {
        // ------------------------------------------------------------ producer
        if (lane == 0) {
            constexpr bool f32 = kF32;
            constexpr bool in8 = kIn8;
            const int nsl = f32 ? (in8 ? kRawI8 : kF32Stages) : kStages;
            uint64_t* fullb = f32 ? sh.f32full : sh.full;
            uint64_t* emptyb = f32 ? sh.f32empty : sh.empty;
            unsigned char* slots = f32 ? smem + (in8 ? kOpStagesI8 : kOpStages2) * kSlot2 : smem;
            const int pitch = f32 ? (in8 ? kRawPitch : kStage2Bytes) : kSlot;
            int g = 0;
            for (int it = blockIdx.x; it < t.n_items && !*abort_flag; it += gridDim.x) {
                const ItemGeo ig = item_geo(t, it);
                const XtSub& s = t.sub[ig.sub];
                for (int st = 0; st < ig.n_stage; ++st, ++g) {
                    const int slot = g % nsl;
                    if (!mbar_wait(&emptyb[slot], ((g / nsl) & 1) ^ 1, t.err, ERR_WAIT_MMA)) {
                        *abort_flag = 1;
                        break;
                    }
                    unsigned char* dst = slots + slot * pitch;
                    if (f32 && s.quad) {
                        // channel-quad layout: one 5-D tensor copy gathers the stage's pieces of channel k
                        // (a last, shorter stage reads zeros past the end and counts the whole box)
                        const CUtensorMap* map = ig.base ? &s.tmap_hi : &s.tmap;
                        if (st == 0) tmap_acquire(map);
                        const int nkb = s.ks / kTbHalf;
                        mbar_arrive_expect_tx(&fullb[slot], static_cast<uint32_t>(nkb) * ig.R * 32);
                        tma_load_5d(dst, map, 0, ig.k & 3, 0, st * nkb, ig.k >> 2, &fullb[slot]);
                    } else if (f32 && in8) {
                        // channel-quad int8 bytes: one 5-D tensor copy gathers the stage's 16-byte pieces
                        // of channel k into [kb][2 n_in rows][8 bytes] (half the fp16 bytes)
                        const CUtensorMap* map = ig.base ? &s.tmap_hi : &s.tmap;
                        if (st == 0) tmap_acquire(map);
                        const int nkb = s.ks / kTbHalf;
                        mbar_arrive_expect_tx(&fullb[slot], static_cast<uint32_t>(nkb) * ig.R * 8);
                        tma_load_5d(dst, map, 0, ig.k & 3, 0, st * nkb, ig.k >> 2, &fullb[slot]);
                    } else if (f32) {
                        // the stage's FP32 K-blocks of channel k are contiguous
                        const int frames = min(s.ks, s.n_int - st * s.ks);
                        const uint32_t bytes = static_cast<uint32_t>(frames) * ig.Rp * 4;
                        const float* src = s.spec32 +
                            (static_cast<int64_t>(ig.k) * ig.ntb32 + st * (s.ks / ig.tb32)) * ig.Rp * ig.tb32;
                        mbar_arrive_expect_tx(&fullb[slot], bytes);
                        bulk_g2s(dst, src, bytes, &fullb[slot]);
                    } else {
                        const int kb0 = st * ig.nkb_stage;
                        const int nkb = min(ig.nkb_stage, ig.ntb - kb0);
                        const uint32_t bytes = static_cast<uint32_t>(nkb) * ig.R * 16;
                        const int64_t off = (static_cast<int64_t>(ig.k) * ig.ntb + kb0) * ig.R * kTbHalf;
                        mbar_arrive_expect_tx(&fullb[slot], bytes);
                        bulk_g2s(dst, s.spec + off, bytes, &fullb[slot]);
                    }
                }
            }
            // let every issued copy land before the CTA can exit
            for (int q = *(volatile int*)&sh.consumed; q < g; ++q)
                mbar_wait(&fullb[q % nsl], (q / nsl) & 1, nullptr, 0);
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer
        // The whole warp runs the loop on warp-uniform values and one elected lane issues, the stage's
        // MMAs unrolled and their descriptors stepped by one addition: the tensor core takes a
        // 128 x 128 x 16 MMA every 64 cycles and a 128 x 256 x 16 one every 128 that way.  Issued in
        // a loop from a `lane == 0` branch, where each instruction's operands are first moved to
        // uniform registers, either came every 129 cycles at best (MMAs alone) and every 220 to 270
        // here (int8 form, MMAs alone: 0.36 -> 0.23 ms).
        int g = 0, cc = 0;
        uint32_t par = 0;                     // bit b: parity of accumulator b's uses so far
        int prev_nbuf = -1;
        constexpr int nsl = kF32 ? (kIn8 ? kOpStagesI8 : kOpStages2) : kStages;
        // the decision to go on is the warp's
        auto wait = [&](uint64_t* bar, uint32_t parity, unsigned bit) {
            if (mbar_wait_warp(bar, parity, t.err, bit)) return true;
            *abort_flag = 1;
            return false;
        };
        const uint32_t smem0 = __shfl_sync(0xffffffffu, smem_u32(smem), 0);
        bool go = true;
        for (int it = blockIdx.x; it < t.n_items && go; it += gridDim.x) {
            const ItemGeo ig = item_geo(t, it);
            const XtSub& s = t.sub[ig.sub];
            const uint32_t idesc = __shfl_sync(0xffffffffu, idesc_f16_f32(128, kPairs ? 256 : ig.N), 0);
            // K-blocks of a paired item: 128 hi rows then 128 lo rows (LBO 4096 bytes)
            const uint32_t lbo = __shfl_sync(0xffffffffu, kPairs ? 4096u : static_cast<uint32_t>(ig.R) * 16, 0);
            const uint32_t offa = __shfl_sync(0xffffffffu, static_cast<uint32_t>(ig.a0) * 16, 0);
            const uint32_t offb = __shfl_sync(0xffffffffu, static_cast<uint32_t>(ig.b0) * 16, 0);
            const uint32_t lo_off = __shfl_sync(0xffffffffu, static_cast<uint32_t>(ig.nkb_stage) * ig.R * 16, 0);
            const uint64_t kstep = (2 * lbo) >> 4;    // 16 frames on, in descriptor units
            const int stages_per_chunk = s.chunk / s.ks;
            bool xfirst = true;                   // next cross-term MMA starts the accumulator
            if (ig.cross) {                       // the previous item's cross terms are drained
                if (!(go = wait(&sh.xe, ((par >> kXBit) & 1) ^ 1, ERR_WAIT_EPI))) break;
                par ^= 1u << kXBit;
            }
            for (int chunk = 0; chunk < ig.n_chunk && go; ++chunk, ++cc) {
                const int b = cc % ig.nbuf;
                // a single-buffered item, or a change of buffering, needs every earlier drain done
                if (!ig.dbl || prev_nbuf != ig.nbuf) {
                    for (int q = 0; q < kAccBufs && go; ++q) go = wait(&sh.acce[q], ((par >> q) & 1) ^ 1, ERR_WAIT_EPI);
                    // (columns 256-383 may have held cross terms; a sep item already waited)
                    if (go && !ig.cross) go = wait(&sh.xe, ((par >> kXBit) & 1) ^ 1, ERR_WAIT_EPI);
                } else {
                    go = wait(&sh.acce[b], ((par >> b) & 1) ^ 1, ERR_WAIT_EPI);
                }
                prev_nbuf = ig.nbuf;
                if (!go) break;
                par ^= 1u << b;
                tc_fence_after();
                const uint32_t dcol = __shfl_sync(0xffffffffu, tmem + (ig.dbl ? b * (kPairs ? 256 : 128) : 0), 0);
                const uint32_t xcol = ig.sep ? tmem + kColX : dcol;
                const int st0 = chunk * stages_per_chunk;
                const int st1 = min(ig.n_stage, st0 + stages_per_chunk);
                bool first = true;
                for (int st = st0; st < st1; ++st, ++g) {
                    const int slot = g % nsl;
                    if (!(go = wait(&sh.full[slot], (g / nsl) & 1, ERR_WAIT_STAGE))) break;
                    tc_fence_after();
                    const int nk = min(ig.nkb_stage, ig.ntb - st * ig.nkb_stage) / 2;   // 16-frame steps
                    const uint32_t base = smem0 + slot * (kF32 ? kSlot2 : kSlot);
                    uint64_t da = smem_desc_noswizzle(base + offa, lbo, 128);
                    uint64_t db = smem_desc_noswizzle(base + offb, lbo, 128);
                    if (elect_one()) {
                        if (kForm == XT_FORM_F32) {
                            uint64_t la = smem_desc_noswizzle(base + lo_off + offa, lbo, 128);
                            uint64_t lb = smem_desc_noswizzle(base + lo_off + offb, lbo, 128);
#pragma unroll 2
                            for (int kk = 0; kk < nk; ++kk) {
                                umma_f16(dcol, da, db, idesc, (first && kk == 0) ? 0u : 1u);
                                umma_f16(xcol, da, lb, idesc, (ig.sep && xfirst && kk == 0) ? 0u : 1u);   // H L^T
                                umma_f16(xcol, la, db, idesc, 1u);                                         // L H^T
                                da += kstep;
                                db += kstep;
                                la += kstep;
                                lb += kstep;
                            }
                        } else {
                            // one product; paired items: [H H^T | H L^T] = H [H; L]^T (N = 256)
#pragma unroll 4
                            for (int kk = 0; kk < nk; ++kk) {
                                umma_f16(dcol, da, db, idesc, (first && kk == 0) ? 0u : 1u);
                                da += kstep;
                                db += kstep;
                            }
                        }
                        umma_commit(&sh.empty[slot]);   // frees the stage once these MMAs finish
                        if (!kF32) sh.consumed = g + 1;
                    }
                    __syncwarp();
                    first = false;
                    xfirst = false;
                }
                if (!go) break;
                if (elect_one()) umma_commit(&sh.accf[b]);   // chunk complete
                __syncwarp();
            }
            if (!go) break;
            if (ig.cross) {                                  // cross terms complete
                if (elect_one()) umma_commit(&sh.xf);
                __syncwarp();
            }
        }
    } else if (kF32) {
        // ------------------------------------------------------------ converters
        convert_stages<kIn8, kPairs>(t, sh, smem, static_cast<int>(threadIdx.x) - (warp < 4 ? 64 : 192));
    }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem, kTmemCols);
    }
}

}  // namespace

bool xengine_tc_encode_quad(XtSub& x) {
    const bool b8 = x.in8 != 0;                    // int8 bytes (16-byte pieces) or FP32 (64-byte pieces)
    static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
    if (!encode) {
        cudaDriverEntryPointQueryResult q{};
        void* fn = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess || !fn)
            return false;
        encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    }
    const cuuint64_t ntb = static_cast<cuuint64_t>(x.n_int / kTbHalf);
    const cuuint64_t piece = b8 ? 16 : 64;         // bytes of one (channel, K-block, input) piece
    const cuuint64_t stride[4] = {piece, 4 * piece, 4 * piece * x.n_in, 4 * piece * x.n_in * ntb};   // bytes, dims 1..4
    const cuuint32_t estride[5] = {1, 1, 1, 1, 1};
    void* base = b8 ? static_cast<void*>(const_cast<__half*>(x.spec)) : static_cast<void*>(const_cast<float*>(x.spec32));
    auto map = [&](CUtensorMap* m, int first) {    // inputs first .. n_in - 1
        const int n = x.n_in - first;
        const cuuint64_t dim[5] = {16, 4, static_cast<cuuint64_t>(n), ntb, static_cast<cuuint64_t>(x.n_chan / 4)};
        const cuuint32_t box[5] = {16, 1, static_cast<cuuint32_t>(n), static_cast<cuuint32_t>(x.ks / kTbHalf), 1};
        return encode(m, b8 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 5,
                      static_cast<char*>(base) + 4 * piece * first, dim, stride, box, estride, CU_TENSOR_MAP_INTERLEAVE_NONE,
                      CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    };
    return map(&x.tmap, 0) && (x.n_in <= 64 || map(&x.tmap_hi, 64));
}

bool xengine_tc_supported(int n_in) { return n_in >= 1 && 2 * n_in <= 256; }

int xengine_tc_max_ks(int n_in) {
    int ks = 512;                                  // stages of at most 512 frames
    while (ks > 16 && (ks / kTbHalf) * 2 * n_in * 16 > kStageMaxBytes) ks /= 2;
    return ks;
}

int xengine_tc_ks_fp32(int n_in) {
    // the FP32 slot holds ks * rows_fp32(n_in) floats; the operand slot's two planes then take
    // ks * 2 n_in * 4 <= that many bytes
    int ks = 512;
    while (ks > 16 && ks * rows_fp32(n_in) * 4 > kStage2Bytes) ks /= 2;
    return ks;
}

cudaError_t launch_xengine_tc_table(const XtBatch* dtab, int n_items, int n_sm, cudaStream_t s, int form) {
    const size_t smem = static_cast<size_t>(smem_bytes(form));
    auto kern = form == XT_FORM_F32  ? xengine_tc_kernel<XT_FORM_F32>
              : form == XT_FORM_F32P ? xengine_tc_kernel<XT_FORM_F32P>
              : form == XT_FORM_I8  ? xengine_tc_kernel<XT_FORM_I8>
                                    : xengine_tc_kernel<XT_FORM_F16>;
    const bool convert = form != XT_FORM_F16;
    cudaError_t e;
    if (convert) {   // the drain warps' registers come out of the launch's: refuse one that has fewer
        cudaFuncAttributes fa{};
        if ((e = cudaFuncGetAttributes(&fa, kern)) != cudaSuccess) return e;
        if (fa.numRegs != kRegsLaunch) return cudaErrorInvalidConfiguration;
    }
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(smem));
    if (e != cudaSuccess) return e;
    const int grid = std::max(1, std::min(n_items, n_sm));
    kern<<<grid, (convert ? kWarps2 : kWarps1) * 32, smem, s>>>(dtab);
    return cudaGetLastError();
}

}  // namespace gbx
