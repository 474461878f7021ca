// Tensor-core execution of the large pairwise contractions of a path (the
// batched complex GEMMs of Sec. III-A's contraction, real and imaginary parts
// split into real GEMMs) on sm_103a: tcgen05.mma with the accumulator in
// tensor memory, operands staged by TMA into 128-byte-swizzled shared memory
// through an mbarrier pipeline.
//
// A step  C[inst][m, n] (h) = sum_k A[m, k] (h) * B[n, k] (h)  runs in two phases:
//  1. pack: each operand is gathered (any bit layout, merged-gate variant,
//     prefix slice) into row-major K-contiguous rows, each value split into a
//     high and a low part in the tensor-core input format F:
//       A rows:  [ hi(re0) hi(im0) hi(re1) ... | lo(re0) lo(im0) ... ]
//       B rows 2n, 2n+1 (the complex product as real dot products):
//         row 2n   = (re, -im) per k,  row 2n+1 = (im, re) per k, each [hi | lo];
//     so that  A_row . B_row(2n) = Re C[m, n]  and  A_row . B_row(2n+1) = Im C[m, n];
//  2. GEMM: D = A_hi B_hi^T + A_hi B_lo^T + A_lo B_hi^T with FP32 accumulation
//     in TMEM (the lo*lo term is dropped) over segments of at most kSegKb
//     k-blocks, the segments added in FP32 by the epilogue; D[m][2n + c] ->
//     C[m, n], written through the step's output strides (any layout).
// Formats (the precision modes of the contraction):
//  - TF32 (PTN_PREC_FP32): hi = x rounded to TF32, lo = (x - hi) rounded to
//    TF32; |x - hi - lo| <= 2^-24 |x|, i.e. FP32-accurate products;
//  - BF16 (PTN_PREC_BF16X3): hi, lo rounded to BF16 (16 significant bits in
//    total, FP32 exponent range);
//  - FP16 (PTN_PREC_FP16X3): hi, lo rounded to FP16 (22 significant bits) after
//    scaling each packed row by a power of two that brings its largest
//    magnitude into [0.5, 1); the epilogue undoes the row and column scales
//    exactly.
// The GEMM kernel is persistent and warp-specialised (see k_gemm).
// Conjugated operands (bra layer) are conjugated while packing.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cstring>

#include "kernels.cuh"
#include "stats.h"

namespace ptn {

namespace {

constexpr int kBM = 128;          // UMMA M (cta_group::1)
constexpr int kBN = 128;          // UMMA N (realified B rows per tile)
constexpr int kRowBytes = 128;    // one swizzle row of every tile
constexpr int kStages = 3;        // pipeline depth (4 tiles of 16 KB per stage)
constexpr int kTileA = kBM * kRowBytes;
constexpr int kTileB = kBN * kRowBytes;
constexpr int kStageBytes = 2 * kTileA + 2 * kTileB;
constexpr int kPairN = 2 * kBN;   // columns of a CTA pair's tile (k_gemm<F, true>): 128 B rows staged by each CTA
// epilogue staging: per epilogue warp a fragment of 32 rows x 8 complex columns.
// Its elements are placed so that a half-warp's 8-byte accesses hit 16 different
// bank pairs both when written by row and when read in the order of the output
// (run_gemm): a 128 x 128 tile's operands already take 1280 clocks of shared memory
// per k-block.  Against rows padded to 9 slots, 2^20 outputs by 128 terms, 40
// trajectories: 16.5 -> 13.9 million wavefronts, 9.8 -> 7.0 million of them counted
// as conflicts; 4096 trajectories 14.2 -> 13.4 ms.
constexpr int kStgElems = 32 * 8;
constexpr int kStgBytes = 8 * kStgElems * 8;
constexpr int kTabBytes = 8192;   // barriers, TMEM slot, per-warp column offsets and FP16 column scales
constexpr int kGemmSmem = 1024 + kStages * kStageBytes + kTabBytes + kStgBytes;   // align slack + stages + tables + staging
constexpr int kMaxPackBits = 40;
constexpr int kSegKb = 16;        // longest run of k-blocks accumulated in TMEM before the epilogue adds it
// k-blocks are spread round-robin over kAcc TMEM accumulators that the
// epilogue adds in FP32: the tensor core's FP32 accumulation truncates, so
// shorter accumulation chains keep the contraction within FP32 accuracy.
constexpr int kAcc = 4;
constexpr uint32_t kTmemCols = kAcc * kBN;   // 512: the whole TMEM of the SM (one CTA per SM)

enum GemmFmt { FMT_TF32 = 0, FMT_BF16 = 1, FMT_FP16 = 2 };

template <int F>
struct Fmt;
template <>
struct Fmt<FMT_TF32> {
    using T = float;
    static constexpr int kBytes = 4;
    static constexpr uint32_t kAB = 2;   // TF32 in the instruction descriptor
};
template <>
struct Fmt<FMT_BF16> {
    using T = __nv_bfloat16;
    static constexpr int kBytes = 2;
    static constexpr uint32_t kAB = 1;   // BF16
};
template <>
struct Fmt<FMT_FP16> {
    using T = __half;
    static constexpr int kBytes = 2;
    static constexpr uint32_t kAB = 0;   // F16
};

struct PackArgs {
    OperandDesc op;
    int32_t pcls;            // instance class the packed operand is addressed by
    int32_t role;            // 0: rows (A), 1: realified (B)
    int32_t n_rb, n_hb, n_kb;
    int32_t Kh;              // elements per half row (hi or lo), a multiple of one swizzle row
    int64_t n_pinst;
    int64_t r_stride[kMaxPackBits];   // operand strides of the row bits
    int64_t h_stride[kMaxPackBits];
    int64_t k_stride[kMaxPackBits];
    void* dst;
    int8_t* row_exp;         // FP16: per packed row and K segment (row-major [row][segment]) the
                             // power-of-two exponent e of the segment's largest |component| (the
                             // segment is stored scaled by 2^-e), else null
    int32_t seg_slots;       // FP16: complex slots per K segment (the GEMM's kSegKb k-blocks)
    const int32_t* inst_map; // cached step: packed instance i is local trajectory inst_map[i] (else i)
    // Outer-product operand (StepDesc.prod): the element is op[o0] * op1[o1], and every
    // stride above holds o0 in its low and o1 in its high 32 bits (sums stay carry-free,
    // each factor having at most 2^31 elements per instance); xconj: conjugate the product
    int32_t prod, xconj;
    OperandDesc op1;
    int32_t run_log;         // k_pack_rows: log2 consecutive units of a warp
};

struct GemmArgs {
    int32_t M, N2, Kh, nkb;
    int32_t n_h;
    int32_t a_pcls, b_pcls, out_cls;
    int32_t n_mb, n_nb, n_hb;
    // Staged stores: the 8 bits of a fragment (5 row bits, 3 column bits) by
    // increasing output stride; a lane stores pairs along bit 0, bits 1-5 run
    // over the lanes, bits 6-7 over its four stores.
    int32_t staged;              // 0: the lowest five output bits are row bits, lanes store their own rows
    int32_t frag_vec;            // bit 0 has stride 1 and every address is even: 16-byte stores
    int32_t frag_sm[8], frag_row[8];   // place in the staged fragment (XOR of the words), row within the 32
    int32_t row_sm[5], col_sm[3];      // places of a fragment's row and column bits
    int64_t frag_out[8];
    int64_t row_hi[2];           // output strides of rows 32 and 64 of a tile
    int32_t pair;                // CTA pairs: an M tile and its odd neighbour run together
    int32_t bn;                  // columns of a tile
    int32_t tm_log, tn_log;      // log2 tiles along M and N (a step's sizes are powers of two)
    int64_t tiles_m, tiles_n, n_inst, n_tiles;
    const int32_t* net_tl;
    // stacked mode: the rows of all networks of one trajectory form one GEMM
    // (rows = network-major (net, m)); tiles never cross trajectories
    int32_t stacked, m_bits;
    int64_t n_groups;
    const int32_t* grp_net0;     // [n_groups + 1] first network of each trajectory group
    const int64_t* grp_tile0;    // [n_groups + 1] first tile of each group
    float2* out;
    int64_t out_size;
    int* err;
    uint64_t wait_ns;            // limit of every pipeline wait (ptn_set_wait_limit)
    const int8_t* exp_a;         // FP16 row exponents of A and B (see PackArgs), else null
    const int8_t* exp_b;
    const int32_t* out_map;      // cached step: instance i writes local trajectory out_map[i] (else i)
    int64_t m_stride[kMaxOut];
    int64_t n_stride[kMaxOut];
    int64_t h_stride[kMaxOut];
};

// Round to the nearest TF32 value (ties away from zero): add half of the 13
// dropped mantissa bits, then clear them.
__device__ __forceinline__ float tf32_rn(float x) {
    return __uint_as_float((__float_as_uint(x) + 0x1000u) & 0xFFFFE000u);
}

template <int F>
__device__ __forceinline__ void split(float x, typename Fmt<F>::T& hi, typename Fmt<F>::T& lo);
template <>
__device__ __forceinline__ void split<FMT_TF32>(float x, float& hi, float& lo) {
    hi = tf32_rn(x);
    lo = tf32_rn(x - hi);
}
template <>
__device__ __forceinline__ void split<FMT_BF16>(float x, __nv_bfloat16& hi, __nv_bfloat16& lo) {
    hi = __float2bfloat16_rn(x);
    lo = __float2bfloat16_rn(x - __bfloat162float(hi));
}
template <>
__device__ __forceinline__ void split<FMT_FP16>(float x, __half& hi, __half& lo) {
    hi = __float2half_rn(x);
    lo = __float2half_rn(x - __half2float(hi));
}

template <int F>
__device__ __forceinline__ void store_pair(typename Fmt<F>::T* d, typename Fmt<F>::T x, typename Fmt<F>::T y);
template <>
__device__ __forceinline__ void store_pair<FMT_TF32>(float* d, float x, float y) {
    *reinterpret_cast<float2*>(d) = make_float2(x, y);
}
template <>
__device__ __forceinline__ void store_pair<FMT_BF16>(__nv_bfloat16* d, __nv_bfloat16 x, __nv_bfloat16 y) {
    *reinterpret_cast<__nv_bfloat162*>(d) = __halves2bfloat162(x, y);
}
template <>
__device__ __forceinline__ void store_pair<FMT_FP16>(__half* d, __half x, __half y) {
    *reinterpret_cast<__half2*>(d) = __halves2half2(x, y);
}

__device__ __forceinline__ const float2* pack_operand_ptr(const OperandDesc& d, int pcls, int64_t inst,
                                                          const ChunkCtx& c) {
    int64_t tl = 0, net = 0;
    if (pcls == CLS_NET) {
        net = inst;
        tl = c.net_tl[inst];
    } else if (pcls == CLS_TRAJ) {
        tl = inst;
    }
    const float2* p;
    if (d.mode == OP_LEAF) {
        int64_t var = 0;
        if (d.leaf_col >= 0) var = c.var_ids[(int64_t)c.chunk_traj[tl] * c.n_var_cols + d.leaf_col];
        p = c.vtab + d.leaf_base + var * d.inst_size;
    } else {
        const int64_t oi = d.cls == CLS_CONST ? 0 : (d.cls == CLS_TRAJ ? rep_inst(d, tl, c) : net);
        p = c.arena[d.arena] + d.arena_off * c.arena_inst[d.arena] + oi * d.inst_size;
    }
    if (pcls == CLS_NET && d.n_slice) {
        const uint64_t* pre = c.net_prefix + net * c.n_words;
        int64_t off = 0;
        for (int s = 0; s < d.n_slice; s++) off += (int64_t)bits_get(pre, d.slice_qubit[s]) * d.slice_stride[s];
        p += off;
    }
    return p;
}

// Packing: one warp per packed row (instance, h, row) when a half row holds
// >= 32 complex slots, else 32 / slots rows per warp.  Every size is a power of
// two, so the row index is decoded with shifts.  The row's base offset is
// formed once per row; the K offsets come from a per-block shared table in two
// levels (bits 0-9 and 10-19; bit 20 and up, rarely used, by a loop), so a
// contiguous K axis turns into coalesced float2 loads.  Stores are float2 /
// 32-bit pairs, consecutive lanes on consecutive slots.  FP16 rows are scaled
// segment by segment: the GEMM accumulates K in segments of kSegKb k-blocks
// (512 complex slots in FP16) and adds them in FP32, so a scale needs to be
// uniform along one segment only.  Each (row, segment) is stored scaled by
// 2^-e, e the exponent of its largest |component|, in one pass: a warp keeps
// the segment in registers between the max and the store.
constexpr int kKTab = 1024;
constexpr int kPackRegRow = 512;   // longest FP16 K segment a warp holds in registers

__device__ __forceinline__ void build_ktab(const PackArgs& a, int64_t* ktab) {
    const int n_lo = a.n_kb < 10 ? a.n_kb : 10;
    const int n_mid = a.n_kb < 20 ? a.n_kb - n_lo : 10;
    for (int i = threadIdx.x; i < 2 * kKTab; i += blockDim.x) {
        const int lvl = i >= kKTab, v = i & (kKTab - 1);
        int64_t off = 0;
        const int nb = lvl ? n_mid : n_lo, b0 = lvl ? 10 : 0;
        for (int t = 0; t < nb; t++)
            if ((v >> t) & 1) off += a.k_stride[b0 + t];
        ktab[i] = off;
    }
}
__device__ __forceinline__ int64_t kofs(const PackArgs& a, const int64_t* ktab, int64_t kc) {
    int64_t off = ktab[kc & (kKTab - 1)] + ktab[kKTab + ((kc >> 10) & (kKTab - 1))];
    for (int t = 20; t < a.n_kb; t++)
        if ((kc >> t) & 1) off += a.k_stride[t];
    return off;
}
// Operand address of packed row jr = (pi * nh + h) * nrow + row; z = pi * nh + h.
// Row offsets from a two-level table like the K offsets (row bits 0-9 and
// 10-19; bit 20 and up by a loop): short rows would otherwise spend most of
// their time forming their base address.
__device__ __forceinline__ void build_rtab(const PackArgs& a, int64_t* rtab) {
    const int n_lo = a.n_rb < 10 ? a.n_rb : 10;
    const int n_mid = a.n_rb < 20 ? a.n_rb - n_lo : 10;
    for (int i = threadIdx.x; i < 2 * kKTab; i += blockDim.x) {
        const int lvl = i >= kKTab, v = i & (kKTab - 1);
        int64_t off = 0;
        const int nb = lvl ? n_mid : n_lo, b0 = lvl ? 10 : 0;
        for (int t = 0; t < nb; t++)
            if ((v >> t) & 1) off += a.r_stride[b0 + t];
        rtab[i] = off;
    }
}
struct PackSrc {
    const float2* b0;        // the operand's row (outer product: factor 0's)
    const float2* b1;        // outer product: factor 1's, else unused
};
constexpr int64_t kLo32 = 0xffffffffll;
__device__ __forceinline__ PackSrc pack_row_base(const PackArgs& a, const ChunkCtx& c, const int64_t* rtab,
                                                 int64_t jr, int64_t& z, int64_t& row) {
    row = jr & (((int64_t)1 << a.n_rb) - 1);
    z = jr >> a.n_rb;
    const int64_t h = z & (((int64_t)1 << a.n_hb) - 1);
    const int64_t pi = a.inst_map ? (int64_t)a.inst_map[z >> a.n_hb] : z >> a.n_hb;
    int64_t off = rtab[row & (kKTab - 1)] + rtab[kKTab + ((row >> 10) & (kKTab - 1))];
    for (int i = 20; i < a.n_rb; i++)
        if ((row >> i) & 1) off += a.r_stride[i];
    for (int i = 0; i < a.n_hb; i++)
        if ((h >> i) & 1) off += a.h_stride[i];
    PackSrc src;
    if (!a.prod) {
        src.b0 = pack_operand_ptr(a.op, a.pcls, pi, c) + off;
        src.b1 = nullptr;
    } else {
        src.b0 = pack_operand_ptr(a.op, a.pcls, pi, c) + (off & kLo32);
        src.b1 = pack_operand_ptr(a.op1, a.pcls, pi, c) + (off >> 32);
    }
    return src;
}
// Element at K offset koff of a row: a plain read, or the product of the two
// factors with the single-term multiply-add sequence of the SIMT contraction
// kernels (so the packed values equal those of the materialised product).
__device__ __forceinline__ float2 pack_load(const PackArgs& a, const PackSrc& src, int64_t koff) {
    if (!a.prod) return src.b0[koff];
    const float2 x = src.b0[koff & kLo32], y = src.b1[koff >> 32];
    const float xi = a.op.conj ? -x.y : x.y, yi = a.op1.conj ? -y.y : y.y;
    float2 r;
    r.x = fmaf(x.x, y.x, 0.f);
    r.x = fmaf(-xi, yi, r.x);
    r.y = fmaf(x.x, yi, 0.f);
    r.y = fmaf(xi, y.x, r.y);
    return r;
}
template <int F>
__device__ __forceinline__ void pack_store(const PackArgs& a, typename Fmt<F>::T* d0, int64_t rowlen, int64_t kc,
                                           float re, float im) {
    using T = typename Fmt<F>::T;
    T rh, rl, ih, il;
    split<F>(re, rh, rl);
    split<F>(im, ih, il);
    if (a.role == 0) {
        store_pair<F>(d0 + 2 * kc, rh, ih);
        store_pair<F>(d0 + a.Kh + 2 * kc, rl, il);
    } else {
        T nih, nil;
        split<F>(-im, nih, nil);
        store_pair<F>(d0 + 2 * kc, rh, nih);
        store_pair<F>(d0 + a.Kh + 2 * kc, rl, nil);
        store_pair<F>(d0 + rowlen + 2 * kc, ih, rh);
        store_pair<F>(d0 + rowlen + a.Kh + 2 * kc, il, rl);
    }
}
__device__ __forceinline__ int row_exponent(float mx) {
    int e = 0;
    if (mx > 0.f) {
        frexpf(mx, &e);
        e = e < -100 ? -100 : (e > 100 ? 100 : e);
    }
    return e;
}

template <int F>
__global__ void __launch_bounds__(256) k_pack(const __grid_constant__ PackArgs a, const __grid_constant__ ChunkCtx c) {
    using T = typename Fmt<F>::T;
    __shared__ int64_t ktab[2 * kKTab];
    __shared__ int64_t rtab[2 * kKTab];
    build_ktab(a, ktab);
    build_rtab(a, rtab);
    __syncthreads();
    T* dst = static_cast<T*>(a.dst);
    const int lk = 31 - __clz(a.Kh / 2);                // log2 complex slots per half row
    const int64_t kcp = (int64_t)1 << lk;
    const int64_t kc_real = (int64_t)1 << a.n_kb;
    const int64_t rowlen = 2 * (int64_t)a.Kh;
    const int rpw = lk >= 5 ? 1 : (32 >> lk);           // rows per warp
    const int lane = threadIdx.x & 31;
    const int sub = lk >= 5 ? 0 : (lane >> lk);         // row of this lane within the warp
    const int lstep = lk >= 5 ? 32 : (int)kcp;          // slots a lane advances by
    const int l0 = lk >= 5 ? lane : (lane & ((int)kcp - 1));
    const int64_t n_rows = a.n_pinst << (a.n_hb + a.n_rb);
    const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const float csign = (a.prod ? a.xconj : a.op.conj) ? -1.f : 1.f;
    if (F == FMT_FP16 && kc_real < 32) {
        // short FP16 rows (fewer real slots than a warp, padded to 32): g =
        // kc_real lanes per row, 32 / g rows per warp, the row maximum
        // reduced within each lane group
        const int lg = a.n_kb, g = 1 << lg;
        const int sub_r = lane >> lg, l0r = lane & (g - 1);
        for (int64_t w = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5); (w << (5 - lg)) < n_rows;
             w += warps) {
            const int64_t jr = (w << (5 - lg)) + sub_r;
            const bool act = jr < n_rows;
            float2 v = make_float2(0.f, 0.f);
            int64_t z = 0, row = 0;
            if (act) {
                const PackSrc src = pack_row_base(a, c, rtab, jr, z, row);
                v = pack_load(a, src, kofs(a, ktab, l0r));
            }
            float mx = fmaxf(fabsf(v.x), fabsf(v.y));
            for (int o = g >> 1; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            if (!act) continue;
            const int e = row_exponent(mx);
            const float sc = ldexpf(1.f, -e);
            if (l0r == 0) a.row_exp[jr] = (int8_t)e;
            T* d0 = a.role == 0 ? dst + jr * rowlen : dst + ((z << (a.n_rb + 1)) + 2 * row) * rowlen;
            pack_store<F>(a, d0, rowlen, l0r, v.x * sc, csign * v.y * sc);
            for (int64_t kc = l0r + g; kc < kcp; kc += g) pack_store<F>(a, d0, rowlen, kc, 0.f, 0.f);   // padding
        }
        return;
    }
    if constexpr (F == FMT_FP16) {
        // units of (row, K segment): a warp holds a segment of at most
        // kPackRegRow slots in registers, reduces its largest |component|,
        // and writes it scaled (rows span at least 32 slots: one unit per warp)
        const int64_t seg = kcp < a.seg_slots ? kcp : a.seg_slots;
        const int lseg = 63 - __clzll(seg);
        const int64_t nseg = kcp >> lseg;
        const int64_t units = n_rows << (lk - lseg);
        for (int64_t w = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5); w < units; w += warps) {
            const int64_t jr = w >> (lk - lseg), sg = w & (nseg - 1);
            int64_t z, row;
            const PackSrc src = pack_row_base(a, c, rtab, jr, z, row);
            T* d0 = a.role == 0 ? dst + jr * rowlen : dst + ((z << (a.n_rb + 1)) + 2 * row) * rowlen;
            const int64_t kc0 = sg << lseg;
            float2 v[kPackRegRow / 32];
            float mx = 0.f;
#pragma unroll
            for (int i = 0; i < kPackRegRow / 32; i++) {
                const int64_t kc = kc0 + lane + 32 * i;
                v[i] = make_float2(0.f, 0.f);
                if (lane + 32 * i < seg && kc < kc_real) v[i] = pack_load(a, src, kofs(a, ktab, kc));
                mx = fmaxf(mx, fmaxf(fabsf(v[i].x), fabsf(v[i].y)));
            }
            for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            const int e = row_exponent(mx);
            const float sc = ldexpf(1.f, -e);
            if (lane == 0) a.row_exp[jr * nseg + sg] = (int8_t)e;
#pragma unroll
            for (int i = 0; i < kPackRegRow / 32; i++)
                if (lane + 32 * i < seg)
                    pack_store<F>(a, d0, rowlen, kc0 + lane + 32 * i, v[i].x * sc, csign * v[i].y * sc);
        }
        return;
    }
    for (int64_t w = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5); w * rpw < n_rows; w += warps) {
        const int64_t jr = w * rpw + sub;                // (pi, h, row), row fastest
        if (jr >= n_rows) continue;
        int64_t z, row;
        const PackSrc src = pack_row_base(a, c, rtab, jr, z, row);
        T* d0 = a.role == 0 ? dst + jr * rowlen : dst + ((z << (a.n_rb + 1)) + 2 * row) * rowlen;
        {
            for (int64_t kc = l0; kc < kcp; kc += lstep) {
                float re = 0.f, im = 0.f;
                if (kc < kc_real) {
                    const float2 v = pack_load(a, src, kofs(a, ktab, kc));
                    re = v.x;
                    im = csign * v.y;
                }
                pack_store<F>(a, d0, rowlen, kc, re, im);
            }
        }
    }
}

// Four real components (two consecutive complex slots) of a packed row: the
// hi and lo stores of a role.
template <int F>
struct Quad;
template <>
struct Quad<FMT_TF32> {
    static __device__ __forceinline__ void store(float* d, float a, float b, float c, float e) {
        *reinterpret_cast<float4*>(d) = make_float4(a, b, c, e);
    }
};
template <>
struct Quad<FMT_BF16> {
    static __device__ __forceinline__ void store(__nv_bfloat16* d, __nv_bfloat16 a, __nv_bfloat16 b, __nv_bfloat16 c,
                                                 __nv_bfloat16 e) {
        __nv_bfloat162 v[2] = {__halves2bfloat162(a, b), __halves2bfloat162(c, e)};
        *reinterpret_cast<uint2*>(d) = *reinterpret_cast<uint2*>(v);
    }
};
template <>
struct Quad<FMT_FP16> {
    static __device__ __forceinline__ void store(__half* d, __half a, __half b, __half c, __half e) {
        __half2 v[2] = {__halves2half2(a, b), __halves2half2(c, e)};
        *reinterpret_cast<uint2*>(d) = *reinterpret_cast<uint2*>(v);
    }
};
// Slots kc, kc + 1 = (re0, im0), (re1, im1) of the row at d0 (the pair of rows, realified).
template <int F, int ROLE>
__device__ __forceinline__ void pack_store2(typename Fmt<F>::T* d0, int64_t Kh, int kc, float re0, float im0, float re1,
                                            float im1) {
    using T = typename Fmt<F>::T;
    T rh0, rl0, ih0, il0, rh1, rl1, ih1, il1;
    split<F>(re0, rh0, rl0);
    split<F>(im0, ih0, il0);
    split<F>(re1, rh1, rl1);
    split<F>(im1, ih1, il1);
    T* d = d0 + 2 * kc;
    if (ROLE == 0) {
        Quad<F>::store(d, rh0, ih0, rh1, ih1);
        Quad<F>::store(d + Kh, rl0, il0, rl1, il1);
    } else {
        T nh0, nl0, nh1, nl1;
        split<F>(-im0, nh0, nl0);
        split<F>(-im1, nh1, nl1);
        Quad<F>::store(d, rh0, nh0, rh1, nh1);
        Quad<F>::store(d + Kh, rl0, nl0, rl1, nl1);
        Quad<F>::store(d + 2 * Kh, ih0, rh0, ih1, rh1);
        Quad<F>::store(d + 3 * Kh, il0, rl0, il1, rl1);
    }
}
// Scale of a segment whose largest |component| over the lanes of a row (g of
// them) is mx, and its exponent.
template <int G>
__device__ __forceinline__ float seg_scale(float mx, int g, int& e) {
#pragma unroll
    for (int o = G >> 1; o > 0; o >>= 1)
        if (o < g) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    e = row_exponent(mx);
    return ldexpf(1.f, -e);
}

// Packing of an operand whose summed axis is contiguous and 16-byte aligned
// (all but a few steps): k_pack above forms an offset and reads 8 bytes per
// slot, keeps 16 registers of slots whatever the row's length, and walks rows
// grid-strided, so short rows spend most of their time on addresses (2.6 TB/s
// at 128 slots per row).  Here a lane takes two consecutive slots per 16-byte
// read, a warp a run of consecutive units (row, segment of at most 512
// slots) so that the instance's address is formed once per run, and NV * UN
// reads per lane are in flight.  Row offsets come from a three-level table of
// 7 bits each.  Same values, scales and layout as k_pack.  It is bound by
// HBM: 4096 trajectories of the middle 30-qubit block, 128 slots per row (74.5 GB)
// 29.0 -> 12.3 ms (6.1 TB/s), 256 slots (23.2 GB) 4.82 -> 3.44 ms.
template <int F, int ROLE, int NV>
__global__ void __launch_bounds__(256) k_pack_rows(const __grid_constant__ PackArgs a, const __grid_constant__ ChunkCtx c) {
    using T = typename Fmt<F>::T;
    constexpr int UN = NV >= 4 ? 1 : 4 / NV;            // units in flight per lane group
    __shared__ int64_t rtab[3 * 128];
    for (int i = threadIdx.x; i < 3 * 128; i += blockDim.x) {
        int64_t off = 0;
        for (int t = 0; t < 7; t++) {
            const int b = (i >> 7) * 7 + t;
            if (b < a.n_rb && ((i >> t) & 1)) off += a.r_stride[b];
        }
        rtab[i] = off;
    }
    __syncthreads();
    T* dst = static_cast<T*>(a.dst);
    const int lane = threadIdx.x & 31;
    const int seg_log = a.n_kb < 9 ? a.n_kb : 9;        // slots of a unit
    const int nseg_log = a.n_kb - seg_log;
    const int g_log = seg_log < 6 ? seg_log - 1 : 5;    // lanes per unit
    const int g = 1 << g_log, l0 = lane & (g - 1), per_log = 5 - g_log;
    const int kcp = a.Kh / 2, pad = kcp - (1 << a.n_kb);   // padding slots (rows of one unit only)
    const int64_t n_units = (a.n_pinst << (a.n_hb + a.n_rb)) << nseg_log;
    const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const float csign = a.op.conj ? -1.f : 1.f;
    int64_t cur_z = -1;
    const float2* base = nullptr;
    const int run = 1 << a.run_log;
    for (int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; (w << a.run_log) < n_units; w += warps) {
        for (int i0 = 0; i0 < run; i0 += UN << per_log) {
            float4 v[UN][NV];
            int64_t unit[UN];
#pragma unroll
            for (int j = 0; j < UN; j++) {
                unit[j] = (w << a.run_log) + i0 + (j << per_log) + (lane >> g_log);
                const bool act = unit[j] < n_units;
                if (!act) unit[j] = -1;
                const int64_t jr = (act ? unit[j] : n_units - 1) >> nseg_log;
                const int64_t row = jr & (((int64_t)1 << a.n_rb) - 1), z = jr >> a.n_rb;
                if (z != cur_z) {
                    cur_z = z;
                    const int64_t h = z & (((int64_t)1 << a.n_hb) - 1);
                    const int64_t pi = a.inst_map ? (int64_t)a.inst_map[z >> a.n_hb] : z >> a.n_hb;
                    base = pack_operand_ptr(a.op, a.pcls, pi, c);
                    for (int t = 0; t < a.n_hb; t++)
                        if ((h >> t) & 1) base += a.h_stride[t];
                }
                int64_t off = rtab[row & 127] + rtab[128 + ((row >> 7) & 127)] + rtab[256 + ((row >> 14) & 127)];
                for (int t = 21; t < a.n_rb; t++)
                    if ((row >> t) & 1) off += a.r_stride[t];
                const float2* src = base + off + ((act ? unit[j] & ((1 << nseg_log) - 1) : 0) << seg_log) + 2 * l0;
#pragma unroll
                for (int q = 0; q < NV; q++)
                    v[j][q] = *reinterpret_cast<const float4*>(src + 2 * (q << g_log));
            }
#pragma unroll
            for (int j = 0; j < UN; j++) {
                float sc = 1.f;
                if constexpr (F == FMT_FP16) {
                    float mx = 0.f;
#pragma unroll
                    for (int q = 0; q < NV; q++)
                        mx = fmaxf(mx, fmaxf(fmaxf(fabsf(v[j][q].x), fabsf(v[j][q].y)),
                                             fmaxf(fabsf(v[j][q].z), fabsf(v[j][q].w))));
                    int e;
                    sc = seg_scale<32>(mx, g, e);
                    if (l0 == 0 && unit[j] >= 0) a.row_exp[unit[j]] = (int8_t)e;
                }
                if (unit[j] >= 0) {
                    const float si = csign * sc;
                    T* d0 = dst + (unit[j] >> nseg_log) * (ROLE ? 4 : 2) * (int64_t)a.Kh;
                    const int k0 = (int)(unit[j] & ((1 << nseg_log) - 1)) << seg_log;
#pragma unroll
                    for (int q = 0; q < NV; q++)
                        pack_store2<F, ROLE>(d0, a.Kh, k0 + 2 * (l0 + (q << g_log)), v[j][q].x * sc, v[j][q].y * si,
                                             v[j][q].z * sc, v[j][q].w * si);
                    for (int k = 2 * l0; k < pad; k += 2 << g_log)
                        pack_store2<F, ROLE>(d0, a.Kh, (1 << a.n_kb) + k, 0.f, 0.f, 0.f, 0.f);
                }
            }
        }
    }
}

// Packing of an outer-product operand: the factors' elements that one packed
// instance's rows read (2^n_rb rows by the summed bits each factor varies
// along) are staged in shared memory in the order of the summed axis, so that
// forming a slot is two conflict-free shared reads instead of two scattered
// global ones with table offsets.  One CTA per packed instance at a time, a
// warp per (row, segment).  Same values as k_pack.  Bound by the HBM writes of
// the packed rows: the middle 30-qubit block's product rows (8 x 4096 slots per
// network) with the trajectory operand they meet, 274 GB, 96.2 -> 43.7 ms (6.3
// TB/s).
constexpr int kProdStage = 1024;      // elements of one factor per packed instance
constexpr int kProdHi = 256;          // combinations of the summed bits above the lowest six
template <int F, int ROLE>
__global__ void __launch_bounds__(256) k_pack_prod(const __grid_constant__ PackArgs a, const __grid_constant__ ChunkCtx c) {
    using T = typename Fmt<F>::T;
    __shared__ float2 st[2][kProdStage];
    __shared__ int16_t hidx[2][kProdHi];
    __shared__ int64_t sbase[2];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // compact index of a factor: its summed bits in order (n_kf of them), rows above
    int n_kf[2] = {0, 0}, lidx[2][2] = {{0, 0}, {0, 0}};   // lane's two slots: index of the low six bits
    for (int t = 0; t < a.n_kb; t++) {
        const int64_t sf[2] = {a.k_stride[t] & kLo32, a.k_stride[t] >> 32};
#pragma unroll
        for (int f = 0; f < 2; f++) {
            if (!sf[f]) continue;
            if (t < 6) {
                lidx[f][0] |= ((2 * lane) >> t & 1) << n_kf[f];
                lidx[f][1] |= ((2 * lane + 1) >> t & 1) << n_kf[f];
            }
            n_kf[f]++;
        }
    }
    const int n_hi = 1 << (a.n_kb - 6);
    for (int i = threadIdx.x; i < 2 * n_hi; i += blockDim.x) {
        const int f = i >= n_hi, v = i & (n_hi - 1);
        int x = 0, n = 0;
        for (int t = 0; t < a.n_kb; t++) {
            if (!(f ? a.k_stride[t] >> 32 : a.k_stride[t] & kLo32)) continue;
            if (t >= 6) x |= (v >> (t - 6) & 1) << n;
            n++;
        }
        hidx[f][v] = (int16_t)x;
    }
    T* dst = static_cast<T*>(a.dst);
    const int seg_log = a.n_kb < 9 ? a.n_kb : 9, nseg_log = a.n_kb - seg_log, nv = 1 << (seg_log - 6);
    const float csign = a.xconj ? -1.f : 1.f;
    const float s0 = a.op.conj ? -1.f : 1.f, s1 = a.op1.conj ? -1.f : 1.f;
    const int64_t nz = a.n_pinst << a.n_hb;
    for (int64_t z = blockIdx.x; z < nz; z += gridDim.x) {
        __syncthreads();   // the previous instance's factors are no longer read
        if (lane == 0 && warp < 2) {
            const int64_t h = z & (((int64_t)1 << a.n_hb) - 1);
            const int64_t pi = a.inst_map ? (int64_t)a.inst_map[z >> a.n_hb] : z >> a.n_hb;
            int64_t off = 0;
            for (int t = 0; t < a.n_hb; t++)
                if ((h >> t) & 1) off += a.h_stride[t];
            sbase[warp] = reinterpret_cast<int64_t>(warp ? pack_operand_ptr(a.op1, a.pcls, pi, c) + (off >> 32)
                                                         : pack_operand_ptr(a.op, a.pcls, pi, c) + (off & kLo32));
        }
        __syncthreads();
#pragma unroll
        for (int f = 0; f < 2; f++) {
            const float2* b = reinterpret_cast<const float2*>(sbase[f]);
            for (int i = threadIdx.x; i < 1 << (n_kf[f] + a.n_rb); i += blockDim.x) {
                int64_t off = 0;
                int n = 0;
                for (int t = 0; t < a.n_kb; t++) {
                    const int64_t sf = f ? a.k_stride[t] >> 32 : a.k_stride[t] & kLo32;
                    if (sf && ((i >> n++) & 1)) off += sf;
                }
                for (int t = 0; t < a.n_rb; t++)
                    if ((i >> (n_kf[f] + t)) & 1) off += f ? a.r_stride[t] >> 32 : a.r_stride[t] & kLo32;
                float2 x = b[off];
                x.y *= f ? s1 : s0;
                st[f][i] = x;
            }
        }
        __syncthreads();
        for (int u = warp; u < 1 << (a.n_rb + nseg_log); u += 8) {
            const int row = u >> nseg_log, sg = u & ((1 << nseg_log) - 1);
            const float2 *f0 = st[0] + (row << n_kf[0]), *f1 = st[1] + (row << n_kf[1]);
            float4 v[8];
            float mx = 0.f;
#pragma unroll
            for (int q = 0; q < 8; q++) {
                if (q >= nv) break;
                const int h0 = hidx[0][(sg << (seg_log - 6)) + q], h1 = hidx[1][(sg << (seg_log - 6)) + q];
                float r[4];
#pragma unroll
                for (int e = 0; e < 2; e++) {
                    const float2 x = f0[lidx[0][e] + h0], y = f1[lidx[1][e] + h1];
                    r[2 * e] = fmaf(-x.y, y.y, fmaf(x.x, y.x, 0.f));
                    r[2 * e + 1] = fmaf(x.y, y.x, fmaf(x.x, y.y, 0.f));
                }
                v[q] = make_float4(r[0], r[1], r[2], r[3]);
                mx = fmaxf(mx, fmaxf(fmaxf(fabsf(r[0]), fabsf(r[1])), fmaxf(fabsf(r[2]), fabsf(r[3]))));
            }
            const int64_t jr = (z << a.n_rb) + row;
            float sc = 1.f;
            if constexpr (F == FMT_FP16) {
                int e;
                sc = seg_scale<32>(mx, 32, e);
                if (lane == 0) a.row_exp[(jr << nseg_log) + sg] = (int8_t)e;
            }
            const float si = csign * sc;
            T* d0 = dst + jr * (ROLE ? 4 : 2) * (int64_t)a.Kh;
#pragma unroll
            for (int q = 0; q < 8; q++) {
                if (q >= nv) break;
                pack_store2<F, ROLE>(d0, a.Kh, (sg << seg_log) + 64 * q + 2 * lane, v[q].x * sc, v[q].y * si, v[q].z * sc,
                                     v[q].w * si);
            }
        }
    }
}

// Packing of an operand whose summed bits lie anywhere in its memory (adjoint
// steps read tensors in the order another step wanted them): tiles of up to 2^11
// elements spanned by the five lowest strides and the six lowest summed bits go
// through shared memory, read 256 consecutive bytes at a time and written as
// rows of consecutive slots.  k_pack reads 8 bytes a lane at the summed bits'
// strides instead (3-4.6 TB/s).  For the formats without per-segment scales.
// Same values and layout as k_pack.  The gradient's adjoint steps, 1024
// trajectories of 16 qubits: 47 GB 10.2 -> 7.6 ms (6.2 TB/s), all packs 52.2 ->
// 46.8 ms.
constexpr int kTileBits = 11;
struct TileArgs {
    int32_t nt;                      // tile bits
    int64_t ld_stride[kTileBits];    // load order: operand strides, place in the staged tile
    int32_t ld_place[kTileBits];
    int64_t st_dst[kTileBits];       // store order (summed bits, then rows): destination of each bit, in elements
    int32_t n_out;                   // bits outside the tile: operand strides and destinations
    int64_t out_stride[2 * kMaxPackBits], out_dst[2 * kMaxPackBits];
};
template <int F, int ROLE>
__global__ void __launch_bounds__(256) k_pack_tile(const __grid_constant__ PackArgs a, const __grid_constant__ TileArgs t,
                                                   const __grid_constant__ ChunkCtx c) {
    using T = typename Fmt<F>::T;
    constexpr int NL = 1 << (kTileBits - 8);
    __shared__ float2 tile[(1 << kTileBits) + (1 << (kTileBits - 6))];   // element i at i + i / 64: rows 65 apart
    __shared__ int64_t sh_src[2], sh_dst[2];
    const int tid = threadIdx.x, n = 1 << t.nt;
    int64_t off_t = 0, dst_t = 0;
    int pl_t = 0;
    for (int b = 0; b < 8 && b < t.nt; b++)
        if ((tid >> b) & 1) {
            off_t += t.ld_stride[b];
            pl_t += t.ld_place[b];
        }
    // a thread stores slot pairs: bit 0 of the store order is the lowest summed bit
    for (int b = 0; b < 8 && b + 1 < t.nt; b++)
        if ((tid >> b) & 1) dst_t += t.st_dst[b + 1];
    const float csign = a.op.conj ? -1.f : 1.f;
    const int64_t n_tiles = (a.n_pinst << a.n_hb) << t.n_out;
    T* dst = static_cast<T*>(a.dst);
    // addresses of tile u into slot s, by one warp (a lane per bit)
    auto locate = [&](int64_t u, int s) {
        const int lane = tid & 31;
        const int64_t z = u >> t.n_out, h = z & (((int64_t)1 << a.n_hb) - 1);
        int64_t p = 0, d = 0;
        for (int b = lane; b < t.n_out; b += 32)
            if ((u >> b) & 1) {
                p += t.out_stride[b];
                d += t.out_dst[b];
            }
        for (int b = lane; b < a.n_hb; b += 32)
            if ((h >> b) & 1) p += a.h_stride[b];
        for (int o = 16; o > 0; o >>= 1) {
            p += __shfl_xor_sync(0xffffffffu, p, o);
            d += __shfl_xor_sync(0xffffffffu, d, o);
        }
        if (lane == 0) {
            const int64_t pi = a.inst_map ? (int64_t)a.inst_map[z >> a.n_hb] : z >> a.n_hb;
            sh_src[s] = reinterpret_cast<int64_t>(pack_operand_ptr(a.op, a.pcls, pi, c) + p);
            sh_dst[s] = d + (z << a.n_rb) * (ROLE ? 4 : 2) * (int64_t)a.Kh;
        }
    };
    float2 v[NL];
    auto load = [&](int s) {
        const float2* src = reinterpret_cast<const float2*>(sh_src[s]) + off_t;
#pragma unroll
        for (int i = 0; i < NL; i++) {
            int64_t off = 0;
#pragma unroll
            for (int b = 8; b < kTileBits; b++)
                if ((i >> (b - 8)) & 1) off += t.ld_stride[b];
            if ((i << 8) + tid < n) v[i] = src[off];
        }
    };
    int64_t u = blockIdx.x;
    if (u >= n_tiles) return;
    if (tid < 32) locate(u, 0);
    else if (tid < 64 && u + gridDim.x < n_tiles) locate(u + gridDim.x, 1);
    __syncthreads();
    load(0);
    for (int s = 0; u < n_tiles; u += gridDim.x, s ^= 1) {
        // the next tile's reads are in flight while this one is stored
        __syncthreads();             // the previous tile has been stored
#pragma unroll
        for (int i = 0; i < NL; i++) {
            int pl = pl_t;
#pragma unroll
            for (int b = 8; b < kTileBits; b++)
                if ((i >> (b - 8)) & 1) pl += t.ld_place[b];
            if ((i << 8) + tid < n) tile[pl + (pl >> 6)] = v[i];
        }
        T* d0 = dst + sh_dst[s] + dst_t;
        __syncthreads();
        if (u + gridDim.x < n_tiles) load(s ^ 1);
        if (tid < 32 && u + 2 * gridDim.x < n_tiles) locate(u + 2 * gridDim.x, s);
#pragma unroll
        for (int i = 0; i < 1 << (kTileBits - 9); i++) {
            int64_t d = 0;
#pragma unroll
            for (int b = 9; b < kTileBits; b++)
                if ((i >> (b - 9)) & 1) d += t.st_dst[b];
            const int e = 2 * ((i << 8) + tid);
            if (e < n) {
                const float2 x = tile[e + (e >> 6)], y = tile[e + 1 + (e >> 6)];
                pack_store2<F, ROLE>(d0 + d, a.Kh, 0, x.x, csign * x.y, y.x, csign * y.y);
            }
        }
    }
}

// ------------------------------------------------------------- PTX helpers --
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
// takes `bytes` that no copy will bring off the current phase of this CTA's barrier
__device__ __forceinline__ void mbar_complete_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.complete_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// the same barrier of CTA `rank` of the cluster (a shared::cluster address)
__device__ __forceinline__ uint32_t mbar_of(uint64_t* bar, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_u32(bar)), "r"(rank));
    return r;
}
// a 64-bit word of CTA `rank`'s shared memory
__device__ __forceinline__ int64_t load_of(const int64_t* p, uint32_t rank) {
    uint32_t a;
    int64_t v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
    asm volatile("ld.shared::cluster.s64 %0, [%1];" : "=l"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t addr) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(addr) : "memory");
}
__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint64_t global_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// Bounded wait (limit_ns of wall time, 2 s by default); false when it gave up
// or another thread of the block aborted.  A limit of 0 gives up at the first
// poll that finds the phase incomplete.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, volatile int* abort, uint64_t limit_ns) {
    if (mbar_try_wait(bar, parity)) return true;
    const uint64_t t0 = global_ns();
    for (uint32_t i = 0;; i++) {
        if ((i & 255u) == 0u) {   // first after a failed poll, then every 256 polls
            if (*abort) return false;
            if (global_ns() - t0 >= limit_ns) return false;
        }
        if (mbar_try_wait(bar, parity)) return true;
    }
}
// Bounded wait that ignores the abort flag (used to drain own async work).
__device__ __forceinline__ bool mbar_wait_plain(uint64_t* bar, uint32_t parity) {
    const uint64_t t0 = global_ns();
    for (uint32_t i = 0;; i++) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((i & 255u) == 255u && global_ns() - t0 > 2000000000ull) return false;
    }
}
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* tm, int x, int y, int z, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(tm)), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
        : "memory");
}
// the same load by a CTA of a pair, its bytes counted by the leader's barrier
__device__ __forceinline__ void tma_load_3d_pair(void* dst, const CUtensorMap* tm, int x, int y, int z, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(tm)), "r"(x), "r"(y), "r"(z), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Shared-memory matrix descriptor: K-major operand tile in the 128-byte swizzle
// layout TMA writes (rows of 128 B, 8-row atoms 1024 B apart).
__device__ __forceinline__ uint64_t sdesc_sw128(uint32_t saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFFu);   // start address
    d |= (uint64_t)1u << 16;                   // leading byte offset (unused for swizzled K-major)
    d |= (uint64_t)(1024u >> 4) << 32;         // stride byte offset: 8 rows x 128 B
    d |= (uint64_t)1u << 46;                   // descriptor version for tcgen05
    d |= (uint64_t)2u << 61;                   // SWIZZLE_128B
    return d;
}

// Instruction descriptor: D = F32, A = B = format F, both K-major, M = 128 (a
// pair: 256, 128 rows per CTA), N = kBN (a pair: kPairN).
template <int F, bool PAIR>
__host__ __device__ constexpr uint32_t idesc() {
    return (1u << 4) | (Fmt<F>::kAB << 7) | (Fmt<F>::kAB << 10) | ((uint32_t)((PAIR ? kPairN : kBN) >> 3) << 17) |
           ((uint32_t)((PAIR ? 2 * kBM : kBM) >> 4) << 24);
}

// One MMA over 32 bytes of K (8 TF32 or 16 BF16/FP16 elements).
template <int F, bool PAIR>
__device__ __forceinline__ void umma(uint32_t taddr, uint64_t ad, uint64_t bd, uint32_t acc) {
    if constexpr (F == FMT_TF32 && !PAIR) {
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "setp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(taddr),
            "l"(ad), "l"(bd), "r"(idesc<F, PAIR>()), "r"(acc)
            : "memory");
    } else if constexpr (F == FMT_TF32) {
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "setp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::2.kind::tf32 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(taddr),
            "l"(ad), "l"(bd), "r"(idesc<F, PAIR>()), "r"(acc)
            : "memory");
    } else if constexpr (!PAIR) {
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "setp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(taddr),
            "l"(ad), "l"(bd), "r"(idesc<F, PAIR>()), "r"(acc)
            : "memory");
    } else {
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "setp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(taddr),
            "l"(ad), "l"(bd), "r"(idesc<F, PAIR>()), "r"(acc)
            : "memory");
    }
}
// bar (a pair: this barrier of both CTAs) arrives when the MMAs issued so far are done
template <bool PAIR>
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
    if constexpr (PAIR) {
        asm volatile(
            "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
                smem_u32(bar)),
            "h"((uint16_t)3)
            : "memory");
    } else {
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                     : "memory");
    }
}

__device__ __forceinline__ void tmem_ld32_issue(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
    tmem_ld32_issue(taddr, r);
    tmem_ld_wait();
}
// Store 32 columns of this warp's 32 TMEM lanes (one register per column) and
// wait until the stores have completed.
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
        "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
        "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};"
        ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
          "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]),
          "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]),
          "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
        : "memory");
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// Persistent warp-specialised GEMM: each CTA (one per SM) walks the tiles
// blockIdx.x, blockIdx.x + gridDim.x, ...  Warp 0 lane 0 streams the K-blocks
// of all its tiles through the kStages shared-memory ring by TMA; warp 1
// lane 0 issues tcgen05.mma into the TMEM accumulators; warps 4-11 (two per
// TMEM lane quadrant) drain a finished item (a tile, or one K segment of a
// long tile) while the producer already loads the next one.  The MMA warp
// starts an item only after the epilogue has released that item's accumulator
// set (acc_empty), and the epilogue starts after the item's last MMA
// completes (acc_full).  Every wait is bounded.
// A warpgroup with the producer and the MMA warp (the other two idle) and two of
// epilogue warps.  At launch 12 warps have 168 registers a thread; the first
// warpgroup keeps kRegsFew and each epilogue thread takes kRegsEpi.  With 168 for
// all (10 warps) the epilogue spilled 28 to 240 bytes, and every step bound by its
// output slowed with the spills, staged or not (16 terms by 2^17 outputs 1.06 ms
// at 68 bytes, 1.15 at 240, 0.97 without); all GEMMs of the 10^6-shot job 113.4 ->
// 110.1 ms together with the placed fragments.
constexpr int kGemmThreads = 384;
constexpr int kRegsFew = 72, kRegsEpi = 208;
static_assert(128 * kRegsFew + 256 * kRegsEpi <= kGemmThreads * 168, "registers of the launch");
constexpr int kPairKb = 8;          // least k-blocks run by CTA pairs (2 segments of 4)
constexpr int64_t kPairRows = 4;    // least M tiles per trajectory of a stacked GEMM run by CTA pairs
struct TileInfo {              // (rows and instances are TMA coordinates: 32 bits)
    int inst, h, row_end, m0, n0, za, zb, out;   // out: instance written (unstacked)
};
__device__ __forceinline__ TileInfo decode_tile(const GemmArgs& g, int64_t tile) {
    TileInfo t;
    if (!g.stacked) {
        const int64_t tm = tile & (((int64_t)1 << g.tm_log) - 1), tn = (tile >> g.tm_log) & (((int64_t)1 << g.tn_log) - 1);
        const int64_t zt = tile >> (g.tm_log + g.tn_log);
        t.inst = (int)(zt >> g.n_hb);
        t.h = (int)(zt & (((int64_t)1 << g.n_hb) - 1));
        t.m0 = (int)(tm * kBM);
        t.n0 = (int)(tn * g.bn);
        t.row_end = g.M;
        t.out = g.out_map ? g.out_map[t.inst] : t.inst;
        const int pa = g.a_pcls == g.out_cls ? t.inst : (g.a_pcls == CLS_TRAJ ? g.net_tl[t.inst] : 0);
        const int pb = g.b_pcls == g.out_cls ? t.inst : (g.b_pcls == CLS_TRAJ ? g.net_tl[t.inst] : 0);
        t.za = pa * g.n_h + t.h;
        t.zb = pb * g.n_h + t.h;
    } else {
        // group (trajectory) of this tile: largest grp with grp_tile0[grp] <= tile
        int64_t lo = 0, hi = g.n_groups - 1;
        while (lo < hi) {
            const int64_t mid = (lo + hi + 1) >> 1;
            if (g.grp_tile0[mid] <= tile) lo = mid;
            else hi = mid - 1;
        }
        const int64_t r = tile - g.grp_tile0[lo];
        const int64_t r0 = (int64_t)g.grp_net0[lo] << g.m_bits, r1 = (int64_t)g.grp_net0[lo + 1] << g.m_bits;
        const int64_t tmg = ((r1 - r0 + kBM - 1) / kBM + g.pair) & ~(int64_t)g.pair;   // pairs: an even number
        t.m0 = (int)(r0 + (r % tmg) * kBM);
        t.n0 = (int)((r / tmg) * g.bn);
        t.inst = (int)lo;     // the trajectory (local index) supplies the B operand
        t.h = t.out = 0;
        t.row_end = (int)r1;
        t.za = 0;
        t.zb = g.b_pcls == CLS_TRAJ ? (int)lo : 0;
    }
    return t;
}

// The tiles of a CTA as a warp sees them: lane l decodes the l-th of the next 32
// at once (a stacked tile's group takes a binary search of dependent reads, so
// one search's latency serves 32 tiles) and the warp takes them by shuffles.
struct TileQueue {
    TileInfo mine;
    int64_t i = 0;
    __device__ __forceinline__ bool next(const GemmArgs& g, int lane, TileInfo& t) {
        const int64_t tile = blockIdx.x + i * gridDim.x;
        if (tile >= g.n_tiles) return false;
        const int l = (int)(i & 31);
        if (l == 0) {
            const int64_t ahead = tile + (int64_t)lane * gridDim.x;
            mine = decode_tile(g, ahead < g.n_tiles ? ahead : tile);
        }
        t.inst = __shfl_sync(0xffffffffu, mine.inst, l);
        t.h = __shfl_sync(0xffffffffu, mine.h, l);
        t.row_end = __shfl_sync(0xffffffffu, mine.row_end, l);
        t.m0 = __shfl_sync(0xffffffffu, mine.m0, l);
        t.n0 = __shfl_sync(0xffffffffu, mine.n0, l);
        t.za = __shfl_sync(0xffffffffu, mine.za, l);
        t.zb = __shfl_sync(0xffffffffu, mine.zb, l);
        t.out = __shfl_sync(0xffffffffu, mine.out, l);
        i++;
        return true;
    }
};
__device__ __forceinline__ float pow2f(int e) { return __int_as_float((127 + e) << 23); }   // |e| <= 126

// PAIR: two CTAs of a cluster work on 256 x 256 tiles (cta_group::2): each
// stages its own 128 A rows and half of the B rows, both tensor cores read both
// halves.  A 128 x 128 tile is bound by shared memory: per k-block its 12 MMAs
// read 96 KB and TMA writes 64 KB, 1280 clocks at 128 bytes each, and takes 1370
// to 1430 where the MMAs alone take 768 (64 clocks each with resident operands);
// a pair of 128 columns measured the same 1380.  With 256 columns a CTA's k-block
// has twice the work for the same 64 KB written.  Two accumulators of a pair fill
// TMEM, so its tiles are summed from segments of one accumulator: the first one
// stays where it is, the others are accumulated beside it and added to it, and the
// two regions change places from tile to tile, so that a tile is stored while the
// next one's first segment runs.  Long contractions have segments anyway; those of
// 8 and 16 k-blocks run their 2 and 4 accumulators (every second, every fourth
// k-block) one after the other.  The even CTA leads: its producer counts both
// CTAs' bytes, its MMA thread issues for both and signals freed stages and finished
// accumulators to both, and both CTAs' epilogue warps free a region at its barrier.
// The products, their order and the order of the sums are those of one CTA, so
// every output is the same.  Measured: the middle 30-qubit block's step of 4096
// terms (FP16 hi/lo) 64.3 -> 51.8 to 53.5 ms (516 to 533 TFLOP/s, 0.95 of the
// sustained peak / 3 with its padded rows), its 256 terms by 2^18 outputs 4.34 ->
// 3.79 ms; of the 16-qubit state (TF32) 512 terms 9.57 -> 6.20 ms (355 TFLOP/s),
// 256 terms 11.26 -> 8.53 ms.
template <int F, bool PAIR>
__global__ void __launch_bounds__(kGemmThreads, 1) k_gemm(const __grid_constant__ CUtensorMap tmA,
                                                          const __grid_constant__ CUtensorMap tmB,
                                                          const __grid_constant__ GemmArgs g) {
    constexpr int kBK = kRowBytes / Fmt<F>::kBytes;   // elements per swizzle row
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t* stage0 = smem;
    constexpr int NST = kStages, TN = PAIR ? kPairN : kBN;   // columns of a tile
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + kStages * kStageBytes);   // a pair: the leader's count
    uint64_t* empty = full + NST;
    uint64_t* acc_full = empty + NST;       // per accumulator set
    uint64_t* acc_empty = acc_full + 2;     // a pair: the leader's count
    uint64_t* drain = acc_empty + 2;
    uint32_t* tslot = reinterpret_cast<uint32_t*>(drain + 1);
    volatile int* abort = reinterpret_cast<volatile int*>(tslot + 1);
    int64_t* issued = reinterpret_cast<int64_t*>(tslot + 2);   // a pair: stages this CTA's producer loaded
    // tables of the 8 epilogue warps, 16-byte aligned (the scales are read four at
    // a time; the barriers before them end 8 bytes past a boundary)
    constexpr int kTabOff = (int)(((2 * NST + 5) * 8 + 16 + 15) & ~15);
    static_assert(kTabOff % 16 == 0 && kTabOff + 8 * (kBN / 2) * 12 <= kTabBytes, "epilogue tables");
    int64_t* noff_all = reinterpret_cast<int64_t*>(smem + kStages * kStageBytes + kTabOff);   // kBN / 2 column offsets each
    float* ucol_all = reinterpret_cast<float*>(noff_all + 8 * (kBN / 2));   // FP16: column scales 2^eb
    float2* stg_all = reinterpret_cast<float2*>(smem + kStages * kStageBytes + kTabBytes);   // staged fragments
    const uint32_t rank = PAIR ? cluster_rank() : 0u;
    // Work items are (tile, K segment) pairs.  A tile's k-blocks run in
    // segments of at most kSegKb; the tensor core's accumulation truncates, so
    // long chains drift: every segment is accumulated on its own and the
    // epilogue adds the segments in FP32 (round to nearest), in order, into a
    // running sum kept in TMEM columns [2 kBN, 3 kBN), then writes the tile
    // once.  Segmented tiles use two accumulator sets of one accumulator, short
    // contractions (at most 8 k-blocks) two sets of kAcc / 2 (the epilogue of
    // one item overlaps the MMAs of the next); the others one set of kAcc.
    // A pair runs the accumulators of a short contraction (k-blocks j, j + n_seg,
    // ... of accumulator j) one after the other, as segments (`split`).
    const bool split = PAIR && g.nkb <= kSegKb;
    const int n_scale = (g.nkb + kSegKb - 1) / kSegKb;   // FP16 scales per row and column
    const int split_acc = g.nkb <= 8 ? kAcc / 2 : kAcc;
    const int seg_kb = split ? g.nkb / split_acc : (g.nkb > kSegKb ? kSegKb : g.nkb);
    const int n_seg = (g.nkb + seg_kb - 1) / seg_kb;
    const int n_sets = !PAIR && (g.nkb <= 8 || n_seg > 1) ? 2 : 1;
    const int acc_per = n_seg > 1 ? 1 : kAcc / n_sets;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 32) {
        for (int s = 0; s < NST; s++) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int k = 0; k < 2; k++) {
            mbar_init(&acc_full[k], 1);
            mbar_init(&acc_empty[k], PAIR ? 16 : 8);   // one arrival per epilogue warp
        }
        mbar_init(drain, 1);
        *abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if constexpr (PAIR) {
        // both CTAs' barriers exist before either signals the other's
        __syncthreads();
        cluster_sync();
        if (warp == 0) {
            asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                         "r"(kTmemCols)
                         : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
        }
        tc_fence_before();
        __syncthreads();
        cluster_sync();              // the peer's accumulators are allocated too
    } else {
        if (warp == 0) {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                         "r"(kTmemCols)
                         : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        }
        tc_fence_before();
        __syncthreads();
    }
    tc_fence_after();
    const uint32_t tmem = *tslot;
    const int64_t n_tiles = g.n_tiles;

    if (warp < 4) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsFew));
        if (warp == 0) {
            int64_t it = 0;
            TileQueue tq;
            TileInfo t;
            while (!__shfl_sync(0xffffffffu, *abort, 0) && tq.next(g, lane, t)) {
                if (lane == 0) {
                    for (int i = 0; i < g.nkb; i++, it++) {
                        const int kb = split ? i % seg_kb * n_seg + i / seg_kb : i;
                        const int s = (int)(it % NST);
                        if (it >= NST && !mbar_wait(&empty[s], (uint32_t)((it / NST) - 1) & 1u, abort, g.wait_ns)) {
                            atomicExch(g.err, 1);
                            *abort = 1;
                            break;
                        }
                        uint8_t* st = stage0 + s * kStageBytes;
                        if constexpr (PAIR) {
                            if (rank == 0) mbar_expect_tx(&full[s], (uint32_t)(2 * kStageBytes));   // both CTAs' copies
                            const uint32_t bar = mbar_of(&full[s], 0);
                            const int n0 = t.n0 + (int)rank * kBN;                                   // this CTA's half of B
                            tma_load_3d_pair(st, &tmA, kb * kBK, t.m0, t.za, bar);
                            tma_load_3d_pair(st + kTileA, &tmA, g.Kh + kb * kBK, t.m0, t.za, bar);
                            tma_load_3d_pair(st + 2 * kTileA, &tmB, kb * kBK, n0, t.zb, bar);
                            tma_load_3d_pair(st + 2 * kTileA + kTileB, &tmB, g.Kh + kb * kBK, n0, t.zb, bar);
                        } else {
                            mbar_expect_tx(&full[s], (uint32_t)kStageBytes);
                            tma_load_3d(st, &tmA, kb * kBK, t.m0, t.za, &full[s]);                          // A hi
                            tma_load_3d(st + kTileA, &tmA, g.Kh + kb * kBK, t.m0, t.za, &full[s]);          // A lo
                            tma_load_3d(st + 2 * kTileA, &tmB, kb * kBK, t.n0, t.zb, &full[s]);             // B hi
                            tma_load_3d(st + 2 * kTileA + kTileB, &tmB, g.Kh + kb * kBK, t.n0, t.zb, &full[s]);   // B lo
                        }
                    }
                }
                __syncwarp();
            }
            if (lane == 0) {
                // let this CTA's own copies land before it exits (on every path: the
                // MMA thread may have stopped early): the last load of every stage
                // is that stage's newest phase
                // (a pair's are counted by the leader: below, when both producers have stopped)
                const int64_t first = it > NST ? it - NST : 0;
                if (PAIR) *issued = it;
                else
                    for (int64_t j = first; j < it; j++) mbar_wait_plain(&full[j % NST], (uint32_t)(j / NST) & 1u);
            }
            __syncwarp();
        } else if (warp == 1) {
            if (lane == 0 && rank == 0) {
                int64_t it = 0, lt = 0;
                bool ok = true;
                uint32_t used = 0, phase = 0, x = 1;   // a pair: regions used, their waits' parities, the tile's sum
                for (int64_t tile = blockIdx.x; tile < n_tiles && !*abort && ok; tile += gridDim.x) {
                    x ^= 1;
                    for (int sg = 0; sg < n_seg && ok; sg++, lt++) {
                        const int set = PAIR ? (int)(sg ? x ^ 1 : x) : (int)(lt % n_sets);
                        const bool again = PAIR ? (used >> set) & 1 : lt >= n_sets;
                        const uint32_t parity = PAIR ? (phase >> set) & 1 : (uint32_t)((lt / n_sets - 1) & 1);
                        if (again) phase ^= 1u << set;
                        used |= 1u << set;
                        // this set's previous item has been drained by the epilogue
                        if (again && !mbar_wait(&acc_empty[set], parity, abort, g.wait_ns)) {
                            atomicExch(g.err, 4);
                            *abort = 1;
                            ok = false;
                            break;
                        }
                        tc_fence_after();
                        const int kb0 = sg * seg_kb, kb1 = kb0 + seg_kb < g.nkb ? kb0 + seg_kb : g.nkb;
                        for (int kb = kb0; kb < kb1; kb++, it++) {
                            const int s = (int)(it % NST);
                            if (!mbar_wait(&full[s], (uint32_t)(it / NST) & 1u, abort, g.wait_ns)) {
                                atomicExch(g.err, 2);
                                *abort = 1;
                                ok = false;
                                break;
                            }
                            tc_fence_after();
                            const uint32_t sa = smem_u32(stage0 + s * kStageBytes);
                            const uint32_t sal = sa + kTileA, sb = sa + 2 * kTileA, sbl = sb + kTileB;
                            const int j = kb - kb0;
                            const uint32_t acc = tmem + (uint32_t)((set * acc_per + j % acc_per) * TN);
                            const bool fresh = j < acc_per;
    #pragma unroll
                            for (int kk = 0; kk < kRowBytes / 32; kk++) {   // 32 bytes of K per MMA
                                const uint32_t o = kk * 32;
                                umma<F, PAIR>(acc, sdesc_sw128(sa + o), sdesc_sw128(sb + o), (fresh && kk == 0) ? 0u : 1u);
                                umma<F, PAIR>(acc, sdesc_sw128(sa + o), sdesc_sw128(sbl + o), 1u);
                                umma<F, PAIR>(acc, sdesc_sw128(sal + o), sdesc_sw128(sb + o), 1u);
                            }
                            umma_commit<PAIR>(&empty[s]);   // stage free once these MMAs have read it
                        }
                        if (!ok) break;
                        umma_commit<PAIR>(&acc_full[set]);  // accumulators complete for this item
                    }
                }
                // MMAs still in flight finish before TMEM is freed (on every path: the
                // epilogue may have stopped early)
                umma_commit<PAIR>(drain);
                mbar_wait_plain(drain, 0u);
            }
            __syncwarp();
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsEpi));
        // epilogue warps 4..11: TMEM lane quadrant q = warp % 4 holds tile rows
        // 32q..32q+31; two warps per quadrant drain half of the tile's columns
        // each (one warp per SM sub-partition leaves its load and store
        // latencies exposed).  Where the lowest five output bits are row bits a
        // lane stores its own row's columns and the warp writes 256 consecutive
        // bytes.  Every other layout goes through a staged fragment whose
        // elements the lanes take in the order of the output (sorting the
        // fragment's row and column bits by stride): a layout of 2^20 outputs
        // by 128 terms with seven low column bits wrote at 1.4 TB/s with four
        // warps staging 16 columns.  4096 trajectories of the middle 30-qubit
        // block: that step 23.9 -> 16.1 ms, one with four hyper bits (55 GB)
        // 12.7 -> 9.1 ms (6.0 TB/s); all GEMMs of the 10^6-shot job 149 -> 132 ms.
        const int ew = warp - 4, q = warp & 3;
        const int c_lo = (ew >> 2) * (TN / 2), c_hi = c_lo + TN / 2;
        // this warp's columns, from c_lo / 2 on (a single CTA's tables have room for all)
        int64_t* noff = noff_all + ew * (kBN / 2) - (PAIR ? c_lo / 2 : 0);
        float* ucol = ucol_all + ew * (kBN / 2) - (PAIR ? c_lo / 2 : 0);
        float2* stg = stg_all + ew * kStgElems;
        int sm_l = 0, row_l = 0, st_l = 0;
        int64_t out_l = (q & 1 ? g.row_hi[0] : 0) + (q & 2 ? g.row_hi[1] : 0);
        for (int b = 0; b < 5; b++)
            if ((lane >> b) & 1) {
                sm_l ^= g.frag_sm[b + 1];
                st_l ^= g.row_sm[b];
                row_l += g.frag_row[b + 1];
                out_l += g.frag_out[b + 1];
            }
        int64_t lt = 0;
        uint32_t phase = 0, x = 1;   // a pair: parities of the regions' waits, the tile's running sum
        bool live = true;
        auto release_set = [&](int set) {
            if constexpr (PAIR) mbar_arrive_cluster(mbar_of(&acc_empty[set], 0));
            else mbar_arrive(&acc_empty[set]);
        };
        TileQueue tq;
        TileInfo t, tn;
        bool more = tq.next(g, lane, tn);
        // FP16: this lane's row and column exponents of a tile's segment 0, read one
        // tile ahead (their latency would precede every tile of a short contraction)
        int ea = 0, eb = 0, eb1 = 0;   // (a pair's warp has 64 columns)
        auto read_exps = [&](const TileInfo& x, int sg, int& a, int& b, int& b1) {
            const int64_t row = (int64_t)x.m0 + q * 32 + lane;
            a = row < x.row_end ? g.exp_a[((int64_t)x.za * g.M + row) * n_scale + sg] : 0;
            const int64_t col = (int64_t)x.zb * (g.N2 >> 1) + (x.n0 >> 1) + (c_lo >> 1) + lane;
            b = g.exp_b[col * n_scale + sg];
            if (PAIR) b1 = g.exp_b[(col + 32) * n_scale + sg];
        };
        if (F == FMT_FP16 && more) read_exps(tn, 0, ea, eb, eb1);
        while (more && live) {
            if (__shfl_sync(0xffffffffu, *abort, 0)) break;   // warp-uniform stop
            t = tn;
            more = tq.next(g, lane, tn);
            // output offsets of this warp's columns (staged: of its fragments' first columns)
            for (int c = c_lo / 2 + lane; c < c_hi / 2; c += 32) {
                const int64_t n = (int64_t)(t.n0 / 2) + c;
                int64_t off = 0;
                for (int i = 0; i < g.n_nb; i++)
                    if ((n >> i) & 1) off += g.n_stride[i];
                noff[c] = off;
            }
            const int64_t row = (int64_t)t.m0 + q * 32 + lane;
            const int64_t row0 = g.staged ? (int64_t)t.m0 : row;   // staged: the tile's first row
            int64_t m = row0, out_inst = t.out;
            if (g.stacked) {
                out_inst = row0 >> g.m_bits;
                m = row0 & (((int64_t)1 << g.m_bits) - 1);
            }
            int64_t moff = 0;
            for (int i = 0; i < g.n_mb; i++)
                if ((m >> i) & 1) moff += g.m_stride[i];
            for (int i = 0; i < g.n_hb; i++)
                if ((t.h >> i) & 1) moff += g.h_stride[i];
            const bool row_ok = row < t.row_end;
            const int row_lim = min(t.row_end - t.m0, 128) - q * 32;   // valid rows of this quadrant
            float2* out = g.out + (row_ok || g.staged ? out_inst : 0) * g.out_size + moff + (g.staged ? out_l : 0);
            __syncwarp();
            x ^= 1;
            float urow = 1.f;
            for (int sg = 0; sg < n_seg; sg++, lt++) {
                const int set = PAIR ? (int)(sg ? x ^ 1 : x) : (int)(lt % n_sets);
                const uint32_t acc0 = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(set * acc_per * TN);
                const int seg_len = (sg + 1) * seg_kb < g.nkb ? seg_kb : g.nkb - sg * seg_kb;
                const int n_acc = seg_len < acc_per ? seg_len : acc_per;
                const bool add = sg > 0;   // later segments add to the running sum
                // FP16: the segment's A row scale 2^ea (packed row za * M + row) and
                // column scales 2^eb; their product 2^(ea + eb) is exact
                if (F == FMT_FP16 && !(split && sg)) {
                    if (sg > 0) read_exps(t, sg, ea, eb, eb1);
                    __syncwarp();        // the previous segment's scales are no longer read
                    ucol[c_lo / 2 + lane] = pow2f(eb);
                    if (PAIR) ucol[c_lo / 2 + 32 + lane] = pow2f(eb1);
                    urow = pow2f(ea);
                    if ((split || sg + 1 == n_seg) && more) read_exps(tn, 0, ea, eb, eb1);
                    __syncwarp();
                }
                // one lane waits and the warp follows its outcome (lanes polling on
                // their own could disagree when a wait gives up)
                int ok = 1;
                const uint32_t parity = PAIR ? (phase >> set) & 1 : (uint32_t)((lt / n_sets) & 1);
                phase ^= 1u << set;
                if (lane == 0) ok = mbar_wait(&acc_full[set], parity, abort, g.wait_ns) ? 1 : 0;
                ok = __shfl_sync(0xffffffffu, ok, 0);
                if (!ok) {
                    if (lane == 0) {
                        atomicExch(g.err, 3);
                        *abort = 1;
                    }
                    live = false;
                    break;
                }
                __syncwarp();
                tc_fence_after();
                // one chunk of 32 columns of this thread's row: v[2j], v[2j+1] = complex
                // column (c0 / 2 + j), written through the output strides
                auto store_chunk = [&](int c0, const float* v) {
                    if (g.staged) {
#pragma unroll
                        for (int f = 0; f < 2; f++) {
#pragma unroll
                            for (int j = 0; j < 8; j++)
                                stg[st_l ^ (j & 1 ? g.col_sm[0] : 0) ^ (j & 2 ? g.col_sm[1] : 0) ^ (j & 4 ? g.col_sm[2] : 0)] =
                                    make_float2(v[16 * f + 2 * j], v[16 * f + 2 * j + 1]);
                            __syncwarp();
                            float2* o = out + noff[(c0 >> 1) + 8 * f];
#pragma unroll
                            for (int i = 0; i < 4; i++) {
                                const int sm = sm_l ^ (i & 1 ? g.frag_sm[6] : 0) ^ (i & 2 ? g.frag_sm[7] : 0);
                                const int rr = row_l + (i & 1 ? g.frag_row[6] : 0) + (i & 2 ? g.frag_row[7] : 0);
                                float2* d = o + ((i & 1 ? g.frag_out[6] : 0) + (i & 2 ? g.frag_out[7] : 0));
                                const float2 x = stg[sm], y = stg[sm ^ g.frag_sm[0]];
                                if (g.frag_vec && rr + g.frag_row[0] < row_lim) {
                                    *reinterpret_cast<float4*>(d) = make_float4(x.x, x.y, y.x, y.y);
                                } else {
                                    if (rr < row_lim) d[0] = x;
                                    if (rr + g.frag_row[0] < row_lim) d[g.frag_out[0]] = y;
                                }
                            }
                            __syncwarp();
                        }
                    } else if (row_ok) {
#pragma unroll
                        for (int j = 0; j < 16; j++) out[noff[(c0 >> 1) + j]] = make_float2(v[2 * j], v[2 * j + 1]);
                    }
                };
                auto scale_chunk = [&](int c0, float (&v)[32]) {   // FP16: by the row's and the columns' scales
#pragma unroll
                    for (int j = 0; j < 16; j += 4) {
                        const float4 u4 = *reinterpret_cast<const float4*>(ucol + (c0 >> 1) + j);
                        const float u[4] = {urow * u4.x, urow * u4.y, urow * u4.z, urow * u4.w};
#pragma unroll
                        for (int i = 0; i < 4; i++) {
                            v[2 * (j + i)] *= u[i];
                            v[2 * (j + i) + 1] *= u[i];
                        }
                    }
                };
                if constexpr (PAIR) {
                    // the tile's first segment stays where it is and the others are
                    // added to it; the other region is free again after each
                    const uint32_t sum = tmem + ((uint32_t)(q * 32) << 16) + x * TN;
                    const bool scale = F == FMT_FP16 && !split;   // per segment (else once, before the stores)
                    if (sg > 0 || scale) {
#pragma unroll 1
                        for (int c0 = c_lo; c0 < c_hi; c0 += 32) {
                            float v[32];
                            uint32_t r[32], r2[32];
                            tmem_ld32_issue(acc0 + (uint32_t)c0, r);
                            if (sg > 0) tmem_ld32_issue(sum + (uint32_t)c0, r2);
                            tmem_ld_wait();
#pragma unroll
                            for (int j = 0; j < 32; j++) v[j] = __uint_as_float(r[j]);
                            if (scale) scale_chunk(c0, v);
                            if (sg > 0) {
#pragma unroll
                                for (int j = 0; j < 32; j++) v[j] += __uint_as_float(r2[j]);
                            }
#pragma unroll
                            for (int j = 0; j < 32; j++) r[j] = __float_as_uint(v[j]);
                            tmem_st32(sum + (uint32_t)c0, r);
                        }
                    }
                    if (sg > 0) {
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) release_set(set);
                    }
                    if (sg + 1 < n_seg) continue;
#pragma unroll 1
                    for (int c0 = c_lo; c0 < c_hi; c0 += 32) {   // the tile, while the next one starts
                        float v[32];
                        uint32_t r[32];
                        tmem_ld32(sum + (uint32_t)c0, r);
                        if (c0 + 32 >= c_hi) {
                            tc_fence_before();
                            __syncwarp();
                            if (lane == 0) release_set((int)x);
                        }
#pragma unroll
                        for (int j = 0; j < 32; j++) v[j] = __uint_as_float(r[j]);
                        if (F == FMT_FP16 && split) scale_chunk(c0, v);
                        store_chunk(c0, v);
                    }
                    continue;
                }
                if (n_seg == 1) {
#pragma unroll 1
                    for (int c0 = c_lo; c0 < c_hi; c0 += 32) {
                        // accumulators two at a time, added in order
                        float v[32];
                        uint32_t r[32], r2[32];
                        tmem_ld32_issue(acc0 + (uint32_t)c0, r);
                        if (n_acc > 1) tmem_ld32_issue(acc0 + (uint32_t)(kBN + c0), r2);
                        tmem_ld_wait();
#pragma unroll
                        for (int j = 0; j < 32; j++) v[j] = __uint_as_float(r[j]);
                        if (n_acc > 1) {
#pragma unroll
                            for (int j = 0; j < 32; j++) v[j] += __uint_as_float(r2[j]);
                        }
                        if (n_acc > 2) {
                            tmem_ld32_issue(acc0 + (uint32_t)(2 * kBN + c0), r);
                            if (n_acc > 3) tmem_ld32_issue(acc0 + (uint32_t)(3 * kBN + c0), r2);
                            tmem_ld_wait();
#pragma unroll
                            for (int j = 0; j < 32; j++) v[j] += __uint_as_float(r[j]);
                            if (n_acc > 3) {
#pragma unroll
                                for (int j = 0; j < 32; j++) v[j] += __uint_as_float(r2[j]);
                            }
                        }
                        if (c0 + 32 >= c_hi) {   // everything read: the set may take its next item while the tile is stored
                            tc_fence_before();
                            __syncwarp();
                            if (lane == 0) release_set(set);
                        }
                        if (F == FMT_FP16) scale_chunk(c0, v);
                        store_chunk(c0, v);
                    }
                } else {
                    // segmented: add this segment to the running sum in TMEM; the
                    // last one writes the tile
#pragma unroll 1
                    for (int c0 = c_lo; c0 < c_hi; c0 += 32) {
                        float v[32];
                        uint32_t r[32];
                        tmem_ld32(acc0 + (uint32_t)c0, r);
#pragma unroll
                        for (int j = 0; j < 32; j++) v[j] = __uint_as_float(r[j]);
                        if (F == FMT_FP16) scale_chunk(c0, v);
                        const uint32_t sa = tmem + ((uint32_t)(q * 32) << 16) + 2 * kBN + (uint32_t)c0;
                        if (add) {
                            tmem_ld32(sa, r);
#pragma unroll
                            for (int j = 0; j < 32; j++) v[j] += __uint_as_float(r[j]);
                        }
                        if (sg + 1 < n_seg) {
#pragma unroll
                            for (int j = 0; j < 32; j++) r[j] = __float_as_uint(v[j]);
                            tmem_st32(sa, r);
                        } else {
                            store_chunk(c0, v);
                        }
                    }
                }
                if (n_seg > 1) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) release_set(set);   // accumulators read: this set may take the next item
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if constexpr (PAIR) {
        // The peer's MMAs read this CTA's shared memory and write its TMEM, its
        // barriers are signalled from here, and the leader's count the copies of
        // both: neither frees or leaves before all of that has ended.
        cluster_sync();              // no wait, load or MMA is started by either from here on
        if (threadIdx.x == 0) {
            if (rank == 0) {
                // After a wait that ran out the producers may have stopped at different
                // stages.  A stage that one of them alone loaded (at most NST: both wait
                // for the same MMAs) is settled for the half that is missing; then the
                // newest phase of every stage ends with the last copy in flight.
                const int64_t mine = *issued, peer = load_of(issued, 1);
                const int64_t lo = mine < peer ? mine : peer, hi = mine < peer ? peer : mine;
                for (int64_t j = lo; j < hi; j++) {
                    if (mine > peer) mbar_complete_tx(&full[j % NST], (uint32_t)kStageBytes);
                    else mbar_expect_tx(&full[j % NST], (uint32_t)kStageBytes);
                }
                for (int64_t j = hi > NST ? hi - NST : 0; j < hi; j++)
                    mbar_wait_plain(&full[j % NST], (uint32_t)(j / NST) & 1u);
            } else {
                mbar_wait_plain(drain, 0u);   // the leader's last commit, signalled to both
            }
        }
        __syncwarp();
    }
    if (warp == 0) {
        tc_fence_after();
        if constexpr (PAIR)
            asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
        else
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
    }
    if constexpr (PAIR) {
        __syncthreads();
        cluster_sync();
    }
}

// Tiles of every trajectory group of a stacked GEMM (cnt[n_groups] = 0, so the
// exclusive scan of cnt ends with the total).
__global__ void k_group_tiles(const int32_t* __restrict__ net0, int64_t n_groups, int m_bits, int64_t tiles_n, int pair,
                              int64_t* __restrict__ cnt) {
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (g > n_groups) return;
    if (g == n_groups) {
        cnt[g] = 0;
        return;
    }
    const int64_t r = (int64_t)(net0[g + 1] - net0[g]) << m_bits;
    cnt[g] = (((r + kBM - 1) / kBM + pair) & ~(int64_t)pair) * tiles_n;
}

// ---------------------------------------------------------- host helpers --
std::atomic<uint64_t> g_wait_ns{2000000000ull};   // limit of the GEMM's pipeline waits
thread_local uint64_t t_gemm_forms = 0;   // this thread's launches since gemm_forms_reset: pairs or single CTAs

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
    // thread-safe one-time lookup (function-local static initialisation)
    static const EncodeTiledFn fn = []() -> EncodeTiledFn {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            return reinterpret_cast<EncodeTiledFn>(p);
        return nullptr;
    }();
    return fn;
}

// 3D map over packed rows: (elements of a row, rows, instances), boxes of one
// 128-byte swizzle row by box_rows rows.
ptn_status make_map(CUtensorMap* m, void* base, CUtensorMapDataType dt, int ebytes, int64_t row_elems, int64_t rows,
                    int64_t zs, int box_rows) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return set_error(PTN_ERR_CUDA, "cuTensorMapEncodeTiled unavailable");
    cuuint64_t dims[3] = {(cuuint64_t)row_elems, (cuuint64_t)rows, (cuuint64_t)zs};
    cuuint64_t strides[2] = {(cuuint64_t)row_elems * ebytes, (cuuint64_t)row_elems * ebytes * (cuuint64_t)rows};
    cuuint32_t box[3] = {(cuuint32_t)(kRowBytes / ebytes), (cuuint32_t)box_rows, 1};
    cuuint32_t es[3] = {1, 1, 1};
    CUresult r = fn(m, dt, 3, base, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return set_error(PTN_ERR_CUDA, "cuTensorMapEncodeTiled failed (%d)", (int)r);
    return PTN_OK;
}

int pack_class(const OperandDesc& d, int step_cls) {
    if (step_cls == CLS_NET && d.n_slice) return CLS_NET;
    if (d.mode == OP_LEAF) return d.leaf_col >= 0 ? CLS_TRAJ : CLS_CONST;
    return d.cls;
}

unsigned grid_of(int64_t n) {
    int64_t b = (n + 255) / 256;
    return (unsigned)(b > 152 * 16 ? 152 * 16 : (b < 1 ? 1 : b));
}

// Whether an operand's summed axis is contiguous and its rows start on 16-byte
// boundaries (k_pack_rows).
bool pack_dense(const PackArgs& p, const ChunkCtx& c) {
    const OperandDesc& d = p.op;
    if (p.prod || p.n_kb < 3) return false;
    for (int t = 0; t < p.n_kb; t++)
        if (p.k_stride[t] != (int64_t)1 << t) return false;
    const int64_t base = d.mode == OP_LEAF ? d.leaf_base : d.arena_off * c.arena_inst[d.arena];
    int64_t odd = base | d.inst_size;
    for (int t = 0; t < p.n_rb; t++) odd |= p.r_stride[t];
    for (int t = 0; t < p.n_hb; t++) odd |= p.h_stride[t];
    for (int t = 0; t < d.n_slice; t++) odd |= d.slice_stride[t];
    return !(odd & 1);
}
// Whether the factors' elements of one packed instance fit k_pack_prod's stages.
bool pack_prod_fits(const PackArgs& p) {
    if (!p.prod || p.n_kb < 6 || (1 << (p.n_kb - 6)) > kProdHi || p.n_rb > 10) return false;
    int n[2] = {p.n_rb, p.n_rb};
    for (int t = 0; t < p.n_kb; t++) {
        n[0] += (p.k_stride[t] & kLo32) != 0;
        n[1] += (p.k_stride[t] >> 32) != 0;
    }
    return (1 << n[0]) <= kProdStage && (1 << n[1]) <= kProdStage;
}
// Tile of k_pack_tile; false where the operand is an outer product, its rows
// are padded, or the four lowest strides are not row bits: with summed bits
// among them k_pack's reads are partly contiguous and a tile has few rows (a
// step's pack at 4.35 TB/s by k_pack, 3.1 here).
bool pack_tile_split(const PackArgs& p, int role, TileArgs& t) {
    memset(&t, 0, sizeof t);
    const int64_t row = (role ? 4 : 2) * (int64_t)p.Kh;   // packed elements per operand row
    if (p.prod || ((int64_t)1 << p.n_kb) * 2 != p.Kh) return false;
    struct Bit {
        int64_t stride, dst;
        bool k, in;
    } bits[2 * kMaxPackBits];        // store order: summed bits, then rows
    int order[2 * kMaxPackBits], place[2 * kMaxPackBits] = {}, nb = 0;
    for (int i = 0; i < p.n_kb; i++) bits[nb++] = {p.k_stride[i], (int64_t)2 << i, true, i < 6};
    for (int i = 0; i < p.n_rb; i++) bits[nb++] = {p.r_stride[i], row << i, false, false};
    for (int i = 0; i < nb; i++) order[i] = i;
    std::sort(order, order + nb, [&](int x, int y) { return bits[x].stride < bits[y].stride; });
    if (nb < 5) return false;
    for (int i = 0; i < 4; i++)
        if (bits[order[i]].stride != (int64_t)1 << i || bits[order[i]].k) return false;
    for (int i = 0; i < 5; i++) bits[order[i]].in = true;
    for (int i = 0; i < nb; i++) {
        if (bits[i].in) {
            place[i] = 1 << t.nt;
            t.st_dst[t.nt++] = bits[i].dst;
        } else {
            t.out_stride[t.n_out] = bits[i].stride;
            t.out_dst[t.n_out++] = bits[i].dst;
        }
    }
    int n = 0;
    for (int i = 0; i < nb; i++)
        if (bits[order[i]].in) {
            t.ld_stride[n] = bits[order[i]].stride;
            t.ld_place[n++] = place[order[i]];
        }
    return true;
}
template <int F, int ROLE>
void launch_pack_rows(PackArgs p, const ChunkCtx& ctx, int64_t n_units, cudaStream_t s) {
    // a warp takes up to 32 consecutive units, fewer (at least what it handles at
    // once) where that would leave some of eight CTAs per SM without work
    const int per_log = p.n_kb < 6 ? 6 - p.n_kb : 0, un_log = p.n_kb <= 6 ? 2 : (p.n_kb == 7 ? 1 : 0);
    p.run_log = 5;
    while (p.run_log > per_log + un_log && (n_units >> p.run_log) < 152 * 8 * 8) p.run_log--;
    const int64_t per_block = (int64_t)8 << p.run_log;
    const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>((n_units + per_block - 1) / per_block, 152 * 8));
    switch (p.n_kb) {
        default: k_pack_rows<F, ROLE, 8><<<(unsigned)blocks, 256, 0, s>>>(p, ctx); break;
        case 8: k_pack_rows<F, ROLE, 4><<<(unsigned)blocks, 256, 0, s>>>(p, ctx); break;
        case 7: k_pack_rows<F, ROLE, 2><<<(unsigned)blocks, 256, 0, s>>>(p, ctx); break;
        case 6: case 5: case 4: case 3: k_pack_rows<F, ROLE, 1><<<(unsigned)blocks, 256, 0, s>>>(p, ctx); break;
    }
}
template <int F, int ROLE>
void launch_pack(const PackArgs& p, const ChunkCtx& ctx, int64_t slots, cudaStream_t s) {
    const int64_t rows = p.n_pinst << (p.n_hb + p.n_rb);
    if constexpr (F != FMT_FP16) {
        TileArgs t;
        if (!pack_dense(p, ctx) && pack_tile_split(p, ROLE, t)) {
            const int64_t tiles = (p.n_pinst << p.n_hb) << t.n_out;
            k_pack_tile<F, ROLE><<<(unsigned)std::min<int64_t>(tiles, 152 * 8), 256, 0, s>>>(p, t, ctx);
            return;
        }
    }
    if (pack_dense(p, ctx)) launch_pack_rows<F, ROLE>(p, ctx, rows << (p.n_kb > 9 ? p.n_kb - 9 : 0), s);
    else if (pack_prod_fits(p))
        k_pack_prod<F, ROLE><<<(unsigned)std::min<int64_t>(p.n_pinst << p.n_hb, 152 * 8), 256, 0, s>>>(p, ctx);
    else k_pack<F><<<grid_of(slots), 256, 0, s>>>(p, ctx);   // (grid_of sizes by complex slots; the kernel strides over rows)
}

template <int F>
ptn_status run_gemm(const StepDesc& st, const ChunkCtx& ctx, int64_t n_inst, void* pack_a, void* pack_b,
                    int* err, const GroupTable& grp, cudaStream_t s, const StepDesc* prod_src) {
    constexpr int kEB = Fmt<F>::kBytes;
    constexpr int kBK = kRowBytes / kEB;
    const CUtensorMapDataType dt = F == FMT_TF32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32
                                   : F == FMT_BF16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16
                                                   : CU_TENSOR_MAP_DATA_TYPE_FLOAT16;
    const bool stacked = st.kind == STEP_GEMM_STACKED;
    const int a = st.gemm_a, b = 1 - a;
    PackArgs pa, pb;
    memset(&pa, 0, sizeof pa);
    memset(&pb, 0, sizeof pb);
    GemmArgs ga;
    memset(&ga, 0, sizeof ga);
    int nm = 0, nn = 0, nh = 0;
    for (int p = 0; p < st.n_out; p++) {
        const int64_t sa = st.out_stride[a][p], sb = st.out_stride[b][p], so = (int64_t)1 << p;
        if (sa && sb) {
            pa.h_stride[nh] = sa;
            pb.h_stride[nh] = sb;
            ga.h_stride[nh] = so;
            nh++;
        } else if (sa) {
            pa.r_stride[nm] = sa;
            ga.m_stride[nm] = so;
            nm++;
        } else {
            pb.r_stride[nn] = sb;
            ga.n_stride[nn] = so;
            nn++;
        }
    }
    for (int q = 0; q < st.n_sum; q++) {
        pa.k_stride[q] = st.sum_stride[a][q];
        pb.k_stride[q] = st.sum_stride[b][q];
    }
    const int64_t M = (int64_t)1 << nm, N = (int64_t)1 << nn, Kc = (int64_t)1 << st.n_sum;
    const int64_t Kh = ((2 * Kc + kBK - 1) / kBK) * kBK;
    // A cached step (trajectory class, never stacked) runs over the chunk's
    // representatives of its slot: its trajectory-class operands are packed
    // for those instances only and its tiles write their trajectories' outputs.
    const int32_t* cmap = (st.cache > 0 && ctx.cache_list) ? ctx.cache_list + (int64_t)(st.cache - 1) * ctx.cache_n
                                                           : nullptr;
    const int64_t inst_of[3] = {1, cmap ? n_inst : ctx.arena_inst[CLS_TRAJ], ctx.arena_inst[CLS_NET]};
    pa.op = st.op[a];
    pb.op = st.op[b];
    pa.pcls = pack_class(st.op[a], st.out_cls);
    pb.pcls = pack_class(st.op[b], st.out_cls);
    if (st.prod) {
        // the operand st.prod - 1 is prod_src's outer product: bit p of it (stride
        // 2^p) is bit p of prod_src's output, at strides out_stride[0 / 1][p] of
        // the two factors, packed into one word (low / high 32 bits)
        if (!prod_src || st.prod < 1 || st.prod > 2)
            return set_error(PTN_ERR_INVALID_ARG, "internal: outer-product operand without its step");
        PackArgs& px = st.prod - 1 == a ? pa : pb;
        bool ok = true;
        auto packed = [&](int64_t v) -> int64_t {
            if (v <= 0 || (v & (v - 1))) {
                ok = false;
                return 0;
            }
            const int p = __builtin_ctzll((unsigned long long)v);
            if (p >= prod_src->n_out) {
                ok = false;
                return 0;
            }
            return prod_src->out_stride[0][p] | (prod_src->out_stride[1][p] << 32);
        };
        const int n_rb = st.prod - 1 == a ? nm : nn;
        for (int i = 0; i < n_rb; i++) px.r_stride[i] = packed(px.r_stride[i]);
        for (int i = 0; i < nh; i++) px.h_stride[i] = packed(px.h_stride[i]);
        for (int i = 0; i < st.n_sum; i++) px.k_stride[i] = packed(px.k_stride[i]);
        if (!ok) return set_error(PTN_ERR_INVALID_ARG, "internal: outer-product operand with a non-dense stride");
        px.prod = 1;
        px.xconj = st.op[st.prod - 1].conj;
        px.op = prod_src->op[0];
        px.op1 = prod_src->op[1];
    }
    pa.role = 0;
    pb.role = 1;
    pa.n_rb = nm;
    pb.n_rb = nn;
    pa.n_hb = pb.n_hb = nh;
    pa.n_kb = pb.n_kb = st.n_sum;
    pa.Kh = pb.Kh = (int32_t)Kh;
    pa.n_pinst = inst_of[pa.pcls];
    pb.n_pinst = inst_of[pb.pcls];
    pa.inst_map = pa.pcls == CLS_TRAJ ? cmap : nullptr;
    pb.inst_map = pb.pcls == CLS_TRAJ ? cmap : nullptr;
    pa.dst = pack_a;
    pb.dst = pack_b;
    ga.M = (int32_t)M;
    ga.N2 = (int32_t)(2 * N);
    ga.Kh = (int32_t)Kh;
    ga.nkb = (int32_t)(Kh / kBK);
    ga.n_h = 1 << nh;
    ga.a_pcls = pa.pcls;
    ga.b_pcls = pb.pcls;
    ga.out_cls = st.out_cls;
    ga.n_mb = nm;
    ga.n_nb = nn;
    ga.n_hb = nh;
    ga.tiles_m = (M + kBM - 1) / kBM;
    // CTA pairs: at least two segments of 4 k-blocks and 256 columns, more 128 x 128
    // tiles than SMs (fewer finish in one wave, where a pair's tile takes longer),
    // and every M tile has a neighbour or (stacked) the trajectories average at
    // least kPairRows tiles of rows, so that few pairs are half empty
    static const int n_sm = [] {
        int dev = 0, n = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        return n > 0 ? n : 148;
    }();
    const int64_t rows_all = stacked ? n_inst * M : ga.tiles_m * kBM * (n_inst << nh);
    ga.pair = ga.nkb >= kPairKb && 2 * N >= kPairN && rows_all / kBM * (2 * N / kBN) > n_sm &&
              (stacked ? n_inst * M >= kPairRows * kBM * grp.n_groups : ga.tiles_m >= 2);
    ga.bn = ga.pair ? kPairN : kBN;
    ga.tiles_n = (2 * N + ga.bn - 1) / ga.bn;
    while ((1ll << ga.tm_log) < ga.tiles_m) ga.tm_log++;
    while ((1ll << ga.tn_log) < ga.tiles_n) ga.tn_log++;
    ga.n_inst = n_inst;
    ga.net_tl = ctx.net_tl;
    ga.out = ctx.arena[st.out_arena] + st.out_off * ctx.arena_inst[st.out_arena];
    ga.out_size = st.out_size;
    {
        // rows' output strides: a stacked tile's rows above m_bits are networks
        auto row_stride = [&](int i) {
            return i < nm ? ga.m_stride[i] : (stacked ? st.out_size << (i - nm) : (int64_t)0);
        };
        bool direct = true;
        for (int i = 0; i < 5; i++) direct = direct && row_stride(i) == (int64_t)1 << i;
        ga.staged = direct ? 0 : 1;
        struct Bit {
            int64_t out;
            int32_t id;   // 0..4 row bits, 5..7 column bits
        } bit[8];
        for (int i = 0; i < 8; i++) bit[i] = {i < 5 ? row_stride(i) : ga.n_stride[i - 5], i};
        std::sort(bit, bit + 8, [](const Bit& x, const Bit& y) { return x.out < y.out; });
        // place of a fragment's element: the XOR of its bits' words.  The low four
        // bits of a place choose the bank pair; row bits 0..3 (a half-warp's lanes
        // when it writes) and the sorted bits 1..4 (when it reads) both span them:
        // a sorted bit that is not among those row bits shares the bank bit of a row
        // bit that is not among the sorted ones.
        int32_t place[8];
        for (int i = 0; i < 8; i++) place[i] = 1 << i;
        int spare = 0;   // next row bit 0..3 that is not a sorted bit 1..4
        for (int i = 1; i <= 4; i++) {
            if (bit[i].id < 4) continue;
            auto sorted = [&](int r) {
                for (int k = 1; k <= 4; k++)
                    if (bit[k].id == r) return true;
                return false;
            };
            while (sorted(spare)) spare++;
            place[bit[i].id] |= 1 << spare++;
        }
        for (int i = 0; i < 8; i++) {
            ga.frag_out[i] = bit[i].out;
            ga.frag_sm[i] = place[bit[i].id];
            ga.frag_row[i] = bit[i].id < 5 ? 1 << bit[i].id : 0;
        }
        for (int i = 0; i < 5; i++) ga.row_sm[i] = place[i];
        for (int i = 0; i < 3; i++) ga.col_sm[i] = place[5 + i];
        ga.row_hi[0] = row_stride(5);
        ga.row_hi[1] = row_stride(6);
        // every bit above stride 1 is even; so must the instances' bases be
        ga.frag_vec = bit[0].out == 1 && !((st.out_off * ctx.arena_inst[st.out_arena] | st.out_size) & 1);
        if (N < kBN / 2) return set_error(PTN_ERR_INVALID_ARG, "internal: tensor-core step narrower than a tile");
    }
    ga.out_map = cmap;
    ga.err = err;
    ga.wait_ns = g_wait_ns.load(std::memory_order_relaxed);
    const int64_t tot_a = pa.n_pinst * (1ll << nh) * M * (Kh / 2);
    const int64_t tot_b = pb.n_pinst * (1ll << nh) * N * (Kh / 2);
    cudaError_t e;
    if (F == FMT_FP16) {
        // row exponents live after the packed rows (the pack buffers are sized for
        // 4-byte elements plus slack, FP16 rows use half of that)
        auto after = [&](void* base, int64_t rows) {
            const int64_t bytes = rows * 2 * Kh * kEB;
            return reinterpret_cast<int8_t*>(static_cast<uint8_t*>(base) + ((bytes + 255) & ~(int64_t)255));
        };
        pa.row_exp = after(pack_a, pa.n_pinst * (1ll << nh) * M);
        pb.row_exp = after(pack_b, pb.n_pinst * (1ll << nh) * 2 * N);   // B rows are realified pairs
        ga.exp_a = pa.row_exp;
        ga.exp_b = pb.row_exp;
        pa.seg_slots = pb.seg_slots = kSegKb * kBK / 2;
        if (Kh / 2 < 32) return set_error(PTN_ERR_INVALID_ARG, "internal: FP16 rows shorter than a warp");
    }
    {
        // algorithmic bytes: every operand element read once (an outer-product
        // operand: its two factors per instance), the hi/lo rows written once
        auto rd = [&](const PackArgs& pk, int64_t tot) {
            return pk.prod ? 8.0 * (double)pk.n_pinst * (double)(pk.op.inst_size + pk.op1.inst_size)
                           : 8.0 * (double)tot;
        };
        StatScope sc(K_PACK, s, rd(pa, tot_a) + rd(pb, tot_b) + 4.0 * kEB * (double)tot_a + 8.0 * kEB * (double)tot_b,
                     0.0);
        launch_pack<F, 0>(pa, ctx, tot_a, s);
        launch_pack<F, 1>(pb, ctx, tot_b, s);
        count_launches(K_PACK);   // two pack kernels under one scope
    }
    CUtensorMap mA, mB;
    int64_t blocks = ga.tiles_m * ga.tiles_n * n_inst * (1ll << nh);
    ptn_status ps;
    if (!stacked) {
        ps = make_map(&mA, pack_a, dt, kEB, 2 * Kh, M, pa.n_pinst * (1ll << nh), kBM);
    } else {
        // rows of all networks, network-major; groups (trajectories) tile separately.
        // The pack buffer holds at least one full tile of rows (planner), so a
        // chunk with fewer rows still spans the TMA box.
        const int64_t rows = pa.n_pinst * M;
        ps = make_map(&mA, pack_a, dt, kEB, 2 * Kh, rows < kBM ? kBM : rows, 1, kBM);
        ga.stacked = 1;
        ga.m_bits = nm;
        ga.n_groups = grp.n_groups;
        ga.grp_net0 = grp.d_net0;
        ga.grp_tile0 = grp.d_tile0;
        int64_t acc = 0;   // the same count the device tile table ends with
        for (int64_t gi = 0; gi < grp.n_groups; gi++) {
            const int64_t r = (int64_t)(grp.h_net0[gi + 1] - grp.h_net0[gi]) * M;
            acc += (((r + kBM - 1) / kBM + ga.pair) & ~(int64_t)ga.pair) * ga.tiles_n;
        }
        blocks = acc;
        count_launches(K_MISC);
        k_group_tiles<<<(unsigned)((grp.n_groups + 256) / 256), 256, 0, s>>>(grp.d_net0, grp.n_groups, nm,
                                                                              ga.tiles_n, ga.pair, grp.d_cnt);
        launch_exclusive_scan(grp.d_cnt, grp.d_tile0, grp.n_groups + 1, grp.d_scan, s);
    }
    if (ps) return ps;
    ps = make_map(&mB, pack_b, dt, kEB, 2 * Kh, 2 * N, pb.n_pinst * (1ll << nh), kBN);
    if (ps) return ps;
    static std::once_flag done[64];
    once_per_device(done, [] {
        cudaFuncSetAttribute(k_gemm<F, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kGemmSmem);
        cudaFuncSetAttribute(k_gemm<F, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kGemmSmem);
    });
    if (blocks <= 0) return PTN_OK;
    const double flops = 8.0 * (double)n_inst * (double)(1ll << nh) * (double)M * (double)N * (double)Kc;
    const double bytes = 8.0 * ((double)n_inst * (1ll << nh) * M * N) +
                         (double)kEB * 2 * Kh * ((double)pa.n_pinst * M + (double)pb.n_pinst * 2 * N) * (1ll << nh);
    StatScope sc(K_CONTRACT_GEMM, s, bytes, flops);
    ga.n_tiles = blocks;
    t_gemm_forms = (t_gemm_forms ^ (uint64_t)(1 + ga.pair)) * 1099511628211ull;
    const int64_t grid = blocks < n_sm ? blocks : n_sm;
    if (ga.pair) {
        cudaLaunchConfig_t lc{};
        lc.gridDim = dim3((unsigned)(grid & ~(int64_t)1));
        lc.blockDim = dim3(kGemmThreads);
        lc.dynamicSmemBytes = kGemmSmem;
        lc.stream = s;
        cudaLaunchAttribute at{};
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = 2;
        at.val.clusterDim.y = at.val.clusterDim.z = 1;
        lc.attrs = &at;
        lc.numAttrs = 1;
        e = cudaLaunchKernelEx(&lc, k_gemm<F, true>, mA, mB, ga);
        if (e != cudaSuccess) return set_error(PTN_ERR_CUDA, "gemm launch: %s", cudaGetErrorString(e));
    } else {
        k_gemm<F, false><<<(unsigned)grid, kGemmThreads, kGemmSmem, s>>>(mA, mB, ga);
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) return set_error(PTN_ERR_CUDA, "gemm launch: %s", cudaGetErrorString(e));
    return PTN_OK;
}

}  // namespace

void gemm_forms_reset() { t_gemm_forms = 14695981039346656037ull; }
uint64_t gemm_forms() { return t_gemm_forms; }

ptn_status launch_gemm_step(const StepDesc& st, const ChunkCtx& ctx, int64_t n_inst, void* pack_a, void* pack_b,
                            int* err, const GroupTable& grp, int precision,
                            cudaStream_t s, const StepDesc* prod_src) {
    // Contractions of at most 16 complex terms run in TF32 hi/lo in every mode:
    // they fill one 128-byte K-block of TF32 exactly where a 16-bit K-block
    // would be half padding, and their time is the epilogue's (FP16 adds
    // per-row and per-column scales there); TF32 hi/lo is FP32-accurate.
    if (precision != PTN_PREC_FP32 && st.n_sum <= 4 &&
        (precision == PTN_PREC_BF16X3 || precision == PTN_PREC_FP16X3))
        precision = PTN_PREC_FP32;
    switch (precision) {
        case PTN_PREC_FP32: return run_gemm<FMT_TF32>(st, ctx, n_inst, pack_a, pack_b, err, grp, s, prod_src);
        case PTN_PREC_BF16X3: return run_gemm<FMT_BF16>(st, ctx, n_inst, pack_a, pack_b, err, grp, s, prod_src);
        case PTN_PREC_FP16X3: return run_gemm<FMT_FP16>(st, ctx, n_inst, pack_a, pack_b, err, grp, s, prod_src);
    }
    return set_error(PTN_ERR_UNSUPPORTED, "precision mode %d", precision);
}

}  // namespace ptn

extern "C" ptn_status ptn_set_wait_limit(double seconds) {
    if (!(seconds >= 0.0 && seconds <= 60.0))
        return ptn::set_error(PTN_ERR_INVALID_ARG, "wait limit %g s outside 0..60", seconds);
    ptn::g_wait_ns.store((uint64_t)(seconds * 1e9), std::memory_order_relaxed);
    return PTN_OK;
}
