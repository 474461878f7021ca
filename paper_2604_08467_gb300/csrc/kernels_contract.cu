// Batched pairwise contraction of block networks (the execution of one path
// step of P^j for every network of a chunk, Sec. III-A) and the marginal
// finalisation of the block's root tensor (Sec. II-B).
//
// k_contract_direct: each output element of one instance is one thread's
// accumulation; the element's operand addresses come from the step's per-bit
// stride tables, so any bit layout of either operand is read without a
// separate permutation pass.  The first operand read of a merged-gate leaf goes through the
// trajectory's variant index: the UPV merge happens as a gather fused into its
// first consumer.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>

#include "kernels.cuh"
#include "stats.h"

namespace ptn {

namespace {

__device__ __forceinline__ const float2* operand_ptr(const OperandDesc& d, int out_cls, int64_t inst,
                                                     const ChunkCtx& c) {
    int64_t tl = 0, net = 0;
    if (out_cls == CLS_NET) {
        net = inst;
        tl = c.net_tl[inst];
    } else if (out_cls == CLS_TRAJ) {
        tl = inst;
    }
    const float2* p;
    if (d.mode == OP_LEAF) {
        int64_t var = 0;
        if (d.leaf_col >= 0) {
            const int64_t g = c.chunk_traj[tl];
            var = c.var_ids[g * c.n_var_cols + d.leaf_col];
        }
        p = c.vtab + d.leaf_base + var * d.inst_size;
    } else {
        const int64_t oi = d.cls == CLS_CONST ? 0 : (d.cls == CLS_TRAJ ? rep_inst(d, tl, c) : net);
        p = c.arena[d.arena] + d.arena_off * c.arena_inst[d.arena] + oi * d.inst_size;
    }
    if (d.n_slice) {
        const uint64_t* pre = c.net_prefix + net * c.n_words;
        int64_t off = 0;
        for (int s = 0; s < d.n_slice; s++) off += (int64_t)bits_get(pre, d.slice_qubit[s]) * d.slice_stride[s];
        p += off;
    }
    return p;
}

// A warp takes tiles of 128 consecutive outputs (instance-major), four per
// lane (lane, lane + 32, ...): four independent accumulation chains, and each
// store instruction of the warp covers 32 consecutive outputs.  Offsets of the
// low 8 output bits and of the low 8 summed bits come from per-block tables;
// higher summed bits are walked in Gray-code order.  OffT is int32_t when
// every in-instance offset fits (the usual case), halving the address math.
constexpr int kDirThreads = 256;
constexpr int kDirU = 4;
template <typename OffT>
__global__ void __launch_bounds__(kDirThreads, 3) k_contract_direct(const StepDesc* __restrict__ gstep, const __grid_constant__ ChunkCtx c,
                                                                 int64_t n_inst) {
    __shared__ __align__(16) StepDesc s;
    {
        const int4* src = reinterpret_cast<const int4*>(gstep);
        int4* dst = reinterpret_cast<int4*>(&s);
        for (int i = threadIdx.x; i < (int)(sizeof(StepDesc) / sizeof(int4)); i += blockDim.x) dst[i] = src[i];
    }
    __syncthreads();
    __shared__ OffT otab[2][256];
    __shared__ OffT ktab[2][256];
    const int lowb = s.n_out < 8 ? s.n_out : 8;
    const int nk = s.n_sum;
    const int klo = nk < 8 ? nk : 8;
    for (int t = threadIdx.x; t < 256; t += blockDim.x) {
        OffT a = 0, b = 0, ka = 0, kb = 0;
        for (int p = 0; p < lowb; p++)
            if ((t >> p) & 1) {
                a += (OffT)s.out_stride[0][p];
                b += (OffT)s.out_stride[1][p];
            }
        for (int p = 0; p < klo; p++)
            if ((t >> p) & 1) {
                ka += (OffT)s.sum_stride[0][p];
                kb += (OffT)s.sum_stride[1][p];
            }
        otab[0][t] = a;
        otab[1][t] = b;
        ktab[0][t] = ka;
        ktab[1][t] = kb;
    }
    __syncthreads();
    const int64_t total = n_inst << s.n_out;
    const int64_t mask = s.out_size - 1;
    const int lowmask = (1 << lowb) - 1;
    const int n_lo = 1 << klo;
    const int64_t n_hi = (int64_t)1 << (nk - klo);
    const float sa = s.op[0].conj ? -1.f : 1.f, sb = s.op[1].conj ? -1.f : 1.f;
    float2* outbase = c.arena[s.out_arena] + s.out_off * c.arena_inst[s.out_arena];
    const int lane = threadIdx.x & 31;
    const int64_t n_tiles = (total + 32 * kDirU - 1) / (32 * kDirU);
    const int64_t warps = (int64_t)gridDim.x * (kDirThreads / 32);
    // A cached step runs over the chunk's representatives: instance i writes
    // trajectory step_inst(i), odelta = (that - i) << n_out (cached steps have
    // n_out >= 7, so a tile of 128 outputs lies within one instance).
    int64_t cur_inst = -1, cur_hi = -1, odelta = 0;
    OffT hia = 0, hib = 0;
    const float2 *A = nullptr, *B = nullptr;
    for (int64_t tile = (int64_t)blockIdx.x * (kDirThreads / 32) + (threadIdx.x >> 5); tile < n_tiles; tile += warps) {
        const float2* pa[kDirU];
        const float2* pb[kDirU];
        float2 acc[kDirU];
#pragma unroll
        for (int u = 0; u < kDirU; u++) {
            acc[u] = make_float2(0.f, 0.f);
            const int64_t g = tile * (32 * kDirU) + u * 32 + lane;
            const int64_t gg = g < total ? g : total - 1;     // tail lanes compute a valid dummy
            const int64_t inst = gg >> s.n_out;
            const int64_t o = gg & mask;
            if (inst != cur_inst) {
                const int64_t tl = step_inst(s.cache, inst, c);
                odelta = (tl - inst) << s.n_out;
                A = operand_ptr(s.op[0], s.out_cls, tl, c);
                B = operand_ptr(s.op[1], s.out_cls, tl, c);
                cur_inst = inst;
            }
            const int64_t hi = o >> lowb;
            if (hi != cur_hi) {
                hia = hib = 0;
                for (int p = lowb; p < s.n_out; p++)
                    if ((o >> p) & 1) {
                        hia += (OffT)s.out_stride[0][p];
                        hib += (OffT)s.out_stride[1][p];
                    }
                cur_hi = hi;
            }
            pa[u] = A + (hia + otab[0][o & lowmask]);
            pb[u] = B + (hib + otab[1][o & lowmask]);
        }
        OffT ha = 0, hb = 0;
        for (int64_t th = 0; th < n_hi; th++) {
            if (th) {
                const int bit = __ffsll(th) - 1;
                const int64_t gray = th ^ (th >> 1);
                const OffT da = (OffT)s.sum_stride[0][klo + bit], db = (OffT)s.sum_stride[1][klo + bit];
                if ((gray >> bit) & 1) {
                    ha += da;
                    hb += db;
                } else {
                    ha -= da;
                    hb -= db;
                }
            }
            for (int tl = 0; tl < n_lo; tl++) {
                const OffT ka = ha + ktab[0][tl], kb = hb + ktab[1][tl];
#pragma unroll
                for (int u = 0; u < kDirU; u++) {
                    const float2 x = pa[u][ka], y = pb[u][kb];
                    const float xi = sa * x.y, yi = sb * y.y;
                    acc[u].x = fmaf(x.x, y.x, acc[u].x);
                    acc[u].x = fmaf(-xi, yi, acc[u].x);
                    acc[u].y = fmaf(x.x, yi, acc[u].y);
                    acc[u].y = fmaf(xi, y.x, acc[u].y);
                }
            }
        }
#pragma unroll
        for (int u = 0; u < kDirU; u++) {
            const int64_t g = tile * (32 * kDirU) + u * 32 + lane;
            if (g < total) outbase[g + odelta] = acc[u];
        }
    }
}

// Register-tiled variant: a thread computes a 2^RA x 2^RB micro-tile of
// outputs spanned by RA output bits along which only A varies and RB bits
// along which only B varies, so every term loads 2^RA + 2^RB operand values
// for 2^(RA+RB) complex multiply-adds.  The remaining output bits (the tile
// origin) run over the lanes, lowest first.
struct MicroBits {
    int32_t ta[2], tb[2];      // output bits of the micro-tile (A-only, B-only)
    int32_t ins[4];            // the same bits in ascending order (zero insertion)
    int32_t n_ins;
};
template <int RA, int RB>
__global__ void __launch_bounds__(kDirThreads, 2) k_contract_micro(const StepDesc* __restrict__ gstep, const __grid_constant__ ChunkCtx c,
                                                                   int64_t n_inst, const MicroBits mb) {
    __shared__ __align__(16) StepDesc s;
    {
        const int4* src = reinterpret_cast<const int4*>(gstep);
        int4* dst = reinterpret_cast<int4*>(&s);
        for (int i = threadIdx.x; i < (int)(sizeof(StepDesc) / sizeof(int4)); i += blockDim.x) dst[i] = src[i];
    }
    __syncthreads();
    __shared__ int32_t otab[2][256];
    __shared__ int32_t ktab[2][256];
    const int lowb = s.n_out < 8 ? s.n_out : 8;
    const int nk = s.n_sum;
    const int klo = nk < 8 ? nk : 8;
    for (int t = threadIdx.x; t < 256; t += blockDim.x) {
        int32_t a = 0, b = 0, ka = 0, kb = 0;
        for (int p = 0; p < lowb; p++)
            if ((t >> p) & 1) {
                a += (int32_t)s.out_stride[0][p];
                b += (int32_t)s.out_stride[1][p];
            }
        for (int p = 0; p < klo; p++)
            if ((t >> p) & 1) {
                ka += (int32_t)s.sum_stride[0][p];
                kb += (int32_t)s.sum_stride[1][p];
            }
        otab[0][t] = a;
        otab[1][t] = b;
        ktab[0][t] = ka;
        ktab[1][t] = kb;
    }
    __syncthreads();
    constexpr int NA = 1 << RA, NB = 1 << RB;
    int32_t da[NA], db[NB];
    int64_t doa[NA], dob[NB];
#pragma unroll
    for (int i = 0; i < NA; i++) {
        da[i] = 0;
        doa[i] = 0;
#pragma unroll
        for (int j = 0; j < RA; j++)
            if ((i >> j) & 1) {
                da[i] += (int32_t)s.out_stride[0][mb.ta[j]];
                doa[i] += (int64_t)1 << mb.ta[j];
            }
    }
#pragma unroll
    for (int i = 0; i < NB; i++) {
        db[i] = 0;
        dob[i] = 0;
#pragma unroll
        for (int j = 0; j < RB; j++)
            if ((i >> j) & 1) {
                db[i] += (int32_t)s.out_stride[1][mb.tb[j]];
                dob[i] += (int64_t)1 << mb.tb[j];
            }
    }
    const int nq = s.n_out - RA - RB;
    const int64_t total = n_inst << nq;
    const int64_t qmask = ((int64_t)1 << nq) - 1;
    const int lowmask = (1 << lowb) - 1;
    const int n_lo = 1 << klo;
    const int64_t n_hi = (int64_t)1 << (nk - klo);
    const float sa = s.op[0].conj ? -1.f : 1.f, sb = s.op[1].conj ? -1.f : 1.f;
    float2* outbase = c.arena[s.out_arena] + s.out_off * c.arena_inst[s.out_arena];
    int64_t cur_inst = -1, cur_hi = -1, cur_tl = 0;
    int32_t hia = 0, hib = 0;
    const float2 *A = nullptr, *B = nullptr;
    for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < total; g += (int64_t)gridDim.x * blockDim.x) {
        const int64_t inst = g >> nq;
        int64_t o = g & qmask;
        for (int z = 0; z < mb.n_ins; z++) {
            const int cbit = mb.ins[z];
            o = ((o >> cbit) << (cbit + 1)) | (o & (((int64_t)1 << cbit) - 1));
        }
        if (inst != cur_inst) {
            cur_tl = step_inst(s.cache, inst, c);   // a cached step runs over representatives
            A = operand_ptr(s.op[0], s.out_cls, cur_tl, c);
            B = operand_ptr(s.op[1], s.out_cls, cur_tl, c);
            cur_inst = inst;
        }
        const int64_t hi = o >> lowb;
        if (hi != cur_hi) {
            hia = hib = 0;
            for (int p = lowb; p < s.n_out; p++)
                if ((o >> p) & 1) {
                    hia += (int32_t)s.out_stride[0][p];
                    hib += (int32_t)s.out_stride[1][p];
                }
            cur_hi = hi;
        }
        const float2* pa = A + (hia + otab[0][o & lowmask]);
        const float2* pb = B + (hib + otab[1][o & lowmask]);
        float2 acc[NA][NB];
#pragma unroll
        for (int i = 0; i < NA; i++)
#pragma unroll
            for (int j = 0; j < NB; j++) acc[i][j] = make_float2(0.f, 0.f);
        int32_t ha = 0, hb = 0;
        for (int64_t th = 0; th < n_hi; th++) {
            if (th) {
                const int bit = __ffsll(th) - 1;
                const int64_t gray = th ^ (th >> 1);
                const int32_t dka = (int32_t)s.sum_stride[0][klo + bit], dkb = (int32_t)s.sum_stride[1][klo + bit];
                if ((gray >> bit) & 1) {
                    ha += dka;
                    hb += dkb;
                } else {
                    ha -= dka;
                    hb -= dkb;
                }
            }
            for (int tl = 0; tl < n_lo; tl++) {
                const int32_t ka = ha + ktab[0][tl], kb = hb + ktab[1][tl];
                float2 av[NA], bv[NB];
#pragma unroll
                for (int i = 0; i < NA; i++) {
                    av[i] = pa[da[i] + ka];
                    av[i].y *= sa;
                }
#pragma unroll
                for (int j = 0; j < NB; j++) {
                    bv[j] = pb[db[j] + kb];
                    bv[j].y *= sb;
                }
#pragma unroll
                for (int i = 0; i < NA; i++)
#pragma unroll
                    for (int j = 0; j < NB; j++) {
                        acc[i][j].x = fmaf(av[i].x, bv[j].x, acc[i][j].x);
                        acc[i][j].x = fmaf(-av[i].y, bv[j].y, acc[i][j].x);
                        acc[i][j].y = fmaf(av[i].x, bv[j].y, acc[i][j].y);
                        acc[i][j].y = fmaf(av[i].y, bv[j].x, acc[i][j].y);
                    }
            }
        }
        float2* out = outbase + cur_tl * s.out_size + o;
#pragma unroll
        for (int i = 0; i < NA; i++)
#pragma unroll
            for (int j = 0; j < NB; j++) out[doa[i] + dob[j]] = acc[i][j];
    }
}

template <int RA, int RB>
static void launch_micro(const StepDesc* d_step, const ChunkCtx& ctx, int64_t n_inst, const MicroBits& mb,
                         int64_t total_q, cudaStream_t s) {
    int64_t blocks = (total_q + kDirThreads - 1) / kDirThreads;
    if (blocks > 152 * 8) blocks = 152 * 8;
    if (blocks < 1) blocks = 1;
    k_contract_micro<RA, RB><<<(unsigned)blocks, kDirThreads, 0, s>>>(d_step, ctx, n_inst, mb);
}

// SIMT contraction staged in shared memory: the rows a CTA needs, 16 terms at a
// time.  The kernels above let each thread walk its own rows, and neighbouring
// lanes' rows lie a whole row apart: at 64 terms (512 bytes) the lines of all
// resident threads exceed L1 and every 8-byte read fetches a sector again (the
// middle 30-qubit block's network step read at 131 GB/s).  Here a row chunk is copied once by consecutive 16-byte cp.async and
// read back two terms at a time; rows are pitched by one extra 16-byte slot, so
// the eight lanes of a 128-bit shared read hit different banks.  Three stages,
// one barrier per chunk: the copies of the chunk after next are in flight while
// a chunk is contracted.  A CTA takes units (instance, sub-tile of the output)
// with the stride of the grid; the operand addresses of a unit are formed by
// one thread per operand an iteration before its first copy is issued.
// Every output is the multiply-add chain of k_contract_direct: terms in
// increasing order within 256, blocks of 256 in Gray-code order.  Measured
// against the micro-tiles: 1024 terms, 4096 trajectories 5.47 -> 1.81 ms (5.3
// TB/s); 64 terms, 1024 outputs, 10,240 networks 0.65 -> 0.18 ms.
// GATHER: an operand whose summed axis is not contiguous (a mirrored buffer, an
// adjoint step) has no 16-byte pieces; its rows are copied 8 bytes at a time,
// lanes over rows, whose strides are the low ones there.  32 terms, 2^14 outputs,
// 1024 trajectories 0.49 -> 0.166 ms.  A variant of its own: the plain copy loop keeps
// its registers.
constexpr int kRowsMax = 10;          // row bits per operand, sub-tile bits, thread-tile bits
constexpr int kRowsChunk = 16;        // terms per stage
constexpr int kRowsStages = 3;
constexpr int kRowsSmem = 110 * 1024; // stages of one CTA (two per SM)
constexpr int kRowsMinSum = 3;        // shortest summed axis (bits)
constexpr int kGroupLog = 3;          // log2 networks contracted together by k_contract_group
constexpr int64_t kGroupMin = 6;      // least networks per unit on average
struct RowsArgs {
    int32_t rb[2];                     // log2 rows staged per operand
    int32_t r_stride[2][kRowsMax];     // operand stride of each row bit
    int32_t n_sub, n_lane, n_sum, kc_log;
    int32_t k_stride[2][8];            // summed strides of an operand whose summed axis is not contiguous
    int32_t gather[2];                 // that operand: its rows are copied 8 bytes at a time
    int32_t sub_stride[2][kMaxOut];    // sub-tile bits: operand strides, output strides
    int64_t sub_out[kMaxOut];
    int32_t lane_row[2][kRowsMax];     // thread index bits: row weights, output strides
    int32_t lane_out[kRowsMax];
    int32_t tile_row_a[2], tile_row_b[2], tile_out_a[2], tile_out_b[2];   // micro-tile bits
};

__device__ __forceinline__ void cp_async8(uint32_t dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

// two consecutive terms of one output
__device__ __forceinline__ void rows_terms(float2& acc, const float4& a, const float4& b) {
    acc.x = fmaf(a.x, b.x, acc.x);
    acc.x = fmaf(-a.y, b.y, acc.x);
    acc.y = fmaf(a.x, b.y, acc.y);
    acc.y = fmaf(a.y, b.x, acc.y);
    acc.x = fmaf(a.z, b.z, acc.x);
    acc.x = fmaf(-a.w, b.w, acc.x);
    acc.y = fmaf(a.z, b.w, acc.y);
    acc.y = fmaf(a.w, b.z, acc.y);
}

template <int RA, int RB, bool GATHER>
__global__ void __launch_bounds__(256) k_contract_rows(const StepDesc* __restrict__ s, const __grid_constant__ ChunkCtx c,
                                                       const int64_t n_inst, const __grid_constant__ RowsArgs r) {
    extern __shared__ __align__(16) uint8_t rows_smem[];
    constexpr int NA = 1 << RA, NB = 1 << RB;
    const int KC = 1 << r.kc_log, pitch = KC + 2;
    const int rows_a = 1 << r.rb[0], rows = rows_a + (1 << r.rb[1]);
    float2* stage0 = reinterpret_cast<float2*>(rows_smem);
    const int stage_elems = rows * pitch;
    int32_t* row_off = reinterpret_cast<int32_t*>(stage0 + kRowsStages * stage_elems);
    __shared__ const float2* ptr[4][2];    // operand addresses of the units in flight
    __shared__ int64_t out_tl[4];
    for (int i = threadIdx.x; i < rows; i += blockDim.x) {
        const int o = i >= rows_a, v = i - (o ? rows_a : 0);
        int32_t off = 0;
        for (int b = 0; b < r.rb[o]; b++)
            if ((v >> b) & 1) off += r.r_stride[o][b];
        row_off[i] = off;
    }
    const int64_t n_units = n_inst << r.n_sub;
    const int chunks_log = r.n_sum - r.kc_log, n_chunk = 1 << chunks_log;
    const int64_t my_units = n_units > blockIdx.x ? (n_units - blockIdx.x + gridDim.x - 1) / gridDim.x : 0;
    const int64_t n_items = my_units << chunks_log;
    auto set_unit = [&](int64_t u) {       // one thread per operand: addresses of this CTA's u-th unit
        const int o = threadIdx.x >> 5;
        const int64_t unit = blockIdx.x + u * gridDim.x, inst = unit >> r.n_sub;
        const int64_t tl = step_inst(s->cache, inst, c);
        int64_t off = 0;
        for (int b = 0; b < r.n_sub; b++)
            if ((unit >> b) & 1) off += r.sub_stride[o][b];
        ptr[u & 3][o] = operand_ptr(s->op[o], s->out_cls, tl, c) + off;
        if (o == 0) out_tl[u & 3] = tl;
    };
    const bool setter = threadIdx.x == 0 || threadIdx.x == 32;
    // copies of item it (its unit's chunk) into stage it % 3
    const int piece_log = r.kc_log - 1;    // 16-byte pieces per row chunk
    auto issue = [&](int64_t it) {
        if (it < n_items) {
            const int64_t u = it >> chunks_log;
            const int ch = (int)(it & (n_chunk - 1));
            int k0 = ch << r.kc_log;
            if (r.n_sum > 8) {             // blocks of 256 terms in Gray-code order
                const int hi = k0 >> 8;
                k0 = ((hi ^ (hi >> 1)) << 8) | (k0 & 255);
            }
            const uint32_t st = static_cast<uint32_t>(__cvta_generic_to_shared(stage0 + (int)(it % kRowsStages) * stage_elems));
            if constexpr (!GATHER) {
                const float2* pa = ptr[u & 3][0] + k0;
                const float2* pb = ptr[u & 3][1] + k0;
                const int n = rows << piece_log;
                for (int i = threadIdx.x; i < n; i += blockDim.x) {
                    const int row = i >> piece_log, pc = i & ((1 << piece_log) - 1);
                    cp_async16(st + (uint32_t)(row * pitch + 2 * pc) * 8u, (row < rows_a ? pa : pb) + row_off[row] + 2 * pc);
                }
            } else {
                for (int o = 0; o < 2; o++) {
                    const float2* p = ptr[u & 3][o];
                    const int row0 = o ? rows_a : 0, n_rows = 1 << r.rb[o];
                    if (!r.gather[o]) {
                        for (int i = threadIdx.x; i < n_rows << piece_log; i += blockDim.x) {
                            const int row = row0 + (i >> piece_log), pc = i & ((1 << piece_log) - 1);
                            cp_async16(st + (uint32_t)(row * pitch + 2 * pc) * 8u, p + k0 + row_off[row] + 2 * pc);
                        }
                    } else {               // lanes over rows: their strides are the low ones here
                        for (int i = threadIdx.x; i < n_rows << r.kc_log; i += blockDim.x) {
                            const int row = row0 + (i & (n_rows - 1)), k = i >> r.rb[o];
                            int ko = 0;
#pragma unroll
                            for (int b = 0; b < 8; b++)
                                if (b < r.n_sum && (((k0 + k) >> b) & 1)) ko += r.k_stride[o][b];
                            cp_async8(st + (uint32_t)(row * pitch + k) * 8u, p + row_off[row] + ko);
                        }
                    }
                }
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    if (setter)
        for (int64_t u = 0; u < 3 && u < my_units; u++) set_unit(u);
    // this thread's rows and output offset
    const bool act = (int)threadIdx.x < (1 << r.n_lane);
    int ra = 0, rb = 0;
    int64_t o0 = 0;
    for (int b = 0; b < r.n_lane; b++)
        if ((threadIdx.x >> b) & 1) {
            ra += r.lane_row[0][b];
            rb += r.lane_row[1][b];
            o0 += r.lane_out[b];
        }
    int da[NA], db[NB];
#pragma unroll
    for (int i = 0; i < NA; i++) {
        da[i] = 0;
#pragma unroll
        for (int j = 0; j < RA; j++)
            if ((i >> j) & 1) da[i] += r.tile_row_a[j];
        da[i] = (ra + da[i]) * pitch;
    }
#pragma unroll
    for (int i = 0; i < NB; i++) {
        db[i] = 0;
#pragma unroll
        for (int j = 0; j < RB; j++)
            if ((i >> j) & 1) db[i] += r.tile_row_b[j];
        db[i] = (rows_a + rb + db[i]) * pitch;
    }
    const float sa = s->op[0].conj ? -1.f : 1.f, sb = s->op[1].conj ? -1.f : 1.f;
    float2* outbase = c.arena[s->out_arena] + s->out_off * c.arena_inst[s->out_arena];
    const int64_t out_size = s->out_size;
    __syncthreads();
    issue(0);
    issue(1);
    float2 acc[NA][NB];
    for (int64_t it = 0; it < n_items; it++) {
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncthreads();                   // chunk `it` has landed; stage (it + 2) % 3 is free
        issue(it + 2);
        if (setter && ((it + 3) & (n_chunk - 1)) == 0 && it + 3 < n_items && ((it + 3) >> chunks_log) >= 3)
            set_unit((it + 3) >> chunks_log);
        const int64_t u = it >> chunks_log;
        const int ch = (int)(it & (n_chunk - 1));
        if (!act) continue;
        if (ch == 0) {
#pragma unroll
            for (int i = 0; i < NA; i++)
#pragma unroll
                for (int j = 0; j < NB; j++) acc[i][j] = make_float2(0.f, 0.f);
        }
        const float2* st = stage0 + (int)(it % kRowsStages) * stage_elems;
#pragma unroll 2
        for (int k = 0; k < KC; k += 2) {
            float4 av[NA], bv[NB];
#pragma unroll
            for (int i = 0; i < NA; i++) {
                av[i] = *reinterpret_cast<const float4*>(st + da[i] + k);
                av[i].y *= sa;
                av[i].w *= sa;
            }
#pragma unroll
            for (int j = 0; j < NB; j++) {
                bv[j] = *reinterpret_cast<const float4*>(st + db[j] + k);
                bv[j].y *= sb;
                bv[j].w *= sb;
            }
#pragma unroll
            for (int i = 0; i < NA; i++)
#pragma unroll
                for (int j = 0; j < NB; j++) rows_terms(acc[i][j], av[i], bv[j]);
        }
        if (ch == n_chunk - 1) {
            const int64_t unit = blockIdx.x + u * gridDim.x;
            int64_t o = out_tl[u & 3] * out_size + o0;
            for (int b = 0; b < r.n_sub; b++)
                if ((unit >> b) & 1) o += r.sub_out[b];
#pragma unroll
            for (int i = 0; i < NA; i++)
#pragma unroll
                for (int j = 0; j < NB; j++) {
                    int64_t t = o;
#pragma unroll
                    for (int q = 0; q < RA; q++)
                        if ((i >> q) & 1) t += r.tile_out_a[q];
#pragma unroll
                    for (int q = 0; q < RB; q++)
                        if ((j >> q) & 1) t += r.tile_out_b[q];
                    outbase[t] = acc[i][j];
                }
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
}

// Networks of one trajectory whose prefixes agree on the bits an operand is
// sliced by read the same rows of it.  k_contract_group takes units
// (trajectory, slice value, sub-tile): it stages the shared operand's rows
// once, lists the unit's networks, and contracts them 2^g at a time, the other
// operand's rows double-buffered.  The middle 30-qubit block's network step (a
// 64-term vector against 512 shared rows per network) read its rows once per
// network, 7.3 GB through L2 for 28,000 networks: 2.98 ms by the micro-tiles,
// 2.43 ms by k_contract_rows, 0.31 ms here (93.7 -> 9.1 ms in the 10^6-shot job).
// Batches of 8 have to be mostly full: with 5 networks per unit 0.053 ms by
// k_contract_rows became 0.130, with 6.6 it went from 0.115 to 0.053.
constexpr int kGroupWin = 512;         // networks scanned at a time
// stages of one CTA: three per SM, but for 4 x 4 micro-tiles (wide steps), whose 194
// registers leave room for two CTAs of 128 threads or one of 256
constexpr int kGroupSmem = 72 * 1024;
struct GroupArgs {
    RowsArgs r;                        // thread, micro-tile and sub-tile bits; the private operand's row
                                       // index has the network's place in the batch above its own rows
    int32_t shared_op, g_log, ns;      // shared operand; log2 networks per batch; its slice bits
    int32_t seg_log;                   // a trajectory's networks are split into 2^seg_log ranges
    int64_t n_groups;
};

template <int RA, int RB>
__global__ void __launch_bounds__(256) k_contract_group(const StepDesc* __restrict__ s, const __grid_constant__ ChunkCtx c,
                                                        const __grid_constant__ GroupArgs ga) {
    extern __shared__ __align__(16) uint8_t rows_smem[];
    constexpr int NA = 1 << RA, NB = 1 << RB;
    const RowsArgs& r = ga.r;
    const int P = ga.shared_op, Q = 1 - P, K = 1 << r.n_sum, pitch = K + 2, G = 1 << ga.g_log;
    const int rows_p = 1 << r.rb[P], rows_q = 1 << r.rb[Q];
    float2* st_p = reinterpret_cast<float2*>(rows_smem);
    float2* st_q0 = st_p + rows_p * pitch;
    const int q_elems = (rows_q << ga.g_log) * pitch;
    const float2** qptr = reinterpret_cast<const float2**>(st_q0 + 2 * q_elems);   // [kGroupWin]
    int32_t* list = reinterpret_cast<int32_t*>(qptr + kGroupWin);                  // [kGroupWin]
    int32_t* row_off = list + kGroupWin;                                           // [rows_p + rows_q]
    __shared__ int cnt;
    __shared__ const float2* pptr;
    for (int i = threadIdx.x; i < rows_p + rows_q; i += blockDim.x) {
        const int o = i < rows_p ? P : Q, v = i < rows_p ? i : i - rows_p;
        int32_t off = 0;
        for (int b = 0; b < r.rb[o]; b++)
            if ((v >> b) & 1) off += r.r_stride[o][b];
        row_off[i] = off;
    }
    const bool act = (int)threadIdx.x < (1 << r.n_lane);
    int row0[2] = {0, 0};
    int64_t o0 = 0;
    for (int b = 0; b < r.n_lane; b++)
        if ((threadIdx.x >> b) & 1) {
            row0[0] += r.lane_row[0][b];
            row0[1] += r.lane_row[1][b];
            o0 += r.lane_out[b];
        }
    int da[NA], db[NB];
#pragma unroll
    for (int i = 0; i < NA; i++) {
        da[i] = row0[0];
#pragma unroll
        for (int j = 0; j < RA; j++)
            if ((i >> j) & 1) da[i] += r.tile_row_a[j];
    }
#pragma unroll
    for (int i = 0; i < NB; i++) {
        db[i] = row0[1];
#pragma unroll
        for (int j = 0; j < RB; j++)
            if ((i >> j) & 1) db[i] += r.tile_row_b[j];
    }
    const OperandDesc& dp = s->op[P];
    const float sa = s->op[0].conj ? -1.f : 1.f, sb = s->op[1].conj ? -1.f : 1.f;
    float2* outbase = c.arena[s->out_arena] + s->out_off * c.arena_inst[s->out_arena];
    const int64_t out_size = s->out_size;
    const int64_t n_units = ga.n_groups << (r.n_sub + ga.ns + ga.seg_log);
    const int piece_log = r.n_sum - 1;
    for (int64_t unit = blockIdx.x; unit < n_units; unit += gridDim.x) {
        const int sub = (int)(unit & ((1 << r.n_sub) - 1));
        const int var = (int)((unit >> r.n_sub) & ((1 << ga.ns) - 1));
        const int seg = (int)((unit >> (r.n_sub + ga.ns)) & ((1 << ga.seg_log) - 1));
        const int64_t grp = unit >> (r.n_sub + ga.ns + ga.seg_log);
        const int g0 = c.grp_net0[grp], gn = c.grp_net0[grp + 1] - g0;
        const int n0 = g0 + (int)(((int64_t)gn * seg) >> ga.seg_log), n1 = g0 + (int)(((int64_t)gn * (seg + 1)) >> ga.seg_log);
        int64_t sub_off[2] = {0, 0}, sub_out = o0;
        for (int b = 0; b < r.n_sub; b++)
            if ((sub >> b) & 1) {
                sub_off[0] += r.sub_stride[0][b];
                sub_off[1] += r.sub_stride[1][b];
                sub_out += r.sub_out[b];
            }
        bool have_p = false;
        for (int w0 = n0; w0 < n1; w0 += kGroupWin) {
            __syncthreads();   // the previous window's list is no longer read
            if (threadIdx.x == 0) cnt = 0;
            __syncthreads();
            const int w1 = min(w0 + kGroupWin, n1);
            for (int net = w0 + (int)threadIdx.x; net < w1; net += blockDim.x) {
                const uint64_t* pre = c.net_prefix + (int64_t)net * c.n_words;
                int key = 0;
                for (int b = 0; b < ga.ns; b++) key |= (int)bits_get(pre, dp.slice_qubit[b]) << b;
                if (key == var) {
                    const int i = atomicAdd(&cnt, 1);
                    list[i] = net;
                    qptr[i] = operand_ptr(s->op[Q], CLS_NET, net, c) + (Q ? sub_off[1] : sub_off[0]);
                    if (i == 0) pptr = operand_ptr(dp, CLS_NET, net, c) + (P ? sub_off[1] : sub_off[0]);
                }
            }
            __syncthreads();
            const int m = cnt;
            if (m == 0) continue;
            if (!have_p) {
                const uint32_t st = static_cast<uint32_t>(__cvta_generic_to_shared(st_p));
                for (int i = threadIdx.x; i < rows_p << piece_log; i += blockDim.x) {
                    const int row = i >> piece_log, pc = i & ((1 << piece_log) - 1);
                    cp_async16(st + (uint32_t)(row * pitch + 2 * pc) * 8u, pptr + row_off[row] + 2 * pc);
                }
                have_p = true;
            }
            auto issue = [&](int batch) {
                const int left = min(G, m - (batch << ga.g_log));
                if (left > 0) {
                    const uint32_t st = static_cast<uint32_t>(__cvta_generic_to_shared(st_q0 + (batch & 1) * q_elems));
                    const int n = (left * rows_q) << piece_log;
                    for (int i = threadIdx.x; i < n; i += blockDim.x) {
                        const int row = i >> piece_log, pc = i & ((1 << piece_log) - 1);
                        const int net = row >> r.rb[Q], rq = row & (rows_q - 1);
                        cp_async16(st + (uint32_t)(row * pitch + 2 * pc) * 8u,
                                   qptr[(batch << ga.g_log) + net] + row_off[rows_p + rq] + 2 * pc);
                    }
                }
                asm volatile("cp.async.commit_group;" ::: "memory");
            };
            const int n_batch = (m + G - 1) >> ga.g_log;
            issue(0);
            for (int batch = 0; batch < n_batch; batch++) {
                issue(batch + 1);
                asm volatile("cp.async.wait_group 1;" ::: "memory");
                __syncthreads();
                if (act) {
                    const float2* sq = st_q0 + (batch & 1) * q_elems;
                    const float2 *base_a = P == 0 ? st_p : sq, *base_b = P == 0 ? sq : st_p;
                    float2 acc[NA][NB];
#pragma unroll
                    for (int i = 0; i < NA; i++)
#pragma unroll
                        for (int j = 0; j < NB; j++) acc[i][j] = make_float2(0.f, 0.f);
#pragma unroll 2
                    for (int k = 0; k < K; k += 2) {
                        float4 av[NA], bv[NB];
#pragma unroll
                        for (int i = 0; i < NA; i++) {
                            av[i] = *reinterpret_cast<const float4*>(base_a + da[i] * pitch + k);
                            av[i].y *= sa;
                            av[i].w *= sa;
                        }
#pragma unroll
                        for (int j = 0; j < NB; j++) {
                            bv[j] = *reinterpret_cast<const float4*>(base_b + db[j] * pitch + k);
                            bv[j].y *= sb;
                            bv[j].w *= sb;
                        }
#pragma unroll
                        for (int i = 0; i < NA; i++)
#pragma unroll
                            for (int j = 0; j < NB; j++) rows_terms(acc[i][j], av[i], bv[j]);
                    }
#pragma unroll
                    for (int i = 0; i < NA; i++)
#pragma unroll
                        for (int j = 0; j < NB; j++) {
                            const int net = (batch << ga.g_log) + ((Q ? db[j] : da[i]) >> r.rb[Q]);
                            if (net >= m) continue;
                            int64_t t = list[net] * out_size + sub_out;
#pragma unroll
                            for (int q = 0; q < RA; q++)
                                if ((i >> q) & 1) t += r.tile_out_a[q];
#pragma unroll
                            for (int q = 0; q < RB; q++)
                                if ((j >> q) & 1) t += r.tile_out_b[q];
                            outbase[t] = acc[i][j];
                        }
                }
                __syncthreads();   // this batch's stage may be refilled
            }
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
}

// Split of a step for k_contract_rows (shared < 0) or, with operand `shared`
// kept for a group of 2^g_log networks, k_contract_group; false where it does
// not apply: 16-byte misaligned rows, more bits than the tables hold, or (a
// group, or more than 256 terms) a summed axis that is not contiguous.
bool rows_split(const StepDesc& h, const ChunkCtx& ctx, int shared, int g_log, RowsArgs& r, int& ra, int& rb, int& smem) {
    memset(&r, 0, sizeof r);
    if (h.n_sum < kRowsMinSum || h.n_out < 1 || h.out_size >= (1ll << 31)) return false;
    // 64-byte rows with few outputs to share them: 0.051 ms by the micro-tiles
    // against 0.070 here (256 outputs per network, 28,000 networks); with 2048
    // outputs 0.156 against 0.111 ms
    if (h.n_sum == 3 && h.n_out < 9) return false;
    for (int o = 0; o < 2; o++) {
        const OperandDesc& d = h.op[o];
        if (d.inst_size >= (1ll << 31)) return false;
        for (int q = 0; q < h.n_sum; q++)
            if (h.sum_stride[o][q] != (int64_t)1 << q) r.gather[o] = 1;
        if (r.gather[o]) {
            if (shared >= 0 || h.n_sum > 8) return false;
            for (int q = 0; q < h.n_sum; q++) r.k_stride[o][q] = (int32_t)h.sum_stride[o][q];
            continue;
        }
        const int64_t base = d.mode == OP_LEAF ? d.leaf_base : d.arena_off * ctx.arena_inst[d.arena];
        if ((base | d.inst_size) & 1) return false;
        for (int p = 0; p < h.n_out; p++)
            if (h.out_stride[o][p] & 1) return false;
        for (int p = 0; p < d.n_slice; p++)
            if (d.slice_stride[p] & 1) return false;
    }
    // bits by who varies along them: 1 operand 0, 2 operand 1, 3 both; the places
    // of a group's networks are extra bits n_out .. of the private operand alone
    const int n_bits = h.n_out + (shared < 0 ? 0 : g_log), priv = 1 - shared;
    int kind[kMaxOut + 8], rbits[2] = {0, 0};
    bool sub[kMaxOut + 8] = {}, tile[kMaxOut + 8] = {};
    for (int p = 0; p < h.n_out; p++) {
        kind[p] = (h.out_stride[0][p] ? 1 : 0) | (h.out_stride[1][p] ? 2 : 0);
        for (int o = 0; o < 2; o++) rbits[o] += (kind[p] >> o) & 1;
    }
    for (int p = h.n_out; p < n_bits; p++) kind[p] = 1 + priv;
    r.n_sum = h.n_sum;
    r.kc_log = shared >= 0 ? h.n_sum : (h.n_sum < 4 ? h.n_sum : 4);
    const int pitch = (1 << r.kc_log) + 2;
    auto bytes = [&] {
        const int rows = (1 << rbits[0]) + (1 << rbits[1]);
        if (shared < 0) return kRowsStages * rows * pitch * 8 + rows * 4;
        return ((1 << rbits[shared]) + (2 << (rbits[priv] + g_log))) * pitch * 8 + kGroupWin * 12 + rows * 4;
    };
    auto free_bits = [&](int k) {
        int n = 0;
        for (int p = 0; p < n_bits; p++) n += kind[p] == k && !sub[p];
        return n;
    };
    // sub-tiles: highest bits of the operand with more rows, until the stages of
    // two (three) CTAs fit an SM and a 4 x 4 micro-tile leaves at most 256 threads
    const int cap = shared < 0 ? kRowsSmem : kGroupSmem;
    for (;;) {
        int left = 0;
        for (int p = 0; p < n_bits; p++) left += !sub[p];
        const int t = std::min(2, free_bits(1)) + std::min(2, free_bits(2));
        if (rbits[0] <= kRowsMax && rbits[1] <= kRowsMax && bytes() <= cap && left - t <= 8) break;
        int pick = -1;
        const int big = rbits[0] >= rbits[1] ? 1 : 2;
        for (int want : {big, 3, 3 - big}) {
            for (int p = h.n_out - 1; p >= 0 && pick < 0; p--)
                if (!sub[p] && kind[p] == want) pick = p;
            if (pick >= 0) break;
        }
        if (pick < 0) return false;
        sub[pick] = true;
        for (int o = 0; o < 2; o++) rbits[o] -= (kind[pick] >> o) & 1;
        r.sub_stride[0][r.n_sub] = (int32_t)h.out_stride[0][pick];
        r.sub_stride[1][r.n_sub] = (int32_t)h.out_stride[1][pick];
        r.sub_out[r.n_sub++] = (int64_t)1 << pick;
    }
    // micro-tile: the highest one-operand bits (a group's networks first), the
    // operand with fewer tile bits first, while more than 128 threads remain
    int left = n_bits - r.n_sub;
    int tb[2] = {0, 0}, tbit[2][2] = {{-1, -1}, {-1, -1}};
    while (left > 7) {
        int pick = -1;
        for (int o : {tb[0] <= tb[1] ? 0 : 1, tb[0] <= tb[1] ? 1 : 0}) {
            if (tb[o] >= 2) continue;
            for (int p = n_bits - 1; p >= 0 && pick < 0; p--)
                if (!sub[p] && !tile[p] && kind[p] == o + 1) pick = p;
            if (pick >= 0) {
                tbit[o][tb[o]++] = pick;
                break;
            }
        }
        if (pick < 0) break;
        tile[pick] = true;
        left--;
    }
    if (left > 8) return false;
    ra = tb[0];
    rb = tb[1];
    int w[2] = {0, 0};
    for (int p = 0; p < n_bits; p++) {
        if (sub[p]) continue;
        int32_t weight[2] = {0, 0};
        for (int o = 0; o < 2; o++)
            if ((kind[p] >> o) & 1) {
                weight[o] = 1 << w[o];
                if (p < h.n_out) r.r_stride[o][w[o]] = (int32_t)h.out_stride[o][p];
                w[o]++;
            }
        const int32_t out = p < h.n_out ? 1 << p : 0;
        if (tile[p]) {
            const int o = kind[p] - 1, j = tbit[o][0] == p ? 0 : 1;
            (o ? r.tile_row_b : r.tile_row_a)[j] = weight[o];
            (o ? r.tile_out_b : r.tile_out_a)[j] = out;
        } else {
            r.lane_row[0][r.n_lane] = weight[0];
            r.lane_row[1][r.n_lane] = weight[1];
            r.lane_out[r.n_lane++] = out;
        }
    }
    r.rb[0] = rbits[0];
    r.rb[1] = rbits[1];
    smem = bytes();
    return true;
}

template <int RA, int RB>
void launch_rows_t(const StepDesc* d_step, const ChunkCtx& ctx, int64_t n_inst, const GroupArgs& g, int smem,
                   cudaStream_t s) {
    static std::once_flag done[64];
    once_per_device(done, [] {
        cudaFuncSetAttribute(k_contract_rows<RA, RB, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kRowsSmem);
        cudaFuncSetAttribute(k_contract_rows<RA, RB, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kRowsSmem);
        cudaFuncSetAttribute(k_contract_group<RA, RB>, cudaFuncAttributeMaxDynamicSharedMemorySize, kGroupSmem);
    });
    const int threads = std::max(64, 1 << g.r.n_lane);
    const int64_t cap = 152ll * std::max(1, std::min(2048 / threads / 2, 220 * 1024 / (smem + 1024)));
    if (g.n_groups) {
        const int64_t units = g.n_groups << (g.r.n_sub + g.ns + g.seg_log);
        k_contract_group<RA, RB><<<(unsigned)std::min(units, cap), threads, smem, s>>>(d_step, ctx, g);
    } else {
        const int64_t units = n_inst << g.r.n_sub;
        const unsigned grid = (unsigned)std::min(units, cap);
        if (g.r.gather[0] | g.r.gather[1])
            k_contract_rows<RA, RB, true><<<grid, threads, smem, s>>>(d_step, ctx, n_inst, g.r);
        else
            k_contract_rows<RA, RB, false><<<grid, threads, smem, s>>>(d_step, ctx, n_inst, g.r);
    }
}

// Arguments of k_contract_group (n_groups set) or k_contract_rows for a step;
// false where neither applies.
bool choose_rows(const StepDesc& h, const ChunkCtx& ctx, int64_t n_inst, GroupArgs& g, int& ra, int& rb, int& smem) {
    memset(&g, 0, sizeof g);
    // shared operand: a trajectory- or circuit-level buffer, the one with more
    // elements per network; grouped where a unit finds at least kGroupMin
    // networks on average
    if (h.out_cls == CLS_NET && ctx.grp_net0 && h.n_sum <= 8) {
        int p = -1;
        int64_t best = 0;
        for (int o = 0; o < 2; o++) {
            const OperandDesc& d = h.op[o];
            const int64_t elems = d.inst_size >> d.n_slice;
            if (d.mode == OP_BUF && d.cls != CLS_NET && d.n_slice <= 12 && elems > best) {
                best = elems;
                p = o;
            }
        }
        const int64_t groups = ctx.arena_inst[CLS_TRAJ];
        if (p >= 0 && n_inst >= kGroupMin * (groups << h.op[p].n_slice) &&
            rows_split(h, ctx, p, kGroupLog, g.r, ra, rb, smem)) {
            g.shared_op = p;
            g.g_log = kGroupLog;
            g.ns = h.op[p].n_slice;
            g.n_groups = groups;
            // ranges of a trajectory's networks: enough units for every CTA slot,
            // each still with kGroupMin networks
            while ((groups << (g.r.n_sub + g.ns + g.seg_log)) < 152 * 6 &&
                   n_inst >= 2 * kGroupMin * (groups << (g.ns + g.seg_log)))
                g.seg_log++;
            return true;
        }
    }
    return rows_split(h, ctx, -1, 0, g.r, ra, rb, smem);
}
bool launch_rows(const StepDesc* d_step, const StepDesc& h, const ChunkCtx& ctx, int64_t n_inst, cudaStream_t s) {
    GroupArgs g;
    int ra, rb, smem;
    if (!choose_rows(h, ctx, n_inst, g, ra, rb, smem)) return false;
    switch (ra * 3 + rb) {
        case 0: launch_rows_t<0, 0>(d_step, ctx, n_inst, g, smem, s); break;
        case 1: launch_rows_t<0, 1>(d_step, ctx, n_inst, g, smem, s); break;
        case 2: launch_rows_t<0, 2>(d_step, ctx, n_inst, g, smem, s); break;
        case 3: launch_rows_t<1, 0>(d_step, ctx, n_inst, g, smem, s); break;
        case 4: launch_rows_t<1, 1>(d_step, ctx, n_inst, g, smem, s); break;
        case 5: launch_rows_t<1, 2>(d_step, ctx, n_inst, g, smem, s); break;
        case 6: launch_rows_t<2, 0>(d_step, ctx, n_inst, g, smem, s); break;
        case 7: launch_rows_t<2, 1>(d_step, ctx, n_inst, g, smem, s); break;
        default: launch_rows_t<2, 2>(d_step, ctx, n_inst, g, smem, s); break;
    }
    return true;
}

// marg[n][x] = Re(root_n[x]) (the double-layer diagonal), or, where the block
// ends with an elementwise or outer product (the ket-only form's |a(x)|^2, a
// network whose last two parts share no bond), that product's real part formed
// from the factors: the closing step is then not launched and its 8-byte
// outputs are neither written nor read.  Z is the row's FP64 total; with
// rowmax, the largest entry of every row is kept too.
// A CTA takes units of 4096 outcomes (a tile of a wide block, or several
// networks of a narrow one).  The root is read in the order of its memory
// (outcome bits sorted by stride) and turned to outcome order in shared
// memory, so reads and writes are both coalesced; one thread per 16 consecutive
// outcomes read 8 bytes per 64-128 byte step, with 64 of 256 threads busy at
// 2^10 outcomes (1.4 TB/s).  Blocks of 2^10 and of 2^12 outcomes and more hold
// their elements in registers (TB): a warp's part of a row is added as 64-bit
// integers scaled by its largest entry (53 bits for it, the accuracy of adding
// FP64 roundings), because this chip adds two FP64 numbers per clock and SM;
// warps and tiles follow in order in FP64.  The others add 16 consecutive
// outcomes per thread the same way and use a shuffle tree; their form takes 107 to
// 128 registers where the two take 64.  The two run through it would take, per
// entry of 16,384 rows, at 2^10 outcomes 5.8 ps for the root (4.6 here), 6.0 for
// |a|^2 (6.2), 8.5 for an outer product (5.4), at 2^12 5.3 (3.0), 5.4 (4.7) and 8.5
// (4.3); 512 rows of 2^20 as an outer product 5.42 ms (2.21).
// Measured: 1.9 M rows of 2^10 outcomes 15.6 -> 8.4 ms with the closing |a|^2
// (6.3 ms, 24.6 GB) gone; 24 rows of 2^28 outcomes, an outer product, 46.1 ms
// and 13.2 ms for the product -> 18.9 ms.
constexpr int kFinThreads = 256, kFinTileLog = 12, kFinTile = 1 << kFinTileLog;
enum FinMode { FIN_ROOT = 0, FIN_SQUARE = 1, FIN_PRODUCT = 2 };
struct FinArgs {
    int32_t b, tb;                 // outcome bits; those within a unit (the rest number tiles)
    int32_t n_it, net_log;         // elements per thread; log2 networks per unit
    int32_t x_bit[kFinTileLog];    // outcome bit of element bit k
    float s0, s1;                  // signs of the factors' imaginary parts
    int64_t stride[2][kFinTileLog];   // operand strides of the element bits
    int64_t hi_stride[2][32];         // of the outcome bits above tb
    int64_t tiles, n_net, n_units;
};

// 2^s as two FP32 factors and 2^-s in FP64, |s| <= 250
struct FixedScale {
    float f1, f2;
    double inv;
    __device__ __forceinline__ explicit FixedScale(int s) {
        const int s1 = s / 2, s2 = s - s1;
        f1 = __int_as_float((127 + s1) << 23);
        f2 = __int_as_float((127 + s2) << 23);
        inv = __longlong_as_double((int64_t)(1023 - s) << 52);
    }
    __device__ __forceinline__ int64_t operator()(float v) const { return __float2ll_rn(v * f1 * f2); }
};
// Sum of 16 floats of a thread.
__device__ __forceinline__ double sum16(const float* v) {
    float m = 0.f;
    bool fin = true;
    for (int k = 0; k < 16; k++) {
        m = fmaxf(m, fabsf(v[k]));
        fin = fin && fabsf(v[k]) < __int_as_float(0x7f800000);
    }
    double acc = 0.0;
    if (!fin) {                    // infinite entries or NaN
        for (int k = 0; k < 16; k++) acc += (double)v[k];
        return acc;
    }
    if (m == 0.f) return 0.0;
    const FixedScale fs(58 - frexp_exp(m));
    int64_t t = 0;
    for (int k = 0; k < 16; k++) t += fs(v[k]);
    return (double)t * fs.inv;
}
// Sum of N floats per lane over a warp (in lane 0), and the largest entry (m, all lanes).
template <int N>
__device__ __forceinline__ double warp_sum(const float* v, float& m) {
    float a = 0.f;
    m = 0.f;
    bool fin = true;
#pragma unroll
    for (int k = 0; k < N; k++) {
        m = fmaxf(m, v[k]);
        a = fmaxf(a, fabsf(v[k]));
        fin = fin && fabsf(v[k]) < __int_as_float(0x7f800000);
    }
    for (int o = 16; o > 0; o >>= 1) {
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        a = fmaxf(a, __shfl_xor_sync(0xffffffffu, a, o));
    }
    if (!__all_sync(0xffffffffu, fin)) {   // infinite entries or NaN
        double acc = 0.0;
        for (int k = 0; k < N; k++) acc += (double)v[k];
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
        return acc;
    }
    if (a == 0.f) return 0.0;
    const FixedScale fs(53 - frexp_exp(a));
    int64_t t = 0;
#pragma unroll
    for (int k = 0; k < N; k++) t += fs(v[k]);
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    return (double)t * fs.inv;
}

template <int TB, int MODE>        // TB: tb = 10 or 12 with 4096 elements per unit; 0: any other
__global__ void __launch_bounds__(kFinThreads) k_finalize(const OperandDesc* __restrict__ op0, const OperandDesc* __restrict__ op1,
                                                          const __grid_constant__ ChunkCtx c,
                                                          const __grid_constant__ FinArgs f, float* __restrict__ marg,
                                                          double* __restrict__ Z, double* __restrict__ part,
                                                          unsigned* __restrict__ rowmax) {
    constexpr int NOP = MODE == FIN_PRODUCT ? 2 : 1, NV = 16;
    __shared__ float sm[kFinTile + kFinTile / 16];   // outcome x at x + x / 16
    __shared__ const float2* ptr[NOP][TB ? 4 : kFinThreads];
    __shared__ double red[4 * kFinThreads / 32];
    const int tid = threadIdx.x, n_it = TB ? NV : f.n_it, tb = TB ? TB : f.tb;
    // element e = it * 256 + tid: its bits below tb select the outcome in the
    // order of the operands' memory, those above the network of the unit
    int64_t off_t[NOP];
    int x_t = 0;
#pragma unroll
    for (int o = 0; o < NOP; o++) off_t[o] = 0;
    for (int k = 0; k < 8; k++)
        if ((tid >> k) & 1) {
#pragma unroll
            for (int o = 0; o < NOP; o++) off_t[o] += f.stride[o][k];
            x_t += 1 << f.x_bit[k];
        }
    const int64_t nx = (int64_t)1 << f.b;
    for (int64_t u = blockIdx.x; u < f.n_units; u += gridDim.x) {
        const int64_t tile = u % f.tiles, net0 = (u / f.tiles) << f.net_log;
        const int nets = (int)min((int64_t)1 << f.net_log, f.n_net - net0);
        __syncthreads();           // the previous unit's addresses and outcomes are no longer read
        if (tid < nets)
#pragma unroll
            for (int o = 0; o < NOP; o++) {
                const float2* p = operand_ptr(o ? *op1 : *op0, CLS_NET, net0 + tid, c);
                for (int t = tb; t < f.b; t++)
                    if ((tile >> (t - tb)) & 1) p += f.hi_stride[o][t];
                ptr[o][tid] = p;
            }
        __syncthreads();
        const int valid = nets << tb;     // elements of the unit
        // every read of the unit in flight before the first is used
        float v[NV];
#pragma unroll
        for (int it = 0; it < NV; it++) {
            const int e = it * kFinThreads + tid;
            v[it] = 0.f;
            if (it < n_it && e < valid) {
                int64_t off[NOP];
#pragma unroll
                for (int o = 0; o < NOP; o++) {
                    off[o] = off_t[o];
#pragma unroll
                    for (int k = 8; k < kFinTileLog; k++)
                        if ((it >> (k - 8)) & 1) off[o] += f.stride[o][k];
                }
                const float2* p = ptr[0][e >> tb] + off[0];
                if constexpr (MODE == FIN_ROOT) {
                    v[it] = p->x;
                } else {
                    const float2 x = *p;
                    float2 y = x;
                    if constexpr (MODE == FIN_PRODUCT) y = ptr[NOP - 1][e >> tb][off[NOP - 1]];
                    v[it] = fmaf(-(f.s0 * x.y), f.s1 * y.y, fmaf(x.x, y.x, 0.f));   // as the SIMT kernels' single term
                }
            }
        }
#pragma unroll
        for (int it = 0; it < NV; it++) {
            int x = x_t;
#pragma unroll
            for (int k = 8; k < kFinTileLog; k++)
                if ((it >> (k - 8)) & 1) x += 1 << f.x_bit[k];
            if (it < n_it) sm[x + (x >> 4)] = v[it];
        }
        __syncthreads();
        float* out = marg + net0 * nx + (tile << tb);
#pragma unroll
        for (int it = 0; it < NV; it++) {
            const int x = it * kFinThreads + tid;
            if (it < n_it) v[it] = sm[x + (x >> 4)];
            if (it < n_it && x < valid) out[x] = v[it];
        }
        // the totals take the outcomes in their own order, whatever the order of the
        // operands' memory: the same row gives the same total in every plan
        if constexpr (TB != 0) {
            constexpr int PER = 1 << (TB - 8), NETS = NV / PER;   // a thread's elements of a network
#pragma unroll
            for (int g = 0; g < NETS; g++) {
                float m;
                const double t = warp_sum<PER>(v + g * PER, m);
                if ((tid & 31) == 0) {
                    red[g * 8 + (tid >> 5)] = t;
                    if (rowmax && m > 0.f && g < nets) atomicMax(&rowmax[net0 + g], __float_as_uint(m));
                }
            }
            __syncthreads();
            if (tid < nets) {
                double t = 0.0;
                for (int w = 0; w < 8; w++) t += red[tid * 8 + w];
                if (f.tiles == 1) Z[net0 + tid] = t;
                else part[(net0 + tid) * f.tiles + tile] = t;
            }
            continue;
        }
        // narrow blocks: threads past the last network drop out (whole trees of them)
        const unsigned mask = __ballot_sync(0xffffffffu, tb >= 9 || 16 * tid < valid);
        if (tb < 9 && 16 * tid >= valid) continue;
        const float* row = sm + 17 * tid;
        if (tb < 4) {              // several networks per thread
            for (int g = 0; g < 16 >> tb && 16 * tid + (g << tb) < valid; g++) {
                double acc = 0.0;
                float m = 0.f;
                for (int k = 0; k < 1 << tb; k++) {
                    acc += (double)row[(g << tb) + k];
                    m = fmaxf(m, row[(g << tb) + k]);
                }
                const int64_t net = net0 + (((16 * tid) >> tb) + g);
                Z[net] = acc;
                if (rowmax && m > 0.f) rowmax[net] = __float_as_uint(m);
            }
            continue;
        }
        double acc = 0.0;
        float m = 0.f;
        if (16 * tid < valid) {
            float r[16];
#pragma unroll
            for (int k = 0; k < 16; k++) {
                r[k] = row[k];
                m = fmaxf(m, r[k]);
            }
            acc = sum16(r);
        }
        const int per = 1 << (tb - 4);                  // threads per network
        const int64_t net = net0 + tid / per;
        const int width = per < 32 ? per : 32;
        for (int o = width >> 1; o > 0; o >>= 1) {
            acc += __shfl_down_sync(mask, acc, o, width);
            m = fmaxf(m, __shfl_down_sync(mask, m, o, width));
        }
        const bool lead = (tid & (width - 1)) == 0 && 16 * tid < valid;
        if (rowmax && lead && m > 0.f) atomicMax(&rowmax[net], __float_as_uint(m));
        if (per <= 32) {
            if (lead) Z[net] = acc;
            continue;
        }
        if ((tid & 31) == 0) red[tid >> 5] = acc;
        __syncthreads();
        if (tid % per == 0 && 16 * tid < valid) {
            double t = 0.0;
            for (int w = 0; w < per / 32; w++) t += red[(tid >> 5) + w];
            if (f.tiles == 1) Z[net] = t;
            else part[net * f.tiles + tile] = t;
        }
    }
}

// Z[net] = sum of its tiles' partials, in tile order
__global__ void k_finalize_sum(const double* __restrict__ part, int64_t tiles, int64_t n_net, double* __restrict__ Z) {
    const int64_t net = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (net >= n_net) return;
    double t = 0.0;
    for (int64_t k = 0; k < tiles; k++) t += part[net * tiles + k];
    Z[net] = t;
}

// A run of consecutive small trajectory-class steps (the gate-level start of a
// block's path: outputs of at most 2^kSmallOutBits elements from operands of
// at most 2^kSmallOpBits) in one launch, one CTA per trajectory.  The run is
// bound by latency, not by its arithmetic (0.2-0.5 M multiply-adds per
// trajectory), so it is walked level by level of its dataflow
// (small_runs.cpp) with one barrier per level instead of step by step: 19
// barriers for the 731 steps of the first 30-qubit block.  The operand and
// output addresses of all its steps are resolved into shared memory first
// (one dependent chain of table reads for the whole run), and a thread takes
// output elements of any step of the level, whose operand offsets were laid
// out by the host.  A CTA touches only its own trajectory's instances, and the
// planner admits a step into a run only if no other CTA's instances can share
// its output's addresses (small_step, fuse_prev).  Every output is the same
// complex multiply-add chain over the summed bits as in k_contract_direct.
// Measured against the walk with two barriers and a 2.7 KB descriptor per
// step: 689 steps of the last 30-qubit block, 131 trajectories 1.67 -> 0.09 ms;
// 731 steps of the first, 4096 trajectories 8.2 -> 2.6 ms.
// Runs of network-level steps (blocks lowered class by class) go the same way,
// one CTA per network: a 100-qubit block's network, 203 launches 1.24 ms -> 2
// launches and the finalisation 0.13 ms.
struct SmallArgs {
    const SmallStep* steps;
    const SmallEnt* ent;
    const int32_t* lvl;
    const uint32_t* ktab;
    const SmallSlice* slices;
    int32_t n_steps, n_lvl, cls;
};
struct SmallRes {
    const float2 *A, *B;
    float2* out;
    uint32_t loop;
    int32_t ktab;
};

__device__ __forceinline__ const float2* small_operand(const SmallOp& d, int64_t tl, int64_t net,
                                                       const SmallSlice* slices, const ChunkCtx& c) {
    int64_t off = 0;
    if (d.n_slice) {
        const uint64_t* pre = c.net_prefix + net * c.n_words;
        for (int s = 0; s < d.n_slice; s++)
            off += (int64_t)bits_get(pre, slices[d.slice0 + s].qubit) * slices[d.slice0 + s].stride;
    }
    if (d.src < 0) {
        int64_t var = 0;
        if (d.col >= 0) var = c.var_ids[(int64_t)c.chunk_traj[tl] * c.n_var_cols + d.col];
        return c.vtab + d.base + var * d.size + off;
    }
    int64_t oi = d.inst == CLS_NET ? net : 0;
    if (d.inst == CLS_TRAJ)
        oi = (d.cache > 0 && c.cache_rep) ? (int64_t)c.cache_rep[(int64_t)(d.cache - 1) * c.cache_n + tl] : tl;
    return c.arena[d.src] + d.base * c.arena_inst[d.src] + oi * d.size + off;
}

__device__ __forceinline__ void small_term(float2& acc, const float2 x, const float2 y, float sa, float sb) {
    const float xi = sa * x.y, yi = sb * y.y;
    acc.x = fmaf(x.x, y.x, acc.x);
    acc.x = fmaf(-xi, yi, acc.x);
    acc.y = fmaf(x.x, yi, acc.y);
    acc.y = fmaf(xi, y.x, acc.y);
}

__global__ void __launch_bounds__(1024) k_small_steps(const SmallArgs a, const __grid_constant__ ChunkCtx c) {
    extern __shared__ __align__(16) uint8_t small_smem[];
    SmallRes* res = reinterpret_cast<SmallRes*>(small_smem);
    const int64_t inst = blockIdx.x, tl = a.cls == CLS_NET ? (int64_t)c.net_tl[inst] : inst;
    for (int t = threadIdx.x; t < 2 * a.n_steps; t += blockDim.x) {
        const SmallStep& s = a.steps[t >> 1];
        const float2* p = small_operand(s.op[t & 1], tl, inst, a.slices, c);
        SmallRes& r = res[t >> 1];
        if (t & 1) {
            r.B = p;
            r.loop = s.loop;
            r.ktab = s.ktab;
        } else {
            r.A = p;
            r.out = c.arena[s.out_arena] + s.out_off * c.arena_inst[s.out_arena] + inst * s.out_size;
        }
    }
    int e1 = a.lvl[0];
    int i = e1 + (int)threadIdx.x;
    for (int l = 0; l < a.n_lvl; l++) {
        e1 = a.lvl[l + 1];
        SmallEnt e = i < e1 ? a.ent[i] : SmallEnt{0, 0, 0};
        __syncthreads();   // addresses resolved; the previous level's outputs are visible
        while (i < e1) {
            const int nx = i + (int)blockDim.x;
            const SmallEnt en = nx < e1 ? a.ent[nx] : SmallEnt{0, 0, 0};
            const SmallRes r = res[e.step];
            const float2 *A = r.A + (e.offs & 0xffffu), *B = r.B + (e.offs >> 16);
            const float sa = (r.loop & kSmallConjA) ? -1.f : 1.f, sb = (r.loop & kSmallConjB) ? -1.f : 1.f;
            const int nk = (int)(r.loop & 0xffffu);
            float2 acc = make_float2(0.f, 0.f);
            if (r.loop & kSmallDense) {
#pragma unroll 4
                for (int k = 0; k < nk; k++) small_term(acc, A[k], B[k], sa, sb);
            } else {
                const uint32_t* kt = a.ktab + r.ktab;
#pragma unroll 4
                for (int k = 0; k < nk; k++) {
                    const uint32_t ko = kt[k];
                    small_term(acc, A[ko & 0xffffu], B[ko >> 16], sa, sb);
                }
            }
            r.out[e.o] = acc;
            i = nx;
            e = en;
        }
        i = e1 + (int)threadIdx.x;
    }
}

}  // namespace

void launch_small_steps(const SmallRuns& sr, std::pair<int32_t, int32_t> parts, const StepDesc* h_steps, int n_steps,
                        const ChunkCtx& ctx, int64_t n_inst, cudaStream_t s) {
    if (n_steps <= 0 || n_inst <= 0) return;
    double bytes = 0.0, flops = 0.0;
    for (int k = 0; k < n_steps; k++) {
        const StepDesc& h = h_steps[k];
        bytes += 8.0 * (double)n_inst * (double)(h.out_size + h.op[0].inst_size + h.op[1].inst_size);
        flops += 8.0 * (double)n_inst * (double)h.out_size * (double)(1ll << h.n_sum);
    }
    StatScope sc(K_CONTRACT_SMALL, s, bytes, flops);
    // up to one instance per SM: the levels' elements over as many threads as a
    // CTA has (latency); more of them: smaller CTAs, several per SM, so that
    // one's barriers and address chains overlap another's arithmetic.  A
    // network's levels have tens of elements.  Up to three instances per SM stay
    // at the middle size: 372 trajectories 0.393 ms at 256 threads, 0.359 at 512.
    const bool net = h_steps[0].out_cls == CLS_NET;
    const int threads = n_inst <= 152 ? (net ? 512 : 1024) : (n_inst <= 456 ? (net ? 256 : 512) : (net ? 64 : 256));
    for (int p = parts.first; p < parts.second; p++) {
        const SmallPart& pt = sr.parts[p];
        const SmallArgs a{sr.d_steps + pt.step0, sr.d_ent, sr.d_lvl + pt.lvl0, sr.d_ktab, sr.d_slices,
                          pt.n_steps, pt.n_lvl, pt.cls};
        if (p > parts.first) count_launches(K_CONTRACT_SMALL);
        k_small_steps<<<(unsigned)n_inst, threads, sizeof(SmallRes) * pt.n_steps, s>>>(a, ctx);
    }
}

bool staged_step(const StepDesc& h, const ChunkCtx& ctx, int64_t n_inst) {
    GroupArgs g;
    int ra, rb, smem;
    return choose_rows(h, ctx, n_inst, g, ra, rb, smem);
}

void launch_contract_step(const StepDesc* d_step, const StepDesc& h, const ChunkCtx& ctx, int64_t n_inst,
                          cudaStream_t s) {
    const int64_t total = n_inst << h.n_out;
    if (total <= 0) return;
    const int64_t tiles = (total + 32 * kDirU - 1) / (32 * kDirU);
    int64_t blocks = (tiles + kDirThreads / 32 - 1) / (kDirThreads / 32);
    const int64_t cap = 152 * 16;
    if (blocks > cap) blocks = cap;
    // 32-bit in-instance offsets when both operands and the output fit
    const bool off32 = h.op[0].inst_size < (1ll << 31) && h.op[1].inst_size < (1ll << 31) &&
                       h.out_size < (1ll << 31);
    // algorithmic traffic: every distinct operand element once, the output once
    // (a cached step reads the operands of its n_inst representatives only)
    double bytes = 8.0 * (double)total;
    const double n_traj_read = (h.cache > 0 && ctx.cache_list) ? (double)n_inst : (double)ctx.arena_inst[CLS_TRAJ];
    for (int o = 0; o < 2; o++) {
        const OperandDesc& d = h.op[o];
        double inst = d.mode == OP_LEAF ? (d.leaf_col >= 0 ? n_traj_read : 1.0)
                                        : (d.cls == CLS_TRAJ ? n_traj_read : (double)ctx.arena_inst[d.cls]);
        bytes += 8.0 * inst * (double)d.inst_size;
    }
    const double flops = 8.0 * (double)total * (double)(1ll << h.n_sum);
    StatScope sc(K_CONTRACT_DIRECT, s, bytes, flops);
    if (!h.tile && launch_rows(d_step, h, ctx, n_inst, s)) return;
    // micro-tile bits: the highest output bits along which only one operand varies
    MicroBits mb;
    memset(&mb, 0, sizeof mb);
    int ra = 0, rb = 0;
    const int ra_max = h.tile ? (h.tile - 1) / 3 : 2, rb_max = h.tile ? (h.tile - 1) % 3 : 2;
    for (int p = h.n_out - 1; p >= 0; p--) {
        const bool va = h.out_stride[0][p] != 0, vb = h.out_stride[1][p] != 0;
        if (va && !vb && ra < ra_max) mb.ta[ra++] = p;
        else if (vb && !va && rb < rb_max) mb.tb[rb++] = p;
    }
    if (off32 && ra + rb > 0) {
        for (int j = 0; j < ra; j++) mb.ins[mb.n_ins++] = mb.ta[j];
        for (int j = 0; j < rb; j++) mb.ins[mb.n_ins++] = mb.tb[j];
        std::sort(mb.ins, mb.ins + mb.n_ins);
        const int64_t tq = n_inst << (h.n_out - ra - rb);
        switch (ra * 3 + rb) {
            case 1: launch_micro<0, 1>(d_step, ctx, n_inst, mb, tq, s); break;
            case 2: launch_micro<0, 2>(d_step, ctx, n_inst, mb, tq, s); break;
            case 3: launch_micro<1, 0>(d_step, ctx, n_inst, mb, tq, s); break;
            case 4: launch_micro<1, 1>(d_step, ctx, n_inst, mb, tq, s); break;
            case 5: launch_micro<1, 2>(d_step, ctx, n_inst, mb, tq, s); break;
            case 6: launch_micro<2, 0>(d_step, ctx, n_inst, mb, tq, s); break;
            case 7: launch_micro<2, 1>(d_step, ctx, n_inst, mb, tq, s); break;
            default: launch_micro<2, 2>(d_step, ctx, n_inst, mb, tq, s); break;
        }
        return;
    }
    if (off32)
        k_contract_direct<int32_t><<<(unsigned)blocks, kDirThreads, 0, s>>>(d_step, ctx, n_inst);
    else
        k_contract_direct<int64_t><<<(unsigned)blocks, kDirThreads, 0, s>>>(d_step, ctx, n_inst);
}

int64_t finalize_tiles(int b) { return (((int64_t)1 << b) + kFinTile - 1) / kFinTile; }

const StepDesc* closing_product(const BlockPlan& bp) {
    if (bp.steps.empty()) return nullptr;
    const StepDesc& h = bp.steps.back();
    const OperandDesc& r = bp.root.op;
    if (h.kind != STEP_DIRECT || h.n_sum != 0 || h.virt || h.fuse_prev || bp.b != h.n_out || h.n_out > 30) return nullptr;
    if (r.mode != OP_BUF || r.n_slice || r.arena != h.out_arena || r.arena_off != h.out_off || r.inst_size != h.out_size)
        return nullptr;
    for (int t = 0; t < bp.b; t++) {
        const int64_t v = bp.root.x_stride[t];
        if (v <= 0 || (v & (v - 1)) || v >= h.out_size) return nullptr;
    }
    return &h;
}

void launch_finalize(const RootRef* d_root, const RootRef& root, const StepDesc* d_prod, const StepDesc* prod,
                     const ChunkCtx& ctx, int b, int64_t n_net, float* marg, double* Z, double* part, unsigned* rowmax,
                     cudaStream_t s) {
    if (n_net <= 0) return;
    FinArgs f;
    memset(&f, 0, sizeof f);
    f.b = b;
    f.tb = std::min(b, kFinTileLog);
    f.net_log = std::min(kFinTileLog - f.tb, 8);
    f.n_it = std::max(1, 1 << (f.tb + f.net_log) >> 8);
    f.n_net = n_net;
    f.tiles = finalize_tiles(b);
    f.n_units = ((n_net + (1ll << f.net_log) - 1) >> f.net_log) * f.tiles;
    f.s0 = f.s1 = 1.f;
    int mode = FIN_ROOT;
    const OperandDesc *op0 = &d_root->op, *op1 = op0;
    if (prod) {
        const OperandDesc &p = prod->op[0], &q = prod->op[1];
        bool same = p.mode == OP_BUF && q.mode == OP_BUF && !p.n_slice && !q.n_slice && p.arena == q.arena &&
                    p.cls == q.cls && p.arena_off == q.arena_off && p.inst_size == q.inst_size && p.cache == q.cache;
        for (int t = 0; t < prod->n_out; t++) same = same && prod->out_stride[0][t] == prod->out_stride[1][t];
        mode = same ? FIN_SQUARE : FIN_PRODUCT;
        op0 = &d_prod->op[0];
        op1 = &d_prod->op[1];
        f.s0 = p.conj ? -1.f : 1.f;
        f.s1 = q.conj ? -1.f : 1.f;
    }
    // stride of outcome bit t in the root, or in a factor of the closing product
    auto stride = [&](int o, int t) {
        const int64_t v = root.x_stride[t];
        return prod ? prod->out_stride[o][__builtin_ctzll((unsigned long long)v)] : v;
    };
    // element order: along the larger operand's memory, then the other's bits
    const int big = mode == FIN_PRODUCT && prod->op[1].inst_size >> prod->op[1].n_slice > prod->op[0].inst_size >> prod->op[0].n_slice;
    int order[kFinTileLog];
    for (int t = 0; t < f.tb; t++) order[t] = t;
    auto key = [&](int t) {
        const int64_t v = stride(big, t);
        return v ? v : ((int64_t)1 << 40) + stride(1 - big, t);
    };
    std::sort(order, order + f.tb, [&](int x, int y) { return key(x) < key(y); });
    for (int k = f.tb; k < kFinTileLog; k++) f.x_bit[k] = k;   // network bits: no stride
    for (int k = 0; k < f.tb; k++) {
        f.x_bit[k] = order[k];
        for (int o = 0; o < 2; o++) f.stride[o][k] = stride(o, order[k]);
    }
    for (int t = f.tb; t < b; t++)
        for (int o = 0; o < 2; o++) f.hi_stride[o][t] = stride(o, t);
    StatScope sc(K_FINALIZE, s, (double)n_net * (double)(1ll << b) * (mode == FIN_PRODUCT ? 4.0 : 12.0), 0.0);
    const unsigned grid = (unsigned)std::min<int64_t>(f.n_units, 152 * 8);
    auto run = [&](auto kernel) { kernel<<<grid, kFinThreads, 0, s>>>(op0, op1, ctx, f, marg, Z, part, rowmax); };
    if (f.tb == 12) {
        if (mode == FIN_ROOT) run(k_finalize<12, FIN_ROOT>);
        else if (mode == FIN_SQUARE) run(k_finalize<12, FIN_SQUARE>);
        else run(k_finalize<12, FIN_PRODUCT>);
    } else if (f.tb == 10) {
        if (mode == FIN_ROOT) run(k_finalize<10, FIN_ROOT>);
        else if (mode == FIN_SQUARE) run(k_finalize<10, FIN_SQUARE>);
        else run(k_finalize<10, FIN_PRODUCT>);
    } else {
        if (mode == FIN_ROOT) run(k_finalize<0, FIN_ROOT>);
        else if (mode == FIN_SQUARE) run(k_finalize<0, FIN_SQUARE>);
        else run(k_finalize<0, FIN_PRODUCT>);
    }
    if (f.tiles > 1) count_launches(K_FINALIZE);
    if (f.tiles > 1) k_finalize_sum<<<(unsigned)((n_net + 127) / 128), 128, 0, s>>>(part, f.tiles, n_net, Z);
}

}  // namespace ptn
