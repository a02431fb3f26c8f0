// Tensor-core (tcgen05) variant of the substitution products for complex64 factors.
//
// A work item computes 128 complex output rows (four factor tile rows) x NT = 32, 64 or 128
// right-hand-side columns of one of the four node products of the substitution (see solve.cu), for the nodes
// whose products are large enough to fill it; smaller nodes of the same tree level run on the
// CUDA-core kernel in the same phase.
//
// The complex product Y = A X is four real products with two accumulators in tensor memory:
//     Yr = Ar Xr - Ai Xi,    Yi = Ai Xr + Ar Xi,
// (the minus sign through the instruction descriptor's negate-A bit).  Each real product runs
// in TF32 with a three-term split of both operands (a = a_hi + a_lo, x = x_hi + x_lo;
// a x ~ a_hi x_hi + a_hi x_lo + a_lo x_hi) and FP32 accumulation, which keeps every product at
// FP32-level accuracy (about 2^-21 relative): 12 MMAs (M = 128, N = NT, K = 8) per 8 complex
// reduction indices.  SPLIT = 1 keeps only a_hi x_hi (plain TF32, about 2^-11 relative; 4 MMAs);
// it is an option (HZ_PRECOND_SPLIT=1) for the local solves inside the preconditioner, whose
// accuracy changes how fast GMRES converges but not the solution it converges to.
//
// Warp-specialized pipeline (16 complex reduction indices per stage, rings of two to six raw and two or
// four converted buffers, every hand-off an mbarrier):
//   4 loader warps    : cp.async 16-byte copies of the factor tiles and vector rows into a raw
//                       buffer (masked rows / absent tiles zero-filled by the copy), completion
//                       signalled with cp.async.mbarrier.arrive;
//   8 converter warps : raw -> split hi/lo TF32 operands in the K-major core-matrix layout
//                       (no swizzle), 16-byte stores, or the factor's in tensor memory;
//   1 MMA warp        : one thread issues the MMAs of a stage and commits them to the mbarrier
//                       that releases the converted buffer.
// Two kernels share these stages:
//   k_subst_tc  (one block per work item, 416 threads): after the last MMA the converter warps
//               stage the accumulators through shared memory and write whole rows;
//   k_subst_tcp (persistent, one block per SM, 544 threads): the block walks the launch's work
//               items with stride gridDim.x; the rings run on across items, the accumulators
//               alternate between two TMEM buffers, and 4 epilogue warps drain item i while the
//               MMA warp accumulates item i+1, so block start-up, pipeline fill and epilogue are
//               paid once per SM instead of once per item.
// Output rule of both: an item that covers the full reduction of its rows stores them; split
// reductions and the updates (FB, BA) accumulate with vector atomics.  Every mbarrier
// wait is bounded (polls and wall time); a wait that gives up raises an abort flag in shared
// memory that ends the block's other waits; the block then records an error flag, waits
// (bounded) for its own MMAs, frees its tensor memory and exits.
#include <algorithm>

#include "hz_internal.cuh"
#include "hz_ctx.cuh"
#include "hz_solve.cuh"
#include "tc_common.cuh"
#include "subst_items.cuh"

namespace hz {

namespace {

using namespace tcc;

// Sizes of one ring stage for NT columns.  NT <= 64 runs the wide form of the MMAs (the output's
// two halves side by side, three vector blocks per term); NT = 128 would need 6 x 8 KB of vector
// operands per stage, which does not fit beside a two-deep raw ring, and fills N = 128 as it is.
// The room that narrow tiles leave goes to the raw ring: the factor stream, 16 KB per stage
// whatever NT is, binds them, and every further stage in flight covers memory latency.
// Measured: a 32-column block of a 128^3 layer 3.10 ms on the CUDA cores, 1.68 in the wide form; 64
// columns, 64^3, 8 layers: 3.98 ms with N = 64 MMAs on a two-deep ring, 2.80 in the wide form.
template <int NT> struct Ring {
    static constexpr bool WIDE = NT <= 64;
    static constexpr int A_MAT = MR * KC * 4;            // one real operand matrix (8 KB)
    static constexpr int X_MAT = NT * KC * 4;
    // Ar_h Ar_l Ai_h Ai_l, then Xr_h Xr_l Xi_h Xi_l, or (WIDE) -Xi_h Xr_h Xi_h -Xi_l Xr_l Xi_l
    static constexpr int CONV = 4 * A_MAT + (WIDE ? 6 : 4) * X_MAT;
    static constexpr int RAW_A = 4 * 32 * TROW;          // large enough for both raw tile layouts
    static constexpr int RAW_X = KC * NT * 8;
    static constexpr int RAW = RAW_A + RAW_X;
    static constexpr int RD = NT == 32 ? 4 : (NT == 64 ? 3 : 2);   // raw ring depth
    static constexpr int BYTES = 2 * CONV + RD * RAW;    // converted operands: two-deep
};

// Columns of one accumulator set: real and imaginary part, and (SEP) the hi x lo terms' own.
template <int NT, int SPLIT, bool SEP> constexpr int acc_cols = (SEP && SPLIT == 3) ? 4 * NT : 2 * NT;

template <int NT, int SPLIT, bool SEP, bool TA>
__device__ __forceinline__ void mma_item_stage(uint32_t conv, uint32_t tm, bool first, uint32_t ta) {
    static_assert(Ring<NT>::WIDE || !TA, "the factor operand is in tensor memory in the wide form only");
    if constexpr (Ring<NT>::WIDE) mma_stage_wide<NT, SPLIT, SEP, TA>(conv, tm, first, ta);
    else mma_stage<NT, SPLIT, SEP>(conv, tm, tm + NT, first);
}

// 16 accumulator columns from c0 on of this warp's lanes, the terms added up.
template <int NT, int SPLIT, bool SEP>
__device__ __forceinline__ void read_acc(uint32_t tm, int c0, uint32_t (&vr)[16], uint32_t (&vi)[16]) {
    tmem_ld16(tm + (uint32_t)c0, tm + (uint32_t)(NT + c0), vr, vi);
    if constexpr (SEP && SPLIT == 3) {
        uint32_t lr[16], li[16];
        tmem_ld16(tm + (uint32_t)(2 * NT + c0), tm + (uint32_t)(3 * NT + c0), lr, li);
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            vr[j] = __float_as_uint(__uint_as_float(vr[j]) + __uint_as_float(lr[j]));
            vi[j] = __float_as_uint(__uint_as_float(vi[j]) + __uint_as_float(li[j]));
        }
    }
}

// Loader part of stage s of an item: the four factor tiles' 16-column halves and 16 vector rows.
template <int NT, int MODE>
__device__ inline void load_stage(unsigned char* rb, const Item& it, TilePtrs<MODE>& tp, int s, int ldc, int t,
                                  const Vrows<NT>& vr) {
    using RG = Ring<NT>;
    constexpr bool TR = (MODE == BA || MODE == BB);  // factor tiles used transposed
    const int hk = s & 1;
    const uint32_t dst = smem_u32(rb) + (TR ? (t >> 3) * TROW + (t & 7) * 16 : t * 16);
#pragma unroll
    for (int oi = 0; oi < 4; ++oi) {   // factor tiles: 1024 chunks of 16 bytes
        const bool ex = tp.exists(oi);
        const char* src = ex ? tp.p[oi] + hk * (TR ? KC * 8 : KC * 32 * 8) : (const char*)it.jb.fac;
        const int n = ex ? 16 : 0;
        constexpr int DT = TR ? 32 * TROW : 4096;
        cp16(dst + oi * DT, src, n);
        cp16(dst + oi * DT + (TR ? 16 * TROW : 2048), ex ? src + (TR ? 16 * 256 : 2048) : src, n);
    }
    if (hk) tp.next();
    const float2* vec = MODE == BB ? it.jb.x : it.jb.acc;
#pragma unroll
    for (int i = 0; i < KC * NT / 2 / NLOAD; ++i) {  // vector rows: KC x NT, raw [k][n]
        const int c = t + NLOAD * i;
        const int k = c / (NT / 2), j = c % (NT / 2);
        const bool v = vr.r[i] >= 0;
        const long long row = v ? vr.r[i] : 0;
        cp16(smem_u32(rb + RG::RAW_A + k * NT * 8 + j * 16), vec + row * ldc + it.col0 + 2 * j, v ? 16 : 0);
    }
}

// Converter part of a stage: raw -> hi (and lo) TF32 operands, the vectors in shared memory, the factor
// there or (TA) in tensor memory from column ta on: converter warp w writes the 32 lanes (rows) of tile
// w % 4 that its place in the block gives it access to, 8 of the 16 columns of each matrix.
// The stage is NTHR threads' work.
template <int NT, int MODE, int SPLIT, bool TA, int NTHR>
__device__ inline void convert_stage(const unsigned char* rb, unsigned char* cv, int ct, uint32_t ta) {
    using RG = Ring<NT>;
    constexpr bool TR = (MODE == BA || MODE == BB);
    if constexpr (TA) {
        static_assert(NLOAD % 128 == 0 && NTHR == 128, "converter warp w must have warp index 4 n + w");
        const int oi = ct >> 5, r = ct & 31;
#pragma unroll
        for (int kh = 0; kh < 2; ++kh) {
            float re[8], im[8];
            if (!TR) {
                const float2* src = (const float2*)(rb + oi * 4096) + 8 * kh * 32 + r;
#pragma unroll
                for (int j = 0; j < 8; ++j) { const float2 a = src[j * 32]; re[j] = a.x; im[j] = a.y; }
            } else {
                const float4* src = (const float4*)(rb + oi * 32 * TROW + r * TROW + kh * 64);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float4 a = src[j];
                    re[2 * j] = a.x; im[2 * j] = a.y; re[2 * j + 1] = a.z; im[2 * j + 1] = a.w;
                }
            }
            float hi[8];
            const uint32_t col = ta + ((uint32_t)(32 * oi) << 16) + 8 * kh;
#pragma unroll
            for (int j = 0; j < 8; ++j) { hi[j] = tf32_hi<SPLIT>(re[j]); re[j] -= hi[j]; }
            tmem_st8(col, hi);
            if (SPLIT == 3) tmem_st8(col + KC, re);
#pragma unroll
            for (int j = 0; j < 8; ++j) { hi[j] = tf32_hi<SPLIT>(im[j]); im[j] -= hi[j]; }
            tmem_st8(col + 2 * KC, hi);
            if (SPLIT == 3) tmem_st8(col + 3 * KC, im);
        }
    }
    for (int id = ct; !TA && id < MR * 4; id += NTHR) {   // factor operand: 128 rows x 16 k, (row, 4 consecutive k)
        const int row = id & 127, kq = id >> 7;
        const int oi = row >> 5, r = row & 31;
        float re[4], im[4];
        if (!TR) {
            const float2* src = (const float2*)(rb + oi * 4096);
#pragma unroll
            for (int j = 0; j < 4; ++j) { float2 a = src[(4 * kq + j) * 32 + r]; re[j] = a.x; im[j] = a.y; }
        } else {
            const float4* src = (const float4*)(rb + oi * 32 * TROW + r * TROW + kq * 32);
            float4 a0 = src[0], a1 = src[1];
            re[0] = a0.x; im[0] = a0.y; re[1] = a0.z; im[1] = a0.w;
            re[2] = a1.x; im[2] = a1.y; re[3] = a1.z; im[3] = a1.w;
        }
        float4 rh, ih;
        rh.x = tf32_hi<SPLIT>(re[0]); rh.y = tf32_hi<SPLIT>(re[1]); rh.z = tf32_hi<SPLIT>(re[2]); rh.w = tf32_hi<SPLIT>(re[3]);
        ih.x = tf32_hi<SPLIT>(im[0]); ih.y = tf32_hi<SPLIT>(im[1]); ih.z = tf32_hi<SPLIT>(im[2]); ih.w = tf32_hi<SPLIT>(im[3]);
        const int off = coff(row, 4 * kq);
        *(float4*)(cv + 0 * RG::A_MAT + off) = rh;
        *(float4*)(cv + 2 * RG::A_MAT + off) = ih;
        if (SPLIT == 3) {
            *(float4*)(cv + 1 * RG::A_MAT + off) = make_float4(re[0] - rh.x, re[1] - rh.y, re[2] - rh.z, re[3] - rh.w);
            *(float4*)(cv + 3 * RG::A_MAT + off) = make_float4(im[0] - ih.x, im[1] - ih.y, im[2] - ih.z, im[3] - ih.w);
        }
    }
    for (int id = ct; id < NT * 4; id += NTHR) {   // vector operand: NT rows x 16 k
        const int n = id % NT, kq = id / NT;
        const float2* src = (const float2*)(rb + RG::RAW_A);
        float re[4], im[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) { float2 a = src[(4 * kq + j) * NT + n]; re[j] = a.x; im[j] = a.y; }
        float4 rh, ih;
        rh.x = tf32_hi<SPLIT>(re[0]); rh.y = tf32_hi<SPLIT>(re[1]); rh.z = tf32_hi<SPLIT>(re[2]); rh.w = tf32_hi<SPLIT>(re[3]);
        ih.x = tf32_hi<SPLIT>(im[0]); ih.y = tf32_hi<SPLIT>(im[1]); ih.z = tf32_hi<SPLIT>(im[2]); ih.w = tf32_hi<SPLIT>(im[3]);
        const int off = (TA ? 0 : 4 * RG::A_MAT) + coff(n, 4 * kq);
        const float4 rl = make_float4(re[0] - rh.x, re[1] - rh.y, re[2] - rh.z, re[3] - rh.w);
        const float4 il = make_float4(im[0] - ih.x, im[1] - ih.y, im[2] - ih.z, im[3] - ih.w);
        if (RG::WIDE) {
            *(float4*)(cv + off + 0 * RG::X_MAT) = make_float4(-ih.x, -ih.y, -ih.z, -ih.w);
            *(float4*)(cv + off + 1 * RG::X_MAT) = rh;
            *(float4*)(cv + off + 2 * RG::X_MAT) = ih;
            if (SPLIT == 3) {
                *(float4*)(cv + off + 3 * RG::X_MAT) = make_float4(-il.x, -il.y, -il.z, -il.w);
                *(float4*)(cv + off + 4 * RG::X_MAT) = rl;
                *(float4*)(cv + off + 5 * RG::X_MAT) = il;
            }
        } else {
            *(float4*)(cv + off + 0 * RG::X_MAT) = rh;
            *(float4*)(cv + off + 2 * RG::X_MAT) = ih;
            if (SPLIT == 3) {
                *(float4*)(cv + off + 1 * RG::X_MAT) = rl;
                *(float4*)(cv + off + 3 * RG::X_MAT) = il;
            }
        }
    }
    if constexpr (TA) {
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    }
}

// Writes one 16-byte column pair y of an output row (global offset base + c) by the output rule;
// d is the row's D^{-1} (FA).
template <int MODE>
__device__ inline void write_pair(const Item& it, long long base, int c, float4 y, float2 d) {
    if (MODE == FB || MODE == BA) {
        atomicAdd((float4*)(it.jb.acc + base + c), make_float4(-y.x, -y.y, -y.z, -y.w));
    } else {
        if (MODE == FA)
            y = make_float4(d.x * y.x - d.y * y.y, d.x * y.y + d.y * y.x, d.x * y.z - d.y * y.w, d.x * y.w + d.y * y.z);
        float4* dst = (float4*)((MODE == FA ? it.jb.x : it.jb.acc) + base + c);
        if (it.unique) *dst = y;
        else atomicAdd(dst, y);
    }
}

// ------------------------------------------------------------------------------------------
// k_subst_tc: one block per work item
// ------------------------------------------------------------------------------------------
template <int NT> struct OneLayout {
    using RG = Ring<NT>;
    static constexpr int NTHREADS = NLOAD + NCONV + 32;
    static constexpr int HALF = NT >= 64 ? NT / 2 : NT;  // output columns staged per epilogue pass
    static constexpr int SP = HALF + 2;                  // staging pitch (complex): 16-byte rows, odd in 16 B
    static_assert(MR * SP * 8 <= RG::BYTES, "staging tile must fit in the ring buffers");
    static constexpr int ROWS_OFF = RG::BYTES;           // long long rowbase[128], float2 dinv[128]
    static constexpr int BAR_OFF = ROWS_OFF + MR * 8 + MR * 8;
    static constexpr int TOTAL = BAR_OFF + (2 * RG::RD + 4) * 8 + 16;
};

template <int NT, int MODE, int SPLIT>
__global__ void __launch_bounds__(OneLayout<NT>::NTHREADS, 1)
k_subst_tc(const Task* __restrict__ tasks, const JobDev<float2>* __restrict__ jobs, int ldc, int nchunks,
           int* flag, long long polls) {
    using RG = Ring<NT>;
    using LY = OneLayout<NT>;
    extern __shared__ __align__(1024) unsigned char smem[];
    unsigned char* conv = smem;                  // [2][CONV]
    unsigned char* raw = smem + 2 * RG::CONV;    // [RD][RAW]
    constexpr int RD = RG::RD;
    constexpr int TCOLS = acc_cols<NT, SPLIT, true>;
    long long* rowbase = (long long*)(smem + LY::ROWS_OFF);
    float2* dinv_s = (float2*)(smem + LY::ROWS_OFF + MR * 8);
    uint64_t* raw_full = (uint64_t*)(smem + LY::BAR_OFF);   // [RD] loaders' copies landed (count NLOAD)
    uint64_t* raw_empty = raw_full + RD;   // [RD] converters done reading (count NCONV)
    uint64_t* conv_full = raw_empty + RD;  // [2] converted operands written (count NCONV)
    uint64_t* conv_empty = conv_full + 2;  // [2] MMAs of the buffer done (tcgen05.commit)
    uint32_t* tptr = (uint32_t*)(conv_empty + 2);
    volatile int* abort = (volatile int*)tptr + 1;
    volatile int* committed = (volatile int*)tptr + 2;   // stages whose MMAs were committed

    const Item it = decode<NT, MODE>(tasks, jobs, blockIdx.x, nchunks);
    const int t = threadIdx.x, w = t >> 5, l = t & 31;
    const int nst = it.nst;
    const int mma_warp = (NLOAD + NCONV) / 32;

    if (w == mma_warp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" :: "r"(smem_u32(tptr)), "r"(TCOLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (t == 0) {
        for (int b = 0; b < RD; ++b) {
            mbar_init(raw_full + b, NLOAD);
            mbar_init(raw_empty + b, NCONV);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(conv_full + b, NCONV);
            mbar_init(conv_empty + b, 1);
        }
        *abort = 0;
        *committed = 0;
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tptr;
    bool ok = true;

    if (t < NLOAD) {
        Vrows<NT> rows = stage_rows<NT, MODE>(it, 0, t);
        TilePtrs<MODE> tp;
        tp.init(it, t);
        for (int s = 0; s < nst && ok; ++s) {
            const int slot = s % RD, use = s / RD;
            const Vrows<NT> next = stage_rows<NT, MODE>(it, s + 1, t);   // looked up ahead
            if (s >= RD) ok = mbar_wait(smem_u32(raw_empty + slot), (uint32_t)((use - 1) & 1), abort, polls);
            if (!ok) break;
            load_stage<NT, MODE>(raw + slot * RG::RAW, it, tp, s, ldc, t, rows);
            cp_async_arrive(raw_full + slot);
            rows = next;
        }
        // row descriptors of the epilogue, fetched while the pipeline drains
        for (int r = t; r < MR; r += NLOAD) {
            const long long base = row_base<MODE>(it, r, ldc);
            rowbase[r] = base;
            if (MODE == FA) dinv_s[r] = base >= 0 ? it.jb.dinv[it.nd.own0 + it.o0 * TILE + r] : make_float2(0.f, 0.f);
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
    } else if (t < NLOAD + NCONV) {
        const int ct = t - NLOAD;
        for (int s = 0; s < nst && ok; ++s) {
            const int slot = s % RD, use = s / RD, cb = s & 1, cuse = s >> 1;
            ok = mbar_wait(smem_u32(raw_full + slot), (uint32_t)(use & 1), abort, polls);
            if (ok && s >= 2) ok = mbar_wait(smem_u32(conv_empty + cb), (uint32_t)((cuse - 1) & 1), abort, polls);
            if (!ok) break;
            convert_stage<NT, MODE, SPLIT, false, NCONV>(raw + slot * RG::RAW, conv + cb * RG::CONV, ct, 0);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            mbar_arrive(raw_empty + slot);
            mbar_arrive(conv_full + cb);
        }
    } else if (l == 0) {
        for (int s = 0; s < nst && ok; ++s) {
            const int cb = s & 1, use = s >> 1;
            ok = mbar_wait(smem_u32(conv_full + cb), (uint32_t)(use & 1), abort, polls);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            mma_item_stage<NT, SPLIT, true, false>(smem_u32(conv + cb * RG::CONV), tmem, s == 0, 0);
            mma_commit(conv_empty + cb);
            *committed = s + 1;
        }
    }

    // every role arrives here (their waits are bounded); make the outcome block-uniform
    ok = __syncthreads_and(ok) != 0;
    bool done = true;
    const int ncommit = *committed;
    if (ncommit > 0) {   // the last committed stage's MMAs, waited for even after an abort
        const int sl = ncommit - 1;
        int no_abort = 0;
        const bool got = mbar_wait(smem_u32(conv_empty + (sl & 1)), (uint32_t)((sl >> 1) & 1), &no_abort);
        done = __syncthreads_and(got) != 0;
    }
    if (!ok || !done) {
        if (t == 0) atomicExch(flag, 1);
        ok = false;
    }
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");

    // ---- epilogue (converter warps), per column half of the tile:
    //  (1) tensor memory -> shared staging tile [128 rows][HALF + 2]; warp w may read TMEM lanes
    //      32 (w % 4) .. +31 (output tile o0 + w % 4); the two warps of a lane quarter split the columns;
    //  (2) each converter warp writes 16 staged rows, lane = pair of columns (16-byte accesses).
    if (ok && t >= NLOAD && t < NLOAD + NCONV) {
        constexpr int HALF = LY::HALF, SP = LY::SP;
        constexpr int CPW = HALF / 2;            // columns per warp per pass
        constexpr int RPW = MR / (NCONV / 32);   // staged rows written per warp
        constexpr int NP = HALF / 2;             // 16-byte column pairs per row and pass
        static_assert(CPW % 16 == 0, "epilogue tiling");
        float2* stg = (float2*)smem;             // operand and raw buffers are free after the MMAs
        const int cw = (t - NLOAD) >> 5;
        const int q4 = w & 3, sub = cw >> 2;
        const int rl = 32 * q4 + l;
        for (int pass = 0; pass < NT / HALF; ++pass) {
            const int cbeg = pass * HALF + sub * CPW;
            for (int c0 = cbeg; c0 < cbeg + CPW; c0 += 16) {
                uint32_t vr[16], vi[16];
                if (nst > 0) {
                    const uint32_t lane_off = (uint32_t)(32 * q4) << 16;
                    read_acc<NT, SPLIT, true>(tmem + lane_off, c0, vr, vi);
                } else {
#pragma unroll
                    for (int j = 0; j < 16; ++j) { vr[j] = 0u; vi[j] = 0u; }
                }
                const int cl = c0 - pass * HALF;
#pragma unroll
                for (int j = 0; j < 16; j += 2)
                    *(float4*)&stg[rl * SP + cl + j] = make_float4(__uint_as_float(vr[j]), __uint_as_float(vi[j]),
                                                                   __uint_as_float(vr[j + 1]), __uint_as_float(vi[j + 1]));
            }
            asm volatile("bar.sync 1, %0;" :: "n"(NCONV) : "memory");   // converter warps only
            const bool lane_on = l < NP;
            const int c = pass * HALF + 2 * l;
#pragma unroll 8
            for (int i = 0; i < RPW; ++i) {
                const int rl2 = cw * RPW + i;
                const long long base = rowbase[rl2];
                if (!lane_on || base < 0) continue;
                const float2 d = (MODE == FA) ? dinv_s[rl2] : make_float2(0.f, 0.f);
                write_pair<MODE>(it, base, c, *(const float4*)&stg[rl2 * SP + 2 * l], d);
            }
            asm volatile("bar.sync 1, %0;" :: "n"(NCONV) : "memory");   // staging reused by the next pass
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (w == mma_warp) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"(TCOLS));
}

// ------------------------------------------------------------------------------------------
// k_subst_tcp: persistent, one block per SM
// ------------------------------------------------------------------------------------------
// The wide tiles (NT <= 64) hold the factor operand in tensor memory: the converters write it there from
// registers, so that of the shared-memory traffic of a stage (NT = 32: 16 KB copied in, 16 read back, 32
// of operands written, 48 + 24 read by the MMAs) the factor's 80 KB of operands go.  The columns that the
// accumulators leave are its ring.  NT = 128 has none left: its two buffers take all 512 columns.
// Measured (128^3 layer, 32 columns / 64^3, 8 layers, 64 columns): operands in shared memory 1.68 / 2.80
// ms, in tensor memory 1.58 / 2.45, with two converter groups 1.53 / 2.33, row look-ups two stages ahead
// and integer rounding 1.48 / 2.24, running tile pointers 1.40 / 2.13; 128 columns (64^3, M_pol) 9.69 ->
// 8.17 from the last three.  A third of the MMAs would save 15 %: the instruction streams of the loaders
// and converters bind the narrow tiles, the shared-memory banks NT = 128.
template <int NT> struct PLayout {
    using RG = Ring<NT>;
    static constexpr bool TA = RG::WIDE;
    // the hi x lo terms' own accumulators fit beside the factor ring at NT = 32
    static constexpr bool SEP = NT == 32;
    static constexpr int CD = NT <= 64 ? 4 : 2;                    // converted operands' ring depth
    static constexpr int RD = NT == 32 ? 6 : NT == 64 ? 4 : 2;     // raw ring depth
    // Two converter groups take alternate stages.  A parity wait tells only the last phase from the one
    // before, so nobody may reach it while an older use of the slot is still open.  With even depths a slot
    // is one group's alone and the group's own previous wait on it has closed that use; with an odd
    // depth it would follow only from the MMAs' commits arriving in the order of the stages.
    static_assert(CD % 2 == 0 && RD % 2 == 0, "a ring slot belongs to one converter group");
    static constexpr int CONV = TA ? 6 * RG::X_MAT : RG::CONV;
    static constexpr int NEPI = 128;                       // epilogue threads (4 warps)
    static constexpr int NTHREADS = NLOAD + NCONV + 32 + NEPI;
    static constexpr int EP = 18;                          // staging pitch (complex) of a 32 x 16 chunk
    static constexpr int STG_OFF = CD * CONV + RD * RG::RAW;   // 4 warps x 32 rows x EP complex
    static constexpr int BAR_OFF = STG_OFF + 4 * 32 * EP * 8;
    static constexpr int TOTAL = BAR_OFF + (2 * RD + 2 * CD + 4) * 8 + 16;
    static_assert(TOTAL <= 232448, "shared memory of one block");
};

template <int NT, int MODE, int SPLIT>
__global__ void __launch_bounds__(PLayout<NT>::NTHREADS, 1)
k_subst_tcp(const Task* __restrict__ tasks, const JobDev<float2>* __restrict__ jobs, int ldc, int nchunks,
            long long nitems, int* flag, long long polls) {
    using RG = Ring<NT>;
    using LY = PLayout<NT>;
    extern __shared__ __align__(1024) unsigned char smem[];
    constexpr int RD = LY::RD, CD = LY::CD, CGRP = NCONV / 2;
    constexpr bool SEP = LY::SEP, TA = LY::TA;
    constexpr int BCOLS = acc_cols<NT, SPLIT, SEP>;          // one accumulator buffer
    constexpr int ACOL = 2 * BCOLS;                          // factor ring (TA): CD x 4 KC columns
    constexpr int TCOLS = TA ? 512 : 2 * BCOLS;
    static_assert(ACOL + (TA ? CD * 4 * KC : 0) <= 512, "tensor memory columns");
    unsigned char* conv = smem;                  // [CD][CONV]
    unsigned char* raw = smem + CD * LY::CONV;   // [RD][RAW]
    uint64_t* raw_full = (uint64_t*)(smem + LY::BAR_OFF);   // [RD] loaders' copies landed (count NLOAD)
    uint64_t* raw_empty = raw_full + RD;   // [RD] converters done reading (count CGRP)
    uint64_t* conv_full = raw_empty + RD;  // [CD] converted operands written (count CGRP)
    uint64_t* conv_empty = conv_full + CD; // [CD] MMAs of the buffer done (tcgen05.commit)
    uint64_t* acc_full = conv_empty + CD;  // [2] all MMAs of an item's accumulator done (tcgen05.commit)
    uint64_t* acc_empty = acc_full + 2;    // [2] epilogue done reading the accumulator (count NEPI)
    uint32_t* tptr = (uint32_t*)(acc_empty + 2);
    volatile int* abort = (volatile int*)tptr + 1;

    const int t = threadIdx.x, w = t >> 5, l = t & 31;
    const int mma_warp = (NLOAD + NCONV) / 32;
    const int epi_warp0 = (NLOAD + NCONV + 32) / 32;

    if (w == mma_warp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" :: "r"(smem_u32(tptr)),
                     "r"(TCOLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (t == 0) {
        for (int b = 0; b < RD; ++b) {
            mbar_init(raw_full + b, NLOAD);
            mbar_init(raw_empty + b, CGRP);
        }
        for (int b = 0; b < CD; ++b) {
            mbar_init(conv_full + b, CGRP);
            mbar_init(conv_empty + b, 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(acc_full + b, 1);
            mbar_init(acc_empty + b, LY::NEPI);
        }
        *abort = 0;
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tptr;
    bool ok = true;
    bool mma_drained = true;

    if (t < NLOAD) {
        // ------------------------------------------------------------ loaders
        // the next item is decoded, and the vector rows of the next two stages (BA: a lookup in the
        // update list) are on their way, while the current stage's copies are issued
        long long gs = 0;  // stage counter across this block's items
        long long item = blockIdx.x;
        Item cur;
        Vrows<NT> rows, rows1;
        if (item < nitems) {
            cur = decode<NT, MODE>(tasks, jobs, item, nchunks);
            rows = stage_rows<NT, MODE>(cur, 0, t);
            rows1 = stage_rows<NT, MODE>(cur, 1, t);   // an item has at least two stages
        }
        for (; item < nitems && ok; item += gridDim.x) {
            const long long nxt_item = item + gridDim.x;
            Item nxt = cur;
            if (nxt_item < nitems) nxt = decode<NT, MODE>(tasks, jobs, nxt_item, nchunks);
            TilePtrs<MODE> tp;
            tp.init(cur, t);
            for (int s = 0; s < cur.nst && ok; ++s, ++gs) {
                const int slot = (int)(gs % RD);
                const long long use = gs / RD;
                Vrows<NT> rows2;
                if (s + 2 < cur.nst) rows2 = stage_rows<NT, MODE>(cur, s + 2, t);
                else if (nxt_item < nitems) rows2 = stage_rows<NT, MODE>(nxt, s + 2 - cur.nst, t);
                if (gs >= RD) ok = mbar_wait(smem_u32(raw_empty + slot), (uint32_t)((use - 1) & 1), abort, polls);
                if (!ok) break;
                load_stage<NT, MODE>(raw + slot * RG::RAW, cur, tp, s, ldc, t, rows);
                cp_async_arrive(raw_full + slot);
                rows = rows1;
                rows1 = rows2;
            }
            cur = nxt;
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
    } else if (t < NLOAD + NCONV) {
        // ------------------------------------------------------------ converters
        // two groups of warps take alternate stages: a stage is a chain of waits, shared-memory loads,
        // operand stores and fences, and two of them overlap
        const int ct = (t - NLOAD) & (CGRP - 1), grp = (t - NLOAD) / CGRP;
        long long gs = 0;
        int nst_next = blockIdx.x < nitems ? decode<NT, MODE>(tasks, jobs, blockIdx.x, nchunks).nst : 0;
        for (long long item = blockIdx.x; item < nitems && ok; item += gridDim.x) {
            const int nst = nst_next;   // decoded one item ahead
            if (item + gridDim.x < nitems) nst_next = decode<NT, MODE>(tasks, jobs, item + gridDim.x, nchunks).nst;
            for (int s = 0; s < nst && ok; ++s, ++gs) {
                if ((int)(gs & 1) != grp) continue;
                const int slot = (int)(gs % RD), cb = (int)(gs % CD);
                const long long use = gs / RD, cuse = gs / CD;
                ok = mbar_wait(smem_u32(raw_full + slot), (uint32_t)(use & 1), abort, polls);
                if (ok && gs >= CD) ok = mbar_wait(smem_u32(conv_empty + cb), (uint32_t)((cuse - 1) & 1), abort, polls);
                if (!TA && !ok) break;
                if (TA) {
                    ok = __all_sync(0xffffffffu, ok);   // the tensor-memory stores are warp-wide
                    if (!ok) break;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                }
                convert_stage<NT, MODE, SPLIT, TA, CGRP>(raw + slot * RG::RAW, conv + cb * LY::CONV, ct, tmem + ACOL + cb * 4 * KC);
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                mbar_arrive(raw_empty + slot);
                mbar_arrive(conv_full + cb);
            }
        }
    } else if (w == mma_warp) {
        // ------------------------------------------------------------ MMA issuer (lane 0)
        if (l == 0) {
            long long gs = 0;
            int nit = 0;  // items of this block so far
            int nst_next = blockIdx.x < nitems ? decode<NT, MODE>(tasks, jobs, blockIdx.x, nchunks).nst : 0;
            for (long long item = blockIdx.x; item < nitems && ok; item += gridDim.x, ++nit) {
                const int nst = nst_next;   // decoded one item ahead
                if (item + gridDim.x < nitems) nst_next = decode<NT, MODE>(tasks, jobs, item + gridDim.x, nchunks).nst;
                const int b = nit & 1;
                if (nit >= 2) ok = mbar_wait(smem_u32(acc_empty + b), (uint32_t)(((nit >> 1) - 1) & 1), abort, polls);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t tm = tmem + (uint32_t)(b * BCOLS);
                for (int s = 0; s < nst && ok; ++s, ++gs) {
                    const int cb = (int)(gs % CD);
                    ok = mbar_wait(smem_u32(conv_full + cb), (uint32_t)((gs / CD) & 1), abort, polls);
                    if (!ok) break;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    mma_item_stage<NT, SPLIT, SEP, TA>(smem_u32(conv + cb * LY::CONV), tm, s == 0, tmem + ACOL + cb * 4 * KC);
                    mma_commit(conv_empty + cb);
                }
                mma_commit(acc_full + b);   // arrives when every MMA issued so far has completed
            }
            // before the tensor memory is freed every issued MMA must have completed: the last
            // item begun (nit - 1; an interrupted one was committed too) is waited for, even
            // after an abort
            if (nit > 0) {
                int no_abort = 0;
                mma_drained = mbar_wait(smem_u32(acc_full + ((nit - 1) & 1)), (uint32_t)(((nit - 1) >> 1) & 1), &no_abort);
            }
        }
    } else {
        // ------------------------------------------------------------ epilogue warps
        // warp w reads TMEM lanes 32 (w % 4) .. +31 = output rows of tile o0 + w % 4 (lane = row);
        // per 16-column chunk: stage 32 x 16 in this warp's shared slice, then write 4 rows per
        // instruction (8 lanes x 16 bytes per row)
        const int q4 = w & 3;
        float2* stg = (float2*)(smem + LY::STG_OFF) + (size_t)(w - epi_warp0) * 32 * LY::EP;
        const int r4 = l >> 3, p = l & 7;   // write phase: row within a group of 4, column pair
        int nit = 0;
        for (long long item = blockIdx.x; item < nitems && ok; item += gridDim.x, ++nit) {
            const Item it = decode<NT, MODE>(tasks, jobs, item, nchunks);
            const int b = nit & 1;
            // this lane's row descriptor, shuffled to the writing lanes below
            const long long my_base = row_base<MODE>(it, 32 * q4 + l, ldc);
            float2 my_d = make_float2(0.f, 0.f);
            if (MODE == FA && my_base >= 0) my_d = it.jb.dinv[it.nd.own0 + it.o0 * TILE + 32 * q4 + l];
            ok = mbar_wait(smem_u32(acc_full + b), (uint32_t)((nit >> 1) & 1), abort, polls);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t lane_off = (uint32_t)(32 * q4) << 16;
            const uint32_t tm = tmem + (uint32_t)(b * BCOLS) + lane_off;
            for (int c0 = 0; c0 < NT; c0 += 16) {
                uint32_t vr[16], vi[16];
                if (it.nst > 0) {
                    read_acc<NT, SPLIT, SEP>(tm, c0, vr, vi);
                } else {
#pragma unroll
                    for (int j = 0; j < 16; ++j) { vr[j] = 0u; vi[j] = 0u; }
                }
#pragma unroll
                for (int j = 0; j < 16; j += 2)
                    *(float4*)&stg[l * LY::EP + j] = make_float4(__uint_as_float(vr[j]), __uint_as_float(vi[j]),
                                                                 __uint_as_float(vr[j + 1]), __uint_as_float(vi[j + 1]));
                __syncwarp();
                const int c = c0 + 2 * p;
#pragma unroll
                for (int g = 0; g < 8; ++g) {
                    const int rr = 4 * g + r4;
                    const long long base = __shfl_sync(0xffffffffu, my_base, rr);
                    float2 d = make_float2(0.f, 0.f);
                    if (MODE == FA) {
                        d.x = __shfl_sync(0xffffffffu, my_d.x, rr);
                        d.y = __shfl_sync(0xffffffffu, my_d.y, rr);
                    }
                    if (base < 0) continue;
                    write_pair<MODE>(it, base, c, *(const float4*)&stg[rr * LY::EP + 2 * p], d);
                }
                __syncwarp();
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            mbar_arrive(acc_empty + b);
        }
    }

    ok = __syncthreads_and(ok && mma_drained) != 0;
    if (!ok && t == 0) atomicExch(flag, 1);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (w == mma_warp) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"(TCOLS));
}

template <int NT, int MODE, int SPLIT>
void launch_one(const Batch& b, const Task* tasks, long long n, const JobDev<float2>* jobs, int ldc, int* flag,
                cudaStream_t st) {
    const int nchunks = (b.job_cols > 0 ? b.job_cols : ldc) / NT;
    const long long nitems = n * nchunks;
    if (b.tc_cfg == 1) {
        const long long grid = std::min<long long>(nitems, b.sms);
        k_subst_tcp<NT, MODE, SPLIT><<<(unsigned)grid, PLayout<NT>::NTHREADS, PLayout<NT>::TOTAL, st>>>(
            tasks, jobs, ldc, nchunks, nitems, flag, b.wait_polls);
    } else {
        k_subst_tc<NT, MODE, SPLIT><<<(unsigned)nitems, OneLayout<NT>::NTHREADS, OneLayout<NT>::TOTAL, st>>>(
            tasks, jobs, ldc, nchunks, flag, b.wait_polls);
    }
    HZ_CHECK_LAUNCH();
}

template <int NT, int MODE, int SPLIT> void allow_smem(int cfg) {
    if (cfg == 1)
        HZ_CUDA(cudaFuncSetAttribute(k_subst_tcp<NT, MODE, SPLIT>, cudaFuncAttributeMaxDynamicSharedMemorySize, PLayout<NT>::TOTAL));
    else
        HZ_CUDA(cudaFuncSetAttribute(k_subst_tc<NT, MODE, SPLIT>, cudaFuncAttributeMaxDynamicSharedMemorySize, OneLayout<NT>::TOTAL));
}
template <int NT, int SPLIT> void allow_smem_modes(int cfg) {
    allow_smem<NT, FA, SPLIT>(cfg);
    allow_smem<NT, FB, SPLIT>(cfg);
    allow_smem<NT, BA, SPLIT>(cfg);
    allow_smem<NT, BB, SPLIT>(cfg);
}

template <int NT, int SPLIT>
void launch_mode(const Batch& b, int h, int mode, int ldc, int* flag, cudaStream_t st) {
    const long long off = b.pair_off[mode][h], n = b.pair_cnt[mode][h];
    if (n == 0) return;
    const Task* tasks = b.d_tasks + off;
    const JobDev<float2>* jobs = (const JobDev<float2>*)b.d_jobs;
    switch (mode) {
        case FA: launch_one<NT, FA, SPLIT>(b, tasks, n, jobs, ldc, flag, st); break;
        case FB: launch_one<NT, FB, SPLIT>(b, tasks, n, jobs, ldc, flag, st); break;
        case BA: launch_one<NT, BA, SPLIT>(b, tasks, n, jobs, ldc, flag, st); break;
        default: launch_one<NT, BB, SPLIT>(b, tasks, n, jobs, ldc, flag, st); break;
    }
}

}  // namespace

int tc_columns(int ldc) {
    if (ldc % 128 == 0) return 128;
    if (ldc % 64 == 0) return 64;
    if (ldc % 32 == 0) return 32;
    return 0;
}

void prepare_tc(const Batch& b, int ldc) {
    const int nt = tc_columns(b.job_cols > 0 ? b.job_cols : ldc);
    if (b.split == 1) {
        if (nt == 128) allow_smem_modes<128, 1>(b.tc_cfg);
        else if (nt == 64) allow_smem_modes<64, 1>(b.tc_cfg);
        else allow_smem_modes<32, 1>(b.tc_cfg);
    } else {
        if (nt == 128) allow_smem_modes<128, 3>(b.tc_cfg);
        else if (nt == 64) allow_smem_modes<64, 3>(b.tc_cfg);
        else allow_smem_modes<32, 3>(b.tc_cfg);
    }
}

void launch_level_tc(const Batch& b, int h, int mode, int ldc, int* flag, cudaStream_t st) {
    const int nt = tc_columns(b.job_cols > 0 ? b.job_cols : ldc);
    if (b.split == 1) {
        if (nt == 128) launch_mode<128, 1>(b, h, mode, ldc, flag, st);
        else if (nt == 64) launch_mode<64, 1>(b, h, mode, ldc, flag, st);
        else launch_mode<32, 1>(b, h, mode, ldc, flag, st);
    } else {
        if (nt == 128) launch_mode<128, 3>(b, h, mode, ldc, flag, st);
        else if (nt == 64) launch_mode<64, 3>(b, h, mode, ldc, flag, st);
        else launch_mode<32, 3>(b, h, mode, ldc, flag, st);
    }
}

}  // namespace hz
