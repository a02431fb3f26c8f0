// Which tiles, vector rows and output rows a tensor-core work item touches: the index arithmetic of
// the kernels of subst_tc.cu, callable on the host too, so that a test can walk every item of a batch.
#pragma once

#include "hz_internal.cuh"
#include "tc_common.cuh"

namespace hz {
namespace tcc {

enum { FA = 0, FB = 1, BA = 2, BB = 3 };

// One work item: 128 output rows (tiles o0 .. o0+3) x NT columns of one node product, reduction
// tiles [kbeg, kend).
struct Item {
    JobDev<float2> jb;
    NodeDev nd;
    int col0, o0, nout_t, nrows_out, nrows_k, kbeg, kend, nst;
    bool unique;
};

template <int NT, int MODE>
__host__ __device__ inline Item decode(const Task* tasks, const JobDev<float2>* jobs, long long item, int nchunks) {
    Item it;
    const Task tk = tasks[item / nchunks];
    it.jb = jobs[tk.job];
    it.nd = it.jb.nodes[tk.node];
    const NodeDev& nd = it.nd;
    it.col0 = (int)(item % nchunks) * NT;
    it.o0 = tk.tile;
    it.nout_t = (MODE == FB) ? nd.upd_t : nd.own_t;
    it.nrows_out = (MODE == FB) ? nd.nupd : nd.nown;
    it.nrows_k = (MODE == BA) ? nd.nupd : nd.nown;
    it.kbeg = tk.k0;
    const int kfull0 = (MODE == BB) ? it.o0 : 0;
    const int kfull1 = (MODE == FA) ? min(it.o0 + 4, nd.own_t) : ((MODE == BA) ? nd.upd_t : nd.own_t);
    it.kend = it.kbeg + tk.klen;
    it.nst = tk.klen * 2;
    it.unique = it.kbeg == kfull0 && it.kend == kfull1 && MODE != FB && MODE != BA;
    return it;
}

// Vector rows a loader thread copies in stage s of an item (-1: beyond the node, zero-filled).
// They are looked up one stage ahead, so that BA's gather through the update index list is not
// on the copy's critical path.
template <int NT> struct Vrows { int r[KC * NT / 2 / NLOAD]; };

template <int NT, int MODE>
__host__ __device__ inline Vrows<NT> stage_rows(const Item& it, int s, int t) {
    Vrows<NT> v;
    const int kt = it.kbeg + (s >> 1), hk = s & 1;
    const int* upd = it.jb.upd_idx + it.nd.upd_off;
#pragma unroll
    for (int i = 0; i < KC * NT / 2 / NLOAD; ++i) {
        const int k = (t + NLOAD * i) / (NT / 2);
        const int rr = kt * TILE + hk * KC + k;
        v.r[i] = -1;
        if (rr < it.nrows_k) v.r[i] = (MODE == BA) ? upd[rr] : it.nd.own0 + rr;
    }
    return v;
}

// The four factor tiles of an item's current reduction tile, as one loader thread copies them: its
// first 16 bytes of each (8 per stage: 4 tiles x 2, 2 KB apart as stored, 16 columns apart where used
// transposed).  Pointers advance from tile to tile; forming every copy's address anew (triangular
// index, 64-bit products) kept a loader warp at some 230 instructions a stage, which bound narrow tiles.
template <int MODE> struct TilePtrs {
    static constexpr bool TR = (MODE == BA || MODE == BB);
    const char* p[4];
    int kt, o0, nout_t;
    long long step;   // bytes to the next reduction tile (BB: of the first one on)

    __host__ __device__ __forceinline__ void init(const Item& it, int t) {
        const NodeDev& nd = it.nd;
        kt = it.kbeg;
        o0 = it.o0;
        nout_t = it.nout_t;
        const int thr = TR ? (t >> 3) * 256 + (t & 7) * 16 : t * 16;
#pragma unroll
        for (int oi = 0; oi < 4; ++oi) {
            const int o = o0 + oi;
            long long toff;
            if (MODE == FA) toff = nd.linv_off + tri_idx(o, kt);
            else if (MODE == FB) toff = nd.l21_off + (long long)o * nd.own_t + kt;
            else if (MODE == BA) toff = nd.l21_off + (long long)kt * nd.own_t + o;
            else toff = nd.linv_off + tri_idx(kt, o);
            p[oi] = (const char*)(it.jb.fac + toff * TILE2) + thr;
        }
        step = (MODE == BA ? (long long)nd.own_t : MODE == BB ? (long long)kt + 1 : 1LL) * (TILE2 * 8);
    }
    __host__ __device__ __forceinline__ void next() {
#pragma unroll
        for (int oi = 0; oi < 4; ++oi) p[oi] += step;
        ++kt;
        if (MODE == BB) step += TILE2 * 8;
    }
    __host__ __device__ __forceinline__ bool exists(int oi) const {
        const int o = o0 + oi;
        return o < nout_t && (MODE != FA || kt <= o) && (MODE != BB || kt >= o);
    }
};

// global offset (row x ldc + chunk column) of local output row r of an item, -1 if absent
template <int MODE>
__host__ __device__ inline long long row_base(const Item& it, int r, int ldc) {
    const int row = it.o0 * TILE + r;
    if ((it.o0 + (r >> 5)) >= it.nout_t || row >= it.nrows_out) return -1;
    const int* upd = it.jb.upd_idx + it.nd.upd_off;
    return ((MODE == FB) ? (long long)upd[row] : (long long)(it.nd.own0 + row)) * ldc + it.col0;
}

}  // namespace tcc
}  // namespace hz
