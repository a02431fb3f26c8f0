// One-launch substitution for complex64 blocks of at most 16 columns.
//
// With few columns a substitution is a chain of 2 H dependent phases (solve.cu) of a few
// microseconds of work each: as one launch per phase, every phase pays a kernel boundary, the chain
// of loads to its first factor tile, and a drained memory system (64^3, one layer, 16 columns: 0.37 ms
// for 0.05 ms worth of factor bytes).  Here one cooperative launch, one block per SM, runs all phases
// with a grid barrier between them, and the factor tiles, which no phase computes, stream past the
// barriers: every warp copies the tiles of its own tasks, of all phases in order, into a private
// ring in shared memory, so that a phase finds its first tiles there and only its vector entries
// (L2) are loaded after the barrier.
//
// A task is one TILE-row slab of one product over a range of reduction indices, and one warp's work:
// lane = output row, all columns in registers, 16 reduction indices (half a tile, 4 KB) per step, no
// synchronisation beyond the warp.  Eight independent warps hide each other's latencies where a phase
// is wide; where it is narrow, half-tile tasks spread it over all SMs.  (One task per block with the
// warps sharing every tile spent 950 cycles a tile on the chain wait - load - multiply, whatever
// the columns.)  Columns are accumulated with packed FP32 FMAs as (ar xr, ar xi) and (ai xr, ai xi),
// combined at the end.  Half tiles used as stored (FA, FB) are one bulk copy; those used transposed
// (BA, BB) are copied with 16-byte cp.async into rows padded by 16 bytes, which makes a lane's 16-byte
// loads of two reduction indices conflict-free.
//
// FB and BA add into acc with vector atomics; FA and BB tasks that cover their whole reduction store,
// and the rows of those that are split are cleared in an earlier phase.  Tasks are dealt to the warps
// per phase, longest first, to the least loaded one (host).  Bound: HBM at 2-4 columns, FP32 FMA issue
// at 16 (512 cycles per tile and SM), barriers where the tree is narrow.  Measured, launches per phase
// against one launch: 64^3, one layer of 8, 2 / 4 / 16 columns 0.201 -> 0.116, 0.236 -> 0.134, 0.373 ->
// 0.228 ms; all 8 layers 1.38 -> 1.11, 1.77 -> 1.18, 3.52 -> 2.30 ms (4 columns: 5.5 TB/s of DRAM); 24^3,
// 2 columns 0.095 -> 0.049 ms.
//
// Every wait is bounded (polls and wall time).  A wait that gives up ends the block's other waits and
// raises the error flag; every warp waits (bounded) for its copies in flight before it leaves, and every
// block still counts itself out, so the barrier counters are back at zero for the next launch.
#include <algorithm>
#include <queue>

#include "hz_internal.cuh"
#include "hz_ctx.cuh"
#include "hz_solve.cuh"
#include "tc_common.cuh"

namespace hz {

namespace {

using tcc::mbar_arrive;
using tcc::mbar_init;
using tcc::mbar_wait;
using tcc::smem_u32;

enum { FA = 0, FB = 1, BA = 2, BB = 3 };

constexpr int SW = 8;                     // warps
constexpr int KU = SKU;                   // reduction indices per step
constexpr int TPITCH = KU + 2;            // transposed half tiles: padded row (complex)
constexpr int SLOT = TILE * TPITCH * 8;   // 4608 bytes
constexpr int DX = 4;                     // vector slices in the ring

template <int RC> struct SLayout {
    static constexpr int XS = KU * RC * 8;                    // one vector slice
    static constexpr int SLOTS = RC == 16 ? 4 : 5;
    static constexpr int WARP = SLOTS * SLOT + DX * XS;       // one warp's rings
    static constexpr int OP = RC * 8 + 16;                    // pitch of the staged outputs (over the vector ring)
    static_assert(TILE * OP <= DX * XS, "staged outputs fit in the vector ring");
    static constexpr int BAR_OFF = SW * WARP;
    static constexpr int TOTAL = BAR_OFF + SW * SLOTS * 8 + 16;
};

__device__ __forceinline__ void bulk_copy(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 :: "r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect(uint32_t bar, uint32_t bytes) {
    asm volatile("{\n.reg .b64 st;\nmbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n}" :: "r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ float2 ffma2(float2 a, float2 b, float2 c) {
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;"
        : "=l"(r)
        : "l"(*(unsigned long long*)&a), "l"(*(unsigned long long*)&b), "l"(*(unsigned long long*)&c));
    return *(float2*)&r;
}
// Barrier of the block that also agrees on the outcome: a thread that gave up still arrives here,
// and all of them then leave together.
__device__ __forceinline__ bool block_and(bool ok) { return __syncthreads_and(ok) != 0; }

// A warp's stream of half tiles over all of its tasks: issue() copies the next one into the ring.
template <int RC> struct TileStream {
    using LY = SLayout<RC>;
    const STask* tasks;
    const JobDev<float2>* jobs;
    unsigned char* ring;
    uint64_t* full;
    int i, i1;             // next task to look at, end of the warp's list
    int left = 0, half, step, dstep;
    bool tr;
    const float2* tile;    // current tile
    unsigned q = 0;        // half tiles issued

    __device__ __forceinline__ void issue(int l) {
        while (left == 0) {
            if (i >= i1) return;
            const STask& tk = tasks[i++];
            left = tk.nunits;
            half = tk.half0;
            step = tk.step;
            dstep = tk.dstep;
            tr = tk.mode == BA || tk.mode == BB;
            tile = jobs[tk.job].fac + tk.tile0 * TILE2;
        }
        const int slot = (int)(q % LY::SLOTS);
        const uint32_t dst = smem_u32(ring + slot * SLOT);
        uint64_t* bar = full + slot;
        if (tr) {   // columns of 16 consecutive reduction indices: 8 pieces each
            const float2* src = tile + half * KU + (l >> 3) * TILE + (l & 7) * 2;
            const uint32_t d = dst + (l >> 3) * TPITCH * 8 + (l & 7) * 16;
#pragma unroll
            for (int c = 0; c < TILE; c += 4) tcc::cp16(d + c * TPITCH * 8, src + c * TILE, 16);
            tcc::cp_async_arrive(bar);
        } else if (l == 0) {
            // the slot was last read, or filled by cp.async, through the generic proxy
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            mbar_expect(smem_u32(bar), KU * TILE * 8);
            bulk_copy(dst, tile + half * KU * TILE, KU * TILE * 8, smem_u32(bar));
        } else {
            mbar_arrive(bar);
        }
        ++q;
        --left;
        if (half) {
            tile += (long long)step * TILE2;
            step += dstep;
        }
        half ^= 1;
    }
};

// One task of one warp.  `enter` runs once the task's first row indices are on their way and before
// its first vector access (the grid barrier of the phase's first task).  u: half tiles consumed.
template <int RC, int MODE, class Enter>
__device__ __forceinline__ bool run_task(const STask& tk, const JobDev<float2>& jb, TileStream<RC>& ts, unsigned char* xs,
                                         unsigned& u, int l, volatile int* abort, long long polls, Enter enter) {
    using LY = SLayout<RC>;
    constexpr bool TR = MODE == BA || MODE == BB;
    constexpr int LPR = RC / 2;                            // 16-byte pieces of a vector row
    constexpr int NP = (KU * LPR + 31) / 32;               // pieces of a slice per lane
    const int* upd = jb.upd_idx + tk.upd_off;
    const float2* vec = MODE == BB ? jb.x : jb.acc;
    const int nu = tk.nunits;
    struct Rows { int r[NP]; };
    auto rows_of = [&](int j) {
        Rows v;
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            const int k = j * KU + (l + 32 * i) / LPR;
            v.r[i] = -1;
            if ((l + 32 * i) / LPR < KU && j < nu && k < tk.nk)
                v.r[i] = MODE == BA ? __ldg(upd + tk.k0 + k) : tk.own0 + tk.k0 + k;
        }
        return v;
    };
    auto load_x = [&](int j, const Rows& v) {
        if (j < nu) {
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                const int p = l + 32 * i;
                if (p < KU * LPR)
                    tcc::cp16(smem_u32(xs + (j % DX) * LY::XS + p * 16),
                              vec + (long long)(v.r[i] < 0 ? 0 : v.r[i]) * RC + 2 * (p % LPR), v.r[i] < 0 ? 0 : 16);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    Rows rows[DX - 1];
#pragma unroll
    for (int j = 0; j < DX - 1; ++j) rows[j] = rows_of(j);
    // the output row of this lane's register sums
    int orow = -1;
    float2 od = make_float2(0.f, 0.f);
    if (l < tk.nrows) {
        orow = MODE == FB ? __ldg(upd + tk.row0 + l) : tk.own0 + tk.row0 + l;
        if (MODE == FA) od = __ldg(jb.dinv + orow);
    }
    if (!enter()) return false;
#pragma unroll
    for (int j = 0; j < DX - 1; ++j) load_x(j, rows[j]);
    Rows next = rows_of(DX - 1);

    float2 a1[RC], a2[RC];   // (ar xr, ar xi), (ai xr, ai xi)
#pragma unroll
    for (int c = 0; c < RC; ++c) { a1[c] = make_float2(0.f, 0.f); a2[c] = make_float2(0.f, 0.f); }
    bool ok = true;
    for (int j = 0; j < nu; ++j) {
        load_x(j + DX - 1, next);
        next = rows_of(j + DX);
        const int slot = (int)(u % LY::SLOTS);
        ok = mbar_wait(smem_u32(ts.full + slot), (u / LY::SLOTS) & 1, abort, polls);
        asm volatile("cp.async.wait_group %0;" :: "n"(DX - 1) : "memory");
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        __syncwarp();   // the slice holds pieces that other lanes copied: a vote orders no memory accesses
        ++u;
        const float2* tile = (const float2*)(ts.ring + slot * SLOT);
        const float2* x = (const float2*)(xs + (j % DX) * LY::XS);
#pragma unroll
        for (int k = 0; k < KU; k += 2) {
            float2 a[2];
            if (TR) {
                const float4 p = *(const float4*)(tile + l * TPITCH + k);
                a[0] = make_float2(p.x, p.y);
                a[1] = make_float2(p.z, p.w);
            } else {
                a[0] = tile[k * TILE + l];
                a[1] = tile[(k + 1) * TILE + l];
            }
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const float2 ar = make_float2(a[e].x, a[e].x), ai = make_float2(a[e].y, a[e].y);
#pragma unroll
                for (int c = 0; c < RC; c += 2) {
                    const float4 v = *(const float4*)(x + (k + e) * RC + c);
                    const float2 v0 = make_float2(v.x, v.y), v1 = make_float2(v.z, v.w);
                    a1[c] = ffma2(ar, v0, a1[c]);
                    a2[c] = ffma2(ai, v0, a2[c]);
                    a1[c + 1] = ffma2(ar, v1, a1[c + 1]);
                    a2[c + 1] = ffma2(ai, v1, a2[c + 1]);
                }
            }
        }
        __syncwarp();   // the half tile and the slice are overwritten from here on
        ts.issue(l);
    }
    if (!ok) return false;
    // stage the slab over the vector ring (the last slice's wait covered all of this task's copies to
    // it), so that rows are written by neighbouring lanes
#pragma unroll
    for (int c = 0; c < RC; c += 2) {
        float2 y0 = make_float2(a1[c].x - a2[c].y, a1[c].y + a2[c].x);
        float2 y1 = make_float2(a1[c + 1].x - a2[c + 1].y, a1[c + 1].y + a2[c + 1].x);
        if (MODE == FA) { y0 = cmul(od, y0); y1 = cmul(od, y1); }
        *(float4*)(xs + l * LY::OP + c * 8) = make_float4(y0.x, y0.y, y1.x, y1.y);
    }
    __syncwarp();
    float2* out = MODE == FA ? jb.x : jb.acc;
    const int c = 2 * (l % LPR);
#pragma unroll
    for (int r0 = 0; r0 < TILE; r0 += 32 / LPR) {
        const int r = r0 + l / LPR;
        const int row = __shfl_sync(0xffffffffu, orow, r);
        if (row < 0) continue;
        const float4 y = *(const float4*)(xs + r * LY::OP + c * 8);
        float4* o = (float4*)(out + (long long)row * RC + c);
        if (MODE == FB || MODE == BA) atomicAdd(o, make_float4(-y.x, -y.y, -y.z, -y.w));
        else if (tk.store) *o = y;
        else atomicAdd(o, y);
    }
    __syncwarp();
    return true;
}

// sync[0]: blocks that have finished a phase, over all phases; sync[1]: blocks that are done.  Warp v
// of the grid (block v % G) has tasks off[v * nph + phase] .. off[v * nph + phase + 1).
template <int RC>
__global__ void __launch_bounds__(32 * SW, 1)
k_subst_stream(const STask* __restrict__ tasks, const int* __restrict__ off, int nph,
               const JobDev<float2>* __restrict__ jobs, unsigned* sync, int* flag, long long polls) {
    using LY = SLayout<RC>;
    extern __shared__ __align__(128) unsigned char smem[];
    const int t = threadIdx.x, w = t >> 5, l = t & 31;
    const unsigned G = gridDim.x;
    const long long v = (long long)w * G + blockIdx.x;
    uint64_t* bars = (uint64_t*)(smem + LY::BAR_OFF);
    volatile int* abort = (volatile int*)(bars + SW * LY::SLOTS);
    if (t == 0) {
        for (int s = 0; s < SW * LY::SLOTS; ++s) mbar_init(bars + s, 32);   // the warp's lanes
        *abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    const int* myoff = off + v * nph;
    TileStream<RC> ts;
    ts.tasks = tasks;
    ts.jobs = jobs;
    ts.ring = smem + w * LY::WARP;
    ts.full = bars + w * LY::SLOTS;
    ts.i = myoff[0];
    ts.i1 = myoff[nph];
    unsigned char* xs = ts.ring + LY::SLOTS * SLOT;
    for (int s = 0; s < LY::SLOTS; ++s) ts.issue(l);
    unsigned u = 0;
    bool ok = true;
    STask next = tasks[ts.i1 > myoff[0] ? myoff[0] : 0];   // looked up one task ahead
    for (int ph = 0; ph < nph; ++ph) {
        // all blocks have finished the phases before ph; polled by one thread.  Every thread of the
        // block comes here exactly once per phase, and all get the same answer.
        auto enter = [&]() -> bool {
            if (ph == 0) return true;
            bool got = true;
            if (t == 0) {
                const unsigned want = (unsigned)ph * G;
                unsigned long long t0 = 0;
                for (long long it = 0; ld_acquire(sync) < want; ++it) {
                    got = it < polls;
                    if (got && (it & 63) == 63) {
                        const unsigned long long now = tcc::global_ns();
                        if (t0 == 0) t0 = now;
                        got = !*abort && now - t0 <= tcc::WAIT_NS;
                    }
                    if (!got) break;
                }
            }
            return block_and(got);
        };
        const int i0 = myoff[ph], i1 = myoff[ph + 1];
        bool entered = false;
        auto first = [&]() -> bool {
            if (entered) return true;
            entered = true;
            return enter();
        };
        if (i0 == i1) ok = first();
        for (int i = i0; i < i1 && ok; ++i) {
            const STask tk = next;
            next = tasks[i + 1];   // the list is padded by one task
            const JobDev<float2> jb = jobs[tk.job];
            if (tk.mode == FA) ok = run_task<RC, FA>(tk, jb, ts, xs, u, l, abort, polls, first);
            else if (tk.mode == FB) ok = run_task<RC, FB>(tk, jb, ts, xs, u, l, abort, polls, first);
            else if (tk.mode == BA) ok = run_task<RC, BA>(tk, jb, ts, xs, u, l, abort, polls, first);
            else if (tk.mode == BB) ok = run_task<RC, BB>(tk, jb, ts, xs, u, l, abort, polls, first);
            else {
                ok = first();
                float2* z = (tk.mode == ST_ZERO_X ? jb.x : jb.acc) + (long long)(tk.own0 + tk.row0) * RC;
                for (int e = l; ok && e < tk.nrows * RC / 2; e += 32) ((float4*)z)[e] = make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
        ok = block_and(ok);   // all of the block's warps are through, or leave together
        if (!ok) break;
        if (t == 0 && ph + 1 < nph) {
            __threadfence();
            atomicAdd(sync, 1u);
        }
    }
    if (!ok) *abort = 1;
    // copies still in flight land before the block's shared memory goes, whoever gave up
    asm volatile("cp.async.wait_all;" ::: "memory");
    int no_abort = 0;
    for (; u < ts.q; ++u) mbar_wait(smem_u32(ts.full + u % LY::SLOTS), (u / LY::SLOTS) & 1, &no_abort);
    __syncthreads();
    if (t == 0) {
        if (!ok) atomicExch(flag, 1);
        __threadfence();
        if (atomicAdd(sync + 1, 1u) == G - 1) {   // the last block out; nobody polls any more
            sync[0] = 0;
            sync[1] = 0;
            __threadfence();
        }
    }
}

template <int RC> void launch_rc(const StreamPlan& p, const void* jobs, unsigned* sync, int* flag, long long polls, cudaStream_t st) {
    const STask* tasks = (const STask*)p.d_tasks;
    const int* off = p.d_off;
    int nph = p.nph;
    const JobDev<float2>* jd = (const JobDev<float2>*)jobs;
    void* args[] = {&tasks, &off, &nph, &jd, &sync, &flag, &polls};
    HZ_CUDA(cudaLaunchCooperativeKernel((const void*)k_subst_stream<RC>, dim3(p.grid), dim3(32 * SW), args,
                                        (size_t)SLayout<RC>::TOTAL, st));
    HZ_CHECK_LAUNCH();
}

// The kernel's shared memory on the current device, and whether a launch of `grid` blocks fits there at
// once: by the occupancy, and by the launch itself (with no phases) where the context has fewer SMs than
// the device.  `zeros`: 128 cleared bytes (they are zero again afterwards).  Outside captures.
template <int RC> bool grid_fits(int grid, void* zeros, cudaStream_t st) {
    HZ_CUDA(cudaFuncSetAttribute(k_subst_stream<RC>, cudaFuncAttributeMaxDynamicSharedMemorySize, SLayout<RC>::TOTAL));
    int per_sm = 0;
    HZ_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_subst_stream<RC>, 32 * SW, SLayout<RC>::TOTAL));
    if (per_sm < 1) return false;
    const STask* tasks = (const STask*)zeros;
    const int* off = (const int*)zeros;
    int nph = 0;
    const JobDev<float2>* jd = nullptr;
    unsigned* sync = (unsigned*)zeros + 16;   // behind the one task that is read
    int* flag = (int*)zeros + 18;
    long long polls = 1;
    void* args[] = {&tasks, &off, &nph, &jd, &sync, &flag, &polls};
    const cudaError_t e = cudaLaunchCooperativeKernel((const void*)k_subst_stream<RC>, dim3(grid), dim3(32 * SW), args,
                                                      (size_t)SLayout<RC>::TOTAL, st);
    if (e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorNotSupported || e == cudaErrorNotPermitted) {
        cudaGetLastError();
        return false;
    }
    HZ_CUDA(e);
    HZ_CHECK_LAUNCH();
    HZ_CUDA(cudaStreamSynchronize(st));
    return true;
}

}  // namespace

bool stream_usable(int ldc) { return ldc >= 2 && ldc <= 16 && (ldc & (ldc - 1)) == 0; }

void launch_stream(const StreamPlan& p, const void* jobs, int ldc, unsigned* sync, int* flag, long long polls, cudaStream_t st) {
    if (p.nph == 0) return;
    switch (ldc) {
        case 2: launch_rc<2>(p, jobs, sync, flag, polls, st); break;
        case 4: launch_rc<4>(p, jobs, sync, flag, polls, st); break;
        case 8: launch_rc<8>(p, jobs, sync, flag, polls, st); break;
        case 16: launch_rc<16>(p, jobs, sync, flag, polls, st); break;
        default: throw Error{HZ_ERR_ARG, "stream substitution width"};
    }
}

// Phases, tasks and their warps for the active products `prods` (mode, level, node of a job).
StreamLists stream_lists(const Ctx& ctx, const std::vector<int>& layers, const std::vector<StreamProduct>& prods, int H,
                         int warps) {
    const int V = warps;
    // phase of a product: FB by level, FA, (clearing acc), BB, BA by level downwards
    const int PFA = std::max(1, H), PZ = PFA + 1, PBB = PFA + 2;
    std::vector<std::vector<const StreamProduct*>> phases(PBB + 1 + H);
    for (const auto& p : prods) {
        const int ph = p.mode == FB ? p.level : p.mode == FA ? PFA : p.mode == BB ? PBB : PBB + 1 + (H - 1 - p.level);
        phases[ph].push_back(&p);
    }
    std::vector<std::vector<STask>> ts(phases.size());
    for (size_t q = 0; q < phases.size(); ++q) {
        const auto& ph = phases[q];
        if (ph.empty()) continue;
        const int mode = ph[0]->mode;
        auto node = [&](const StreamProduct* p) -> const Node& {
            return ctx.shapes[ctx.layers[layers[p->job]].shape].nodes[p->node];
        };
        long long units = 0;
        for (auto* p : ph) {
            const Node& nd = node(p);
            units += (mode == FA || mode == BB) ? (long long)nd.own_t * (nd.own_t + 1) : 2LL * nd.own_t * nd.upd_t;
        }
        // reductions split so that every warp gets work: half a tile a task where the level is
        // narrow, up to 32 half tiles where it is wide
        const int ks = (int)std::max<long long>(1, std::min<long long>(32, (units + V - 1) / V));
        for (auto* p : ph) {
            const Node& nd = node(p);
            const int out_t = mode == FB ? nd.upd_t : nd.own_t, nout = mode == FB ? nd.nupd : nd.nown;
            const int red = mode == BA ? nd.nupd : nd.nown;
            for (int o = 0; o < out_t; ++o) {
                STask s{};
                s.mode = mode;
                s.job = p->job;
                s.upd_off = nd.upd_off;
                s.own0 = nd.own0;
                s.row0 = o * TILE;
                s.nrows = std::min(TILE, nout - s.row0);
                const int rb = mode == BB ? o * TILE : 0, re = mode == FA ? std::min(red, (o + 1) * TILE) : red;
                const int ub = rb / KU, ue = (re + KU - 1) / KU;
                // whole reductions of FA and BB are stored: worth up to 8 half tiles in one warp
                const bool whole = (mode == FA || mode == BB) && ue - ub <= std::max(8, ks);
                const int len = whole ? ue - ub : ks;
                s.store = whole;
                if ((mode == FA || mode == BB) && !whole) {
                    STask z = s;
                    z.mode = mode == FA ? ST_ZERO_X : ST_ZERO_ACC;
                    ts[mode == FA ? 0 : PZ].push_back(z);
                }
                for (int k = ub; k < ue; k += len) {
                    s.nunits = std::min(len, ue - k);
                    s.half0 = k & 1;
                    s.k0 = k * KU;
                    s.nk = re - s.k0;
                    const long long kt = k / 2;
                    if (mode == FA) { s.tile0 = nd.linv_off + (long long)o * (o + 1) / 2 + kt; s.step = 1; s.dstep = 0; }
                    else if (mode == FB) { s.tile0 = nd.l21_off + (long long)o * nd.own_t + kt; s.step = 1; s.dstep = 0; }
                    else if (mode == BA) { s.tile0 = nd.l21_off + kt * nd.own_t + o; s.step = nd.own_t; s.dstep = 0; }
                    else { s.tile0 = nd.linv_off + kt * (kt + 1) / 2 + o; s.step = (int)kt + 1; s.dstep = 1; }
                    ts[q].push_back(s);
                }
            }
        }
    }
    std::vector<std::vector<std::vector<STask>>> dealt;   // [phase][warp]
    for (auto& ph : ts) {
        if (ph.empty()) continue;
        std::stable_sort(ph.begin(), ph.end(), [](const STask& a, const STask& c) { return a.nunits > c.nunits; });
        // longest first to the least loaded warp (warp v in block v % grid, so the first `grid` tasks go
        // to different SMs); a task's fixed cost counts as two half tiles
        dealt.emplace_back(V);
        std::priority_queue<std::pair<long long, int>, std::vector<std::pair<long long, int>>, std::greater<>> load;
        for (int g = 0; g < V; ++g) load.push({0, g});
        for (const STask& s : ph) {
            auto [ld, g] = load.top();
            load.pop();
            dealt.back()[g].push_back(s);
            load.push({ld + s.nunits + 2, g});
        }
    }
    StreamLists out;   // by warp, then phase: a warp walks one contiguous list
    for (int g = 0; g < V; ++g)
        for (const auto& ph : dealt) {
            out.off.push_back((int)out.tasks.size());
            out.tasks.insert(out.tasks.end(), ph[g].begin(), ph[g].end());
        }
    out.off.push_back((int)out.tasks.size());
    out.tasks.push_back(STask{});   // read ahead, never run
    out.nph = (int)dealt.size();
    return out;
}

bool stream_fits(const Ctx& ctx, int ldc) {
    int coop = 0, sms = 0;
    HZ_CUDA(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, ctx.device));
    HZ_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx.device));
    if (!coop) return false;
    void* zeros = ctx.d_flag + Ctx::FLAG_ZEROS;
    if (ldc == 2) return grid_fits<2>(sms, zeros, ctx.stream);
    if (ldc == 4) return grid_fits<4>(sms, zeros, ctx.stream);
    if (ldc == 8) return grid_fits<8>(sms, zeros, ctx.stream);
    return grid_fits<16>(sms, zeros, ctx.stream);
}

void build_stream(const Ctx& ctx, const std::vector<int>& layers, const std::vector<StreamProduct>& prods, int H,
                  StreamPlan& plan) {
    int sms = 0;
    HZ_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx.device));
    const StreamLists ls = stream_lists(ctx, layers, prods, H, sms * SW);
    plan.nph = ls.nph;
    plan.grid = sms;
    auto up = [&](const void* src, size_t bytes) -> void* {
        void* d = nullptr;
        if (cudaMalloc(&d, std::max<size_t>(16, bytes)) != cudaSuccess) {
            cudaGetLastError();
            throw Error{HZ_ERR_OOM, "substitution task lists"};
        }
        HZ_CUDA(cudaMemcpyAsync(d, src, bytes, cudaMemcpyHostToDevice, ctx.stream));
        HZ_CUDA(cudaStreamSynchronize(ctx.stream));
        return d;
    };
    plan.d_tasks = up(ls.tasks.data(), ls.tasks.size() * sizeof(STask));
    plan.d_off = (int*)up(ls.off.data(), ls.off.size() * sizeof(int));
}

}  // namespace hz
