// Walks every task of the substitution's and the factorization's work lists for one problem on the host
// and checks that it stays inside its arrays: factor tiles inside the node's, vector rows and update
// indices inside the slot, cleared rows inside the vector, and that the tasks of a product cover each of
// its tile pairs exactly once.  Arguments: nx ny nz npml layers leaf.  Prints the counts, or the first
// fault with status 1.
#include <cstdio>
#include <cstdlib>
#include <map>
#include <set>

#include "hz_internal.cuh"
#include "hz_ctx.cuh"
#include "hz_solve.cuh"
#include "subst_items.cuh"

using namespace hz;
using tcc::FA;
using tcc::FB;
using tcc::BA;
using tcc::BB;

static std::string where;
static long long n_stages = 0, n_units = 0, n_tasks = 0;

#define CHECK(cond)                                                                          \
    do {                                                                                     \
        if (!(cond)) {                                                                       \
            std::printf("%s:%d: %s [%s]\n", __FILE__, __LINE__, #cond, where.c_str());       \
            std::exit(1);                                                                    \
        }                                                                                    \
    } while (0)

static const Shape& shape_of(const Ctx& c, int layer) { return c.shapes[c.layers[layer].shape]; }

// reduction tiles that output tile o of a node product needs: [lo, hi)
static int red_lo(int mode, int o) { return mode == BB ? o : 0; }
static int red_hi(int mode, const Node& nd, int o) { return mode == FA ? o + 1 : mode == BA ? nd.upd_t : nd.own_t; }
static int out_tiles(int mode, const Node& nd) { return mode == FB ? nd.upd_t : nd.own_t; }

// the stored tile of (output tile o, reduction tile k), and whether an offset is one of the node's
static long long tile_of(int mode, const Node& nd, int o, int k) {
    if (mode == FA) return nd.linv_off + tcc::tri_idx(o, k);
    if (mode == FB) return nd.l21_off + (long long)o * nd.own_t + k;
    if (mode == BA) return nd.l21_off + (long long)k * nd.own_t + o;
    return nd.linv_off + tcc::tri_idx(k, o);
}
static bool owns_tile(int mode, const Node& nd, long long t) {
    if (mode == FA || mode == BB) return t >= nd.linv_off && t < nd.linv_off + (long long)nd.own_t * (nd.own_t + 1) / 2;
    return t >= nd.l21_off && t < nd.l21_off + (long long)nd.own_t * nd.upd_t;
}

using Key = std::array<int, 3>;                       // job, node, mode
struct Cover { std::vector<int> n; std::vector<char> whole; };   // per (o, k); per o: stored by one task

static Cover& cover(std::map<Key, Cover>& cov, int job, int node, int mode, const Node& nd) {
    Cover& c = cov[{job, node, mode}];
    if (c.n.empty()) {
        c.n.assign((size_t)out_tiles(mode, nd) * std::max({1, nd.own_t, nd.upd_t}), 0);
        c.whole.assign(out_tiles(mode, nd), 0);
    }
    return c;
}

static void check_node(const Shape& sh, const Node& nd) {
    CHECK(nd.own0 >= 0 && nd.nown > 0 && nd.own0 + (long long)nd.nown <= sh.N);
    CHECK(nd.upd_off >= 0 && nd.upd_off + nd.nupd <= (long long)sh.upd_idx.size());
    CHECK(nd.own_t == cdiv(nd.nown, TILE) && nd.upd_t == cdiv(nd.nupd, TILE));
    CHECK(nd.linv_off >= 0 && nd.linv_off + (long long)nd.own_t * (nd.own_t + 1) / 2 <= sh.factor_tiles);
    CHECK(nd.l21_off >= 0 && nd.l21_off + (long long)nd.own_t * nd.upd_t <= sh.factor_tiles);
    for (int i = 0; i < nd.nupd; ++i) {
        const int u = sh.upd_idx[nd.upd_off + i];
        CHECK(u >= nd.own0 + nd.nown && u < sh.N);   // ancestors come later in the elimination
    }
}

// every active product covered exactly once (sparse == 0: all of them active)
static void check_cover(const Ctx& c, const std::vector<int>& layers, int nblk, int sparse, bool m21,
                        std::map<Key, Cover>& cov) {
    for (auto& kv : cov) {
        const Node& nd = shape_of(c, layers[kv.first[0] / nblk]).nodes[kv.first[1]];
        const int mode = kv.first[2], w = std::max({1, nd.own_t, nd.upd_t});
        for (int o = 0; o < out_tiles(mode, nd); ++o)
            for (int k = 0; k < w; ++k) {
                const bool need = k >= red_lo(mode, o) && k < red_hi(mode, nd, o);
                CHECK(kv.second.n[(size_t)o * w + k] == (need ? 1 : 0));
            }
    }
    if (sparse) return;
    for (int j = 0; j < (int)layers.size(); ++j) {
        const Shape& sh = shape_of(c, layers[j]);
        for (int n = 0; n < (int)sh.nodes.size(); ++n)
            for (int mode = 0; mode < 4; ++mode) {
                const Node& nd = sh.nodes[n];
                const bool any = out_tiles(mode, nd) > 0 && !(m21 && mode == BA && nd.nupd == 0);
                CHECK(cov.count({j, n, mode}) == (any ? 1u : 0u));
            }
    }
}

// host stand-ins for the device arrays of a batch; addresses are formed, never read
struct HostJobs {
    std::vector<std::vector<NodeDev>> nodes;
    std::vector<JobDev<float2>> jobs;
    HostJobs(const Ctx& c, const std::vector<int>& layers, int nblk) {
        for (auto& sh : c.shapes) {
            std::vector<NodeDev> v;
            for (auto& nd : sh.nodes) v.push_back({nd.own0, nd.nown, nd.nupd, nd.own_t, nd.upd_t, 0, nd.upd_off, nd.linv_off, nd.l21_off});
            nodes.push_back(v);
        }
        for (int l : layers)
            for (int q = 0; q < nblk; ++q) {
                JobDev<float2> j{};
                j.fac = (const float2*)(uintptr_t)(1ull << 40);
                j.nodes = nodes[c.layers[l].shape].data();
                j.upd_idx = shape_of(c, l).upd_idx.data();
                jobs.push_back(j);
            }
    }
};

// one tensor-core item as the loaders and the epilogue walk it
template <int NT, int MODE>
static void walk_item(const Ctx& c, const std::vector<int>& layers, const HostJobs& hj, const Task& tk, int ldc, int width,
                      int nblk, std::map<Key, Cover>& cov) {
    const Shape& sh = shape_of(c, layers[tk.job / nblk]);
    const Node& nd = sh.nodes[tk.node];
    const int nchunks = width / NT;
    CHECK(width % NT == 0 && nchunks >= 1 && tk.klen > 0 && tk.tile >= 0 && tk.tile < out_tiles(MODE, nd));
    Cover& cv = cover(cov, tk.job, tk.node, MODE, nd);
    const int w = std::max({1, nd.own_t, nd.upd_t});
    for (int chunk = 0; chunk < nchunks; chunk += std::max(1, nchunks - 1)) {
        const tcc::Item it = tcc::decode<NT, MODE>(&tk, hj.jobs.data(), chunk, nchunks);
        CHECK(it.col0 + NT <= width && it.nst == 2 * tk.klen);
        for (int t = 0; t < tcc::NLOAD; t += 16) {   // every vector row of a stage, first and last tile piece
            tcc::TilePtrs<MODE> tp;
            tp.init(it, t);
            const int thr = tcc::TilePtrs<MODE>::TR ? (t >> 3) * 256 + (t & 7) * 16 : t * 16;
            for (int s = 0; s < it.nst + 2; ++s) {   // the look-ahead reaches two stages past the end
                const tcc::Vrows<NT> v = tcc::stage_rows<NT, MODE>(it, s, t);
                for (int r : v.r) CHECK(r >= -1 && r < sh.N);
                if (s >= it.nst) continue;
                ++n_stages;
                for (int oi = 0; oi < 4; ++oi) {
                    if (!tp.exists(oi)) continue;
                    const long long byte = tp.p[oi] - thr - (const char*)it.jb.fac;
                    CHECK(byte % (TILE2 * 8) == 0 && byte / (TILE2 * 8) == tile_of(MODE, nd, it.o0 + oi, tp.kt));
                    CHECK(owns_tile(MODE, nd, byte / (TILE2 * 8)));
                    if (chunk == 0 && t == 0 && !(s & 1)) cv.n[(size_t)(it.o0 + oi) * w + tp.kt]++;
                }
                if (s & 1) tp.next();
            }
        }
        for (int r = 0; r < tcc::MR; ++r) {
            const long long b = tcc::row_base<MODE>(it, r, ldc);
            CHECK(b >= -1 && (b < 0 || b + NT <= sh.N * (long long)ldc));
            CHECK((b >= 0) == (it.o0 * TILE + r < it.nrows_out));
        }
        if (it.unique)
            for (int oi = 0; oi < 4 && it.o0 + oi < it.nout_t; ++oi) cv.whole[it.o0 + oi] = 1;
    }
}

template <int NT>
static void walk_mode(const Ctx& c, const std::vector<int>& layers, const HostJobs& hj, const Task& tk, int mode, int ldc,
                      int width, int nblk, std::map<Key, Cover>& cov) {
    if (mode == FA) walk_item<NT, FA>(c, layers, hj, tk, ldc, width, nblk, cov);
    else if (mode == FB) walk_item<NT, FB>(c, layers, hj, tk, ldc, width, nblk, cov);
    else if (mode == BA) walk_item<NT, BA>(c, layers, hj, tk, ldc, width, nblk, cov);
    else walk_item<NT, BB>(c, layers, hj, tk, ldc, width, nblk, cov);
}

static void check_lists(const Ctx& c, const std::vector<int>& layers, size_t elem, int ncols, int KS, bool tc, int KS_tc,
                        int min_t, int sparse) {
    const bool dbl = elem == 16;
    const int ldc = padded_ldc(dbl, ncols), nblk = block_count(sparse);
    const int width = nblk > 1 ? ncols / nblk : ldc;
    const BatchLists ls = batch_lists(c, layers, elem, KS, tc, KS_tc, min_t, sparse, false);
    const HostJobs hj(c, layers, nblk);
    std::map<Key, Cover> cov;
    std::set<std::array<int, 3>> cleared;   // layer position, x, own0
    for (const ZeroRows& z : ls.zero) {
        const Shape& sh = shape_of(c, layers[z.layer]);
        CHECK(z.own0 >= 0 && z.nown > 0 && z.own0 + (long long)z.nown <= sh.N);
        cleared.insert({z.layer, z.x, z.own0});
    }
    for (int mode = 0; mode < 4; ++mode)
        for (int h = 0; h < ls.H; ++h) {
            for (const Task& tk : ls.lists[mode][h]) {
                ++n_tasks;
                CHECK(tk.job >= 0 && tk.job < (int)layers.size() * nblk);
                const Shape& sh = shape_of(c, layers[tk.job / nblk]);
                CHECK(tk.node >= 0 && tk.node < (int)sh.nodes.size());
                const Node& nd = sh.nodes[tk.node];
                CHECK(tk.tile >= 0 && tk.tile < out_tiles(mode, nd));
                if (elem == 16 || mode == FB || mode == BA) CHECK(nd.height == h);
                CHECK(tk.klen > 0 || (mode == BA && nd.nupd == 0));
                Cover& cv = cover(cov, tk.job, tk.node, mode, nd);
                for (int k = tk.k0; k < tk.k0 + tk.klen; ++k) {
                    CHECK(k >= red_lo(mode, tk.tile) && k < red_hi(mode, nd, tk.tile));
                    CHECK(owns_tile(mode, nd, tile_of(mode, nd, tk.tile, k)));
                    cv.n[(size_t)tk.tile * std::max({1, nd.own_t, nd.upd_t}) + k]++;
                }
                if (tk.k0 == red_lo(mode, tk.tile) && tk.k0 + tk.klen == red_hi(mode, nd, tk.tile)) cv.whole[tk.tile] = 1;
            }
            for (const Task& tk : ls.quads[mode][h]) {
                ++n_tasks;
                CHECK(tc && tk.job >= 0 && tk.job < (int)layers.size() * nblk);
                const Shape& sh = shape_of(c, layers[tk.job / nblk]);
                CHECK(tk.node >= 0 && tk.node < (int)sh.nodes.size());
                if (mode == FB || mode == BA) CHECK(sh.nodes[tk.node].height == h);
                const int nt = tc_columns(width);
                if (nt == 128) walk_mode<128>(c, layers, hj, tk, mode, ldc, width, nblk, cov);
                else if (nt == 64) walk_mode<64>(c, layers, hj, tk, mode, ldc, width, nblk, cov);
                else { CHECK(nt == 32); walk_mode<32>(c, layers, hj, tk, mode, ldc, width, nblk, cov); }
            }
        }
    check_cover(c, layers, nblk, sparse, !dbl, cov);
    if (dbl) return;   // whole vectors are cleared
    for (auto& kv : cov) {   // rows of a split reduction are added into, so they are cleared
        const int mode = kv.first[2], j = kv.first[0] / nblk;
        if (mode == FB || mode == BA) continue;
        for (char whole : kv.second.whole)
            if (!whole) CHECK(cleared.count({j, mode == FA, shape_of(c, layers[j]).nodes[kv.first[1]].own0}) == 1);
    }
}

static void check_stream(const Ctx& c, const std::vector<int>& layers, int sparse, int warps) {
    const BatchLists ls = batch_lists(c, layers, 8, 0, false, 1 << 30, 0, sparse, true);
    const StreamLists st = stream_lists(c, layers, ls.prods, ls.H, warps);
    CHECK((long long)st.off.size() == (long long)warps * st.nph + 1 && st.off[0] == 0);
    CHECK((size_t)st.off.back() + 1 == st.tasks.size());   // one task of padding, read ahead
    std::map<Key, Cover> cov;                              // per half tile of the reduction
    std::map<std::array<int, 4>, int> writer, zeroed;      // job, x, first row, rows -> phase
    std::map<std::array<int, 3>, std::set<int>> phase;     // job, node, mode -> phases
    std::vector<std::map<int, int>> node_at(c.shapes.size());   // own0 -> node
    for (size_t s = 0; s < c.shapes.size(); ++s)
        for (size_t n = 0; n < c.shapes[s].nodes.size(); ++n) node_at[s][c.shapes[s].nodes[n].own0] = (int)n;
    for (int g = 0; g < warps; ++g)
        for (int ph = 0; ph < st.nph; ++ph) {
            const size_t o = (size_t)g * st.nph + ph;
            CHECK(st.off[o] <= st.off[o + 1]);
            for (int i = st.off[o]; i < st.off[o + 1]; ++i) {
                const STask& tk = st.tasks[i];
                CHECK(tk.job >= 0 && tk.job < (int)layers.size());
                const Layer& ly = c.layers[layers[tk.job]];
                const Shape& sh = c.shapes[ly.shape];
                CHECK(node_at[ly.shape].count(tk.own0) == 1);
                const int n = node_at[ly.shape][tk.own0];
                const Node& nd = sh.nodes[n];
                CHECK(tk.upd_off == nd.upd_off && tk.row0 >= 0 && tk.row0 % TILE == 0 && tk.nrows > 0 && tk.nrows <= TILE);
                if (tk.mode == ST_ZERO_ACC || tk.mode == ST_ZERO_X) {
                    CHECK(tk.nunits == 0 && tk.row0 + tk.nrows <= nd.nown);
                    CHECK(zeroed.insert({{tk.job, tk.mode == ST_ZERO_X, tk.own0 + tk.row0, tk.nrows}, ph}).second);
                    continue;
                }
                const int mode = tk.mode, slab = tk.row0 / TILE, nout = mode == FB ? nd.nupd : nd.nown;
                const int red = mode == BA ? nd.nupd : nd.nown;
                CHECK(tk.row0 + tk.nrows == std::min(nout, (slab + 1) * TILE));
                CHECK(tk.nunits > 0 && tk.k0 % SKU == 0 && tk.half0 == ((tk.k0 / SKU) & 1) && tk.nk > 0);
                CHECK(tk.k0 + tk.nk <= red);
                phase[{tk.job, n, mode}].insert(ph);
                Cover& cv = cov[{tk.job, n, mode}];
                const int w = 2 * std::max(nd.own_t, nd.upd_t);
                cv.n.resize((size_t)out_tiles(mode, nd) * w);
                long long tile = tk.tile0, step = tk.step;
                int half = tk.half0;
                for (int j = 0; j < tk.nunits; ++j) {   // as a warp's tile stream advances
                    ++n_units;
                    const int k = tk.k0 / SKU + j;
                    CHECK(half == (k & 1) && tile == tile_of(mode, nd, slab, k / 2) && owns_tile(mode, nd, tile));
                    CHECK(k * SKU < red);                // a step has at least one reduction row
                    cv.n[(size_t)slab * w + k]++;
                    if (half) { tile += step; step += tk.dstep; }
                    half ^= 1;
                }
                if (mode == FA || mode == BB) {
                    const std::array<int, 4> rows{tk.job, mode == FA, tk.own0 + tk.row0, tk.nrows};
                    if (tk.store) CHECK(writer.insert({rows, ph}).second && !zeroed.count(rows));
                    else writer[rows] = ph;
                }
            }
        }
    for (auto& kv : cov) {
        const Node& nd = shape_of(c, layers[kv.first[0]]).nodes[kv.first[1]];
        const int mode = kv.first[2], w = 2 * std::max(nd.own_t, nd.upd_t);
        const int red = mode == BA ? nd.nupd : nd.nown;
        for (int o = 0; o < out_tiles(mode, nd); ++o)
            for (int k = 0; k < w; ++k) {
                const bool need = k / 2 >= red_lo(mode, o) && k / 2 < red_hi(mode, nd, o) && k * SKU < red;
                CHECK(kv.second.n[(size_t)o * w + k] == (need ? 1 : 0));
            }
        CHECK((phase[{kv.first[0], kv.first[1], mode}].size() == 1));
    }
    auto at = [&](int j, int n, int mode, int none) {
        auto it = phase.find({j, n, mode});
        return it == phase.end() ? none : *it->second.begin();
    };
    int fa = -1, bb = -1;
    for (auto& kv : phase) {
        if (kv.first[2] == FA) { CHECK(fa < 0 || fa == *kv.second.begin()); fa = *kv.second.begin(); }
        if (kv.first[2] == BB) { CHECK(bb < 0 || bb == *kv.second.begin()); bb = *kv.second.begin(); }
    }
    for (int j = 0; j < (int)layers.size(); ++j) {
        const Shape& sh = shape_of(c, layers[j]);
        for (int n = 0; n < (int)sh.nodes.size(); ++n) {
            const int p = sh.nodes[n].parent;
            if (p >= 0) {   // updates go up a level at a time, gathers come down one
                CHECK(at(j, n, FB, -1) < at(j, p, FB, 1 << 30));
                CHECK(at(j, n, BA, 1 << 30) > at(j, p, BA, -1));
            }
            if (fa >= 0) CHECK(at(j, n, FB, -1) < fa && at(j, n, BA, 1 << 30) > bb && fa < bb);
            if (!sparse)
                for (int mode = 0; mode < 4; ++mode)
                    CHECK(cov.count({j, n, mode}) == (((mode == FA || mode == BB) || sh.nodes[n].nupd > 0) ? 1u : 0u));
        }
    }
    for (auto& kv : zeroed) {   // cleared before they are added into; acc not before FA has read it
        CHECK(writer.count(kv.first) == 1 && kv.second < writer[kv.first]);
        if (!kv.first[1]) CHECK(kv.second > fa);
    }
    std::map<std::array<int, 4>, int> stored;
    for (size_t i = 0; i + 1 < st.tasks.size(); ++i) {
        const STask& tk = st.tasks[i];
        if ((tk.mode == FA || tk.mode == BB) && !tk.store) {
            const std::array<int, 4> rows{tk.job, tk.mode == FA, tk.own0 + tk.row0, tk.nrows};
            CHECK(zeroed.count(rows) == 1);
        }
    }
}

// the three products of the tensor-core fronts: every tile and front element that a loader or the
// epilogue touches, by the conditions of the kernel
static void check_front_items(const Ctx& c, int min_upd) {
    for (const Shape& sh : c.shapes)
        for (auto& level : sh.levels) {
            std::vector<FrontGemmDesc> fr;
            for (int n : level) {
                const Node& nd = sh.nodes[n];
                if (!front_gemm_eligible(nd.nown, nd.nupd, min_upd)) continue;
                FrontGemmDesc g{};
                g.linv_off = nd.linv_off;
                g.l21_off = nd.l21_off;
                g.m = nd.m; g.nown = nd.nown; g.nupd = nd.nupd; g.own0 = nd.own0;
                g.own_t = nd.own_t; g.upd_t = nd.upd_t;
                fr.push_back(g);
            }
            std::vector<GemmItem> items[3];
            front_gemm_items(fr, items[0], items[1], items[2]);
            for (int mode = 0; mode < 3; ++mode)
                for (const GemmItem& it : items[mode]) {
                    CHECK(it.front >= 0 && it.front < (int)fr.size() && it.nst > 0 && it.nst % 2 == 0);
                    const FrontGemmDesc& f = fr[it.front];
                    const long long linv1 = f.linv_off + (long long)f.own_t * (f.own_t + 1) / 2;
                    const long long l211 = f.l21_off + (long long)f.own_t * f.upd_t;
                    CHECK(it.ti >= 0 && it.ti * 128 < f.nupd && it.tj >= 0 && it.tj * 128 < (mode == 1 ? f.nupd : f.nown));
                    for (int s = 0; s < it.nst; s += 2) {
                        ++n_stages;
                        const int kt = s / 2 + (mode == 2 ? it.tj * 4 : 0);
                        CHECK(kt < f.own_t);
                        for (int oi = 0; oi < 4; ++oi) {
                            const int ra = it.ti * 4 + oi, rb = it.tj * 4 + oi;
                            if (mode != 0 && ra < f.upd_t) CHECK(f.l21_off + (long long)ra * f.own_t + kt < l211);
                            if (mode == 0 && rb < f.own_t && kt <= rb) CHECK(f.linv_off + tcc::tri_idx(rb, kt) < linv1);
                            if (mode == 1 && rb < f.upd_t) CHECK(f.l21_off + (long long)rb * f.own_t + kt < l211);
                            if (mode == 2 && rb < f.own_t && rb <= kt) CHECK(f.linv_off + tcc::tri_idx(kt, rb) < linv1);
                        }
                    }
                    if (mode == 2) CHECK(it.tj * 4 + it.nst / 2 == f.own_t);   // reduction up to the last own tile
                }
        }
}

int main(int argc, char** argv) {
    if (argc != 7) return 2;
    int a[6];
    for (int i = 0; i < 6; ++i) a[i] = std::atoi(argv[i + 1]);
    Ctx c;
    c.nx = a[0]; c.ny = a[1]; c.nz = a[2]; c.npml = c.npml_loc = a[3]; c.L = a[4];
    c.prec = HZ_PREC_MIXED;
    std::map<int, int> shape_of_nz;
    const int nphys = c.nz - 2 * c.npml, q = nphys / c.L, rem = nphys % c.L;
    for (int l = 0, start = c.npml; l < c.L; ++l) {   // the layers as the solver partitions them
        Layer ly;
        ly.lo = start;
        ly.hi = start + q + (l < rem) - 1;
        start = ly.hi + 1;
        if (l == 0) ly.lo = 0;
        if (l == c.L - 1) ly.hi = c.nz - 1;
        ly.zlo = l > 0 ? ly.lo - c.npml : ly.lo;
        ly.zhi = l < c.L - 1 ? ly.hi + c.npml : ly.hi;
        ly.nzl = ly.zhi - ly.zlo + 1;
        if (!shape_of_nz.count(ly.nzl)) {
            shape_of_nz[ly.nzl] = (int)c.shapes.size();
            Shape sh;
            build_shape(sh, c.nx, c.ny, ly.nzl, a[5]);
            for (const Node& nd : sh.nodes) check_node(sh, nd);
            c.shapes.push_back(std::move(sh));
        }
        ly.shape = shape_of_nz[ly.nzl];
        c.layers.push_back(ly);
    }
    std::vector<std::vector<int>> sets{{}};
    for (int l = 0; l < c.L; ++l) sets[0].push_back(l);
    if (c.L > 1) { sets.push_back({0}); sets.push_back({c.L - 1}); }
    if (c.L > 2) sets.push_back({c.L / 2});
    const int one_code[4] = {0, sparse_code(SP_TOP, SP_BOT), sparse_code(SP_BOT, SP_TOP), sparse_code(SP_BOTH, SP_BOTH)};
    const int blocks[4] = {sparse_code(SP_TOP, SP_BOT), sparse_code(SP_TOP, SP_BOTH), sparse_code(SP_BOT, SP_TOP), sparse_code(SP_BOT, SP_BOTH)};
    std::set<std::array<int, 7>> seen;
    for (auto& layers : sets)
        for (int code : one_code) {
            for (int warps : {8, 148 * 8, 152 * 8}) {
                where = "one launch, " + std::to_string(layers.size()) + " layers from " + std::to_string(layers[0]) + ", code " + std::to_string(code);
                check_stream(c, layers, code, warps);
            }
            for (int prec : {(int)HZ_PREC_MIXED, (int)HZ_PREC_MIXED_FP64_FACTOR, (int)HZ_PREC_FP64}) {
                c.prec = (hz_precision)prec;
                const size_t elem = prec == HZ_PREC_FP64 ? 16 : 8;
                for (int ncols : {1, 2, 3, 13, 16, 17, 33, 52, 64, 128, 192, 256}) {
                    auto cands = tune_candidates(c, elem == 16, ncols);
                    for (int ks : {8, 1 << 30}) cands.push_back({ks, 0, 0, 1 << 30, 0, 0});   // untuned
                    if (tc_columns(padded_ldc(elem == 16, ncols)) && elem == 8)
                        for (int ks : {4, 1 << 30}) cands.push_back({ks == 4 ? 8 : 1 << 30, 0, 1, ks, c.tc_min_tiles, 0});
                    for (auto& cd : cands) {
                        // the lists depend on the widths through the tile width alone
                        const int nt = cd.tc ? tc_columns(padded_ldc(false, ncols)) : 0;
                        if (!seen.insert({layers[0], (int)layers.size(), code, (int)elem, cd.tc ? cd.KS_tc : -1, cd.KS, nt * 100 + cd.min_t}).second) continue;
                        where = "prec " + std::to_string(prec) + ", " + std::to_string(ncols) + " columns, " + std::to_string(layers.size()) + " layers from " + std::to_string(layers[0]) + ", code " + std::to_string(code) + ", KS " + std::to_string(cd.KS) + "/" + std::to_string(cd.KS_tc) + ", tc " + std::to_string(cd.tc) + ", min " + std::to_string(cd.min_t);
                        check_lists(c, layers, elem, ncols, cd.KS, cd.tc != 0, cd.KS_tc, cd.min_t, code);
                    }
                }
            }
        }
    for (int ncols : {256, 512})   // four blocks of 64 and 128 columns with codes of their own
        for (int kst : {2, 16, 1 << 30}) {
            where = "blocks, " + std::to_string(ncols) + " columns, KS " + std::to_string(kst);
            check_lists(c, sets[0], 8, ncols, 8, true, kst, 2, blocked_code(4, blocks));
            check_lists(c, sets[0], 8, ncols, 1 << 30, false, 1 << 30, 0, blocked_code(4, blocks));
        }
    where = "route";   // a device that holds the grid at once takes the one launch, another the tuner's choice
    for (int ldc : {2, 4, 8, 16}) {
        c.one_launch_fits[ldc] = true;
        CHECK(use_one_launch(c, ldc, 0) && use_one_launch(c, ldc, one_code[1]));
        c.one_launch_fits[ldc] = false;
        CHECK(!use_one_launch(c, ldc, 0) && !tune_candidates(c, false, ldc).empty());
        c.one_launch_fits[ldc] = true;
        c.one_launch = false;
        CHECK(!use_one_launch(c, ldc, 0));
        c.one_launch = true;
    }
    for (int ldc : {1, 32, 64, 128}) CHECK(!use_one_launch(c, ldc, 0));
    where = "tuner";   // a minimum of output tiles that the caller set is timed, whatever its value
    for (int ncols : {17, 64, 128})
        for (int set : {1, 4, 8, 16}) {
            auto has = [&](int t) {
                for (auto& cd : tune_candidates(c, false, ncols))
                    if (cd.tc && cd.min_t == t) return true;
                return false;
            };
            c.prec = HZ_PREC_MIXED;
            c.tc_min_tiles = set;
            c.tc_min_set = true;
            CHECK(has(set) && has(2));
            c.tc_min_tiles = 8;
            c.tc_min_set = false;
            CHECK(!has(8) && has(2));
        }
    where = "fronts";
    for (int min_upd : {1, 128}) check_front_items(c, min_upd);
    std::printf("%lld tasks, %lld tensor-core stages, %lld half tiles\n", n_tasks, n_stages, n_units);
    return 0;
}
