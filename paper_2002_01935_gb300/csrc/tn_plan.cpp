// tn_plan.cpp -- node planning, workspace liveness and the per-call runtime
// of libtn.so.  See tn_api.cpp for the overview.
#include "tn_plan.h"

#include <algorithm>
#include <climits>
#include <cmath>
#include <cstring>
#include <cstdlib>
#include <map>
#include <tuple>

namespace tn {

namespace {

struct SubCount {
    std::vector<std::pair<int, int>> c;  // (label, leaves of the subtree holding it)
    int get(int l) const {
        for (auto& x : c)
            if (x.first == l) return x.second;
        return 0;
    }
};

int64_t stride_in(const std::vector<int>& lab, const std::vector<int64_t>& st, int l) {
    for (size_t i = 0; i < lab.size(); ++i)
        if (lab[i] == l) return st[i];
    return 0;
}

bool has(const std::vector<int>& v, int x) { return std::find(v.begin(), v.end(), x) != v.end(); }

// Best-fit workspace allocator over element offsets (liveness planning).
struct Arena {
    std::map<int64_t, int64_t> free_;  // offset -> length
    int64_t end = 0;
    static int64_t round(int64_t n) { return (n + 63) / 64 * 64; }
    int64_t alloc(int64_t n) {
        n = round(n);
        auto best = free_.end();
        for (auto it = free_.begin(); it != free_.end(); ++it)
            if (it->second >= n && (best == free_.end() || it->second < best->second)) best = it;
        if (best != free_.end()) {
            int64_t off = best->first, len = best->second;
            free_.erase(best);
            if (len > n) free_[off + n] = len - n;
            return off;
        }
        // extend, merging a free tail block
        if (!free_.empty()) {
            auto last = std::prev(free_.end());
            if (last->first + last->second == end) {
                int64_t off = last->first;
                free_.erase(last);
                end = off + n;
                return off;
            }
        }
        int64_t off = end;
        end += n;
        return off;
    }
    void release(int64_t off, int64_t n) {
        n = round(n);
        auto it = free_.emplace(off, n).first;
        auto nx = std::next(it);
        if (nx != free_.end() && it->first + it->second == nx->first) {
            it->second += nx->second;
            free_.erase(nx);
        }
        if (it != free_.begin()) {
            auto pv = std::prev(it);
            if (pv->first + pv->second == it->first) {
                pv->second += it->second;
                free_.erase(it);
            }
        }
    }
};

bool pow2(int64_t x) { return x >= 1 && (x & (x - 1)) == 0; }
int ilog2(int64_t x) {
    int r = 0;
    while ((int64_t(1) << r) < x) ++r;
    return r;
}

// Real nodes take 128 x 128 tiles (64 outputs per thread) where these alone
// give every SM one: 2^11 x 2^11 x 2^10 256 against 289 us with 64 x 64 tiles,
// 2^12 x 2^12 x 2^10 882 against 1055; with fewer tiles the smaller ones win
// (2^9 x 2^9 x 2^9: 39 against 30 us).  A complex thread tile of that size
// does not fit the registers.
bool large_real_tiles(const NetDesc& d, int64_t nbatch, int64_t M, int64_t N) {
    return !d.is_complex() && M >= 128 && N >= 128 && ((M + 127) / 128) * ((N + 127) / 128) * nbatch >= sm_count();
}

// An operand whose offsets reach 2^31 entries.  Labels of a sliced leaf keep
// the strides of the whole leaf, so that its slice may be small and yet
// spread over more than that.
bool wide_operand(const NetDesc& d, const Plan& p, int c) {
    if (c < 0) return false;
    double last = 0;
    for (size_t i = 0; i < p.vlab[c].size(); ++i) last += (double)(d.dims[p.vlab[c][i]] - 1) * (double)p.vstride[c][i];
    return last >= 2147483648.0;
}

// Inner-product nodes: one CTA per output (and K part) instead of one for all
// outputs.  tiles: 1024 products of one output.
//  - One output: always.
//  - Few tiles, two per SM: the outputs side by side are then faster than one
//    after the other (8 x 8 outputs over K = 2^9: 8.8 us against 17, 2 x 2 over
//    2^14 13 against 17; from 512 tiles on 17 to 20 either way or worse).
//  - One row (column) whose operand does not fit L2 and is contiguous along K
//    (at most 4 outputs or batch entries among 32 neighbours): it is read once
//    in either form, in whole lines here (64 outputs over K = 2^18, real, 67 MB:
//    54 us against 79; below 8192 tiles 1.2 to 3 times slower).
bool dot_each_output(const TileArgs& t, int copies) {
    if (t.nm + t.nn == 0) return true;
    const int64_t tiles = (t.nbatch << (t.nm + t.nn)) * copies * std::max<int64_t>(1, (int64_t(1) << t.nk) / 1024);
    if (tiles <= 2 * (int64_t)sm_count()) return true;
    if (std::min(t.nm, t.nn) > 0 || tiles < 8192) return false;
    const bool b = t.nm == 0;  // the operand that holds the outputs
    int low = 0;
    for (int i = 0; i < (b ? t.nn : t.nm); ++i) low += (b ? t.b_n : t.a_m)[i] < 5;
    for (int i = 0; i < t.nb; ++i) low += (b ? t.b_b : t.a_b)[i] < 5;
    return low <= 2;
}

// Tiled-kernel plan of a node whose labels and strides are all powers of
// two: index bits per group, K order, load directions, tile shape and K
// split.  Returns false (generic kernel) when a limit is exceeded.
bool plan_tile(const NetDesc& d, const Plan& p, Node& nd, int64_t& split_elems, int force_cfg = 0) {
    static const std::vector<int> none;
    static const std::vector<int64_t> nones;
    const std::vector<int>& la = nd.ca >= 0 ? p.vlab[nd.ca] : none;
    const std::vector<int>& lb = nd.cb >= 0 ? p.vlab[nd.cb] : none;
    const std::vector<int64_t>& sa = nd.ca >= 0 ? p.vstride[nd.ca] : nones;
    const std::vector<int64_t>& sb = nd.cb >= 0 ? p.vstride[nd.cb] : nones;
    for (size_t i = 0; i < la.size(); ++i)
        if (!pow2(d.dims[la[i]]) || !pow2(sa[i])) return false;
    for (size_t i = 0; i < lb.size(); ++i)
        if (!pow2(d.dims[lb[i]]) || !pow2(sb[i])) return false;
    TileArgs t;
    memset(&t, 0, sizeof(t));
    auto push = [&](uint8_t* arr, int& nbits, int l, int64_t stride) -> bool {
        const int j = ilog2(d.dims[l]);
        for (int r = 0; r < j; ++r) {
            if (nbits >= kMaxBits) return false;
            arr[nbits++] = stride ? (uint8_t)(ilog2(stride) + r) : kNoBit;
        }
        return true;
    };
    // batch, M, N: fastest label first (the lists are slowest first)
    int nb2 = 0;
    for (auto it = nd.gb.rbegin(); it != nd.gb.rend(); ++it) {
        int tmp = t.nb;
        if (!push(t.a_b, t.nb, *it, stride_in(la, sa, *it))) return false;
        if (!push(t.b_b, tmp, *it, stride_in(lb, sb, *it))) return false;
        nb2 = tmp;
    }
    (void)nb2;
    for (auto it = nd.gm.rbegin(); it != nd.gm.rend(); ++it)
        if (!push(t.a_m, t.nm, *it, stride_in(la, sa, *it))) return false;
    for (auto it = nd.gn.rbegin(); it != nd.gn.rend(); ++it)
        if (!push(t.b_n, t.nn, *it, stride_in(lb, sb, *it))) return false;
    // K (shared and summed-only labels): order by the stride of the operand
    // whose fastest label is a K label, so its loads stay contiguous
    std::vector<int> ks = nd.gk;
    ks.insert(ks.end(), nd.gsa.begin(), nd.gsa.end());
    ks.insert(ks.end(), nd.gsb.begin(), nd.gsb.end());
    auto fastest = [&](const std::vector<int>& lab, const std::vector<int64_t>& st) {
        int best = -1;
        int64_t bs = INT64_MAX;
        for (size_t i = 0; i < lab.size(); ++i)
            if (d.dims[lab[i]] > 1 && st[i] < bs) {
                bs = st[i];
                best = lab[i];
            }
        return best;
    };
    const int fa = fastest(la, sa), fb = fastest(lb, sb);
    const bool fa_k = fa >= 0 && has(ks, fa), fb_k = fb >= 0 && has(ks, fb);
    // K follows the strides of the operand that needs it for contiguous
    // loads; when both or neither do, the larger operand wins
    int64_t size_a = 1, size_b = 1;
    for (int l : la) size_a *= d.dims[l];
    for (int l : lb) size_b *= d.dims[l];
    const bool by_a = (fa_k && !fb_k) || (fa_k == fb_k && size_a > size_b);
    const int64_t big = INT64_MAX / 4;
    std::sort(ks.begin(), ks.end(), [&](int x, int y) {
        int64_t sx = by_a ? stride_in(la, sa, x) : stride_in(lb, sb, x);
        int64_t sy = by_a ? stride_in(la, sa, y) : stride_in(lb, sb, y);
        if (!sx) sx = big;
        if (!sy) sy = big;
        return sx < sy;
    });
    for (int l : ks) {
        int tmp = t.nk;
        if (!push(t.a_k, t.nk, l, stride_in(la, sa, l))) return false;
        if (!push(t.b_k, tmp, l, stride_in(lb, sb, l))) return false;
    }
    if (t.nb > 16 || t.nm > 31 || t.nn > 31 || t.nk > 40 || t.nm + t.nn > 40) return false;
    t.wide = wide_operand(d, p, nd.ca) || wide_operand(d, p, nd.cb);
    for (const std::vector<int>* lab : {&la, &lb}) {
        int64_t sz = 1;
        for (int l : *lab) sz *= d.dims[l];
        if (sz >= (int64_t(1) << 31)) return false;
    }
    t.nbatch = int64_t(1) << t.nb;
    t.a_mfast = fa >= 0 && has(nd.gm, fa);
    t.b_nfast = fb >= 0 && has(nd.gn, fb);
    const int64_t M = int64_t(1) << t.nm, N = int64_t(1) << t.nn, K = int64_t(1) << t.nk;
    int TM = 64, TN = 64, TK = 16;
    const bool dot = M * N <= 64 && K >= 512;
    if (force_cfg >= kTile64x64 && force_cfg <= kTile128x128 && force_cfg != kTileDot && !dot) {
        // a shape forced by the autotuner (any shape is valid: tiles clip)
        static const int shapes[8][3] = {{0, 0, 0},     {64, 64, 16}, {16, 256, 16}, {4, 1024, 4},
                                         {256, 16, 16}, {0, 0, 0},    {128, 64, 16}, {128, 128, 16}};
        t.cfg = force_cfg;
        TM = shapes[force_cfg][0];
        TN = shapes[force_cfg][1];
        TK = shapes[force_cfg][2];
    } else if (dot) {
        t.cfg = kTileDot;
        t.dot_each = t.wide || dot_each_output(t, p.copies);
        TM = (int)M;
        TN = (int)N;
    } else if (t.nm <= 2 && t.nn >= 10) {
        t.cfg = kTile4x1024;
        TM = 4;
        TN = 1024;
        TK = 4;
    } else if (t.nm <= 5 && t.nn >= 8) {  // 64-row tiles would run half empty at M = 32
        t.cfg = kTile16x256;
        TM = 16;
        TN = 256;
    } else if (t.nn <= 5 && t.nm >= 8) {
        t.cfg = kTile256x16;
        TM = 256;
        TN = 16;
    } else if (large_real_tiles(d, p.copies * t.nbatch, M, N)) {
        t.cfg = kTile128x128;
        TM = 128;
        TN = 128;
    } else {
        t.cfg = kTile64x64;
    }
    t.split = 1;
    t.kchunk = K;
    if (t.cfg != kTileDot) {
        const int64_t tiles = ((M + TM - 1) / TM) * ((N + TN - 1) / TN) * t.nbatch;
        const int64_t ktiles = (K + TK - 1) / TK;
        int split = 1;
        while (tiles * p.copies * split < 2 * sm_count() && split * 16 <= ktiles && split < 64 &&
               t.nbatch * split * 2 <= 65535)
            split *= 2;
        t.split = split;
        t.kchunk = ((ktiles + split - 1) / split) * TK;
        if (split > 1) split_elems = std::max(split_elems, (int64_t)split * t.nbatch * M * N);
    } else {
        if (t.nbatch > 65535) return false;
        const int64_t outs = M * N * t.nbatch;
        int split = 1;
        // a K tile (2^11 entries of both operands) or more per part, four where a
        // part reduces several outputs; at least eight parts (times outputs, with
        // a CTA each) per SM in all: several CTAs per SM keep enough loads in
        // flight for HBM.  4 x 4 outputs over 2^18 in eight slices: 161 us with
        // parts of one tile, 89 with four.
        const int64_t tiles = t.dot_each ? K >> dot_tile_bits(0, 0, t.nk) : (K >> dot_tile_bits(t.nm, t.nn, t.nk)) / 4;
        while ((t.dot_each ? outs : t.nbatch) * p.copies * split < 8 * (int64_t)sm_count() && split * 2 <= tiles && split < 4096 &&
               (int64_t)split * 2 * p.copies <= 65535)
            split *= 2;
        t.split = split;
        t.kchunk = ((K / split + 255) / 256) * 256;
        if (split > 1) split_elems = std::max(split_elems, (int64_t)split * outs);
    }
    t.a_leaf = nd.ca >= 0 && nd.ca < d.n ? nd.ca : -1;
    t.b_leaf = nd.cb >= 0 && nd.cb < d.n ? nd.cb : -1;
    nd.tile = t;
    nd.kind = kTiled;
    return true;
}

}  // namespace

// A node contracting vertices a and b (tree ids, -1 = the unit scalar) into
// the labels in keep: label groups and the [batch][M][N] output layout.
// The larger operand takes the B role (its labels are the fastest).
Node build_node(const NetDesc& d, const Plan& p, int id, int a, int b, const std::vector<int>& keep) {
    auto log2size = [&](const std::vector<int>& lab) {
        double s = 0;
        for (int l : lab) s += std::log2((double)d.dims[l]);
        return s;
    };
    // a, b: tree ids or -1 (unit scalar: no labels)
    static const std::vector<int> none;
    static const std::vector<int64_t> nones;
    const std::vector<int>& la = a >= 0 ? p.vlab[a] : none;
    const std::vector<int>& lb = b >= 0 ? p.vlab[b] : none;
    const std::vector<int64_t>& sa = a >= 0 ? p.vstride[a] : nones;
    const std::vector<int64_t>& sb = b >= 0 ? p.vstride[b] : nones;
    int64_t size_a = 1, size_b = 1;
    for (int l : la) size_a *= d.dims[l];
    for (int l : lb) size_b *= d.dims[l];
    // role: the larger operand takes the B (inner, fastest output) role
    bool swap = size_a > size_b;
    Node nd;
    nd.id = id;
    nd.ca = swap ? b : a;
    nd.cb = swap ? a : b;
    const std::vector<int>& A = swap ? lb : la;
    const std::vector<int>& B = swap ? la : lb;
    const std::vector<int64_t>& SA = swap ? sb : sa;
    const std::vector<int64_t>& SB = swap ? sa : sb;
    for (int l : A) {
        bool inb = has(B, l), kept = has(keep, l);
        if (inb && kept) nd.gb.push_back(l);
        else if (inb) nd.gk.push_back(l);
        else if (kept) nd.gm.push_back(l);
        else nd.gsa.push_back(l);
    }
    for (int l : B) {
        if (has(A, l)) continue;
        if (has(keep, l)) nd.gn.push_back(l);
        else nd.gsb.push_back(l);
    }
    auto by_desc = [&](const std::vector<int64_t>& S, const std::vector<int>& lab) {
        return [&](int x, int y) { return stride_in(lab, S, x) > stride_in(lab, S, y); };
    };
    std::sort(nd.gb.begin(), nd.gb.end(), by_desc(SA, A));
    std::sort(nd.gm.begin(), nd.gm.end(), by_desc(SA, A));
    std::sort(nd.gn.begin(), nd.gn.end(), by_desc(SB, B));
    std::sort(nd.gk.begin(), nd.gk.end(), by_desc(SB, B));
    nd.lab = nd.gb;
    nd.lab.insert(nd.lab.end(), nd.gm.begin(), nd.gm.end());
    nd.lab.insert(nd.lab.end(), nd.gn.begin(), nd.gn.end());
    nd.stride.assign(nd.lab.size(), 1);
    nd.size = 1;
    for (int i = (int)nd.lab.size() - 1; i >= 0; --i) {
        nd.stride[i] = nd.size;
        nd.size *= d.dims[nd.lab[i]];
    }
    std::vector<int> uni = A;
    for (int l : B)
        if (!has(uni, l)) uni.push_back(l);
    nd.vc = log2size(uni);
    return nd;
}

// The tile kernel for sizes of any kind.  The shape follows the rule of
// plan_tile (4 x 1024 up to 4 rows, 16 x 256 up to 32, 256 x 16 up to 32
// columns, else 64 x 64); the K split gives every SM a tile, each part at
// least 16 entries.  A node takes it where the estimates below say that it is
// faster than one thread per output: 3^14 multiply-adds 26 us against 19, 5^12
// 562 against 79, 7 x 5 outputs over K = 3^8 1809 against 28.  Tiles that
// batch labels leave nearly empty cost about 6 us a round of resident blocks
// all the same (3^9 entries of 3 x 3 outputs over K = 3: 275 us, 13 with one
// thread per output; 3^10 entries of one product each: 752 and 8), as do short
// sums of few outputs (9.6 us against 11-12 below 2^13 multiply-adds).
//
// Microseconds, fitted to nodes of 1 to 10^7 outputs over K = 1 to 3^10:
// rounds of resident blocks, each with its setup and its K steps ...
static double any_tile_us(const NetDesc& d, int cfg, double blocks, int64_t kchunk, int split) {
    const double slots = (cfg == kTile64x64 ? 3.0 : 2.0) * sm_count();
    const double steps = std::ceil((double)kchunk / (cfg == kTile4x1024 ? 4.0 : 8.0));
    return 3.5 + std::ceil(blocks / slots) * (6.0 + steps * (d.is_complex() ? 1.2 : 0.6)) + (split > 1 ? 6.0 : 0.0);
}
// ... and one thread's serial sum, or all products at the launch's rate.
static double any_generic_us(double outputs, double K) { return 7.0 + std::max(0.19 * K, outputs * (K + 3.0) / 220e3); }

void plan_any_tile(const NetDesc& d, const Plan& p, Node& nd, int64_t& split_elems, int copies) {
    nd.any_cfg = 0;
    nd.any_split = 1;
    auto volume = [&](std::initializer_list<const std::vector<int>*> groups) {
        double v = 1;
        for (auto* g : groups)
            for (int l : *g) v *= (double)d.dims[l];
        return v;
    };
    const double lim = 2147483648.0;  // the kernel's indices and offsets are 32-bit
    if (wide_operand(d, p, nd.ca) || wide_operand(d, p, nd.cb)) return;
    const double M = volume({&nd.gm}), N = volume({&nd.gn}), B = volume({&nd.gb}), K = volume({&nd.gk, &nd.gsa, &nd.gsb});
    const double size_a = volume({&nd.gb, &nd.gm, &nd.gk, &nd.gsa}), size_b = volume({&nd.gb, &nd.gn, &nd.gk, &nd.gsb});
    if (M * N * K * B < 8192.0 || std::max(std::max(size_a, size_b), std::max(K, std::max(M, N))) >= lim) return;
    int cfg = kTile64x64, TM = 64, TN = 64, TK = 16;
    if (M <= 4 && N >= 1024) {
        cfg = kTile4x1024;
        TM = 4;
        TN = 1024;
        TK = 4;
    } else if (M <= 32 && N >= 256) {
        cfg = kTile16x256;
        TM = 16;
        TN = 256;
    } else if (N <= 32 && M >= 256) {
        cfg = kTile256x16;
        TM = 256;
        TN = 16;
    } else if (large_real_tiles(d, (int64_t)B * copies, (int64_t)M, (int64_t)N)) {
        cfg = kTile128x128;
        TM = TN = 128;
    }
    const double tiles = std::ceil(M / TM) * std::ceil(N / TN) * B;
    if (B * copies > 65535 || std::ceil(M / TM) * std::ceil(N / TN) >= lim) return;  // launch grid limits
    const int64_t ktiles = ((int64_t)K + TK - 1) / TK;
    int split = 1;
    // (several CTAs share an SM: a split that only fills the second one costs
    // more in its reduction -- 270 tiles over K = 180: 68 + 21 us in two parts)
    while (tiles * copies * split < sm_count() && split * 2 <= ktiles && split < 64 &&
           B * split * 2 * copies <= 65535)
        split *= 2;
    const int64_t kchunk = ((ktiles + split - 1) / split) * TK;
    if (any_tile_us(d, cfg, tiles * copies * split, std::min(kchunk, (int64_t)K), split) >=
        any_generic_us(M * N * B * copies, K))
        return;
    nd.any_cfg = cfg;
    nd.any_kchunk = kchunk;
    nd.any_split = (int)(((int64_t)K + nd.any_kchunk - 1) / nd.any_kchunk);  // no empty part
    if (nd.any_split > 1) split_elems = std::max(split_elems, (int64_t)nd.any_split * (int64_t)(B * M * N));
}

// Work items of a node in the persistent launch (per instance).
static int64_t persistent_items(const Node& nd) {
    if (nd.tile.cfg == kTile64x64 && tile_item_node(nd)) {
        const int64_t M = int64_t(1) << nd.tile.nm, N = int64_t(1) << nd.tile.nn;
        return ((M + 63) / 64) * ((N + 63) / 64) * nd.tile.nbatch;
    }
    const int64_t chunk = wave_chunk(nd, 2);
    return (nd.size + chunk - 1) / chunk;
}

static tn_status fill_generic(const NetDesc& d, const Plan& p, const Node& nd, GenericArgs& g, std::string& err);

// ---- subtree regions (tn_region.cu)

// Small enough for a region: at most 2^14 multiply-adds (64 per thread of a
// 256-thread block, 32 of a 512-thread one: about a microsecond; waves spread
// larger ones over the GPU) and 2^10 outputs, operands that can be staged.  Sizes of other kinds: the nodes that would take a
// launch of one thread per output each.
static bool region_node(const RegionView& v, const Node& nd) {
    const NetDesc& d = *v.d;
    if (nd.size > 1024 || nd.vc > 14.0 || nd.ca < 0 || nd.cb < 0) return false;
    for (int c : {nd.ca, nd.cb})
        if (v.operand(c).size > (c < d.n ? 256 : 1024)) return false;
    if (nd.kind == kTiled) return wave_node(nd, v.copies);
    if (nd.kind != kGeneric || nd.any_cfg) return false;
    double k = 1;
    for (const std::vector<int>* g : {&nd.gk, &nd.gsa, &nd.gsb})
        for (int l : *g) k *= (double)d.dims[l];
    return k <= 64;
}

static int64_t region_k(const NetDesc& d, const Node& nd) {
    int64_t k = 1;
    for (const std::vector<int>* g : {&nd.gk, &nd.gsa, &nd.gsb})
        for (int l : *g) k *= d.dims[l];
    return k;
}

// Connected pieces of region nodes, bottom up: a node joins its children's
// pieces while the union fits one CTA's shared memory, program and 2^16
// multiply-adds (a few microseconds).  Pieces of fewer than four nodes stay
// with the waves.  (An adjoint node joins its parent adjoint's piece: that is
// the operand of its own list.)
void find_regions(const RegionView& v, int k0, int k1, std::vector<int>& of, std::vector<std::vector<int>>& regions) {
    const NetDesc& d = *v.d;
    struct Size {
        int64_t out = 0, elems = 0, macs = 0, words = 0;
        int nodes = 0, ext = 0;
    };
    std::vector<Size> size;
    std::vector<std::vector<int>> members;
    std::vector<int> mine(k1 - k0, -1);  // piece of each node so far
    for (int k = k0; k < k1; ++k) {
        const Node& nd = v.node(k);
        if (!region_node(v, nd)) continue;
        const int64_t K = region_k(d, nd);
        const RegionOperand op[2] = {v.operand(nd.ca), v.operand(nd.cb)};
        int child[2];
        for (int s = 0; s < 2; ++s)
            child[s] = op[s].producer >= k0 && op[s].producer < k1 ? mine[op[s].producer - k0] : -1;
        // candidates: both operands' pieces, the larger one, the other, none
        int tries[4][2] = {{1, 1}, {1, 0}, {0, 1}, {0, 0}};
        if (child[0] >= 0 && child[1] >= 0 && size[child[1]].macs > size[child[0]].macs) {
            std::swap(tries[1][0], tries[2][0]);
            std::swap(tries[1][1], tries[2][1]);
        }
        for (auto& t : tries) {
            if ((t[0] && child[0] < 0) || (t[1] && child[1] < 0)) continue;
            if (t[0] && t[1] && child[0] == child[1]) continue;  // (no tree has it)
            Size z;
            z.out = nd.size;
            z.macs = nd.size * K;
            z.nodes = 1;
            z.words = 2 * nd.size + K + 8 + 4 + 6;  // at most one step and one store each
            for (int s = 0; s < 2; ++s) {
                if (t[s]) {
                    const Size& y = size[child[s]];
                    z.out += y.out;
                    z.elems += y.elems;
                    z.macs += y.macs;
                    z.words += y.words;
                    z.nodes += y.nodes;
                    z.ext += y.ext;
                } else {
                    z.elems += op[s].size;
                    z.ext += 1;
                    z.words += 8 + op[s].size / 2 + 1;
                }
            }
            if (z.out + z.elems > kRegionArena || z.nodes > kRegionNodes || z.ext > kRegionExt ||
                z.words + 32 > kRegionWords || z.macs > (1 << 16))
                continue;
            // the piece takes the place of the first one it joins
            const int r = t[0] ? child[0] : (t[1] ? child[1] : (int)size.size());
            if (r == (int)size.size()) {
                size.emplace_back();
                members.emplace_back();
            }
            if (t[0] && t[1]) {
                for (int q : members[child[1]]) mine[q - k0] = r;
                members[r].insert(members[r].end(), members[child[1]].begin(), members[child[1]].end());
                members[child[1]].clear();
            }
            size[r] = z;
            members[r].push_back(k);
            mine[k - k0] = r;
            break;
        }
    }
    for (auto& m : members) {
        if (m.empty()) continue;
        bool any = false;
        for (int k : m) any |= v.node(k).kind == kGeneric;
        if (m.size() < 4 && !any) continue;
        std::sort(m.begin(), m.end());
        for (int k : m) of[k] = (int)regions.size();
        regions.push_back(m);
    }
}

// Offsets of every output and K index of a node in its operands, in the order
// of the kernel that runs it outside a region: written to every second word of
// out, and to kt.
static void region_tables(const NetDesc& d, const Plan& p, const Node& nd, int64_t K, int32_t* out, int32_t* kt) {
    auto pack = [](int64_t a, int64_t b) { return (int32_t)((uint32_t)a | ((uint32_t)b << 16)); };
    if (nd.kind == kTiled) {
        const TileArgs& t = nd.tile;
        // offsets double with every index bit: entry x + 2^i is entry x plus bit i
        auto grow = [&](int32_t* v, int step, int64_t& have, const uint8_t* sa, const uint8_t* sb, int nb) {
            for (int i = 0; i < nb; ++i, have *= 2) {
                const int32_t add = pack(sa && sa[i] != kNoBit ? int64_t(1) << sa[i] : 0,
                                         sb && sb[i] != kNoBit ? int64_t(1) << sb[i] : 0);
                for (int64_t x = 0; x < have; ++x) v[(have + x) * step] = (int32_t)((uint32_t)v[x * step] + (uint32_t)add);
            }
        };
        int64_t have = 1;
        out[0] = 0;
        grow(out, 2, have, nullptr, t.b_n, t.nn);
        grow(out, 2, have, t.a_m, nullptr, t.nm);
        grow(out, 2, have, t.a_b, t.b_b, t.nb);
        have = 1;
        kt[0] = 0;
        grow(kt, 1, have, t.a_k, t.b_k, t.nk);
        return;
    }
    GenericArgs g;
    std::string err;
    fill_generic(d, p, nd, g, err);  // ranks were checked when the plan was made
    for (int64_t o = 0; o < nd.size; ++o) {
        int64_t rem = o, a = 0, b = 0;
        for (int i = 0; i < g.n_od; ++i) {
            a += rem % g.od_dim[i] * g.od_sa[i];
            b += rem % g.od_dim[i] * g.od_sb[i];
            rem /= g.od_dim[i];
        }
        out[2 * o] = pack(a, b);
    }
    for (int64_t k = 0; k < K; ++k) {
        int64_t rem = k, a = 0, b = 0;
        for (int i = 0; i < g.n_kd; ++i) {
            a += rem % g.kd_dim[i] * g.kd_sa[i];
            b += rem % g.kd_dim[i] * g.kd_sb[i];
            rem /= g.kd_dim[i];
        }
        kt[k] = pack(a, b);
    }
}

// Program of one region (layout: RegionHdr), appended to the plan's.
// at: one entry per node of the list, all -1 before and after (scratch).
void emit_region(const RegionView& v, const std::vector<int>& members, const std::vector<std::pair<int, int>>& stored,
                 std::vector<int>& at, std::vector<RegionHdr>& hdr, std::vector<int32_t>& P) {
    const NetDesc& d = *v.d;
    // order: tree level within the region, then how a node's sums are shared
    struct Item {
        int k, level, lg, accs;
        int64_t K;
    };
    std::vector<Item> items;
    items.reserve(members.size());
    for (int k : members) {
        const Node& nd = v.node(k);
        int lv = 0;
        for (int c : {nd.ca, nd.cb}) {
            const int pr = v.operand(c).producer;
            if (pr >= 0 && at[pr] >= 0) lv = std::max(lv, at[pr]);
        }
        at[k] = lv + 1;  // level for now
        // the wave kernel's g partial sums per output: lanes x sums per lane
        int64_t g = 1, K = region_k(d, nd);
        if (nd.kind == kTiled) {
            const int64_t O = wave_chunk(nd, v.copies);
            g = std::min<int64_t>(O >= 256 ? 1 : 256 / O, K);
        }
        int64_t L = std::max<int64_t>(1, g / 8);
        while (L < g && L < 32 && K / L > 16) L *= 2;
        items.push_back({k, lv + 1, ilog2(L), (int)(g / L), K});
    }
    std::stable_sort(items.begin(), items.end(), [](const Item& x, const Item& y) {
        return std::tie(x.level, x.lg, x.accs) < std::tie(y.level, y.lg, y.accs);
    });
    for (size_t i = 0; i < items.size(); ++i) at[items[i].k] = (int)i;  // place in the program
    std::vector<RegionExt> ext;
    std::vector<uint16_t> elem;
    std::vector<int64_t> q0(items.size());
    int64_t n_out = 0, n_k = 0;
    for (size_t i = 0; i < items.size(); ++i) {
        q0[i] = n_out;
        n_out += v.node(items[i].k).size;
        n_k += items[i].K;
    }
    // the blob starts with the outputs and the K tables
    RegionHdr h;
    memset(&h, 0, sizeof(h));
    h.blob = (int)P.size();
    h.o_k = (int)((2 * n_out + 3) / 4 * 4);
    P.resize(P.size() + h.o_k + n_k);
    int32_t* const outs = P.data() + h.blob;
    int32_t* const kts = outs + h.o_k;
    n_k = 0;
    std::vector<RegionNode> nodes(items.size());
    std::vector<RegionStep> steps;
    for (size_t i = 0; i < items.size(); ++i) {
        const Node& nd = v.node(items[i].k);
        RegionNode& r = nodes[i];
        r.kbase = (int)n_k;
        r.k = (int)items[i].K;
        region_tables(d, *v.p, nd, r.k, outs + 2 * q0[i], kts + n_k);
        for (int64_t q = q0[i]; q < q0[i] + nd.size; ++q) outs[2 * q + 1] = (int32_t)i;
        n_k += r.k;
        r.q0 = (int)q0[i];
        r.conj = (nd.tile.conj_a ? 1 : 0) | (nd.tile.conj_b ? 2 : 0);
        for (int s = 0; s < 2; ++s) {
            const RegionOperand op = v.operand(s ? nd.cb : nd.ca);
            int ref, slot;
            if (op.producer >= 0 && at[op.producer] >= 0) {
                const int j = at[op.producer];
                ref = -1 - (int)q0[j];  // the arena's outputs; the staged entries are added below
                slot = -1 - j;
            } else {
                RegionExt e;
                memset(&e, 0, sizeof(e));
                e.leaf = op.leaf;
                e.first = (int)elem.size();
                e.node = op.leaf >= 0 ? 0 : op.slot;
                e.ws_off = op.leaf >= 0 ? 0 : op.ws_off;
                elem.insert(elem.end(), op.size, (uint16_t)ext.size());
                ref = slot = (int)ext.size();
                ext.push_back(e);
            }
            (s ? r.b : r.a) = ref;
            (s ? r.sb : r.sa) = slot;
        }
        const bool new_level = i == 0 || items[i].level != items[i - 1].level;
        if (new_level || items[i].lg != items[i - 1].lg || items[i].accs != items[i - 1].accs)
            steps.push_back({(int)q0[i], (int)q0[i], items[i].lg, new_level ? -items[i].accs : items[i].accs});
        steps.back().q1 = (int)(q0[i] + nd.size);
    }
    const int n_elem = (int)elem.size(), n_ext = (int)ext.size();
    for (RegionNode& r : nodes) {
        if (r.a < 0) r.a = ~(n_elem + (-1 - r.a));
        if (r.b < 0) r.b = ~(n_elem + (-1 - r.b));
        if (r.sa < 0) r.sa = n_ext + (-1 - r.sa);
        if (r.sb < 0) r.sb = n_ext + (-1 - r.sb);
    }
    std::vector<RegionStore> stores;
    for (auto& st : stored) stores.push_back({at[st.first], st.second, v.node(st.first).ws_off, -1, 0});
    for (int k : members) at[k] = -1;
    auto put = [&](const void* src, size_t words) {
        while ((P.size() - h.blob) % 4) P.push_back(0);
        const int at = (int)P.size() - h.blob;
        const int32_t* w = static_cast<const int32_t*>(src);
        P.insert(P.end(), w, w + words);
        return at;
    };
    if (elem.size() % 2) elem.push_back(0);
    h.o_nodes = put(nodes.data(), nodes.size() * sizeof(RegionNode) / 4);
    h.o_ext = put(ext.data(), ext.size() * sizeof(RegionExt) / 4);
    h.o_elem = put(elem.data(), elem.size() / 2);
    h.o_steps = put(steps.data(), steps.size() * sizeof(RegionStep) / 4);
    h.o_store = put(stores.data(), stores.size() * sizeof(RegionStore) / 4);
    while ((P.size() - h.blob) % 4) P.push_back(0);
    h.words = (int)P.size() - h.blob;
    h.n_out = (int)n_out;
    h.n_nodes = (int)nodes.size();
    h.n_ext = n_ext;
    h.n_elem = n_elem;
    h.n_steps = (int)steps.size();
    h.n_store = (int)stores.size();
    hdr.push_back(h);
}

void set_regions(RegionArgs& ra, const std::vector<RegionHdr>& hdr, int begin, int count) {
    ra.hdr += begin;
    ra.n_regions = count;
    ra.words = ra.entries = 0;
    for (int r = begin; r < begin + count; ++r) {
        ra.words = std::max(ra.words, hdr[r].words);
        ra.entries = std::max(ra.entries, hdr[r].n_elem + hdr[r].n_out);
    }
}

cudaError_t upload_regions(const std::vector<RegionHdr>& hdr, const std::vector<int32_t>& prog,
                           const std::vector<SliceDigits>& leaf_sl, const std::vector<int64_t>& leaf_is, void** dev,
                           int64_t** leaf_is_dev, RegionArgs& ra) {
    const size_t hb = (hdr.size() * sizeof(RegionHdr) + 255) / 256 * 256;
    const size_t pb = (prog.size() * 4 + 255) / 256 * 256;
    const size_t sb = (leaf_sl.size() * sizeof(SliceDigits) + 255) / 256 * 256;
    std::vector<char> img(hb + pb + sb + sizeof(int64_t) * leaf_is.size());
    memcpy(img.data(), hdr.data(), hdr.size() * sizeof(RegionHdr));
    memcpy(img.data() + hb, prog.data(), prog.size() * 4);
    memcpy(img.data() + hb + pb, leaf_sl.data(), leaf_sl.size() * sizeof(SliceDigits));
    memcpy(img.data() + hb + pb + sb, leaf_is.data(), sizeof(int64_t) * leaf_is.size());
    cudaError_t e = cudaMalloc(dev, img.size());
    if (e != cudaSuccess) return e;
    e = cudaMemcpy(*dev, img.data(), img.size(), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) return e;
    char* q = static_cast<char*>(*dev);
    *leaf_is_dev = reinterpret_cast<int64_t*>(q + hb + pb + sb);
    ra.hdr = reinterpret_cast<const RegionHdr*>(q);
    ra.prog = reinterpret_cast<const int32_t*>(q + hb);
    ra.leaf_sl = reinterpret_cast<const SliceDigits*>(q + hb + pb);
    ra.leaf_is = *leaf_is_dev;
    return cudaSuccess;
}

tn_status build_plan(const NetDesc& d, Plan& p, std::string& err) {
    const int n = d.n;
    // diagnostics: TN_FORCE_GENERIC=1 runs every node on the generic kernel,
    // TN_NO_WAVES=1 launches every node separately, TN_NO_FLOW=1 one launch
    // per wave level
    if (const char* e = getenv("TN_FORCE_GENERIC")) p.force_generic = e[0] == '1';
    if (const char* e = getenv("TN_NO_WAVES")) p.no_waves = e[0] == '1';
    if (const char* e = getenv("TN_NO_FLOW")) p.no_flow = e[0] == '1';
    if (const char* e = getenv("TN_NO_TENSOR_CORES")) p.no_tensor_cores = e[0] == '1';
    const int L = (int)d.dims.size();
    // ---- tree validation (Sec. 2: leaves first, children before parents)
    if ((int64_t)p.pairs.size() != 2 * (int64_t)(n - 1)) {
        err = "tree must have n_tensors-1 pairs";
        return TN_EINVAL;
    }
    std::vector<char> used(2 * n, 0);
    for (int k = 0; k < n - 1; ++k) {
        int me = n + k;
        for (int j = 0; j < 2; ++j) {
            int c = p.pairs[2 * k + j];
            if (c < 0 || c >= me) {
                err = "tree child id out of range";
                return TN_EINVAL;
            }
            if (used[c]) {
                err = "tree id used twice";
                return TN_EINVAL;
            }
            used[c] = 1;
        }
    }
    // ---- sliced labels (Sec. 4.7.1)
    std::vector<char> is_open(L, 0), is_sl(L, 0);
    for (int l : d.open) is_open[l] = 1;
    p.sliced.clear();
    p.d_sliced = 1;
    for (int64_t id : p.sliced_ids) {
        auto it = d.id2d.find(id);
        if (it == d.id2d.end()) {
            err = "unknown sliced label";
            return TN_EINVAL;
        }
        int l = it->second;
        if (is_open[l]) {
            err = "sliced label is open";
            return TN_EINVAL;
        }
        if (is_sl[l]) {
            err = "sliced label repeated";
            return TN_EINVAL;
        }
        is_sl[l] = 1;
        p.sliced.push_back(l);
        if (p.d_sliced > (INT64_MAX / 4) / d.dims[l]) {
            err = "too many slices";
            return TN_EUNSUPPORTED;
        }
        p.d_sliced *= d.dims[l];
    }
    const int ns = (int)p.sliced.size();
    std::vector<int64_t> sdiv(ns, 1);
    for (int j = ns - 2; j >= 0; --j) sdiv[j] = sdiv[j + 1] * d.dims[p.sliced[j + 1]];

    // ---- per-vertex labels after slicing
    const int NV = 2 * n - 1;
    p.vlab.assign(NV, {});
    p.vstride.assign(NV, {});
    p.leaf_sl.assign(n, SliceDigits{});
    std::vector<int> total(L, 0);
    std::vector<SubCount> sub(NV);
    for (int v = 0; v < n; ++v) {
        const LeafDesc& lf = d.leaves[v];
        SliceDigits& sd = p.leaf_sl[v];
        sd.n = 0;
        for (size_t i = 0; i < lf.lab.size(); ++i) {
            int l = lf.lab[i];
            if (is_sl[l]) {
                if (sd.n >= kMaxSliceDigits) {
                    err = "too many sliced labels in one tensor";
                    return TN_EUNSUPPORTED;
                }
                int j = (int)(std::find(p.sliced.begin(), p.sliced.end(), l) - p.sliced.begin());
                sd.div[sd.n] = sdiv[j];
                sd.dim[sd.n] = d.dims[l];
                sd.stride[sd.n] = lf.stride[i];
                sd.n++;
                continue;
            }
            p.vlab[v].push_back(l);
            p.vstride[v].push_back(lf.stride[i]);
            total[l]++;
            sub[v].c.push_back({l, 1});
        }
    }
    // ---- nodes
    p.nodes.clear();
    p.nodes.reserve(std::max(n - 1, 1));  // nodes are large: no copies while the list grows
    double W = 0, C = 0;
    auto log2size = [&](const std::vector<int>& lab) {
        double s = 0;
        for (int l : lab) s += std::log2((double)d.dims[l]);
        return s;
    };
    for (int v = 0; v < n; ++v) W = std::max(W, log2size(p.vlab[v]));
    auto make_node = [&](int id, int a, int b, const std::vector<int>& keep) -> Node {
        return build_node(d, p, id, a, b, keep);
    };
    if (n == 1) {
        std::vector<int> keep = d.open;
        Node nd = make_node(n, 0, -1, keep);
        // the unit operand is smaller: make sure the leaf is an operand
        p.vlab.push_back(nd.lab);
        p.vstride.push_back(nd.stride);
        W = std::max(W, log2size(nd.lab));
        // one leaf has no contraction vertex, so C = 0 (Sec. 2); the node
        // only sums the leaf's own summed labels and orders the open axes
        p.nodes.push_back(nd);
    } else {
        for (int k = 0; k < n - 1; ++k) {
            int a = p.pairs[2 * k], b = p.pairs[2 * k + 1], me = n + k;
            std::vector<int> keep;
            SubCount sc;
            auto visit = [&](int c, int other) {
                for (auto& x : sub[c].c) {
                    int l = x.first;
                    if (c == b && sub[a].get(l)) continue;
                    int cnt = x.second + (c == a ? sub[b].get(l) : 0);
                    if (is_open[l] || cnt < total[l]) {
                        keep.push_back(l);
                        sc.c.push_back({l, cnt});
                    }
                }
                (void)other;
            };
            visit(a, b);
            visit(b, a);
            // sizes are formed in int64 below: refuse what could overflow them
            std::vector<int> uni = p.vlab[a];
            for (int l : p.vlab[b])
                if (std::find(uni.begin(), uni.end(), l) == uni.end()) uni.push_back(l);
            if (log2size(keep) > kMaxLog2Entries) {
                err = "an intermediate of the sliced tree has more than 2^40 entries";
                return TN_EUNSUPPORTED;
            }
            if (log2size(uni) > kMaxLog2Work) {
                err = "a node of the sliced tree needs more than 2^62 multiply-adds";
                return TN_EUNSUPPORTED;
            }
            sub[me] = sc;
            sub[a].c.clear();
            sub[b].c.clear();
            Node nd = make_node(me, a, b, keep);
            p.vlab[me] = nd.lab;
            p.vstride[me] = nd.stride;
            W = std::max(W, log2size(nd.lab));
            C += std::pow(2.0, nd.vc);
            p.nodes.push_back(std::move(nd));
        }
    }
    // root labels must be exactly the open labels
    const Node& root = p.nodes.back();
    if (root.lab.size() != d.open.size()) {
        err = "internal: root labels differ from the open labels";
        return TN_EINVAL;
    }
    p.W = W;
    p.C = C;
    // ---- kernel choice per node: large GEMM-shaped nodes go to the tensor
    // cores in the reduced-precision modes (M >= 128 rows, N >= 128 real
    // accumulator columns, K >= 16); everything else on CUDA cores
    int64_t split_elems = 0;
    for (size_t k = 0; k < p.nodes.size(); ++k) {
        Node& nd = p.nodes[k];
        nd.kind = kGeneric;
        if (p.force_generic || !plan_tile(d, p, nd, split_elems)) {
            if (p.persistent) {
                err = "the persistent launch needs power-of-two label sizes on every node";
                return TN_EUNSUPPORTED;
            }
            if (!p.force_generic) plan_any_tile(d, p, nd, split_elems, p.copies);
            continue;
        }
        if (p.persistent) {
            // tile items: 64 x 64 tiles, all of K in one item (no K split)
            if (tile_item_node(nd)) {
                int64_t unused = 0;
                Node t = nd;
                if (plan_tile(d, p, t, unused, kTile64x64)) {
                    t.tile.split = 1;
                    t.tile.kchunk = int64_t(1) << t.tile.nk;
                    nd = t;
                }
            }
            continue;
        }
        if (!p.no_tensor_cores) make_tensor_core(d, p.mode, nd, split_elems, p.copies);
    }
    p.split_bytes = (split_elems * (int64_t)d.elem_bytes() + 1023) / 1024 * 1024;
    // ---- launch schedule: tree levels; per level one wave launch for the
    // small tiled nodes, then one launch per remaining node
    std::vector<int> level(2 * n, 0);
    int max_level = 0;
    // subtrees of small nodes: one region each, a single step of the schedule
    std::vector<std::vector<int>> regions;
    std::vector<int> region_of(p.nodes.size(), -1);
    RegionView view;
    view.d = &d;
    view.p = &p;
    view.copies = p.copies;
    view.node = [&p](int k) -> const Node& { return p.nodes[k]; };
    view.operand = [&d, &p, n](int c) -> RegionOperand {
        if (c < n) return {-1, c, 0, d.leaves[c].size, 0};
        return {c - n, -1, c - n, p.nodes[c - n].size, 0};  // workspace offsets follow below
    };
    if (!p.no_regions && !p.no_waves && !p.no_flow && !p.force_generic && !p.persistent)
        find_regions(view, 0, (int)p.nodes.size(), region_of, regions);
    for (size_t k = 0; k < p.nodes.size(); ++k) {
        const Node& nd = p.nodes[k];
        const int r = region_of[k];
        int lv = 0;
        if (r < 0) {
            for (int c : {nd.ca, nd.cb})
                if (c >= n) lv = std::max(lv, level[c]);
        } else if (regions[r].back() == (int)k) {
            // the region's root, its last node: after everything it reads from outside
            for (int q : regions[r])
                for (int c : {p.nodes[q].ca, p.nodes[q].cb})
                    if (c >= n && region_of[c - n] != r) lv = std::max(lv, level[c]);
            for (int q : regions[r]) level[n + q] = lv + 1;
        } else {
            continue;
        }
        level[n + k] = 1 + lv;
        max_level = std::max(max_level, level[n + k]);
    }
    p.node_level.assign(level.begin() + n, level.begin() + n + p.nodes.size());
    p.steps.clear();
    p.items.clear();
    if (p.persistent) {
        // one dataflow launch over the whole tree, level by level
        Step w;
        w.wave = 1;
        w.flow = 1;
        w.item_begin = 0;
        for (int L = 1; L <= max_level; ++L)
            for (size_t k = 0; k < p.nodes.size(); ++k) {
                if (level[n + k] != L) continue;
                const Node& nd = p.nodes[k];
                const int64_t cnt = persistent_items(nd);
                for (int64_t i = 0; i < cnt; ++i) {
                    WaveItem it;
                    it.node = (int)k;
                    it.pad = 0;
                    if (nd.tile.cfg == kTile64x64 && tile_item_node(nd)) {
                        it.o_begin = i;
                        it.o_count = -1;
                    } else {
                        const int64_t chunk = wave_chunk(nd, 2);
                        it.o_begin = i * chunk;
                        it.o_count = std::min(chunk, nd.size - i * chunk);
                    }
                    p.items.push_back(it);
                }
                w.nodes.push_back((int)k);
            }
        w.item_count = (int)p.items.size();
        if ((int64_t)p.items.size() > (int64_t(1) << 30)) {
            err = "the persistent launch would need more than 2^30 work items";
            return TN_EUNSUPPORTED;
        }
        p.steps.push_back(w);
    }
    p.region_hdr.clear();
    p.region_prog.clear();
    std::vector<int> scratch(p.nodes.size(), -1);
    for (int L = 1; L <= max_level && !p.persistent; ++L) {
        Step rs;
        for (size_t r = 0; r < regions.size(); ++r) {
            if (level[n + regions[r].back()] != L) continue;
            if (rs.regions == 0) rs.region_begin = (int)p.region_hdr.size();
            // the root, its last member, is read outside
            emit_region(view, regions[r], {{regions[r].back(), regions[r].back()}}, scratch, p.region_hdr, p.region_prog);
            ++rs.regions;
            rs.nodes.insert(rs.nodes.end(), regions[r].begin(), regions[r].end());
        }
        if (rs.regions) p.steps.push_back(rs);
        Step w;
        w.wave = 1;
        w.item_begin = (int)p.items.size();
        std::vector<int> singles;
        for (size_t k = 0; k < p.nodes.size(); ++k) {
            if (level[n + k] != L || region_of[k] >= 0) continue;
            const Node& nd = p.nodes[k];
            const bool small = wave_node(nd, p.copies) && !p.no_waves;
            if (!small) {
                singles.push_back((int)k);
                continue;
            }
            const int64_t chunk = wave_chunk(nd, p.copies);
            for (int64_t o = 0; o < nd.size; o += chunk) {
                WaveItem it;
                it.node = (int)k;
                it.pad = 0;
                it.o_begin = o;
                it.o_count = chunk;
                p.items.push_back(it);
            }
            w.nodes.push_back((int)k);
        }
        w.item_count = (int)p.items.size() - w.item_begin;
        if (w.item_count > 0) p.steps.push_back(w);
        for (int k : singles) {
            Step s;
            s.node = k;
            s.nodes.push_back(k);
            p.steps.push_back(s);
        }
    }
    // ---- consecutive wave levels become one dataflow launch (their items
    // are contiguous); a node waits for its children in the same launch
    if (!p.no_flow && !p.persistent) {
        std::vector<Step> merged;
        for (Step& st : p.steps) {
            if (st.wave && !merged.empty() && merged.back().wave &&
                merged.back().item_begin + merged.back().item_count == st.item_begin) {
                Step& m = merged.back();
                m.item_count += st.item_count;
                m.nodes.insert(m.nodes.end(), st.nodes.begin(), st.nodes.end());
                m.flow = 1;
            } else {
                merged.push_back(st);
            }
        }
        p.steps = merged;
    }
    p.flow_deps.assign(4 * p.nodes.size(), -1);
    for (const Step& st : p.steps) {
        if (!st.flow) continue;
        std::vector<char> in_step(p.nodes.size(), 0);
        for (int k : st.nodes) in_step[k] = 1;
        for (int k : st.nodes) {
            const Node& nd = p.nodes[k];
            int slot = 0;
            for (int c : {nd.ca, nd.cb}) {
                if (c >= n && in_step[c - n]) {
                    const Node& ch = p.nodes[c - n];
                    const int64_t chunk = wave_chunk(ch, p.copies);
                    p.flow_deps[4 * k + 2 * slot] = c - n;
                    p.flow_deps[4 * k + 2 * slot + 1] =
                        p.persistent ? (int)persistent_items(ch) : (int)((ch.size + chunk - 1) / chunk);
                }
                ++slot;
            }
        }
    }
    // ---- workspace liveness in execution order: a step's outputs are all
    // allocated before any of its operands is released (they run at once).  Of a
    // region only the root is stored.
    Arena ar;
    for (const Step& st : p.steps) {
        auto inside = [&](int k) { return region_of[k] >= 0 && regions[region_of[k]].back() != k; };
        for (int k : st.nodes)
            if (!inside(k)) p.nodes[k].ws_off = ar.alloc(p.nodes[k].size);
        for (int k : st.nodes)
            for (int c : {p.nodes[k].ca, p.nodes[k].cb})
                if (c >= n && !inside(c - n)) {
                    const Node& ch = p.nodes[c - n];
                    ar.release(ch.ws_off, ch.size);
                }
    }
    p.ws_elems = std::max<int64_t>(ar.end, 64);
    // the programs' workspace offsets
    for (const RegionHdr& h : p.region_hdr) {
        RegionExt* ext = reinterpret_cast<RegionExt*>(p.region_prog.data() + h.blob + h.o_ext);
        for (int e = 0; e < h.n_ext; ++e)
            if (ext[e].leaf < 0) ext[e].ws_off = p.nodes[ext[e].node].ws_off;
        RegionStore* st = reinterpret_cast<RegionStore*>(p.region_prog.data() + h.blob + h.o_store);
        for (int i = 0; i < h.n_store; ++i) st[i].ws_off = p.nodes[st[i].slot].ws_off;
    }
    p.n_out = 1;
    for (int l : d.open) p.n_out *= d.dims[l];
    return TN_OK;
}

static tn_status fill_generic(const NetDesc& d, const Plan& p, const Node& nd, GenericArgs& g,
                              std::string& err) {
    memset(&g, 0, sizeof(g));
    const int n = d.n;
    static const std::vector<int> none;
    static const std::vector<int64_t> nones;
    const std::vector<int>& la = nd.ca >= 0 ? p.vlab[nd.ca] : none;
    const std::vector<int>& lb = nd.cb >= 0 ? p.vlab[nd.cb] : none;
    const std::vector<int64_t>& sa = nd.ca >= 0 ? p.vstride[nd.ca] : nones;
    const std::vector<int64_t>& sb = nd.cb >= 0 ? p.vstride[nd.cb] : nones;
    if ((int)nd.lab.size() > kMaxDigits) {
        err = "node rank exceeds the generic kernel limit";
        return TN_EUNSUPPORTED;
    }
    g.n_out = nd.size;
    g.n_od = (int)nd.lab.size();
    for (int i = 0; i < g.n_od; ++i) {
        int l = nd.lab[nd.lab.size() - 1 - i];
        g.od_dim[i] = (int32_t)d.dims[l];
        g.od_sa[i] = stride_in(la, sa, l);
        g.od_sb[i] = stride_in(lb, sb, l);
    }
    std::vector<int> ks = nd.gk;
    ks.insert(ks.end(), nd.gsa.begin(), nd.gsa.end());
    ks.insert(ks.end(), nd.gsb.begin(), nd.gsb.end());
    std::sort(ks.begin(), ks.end(), [&](int x, int y) {
        return stride_in(lb, sb, x) + stride_in(la, sa, x) < stride_in(lb, sb, y) + stride_in(la, sa, y);
    });
    if ((int)ks.size() > kMaxDigits) {
        err = "too many summed labels in one node";
        return TN_EUNSUPPORTED;
    }
    g.n_kd = (int)ks.size();
    g.n_sum = 1;
    for (int i = 0; i < g.n_kd; ++i) {
        int l = ks[i];
        g.kd_dim[i] = (int32_t)d.dims[l];
        g.kd_sa[i] = stride_in(la, sa, l);
        g.kd_sb[i] = stride_in(lb, sb, l);
        g.n_sum *= d.dims[l];
    }
    if (nd.ca >= 0 && nd.ca < n) g.sla = p.leaf_sl[nd.ca];
    if (nd.cb >= 0 && nd.cb < n) g.slb = p.leaf_sl[nd.cb];
    g.nbatch = g.M = g.N = 1;
    g.split = 1;
    if (nd.kind == kGeneric && nd.any_cfg) {
        g.cfg = nd.any_cfg;
        g.split = nd.any_split;
        g.kchunk = nd.any_kchunk;
        g.n_nd = (int)nd.gn.size();
        g.n_md = (int)nd.gm.size();
        for (int l : nd.gn) g.N *= d.dims[l];
        for (int l : nd.gm) g.M *= d.dims[l];
        for (int l : nd.gb) g.nbatch *= d.dims[l];
        // load along the rows (columns) where they hold the operand's fastest label
        auto fast = [&](const std::vector<int>& lab, const std::vector<int64_t>& st, const std::vector<int>& group) {
            int best = -1;
            int64_t bs = INT64_MAX;
            for (size_t i = 0; i < lab.size(); ++i)
                if (d.dims[lab[i]] > 1 && st[i] < bs) {
                    bs = st[i];
                    best = lab[i];
                }
            return best >= 0 && has(group, best);
        };
        g.a_mfast = fast(la, sa, nd.gm);
        g.b_nfast = fast(lb, sb, nd.gn);
    }
    return TN_OK;
}

tn_status alloc_plan(NetDesc& d, Plan& p, void* unit, std::string& err) {
    const size_t eb = d.elem_bytes();
    const int nn = (int)p.nodes.size();
    auto ck = [&](cudaError_t e, const char* what) {
        if (e != cudaSuccess) {
            err = std::string(what) + ": " + cudaGetErrorString(e);
            return false;
        }
        return true;
    };
    const int G = std::max(p.alloc_inst, 1);
    if (!ck(cudaMalloc(&p.ws, (size_t)p.ws_elems * eb * G), "workspace allocation")) return TN_ENOMEM;
    // node maxima of every instance, then the dataflow counters (done per
    // node and instance, one item head per step): one region, cleared by one
    // memset per slice
    const size_t flow_cnt = (size_t)nn * G + p.steps.size() + 1;
    if (!ck(cudaMalloc(&p.maxabs, sizeof(unsigned) * ((size_t)nn * G + flow_cnt)), "cudaMalloc"))
        return TN_ENOMEM;
    p.flow_cnt_dev = p.maxabs + (size_t)nn * G;
    if (!ck(cudaMalloc(&p.exps, sizeof(int64_t) * nn * G), "cudaMalloc")) return TN_ENOMEM;
    if (!ck(cudaMalloc(&p.inst_roots_dev, sizeof(BatchRoot) * G), "cudaMalloc")) return TN_ENOMEM;
    if (!ck(cudaMalloc(&p.inst_out_dev, sizeof(double) * 2 * G), "cudaMalloc")) return TN_ENOMEM;
    if (!ck(cudaMalloc(&p.inst_exp_dev, sizeof(int64_t) * G), "cudaMalloc")) return TN_ENOMEM;
    if (!ck(cudaMalloc(&p.ctl, sizeof(Control)), "cudaMalloc")) return TN_ENOMEM;
    // a call of an unsliced tree folds straight into the caller's output
    size_t acc_doubles = (size_t)p.n_out * (d.is_complex() ? 2 : 1);
    if (p.d_sliced > 1 && !ck(cudaMalloc(&p.acc, sizeof(double) * acc_doubles), "cudaMalloc")) return TN_ENOMEM;
    if (!ck(cudaStreamCreateWithFlags(&p.cap_stream, cudaStreamNonBlocking), "stream")) return TN_ECUDA;
    if (!ck(cudaMalloc(&p.leafmax, sizeof(unsigned) * d.n), "cudaMalloc")) return TN_ENOMEM;
    if (!ck(cudaMalloc((void**)&p.leaf_ptr_dev, sizeof(void*) * d.n), "cudaMalloc")) return TN_ENOMEM;
    if (!ck(cudaMalloc(&p.leaf_nfloat_dev, sizeof(int64_t) * d.n), "cudaMalloc")) return TN_ENOMEM;
    {
        std::vector<int64_t> nf(d.n);
        for (int v = 0; v < d.n; ++v) nf[v] = d.leaves[v].size * (d.is_complex() ? 2 : 1);
        if (!ck(cudaMemcpy(p.leaf_nfloat_dev, nf.data(), sizeof(int64_t) * d.n,
                           cudaMemcpyHostToDevice), "cudaMemcpy"))
            return TN_ECUDA;
        p.leaf_nfloat_uploaded = nf;
    }
    if (p.split_bytes > 0 && !ck(cudaMalloc(&p.split_buf, p.split_bytes * G), "split-K buffer"))
        return TN_ENOMEM;
    // node launch arguments; leaf pointers are patched per call
    p.gen.resize(nn);
    const int n = d.n;
    for (int k = 0; k < nn; ++k) {
        const Node& nd = p.nodes[k];
        GenericArgs& g = p.gen[k];
        tn_status st = fill_generic(d, p, nd, g, err);
        if (st != TN_OK) return st;
        char* ws = (char*)p.ws;
        g.C = ws + nd.ws_off * eb;
        g.A = nd.ca >= n ? (const void*)(ws + p.nodes[nd.ca - n].ws_off * eb) : nullptr;
        g.B = nd.cb >= n ? (const void*)(ws + p.nodes[nd.cb - n].ws_off * eb) : nullptr;
        if (nd.ca < 0) g.A = unit;
        if (nd.cb < 0) g.B = unit;
        g.P = p.split_buf;
        g.ctl = p.ctl;
        // leaves: renormalised by their own max, stored exponent 0
        g.sc.max_a = nd.ca >= n ? p.maxabs + (nd.ca - n) : (nd.ca >= 0 ? p.leafmax + nd.ca : nullptr);
        g.sc.exp_a = nd.ca >= n ? p.exps + (nd.ca - n) : nullptr;
        g.sc.max_b = nd.cb >= n ? p.maxabs + (nd.cb - n) : (nd.cb >= 0 ? p.leafmax + nd.cb : nullptr);
        g.sc.exp_b = nd.cb >= n ? p.exps + (nd.cb - n) : nullptr;
        g.sc.max_c = p.maxabs + k;
        g.sc.exp_c = p.exps + k;
        Node& ndm = p.nodes[k];
        if (ndm.kind == kTiled || ndm.kind == kTensorCore) {
            TileArgs& t = ndm.tile;
            t.A = g.A;
            t.B = g.B;
            t.C = g.C;
            t.P = p.split_buf;
            t.sla = g.sla;
            t.slb = g.slb;
            t.ctl = g.ctl;
            t.sc = g.sc;
        }
    }
    {
        // dataflow waves: dependencies, and completion / item counters
        if (!ck(cudaMalloc(&p.flow_deps_dev, sizeof(int) * 4 * std::max(nn, 1)), "cudaMalloc")) return TN_ENOMEM;
        if (!ck(cudaMemcpy(p.flow_deps_dev, p.flow_deps.data(), sizeof(int) * p.flow_deps.size(),
                           cudaMemcpyHostToDevice), "cudaMemcpy"))
            return TN_ECUDA;
    }
    if (!p.items.empty()) {  // filled by configure_instances, before every first run
        if (!ck(cudaMalloc(&p.descs_dev, sizeof(TileArgs) * nn), "cudaMalloc")) return TN_ENOMEM;
        if (!ck(cudaMalloc(&p.items_dev, sizeof(WaveItem) * p.items.size() * G), "cudaMalloc"))
            return TN_ENOMEM;
    }
    if (!p.region_hdr.empty()) {
        RegionArgs& ra = p.region_args;
        memset(&ra, 0, sizeof(ra));
        p.leaf_is_uploaded.assign(n, 0);
        if (!ck(upload_regions(p.region_hdr, p.region_prog, p.leaf_sl, p.leaf_is_uploaded, &p.region_dev,
                               &p.leaf_is_dev, ra), "region programs"))
            return TN_ENOMEM;
        ra.leaf_ptrs = reinterpret_cast<const void* const*>(p.leaf_ptr_dev);
        ra.leafmax = p.leafmax;
        ra.ws = p.ws;
        ra.ws_is = p.ws_elems;
        ra.maxabs = p.maxabs;
        ra.exps = p.exps;
        ra.slot_is = nn;
        ra.ctl = p.ctl;
    }
    // root accumulation: user open-label order -> root layout
    const Node& root = p.nodes.back();
    AccumArgs& a = p.acc_args;
    memset(&a, 0, sizeof(a));
    a.R = (char*)p.ws + root.ws_off * eb;
    a.n_out = p.n_out;
    if ((int)d.open.size() > kMaxDigits) {
        err = "too many open labels";
        return TN_EUNSUPPORTED;
    }
    for (int i = (int)d.open.size() - 1; i >= 0; --i)
        push_fold_digit(a, d.dims[d.open[i]], stride_in(root.lab, root.stride, d.open[i]));
    a.direct = 1;
    a.max_r = p.maxabs + (nn - 1);
    a.exp_r = p.exps + (nn - 1);
    a.acc = p.acc;
    a.ctl = p.ctl;
    a.n_inst = 1;
    a.r_is = p.ws_elems;
    a.s_is = nn;
    p.cfg_inst = -1;  // instance layout not yet written to the arguments
    return TN_OK;
}

// Write the instance layout (G instances; step 1: instance i = slice s+i,
// step 0: independent copies whose leaf v sits leaf_is[v] elements apart)
// into every node's launch arguments, the wave items and the accumulator.
// The device tables are written in the stream's order: earlier calls on it may
// still be reading them.
static tn_status configure_instances(const NetDesc& d, Plan& p, int G, int step,
                                     const std::vector<int64_t>& leaf_is, cudaStream_t stream, std::string& err) {
    if (p.cfg_inst == G && p.cfg_step == step && p.cfg_leaf_is == leaf_is) return TN_OK;
    const int n = d.n;
    const int nn = (int)p.nodes.size();
    const int64_t p_is = p.split_bytes / (int64_t)d.elem_bytes();
    for (int k = 0; k < nn; ++k) {
        Node& nd = p.nodes[k];
        InstanceInfo in;
        memset(&in, 0, sizeof(in));
        in.n_inst = G;
        in.slice_step = step;
        in.c_is = p.ws_elems;
        in.sc_is = nn;
        in.p_is = p_is;
        auto set = [&](int c, int64_t& is, int32_t& sis) {
            if (c >= n) {
                is = p.ws_elems;
                sis = nn;
            } else if (c >= 0) {
                is = leaf_is.empty() ? 0 : leaf_is[c];
                sis = 0;
            }
        };
        set(nd.ca, in.a_is, in.sa_is);
        set(nd.cb, in.b_is, in.sb_is);
        p.gen[k].in = in;
        nd.tile.in = in;
        // the launch grid's z extent (batch x K splits x instances) is at most
        // 65535: fewer K splits when many instances run side by side
        if (!p.persistent && (nd.kind == kTiled || nd.kind == kTensorCore)) {
            TileArgs& t = nd.tile;
            if (t.nbatch * (int64_t)G > 65535) {
                err = "too many instances for a node with " + std::to_string(t.nbatch) + " batch entries";
                return TN_EUNSUPPORTED;
            }
            if (t.split > 1 && t.nbatch * (int64_t)t.split * G > 65535) {
                int split = t.split;
                while (split > 1 && t.nbatch * (int64_t)split * G > 65535) split /= 2;
                const int64_t K = int64_t(1) << t.nk;
                const int64_t gran = t.cfg == kTileDot ? 256 : (t.cfg == kTile4x1024 ? 4 : 16);
                const int64_t units = (K + gran - 1) / gran;
                t.split = split;
                t.kchunk = ((units + split - 1) / split) * gran;
            }
        }
        if (!p.persistent && nd.kind == kGeneric) {
            if (G > 65535) {
                err = "too many instances";
                return TN_EUNSUPPORTED;
            }
            // the tile kernel's grid z likewise; one thread per output otherwise
            GenericArgs& g = p.gen[k];
            g.cfg = g.nbatch * (int64_t)nd.any_split * G > 65535 ? 0 : nd.any_cfg;
        }
    }
    if (!p.items.empty()) {
        std::vector<TileArgs> descs(nn);
        for (int k = 0; k < nn; ++k) descs[k] = p.nodes[k].tile;
        std::vector<WaveItem> items;
        items.reserve(p.items.size() * G);
        // within each step: level by level, every instance's items of a
        // level before the next level (the instances' dependency chains
        // advance together; a node's children always come earlier)
        std::vector<int> level(nn, 0);
        for (int k = 0; k < nn; ++k) {
            const Node& nd = p.nodes[k];
            const int la = nd.ca >= n ? level[nd.ca - n] : 0, lb = nd.cb >= n ? level[nd.cb - n] : 0;
            level[k] = 1 + std::max(la, lb);
        }
        p.inst_items_begin.assign(p.steps.size(), 0);
        for (size_t s = 0; s < p.steps.size(); ++s) {
            const Step& st = p.steps[s];
            p.inst_items_begin[s] = (int)items.size();
            if (!st.wave) continue;
            int j0 = 0;
            while (j0 < st.item_count) {
                const int L = level[p.items[st.item_begin + j0].node];
                int j1 = j0;
                while (j1 < st.item_count && level[p.items[st.item_begin + j1].node] == L) ++j1;
                for (int i = 0; i < G; ++i)
                    for (int j = j0; j < j1; ++j) {
                        WaveItem it = p.items[st.item_begin + j];
                        it.pad = i;
                        items.push_back(it);
                    }
                j0 = j1;
            }
        }
        cudaError_t e = cudaMemcpyAsync(p.descs_dev, descs.data(), sizeof(TileArgs) * nn, cudaMemcpyHostToDevice, stream);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(p.items_dev, items.data(), sizeof(WaveItem) * items.size(), cudaMemcpyHostToDevice, stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(stream);  // the lists end with this block
        if (e != cudaSuccess) {
            err = std::string("instance layout upload: ") + cudaGetErrorString(e);
            return TN_ECUDA;
        }
    }
    if (p.leaf_is_dev) {
        const std::vector<int64_t> is = leaf_is.empty() ? std::vector<int64_t>(n, 0) : leaf_is;
        if (is != p.leaf_is_uploaded) {
            cudaError_t e = cudaMemcpyAsync(p.leaf_is_dev, is.data(), sizeof(int64_t) * n, cudaMemcpyHostToDevice, stream);
            if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
            if (e != cudaSuccess) {
                err = std::string("instance layout upload: ") + cudaGetErrorString(e);
                return TN_ECUDA;
            }
            p.leaf_is_uploaded = is;
        }
        p.region_args.n_inst = G;
        p.region_args.slice_step = step;
    }
    p.acc_args.n_inst = step == 1 ? G : 1;
    p.graph_inst = p.graph_inst_h = -2;  // captured sequences hold the old layout
    p.cfg_inst = G;
    p.cfg_step = step;
    p.cfg_leaf_is = leaf_is;
    return TN_OK;
}

// One launch group: reset the node maxima of all instances, run every node
// (each launch covers all instances), then either fold the instances' roots
// (consecutive slices) into the FP64 accumulator and advance the slice
// counter, or write each independent instance's root to its output.
// ev: optional timing events around launch steps [pf, pf + pc).
static cudaError_t enqueue_slice(const NetDesc& d, Plan& p, cudaStream_t s, const cudaEvent_t* ev,
                                 int pf, int pc) {
    const int G = std::max(p.cfg_inst, 1);
    const int nn = (int)p.nodes.size();
    bool any_flow = false;
    for (const Step& st : p.steps) any_flow |= st.flow != 0;
    // the node maxima and (dataflow) the counters that follow them
    const size_t n_zero = any_flow ? (size_t)(p.flow_cnt_dev - p.maxabs) + (size_t)nn * G + p.steps.size()
                                   : (size_t)nn * G;
    cudaError_t e = cudaMemsetAsync(p.maxabs, 0, sizeof(unsigned) * n_zero, s);
    if (e != cudaSuccess) return e;
    const bool c = d.is_complex();
    for (int k = 0; k < (int)p.steps.size(); ++k) {
        // External records become event-record nodes under stream capture.
        if (ev && k >= pf && k < pf + pc &&
            (e = cudaEventRecordWithFlags(ev[k - pf], s, cudaEventRecordExternal)) != cudaSuccess)
            return e;
        const Step& st = p.steps[k];
        if (st.regions) {
            RegionArgs ra = p.region_args;
            set_regions(ra, p.region_hdr, st.region_begin, st.regions);
            e = launch_regions(ra, c, s);
        } else if (st.wave) {
            if (st.flow)
                e = launch_wave(p.items_dev + p.inst_items_begin[k], st.item_count * G, p.descs_dev,
                                reinterpret_cast<const void* const*>(p.leaf_ptr_dev), c, s,
                                reinterpret_cast<const int4*>(p.flow_deps_dev), p.flow_cnt_dev,
                                p.flow_cnt_dev + (size_t)nn * G + k, G, p.persistent);
            else
                e = launch_wave(p.items_dev + p.inst_items_begin[k], st.item_count * G, p.descs_dev,
                                reinterpret_cast<const void* const*>(p.leaf_ptr_dev), c, s);
        } else {
            const Node& nd = p.nodes[st.node];
            if (nd.kind == kTensorCore)
                e = launch_tc(nd.tile, tc_prec_of_mode(p.mode),
                              c, s);
            else if (nd.kind == kTiled)
                e = launch_tile(nd.tile, c, s);
            else
                e = launch_generic(p.gen[st.node], c, s);
        }
        if (e != cudaSuccess) return e;
        if (ev && k == pf + pc - 1 &&
            (e = cudaEventRecordWithFlags(ev[pc], s, cudaEventRecordExternal)) != cudaSuccess)
            return e;
    }
    if (p.cfg_step == 0)
        return launch_batch_finish(p.inst_roots_dev, G, p.inst_out_dev, p.inst_exp_dev, nullptr, nullptr,
                                   nullptr, s);
    return launch_accumulate(p.acc_args, c, s, G);
}

#define CK(x)                                                     \
    do {                                                          \
        cudaError_t e_ = (x);                                     \
        if (e_ != cudaSuccess) {                                  \
            err = std::string(#x) + ": " + cudaGetErrorString(e_); \
            return e_ == cudaErrorMemoryAllocation ? TN_ENOMEM : TN_ECUDA; \
        }                                                         \
    } while (0)

// Leaf pointers of this call (host leaves are staged into library memory),
// patched into the node arguments and the device leaf table.
static tn_status prepare_leaves(NetDesc& d, Plan& p, bool capturing, std::vector<const void*>& lp,
                                cudaStream_t stream, std::string& err) {
    const int n = d.n;
    const size_t eb = d.elem_bytes();
    lp.assign(n, nullptr);
    // several host leaves outside capture: one page-locked image, one copy
    int n_host = 0;
    int64_t total = 0;
    for (int v = 0; v < n; ++v)
        if (d.leaves[v].mem == TN_MEM_HOST) {
            ++n_host;
            total += (d.leaves[v].size * (int64_t)eb + 15) / 16 * 16;
        }
    if (!capturing && n_host > 1) {
        if (d.stage_bytes < total) {
            if (d.stage_pending) CK(cudaEventSynchronize(d.stage_done));
            d.stage_pending = false;
            if (d.stage_host) CK(cudaFreeHost(d.stage_host));
            if (d.stage_dev) CK(cudaFree(d.stage_dev));
            d.stage_host = d.stage_dev = nullptr;
            d.stage_bytes = 0;
            CK(cudaMallocHost(&d.stage_host, total));
            CK(cudaMalloc(&d.stage_dev, total));
            d.stage_bytes = total;
            if (!d.stage_done) CK(cudaEventCreateWithFlags(&d.stage_done, cudaEventDisableTiming));
        }
        // the image may still be read by the previous call's copy
        if (d.stage_pending) CK(cudaEventSynchronize(d.stage_done));
        int64_t off = 0;
        for (int v = 0; v < n; ++v) {
            LeafDesc& lf = d.leaves[v];
            if (lf.mem == TN_MEM_HOST) {
                memcpy((char*)d.stage_host + off, lf.ptr, lf.size * eb);
                lp[v] = (char*)d.stage_dev + off;
                off += (lf.size * (int64_t)eb + 15) / 16 * 16;
            } else {
                lp[v] = lf.ptr;
            }
        }
        CK(cudaMemcpyAsync(d.stage_dev, d.stage_host, off, cudaMemcpyHostToDevice, stream));
        CK(cudaEventRecord(d.stage_done, stream));
        d.stage_pending = true;
    }
    for (int v = 0; v < n; ++v) {
        LeafDesc& lf = d.leaves[v];
        if (lf.mem == TN_MEM_HOST && lp[v]) continue;  // staged above
        if (lf.mem == TN_MEM_HOST) {
            int64_t bytes = std::max<int64_t>(lf.size * (int64_t)eb, 16);
            if (lf.staged_bytes < bytes) {
                if (capturing) {
                    err = "host leaves need a first call outside stream capture";
                    return TN_EUNSUPPORTED;
                }
                if (lf.staged) CK(cudaFree(lf.staged));
                lf.staged = nullptr;
                CK(cudaMalloc(&lf.staged, bytes));
                lf.staged_bytes = bytes;
            }
            CK(cudaMemcpyAsync(lf.staged, lf.ptr, lf.size * eb, cudaMemcpyHostToDevice, stream));
            lp[v] = lf.staged;
        } else {
            lp[v] = lf.ptr;
        }
    }
    for (size_t k = 0; k < p.nodes.size(); ++k) {
        Node& nd = p.nodes[k];
        if (nd.ca >= 0 && nd.ca < n) p.gen[k].A = nd.tile.A = lp[nd.ca];
        if (nd.cb >= 0 && nd.cb < n) p.gen[k].B = nd.tile.B = lp[nd.cb];
    }
    if (capturing && p.leaf_ptr_uploaded != lp) {
        err = "re-attached leaves need a first call outside stream capture";
        return TN_EUNSUPPORTED;
    }
    // The pointer table changes only when leaves are re-attached; the stream
    // orders the write between the calls that read the table.  A captured
    // call writes its own pointers at every replay, so once there is one,
    // direct calls write theirs every time.
    p.captured |= capturing;
    if (p.captured || p.leaf_ptr_uploaded != lp) {
        CK(launch_leaf_table(lp.data(), n, reinterpret_cast<const void**>(p.leaf_ptr_dev), stream));
        p.leaf_ptr_uploaded = lp;
    }
    return TN_OK;
}

// The pointers that a captured sequence holds: those of leaves read by nodes
// with a launch of their own.  Waves read theirs from the device table, so
// re-attaching the others (the output states of another bitstring, say) does
// not recapture the graph.
static std::vector<const void*> captured_leaves(const NetDesc& d, const Plan& p, const std::vector<const void*>& lp) {
    std::vector<const void*> got;
    for (const Step& st : p.steps) {
        if (st.wave || st.regions) continue;
        const Node& nd = p.nodes[st.node];
        for (int c : {nd.ca, nd.cb})
            if (c >= 0 && c < d.n) got.push_back(lp[c]);
    }
    return got;
}

// (Re)capture the per-group graph when the leaves, the timing hooks or the
// instance layout changed.
static tn_status ensure_graph(const NetDesc& d, Plan& p, const std::vector<const void*>& all_leaves, int pf,
                              int pc, std::string& err) {
    const bool h = pc > 0;
    const std::vector<const void*> lp = captured_leaves(d, p, all_leaves);
    cudaGraph_t& graph = h ? p.graph_h : p.graph;
    cudaGraphExec_t& gexec = h ? p.gexec_h : p.gexec;
    std::vector<const void*>& gptrs = h ? p.graph_ptrs_h : p.graph_ptrs;
    int& gpf = h ? p.graph_prof_first_h : p.graph_prof_first;
    int& gpc = h ? p.graph_prof_count_h : p.graph_prof_count;
    int& ginst = h ? p.graph_inst_h : p.graph_inst;
    int& gstep = h ? p.graph_step_h : p.graph_step;
    if (gexec && gptrs == lp && gpf == pf && gpc == pc && ginst == p.cfg_inst && gstep == p.cfg_step)
        return TN_OK;
    if (gexec) CK(cudaGraphExecDestroy(gexec));
    if (graph) CK(cudaGraphDestroy(graph));
    gexec = nullptr;
    graph = nullptr;
    while ((int)p.prof_placeholder.size() < pc + 1) {
        cudaEvent_t ev;
        CK(cudaEventCreate(&ev));
        p.prof_placeholder.push_back(ev);
    }
    CK(cudaStreamBeginCapture(p.cap_stream, cudaStreamCaptureModeThreadLocal));
    cudaError_t e = enqueue_slice(d, p, p.cap_stream, pc ? p.prof_placeholder.data() : nullptr, pf, pc);
    cudaError_t e2 = cudaStreamEndCapture(p.cap_stream, &graph);
    CK(e);
    CK(e2);
    CK(cudaGraphInstantiate(&gexec, graph, 0));
    gptrs = lp;
    gpf = pf;
    gpc = pc;
    ginst = p.cfg_inst;
    gstep = p.cfg_step;
    if (!h) return TN_OK;
    p.prof_nodes.assign(pc + 1, nullptr);
    if (pc) {
        size_t nn = 0;
        CK(cudaGraphGetNodes(graph, nullptr, &nn));
        std::vector<cudaGraphNode_t> all(nn);
        CK(cudaGraphGetNodes(graph, all.data(), &nn));
        for (auto g : all) {
            cudaGraphNodeType t;
            CK(cudaGraphNodeGetType(g, &t));
            if (t != cudaGraphNodeTypeEventRecord) continue;
            cudaEvent_t ev;
            CK(cudaGraphEventRecordNodeGetEvent(g, &ev));
            for (int i = 0; i <= pc; ++i)
                if (p.prof_placeholder[i] == ev) p.prof_nodes[i] = g;
        }
        for (auto g : p.prof_nodes)
            if (!g) {
                err = "internal: timing event node missing from the captured graph";
                return TN_ECUDA;
            }
    }
    return TN_OK;
}

static tn_status upload_leaf_sizes(const NetDesc& d, Plan& p, int G, const std::vector<int64_t>& leaf_is,
                                   cudaStream_t stream, std::string& err) {
    std::vector<int64_t> nf(d.n);
    for (int v = 0; v < d.n; ++v) {
        const int64_t is = leaf_is.empty() ? 0 : leaf_is[v];
        nf[v] = ((int64_t)(G - 1) * is + d.leaves[v].size) * (d.is_complex() ? 2 : 1);
    }
    if (nf == p.leaf_nfloat_uploaded) return TN_OK;
    CK(cudaMemcpyAsync(p.leaf_nfloat_dev, nf.data(), sizeof(int64_t) * d.n, cudaMemcpyHostToDevice, stream));
    CK(cudaStreamSynchronize(stream));
    p.leaf_nfloat_uploaded = nf;
    return TN_OK;
}

constexpr int64_t kHostOneCopy = int64_t(1) << 13;  // doubles of a host result that is copied together with its exponent

tn_status run_plan(NetDesc& d, Plan& p, void* unit, int64_t begin, int64_t count,
                   const tn_options& o, void* out, int out_mem, int64_t* out_exp2,
                   cudaStream_t stream, std::string& err) {
    (void)unit;
    const int n = d.n;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    CK(cudaStreamIsCapturing(stream, &cap));
    const bool capturing = cap != cudaStreamCaptureStatusNone;
    // profiling hooks
    int pf = 0, pc = 0;
    const cudaEvent_t* uev = nullptr;
    if (o.prof_events && o.prof_count > 0) {
        pf = o.prof_first;
        pc = o.prof_count;
        if (pf < 0 || pf + pc > (int)p.steps.size()) {
            err = "profiling step range out of bounds";
            return TN_EINVAL;
        }
        uev = reinterpret_cast<const cudaEvent_t*>(o.prof_events);
    }
    // slices per launch group (instances); the device state was sized for it
    int G = o.slice_batch > 1 ? o.slice_batch : 1;
    if (G > count) G = (int)count;
    if (G > p.alloc_inst) {
        err = "internal: slice batch exceeds the allocated instances";
        return TN_ECUDA;
    }
    if (capturing && (p.cfg_inst != G || p.cfg_step != 1)) {
        err = "the first call with a new slice batch must run outside stream capture";
        return TN_EUNSUPPORTED;
    }
    tn_status st = configure_instances(d, p, G, 1, std::vector<int64_t>(), stream, err);
    if (st != TN_OK) return st;
    if (!capturing) {
        st = upload_leaf_sizes(d, p, 1, std::vector<int64_t>(), stream, err);
        if (st != TN_OK) return st;
    }
    std::vector<const void*> lp;
    st = prepare_leaves(d, p, capturing, lp, stream, err);
    if (st != TN_OK) return st;
    const int64_t n_acc = p.n_out * (d.is_complex() ? 2 : 1);
    // the last group's fold writes the result: to the caller's device buffers,
    // or (host outputs) to a staging buffer [result | exponent] for one copy
    double* res = static_cast<double*>(out);
    int64_t* res_exp = out_exp2;
    if (out_mem == TN_MEM_HOST) {
        if (!p.out_stage) CK(cudaMalloc(&p.out_stage, sizeof(double) * (n_acc + 1)));
        res = p.out_stage;
        res_exp = reinterpret_cast<int64_t*>(p.out_stage + n_acc);
    }
    CK(launch_call_begin(p.leaf_ptr_dev, p.leaf_nfloat_dev, p.leaf_nfloat_uploaded.data(), p.leafmax, n, p.ctl, begin,
                         begin + count, nullptr, 0, res, res_exp, stream));
    const int64_t groups = (count + G - 1) / G;
    const bool use_graph = !o.no_graph && !capturing;
    if (use_graph) {
        st = ensure_graph(d, p, lp, pf, pc, err);
        if (st != TN_OK) return st;
        cudaGraphExec_t gx = pc ? p.gexec_h : p.gexec;
        for (int i = 0; i < pc + (pc ? 1 : 0); ++i)
            CK(cudaGraphExecEventRecordNodeSetEvent(gx, p.prof_nodes[i], uev[i]));
        for (int64_t s = 0; s < groups; ++s) CK(cudaGraphLaunch(gx, stream));
    } else {
        for (int64_t s = 0; s < groups; ++s) CK(enqueue_slice(d, p, stream, uev, pf, pc));
    }
    if (out_mem == TN_MEM_HOST) {
        // few outputs: value and exponent in one copy; many: straight into the
        // caller's memory (a second pass over them on the host costs more than
        // the second copy: 2^22 complex outputs 8.8 ms, 3.9 this way;
        // 2^12 the same)
        const bool few = n_acc <= kHostOneCopy;
        std::vector<double> host(few ? (size_t)n_acc + 1 : 1);
        if (!few) CK(cudaMemcpyAsync(host.data(), res_exp, sizeof(double), cudaMemcpyDeviceToHost, stream));
        CK(cudaMemcpyAsync(few ? host.data() : static_cast<double*>(out), p.out_stage,
                           sizeof(double) * (few ? n_acc + 1 : n_acc), cudaMemcpyDeviceToHost, stream));
        CK(cudaStreamSynchronize(stream));
        if (few) std::memcpy(out, host.data(), sizeof(double) * n_acc);
        std::memcpy(out_exp2, &host.back(), sizeof(int64_t));
    }
    return TN_OK;
}

tn_status run_instances(NetDesc& d, Plan& p, void* unit, int n_inst, const int64_t* leaf_is_arr,
                        double* out, int64_t* out_exp2, int out_mem, cudaStream_t stream,
                        std::string& err) {
    (void)unit;
    const int n = d.n;
    const int nn = (int)p.nodes.size();
    const size_t eb = d.elem_bytes();
    if (p.d_sliced != 1 || p.n_out != 1) {
        err = "tn_contract_instances: the network must be scalar and the tree unsliced";
        return TN_EUNSUPPORTED;
    }
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    CK(cudaStreamIsCapturing(stream, &cap));
    if (cap != cudaStreamCaptureStatusNone) {
        err = "tn_contract_instances: not available during stream capture";
        return TN_EUNSUPPORTED;
    }
    const int G = n_inst;
    if (G > p.alloc_inst) {
        err = "internal: instances exceed the allocation";
        return TN_ECUDA;
    }
    std::vector<int64_t> leaf_is(n, 0);
    if (leaf_is_arr)
        for (int v = 0; v < n; ++v) leaf_is[v] = leaf_is_arr[v];
    tn_status st = configure_instances(d, p, G, 0, leaf_is, stream, err);
    if (st != TN_OK) return st;
    st = upload_leaf_sizes(d, p, G, leaf_is, stream, err);
    if (st != TN_OK) return st;
    if (p.inst_roots_n != G) {
        const Node& root = p.nodes.back();
        std::vector<BatchRoot> roots(G);
        for (int i = 0; i < G; ++i) {
            roots[i].root = (char*)p.ws + ((int64_t)i * p.ws_elems + root.ws_off) * eb;
            roots[i].exp = p.exps + (int64_t)i * nn + (nn - 1);
            roots[i].max = p.maxabs + (int64_t)i * nn + (nn - 1);
            roots[i].is_c = d.is_complex();
            roots[i].pad = 0;
        }
        CK(cudaMemcpyAsync(p.inst_roots_dev, roots.data(), sizeof(BatchRoot) * G, cudaMemcpyHostToDevice, stream));
        CK(cudaStreamSynchronize(stream));
        p.inst_roots_n = G;
    }
    std::vector<const void*> lp;
    st = prepare_leaves(d, p, false, lp, stream, err);
    if (st != TN_OK) return st;
    CK(launch_call_begin(p.leaf_ptr_dev, p.leaf_nfloat_dev, p.leaf_nfloat_uploaded.data(), p.leafmax, n, p.ctl, 0, 1,
                         nullptr, 0, nullptr, nullptr, stream));
    st = ensure_graph(d, p, lp, 0, 0, err);
    if (st != TN_OK) return st;
    CK(cudaGraphLaunch(p.gexec, stream));
    cudaMemcpyKind kind = out_mem == TN_MEM_HOST ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice;
    CK(cudaMemcpyAsync(out, p.inst_out_dev, sizeof(double) * 2 * G, kind, stream));
    CK(cudaMemcpyAsync(out_exp2, p.inst_exp_dev, sizeof(int64_t) * G, kind, stream));
    if (out_mem == TN_MEM_HOST) CK(cudaStreamSynchronize(stream));
    return TN_OK;
}


tn_status make_generic_args_node(const NetDesc& d, const Plan& p, const Node& nd, GenericArgs& g,
                                 std::string& err) {
    return fill_generic(d, p, nd, g, err);
}

// Tensor-core choice for a tiled node in a reduced-precision mode: the
// GEMM tile needs >= 128 accumulator rows, >= 128 real accumulator columns
// (a complex node: >= 64, its 32 complex columns expand to 64 real ones that
// fill half of the 128-column tile, the rest is padding the epilogue drops)
// and K >= 16.  A complex node puts its larger
// operand in the row role (the column operand is expanded to two real rows
// per column).  The packed operands live in the shared P buffer, which
// grows to hold them.
bool make_tensor_core(const NetDesc& d, tn_mode mode, Node& nd, int64_t& split_elems, int copies) {
    TileArgs& t = nd.tile;
    if (mode == TN_MODE_FP32 || t.cfg == kTileDot || t.nk < 4 || t.nbatch > 65535) return false;
    const bool c = d.is_complex();
    int swap = 0;
    if (c) {
        if (std::max(t.nm, t.nn) < 7 || std::min(t.nm, t.nn) < 5) return false;
        swap = t.nn > t.nm ? 1 : 0;
    } else if (t.nm < 7 || t.nn < 7) {
        return false;
    }
    t.tc_swap = swap;
    t.split = 1;
    t.kchunk = int64_t(1) << t.nk;
    const int prec = tc_prec_of_mode(mode);
    // the planar layout (asked for by the autotuner's planar variant, or for
    // every eligible node by the diagnostic switch TN_PLANAR=1, read when a
    // plan is built) needs a complex node in a split precision with >= 128
    // complex rows and columns
    if (const char* e = getenv("TN_PLANAR"))
        if (e[0] == '1') t.tc_planar = 1;
    // 256-column GEMMs run on CTA pairs (pair MMA) where the row tiles pair
    // up; the diagnostic switch TN_NO_PAIR=1, read when a plan is built,
    // keeps the single-CTA GEMM
    t.tc_nopair = 0;
    if (const char* e = getenv("TN_NO_PAIR"))
        if (e[0] == '1') t.tc_nopair = 1;
    t.tc_planar = (t.tc_planar && c && (prec == 1 || prec == 2 || prec == 4) && t.nm >= 7 && t.nn >= 7 &&
                   !t.tc_bn128) ? 1 : 0;
    // K split: the grid should fill whole waves of the SMs (one CTA
    // each); split only while every part keeps >= 8 k-blocks
    {
        const TcGeom g0 = tc_geom(t, c, prec);
        const double tiles = (double)t.nbatch * (g0.rows_r / 128) * (g0.cols_q / g0.bn) * copies;
        double best = 0.0;
        for (int s = 1; s <= 16 && g0.nkb / s >= 8; s *= 2) {
            const double w = tiles * s / (double)sm_count();
            const double eff = w / std::ceil(w);
            if (eff > best + 0.03) {
                best = eff;
                t.split = s;
            }
        }
        if (t.nbatch * (int64_t)t.split > 65535) t.split = 1;
        // partials that do not fit L2 cost HBM traffic (written, read, and the
        // sum written): split only if the fuller waves gain more.  Times in us:
        // a k-block of a tile on the tensor pipe at 1.9 GHz per product of the
        // precision, bytes at 6.5 TB/s.  A 2^13 x 2^12 x 2^10 node, 13.5 waves:
        // 17 us of GEMM gained by two parts against 125 us of reduction and
        // as many partial stores again (call 1191 -> 1050 us without them).
        // Several copies per launch keep their split: a gradient step of 64
        // copies is 2% faster without, but the other order of its sums showed
        // as 1.6e-5 instead of 1.1e-5 error on an ill-conditioned loss.
        const double out_bytes = (double)t.nbatch * (double)(int64_t(1) << (t.nm + t.nn)) * d.elem_bytes();
        if (t.split > 1 && copies == 1 && t.split * out_bytes > 126e6) {
            const double products = prec == 0 ? 1.0 : (g0.planar ? 4.0 : 3.0);
            const double t_kb = 0.27 * products * g0.bn / 256.0;
            auto gemm_us = [&](int s) {
                return std::ceil(tiles * s / (double)sm_count()) * (double)(g0.nkb / s) * t_kb;
            };
            if (gemm_us(1) - gemm_us(t.split) < 2.0 * t.split * out_bytes / 6.5e6) t.split = 1;
        }
    }
    const int64_t eb = d.elem_bytes();
    split_elems = std::max(split_elems, (tc_geom(t, c, prec).total + eb - 1) / eb);
    nd.kind = kTensorCore;
    return true;
}

// ---- autotuner: the kernel of every node that runs alone in its launch
// step is chosen by timing each candidate on the device.
static cudaError_t launch_node(const NetDesc& d, const Plan& p, const Node& nd, cudaStream_t s) {
    if (nd.kind == kTensorCore)
        return launch_tc(nd.tile, tc_prec_of_mode(p.mode),
                         d.is_complex(), s);
    return launch_tile(nd.tile, d.is_complex(), s);
}

// Node k rebuilt as variant v (1..4: tile shape, kVariantTC: tensor core),
// keeping its device bindings; false if the variant does not apply.
static bool make_variant(const NetDesc& d, const Plan& p, int k, int v, Node& out, int64_t& split_elems,
                         int split_mult = 1) {
    const Node& nd = p.nodes[k];
    Node t = nd;
    const bool tcv = v == kVariantTC || v == kVariantTC128 || v == kVariantTCPlanar;
    if (!plan_tile(d, p, t, split_elems, tcv ? 0 : v)) return false;
    if (v == kVariantTC128) t.tile.tc_bn128 = 1;
    if (v == kVariantTCPlanar) t.tile.tc_planar = 1;
    if (t.tile.cfg == kTileDot) return false;
    t.kind = kTiled;
    if (tcv && !make_tensor_core(d, p.mode, t, split_elems)) return false;
    if (!tcv && split_mult > 1) {
        // finer K split: more blocks for short grids over long K (>= 2 K tiles each)
        TileArgs& a = t.tile;
        const int TK = a.cfg == kTile4x1024 ? 4 : 16;
        const int64_t K = int64_t(1) << a.nk, ktiles = (K + TK - 1) / TK;
        const int split = a.split * split_mult;
        if (split > 256 || ktiles / split < 2 || a.nbatch * (int64_t)split > 65535) return false;
        a.split = split;
        a.kchunk = ((ktiles + split - 1) / split) * TK;
        split_elems = std::max(split_elems, (int64_t)split * a.nbatch * (int64_t(1) << (a.nm + a.nn)));
    }
    TileArgs& a = t.tile;
    const TileArgs& o = nd.tile;
    a.A = o.A;
    a.B = o.B;
    a.C = o.C;
    a.P = o.P;
    a.sla = o.sla;
    a.slb = o.slb;
    a.ctl = o.ctl;
    a.sc = o.sc;
    a.conj_a = o.conj_a;
    a.conj_b = o.conj_b;
    a.t_done = o.t_done;
    a.in = o.in;
    out = t;
    return true;
}

tn_status autotune_plan(NetDesc& d, Plan& p, int reps, int32_t* choice, cudaStream_t s, std::string& err) {
    const int nn = (int)p.nodes.size();
    if (choice)
        for (int k = 0; k < nn; ++k) choice[k] = 0;
    if (reps < 1) reps = 1;
    // nodes that run alone in their step, on a tiled or tensor-core kernel
    std::vector<int> tune;
    for (const Step& st : p.steps)
        if (!st.wave && !st.regions) {
            const Node& nd = p.nodes[st.node];
            if ((nd.kind == kTiled && nd.tile.cfg != kTileDot) || nd.kind == kTensorCore) tune.push_back(st.node);
        }
    if (tune.empty()) return TN_OK;
    // bind this call's leaves (their values do not matter for timing)
    tn_status st = configure_instances(d, p, 1, 1, std::vector<int64_t>(), s, err);
    if (st != TN_OK) return st;
    st = upload_leaf_sizes(d, p, 1, std::vector<int64_t>(), s, err);
    if (st != TN_OK) return st;
    std::vector<const void*> lp;
    st = prepare_leaves(d, p, false, lp, s, err);
    if (st != TN_OK) return st;
    CK(launch_leaf_max(p.leaf_ptr_dev, p.leaf_nfloat_dev, p.leaf_nfloat_uploaded.data(), p.leafmax, d.n, s));
    // candidates and the shared P buffer they need
    std::vector<std::vector<std::pair<int, Node>>> cand(nn);
    int64_t split_elems = 0;
    for (int k : tune) {
        const Node& nd = p.nodes[k];
        const int vc = nd.tile.nm + nd.tile.nn + nd.tile.nk + nd.tile.nb;  // log2 of the products
        Node tc;
        const bool has_tc = !p.no_tensor_cores && make_variant(d, p, k, kVariantTC, tc, split_elems);
        if (has_tc) {
            cand[k].push_back({kVariantTC, tc});
            if (tc.tile.split > 1) {  // the same GEMM without its K split (no reduction launch)
                Node t1 = tc;
                t1.tile.split = 1;
                cand[k].push_back({kVariantTC, t1});
            }
            // the planar layout (complex nodes in a split precision)
            Node tpl;
            if (make_variant(d, p, k, kVariantTCPlanar, tpl, split_elems) && tpl.tile.tc_planar) {
                cand[k].push_back({kVariantTCPlanar, tpl});
                if (tpl.tile.split > 1) {
                    Node t1 = tpl;
                    t1.tile.split = 1;
                    cand[k].push_back({kVariantTCPlanar, t1});
                }
            }
            // 128-column tiles where 256 were chosen: twice the CTAs
            Node tn;
            const TcGeom g_tc = tc_geom(tc.tile, d.is_complex(), tc_prec_of_mode(p.mode));
            if (g_tc.bn == 256 &&
                make_variant(d, p, k, kVariantTC128, tn, split_elems)) {
                cand[k].push_back({kVariantTC128, tn});
                if (tn.tile.split > 1) {
                    Node t1 = tn;
                    t1.tile.split = 1;
                    cand[k].push_back({kVariantTC128, t1});
                }
            }
        }
        // CUDA-core shapes, unless the node is so large that they cannot win
        if (!has_tc || vc < 32)
            for (int v : {int(kTile64x64), int(kTile16x256), int(kTile4x1024), int(kTile256x16), int(kTile128x64),
                          int(kTile128x128)})
                for (int mult : {1, 4}) {
                    Node t;
                    if (v == kTile128x128 && d.is_complex()) continue;  // real nodes only
                    // both 128-row shapes are reported as 6
                    if (make_variant(d, p, k, v, t, split_elems, mult))
                        cand[k].push_back({v == kTile128x128 ? int(kTile128x64) : v, t});
                }
    }
    const int64_t need = (split_elems * (int64_t)d.elem_bytes() + 1023) / 1024 * 1024;
    const int G = std::max(p.alloc_inst, 1);
    if (need > p.split_bytes) {
        CK(cudaStreamSynchronize(s));
        if (p.split_buf) CK(cudaFree(p.split_buf));
        p.split_buf = nullptr;
        CK(cudaMalloc(&p.split_buf, need * G));
        p.split_bytes = need;
        for (auto& nd : p.nodes) nd.tile.P = p.split_buf;
        for (auto& g : p.gen) g.P = p.split_buf;
        for (auto& cs : cand)
            for (auto& c : cs) c.second.tile.P = p.split_buf;
    }
    // a valid control block (slice 0 of the range) for the single-node launches
    CK(launch_begin_call(p.ctl, 0, p.d_sliced, nullptr, 0, s));
    cudaEvent_t e0, e1;
    CK(cudaEventCreate(&e0));
    CK(cudaEventCreate(&e1));
    for (int k : tune) {
        float best = 1e30f;
        int best_v = 0;
        Node best_node = p.nodes[k];
        for (auto& c : cand[k]) {
            c.second.tile.in = p.nodes[k].tile.in;
            cudaError_t e = launch_node(d, p, c.second, s);
            if (e == cudaSuccess) e = cudaEventRecord(e0, s);
            for (int r = 0; r < reps && e == cudaSuccess; ++r) e = launch_node(d, p, c.second, s);
            if (e == cudaSuccess) e = cudaEventRecord(e1, s);
            if (e == cudaSuccess) e = cudaEventSynchronize(e1);
            float ms = 0.f;
            if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
            if (e != cudaSuccess) {
                cudaEventDestroy(e0);
                cudaEventDestroy(e1);
                err = std::string("autotune: ") + cudaGetErrorString(e);
                return TN_ECUDA;
            }
            // the planner's choice stays unless another is clearly faster
            const bool planned = c.second.kind == p.nodes[k].kind &&
                                 (c.second.kind == kTensorCore || c.second.tile.cfg == p.nodes[k].tile.cfg);
            const float eff = planned ? ms * 0.95f : ms;
            if (eff < best) {
                best = eff;
                best_v = c.first;
                best_node = c.second;
            }
        }
        p.nodes[k] = best_node;
        if (choice) choice[k] = best_v;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    // the control block must not look like a finished call; the next call
    // rebuilds the instance configuration and the captured graph
    CK(cudaStreamSynchronize(s));
    Control zero{};
    CK(cudaMemcpy(p.ctl, &zero, sizeof(Control), cudaMemcpyHostToDevice));
    if (p.descs_dev) {
        std::vector<TileArgs> descs(nn);
        for (int k = 0; k < nn; ++k) descs[k] = p.nodes[k].tile;
        CK(cudaMemcpy(p.descs_dev, descs.data(), sizeof(TileArgs) * nn, cudaMemcpyHostToDevice));
    }
    p.cfg_inst = -1;
    p.graph_inst = p.graph_inst_h = -2;
    p.tuned = true;
    return TN_OK;
}

#undef CK

bool plan_tile_node(const NetDesc& d, const Plan& p, Node& nd, int64_t& split_elems) {
    return plan_tile(d, p, nd, split_elems);
}

tn_status make_generic_args(const NetDesc& d, const Plan& p, int k, GenericArgs& g, std::string& err) {
    return fill_generic(d, p, p.nodes[k], g, err);
}

void plan_info(const NetDesc& d, const Plan& p, int64_t ws_elems, double out[8]) {
    out[0] = p.W;
    out[1] = p.C;
    out[2] = (double)p.d_sliced;
    out[3] = (d.is_complex() ? 8.0 : 2.0) * p.C * (double)p.d_sliced;
    out[4] = (double)std::max(p.ws_elems, ws_elems) * (double)d.elem_bytes();
    int cnt[3] = {0, 0, 0};
    for (auto& nd : p.nodes) cnt[nd.kind]++;
    out[5] = cnt[kTiled];
    out[6] = cnt[kTensorCore];
    out[7] = cnt[kGeneric];
}

void free_device(Plan& p) {
    free_grad(p);
    if (p.gexec) cudaGraphExecDestroy(p.gexec);
    if (p.graph) cudaGraphDestroy(p.graph);
    if (p.gexec_h) cudaGraphExecDestroy(p.gexec_h);
    if (p.graph_h) cudaGraphDestroy(p.graph_h);
    p.gexec_h = nullptr;
    p.graph_h = nullptr;
    p.graph_ptrs_h.clear();
    p.graph_inst_h = p.graph_step_h = -1;
    for (auto ev : p.prof_placeholder) cudaEventDestroy(ev);
    p.prof_placeholder.clear();
    p.prof_nodes.clear();
    p.graph = nullptr;
    if (p.cap_stream) cudaStreamDestroy(p.cap_stream);
    if (p.ws) cudaFree(p.ws);
    if (p.maxabs) cudaFree(p.maxabs);
    if (p.exps) cudaFree(p.exps);
    if (p.ctl) cudaFree(p.ctl);
    if (p.acc) cudaFree(p.acc);
    if (p.out_stage) cudaFree(p.out_stage);
    p.out_stage = nullptr;
    if (p.leafmax) cudaFree(p.leafmax);
    if (p.split_buf) cudaFree(p.split_buf);
    p.split_buf = nullptr;
    if (p.descs_dev) cudaFree(p.descs_dev);
    if (p.items_dev) cudaFree(p.items_dev);
    if (p.flow_deps_dev) cudaFree(p.flow_deps_dev);
    if (p.region_dev) cudaFree(p.region_dev);
    p.region_dev = nullptr;
    p.leaf_is_dev = nullptr;
    p.flow_deps_dev = nullptr;
    p.flow_cnt_dev = nullptr;
    if (p.inst_roots_dev) cudaFree(p.inst_roots_dev);
    if (p.inst_out_dev) cudaFree(p.inst_out_dev);
    if (p.inst_exp_dev) cudaFree(p.inst_exp_dev);
    p.inst_roots_dev = nullptr;
    p.inst_out_dev = nullptr;
    p.inst_exp_dev = nullptr;
    p.cfg_inst = -1;
    p.inst_roots_n = 0;
    p.graph_inst = -1;
    p.graph_step = -1;
    p.leaf_nfloat_uploaded.clear();
    p.descs_dev = nullptr;
    p.items_dev = nullptr;
    if (p.leaf_ptr_dev) cudaFree(p.leaf_ptr_dev);
    if (p.leaf_nfloat_dev) cudaFree(p.leaf_nfloat_dev);
    p.leafmax = nullptr;
    p.leaf_ptr_dev = nullptr;
    p.leaf_nfloat_dev = nullptr;
    p.leaf_ptr_uploaded.clear();
    p.captured = false;
    p.gexec = nullptr;
    p.cap_stream = nullptr;
    p.ws = nullptr;
    p.maxabs = nullptr;
    p.exps = nullptr;
    p.ctl = nullptr;
    p.acc = nullptr;
    p.graph_ptrs.clear();
}

}  // namespace tn
