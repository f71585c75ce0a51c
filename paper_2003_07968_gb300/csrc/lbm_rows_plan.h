// lbm_rows_plan.h -- host side of the row kernels (lbm_rows.cuh): how lattices
// are cut into strips of columns and bands of rows.
#pragma once
#include <algorithm>
#include <vector>

#include "lbm_device.cuh"

namespace pplbm {

constexpr int kRowCols = 60;  // columns a warp advances at most (it holds 64)

// First column of strip k of the n = strip_count(nx, cols) strips over nx columns:
// even, two of them at most `cols` (an even number) apart, as equal as that allows.
inline int strip_edge(int nx, int n, int k) {
    const int pairs = (nx + 1) / 2;
    return std::min(nx, 2 * (int)(((int64_t)pairs * k + n - 1) / n));
}
inline int strip_count(int nx, int cols = kRowCols) { return (nx + cols - 1) / cols; }
inline int band_edge(int ny, int n, int k) { return (int)((int64_t)ny * k / n); }

// ---- one step a launch (k_rows): row items, each the work of one warp
constexpr int kRowWarps = 4;  // warps of a block, each on an item of its own
// entry of an item list: (lattice, x0, y0, rows | width << 24)
inline int pack_rows(int rows, int width) { return rows | (width << 24); }

// Rows of an item: one wave of the `warps` the GPU holds where that makes
// items of at most 16 rows (a second, partly filled wave costs more than the
// three extra rows an item pulls and computes psi for), else about five
// waves, of at most 64 rows.
inline int row_item_height(const std::vector<LatDev>& lats, int64_t warps) {
    int64_t units = 0;
    for (const LatDev& L : lats) units += (int64_t)strip_count(L.nx) * L.ny;
    for (int h = 2; h <= 16; ++h) {
        int64_t n = 0;
        for (const LatDev& L : lats) n += (int64_t)strip_count(L.nx) * ((L.ny + h - 1) / h);
        if (n <= warps) return h;
    }
    return (int)std::min<int64_t>(64, std::max<int64_t>(8, units / (5 * warps)));
}
// The items of one lattice, bands one after another, a band's strips side by side.
inline void row_items(const LatDev& L, int lattice, int h, std::vector<int4>& out,
                      int cols = kRowCols) {
    const int ns = strip_count(L.nx, cols), nb = (L.ny + h - 1) / h;
    for (int b = 0; b < nb; ++b) {
        const int y0 = band_edge(L.ny, nb, b), y1 = band_edge(L.ny, nb, b + 1);
        for (int s = 0; s < ns; ++s) {
            const int x0 = strip_edge(L.nx, ns, s), x1 = strip_edge(L.nx, ns, s + 1);
            out.push_back(make_int4(lattice, x0, y0, pack_rows(y1 - y0, x1 - x0)));
        }
    }
}

// ---- two steps a launch (k_rows2): an item is the work of a pair of warps
constexpr int kPairCols = 56;   // columns of an item at most (64 held, 4 lost a side)
constexpr int kPairDepth = 8;   // rows of the ring between a pair's warps
constexpr int kPairs = 4;       // pairs of a block
constexpr size_t kPairSmem = (size_t)kPairs * kPairDepth * 9 * 64 * sizeof(float);

// Rows of an item, `pairs`: the pairs of warps the GPU holds.  One wave while
// that makes items of about 100 rows at most, then even waves of about 72
// rows, for one lattice 4 at most (a last wave that is nearly empty costs
// more than the rows that items share).  Measured per step: 2100 x 1700 46 us
// in one wave of 53 rows, 53-60 in items of 32 to 64; 3000^2 106 us in two
// waves of 67, 112-144 in items of 48 to 192; 512 lattices 726 us in items of
// 96 rows, 793 in four waves of 230.
//
// Lattices of few rows make an item however low it is, and beside many of them
// no height, or only a large one, keeps the count of items within the waves: a
// taller lattice's items would then run on long after all others.  So the
// height is at most twice an even share of the rows, and beyond that the one
// at which the lattices' work, not their items, fills the waves.  2000 lattices
// of 16^2 and one of 512^2: items of 512 rows 288 us a step, of 31 43 (tile
// kernel 78); 5000 of 32^2 and one of 2048^2: 1221 and 200 us (478).
inline int pair_item_height(const std::vector<LatDev>& lats, int64_t pairs) {
    int64_t units = 0, most = 0;
    for (const LatDev& L : lats) {
        units += (int64_t)strip_count(L.nx, kPairCols) * L.ny;
        most = std::max<int64_t>(most, L.ny);
    }
    const bool one = lats.size() == 1;
    int64_t waves = std::max<int64_t>(1, (units + 36 * pairs) / (72 * pairs));
    if (one) waves = std::min<int64_t>(waves, 4);
    const int64_t share = std::max<int64_t>(4, units / (waves * pairs));
    for (int64_t h = share; h < most && (one || h <= 2 * share); ++h) {
        int64_t n = 0;  // items
        for (const LatDev& L : lats) n += strip_count(L.nx, kPairCols) * ((L.ny + h - 1) / h);
        if (n <= waves * pairs) return (int)h;
    }
    if (one || 2 * share >= most) return (int)most;
    for (int64_t h = share; h < most; ++h) {
        int64_t rows = 0;  // a lattice below h counts with its rows, others with whole items
        for (const LatDev& L : lats)
            rows += strip_count(L.nx, kPairCols) * (L.ny < h ? L.ny : (L.ny + h - 1) / h * h);
        if (rows <= waves * pairs * h) return (int)h;
    }
    return (int)most;
}
// ---- row kernel or tile kernel
// Estimated microseconds of a step on the row kernel of the storage (one: one
// lattice, by value; else the batch instance) over items of `height` rows, and
// on the tile kernel the handle has (tensor: the TMA kernel's 32 x 16 tiles;
// else plain loads).  A warp's rows come one after another, whatever the
// others do, so a launch lasts as long as its tallest item or its waves of
// items; what the warps of an SM share (the FP32 pipe) adds a part by the total
// of rows.  A strip costs its 64 columns even if it holds 32 (a lattice 64
// columns wide is two such strips and four tiles), which is where the tile
// kernel wins.  Fitted to 65 shapes in each storage, BGK and MRT, from one
// lattice to 5000 and 16 k to 17 M sites: nine of ten of the row kernels' times
// lie within 12 %, of the tile kernels' within 20 % (theirs vary with the pitch).
inline double rows_us(const std::vector<LatDev>& lats, int height, bool f16, bool mrt, bool one,
                      int64_t sms) {
    const int cols = f16 ? kRowCols : kPairCols, halo = f16 ? 3 : 6;
    const int64_t slots = sms * (f16 ? 4 * kRowWarps : 2 * kPairs);
    int64_t n = 0, work = 0, tallest = 0;
    for (const LatDev& L : lats) {
        const int64_t ns = strip_count(L.nx, cols), nb = (L.ny + height - 1) / height;
        n += ns * nb;
        work += ns * (L.ny + halo * nb);
        tallest = std::max<int64_t>(tallest, (L.ny + nb - 1) / nb + halo);
    }
    const double waves = (double)((n + slots - 1) / slots);
    const double chain = std::max((double)tallest, waves * (double)work / (double)n);
    const double start = f16 ? (one ? 7.0 : 5.0) : 0.5;
    const double per_row = f16 ? (one ? 0.3 : 0.09) : (one ? 0.43 : 0.61);
    const double shared = f16 ? (one ? 1.09 : 1.5) : (one ? 0.35 : 0.25);
    return start + (chain * per_row + (double)work / (double)slots * shared) *
                       (mrt ? (one ? 1.17 : 1.12) : 1.0);
}
inline double tiles_us(const std::vector<LatDev>& lats, bool mrt, bool tensor) {
    double us = 0.0;
    for (const LatDev& L : lats) {
        const double across = (L.nx + 31) / 32, down = (L.ny + 15) / 16;
        if (lats.size() == 1)  // a tile cut at the right edge is stored without the TMA
            us += down * (0.0088 * (L.nx / 32) + 0.0112 * (across - L.nx / 32));
        else if (tensor)
            us += 0.009 * across * down;
        else
            us += 0.0052 * across * down + 0.0138 / 512.0 * L.nx * L.ny;
    }
    return 4.6 + us * (mrt ? 1.1 : 1.0);
}
// Whether the row kernel takes the lattices.  Measured per step, tile kernel
// against row kernel: 310 lattices of 64^2 30 and 60 us (FP16 storage 32 and
// 42), 400 of 60^2 39 and 59, 1000 of 32^2 26 and 34, one of 64 x 62500 in FP16
// 84 and 116: tiles.  400 of 56^2 39 and 23, 100 of 128^2 38 and 34, 200 of
// 100^2 62 and 37: rows.  Estimates up to 5 % above go to the rows too (their
// errors there: 128^2 takes 10 % less on them in either storage), and one
// FP32 lattice up to 15 % above (61 x 21001: 32 us on either).
inline bool rows_pay(const std::vector<LatDev>& lats, int height, bool f16, bool mrt, bool one,
                     bool tensor, int64_t sms) {
    return rows_us(lats, height, f16, mrt, one, sms) <
           (one && !f16 ? 1.15 : 1.05) * tiles_us(lats, mrt, tensor);
}

// 32-bit offsets of k_rows2: a lattice's rows in a plane take less than 4 GB
inline bool rows_fit(const LatDev& L, int es) {
    return ((int64_t)L.ny + 2 * GY) * L.pitch * es < (int64_t)1 << 32;
}

// ---- resident lattices: one tile a block, kept in shared memory for many steps
constexpr int kResWarps = 8;            // warps of a block, one row each at a time
// shared memory of a block: half an SM's, whatever its tile needs, so that any
// two blocks of any launches share an SM (launches in flight are counted so)
constexpr int kResSmem = 113 * 1024;
constexpr int kResRows = 96;            // rows of a tile at most
constexpr int kResMail = 1088;          // packets of a mailbox slot at most
constexpr int kResBlocks = 480;         // blocks of a launch at most

// packets of a tile's halo (three values each; see k_resident)
constexpr int res_packets(int rows, int wd) { return 20 * ((wd + 2) / 3 + (rows + 2) / 3) + 40; }
static_assert(res_packets(kResRows, kRowCols) <= kResMail, "a tile's halo fits its mailbox");
static_assert((int64_t)kResBlocks * 2 * kResMail < 1 << 20, "a packet's place takes 20 bits");
// shared memory of a tile: psi, packet table, lattice constants, the box (and
// the elements a line's last packet may read past it)
inline size_t res_smem(int rows, int wd, int es) {
    return (size_t)(rows + 2) * 256 + (size_t)res_packets(rows, wd) * 8 + sizeof(LatDev) +
           (size_t)9 * (rows + 4) * 64 * es + 256 * es;
}
// rows of the tallest tile that fits
inline int res_rows(int es) {
    int r = 2;
    while (r < kResRows && res_smem(r + 1, kRowCols, es) <= (size_t)kResSmem &&
           9 * (r + 5) * 64 <= 65536)
        ++r;
    return r;
}

struct ResTile {
    int32_t lattice, x0, wd, y0, rows;
    int32_t nbr[8];  // tiles above left, above, above right, left, right, below left, below, below right
    int32_t wd_w, wd_e;  // widths of the left and right neighbours
    int32_t gr_n, gr_s;  // (rows + 2) / 3 of the tiles above and below
};
struct ResArgs {
    StepArgs a;
    const ResTile* tiles;
    uint4* mail;      // [tile][2][slot]
    uint32_t* epoch;  // per tile: steps so far (all equal between launches)
    int slot;         // packets of a mailbox slot
    int nsteps;
};

// Bands of a lattice of ny rows when tiles of about `rows` rows are aimed at.
inline int res_bands(int ny, int rows) { return std::max(1, std::min((ny + rows - 1) / rows, ny / 2)); }

// Rows of the tiles that a launch takes beside others: with psi's two more they
// are two rounds of the eight warps.
constexpr int kResBeside = 14;

struct ResPlan {
    std::vector<ResTile> tiles;  // none: no plan
    int rows = 0;  // of the tallest tile
};

// The tiles of a handle's lattices if each block of a launch of at most
// `blocks` can keep one: the flattest tiles (of about `low` rows or more) that
// fit.  Flat tiles spread the rows over all SMs, and a step is latency: 256^2
// takes 2.73 us a step in 260 tiles of 4 rows, 2.95 in 145 of 8 and 4.3 in 60
// of 21.
inline ResPlan plan_resident(const std::vector<LatDev>& lats, int blocks, int es, int low = 2) {
    ResPlan P;
    const int most = res_rows(es);
    int h = 0;  // the smallest height whose tiles fit
    for (int rows = low; rows <= most && !h; ++rows) {
        int64_t n = 0;
        int tallest = 0;
        for (const LatDev& L : lats) {
            const int nb = res_bands(L.ny, rows);
            n += (int64_t)strip_count(L.nx) * nb;
            tallest = std::max(tallest, (L.ny + nb - 1) / nb);
            if (n > blocks) break;
        }
        if (n <= blocks && tallest <= most) {
            h = rows;
            P.rows = tallest;
        }
    }
    if (!h) return P;
    for (size_t l = 0; l < lats.size(); ++l) {
        const int nx = lats[l].nx, ny = lats[l].ny;
        const int ns = strip_count(nx), nb = res_bands(ny, h), t0 = (int)P.tiles.size();
        auto width = [&](int s) {
            s = (s + ns) % ns;
            return strip_edge(nx, ns, s + 1) - strip_edge(nx, ns, s);
        };
        auto groups = [&](int b) {
            b = (b + nb) % nb;
            return (band_edge(ny, nb, b + 1) - band_edge(ny, nb, b) + 2) / 3;
        };
        for (int s = 0; s < ns; ++s)
            for (int b = 0; b < nb; ++b) {
                ResTile t{};
                t.lattice = (int)l;
                t.x0 = strip_edge(nx, ns, s);
                t.wd = width(s);
                t.y0 = band_edge(ny, nb, b);
                t.rows = band_edge(ny, nb, b + 1) - t.y0;
                int k = 0;
                for (int db = -1; db <= 1; ++db)
                    for (int ds = -1; ds <= 1; ++ds)
                        if (ds || db)
                            t.nbr[k++] = t0 + (s + ds + ns) % ns * nb + (b + db + nb) % nb;
                t.wd_w = width(s - 1);
                t.wd_e = width(s + 1);
                t.gr_n = groups(b - 1);
                t.gr_s = groups(b + 1);
                P.tiles.push_back(t);
            }
    }
    return P;
}

}  // namespace pplbm
