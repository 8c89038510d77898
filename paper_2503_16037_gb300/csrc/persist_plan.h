// The persistent solve's division of the grid (host and device, no CUDA
// types): which groups a block owns, the tile of source values it keeps, and
// every index into it.
//
// Groups of 128 rows are taken strip by strip (strip q: group q of every
// layer) and, inside a strip, in the order zz = 0 (the ground), 1 (layer 0),
// 2, ...: a row gathers from at most R positions of zz away, so the groups
// of one block need, per strip they touch, a box of consecutive zz ("chunks"
// of tl elements: the strip's rows and H rows on either side, whole haloed
// rows of one layer).
#pragma once

#include <stddef.h>
#include <stdint.h>

#include <vector>

#ifdef __CUDACC__
#define PS_HD __host__ __device__ inline
#else
#define PS_HD inline
#endif

namespace tk {

constexpr int kPsRows = 128;      // rows of a group
constexpr int kPsW = 16;          // warps per block
constexpr int kPsMaxSeg = 8;      // strips a block's groups may touch
constexpr int kPsMaxChunk = 96;   // chunks of a block's tile
constexpr int kPsMaxGroups = 64;  // groups of a block
constexpr int kPsDots = 8;        // sums exchanged per publication

struct PsGeom {
    int nx, ny, nz, nxy, gpl, H, nxp, lp, R;
};

struct PsPlan {
    int nb = 0;            // blocks (0: the scene does not fit the persistent solve)
    int nl = 0;            // most groups of a block
    int tl = 0;            // elements per chunk
    int nchunk = 0;        // most chunks of a block
    int wpg = 0;           // warps that share a group: warp wi adds its slots wi, wi + wpg, ...
    int it = 0;            // most slots of a warp and group (a multiple of 8)
    int kcap = 0;          // slot rows (128 values) of K a block can keep in shared memory
    int near = 0;          // slot rows of a block's streamed groups that L2 can hold
    size_t smem = 0;       // dynamic shared memory
    std::vector<int> run;  // [nb + 1] first group of each block, in strip order
};

// byte offsets of the dynamic shared memory
struct PsLayout {
    size_t a, b, part, r0, d, so, toff, k;
};
PS_HD PsLayout ps_layout(int es, int nl, int tl, int nchunk, int wpg, int it) {
    PsLayout L;
    size_t o = 0;
    const size_t tile = ((size_t)(nchunk + 1) * tl * es + 15) / 16 * 16;  // one chunk of zeros last
    const size_t rows = (size_t)nl * kPsRows * es;
    L.a = o;
    o += tile;
    L.b = o;
    o += tile;
    L.part = o;  // per warp [4][32], or [8][32] (the FP32-pair residual)
    o += (size_t)kPsW * (es == 4 ? 8 : 4) * 32 * es;
    L.r0 = o;
    o += rows;
    L.d = o;
    o += rows;
    L.so = o;
    o += rows;
    L.toff = o;
    o += (size_t)nl * wpg * it * sizeof(int);
    L.k = o;
    return L;
}

// strip and position of group e in strip order, and its layer (nz: the ground)
PS_HD int ps_strip(const PsGeom &g, int e) { return e / (g.nz + 1); }
PS_HD int ps_zz(const PsGeom &g, int e) { return e % (g.nz + 1); }
PS_HD int ps_layer(const PsGeom &g, int zz) { return zz == 0 ? g.nz : zz - 1; }
PS_HD int ps_y0(const PsGeom &g, int q) { return q * kPsRows / g.nx; }
PS_HD int ps_y1(const PsGeom &g, int q) {
    const int r = q * kPsRows + kPsRows - 1;
    return (r < g.nxy ? r : g.nxy - 1) / g.nx;
}

// The chunks of the groups [e0, e1): strips (q, first chunk, first zz),
// chunks (haloed index of the first element, elements copied) and each
// group's strip.  Returns the number of chunks, or -1 when the block exceeds
// the limits above (the arrays hold that many entries).
PS_HD int ps_walk(const PsGeom &g, int e0, int e1, int *nseg, int *segq, int *segc, int *segz, int *cbase, int *clen,
                  int *gseg) {
    int ns = 0, nc = 0;
    if (e1 - e0 > kPsMaxGroups) return -1;
    for (int e = e0; e < e1; ++e) {
        const int zz = ps_zz(g, e);
        if (e == e0 || zz == 0) {
            if (ns >= kPsMaxSeg) return -1;
            const int q = ps_strip(g, e);
            const int last = zz + (e1 - 1 - e) < g.nz ? zz + (e1 - 1 - e) : g.nz;
            const int za = zz > g.R ? zz - g.R : 0, zb = last + g.R < g.nz ? last + g.R : g.nz;
            segq[ns] = q;
            segc[ns] = nc;
            segz[ns] = za;
            for (int c = za; c <= zb; ++c, ++nc) {
                if (nc >= kPsMaxChunk) return -1;
                cbase[nc] = ps_layer(g, c) * g.lp + ps_y0(g, q) * g.nxp;
                clen[nc] = (ps_y1(g, q) - ps_y0(g, q) + 1 + 2 * g.H) * g.nxp;
            }
            ++ns;
        }
        gseg[e - e0] = ns - 1;
    }
    *nseg = ns;
    return nc;
}

// Row r of strip q: its offset inside a chunk, less the halo (rows past the
// layer's end: 0), and its haloed in-layer position with flags (0: past the
// end); a gathered source of the row sits at ps_off(...) + ps_row_off(...).
constexpr unsigned kPsValid = 1u << 27, kPsXl = 1u << 28, kPsXr = 1u << 29, kPsYl = 1u << 30, kPsYr = 1u << 31;
constexpr unsigned kPsPos = kPsValid - 1;
PS_HD int ps_row_off(const PsGeom &g, int q, int r) {
    const int rr = q * kPsRows + r;
    if (rr >= g.nxy) return 0;
    const int y = rr / g.nx;
    return (y - ps_y0(g, q)) * g.nxp + rr - y * g.nx;
}
PS_HD unsigned ps_row_pos(const PsGeom &g, int q, int r) {
    const int rr = q * kPsRows + r;
    if (rr >= g.nxy) return 0;
    const int y = rr / g.nx, x = rr - y * g.nx;
    unsigned p = (unsigned)((y + g.H) * g.nxp + x + g.H) | kPsValid;
    if (x < g.H) p |= kPsXl;
    else if (x >= g.nx - g.H) p |= kPsXr;
    if (y < g.H) p |= kPsYl;
    else if (y >= g.ny - g.H) p |= kPsYr;
    return p;
}
// tile offset of a source at position zz and in-layer haloed offset off from
// the row, for a strip whose box starts at chunk segc and position segz
PS_HD int ps_off(const PsGeom &g, int tl, int segc, int segz, int zz, int off) {
    return (segc + zz - segz) * tl + off + g.H * g.nxp + g.H;
}

// The warps that share a group walk the same number of slots, in FP32 a
// multiple of 4, so that the loop has no conditions: the slots past the last
// one gather from a chunk of zeros (and, streamed, read the values that
// follow the group's).  In FP64 a slot costs its multiply-adds (2 per clock
// and SM), so it walks no more than it has to.
PS_HD int ps_padded(int nt, int wpg, int es) {
    const int m = wpg * (es == 4 ? 4 : 1);
    return (nt + m - 1) / m * m;
}

// first of the groups [e0, e1) whose values stay in shared memory (whole
// groups, from the last one back, their padding set to zero); nt(e): slots
// of group e
template <class F>
PS_HD int ps_first_resident(int e0, int e1, int kcap, int wpg, int es, F nt) {
    int e = e1;
    while (e > e0 && ps_padded(nt(e - 1), wpg, es) <= kcap) {
        kcap -= ps_padded(nt(e - 1), wpg, es);
        --e;
    }
    return e;
}

// values past a scene's last one that a block may read (finite, and times
// zero): a step of all warps from the last group on
constexpr size_t kPsPad = (size_t)2 * kPsW * 8 * kPsRows;

// Plan for a grid whose layer z (nz: the ground) has nt[z] slots per row;
// es: bytes of the compute type, fixed_smem: the kernel's static shared
// memory.  nb = 0 when the scene does not fit.
PsPlan ps_plan(const PsGeom &g, const std::vector<int> &nt, int es, int nsm, size_t smem_max, size_t fixed_smem);

// ---- Rounds of the streamed passes (k_run in stage.cuh), for scenes the
// persistent solve does not take: a block walks its groups in rounds of at most
// kRunGroups consecutive ones (strip order) whose chunks fit a tile of nc.
constexpr int kRunGroups = 8;     // groups of a round, two warps each
constexpr int kRunMaxChunk = 20;  // chunks of a round's tile
constexpr int kRunMaxRounds = 128, kRunMaxNz = 510;  // tables in shared memory (at most 24 KB)
struct RunPlan {
    int nb = 0;              // blocks (0: the passes run a block per group)
    int tl = 0, nc = 0;      // elements per chunk, chunks per tile
    int near = 0;            // rounds of each block whose values L2 can hold
    int rmax = 0;            // most rounds of a block
    std::vector<int> first;  // [nb + 1] first round of each block
    std::vector<int> round;  // per round: first group, groups, first chunk, chunks
    std::vector<int> chunk;  // per chunk: haloed index of its first element, elements
    std::vector<int> own;    // [rounds][kRunGroups] the chunk of each group's own rows
};
// tile_bytes: shared memory one tile (of one vector) may take
RunPlan run_plan(const PsGeom &g, const std::vector<int> &nt, int nsm, size_t tile_bytes);

}  // namespace tk
