// The persistent solve: BiCGStab (van der Vorst 1992) inside FP64 residual
// refinement, in one cooperative launch.
//
// Why one launch.  With a pass per launch, K comes from HBM and L2 again for
// every product (12.9 us per FP32 pass on the 64 x 64 x 32 plume, 67 MB), and
// the refinements' read-backs and host decisions add about 30 us each: 668 us
// per solve.  Here every block owns the same groups of 128 rows for the whole
// solve.  The values of its last groups stay in shared memory; the others are
// streamed from L2, where they stay because a line is only ever read by one
// SM: measured on GB300, a set read with a fixed mapping of blocks to data
// stays in L2 up to 100 MB (11 to 18 TB/s), and only up to 60 MB when the
// mapping changes from pass to pass (both dies then keep copies).
//
// Why BiCGStab.  It takes two products per step and no spectrum estimate: on
// the plume 32 products in 2 refinements against 38 in 3 (4 sweeps and 30
// Chebyshev steps), on scenes where the interval was missed and GMRES took
// over 50 against 62 with 10 Arnoldi steps' host round trips.  Each block
// keeps r and p on its rows and on every node its rows gather from (its tile,
// updated redundantly), so a product needs one exchange: the block publishes
// its part of A p (or A s) and its shares of the dot products, meets the grid
// barrier (1.3 us over 152 blocks), and reads the others' parts.
//
// What bounds a product: its shared-memory wavefronts, 8 per slot of 128 rows
// (4 for the values, 4 for the gathers; 3.6 us for 7 groups), then the
// exchange.  Measured on the plume, per step of two products: 6.4 and 6.6 us
// of products, 1.5 and 2.0 us of barriers, 1.5 and 2.7 us of vector updates.
// Whole solve 373 us (plume), 395 us (random 45 x 37 x 29: 1160 us with passes
// and GMRES), 120 us (plume 16^3), 1.2 ms (96 x 96 x 32, 150 MB of values
// of which L2 keeps 80).  FP64 is kept off the common path of FP32
// scenes (an FP64 warp operation takes 16 issue slots of the SM): dot products
// are FP32 pairs, 48 bits, and the outer loop's scalars are one thread's.
//
// Sums run in a fixed order that depends on the plan only, so a solve's bits
// do not depend on what else is in the launch.
#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

#include "dots.cuh"
#include "kern.h"
#include "persist.h"

namespace tk {

constexpr int kPsThreads = 32 * kPsW;
static_assert(kPsRows == kGroup, "groups");
constexpr long long kPsPolls = 1ll << 21;  // polls of one barrier: about 1.5 s

// ---- grid barrier over the job's blocks: one release-add and an acquire
// poll; false once a wait has run out (the block then leaves the kernel)
__device__ __forceinline__ bool ps_barrier(unsigned *bar, unsigned target, int *status, int *ok_sh) {
    __syncthreads();
    if (threadIdx.x == 0) {
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
        int ok = 0;
        for (long long i = 0; i < kPsPolls; ++i) {
            unsigned v;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
            if ((int)(v - target) >= 0) {
                ok = 1;
                break;
            }
        }
        if (!ok) atomicOr(status, STATUS_TIMEOUT);
        *ok_sh = ok;
    }
    __syncthreads();
    return *ok_sh != 0;
}

// the FP32-pair accumulation of the refinement residual (see OpResidDS)
__device__ __forceinline__ void ps_ds(float &hi, float &lo, float v, float xh, float xl) {
    const float p = __fmul_rn(v, xh);
    const float e = fmaf(v, xh, -p);
    const float s = __fadd_rn(hi, p);
    const float bb = __fsub_rn(s, hi);
    const float err = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(p, bb));
    hi = s;
    lo = __fadd_rn(lo, __fadd_rn(__fadd_rn(err, e), __fmul_rn(v, xl)));
}

__device__ __forceinline__ void ps_quad(const float *p, float (&v)[4]) {
    const float4 q = *reinterpret_cast<const float4 *>(p);
    v[0] = q.x;
    v[1] = q.y;
    v[2] = q.z;
    v[3] = q.w;
}
__device__ __forceinline__ void ps_quad(const double *p, double (&v)[4]) {
    const double2 a = reinterpret_cast<const double2 *>(p)[0], b = reinterpret_cast<const double2 *>(p)[1];
    v[0] = a.x;
    v[1] = a.y;
    v[2] = b.x;
    v[3] = b.y;
}
// the same from global memory, with an L2 policy, past L1 (what the tiles leave
// of it would only be turned over: 16 mixed requests 15.6 -> 15.25 ms)
__device__ __forceinline__ void ps_quad_g(const float *p, unsigned long long pol, float (&v)[4]) {
    asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.v4.f32 {%0, %1, %2, %3}, [%4], %5;"
        : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3])
        : "l"(p), "l"(pol));
}
__device__ __forceinline__ void ps_quad_g(const double *p, unsigned long long pol, double (&v)[4]) {
    asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.v2.f64 {%0, %1}, [%2], %3;" : "=d"(v[0]), "=d"(v[1]) : "l"(p), "l"(pol));
    asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.v2.f64 {%0, %1}, [%2], %3;" : "=d"(v[2]), "=d"(v[3]) : "l"(p + 2), "l"(pol));
}

// what a block knows of one of its groups
struct PsGroup {
    long long vb;   // first value
    int nt, zz, z;  // slots, position, layer
    int seg;        // strip
    int own;        // tile offset of the group's own rows (added to rlt)
    int ks;         // its values in shared memory (slot rows), -1: streamed from L2, -2: from HBM
};

struct PsShared {
    PsGroup grp[kPsMaxGroups];
    int cbase[kPsMaxChunk], clen[kPsMaxChunk];
    uint16_t rlt[kPsMaxSeg][kGroup];   // a row's offset inside one chunk (ps_row_off)
    unsigned hp[kPsMaxSeg][kGroup];    // its haloed in-layer position and flags (ps_row_pos)
    int segq[kPsMaxSeg], segc[kPsMaxSeg], segz[kPsMaxSeg], segk[kPsMaxSeg];  // strip, first chunk, first zz, row blocks
    double red[kPsW][kPsDots];
    double sc[kPsDots];
    int gseg[kPsMaxGroups];
    int nseg, nchunk, ok;
    // the outer loop's scalars (thread 0) and one step's (FP64 scenes)
    double sn, rel, bb, stop2;
    int ex, state, stalls;
    double sc_out[4];
};

struct PsBatch {
    int njobs, pad[3];
    PsJob job[kPsMaxJobs];
};

enum { PS_V = 0, PS_T = 1, PS_RES = 2 };

template <typename T, int wpg>
__global__ void __launch_bounds__(kPsThreads, 1) k_persist(const __grid_constant__ PsBatch B) {
    constexpr int PF = sizeof(T) == 4 ? 8 : 4;  // slots of a warp in flight
    extern __shared__ __align__(16) unsigned char ps_dyn[];
    __shared__ PsShared S;
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    int jb = 0;
    while (jb + 1 < B.njobs && (int)blockIdx.x >= B.job[jb + 1].block0) ++jb;
    const PsJob &J = B.job[jb];
    const int blk = blockIdx.x - J.block0, nb = J.nb;
    const int nx = J.g.nx, ny = J.g.ny, nz = J.g.nz, nxy = J.g.nxy, H = J.g.H, nxp = J.g.nxp, lp = J.g.lp;
    const int tl = J.tl, it = J.it;
    constexpr int nsets = kPsW / wpg;
    constexpr int step = wpg * kGroup;  // values between a warp's slots
    const int set = w / wpg, wi = w - set * wpg;  // set >= nsets: no groups
    const PsLayout L = ps_layout(sizeof(T), J.nl, tl, J.nchunk, wpg, it);
    T *tA = (T *)(ps_dyn + L.a), *tB = (T *)(ps_dyn + L.b);
    T *sR0 = (T *)(ps_dyn + L.r0), *sD = (T *)(ps_dyn + L.d), *sS = (T *)(ps_dyn + L.so);
    T *sPart = (T *)(ps_dyn + L.part);
    int *toff = (int *)(ps_dyn + L.toff);
    T *sm = (T *)ps_dyn;
    T *sK = (T *)(ps_dyn + L.k);
    const T *val = (const T *)J.val;
    const T *src_s = (const T *)J.s;
    const int e0 = __ldg(J.run + blk), e1 = __ldg(J.run + blk + 1), nl = e1 - e0;

    const PsGeom geo{nx, ny, nz, nxy, J.g.gpl, H, nxp, lp, J.g.R};

    // ---- the block's groups, strips and tile chunks
    if (tid == 0) {
        S.stalls = 0;
        S.rel = 1.0;
        S.nchunk = ps_walk(geo, e0, e1, &S.nseg, S.segq, S.segc, S.segz, S.cbase, S.clen, S.gseg);
        for (int l = 0; l < nl; ++l) {
            PsGroup G;
            G.zz = ps_zz(geo, e0 + l);
            G.z = ps_layer(geo, G.zz);
            G.seg = S.gseg[l];
            G.nt = __ldg(J.tstart + G.z + 1) - __ldg(J.tstart + G.z);
            G.vb = __ldg(J.voff + G.z) + (long long)S.segq[G.seg] * G.nt * kGroup;
            G.own = ps_off(geo, tl, S.segc[G.seg], S.segz[G.seg], G.zz, 0);
            G.ks = -1;
            S.grp[l] = G;
        }
        for (int i = 0; i < S.nseg; ++i) S.segk[i] = min(4, (nxy - S.segq[i] * kGroup + 31) / 32);
        const int er = ps_first_resident(0, nl, J.kcap, wpg, (int)sizeof(T), [&](int l) { return S.grp[l].nt; });
        // streamed groups beyond what L2 holds for all blocks come from HBM
        // every time, marked to leave L2 first, so that they do not push the
        // others out
        int near = J.near;
        for (int l = er - 1; l >= 0; --l) {
            near -= S.grp[l].nt;
            if (near < 0) S.grp[l].ks = -2;
        }
        int ks = 0;
        for (int l = er; l < nl; ++l) {
            S.grp[l].ks = ks;
            ks += ps_padded(S.grp[l].nt, wpg, (int)sizeof(T));
        }
    }
    __syncthreads();
    const int nseg = S.nseg, ntile = S.nchunk * tl;
    for (int i = tid; i < nseg * kGroup; i += kPsThreads) {
        const int sg = i / kGroup, r = i - sg * kGroup;
        S.rlt[sg][r] = (uint16_t)ps_row_off(geo, S.segq[sg], r);
        S.hp[sg][r] = ps_row_pos(geo, S.segq[sg], r);
    }
    // a slot's tile offset from its row's rlt: [group][warp][step], slot = wi + wpg * i
    for (int i = tid; i < nl * wpg * it; i += kPsThreads) {
        const int l = i / (wpg * it), rem = i - l * wpg * it, ww = rem / it, k = rem - ww * it, t = ww + wpg * k;
        const PsGroup &G = S.grp[l];
        int o = ps_off(geo, tl, J.nchunk, 0, 0, 0);  // past the last slot: the zeros
        if (t < G.nt) {
            const int2 p = __ldg(J.tpos + __ldg(J.tstart + G.z) + t);
            o = ps_off(geo, tl, S.segc[G.seg], S.segz[G.seg], p.x, p.y);
        }
        toff[i] = o;
    }
    // ---- the resident values
    for (int l = 0; l < nl; ++l) {
        const PsGroup &G = S.grp[l];
        if (G.ks < 0) continue;
        constexpr int per = 16 / sizeof(T);
        const int n = G.nt * kGroup / per;
        const uint4 *src = reinterpret_cast<const uint4 *>(val + G.vb);
        uint4 *dst = reinterpret_cast<uint4 *>(sK + (size_t)G.ks * kGroup);
#pragma unroll 8
        for (int i = tid; i < n; i += kPsThreads) dst[i] = __ldg(src + i);
        for (int i = n + tid; i < ps_padded(G.nt, wpg, (int)sizeof(T)) * kGroup / per; i += kPsThreads) dst[i] = make_uint4(0, 0, 0, 0);
    }
    for (int i = tid; i < tl; i += kPsThreads) tA[J.nchunk * tl + i] = tB[J.nchunk * tl + i] = T(0);
    // The next PF slots of this warp, loaded ahead of their use: pf holds the
    // first slots of a streamed group by the time the group's turn comes,
    // across groups and across the barrier into the next product.
    T pf[PF][4];
    auto stream = [&](int l) -> const T * {  // the warp's first value of group l, null: not streamed
        return l < nl && S.grp[l].ks < 0 ? val + S.grp[l].vb + wi * kGroup + 4 * lane : nullptr;
    };
    unsigned long long keep, pass_by;
    asm("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(keep));
    asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pass_by));
    auto policy = [&](int l) { return l < nl && S.grp[l].ks == -2 ? pass_by : keep; };
    {
        const int l = set < nsets ? set : nl;
        const T *p = stream(l);
        if (p) {
            const unsigned long long pol = policy(l);
#pragma unroll
            for (int i = 0; i < PF; ++i) ps_quad_g(p + i * step, pol, pf[i]);
        }
    }
    // the first EB tile elements of this thread: where they come from
    constexpr int EB = sizeof(T) == 4 ? 10 : 6;
    // own rows: initial right-hand side b = s, published
    unsigned gen = 0;  // publications (and barriers) so far
    // a row's value at its haloed position and at its halo copies
    auto publish = [&](auto *v, int z, unsigned hp, auto a) {
        auto *p = v + (size_t)z * lp + (hp & kPsPos);
        *p = a;
        const int ax = (hp & kPsXl) ? nx : (hp & kPsXr) ? -nx : 0;
        const int ay = (hp & kPsYl) ? ny * nxp : (hp & kPsYr) ? -ny * nxp : 0;
        if (ax) p[ax] = a;
        if (ay) {
            p[ay] = a;
            if (ax) p[ax + ay] = a;
        }
    };
    // node number (natural order) of row r of group G
    auto node = [&](const PsGroup &G, int r) { return G.z * nxy + S.segq[G.seg] * kGroup + r; };
    // The block's sums of nd values already summed per warp (S.red, as Dot
    // bits) go to the job's partials of the current publication; sums_of reads
    // the job's sums of the last one into S.sc.  FP32 scenes stay in FP32
    // pairs: an FP64 operation costs a warp 16 issue slots on this GPU, and
    // FP64 scalars in every thread took 7 us per step here.
    auto put_sums = [&](int nd) {
        __syncthreads();
        if (w < nd) {
            Dot<T> v;
            if (lane < kPsW) v = Dot<T>::from(S.red[lane][w]);
#pragma unroll
            for (int o = kPsW / 2; o >= 1; o >>= 1) v.join(v.xch(o));
            if (lane == 0) J.part[((size_t)(gen % 3) * kPsDots + w) * nb + blk] = v.bits();
        }
    };
    auto sums_of = [&](int nd) {
        if (w < nd) {
            const double *p = J.part + ((size_t)((gen - 1) % 3) * kPsDots + w) * nb;
            Dot<T> v;
            for (int i = lane; i < nb; i += 32) v.join(Dot<T>::from(__ldcg(p + i)));
#pragma unroll
            for (int o = 16; o >= 1; o >>= 1) v.join(v.xch(o));
            if (lane == 0) S.sc[w] = v.bits();
        }
        __syncthreads();
    };
    // the same for one FP64 value per thread (the refinement's ||r||^2)
    auto put_norm = [&](double v) {
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) S.red[w][0] = v;
        __syncthreads();
        if (tid == 0) {
            double t = 0.0;
            for (int q = 0; q < kPsW; ++q) t += S.red[q][0];
            J.part[(size_t)(gen % 3) * kPsDots * nb + blk] = t;
        }
    };
    auto norm_of = [&]() {  // in thread 0's S.sc[0]
        if (w == 0) {
            const double *p = J.part + (size_t)((gen - 1) % 3) * kPsDots * nb;
            double t = 0.0;
            for (int i = lane; i < nb; i += 32) t += __ldcg(p + i);
            for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
            if (lane == 0) S.sc[0] = t;
        }
    };
    const unsigned tl_magic = (unsigned)((0x100000000ull + tl - 1) / tl);
    auto tile_src = [&](int j) -> int {  // haloed index of tile element j, -1: none
        const int c = (int)__umulhi((unsigned)j, tl_magic);
        const int o = j - c * tl;
        return o < S.clen[c] ? S.cbase[c] + o : -1;
    };
    int tsrc[EB];
#pragma unroll
    for (int e = 0; e < EB; ++e) {
        const int j = tid + e * kPsThreads;
        tsrc[e] = j < ntile ? tile_src(j) : -1;
    }

    // One product over the block's rows from the tile (PS_V: v = A p from tB,
    // PS_T: t = A s from tA, PS_RES: r = s - x + K x from tA (and tB)),
    // published with its dot products.
    auto set_sync = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(1 + set), "r"(32 * wpg) : "memory"); };
    auto pass = [&](auto mode_c) {
        constexpr int MODE = decltype(mode_c)::value;
        constexpr bool DS = MODE == PS_RES && sizeof(T) == 4;
        constexpr int NA = DS ? 8 : 4;
        const T *tile = MODE == PS_V ? tB : tA;
        Dot<T> dot[8];
        double rr = 0.0;
        T *pub = (T *)J.pub[gen % 3];
        T *pw = sPart + (size_t)(set < nsets ? set : 0) * wpg * NA * 32;  // the set's partial sums [wpg][NA][32]
        // row 32 k + lane of group l from the set's partial sums
        auto finish = [&](int l, int k) {
            const PsGroup &G = S.grp[l];
            const int r = 32 * k + lane;
            const unsigned hp = S.hp[G.seg][r];
            if (!(hp & kPsValid)) return;
            if constexpr (MODE == PS_RES) {
                double kx;
                if constexpr (DS) {
                    float h = 0.f, lo = 0.f;
#pragma unroll
                    for (int q = 0; q < wpg; ++q) {
                        const float pp = pw[(q * NA + k) * 32 + lane];
                        const float ss = __fadd_rn(h, pp);
                        const float bb = __fsub_rn(ss, h);
                        lo = __fadd_rn(lo, __fadd_rn(__fadd_rn(__fsub_rn(h, __fsub_rn(ss, bb)), __fsub_rn(pp, bb)),
                                                     pw[(q * NA + k + 4) * 32 + lane]));
                        h = ss;
                    }
                    kx = (double)h + (double)lo;
                } else {
                    kx = 0.0;
#pragma unroll
                    for (int q = 0; q < wpg; ++q) kx += pw[(q * NA + k) * 32 + lane];
                }
                const double r64 = (double)src_s[node(G, r)] - J.x[(size_t)G.z * lp + (hp & kPsPos)] + kx;
                publish(pub, G.z, hp, (T)r64);
                rr = fma(r64, r64, rr);
            } else {
                T a = T(0);
#pragma unroll
                for (int q = 0; q < wpg; ++q) a += pw[(q * NA + k) * 32 + lane];
                const T o = tile[G.own + S.rlt[G.seg][r]];
                const T y = o - a;
                publish(pub, G.z, hp, y);
                const T q0 = sR0[l * kGroup + r];
                if constexpr (MODE == PS_V) {
                    dot[0].add(q0, y);
                } else {
                    sS[l * kGroup + r] = o;
                    dot[0].add(y, o);   // t.s
                    dot[1].add(y, y);   // t.t
                    dot[2].add(q0, o);  // r0.s
                    dot[3].add(q0, y);  // r0.t
                    dot[4].add(o, o);   // s.s
                }
            }
        };
        int seg = -1;
        int ia[4] = {0, 0, 0, 0}, ib[4] = {0, 0, 0, 0};  // the lane's rows in the tile (and in tB for DS)
        for (int l = set < nsets ? set : nl; l < nl; l += nsets) {
            const PsGroup &G = S.grp[l];
            if (G.seg != seg) {
                seg = G.seg;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int o = S.rlt[seg][lane + 32 * k];
                    ia[k] = (int)(tile - sm) + o;
                    if (DS) ib[k] = (int)(tB - sm) + o;
                }
            }
            T acc[NA];
#pragma unroll
            for (int m = 0; m < NA; ++m) acc[m] = T(0);
            const int kb = sizeof(T) == 8 ? S.segk[G.seg] : 4;  // row blocks with rows
            auto add = [&](const T (&v)[4], int off) {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    if constexpr (DS)
                        ps_ds(acc[k], acc[4 + k], v[k], sm[off + ia[k]], sm[off + ib[k]]);
                    else if (sizeof(T) == 4 || k < kb)
                        acc[k] += v[k] * sm[off + ia[k]];
                }
            };
            const int *to = toff + (l * wpg + wi) * it;
            const int n = ps_padded(G.nt, wpg, (int)sizeof(T)) / wpg;  // the warp's slots
            const T *nx_ = stream(l + nsets < nl ? l + nsets : set);
            const unsigned long long pol = policy(l), poln = policy(l + nsets < nl ? l + nsets : set);
            if (G.ks >= 0) {  // in shared memory
                const T *ksm = sK + (size_t)G.ks * kGroup + wi * kGroup + 4 * lane;
                auto round = [&](auto cnt_c, int i0) {
                    constexpr int N = decltype(cnt_c)::value;
                    T q[N][4];
                    int off[N];
#pragma unroll
                    for (int i = 0; i < N; i += 4) {
                        const int4 t = *reinterpret_cast<const int4 *>(to + i0 + i);
                        off[i] = t.x;
                        off[i + 1] = t.y;
                        off[i + 2] = t.z;
                        off[i + 3] = t.w;
                    }
#pragma unroll
                    for (int i = 0; i < N; ++i) ps_quad(ksm + (i0 + i) * step, q[i]);
#pragma unroll
                    for (int i = 0; i < N; ++i) add(q[i], off[i]);
                };
                int i0 = 0;
                if constexpr (sizeof(T) == 4 && !DS) {
                    for (; i0 + 8 <= n; i0 += 8) round(std::integral_constant<int, 8>(), i0);
                }
                for (; i0 + 4 <= n; i0 += 4) round(std::integral_constant<int, 4>(), i0);
                for (; sizeof(T) == 8 && i0 < n; ++i0) {
                    T q[4];
                    ps_quad(ksm + i0 * step, q);
                    add(q, to[i0]);
                }
                if (nx_) {
#pragma unroll
                    for (int i = 0; i < PF; ++i) ps_quad_g(nx_ + i * step, poln, pf[i]);
                }
            } else {  // streamed from L2: PF slots are there; each one's successor is requested as it is used
                const T *kg = val + G.vb + wi * kGroup + 4 * lane;
                for (int i0 = 0; i0 < n; i0 += PF) {
                    const T *p = i0 + PF < n ? kg + (i0 + PF) * step : nx_ ? nx_ : kg;
                    const unsigned long long pp = i0 + PF < n || !nx_ ? pol : poln;
                    int off[PF];
#pragma unroll
                    for (int i = 0; i < PF; i += 4) {
                        const int4 t = *reinterpret_cast<const int4 *>(to + i0 + i);
                        off[i] = t.x;
                        off[i + 1] = t.y;
                        off[i + 2] = t.z;
                        off[i + 3] = t.w;
                    }
#pragma unroll
                    for (int i = 0; i < PF; ++i) {
                        if (sizeof(T) == 4 || i0 + i < n) add(pf[i], off[i]);
                        ps_quad_g(p + i * step, pp, pf[i]);
                    }
                }
            }
#pragma unroll
            for (int m = 0; m < NA; ++m) pw[(wi * NA + m) * 32 + lane] = acc[m];
            set_sync();
            for (int k = wi; k < 4; k += wpg) finish(l, k);
            if (l + nsets < nl) set_sync();
        }
        const bool any = set < nsets && set < nl && wi < 4;  // the warp has finished rows
        if constexpr (MODE == PS_T) {
            if (any) {
                const Dot<T> v = warp_dots8<T>(dot);
                if ((lane & 3) == 0 && (lane >> 2) < 5) S.red[w][lane >> 2] = v.bits();
            } else if (lane < 5) {
                S.red[w][lane] = 0.0;
            }
            put_sums(5);
        } else if constexpr (MODE == PS_V) {
            if (any) {
                const Dot<T> v = warp_dot1<T>(dot[0]);
                if (lane == 0) S.red[w][0] = v.bits();
            } else if (lane == 0) {
                S.red[w][0] = 0.0;
            }
            put_sums(1);
        } else {
            put_norm(rr);
        }
    };
    auto barrier = [&]() -> bool {
        ++gen;
        return ps_barrier(J.bar, gen * (unsigned)nb, J.status, &S.ok);
    };

    // ---- r = s (x = 0)
    {
        double rr = 0.0;
        T *pub = (T *)J.pub[gen % 3];
        for (int i = tid; i < nl * kGroup; i += kPsThreads) {
            const PsGroup &G = S.grp[i / kGroup];
            const unsigned hp = S.hp[G.seg][i % kGroup];
            if (!(hp & kPsValid)) continue;
            const T b = src_s[node(G, i % kGroup)];
            publish(pub, G.z, hp, b);
            rr = fma((double)b, (double)b, rr);
        }
        put_norm(rr);
    }
    int iters = 0, refinements = 0, state = PS_RUNNING;  // iters: steps and residuals
    for (;;) {
        // ---- the residual r of the current x is published: its norm, and the tile
        if (!barrier()) return;
        norm_of();
        if (tid == 0) {  // FP64 in one thread (every thread's would cost 10 us here)
            const double rr = S.sc[0], prev = S.rel;
            if (refinements == 0) {
                S.sn = sqrt(rr);
                S.rel = S.sn == 0.0 ? 0.0 : 1.0;
            } else {
                S.rel = sqrt(rr) / S.sn;
            }
            int st = PS_RUNNING;
            if (S.rel <= J.rtol)
                st = PS_CONVERGED;
            else if (!(S.rel <= 1e30))
                st = PS_GAVE_UP;
            else if (iters >= J.max_iter)
                st = PS_MAX_ITER;
            else if (refinements > 0 && !(S.rel <= 0.5 * prev) && ++S.stalls > 1)
                st = PS_GAVE_UP;
            S.state = st;
            // the correction is solved for at unit scale (a power of two), so that
            // FP32 squares neither overflow nor underflow
            S.ex = st == PS_RUNNING ? min(120, max(-120, ilogb(sqrt(rr)))) : 0;
            const double tol = fmax(0.3 * J.rtol / S.rel, sizeof(T) == 8 ? 1e-15 : 2e-6);
            S.bb = ldexp(rr, -2 * S.ex);
            S.stop2 = tol * tol * S.bb;
        }
        __syncthreads();
        state = S.state;
        if (state != PS_RUNNING) break;
        const int ex = S.ex;
        const T down = sizeof(T) == 4 ? (T)ldexpf(1.f, -ex) : (T)ldexp(1.0, -ex);
        const T bb = (T)S.bb, stop2 = (T)S.stop2;
        {
            const T *pb = (const T *)J.pub[(gen - 1) % 3];
            for (int j = tid; j < ntile; j += kPsThreads) {
                const int a = tile_src(j);
                const T v = a >= 0 ? down * __ldcg(pb + a) : T(0);
                tA[j] = v;
                tB[j] = v;
            }
        }
        __syncthreads();
        for (int i = tid; i < nl * kGroup; i += kPsThreads) {
            const PsGroup &G = S.grp[i / kGroup];
            sR0[i] = tA[G.own + S.rlt[G.seg][i % kGroup]];
            sD[i] = T(0);
        }
        __syncthreads();
        // ---- BiCGStab on (I - K) d = b
        T rho = bb, best = bb;
        int since = 0;
        for (;;) {
            pass(std::integral_constant<int, PS_V>());
            if (!barrier()) return;
            T alpha;
            {
                const T *pv = (const T *)J.pub[(gen - 1) % 3];
                T buf[EB];
#pragma unroll
                for (int e = 0; e < EB; ++e) {
                    buf[e] = tsrc[e] >= 0 ? __ldcg(pv + tsrc[e]) : T(0);
                }
                sums_of(1);
                auto scalars = [&](T *o) {
                    const T r0v = Dot<T>::from(S.sc[0]).value();
                    o[0] = r0v != T(0) ? rho / r0v : T(0);
                };
                T sv[1];
                if constexpr (sizeof(T) == 4) {
                    scalars(sv);
                } else {
                    if (tid == 0) scalars(S.sc_out);
                    __syncthreads();
                    sv[0] = S.sc_out[0];
                }
                alpha = sv[0];
                for (int i = tid; i < nl * kGroup; i += kPsThreads) {
                    const PsGroup &G = S.grp[i / kGroup];
                    sD[i] += alpha * tB[G.own + S.rlt[G.seg][i % kGroup]];
                }
#pragma unroll
                for (int e = 0; e < EB; ++e) {
                    if (tsrc[e] >= 0) tA[tid + e * kPsThreads] -= alpha * buf[e];
                }
#pragma unroll 4
                for (int j = tid + EB * kPsThreads; j < ntile; j += kPsThreads) {
                    const int a = tile_src(j);
                    if (a >= 0) tA[j] -= alpha * __ldcg(pv + a);
                }
            }
            __syncthreads();
            pass(std::integral_constant<int, PS_T>());
            if (!barrier()) return;
            ++iters;
            bool stop;
            {
                const T *pv = (const T *)J.pub[(gen - 2) % 3], *pt = (const T *)J.pub[(gen - 1) % 3];
                T bv[EB], bt[EB];
#pragma unroll
                for (int e = 0; e < EB; ++e) {
                    bv[e] = tsrc[e] >= 0 ? __ldcg(pv + tsrc[e]) : T(0);
                    bt[e] = tsrc[e] >= 0 ? __ldcg(pt + tsrc[e]) : T(0);
                }
                sums_of(5);
                auto scalars = [&](T *o) {  // omega, beta, the new rho, ||r||^2
                    const Dot<T> ts = Dot<T>::from(S.sc[0]), tt = Dot<T>::from(S.sc[1]), r0t = Dot<T>::from(S.sc[3]);
                    Dot<T> r0r = Dot<T>::from(S.sc[2]), rn = Dot<T>::from(S.sc[4]);
                    const T om = tt.value() > T(0) ? ts.value() / tt.value() : T(0);
                    r0t.add_to(r0r, -om);          // r0.r = r0.s - omega r0.t
                    ts.add_to(rn, T(-2) * om);     // r.r = s.s - 2 omega t.s + omega^2 t.t
                    Dot<T> ott;
                    tt.add_to(ott, om);
                    ott.add_to(rn, om);
                    o[0] = om;
                    o[2] = r0r.value();
                    o[3] = rn.value();
                    o[1] = (rho != T(0) && om != T(0)) ? (o[2] / rho) * (alpha / om) : T(0);
                };
                T sv[4];
                if constexpr (sizeof(T) == 4) {
                    scalars(sv);
                } else {
                    if (tid == 0) scalars(S.sc_out);
                    __syncthreads();
#pragma unroll
                    for (int k = 0; k < 4; ++k) sv[k] = S.sc_out[k];
                }
                const T omega = sv[0], beta = sv[1], rnv = sv[3];
                const T rho1 = sv[2];
                rho = rho1;
                // (as they are: FP64 conversions here cost FP32 scenes 0.7 % of a solve)
                if (iters <= kPsRec && tid == 0 && blk == 0) {
                    J.info->coef<T>()[iters - 1] = alpha;
                    J.info->coef<T>()[kPsRec + iters - 1] = beta;
                }
                if (rnv < best) {
                    best = rnv;
                    since = 0;
                } else {
                    ++since;
                }
                stop = !(rnv > stop2) || omega == T(0) || !(fabs(beta) > T(0)) || since > 40 ||
                       iters + 1 >= J.max_iter;
                for (int i = tid; i < nl * kGroup; i += kPsThreads) sD[i] += omega * sS[i];
                if (!stop) {
                    auto upd = [&](int j, T v, T t) {
                        const T r = tA[j] - omega * t;
                        tB[j] = r + beta * (tB[j] - omega * v);
                        tA[j] = r;
                    };
#pragma unroll
                    for (int e = 0; e < EB; ++e) {
                        if (tsrc[e] >= 0) upd(tid + e * kPsThreads, bv[e], bt[e]);
                    }
#pragma unroll 4
                    for (int j = tid + EB * kPsThreads; j < ntile; j += kPsThreads) {
                        const int a = tile_src(j);
                        if (a >= 0) upd(j, __ldcg(pv + a), __ldcg(pt + a));
                    }
                }
            }
            __syncthreads();
            if (stop) break;
        }
        // ---- x += d (own rows; the FP32 pair of x, or x itself, is published)
        const T up = sizeof(T) == 4 ? (T)ldexpf(1.f, ex) : (T)ldexp(1.0, ex);
        for (int i = tid; i < nl * kGroup; i += kPsThreads) {
            const PsGroup &G = S.grp[i / kGroup];
            const unsigned hp = S.hp[G.seg][i % kGroup];
            if (!(hp & kPsValid)) continue;
            double v = (double)(up * sD[i]);
            if (refinements > 0) v += J.x[(size_t)G.z * lp + (hp & kPsPos)];
            publish(J.x, G.z, hp, v);
            if (sizeof(T) == 4) {
                const float h = (float)v;
                publish(J.xh, G.z, hp, h);
                publish(J.xl, G.z, hp, (float)(v - (double)h));
            }
        }
        if (!barrier()) return;
#pragma unroll 4
        for (int j = tid; j < ntile; j += kPsThreads) {
            const int a = tile_src(j);
            if constexpr (sizeof(T) == 4) {
                tA[j] = a >= 0 ? __ldcg(J.xh + a) : 0.f;
                tB[j] = a >= 0 ? __ldcg(J.xl + a) : 0.f;
            } else {
                tA[j] = a >= 0 ? __ldcg(J.x + a) : 0.0;
            }
        }
        __syncthreads();
        pass(std::integral_constant<int, PS_RES>());
        ++iters;
        ++refinements;
    }
    if (state == PS_CONVERGED && refinements == 0) {  // s = 0 (or rtol >= 1): x = 0
        for (int i = tid; i < nl * kGroup; i += kPsThreads) {
            const PsGroup &G = S.grp[i / kGroup];
            const unsigned hp = S.hp[G.seg][i % kGroup];
            if (!(hp & kPsValid)) continue;
            publish(J.x, G.z, hp, 0.0);
            if (sizeof(T) == 4) {
                publish(J.xh, G.z, hp, 0.f);
                publish(J.xl, G.z, hp, 0.f);
            }
        }
    }
    if (blk == 0 && tid == 0) {
        J.info->iters = iters;
        J.info->refinements = refinements;
        J.info->state = state;
        J.info->rel = S.rel;
        J.info->sn = S.sn;
    }
}

// ---------------------------------------------------------------------------

PsGeom ps_geom(const GridC &g) { return PsGeom{g.nx, g.ny, g.nz, g.nxy, g.gpl, g.H, g.nxp, g.lp, g.R}; }
size_t ps_fixed_smem() { return sizeof(PsShared) + 2048; }

cudaError_t launch_persist(cudaStream_t st, const PsJob *jobs, int njobs, int blocks, size_t smem, bool fp64) {
    if (njobs < 1 || njobs > kPsMaxJobs) return cudaErrorInvalidValue;
    PsBatch B;
    B.njobs = njobs;
    B.pad[0] = B.pad[1] = B.pad[2] = 0;
    for (int i = 0; i < njobs; ++i) B.job[i] = jobs[i];
    auto kernel = [&](auto t) -> const void * {
        using T = decltype(t);
        switch (jobs[0].wpg) {
            case 2: return (const void *)k_persist<T, 2>;
            case 3: return (const void *)k_persist<T, 3>;
            case 4: return (const void *)k_persist<T, 4>;
            case 5: return (const void *)k_persist<T, 5>;
            case 8: return (const void *)k_persist<T, 8>;
            case 16: return (const void *)k_persist<T, 16>;
        }
        return nullptr;
    };
    const void *k = fp64 ? kernel(0.0) : kernel(0.f);
    if (!k) return cudaErrorInvalidValue;
    for (int i = 1; i < njobs; ++i)
        if (jobs[i].wpg != jobs[0].wpg) return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    void *args[] = {(void *)&B};
    return cudaLaunchCooperativeKernel(k, dim3(blocks), dim3(kPsThreads), args, smem, st);
}

// the self-test: every block meets one barrier that expects `expect` arrivals
__global__ void k_barrier_test(unsigned *bar, unsigned expect) {
    __shared__ int ok;
    ps_barrier(bar, expect, (int *)(bar + 1), &ok);
}

int barrier_selftest(cudaStream_t st, int blocks, int arrive) {
    unsigned *bar = nullptr;
    if (cudaMalloc((void **)&bar, 2 * sizeof(unsigned)) != cudaSuccess) return -1;
    int result = -1;
    unsigned h[2] = {0, 0};
    if (cudaMemsetAsync(bar, 0, sizeof(h), st) == cudaSuccess) {
        unsigned expect = (unsigned)blocks + (arrive ? 0u : 1u);
        void *args[] = {(void *)&bar, (void *)&expect};
        if (cudaLaunchCooperativeKernel((const void *)k_barrier_test, dim3(blocks), dim3(32), args, 0, st) ==
                cudaSuccess &&
            cudaMemcpyAsync(h, bar, sizeof(h), cudaMemcpyDeviceToHost, st) == cudaSuccess &&
            cudaStreamSynchronize(st) == cudaSuccess)
            result = (int)h[1] & STATUS_TIMEOUT;
    }
    cudaFree(bar);
    return result;
}

}  // namespace tk
