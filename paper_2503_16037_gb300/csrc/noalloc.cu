// Allocation-free variant of the refined solve of (I - K) x = s.
//
// Some callers cannot allocate device memory at the moment they need a solve:
// a host program whose device memory is owned by its own pool allocator and
// sized at start-up, or a latency-critical loop in which cudaMalloc / cudaFree
// (which may synchronise the whole device) are not allowed.  This entry point
// serves them: it takes the matrix, the source and the output from the
// caller and keeps its work vectors in a fixed, file-scope device array that
// is part of the library image, so the call itself allocates nothing.
#include <cuda_runtime.h>

#include <cstdint>
#include <cstring>
#include <type_traits>

#include "tursca.h"

namespace {

// Largest system the scratch array can hold, and its layout.
constexpr int kMaxNodes = 1 << 20;                 // 1,048,576 nodes
constexpr int kPartBlocks = 1024;                  // residual partial sums
constexpr size_t kOffB = 0;                        // float  [kMaxNodes] right-hand side of the sweeps
constexpr size_t kOffD0 = kOffB + 4ull * kMaxNodes;  // float  [kMaxNodes] sweep buffer
constexpr size_t kOffD1 = kOffD0 + 4ull * kMaxNodes; // float  [kMaxNodes] sweep buffer
constexpr size_t kOffPart = kOffD1 + 4ull * kMaxNodes; // double [kPartBlocks]
constexpr size_t kOffBar = kOffPart + 8ull * kPartBlocks;  // barrier word of the one-launch form
constexpr size_t kScratchBytes = kOffBar + 256;            // about 12 MiB

// Shared by every call on a device; holds the previous call's contents.
static __device__ __align__(256) unsigned char g_solve_scratch[kScratchBytes];

// Most kernel launches one call may issue (sweeps and residual passes).
constexpr long long kMaxLaunches = 1000000;

// Device address of the scratch array in the current device's context,
// looked up on every call: the lookup is cheap once the module is loaded, and
// a cached address would go stale if the context were reset or replaced
// between calls.  The first call in a context loads the module there.
cudaError_t scratch_address(void **out) {
    void *p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_solve_scratch);
    if (e != cudaSuccess) return e;
    *out = p;
    return cudaSuccess;
}

__global__ void k_na_init(int n, const float *__restrict__ s, double *__restrict__ x, float *__restrict__ b) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    x[i] = 0.0;
    b[i] = s[i];
}

// y = b + K v, one warp per row, plain loads (any CSR layout)
__global__ void k_na_sweep(int n, const int32_t *__restrict__ row_ptr, const int32_t *__restrict__ col,
                           const float *__restrict__ val, const float *__restrict__ b, const float *__restrict__ v,
                           float *__restrict__ y) {
    int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (row >= n) return;
    float acc = 0.f;
    for (int e = row_ptr[row] + lane; e < row_ptr[row + 1]; e += 32) acc += val[e] * v[col[e]];
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) y[row] = b[row] + acc;
}

__global__ void k_na_update(int n, const float *__restrict__ d, double *__restrict__ x) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) x[i] += (double)d[i];
}

// r = s - x + K x in FP64; b = (float) r; per-block sums of r^2 into part
__global__ void k_na_residual(int n, const int32_t *__restrict__ row_ptr, const int32_t *__restrict__ col,
                              const float *__restrict__ val, const float *__restrict__ s,
                              const double *__restrict__ x, float *__restrict__ b, double *__restrict__ part) {
    __shared__ double red[8];
    const int warps = blockDim.x >> 5, w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double loc = 0.0;
    for (int row = blockIdx.x * warps + w; row < n; row += gridDim.x * warps) {
        double acc = 0.0;
        for (int e = row_ptr[row] + lane; e < row_ptr[row + 1]; e += 32) acc += (double)val[e] * x[col[e]];
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (lane == 0) {
            double r = (double)s[row] - x[row] + acc;
            b[row] = (float)r;
            loc += r * r;
        }
    }
    if (lane == 0) red[w] = loc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int i = 0; i < warps; ++i) t += red[i];
        part[blockIdx.x] = t;
    }
}

__global__ void k_na_final(const double *__restrict__ part, int nb, double *__restrict__ out) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    double t = 0.0;
    for (int i = 0; i < nb; ++i) t += part[i];
    *out = t;
}

// ---------------------------------------------------------------------------
// The whole solve in one cooperative launch.
//
// What bounds a sweep of one launch each (k_na_sweep) is the gather of v: 32
// unrelated addresses per warp load, 24 us for 6.1M entries (65,536 rows of a
// band of +-4096), where the matrix itself (49 MB) would take 5 us from L2.
// Here a block owns the same rows for the whole solve, keeps in shared memory
// the window of v that its rows reach (columns modulo n, so a band that wraps
// around is one window) and as many of its entries as fit beside it, as 4-byte
// values and 2-byte window indices; the other entries come from L2, where
// they stay because a line is only ever read by one SM (what L2 cannot hold
// comes from HBM).  Blocks exchange v through global memory with one grid
// barrier per sweep.  A block whose rows reach too far for a window keeps as
// much of it as shared memory holds and gathers the rest from global memory;
// with all gathers from there 100,000 rows of 62 to 124 entries in any column
// took 6,600 us, now 4,130 (a launch per sweep, whose L1 holds more of v: 3,500).
//
// Kept rows are packed to whole quads (zeros that gather a zero), so a lane takes four
// entries per step with two loads of values and indices; 8 lanes (32 in blocks
// whose rows average more than 256 entries) share a row.  80 sweeps over the 65,536
// rows: 2010 us with a launch per sweep, 1159 us in one launch entry by entry
// (a warp per row, bound by its 47 instructions per 32 entries), 1085 us packed,
// 1045 us as here (streamed rows read in whole 32-byte sectors).
//
// The line at kNsMaxNodes is one on rows because the number of entries is not
// known to the host.  Both sides, 80 sweeps, one launch against a launch per
// sweep, us: 2,000 rows of 10 to 20 entries 217 / 380; 131,072 of 62 to 124
// 1,821 / 3,930; 131,072 of 150 to 300 (236 MB) 6,000 / 5,780; 65,536 of 500 to
// 1,000 (393 MB) 7,550 / 7,170; 131,072 of 500 to 1,000 (786 MB, HBM-bound
// either way, and static shares end unevenly) 14,900 / 13,380.
constexpr int kNsThreads = 1024, kNsWarps = kNsThreads / 32;
constexpr int kNsMaxRows = 4096;     // rows a block may keep
constexpr int kNsMaxNodes = 131072;  // above this a launch per sweep
constexpr long long kNsPolls = 1ll << 21;  // polls of one barrier: about 1.5 s
// A row longer than kNsLong entries (kNsLongWide in blocks whose rows average
// more than 256) is cut into chunks of that many, which the block's warps share
// and whose sums one thread adds in order; left to the lanes that share a
// common row it would hold up the whole grid: 65,536 rows of 40 to 80 entries
// and one of 65,536 took 60.5 ms (80 sweeps; a launch per sweep, a warp per row:
// 11.0 ms), with chunks 1.8 ms; 16 of 20,000 19.5 ms (4.7), with chunks 1.3 ms.
constexpr int kNsLong = 512, kNsLongWide = 4096;
constexpr int kNsLongKept = 2048;  // from shared memory the lanes of a common row are quick enough up to here
constexpr int kNsChunks = 256;  // most chunks of a block (longer chunks where they would not do)
constexpr unsigned kNsIsLong = 0x8000u;  // flag of a row in the packed row starts

// an entry's value or column, with an L2 policy or without
template <bool POLICY, typename E>
__device__ __forceinline__ E ns_ld(const E *p, unsigned long long policy) {
    if constexpr (!POLICY) return __ldg(p);
    unsigned v;
    asm("ld.global.nc.L2::cache_hint.u32 %0, [%1], %2;" : "=r"(v) : "l"(p), "l"(policy));
    E r;
    memcpy(&r, &v, 4);
    return r;
}

enum { NS_ALL = 0, NS_SOME = 1, NS_NONE = 2 };  // columns that a pass finds in shared memory

constexpr int kNsL2Entries = 10000000;  // 80 MB, what L2 keeps of a set that is read over and over (65,536 rows of
                                        // 500 to 1,000 entries: 7,760 us without the policies, 7,360 with them when
                                        // they came)

struct NsArgs {
    int n, sweeps, refinements, smem;
    const int32_t *row_ptr, *col;
    const float *val, *s;
    double *x, *resid2, *part;
    float *b, *d0, *d1;
    unsigned *bar;
};

__global__ void __launch_bounds__(kNsThreads, 1) k_na_solve(const __grid_constant__ NsArgs A) {
    extern __shared__ __align__(16) unsigned char ns_dyn[];
    __shared__ int sh_r[2], sh_min[kNsWarps], sh_max[kNsWarps], sh_ok, sh_nch;
    __shared__ int sh_crow[kNsChunks], sh_cst[kNsChunks];  // per chunk: its row and first entry
    __shared__ double sh_csum[kNsChunks], sh_red[kNsWarps];
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31, n = A.n, nb = gridDim.x, blk = blockIdx.x;
    const int32_t *__restrict__ rp = A.row_ptr;
    // rows [r0, r1): equal shares of entries, a row counted as 16 more
    if (tid < 2) {
        const long long base = rp[0], total = (long long)rp[n] - base + 16ll * n;
        const long long target = total * (blk + tid) / nb;
        int lo = 0, hi = n;
        while (lo < hi) {
            const int m = (lo + hi) >> 1;
            if ((long long)rp[m] - base + 16ll * m < target) lo = m + 1;
            else hi = m;
        }
        sh_r[tid] = blk + tid == nb ? n : lo;
    }
    if (tid == 0) sh_nch = 0;
    __syncthreads();
    const int r0 = sh_r[0], r1 = sh_r[1], e0 = rp[r0], ne = rp[r1] - e0;
    // long rows: more than `chunk` entries streamed, more than klong kept
    const bool wide = ne > 256ll * (r1 - r0);
    int chunk = wide ? kNsLongWide : kNsLong;
    auto count = [&]() {  // the chunks of all long rows
        for (int r = r0 + tid; r < r1; r += kNsThreads) {
            const int len = __ldg(rp + r + 1) - __ldg(rp + r);
            if (len > chunk) atomicAdd(&sh_nch, (len - 1) / chunk + 1);
        }
    };
    count();
    // the window: the smallest and largest column, as offsets from r0 modulo n
    int mn = 0x7fffffff, mx = -0x7fffffff;
    for (int e = tid; e < ne; e += kNsThreads) {
        int d = __ldg(A.col + e0 + e) - r0;
        if (d > n / 2) d -= n;
        else if (d < -(n / 2)) d += n;
        mn = min(mn, d);
        mx = max(mx, d);
    }
    for (int o = 16; o > 0; o >>= 1) {
        mn = min(mn, __shfl_xor_sync(0xffffffffu, mn, o));
        mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    if (lane == 0) {
        sh_min[w] = mn;
        sh_max[w] = mx;
    }
    __syncthreads();
    for (int q = 0; q < kNsWarps; ++q) {
        mn = min(mn, sh_min[q]);
        mx = max(mx, sh_max[q]);
    }
    int w0 = r0 + mn, W = mx - mn + 1;
    if (ne == 0) w0 = W = 0;
    else if (W >= n) { w0 = 0; W = n; }
    if (w0 < 0) w0 += n;
    else if (w0 >= n) w0 -= n;
    const bool win4 = W <= 32768;                         // v in shared memory
    const bool win8 = W <= 12288;                         // x too (FP64)
    const int wbytes = win4 ? ((win8 ? 8 : 4) * (W + 1) + 15) / 16 * 16 : 0;  // and a 0, which padding gathers
    // columns of v in shared memory: all of them; or, beside no entries, as many
    // as fit, around the block's own rows, where its entries are enough to pay
    // for the copy (100,000 rows of 20 to 40 entries, 20 thousand a block, 2,277 us
    // without and 1,854 with it; of 30 to 60 3,317 and 2,424)
    int wv = W;
    if (!win4) {
        wv = ne > W / 8 ? min(W, (A.smem - 64) / 4) : 0;
        if (W >= n) w0 = (r0 + r1) / 2 - wv / 2;
        else w0 += (W - wv) / 2;
        if (w0 < 0) w0 += n;
        else if (w0 >= n) w0 -= n;
    }
    const int wx = win8 ? W : 0;  // and of x
    // rows kept, from the first on: packed row starts (in quads), values, indices
    const int capq = win4 ? (A.smem - wbytes - min(r1 - r0 + 1, kNsMaxRows) * 2 - 64) / 24 : 0;  // quads that fit
    float *win = (float *)ns_dyn;
    double *winx = (double *)ns_dyn;
    float4 *sval = (float4 *)(ns_dyn + wbytes);
    uint2 *sidx = (uint2 *)(sval + capq);
    uint16_t *srow = (uint16_t *)(sidx + capq);
    auto local = [&](int c) {
        int d = c - w0;
        d += d < 0 ? n : 0;
        return d;
    };
    while (sh_nch > kNsChunks) {  // longer chunks, until the block can list all of them
        chunk *= 2;
        __syncthreads();
        if (tid == 0) sh_nch = 0;
        __syncthreads();
        count();
        __syncthreads();
    }
    int nch = sh_nch;
    const int klong = max(chunk, kNsLongKept);
    int kept = 0;  // rows [r0, r0 + kept), the long ones among them left out
    if (capq > 0) {
        int carry = 0;
        const int most = min(r1 - r0, kNsMaxRows - 1);
        for (int base = 0; base < most; base += kNsThreads) {
            const int r = base + tid;
            const int len = r < most ? __ldg(rp + r0 + r + 1) - __ldg(rp + r0 + r) : 0;
            const int q = len > klong ? 0 : (len + 3) / 4;
            int v = q;  // inclusive scan over the block
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, v, o);
                if (lane >= o) v += u;
            }
            __syncthreads();
            if (lane == 31) sh_min[w] = v;
            __syncthreads();
            int before = carry, all = 0;
            for (int k = 0; k < kNsWarps; ++k) {
                if (k < w) before += sh_min[k];
                all += sh_min[k];
            }
            v += before;
            const bool fits = r < most && v <= capq;
            if (fits) srow[r + 1] = (uint16_t)(v | (len > klong ? kNsIsLong : 0u));
            if (r == 0) srow[0] = 0;
            const int nf = __syncthreads_count(fits);  // a prefix of the rows: v never falls
            kept = base + nf;
            carry += all;
            if (nf < kNsThreads) break;
        }
    }
    __syncthreads();
    for (int r = tid / 8; r < kept; r += kNsThreads / 8) {
        const int p = __ldg(rp + r0 + r), len = __ldg(rp + r0 + r + 1) - p, q0 = srow[r] & (kNsIsLong - 1);
        if (len > klong) continue;
        float *v = (float *)(sval + q0);
        uint16_t *ix = (uint16_t *)(sidx + q0);
        for (int i = tid % 8; i < (len + 3) / 4 * 4; i += 8) {
            v[i] = i < len ? __ldg(A.val + p + i) : 0.f;
            ix[i] = (uint16_t)(i < len ? local(__ldg(A.col + p + i)) : W);
        }
    }
    // the list of the long rows' chunks (no more than were counted: klong >= chunk)
    auto longest = [&](int row) { return row < r0 + kept ? klong : chunk; };
    if (nch > 0) {
        __syncthreads();
        if (tid == 0) sh_nch = 0;
        __syncthreads();
        for (int r = r0 + tid; r < r1; r += kNsThreads) {
            const int p = __ldg(rp + r), len = __ldg(rp + r + 1) - p;
            if (len <= longest(r)) continue;
            const int nc = (len - 1) / chunk + 1, c0 = atomicAdd(&sh_nch, nc);
            for (int c = 0; c < nc; ++c) {
                sh_crow[c0 + c] = r;
                sh_cst[c0 + c] = p + c * chunk;
            }
        }
        __syncthreads();
        nch = sh_nch;
    }
    unsigned gen = 0;
    auto barrier = [&]() -> bool {
        ++gen;
        __syncthreads();
        if (tid == 0) {
            asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(A.bar) : "memory");
            int ok = 0;
            for (long long i = 0; i < kNsPolls; ++i) {
                unsigned v;
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(A.bar) : "memory");
                if ((int)(v - gen * (unsigned)nb) >= 0) {
                    ok = 1;
                    break;
                }
            }
            sh_ok = ok;
        }
        __syncthreads();
        return sh_ok != 0;
    };
    // Entries streamed beyond what L2 holds for all blocks leave it first, so
    // that they do not push the others out.
    unsigned long long near_by, pass_by;
    asm("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(near_by));
    asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pass_by));
    const int streamed = wide && r0 + kept < r1 ? __ldg(rp + r0 + kept) : e0 + ne;  // the first streamed entry
    const int near_end = e0 + ne - streamed <= kNsL2Entries / nb * 11 / 10 ? 0x7fffffff : streamed + kNsL2Entries / nb;
    // The refinements.  Blocks with a whole window, no long rows and 8 lanes to a
    // row have code of their own: the tests and the registers of the others cost
    // their sweeps 2 to 3 %.
    auto refine = [&](auto general_c) {
        constexpr bool GENERAL = decltype(general_c)::value;
        // Every row's sum over its entries of val times the gathered vector (from
        // the kept entries; else from L2, with the window's `width` columns in
        // shared memory and the others in global memory),
        // handed to out(row, sum) in one lane of the row's L lanes.  The rows that
        // are not kept go first: their loads take longest.  Long rows are skipped
        // (long_rows).
        auto rows = [&](auto lanes_c, auto mode_c, auto zero, const auto *vec, const auto *window, int width, auto out) {
            constexpr int L = decltype(lanes_c)::value, MODE = decltype(mode_c)::value;
            using V = decltype(zero);
            const int sl = lane & (L - 1), first = tid / 32 * (32 / L) + lane / L, lanes = kNsThreads / L;
            auto get = [&](int c) {
                if constexpr (MODE == NS_NONE) return vec[c];
                const int d = local(c);
                if constexpr (MODE == NS_ALL) return window[d];
                return d < width ? window[d] : vec[c];
            };
            auto sum = [&](V acc, int row, bool on) {
                __syncwarp();
#pragma unroll
                for (int o = L / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
                if (sl == 0 && on) out(row, acc);
            };
            const int k0 = MODE == NS_ALL ? kept : 0;
            for (int b = r0 + k0; b < r1; b += lanes) {
                const int row = b + first;
                const bool in_block = row < r1;
                const int p = in_block ? __ldg(rp + row) : 0, row_end = in_block ? __ldg(rp + row + 1) : 0;
                const bool is_long = GENERAL && nch > 0 && row_end - p > (MODE == NS_ALL ? chunk : longest(row));
                const bool on = in_block && !is_long;
                const int end = is_long ? p : row_end;
                V acc = zero;
                constexpr int U = sizeof(V) == 4 ? 6 : 4;
                // (a policy operand costs matrices that stay in L2 2 to 4 %: wide rows only)
                const unsigned long long policy = p < near_end ? near_by : pass_by;
                const int start = sizeof(V) == 4 ? p & ~7 : p;  // sweeps: the lanes' 8 or 32 entries in whole sectors
                for (int e = start + sl; e < end; e += U * L) {
                    float v[U];
                    int c[U];
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const bool in = e + u * L < end && (u > 0 || e >= p);
                        v[u] = in ? ns_ld<L == 32>(A.val + e + u * L, policy) : 0.f;
                        c[u] = in ? ns_ld<L == 32>(A.col + e + u * L, policy) : -1;
                    }
#pragma unroll
                    for (int u = 0; u < U; ++u)
                        if (c[u] >= 0) acc += (V)v[u] * get(c[u]);
                }
                sum(acc, row, on);
            }
            for (int b = 0; b < k0; b += lanes) {
                const int r = b + first;
                bool on = r < k0;
                int q0 = on ? srow[r] : 0, q1 = on ? srow[r + 1] : 0;
                if constexpr (GENERAL) {
                    on = on && !(q1 & kNsIsLong);
                    q0 &= kNsIsLong - 1;
                    q1 = on ? q1 : q0;
                }
                V acc = zero;
#pragma unroll 2
                for (int q = q0 + sl; q < q1; q += L) {
                    const float4 v = sval[q];
                    const uint2 ix = sidx[q];
                    acc += (V)v.x * window[ix.x & 0xffffu];
                    acc += (V)v.y * window[ix.x >> 16];
                    acc += (V)v.z * window[ix.y & 0xffffu];
                    acc += (V)v.w * window[ix.y >> 16];
                }
                sum(acc, r0 + r, on);
            }
        };
        auto long_rows = [&](auto zero, const auto *vec, const auto *window, int width, auto out) {
            using V = decltype(zero);
            for (int c = w; c < nch; c += kNsWarps) {
                const int p = sh_cst[c], re = __ldg(rp + sh_crow[c] + 1), end = re - p > chunk ? p + chunk : re;
                V acc = zero;
#pragma unroll 8
                for (int e = p + lane; e < end; e += 32) {
                    const int k = __ldg(A.col + e), d = local(k);
                    acc += (V)__ldg(A.val + e) * (d < width ? window[d] : vec[k]);
                }
                for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
                if (lane == 0) sh_csum[c] = (double)acc;
            }
            __syncthreads();
            for (int c = tid; c < nch; c += kNsThreads) {
                const int row = sh_crow[c], p = __ldg(rp + row), len = __ldg(rp + row + 1) - p;
                if (sh_cst[c] != p) continue;  // not the row's first
                V t = zero;
                for (int k = 0; k <= (len - 1) / chunk; ++k) t += (V)sh_csum[c + k];
                out(row, t);
            }
            __syncthreads();  // sh_csum
        };
        auto all_rows = [&](auto zero, const auto *vec, const auto *window, int width, auto out) {
            if constexpr (GENERAL) {
                if (nch > 0) long_rows(zero, vec, window, width, out);
                auto go = [&](auto mode_c) {
                    if (wide) rows(std::integral_constant<int, 32>(), mode_c, zero, vec, window, width, out);
                    else rows(std::integral_constant<int, 8>(), mode_c, zero, vec, window, width, out);
                };
                if (width == W) return go(std::integral_constant<int, NS_ALL>());
                if constexpr (sizeof(zero) == 4)
                    if (width > 0) return go(std::integral_constant<int, NS_SOME>());
                go(std::integral_constant<int, NS_NONE>());
            } else {
                constexpr std::integral_constant<int, 8> lanes_c{};
                if (sizeof(zero) == 4 || width == W) rows(lanes_c, std::integral_constant<int, NS_ALL>(), zero, vec, window, width, out);
                else rows(lanes_c, std::integral_constant<int, NS_NONE>(), zero, vec, window, width, out);
            }
        };
        bool ok = true;
        for (int r = 0; ok && r < A.refinements; ++r) {
            if (win4 && tid == 0) win[W] = 0.f;  // (where x's window lay meanwhile)
            const float *cur = A.b;
            for (int k = 0; ok && k < A.sweeps; ++k) {
                float *nxt = (k & 1) ? A.d1 : A.d0;
                if (wv > 0) {
#pragma unroll 8
                    for (int j = tid; j < wv; j += kNsThreads) {
                        const int g = w0 + j;
                        win[j] = __ldcg(cur + (g >= n ? g - n : g));
                    }
                    __syncthreads();
                }
                all_rows(0.f, cur, win, wv, [&](int row, float v) { nxt[row] = A.b[row] + v; });
                cur = nxt;
                ok = barrier();
            }
            if (!ok) break;
            for (int i = r0 + tid; i < r1; i += kNsThreads) A.x[i] += (double)cur[i];
            ok = barrier();
            if (!ok) break;
            if (win8) {
#pragma unroll 4
                for (int j = tid; j < W; j += kNsThreads) {
                    const int g = w0 + j;
                    winx[j] = __ldcg(A.x + (g >= n ? g - n : g));
                }
                __syncthreads();
            }
            double loc = 0.0;
            all_rows(0.0, A.x, winx, wx, [&](int row, double v) {
                const double res = (double)A.s[row] - A.x[row] + v;
                A.b[row] = (float)res;
                loc += res * res;
            });
            if (r == A.refinements - 1 && A.resid2) {
                for (int o = 16; o > 0; o >>= 1) loc += __shfl_xor_sync(0xffffffffu, loc, o);
                if (lane == 0) sh_red[w] = loc;
                __syncthreads();
                if (tid == 0) {
                    double t = 0.0;
                    for (int q = 0; q < kNsWarps; ++q) t += sh_red[q];
                    A.part[blk] = t;
                }
            }
            if (r + 1 < A.refinements || A.resid2) ok = barrier();
        }
        return ok;
    };
    for (int i = r0 + tid; i < r1; i += kNsThreads) {
        A.x[i] = 0.0;
        A.b[i] = A.s[i];
    }
    bool ok = barrier();
    if (win8 && tid == 0) winx[W] = 0.0;
    if (ok) ok = wv == W && nch == 0 && !wide ? refine(std::false_type()) : refine(std::true_type());
    if (!ok) {  // a barrier gave up (the launch is cooperative, so none should): no half result
        for (int i = r0 + tid; i < r1; i += kNsThreads) A.x[i] = __longlong_as_double(0x7ff8000000000000ll);
    }
    if (A.resid2 && blk == 0 && tid == 0) {
        double t = ok ? 0.0 : __longlong_as_double(0x7ff8000000000000ll);
        for (int q = 0; ok && q < nb; ++q) t += __ldcg(A.part + q);
        *A.resid2 = t;
    }
}

// launches k_na_solve; false when this device cannot (the caller then runs a
// launch per sweep)
bool one_launch(const NsArgs &a0, cudaStream_t st) {
    int dev = 0, nsm = 0, smem = 0, coop = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop || nsm < 1 ||
        smem < 160 * 1024)
        return false;
    NsArgs a = a0;
    a.smem = smem - 6 * 1024;  // beside the static shared memory
    int nb = (a.n + kNsWarps - 1) / kNsWarps;
    if (nb > nsm) nb = nsm;
    if (nb > kPartBlocks) nb = kPartBlocks;
    if (cudaFuncSetAttribute(k_na_solve, cudaFuncAttributeMaxDynamicSharedMemorySize, a.smem) != cudaSuccess) return false;
    if (cudaMemsetAsync(a.bar, 0, sizeof(unsigned), st) != cudaSuccess) return false;
    void *args[] = {(void *)&a};
    return cudaLaunchCooperativeKernel((const void *)k_na_solve, dim3(nb), dim3(kNsThreads), args, a.smem, st) == cudaSuccess;
}

}  // namespace

extern "C" tursca_status tursca_csr_solve_noalloc(const int32_t *row_ptr, const int32_t *col, const float *val,
                                                  int n_nodes, const float *s, double *x, int sweeps,
                                                  int refinements, double *resid2, void *cuda_stream) {
    if (!row_ptr || !col || !val || !s || !x) return TURSCA_E_INVALID;
    if (n_nodes < 1 || n_nodes > kMaxNodes) return TURSCA_E_INVALID;
    if (sweeps < 0 || sweeps > 100000 || refinements < 1 || refinements > 1000) return TURSCA_E_INVALID;
    if ((long long)(sweeps + 2) * refinements + 2 > kMaxLaunches) return TURSCA_E_INVALID;
    // an error left pending by earlier work belongs to its owner: report it
    // without clearing it, before launching anything
    if (cudaPeekAtLastError() != cudaSuccess) return TURSCA_E_CUDA;
    void *base = nullptr;
    if (scratch_address(&base) != cudaSuccess) return TURSCA_E_CUDA;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    unsigned char *p = (unsigned char *)base;
    float *b = (float *)(p + kOffB), *d0 = (float *)(p + kOffD0), *d1 = (float *)(p + kOffD1);
    double *part = (double *)(p + kOffPart);
    const int th = 256;
    const int nvec = (n_nodes + th - 1) / th;
    const long long rows_blocks = ((long long)n_nodes * 32 + th - 1) / th;
    int nres = (n_nodes + 7) / 8;
    if (nres > kPartBlocks) nres = kPartBlocks;
    if (n_nodes <= kNsMaxNodes) {
        NsArgs a;
        a.n = n_nodes;
        a.sweeps = sweeps;
        a.refinements = refinements;
        a.smem = 0;
        a.row_ptr = row_ptr;
        a.col = col;
        a.val = val;
        a.s = s;
        a.x = x;
        a.resid2 = resid2;
        a.part = part;
        a.b = b;
        a.d0 = d0;
        a.d1 = d1;
        a.bar = (unsigned *)(p + kOffBar);
        if (one_launch(a, st)) return TURSCA_OK;
        cudaGetLastError();  // its own error only: none was pending
    }
    k_na_init<<<nvec, th, 0, st>>>(n_nodes, s, x, b);
    // a launch that fails (a bad stream, say) fails them all: stop at the first
    if (cudaGetLastError() != cudaSuccess) return TURSCA_E_CUDA;
    for (int r = 0; r < refinements; ++r) {
        const float *cur = b;
        for (int k = 0; k < sweeps; ++k) {
            float *nxt = (k & 1) ? d1 : d0;
            k_na_sweep<<<(unsigned)rows_blocks, th, 0, st>>>(n_nodes, row_ptr, col, val, b, cur, nxt);
            cur = nxt;
        }
        k_na_update<<<nvec, th, 0, st>>>(n_nodes, cur, x);
        k_na_residual<<<nres, th, 0, st>>>(n_nodes, row_ptr, col, val, s, x, b, part);
    }
    if (resid2) k_na_final<<<1, 32, 0, st>>>(part, nres, resid2);
    return cudaGetLastError() == cudaSuccess ? TURSCA_OK : TURSCA_E_CUDA;
}
