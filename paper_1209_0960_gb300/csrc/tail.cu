// The small levels of the V-cycle as one thread-block cluster.
//
// On a level of a few thousand rows a colour pass has a few hundred rows, and
// as a launch of its own it takes about 2 us, nearly all of it launch, grid
// completion and one chain of dependent loads; a V-cycle has 4 C - 2 such
// passes per level of C colours.  Here one cluster of up to 16 blocks runs the
// whole part of the V-cycle from such a level down: pre-smoothing, residual,
// restriction, the levels below, the solve of a small coarsest level,
// prolongation and post-smoothing (two launches around the coarsest solve
// where that one needs all SMs).
//
// Layout.  The rows of a colour are cut into one chunk per block.  Everything a
// block needs for its own rows (entries with 16-bit columns, 1/A_ii, transfer
// lists, its slice of the coarsest inverse) is packed at setup into one image
// per block, which the block copies into its shared memory before it waits for
// the kernel before it: an L2 round trip takes about 1000 cycles, more than a
// whole pass.  Every block also holds the solution vectors of the tail's levels.
// After updating its chunk a block stores a new value into its own copy and
// into those of the blocks that own a neighbour of the row (a bit mask per
// row), and the hardware cluster barrier ends the pass, so every gather is a
// local shared-memory load.  Residuals cross blocks through global memory, once
// per level.
//
// What bounds it, measured on GB300: the cluster barrier takes 0.30 us whatever
// the block count, storing every value to all 16 blocks another 0.25 to 0.45
// us, and float64 arithmetic about 64 cycles per warp instruction on one of the
// four sub-partitions (two lanes a clock per SM), which is why float64 rows
// take two lanes and float32 rows four (eight lanes of either were slower).  A
// pass takes about 0.9 us in float32 and 1.4 us in float64 on a level of 4,000
// to 7,000 rows, against 1.7 to 2.1 us as a launch; with the entries left in
// L2 and loaded one pass ahead it took 1.3 and 2.5 us.  PCG iterations, tail
// against one launch per pass: 64x64 Poisson 98.4 -> 75 us, 61x47x70 mixed 169.7
// -> 148.5 us, 81x64x77 float64 236.0 -> 232.7 us.  (An earlier form that kept x distributed and
// gathered neighbours from the other blocks' shared memory was several times
// slower: remote loads of single values run at about one per ten cycles and SM.)
//
// The rows are updated with the arithmetic of split levels (RowPart).  No
// kernel here spins: blocks wait for each other at barrier.cluster only, which
// every thread of the cluster reaches the same number of times.

#include <algorithm>
#include <cstring>
#include <type_traits>

#include "device.h"
#include "device_util.cuh"

namespace amg {

namespace {

constexpr int kTailThreads = 256;
constexpr int kTailMaxLevels = 12;
// dynamic shared memory a block may use (227 KB less the static part)
constexpr int64_t kTailSmem = 220 * 1024;

// A colour of a level: its rows [r0, r0 + cnt) are cut into chunks of `chunk`
// rows, one per block; a block's rows start at lo among its own rows.
struct TailBlk {
    int32_t r0, cnt, chunk, lo;
};
// Where a block's rows of a colour start in its image: entries, and members of
// the rows' aggregates (levels below the first).
struct TailAt {
    int32_t ent, mem;
};

// One of a block's own rows: position (0xffff: none, in a short last chunk),
// the other blocks that read it, the lengths of its two parts and the place of
// its entries in the image (lower part first).
struct OwnRow {
    uint16_t row, mask, low, up;
    uint32_t e0, members;   // members: of its aggregate on the level above
};

template <typename T>
struct TailLevel {
    // in global memory
    const uint16_t *rlen, *rlow;
    const int32_t* scol;
    const T* sval;
    const T* dinv;
    const int32_t *agg, *rptr, *ridx, *nrp;
    const T* t;
    T *b, *x, *r;
    int64_t sw;
    int32_t n, nc, last, ncolours;    // last: last slot of a slice
    int32_t xoff;                     // its solution in the block's shared memory (elements)
    int32_t own0, nown;               // its own rows among the block's own rows
    int32_t blk0;                     // its colours (the coarsest level: one)
};

template <typename T>
struct TailDesc {
    TailLevel<T> lev[kTailMaxLevels + 1];   // the tail's levels, then the coarsest
    int32_t nlev, nblk, nown, nall;         // own rows without / with the coarsest level's
    int32_t down, up;                       // 1: this launch descends / ascends (both: with the solve)
    int32_t nL, ldM, m32;                   // coarsest rows; row stride and type of M
    int32_t rows_x;                         // elements of all solution vectors
    // byte offsets in a block's shared memory; the image is [img, img + img_bytes)
    int32_t o_bs, o_ps, o_ob, o_os, img, img_bytes;
    int32_t o_row, o_dinv, o_agg, o_aggw, o_mptr, o_mem, o_memw, o_val, o_col, o_M;
    double omega;
    const void* M;
    const TailBlk* blk;
    const TailAt* at;                       // [blocks][nblk]
    unsigned char* image;                   // one image per block
    int32_t* err;
};

// What an index outside its level becomes in an image: positions have 16 bits
// there, and a cut one could fall inside the level again.  It is past the rows
// of every level (kTailMaxRows), so the checked build's kernel reports it each
// time it meets it, as the other kernels do.
constexpr uint16_t kTailOut = 0xfffe;

struct TailBatch {
    const void* desc[kMaxVBatch];
};

template <int NC>
__device__ __forceinline__ void tail_sync() {
    if (NC == 1) {
        __syncthreads();
    } else {
        cluster_arrive();
        cluster_wait();
    }
}

// Lanes per row: with several blocks a chunk is a few dozen rows, and two
// (float64) or four (float32) lanes shorten a row's chain of sums; float64
// sums across more lanes would cost more of the pipe than they save.  A block
// alone has enough rows for one lane each.
template <typename T, int NC>
__host__ __device__ constexpr int tail_lanes() {
    return NC == 1 ? 1 : std::is_same<T, double>::value ? 2 : 4;
}

template <typename T, int NC>
__global__ void __launch_bounds__(kTailThreads, 1) k_tail(const TailBatch batch) {
    constexpr int G = tail_lanes<T, NC>();
    constexpr int kPer = kTailThreads / G;   // rows a block updates at once
    using Lower = std::integral_constant<int, kPartLower>;
    using Upper = std::integral_constant<int, kPartUpper>;
    using Both = std::integral_constant<int, kPartBoth>;
    extern __shared__ __align__(16) unsigned char tsm[];
    __shared__ TailLevel<T> lev[kTailMaxLevels + 1];
    pdl_launch_dependents();
    const TailDesc<T>& D = *static_cast<const TailDesc<T>*>(batch.desc[blockIdx.x / NC]);
    const int rank = (int)(blockIdx.x % NC), tid = (int)threadIdx.x;
    const int slot = tid / G, lane = tid % G;
    // the image (setup-time data only)
    {
        const int4* src = reinterpret_cast<const int4*>(D.image + (size_t)rank * D.img_bytes);
        int4* to = reinterpret_cast<int4*>(tsm + D.img);
        const int m = D.img_bytes >> 4;
#pragma unroll 8
        for (int i = tid; i < m; i += kTailThreads) to[i] = __ldg(src + i);
    }
    const int nlev = D.nlev, nL = D.nL;
    const bool down = D.down != 0, up = D.up != 0, m32 = D.m32 != 0;
    int32_t* const err = D.err;
    T* const xs = reinterpret_cast<T*>(tsm);
    double* const bs = reinterpret_cast<double*>(tsm + D.o_bs);
    double* const ps = reinterpret_cast<double*>(tsm + D.o_ps);
    T* const ob = reinterpret_cast<T*>(tsm + D.o_ob);
    T* const os = reinterpret_cast<T*>(tsm + D.o_os);
    const OwnRow* const orow = reinterpret_cast<const OwnRow*>(tsm + D.o_row);
    const T* const od = reinterpret_cast<const T*>(tsm + D.o_dinv);
    const uint16_t* const oagg = reinterpret_cast<const uint16_t*>(tsm + D.o_agg);
    const T* const oaggw = reinterpret_cast<const T*>(tsm + D.o_aggw);
    const uint32_t* const mptr = reinterpret_cast<const uint32_t*>(tsm + D.o_mptr);
    const uint16_t* const mem = reinterpret_cast<const uint16_t*>(tsm + D.o_mem);
    const T* const memw = reinterpret_cast<const T*>(tsm + D.o_memw);
    const T* const val = reinterpret_cast<const T*>(tsm + D.o_val);
    const uint16_t* const col = reinterpret_cast<const uint16_t*>(tsm + D.o_col);
    constexpr bool kScaled = std::is_same<T, float>::value;
    const T omega = (T)D.omega;
    for (int i = tid; i < (nlev + 1) * (int)(sizeof(TailLevel<T>) / 4); i += kTailThreads)
        reinterpret_cast<uint32_t*>(lev)[i] = reinterpret_cast<const uint32_t*>(D.lev)[i];
    TailBlk* const blk = reinterpret_cast<TailBlk*>(tsm + D.img + D.img_bytes);
    for (int i = tid; i < D.nblk * (int)(sizeof(TailBlk) / 4); i += kTailThreads)
        reinterpret_cast<uint32_t*>(blk)[i] = reinterpret_cast<const uint32_t*>(D.blk)[i];
    const uint32_t xs_addr = smem_u32(xs);
    // the value of own row o of a level (element k of the solutions), from the
    // lanes of the row
    auto publish = [&](const OwnRow& o, int k, T v) {
        if (lane == 0) xs[k] = v;
        if (NC > 1) {
            const uint32_t a = xs_addr + (uint32_t)(k * (int)sizeof(T));
#pragma unroll
            for (int d = 0; d < (NC + G - 1) / G; ++d) {
                const int q = d * G + lane;
                if (q < NC && (o.mask >> q & 1)) st_cluster(map_rank(a, (uint32_t)q), v);
            }
        }
    };
    __syncthreads();

    // acc - the entries of one part of own row o times x
    auto part = [&](T acc, const OwnRow& o, bool upper, int n, const T* x) {
        const int cnt = upper ? o.up : o.low;
        const uint32_t e0 = o.e0 + (upper ? o.low : 0);
#pragma unroll 4
        for (int t = lane; t < cnt; t += G) {
            const int j = col[e0 + t];
            if (index_ok(j, n, err)) acc = fmad(-val[e0 + t], x[j], acc);
        }
        __syncwarp();
        return acc;
    };
    auto sum = [&](T s) {
#pragma unroll
        for (int off = G >> 1; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
        return s;
    };
    // whether this warp has rows of [k0, end) (the others go straight to the barrier)
    auto warp_has = [&](int end, int k0) { return k0 + ((tid & ~31) / G) < end; };

    // one colour pass
    auto pass = [&](const TailLevel<T>& L, int c, auto part_tag) {
        constexpr int which = decltype(part_tag)::value;
        const TailBlk q = blk[L.blk0 + c];
        const T* x = xs + L.xoff;
        const int base = L.own0 + q.lo;
        for (int k0 = 0; warp_has(q.chunk, k0); k0 += kPer) {
            const int k = k0 + slot;
            OwnRow o = {0xffff, 0, 0, 0, 0u, 0u};
            if (k < q.chunk) o = orow[base + k];
            const bool has = o.row != 0xffff, lead = has && lane == 0;
            const int oi = base + (has ? k : 0);
            T s = T(0), w = T(0);
            if (which != kPartUpper) {
                s = sum(part(lead ? ob[oi] : T(0), o, false, L.n, x));
                if (lead) os[oi] = s;
            }
            if (which != kPartLower) {
                const T a0 = (lead && which == kPartUpper) ? (c == 0 ? ob[oi] : os[oi]) : T(0);
                w = sum(part(a0, o, true, L.n, x));
            }
            if (has) {
                const T sx = which == kPartLower ? s : which == kPartBoth ? s + w : w;
                publish(o, L.xoff + o.row, sx * od[oi]);
            }
        }
        tail_sync<NC>();
    };

    pdl_wait();
    if (down) {
        const TailLevel<T>& L = lev[0];
        for (int i = tid; i < L.nown; i += kTailThreads) {
            const int row = orow[L.own0 + i].row;
            if (row != 0xffff) ob[L.own0 + i] = L.b[row];
        }
    } else {
        // the descent's launch left x and b of every level in global memory
        for (int l = 0; l <= nlev; ++l) {
            const TailLevel<T>& L = lev[l];
            T* x = xs + L.xoff;
#pragma unroll 8
            for (int i = tid; i < L.n; i += kTailThreads) x[i] = L.x[i];
            if (l == nlev) break;
            for (int i = tid; i < L.nown; i += kTailThreads) {
                const int row = orow[L.own0 + i].row;
                if (row != 0xffff) ob[L.own0 + i] = L.b[row];
            }
        }
    }
    // every block of the cluster has started and holds its data
    tail_sync<NC>();

    if (down) {
#pragma unroll 1
        for (int l = 0; l < nlev; ++l) {
            const TailLevel<T>& L = lev[l];
            const int C = L.ncolours;
            {   // colour 0 from a zero guess
                const TailBlk q = blk[L.blk0];
                for (int k = slot; k < q.chunk; k += kPer) {
                    const int oi = L.own0 + q.lo + k;
                    const OwnRow o = orow[oi];
                    if (o.row != 0xffff) publish(o, L.xoff + o.row, ob[oi] * od[oi]);
                }
                tail_sync<NC>();
            }
#pragma unroll 1
            for (int c = 1; c < C; ++c) pass(L, c, Lower());
#pragma unroll 1
            for (int c = C - 2; c >= 0; --c) pass(L, c, Upper());
            {   // residual of the own rows of colour >= 1, into global memory
                const T* x = xs + L.xoff;
                for (int k0 = blk[L.blk0 + 1].lo; warp_has(L.nown, k0); k0 += kPer) {
                    const int oi = L.own0 + k0 + slot;
                    OwnRow o = {0xffff, 0, 0, 0, 0u, 0u};
                    if (k0 + slot < L.nown) o = orow[oi];
                    const bool lead = o.row != 0xffff && lane == 0;
                    const T s = sum(part(lead ? ob[oi] - os[oi] : T(0), o, false, L.n, x));
                    if (lead) L.r[o.row] = s;
                }
                tail_sync<NC>();
            }
            // right-hand side of the own rows of the next level
            const TailLevel<T>& N = lev[l + 1];
            const bool coarsest = l + 1 == nlev;
            for (int i = tid; i < N.nown; i += kTailThreads) {
                const int oi = N.own0 + i;
                const OwnRow o = orow[oi];
                if (o.row == 0xffff) continue;
                const int kb = (int)mptr[oi], k1 = kb + (int)o.members;
                T s = T(0);
                for (int k = kb; k < k1; k += 8) {
                    T v[8];
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        v[u] = T(0);
                        if (k + u < k1) {
                            const int m = mem[k + u];
                            if (index_ok(m, L.n, err)) v[u] = __ldcg(L.r + m);
                        }
                    }
#pragma unroll
                    for (int u = 0; u < 8; ++u)
                        if (k + u < k1) s += kScaled ? memw[k + u] * v[u] : v[u];
                }
                if (!coarsest) ob[oi] = s;
                if (!up) {
                    N.b[o.row] = s;
                } else if (coarsest) {
                    // every block's share of the solve reads all of b
                    if (m32) {
                        float* at = reinterpret_cast<float*>(bs) + o.row;
                        if (NC == 1) *at = (float)s;
                        else
                            for (int q = 0; q < NC; ++q) st_cluster(map_rank(smem_u32(at), (uint32_t)q), (float)s);
                    } else {
                        double* at = bs + o.row;
                        if (NC == 1) *at = (double)s;
                        else
                            for (int q = 0; q < NC; ++q) st_cluster(map_rank(smem_u32(at), (uint32_t)q), (double)s);
                    }
                }
            }
            if (coarsest) tail_sync<NC>();
            else __syncthreads();
        }
    }
    if (down && up) {
        // e = M b, a chunk of rows per block: groups of 32 rows, the columns of
        // a group split over the warps that are left, partial sums combined in
        // order.  M is symmetric: the image holds the block's rows of M^T, so the
        // lanes of a warp read consecutive values.
        const TailLevel<T>& E = lev[nlev];
        const int chunk = E.nown, groups = (chunk + 31) >> 5;
        const int splits = max(1, (kTailThreads / 32) / groups);
        const int warp = tid >> 5, ln = tid & 31;
        for (int g0 = 0; g0 < groups; g0 += kTailThreads / 32) {
            const int g = splits > 1 ? warp % groups : g0 + warp, sp = splits > 1 ? warp / groups : 0;
            const int q = g * 32 + ln;
            OwnRow o = {0xffff, 0, 0, 0, 0u, 0u};
            if (g < groups && sp < splits && q < chunk) o = orow[E.own0 + q];
            const bool valid = o.row != 0xffff;
            double acc = 0.0;
            if (valid) {
                const int c0 = nL * sp / splits, c1 = nL * (sp + 1) / splits;
                if (m32) {
                    const float* m = reinterpret_cast<const float*>(tsm + D.o_M) + q;
                    const float* bf = reinterpret_cast<const float*>(bs);
                    float a0 = 0.f;
#pragma unroll 4
                    for (int c = c0; c < c1; ++c) a0 = fmaf(m[c * chunk], bf[c], a0);
                    acc = (double)a0;
                } else {
                    const double* m = reinterpret_cast<const double*>(tsm + D.o_M) + q;
#pragma unroll 4
                    for (int c = c0; c < c1; ++c) acc = fmad(m[c * chunk], bs[c], acc);
                }
            }
            ps[tid] = acc;
            __syncthreads();
            if (valid && sp == 0) {
                for (int k = 1; k < splits; ++k) acc += ps[tid + 32 * groups * k];
                const int k = E.xoff + o.row;
                xs[k] = (T)acc;
                if (NC > 1)
                    for (int r = 0; r < NC; ++r)
                        if (o.mask >> r & 1)
                            st_cluster(map_rank(xs_addr + (uint32_t)(k * (int)sizeof(T)), (uint32_t)r), (T)acc);
            }
            __syncthreads();
        }
        tail_sync<NC>();
    }
    if (up) {
#pragma unroll 1
        for (int l = nlev - 1; l >= 0; --l) {
            const TailLevel<T>& L = lev[l];
            const int C = L.ncolours;
            const T* e = xs + lev[l + 1].xoff;
            // x += omega P e on the own rows of colour >= 1.  All lanes of a row
            // read its x; lane 0 replaces it once they have (the other lanes
            // send the sum to the blocks that read the row).
            for (int k0 = blk[L.blk0 + 1].lo; warp_has(L.nown, k0); k0 += kPer) {
                const int oi = L.own0 + k0 + slot;
                OwnRow o = {0xffff, 0, 0, 0, 0u, 0u};
                if (k0 + slot < L.nown) o = orow[oi];
                const int g = o.row != 0xffff ? oagg[oi] : 0xffff;
                const bool has = g != 0xffff && index_ok(g, L.nc, err);
                T v = T(0);
                if (has) v = fmad(kScaled ? omega * oaggw[oi] : omega, e[g], xs[L.xoff + o.row]);
                __syncwarp();
                if (has) publish(o, L.xoff + o.row, v);
            }
            tail_sync<NC>();
#pragma unroll 1
            for (int c = 0; c < C; ++c) pass(L, c, Both());
#pragma unroll 1
            for (int c = C - 2; c >= 0; --c) pass(L, c, Upper());
        }
    }
    // results: x of the first level, or of every level for the ascent's launch
    const int lout = up ? 1 : nlev;
    for (int l = 0; l < lout; ++l) {
        const TailLevel<T>& L = lev[l];
        for (int i = tid; i < L.nown; i += kTailThreads) {
            const int row = orow[L.own0 + i].row;
            if (row != 0xffff) L.x[row] = xs[L.xoff + row];
        }
    }
}

// ---------------------------------------------------------------------------
// The blocks' images, read from the levels' arrays: blockIdx.y = block of the
// cluster, one thread per own row (colour by colour its chunk of each level, the
// coarsest level's rows as one colour last).
// ---------------------------------------------------------------------------
__device__ __forceinline__ int tail_owner(const TailBlk* blk, int nblk, int row) {
    int c = 0;
    while (c + 1 < nblk && row >= blk[c + 1].r0) ++c;
    return blk[c].chunk > 0 ? (row - blk[c].r0) / blk[c].chunk : 0;
}

constexpr int kPackThreads = 128;

template <typename T>
__global__ void __launch_bounds__(kPackThreads) k_tail_pack(const TailDesc<T>* Dp) {
    const TailDesc<T>& D = *Dp;
    const int rank = (int)blockIdx.y, gi = (int)(blockIdx.x * kPackThreads + threadIdx.x);
    unsigned char* img = D.image + (size_t)rank * D.img_bytes - D.img;   // offsets are shared-memory ones
    constexpr bool kScaled = std::is_same<T, float>::value;
    if (gi < D.nall) {
        int l = 0;
        while (l < D.nlev && gi >= D.lev[l + 1].own0) ++l;
        const TailLevel<T>& L = D.lev[l];
        const bool coarsest = l == D.nlev;
        const TailBlk* blk = D.blk + L.blk0;
        int c = L.ncolours - 1;
        while (c > 0 && gi - L.own0 < blk[c].lo) --c;
        const int first = blk[c].r0 + rank * blk[c].chunk;   // the block's first row of the colour
        const int row = first + (gi - L.own0 - blk[c].lo);
        const bool has = row < blk[c].r0 + blk[c].cnt;
        const TailAt at = D.at[rank * D.nblk + L.blk0 + c];
        OwnRow o = {0xffff, 0, 0, 0, 0u, 0u};
        uint32_t mask = 0, m0 = (uint32_t)at.mem;
        if (has) {
            o.row = (uint16_t)row;
            if (!coarsest) {
                o.low = L.rlow[row];
                o.up = (uint16_t)(L.rlen[row] - o.low);
                o.e0 = (uint32_t)(at.ent + L.nrp[row] - L.nrp[first]);
                T* val = reinterpret_cast<T*>(img + D.o_val) + o.e0;
                uint16_t* col = reinterpret_cast<uint16_t*>(img + D.o_col) + o.e0;
                const int64_t base = (int64_t)(row >> 5) * L.sw + (row & 31);
                for (int t = 0; t < o.low + o.up; ++t) {
                    const int64_t e = base + 32 * (int64_t)(t < o.low ? t : L.last - (t - o.low));
                    const int j = L.scol[e];
                    const bool in = index_ok(j, L.n, D.err);
                    col[t] = in ? (uint16_t)j : kTailOut;
                    val[t] = L.sval[e];
                    if (in) mask |= 1u << tail_owner(blk, L.ncolours, j);
                }
            }
            if (l > 0) {   // the row's value goes to its members, its right-hand side comes from them
                const TailLevel<T>& F = D.lev[l - 1];
                const int kb = F.rptr[row], k1 = F.rptr[row + 1];
                m0 += (uint32_t)(kb - F.rptr[first]);
                uint16_t* mem = reinterpret_cast<uint16_t*>(img + D.o_mem) + m0;
                T* memw = reinterpret_cast<T*>(img + D.o_memw) + m0;
                for (int k = kb; k < k1; ++k) {
                    const int m = F.ridx[k];
                    const bool in = index_ok(m, F.n, D.err);
                    mem[k - kb] = in ? (uint16_t)m : kTailOut;
                    if (kScaled) memw[k - kb] = in ? F.t[m] : T(0);
                    if (in) mask |= 1u << tail_owner(D.blk + F.blk0, F.ncolours, m);
                }
                o.members = (uint32_t)(k1 - kb);
            }
            o.mask = (uint16_t)(mask & ~(1u << rank));
        }
        reinterpret_cast<OwnRow*>(img + D.o_row)[gi] = o;
        reinterpret_cast<uint32_t*>(img + D.o_mptr)[gi] = m0;
        if (!coarsest) {
            reinterpret_cast<T*>(img + D.o_dinv)[gi] = has ? L.dinv[row] : T(0);
            const int g = has ? L.agg[row] : -1;
            const bool in = g < 0 || index_ok(g, L.nc, D.err);
            reinterpret_cast<uint16_t*>(img + D.o_agg)[gi] = g < 0 ? (uint16_t)0xffff
                                                             : in  ? (uint16_t)g
                                                                   : kTailOut;
            if (kScaled) reinterpret_cast<T*>(img + D.o_aggw)[gi] = g >= 0 ? L.t[row] : T(0);
        }
    }
    if (D.down && D.up) {
        const int chunk = D.lev[D.nlev].nown;
        for (int k = gi; k < chunk * D.nL; k += (int)(gridDim.x * kPackThreads)) {
            const int c = k / chunk, row = rank * chunk + k % chunk;
            if (D.m32)
                reinterpret_cast<float*>(img + D.o_M)[k] =
                    row < D.nL ? static_cast<const float*>(D.M)[(size_t)row * D.ldM + c] : 0.f;
            else
                reinterpret_cast<double*>(img + D.o_M)[k] =
                    row < D.nL ? static_cast<const double*>(D.M)[(size_t)row * D.ldM + c] : 0.0;
        }
    }
}

template <typename T>
struct TailArrays;
template <>
struct TailArrays<double> {
    static void fill(TailLevel<double>& t, const DevLevel& L) {
        t.sval = L.sval, t.dinv = L.dinv, t.t = nullptr, t.b = L.b, t.x = L.x, t.r = L.r;
    }
};
template <>
struct TailArrays<float> {
    static void fill(TailLevel<float>& t, const DevLevel& L) {
        t.sval = L.sval32, t.dinv = L.dinv32, t.t = L.t32, t.b = L.b32, t.x = L.x32, t.r = L.r32;
    }
};

// Least blocks of the cluster for a tail whose first level has n rows.  More
// blocks share the float64 work and the entries; one block needs no cluster
// barrier.  Measured per PCG iteration: 64x64 Poisson (tail from 983 rows) 80.8
// us with one block, 75.4 with 8, 76.7 with 16; 61x47x70 mixed (4,191 rows)
// 148.3 us with 16, 156.8 with 8.
inline int tail_blocks(int32_t n) { return n <= 300 ? 1 : n <= 2000 ? 8 : 16; }

template <typename T, int NC>
void tail_launch(const TailBatch& b, int nrec, size_t smem, cudaStream_t s) {
    void (*kern)(const TailBatch) = k_tail<T, NC>;
    raise_dyn_smem(kern, smem);
    if (NC > 8) {
        const cudaError_t e = cudaFuncSetAttribute(reinterpret_cast<const void*>(kern),
                                                   cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) {
            cudaGetLastError();
            throw Error{AMG_ECUDA, std::string("cluster size of the small levels: ") + cudaGetErrorString(e)};
        }
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(NC * nrec));
    cfg.blockDim = dim3(kTailThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = NC;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    unsigned na = 1;
    if (t_launch_overlap) {
        attr[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[na].val.programmaticStreamSerializationAllowed = 1;
        ++na;
    }
    cfg.attrs = attr;
    cfg.numAttrs = na;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, b);
    if (e != cudaSuccess) {
        cudaGetLastError();
        throw Error{AMG_ECUDA, std::string("launch of the small levels (") + std::to_string(NC) +
                                   " blocks, shared " + std::to_string(smem) +
                                   " B) failed: " + cudaGetErrorString(e)};
    }
}

template <typename T, int NC>
void tail_batch(const VRec* const* recs, int n, cudaStream_t s) {
    TailBatch b = {};
    size_t smem = 0;
    for (int k = 0; k < n; ++k) {
        b.desc[k] = recs[k]->a.dv;
        smem = std::max(smem, recs[k]->smem);
    }
    tail_launch<T, NC>(b, n, smem, s);
}

template <typename T>
VBatchLauncher tail_launcher(int nc) {
    return nc == 1 ? &tail_batch<T, 1> : nc == 8 ? &tail_batch<T, 8> : &tail_batch<T, 16>;
}

inline int64_t align16(int64_t v) { return (v + 15) & ~int64_t(15); }

// Lays out the tail from level l0 for a cluster of `blocks` blocks.
template <typename T>
struct TailPlan {
    TailDesc<T> d = {};
    std::vector<TailBlk> blk;
    std::vector<TailAt> at;   // [blocks][colours of all levels]
    int64_t smem = 0;
    int nc;

    // down, up: which half (both: with the coarsest solve in between)
    TailPlan(const std::vector<DevLevel>& dl, int l0, int blocks, bool down, bool up, bool m32)
        : nc(blocks) {
        const int nlev = (int)dl.size(), m = nlev - 1 - l0;
        d.nlev = m;
        d.down = down ? 1 : 0;
        d.up = up ? 1 : 0;
        d.nL = dl[nlev - 1].n;
        d.m32 = m32 ? 1 : 0;
        for (int k = 0; k <= m; ++k) {
            const DevLevel& L = dl[l0 + k];
            TailLevel<T>& t = d.lev[k];
            TailArrays<T>::fill(t, L);
            t.n = L.n;
            t.xoff = d.rows_x;
            d.rows_x += L.n;
            t.own0 = d.nall;
            t.blk0 = (int32_t)blk.size();
            t.ncolours = k < m ? L.ncolours : 1;
            int32_t lo = 0;
            for (int c = 0; c < t.ncolours; ++c) {
                TailBlk q;
                q.r0 = k < m ? L.cptr[c] : 0;
                q.cnt = (k < m ? L.cptr[c + 1] : L.n) - q.r0;
                q.chunk = (q.cnt + nc - 1) / nc;
                q.lo = lo;
                lo += q.chunk;
                blk.push_back(q);
            }
            t.nown = lo;
            d.nall += lo;
            if (k == m) break;
            t.nc = L.n_coarse;
            t.last = L.width - 1;
            t.sw = L.sw;
            t.rlen = L.rlen;
            t.rlow = L.rlow;
            t.scol = L.scol;
            t.agg = L.agg;
            t.rptr = L.rptr;
            t.ridx = L.ridx;
            t.nrp = L.nrp;
        }
        // where each block's colours start in its image
        d.nblk = (int32_t)blk.size();
        at.resize((size_t)nc * d.nblk);
        int64_t E = 0, M = 0;
        for (int r = 0; r < nc; ++r) {
            int64_t e = 0, mm = 0;
            for (int k = 0; k <= m; ++k)
                for (int c = 0; c < d.lev[k].ncolours; ++c) {
                    const int i = d.lev[k].blk0 + c;
                    const TailBlk& q = blk[i];
                    const int32_t a = q.r0 + std::min(q.cnt, r * q.chunk), z = q.r0 + std::min(q.cnt, (r + 1) * q.chunk);
                    at[(size_t)r * d.nblk + i] = {(int32_t)e, (int32_t)mm};
                    if (k < m) e += dl[l0 + k].nrp_host[z] - dl[l0 + k].nrp_host[a];
                    if (k > 0) mm += dl[l0 + k - 1].rptr_host[z] - dl[l0 + k - 1].rptr_host[a];
                }
            E = std::max(E, e);
            M = std::max(M, mm);
        }
        d.nown = d.lev[m].own0;
        const bool dense = down && up;
        int64_t pos = align16((int64_t)d.rows_x * sizeof(T));
        auto take = [&](int32_t& off, int64_t bytes) {
            off = (int32_t)pos;
            pos = align16(pos + bytes);
        };
        take(d.o_bs, dense ? 8 * (int64_t)d.nL : 0);
        take(d.o_ps, dense ? 8 * kTailThreads : 0);
        take(d.o_ob, (int64_t)d.nown * sizeof(T));
        take(d.o_os, (int64_t)d.nown * sizeof(T));
        d.img = (int32_t)pos;
        take(d.o_row, (int64_t)d.nall * sizeof(OwnRow));
        take(d.o_dinv, (int64_t)d.nown * sizeof(T));
        take(d.o_agg, (int64_t)d.nown * 2);
        take(d.o_aggw, std::is_same<T, float>::value ? (int64_t)d.nown * sizeof(T) : 0);
        take(d.o_mptr, 4 * (int64_t)d.nall);
        take(d.o_mem, 2 * M);
        take(d.o_memw, std::is_same<T, float>::value ? M * (int64_t)sizeof(T) : 0);
        take(d.o_val, E * (int64_t)sizeof(T));
        take(d.o_col, E * 2);
        take(d.o_M, dense ? (int64_t)d.nL * d.lev[m].nown * (m32 ? 4 : 8) : 0);
        d.img_bytes = (int32_t)(pos - d.img);
        smem = pos + (int64_t)d.nblk * sizeof(TailBlk);
    }
};

// Whether the coarsest solve joins the cluster's launch: 16 SMs have a tenth of
// the float64 rate, so a solve of many rows is a launch over all SMs.
inline bool tail_dense(int32_t nL) { return nL <= kTailDenseMax; }

template <typename T>
const void* tail_kernel(int nc) {
    void (*k)(const TailBatch) = nc == 1 ? &k_tail<T, 1> : nc == 8 ? &k_tail<T, 8> : &k_tail<T, 16>;
    return reinterpret_cast<const void*>(k);
}

// Blocks of the cluster for the tail from level l0; 0 if it does not fit: in
// shared memory, or on a device (or a part of one) that cannot hold the cluster.
template <typename T>
int tail_cluster(const amg_ctx* c, int l0, bool m32) {
    const int nlev = (int)c->dl.size(), m = nlev - 1 - l0;
    if (m < 1 || m > kTailMaxLevels) return 0;
    int64_t rows = 0;
    for (int l = l0; l < nlev; ++l) {
        if (l < nlev - 1 && !c->dl[l].split) return 0;
        if (c->dl[l].n >= kTailMaxRows || (l < nlev - 1 && !c->dl[l].nrp)) return 0;
        rows += c->dl[l].n;
    }
    if (rows * (int64_t)sizeof(T) > kTailSmem) return 0;
    const bool one = tail_dense(c->nL);
    for (int nc : {1, 8, 16}) {
        if (nc < tail_blocks(c->dl[l0].n)) continue;
        int64_t smem = TailPlan<T>(c->dl, l0, nc, true, one, m32).smem;
        if (!one) smem = std::max(smem, TailPlan<T>(c->dl, l0, nc, false, true, m32).smem);
        if (smem <= kTailSmem && resident_clusters(tail_kernel<T>(nc), nc, kTailThreads, (size_t)smem) > 0)
            return nc;
    }
    return 0;
}

// The device descriptor of one launch.  image: of the other half, whose layout
// is the same, or null to pack one.
template <typename T>
TailHalf upload_tail(amg_ctx* c, TailPlan<T>& p, const void* M, int ld, unsigned char** image) {
    cudaStream_t s = c->stream;
    const bool pack = !*image;
    if (pack) *image = c->mem.alloc<unsigned char>((size_t)p.d.img_bytes * p.nc);
    // one copy: descriptor, colours, image offsets
    const size_t b0 = sizeof(TailDesc<T>), b1 = b0 + sizeof(TailBlk) * p.blk.size(),
                 b2 = b1 + sizeof(TailAt) * p.at.size();
    unsigned char* dev = c->mem.alloc<unsigned char>(b2);
    p.d.image = *image;
    p.d.blk = reinterpret_cast<const TailBlk*>(dev + b0);
    p.d.at = reinterpret_cast<const TailAt*>(dev + b1);
    p.d.M = M;
    p.d.ldM = ld;
    p.d.omega = c->p.omega;
    p.d.err = c->dl[0].err;
    std::vector<unsigned char> host(b2);
    std::memcpy(host.data(), &p.d, b0);
    std::memcpy(host.data() + b0, p.blk.data(), b1 - b0);
    std::memcpy(host.data() + b1, p.at.data(), b2 - b1);
    // (a copy from pageable memory has left the host buffer when it returns)
    AMG_CUDA_TRY(cudaMemcpyAsync(dev, host.data(), b2, cudaMemcpyHostToDevice, s));
    if (pack) {
        k_tail_pack<T><<<dim3((unsigned)((p.d.nall + kPackThreads - 1) / kPackThreads), (unsigned)p.nc),
                         kPackThreads, 0, s>>>(reinterpret_cast<const TailDesc<T>*>(dev));
        AMG_CUDA_TRY(cudaGetLastError());
    }
    TailHalf h;
    h.desc = dev;
    h.smem = (size_t)p.smem;
    h.blocks = p.nc;
    return h;
}

template <typename T>
Tail make_tail(amg_ctx* c, int l0) {
    const bool f32 = std::is_same<T, float>::value;
    const bool m32 = f32 && c->Ainv_s32;
    const void* M = m32 ? (const void*)c->Ainv_s32 : f32 ? (const void*)c->Ainv_s : (const void*)c->Ainv;
    const int ld = m32 ? c->ld32 : c->nL;
    const int nc = tail_cluster<T>(c, l0, m32);
    if (nc == 0) throw Error{AMG_EINVAL, "the levels do not fit in one cluster"};
    Tail t;
    t.one = tail_dense(c->nL);
    unsigned char* image = nullptr;
    TailPlan<T> p(c->dl, l0, nc, true, t.one, m32);
    t.down = upload_tail<T>(c, p, M, ld, &image);
    if (!t.one) {
        TailPlan<T> q(c->dl, l0, nc, false, true, m32);
        t.up = upload_tail<T>(c, q, M, ld, &image);
    }
    return t;
}

}  // namespace

bool tail_fits(const amg_ctx* c, int l0, bool f32) {
    return (f32 ? tail_cluster<float>(c, l0, c->p.coarsest_fp32 != 0) : tail_cluster<double>(c, l0, false)) > 0;
}

const Tail& tail_of(amg_ctx* c, int l0, bool f32) {
    auto& m = c->tails[f32 ? 1 : 0];
    auto it = m.find(l0);
    if (it == m.end()) it = m.emplace(l0, f32 ? make_tail<float>(c, l0) : make_tail<double>(c, l0)).first;
    return it->second;
}

void launch_tail(const TailHalf& h, bool f32, cudaStream_t s) {
    const VBatchLauncher f = f32 ? tail_launcher<float>(h.blocks) : tail_launcher<double>(h.blocks);
    VRec r;
    r.launch = f;
    r.grid = h.blocks;
    r.block = kTailThreads;
    r.smem = h.smem;
    r.a.dv = h.desc;
    if (t_vrecord) {
        r.phase = t_vkey.phase;
        r.level = t_vkey.level;
        r.step = t_vkey.step++;
        t_vrecord->push_back(r);
        return;
    }
    const VRec* one = &r;
    f(&one, 1, s);
}

}  // namespace amg
