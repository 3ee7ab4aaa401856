// Octree over Morton-sorted members (Section 2.2.2: cubic cells divided into
// 8 subcells until a cell holds at most `leaf` members, one radiation source
// per cell for the source tree) and its luminosity moments (L = sum L_j,
// r = sum L_j r_j / sum L_j; the same form with N_rec for emitters, Eq. ssum).
//
// Depth-first pre-order with children in octant order is the order of (first
// member, level), so the tree needs no level-by-level construction: one
// thread per sorted key counts the cells that start at it, a scan of the
// counts gives every cell its pre-order index, and a second pass writes the
// records -- the end of a cell's keys is found by a galloping search, its skip
// pointer is the scan at that end, its parent the cell of the next coarser
// level that holds its first key.  (Level by level -- children counted, scanned
// and emitted, then subtree sizes and positions -- took eight launches and
// seven chained binary searches per cell and level: 0.62 ms for 2^20 members,
// 0.38 ms for 23 k, against 0.16 and 0.06 ms.)
//
// The members of a batch of problems lie one problem after the other (Segs);
// the same passes then build the forest of their trees.
#include "common.cuh"

namespace st {

__device__ __forceinline__ u32 compact3(u64 v)
{
    v &= 0x1249249249249249ull;
    v = (v | (v >> 2)) & 0x10c30c30c30c30c3ull;
    v = (v | (v >> 4)) & 0x100f00f00f00f00full;
    v = (v | (v >> 8)) & 0x1f0000ff0000ffull;
    v = (v | (v >> 16)) & 0x1f00000000ffffull;
    v = (v | (v >> 32)) & 0x1fffffull;
    return (u32)v;
}

// First index in [lo, hi) whose key is >= v (hi when none).
__device__ __forceinline__ u32 lower_key(const u64 *keys, u32 lo, u32 hi, u64 v)
{
    while (lo < hi) {
        u32 mid = lo + ((hi - lo) >> 1);
        if (keys[mid] < v) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// First index in (k, hi] whose key is >= v, keys[k] < v: galloping from k, for
// most cells hold few keys.
__device__ __forceinline__ u32 end_key(const u64 *keys, u32 k, u32 hi, u64 v)
{
    u32 a = k, step = 1;
    while (step < hi - a && keys[a + step] < v) {
        a += step;
        step <<= 1;
    }
    return lower_key(keys, a + 1, step < hi - a ? a + step : hi, v);
}

// First index in [lo, k] whose key is >= v, keys[k] >= v.
__device__ __forceinline__ u32 start_key(const u64 *keys, u32 lo, u32 k, u64 v)
{
    u32 a = k, step = 1;
    while (step <= a - lo && keys[a - step] >= v) {
        a -= step;
        step <<= 1;
    }
    return lower_key(keys, step <= a - lo ? a - step + 1 : lo, a, v);
}

__device__ __forceinline__ int level_shift(int l) { return 3 * (kLevels - l); }

// Cells that start at every key: a cell of level l starts at key k iff k is
// the first key of its level-l prefix and its parent holds more than `leaf`
// keys (then every ancestor does too, so the parent exists and is split); a
// cell of at most `leaf` keys, or of level kLevels, is a leaf.  cnt[k] cells
// of levels lst[k], lst[k] + 1, ... start at k; hist[l] += the cells of level l.
__global__ void __launch_bounds__(256) k_tree_census(const u64 *keys, long long n, int leaf,
                                                     Segs segs, u32 *cnt, unsigned char *lst,
                                                     unsigned long long *hist)
{
    __shared__ unsigned sh[kLevels + 1];
    if (threadIdx.x <= kLevels) sh[threadIdx.x] = 0u;
    __syncthreads();
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < n) {
        const u32 k = (u32)t;
        u32 lo = 0u, hi = (u32)n;
        segs.range(k, lo, hi);
        const u64 key = keys[k];
        int l = 0;
        if (k > lo) {
            const u64 x = keys[k - 1] ^ key;   // keys hold 3 kLevels bits
            const int lcp = x ? (__clzll((long long)x) - (64 - 3 * kLevels)) / 3 : kLevels;
            l = lcp + 1;
            if (l <= kLevels) {   // the level-lcp cell holding keys k - 1 and k
                const int s3 = level_shift(lcp);
                const u64 p = key >> s3;
                const u32 en = end_key(keys, k, hi, (p + 1) << s3);
                if (en - k < (u32)leaf &&   // a leaf: nothing starts here
                    en - start_key(keys, lo, k, p << s3) <= (u32)leaf)
                    l = kLevels + 1;
            }
        }
        lst[k] = (unsigned char)l;
        u32 c = 0, e = hi;
        for (; l <= kLevels; ++l) {
            ++c;
            atomicAdd(&sh[l], 1u);
            if (l > 0) e = end_key(keys, k, e, ((key >> level_shift(l)) + 1) << level_shift(l));
            if (e - k <= (u32)leaf) break;
        }
        cnt[k] = c;
    }
    __syncthreads();
    if (threadIdx.x <= kLevels && sh[threadIdx.x])
        atomicAdd(&hist[threadIdx.x], (unsigned long long)sh[threadIdx.x]);
}

// The records of every cell (pos: exclusive scan of the counts, pos[n] their
// total) and, when lnode is set, the cells grouped by level: level l's from
// the sum of the coarser levels' counts on, in no particular order.
__global__ void __launch_bounds__(256) k_tree_emit(const u64 *keys, long long n, Segs segs,
                                                   const FrameRec *frames, const u32 *pos,
                                                   const unsigned char *lst, float4 *box,
                                                   uint4 *meta, double *cube, int *lev,
                                                   u32 *parent, u32 *leafof, u32 *lnode,
                                                   const unsigned long long *hist, u32 *cursor)
{
    __shared__ u32 sh[kLevels + 1], base[kLevels + 1];
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const u32 k = (u32)t;
    u32 p0 = 0, m = 0;
    int l0 = 0;
    if (t < n) {
        p0 = pos[k];
        m = pos[k + 1] - p0;
        l0 = lst[k];
    }
    if (lnode) {   // this block's places in the level lists
        if (threadIdx.x <= kLevels) sh[threadIdx.x] = 0u;
        __syncthreads();
        for (u32 j = 0; j < m; ++j) atomicAdd(&sh[l0 + j], 1u);
        __syncthreads();
        if (threadIdx.x <= kLevels) {
            u32 off = 0;
            for (int l = 0; l < (int)threadIdx.x; ++l) off += (u32)hist[l];
            base[threadIdx.x] =
                off + (sh[threadIdx.x] ? atomicAdd(&cursor[threadIdx.x], sh[threadIdx.x]) : 0u);
        }
        __syncthreads();
        if (threadIdx.x <= kLevels) sh[threadIdx.x] = 0u;
        __syncthreads();
    }
    if (m == 0) return;
    u32 lo = 0u, hi = (u32)n;
    const u32 b = segs.range(k, lo, hi);
    const FrameRec fr = frames[b];
    const u64 key = keys[k];
    u32 e = hi, par = 0xffffffffu;
    if (l0 > 0) {
        const u32 st = start_key(keys, lo, k, (key >> level_shift(l0 - 1)) << level_shift(l0 - 1));
        par = pos[st] + (u32)(l0 - 1 - lst[st]);
    }
    for (u32 j = 0; j < m; ++j) {
        const int l = l0 + (int)j;
        const u32 i = p0 + j;
        if (l > 0) e = end_key(keys, k, e, ((key >> level_shift(l)) + 1) << level_shift(l));
        const u64 prefix = key >> level_shift(l);   // 0 at the root: keys hold 3 kLevels bits
        const u32 ix = compact3(prefix >> 2), iy = compact3(prefix >> 1), iz = compact3(prefix);
        const double s = ldexp(fr.side, -l);
        const double cx = __dadd_rn(fr.lo[0], __dmul_rn((double)ix, s));
        const double cy = __dadd_rn(fr.lo[1], __dmul_rn((double)iy, s));
        const double cz = __dadd_rn(fr.lo[2], __dmul_rn((double)iz, s));
        double2 *cb = reinterpret_cast<double2 *>(cube + 4 * (size_t)i);
        cb[0] = make_double2(cx, cy);
        cb[1] = make_double2(cz, s);
        box[i] = make_float4(__double2float_rn(cx), __double2float_rn(cy), __double2float_rn(cz),
                             __double2float_rn(s));
        const bool leaf = j + 1 == m;
        meta[i] = make_uint4(pos[e], k, e - k, leaf ? 1u : 0u);
        lev[i] = l;
        parent[i] = j ? i - 1 : par;
        if (leaf)
            for (u32 r = k; r < e; ++r) leafof[r] = i;
        if (lnode) lnode[base[l] + atomicAdd(&sh[l], 1u)] = i;
    }
}

// Issues the census of a tree over n sorted keys and the scan of its counts;
// the counts per level (kLevels + 1) go to hist, which the caller cleared.
int tree_census(start_ctx *c, Tree &t, const u64 *keys, long long n, int leaf, const Segs &segs,
                unsigned long long *hist)
{
    t.n = 0;
    t.lvl_off.clear();
    if (n <= 0) return START_OK;
    if (ensure(t.pos, (n + 1) * sizeof(u32)) || ensure(t.lst, n))
        return set_err(c, START_ENOMEM, "out of device memory (octree)");
    k_tree_census<<<grid_for(n, 256), 256, 0, c->stream>>>(keys, n, leaf, segs, t.pos.as<u32>(),
                                                           t.lst.as<unsigned char>(), hist);
    ++c->launches;
    ST_CUDA(c, cudaGetLastError());
    return exclusive_scan_u32(c, t.pos.as<u32>(), t.pos.as<u32>(), n, t.pos.as<u32>() + n);
}

// Writes the tree's records; hist: the census on the host and on the device,
// cursor: kLevels + 1 cleared counters.  by_level: also group the cells by
// level (tree_moments needs it).
int tree_emit(start_ctx *c, Tree &t, const u64 *keys, long long n, const Segs &segs,
              const FrameRec *frames, const unsigned long long *hist,
              const unsigned long long *hist_dev, u32 *cursor, bool by_level)
{
    if (n <= 0) return START_OK;
    unsigned long long total = 0;
    for (int l = 0; l <= kLevels && hist[l]; ++l) {
        t.lvl_off.push_back((long long)total);
        total += hist[l];
    }
    t.lvl_off.push_back((long long)total);
    if (hist[0] != (unsigned long long)segs.trees || total >= (1ull << 31))
        return set_err(c, START_ECUDA, "octree census");
    if (ensure(t.box, total * sizeof(float4)) || ensure(t.meta, total * sizeof(uint4)) ||
        ensure(t.cube, total * 4 * sizeof(double)) || ensure(t.level, total * sizeof(int)) ||
        ensure(t.parent, total * sizeof(u32)) || ensure(t.leafof, n * sizeof(u32)) ||
        (by_level && ensure(t.lnode, total * sizeof(u32))))
        return set_err(c, START_ENOMEM, "out of device memory (octree)");
    k_tree_emit<<<grid_for(n, 256), 256, 0, c->stream>>>(
        keys, n, segs, frames, t.pos.as<u32>(), t.lst.as<unsigned char>(), t.box.as<float4>(),
        t.meta.as<uint4>(), t.cube.as<double>(), t.level.as<int>(), t.parent.as<u32>(),
        t.leafof.as<u32>(), by_level ? t.lnode.as<u32>() : nullptr, hist_dev, cursor);
    ++c->launches;
    t.n = (long long)total;
    return cuda_check(c, cudaGetLastError(), "k_tree_emit");
}

// ---------------------------------------------------------------- moments
// One cell.  A leaf sums its members in sorted order; an inner cell sums its
// children in octant order (FP64, never contracted): the first child follows
// its parent, each further one its sibling's subtree.
__device__ __forceinline__ void node_moments(u32 i, const uint4 *meta, const float4 *mem_pos,
                                             const double *mem_L, const double *cube,
                                             double L_unit, double *L, double *M, float4 *vsrc)
{
    const uint4 mt = meta[i];
    double S = 0.0, Mx = 0.0, My = 0.0, Mz = 0.0;
    const u32 f = mt.y, n = mt.z;
    if (mt.w) {
        for (u32 r = f; r < f + n; ++r) {
            double Lj = mem_L[r];
            float4 p = mem_pos[r];
            S = __dadd_rn(S, Lj);
            Mx = __dadd_rn(Mx, __dmul_rn(Lj, (double)p.x));
            My = __dadd_rn(My, __dmul_rn(Lj, (double)p.y));
            Mz = __dadd_rn(Mz, __dmul_rn(Lj, (double)p.z));
        }
    } else {
        for (u32 j = i + 1; j < mt.x; j = meta[j].x) {
            S = __dadd_rn(S, L[j]);
            Mx = __dadd_rn(Mx, M[3 * (size_t)j + 0]);
            My = __dadd_rn(My, M[3 * (size_t)j + 1]);
            Mz = __dadd_rn(Mz, M[3 * (size_t)j + 2]);
        }
    }
    L[i] = S;
    M[3 * (size_t)i + 0] = Mx;
    M[3 * (size_t)i + 1] = My;
    M[3 * (size_t)i + 2] = Mz;
    float4 v;
    if (n == 1) {
        float4 p = mem_pos[f];
        v = make_float4(p.x, p.y, p.z, 0.f);
    } else if (S > 0.0) {
        v = make_float4(__double2float_rn(__ddiv_rn(Mx, S)), __double2float_rn(__ddiv_rn(My, S)),
                        __double2float_rn(__ddiv_rn(Mz, S)), 0.f);
    } else {
        double l = cube[4 * (size_t)i + 3];
        v = make_float4(__double2float_rn(__dadd_rn(cube[4 * (size_t)i + 0], __dmul_rn(0.5, l))),
                        __double2float_rn(__dadd_rn(cube[4 * (size_t)i + 1], __dmul_rn(0.5, l))),
                        __double2float_rn(__dadd_rn(cube[4 * (size_t)i + 2], __dmul_rn(0.5, l))),
                        0.f);
    }
    v.w = __double2float_rn(__ddiv_rn(S, L_unit));
    vsrc[i] = v;
}

// One level, deepest first.
__global__ void k_moments_level(const u32 *lnode, long long m, const uint4 *meta,
                                const float4 *mem_pos, const double *mem_L, const double *cube,
                                double L_unit, double *L, double *M, float4 *vsrc)
{
    long long b = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= m) return;
    node_moments(lnode[b], meta, mem_pos, mem_L, cube, L_unit, L, M, vsrc);
}

// All levels of a small tree by one block, deepest first.
struct LevelOffsets {
    u32 off[kLevels + 2];
    int levels;
};

constexpr long long kSmallMoments = 8192;   // cells of a tree that one block sums

__global__ void __launch_bounds__(512) k_moments_small(const u32 *lnode, LevelOffsets lo,
                                                       const uint4 *meta, const float4 *mem_pos,
                                                       const double *mem_L, const double *cube,
                                                       double L_unit, double *L, double *M,
                                                       float4 *vsrc)
{
    for (int l = lo.levels - 1; l >= 0; --l) {
        for (u32 b = lo.off[l] + threadIdx.x; b < lo.off[l + 1]; b += blockDim.x)
            node_moments(lnode[b], meta, mem_pos, mem_L, cube, L_unit, L, M, vsrc);
        __syncthreads();
    }
}

int tree_moments(start_ctx *c, Tree &t, const float4 *mem_pos, const double *mem_L, double L_unit)
{
    if (t.n == 0) return START_OK;
    if (ensure(t.L, t.n * sizeof(double)) || ensure(t.M, t.n * 3 * sizeof(double)) ||
        ensure(t.vsrc, t.n * sizeof(float4)))
        return set_err(c, START_ENOMEM, "out of device memory (moments)");
    const int levels = (int)t.lvl_off.size() - 1;
    if (t.n <= kSmallMoments) {
        LevelOffsets lo{};
        for (int l = 0; l <= levels; ++l) lo.off[l] = (u32)t.lvl_off[l];
        lo.levels = levels;
        k_moments_small<<<1, 512, 0, c->stream>>>(t.lnode.as<u32>(), lo, t.meta.as<uint4>(),
                                                  mem_pos, mem_L, t.cube.as<double>(), L_unit,
                                                  t.L.as<double>(), t.M.as<double>(),
                                                  t.vsrc.as<float4>());
        ++c->launches;
        return cuda_check(c, cudaGetLastError(), "k_moments_small");
    }
    for (int l = levels - 1; l >= 0; --l) {
        const long long o = t.lvl_off[l], m = t.lvl_off[l + 1] - o;
        k_moments_level<<<grid_for(m, 256), 256, 0, c->stream>>>(
            t.lnode.as<u32>() + o, m, t.meta.as<uint4>(), mem_pos, mem_L, t.cube.as<double>(),
            L_unit, t.L.as<double>(), t.M.as<double>(), t.vsrc.as<float4>());
        ++c->launches;
    }
    return cuda_check(c, cudaGetLastError(), "k_moments_level");
}

void tree_release(Tree &t)
{
    DBuf *all[] = {&t.box, &t.meta, &t.cube, &t.level, &t.parent, &t.leafof,
                   &t.vsrc, &t.L, &t.M, &t.pos, &t.lst, &t.lnode};
    for (DBuf *b : all) release(*b);
    t.n = 0;
    t.lvl_off.clear();
}

}  // namespace st
