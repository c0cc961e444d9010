// Tiled forward (hash + gather + sum-pool) and backward scatter kernels.
//
// The forward gives each warp its own tile (see k_forward_warp).  The atomic
// backward scatter gives each CTA a TILE of `tb` consecutive bags of one table
// (bag slots t*B + b0 .. t*B + b0 + tb - 1, so the table id is uniform):
//   stage:  the tile's offsets go to shared memory; then every (id, chunk)
//           pair of the tile is hashed ONCE, by one thread, into a shared
//           array of block buckets x (loc = G*x).  Long tiles are staged in
//           chunks of `qc` ids.
//   gather / scatter: groups of gs lanes own consecutive bags of the tile and
//           walk their ids in order, U ids at a time so that U independent
//           16-byte loads per lane are in flight; a bag's row is stored when
//           its last id has been added (empty bags store zeros).
// Everything is index arithmetic on the CSR batch; no sort, no atomics in the
// forward.  The backward adds each bag's upstream-gradient row into every
// block the bag read (the dense branch of Algorithm 1) with global reductions:
// 16-byte fp32 vector reductions, or one fp64 reduction per element with
// consecutive lanes on consecutive elements (8 sectors per instruction).
#include <climits>
#include <type_traits>

#include "pss_device.cuh"
#include "pss_internal.h"
#include "pss_tiles.h"

namespace pss {
namespace {

constexpr int kU = 4;            // ids in flight per group
// ids in flight per group in the multi-id forward (4 or 8; measured on GB300
// at the multi-hot shape: 8 took 0.398 ms per forward with spills and 0.381
// at 3 CTAs per SM, against 0.334 ms with 4)
constexpr int kUM = 4;
static_assert(kUM == 4, "the multi-id forward sums 4 values per round as a tree");
constexpr int kBagsPerGroup = 16;

template <typename XT>
struct Invalid;
template <>
struct Invalid<uint32_t> {
    static constexpr uint32_t v = 0xffffffffu;
};
template <>
struct Invalid<uint64_t> {
    static constexpr uint64_t v = ~uint64_t(0);
};

struct TileGeom {
    int tb;               // bags per tile
    int qc;               // ids per staging chunk
    int tiles_per_table;  // ceil(B / tb)
};

// Stage the offsets of tile (t, b0) into s_off; returns false (and zeroes the
// tile's rows when `out` is given) if the offsets are malformed.
// s_flags bit 0: malformed offsets; bit 1: some bag holds more than one id.
__device__ __forceinline__ bool stage_offsets(const int64_t* __restrict__ off, int64_t s0, int nb,
                                              int64_t nnz, int64_t* s_off, int* s_flags,
                                              DevError* err, bool* one_hot = nullptr) {
    if (threadIdx.x == 0) *s_flags = 0;
    for (int i = threadIdx.x; i <= nb; i += kThreads) s_off[i] = __ldg(off + s0 + i);
    __syncthreads();
    int f = 0;
    for (int i = threadIdx.x; i < nb; i += kThreads) {
        const int64_t a = s_off[i], c = s_off[i + 1];
        if (a < 0 || c < a || c > nnz) f |= 1;
        if (c - a > 1) f |= 2;
    }
    if (f) atomicOr(s_flags, f);
    __syncthreads();
    const int flags = *s_flags;
    if ((flags & 1) && threadIdx.x == 0) record_bad_offsets(err);
    if (one_hot) *one_hot = (flags & 2) == 0;
    return !(flags & 1);
}

// Hash every (id, chunk) pair of ids [qc0, qc0 + nq) of table t into s_x
// (CTA-cooperative; used by the atomic backward scatter).  With TOUCH every
// distinct bucket is also recorded in the touched bitmap / list, with one
// list-counter atomic per warp.
template <typename XT, bool TOUCH>
__device__ __forceinline__ void stage_buckets(const DevParams& p, const int64_t* __restrict__ idx,
                                              int t, uint64_t card, int64_t qc0, int nq, XT* s_x,
                                              DevError* err, const Touched& tc) {
    const int npairs = nq * p.J;
    const int lane = threadIdx.x & 31;
    for (int base = threadIdx.x & ~31; base < npairs; base += kThreads) {   // warp-uniform
        const int k = base + lane;
        XT x = Invalid<XT>::v;
        if (k < npairs) {
            const int qi = k / p.J;
            const int j = k - qi * p.J;
            const int64_t q = qc0 + qi;
            const int64_t id = __ldg(idx + q);
            if ((uint64_t)id < card) {
                const uint64_t key = hash_key(p, (uint64_t)id, t, j);
                x = (XT)hash_bucket(p, key) | (XT)hash_sign_bit(p, key);
            } else if (j == 0) {
                record_bad_id(err, q);
            }
            s_x[k] = x;
        }
        if (TOUCH)
            mark_touched_warp(tc, (uint64_t)(x & ~(XT)p.smask), x != Invalid<XT>::v, lane);
    }
}

// One VW-wide load of the block of a staged bucket x; wz points at the column
// in the array's first block, Gb is the bytes between block starts (below 2^32
// with 32-bit buckets: one multiply-add).  With signed hashing (SG) the bucket
// carries the sign in bit 31, applied to the value.
template <bool SG, typename V, typename XT>
__device__ __forceinline__ typename V::T gather(const float* __restrict__ wz, uint64_t Gb, XT x) {
    const XT xb = SG ? (x & ~(XT)0x80000000u) : x;
    const uint64_t off = (sizeof(XT) == 4) ? (uint64_t)(uint32_t)Gb * (uint32_t)xb
                                           : Gb * (uint64_t)xb;
    const auto v = V::ldg(reinterpret_cast<const float*>(reinterpret_cast<const char*>(wz) + off));
    return SG ? sign_by(v, (uint32_t)x & 0x80000000u) : v;
}

// ---------------------------------------------------------------------------
// Forward.  Each WARP owns a tile of `wb` consecutive bags of one table and
// stages it in its own slice of shared memory, so warps never wait for each
// other (no CTA-wide barrier): the lanes hash the tile's (id, chunk) pairs
// 32 at a time, then the lane groups gather and sum-pool their bags.
constexpr int kIdU = 4;           // ids in flight per lane while a window is hashed


// Variants of the forward (MODE): rows in flight per lane group in one-id
// tiles, and CTAs per SM.  Measured on GB300, us per forward with the kernel
// compiled for 3, 2 and 4 CTAs per SM (and 4, 16 and 4 rows in flight):
//                                 3      2      4
//   Criteo-TB shape, B = 65536  154    152    199
//   M = 2^26, B = 16384          63     57     99
//   Criteo-TB shape, B = 2048   9.4   10.0   10.3
//   multi-hot, 20 ids per bag   261    288    247
//   multi-hot, 5 ids per bag    148    ---    138
// HBM takes the rows of few warps that write many at a time best; long bags
// want warps.
constexpr int kFwdShort = 0;   // one-id bags
constexpr int kFwdMany = 1;    // many one-id bags, rows of a whole warp
constexpr int kFwdLong = 2;    // bags of several ids
constexpr int fwd_rows(int mode) { return mode == kFwdMany ? 16 : 4; }
constexpr int fwd_min_ctas(int VW, int KC, int mode) {
    return KC * VW > 4 ? (KC * VW <= 8 ? 2 : 1)
                       : mode == kFwdMany ? 2 : mode == kFwdLong && KC == 1 ? 4 : 3;
}

// Bucket of a pair from its hash s = (A*key + B0) mod P: s mod R, the same
// integers as hash_bucket.  For R <= 2^30, q is floor(s / R) or up to 3 less:
// Barrett's quotient loses 1 (see hash_bucket) and the three dropped parts of
// the 64 x 64-bit product lose less than 1 each; so s - q*R < 4R <= 2^32 and
// 32-bit arithmetic modulo 2^32 gives it.
template <typename XT>
__device__ __forceinline__ XT mod_R(const DevParams& p, uint64_t s) {
    if (sizeof(XT) == 4 && p.R <= (uint64_t(1) << 30)) {
        const uint32_t sh = (uint32_t)(s >> 32), sl = (uint32_t)s;
        const uint32_t rh = (uint32_t)(p.Rinv >> 32), rl = (uint32_t)p.Rinv;
        const uint32_t R = (uint32_t)p.R;
        const uint32_t q = sh * rh + __umulhi(sh, rl) + __umulhi(sl, rh);
        uint32_t r = sl - q * R;
        r = min(r, r - 2u * R);   // (wraps above r when r is the smaller)
        return (XT)min(r, r - R);
    }
    const uint64_t q = __umul64hi(s, p.Rinv);
    const uint64_t R = sizeof(XT) == 4 ? (uint64_t)(uint32_t)p.R : p.R;
    const uint64_t r = s - q * R;
    return (XT)(r >= R ? r - R : r);
}

// a + b mod P for a, b < P
__device__ __forceinline__ uint64_t add_p61(uint64_t a, uint64_t b) {
    const uint64_t s = a + b;
    return s >= kP61 ? s - kP61 : s;
}

// Two fp32 operations per instruction (each rounded as the scalar one).
__device__ __forceinline__ uint64_t pack2(float a, float b) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& a, float& b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b) {   // a - b = fma(b, -1, a)
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(b), "l"(0xbf800000bf800000ull), "l"(a));
    return r;
}

// Compensated sums of VW-wide columns: add(v) is kahan_add per element,
// add4 the tree sum of four values first; merge adds another lane's sum, and its
// compensation the same way (added plainly, 32 groups' sums were off by 2% more:
// rms 5.3e-8 against 5.2e-8).
template <int VW>
struct Sum;
template <>
struct Sum<4> {
    uint64_t s0 = 0, s1 = 0, c0 = 0, c1 = 0;
    static __device__ __forceinline__ void kahan(uint64_t& s, uint64_t& c, uint64_t x) {
        const uint64_t y = sub2(x, c);
        const uint64_t t = add2(s, y);
        c = sub2(sub2(t, s), y);
        s = t;
    }
    __device__ __forceinline__ void add4(const float4& a, const float4& b, const float4& c,
                                         const float4& d) {
        kahan(s0, c0, add2(add2(pack2(a.x, a.y), pack2(b.x, b.y)),
                           add2(pack2(c.x, c.y), pack2(d.x, d.y))));
        kahan(s1, c1, add2(add2(pack2(a.z, a.w), pack2(b.z, b.w)),
                           add2(pack2(c.z, c.w), pack2(d.z, d.w))));
    }
    __device__ __forceinline__ void merge(int o) {
        const uint64_t t0 = __shfl_xor_sync(0xffffffffu, s0, o);
        const uint64_t t1 = __shfl_xor_sync(0xffffffffu, s1, o);
        const uint64_t d0 = __shfl_xor_sync(0xffffffffu, c0, o);
        const uint64_t d1 = __shfl_xor_sync(0xffffffffu, c1, o);
        constexpr uint64_t kNeg = 0x8000000080000000ull;
        kahan(s0, c0, t0);
        kahan(s1, c1, t1);
        kahan(s0, c0, d0 ^ kNeg);
        kahan(s1, c1, d1 ^ kNeg);
    }
    __device__ __forceinline__ float4 value() const {
        float4 v;
        unpack2(sub2(s0, c0), v.x, v.y);
        unpack2(sub2(s1, c1), v.z, v.w);
        return v;
    }
};
template <>
struct Sum<1> {
    float s = 0.f, c = 0.f;
    __device__ __forceinline__ void add4(float a, float b, float x, float y) {
        kahan_add(s, c, (a + b) + (x + y));
    }
    __device__ __forceinline__ void merge(int o) {
        const float os = __shfl_xor_sync(0xffffffffu, s, o);
        const float oc = __shfl_xor_sync(0xffffffffu, c, o);
        kahan_add(s, c, os);
        kahan_add(s, c, -oc);
    }
    __device__ __forceinline__ float value() const { return s - c; }
};

// How a forward's work is cut.  One-id bags: tiles of wb consecutive bags of
// one table; 2^log2pw >= wb lanes own one bag each (32 >> log2pw lanes per
// bag).  Longer bags: 2^log2pi ids are hashed at a time, 32 >> log2pi lanes
// each.  stepA[k] and stepA2[k] are A and A2 times the lanes per bag (k = 0)
// or id (1), mod P.
struct FwdGeom {
    int wb, log2pw, log2pi, tiles_per_table;
    bool by_table;        // tiles in the order of the tables, else of the bags
    uint64_t stepA[2], stepA2[2];
    uint64_t TJ;          // T * J: keys of consecutive ids
    uint64_t Gb;          // bytes between block starts
};

// Buckets of chunks j0, j0 + lpi, ... of one id into sx[0 .. J), Invalid for a
// bad id: one product A*key per lane, chunk j + lpi has step = A*lpi more.
template <typename XT, bool SG>
__device__ __forceinline__ void hash_id(const DevParams& p, uint64_t TJ, uint64_t id, uint64_t tJ,
                                        bool valid, int j0, int lpi, uint64_t step, uint64_t step2,
                                        XT* sx) {
    const uint64_t key = id * TJ + tJ + (uint32_t)j0;   // hash_key; tJ = t*J
    uint64_t s = affine_mod_p61(p.A, key, p.B0);
    uint64_t s2 = SG ? affine_mod_p61(p.A2, key, p.B2) : 0ull;
    for (int j = j0; j < p.J; j += lpi) {
        XT x = mod_R<XT>(p, s);
        s = add_p61(s, step);
        if (SG) {
            x |= (XT)((uint32_t)(s2 & 1u) << 31);
            s2 = add_p61(s2, step2);
        }
        sx[j] = valid ? x : Invalid<XT>::v;
    }
}

// n staged buckets to pair_x + at, whose ids are consecutive.
template <typename XT>
__device__ __forceinline__ void emit_pairs(const XT* s_x, int n, int J, uint32_t* __restrict__ px,
                                           int lane) {
    if (sizeof(XT) == 4 && (J & 3) == 0) {
        for (int k = lane; k < n / 4; k += 32)
            reinterpret_cast<uint4*>(px)[k] = reinterpret_cast<const uint4*>(s_x)[k];
    } else if (sizeof(XT) == 4 && (J & 1) == 0) {
        for (int k = lane; k < n / 2; k += 32)
            reinterpret_cast<uint2*>(px)[k] = reinterpret_cast<const uint2*>(s_x)[k];
    } else {
        for (int k = lane; k < n; k += 32) px[k] = (uint32_t)s_x[k];
    }
}

// Bags of any length: pools the nb bags of a tile, lane l holding the offsets
// [q0, q1) of bag l (mod the power of two at or above the tile's bags), all
// ids within [qa, qb).  The ids are staged and hashed in windows.  Bags of
// similar length that lie inside a window go one to a lane group, ng at a
// time.  Other bags take the whole warp, one at a time: its ng lane groups add
// ng consecutive ids of the bag in parallel, kUM steps per round.  A round's kUM values are summed
// as a tree and added with compensation; at the end of the bag the groups'
// sums are merged the same way and group 0 stores the row.
// (One bag per lane group, GROUPS, needs no merge and fewer partly filled
// rounds: 234 us per multi-hot forward against 244 with the whole warp on
// every bag.  The variants for one-id bags leave it out: its registers cost
// them 10-40%.)
// What bounds it: instruction issue, then the L2 gathers.  So whole rounds of
// valid ids run without tests, the sums take two elements per instruction, an
// id's chunks are hashed from one product, and a bag's bounds in the window
// are 32-bit numbers that the lanes compute together.
template <int VW, int KC, typename XT, bool SG, bool GROUPS>
__device__ __forceinline__ void
forward_bags(const DevParams& p, const FwdGeom& fg, const int64_t* __restrict__ idx, uint64_t tJ,
             uint64_t card, int64_t q0, int64_t q1, int nb, XT* s_x,
             const float* const (&wz)[KC], const Cols<VW, KC>& col, float* orow, int64_t ostride,
             uint32_t row, DevError* err, uint32_t* __restrict__ pair_x,
             uint32_t* __restrict__ q_row, int log2gs, int lane) {
    using V = Vec<VW>;
    using VT = typename V::T;
    const int gs = 1 << log2gs;
    const int g = lane >> log2gs;
    const int ng = 32 >> log2gs;
    const int J = p.J;
    const int sJ = ng * J;                   // staged buckets from one of a lane's ids to the next
    const int gJ = g * J;
    const int qcw = kWarpPairs / J;          // ids per staged window
    const int ids = 1 << fg.log2pi, lpi = 32 >> fg.log2pi;
    const int64_t qb = __shfl_sync(0xffffffffu, q1, nb - 1);
    int64_t sw0 = __shfl_sync(0xffffffffu, q0, 0);
    int bi = 0;
    bool begun = false;              // bag bi has ids in an earlier window
    Sum<VW> acc[KC];
    for (;;) {
        // stage the window [sw0, sw0 + n)
        const int n = (int)((qb - sw0) < qcw ? (qb - sw0) : qcw);
        bool ok = true;
        for (int i0 = lane & (ids - 1); i0 < n; i0 += ids * kIdU) {
            int64_t id[kIdU];   // loads in flight together
#pragma unroll
            for (int u = 0; u < kIdU; ++u)
                id[u] = i0 + u * ids < n ? __ldg(idx + sw0 + i0 + u * ids) : 0;
#pragma unroll
            for (int u = 0; u < kIdU; ++u) {
                const int i = i0 + u * ids;
                if (i >= n) break;
                const bool valid = (uint64_t)id[u] < card;
                ok &= valid;
                if (!valid && lane < ids) record_bad_id(err, sw0 + i);
                hash_id<XT, SG>(p, fg.TJ, (uint64_t)id[u], tJ, valid, lane >> fg.log2pi, lpi,
                                fg.stepA[1], fg.stepA2[1], s_x + i * J);
            }
        }
        const bool clean = __all_sync(0xffffffffu, ok);   // every id valid
        __syncwarp();
        if (pair_x) emit_pairs<XT>(s_x, n * J, J, pair_x + sw0 * J, lane);
        // this lane's bag inside the window, and whether it ends there
        const int64_t a = q0 - sw0, c = q1 - sw0;
        const int lo = (int)(a < 0 ? 0 : a < n ? a : n), hi = (int)(c < n ? c : n);
        const unsigned ends = __ballot_sync(0xffffffffu, c <= n);
        while (bi < nb) {
            if (GROUPS && ng > 1 && clean && bi + ng <= nb && ((ends >> (bi + ng - 1)) & 1u)) {
                // ng bags that end in this window, the first not begun before
                // it: one per lane group, unless one is much longer than the rest
                const int b0 = __shfl_sync(0xffffffffu, lo, bi + g);
                const int m = __shfl_sync(0xffffffffu, hi, bi + g) - b0;
                int mx = m, mn = m, sum = m;
                for (int o = gs; o < 32; o <<= 1) {
                    mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
                    mn = min(mn, __shfl_xor_sync(0xffffffffu, mn, o));
                    sum += __shfl_xor_sync(0xffffffffu, sum, o);
                }
                if (!begun && mx * ng <= 2 * sum + 8 * ng) {
                    if (q_row)
                        for (int i = lane & (gs - 1); i < m; i += gs)
                            q_row[sw0 + b0 + i] = row + (uint32_t)g * (uint32_t)p.T;
                    Sum<VW> ga[KC];
                    const XT* sx = s_x + b0 * J;
                    int left = mn;
                    for (; left >= kUM; left -= kUM) {   // rounds that every bag fills
                        VT v[kUM][KC];
#pragma unroll
                        for (int u = 0; u < kUM; ++u)
#pragma unroll
                            for (int k = 0; k < KC; ++k)
                                v[u][k] = gather<SG, V>(wz[k], fg.Gb, sx[u * J + col.js[k]]);
                        sx += kUM * J;
#pragma unroll
                        for (int k = 0; k < KC; ++k) ga[k].add4(v[0][k], v[1][k], v[2][k], v[3][k]);
                    }
                    // the rest: groups past their bag load the window's first id
                    // and drop it
                    const int done = mn - left;
                    for (int i = done; i < mx; i += kUM) {
                        VT v[kUM][KC];
#pragma unroll
                        for (int u = 0; u < kUM; ++u) {
                            const bool in = i + u < m;
                            const XT* su = in ? sx + u * J : s_x;
#pragma unroll
                            for (int k = 0; k < KC; ++k) {
                                v[u][k] = gather<SG, V>(wz[k], fg.Gb, su[col.js[k]]);
#pragma unroll
                                for (int c = 0; c < VW; ++c)
                                    V::set(v[u][k], c, in ? V::get(v[u][k], c) : 0.f);
                            }
                        }
                        sx += kUM * J;
#pragma unroll
                        for (int k = 0; k < KC; ++k) ga[k].add4(v[0][k], v[1][k], v[2][k], v[3][k]);
                    }
                    float* og = orow + g * ostride;
#pragma unroll
                    for (int k = 0; k < KC; ++k)
                        if (col.v[k]) V::stcs(og + col.e[k], ga[k].value());
                    orow += ng * ostride;
                    row += (uint32_t)(ng * p.T);
                    bi += ng;
                    continue;
                }
            }
            const int b0 = __shfl_sync(0xffffffffu, lo, bi), b1 = __shfl_sync(0xffffffffu, hi, bi);
            if (q_row)   // the bag's ids' output row, one store per lane
                for (int i = b0 + lane; i < b1; i += 32) q_row[sw0 + i] = row;
            const XT* sx = s_x + b0 * J;
            int left = b1 - b0;   // ids to add
            if (clean) {
                // whole rounds: every group has kUM ids
                for (; left >= kUM * ng; left -= kUM * ng) {
                    VT v[kUM][KC];
#pragma unroll
                    for (int u = 0; u < kUM; ++u)
#pragma unroll
                        for (int k = 0; k < KC; ++k)
                            v[u][k] = gather<SG, V>(wz[k], fg.Gb, sx[gJ + u * sJ + col.js[k]]);
                    sx += kUM * sJ;
#pragma unroll
                    for (int k = 0; k < KC; ++k) acc[k].add4(v[0][k], v[1][k], v[2][k], v[3][k]);
                }
                // the rest: lanes past the bag load its next id and drop it
                if (left > 0) {
                    VT v[kUM][KC];
#pragma unroll
                    for (int u = 0; u < kUM; ++u) {
                        const bool in = g + u * ng < left;
                        const int o = in ? gJ + u * sJ : 0;
#pragma unroll
                        for (int k = 0; k < KC; ++k) {
                            v[u][k] = gather<SG, V>(wz[k], fg.Gb, sx[o + col.js[k]]);
#pragma unroll
                            for (int i = 0; i < VW; ++i)
                                V::set(v[u][k], i, in ? V::get(v[u][k], i) : 0.f);
                        }
                    }
#pragma unroll
                    for (int k = 0; k < KC; ++k) acc[k].add4(v[0][k], v[1][k], v[2][k], v[3][k]);
                }
            } else {
                for (int i0 = g; i0 - g < left; i0 += kUM * ng) {
                    VT v[kUM][KC];
#pragma unroll
                    for (int u = 0; u < kUM; ++u)
#pragma unroll
                        for (int k = 0; k < KC; ++k) {
#pragma unroll
                            for (int i = 0; i < VW; ++i) V::set(v[u][k], i, 0.f);
                            if (i0 + u * ng < left) {
                                const XT x = sx[(i0 + u * ng) * J + col.js[k]];
                                if (x != Invalid<XT>::v) v[u][k] = gather<SG, V>(wz[k], fg.Gb, x);
                            }
                        }
#pragma unroll
                    for (int k = 0; k < KC; ++k) acc[k].add4(v[0][k], v[1][k], v[2][k], v[3][k]);
                }
            }
            begun = !((ends >> bi) & 1u);
            if (begun) break;   // it goes on in the next window
            for (int o = gs; o < 32; o <<= 1)
#pragma unroll
                for (int k = 0; k < KC; ++k) acc[k].merge(o);
            if (g == 0) {
#pragma unroll
                for (int k = 0; k < KC; ++k)
                    if (col.v[k]) V::stcs(orow + col.e[k], acc[k].value());
            }
            orow += ostride;
            row += (uint32_t)p.T;
#pragma unroll
            for (int k = 0; k < KC; ++k) acc[k] = Sum<VW>();
            ++bi;
        }
        if (bi >= nb) break;
        sw0 += n;
        __syncwarp();   // s_x is staged again
    }
}

// The two cases in which an id has no pair, whose buckets become Invalid.  Both
// are rare and kept out of the forward's code: inlined, they cost the one-id
// variant 3 us of 155 (Criteo-TB shape).
// (1) Ids before the first bag and after the last: a and b are the batch's first
// and last offset, and one warp of every CTA calls this.
__device__ __noinline__ void drop_unused(int64_t a, int64_t b, int64_t nnz, int J,
                                         uint32_t* __restrict__ pair_x, int lane) {
    // (malformed offsets are any 64-bit numbers: into [0, nnz] before a product)
    const int64_t head = (a < 0 ? 0 : a < nnz ? a : nnz) * J;
    const int64_t tail = (b < 0 ? 0 : b < nnz ? b : nnz) * J;
    const int64_t stride = (int64_t)gridDim.x * 32, k0 = (int64_t)blockIdx.x * 32 + lane;
    for (int64_t k = k0; k < head; k += stride) pair_x[k] = Invalid<uint32_t>::v;
    for (int64_t k = tail + k0; k < nnz * J; k += stride) pair_x[k] = Invalid<uint32_t>::v;
}
// (2) The ids [qa, qb) of a tile with malformed offsets, as far as those tell
// them (the sorts check the bounds of what else malformed offsets leave; ranges
// that may enclose the whole batch, for every such tile, are left).
__device__ __noinline__ void drop_tile(int64_t qa, int64_t qb, int64_t nnz, int J,
                                       uint32_t* __restrict__ pair_x, int lane) {
    constexpr int64_t kMost = 1 << 16;   // pairs
    if (qa < 0 || qb < qa || qb > nnz || (qb - qa) * J > kMost) return;
    for (int64_t k = qa * J + lane; k < qb * J; k += 32) pair_x[k] = Invalid<uint32_t>::v;
}

// What bounds it with one-id bags: the pooled rows' stores to HBM at d = 128
// (one 16-byte load and store per lane and row), and the latency of the chain
// offsets -> ids -> hash -> blocks behind them.  So a warp loads the offsets
// of the tile after next and the ids of the next tile before it gathers its
// own, and in tiles whose bags all hold one valid id a row costs one
// shared-memory load, one multiply-add, one load and one store.  Tiles run
// over the tables of a range of bags first, so that the rows that the GPU
// writes at a time are one contiguous piece of the output (large arrays: over
// the bags of a table first, see kByTableMinM).
template <int VW, int KC, typename XT, bool SG, int MODE>
__global__ void __launch_bounds__(kThreads, fwd_min_ctas(VW, KC, MODE))
k_forward_warp(const __grid_constant__ DevParams p, const int64_t* __restrict__ idx, int64_t nnz,
               const int64_t* __restrict__ off, int64_t B, const float* __restrict__ w,
               float* __restrict__ out, DevError* err, uint32_t* __restrict__ pair_x,
               uint32_t* __restrict__ q_row, int log2gs, const __grid_constant__ FwdGeom fg,
               int64_t b_lo, int64_t b_hi) {
    pdl_prologue();
    using V = Vec<VW>;
    using VT = typename V::T;
    extern __shared__ __align__(16) unsigned char smem[];
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    XT* s_x = reinterpret_cast<XT*>(smem) + warp * kWarpPairs;
    const int gs = 1 << log2gs;
    const int lg = lane & (gs - 1);
    const int g = lane >> log2gs;
    const int wb = fg.wb;
    const int bpg = wb >> (5 - log2gs);      // bags per group
    const Cols<VW, KC> col(p, lg, gs);
    const float* wz[KC];
#pragma unroll
    for (int k = 0; k < KC; ++k) wz[k] = w + col.zs[k];
    const int J = p.J;
    const int64_t ostride = (int64_t)p.T * p.d;
    const int bag = lane & ((1 << fg.log2pw) - 1);   // this lane's bag of the tile
    const int j0 = lane >> fg.log2pw;                // its first chunk
    const int lpb = 32 >> fg.log2pw;                 // lanes per bag

    // tiles of this warp, and the place of the lane's bag in the offsets
    const TileWalk walk(gridDim.x * kWarps, (uint32_t)p.T, (uint32_t)fg.tiles_per_table, B, wb,
                        fg.by_table);
    uint32_t t, r;
    walk.first(blockIdx.x * kWarps + warp, t, r);
    if (!walk.inside(t, r)) return;
    const int64_t* po = off + (int64_t)t * B + b_lo + (int64_t)r * wb + bag;
    const int64_t nbags = b_hi - b_lo;
    // offsets of this lane's bag of tile (tt, rr) at po: a zero-length bag past the end
    auto load_offsets = [&](uint32_t tt, uint32_t rr, int64_t& q0, int64_t& q1) {
        q0 = q1 = 0;
        if (bag < wb && tt < walk.T && (int64_t)rr * wb + bag < nbags) {
            q0 = __ldg(po);
            q1 = __ldg(po + 1);
        }
    };
    // the id of a bag that holds exactly one (offsets in range), else -1
    auto load_id = [&](int64_t q0, int64_t q1) -> int64_t {
        return (q0 >= 0 && q0 < nnz && q1 == q0 + 1) ? __ldg(idx + q0) : -1;
    };

    int64_t q0, q1, q0n, q1n;
    load_offsets(t, r, q0, q1);
    uint32_t t1 = t, r1 = r;
    po += walk.advance(t1, r1);
    load_offsets(t1, r1, q0n, q1n);
    if (pair_x && warp == 0 && b_lo == 0) {   // (these loads arrive with the tile's offsets)
        const int64_t a = __ldg(off), b = __ldg(off + (int64_t)p.T * B);
        if (a > 0 || b < nnz) drop_unused(a, b, nnz, J, pair_x, lane);
    }
    int64_t id = load_id(q0, q1);
    while (walk.inside(t, r)) {
        uint32_t t2 = t1, r2 = r1;
        po += walk.advance(t2, r2);
        const int64_t idn = load_id(q0n, q1n);
        int64_t q0m, q1m;
        load_offsets(t2, r2, q0m, q1m);

        const int64_t b0 = b_lo + (int64_t)r * wb;
        const int nb = (int)((b_hi - b0) < wb ? (b_hi - b0) : wb);
        float* obase = out + b0 * ostride + (int64_t)t * p.d;
        const uint32_t row0 = (uint32_t)b0 * (uint32_t)p.T + t;
        const uint64_t tJ = (uint64_t)t * (uint32_t)J;
        const uint64_t card = (uint64_t)__ldg(p.cards + t);
        const bool has = q1 > q0;
        const unsigned odd = __ballot_sync(0xffffffffu, q0 < 0 || q1 < q0 || q1 > nnz);
        const bool multi = __any_sync(0xffffffffu, q1 - q0 > 1) || nb * J > kWarpPairs;
        if (odd | (unsigned)multi) {
            if (odd) {
                if (lane == 0) record_bad_offsets(err);
                for (int bi = g; bi < nb; bi += 32 >> log2gs)
#pragma unroll
                    for (int k = 0; k < KC; ++k) {
                        if (!col.v[k]) continue;
                        VT z;
#pragma unroll
                        for (int i = 0; i < VW; ++i) V::set(z, i, 0.f);
                        V::stcs(obase + bi * ostride + col.e[k], z);
                    }
                if (pair_x)
                    drop_tile(__shfl_sync(0xffffffffu, q0, 0), __shfl_sync(0xffffffffu, q1, nb - 1),
                              nnz, J, pair_x, lane);
            } else {
                forward_bags<VW, KC, XT, SG, MODE == kFwdLong>(
                    p, fg, idx, tJ, card, q0, q1, nb, s_x, wz, col, obase, ostride, row0, err,
                    pair_x, q_row, log2gs, lane);
            }
        } else {
            // every bag holds at most one id: s_x[bag*J + j] is the bucket of
            // chunk j of the bag's id (Invalid for an empty bag or a bad id),
            // one load per bag, no accumulation
            const bool mine = bag < nb;
            const bool valid = has && (uint64_t)id < card;
            if (mine)
                hash_id<XT, SG>(p, fg.TJ, (uint64_t)id, tJ, valid, j0, lpb, fg.stepA[0],
                                fg.stepA2[0], s_x + bag * J);
            if (has && j0 == 0) {
                if (!valid) record_bad_id(err, q0);
                if (q_row) q_row[q0] = row0 + (uint32_t)bag * (uint32_t)p.T;
            }
            __syncwarp();
            if (pair_x) {
                // the bags' ids are consecutive; empty bags have no pair
                if (__all_sync(0xffffffffu, has || !mine)) {
                    emit_pairs<XT>(s_x, nb * J, J,
                                   pair_x + __shfl_sync(0xffffffffu, q0, 0) * J, lane);
                } else if (has) {
                    for (int j = j0; j < J; j += lpb)
                        pair_x[q0 * J + j] = (uint32_t)s_x[bag * J + j];
                }
            }
            const int gb0 = min(g * bpg, nb);
            float* orow = obase + gb0 * ostride;
            const XT* sx = s_x + gb0 * J;
            int n = min(bpg, nb - gb0);
            if (nb == wb && __all_sync(0xffffffffu, valid || !mine)) {
                // whole tile, all ids valid: no tests in the rows' loops
                auto rows = [&](auto nu) {
                    constexpr int U = decltype(nu)::value;
                    VT v[U][KC];
#pragma unroll
                    for (int u = 0; u < U; ++u) {
#pragma unroll
                        for (int k = 0; k < KC; ++k)
                            v[u][k] = gather<SG, V>(wz[k], fg.Gb, sx[col.js[k]]);
                        sx += J;
                    }
#pragma unroll
                    for (int u = 0; u < U; ++u) {
#pragma unroll
                        for (int k = 0; k < KC; ++k)
                            if (col.v[k]) V::stcs(orow + col.e[k], v[u][k]);
                        orow += ostride;
                    }
                    n -= U;
                };
                constexpr int kRows = fwd_rows(MODE);
                if (kRows > 4)
                    while (n >= kRows) rows(std::integral_constant<int, kRows>());
                while (n >= 4) rows(std::integral_constant<int, 4>());
            }
            constexpr int kU4 = 4;
            for (; __any_sync(0xffffffffu, n > 0); n -= kU4) {
                VT v[kU4][KC];
#pragma unroll
                for (int u = 0; u < kU4; ++u)
#pragma unroll
                    for (int k = 0; k < KC; ++k) {
#pragma unroll
                        for (int i = 0; i < VW; ++i) V::set(v[u][k], i, 0.f);
                        if (u < n && col.v[k]) {
                            const XT x = sx[u * J + col.j[k]];
                            if (x != Invalid<XT>::v) v[u][k] = gather<SG, V>(wz[k], fg.Gb, x);
                        }
                    }
#pragma unroll
                for (int u = 0; u < kU4; ++u)
#pragma unroll
                    for (int k = 0; k < KC; ++k)
                        if (u < n && col.v[k]) V::stcs(orow + u * ostride + col.e[k], v[u][k]);
                sx += kU4 * J;
                orow += kU4 * ostride;
            }
        }
        __syncwarp();   // s_x is reused by the next tile
        t = t1;
        r = r1;
        t1 = t2;
        r1 = r2;
        q0 = q0n;
        q1 = q1n;
        id = idn;
        q0n = q0m;
        q1n = q1m;
    }
}

// ---------------------------------------------------------------------------
// Backward scatter: target[G*x + z] += scale * grad_out row chunk.
template <int VW, int KC, typename XT, typename AT, bool TOUCH>
__global__ void __launch_bounds__(kThreads)
k_scatter_tiled(DevParams p, const int64_t* __restrict__ idx, int64_t nnz,
                const int64_t* __restrict__ off, int64_t B, const float* __restrict__ gout,
                float scale, AT* __restrict__ target, Touched tc, DevError* err, int log2gs,
                TileGeom tg) {
    pdl_prologue();
    using V = Vec<VW>;
    using VT = typename V::T;
    extern __shared__ __align__(16) unsigned char smem[];
    int64_t* s_off = reinterpret_cast<int64_t*>(smem);
    XT* s_x = reinterpret_cast<XT*>(s_off + tg.tb + 1);
    __shared__ int s_bad;

    const int lane = threadIdx.x & 31;
    const int gs = 1 << log2gs;
    const int lg = lane & (gs - 1);
    const int grp = (threadIdx.x >> 5) * (32 >> log2gs) + (lane >> log2gs);
    const Cols<VW, KC> col(p, lg, gs);
    const uint64_t G = (uint64_t)p.G;
    const int J = p.J;
    const int64_t ntiles = (int64_t)p.T * tg.tiles_per_table;

    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int t = (int)(tile / tg.tiles_per_table);
        const int64_t b0 = (tile - (int64_t)t * tg.tiles_per_table) * tg.tb;
        const int nb = (int)((B - b0) < tg.tb ? (B - b0) : tg.tb);
        const int64_t s0 = (int64_t)t * B + b0;
        const int gb0 = min(grp * kBagsPerGroup, nb);
        const int gb1 = min(gb0 + kBagsPerGroup, nb);
        const float* gbase = gout + ((b0 * p.T) + t) * (int64_t)p.d;
        const int64_t gstride = (int64_t)p.T * p.d;

        if (!stage_offsets(off, s0, nb, nnz, s_off, &s_bad, err)) {
            __syncthreads();
            continue;
        }
        const uint64_t card = (uint64_t)__ldg(p.cards + t);
        const int64_t qa = s_off[0], qb = s_off[nb];
        const int64_t gq0 = s_off[gb0], gq1 = s_off[gb1];
        int bi = gb0;                       // bag of the next id
        int64_t qend = (gb0 < gb1) ? s_off[gb0 + 1] : 0;
        int have = -1;                      // bag whose row is in `row`
        VT row[KC];

        for (int64_t qc0 = qa; qc0 < qb; qc0 += tg.qc) {
            const int nq = (int)((qb - qc0) < tg.qc ? (qb - qc0) : tg.qc);
            stage_buckets<XT, TOUCH>(p, idx, t, card, qc0, nq, s_x, err, tc);
            __syncthreads();
            const int64_t qlo = gq0 > qc0 ? gq0 : qc0;
            const int64_t qhi = gq1 < qc0 + nq ? gq1 : qc0 + nq;
            for (int64_t q = qlo; q < qhi; q += kU) {
                // bags of the next kU ids, and their rows (independent loads)
                int ub[kU];
                VT r[kU][KC];
#pragma unroll
                for (int u = 0; u < kU; ++u) {
                    ub[u] = -1;
                    if (q + u < qhi) {
                        while (q + u >= qend) {
                            ++bi;
                            qend = s_off[bi + 1];
                        }
                        ub[u] = bi;
                    }
                }
#pragma unroll
                for (int u = 0; u < kU; ++u) {
                    if (ub[u] < 0) continue;
                    const bool same_prev = (u > 0) ? (ub[u] == ub[u - 1]) : (ub[u] == have);
                    if (same_prev) continue;
#pragma unroll
                    for (int k = 0; k < KC; ++k)
                        if (col.v[k])
                            r[u][k] = V::scale(V::ldcs(gbase + ub[u] * gstride + col.e[k]), scale);
                }
#pragma unroll
                for (int u = 0; u < kU; ++u) {
                    if (ub[u] < 0) break;
                    const bool same_prev = (u > 0) ? (ub[u] == ub[u - 1]) : (ub[u] == have);
                    if (!same_prev) {
#pragma unroll
                        for (int k = 0; k < KC; ++k) row[k] = r[u][k];
                        have = ub[u];
                    }
#pragma unroll
                    for (int k = 0; k < KC; ++k) {
                        if (!col.v[k]) continue;
                        const XT x = s_x[(int)(q + u - qc0) * J + col.j[k]];
                        if (x != Invalid<XT>::v)
                            Acc<VW, AT>::red(target + G * (uint64_t)(x & ~(XT)p.smask) + col.z[k],
                                             sign_by(row[k], (uint32_t)x & p.smask));
                    }
                }
            }
            __syncthreads();
        }
        __syncthreads();
    }
}

constexpr int kStageBytes = 16384;   // staged buckets of the scatter

TileGeom tile_geom(const DevParams& p, const RowLayout& lay, int64_t B, size_t xbytes) {
    TileGeom g;
    const int ng = 32 >> lay.log2gs;
    g.tb = kWarps * ng * kBagsPerGroup;
    g.qc = kStageBytes / (int)(xbytes * (size_t)p.J);
    if (g.qc < 1) g.qc = 1;
    g.tiles_per_table = (int)((B + g.tb - 1) / g.tb);
    return g;
}

size_t tile_smem(const TileGeom& g, const DevParams& p, size_t xbytes) {
    return sizeof(int64_t) * (size_t)(g.tb + 1) + xbytes * (size_t)g.qc * (size_t)p.J;
}

// Arrays from this many elements on take their tiles table by table: the larger
// the array, the better the blocks of one table's hot ids stay in the L2 than
// those of all tables at once; smaller arrays take them bag by bag, whose rows HBM
// writes better.  The line is where the two cross.  Measured on GB300, us per
// serving forward, bag by bag against table by table: 65536 rows of one id (d =
// 128) M = 2^20 143 / 150, 2^22 148 / 156, 2^23 161 / 164, 2^24 182 / 178, 2^25
// 194 / 191, 2^26 208 / 199, 2^28 219 / 203; 16384 rows of 20 ids per bag (d = 64)
// 2^22 211 / 211, 2^24 238 / 225, 2^26 254 / 231.
constexpr int64_t kByTableMinM = int64_t(1) << 24;

// The largest of all shapes: 32 lane groups per warp (a chunk's buckets fit:
// J <= 512).
constexpr size_t kTileSmemMost =
    sizeof(int64_t) * (kWarps * 32 * kBagsPerGroup + 1) + kStageBytes;

template <int VW, int KC, typename XT, bool SG, int MODE>
cudaError_t fwd_mode(const DevParams& p, const RowLayout& lay, const int64_t* idx, int64_t nnz,
                     const int64_t* off, int64_t B, const float* w, float* out, DevError* err,
                     uint32_t* pair_x, uint32_t* q_row, int64_t b_lo, int64_t b_hi, int sm_count,
                     cudaStream_t st) {
    const auto kern = k_forward_warp<VW, KC, XT, SG, MODE>;
    const size_t smem = sizeof(XT) * (size_t)kWarps * (size_t)kWarpPairs;
    const int64_t rows = b_hi - b_lo;
    const int max_grid = grid_for(kern, sm_count, INT32_MAX, smem);
    FwdGeom fg;
    fg.wb = tile_bags(p.T, p.J, lay.log2gs, rows, (int64_t)max_grid * kWarps);
    if (fg.wb > kMaxTileBags) return cudaErrorInvalidValue;   // a bag without a lane
    fg.log2pw = ceil_log2(fg.wb);
    fg.log2pi = 0;
    while (fg.log2pi < 5 && (2 << fg.log2pi) * p.J <= kWarpPairs) ++fg.log2pi;
    const int64_t tpt = (rows + fg.wb - 1) / fg.wb;
    const int64_t ntiles = (int64_t)p.T * tpt;
    if (ntiles >= kMaxTiles) return cudaErrorInvalidValue;
    fg.tiles_per_table = (int)tpt;
    fg.by_table = p.M >= kByTableMinM;
    fg.TJ = (uint64_t)p.T * (uint64_t)p.J;
    fg.Gb = (uint64_t)p.G * sizeof(float);
    for (int k = 0; k < 2; ++k) {
        const unsigned lanes = 32u >> (k ? fg.log2pi : fg.log2pw);
        fg.stepA[k] = (uint64_t)((unsigned __int128)p.A * lanes % kP61);
        fg.stepA2[k] = (uint64_t)((unsigned __int128)p.A2 * lanes % kP61);
    }
    const int64_t blocks = (ntiles + kWarps - 1) / kWarps;
    const int grid = blocks < max_grid ? (int)blocks : max_grid;
    return launch_k(kern, dim3(grid), dim3(kThreads), smem, st, p, idx, nnz, off, B, w, out, err,
                    pair_x, q_row, lay.log2gs, fg, b_lo, b_hi);
}

template <int VW, int KC, typename XT, typename AT, bool TOUCH>
cudaError_t sc_inst(const DevParams& p, const RowLayout& lay, const int64_t* idx, int64_t nnz,
                    const int64_t* off, int64_t B, const float* gout, float scale, AT* target,
                    const Touched& tc, DevError* err, int sm_count, cudaStream_t st) {
    const TileGeom tg = tile_geom(p, lay, B, sizeof(XT));
    const size_t smem = tile_smem(tg, p, sizeof(XT));
    const int64_t ntiles = (int64_t)p.T * tg.tiles_per_table;
    const int grid =
        grid_for(k_scatter_tiled<VW, KC, XT, AT, TOUCH>, sm_count, ntiles, smem, kTileSmemMost);
    return launch_k(k_scatter_tiled<VW, KC, XT, AT, TOUCH>, dim3(grid), dim3(kThreads), smem, st, p,
                    idx, nnz, off, B, gout, scale, target, tc, err, lay.log2gs, tg);
}

template <int VW, int KC, typename XT, bool SG>
cudaError_t fwd_inst(const DevParams& p, const RowLayout& lay, const int64_t* idx, int64_t nnz,
                     const int64_t* off, int64_t B, const float* w, float* out, DevError* err,
                     uint32_t* pair_x, uint32_t* q_row, int64_t b_lo, int64_t b_hi, int sm_count,
                     cudaStream_t st) {
    // wider rows and 64-bit buckets have one variant
    constexpr bool kModes = KC * VW <= 4 && sizeof(XT) == 4;
    if (kModes && nnz > p.T * B)
        return fwd_mode<VW, KC, XT, SG, kModes ? kFwdLong : kFwdShort>(
            p, lay, idx, nnz, off, B, w, out, err, pair_x, q_row, b_lo, b_hi, sm_count, st);
    // (8 rounds of 16 bags for the warps of 2 CTAs per SM)
    if (kModes && lay.log2gs == 5 && p.T * (b_hi - b_lo) >= (int64_t)8 * 16 * 2 * kWarps * sm_count)
        return fwd_mode<VW, KC, XT, SG, kModes ? kFwdMany : kFwdShort>(
            p, lay, idx, nnz, off, B, w, out, err, pair_x, q_row, b_lo, b_hi, sm_count, st);
    return fwd_mode<VW, KC, XT, SG, kFwdShort>(p, lay, idx, nnz, off, B, w, out, err, pair_x, q_row,
                                               b_lo, b_hi, sm_count, st);
}

template <int VW, int KC>
cudaError_t fwd_x(const DevParams& p, const RowLayout& lay, const int64_t* idx, int64_t nnz,
                  const int64_t* off, int64_t B, const float* w, float* out, DevError* err,
                  uint32_t* pair_x, uint32_t* q_row, int64_t b_lo, int64_t b_hi, int sm_count,
                  cudaStream_t st) {
    // 32-bit buckets, and block starts below 2^32 bytes apart
    if (p.R < 0xffffffffull && p.G < (int64_t(1) << 30))
        return p.smask ? fwd_inst<VW, KC, uint32_t, true>(p, lay, idx, nnz, off, B, w, out, err,
                                                           pair_x, q_row, b_lo, b_hi, sm_count, st)
                       : fwd_inst<VW, KC, uint32_t, false>(p, lay, idx, nnz, off, B, w, out, err,
                                                            pair_x, q_row, b_lo, b_hi, sm_count,
                                                            st);
    return p.smask ? fwd_inst<VW, KC, uint64_t, true>(p, lay, idx, nnz, off, B, w, out, err,
                                                       pair_x, q_row, b_lo, b_hi, sm_count, st)
                   : fwd_inst<VW, KC, uint64_t, false>(p, lay, idx, nnz, off, B, w, out, err,
                                                        pair_x, q_row, b_lo, b_hi, sm_count, st);
}

template <int VW, int KC, typename AT>
cudaError_t sc_x(const DevParams& p, const RowLayout& lay, const int64_t* idx, int64_t nnz,
                 const int64_t* off, int64_t B, const float* gout, float scale, AT* target,
                 const Touched* tc, DevError* err, int sm_count, cudaStream_t st) {
    const Touched none{};
    const bool wide = p.R >= 0xffffffffull;
    if (tc) {
        if (wide)
            return sc_inst<VW, KC, uint64_t, AT, true>(p, lay, idx, nnz, off, B, gout, scale, target,
                                                        *tc, err, sm_count, st);
        return sc_inst<VW, KC, uint32_t, AT, true>(p, lay, idx, nnz, off, B, gout, scale, target,
                                                    *tc, err, sm_count, st);
    }
    if (wide)
        return sc_inst<VW, KC, uint64_t, AT, false>(p, lay, idx, nnz, off, B, gout, scale, target,
                                                     none, err, sm_count, st);
    return sc_inst<VW, KC, uint32_t, AT, false>(p, lay, idx, nnz, off, B, gout, scale, target, none,
                                                 err, sm_count, st);
}

}  // namespace

cudaError_t launch_forward(const DevParams& p, const RowLayout& lay, const int64_t* idx,
                           int64_t nnz, const int64_t* off, int64_t B, const float* w, float* out,
                           DevError* err, uint32_t* pair_x, uint32_t* q_row, int64_t b_lo,
                           int64_t b_hi, int sm_count, cudaStream_t st) {
    if (b_lo < 0 || b_hi > B || b_lo >= b_hi) return cudaErrorInvalidValue;
#define PSS_FW(VW, KC)                                                                        \
    return fwd_x<VW, KC>(p, lay, idx, nnz, off, B, w, out, err, pair_x, q_row, b_lo, b_hi, \
                         sm_count, st)
    if (lay.vw == 4) {
        switch (lay.kc) {
            case 1: PSS_FW(4, 1);
            case 2: PSS_FW(4, 2);
            case 4: PSS_FW(4, 4);
        }
    } else {
        switch (lay.kc) {
            case 1: PSS_FW(1, 1);
            case 2: PSS_FW(1, 2);
            case 4: PSS_FW(1, 4);
            case 8: PSS_FW(1, 8);
            case 16: PSS_FW(1, 16);
        }
    }
#undef PSS_FW
    return cudaErrorInvalidValue;
}

cudaError_t launch_scatter(const DevParams& p, const RowLayout& lay, const int64_t* idx,
                           int64_t nnz, const int64_t* off, int64_t B, const float* grad_out,
                           float scale, float* target, const Touched* touched, DevError* err,
                           int sm_count, cudaStream_t st) {
#define PSS_SC(VW, KC) \
    return sc_x<VW, KC, float>(p, lay, idx, nnz, off, B, grad_out, scale, target, touched, err, \
                               sm_count, st)
    if (lay.vw == 4) {
        switch (lay.kc) {
            case 1: PSS_SC(4, 1);
            case 2: PSS_SC(4, 2);
            case 4: PSS_SC(4, 4);
        }
    } else {
        switch (lay.kc) {
            case 1: PSS_SC(1, 1);
            case 2: PSS_SC(1, 2);
            case 4: PSS_SC(1, 4);
            case 8: PSS_SC(1, 8);
            case 16: PSS_SC(1, 16);
        }
    }
#undef PSS_SC
    return cudaErrorInvalidValue;
}

cudaError_t launch_scatter64(const DevParams& p, const RowLayout& lay_in, const int64_t* idx,
                             int64_t nnz, const int64_t* off, int64_t B, const float* grad_out,
                             double* target, const Touched* touched, DevError* err, int sm_count,
                             cudaStream_t st) {
    // fp64 reductions are scalar: lanes on consecutive elements
    const RowLayout lay = choose_layout(p.d, 1, 1);
    (void)lay_in;
#define PSS_SC(KC) \
    return sc_x<1, KC, double>(p, lay, idx, nnz, off, B, grad_out, 1.0f, target, touched, err, \
                               sm_count, st)
    switch (lay.kc) {
        case 1: PSS_SC(1);
        case 2: PSS_SC(2);
        case 4: PSS_SC(4);
        case 8: PSS_SC(8);
        case 16: PSS_SC(16);
    }
#undef PSS_SC
    return cudaErrorInvalidValue;
}

}  // namespace pss
