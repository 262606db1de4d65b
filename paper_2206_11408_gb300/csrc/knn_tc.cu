// Exact K-nearest-neighbour ground truth on the 5th-generation tensor cores.
//
// The distance matrix is a dense contraction: ||q - x||^2 = ||q||^2 + ||x||^2
// - 2 q.x.  q.x runs on tcgen05.mma (kind::f16, BF16 operands, FP32
// accumulators in tensor memory) with each FP32 operand split into a BF16 high
// part and a BF16 low part: q.x ~ qh.xh + qh.xl + ql.xh (the dropped ql.xl and
// the rounding of the parts are at most 2^-15 of |q||x|).  Every query row keeps the
// K' smallest approximate distances of its share of the base; a second kernel
// takes the K' smallest of all shares, recomputes their distances exactly in
// FP32 (sum of (q - x)^2) and returns the K best by (distance, id).  A query for
// which the approximation's error leaves open whether another row is nearer is done
// again by the FP32 kernel.
//
// k_knn_tc is persistent (one CTA per SM) and warp-specialised:
//   warp 0     TMA producer: 64-column (128-byte, SWIZZLE_128B) chunks of the base
//              tiles (hi, lo) into a ring; rows above 128 dimensions stream the
//              query tile's chunks through it as well
//   warp 1     MMA issuer (one elected lane): 3 products x 4 K-steps per chunk
//              into one of two 128x128 FP32 accumulators in tensor memory.  Up to
//              128 dimensions the query tile is the A operand from tensor memory: with
//              both operands in shared memory a 128 x 128 x 16 product reads all the
//              128 bytes per cycle it gives, and the epilogue's own accesses starve
//   warps 2-5  epilogue: tcgen05.ld of the accumulator (thread = query row),
//              distances and their minimum against the row's K'-th distance;
//              where some row of the warp has a smaller one, every thread
//              appends its own to its row's pending buffer; they also load the
//              query tiles
// A row's K' candidates are (distance, id) pairs in shared memory, in eight
// groups whose largest keys its thread holds in registers; once some row of a
// warp has more than 16 pending, all 32 rows insert theirs side by side, a thread
// per row (replace the largest key, find its group's next, then the row's).  A
// warp-wide insertion of one candidate into one row's sorted list took 260 cycles
// and bounded the launch: the causal candidate search over 200k x 128 rows spent
// 145 ms there; now 27 ms (an insertion for 32 rows at once takes 500 cycles).
//
// Work is dealt out in items of one query tile and one base segment: contiguous
// segments for a kNN launch, base tiles s, s + nseg, ... for the causal one.  Every mbarrier wait is bounded: on a timeout the kernel raises an
// error flag, every role leaves its loop, and tensor memory is released.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <vector>

#include "internal.cuh"

namespace fg {

namespace {

constexpr int TQ = 128;                      // query rows per tile (MMA M)
constexpr int TB = 128;                      // base rows per tile (MMA N)
constexpr int KCH = 64;                      // K elements per chunk (128 bytes of BF16)
constexpr int PART = TQ * 128;               // one 128-row x 128-byte operand part: 16 KB
constexpr int MAX_STAGES = 5;
constexpr int PEND = 32;                     // pending candidates per row
constexpr int QRES_CHUNKS = 2;               // query tiles up to this many chunks stay resident
constexpr int TC_THREADS = 192;
constexpr long WAIT_TRIES = 1L << 21;

using u64 = unsigned long long;
// candidate key: distance bits mapped to unsigned order, then the id (a kept
// distance is finite).  NO_KEY and above: none
constexpr u64 NO_KEY = KNN_NO_KEY;

__device__ __forceinline__ uint32_t ord_of(float d) {
    const uint32_t b = __float_as_uint(d);
    return b ^ ((uint32_t)((int32_t)b >> 31) | 0x80000000u);
}
__device__ __forceinline__ float dist_of(u64 k) {
    const uint32_t o = (uint32_t)(k >> 32);
    return __uint_as_float(o ^ (o & 0x80000000u ? 0x80000000u : 0xFFFFFFFFu));
}

// Bound on |approximate - true| squared distance for norms nq and nx and m dimensions
// (u = 2^-24, an FP32 rounding):
//   2 |q| |x| (2^-15 + 3 ceil(m / 16) 4 u): a low part is at most 2^-8 of its value (half a
//     unit of BF16's 8 bits) and what both parts leave out 2^-17, so ql.xl and the two
//     remainders' products make 2^-15 |q| |x| (Cauchy-Schwarz); and 4 u for each product added
//     in tensor memory, whose additions are not IEEE ones (an assumption: the largest error
//     found, over 48 distributions of m = 8 to 1024, was 0.74 of this term)
//   (ceil(m / 32) + 12) u (|q|^2 + |x|^2): the norms' sums (m / 32 + 4 per lane, 5 between
//     lanes) and the two roundings that put the distance together
// +inf where a distance could overflow.
__host__ __device__ constexpr float product_error(int m) {
    return 2.f * (0x1p-15f + 3.f * ((m + 15) / 16) * 0x1p-22f);
}
__host__ __device__ constexpr float norm_error(int m) { return ((m + 31) / 32 + 12) * 0x1p-24f; }
__device__ __forceinline__ float split_error(float nq, float nx, int m) {
    return product_error(m) * sqrtf(nq) * sqrtf(nx) + 0.25f * norm_error(m) * (4.f * (nq + nx));
}

// Bound on the relative error of an exact distance, the FP32 sum of (q - x)^2 in any
// order: m additions, a subtraction's error twice, a product's
__host__ __device__ constexpr float sum_error(int m) { return (m + 8) * 0x1p-24f; }

// Every row whose approximate distance is v or more, with error err, has an exact one above
// any that is less than this
__device__ __forceinline__ float below(float v, float err, int m) {
    return (v - err) * (1.f - sum_error(m));
}

// split_error for the rows that may lie at a squared distance of at most d: their length
// is at most |q| + sqrt(d) (2^-7 for the roundings), whatever other rows there are
__device__ __forceinline__ float near_error(const NormMax& x, float nq, float d, int m) {
    const float r = sqrtf(nq) + sqrtf(d);
    return split_error(nq, fminf(x.finite, (1.f + 0x1p-7f) * r * r), m);
}

// Whether a row of infinite norm may be nearer than kth: its length is at least
// 1.8e19 (the root of the largest float, less 2 %), so |q - x| >= 1.8e19 - |q|.
// (A NaN or infinite nq or kth: it may.)
__device__ __forceinline__ bool inf_rows_reach(const NormMax& x, float nq, float kth) {
    const float gap = 1.8e19f - 1.01f * sqrtf(nq);
    return x.inf && !(gap > 0.f && kth < 0.99f * gap * gap);
}

struct TcArgs {
    int64_t nq, n;
    int nchunk;           // ceil(m / 64)
    int nbt;              // base tiles
    int nseg;             // segments of the base: contiguous, or the tiles s, s + nseg, ...
    int interleaved;
    int nqt;              // query tiles
    int causal;           // 1: queries are the base rows, row i sees base rows < i
    int pilot;            // > 0 (causal): a CTA takes a query tile's segments one after the
                          // other, and `pilot` full lists hold as many keys as are wanted
    int stages;
    const __nv_bfloat16 *qh, *ql;   // the queries' BF16 parts, row stride ms
    int ms;
    const float* qn;      // ||q||^2 (FP32), nq
    const float* xn;      // ||x||^2 (FP32), n
    u64* keys;            // nq x nseg x KP candidate keys
    float cap_scale, cap_norm;   // with bound: see margins()
    uint32_t* bound;      // optional: per row, the smallest K'-th distance of its finished
                          // segments (ord_of), 0xFFFFFFFF before the first
    int* err;             // device status word (FINGER_ERR_LIMIT on a wait timeout)
};

// a CTA's jobs, the same sequence for every role: (query tile, segment) items
struct Jobs {
    const TcArgs& a;
    int at, round;
    __device__ __forceinline__ explicit Jobs(const TcArgs& a_)
        : a(a_), at(a_.pilot ? 0 : blockIdx.x), round(0) {}
    // query tile, base tiles b0, b0 + step, ... < b1, segment
    __device__ __forceinline__ bool next(int& qt, int& b0, int& b1, int& step, int& seg) {
        if (a.pilot) {   // the largest tiles first, every other round dealt backwards
            const int b = blockIdx.x, G = gridDim.x;
            if (at == a.nseg) {
                at = 0;
                ++round;
            }
            qt = a.nqt - 1 - (round * G + (round & 1 ? G - 1 - b : b));
            if (qt < 0) return false;   // (a CTA's tiles only get smaller)
            seg = b0 = at++;
            b1 = min(a.nbt, qt + 1);
            step = a.nseg;
            return true;
        }
        if (at >= a.nqt * a.nseg) return false;
        if (a.causal) {   // the largest items first
            qt = a.nqt - 1 - at / a.nseg;
            seg = at % a.nseg;
            b0 = seg;
            b1 = min(a.nbt, qt + 1);
            step = a.nseg;
        } else {          // the query tiles of one segment next to each other
            qt = at % a.nqt;
            seg = at / a.nqt;
            b0 = a.interleaved ? seg : (int)((int64_t)a.nbt * seg / a.nseg);
            b1 = a.interleaved ? a.nbt : (int)((int64_t)a.nbt * (seg + 1) / a.nseg);
            step = a.interleaved ? a.nseg : 1;
        }
        at += gridDim.x;
        return true;
    }
};

__device__ __forceinline__ uint32_t s32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

// true in one lane of the (converged) warp, always the same one
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile(
        "{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(p));
    return p != 0;
}

// bounded parity wait; false (and the abort flag raised) on timeout
__device__ __forceinline__ bool wait_bar(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                         int* err) {
    for (long it = 0; it < WAIT_TRIES; ++it) {
        uint32_t ok;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
            " selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
        if (ok) return true;
        if (*abort_flag) return false;
    }
    *abort_flag = 1;
    atomicOr(err, (int)FINGER_ERR_LIMIT);
    return false;
}

// shared-memory matrix descriptor: K-major operand, 128-byte swizzle, 8-row
// atoms of 1024 bytes stacked along M/N
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr) {
    return (uint64_t)((saddr >> 4) & 0x3FFF) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

__device__ __forceinline__ void mma_bf16_tc(uint32_t tmem, uint64_t ad, uint64_t bd, uint32_t idesc,
                                            uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
        "l"(ad), "l"(bd), "r"(idesc), "r"(accumulate));
}

// the same with A (128 rows, one per lane, two BF16 of K per column) in tensor memory
__device__ __forceinline__ void mma_bf16_ts(uint32_t tmem, uint32_t at, uint64_t bd, uint32_t idesc,
                                            uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(tmem),
        "r"(at), "l"(bd), "r"(idesc), "r"(accumulate));
}

__device__ __forceinline__ void tma_2d(uint32_t dst, const CUtensorMap* map, int x, int y,
                                       uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
            dst),
        "l"((uint64_t)map), "r"(x), "r"(y), "r"(bar)
        : "memory");
}

// 32 columns of this thread's tensor-memory lane; the registers hold them after
// tmem_wait32, which takes them as operands so that no use moves ahead of it
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,"
        "%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
          "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]),
          "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]),
          "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait32(uint32_t (&r)[32]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]),
                   "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]),
                   "+r"(r[14]), "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]),
                   "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]),
                   "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31]));
}

// 32 columns of this thread's tensor-memory lane from registers (wait::st ends it)
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,"
        "%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};" ::"r"(taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
        "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]),
        "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]),
        "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]),
        "r"(r[29]), "r"(r[30]), "r"(r[31])
        : "memory");
}

// (qn + xa) - 2 ra, (qn + xb) - 2 rb, each rounded as its scalar form is
__device__ __forceinline__ void dist2(float qn, float xa, float xb, uint32_t ra, uint32_t rb,
                                      float& va, float& vb) {
    asm("{\n .reg .b64 q, x, r, n;\n mov.b64 q, {%2, %2};\n mov.b64 x, {%3, %4};\n"
        " mov.b64 r, {%5, %6};\n mov.b64 n, {%7, %7};\n add.rn.f32x2 x, q, x;\n"
        " fma.rn.f32x2 x, n, r, x;\n mov.b64 {%0, %1}, x;\n}\n"
        : "=f"(va), "=f"(vb)
        : "f"(qn), "f"(xa), "f"(xb), "r"(ra), "r"(rb), "f"(-2.f));
}

// Candidates of one row: slot i is dist[128 i] (ord_of bits) and id[128 i], group g
// holds the slots g GS .. g GS + GS - 1; gm: the groups' largest distances, gs:
// their places (4 bits each).  The choices go by distance alone, one 32-bit
// maximum per step; equal ones are told apart by id on a path of their own.
template <int KP>
struct RowTop {
    static constexpr int GS = KP / 8;
    uint32_t *dist, *id;
    uint32_t gm[8], root, gs;
    int g;   // group of the root

    __device__ __forceinline__ uint32_t* id_at(int grp, int place) const {
        return id + 128 * (GS * grp + place);
    }
    __device__ __forceinline__ uint32_t place_of(int grp) const { return (gs >> (4 * grp)) & 15u; }
    __device__ __forceinline__ uint32_t root_id() const { return *id_at(g, place_of(g)); }
    __device__ __forceinline__ void clear() {
        for (int i = 0; i < KP; ++i) {
            dist[128 * i] = 0xFFFFFFFFu - i;   // above +inf, and distinct
            id[128 * i] = 0xFFFFFFFFu;
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) gm[i] = 0xFFFFFFFFu - i * GS;
        gs = 0u;
        root = 0xFFFFFFFFu;
        g = 0;
    }
    // the largest key gives way to (d, i), which is smaller
    __device__ __forceinline__ void insert(uint32_t d, uint32_t i) {
        const int at = 128 * (GS * g + (int)place_of(g));
        dist[at] = d;
        id[at] = i;
        const uint32_t* grp = dist + 128 * GS * g;
        uint32_t k[GS], m = 0u, same = 0u;
#pragma unroll
        for (int j = 0; j < GS; ++j) k[j] = grp[128 * j];
#pragma unroll
        for (int j = 0; j < GS; ++j) m = max(m, k[j]);
#pragma unroll
        for (int j = 0; j < GS; ++j) same |= k[j] == m ? 1u << j : 0u;
        int p = __ffs(same) - 1;
        for (same &= same - 1; same; same &= same - 1) {   // equal distances: the larger id
            const int o = __ffs(same) - 1;
            if (*id_at(g, o) > *id_at(g, p)) p = o;
        }
        gs = (gs & ~(15u << (4 * g))) | ((uint32_t)p << (4 * g));
        root = 0u;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            gm[j] = j == g ? m : gm[j];
            root = max(root, gm[j]);
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) same |= gm[j] == root ? 1u << j : 0u;
        g = __ffs(same) - 1;
        for (same &= same - 1; same; same &= same - 1) {
            const int o = __ffs(same) - 1;
            if (*id_at(o, place_of(o)) > root_id()) g = o;
        }
    }
};

template <int KP, bool QRES>
__global__ void __launch_bounds__(TC_THREADS, 1)
    k_knn_tc(const __grid_constant__ CUtensorMap tqh, const __grid_constant__ CUtensorMap tql,
             const __grid_constant__ CUtensorMap txh, const __grid_constant__ CUtensorMap txl,
             TcArgs a) {
    static_assert(KP == 32 || KP == 64, "candidate lists of 32 or 64");
    // tensor memory: two 128-column accumulators, then two query tiles of 2 x 64 columns
    constexpr int TMEM_COLS = QRES ? 512 : 256, QCOL = 2 * TB, QBUF = 128;
    constexpr int XOFF = QRES ? 0 : 2 * PART;                      // a stage: [qh, ql,] xh, xl
    constexpr int STAGE_BYTES = XOFF + 2 * PART;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* sm = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    unsigned char* stages = sm;
    uint32_t* lists = reinterpret_cast<uint32_t*>(stages + (size_t)a.stages * STAGE_BYTES);
    // lists: KP x 128 distances, then ids; PEND x 128 pending (distance, id)
    uint2* pend = reinterpret_cast<uint2*>(lists + 2 * KP * TQ);
    float* xns = reinterpret_cast<float*>(pend + PEND * TQ);                        // 4 x 64 norms
    uint64_t* bars = reinterpret_cast<uint64_t*>(xns + 4 * 64);
    // full[], empty[], accf[2], acce[2], qfull[2]
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * MAX_STAGES + 6);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const uint32_t ring = s32(stages);
    const uint32_t full0 = s32(bars), empty0 = s32(bars + MAX_STAGES),
                   accf0 = s32(bars + 2 * MAX_STAGES), acce0 = accf0 + 16, qfull0 = accf0 + 32;

    if (threadIdx.x == 0) {
        for (int i = 0; i < 2 * MAX_STAGES + 6; ++i) {
            const int count = i >= 2 * MAX_STAGES + 2 ? 128 : 1;   // acce, qfull: the epilogue
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(full0 + 8 * i), "r"(count));
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         s32(tmem_slot)),
                     "n"(TMEM_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);
    Jobs jobs(a);
    int qt, b0, b1, step, seg;

    // The producer and the MMA warp run their loops whole, with one elected lane for
    // the asynchronous instructions only: descriptors, barriers and coordinates then
    // stay in uniform registers, where those instructions take them.  (On one
    // lane alone the issue of a tile's products took 1,800 cycles for 1,400 of work.)
    const bool leader = elect_one();
    auto wait_all = [&](uint32_t bar, uint32_t parity) {
        return __all_sync(0xffffffffu, wait_bar(bar, parity, abort_flag, a.err)) != 0;
    };
    if (warp == 0) {
        uint32_t s = 0, ph = 1u;   // ring slot and its parity for `empty`
        bool ok = true;
        while (ok && jobs.next(qt, b0, b1, step, seg))
            for (int bt = b0; ok && bt < b1; bt += step)
                for (int c = 0; c < a.nchunk; ++c) {
                    ok = wait_all(empty0 + 8 * s, ph);
                    if (!ok) break;
                    const uint32_t fb = full0 + 8 * s;
                    const uint32_t dst = ring + s * STAGE_BYTES;
                    if (leader) {
                        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(fb),
                                     "r"(STAGE_BYTES)
                                     : "memory");
                        if (!QRES) {
                            tma_2d(dst, &tqh, c * KCH, qt * TQ, fb);
                            tma_2d(dst + PART, &tql, c * KCH, qt * TQ, fb);
                        }
                        tma_2d(dst + XOFF, &txh, c * KCH, bt * TB, fb);
                        tma_2d(dst + XOFF + PART, &txl, c * KCH, bt * TB, fb);
                    }
                    __syncwarp();
                    if (++s == (uint32_t)a.stages) {
                        s = 0;
                        ph ^= 1u;
                    }
                }
    } else if (warp == 1) {
        // D F32, A BF16, B BF16, K-major A and B, N = 128, M = 128
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(TB >> 3) << 17) |
                               ((uint32_t)(TQ >> 4) << 24);
        uint32_t s = 0, ph = 0u, job = 0, tile = 0;
        bool ok = true;
        while (ok && jobs.next(qt, b0, b1, step, seg)) {
            if (b0 >= b1) continue;
            uint32_t qt0 = 0;
            if (QRES) {
                ok = wait_all(qfull0 + 8 * (job & 1u), (job >> 1) & 1u);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                qt0 = tmem + QCOL + (job & 1u) * QBUF;
                ++job;
            }
            for (int bt = b0; ok && bt < b1; bt += step, ++tile) {
                const uint32_t b = tile & 1u, tph = (tile >> 1) & 1u;
                ok = wait_all(acce0 + 8 * b, tph ^ 1u);
                if (!ok) break;
                const uint32_t d = tmem + b * TB;
                for (int c = 0; c < a.nchunk; ++c) {
                    ok = wait_all(full0 + 8 * s, ph);
                    if (!ok) break;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t st = ring + s * STAGE_BYTES;
                    const uint64_t xd = sdesc(st + XOFF), qd = sdesc(st);   // + 2 per 32 bytes
                    if (leader) {
#pragma unroll
                        for (int k = 0; k < KCH / 16; ++k) {
                            const uint64_t xh = xd + 2 * k, xl = xd + (PART >> 4) + 2 * k;
                            if constexpr (QRES) {   // 8 columns per K step; low parts from column 64
                                const uint32_t qh = qt0 + (KCH / 2) * c + 8 * k, ql = qh + 64;
                                mma_bf16_ts(d, qh, xh, idesc, (c | k) != 0);
                                mma_bf16_ts(d, qh, xl, idesc, 1u);
                                mma_bf16_ts(d, ql, xh, idesc, 1u);
                            } else {
                                const uint64_t qh = qd + 2 * k, ql = qd + (PART >> 4) + 2 * k;
                                mma_bf16_tc(d, qh, xh, idesc, (c | k) != 0);
                                mma_bf16_tc(d, qh, xl, idesc, 1u);
                                mma_bf16_tc(d, ql, xh, idesc, 1u);
                            }
                        }
                        asm volatile(
                            "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                                empty0 + 8 * s)
                            : "memory");
                        if (c + 1 == a.nchunk)
                            asm volatile(
                                "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                                    accf0 + 8 * b)
                                : "memory");
                    }
                    __syncwarp();
                    if (++s == (uint32_t)a.stages) {
                        s = 0;
                        ph ^= 1u;
                    }
                }
            }
        }
    } else {
        // epilogue: warp w owns the query rows 32 (w % 4) + lane of every tile
        // (the tensor-memory lanes it may read), thread = row
        const int quarter = warp & 3;
        const int row = 32 * quarter + lane;
        RowTop<KP> top;
        top.dist = lists + row;
        top.id = lists + KP * TQ + row;
        uint2* pr = pend + row;
        float* xs = xns + 64 * quarter;
        uint32_t tile = 0;
        bool stop = false;   // a wait timed out (the same in all lanes: they vote below)
        // Query tile of the next job that has tiles into tensor memory: this thread's row
        // (zeros beyond the rows and columns there are).  Two buffers: a job's tile
        // goes in while the job before it runs, when the one before that is done (its
        // last accumulator has been waited for).
        Jobs ahead(a);
        uint32_t loaded = 0;
        // the largest K'-th distance of the row's first `pilot` segments: as many keys as
        // are wanted lie at or below it, so that the others need none above
        uint32_t pilots = 0u;
        auto load_queries = [&]() {
            int nqt_, f0, f1, fs, fseg;
            do {
                if (!ahead.next(nqt_, f0, f1, fs, fseg)) return;
            } while (f0 >= f1);
            const int64_t qr = (int64_t)nqt_ * TQ + row;
            const uint32_t at = tmem + ((uint32_t)(32 * quarter) << 16) + QCOL + (loaded & 1u) * QBUF;
#pragma unroll 1
            for (int part = 0; part < 2; ++part)
#pragma unroll 1
                for (int c = 0; c < a.nchunk; ++c) {
                    const uint4* src =
                        reinterpret_cast<const uint4*>((part ? a.ql : a.qh) + qr * a.ms) + 8 * c;
                    uint32_t r[32];
#pragma unroll
                    for (int p = 0; p < 8; ++p) {
                        const uint4 v = qr < a.nq && c * KCH + 8 * p < a.ms ? __ldg(src + p)
                                                                           : make_uint4(0u, 0u, 0u, 0u);
                        r[4 * p] = v.x;
                        r[4 * p + 1] = v.y;
                        r[4 * p + 2] = v.z;
                        r[4 * p + 3] = v.w;
                    }
                    tmem_st32(at + 64 * part + (KCH / 2) * c, r);
                }
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(qfull0 + 8 * (loaded & 1u))
                         : "memory");
            ++loaded;
        };
        if (QRES) load_queries();
        while (!stop && jobs.next(qt, b0, b1, step, seg)) {
            if (QRES && b0 < b1) load_queries();   // the next job's
            const int64_t q0 = (int64_t)qt * TQ;
            const int64_t qi = q0 + row;
            const int64_t id_end = a.causal ? min(qi, a.n) : a.n;   // ids below this count
            const int64_t lim = a.causal ? min(q0, a.n) : a.n;      // smallest id_end of the tile
            const float qn = qi < a.nq ? a.qn[qi] : 0.f;
            // only distances below thr count: the row's K'-th here, and from the start
            // what the row's finished segments say (their K'-th smallest is no
            // smaller than the whole base's; equal distances still count, by id)
            if (seg == 0) pilots = 0u;
            uint32_t bound = 0xFF800000u;
            if (a.pilot && seg >= a.pilot) bound = min(bound, pilots);
            if (a.bound && qi < a.nq) bound = min(bound, *(volatile uint32_t*)(a.bound + qi));
            float cap = bound < 0xFF800000u ? dist_of((u64)(bound + 1u) << 32) : INFINITY;
            // (a kNN launch keeps what the approximation may have misplaced, see margins())
            if (a.bound) cap = fmaf(fmaxf(cap, 0.f), a.cap_scale, qn * a.cap_norm);
            float thr = qi < a.nq ? cap : -INFINITY;
            int cnt = 0;                                    // pending candidates of the row
            top.clear();
            auto flush = [&]() {
                const int most = __reduce_max_sync(0xffffffffu, cnt);
                for (int p = 0; p < most; ++p) {
                    if (p >= cnt) continue;
                    const uint2 e = pr[128 * p];
                    const uint32_t d = ord_of(__uint_as_float(e.x));
                    if (d < top.root || (d == top.root && e.y < top.root_id())) top.insert(d, e.y);
                }
                cnt = 0;
                // (a list that is not full: its root is a NaN's bits, and cap stays)
                if (qi < a.nq) thr = fminf(cap, dist_of((u64)top.root << 32));
            };
            // a tile's 128 base norms, four per lane, requested two tiles ahead: behind
            // the base tiles' own traffic a load takes over 1,000 cycles (half a tile
            // ahead the epilogue waited for them, 8.3 ms of a launch of 10.9)
            auto norms = [&](int bt) {
                const int64_t id = (int64_t)bt * TB + 4 * lane;
                if (id + 4 <= a.n) return __ldg(reinterpret_cast<const float4*>(a.xn + id));
                return make_float4(id < a.n ? __ldg(a.xn + id) : 0.f,
                                   id + 1 < a.n ? __ldg(a.xn + id + 1) : 0.f,
                                   id + 2 < a.n ? __ldg(a.xn + id + 2) : 0.f, 0.f);
            };
            float4 xnow, x1 = norms(b0), x2 = norms(b0 + step);
            for (int bt = b0; bt < b1; bt += step, ++tile) {
                const uint32_t b = tile & 1u, tph = (tile >> 1) & 1u;
                xnow = x1;
                x1 = x2;
                x2 = norms(bt + 2 * step);
                // norms of 32 columns, read ahead of the accumulator's load: behind it in
                // the same queue they took 250 cycles a step
                float4 x[8];
                auto put = [&](int half) {   // half a tile's norms into shared memory
                    __syncwarp();
                    if (lane >> 4 == half) reinterpret_cast<float4*>(xs)[lane & 15] = xnow;
                    __syncwarp();
                };
                auto get = [&](int c) {
#pragma unroll
                    for (int j = 0; j < 8; ++j) x[j] = reinterpret_cast<const float4*>(xs + (c & 32))[j];
                };
                put(0);
                get(0);
                stop = !__all_sync(0xffffffffu, wait_bar(accf0 + 8 * b, tph, abort_flag, a.err));
                if (stop) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t tbase = tmem + ((uint32_t)(32 * quarter) << 16) + b * TB;
                const bool masked = (int64_t)(bt + 1) * TB > lim;
                uint32_t r[32];
                tmem_ld32(tbase, r);
                // one warp per scheduler: 32 columns per step for independent work, and
                // a loop that fits the instruction cache (unrolled over the tile the
                // launch took 1.5x)
#pragma unroll 1
                for (int c = 0; c < TB; c += 32) {
                    const int64_t id0 = (int64_t)bt * TB + c;
                    tmem_wait32(r);
                    float v[32];
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        dist2(qn, x[j].x, x[j].y, r[4 * j], r[4 * j + 1], v[4 * j], v[4 * j + 1]);
                        dist2(qn, x[j].z, x[j].w, r[4 * j + 2], r[4 * j + 3], v[4 * j + 2], v[4 * j + 3]);
                    }
                    if (masked) {   // (norms() fills the last tile's padding with 0)
#pragma unroll
                        for (int j = 0; j < 32; ++j) v[j] = id0 + j < id_end ? v[j] : INFINITY;
                    }
                    if (c + 32 < TB) {   // the next columns, behind the checks
                        if (c == 32) put(1);
                        get(c + 32);
                        tmem_ld32(tbase + c + 32, r);
                    }
                    float mn[2];
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        float t[4];
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            t[j] = fminf(fminf(v[16 * h + j], v[16 * h + 4 + j]),
                                         fminf(v[16 * h + 8 + j], v[16 * h + 12 + j]));
                        mn[h] = fminf(fminf(t[0], t[1]), fminf(t[2], t[3]));
                    }
                    if (!__any_sync(0xffffffffu, fminf(mn[0], mn[1]) < thr)) continue;
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        if (!__any_sync(0xffffffffu, mn[h] < thr)) continue;
                        // append (at most 16 pending here, 32 afterwards).  Ids grow along the
                        // scan, so an equal distance already listed comes first.
                        uint2* w = pr + 128 * cnt;
#pragma unroll
                        for (int j = 16 * h; j < 16 * h + 16; ++j) {
                            const bool hit = v[j] < thr;
                            if (hit) *w = make_uint2(__float_as_uint(v[j]), (uint32_t)id0 + j);
                            w += hit ? 128 : 0;
                        }
                        cnt = (int)(w - pr) >> 7;
                        if (__any_sync(0xffffffffu, cnt > PEND - 16)) flush();
                    }
                }
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(acce0 + 8 * b) : "memory");
            }
            flush();
            if (qi < a.nq) {
                if (seg < a.pilot) pilots = max(pilots, top.root);
                if (a.bound) atomicMin(a.bound + qi, top.root);
                u64* out = a.keys + ((size_t)qi * a.nseg + seg) * KP;
                for (int k = 0; k < KP; k += 2)
                    *reinterpret_cast<uint4*>(out + k) =
                        make_uint4(top.id[128 * k], top.dist[128 * k], top.id[128 * (k + 1)],
                                   top.dist[128 * (k + 1)]);
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(TMEM_COLS));
}

// FP32 rows -> BF16 high and low parts (row stride ms, zero padded) and the
// FP32 squared norm of every row; one warp per row.  With bound (the queries of a kNN
// launch): their bounds start at none, and the count of redo at 0
__global__ void k_split_bf16(const float* __restrict__ X, int64_t rows, int m, int64_t x_stride,
                             int ms, __nv_bfloat16* hi, __nv_bfloat16* lo, float* norm2,
                             uint32_t* bound = nullptr, int32_t* redo = nullptr) {
    const int lane = threadIdx.x & 31;
    const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (w >= rows) return;
    float acc = 0.f;
    for (int k = lane; k < ms; k += 32) {
        const float x = k < m ? X[w * x_stride + k] : 0.f;
        const __nv_bfloat16 h = __float2bfloat16_rn(x);
        hi[w * ms + k] = h;
        lo[w * ms + k] = __float2bfloat16_rn(x - __bfloat162float(h));
        acc = fmaf(x, x, acc);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (norm2 && lane == 0) norm2[w] = acc;
    if (bound && lane == 0) {
        bound[w] = 0xFFFFFFFFu;
        if (w == 0) redo[0] = 0;
    }
}

__device__ __forceinline__ u64 warp_min(u64 k) {
    const uint32_t hi = __reduce_min_sync(0xffffffffu, (uint32_t)(k >> 32));
    const uint32_t lo =
        __reduce_min_sync(0xffffffffu, (uint32_t)(k >> 32) == hi ? (uint32_t)k : 0xFFFFFFFFu);
    return (u64)hi << 32 | lo;
}

// The R smallest of a warp's 32 E distinct keys (E per lane, destroyed), ascending,
// into out[0..R); NO_KEY where there are fewer
template <int E>
__device__ __forceinline__ void warp_smallest(u64 (&k)[E], int R, u64* out, int lane) {
    for (int r = 0; r < R; ++r) {
        u64 m = k[0];
#pragma unroll
        for (int j = 1; j < E; ++j) m = k[j] < m ? k[j] : m;
        m = warp_min(m);
        if (m >= NO_KEY) {
            for (int i = r + lane; i < R; i += 32) out[i] = NO_KEY;
            break;
        }
#pragma unroll
        for (int j = 0; j < E; ++j) k[j] = k[j] == m ? NO_KEY : k[j];
        if (lane == 0) out[r] = m;
    }
    __syncwarp();
}

// The KP smallest of the nc keys kr[], ascending, into sel[].  W warps (this one is wq;
// part: W KP keys of shared memory), E keys per lane: nc <= 32 E W.
template <int W, int E>
__device__ __forceinline__ void pick(const u64* kr, int nc, int KP, u64* sel, u64* part, int wq, int lane) {
    u64 k[E];
#pragma unroll
    for (int j = 0; j < E; ++j) {
        const int c = (j * W + wq) * 32 + lane;
        k[j] = c < nc ? kr[c] : NO_KEY;
    }
    if constexpr (W == 1) {
        warp_smallest<E>(k, KP, sel, lane);
    } else {
        warp_smallest<E>(k, KP, part + wq * KP, lane);
        __syncthreads();
        if (wq == 0) {
            u64 k2[2 * W];
#pragma unroll
            for (int j = 0; j < 2 * W; ++j)
                k2[j] = 32 * j + lane < W * KP ? part[32 * j + lane] : NO_KEY;
            warp_smallest<2 * W>(k2, KP, sel, lane);
        }
        __syncthreads();
    }
}

// the distance of each key of sel[] gives way to its row's exact one, sum of (q - x)^2 in
// FP32; four rows in flight per warp
template <int W>
__device__ __forceinline__ void exact_keys(const float4* __restrict__ X, int m4, const float* qr, int m,
                                           u64* sel, int KP, int wq, int lane) {
    constexpr int U = 4;
    for (int i = wq * U; i < KP; i += W * U) {
        uint32_t id[U];
        float acc[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            id[u] = (uint32_t)sel[i + u];
            acc[u] = 0.f;
        }
        for (int c = lane; c < m4; c += 32) {
            float4 x[U];
#pragma unroll
            for (int u = 0; u < U; ++u)
                x[u] = (int32_t)id[u] >= 0 ? __ldg(X + (size_t)id[u] * m4 + c)
                                           : make_float4(0.f, 0.f, 0.f, 0.f);
            const int e = 4 * c;
            float qv[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) qv[t] = e + t < m ? qr[e + t] : 0.f;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                float dlt;
                dlt = qv[0] - x[u].x; acc[u] = fmaf(dlt, dlt, acc[u]);
                dlt = qv[1] - x[u].y; acc[u] = fmaf(dlt, dlt, acc[u]);
                dlt = qv[2] - x[u].z; acc[u] = fmaf(dlt, dlt, acc[u]);
                dlt = qv[3] - x[u].w; acc[u] = fmaf(dlt, dlt, acc[u]);
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int u = 0; u < U; ++u) acc[u] += __shfl_xor_sync(0xffffffffu, acc[u], o);
        __syncwarp();
        if (lane < U && (int32_t)(uint32_t)sel[i + lane] >= 0) {
            const float d = lane == 0 ? acc[0] : lane == 1 ? acc[1] : lane == 2 ? acc[2] : acc[3];
            sel[i + lane] = (u64)ord_of(d) << 32 | (uint32_t)sel[i + lane];
        }
    }
    if constexpr (W == 1) __syncwarp();
    else __syncthreads();
}

// the K-th smallest key of sel[0..KP) (one warp); NO_KEY or above if there are fewer
__device__ __forceinline__ u64 kth_key(const u64* sel, int KP, int K, int lane) {
    u64 kth = ~0ull;
    for (int i = lane; i < KP; i += 32) {
        int rank = 0;
        for (int j = 0; j < KP; ++j) rank += sel[j] < sel[i];
        if (rank == K - 1) kth = sel[i];
    }
    return warp_min(kth);
}

// the K smallest keys of sel[0..KP) in order (one warp)
__device__ __forceinline__ void put_best(const u64* sel, int KP, int K, int64_t* out_ids, float* out_d,
                                         int lane) {
    for (int i = lane; i < KP; i += 32) {
        const u64 ki = sel[i];
        int rank = 0;
        for (int j = 0; j < KP; ++j) {
            const u64 kj = sel[j];
            rank += kj < ki || (kj == ki && j < i);   // (only NO_KEYs are equal)
        }
        if (rank < K) {
            const bool ok = (int32_t)(uint32_t)ki >= 0;
            out_ids[rank] = ok ? (int64_t)(uint32_t)ki : (int64_t)-1;
            out_d[rank] = ok ? dist_of(ki) : INFINITY;
        }
    }
}

// Final step of a kNN launch: the KP smallest approximate keys of a query's lists,
// their exact FP32 distances, the K best by (distance, id).  A row outside the lists has
// an approximate distance of at least the KP-th, so an exact one of at least that less
// the approximation's error: the K-th exact distance lies below, and the result stands.
// Where it does not (rows far from the origin, many equal distances), the lists' other
// keys get their exact distances too, and the nearest row that a full list may have
// dropped takes the place of the KP-th.  A query that still does not stand, or whose
// approximate distances may not be finite, goes on `redo` (count in redo[0]) for
// launch_knn_parts and k_redo_rank.  W warps per query (E keys per lane: 32 E W >= the
// query's keys); with W = 1 four queries per block.
template <int W, int E>
__global__ void __launch_bounds__(W == 1 ? 128 : 32 * W)
    k_rerank(const float4* __restrict__ X, int m4, const float* __restrict__ Q, int m, int64_t nq,
             const u64* __restrict__ keys, int nc, int KP, int K, const float* __restrict__ qn,
             const NormMax* __restrict__ xmax, int64_t* out_ids, float* out_d, int32_t* redo) {
    constexpr int QPB = W == 1 ? 4 : 1;
    __shared__ u64 sel_s[QPB][64];
    __shared__ u64 part_s[W == 1 ? 1 : W * 64];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int64_t q = W == 1 ? (int64_t)blockIdx.x * 4 + wib : (int64_t)blockIdx.x;
    const int wq = W == 1 ? 0 : wib;
    if (q >= nq) return;
    u64* sel = sel_s[W == 1 ? wib : 0];
    const u64* kr = keys + (size_t)q * nc;
    const float* qr = Q + (size_t)q * m;
    pick<W, E>(kr, nc, KP, sel, part_s, wq, lane);
    const u64 last = sel[KP - 1];   // the KP-th approximate key
    if constexpr (W == 1) __syncwarp();
    else __syncthreads();
    exact_keys<W>(X, m4, qr, m, sel, KP, wq, lane);
    if (wq != 0) return;
    const float nrm = qn[q];
    const u64 k0 = kth_key(sel, KP, K, lane);
    const float kth = k0 < NO_KEY ? dist_of(k0) : INFINITY;
    const float err = near_error(*xmax, nrm, kth, m);
    bool stands = err < INFINITY && !inf_rows_reach(*xmax, nrm, kth);
    if (!stands && !(nrm < INFINITY)) {   // a query that is not finite has no neighbours
        bool bad = false;
        for (int i = lane; i < m; i += 32) bad |= !(fabsf(qr[i]) < INFINITY);
        stands = __any_sync(0xffffffffu, bad);
    }
    if (stands && last < NO_KEY && !(kth < below(dist_of(last), err, m))) {
        const float lim = kth * (1.f + 2.f * sum_error(m)) + err;   // above it no key can be nearer
        uint32_t most = 0;             // the largest distance of the list so far
        float edge = INFINITY;         // the smallest of the full lists' largest
        for (int c0 = 0; c0 < nc; c0 += 32) {
            const u64 kc = kr[c0 + lane];   // (nc and KP: multiples of 32)
            most = max(most, __reduce_max_sync(0xffffffffu, (uint32_t)(kc >> 32)));
            if ((c0 + 32) % KP == 0) {
                if (most < (uint32_t)(NO_KEY >> 32)) edge = fminf(edge, dist_of((u64)most << 32));
                most = 0;
            }
            unsigned more = __ballot_sync(0xffffffffu,
                                          kc < NO_KEY && kc > last && !(dist_of(kc) > lim));
            while (more) {
                const uint32_t id = __shfl_sync(0xffffffffu, (uint32_t)kc, __ffs(more) - 1);
                more &= more - 1;
                float acc = 0.f;
                for (int c = lane; c < m4; c += 32) {
                    const float4 x = __ldg(X + (size_t)id * m4 + c);
                    const int e = 4 * c;
                    float dlt;
                    dlt = (e < m ? qr[e] : 0.f) - x.x; acc = fmaf(dlt, dlt, acc);
                    dlt = (e + 1 < m ? qr[e + 1] : 0.f) - x.y; acc = fmaf(dlt, dlt, acc);
                    dlt = (e + 2 < m ? qr[e + 2] : 0.f) - x.z; acc = fmaf(dlt, dlt, acc);
                    dlt = (e + 3 < m ? qr[e + 3] : 0.f) - x.w; acc = fmaf(dlt, dlt, acc);
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
                // in the place of the largest kept key, if it is smaller
                const u64 key = (u64)ord_of(acc) << 32 | id;
                const u64 a = sel[lane], b = KP > 32 ? sel[lane + 32] : 0ull;
                const u64 top = ~warp_min(~(a > b ? a : b));
                __syncwarp();
                if (key < top) {
                    if (a == top) sel[lane] = key;
                    else if (KP > 32 && b == top) sel[lane + 32] = key;
                }
                __syncwarp();
            }
        }
        stands = dist_of(kth_key(sel, KP, K, lane)) < below(edge, err, m);
    }
    if (stands) put_best(sel, KP, K, out_ids + (size_t)q * K, out_d + (size_t)q * K, lane);
    else if (lane == 0) redo[1 + atomicAdd(redo, 1)] = (int32_t)q;
}

// The queries on `redo` from the FP32 kernel's lists (launch_knn_parts with this grid
// and room): KP smallest keys of all parts, then as k_rerank, whose sums they get.  10,000
// queries x 1M x 128, K = 10: 6.35 ms with none, 8.11 with one, 227 with all of them (the
// rows 10,000 from the origin in every dimension; at 1,000 most stand, 8.5 ms).
__global__ void __launch_bounds__(256)
    k_redo_rank(const float4* __restrict__ X, int64_t n, int m4, const float* __restrict__ Q, int m,
                const u64* __restrict__ parts, int grid, int64_t room, int KP, int K,
                const int32_t* __restrict__ redo, int64_t* out_ids, float* out_d) {
    constexpr int W = 8, E = 16;
    static_assert(32 * E * W >= 64 * REDO_PARTS, "the keys of a query's parts");
    __shared__ u64 sel[64], part_s[W * 64];
    const int lane = threadIdx.x & 31, wq = threadIdx.x >> 5;
    const int count = redo[0], nc = redo_parts(count, grid, room, n) * KP;
    for (int i = blockIdx.x; i < count; i += gridDim.x) {
        const int64_t q = redo[1 + i];
        pick<W, E>(parts + (size_t)i * nc, nc, KP, sel, part_s, wq, lane);
        exact_keys<W>(X, m4, Q + (size_t)q * m, m, sel, KP, wq, lane);
        if (wq == 0) put_best(sel, KP, K, out_ids + (size_t)q * K, out_d + (size_t)q * K, lane);
        __syncthreads();
    }
}

// Final step of a launch with K > 40, where no single list holds K' = K + 32 keys: a
// block per query sorts the keys of its nseg lists of 64 (np: their count rounded
// up to a power of two), takes the R = K' smallest, sums their exact distances in
// the order of the FP32 kernel (a thread per row, dimension after dimension, so
// both paths return the same bits) and ranks them.  A row that is not among the R has
// an approximate distance of at least the R-th and an exact one of at least that less
// both errors, so the K-th exact distance has to lie below.  A query for
// which it does not, that has fewer than R candidates (rows before it, or finite
// distances), or a full list whose keys are all among the R (it may have dropped
// more) goes on `redo` (count in redo[0]) for the FP32 kernel.
__global__ void __launch_bounds__(256)
    k_rerank_big(const float4* __restrict__ X, int m4, const float* __restrict__ Q,
                 int64_t q_stride, int q_m, const u64* __restrict__ keys, int nseg, int np, int R,
                 int K, const int32_t* __restrict__ remap, const float* __restrict__ qn,
                 const NormMax* __restrict__ xmax, int64_t* out_ids, float* out_d, int32_t* redo) {
    extern __shared__ __align__(16) float4 rb_s[];
    float* qs = reinterpret_cast<float*>(rb_s);          // 4 m4: the query, zero padded
    u64* bk = reinterpret_cast<u64*>(rb_s + m4);         // np keys
    u64* top = bk + np;                                  // nseg: a full list's largest key
    u64* ex = top + nseg;                                // R exact keys
    const int t = threadIdx.x, nc = nseg * 64;
    const int64_t q = blockIdx.x;
    for (int i = t; i < np; i += 256) bk[i] = i < nc ? keys[(size_t)q * nc + i] : ~0ull;
    for (int i = t; i < 4 * m4; i += 256) qs[i] = i < q_m ? Q[q * q_stride + i] : 0.f;
    __syncthreads();
    for (int s = t; s < nseg; s += 256) {
        u64 m = 0;
        for (int k = 0; k < 64; ++k) m = max(m, bk[64 * s + ((k + s) & 63)]);
        top[s] = m;
    }
    for (int size = 2; size <= np; size <<= 1)
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            __syncthreads();
            for (int i = t; i < np / 2; i += 256) {
                const int lo = 2 * i - (i & (stride - 1)), hi = lo + stride;
                const u64 a = bk[lo], b = bk[hi];
                if ((a > b) == ((lo & size) == 0)) {
                    bk[lo] = b;
                    bk[hi] = a;
                }
            }
        }
    __syncthreads();
    const u64 last = bk[min(R, np) - 1];
    bool lost = last >= NO_KEY;
    for (int s = t; s < nseg; s += 256) lost |= top[s] < NO_KEY && top[s] <= last;
    if (__syncthreads_or(lost)) {
        if (t == 0) redo[1 + atomicAdd(redo, 1)] = (int32_t)q;
        return;
    }
    // the result stands where the K-th exact distance lies below this (the error taken for
    // rows as far as the R-th)
    const float vr = dist_of(last), nq = qn[q];
    const float proof = inf_rows_reach(*xmax, nq, vr)
                            ? -1.f
                            : below(vr, near_error(*xmax, nq, fmaxf(vr, 0.f), q_m), q_m);
    for (int i = t; i < R; i += 256) {
        const u64 k = i < np ? bk[i] : ~0ull;
        u64 e = ~0ull;
        if (k < NO_KEY) {
            const float4* row = X + (size_t)(uint32_t)k * m4;
            float acc = 0.f;
#pragma unroll 4
            for (int c = 0; c < m4; ++c) {
                const float4 x = __ldg(row + c);
                const float4 y = reinterpret_cast<const float4*>(qs)[c];
                float d;
                d = y.x - x.x; acc = fmaf(d, d, acc);
                d = y.y - x.y; acc = fmaf(d, d, acc);
                d = y.z - x.z; acc = fmaf(d, d, acc);
                d = y.w - x.w; acc = fmaf(d, d, acc);
            }
            e = (u64)ord_of(acc) << 32 | (uint32_t)k;
        }
        ex[i] = e;
    }
    __syncthreads();
    for (int i = t; i < R; i += 256) {
        const u64 k = ex[i];
        int rank = 0;
        for (int j = 0; j < R; ++j) rank += ex[j] < k || (ex[j] == k && j < i);
        if (rank == K - 1 && !(dist_of(k) < proof)) redo[1 + atomicAdd(redo, 1)] = (int32_t)q;
        if (rank < K) {
            const int32_t id = (int32_t)(uint32_t)k;
            out_ids[(size_t)q * K + rank] = id < 0 ? (int64_t)-1 : (int64_t)(remap ? remap[id] : id);
            out_d[(size_t)q * K + rank] = id < 0 ? INFINITY : dist_of(k);
        }
    }
}

// the NormMax of n norms (zeroed before)
__global__ void k_max_norm(const float* __restrict__ xn, int64_t n, NormMax* out) {
    uint32_t m = 0, inf = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const float x = xn[i];
        if (x < INFINITY) m = max(m, __float_as_uint(x));
        inf |= x == INFINITY;
    }
    m = __reduce_max_sync(0xffffffffu, m);
    inf = __reduce_or_sync(0xffffffffu, inf);
    if ((threadIdx.x & 31) == 0) {
        atomicMax(reinterpret_cast<uint32_t*>(&out->finite), m);
        if (inf) atomicOr(&out->inf, 1u);
    }
}

// ascending bitonic sort of a warp's 32 E keys; lane l holds places E l .. E l + E - 1
template <int E>
__device__ __forceinline__ void warp_sort(u64 (&k)[E], int lane) {
#pragma unroll
    for (int size = 2; size <= 32 * E; size <<= 1) {
#pragma unroll
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            if (stride >= E) {   // between lanes
                const int ls = stride / E;
                const bool up = (lane & (size / E)) == 0;
                const bool low = (lane & ls) == 0;
#pragma unroll
                for (int j = 0; j < E; ++j) {
                    const u64 o = __shfl_xor_sync(0xffffffffu, k[j], ls);
                    k[j] = (up == low) == (o < k[j]) ? o : k[j];
                }
            } else {   // within the lane
#pragma unroll
                for (int j = 0; j < E; ++j)
                    if (!(j & stride)) {
                        const bool up = size < E ? (j & size) == 0 : (lane & (size / E)) == 0;
                        const u64 x = k[j], y = k[j | stride];
                        const bool sw = up == (y < x);
                        k[j] = sw ? y : x;
                        k[j | stride] = sw ? x : y;
                    }
            }
        }
    }
}

// The K smallest keys of every row's 512 candidates, ascending, as int64 ids (-1
// padded) and approximate distances; one warp per row sorts them in registers
// (ranking every candidate against all others took 20 ms for 200k rows)
__global__ void __launch_bounds__(128) k_merge_topk(const u64* __restrict__ keys, int64_t rows,
                                                    int K, int64_t* out_ids, float* out_d) {
    constexpr int E = 16;
    __shared__ u64 s[4][32 * (E + 1)];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int64_t w = (int64_t)blockIdx.x * 4 + wib;
    if (w >= rows) return;
    u64 k[E];
#pragma unroll
    for (int j = 0; j < E; ++j) k[j] = keys[(size_t)w * 32 * E + 32 * j + lane];
    warp_sort<E>(k, lane);
#pragma unroll
    for (int j = 0; j < E; ++j) s[wib][lane * (E + 1) + j] = k[j];
    __syncwarp();
    for (int i = lane; i < K; i += 32) {
        const u64 x = s[wib][i / E * (E + 1) + i % E];
        const bool ok = (int32_t)(uint32_t)x >= 0;
        out_ids[(size_t)w * K + i] = ok ? (int64_t)(uint32_t)x : (int64_t)-1;
        out_d[(size_t)w * K + i] = ok ? dist_of(x) : INFINITY;
    }
}

PFN_cuTensorMapEncodeTiled_v12000 get_encode() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        cudaDriverEntryPointQueryResult q;
        void* p = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                             &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    }
    return fn;
}

bool make_map(CUtensorMap* map, const void* base, int64_t rows, int m, int ms) {
    auto enc = get_encode();
    if (!enc) return false;
    cuuint64_t dims[2] = {(cuuint64_t)m, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)ms * 2};
    cuuint32_t box[2] = {KCH, TQ};
    cuuint32_t es[2] = {1, 1};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides,
               box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
               CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// ring stages that the shared memory beside the lists and pending buffers holds
template <int KP, bool QRES>
cudaError_t run_tc(const CUtensorMap* maps, TcArgs a, int grid, cudaStream_t s) {
    const size_t fixed = 1024 + (size_t)(KP + PEND) * TQ * 8 + 4 * 64 * 4 + 8 * (2 * MAX_STAGES + 6) +
                         16;
    const size_t stage = (QRES ? 2 : 4) * PART;
    a.stages = (int)std::min<size_t>(MAX_STAGES, (227 * 1024 - fixed) / stage);
    const size_t smem = fixed + a.stages * stage;
    cudaError_t e = cudaFuncSetAttribute(k_knn_tc<KP, QRES>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_knn_tc<KP, QRES><<<grid, TC_THREADS, smem, s>>>(maps[0], maps[1], maps[2], maps[3], a);
    return cudaGetLastError();
}

}  // namespace

// Largest K the tensor-core path serves (its candidate lists hold 32 or 64).
int knn_tc_max_k() { return 40; }

namespace {

bool capturing(cudaStream_t s) {
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    return cudaStreamIsCapturing(s, &st) != cudaSuccess || st != cudaStreamCaptureStatusNone;
}

cudaError_t max_norm(const float* xn, int64_t n, NormMax* out, cudaStream_t s) {
    const cudaError_t e = cudaMemsetAsync(out, 0, sizeof(NormMax), s);
    if (e != cudaSuccess) return e;
    k_max_norm<<<256, 256, 0, s>>>(xn, n, out);
    return cudaGetLastError();
}

// BF16 split and largest norm of the base rows, made once per index
cudaError_t ensure_split(finger_index* ix, cudaStream_t s) {
    if (ix->xs_hi) return cudaSuccess;
    const int m = ix->m, ms = (m + 7) & ~7;
    const int64_t n = ix->n;
    __nv_bfloat16 *hi = nullptr, *lo = nullptr;
    NormMax* mx = nullptr;
    cudaError_t e = cudaErrorMemoryAllocation;
    if (cudaMalloc(&hi, sizeof(__nv_bfloat16) * (size_t)n * ms) == cudaSuccess &&
        cudaMalloc(&lo, sizeof(__nv_bfloat16) * (size_t)n * ms) == cudaSuccess &&
        cudaMalloc(&mx, sizeof(NormMax)) == cudaSuccess) {
        k_split_bf16<<<(unsigned)((n * 32 + 255) / 256), 256, 0, s>>>(ix->X, n, m, ix->m_pad, ms, hi, lo,
                                                                      nullptr);
        e = cudaGetLastError();
        if (e == cudaSuccess) e = max_norm(ix->xnorm2, n, mx, s);
        // done before a call on another stream finds it there
        if (e == cudaSuccess && !capturing(s)) e = cudaStreamSynchronize(s);
    }
    if (e != cudaSuccess) {
        cudaFree(hi);
        cudaFree(lo);
        cudaFree(mx);
        cudaGetLastError();
        return e;
    }
    ix->xs_hi = hi;
    ix->xs_lo = lo;
    ix->xs_max = mx;
    return cudaSuccess;
}

// what a launch needs of the base rows (BF16 parts with row stride m rounded to 8)
struct TcBase {
    const __nv_bfloat16 *hi, *lo;
    const float* xn;
    const NormMax* xmax;
    int64_t n;
    int m;
};

TcBase base_of(const finger_index* ix) {
    return {ix->xs_hi, ix->xs_lo, ix->xnorm2, ix->xs_max, ix->n, ix->m};
}

enum TcOrder { CONTIGUOUS, INTERLEAVED, CAUSAL };

// What a finished segment's K'-th approximate distance c lets the row's other segments drop:
// K' rows have exact distances of at most c plus both errors, so that a row is no
// result whose approximate distance is above c + 2 split_error + the sums' errors, for
// rows that may be as near (the others are farther by their length).  With |x| <= |q| +
// sqrt(d), |q| |x| is at most 1.5 |q|^2 + d / 2 and |x|^2 at most 2 |q|^2 + 2 d, where d <=
// 1.001 (c + 0.001 |q|^2) as the error is below 2^-11 (|q|^2 + |x|^2): a line in c and |q|^2.
// (With square roots in the kernel 10,000 queries x 1M x 128 took 6.08 ms there instead of
// 6.04.)
void margins(int m, TcArgs* a) {
    const double p = product_error(m), e = norm_error(m), s = 1 + 4 * (double)sum_error(m);
    const double A = 1.5 * p + 3 * e, B = 0.5 * p + 2 * e, up = 1 + 0x1p-20;
    a->cap_scale = (float)((1 + 2.002 * B) * s * up);
    a->cap_norm = (float)((2 * A + 0.002002 * B) * s * up);
}

// one launch of k_knn_tc over nq query rows (BF16 parts qh/ql) against the base
cudaError_t run_items(finger_index* ix, const TcBase& x, const __nv_bfloat16* qh,
                      const __nv_bfloat16* ql, const float* qn, int64_t nq, int KP, int nseg,
                      TcOrder order, u64* keys, uint32_t* bound, cudaStream_t s,
                      int want = 0) {
    const int ms = (x.m + 7) & ~7;
    CUtensorMap maps[4];
    if (!make_map(&maps[0], qh, nq, x.m, ms) || !make_map(&maps[1], ql, nq, x.m, ms) ||
        !make_map(&maps[2], x.hi, x.n, x.m, ms) || !make_map(&maps[3], x.lo, x.n, x.m, ms))
        return cudaErrorInvalidValue;
    TcArgs a{};
    a.nq = nq;
    a.n = x.n;
    a.nchunk = (x.m + KCH - 1) / KCH;
    a.nbt = (int)((x.n + TB - 1) / TB);
    a.nseg = nseg;
    a.interleaved = order != CONTIGUOUS;
    a.nqt = (int)((nq + TQ - 1) / TQ);
    a.causal = order == CAUSAL ? 1 : 0;
    a.qh = qh;
    a.ql = ql;
    a.ms = ms;
    a.qn = qn;
    a.xn = x.xn;
    a.keys = keys;
    a.bound = bound;
    margins(x.m, &a);
    a.err = ix->err;
    // want > 0: the smallest `want` keys of a causal launch's lists are used.  With query
    // tiles enough for all SMs a CTA keeps a tile's segments, and the first of them
    // bound the others (200k x 128 rows, 8 lists of 64 for 200 keys: 33.6 -> 27.3 ms; whole
// builds without / with: 120k x 128 29.9 / 26.7 ms, 80k 19.1 / 17.2, 80k x 960 36.8 /
// 35.9.  Below, the items of few tiles fill the GPU unevenly: 20k x 960 9.13 / 9.47, 10k
// x 128 4.10 / 4.37, though 40k x 128 would gain, 10.8 / 10.0)
    if (order == CAUSAL && want > 0 && a.nqt >= 4 * ix->num_sms) a.pilot = (want + 63) / 64;
    const int grid = (int)std::min<int64_t>(ix->num_sms, (int64_t)a.nqt * (a.pilot ? 1 : nseg));
    const bool res = a.nchunk <= QRES_CHUNKS;
    if (KP == 32) return res ? run_tc<32, true>(maps, a, grid, s) : run_tc<32, false>(maps, a, grid, s);
    return res ? run_tc<64, true>(maps, a, grid, s) : run_tc<64, false>(maps, a, grid, s);
}

// How a kNN of K <= 40 is divided: queries per pass, and base segments.  The items
// (query tile, segment) are dealt to one CTA per SM in waves, segment by segment, so
// the CTAs of a wave scan the same rows at the same time: a segment of at most 48 MB of
// BF16 parts stays in L2 for them.  (One equal range of the (query tile, base tile)
// sequence per CTA balances without waves, but each CTA then scans rows of its own and
// DRAM bounds it: 10,000 queries x 1M x 128 took 11.6 ms; with segments of 12 MB 7.9, of 24
// 7.1, of 48 to 192 6.5.)  From there the smallest
// count whose last wave costs at most 3 %, or the best of the next 32; each segment
// adds a list of K' per row to fill and to merge.  Above MAX_KEYS / K' such segments
// (12.9 or 25.8 GB of parts) they grow instead: k_rerank takes MAX_KEYS keys per query
// and each pass reads the base from DRAM anyway.  Passes keep the lists below twice
// LIST_BYTES for any number of queries; one still has 4,096 items or more.
constexpr int MAX_KEYS = 16 * 32 * 32;   // the widest k_rerank: 16 warps of 32 keys per lane
constexpr int64_t LIST_BYTES = 256 << 20;

struct KnnPlan {
    int KP, nseg;
    int64_t chunk;   // queries per pass
};

KnnPlan knn_plan(int64_t n, int m, int64_t nq, int K, int num_sms, int64_t most) {
    KnnPlan p;
    p.KP = K <= 16 ? 32 : 64;
    const int64_t nbt = (n + TB - 1) / TB, G = num_sms;
    const int64_t bytes = nbt * TB * ((m + 7) & ~7) * 4;
    const int64_t top = std::min<int64_t>(nbt, MAX_KEYS / p.KP);
    const int64_t lo = std::min<int64_t>(top, std::max<int64_t>(bytes / (48 << 20), 1));
    const int64_t row = 8 * p.KP;   // list bytes per query and segment
    int64_t c = std::min(nq, std::min(most, std::max<int64_t>(TQ, LIST_BYTES / (row * lo))));
    const int64_t passes = (nq + c - 1) / c;
    c = std::min(nq, ((nq + passes - 1) / passes + TQ - 1) / TQ * TQ);
    p.chunk = c;
    const int64_t nqt = (c + TQ - 1) / TQ;
    const int64_t hi = std::min(std::min(top, std::max(lo + 32, (G + nqt - 1) / nqt)),
                                std::max(lo, 2 * LIST_BYTES / (row * c)));
    p.nseg = (int)lo;
    double best_eff = 0;
    for (int64_t S = lo; S <= hi; ++S) {
        const int64_t items = nqt * S;
        const double eff = (double)items / ((items + G - 1) / G * G);
        if (eff > best_eff + 0.002) {
            best_eff = eff;
            p.nseg = (int)S;
        }
        if (best_eff >= 0.97) break;
    }
    return p;
}

}  // namespace

// the plan of a call, for tests on the host: {K', segments, queries per pass, most keys}
extern "C" void fg_knn_plan(int64_t n, int m, int64_t nq, int K, int num_sms, int64_t* out) {
    const KnnPlan p = knn_plan(n, m, nq, K, num_sms, nq);
    out[0] = p.KP;
    out[1] = p.nseg;
    out[2] = p.chunk;
    out[3] = MAX_KEYS;
}

cudaError_t launch_knn_tc(finger_index* ix, const float* Q, int64_t nq, int K, int64_t* out_ids,
                          float* out_d, cudaStream_t s) {
    if (nq <= 0) return cudaSuccess;
    const int m = ix->m, ms = (m + 7) & ~7;
    const int64_t n = ix->n;
    cudaError_t e = ensure_split(ix, s);
    if (e != cudaSuccess) return e;
    // one stream-ordered allocation for all temporaries (a pool that keeps nothing between
    // calls maps each of them anew)
    unsigned char* tmp = nullptr;
    KnnPlan p;
    size_t at[6];
    for (int64_t most = nq;; most = p.chunk / 2) {   // fewer queries per pass where memory is short
        p = knn_plan(n, m, nq, K, ix->num_sms, most);
        const size_t c = (size_t)p.chunk;
        const size_t bytes[6] = {8 * c * p.nseg * p.KP, 4 * c, 2 * c * ms, 2 * c * ms, 4 * c, 4 * (c + 1)};
        size_t total = 0;
        for (int i = 0; i < 6; ++i) {
            at[i] = total;
            total += (bytes[i] + 255) & ~size_t(255);
        }
        if (cudaMallocAsync(&tmp, total, s) == cudaSuccess) break;
        cudaGetLastError();
        if (p.chunk <= TQ) return cudaErrorMemoryAllocation;
    }
    u64* keys = reinterpret_cast<u64*>(tmp + at[0]);
    uint32_t* bound = reinterpret_cast<uint32_t*>(tmp + at[1]);
    __nv_bfloat16* qh = reinterpret_cast<__nv_bfloat16*>(tmp + at[2]);
    __nv_bfloat16* ql = reinterpret_cast<__nv_bfloat16*>(tmp + at[3]);
    float* qn = reinterpret_cast<float*>(tmp + at[4]);
    int32_t* redo = reinterpret_cast<int32_t*>(tmp + at[5]);
    const int nc = p.nseg * p.KP, KP = p.KP;
    const float4* X = reinterpret_cast<const float4*>(ix->X);
    for (int64_t lo = 0; lo < nq && e == cudaSuccess; lo += p.chunk) {
        const int64_t c = std::min(p.chunk, nq - lo);
        const float* q = Q + lo * m;
        k_split_bf16<<<(unsigned)((c * 32 + 255) / 256), 256, 0, s>>>(q, c, m, m, ms, qh, ql, qn, bound,
                                                                      redo);
        if ((e = cudaGetLastError()) != cudaSuccess) break;
        if ((e = run_items(ix, base_of(ix), qh, ql, qn, c, KP, p.nseg, CONTIGUOUS, keys, bound, s)) !=
            cudaSuccess)
            break;
        // a query tile's lists: a few for large batches, up to one per SM for small ones
#define FG_RERANK(W_, E_)                                                                     \
    k_rerank<W_, E_><<<(unsigned)(W_ == 1 ? (c + 3) / 4 : c), W_ == 1 ? 128 : 32 * W_, 0, s>>>( \
        X, ix->m4, q, m, c, keys, nc, KP, K, qn, ix->xs_max, out_ids + lo * K, out_d + lo * K, redo)
        if (nc <= 32 * 4) FG_RERANK(1, 4);
        else if (nc <= 32 * 16) FG_RERANK(1, 16);
        else if (nc <= 8 * 32 * 16) FG_RERANK(8, 16);
        else FG_RERANK(16, 32);   // up to MAX_KEYS
#undef FG_RERANK
        if ((e = cudaGetLastError()) != cudaSuccess) break;
        // the lists are done with: their buffer takes those of the queries on redo
        const int64_t room = p.chunk * p.nseg;
        int grid = 0;
        if ((e = launch_knn_parts(X, n, ix->m4, q, m, c, KP, redo, keys, room, &grid, s)) != cudaSuccess)
            break;
        k_redo_rank<<<(unsigned)std::min<int64_t>(c, 2 * ix->num_sms), 256, 0, s>>>(
            X, n, ix->m4, q, m, keys, grid, room, KP, K, redo, out_ids + lo * K, out_d + lo * K);
        e = cudaGetLastError();
    }
    cudaFreeAsync(tmp, s);   // in stream order: when the kernels above are done
    return e;
}

// Causal candidates of the graph builder on the tensor cores: for every base
// row i, the K (<= 256) smallest approximate distances to the rows j < i,
// ascending by (distance, id), int64 ids padded with -1.  Eight interleaved
// base segments keep 64 each: with random ids a node's K nearest spread over
// the segments (for K = 256, 32 per segment on average), so the merged lists
// are its K nearest; only the first rows (fewer than 8 x 128 predecessors)
// can lose candidates beyond 64 of one tile.  Distances carry the BF16-split
// error (~1e-5 relative), which candidate selection tolerates.
cudaError_t launch_knn_tc_causal(finger_index* ix, int K, int64_t* out_ids, float* out_d,
                                 cudaStream_t s) {
    const int64_t n = ix->n;
    if (n <= 1) return cudaSuccess;
    cudaError_t e = ensure_split(ix, s);
    if (e != cudaSuccess) return e;
    constexpr int KP = 64, NSEG = 8;
    u64* keys = nullptr;
    if (cudaMallocAsync(&keys, sizeof(u64) * (size_t)n * NSEG * KP, s) != cudaSuccess) {
        e = cudaErrorMemoryAllocation;
        goto done;
    }
    if ((e = run_items(ix, base_of(ix), ix->xs_hi, ix->xs_lo, ix->xnorm2, n, KP, NSEG, CAUSAL, keys,
                       nullptr, s, K)) != cudaSuccess)
        goto done;
    k_merge_topk<<<(unsigned)((n + 3) / 4), 128, 0, s>>>(keys, n, K, out_ids, out_d);
    e = cudaGetLastError();
done:
    if (keys) cudaFreeAsync(keys, s);
    return e;
}

// Exact kNN for 40 < K <= 256 on the tensor cores: interleaved base segments keep 64
// candidates each (rows near one another in the base fall into different
// segments), k_rerank_big merges them, and the queries whose lists may have
// dropped a neighbour are done again by the FP32 kernel; same keys as launch_knn
// either way.  Base rows Xb (n x m4 chunks, norms xn, BF16 parts hi / lo); causal:
// the queries are the base rows and row i sees rows j < i, reported as remap[j].
// Falls back to launch_knn where the base is small or memory for the lists is not
// to be had.  1,000 queries x 100k x 960, K = 100: 75.6 ms with the FP32 kernel, 0.88
// here; the 12.5k rows of the first upper layer of a 200k x 128 graph, 256
// candidates: 13.6 ms and 3.4 (0.8 lists, 1.1 merge, 1.5 the first 500 rows again).
namespace {

cudaError_t knn_big(finger_index* ix, const TcBase& x, const float4* Xb, int m4, const float* Q,
                    int64_t q_stride, int q_m, int64_t nq, int K, const int32_t* remap,
                    int64_t* out_ids, float* out_d, bool causal, cudaStream_t s) {
    const int ms = (x.m + 7) & ~7;
    const int nbt = (int)((x.n + TB - 1) / TB), R = K + 32;
    // queries per round: the lists of one take 8 to 32 KB
    const int64_t chunk = causal ? nq : std::min<int64_t>(nq, 16384);
    const int nqt = (int)((chunk + TQ - 1) / TQ);
    int nseg = 16;
    if (!causal) {   // 16 to 64 segments, the smallest count whose waves are full
        double best = 0;
        for (int S = 16; S <= std::min(nbt, 64); ++S) {
            const int64_t items = (int64_t)nqt * S, G = ix->num_sms;
            const double eff = (double)items / ((items + G - 1) / G * G);
            if (eff > best + 0.002) {
                best = eff;
                nseg = S;
            }
            if (best >= 0.97) break;
        }
    }
    int np = 1;
    while (np < nseg * 64) np <<= 1;
    const size_t smem = 8 * (size_t)(np + nseg + R) + 16 * (size_t)m4;
    __nv_bfloat16 *qh = nullptr, *ql = nullptr;
    float* qn = nullptr;
    u64* keys = nullptr;
    int32_t* redo = nullptr;
    cudaError_t e = cudaSuccess;
    if ((!causal && (cudaMallocAsync(&qh, 2 * (size_t)chunk * ms, s) != cudaSuccess ||
                     cudaMallocAsync(&ql, 2 * (size_t)chunk * ms, s) != cudaSuccess ||
                     cudaMallocAsync(&qn, sizeof(float) * (size_t)chunk, s) != cudaSuccess)) ||
        cudaMallocAsync(&keys, sizeof(u64) * (size_t)chunk * nseg * 64, s) != cudaSuccess ||
        cudaMallocAsync(&redo, sizeof(int32_t) * (size_t)(chunk + 1), s) != cudaSuccess ||
        cudaFuncSetAttribute(k_rerank_big, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
            cudaSuccess) {
        cudaGetLastError();
        e = launch_knn(Xb, x.n, m4, Q, q_stride, q_m, nq, K, causal, remap, out_ids, out_d, s, causal);
        goto done;
    }
    for (int64_t lo = 0; lo < nq && e == cudaSuccess; lo += chunk) {
        const int64_t c = std::min(chunk, nq - lo);
        const float* q = Q + lo * q_stride;
        if (!causal)
            k_split_bf16<<<(unsigned)((c * 32 + 255) / 256), 256, 0, s>>>(q, c, q_m, q_stride, ms, qh,
                                                                          ql, qn);
        if ((e = cudaGetLastError()) != cudaSuccess) break;
        if ((e = cudaMemsetAsync(redo, 0, sizeof(int32_t), s)) != cudaSuccess) break;
        e = run_items(ix, x, causal ? x.hi : qh, causal ? x.lo : ql, causal ? x.xn : qn, c, 64, nseg,
                      causal ? CAUSAL : INTERLEAVED, keys, nullptr, s);
        if (e != cudaSuccess) break;
        k_rerank_big<<<(unsigned)c, 256, smem, s>>>(Xb, m4, q, q_stride, q_m, keys, nseg, np, R, K,
                                                    remap, causal ? x.xn : qn, x.xmax, out_ids + lo * K,
                                                    out_d + lo * K, redo);
        if ((e = cudaGetLastError()) != cudaSuccess) break;
        e = launch_knn(Xb, x.n, m4, q, q_stride, q_m, c, K, causal, remap, out_ids + lo * K,
                       out_d + lo * K, s, causal, redo);
    }
done:
    if (qh) cudaFreeAsync(qh, s);
    if (ql) cudaFreeAsync(ql, s);
    if (qn) cudaFreeAsync(qn, s);
    if (keys) cudaFreeAsync(keys, s);
    if (redo) cudaFreeAsync(redo, s);
    return e;
}

// rows from which the tensor cores serve K > 40: 32 tiles, two per segment (K = 100, FP32 /
// tensor cores: 4,096 x 64, one query 464 / 289 us, 2,000 queries 1,378 / 550; 1,024 x 64 245 /
// 291 and 816 / 379)
constexpr int64_t BIG_MIN_ROWS = 32 * TB;

}  // namespace

cudaError_t launch_knn_big(finger_index* ix, const float* Q, int64_t nq, int K, int64_t* out_ids,
                           float* out_d, cudaStream_t s) {
    const float4* Xb = reinterpret_cast<const float4*>(ix->X);
    // (a captured launch stays a single kernel: no allocation of the base's split)
    if (nq == 0) return cudaSuccess;
    if (ix->n < BIG_MIN_ROWS || capturing(s) || ensure_split(ix, s) != cudaSuccess) {
        cudaGetLastError();
        return launch_knn(Xb, ix->n, ix->m4, Q, ix->m, ix->m, nq, K, false, nullptr, out_ids, out_d, s);
    }
    return knn_big(ix, base_of(ix), Xb, ix->m4, Q, ix->m, ix->m, nq, K, nullptr, out_ids, out_d,
                   false, s);
}

// Candidates of a gathered layer (graph builder's upper levels): row i of X (cnt x m4
// chunks) against the rows j < i, ids remap[j]
cudaError_t launch_knn_layer(finger_index* ix, const float4* X, int64_t cnt, int K,
                             const int32_t* remap, int64_t* out_ids, float* out_d, cudaStream_t s) {
    const float* Xf = reinterpret_cast<const float*>(X);
    const int m = ix->m, ms = (m + 7) & ~7;
    __nv_bfloat16 *hi = nullptr, *lo = nullptr;
    float* xn = nullptr;
    NormMax* xmax = nullptr;
    cudaError_t e;
    if (cnt < BIG_MIN_ROWS || K <= 40 ||
        cudaMallocAsync(&hi, 2 * (size_t)cnt * ms, s) != cudaSuccess ||
        cudaMallocAsync(&lo, 2 * (size_t)cnt * ms, s) != cudaSuccess ||
        cudaMallocAsync(&xmax, sizeof(NormMax), s) != cudaSuccess ||
        cudaMallocAsync(&xn, sizeof(float) * (size_t)cnt, s) != cudaSuccess) {
        cudaGetLastError();
        e = launch_knn(X, cnt, ix->m4, Xf, ix->m_pad, ix->m_pad, cnt, K, true, remap, out_ids, out_d, s,
                       true);
    } else {
        k_split_bf16<<<(unsigned)((cnt * 32 + 255) / 256), 256, 0, s>>>(Xf, cnt, m, ix->m_pad, ms, hi,
                                                                        lo, xn);
        e = cudaGetLastError();
        if (e == cudaSuccess) e = max_norm(xn, cnt, xmax, s);
        if (e == cudaSuccess)
            e = knn_big(ix, {hi, lo, xn, xmax, cnt, m}, X, ix->m4, Xf, ix->m_pad, ix->m_pad, cnt, K, remap,
                        out_ids, out_d, true, s);
    }
    if (hi) cudaFreeAsync(hi, s);
    if (lo) cudaFreeAsync(lo, s);
    if (xn) cudaFreeAsync(xn, s);
    if (xmax) cudaFreeAsync(xmax, s);
    return e;
}

}  // namespace fg
