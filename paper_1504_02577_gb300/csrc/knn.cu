// Panther++ (Sec. 3.3, Algorithm 2): feature vectors theta(v) and exact
// k-nearest neighbours under Euclidean distance.
//
// theta(v) = the D largest counts cnt(v,u), u != v (the counting kernels of
// topk.cu with k = D, counts only).
//
// Nearest neighbours. For query a and candidate b (integer vectors) the
// squared distance is d = |a|^2 + y with y = |b|^2 - 2 a.b; ranking by d is
// ranking by y. y is screened on the tensor cores:
//   A row (query)      = [bf16(a_0..a_{D-1}), 1 x 8, 0 ...]
//   B row (candidate)  = [-2 bf16(b_0..b_{D-1}), p_0 .. p_7, 0 ...]
// where p_i = ((|b|^2 >> 8i) & 255) << 8i are the eight 8-bit pieces of the
// exact squared norm (each exactly representable in BF16). Rows have K = 64
// columns for D <= 56, 128 for D <= 120 and 192 for D <= 128. One tcgen05.mma
// chain (M=128 queries, N=256 candidates, K, FP32 accumulation in TMEM)
// produces y_hat = |b|^2 - 2 a_hat.b_hat directly.
//
// Error bound. With u = 2^-8 (BF16 round to nearest), gamma = K * 2^-22 (K
// additions at a conservative 2^-22 each) and s = a.b <= |a||b|:
//   |y_hat - y| <= [2(2u+u^2) + 2 gamma (1+u)^2] |a||b| + gamma |b|^2
// If every entry of a and of b is <= 256, the BF16 inputs are exact and every
// partial sum is an integer of magnitude at most 2 D 2^16 <= 2^24, so y_hat = y
// exactly.
//
// Selection (two threads per query row of the tile, half of the columns each)
// keeps the k best keys in shared memory: exact pairs insert (y, id); other
// pairs are kept while their lower bound y_hat - E does not exceed the k-th
// key, insert (y_hat + E, id) and are appended to a per-query shortlist.
// Afterwards every kept candidate is re-ranked with exact uint64 arithmetic on
// the integer vectors, so the answer is exact. Candidates (and queries) are
// stored exact rows first, so whole 256-candidate tiles take the fast path:
// the minimum of 32 columns, which comes with the TMEM load.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <math.h>

#include <algorithm>
#include <numeric>

#include "internal.cuh"

panther_status topk_counts_all(panther_ctx* ctx, const panther_index* ix, const panther_paths* p, int D,
                               uint32_t* theta);

namespace {

constexpr int KN_M = 128;          // queries per tile
constexpr int KN_N = 256;          // candidates per tile
constexpr int KN_K = 64;           // columns of one operand block (128 bytes of bf16)
constexpr int KN_INFO = 4;         // candidate-information stages (tiles)
constexpr int KN_MIN_RUN = 4;      // candidate tiles per work item at least
// operand blocks of a row: the entries and the eight pieces of the squared norm
__host__ __device__ constexpr int kn_blocks(int D) { return (D + 8 + KN_K - 1) / KN_K; }
// ring stages of one 32 KB candidate block each: as many as fit next to A
__host__ __device__ constexpr int kn_stages(int kb) { return kb == 1 ? 4 : 3; }
constexpr int KN_KMAX = 32;
constexpr int KN_SCAP = 256;       // shortlist capacity per query
constexpr int KN_SPLIT = 2;        // selection warps per TMEM lane quarter (each takes one column slice)
constexpr int KN_THREADS = 64 + 128 * KN_SPLIT;   // warp 0 TMA, warp 1 MMA, then the selection warps
// >= 2(2u+u^2) + 2 gamma (1+u)^2 and >= gamma for K = 64, 128, 192
__host__ __device__ constexpr float kn_alpha(int kb) { return kb == 1 ? 0.0157f : kb == 2 ? 0.01573f : 0.01576f; }
__host__ __device__ constexpr float kn_beta(int kb) { return kb == 1 ? 1.6e-5f : kb == 2 ? 3.1e-5f : 4.6e-5f; }
constexpr uint32_t MAX_EXACT = 256;

struct VecMeta {
    int64_t n, npad;                 // vertices, padded to a multiple of 256
    int D;
};

// round a uint32 to 8 significant bits, nearest, ties to even (bf16 of an integer)
__device__ __forceinline__ uint32_t round8(uint32_t x) {
    if (x < 256) return x;
    int p = 31 - __clz(x);           // leading bit
    int sh = p - 7;
    uint32_t q = x >> sh, rem = x & ((1u << sh) - 1), half = 1u << (sh - 1);
    if (rem > half || (rem == half && (q & 1))) ++q;
    return q << sh;                  // may carry to 2^(p+1): still 8 significant bits
}

__device__ __forceinline__ uint16_t bf16_bits_of(float f) {   // f exactly representable
    return (uint16_t)(__float_as_uint(f) >> 16);
}

// per-vertex statistics and the exact-row flag: eight lanes per row (coalesced
// sectors and several rows in flight per warp; a thread per row strides by D),
// one maximum per warp
__global__ void __launch_bounds__(256) vec_stats_kernel(const uint32_t* __restrict__ theta, int64_t n, int D,
                                                        uint64_t* __restrict__ norm2, float* __restrict__ nrm,
                                                        uint8_t* __restrict__ exact, int64_t* __restrict__ flag,
                                                        unsigned* __restrict__ maxv) {
    const int sub = threadIdx.x & 7;
    const int64_t nrows = (int64_t)gridDim.x * blockDim.x / 8;
    uint32_t top = 0;
    for (int64_t v = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / 8; __any_sync(0xffffffffu, v < n);
         v += nrows) {
        uint64_t s = 0;
        uint32_t mx = 0;
        if (v < n) {
#pragma unroll 8
            for (int d = sub; d < D; d += 8) {
                const uint32_t x = theta[v * D + d];
                s += (uint64_t)x * x;
                mx = x > mx ? x : mx;
            }
        }
#pragma unroll
        for (int o = 4; o; o >>= 1) {
            s += __shfl_xor_sync(0xffffffffu, s, o);
            mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        }
        top = max(top, mx);
        if (sub == 0 && v < n) {
            norm2[v] = s;
            const float r = sqrtf(__ull2float_ru(s));
            nrm[v] = r * (1.0f + 1.0f / (1 << 21));
            const uint8_t e = mx <= MAX_EXACT;
            exact[v] = e;
            flag[v] = e;
        }
    }
    top = __reduce_max_sync(0xffffffffu, top);
    if ((threadIdx.x & 31) == 0 && top) atomicMax(maxv, top);
}

// position of every vertex: exact rows first (id ascending), then the rest
__global__ void vec_perm_kernel(const uint8_t* __restrict__ exact, const int64_t* __restrict__ exscan, int64_t n,
                                int64_t nexact, int32_t* __restrict__ perm) {
    int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= n) return;
    int64_t p = exact[v] ? exscan[v] : nexact + (v - exscan[v]);
    perm[p] = (int32_t)v;
}

// B rows (candidate role) in permuted order + SoA candidate info: eight lanes
// per row, each writing eight columns as one 16-byte store (1.5M rows of D = 50:
// 961 us with a thread per row, 320 with a warp per row)
__global__ void __launch_bounds__(256) vec_brow_kernel(const uint32_t* __restrict__ theta,
                                                       const uint64_t* __restrict__ norm2,
                                                       const float* __restrict__ nrm,
                                                       const int32_t* __restrict__ perm, VecMeta M,
                                                       uint16_t* __restrict__ B, int32_t* __restrict__ cid,
                                                       float* __restrict__ cnrm, float* __restrict__ cncf) {
    const int64_t p = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / 8;
    const int sub = threadIdx.x & 7, kb = kn_blocks(M.D);
    if (p >= M.npad) return;
    const bool pad = p >= M.n;
    const int32_t v = pad ? -1 : perm[p];
    const uint64_t n2 = pad ? 0 : norm2[v];
    for (int blk = 0; blk < kb; ++blk) {
        uint32_t c[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int d = blk * KN_K + sub * 8 + j;
            c[j] = !pad && d < M.D ? theta[(int64_t)v * M.D + d] : 0u;
        }
        uint32_t out[4];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int d = blk * KN_K + sub * 8 + j;
            float f = -2.0f * (float)round8(c[j]);
            if (pad) f = d == M.D ? 1099511627776.0f : 0.f;   // padding: y = 2^40 for every query, id -1
            else if (d >= M.D) f = d < M.D + 8 ? ldexpf((float)((n2 >> (8 * (d - M.D))) & 255ull), 8 * (d - M.D)) : 0.f;
            const uint32_t b = bf16_bits_of(f);
            out[j / 2] = j & 1 ? out[j / 2] | (b << 16) : b;
        }
        if (B) ((uint4*)(B + (p * kb + blk) * KN_K))[sub] = make_uint4(out[0], out[1], out[2], out[3]);
    }
    if (sub == 0) {
        cid[p] = v;
        cnrm[p] = pad ? 0.f : nrm[v];
        cncf[p] = pad ? 1099511627776.0f : __ull2float_ru(n2);
    }
}

// A rows (query role) for a list of query slots, a warp per row
__global__ void __launch_bounds__(256) vec_arow_kernel(const uint32_t* __restrict__ theta,
                                                       const int32_t* __restrict__ qv, int64_t qpad, int D,
                                                       uint16_t* __restrict__ A) {
    const int64_t s = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31, kb = kn_blocks(D);
    if (s >= qpad) return;                           // warp-uniform
    const int32_t v = qv[s];
    auto col = [&](int d) -> uint32_t {
        float f = 0.f;
        if (v >= 0 && d < D) f = (float)round8(theta[(int64_t)v * D + d]);
        else if (v >= 0 && d < D + 8) f = 1.0f;
        return bf16_bits_of(f);
    };
    for (int blk = 0; blk < kb; ++blk) {
        const int d = blk * KN_K + 2 * lane;
        ((uint32_t*)(A + (s * kb + blk) * KN_K))[lane] = col(d) | (col(d + 1) << 16);
    }
}

// largest norm and squared norm of each candidate tile (a warp per tile): the
// error bound of any of its pairs is at most the one with these
__global__ void __launch_bounds__(256) tile_max_kernel(const int32_t* __restrict__ cid, const float* __restrict__ cnrm,
                                                       const float* __restrict__ cncf, float2* __restrict__ out,
                                                       int64_t ntiles) {
    const int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (t >= ntiles) return;                         // warp-uniform
    float a = 0.f, b = 0.f;
#pragma unroll
    for (int j = 0; j < KN_N / 32; ++j) {
        const int64_t i = t * KN_N + j * 32 + (threadIdx.x & 31);
        if (cid[i] >= 0) {                           // padding has no pairs
            a = fmaxf(a, cnrm[i]);
            b = fmaxf(b, cncf[i]);
        }
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        a = fmaxf(a, __shfl_xor_sync(0xffffffffu, a, o));
        b = fmaxf(b, __shfl_xor_sync(0xffffffffu, b, o));
    }
    if ((threadIdx.x & 31) == 0) out[t] = make_float2(a, b);
}

// out[t] = every id of tile t is padding or an exact row (a warp per tile)
__global__ void __launch_bounds__(256) tile_flags_kernel(const uint8_t* __restrict__ exact,
                                                         const int32_t* __restrict__ ids, int64_t count, int tile,
                                                         uint8_t* __restrict__ out, int64_t ntiles) {
    const int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (t >= ntiles) return;                         // warp-uniform
    bool all = true;
    for (int64_t i = t * tile + (threadIdx.x & 31); i < (t + 1) * tile && i < count; i += 32) {
        const int32_t v = ids[i];
        all &= v < 0 || exact[v] != 0;
    }
    all = __all_sync(0xffffffffu, all);
    if ((threadIdx.x & 31) == 0) out[t] = all ? 1 : 0;
}

// ----------------------------------------------------------- PTX helpers ---
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// wait for a phase that is certain to complete (copies or MMAs already in
// flight), bounded all the same; used only to drain after an abort
__device__ __forceinline__ void mbar_drain(uint32_t bar, uint32_t parity) {
    const long long t0 = clock64();
    while (!mbar_try(bar, parity) && clock64() - t0 < (1ll << 31)) {
    }
}
// bounded wait: about one second of SM clocks, then report and give up
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, uint32_t* status, volatile int* abort_flag) {
    if (mbar_try(bar, parity)) return true;
    long long t0 = clock64();
    while (!mbar_try(bar, parity)) {
        if (*abort_flag) return false;
        if (clock64() - t0 > (1ll << 31)) {
            flag_status(status, ST_TIMEOUT);
            *abort_flag = 1;
            return false;
        }
    }
    return true;
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
            dst),
        "l"(map), "r"(x), "r"(y), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}

// tcgen05 shared-memory descriptor: K-major, 128-byte swizzle, 8-row groups 1024 B apart
__device__ __forceinline__ uint64_t sw128_desc(uint32_t saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFF) >> 4);          // start address
    d |= (uint64_t)(16 >> 4) << 16;                    // leading byte offset (unused for this layout)
    d |= (uint64_t)(1024 >> 4) << 32;                  // stride byte offset
    d |= (uint64_t)1 << 46;                            // descriptor version
    d |= (uint64_t)2 << 61;                            // SWIZZLE_128B
    return d;
}

// kind::f16 instruction descriptor: D f32, A/B bf16, both K-major, N = 256, M = 128
constexpr uint32_t KN_IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(KN_N >> 3) << 17) |
                              ((uint32_t)(KN_M >> 4) << 24);

__device__ __forceinline__ void umma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(KN_IDESC), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void umma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// 32 columns of this thread's TMEM lane into r and the smallest of them as
// floats into m (asynchronous: wait before use). The minimum comes with the
// load: taken by FMNMX instructions it was three quarters of the selection
// warps' work.
__device__ __forceinline__ void tmem_ld32_min_async(uint32_t taddr, uint32_t (&r)[32], float& m) {
    asm volatile(
        "tcgen05.ld.red.sync.aligned.32x32b.x32.min.f32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, %32, [%33];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31]),
          "=f"(m)
        : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
// ties the registers to a point after the wait, so no use is scheduled before it
__device__ __forceinline__ void reg_fence(uint32_t (&r)[32], float& m) {
    asm volatile(""
                 : "+f"(m), "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]),
                   "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]),
                   "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]),
                   "+r"(r[29]), "+r"(r[30]), "+r"(r[31]));
}

// ---------------------------------------------------------- selection ---
// Per query row: the k best keys live in shared memory (ascending by
// (key, id)); only the k-th key and id stay in registers for the fast test.
struct Row {
    float thr;       // key of the k-th entry (+inf until k entries)
    int thr_id;
    int n;           // entries held
    int scount;      // shortlist entries appended
};

struct RowConst {
    int qid;         // query vertex (-1: padding row)
    int self;        // candidate id excluded from the answer (the query itself; -2 across graphs)
    bool exact;
    float anrm;      // kn_alpha * |a| (BF16) or 2 eps |a| (FP32)
    float beta;      // kn_beta (BF16 only)
    float2* list;    // k entries {key, id bits}
    int32_t* sl;     // shortlist
    int* overflow;
    int k;
};

// insert (key, id) (caller checked it beats the k-th entry); out of line: rare
__device__ __noinline__ Row row_insert(Row r, const RowConst& c, float key, int id) {
    int i = r.n < c.k ? r.n : c.k - 1;
    if (r.n < c.k) ++r.n;
    while (i > 0) {
        float2 e = c.list[i - 1];
        int eid = __float_as_int(e.y);
        if (e.x < key || (e.x == key && eid < id)) break;
        c.list[i] = e;
        --i;
    }
    c.list[i] = make_float2(key, __int_as_float(id));
    if (r.n == c.k) {
        float2 last = c.list[c.k - 1];
        r.thr = last.x;
        r.thr_id = __float_as_int(last.y);
    }
    return r;
}

__device__ __forceinline__ Row take_exact(Row r, const RowConst& c, float y, int cid) {
    if (cid < 0 || cid == c.self) return r;
    if (y < r.thr || (y == r.thr && cid < r.thr_id)) r = row_insert(r, c, y, cid);
    return r;
}

// a pair whose screened value carries an error bound E
__device__ __noinline__ Row take_bounded(Row r, const RowConst& c, float y, float E, int cid, bool cexact) {
    if (cid < 0 || cid == c.self) return r;
    if (c.exact && cexact) return take_exact(r, c, y, cid);
    if (__fsub_rd(y, E) > r.thr) return r;
    if (r.scount < KN_SCAP) c.sl[r.scount] = cid; else *c.overflow = 1;
    ++r.scount;
    float ub = __fadd_ru(y, E);
    if (ub < r.thr || (ub == r.thr && cid < r.thr_id)) r = row_insert(r, c, ub, cid);
    return r;
}

// an upper bound of a group's smallest key (SEED), from the smallest of its
// values and the tile's error bound (+inf when it may be padding's, 2^40)
__device__ __forceinline__ float seed_key(float m, float E) {
    return m < 1099511627776.0f ? __fadd_ru(m, E) : __int_as_float(0x7f800000);
}

// One group of 32 screened values y of an exact tile, for the 32 rows of a
// warp (every lane calls it; `live` marks query rows). Exact tiles hold exact
// rows in ascending id order, after every row already in the list, so a
// candidate tied with the k-th key never wins its tie: only y < thr can enter.
// Mostly one row of the warp has one such candidate, so the warp inserts it
// together, lane l holding entry l of the row's list: an insertion by the
// row's own lane is a chain of up to k loads and stores the tile's other warps
// soon wait for, and a call there saves the group's registers. While lists
// fill, most rows have one: with LANES and more than 1 + k/4 such rows (the chain
// costs about 70 cycles a link, the warp's insertion about as much as three, and
// half-full lists have short chains) every lane inserts its own. That costs
// registers (72 bytes spilled
// instead of 36; 100,000 queries against as many vertices 8.4 instead of 6.4 ms),
// so only the form for few candidate tiles has it (FILL below).
template <bool LANES>
__device__ __forceinline__ Row select_exact(Row r, const RowConst& c, const uint32_t (&y)[32], const int32_t* cid,
                                            bool live, float2* warp_lists) {
    const int lane = threadIdx.x & 31;
    int last = -1;
    for (;;) {
        // this row's next column below thr
        float key = 0.f;
        int at = -1;
#pragma unroll
        for (int j = 31; j >= 0; --j)
            if (__uint_as_float(y[j]) < r.thr && j > last) {
                key = __uint_as_float(y[j]);
                at = j;
            }
        unsigned rows = __ballot_sync(0xffffffffu, live && at >= 0);
        if (!rows) return r;
        const int id = at >= 0 ? cid[at] : -1;
        last = at >= 0 ? at : 32;
        rows &= __ballot_sync(0xffffffffu, id >= 0 && id != c.self);
        if (LANES && __popc(rows) > 1 + c.k / 4) {
            if ((rows >> lane) & 1u) {
                float2* list = warp_lists + lane * (KN_SPLIT * KN_KMAX);
                int i = r.n < c.k ? r.n : c.k - 1;   // the entries worse than it move up one
                r.n = i + 1;
                float2 worst = make_float2(key, __int_as_float(id));
#pragma unroll 1
                for (bool top = true; i > 0; --i, top = false) {
                    const float2 e = list[i - 1];
                    if (e.x < key || (e.x == key && __float_as_int(e.y) < id)) break;
                    list[i] = e;
                    worst = top ? e : worst;
                }
                list[i] = make_float2(key, __int_as_float(id));
                if (r.n == c.k) {
                    r.thr = worst.x;
                    r.thr_id = __float_as_int(worst.y);
                }
            }
            __syncwarp();
            continue;
        }
        while (rows) {                               // warp-uniform
            const int l = __ffs(rows) - 1;
            rows &= rows - 1;
            const float nk = __shfl_sync(0xffffffffu, key, l);
            const int ni = __shfl_sync(0xffffffffu, id, l), n = __shfl_sync(0xffffffffu, r.n, l);
            float2* list = warp_lists + l * (KN_SPLIT * KN_KMAX);
            float2 e = make_float2(0.f, 0.f);
            if (lane < n) e = list[lane];
            const bool before = lane < n && (e.x < nk || (e.x == nk && __float_as_int(e.y) < ni));
            const int pos = __popc(__ballot_sync(0xffffffffu, before));
            float2 up;
            up.x = __shfl_up_sync(0xffffffffu, e.x, 1);
            up.y = __shfl_up_sync(0xffffffffu, e.y, 1);
            const int n1 = n < c.k ? n + 1 : n;
            e = lane < pos ? e : lane == pos ? make_float2(nk, __int_as_float(ni)) : up;
            __syncwarp();
            if (lane >= pos && lane < n1) list[lane] = e;
            __syncwarp();
            const float wk = __shfl_sync(0xffffffffu, e.x, c.k - 1);
            const float wi = __shfl_sync(0xffffffffu, e.y, c.k - 1);
            if (lane == l) {
                r.n = n1;
                if (n1 == c.k) {
                    r.thr = wk;
                    r.thr_id = __float_as_int(wi);
                }
            }
        }
    }
}

// one group of 32 screened values y (columns pos0 .. pos0+31) with error bounds
__device__ __forceinline__ Row select_bounded(Row r, const RowConst& c, const uint32_t (&y)[32], const int32_t* cid,
                                              const float* cnrm, const float* cncf, int64_t pos0, int64_t nexact) {
#pragma unroll
    for (int j = 0; j < 32; ++j) {
        const float E = fmaf(c.anrm, cnrm[j], fmaf(c.beta, cncf[j], 1.0f)) * 1.0001f;
        if (__fsub_rd(__uint_as_float(y[j]), E) <= r.thr)
            r = take_bounded(r, c, __uint_as_float(y[j]), E, cid[j], pos0 + j < nexact);
    }
    return r;
}

// The screen's work, query tiles x candidate tiles in query-tile order, is cut
// into G equal runs, one per CTA: a run crosses query tiles and a query tile is
// cut into at most `nseg` segments, each with lists of its own. (Whole query
// tiles per CTA leave SMs idle when their number is a little above a multiple
// of the SM count: 157 tiles on 152 SMs took two waves.) With G = 0 a CTA
// takes whole query tiles in turn (nseg = 1; the FP32 form's own candidate
// ranges are nseg segments of every tile).
struct Split {
    int64_t nqt, nct, G;
    int64_t nseg;
    __host__ __device__ int64_t begin(int64_t g) const { return g * (nqt * nct) / G; }
    __host__ __device__ int64_t owner(int64_t unit) const { return ((unit + 1) * G - 1) / (nqt * nct); }
    __host__ __device__ int64_t first(int64_t qt) const { return G ? owner(qt * nct) : 0; }
    __host__ __device__ int64_t segments(int64_t qt) const {
        return G ? owner((qt + 1) * nct - 1) - owner(qt * nct) + 1 : nseg;
    }
};

// work item j of CTA c: a query tile, its segment and the candidate tiles of it
struct Item {
    int64_t qt, seg, ct0, ct1;
};
__device__ __forceinline__ bool split_item(const Split& W, int64_t c, int64_t grid, int64_t j, Item* it) {
    if (!W.G) {
        it->qt = c + j * grid;
        it->seg = 0;
        it->ct0 = 0;
        it->ct1 = W.nct;
        return it->qt < W.nqt;
    }
    const int64_t u0 = W.begin(c), u1 = W.begin(c + 1);
    if (u0 >= u1) return false;
    const int64_t qt = u0 / W.nct + j;
    const int64_t a = qt * W.nct;
    if (a >= u1) return false;
    it->qt = qt;
    it->seg = c - W.first(qt);
    it->ct0 = u0 > a ? u0 - a : 0;
    it->ct1 = u1 < a + W.nct ? u1 - a : W.nct;
    return true;
}

struct ScreenArgs {
    const int32_t* cid;      // [npad] candidate vertex per position
    const float* cnrm;       // [npad]
    const float* cncf;       // [npad]
    const uint8_t* ctile;    // [npad/256] all-exact flags
    const float2* ctmax;     // [npad/256] largest norm and squared norm
    Split W;                 // nct of it: candidate tiles screened (SEED: of the sample)
    uint32_t seed_step, seed_mul;   // SEED: tile j of the sample is candidate tile (j * mul mod nct) * step
    const float* thr0;       // [qpad] upper bound of the k-th key, or null
    int64_t nexact;          // exact candidate positions
    const int32_t* qv;       // [qpad] query vertex per slot (-1 pad)
    const float* qnrm;       // [qpad]
    const uint8_t* qexact;   // [qpad]
    const uint8_t* qtile;    // [qpad/128] all-exact flags
    int k;
    float2* lists;           // [qpad][nseg][KN_SPLIT][k]
    int32_t* shortlist;      // [qpad][nseg][KN_SPLIT][KN_SCAP]
    int32_t* scount;         // [qpad][nseg][KN_SPLIT]
    float* smin;             // SEED: [qpad][nseg][KN_SPLIT][seed_keys]
    int seed_keys;           // SEED: minima written per segment and column slice: 20, 4 or 1
    int* overflow;           // [qpad]
    uint32_t* status;
    bool exclude_self;       // queries and candidates are the same vertices
    float* dump;             // DUMP form only: y_hat of every pair, [q][npad] by query index
    const int32_t* qidx;     // DUMP form only: query index of each slot
    int64_t npad;
};

// shared memory map (offsets from a 1024-aligned base)
template <int KB>
struct Smem {
    static constexpr int ST = kn_stages(KB);
    static constexpr uint32_t A = 0;                                     // KB x 16 KB
    static constexpr uint32_t B = A + KB * KN_M * KN_K * 2;              // ST x 32 KB
    static constexpr uint32_t INFO = B + ST * KN_N * KN_K * 2;           // KN_INFO x 3 KB
    static constexpr uint32_t LIST = INFO + KN_INFO * KN_N * 12;         // 128 x SPLIT x KMAX x 8 B
    static constexpr uint32_t BAR = LIST + KN_M * KN_SPLIT * KN_KMAX * 8;   // barriers
    static constexpr uint32_t BYTES = BAR + 256 + 1024;
    static_assert(BYTES <= 232448, "shared memory of one CTA");
};

// SCREEN is the k-NN path. DUMP is the measurement form
// (pantherpp_debug_screen): it also writes every screened value y_hat to
// S.dump. SEED screens a sample of the candidate tiles first, in an order
// scattered over them, to bound each query's k-th key from above (S.thr0 of
// the SCREEN launch). Without it a query meets the candidates by ascending id,
// which real ids make a bad order (low ids, high degrees: every candidate is
// nearer than all before it and enters the list). 48 queries against 1M
// vertices: 589 us without the sample and with insertions by single lanes, 10 +
// 74 now; 20,011 against 1.5M: 17.4 ms, 0.13 + 4.16 now (5.7 with single-lane
// insertions, 3.1 with none). Taking all tiles in the scattered order was 18 ms:
// the few candidates that enter then no longer come in the same tiles for many
// rows, and ties at the k-th key enter by id. The sample keeps no
// lists (a new list takes every candidate of its first tiles): only the minima
// of SEED_T * 4 disjoint shares of each segment's column slice, whose
// (k+1)-th smallest over the query bounds its k-th key (one of them may be the
// query itself).
constexpr int SEED_T = 5;
// FILL is the SCREEN form below 16 candidate tiles, where there is no sample and
// filling the lists is the work: 1,000 queries against 1,000 vertices, k = 10,
// 874 us with warp insertions alone, 310 with the lanes' own.
enum { SCREEN = 0, DUMP_FORM = 1, SEED = 2, FILL = 3 };
constexpr int64_t FILL_TILES = 16;

template <int MODE, int KB>
__global__ void __launch_bounds__(KN_THREADS, 1)
    screen_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, ScreenArgs S) {
    constexpr bool DUMP = MODE == DUMP_FORM;
    auto tile_at = [&](int64_t ct) -> int64_t {
        if (MODE != SEED) return ct;
        return (int64_t)((uint64_t)((uint32_t)ct) * S.seed_mul % (uint32_t)S.W.nct) * S.seed_step;
    };
    extern __shared__ uint8_t smraw[];
    const uint32_t raw = smem_u32(smraw);
    const uint32_t base = (raw + 1023) & ~1023u;
    uint8_t* gbase = smraw + (base - raw);
    using SM = Smem<KB>;
    constexpr int ST = SM::ST;
    // barriers: full[ST], empty[ST], tfull[2], tempty[2], ifull, iempty[KN_INFO], afull, aempty, drain
    const uint32_t bar0 = base + SM::BAR;
    auto FULL = [&](int s) { return bar0 + 8 * s; };
    auto EMPTY = [&](int s) { return bar0 + 8 * (ST + s); };
    auto TFULL = [&](int b) { return bar0 + 8 * (2 * ST + b); };
    auto TEMPTY = [&](int b) { return bar0 + 8 * (2 * ST + 2 + b); };
    auto IFULL = [&](int i) { return bar0 + 8 * (2 * ST + 4 + i); };
    auto IEMPTY = [&](int i) { return bar0 + 8 * (2 * ST + 4 + KN_INFO + i); };
    constexpr int NB = 2 * ST + 4 + 2 * KN_INFO;
    const uint32_t AFULL = bar0 + 8 * NB, AEMPTY = AFULL + 8;
    const uint32_t DRAIN = bar0 + 8 * (NB + 2);              // completion of this CTA's MMAs after an abort
    volatile int* abort_flag = (volatile int*)(gbase + SM::BAR + 8 * (NB + 3));
    uint32_t* tmem_slot = (uint32_t*)(gbase + SM::BAR + 8 * (NB + 4));
    static_assert(8 * (NB + 5) <= 256, "barrier area");

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < ST; ++s) {
            mbar_init(FULL(s), 1);
            mbar_init(EMPTY(s), 1);                  // the MMAs that read the block
        }
        for (int i = 0; i < KN_INFO; ++i) {
            mbar_init(IFULL(i), 1);
            mbar_init(IEMPTY(i), 4 * KN_SPLIT);      // the selection warps
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(TFULL(b), 1);
            mbar_init(TEMPTY(b), 4 * KN_SPLIT);
        }
        mbar_init(AFULL, 1);
        mbar_init(AEMPTY, 1);
        mbar_init(DRAIN, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tmem_slot)));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    // what was issued, for the drain after an abort: the parity of the last A
    // load and of the last B load per stage (-1: none), and whether MMAs ran
    int last_a = -1;
    int last_b[ST], last_i[KN_INFO];
    for (int st = 0; st < ST; ++st) last_b[st] = -1;
    for (int i = 0; i < KN_INFO; ++i) last_i[i] = -1;
    bool mma_issued = false;
    if (warp == 0) {
        // ------------------------------------------------ TMA producer ---
        if (lane == 0) {
            uint32_t it = 0, ib = 0;                 // tiles, operand blocks
            int j = 0;
            bool ok = true;
            Item w;
            for (; ok && split_item(S.W, blockIdx.x, gridDim.x, j, &w); ++j) {
                if (!mbar_wait(AEMPTY, (j & 1) ^ 1, S.status, abort_flag)) {
                    ok = false;
                    break;
                }
                mbar_expect_tx(AFULL, KB * KN_M * KN_K * 2);
                for (int blk = 0; blk < KB; ++blk)
                    tma_load_2d(base + SM::A + blk * (KN_M * KN_K * 2), &tmA, blk * KN_K, (int)(w.qt * KN_M), AFULL);
                last_a = j & 1;
                for (int64_t c = w.ct0; c < w.ct1 && ok; ++c, ++it) {
                    const int64_t ct = tile_at(c);
                    const int si = (int)(it % KN_INFO);
                    const uint32_t pi = (it / KN_INFO) & 1;
                    if (!mbar_wait(IEMPTY(si), pi ^ 1, S.status, abort_flag)) { ok = false; break; }
                    mbar_expect_tx(IFULL(si), 3 * KN_N * 4);
                    const uint32_t info = base + SM::INFO + si * (KN_N * 12);
                    bulk_load(info, S.cid + ct * KN_N, KN_N * 4, IFULL(si));
                    bulk_load(info + KN_N * 4, S.cnrm + ct * KN_N, KN_N * 4, IFULL(si));
                    bulk_load(info + KN_N * 8, S.cncf + ct * KN_N, KN_N * 4, IFULL(si));
                    last_i[si] = (int)pi;
                    for (int blk = 0; blk < KB; ++blk, ++ib) {
                        const int s = (int)(ib % ST);
                        const uint32_t ph = (ib / ST) & 1;
                        if (!mbar_wait(EMPTY(s), ph ^ 1, S.status, abort_flag)) { ok = false; break; }
                        mbar_expect_tx(FULL(s), KN_N * KN_K * 2);
                        tma_load_2d(base + SM::B + s * (KN_N * KN_K * 2), &tmB, blk * KN_K, (int)(ct * KN_N), FULL(s));
                        last_b[s] = (int)ph;
                    }
                }
            }
        }
    } else if (warp == 1) {
        // --------------------------------------------------- MMA issuer ---
        if (lane == 0) {
            uint32_t it = 0, ib = 0;
            int j = 0;
            Item w;
            for (; split_item(S.W, blockIdx.x, gridDim.x, j, &w); ++j) {
                if (!mbar_wait(AFULL, j & 1, S.status, abort_flag)) break;
                bool ok = true;
                for (int64_t c = w.ct0; c < w.ct1 && ok; ++c, ++it) {
                    const int b = (int)(it & 1);
                    const uint32_t pb = (it >> 1) & 1;
                    if (!mbar_wait(TEMPTY(b), pb ^ 1, S.status, abort_flag)) {
                        ok = false;
                        break;
                    }
                    for (int blk = 0; blk < KB; ++blk, ++ib) {
                        const int s = (int)(ib % ST);
                        if (!mbar_wait(FULL(s), (ib / ST) & 1, S.status, abort_flag)) {
                            ok = false;
                            break;
                        }
                        tc_fence_after();
                        const uint32_t a0 = base + SM::A + blk * (KN_M * KN_K * 2), b0 = base + SM::B + s * (KN_N * KN_K * 2);
#pragma unroll
                        for (int kk = 0; kk < KN_K / 16; ++kk)
                            umma_bf16(tmem + b * KN_N, sw128_desc(a0 + kk * 32), sw128_desc(b0 + kk * 32),
                                      blk > 0 || kk > 0);
                        umma_commit(EMPTY(s));
                        mma_issued = true;
                    }
                    // the tile's information has landed before the tile is
                    // handed on: selection warps release its stage without
                    // looking at it, and no copy is in flight when the CTA ends
                    if (ok && !mbar_wait(IFULL(it % KN_INFO), (it / KN_INFO) & 1, S.status, abort_flag)) ok = false;
                    if (ok) umma_commit(TFULL(b));
                }
                umma_commit(AEMPTY);
                if (!ok) break;
            }
            // the last commit has arrived before the CTA's shared memory goes
            if (j > 0 && !*abort_flag) mbar_wait(AEMPTY, (j - 1) & 1, S.status, abort_flag);
        }
    } else {
        // --------------------------------------------------- selection ---
        const int quarter = warp & 3;             // TMEM lanes 32*quarter .. +31
        const int half = (warp - 2) >> 2;         // column slice of every tile this warp screens
        const int row = quarter * 32 + lane;
        float2* mylist = (float2*)(gbase + SM::LIST) + (row * KN_SPLIT + half) * KN_KMAX;
        uint32_t it = 0;
        Item w;
        for (int64_t wj = 0; split_item(S.W, blockIdx.x, gridDim.x, wj, &w); ++wj) {
            const int64_t slot = w.qt * KN_M + row;
            // keys up to thr0 (the k-th key is no larger) enter until k are held
            Row r{S.thr0 ? nextafterf(S.thr0[slot], __int_as_float(0x7f800000)) : __int_as_float(0x7f800000),
                  0x7fffffff, 0, 0};
            const int64_t state = (slot * S.W.nseg + w.seg) * KN_SPLIT + half;
            const RowConst rc{S.qv[slot], S.exclude_self ? S.qv[slot] : -2, S.qexact[slot] != 0,
                              kn_alpha(KB) * S.qnrm[slot], kn_beta(KB), mylist,
                              S.shortlist + state * KN_SCAP, S.overflow + slot, S.k};
            const bool qtile_exact = S.qtile[w.qt] != 0;
            float acc[SEED_T * 4];
            int turn = 0;
            if (MODE == SEED)
#pragma unroll
                for (int i = 0; i < SEED_T * 4; ++i) acc[i] = __int_as_float(0x7f800000);
            bool ok = true;
            bool flag = S.ctile[tile_at(w.ct0)] != 0;    // of the coming tile, loaded a tile ahead
            float2 top = S.ctmax[tile_at(w.ct0)];
            for (int64_t c = w.ct0; c < w.ct1; ++c, ++it) {
                const int64_t ct = tile_at(c);
                const int si = (int)(it % KN_INFO);
                const uint32_t pi = (it / KN_INFO) & 1;
                const int b = (int)(it & 1);
                const uint32_t pb = (it >> 1) & 1;
                const bool fast = qtile_exact && flag;
                // at least the error bound of any pair of this row and the tile
                const float E = rc.exact && flag ? 0.f : fmaf(rc.anrm, top.x, fmaf(rc.beta, top.y, 1.0f)) * 1.0001f;
                if (c + 1 < w.ct1) {
                    flag = S.ctile[tile_at(c + 1)] != 0;
                    top = S.ctmax[tile_at(c + 1)];
                }
                if (!__all_sync(0xffffffffu, mbar_wait(TFULL(b), pb, S.status, abort_flag))) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint8_t* info = gbase + SM::INFO + si * (KN_N * 12);
                const int c0 = half * 128;                // 128 columns per selection warp
                const int32_t* cid = (const int32_t*)info + c0;
                const float* cnrm = (const float*)(info + KN_N * 4) + c0;
                const float* cncf = (const float*)(info + KN_N * 8) + c0;
                const uint32_t tbase = tmem + ((uint32_t)(quarter * 32) << 16) + b * KN_N + c0;
                // the candidates' ids and norms of the tile, needed by few tiles
                // (they have landed: the wait makes them visible)
                auto info_ready = [&]() { return mbar_wait(IFULL(si), pi, S.status, abort_flag); };
                // may a pair with a value from v up enter the list? (E = 0: exact
                // pairs, of which a tie with the k-th key does not, as above)
                auto may_enter = [&](float v) { return E == 0.f ? v < r.thr : __fsub_rd(v, E) <= r.thr; };
                uint32_t u[4][32];
                float m[4];
                __syncwarp();
#pragma unroll
                for (int g = 0; g < 4; ++g) tmem_ld32_min_async(tbase + g * 32, u[g], m[g]);
                tmem_wait_ld();
#pragma unroll
                for (int g = 0; g < 4; ++g) reg_fence(u[g], m[g]);
                // the values are in registers: the buffer goes back to the MMA
                // warp now, so that selection overlaps the next tile's MMAs
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(TEMPTY(b));
                if (DUMP && rc.qid >= 0) {
#pragma unroll
                    for (int g = 0; g < 4; ++g) {
                        float* dst = S.dump + (int64_t)S.qidx[slot] * S.npad + ct * KN_N + c0 + g * 32;
#pragma unroll
                        for (int i = 0; i < 32; ++i) dst[i] = __uint_as_float(u[g][i]);
                    }
                }
                if constexpr (MODE == SEED) {
                    float v[4];
#pragma unroll
                    for (int g = 0; g < 4; ++g) v[g] = seed_key(m[g], E);
#pragma unroll
                    for (int i = 0; i < SEED_T * 4; ++i)
                        if (turn == i / 4) acc[i] = fminf(acc[i], v[i & 3]);
                    turn = turn + 1 == SEED_T ? 0 : turn + 1;
                } else if (fast) {                        // warp-uniform
                    const bool live = rc.qid >= 0;
                    const float mt = live ? r.thr : -__int_as_float(0x7f800000);
                    if (__any_sync(0xffffffffu, fminf(fminf(m[0], m[1]), fminf(m[2], m[3])) < mt) &&
                        __all_sync(0xffffffffu, info_ready())) {
#pragma unroll
                        for (int g = 0; g < 4; ++g)
                            if (__any_sync(0xffffffffu, live && m[g] < r.thr))
                                r = select_exact<MODE == FILL>(r, rc, u[g], cid + g * 32, live, mylist - lane * (KN_SPLIT * KN_KMAX));
                    }
                } else if (rc.qid >= 0 && r.scount <= KN_SCAP &&
                           may_enter(fminf(fminf(m[0], m[1]), fminf(m[2], m[3]))) && info_ready()) {
                    // (a row whose shortlist overflowed is brute_force's; few groups hold a pair that the tile's bound cannot rule
                    // out; with a bound per pair one query beyond BF16-exact
                    // values among 20,011 made the call 50 ms instead of 4.9: its
                    // query tile took 15 times as long as the others. 6.4 now.)
#pragma unroll
                    for (int g = 0; g < 4; ++g)
                        if (may_enter(m[g]))
                            r = select_bounded(r, rc, u[g], cid + g * 32, cnrm + g * 32, cncf + g * 32,
                                               ct * KN_N + c0 + g * 32, S.nexact);
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(IEMPTY(si));
            }
            if (!ok) break;
            if constexpr (MODE == SEED) {
                float* out = S.smin + state * S.seed_keys;
                float g4[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    g4[i] = acc[i];
#pragma unroll
                    for (int t = 1; t < SEED_T; ++t) g4[i] = fminf(g4[i], acc[t * 4 + i]);
                }
                if (S.seed_keys == SEED_T * 4) {
#pragma unroll
                    for (int i = 0; i < SEED_T * 4; ++i) out[i] = acc[i];
                } else if (S.seed_keys == 4) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) out[i] = g4[i];
                } else {
                    out[0] = fminf(fminf(g4[0], g4[1]), fminf(g4[2], g4[3]));
                }
            } else {
                for (int i = 0; i < S.k; ++i)
                    S.lists[state * S.k + i] = i < r.n ? mylist[i] : make_float2(0.f, __int_as_float(-1));
                S.scount[state] = r.scount;
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (*abort_flag) {
        // a wait ran out somewhere in the CTA: the copies issued into shared
        // memory land and the MMAs issued complete before the CTA releases
        // TMEM and exits (each drain is bounded too)
        if (warp == 0 && lane == 0) {
            if (last_a >= 0) mbar_drain(AFULL, (uint32_t)last_a);
            for (int st = 0; st < ST; ++st)
                if (last_b[st] >= 0) mbar_drain(FULL(st), (uint32_t)last_b[st]);
            for (int i = 0; i < KN_INFO; ++i)
                if (last_i[i] >= 0) mbar_drain(IFULL(i), (uint32_t)last_i[i]);
        }
        if (warp == 1 && lane == 0 && mma_issued) {
            umma_commit(DRAIN);
            mbar_drain(DRAIN, 0);
        }
        tc_fence_before();
        __syncthreads();
    }
    tc_fence_after();
    if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem));
}

// ------------------------------------------------ FP32 comparison form ---
// One thread per query row, candidates streamed through shared memory in
// tiles of 256; y = |b|^2 - 2 a.b with the dot product in FP32 FMAs. Bound:
// |y_hat - y| <= (D+3) 2^-23 (2|a||b| + |b|^2) + 1.
constexpr int F_T = 128, F_TILE = 32;

// KK: padded vector length, 64 (D <= 64) or 128 (D <= 128)
template <int KK>
__global__ void __launch_bounds__(F_T) fp32_kernel(const uint32_t* __restrict__ theta_q,
                                                   const uint32_t* __restrict__ theta_c, bool exclude_self, int D,
                                                   const int32_t* __restrict__ qv,
                                                   const uint8_t* __restrict__ qexact, const float* __restrict__ qnrm,
                                                   int64_t qpad, int64_t nexact,
                                                   const int32_t* __restrict__ cidv, const float* __restrict__ cnrmv,
                                                   const float* __restrict__ cncfv, int64_t npad, int k,
                                                   float2* __restrict__ lists, int32_t* __restrict__ shortlist,
                                                   int32_t* __restrict__ scount, int* __restrict__ overflow) {
    __shared__ float cb[F_TILE][KK];
    __shared__ float cn2[F_TILE], cnr[F_TILE];
    __shared__ int cidx[F_TILE];
    __shared__ float2 lst[F_T * KN_KMAX];
    const int64_t slot = (int64_t)blockIdx.x * F_T + threadIdx.x;
    // candidate range blockIdx.y of gridDim.y (whole 256-candidate tiles)
    const int64_t nch = gridDim.y, ch = blockIdx.y, nct = npad / 256;
    const int64_t cbeg = ch * nct / nch * 256, cend = (ch + 1) * nct / nch * 256;
    const int64_t state = slot * nch + ch;
    const float epsD = (float)(D + 3) * (1.0f / 8388608.0f);
    const int qid = slot < qpad ? qv[slot] : -1;
    // rows with every entry <= 256 give exact FP32 products and partial sums
    // (all integers below 2^24); other pairs carry the bound
    const bool qex = slot < qpad && qexact[slot] != 0;
    const RowConst rc{qid, exclude_self ? qid : -2, qex, 2.0f * epsD * (slot < qpad ? qnrm[slot] : 0.f), 0.f,
                      lst + threadIdx.x * KN_KMAX, shortlist + (slot < qpad ? state : 0) * KN_SPLIT * KN_SCAP,
                      overflow + (slot < qpad ? slot : 0), k};
    Row r{__int_as_float(0x7f800000), 0x7fffffff, 0, 0};
    float a[KK];
#pragma unroll
    for (int d = 0; d < KK; ++d) a[d] = (qid >= 0 && d < D) ? (float)theta_q[(int64_t)qid * D + d] : 0.f;
    for (int64_t c0 = cbeg; c0 < cend; c0 += F_TILE) {
        __syncthreads();
        for (int i = threadIdx.x; i < F_TILE * KK; i += F_T) {
            int c = i / KK, d = i % KK;
            int32_t v = cidv[c0 + c];
            cb[c][d] = (v >= 0 && d < D) ? (float)theta_c[(int64_t)v * D + d] : 0.f;
        }
        if (threadIdx.x < F_TILE) {
            cidx[threadIdx.x] = cidv[c0 + threadIdx.x];
            cn2[threadIdx.x] = cncfv[c0 + threadIdx.x];
            cnr[threadIdx.x] = cnrmv[c0 + threadIdx.x];
        }
        __syncthreads();
        if (qid < 0) continue;
        for (int c = 0; c < F_TILE; ++c) {
            float s = 0.f;
#pragma unroll
            for (int d = 0; d < KK; ++d) s = fmaf(a[d], cb[c][d], s);
            float y = fmaf(-2.0f, s, cn2[c]);
            float E = (fmaf(rc.anrm, cnr[c], epsD * cn2[c]) + 1.0f) * 1.0001f;
            if (__fsub_rd(y, E) <= r.thr) r = take_bounded(r, rc, y, E, cidx[c], c0 + c < nexact);
        }
    }
    if (slot < qpad) {
        for (int i = 0; i < k; ++i) {
            lists[(state * KN_SPLIT) * k + i] = i < r.n ? rc.list[i] : make_float2(0.f, __int_as_float(-1));
            for (int h = 1; h < KN_SPLIT; ++h) lists[(state * KN_SPLIT + h) * k + i] = make_float2(0.f, __int_as_float(-1));
        }
        scount[state * KN_SPLIT] = r.scount;
        for (int h = 1; h < KN_SPLIT; ++h) scount[state * KN_SPLIT + h] = 0;
    }
}

// ------------------------------------------------------------- rerank ---
// exact squared distance between row a of theta_q and row b of theta_c
__device__ __forceinline__ uint64_t exact_d2(const uint32_t* __restrict__ theta_q, const uint32_t* __restrict__ theta_c,
                                             int D, int32_t a, int32_t b) {
    uint64_t s = 0;
    const uint32_t* x = theta_q + (int64_t)a * D;
    const uint32_t* y = theta_c + (int64_t)b * D;
    auto add = [&](uint32_t p, uint32_t q) {
        const int64_t t = (int64_t)p - (int64_t)q;
        s += (uint64_t)(t * t);
    };
    if ((D & 1) == 0) {                              // rows are 8-byte aligned
        const uint2 *x2 = (const uint2*)x, *y2 = (const uint2*)y;
#pragma unroll 8
        for (int d = 0; d < D / 2; ++d) {
            const uint2 p = __ldg(x2 + d), q = __ldg(y2 + d);
            add(p.x, q.x);
            add(p.y, q.y);
        }
    } else {
#pragma unroll 8
        for (int d = 0; d < D; ++d) add(__ldg(x + d), __ldg(y + d));
    }
    return s;
}

__device__ __forceinline__ bool pair_less(uint64_t d1, int i1, uint64_t d2, int i2) {
    return d1 < d2 || (d1 == d2 && i1 < i2);
}

constexpr int RERANK_ALL = (KN_SPLIT * (KN_KMAX + KN_SCAP) + 31) / 32, RERANK_FEW = 2;

// One warp per (query slot, candidate range): exact distances of every kept
// candidate, top-k of the range. With one range per query the rows go to the
// output; otherwise to part_d2 / part_id ([qpad][nchunk][k]) for chunk_merge.
// PER: candidates held per lane, the first 32 * PER of the query's; a launch
// with PER = 1 leaves the queries that keep more to one with every candidate.
template <int PER>
__global__ void rerank_kernel(const uint32_t* __restrict__ theta_q, const uint32_t* __restrict__ theta_c, int D,
                              const int32_t* __restrict__ qv,
                              const int32_t* __restrict__ qidx, int64_t qpad, Split W, int k,
                              const float2* __restrict__ lists, const int32_t* __restrict__ shortlist,
                              const int32_t* __restrict__ scount, const int* __restrict__ overflow,
                              int32_t* __restrict__ out_ids, uint64_t* __restrict__ out_d2,
                              int32_t* __restrict__ part_id, uint64_t* __restrict__ part_d2) {
    const int64_t grp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    const int64_t nchunk = W.nseg;
    if (grp >= qpad * nchunk) return;
    const int64_t slot = grp / nchunk;
    const int32_t v = qv[slot];
    if (v < 0 || overflow[slot]) return;   // padding, or handled by the brute-force fallback
    if (grp % nchunk >= W.segments(slot / KN_M)) return;   // the tile has fewer segments
    int32_t* oid = nchunk == 1 ? out_ids + (int64_t)qidx[slot] * k : part_id + grp * k;
    uint64_t* od = nchunk == 1 ? out_d2 + (int64_t)qidx[slot] * k : part_d2 + grp * k;
    // candidates: the lists of the column slices, then their shortlists
    int ns[KN_SPLIT];
    int nst = 0;
#pragma unroll
    for (int h = 0; h < KN_SPLIT; ++h) {
        ns[h] = min(scount[grp * KN_SPLIT + h], KN_SCAP);
        nst += ns[h];
    }
    const int nl = KN_SPLIT * k;
    const int total = nl + nst;
    if (PER < RERANK_ALL ? total > 32 * PER : total <= 32 * RERANK_FEW) return;
    uint64_t dd[PER];
    int id[PER];
#pragma unroll
    for (int t = 0; t < PER; ++t) {
        int i = lane + 32 * t;
        id[t] = -1;
        dd[t] = ~0ull;
        if (i < total) {
            int c;
            if (i < nl) {
                c = __float_as_int(lists[grp * nl + i].y);
            } else {
                int j = i - nl, h = 0;
                while (h < KN_SPLIT - 1 && j >= ns[h]) j -= ns[h++];
                c = shortlist[(grp * KN_SPLIT + h) * KN_SCAP + j];
            }
            if (c >= 0) {
                id[t] = c;
                dd[t] = exact_d2(theta_q, theta_c, D, v, c);
            }
        }
    }
    uint64_t lastd = 0;
    int lasti = -1;
    bool first = true;
    for (int r = 0; r < k; ++r) {
        uint64_t bd = ~0ull;
        int bi = 0x7fffffff;
#pragma unroll
        for (int t = 0; t < PER; ++t) {
            if (id[t] < 0) continue;
            bool after = first || pair_less(lastd, lasti, dd[t], id[t]);
            if (after && pair_less(dd[t], id[t], bd, bi)) {
                bd = dd[t];
                bi = id[t];
            }
        }
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            uint64_t od = __shfl_xor_sync(0xffffffffu, bd, o);
            int oi = __shfl_xor_sync(0xffffffffu, bi, o);
            if (pair_less(od, oi, bd, bi)) {
                bd = od;
                bi = oi;
            }
        }
        if (lane == 0) {
            oid[r] = bi == 0x7fffffff ? -1 : bi;
            od[r] = bi == 0x7fffffff ? ~0ull : bd;
        }
        if (bi == 0x7fffffff) {
            for (int rr = r + 1; rr < k && lane == 0; ++rr) {
                oid[rr] = -1;
                od[rr] = ~0ull;
            }
            break;
        }
        lastd = bd;
        lasti = bi;
        first = false;
    }
}

// one CTA per query slot: top-k of the nchunk exact top-k lists of its ranges
// (the ranges are disjoint, so no candidate appears twice)
// With `slots` given, entry i of the lists belongs to query slot slots[i]
// (the brute-force fallback); otherwise to slot i, skipping overflowed slots.
__global__ void __launch_bounds__(256) chunk_merge_kernel(const int32_t* __restrict__ qv,
                                                          const int32_t* __restrict__ qidx,
                                                          const int* __restrict__ overflow,
                                                          const int32_t* __restrict__ slots, int64_t count,
                                                          Split W, int64_t nchunk, int k,
                                                          const int32_t* __restrict__ part_id,
                                                          const uint64_t* __restrict__ part_d2,
                                                          int32_t* __restrict__ out_ids,
                                                          uint64_t* __restrict__ out_d2) {
    __shared__ uint64_t sd[2][8];
    __shared__ int si[2][8];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int HELD = 8;                           // entries kept in registers per thread
    for (int64_t e = blockIdx.x; e < count; e += gridDim.x) {
        const int64_t slot = slots ? slots[e] : e;
        if (qv[slot] < 0 || (!slots && overflow[slot])) continue;
        const int64_t qi = qidx[slot], base = e * nchunk * k;
        const int64_t total = (slots ? nchunk : W.segments(slot / KN_M)) * k;
        uint64_t hd[HELD];
        int hi[HELD];
#pragma unroll
        for (int j = 0; j < HELD; ++j) {
            const int64_t t = threadIdx.x + 256 * j;
            hi[j] = t < total ? part_id[base + t] : -1;
            hd[j] = hi[j] >= 0 ? part_d2[base + t] : ~0ull;
        }
        uint64_t lastd = 0;
        int lasti = -1;
        for (int r = 0; r < k; ++r) {
            uint64_t bd = ~0ull;
            int bi = 0x7fffffff;
            auto offer = [&](uint64_t d, int id) {
                if (id >= 0 && (r == 0 || pair_less(lastd, lasti, d, id)) && pair_less(d, id, bd, bi)) {
                    bd = d;
                    bi = id;
                }
            };
#pragma unroll
            for (int j = 0; j < HELD; ++j) offer(hd[j], hi[j]);
            for (int64_t t = threadIdx.x + 256 * HELD; t < total; t += 256) {
                const int id = part_id[base + t];
                if (id >= 0) offer(part_d2[base + t], id);
            }
#pragma unroll
            for (int o = 16; o; o >>= 1) {
                uint64_t od = __shfl_xor_sync(0xffffffffu, bd, o);
                int oi = __shfl_xor_sync(0xffffffffu, bi, o);
                if (pair_less(od, oi, bd, bi)) {
                    bd = od;
                    bi = oi;
                }
            }
            if (lane == 0) {
                sd[r & 1][warp] = bd;
                si[r & 1][warp] = bi;
            }
            __syncthreads();                          // (two buffers: one barrier a rank)
            bd = sd[r & 1][0];
            bi = si[r & 1][0];
#pragma unroll
            for (int w = 1; w < 8; ++w)
                if (pair_less(sd[r & 1][w], si[r & 1][w], bd, bi)) {
                    bd = sd[r & 1][w];
                    bi = si[r & 1][w];
                }
            if (threadIdx.x == 0) {
                out_ids[qi * k + r] = bi == 0x7fffffff ? -1 : bi;
                out_d2[qi * k + r] = bi == 0x7fffffff ? ~0ull : bd;
            }
            lastd = bd;
            lasti = bi;
        }
        __syncthreads();
    }
}

// the same with a warp per query slot, for at most 256 entries
__global__ void __launch_bounds__(256) chunk_merge_warp_kernel(const int32_t* __restrict__ qv,
                                                               const int32_t* __restrict__ qidx,
                                                               const int* __restrict__ overflow, int64_t qpad, Split W,
                                                               int k, const int32_t* __restrict__ part_id,
                                                               const uint64_t* __restrict__ part_d2,
                                                               int32_t* __restrict__ out_ids,
                                                               uint64_t* __restrict__ out_d2) {
    const int64_t slot = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (slot >= qpad || qv[slot] < 0 || overflow[slot]) return;      // warp-uniform
    const int64_t qi = qidx[slot], base = slot * W.nseg * k;
    const int total = (int)W.segments(slot / KN_M) * k;
    constexpr int HELD = 8;
    uint64_t hd[HELD];
    int hi[HELD];
#pragma unroll
    for (int j = 0; j < HELD; ++j) {
        const int t = lane + 32 * j;
        hi[j] = t < total ? part_id[base + t] : -1;
        hd[j] = hi[j] >= 0 ? part_d2[base + t] : ~0ull;
    }
    for (int r = 0; r < k; ++r) {
        uint64_t bd = ~0ull;
        int bi = 0x7fffffff;
#pragma unroll
        for (int j = 0; j < HELD; ++j)
            if (hi[j] >= 0 && pair_less(hd[j], hi[j], bd, bi)) {
                bd = hd[j];
                bi = hi[j];
            }
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            const uint64_t od = __shfl_xor_sync(0xffffffffu, bd, o);
            const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
            if (pair_less(od, oi, bd, bi)) {
                bd = od;
                bi = oi;
            }
        }
#pragma unroll
        for (int j = 0; j < HELD; ++j) hi[j] = hi[j] == bi ? -1 : hi[j];   // ids are distinct
        if (lane == 0) {
            out_ids[qi * k + r] = bi == 0x7fffffff ? -1 : bi;
            out_d2[qi * k + r] = bi == 0x7fffffff ? ~0ull : bd;
        }
    }
}

// Exact brute force for the queries whose shortlist overflowed, few of them
// (below BRUTE_TILE): the vertex range of each is cut into nparts pieces, one warp each.
// A warp keeps its k best (d2, id) sorted across its lanes (lane l holds rank
// l); a batch of 32 candidates costs one compare and a ballot unless one of
// them beats the k-th entry. The nparts lists go through chunk_merge_kernel.
__global__ void __launch_bounds__(256) brute_warp_kernel(const uint32_t* __restrict__ theta_q,
                                                         const uint32_t* __restrict__ theta_c, bool exclude_self,
                                                         int D, int64_t n,
                                                         const int32_t* __restrict__ qv,
                                                         const int32_t* __restrict__ ovslots, int64_t nov,
                                                         int64_t nparts, int k, int32_t* __restrict__ part_id,
                                                         uint64_t* __restrict__ part_d2) {
    const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (gw >= nov * nparts) return;
    const int64_t oi = gw / nparts, part = gw % nparts;
    const int32_t v = qv[ovslots[oi]];
    const int64_t u0 = part * n / nparts, u1 = (part + 1) * n / nparts;
    uint64_t ld = ~0ull;   // this lane's rank of the list
    int li = 0x7fffffff;
    for (int64_t base = u0; base < u1; base += 32) {
        const int64_t u = base + lane;
        uint64_t d = ~0ull;
        const bool cand = u < u1 && (!exclude_self || u != v);
        if (cand) d = exact_d2(theta_q, theta_c, D, v, (int32_t)u);
        const uint64_t td = __shfl_sync(0xffffffffu, ld, k - 1);
        const int ti = __shfl_sync(0xffffffffu, li, k - 1);
        unsigned pass = __ballot_sync(0xffffffffu, cand && pair_less(d, (int)u, td, ti));
        while (pass) {
            const int src = __ffs(pass) - 1;
            pass &= pass - 1;
            const uint64_t nd = __shfl_sync(0xffffffffu, d, src);
            const int ni = (int)__shfl_sync(0xffffffffu, (int)u, src);
            // entries at or after the insertion point move up one lane
            const bool after = pair_less(nd, ni, ld, li);
            const unsigned am = __ballot_sync(0xffffffffu, after);
            const uint64_t upd = __shfl_up_sync(0xffffffffu, ld, 1);
            const int upi = __shfl_up_sync(0xffffffffu, li, 1);
            if (am) {
                const int pos = __ffs(am) - 1;
                if (lane == pos) {
                    ld = nd;
                    li = ni;
                } else if (lane > pos) {
                    ld = upd;
                    li = upi;
                }
            }
            // candidates of this batch that no longer beat the k-th entry drop out
            const uint64_t td2 = __shfl_sync(0xffffffffu, ld, k - 1);
            const int ti2 = __shfl_sync(0xffffffffu, li, k - 1);
            pass &= __ballot_sync(0xffffffffu, pair_less(d, (int)u, td2, ti2));
        }
    }
    if (lane < k) {
        part_id[gw * k + lane] = li == 0x7fffffff ? -1 : li;
        part_d2[gw * k + lane] = ld;
    }
}

// The same for many queries: a thread per query, its row in registers, the
// candidates of range blockIdx.y through shared memory, four dot products at a
// time. Entries are non-negative, so d2 <= |a|^2 + |b|^2; while that is below
// 2^32 the distance is exact in 32-bit arithmetic modulo 2^32 whatever the
// entries. Other pairs are computed in 64 bits unless the norms alone,
// (|a| - |b|)^2 <= d2, keep them from the list. A network whose counts are
// mostly beyond BF16-exact values sends most of its queries here (all of 20,000,
// D = 57, k = 10, R = 4e7, whole call: 31.5 ms with a warp per query and range,
// 6.3 with this); the warp form reads every candidate row once per query.
// A CTA costs the same for 1 and 128 queries, and its lists more the longer they
// are: with k = 10 about what the warp form takes for 10 to 20 queries at
// n = 200,000 (D = 128, 30 queries: 1.5 ms against 0.4) and for 60 to 130 at
// n = 20,000, with k = 32 for 30 to 50 and for more than 160.
constexpr int BT_T = 128, BT_C = 32;
constexpr int64_t BRUTE_TILE = int64_t(1) << 18;      // queries x candidates / k from which it is taken
template <int KK>
struct BruteSmem {
    uint32_t row[BT_C][KK];
    uint64_t n2[BT_C];
    float nrm[BT_C];
    int id[BT_C];                      // -1: none
    uint64_t ld[KN_KMAX][BT_T];        // the queries' lists, entry by entry
    int li[KN_KMAX][BT_T];
};

template <int KK>
__global__ void __launch_bounds__(BT_T) brute_tile_kernel(const uint32_t* __restrict__ theta_q,
                                                          const uint64_t* __restrict__ norm2_q,
                                                          const float* __restrict__ nrm_q,
                                                          const uint32_t* __restrict__ theta_c,
                                                          const uint64_t* __restrict__ norm2_c,
                                                          const float* __restrict__ nrm_c, bool exclude_self, int D,
                                                          int64_t n, const int32_t* __restrict__ qv,
                                                          const int32_t* __restrict__ ovslots, int64_t nov, int k,
                                                          int32_t* __restrict__ part_id,
                                                          uint64_t* __restrict__ part_d2) {
    extern __shared__ __align__(16) uint8_t bsm[];
    BruteSmem<KK>& S = *(BruteSmem<KK>*)bsm;
    const int t = threadIdx.x;
    const int64_t q = (int64_t)blockIdx.x * BT_T + t, nparts = gridDim.y, part = blockIdx.y;
    const int64_t u0 = part * n / nparts, u1 = (part + 1) * n / nparts;
    const bool live = q < nov;
    const int32_t v = live ? qv[ovslots[q]] : -1;
    uint32_t a[KK];
#pragma unroll
    for (int d = 0; d < KK; ++d) a[d] = live && d < D ? theta_q[(int64_t)v * D + d] : 0u;
    const uint64_t na2 = live ? norm2_q[v] : 0;
    const float na = live ? nrm_q[v] : 0.f;
    int held = 0;
    uint64_t thr = ~0ull;              // the k-th entry (held == k)
    int thr_id = 0x7fffffff;
    for (int64_t c0 = u0; c0 < u1; c0 += BT_C) {
        __syncthreads();
        const int cnt = (int)(u1 - c0 < BT_C ? u1 - c0 : BT_C);
        for (int i = t; i < BT_C * KK; i += BT_T) {
            const int c = i / KK, d = i % KK;
            S.row[c][d] = c < cnt && d < D ? theta_c[(c0 + c) * D + d] : 0u;
        }
        if (t < BT_C) {
            S.id[t] = t < cnt ? (int)(c0 + t) : -1;
            S.n2[t] = t < cnt ? norm2_c[c0 + t] : 0;
            S.nrm[t] = t < cnt ? nrm_c[c0 + t] : 0.f;
        }
        __syncthreads();
        if (!live) continue;
        for (int c = 0; c < BT_C; c += 4) {
            uint32_t dot[4] = {0, 0, 0, 0};
#pragma unroll
            for (int d = 0; d < KK; d += 4)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const uint4 b = *(const uint4*)&S.row[c + j][d];
                    dot[j] += a[d] * b.x + a[d + 1] * b.y + a[d + 2] * b.z + a[d + 3] * b.w;
                }
#pragma unroll 1
            for (int j = 0; j < 4; ++j) {
                const int u = S.id[c + j];
                if (u < 0 || (exclude_self && u == v)) continue;
                const uint64_t nb2 = S.n2[c + j], sum = na2 + nb2;
                const uint32_t dj = j == 0 ? dot[0] : j == 1 ? dot[1] : j == 2 ? dot[2] : dot[3];
                uint64_t d2;
                if ((na2 | nb2 | sum) >> 32) {       // (sum alone may wrap)
                    const float gap = fabsf(na - S.nrm[c + j]) - 1e-6f * (na + S.nrm[c + j]);
                    if (gap > 0.f && __fmul_rd(gap, gap) > __ull2float_ru(thr)) continue;
                    d2 = exact_d2(theta_q, theta_c, D, v, u);
                } else {
                    d2 = (uint32_t)sum - 2u * dj;
                }
                if (!pair_less(d2, u, thr, thr_id)) continue;
                int i = held < k ? held : k - 1;
                held = i + 1;
                for (; i > 0; --i) {
                    const uint64_t ed = S.ld[i - 1][t];
                    const int ei = S.li[i - 1][t];
                    if (pair_less(ed, ei, d2, u)) break;
                    S.ld[i][t] = ed;
                    S.li[i][t] = ei;
                }
                S.ld[i][t] = d2;
                S.li[i][t] = u;
                if (held == k) {
                    thr = S.ld[k - 1][t];
                    thr_id = S.li[k - 1][t];
                }
            }
        }
    }
    if (live)
        for (int i = 0; i < k; ++i) {
            part_id[(q * nparts + part) * k + i] = i < held ? S.li[i][t] : -1;
            part_d2[(q * nparts + part) * k + i] = i < held ? S.ld[i][t] : ~0ull;
        }
}

// query slots: exact queries first (stable), padded to a multiple of 128.
// exscan = exclusive scan of the queries' exact flags (an out-of-range query
// counts as exact); the number of exact queries is read off its last entry, so
// the host does not wait for it. Also each slot's query information.
struct QuerySlots {
    int32_t* qv;             // [qpad] query vertex (-1: padding or not a vertex)
    int32_t* qidx;           // [qpad] query index
    uint8_t* qexact;         // [qpad]
    float* qnrm;             // [qpad]
    int* overflow;           // [qpad], cleared
    unsigned long long* sums;   // [0] kept pairs, [1] overflowed queries, cleared
};

__device__ __forceinline__ bool exact_query(int32_t v, const uint8_t* exact, int64_t n) {
    return v < 0 || v >= n || exact[v] != 0;
}

__device__ __forceinline__ void put_slot(const QuerySlots& Q, int64_t p, int32_t v, int32_t i, bool bad,
                                         const uint8_t* exact, const float* nrm) {
    Q.qv[p] = bad ? -1 : v;
    Q.qidx[p] = i;
    Q.qexact[p] = bad ? 1 : exact[v];
    Q.qnrm[p] = bad ? 0.f : nrm[v];
}

__global__ void query_slots_kernel(const int32_t* __restrict__ queries, int64_t q, int64_t qpad,
                                   const uint8_t* __restrict__ exact, const float* __restrict__ nrm, int64_t n,
                                   const int64_t* __restrict__ exscan, QuerySlots Q, uint32_t* status) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= qpad) return;
    Q.overflow[i] = 0;
    if (i < 2) Q.sums[i] = 0;
    if (i >= q) {
        put_slot(Q, i, -1, 0, true, exact, nrm);
        return;
    }
    const int32_t lastv = queries ? queries[q - 1] : (int32_t)(q - 1);
    const int64_t nexq = exscan[q - 1] + (exact_query(lastv, exact, n) ? 1 : 0);
    const int32_t v = queries ? queries[i] : (int32_t)i;
    const bool bad = v < 0 || v >= n;
    if (bad) flag_status(status, ST_BAD_QUERY);
    const int64_t p = exact_query(v, exact, n) ? exscan[i] : nexq + (i - exscan[i]);
    put_slot(Q, p, v, (int32_t)i, bad, exact, nrm);
}

__global__ void exact_flags_of_queries(const int32_t* __restrict__ queries, int64_t q, const uint8_t* __restrict__ exact,
                                       int64_t n, int64_t* __restrict__ f) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= q) return;
    f[i] = exact_query(queries ? queries[i] : (int32_t)i, exact, n) ? 1 : 0;
}

// the same for up to SLOTS_SMALL queries, flags, scan, slots and tile flags in
// one CTA instead of seven launches
constexpr int SLOTS_SMALL = 4096;
__global__ void __launch_bounds__(1024) query_slots_small_kernel(const int32_t* __restrict__ queries, int q, int qpad,
                                                                 const uint8_t* __restrict__ exact,
                                                                 const float* __restrict__ nrm, int64_t n,
                                                                 QuerySlots Q, uint8_t* __restrict__ qtile,
                                                                 uint32_t* status) {
    __shared__ int wsum[32];
    constexpr int PER = SLOTS_SMALL / 1024;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    int32_t v[PER];
    bool ex[PER];
    int mine = 0;
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const int i = t * PER + j;
        v[j] = i < q ? queries[i] : -1;
        ex[j] = i < q && exact_query(v[j], exact, n);
        mine += ex[j] ? 1 : 0;
    }
    int inc = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) wsum[w] = inc;
    for (int i = t; i < qpad; i += 1024) Q.overflow[i] = 0;
    for (int i = t; i < qpad / KN_M; i += 1024) qtile[i] = 1;
    if (t < 2) Q.sums[t] = 0;
    __syncthreads();
    int before = inc - mine, nexq = 0;
    for (int i = 0; i < 32; ++i) {
        before += i < w ? wsum[i] : 0;
        nexq += wsum[i];
    }
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const int i = t * PER + j;
        if (i < q) {
            const bool bad = v[j] < 0 || v[j] >= n;
            if (bad) flag_status(status, ST_BAD_QUERY);
            const int p = ex[j] ? before : nexq + (i - before);
            put_slot(Q, p, v[j], i, bad, exact, nrm);
            if (!ex[j]) qtile[p / KN_M] = 0;
            before += ex[j] ? 1 : 0;
        }
    }
    for (int i = q + t; i < qpad; i += 1024) put_slot(Q, i, -1, 0, true, exact, nrm);
}

// thr0[slot] = the (k+1)-th smallest of the slot's sample minima (of disjoint
// candidate sets; at most one is the query itself), +inf when there are fewer:
// an upper bound of the k-th key over all candidates. A warp per slot, at most
// 512 minima (seed_keys per segment and column slice).
__global__ void __launch_bounds__(256) seed_bound_kernel(const float* __restrict__ smin, int64_t qpad, Split W,
                                                         int seed_keys, int k, float* __restrict__ thr0) {
    const int64_t slot = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (slot >= qpad) return;                        // warp-uniform
    constexpr int PER = 16;
    const int total = (int)W.segments(slot / KN_M) * KN_SPLIT * seed_keys;
    const float* mine = smin + slot * W.nseg * KN_SPLIT * seed_keys;
    const float inf = __int_as_float(0x7f800000);
    float key[PER];
#pragma unroll
    for (int j = 0; j < PER; ++j) key[j] = lane + 32 * j < total ? mine[lane + 32 * j] : inf;
    // k+1 times the smallest; equal ones count one by one (the lowest lane that
    // holds it drops one)
    float best = inf;
    for (int r = 0; r <= k; ++r) {
        float m = inf;
#pragma unroll
        for (int j = 0; j < PER; ++j) m = fminf(m, key[j]);
        best = m;
#pragma unroll
        for (int o = 16; o; o >>= 1) best = fminf(best, __shfl_xor_sync(0xffffffffu, best, o));
        if (best == inf) break;                      // warp-uniform
        const unsigned have = __ballot_sync(0xffffffffu, m == best);
        if (lane == __ffs(have) - 1) {
            bool gone = false;
#pragma unroll
            for (int j = 0; j < PER; ++j)
                if (!gone && key[j] == best) {
                    key[j] = inf;
                    gone = true;
                }
        }
    }
    if (lane == 0) thr0[slot] = best;
}

// kept pairs and overflowed slots of a call (their order does not matter)
__global__ void knn_sums_kernel(const int32_t* __restrict__ scount, int64_t nstate, const int* __restrict__ overflow,
                                int64_t qpad, unsigned long long* __restrict__ sums, int32_t* __restrict__ ovslots) {
    unsigned long long kept = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nstate; i += (int64_t)gridDim.x * blockDim.x) {
        kept += (unsigned)scount[i];
        if (i < qpad && overflow[i]) ovslots[atomicAdd(&sums[1], 1ull)] = (int32_t)i;
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) kept += __shfl_xor_sync(0xffffffffu, kept, o);
    if ((threadIdx.x & 31) == 0 && kept) atomicAdd(&sums[0], kept);
}

}  // namespace

// ---------------------------------------------------------------- host ---
static PFN_cuTensorMapEncodeTiled_v12000 encode_fn(panther_ctx* ctx) {
    // looked up once (thread-safe static initialisation: serving workers race here)
    static const PFN_cuTensorMapEncodeTiled_v12000 fn = []() -> PFN_cuTensorMapEncodeTiled_v12000 {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            return (PFN_cuTensorMapEncodeTiled_v12000)p;
        return nullptr;
    }();
    if (!fn) set_err(ctx, PANTHER_ECUDA, "cuTensorMapEncodeTiled is not available");
    return fn;
}

static bool make_map(panther_ctx* ctx, CUtensorMap* m, const void* base, int64_t rows, int box_rows, int kb) {
    auto fn = encode_fn(ctx);
    if (!fn) return false;
    cuuint64_t dims[2] = {(cuuint64_t)KN_K * kb, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)KN_K * kb * 2};
    cuuint32_t box[2] = {(cuuint32_t)KN_K, (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        set_err(ctx, PANTHER_ECUDA, "cuTensorMapEncodeTiled failed (%d)", (int)r);
        return false;
    }
    return true;
}

extern "C" panther_status pantherpp_vectors(panther_ctx* ctx, const panther_index* ix, const panther_paths* p, int D,
                                            pantherpp_vecs** out) {
    if (!ctx || !ix || !p || !out) return PANTHER_EINVAL;
    *out = nullptr;
    if (D < 1 || D > 128) return set_err(ctx, PANTHER_EINVAL, "D must be in [1, 128]");
    if (ix->n != p->n || ix->R != p->R)
        return set_err(ctx, PANTHER_EINVAL, "index and paths do not belong together");
    cudaSetDevice(ctx->device);
    cudaStream_t s = ctx->stream;
    const int64_t n = ix->n;
    pantherpp_vecs* v = new pantherpp_vecs();
    v->ctx = ctx;
    v->n = n;
    v->D = D;
    panther_status st;
    int64_t* flag = nullptr;
    unsigned* maxv = nullptr;
    auto fail = [&](panther_status x) {
        dev_free(ctx, flag);
        dev_free(ctx, maxv);
        pantherpp_free_vecs(v);
        return x;
    };
    if ((st = dev_alloc(ctx, (void**)&v->theta, sizeof(uint32_t) * n * D))) return fail(st);
    if ((st = topk_counts_all(ctx, ix, p, D, v->theta))) return fail(st);
    if ((st = dev_alloc(ctx, (void**)&v->norm2, sizeof(uint64_t) * n)) ||
        (st = dev_alloc(ctx, (void**)&v->nrm, sizeof(float) * n)) ||
        (st = dev_alloc(ctx, (void**)&v->exact, n)) || (st = dev_alloc(ctx, (void**)&flag, sizeof(int64_t) * n)) ||
        (st = dev_alloc(ctx, (void**)&maxv, 4)))
        return fail(st);
    PCK(ctx, cudaMemsetAsync(maxv, 0, 4, s));
    unsigned gb = (unsigned)ceil_div(n, 256);
    vec_stats_kernel<<<(unsigned)std::min<int64_t>(ceil_div(n, 32), (int64_t)ctx->num_sms * 16), 256, 0, s>>>(v->theta, n, D, v->norm2, v->nrm, v->exact, flag, maxv);
    ctx->launches++;
    // number of exact rows = sum of flags (read before the scan overwrites them)
    if ((st = scan_exclusive_i64(ctx, flag, n))) return fail(st);
    int64_t last_scan = 0;
    uint8_t last_flag = 0;
    unsigned hmax = 0;
    PCK(ctx, cudaMemcpyAsync(&last_scan, flag + n - 1, 8, cudaMemcpyDeviceToHost, s));
    PCK(ctx, cudaMemcpyAsync(&last_flag, v->exact + n - 1, 1, cudaMemcpyDeviceToHost, s));
    PCK(ctx, cudaMemcpyAsync(&hmax, maxv, 4, cudaMemcpyDeviceToHost, s));
    PCK(ctx, cudaStreamSynchronize(s));
    v->max_val = hmax;
    if ((unsigned __int128)hmax * hmax * (unsigned)D >= ((unsigned __int128)1 << 64))
        return fail(set_err(ctx, PANTHER_EOVERFLOW, "max count^2 * D reaches 2^64: squared distances could overflow"));
    pantherpp_vecs& x = *v;
    x.nexact = last_scan + last_flag;
    x.npad = ceil_div(n, KN_N) * KN_N;
    int32_t* perm = nullptr;
    // Without memory for the operand rows of wide vectors (256 or 384 bytes per
    // vertex) k-NN takes the FP32 form, which reads theta alone.
    st = dev_alloc(ctx, (void**)&x.B, (size_t)x.npad * kn_blocks(D) * KN_K * 2);
    if (st && (st != PANTHER_ENOMEM || kn_blocks(D) == 1)) return fail(st);
    if ((st = dev_alloc(ctx, (void**)&perm, sizeof(int32_t) * x.npad)) ||
        (st = dev_alloc(ctx, (void**)&x.cid, sizeof(int32_t) * x.npad)) ||
        (st = dev_alloc(ctx, (void**)&x.cnrm, sizeof(float) * x.npad)) ||
        (st = dev_alloc(ctx, (void**)&x.cncf, sizeof(float) * x.npad)) ||
        (st = dev_alloc(ctx, (void**)&x.ctile, x.npad / KN_N)) ||
        (st = dev_alloc(ctx, (void**)&x.ctmax, sizeof(float2) * (x.npad / KN_N)))) {
        dev_free(ctx, perm);
        return fail(st);
    }
    vec_perm_kernel<<<gb, 256, 0, s>>>(v->exact, flag, n, x.nexact, perm);
    vec_brow_kernel<<<(unsigned)ceil_div(x.npad, 32), 256, 0, s>>>(v->theta, v->norm2, v->nrm, perm,
                                                                    VecMeta{n, x.npad, D}, x.B, x.cid,
                                                                    x.cnrm, x.cncf);
    tile_flags_kernel<<<(unsigned)ceil_div(x.npad / KN_N, 8), 256, 0, s>>>(v->exact, x.cid, x.npad, KN_N, x.ctile,
                                                                             x.npad / KN_N);
    tile_max_kernel<<<(unsigned)ceil_div(x.npad / KN_N, 8), 256, 0, s>>>(x.cid, x.cnrm, x.cncf, x.ctmax, x.npad / KN_N);
    ctx->launches += 4;
    dev_free(ctx, perm);
    dev_free(ctx, flag);
    dev_free(ctx, maxv);
    flag = nullptr;
    maxv = nullptr;
    cudaError_t ce = cudaStreamSynchronize(s);
    if (ce) return fail(cuda_err(ctx, ce, "vector preparation"));
    *out = v;
    return PANTHER_OK;
}

// The BF16 screen's work in equal runs, one per CTA, of at least KN_MIN_RUN
// candidate tiles or a whole query tile. From 16 query tiles per SM on, whole tiles per CTA: the last
// wave then costs at most 6%, and every segment more of a tile costs lists and
// a shortlist of 2 KB per query.
static Split knn_split(int64_t nqt, int64_t nct, int num_sms) {
    Split W{nqt, nct, 0, 1};
    if (nqt >= 16 * (int64_t)num_sms) return W;
    W.G = std::min<int64_t>(num_sms, std::max(nqt, nqt * nct / KN_MIN_RUN));
    for (int64_t t = 0; t < nqt; ++t) W.nseg = std::max(W.nseg, W.segments(t));
    return W;
}

// The FP32 form's candidate ranges: with fewer query tiles than SMs the choice
// minimises waves x range length, at least KN_MIN_RUN candidate tiles per range.
static Split knn_ranges(int64_t nqt, int64_t nct, int num_sms) {
    Split W{nqt, nct, 0, 1};
    if (nqt >= num_sms) return W;
    const int64_t pmax = std::max<int64_t>(1, std::min<int64_t>(nct / KN_MIN_RUN, 256));
    double best_cost = (double)ceil_div(nqt, num_sms);
    for (int64_t p = 2; p <= pmax; ++p) {
        const double cost = (double)ceil_div(nqt * p, num_sms) / (double)p;
        if (cost < best_cost * 0.999) {
            W.nseg = p;
            best_cost = cost;
        }
    }
    return W;
}

// Candidate tiles of the sample that bounds the k-th keys (0: none): a 32nd of
// the candidate tiles, a 16th of fewer than 2,048, an eighth of fewer than 128
// but at least five (eight minima a tile; a bound for k = 32 needs 33). Below 16
// tiles the sample would be as long as the screen. (32,000 queries against as
// many vertices, 125 tiles, k = 10: 5.3 ms without a sample, 1.4 with one.
// A 16th instead of an eighth leaves k = 32 without a bound at 16,000 vertices,
// 4.8 ms instead of 2.0.)
static int64_t seed_tiles(int64_t nct) {
    if (nct < FILL_TILES) return 0;
    if (nct < 128) return std::max<int64_t>(5, nct / 8);
    return nct / (nct < 2048 ? 16 : 32);
}

template <int MODE, int KB>
static panther_status launch_screen(panther_ctx* ctx, unsigned grid, const CUtensorMap& tmA, const CUtensorMap& tmB,
                                    const ScreenArgs& S) {
    PCK(ctx, cudaFuncSetAttribute(screen_kernel<MODE, KB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)Smem<KB>::BYTES));
    screen_kernel<MODE, KB><<<grid, KN_THREADS, Smem<KB>::BYTES, ctx->stream>>>(tmA, tmB, S);
    PLAUNCH(ctx);
    return PANTHER_OK;
}

template <int KK>
static panther_status launch_brute(panther_ctx* ctx, const pantherpp_vecs* vq, const pantherpp_vecs* vc, bool same,
                                   const int32_t* qv, const int32_t* ovslots, int64_t over, int64_t nparts, int k,
                                   int32_t* part_id, uint64_t* part_d2) {
    constexpr int smem = (int)sizeof(BruteSmem<KK>);
    PCK(ctx, cudaFuncSetAttribute(brute_tile_kernel<KK>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    brute_tile_kernel<KK><<<dim3((unsigned)ceil_div(over, BT_T), (unsigned)nparts), BT_T, smem, ctx->stream>>>(
        vq->theta, vq->norm2, vq->nrm, vc->theta, vc->norm2, vc->nrm, same, vq->D, vc->n, qv, ovslots, over, k, part_id,
        part_d2);
    PLAUNCH(ctx);
    return PANTHER_OK;
}

// queries are vertices of vq, candidates every vertex of vc; `same` excludes
// the candidate with the query's id (one graph: the query itself)
static panther_status knn_run(panther_ctx* ctx, const pantherpp_vecs* vq, const pantherpp_vecs* vc, bool same,
                              const int32_t* queries, int64_t q, int k, int32_t* ids, uint64_t* d2, bool fp32,
                              float* dump = nullptr) {
    const pantherpp_vecs& x = *vc;
    if (!x.B) fp32 = true;
    const pantherpp_vecs* v = vq;
    cudaStream_t s = ctx->stream;
    const int64_t n = vq->n;
    const int64_t qpad = ceil_div(q, KN_M) * KN_M, nqt = qpad / KN_M, nct = x.npad / KN_N;
    const Split W = fp32 ? knn_ranges(nqt, nct, ctx->num_sms) : knn_split(nqt, nct, ctx->num_sms);
    const int64_t nch = W.nseg;
    const int64_t ns = (fp32 || dump) ? 0 : seed_tiles(nct);
    const Split WS = ns ? knn_split(nqt, ns, ctx->num_sms) : W;
    // minima per segment and column slice: at most 512 a query, at least 40
    const int seed_keys = WS.nseg <= 12 ? SEED_T * 4 : WS.nseg <= 64 ? 4 : 1;
    panther_status st;
    int64_t* qf = nullptr;
    int32_t *sl = nullptr, *sc = nullptr, *pid = nullptr, *ovs = nullptr;
    uint8_t* qtile = nullptr;
    float2* lists = nullptr;
    float *smin = nullptr, *thr0 = nullptr;
    uint16_t* A = nullptr;
    uint64_t* pd = nullptr;
    QuerySlots Q{};
    auto cleanup = [&]() {
        dev_free(ctx, qf); dev_free(ctx, Q.qv); dev_free(ctx, Q.qidx); dev_free(ctx, sl); dev_free(ctx, sc);
        dev_free(ctx, Q.overflow); dev_free(ctx, Q.qexact); dev_free(ctx, qtile); dev_free(ctx, Q.qnrm);
        dev_free(ctx, lists); dev_free(ctx, smin); dev_free(ctx, thr0); dev_free(ctx, A); dev_free(ctx, pid);
        dev_free(ctx, pd); dev_free(ctx, ovs); dev_free(ctx, Q.sums);
    };
    const int64_t nstate = qpad * nch * KN_SPLIT;
    const bool small = q <= SLOTS_SMALL && queries;
    if ((!small && (st = dev_alloc(ctx, (void**)&qf, sizeof(int64_t) * q))) ||
        (st = dev_alloc(ctx, (void**)&Q.qv, sizeof(int32_t) * qpad)) ||
        (st = dev_alloc(ctx, (void**)&Q.qidx, sizeof(int32_t) * qpad)) ||
        (st = dev_alloc(ctx, (void**)&sl, sizeof(int32_t) * nstate * KN_SCAP)) ||
        (st = dev_alloc(ctx, (void**)&sc, sizeof(int32_t) * nstate)) ||
        (st = dev_alloc(ctx, (void**)&Q.overflow, sizeof(int) * qpad)) ||
        (st = dev_alloc(ctx, (void**)&ovs, sizeof(int32_t) * qpad)) ||
        (st = dev_alloc(ctx, (void**)&Q.sums, 2 * sizeof(unsigned long long))) ||
        (st = dev_alloc(ctx, (void**)&Q.qexact, qpad)) || (st = dev_alloc(ctx, (void**)&qtile, nqt)) ||
        (st = dev_alloc(ctx, (void**)&Q.qnrm, sizeof(float) * qpad)) ||
        (st = dev_alloc(ctx, (void**)&lists, sizeof(float2) * nstate * k)) ||
        (nch > 1 && ((st = dev_alloc(ctx, (void**)&pid, sizeof(int32_t) * qpad * nch * k)) ||
                     (st = dev_alloc(ctx, (void**)&pd, sizeof(uint64_t) * qpad * nch * k)))) ||
        (ns && ((st = dev_alloc(ctx, (void**)&smin, sizeof(float) * qpad * WS.nseg * KN_SPLIT * seed_keys)) ||
                (st = dev_alloc(ctx, (void**)&thr0, sizeof(float) * qpad)))) ||
        (!fp32 && (st = dev_alloc(ctx, (void**)&A, (size_t)qpad * kn_blocks(vq->D) * KN_K * 2)))) {
        cleanup();
        return st;
    }
    if (small) {
        query_slots_small_kernel<<<1, 1024, 0, s>>>(queries, (int)q, (int)qpad, v->exact, v->nrm, n, Q, qtile,
                                                    ctx->d_status);
        ctx->launches++;
    } else {
        exact_flags_of_queries<<<(unsigned)ceil_div(q, 256), 256, 0, s>>>(queries, q, v->exact, n, qf);
        if ((st = scan_exclusive_i64(ctx, qf, q))) { cleanup(); return st; }
        query_slots_kernel<<<(unsigned)ceil_div(qpad, 256), 256, 0, s>>>(queries, q, qpad, v->exact, v->nrm, n, qf, Q,
                                                                         ctx->d_status);
        tile_flags_kernel<<<(unsigned)ceil_div(nqt, 8), 256, 0, s>>>(v->exact, Q.qv, qpad, KN_M, qtile, nqt);
        ctx->launches += 3;
    }
    PCK(ctx, cudaMemsetAsync(sc, 0, sizeof(int32_t) * nstate, s));
    if (!fp32) {
        vec_arow_kernel<<<(unsigned)ceil_div(qpad, 8), 256, 0, s>>>(v->theta, Q.qv, qpad, v->D, A);
        ctx->launches++;
        const int kb = kn_blocks(v->D);
        CUtensorMap tmA, tmB;
        if (!make_map(ctx, &tmA, A, qpad, KN_M, kb) || !make_map(ctx, &tmB, x.B, x.npad, KN_N, kb)) {
            cleanup();
            return PANTHER_ECUDA;
        }
        ScreenArgs S{x.cid, x.cnrm, x.cncf, x.ctile, x.ctmax, W, 0, 0, nullptr, x.nexact, Q.qv, Q.qnrm, Q.qexact, qtile,
                     k, lists, sl, sc, nullptr, 0, Q.overflow, ctx->d_status, same, dump, Q.qidx, x.npad};
        auto grid = [&](const Split& w) {
            return (unsigned)(w.G ? w.G : std::min<int64_t>(nqt, ctx->num_sms));
        };
        if (dump) {                                  // (D <= 56)
            if ((st = launch_screen<DUMP_FORM, 1>(ctx, grid(W), tmA, tmB, S))) { cleanup(); return st; }
        } else {
            if (ns) {
                ScreenArgs SS = S;
                SS.W = WS;
                SS.seed_step = (uint32_t)(nct / ns);
                SS.seed_mul = (uint32_t)std::max<int64_t>(1, ns * 618 / 1000);   // coprime to ns: a permutation
                while (std::gcd(SS.seed_mul, (uint32_t)ns) != 1) ++SS.seed_mul;
                SS.smin = smin;
                SS.seed_keys = seed_keys;
                st = kb == 1 ? launch_screen<SEED, 1>(ctx, grid(WS), tmA, tmB, SS)
                   : kb == 2 ? launch_screen<SEED, 2>(ctx, grid(WS), tmA, tmB, SS)
                             : launch_screen<SEED, 3>(ctx, grid(WS), tmA, tmB, SS);
                if (st) { cleanup(); return st; }
                seed_bound_kernel<<<(unsigned)ceil_div(qpad, 8), 256, 0, s>>>(smin, qpad, WS, seed_keys, k, thr0);
                ctx->launches++;
                S.thr0 = thr0;
            }
            if (nct < FILL_TILES)
                st = kb == 1 ? launch_screen<FILL, 1>(ctx, grid(W), tmA, tmB, S)
                   : kb == 2 ? launch_screen<FILL, 2>(ctx, grid(W), tmA, tmB, S)
                             : launch_screen<FILL, 3>(ctx, grid(W), tmA, tmB, S);
            else
                st = kb == 1 ? launch_screen<SCREEN, 1>(ctx, grid(W), tmA, tmB, S)
                   : kb == 2 ? launch_screen<SCREEN, 2>(ctx, grid(W), tmA, tmB, S)
                             : launch_screen<SCREEN, 3>(ctx, grid(W), tmA, tmB, S);
            if (st) { cleanup(); return st; }
        }
    } else {
        const dim3 fg((unsigned)(qpad / F_T), (unsigned)nch);
        if (v->D <= KN_K)
            fp32_kernel<64><<<fg, F_T, 0, s>>>(vq->theta, vc->theta, same, v->D, Q.qv, Q.qexact, Q.qnrm, qpad,
                                               x.nexact, x.cid, x.cnrm, x.cncf, x.npad, k, lists, sl, sc, Q.overflow);
        else
            fp32_kernel<128><<<fg, F_T, 0, s>>>(vq->theta, vc->theta, same, v->D, Q.qv, Q.qexact, Q.qnrm, qpad,
                                                x.nexact, x.cid, x.cnrm, x.cncf, x.npad, k, lists, sl, sc, Q.overflow);
        ctx->launches++;
    }
    PCK(ctx, cudaGetLastError());
    // (every list fits 64 candidates; a query with a shortlist may keep more)
    const unsigned rg = (unsigned)ceil_div(qpad * nch * 32, 256);
    rerank_kernel<RERANK_FEW><<<rg, 256, 0, s>>>(vq->theta, vc->theta, v->D, Q.qv, Q.qidx, qpad, W, k, lists, sl, sc,
                                                 Q.overflow, ids, d2, pid, pd);
    rerank_kernel<RERANK_ALL><<<rg, 256, 0, s>>>(vq->theta, vc->theta, v->D, Q.qv, Q.qidx, qpad, W, k, lists, sl, sc,
                                                 Q.overflow, ids, d2, pid, pd);
    ctx->launches++;
    ctx->launches++;
    if (nch > 1 && nch * k <= 256) {
        chunk_merge_warp_kernel<<<(unsigned)ceil_div(qpad, 8), 256, 0, s>>>(Q.qv, Q.qidx, Q.overflow, qpad, W, k, pid,
                                                                            pd, ids, d2);
        ctx->launches++;
    } else if (nch > 1) {
        chunk_merge_kernel<<<(unsigned)std::min<int64_t>(qpad, 8 * ctx->num_sms), 256, 0, s>>>(
            Q.qv, Q.qidx, Q.overflow, nullptr, qpad, W, nch, k, pid, pd, ids, d2);
        ctx->launches++;
    }
    knn_sums_kernel<<<(unsigned)std::min<int64_t>(ceil_div(nstate, 256), 4 * ctx->num_sms), 256, 0, s>>>(
        sc, nstate, Q.overflow, qpad, Q.sums, ovs);
    ctx->launches++;
    PCK(ctx, cudaGetLastError());
    // screening statistics: pairs kept for rerank, overflowed queries
    unsigned long long* hsum = (unsigned long long*)ctx->h_counts;      // pinned
    PCK(ctx, cudaMemcpyAsync(hsum, Q.sums, 2 * sizeof(unsigned long long), cudaMemcpyDeviceToHost, s));
    PCK(ctx, cudaStreamSynchronize(s));
    const int64_t kept = (int64_t)hsum[0], over = (int64_t)hsum[1];
    if (over) {
        // the overflowed queries: exact brute force over all vertices, spread
        // over the GPU. A warp takes 4,096 vertices of a query, 512 when there
        // are few queries (one query of 1.5M vertices kept 366 warps busy); a
        // CTA of the many-query form 256 or more, three CTAs an SM
        const bool tile = over >= 8 && over * vc->n >= BRUTE_TILE * k;
        const int64_t nparts =
            tile ? std::max<int64_t>(1, std::min<int64_t>(ceil_div(vc->n, 256), 3 * ctx->num_sms / ceil_div(over, BT_T)))
                 : std::max({int64_t(1), std::min<int64_t>(1024, ceil_div(vc->n, 4096)),
                             std::min<int64_t>(ceil_div(vc->n, 512), 32768 / over)});
        int32_t* bid = nullptr;
        uint64_t* bd = nullptr;
        auto bfree = [&]() { dev_free(ctx, bid); dev_free(ctx, bd); };
        if ((st = dev_alloc(ctx, (void**)&bid, sizeof(int32_t) * over * nparts * k)) ||
            (st = dev_alloc(ctx, (void**)&bd, sizeof(uint64_t) * over * nparts * k))) {
            bfree();
            cleanup();
            return st;
        }
        if (tile) {
            st = v->D <= 64 ? launch_brute<64>(ctx, vq, vc, same, Q.qv, ovs, over, nparts, k, bid, bd)
                            : launch_brute<128>(ctx, vq, vc, same, Q.qv, ovs, over, nparts, k, bid, bd);
        } else {
            brute_warp_kernel<<<(unsigned)ceil_div(over * nparts * 32, 256), 256, 0, s>>>(
                vq->theta, vc->theta, same, v->D, vc->n, Q.qv, ovs, over, nparts, k, bid, bd);
            ctx->launches++;
        }
        if (st) {
            bfree();
            cleanup();
            return st;
        }
        chunk_merge_kernel<<<(unsigned)std::min<int64_t>(over, 8 * ctx->num_sms), 256, 0, s>>>(
            Q.qv, Q.qidx, Q.overflow, ovs, over, W, nparts, k, bid, bd, ids, d2);
        ctx->launches++;
        const cudaError_t ce = cudaGetLastError();
        bfree();
        if (ce) {
            cleanup();
            return cuda_err(ctx, ce, "k-NN brute-force fallback");
        }
    }
    ctx->knn_stats[0] = q * vc->n;
    ctx->knn_stats[1] = kept;
    ctx->knn_stats[2] = over;
    ctx->knn_stats[3] = x.nexact;
    cleanup();
    return PANTHER_OK;
}

static panther_status knn_entry(panther_ctx* ctx, const pantherpp_vecs* v, const pantherpp_vecs* vc, bool same,
                                const int32_t* queries, int64_t q, int k, int32_t* out_ids, uint64_t* out_dist2,
                                int flags) {
    if (!ctx || !v || !vc) return PANTHER_EINVAL;
    if (vc->D != v->D) return set_err(ctx, PANTHER_EINVAL, "query and candidate vectors differ in D");
    if (q < 0 || q > 0x7fffffffLL) return set_err(ctx, PANTHER_EINVAL, "q must be in [0, 2^31)");
    if (k < 1 || k > KN_KMAX) return set_err(ctx, PANTHER_EINVAL, "k must be in [1, 32]");
    int mode = flags & 0xff;
    if (mode != PANTHER_KNN_BF16_SCREEN && mode != PANTHER_KNN_FP32) return set_err(ctx, PANTHER_EINVAL, "bad flags");
    const bool fp32 = mode == PANTHER_KNN_FP32;
    auto run = [&](const int32_t* qs, int32_t* oi, uint64_t* od) {
        return knn_run(ctx, v, vc, same, qs, q, k, oi, od, fp32);
    };
    if (q == 0) return PANTHER_OK;
    if (!queries || !out_ids || !out_dist2) return set_err(ctx, PANTHER_EINVAL, "null query or output array");
    cudaSetDevice(ctx->device);
    cudaStream_t s = ctx->stream;
    if (flags & PANTHER_IO_HOST) {
        int32_t* buf = nullptr;
        size_t qb = ((sizeof(int32_t) * q + 15) / 16) * 16, ib = sizeof(int32_t) * q * k, db = sizeof(uint64_t) * q * k;
        panther_status st = dev_alloc(ctx, (void**)&buf, qb + ib + db + 16);
        if (st) return st;
        uint64_t* dd = (uint64_t*)((char*)buf + qb + ((ib + 15) / 16) * 16);
        int32_t* di = (int32_t*)((char*)buf + qb);
        PCK(ctx, cudaMemcpyAsync(buf, queries, sizeof(int32_t) * q, cudaMemcpyHostToDevice, s));
        st = run(buf, di, dd);
        if (!st) {
            PCK(ctx, cudaMemcpyAsync(out_ids, di, ib, cudaMemcpyDeviceToHost, s));
            PCK(ctx, cudaMemcpyAsync(out_dist2, dd, db, cudaMemcpyDeviceToHost, s));
            PCK(ctx, cudaStreamSynchronize(s));
        }
        dev_free(ctx, buf);
        return st;
    }
    return run(queries, out_ids, out_dist2);
}

extern "C" panther_status pantherpp_knn(panther_ctx* ctx, const pantherpp_vecs* v, const int32_t* queries, int64_t q,
                                        int k, int32_t* out_ids, uint64_t* out_dist2, int flags) {
    return knn_entry(ctx, v, v, true, queries, q, k, out_ids, out_dist2, flags);
}

extern "C" panther_status pantherpp_knn_cross(panther_ctx* ctx, const pantherpp_vecs* vq, const pantherpp_vecs* vc,
                                              const int32_t* queries, int64_t q, int k, int32_t* out_ids,
                                              uint64_t* out_dist2, int flags) {
    return knn_entry(ctx, vq, vc, false, queries, q, k, out_ids, out_dist2, flags);
}

extern "C" panther_status pantherpp_knn_stats(panther_ctx* ctx, int64_t stats[4]) {
    if (!ctx || !stats) return PANTHER_EINVAL;
    for (int i = 0; i < 4; ++i) stats[i] = ctx->knn_stats[i];
    return PANTHER_OK;
}

// Measurement of the BF16 screening error (no counterpart in the paper): the
// tensor-core screen of up to 128 queries against every candidate, keeping
// every screened value. out_y[i][p] = y_hat = |b|^2 - 2 a_hat.b_hat for query
// i and the candidate at position p (out_cid[p], -1 for padding); the exact
// value is |b|^2 - 2 a.b, so d_hat = |a|^2 + y_hat.
extern "C" panther_status pantherpp_debug_screen(panther_ctx* ctx, const pantherpp_vecs* v, const int32_t* queries,
                                                 int64_t q, float* out_y, int32_t* out_cid, int64_t* npad) {
    if (!ctx || !v || !npad) return PANTHER_EINVAL;
    *npad = v->npad;
    if (!out_y && !out_cid) return PANTHER_OK;
    if (!queries || !out_y || !out_cid || q < 1 || q > KN_M)
        return set_err(ctx, PANTHER_EINVAL, "1 <= q <= 128 queries and both outputs are needed");
    if (kn_blocks(v->D) > 1) return set_err(ctx, PANTHER_EINVAL, "BF16 screening values are kept for D <= 56 only");
    cudaSetDevice(ctx->device);
    cudaStream_t s = ctx->stream;
    int32_t* ids = nullptr;
    uint64_t* d2 = nullptr;
    panther_status st;
    if ((st = dev_alloc(ctx, (void**)&ids, sizeof(int32_t) * q)) || (st = dev_alloc(ctx, (void**)&d2, 8 * q))) {
        dev_free(ctx, ids);
        return st;
    }
    PCK(ctx, cudaMemsetAsync(out_y, 0xff, sizeof(float) * q * v->npad, s));   // NaN where nothing is screened
    st = knn_run(ctx, v, v, true, queries, q, 1, ids, d2, false, out_y);
    if (!st) {
        cudaError_t e = cudaMemcpyAsync(out_cid, v->cid, sizeof(int32_t) * v->npad, cudaMemcpyDeviceToDevice, s);
        if (!e) e = cudaStreamSynchronize(s);
        if (e) st = cuda_err(ctx, e, "screen dump");
    }
    dev_free(ctx, ids);
    dev_free(ctx, d2);
    return st;
}
