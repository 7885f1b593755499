// CUDA-core kernels of the contraction engine: element-wise contraction of small steps, slice
// binding of the leaves (Sec. 3.2), FP64 cross-slice accumulation and readout (Eq. lxeb_2), and
// the per-tensor power-of-two scaling into planar 16-bit storage (Sec. 4.2, dynamic scaling).
#include <cuda_fp16.h>
#include <cuda_bf16.h>

#include <type_traits>

#include "tn_internal.h"
#include "tn_planar_out.cuh"

namespace tn {

namespace {

__device__ __forceinline__ uint64_t deposit(uint64_t x, int n, const int8_t *pos) {
    uint64_t r = 0;
    for (int i = 0; i < n; ++i)
        if (((x >> i) & 1ull) && pos[i] >= 0) r |= 1ull << pos[i];
    return r;
}

// Operand offsets of output bits.  An element-wise kernel's thread takes outputs tid + 256 t of a
// chunk of 2^LB (LB <= 10) consecutive ones: an offset is the OR of the thread's part (bits 0-7,
// set up once), of t's (bits 8, 9) and of the chunk's (bits LB and up, one bit per lane of the
// warp).  A block's set-up is then a few dozen instructions; tables of all 2^LB offsets in shared
// memory took longer to build than a small step's outputs.
struct Offsets {  // of A and of B
    uint64_t a, b;
};
// bits 0 .. n - 1 of x, both operands in one pass (unrolled: a step's set-up waits for these loads)
__device__ __forceinline__ Offsets deposit2(uint32_t x, int n, const int8_t *pa, const int8_t *pb) {
    Offsets r{0, 0};
#pragma unroll 4
    for (int i = 0; i < n; ++i) {
        const int qa = pa[i], qb = pb[i];
        const uint64_t bit = (x >> i) & 1u;
        r.a |= qa >= 0 ? bit << qa : 0;
        r.b |= qb >= 0 ? bit << qb : 0;
    }
    return r;
}
struct LowOffsets {
    Offsets own, bit8{0, 0}, bit9{0, 0};
    __device__ __forceinline__ LowOffsets(const GenericDesc &d, int lb)
        : own(deposit2(threadIdx.x & ((1u << (lb < 8 ? lb : 8)) - 1), lb < 8 ? lb : 8, d.posA_c,
                       d.posB_c)) {
        if (lb > 8) bit8 = deposit2(1, 1, d.posA_c + 8, d.posB_c + 8);
        if (lb > 9) bit9 = deposit2(1, 1, d.posA_c + 9, d.posB_c + 9);
    }
    __device__ __forceinline__ uint64_t a(int t) const {
        return own.a | ((t & 1) ? bit8.a : 0) | ((t & 2) ? bit9.a : 0);
    }
    __device__ __forceinline__ uint64_t b(int t) const {
        return own.b | ((t & 1) ? bit8.b : 0) | ((t & 2) ? bit9.b : 0);
    }
};
// the offsets of the contracted index's n lowest bits, up to 10, in shared memory
__device__ __forceinline__ void k_offsets(const GenericDesc &d, int n, uint64_t *ka, uint64_t *kb) {
    for (int k = threadIdx.x; k < (1 << n); k += 256) {
        const Offsets o = deposit2((uint32_t)k, n, d.posA_k, d.posB_k);
        ka[k] = o.a;
        kb[k] = o.b;
    }
}
// of bits lb .. n - 1 of x, the same x in every lane of the warp: lane i keeps the places of bits
// lb + i and lb + i + 32 (kernel parameters indexed by the lane are read one lane at a time, so
// not once per chunk)
struct HighOffsets {
    int shift, qa[2], qb[2];
    __device__ __forceinline__ HighOffsets(const GenericDesc &d, int lb)
        : shift(lb + (threadIdx.x & 31)) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int i = shift + 32 * h;
            qa[h] = i < d.rank_c ? d.posA_c[i] : -1;
            qb[h] = i < d.rank_c ? d.posB_c[i] : -1;
        }
    }
    __device__ __forceinline__ Offsets at(uint64_t x) const {
        uint64_t a = 0, b = 0;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint64_t bit = shift + 32 * h < 64 ? (x >> (shift + 32 * h)) & 1ull : 0;
            a |= qa[h] >= 0 ? bit << qa[h] : 0;
            b |= qb[h] >= 0 ? bit << qb[h] : 0;
        }
        auto all = [](uint64_t v) {
            return ((uint64_t)__reduce_or_sync(0xffffffffu, (uint32_t)(v >> 32)) << 32) |
                   __reduce_or_sync(0xffffffffu, (uint32_t)v);
        };
        return Offsets{all(a), all(b)};
    }
};

// One output: the sum over 2^nk consecutive elements of A and B.
// UNROLL: pairs of k whose loads are in flight at once; INDEX counts them.
template <int UNROLL, class INDEX = int>
__device__ __forceinline__ float2 chain_sum(const float2 *A, const float2 *B, int nk,
                                            uint32_t flags) {
    float re = 0.f, im = 0.f;
    auto mac = [&](float ax, float ay, float bx, float by) {
        re = fmaf(ax, bx, re);
        re = fmaf(-ay, by, re);
        im = fmaf(ax, by, im);
        im = fmaf(ay, bx, im);
    };
    if (nk == 0) {
        const float2 a = *A, b = *B;
        if (flags & kChainFused) {
            re = fmaf(a.x, b.x, -a.y * b.y);
            im = fmaf(a.x, b.y, a.y * b.x);
        } else {
            mac(a.x, a.y, b.x, b.y);
        }
        return make_float2(re, im);
    }
    const float4 *A4 = reinterpret_cast<const float4 *>(A);
    const float4 *B4 = reinterpret_cast<const float4 *>(B);
    if (flags & kChainBlocked) {
        float2 sum = make_float2(0.f, 0.f);
        for (int k = 0; k < (1 << (nk - 1)); k += 8) {
            re = im = 0.f;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const float4 a = A4[k + q], b = B4[k + q];
                mac(a.x, a.y, b.x, b.y);
                mac(a.z, a.w, b.z, b.w);
            }
            sum.x += re;
            sum.y += im;
        }
        return sum;
    }
#pragma unroll UNROLL
    for (INDEX k = 0; k < (INDEX)1 << (nk - 1); ++k) {
        const float4 a = A4[k], b = B4[k];
        mac(a.x, a.y, b.x, b.y);
        mac(a.z, a.w, b.z, b.w);
    }
    return make_float2(re, im);
}

// One thread per output element of C (in C's own memory order, so stores are coalesced),
// summing over the contracted elements, which the layout pass puts last and in one order in both
// operands (16-byte loads of two); a block walks chunks of 2^LB consecutive outputs (see
// LowOffsets).  2^22 outputs of 2 terms: 57 -> 32 us against tables of K and of the chunk.
__global__ void __launch_bounds__(256) k_generic(GenericDesc d, int64_t total) {
    const int lb = d.rank_c < 10 ? d.rank_c : 10;
    const LowOffsets low(d, lb);
    const HighOffsets high(d, lb);
    const uint64_t cmask = (d.rank_c >= 63) ? ~0ull : ((1ull << d.rank_c) - 1);
    const int64_t nchunks = total >> lb;
    for (int64_t ch = blockIdx.x; ch < nchunks; ch += gridDim.x) {
        const int64_t base = ch << lb;
        const int64_t s = base >> d.rank_c;
        const uint64_t c0 = (uint64_t)base & cmask;
        const Offsets h = high.at(c0);
        const float2 *Ab = d.A + s * d.sA + h.a;
        const float2 *Bb = d.B + s * d.sB + h.b;
        float2 *Cb = d.C + s * d.sC + (int64_t)c0;
        float amx = 0.f;
#pragma unroll 2
        for (int t = 0; (t << 8) + (int)threadIdx.x < (1 << lb); ++t) {
            const float2 v = chain_sum<4, int64_t>(Ab + low.a(t), Bb + low.b(t), d.nk, 0);
            Cb[(t << 8) + threadIdx.x] = v;
            amx = fmaxf(amx, fmaxf(fabsf(v.x), fabsf(v.y)));
        }
        if (d.amax_out) amax_publish(d.amax_out + s, amx);
    }
}

// Steps with nothing contracted (outer products, with or without batch labels): C[c] = A[a(c)]
// B[b(c)].  Pure streams of stores, so the per-output work is cut to the bone: a thread takes pairs
// of consecutive outputs (16-byte stores), PER of them in each chunk of 512 PER outputs, whose
// operand offsets it keeps in registers (the same in every chunk); the chunk's high-bit offsets come
// from a warp-parallel deposit, and the max-abs is published once per slice a block touches.
// 2^26 x 2^2 outputs: 1.07 -> 0.50 ms (5.4 TB/s) against 8-byte stores in 1024-output chunks.
template <int PER>
__global__ void __launch_bounds__(256) k_generic_k1(GenericDesc d, int64_t total) {
    constexpr int LB = PER == 2 ? 10 : 12;
    static_assert((1 << LB) == 512 * PER, "outputs of a chunk");
    // bit 0 (the pair), then the thread's bits 1-8, then t's
    const Offsets own = deposit2(2 * threadIdx.x, 9, d.posA_c, d.posB_c);
    const Offsets pair = deposit2(1, 1, d.posA_c, d.posB_c);
    const HighOffsets high(d, LB);
    uint64_t oa[PER], ob[PER];
#pragma unroll
    for (int t = 0; t < PER; ++t) {
        const Offsets o = deposit2(t, LB - 9, d.posA_c + 9, d.posB_c + 9);
        oa[t] = own.a | o.a;
        ob[t] = own.b | o.b;
    }
    const uint64_t cmask = (d.rank_c >= 63) ? ~0ull : ((1ull << d.rank_c) - 1);
    const int64_t nchunks = total >> LB;
    int64_t cur_s = -1;
    float amx = 0.f;
    for (int64_t ch = blockIdx.x; ch < nchunks; ch += gridDim.x) {
        const int64_t base = ch << LB;
        const int64_t s = base >> d.rank_c;
        const uint64_t c0 = (uint64_t)base & cmask;
        if (s != cur_s) {
            if (cur_s >= 0 && d.amax_out) amax_publish(d.amax_out + cur_s, amx);
            amx = 0.f;
            cur_s = s;
        }
        const Offsets h = high.at(c0);
        const float2 *Ab = d.A + s * d.sA + h.a;
        const float2 *Bb = d.B + s * d.sB + h.b;
        float4 *Cb = reinterpret_cast<float4 *>(d.C + s * d.sC + (int64_t)c0) + threadIdx.x;
        float2 a[PER][2], b[PER][2];
#pragma unroll
        for (int t = 0; t < PER; ++t) {
            a[t][0] = Ab[oa[t]];
            a[t][1] = Ab[oa[t] | pair.a];
            b[t][0] = Bb[ob[t]];
            b[t][1] = Bb[ob[t] | pair.b];
        }
#pragma unroll
        for (int t = 0; t < PER; ++t) {
            float2 v[2];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                v[q].x = fmaf(a[t][q].x, b[t][q].x, -a[t][q].y * b[t][q].y);
                v[q].y = fmaf(a[t][q].x, b[t][q].y, a[t][q].y * b[t][q].x);
                amx = fmaxf(amx, fmaxf(fabsf(v[q].x), fabsf(v[q].y)));
            }
            Cb[256 * t] = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
        }
    }
    if (cur_s >= 0 && d.amax_out) amax_publish(d.amax_out + cur_s, amx);
}

// Runs of small steps in one launch.  The steps are sorted by their depth in the run (level 0 reads
// only what earlier launches wrote), so all outputs of a level are independent: the threads of a
// slice's blocks share them out, and a barrier separates the levels.  The plan gives all tensors
// a run touches pairwise disjoint memory, so nothing else orders the work.  Bound by the latency
// of a level, not by its work.

// Global-memory form, for runs with a connected part too large for shared memory: quarter warps take
// items of 8 outputs; a cluster of blocks per slice with a cluster barrier per level, or one
// block.  ~1.1 us a level: 402 steps of a 20-qubit circuit, 16 levels, take 25 us (1205 us by one
// block, step after step).
__device__ __forceinline__ uint4 ldg_item(const uint4 *p) {
    uint4 v;
    asm volatile("ld.global.nc.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p));
    return v;
}

// bits of x at the set positions of the mask m of an item's lanes, packed
__device__ __forceinline__ uint32_t pack_lane(uint32_t x, uint32_t m) {
    uint32_t r = 0, sh = 0;
#pragma unroll
    for (int i = 0; i < kChainItemBits; ++i) {
        const uint32_t in = (m >> i) & 1u;
        r |= ((x >> i) & in) << sh;
        sh += in;
    }
    return r;
}

// max of v over the item's lanes into amax[block][slice], for the items that record it
__device__ __forceinline__ void chain_amax(unsigned int *amax, int64_t sb, int64_t s, uint32_t meta,
                                           int lane, float v) {
    if (!__any_sync(0xffffffffu, meta != 0)) return;
    for (int o = kChainItemLanes / 2; o > 0; o >>= 1)
        v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    if (meta != 0 && lane == 0)
        atomicMax(amax + (int64_t)(meta - 1) * sb + s, __float_as_uint(v));
}

__global__ void __launch_bounds__(kChainThreads)
    k_chain(const ChainItem *items, const int32_t *levels, int32_t nlevels, float2 *arena,
            unsigned int *amax, int64_t sb, int32_t cluster) {
    constexpr int kTeams = kChainThreads / kChainItemLanes;
    const int64_t s = blockIdx.x / cluster;
    const int lane = threadIdx.x % kChainItemLanes;
    const int team = (blockIdx.x % cluster) * kTeams + threadIdx.x / kChainItemLanes;
    const int stride = cluster * kTeams;
    auto load = [&](int i, uint4 &x, uint4 &y) {
        const uint4 *p = reinterpret_cast<const uint4 *>(items + i);
        x = ldg_item(p);
        y = ldg_item(p + 1);
    };
    int hi = levels[1];
    int i = levels[0] + team;
    uint4 x = make_uint4(0, 0, 0, 0), y = x;
    if (i < hi) load(i, x, y);
    for (int l = 0; l < nlevels; ++l) {
        const int nhi = l + 1 < nlevels ? levels[l + 2] : hi;
        while (__any_sync(0xffffffffu, i < hi)) {  // the warp's teams go on together
            uint4 nx = x, ny = y;
            if (i + stride < hi) load(i + stride, nx, ny);
            const uint32_t ra = y.y & 0xffu, rb = (y.y >> 8) & 0xffu, rc = (y.y >> 16) & 0xffu;
            const int lanes = (y.y >> 24) & 15, nk = y.y >> 28;
            float amx = 0.f;
            if (i < hi && lane < (1 << lanes)) {
                auto at = [&](uint32_t base, uint32_t off, uint32_t r) {
                    return arena + ((int64_t)base << 5) + off + (r == kChainShared ? 0 : s << r);
                };
                const uint32_t oa = (x.w & 0xffffu) + (pack_lane(lane, (y.x >> 16) & 0xffu) << nk);
                const uint32_t ob = (x.w >> 16) + (pack_lane(lane, y.x >> 24) << nk);
                const float2 v = chain_sum<8>(at(x.x, oa, ra), at(x.y, ob, rb), nk, y.w);
                *at(x.z, (y.x & 0xffffu) + lane, rc) = v;
                amx = fmaxf(fabsf(v.x), fabsf(v.y));
            }
            chain_amax(amax, sb, rc == kChainShared ? 0 : s, i < hi ? y.z : 0, lane, amx);
            i += stride;
            x = nx;
            y = ny;
        }
        if (l + 1 < nlevels) {
            i = hi + team;
            hi = nhi;
            if (i < hi) load(i, x, y);
            // both barriers make the level's results visible to every warp of the slice
            if (cluster == 1)
                __syncthreads();
            else
                asm volatile("barrier.cluster.arrive.release.aligned;\n\t"
                             "barrier.cluster.wait.acquire.aligned;" ::
                                 : "memory");
        }
    }
}

// Shared-memory form: each block works one group of connected steps of one slice.  Everything a level
// touches (operands, records, results) is in shared memory, so a level is a record load, the
// operand loads, the sum and a block barrier.  Measured: the 12-qubit circuit (146 steps, 24 levels)
// in one launch of 20 us, 340 us by one block step after step, ~29 us in the global-memory form
// with two launches for its GEMM steps; 402 steps of the 20-qubit circuit 8.8 us (25 us global).
__global__ void __launch_bounds__(kChainShmThreads)
    k_chain_shm(const ChainGroup *groups, int32_t ngroups, const ChainCopy *copies,
                const ChainRec *recs, const int32_t *levels, float2 *arena, unsigned int *amax,
                int64_t sb) {
    extern __shared__ __align__(16) float2 chain_mem[];
    __shared__ int32_t bounds[kChainShmLevels + 1];
    const int64_t s = blockIdx.x / ngroups;
    const ChainGroup g = groups[blockIdx.x % ngroups];
    const int tid = threadIdx.x, lane = tid % kChainItemLanes;
    constexpr int kTeams = kChainShmThreads / kChainItemLanes;
    float2 *rec_mem = chain_mem + g.elems;
    auto place = [&](const ChainCopy &c) {
        return arena + ((int64_t)c.base << 5) + c.off + lane + (c.r == kChainShared ? 0 : s << c.r);
    };
    for (int i = tid; i <= g.n_levels; i += kChainShmThreads) bounds[i] = levels[g.levels + i];
    {
        const uint4 *src = reinterpret_cast<const uint4 *>(recs + g.recs);
        uint4 *dst = reinterpret_cast<uint4 *>(rec_mem);
        for (int i = tid; i < g.n_recs / 2; i += kChainShmThreads) dst[i] = src[i];
    }
    for (int i = tid / kChainItemLanes; i < g.n_in; i += kTeams) {
        const ChainCopy c = copies[g.copies + i];
        if (lane < (1 << c.lanes)) chain_mem[c.shm + lane] = *place(c);
    }
    __syncthreads();
    for (int l = 0; l < g.n_levels; ++l) {
        const int hi = bounds[l + 1];
        for (int i = bounds[l] + tid; i < hi; i += kChainShmThreads) {
            const ChainRec r = reinterpret_cast<const ChainRec *>(rec_mem)[i];
            chain_mem[r.c] = chain_sum<4>(chain_mem + r.a, chain_mem + r.b, r.nk_flags & 15,
                                          r.nk_flags);
        }
        __syncthreads();
    }
    const int i0 = tid / kChainItemLanes;
    for (int i = i0; __any_sync(0xffffffffu, i < g.n_out); i += kTeams) {
        uint32_t meta = 0;
        int64_t ms = 0;
        float amx = 0.f;
        if (i < g.n_out) {
            const ChainCopy c = copies[g.copies + g.n_in + i];
            meta = c.meta;
            ms = c.r == kChainShared ? 0 : s;
            if (lane < (1 << c.lanes)) {
                const float2 v = chain_mem[c.shm + lane];
                *place(c) = v;
                amx = fmaxf(fabsf(v.x), fabsf(v.y));
            }
        }
        chain_amax(amax, sb, ms, meta, lane, amx);
    }
}

// Sparse-state leaves (Sec. 3.3): grid (leaf, chunk); block (leaf, chunk) writes a strided part
// of that leaf's configurations x dense elements.
__global__ void k_sparse_leaves(const SparseLeafDesc *leaves) {
    const SparseLeafDesc &d = leaves[blockIdx.x];
    const int64_t nd = 1ll << d.rank_d;
    const int64_t total = d.nconf * nd;
    for (int64_t i = blockIdx.y * (int64_t)blockDim.x + threadIdx.x; i < total;
         i += (int64_t)gridDim.y * blockDim.x) {
        const int64_t c = i >> d.rank_d;
        const uint64_t j = (uint64_t)(i & (nd - 1));
        const double2 v = d.src[d.cfg_off[c] | (int64_t)deposit(j, d.rank_d, d.pos_d)];
        d.dst[i] = make_float2((float)v.x, (float)v.y);
    }
}

// One sparse-state step, summing over the contracted dense bits in increasing order; the operand
// entries are the configurations gA[c], gB[c] (the projections of c onto each operand's open
// labels).  A block walks chunks of 2^LB consecutive outputs (see LowOffsets; chunks never leave a
// configuration, those of less than 256 outputs go several at a time), and the sum 2^10 terms at a
// time, whose offsets are in shared memory (one output of 2^20 terms: 1.7 ms, 13-19 ms with offsets
// computed for every term; LONG, so that the many small steps don't load that code).  Bound by the
// instructions per output: a deposit per output made the 2^24-output steps take 4 times as long.
template <bool LONG>
__global__ void __launch_bounds__(256) k_sparse_step(GenericDesc d, const int32_t *gA,
                                                     const int32_t *gB, int64_t nconf) {
    __shared__ uint64_t koffA[1024], koffB[1024];
    const int nk = d.nk, kb = LONG ? 10 : nk;
    const int lb = d.rank_c < 10 ? d.rank_c : 10;
    const LowOffsets low(d, lb);
    const HighOffsets high(d, lb);
    k_offsets(d, kb, koffA, koffB);
    __syncthreads();
    const int64_t chunks = nconf << (d.rank_c - lb);
    const int together = lb < 8 ? 256 >> lb : 1;  // chunks a block takes at once
    const int j0 = together > 1 ? threadIdx.x & ((1 << lb) - 1) : threadIdx.x;
    for (int64_t ch0 = (int64_t)blockIdx.x * together; ch0 < chunks;
         ch0 += (int64_t)gridDim.x * together) {
        const int64_t ch = ch0 + (together > 1 ? (int)threadIdx.x >> lb : 0);
        const uint64_t hi = ((uint64_t)ch << lb) & ((1ull << d.rank_c) - 1);
        Offsets h{0, 0};
        if (d.rank_c > lb) h = high.at(hi);  // one chunk at a time: the same for every thread
        if (ch >= chunks) continue;
        const int64_t c = ch >> (d.rank_c - lb);
        const float2 *Ab = d.A + (int64_t)gA[c] * d.sA + h.a;
        const float2 *Bb = d.B + (int64_t)gB[c] * d.sB + h.b;
        float2 *Cb = d.C + c * d.sC + (int64_t)hi;
        for (int t = 0; (t << 8) + j0 < (1 << lb); ++t) {
            const float2 *A = Ab + low.a(t);
            const float2 *B = Bb + low.b(t);
            float re = 0.f, im = 0.f;
            auto sum = [&](const float2 *Ak, const float2 *Bk) {
#pragma unroll 4
                for (int k = 0; k < 1 << kb; ++k) {
                    const float2 a = Ak[koffA[k]], b = Bk[koffB[k]];
                    re = fmaf(a.x, b.x, re);
                    re = fmaf(-a.y, b.y, re);
                    im = fmaf(a.x, b.y, im);
                    im = fmaf(a.y, b.x, im);
                }
            };
            if constexpr (LONG) {
                for (int64_t k0 = 0; k0 < 1ll << (nk - kb); ++k0) {
                    const Offsets o = deposit2((uint32_t)k0, nk - kb, d.posA_k + kb, d.posB_k + kb);
                    sum(A + o.a, B + o.b);
                }
            } else {
                sum(A, B);
            }
            Cb[(t << 8) + j0] = make_float2(re, im);
        }
    }
}

__global__ void k_sparse_amps(const float2 *root, const int32_t *idx, int64_t n, double2 *amps) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const float2 v = root[idx[i]];
        amps[i].x += (double)v.x;
        amps[i].y += (double)v.y;
    }
}

// Conversions between FP32 and FP64 in integer operations.  GB300 runs conversion instructions
// from and to 64 bits at the rate of its FP64 units, 2 a clock and SM: a complex128 leaf of 2^23
// elements took 28 us for them alone, its memory traffic takes 30.  Normal numbers and zeros are
// rounded (to nearest, ties to even) or widened here, the rest by the instruction.
__device__ __forceinline__ float narrow(double x) {
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    const uint32_t sign = hi & 0x80000000u, mag = hi ^ sign;
    if ((mag | lo) == 0) return __uint_as_float(sign);
    if ((mag >> 20) - 897u > 253u) return (float)x;  // outside FP32's normal range
    const uint32_t m = (mag - (896u << 20)) << 3 | lo >> 29;
    const uint32_t up = (lo & 0x1fffffffu) + (m & 1u) > 0x10000000u;
    return __uint_as_float(sign | (m + up));
}
__device__ __forceinline__ double widen_normal(float x) {
    const uint32_t u = __float_as_uint(x), sign = u & 0x80000000u, mag = u ^ sign;
    return __hiloint2double((int)(sign | (mag ? (mag >> 3) + (896u << 20) : 0u)), (int)(u << 29));
}
__device__ __forceinline__ bool odd(float x) {  // subnormal, infinite or NaN
    const uint32_t u = __float_as_uint(x) << 1;
    return (u >> 24) - 1u > 253u && u != 0;
}
// N values under one test: with a branch for each, the adds that follow wait for one another (one
// slice of 2^24 amplitudes onto others: 189 us).
template <int N>
__device__ __forceinline__ void widen(const float (&v)[N], double (&d)[N]) {
    bool any = false;
#pragma unroll
    for (int i = 0; i < N; ++i) any = any || odd(v[i]);
    if (any) {
#pragma unroll
        for (int i = 0; i < N; ++i) d[i] = (double)v[i];
    } else {
#pragma unroll
        for (int i = 0; i < N; ++i) d[i] = widen_normal(v[i]);
    }
}
// a += v for two amplitudes.  Amplitudes that are all still +0, as before their first slice, take v as
// it is (-0 as +0) and need no FP64 unit.
__device__ __forceinline__ void add_widened2(double2 &a, double2 &b, float4 v) {
    double2 p, q;
    if (odd(v.x) || odd(v.y) || odd(v.z) || odd(v.w)) {
        p = make_double2((double)v.x, (double)v.y);
        q = make_double2((double)v.z, (double)v.w);
    } else {
        p = make_double2(widen_normal(v.x), widen_normal(v.y));
        q = make_double2(widen_normal(v.z), widen_normal(v.w));
    }
    const auto bits = [](double x) { return __double_as_longlong(x); };
    if ((bits(a.x) | bits(a.y) | bits(b.x) | bits(b.y)) == 0) {
        const auto plus = [&](double x) {
            return __longlong_as_double(bits(x) == bits(-0.0) ? 0 : bits(x));
        };
        a = make_double2(plus(p.x), plus(p.y));
        b = make_double2(plus(q.x), plus(q.y));
    } else {
        a = make_double2(a.x + p.x, a.y + p.y);
        b = make_double2(b.x + q.x, b.y + q.y);
    }
}

// Leaf binding: grid (item, slice, chunk); the blocks of one (item, slice) share its elements.
__global__ void k_bind(const BindItem *items, const double2 *src, float2 *arena,
                       int64_t slice_begin) {
    const BindItem it = items[blockIdx.x];
    const int64_t s = blockIdx.y;
    const uint64_t sigma = (uint64_t)(slice_begin + s);
    uint64_t soff = 0;
    for (int t = 0; t < it.nsl; ++t)
        if ((sigma >> it.sl_bit[t]) & 1ull) soff |= 1ull << it.sl_pos[t];
    const int64_t n = 1ll << it.rank;
    float2 *dst = arena + it.dst_off + s * it.dst_sstride;
    for (int64_t i = blockIdx.z * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.z * blockDim.x) {
        const uint64_t so = deposit((uint64_t)i, it.rank, it.pos_src) | soff;
        const double2 v = src[it.src_off + (int64_t)so];
        dst[i] = make_float2(narrow(v.x), narrow(v.y));
    }
}

// Tiled leaf binding (see BindTiled).  Shared memory holds one tile of up to MAXN complex64
// (2^11, or 2^12 when the six lowest source bits all lie above destination bit 5); the element
// of tile index tau sits at tau ^ (((tau >> 6) & 31) << 1).  The XOR changes bits 1-5 only, so
// the two elements of a destination pair stay adjacent and 16-byte aligned, and when the
// source's low bits land on tile bits 6-10 the 32 lanes of a read still write 32 distinct
// 16-byte slots of one 512-byte row.
__device__ __forceinline__ int tile_slot(int tau) { return tau ^ (((tau >> 6) & 31) << 1); }

// A thread has eight 16-byte loads in flight.  HBM bounds the kernel (24 bytes per element, and
// the max-abs of the leaf costs no pass of its own): 2^23 elements in
// 34.5 us (5.8 TB/s), 66 us with one load in flight and a pass for the max-abs.
template <int T>
__global__ void __launch_bounds__(256, 4)
    k_bind_tiled(const __grid_constant__ BindTiled b, const double2 *__restrict__ src,
                 float2 *__restrict__ arena, unsigned int *__restrict__ amax,
                 int64_t slice_begin) {
    __shared__ __align__(16) float2 tile[1 << T];
    __shared__ float wmax[8];
    const int64_t s = blockIdx.y;
    const uint64_t sigma = (uint64_t)(slice_begin + s);
    uint64_t soff = 0;
    for (int j = 0; j < b.nsl; ++j)
        if ((sigma >> b.sl_bit[j]) & 1ull) soff |= 1ull << b.sl_pos[j];
    const double2 *S = src + b.src_off + soff;
    float2 *D = arena + b.dst_off + s * b.dst_sstride;
    const int tid = threadIdx.x;
    // read-order index e = tid + 256 k: its tile index and source offset are those of tid OR'ed
    // with those of 256 k (disjoint bits)
    int tau0 = 0;
    uint64_t so0 = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q)
        if ((tid >> q) & 1) {
            tau0 |= 1 << b.e2t[q];
            so0 |= 1ull << b.e2s[q];
        }
    // write-order pair j = tid + 256 k covers tile indices 2 j, 2 j + 1; destination bits of
    // tile bits 6-8 come from tid, those of tile bits 9 and up from k
    uint64_t dw0 = (2 * tid) & 63;
#pragma unroll
    for (int q = 6; q < 9; ++q)
        if (((2 * tid) >> q) & 1) dw0 |= 1ull << b.t2d[q];
    float m = 0.f;
    for (int64_t w = blockIdx.x; w < b.ntiles; w += gridDim.x) {
        uint64_t dbase = dw0, sbase = so0;
        for (int u = 0; u < b.nrest; ++u)
            if ((w >> u) & 1) {
                dbase |= 1ull << b.rest_d[u];
                sbase |= 1ull << b.rest_s[u];
            }
#pragma unroll
        for (int k0 = 0; k0 < (1 << (T - 8)); k0 += 8) {
            double2 v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                uint64_t so = sbase;
#pragma unroll
                for (int q = 8; q < T; ++q)
                    if (((k0 + k) >> (q - 8)) & 1) so |= 1ull << b.e2s[q];
                v[k] = S[so];
            }
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                int tau = tau0;
#pragma unroll
                for (int q = 8; q < T; ++q)
                    if (((k0 + k) >> (q - 8)) & 1) tau |= 1 << b.e2t[q];
                const float2 f = make_float2(narrow(v[k].x), narrow(v[k].y));
                m = fmaxf(m, fmaxf(fabsf(f.x), fabsf(f.y)));
                tile[tile_slot(tau)] = f;
            }
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < (1 << (T - 9)); ++k) {
            uint64_t doff = dbase;
#pragma unroll
            for (int q = 9; q < T; ++q)
                if ((k >> (q - 9)) & 1) doff |= 1ull << b.t2d[q];
            *reinterpret_cast<float4 *>(D + doff) =
                *reinterpret_cast<const float4 *>(&tile[tile_slot(2 * (tid + (k << 8)))]);
        }
        __syncthreads();
    }
    if (!amax) return;
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((tid & 31) == 0) wmax[tid >> 5] = m;
    __syncthreads();
    if (tid == 0) {
        for (int i = 1; i < 8; ++i) m = fmaxf(m, wmax[i]);
        atomicMax(amax + (b.dst_sstride ? s : 0), __float_as_uint(m));
    }
}

// amps[x] += sum over slices s (in increasing order) of root[s][x], in FP64.  One slice: a thread takes
// two amplitudes and HBM bounds it (40 bytes per amplitude), 2^24 amplitudes in 97 us (6.9 TB/s),
// added to others as to zeros; 128 us when the FP64 units widened the root's values too.
__global__ void __launch_bounds__(256) k_accumulate(const float2 *root, int64_t n, double2 *amps) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < (n >> 1);
         i += (int64_t)gridDim.x * blockDim.x) {
        double2 a = amps[2 * i], b = amps[2 * i + 1];
        const float4 v = reinterpret_cast<const float4 *>(root)[i];
        add_widened2(a, b, v);
        amps[2 * i] = a;
        amps[2 * i + 1] = b;
    }
}

// Several slices: a thread takes PER consecutive amplitudes and reads AHEAD slices at once.  What bounds
// it is the way to memory and back (few amplitudes), the FP64 adds or HBM (many).
template <int PER, int AHEAD>
__global__ void __launch_bounds__(256) k_accumulate_slices(const float2 *root, int64_t sstride,
                                                           int64_t n, int64_t slices,
                                                           double2 *amps) {
    using V = typename std::conditional<PER == 2, float4, float2>::type;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n / PER;
         i += (int64_t)gridDim.x * blockDim.x) {
        double2 a[PER];
#pragma unroll
        for (int q = 0; q < PER; ++q) a[q] = amps[PER * i + q];
        for (int64_t s = 0; s < slices; s += AHEAD) {
            float v[2 * PER * AHEAD] = {};
            double d[2 * PER * AHEAD];
#pragma unroll
            for (int j = 0; j < AHEAD; ++j)
                if (s + j < slices)
                    *reinterpret_cast<V *>(v + 2 * PER * j) =
                        reinterpret_cast<const V *>(root + (s + j) * sstride)[i];
            widen(v, d);
#pragma unroll
            for (int j = 0; j < AHEAD; ++j)
                if (s + j < slices)
#pragma unroll
                    for (int q = 0; q < PER; ++q) {
                        a[q].x += d[2 * (PER * j + q)];
                        a[q].y += d[2 * (PER * j + q) + 1];
                    }
        }
#pragma unroll
        for (int q = 0; q < PER; ++q) amps[PER * i + q] = a[q];
    }
}

// The same with sliced open labels (amplitude batches, Sec. 3.2 slicing applied to open
// bonds): slice s0 + s adds its root into the block of amps that its bits for those labels (the
// set bits of `open`) select.  Slices that differ in them write different amplitudes, so a thread
// takes one root element of one block and walks that block's slices in flight in increasing
// order.
//
// The first id from s0 on whose open bits are o, and the next one with the same open bits; the others
// count the slices of a block.  An id past the last one wraps to below s0.
__device__ __forceinline__ uint64_t block_first(uint64_t s0, uint64_t open, uint64_t o) {
    const uint64_t d = (s0 ^ o) & open;
    if (d == 0) return s0;
    const int q = 63 - __clzll((long long)d);  // below 40, the most sliced labels
    const uint64_t hi = ~0ull << (q + 1);
    if ((o >> q) & 1ull) return (s0 & hi) | (o & ~hi);
    const uint64_t rest = ~open & hi;
    return (((s0 | ~rest) + 1) & rest) | o;
}
__device__ __forceinline__ uint64_t block_next(uint64_t sig, uint64_t open) {
    return (((sig | open) + 1) & ~open) | (sig & open);
}

// AHEAD: slices read at once.  The threads of a root element, 2^log2_g of them, share its blocks out.
// These are numbered by the open bits that vary among the slices in flight (kByBlock, `vary`), or the
// slices are, each a block of its own (kOwnBlock) or, with fewer slices than numbers of blocks, with the
// first of each block going on (kFirstOfBlock).
enum { kByBlock, kOwnBlock, kFirstOfBlock };
template <int AHEAD>
__global__ void __launch_bounds__(256)
    k_accumulate_batched(const float2 *root, int64_t sstride, int log2_n, int64_t slices,
                         int64_t s0_, const AccMap m, uint64_t open, uint64_t vary, int number,
                         int log2_g, double2 *amps) {
    const uint64_t s0 = (uint64_t)s0_, end = s0 + (uint64_t)slices;
    const int64_t blocks = number == kByBlock ? 1ll << __popcll((long long)vary) : slices;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i >> (log2_n + log2_g) == 0;
         i += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t x = (uint64_t)i & ((1ull << log2_n) - 1);
        const uint64_t ox = deposit(x, m.nroot, m.root_pos);
        for (int64_t g = i >> log2_n; g < blocks; g += 1ll << log2_g) {
            uint64_t sig = s0 + (uint64_t)g;
            if (number == kByBlock) {
                uint64_t o = s0 & open & ~vary;
                for (int j = 0, c = 0; j < m.nb; ++j)
                    if ((vary >> m.bj[j]) & 1ull) o |= (((uint64_t)g >> c++) & 1ull) << m.bj[j];
                sig = block_first(s0, open, o);
                if (sig < s0 || sig >= end) continue;
            } else if (number == kFirstOfBlock && block_first(s0, open, sig & open) != sig) {
                continue;
            }
            uint64_t o = ox;
            for (int j = 0; j < m.nb; ++j)
                if ((sig >> m.bj[j]) & 1ull) o |= 1ull << m.bpos[j];
            double2 a = amps[o];
            while (sig < end) {
                float v[2 * AHEAD] = {};
                double d[2 * AHEAD];
                uint64_t t = sig;
#pragma unroll
                for (int j = 0; j < AHEAD; ++j)
                    if (t < end) {
                        const float2 f = root[(int64_t)(t - s0) * sstride + (int64_t)x];
                        v[2 * j] = f.x;
                        v[2 * j + 1] = f.y;
                        t = block_next(t, open);
                    }
                widen(v, d);
#pragma unroll
                for (int j = 0; j < AHEAD; ++j)
                    if (sig < end) {
                        a.x += d[2 * j];
                        a.y += d[2 * j + 1];
                        sig = block_next(sig, open);
                    }
            }
            amps[o] = a;
        }
    }
}

// FP64 readout (Eq. lxeb_2): sums of p = |a|^2 and p^2.  Each thread sums a strided share in index
// order, a block its threads in a fixed tree, pass 2 the blocks likewise.  Four FP64 operations
// per amplitude against GB300's 1/64-rate FP64 units bound it, not memory: 2^24 amplitudes cannot
// take less than ~112 us (40 us of HBM time), so the grid covers every SM.  A readout
// of them with its copy to the host: 164 us; 348 us with 64 blocks and a serial second pass.
__device__ __forceinline__ void block_sum2(double &a1, double &a2, double *s1, double *s2) {
    s1[threadIdx.x] = a1;
    s2[threadIdx.x] = a2;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) {
            s1[threadIdx.x] += s1[threadIdx.x + w];
            s2[threadIdx.x] += s2[threadIdx.x + w];
        }
        __syncthreads();
    }
    a1 = s1[0];
    a2 = s2[0];
}

__global__ void __launch_bounds__(256) k_readout_partial(const double2 *amps, int64_t n,
                                                         double *partial) {
    __shared__ double s1[256], s2[256];
    double a1 = 0.0, a2 = 0.0;
    const int64_t stride = (int64_t)gridDim.x * 256;
#pragma unroll 4
    for (int64_t x = blockIdx.x * (int64_t)256 + threadIdx.x; x < n; x += stride) {
        const double2 v = amps[x];
        const double p = v.x * v.x + v.y * v.y;
        a1 += p;
        a2 += p * p;
    }
    block_sum2(a1, a2, s1, s2);
    if (threadIdx.x == 0) {
        partial[2 * blockIdx.x] = a1;
        partial[2 * blockIdx.x + 1] = a2;
    }
}

// Pass 2, one block: the sums go to partial[0] and partial[1].
__global__ void __launch_bounds__(256) k_readout_final(double *partial, int32_t n_partial) {
    __shared__ double s1[256], s2[256];
    double a1 = 0.0, a2 = 0.0;
    for (int i = threadIdx.x; i < n_partial; i += 256) {
        a1 += partial[2 * i];
        a2 += partial[2 * i + 1];
    }
    block_sum2(a1, a2, s1, s2);  // its barriers also separate the reads from the write below
    if (threadIdx.x == 0) {
        partial[0] = a1;
        partial[1] = a2;
    }
}

__global__ void k_zero_f64(double2 *p, int64_t n) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        p[i] = make_double2(0.0, 0.0);
}

// max(|re|, |im|) per slice, as float bits (non-negative floats order like unsigned ints).
__global__ void __launch_bounds__(256) k_amax(ConvertDesc d) {
    const int64_t s = blockIdx.y;
    const float4 *src = reinterpret_cast<const float4 *>(d.src + s * d.src_sstride);
    const int64_t n2 = d.n >> 1;  // two complex numbers per float4
    float m = 0.f;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n2;
         i += (int64_t)gridDim.x * blockDim.x) {
        const float4 v = src[i];
        m = fmaxf(m, fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w))));
    }
    if ((d.n & 1) && blockIdx.x == 0 && threadIdx.x == 0) {
        const float2 v = d.src[s * d.src_sstride + d.n - 1];
        m = fmaxf(m, fmaxf(fabsf(v.x), fabsf(v.y)));
    }
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(d.amax + s, __float_as_uint(m));
}

__device__ __forceinline__ int scale_exponent(unsigned int amax_bits) {
    const float a = __uint_as_float(amax_bits);
    if (!(a > 0.f) || !isfinite(a)) return 0;
    return ilogbf(a) - 14;  // stored max lands in [2^14, 2^15): inside FP16's range
}

// complex64 -> planar 16-bit: stored = value * 2^-e (exact power-of-two scaling).  With three
// planes the third holds re + im, summed in FP32 and rounded once; with four, planes 2 and 3 hold
// the residuals re - hi(re) and im - hi(im) (the "lo" halves of a compensated product).
template <typename T2>
__device__ __forceinline__ T2 pack2(float a, float b);
template <>
__device__ __forceinline__ __half2 pack2<__half2>(float a, float b) {
    return __floats2half2_rn(a, b);
}
template <>
__device__ __forceinline__ __nv_bfloat162 pack2<__nv_bfloat162>(float a, float b) {
    return __floats2bfloat162_rn(a, b);
}

template <>
__device__ __forceinline__ float2 pack2<float2>(float a, float b) {
    return make_float2(round_tf32(a), round_tf32(b));
}

__device__ __forceinline__ float2 unpack2(__half2 h) { return __half22float2(h); }
__device__ __forceinline__ float2 unpack2(__nv_bfloat162 h) { return __bfloat1622float2(h); }
__device__ __forceinline__ float2 unpack2(float2 h) { return h; }

// Four complex64 (32 bytes) in one load.
struct Quad {
    float re[4], im[4];
};
__device__ __forceinline__ Quad load_quad(const float2 *p) {
    Quad q;
    asm("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=f"(q.re[0]), "=f"(q.im[0]), "=f"(q.re[1]), "=f"(q.im[1]), "=f"(q.re[2]),
          "=f"(q.im[2]), "=f"(q.re[3]), "=f"(q.im[3])
        : "l"(p)
        : "memory");
    return q;
}

// T2 is a pair of stored elements (two 16-bit numbers, or two FP32 for TF32); the planes and
// strides of d count elements.  A thread takes four elements (d.n is a multiple of four): a
// 32-byte load and an 8-byte store per plane (16 for TF32), each a whole number of sectors per
// warp.  HBM bounds it: 2^23 elements into four planes in 23 us (5.8 TB/s),
// 29.5 us with pairs.
template <typename T2>
__device__ __forceinline__ void convert_body(const ConvertDesc &d, int64_t s, int e) {
    using T = decltype(T2().x);
    struct alignas(2 * sizeof(T2)) T4 {
        T2 lo, hi;
    };
    const Pow2 pe = pow2_of(-e);
    const float2 *src = d.src + s * d.src_sstride;
    T *base = reinterpret_cast<T *>(d.dst) + s * d.dst_sstride;
    T4 *re = reinterpret_cast<T4 *>(base);
    T4 *im = reinterpret_cast<T4 *>(base + d.plane_stride);
    T4 *sm = reinterpret_cast<T4 *>(base + 2 * d.plane_stride);
    T4 *il = reinterpret_cast<T4 *>(base + 3 * d.plane_stride);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < (d.n >> 2);
         i += (int64_t)gridDim.x * blockDim.x) {
        Quad q = load_quad(src + 4 * i);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            q.re[j] = scale_pow2(q.re[j], pe);
            q.im[j] = scale_pow2(q.im[j], pe);
        }
        const T4 rh{pack2<T2>(q.re[0], q.re[1]), pack2<T2>(q.re[2], q.re[3])};
        const T4 ih{pack2<T2>(q.im[0], q.im[1]), pack2<T2>(q.im[2], q.im[3])};
        re[i] = rh;
        im[i] = ih;
        if (d.planes == 3)
            sm[i] = T4{pack2<T2>(q.re[0] + q.im[0], q.re[1] + q.im[1]),
                       pack2<T2>(q.re[2] + q.im[2], q.re[3] + q.im[3])};
        if (d.planes == 4) {
            // lo planes: the rounding residuals x - hi (exact in FP32), rounded again
            const float2 r0 = unpack2(rh.lo), r1 = unpack2(rh.hi);
            const float2 i0 = unpack2(ih.lo), i1 = unpack2(ih.hi);
            sm[i] = T4{pack2<T2>(q.re[0] - r0.x, q.re[1] - r0.y),
                       pack2<T2>(q.re[2] - r1.x, q.re[3] - r1.y)};
            il[i] = T4{pack2<T2>(q.im[0] - i0.x, q.im[1] - i0.y),
                       pack2<T2>(q.im[2] - i1.x, q.im[3] - i1.y)};
        }
    }
}

__global__ void __launch_bounds__(256) k_convert16(ConvertDesc d) {
    const int64_t s = blockIdx.y;
    const int e = scale_exponent(d.amax[s]);
    if (blockIdx.x == 0 && threadIdx.x == 0) d.exps[s] = e;
    if (d.dtype == 2) convert_body<float2>(d, s, e);
    else if (d.dtype == 1) convert_body<__nv_bfloat162>(d, s, e);
    else convert_body<__half2>(d, s, e);
}

int grid_for(int64_t work, int threads) {
    int64_t b = (work + threads - 1) / threads;
    if (b < 1) b = 1;
    if (b > 152 * 64) b = 152 * 64;
    return (int)b;
}

}  // namespace

cudaError_t launch_generic(const GenericDesc &d, int64_t slices, cudaStream_t st) {
    const int64_t total = slices << d.rank_c;
    const int lb = d.rank_c < 10 ? d.rank_c : 10;
    int64_t blocks = total >> lb;
    if (blocks > 152 * 16) blocks = 152 * 16;
    if (d.nk == 0 && d.rank_c >= 10) {
        // large products: chunks of 4096 outputs; small ones keep more blocks busy with 1024
        if (d.rank_c >= 12 && total >= (int64_t)1 << 23) {
            blocks = total >> 12;
            if (blocks > 152 * 8) blocks = 152 * 8;
            k_generic_k1<8><<<(unsigned)blocks, 256, 0, st>>>(d, total);
        } else {
            k_generic_k1<2><<<(unsigned)blocks, 256, 0, st>>>(d, total);
        }
    } else {
        k_generic<<<(unsigned)blocks, 256, 0, st>>>(d, total);
    }
    return cudaGetLastError();
}

cudaError_t chain_prepare() {
    return cudaFuncSetAttribute(k_chain_shm, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                kChainShmElems * 8);
}

cudaError_t launch_chain_shm(const ChainGroup *groups, int32_t ngroups, const ChainCopy *copies,
                             const ChainRec *recs, const int32_t *levels, int64_t elems,
                             float2 *arena, unsigned int *amax, int64_t sb, int64_t slices,
                             cudaStream_t st) {
    if (ngroups <= 0 || slices <= 0) return cudaSuccess;
    if (elems > kChainShmElems || slices * ngroups > 0x7fffffff) return cudaErrorInvalidValue;
    k_chain_shm<<<(unsigned)(slices * ngroups), kChainShmThreads, (size_t)elems * 8, st>>>(
        groups, ngroups, copies, recs, levels, arena, amax, sb);
    return cudaGetLastError();
}

cudaError_t launch_chain(const ChainItem *items, const int32_t *levels, int32_t nlevels,
                         float2 *arena, unsigned int *amax, int64_t sb, int64_t slices,
                         int32_t cluster, cudaStream_t st) {
    if (nlevels <= 0 || slices <= 0) return cudaSuccess;
    if (cluster < 1 || cluster > kChainMaxCluster || slices * cluster > 0x7fffffff)
        return cudaErrorInvalidValue;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(slices * cluster));
    cfg.blockDim = dim3(kChainThreads);
    cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)cluster;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_chain, items, levels, nlevels, arena, amax, sb, cluster);
}

cudaError_t launch_sparse_leaves(const SparseLeafDesc *leaves_dev, int32_t n, int32_t max_rank,
                                 cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    int64_t chunks = ((1ll << (max_rank < 24 ? max_rank : 24)) + 255) / 256;
    if (chunks > 1024) chunks = 1024;
    if (chunks < 1) chunks = 1;
    k_sparse_leaves<<<dim3((unsigned)n, (unsigned)chunks), 256, 0, st>>>(leaves_dev);
    return cudaGetLastError();
}

cudaError_t launch_sparse_step(const GenericDesc &d, const int32_t *gA, const int32_t *gB,
                               int64_t nconf, cudaStream_t st) {
    if (nconf <= 0) return cudaSuccess;
    const int lb = d.rank_c < 10 ? d.rank_c : 10;
    const int64_t chunks = nconf << (d.rank_c - lb);
    int64_t blocks = lb < 8 ? (chunks + (256 >> lb) - 1) >> (8 - lb) : chunks;
    if (blocks > 152 * 8) blocks = 152 * 8;
    (d.nk > 10 ? k_sparse_step<true> : k_sparse_step<false>)<<<(unsigned)blocks, 256, 0, st>>>(
        d, gA, gB, nconf);
    return cudaGetLastError();
}

cudaError_t launch_sparse_amps(const float2 *root, const int32_t *idx, int64_t n, double2 *amps,
                               cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    k_sparse_amps<<<grid_for(n, 256), 256, 0, st>>>(root, idx, n, amps);
    return cudaGetLastError();
}

cudaError_t launch_bind(const BindItem *items_dev, int32_t n_items, const double2 *src,
                        float2 *arena, int64_t slice_begin, int64_t slices, int32_t max_rank,
                        cudaStream_t st) {
    if (n_items == 0 || slices == 0) return cudaSuccess;
    const int threads = max_rank >= 8 ? 256 : (max_rank >= 6 ? 64 : 32);
    int64_t chunks = ((1ll << max_rank) + threads * 8 - 1) / (threads * 8);
    if (chunks > 1024) chunks = 1024;
    if (chunks < 1) chunks = 1;
    k_bind<<<dim3((unsigned)n_items, (unsigned)slices, (unsigned)chunks), threads, 0, st>>>(
        items_dev, src, arena, slice_begin);
    return cudaGetLastError();
}

cudaError_t launch_bind_tiled(const BindTiled &b, const double2 *src, float2 *arena,
                              unsigned int *amax, int64_t slice_begin, int64_t slices,
                              cudaStream_t st) {
    if (slices <= 0) return cudaSuccess;
    if (b.t < 11 || b.t > 12 || slices > 65535 || b.ntiles < 1) return cudaErrorInvalidValue;
    int64_t gx = (152 * 4 + slices - 1) / slices;  // four resident blocks per SM
    if (gx > b.ntiles) gx = b.ntiles;
    const dim3 grid((unsigned)gx, (unsigned)slices);
    if (b.t == 11)
        k_bind_tiled<11><<<grid, 256, 0, st>>>(b, src, arena, amax, slice_begin);
    else
        k_bind_tiled<12><<<grid, 256, 0, st>>>(b, src, arena, amax, slice_begin);
    return cudaGetLastError();
}

cudaError_t launch_accumulate(const float2 *root, int64_t root_sstride, int64_t n, int64_t slices,
                              double2 *amps, cudaStream_t st) {
    // 64 slices of 2^14 / 2^16 amplitudes 15 / 23 us, 4 of 2^20 and 2 of 2^21 19 us: FP64 adds and
    // their latency, then HBM.  (Widened by the FP64 units, a slice after the other: 21 / 38, 33, 33.)
    if (slices == 1 && n > 1)
        k_accumulate<<<grid_for(n >> 1, 256), 256, 0, st>>>(root, n, amps);
    else if (n >= 1 << 18)
        (slices <= 2 ? k_accumulate_slices<2, 2> : k_accumulate_slices<2, 4>)
            <<<grid_for(n >> 1, 256), 256, 0, st>>>(root, root_sstride, n, slices, amps);
    else
        (slices <= 8 ? k_accumulate_slices<1, 4> : k_accumulate_slices<1, 16>)
            <<<grid_for(n, 256), 256, 0, st>>>(root, root_sstride, n, slices, amps);
    return cudaGetLastError();
}

cudaError_t launch_accumulate_batched(const float2 *root, int64_t root_sstride, int64_t n,
                                      int64_t slices, int64_t s0, const AccMap &m,
                                      double2 *amps, cudaStream_t st) {
    if (slices <= 0) return cudaSuccess;
    uint64_t open = 0, vary = (uint64_t)(s0 ^ (s0 + slices - 1));
    for (int j = 0; j < m.nb; ++j) open |= 1ull << m.bj[j];
    for (int j = 1; j < 64; j *= 2) vary |= vary >> j;  // every bit up to the highest that changes
    // setting a thread up costs as much as a few slices, walking a block several at a time costs
    // registers.  Against a thread per root element that walks every slice: 2^16 elements of 128
    // slices, 1 / 6 / 7 of their labels open: 48 / 68 / 76 us (78 / 109 / 130); 2^20 of 4, both
    // open: 37 (36); 2^12 of 256, two open: 19 (123).
    const bool own = (vary & ~open) == 0;
    vary &= open;
    const int log2_n = __builtin_ctzll((uint64_t)n);
    const int nb = __builtin_popcountll(vary);
    const int number = own                                       ? kOwnBlock
                       : nb < 62 && ((int64_t)1 << nb) <= slices ? kByBlock
                                                                 : kFirstOfBlock;
    const int64_t blocks = number == kByBlock ? (int64_t)1 << nb : slices;
    int log2_g = 0;  // threads of a root element: as many as keep the GPU busy
    while (((int64_t)1 << log2_g) < blocks && log2_n + log2_g < 19) ++log2_g;
    auto kernel = own || (slices >> nb) <= 1 ? k_accumulate_batched<1>
                  : (slices >> nb) <= 4 ? k_accumulate_batched<2>
                                        : k_accumulate_batched<16>;
    kernel<<<grid_for((int64_t)1 << (log2_n + log2_g), 256), 256, 0, st>>>(
        root, root_sstride, log2_n, slices, s0, m, open, vary, number, log2_g, amps);
    return cudaGetLastError();
}

cudaError_t launch_readout(const double2 *amps, int64_t n, double *partial, cudaStream_t st) {
    // a block per 1024 amplitudes, up to 4 per SM
    int64_t blocks = (n + 1023) / 1024;
    if (blocks > kReadoutBlocks) blocks = kReadoutBlocks;
    k_readout_partial<<<(unsigned)blocks, 256, 0, st>>>(amps, n, partial);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || blocks == 1) return e;
    k_readout_final<<<1, 256, 0, st>>>(partial, (int32_t)blocks);
    return cudaGetLastError();
}

cudaError_t launch_zero_f64(double2 *p, int64_t n, cudaStream_t st) {
    k_zero_f64<<<grid_for(n, 256), 256, 0, st>>>(p, n);
    return cudaGetLastError();
}

cudaError_t launch_amax(const ConvertDesc &d, int64_t slices, cudaStream_t st) {
    const int gx = grid_for((d.n + 1) / 2, 256);
    const int g = gx > 1024 ? 1024 : gx;
    k_amax<<<dim3((unsigned)g, (unsigned)slices), 256, 0, st>>>(d);
    return cudaGetLastError();
}

cudaError_t launch_convert16(const ConvertDesc &d, int64_t slices, cudaStream_t st) {
    if (d.n & 3) return cudaErrorInvalidValue;
    const int gx = grid_for(d.n / 4, 256);
    const int g = gx > 2048 ? 2048 : gx;
    k_convert16<<<dim3((unsigned)g, (unsigned)slices), 256, 0, st>>>(d);
    return cudaGetLastError();
}

}  // namespace tn
