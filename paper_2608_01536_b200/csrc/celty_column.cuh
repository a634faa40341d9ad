// The SpMSpV kernel for the COLUMN layout: the formulation of Sections 3.1-3.3 as published, whole columns decoded
// with the intra-warp prefix sum of Algorithm 1 (included by celty_kernels.cu inside its anonymous namespace, after
// celty_fused.cuh).
//
// A thread block takes an equal share of the surviving columns; inside it, groups of W warps take one column at a
// time, warp w of a group the chunks w, W + w, ... of 256 entries.  The entries of one column are different rows, so
// the warps of a group add into one accumulator of M floats with plain load / fma / store: no two of them ever hold
// the same row, and no atomics are needed (a shared-memory FP32 atomic add is a compare-and-swap loop).  What the
// warps do exchange is where their chunk starts: each scans its own chunk (Algorithm 1), posts the rows it spans and
// meets the others at a named barrier, which also keeps the group's columns apart (nobody scatters column i + 1
// before everybody has scattered column i).  Two chunks per warp are loaded ahead of the one being scattered.
//
// What bounds it: shared memory.  The rows of the 32 lanes fall on the banks as good as at random (8 entries, or
// some 16 rows at 50 % density, lie between two lanes), so a load or store takes 3 to 4 wavefronts where the lane
// tiles' takes one; entries per SM / 32 x 7 wavefronts is 3.2 us at 4096 x 4096, 50 % / 50 %.  Measured there:
// 11.6 us against 41.6 us for warps that each took whole columns and added with shared-memory atomics, behind a
// one-block compaction kernel; 10.2 with dealt columns.
//
// kDealt (column_dealt says where): a block's columns as in k_spmspv_direct, dealt to groups of blocks that share the survivors, instead of
// every block ranking all of x and looking its share up behind five block barriers.  Device time in us, ranked -> dealt: 4096 x 4096 at 10 % /
// 50 % 6.88 -> 5.55, 11.59 -> 10.24;  1000 x 1000 5.81 -> 4.15;  2048 x 8192 at 30 % 8.80 -> 7.68;  7000 x 2300 11.41 -> 10.84.  (The next
// chunk's scan moved under this one's loads: 0.1 to 0.3 us slower, with the loads of x ahead by one chunk more or not.)
//
// a0: k_clear clears y ahead of this kernel (11.4 us where every block cleared its share and all waited for one
// another's ticket, but a call must not need all SMs at once).  a1 as in the fused kernel: every block thresholds all of
// x; where K's keep words leave no room the list comes from k_compact, which also clears y.

struct ColumnParams {
    const uint2 *meta;          // [K] {offset/16, entries}
    const uint8_t *stream;
    const uint16_t *x;
    float tau;
    int32_t *idx;               // the compacted list: written here, or read when own_list is 0
    uint16_t *val;
    int32_t *count;
    float *y;                   // zero: the kernel before this one cleared it
    uint32_t *status;
    int M, K;
    int W, groups;              // warps per column, columns in flight per block (W * groups <= 32, groups <= 15 if W > 1)
    int cap;                    // columns a block looks up at a time
    int own_list;               // 1: threshold x here
    // kDealt: columns are dealt to groups of blocks as in k_spmspv_direct
    celty::DirectSizes sizes;
    int rankers;
    float rankers_inv;
    uint32_t dealt;             // where the block's columns go in shared memory, {column, x bits} of most, then {offset/16, entries}
    int most;
};

constexpr int kColumnThreads = 1024;

// The group of 8 activations that the end of x cuts short (K not a multiple of 8), zero-filled.  Out of line: one
// thread of a block needs it, if any, and the thresholding pass is unrolled four times around the call.
__device__ __noinline__ uint4 ragged_group(const uint16_t *x, int K, int q)
{
    uint32_t h[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const uint32_t lo = (8 * q + 2 * k < K) ? x[8 * q + 2 * k] : 0u;
        const uint32_t hi = (8 * q + 2 * k + 1 < K) ? x[8 * q + 2 * k + 1] : 0u;
        h[k] = lo | (hi << 16);
    }
    return make_uint4(h[0], h[1], h[2], h[3]);
}

// One keep bit per activation of x[32w .. 32w+31] (zero past the end of x).  Plain loads, as in the fused kernel: x may be
// the work of a kernel that has not ended when this one starts.
__device__ __forceinline__ uint32_t keep_word(const uint16_t *x, int K, int w, __half2 tau2)
{
    const int ngroups = (K + 7) >> 3;
    uint32_t word = 0;
    uint4 h[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const int q = 4 * w + c;
        h[c] = make_uint4(0u, 0u, 0u, 0u);                          // never kept (tau >= 0)
        if (8 * q + 8 <= K) h[c] = *reinterpret_cast<const uint4 *>(x + 8 * q);
        else if (q < ngroups) h[c] = ragged_group(x, K, q);
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const uint32_t v[4] = {h[c].x, h[c].y, h[c].z, h[c].w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t le = __hle2_mask(__habs2(*reinterpret_cast<const __half2 *>(&v[k])), tau2);
            word |= ((~le & 1u) | ((~le >> 15) & 2u)) << (8 * c + 2 * k);
        }
    }
    if (32 * w + 32 > K) word &= 32 * w < K ? 0xFFFFFFFFu >> (32 * w + 32 - K) : 0u;
    return word;
}

template <bool kDealt>
__global__ void __launch_bounds__(kColumnThreads, 1) k_spmspv_column(const ColumnParams p)
{
    extern __shared__ __align__(128) uint8_t smem[];
    const ColumnSmem lay = column_smem_layout(p.M, p.K, p.groups, p.cap, p.own_list);
    float *acc = reinterpret_cast<float *>(smem + lay.acc);
    int2 *items = reinterpret_cast<int2 *>(smem + (kDealt ? p.dealt : lay.items));
    uint2 *imeta = kDealt ? reinterpret_cast<uint2 *>(items + p.most) : reinterpret_cast<uint2 *>(smem + lay.imeta);
    int *warp_tot = reinterpret_cast<int *>(smem + lay.warps);
    uint32_t *keep = reinterpret_cast<uint32_t *>(smem + lay.keep);
    int *rank = reinterpret_cast<int *>(smem + lay.rank);
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(kFull, tid >> 5, 0);
    const int Mp = (p.M + 3) & ~3;

    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const float nK_inv = __fdividef(1.f, (float)gridDim.x);
    const DirectGroup group = kDealt ? direct_group((int)blockIdx.x, p.sizes) : DirectGroup{};
    const int column = kDealt && warp < p.rankers ? direct_held(tid, group, (int)gridDim.x, nK_inv) : p.K;      // (K or more: none)
    uint2 place = make_uint2(0u, 0u);
    if (kDealt && column < p.K) place = __ldg(p.meta + column);
    if (kDealt && tid == 0) *warp_tot = 0;                         // columns that the block has taken
    for (int i = tid; i < p.groups * Mp / 4; i += kColumnThreads)
        reinterpret_cast<float4 *>(acc)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    // The block's columns lie around the same fraction of K as the block in the grid: their offsets are fetched now.
    // (The table is part of the image, which no kernel writes.)
    uint2 *const window = reinterpret_cast<uint2 *>(smem + lay.window);
    const int win0 = max(0, min(p.K - kColumnWindow, (int)((float)(2 * blockIdx.x + 1) * (float)p.K / (float)(2 * gridDim.x)) - kColumnWindow / 2));
    if (!kDealt && p.own_list && tid < kColumnWindow && win0 + tid < p.K) window[tid] = __ldg(p.meta + win0 + tid);
    if (kDealt) __syncthreads();
    asm volatile("griddepcontrol.wait;" ::: "memory");

    int n = 0;
    if (kDealt) {
        // ---- a1 as in k_spmspv_direct: the lanes of the ranking warps threshold the columns of the block's group, and every
        // size-th survivor is this block's.  The list for the API comes from the warps that do not stream, in a few blocks.
        if (warp < p.rankers) {
            const uint32_t xb = column < p.K ? p.x[column] : 0u;
            const bool kept = column < p.K && !(fabsf(__half2float(__ushort_as_half((uint16_t)xb))) <= p.tau);
            const uint32_t word = __ballot_sync(kFull, kept);
            if (kept && direct_taker(__popc(word & ((1u << lane) - 1u)), warp, p.rankers_inv, group) == (int)blockIdx.x - group.first) {
                const int i = atomicAdd(warp_tot, 1);
                items[i] = make_int2(column, (int)xb);
                imeta[i] = place;
            }
        }
        __syncthreads();
        n = *warp_tot;
        const int streaming = p.W * p.groups, helpers = 32 - streaming, nwords = (p.K + 31) >> 5;
        const int list_blocks = min((int)gridDim.x, idiv_small(nwords + 2 * helpers - 1, 2 * helpers));
        if (warp >= streaming && (int)blockIdx.x < list_blocks) {
            const __half2 tau2 = __half2half2(__float2half_rd(p.tau));
#pragma unroll 1
            for (int w = tid - 32 * streaming; w < nwords; w += 32 * helpers) keep[w] = keep_word(p.x, p.K, w, tau2);
            asm volatile("bar.sync 15, %0;" ::"r"(32 * helpers) : "memory");
#pragma unroll 1
            for (int w = (int)blockIdx.x + list_blocks * (warp - streaming); w < nwords; w += list_blocks * helpers) {
                uint32_t before = 0;
                for (int e = lane; e < w; e += 32) before += (uint32_t)__popc(keep[e]);
                before = __reduce_add_sync(kFull, before);
                const uint32_t word = keep[w];
                if (word >> lane & 1u) {
                    const int pos = (int)before + __popc(word & ((1u << lane) - 1u)), j = 32 * w + lane;
                    p.idx[pos] = j;
                    p.val[pos] = p.x[j];
                }
                if (w == nwords - 1 && lane == 0) *p.count = (int)before + __popc(word);
            }
        }
    } else if (p.own_list) {
        // ---- a1: keep words and the survivors before each of them
        const __half2 tau2 = __half2half2(__float2half_rd(p.tau));   // |x| > tau decided in FP16, as in the fused kernel
        const int nwords = (p.K + 31) >> 5;
        for (int w0 = 0; w0 < nwords; w0 += kColumnThreads) {          // the same trip count for every thread
            const int w = w0 + tid;
            const uint32_t word = w < nwords ? keep_word(p.x, p.K, w, tau2) : 0u;
            const int cnt = __popc(word);
            int incl = cnt;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int up = __shfl_up_sync(kFull, incl, d);
                if (lane >= d) incl += up;
            }
            if (lane == 31) warp_tot[warp] = incl;
            __syncthreads();
            const int t = warp_tot[lane];
            const int before = __reduce_add_sync(kFull, lane < warp ? t : 0), all = __reduce_add_sync(kFull, t);
            if (w < nwords) {
                keep[w] = word;
                rank[w] = n + before + incl - cnt;
            }
            n += all;
            __syncthreads();
        }
        if (blockIdx.x == 0 && tid == 0) *p.count = n;
    } else {
        n = __ldcg(p.count);
    }

    // n / blocks columns each, the first n mod blocks one more
    const int share = n / (int)gridDim.x, extra = n - share * (int)gridDim.x, b = (int)blockIdx.x;
    const int p0 = kDealt ? 0 : b * share + min(b, extra), p1 = kDealt ? n : p0 + share + (b < extra ? 1 : 0);
    const int g = idiv_small(warp, p.W), w = warp - g * p.W;
    const bool works = g < p.groups;
    float *const a = acc + (size_t)(works ? g : 0) * Mp;
    volatile uint32_t *const spans = reinterpret_cast<uint32_t *>(smem + lay.spans) + (works ? g * p.W : 0);
    const uint32_t acc0 = smem_u32(a), dump = smem_u32(smem + lay.dump) + 4u * lane;
    uint32_t parity = 0;
    bool out_of_range = false;
    for (int b0 = p0; b0 < p1; b0 += kDealt ? n : p.cap) {
        // ---- the columns of ranks b0 .. b0 + cnt - 1
        const int cnt = kDealt ? n : min(p.cap, p1 - b0);
        if (kDealt) {
        } else if (p.own_list) {
            const int nwords = (p.K + 31) >> 5;
            for (int i = tid; i < cnt; i += kColumnThreads) {
                // the last word with rank[] <= r, then the bit: halve the word, keep the half with the wanted set bit
                const int r = b0 + i;
                int at = 0;
                for (int step = 1 << (31 - __clz(nwords)); step; step >>= 1)
                    if (at + step < nwords && rank[at + step] <= r) at += step;
                int k = r - rank[at], pos = 0;
                const uint32_t word = keep[at];
#pragma unroll
                for (int sh = 16; sh; sh >>= 1) {
                    const int c = __popc((word >> pos) & ((1u << sh) - 1u));
                    if (k >= c) { k -= c; pos += sh; }
                }
                const int j = 32 * at + pos;
                const uint16_t xb = p.x[j];
                items[i] = make_int2(j, (int)xb);
                imeta[i] = j >= win0 && j < win0 + kColumnWindow ? window[j - win0] : __ldg(p.meta + j);
                p.idx[r] = j;
                p.val[r] = xb;
            }
        } else {
            for (int i = tid; i < cnt; i += kColumnThreads) {
                const int j = __ldcg(p.idx + b0 + i);
                items[i] = make_int2(j, (int)__ldcg(p.val + b0 + i));
                imeta[i] = __ldg(p.meta + j);
            }
        }
        if (!kDealt) __syncthreads();
        // ---- a2 - a4: this group's columns of the batch
        if (works) {
            const int i1 = idiv_small((g + 1) * cnt, p.groups);          // cnt <= 1024
            int li = idiv_small(g * cnt, p.groups), lc = 0;            // what is loaded next: column, first chunk
            int pi = li, pc = 0;                                       // what is scattered next
            struct Chunk { uint4 v; uint32_t runs; };
            auto next = [&](int &i, int &c) {                          // the group's next W chunks
                c += p.W;
                if ((uint32_t)c * (kChunkGroups * kGroup) >= imeta[i].y) { ++i; c = 0; }
            };
            auto load = [&](Chunk &ch) {
                ch.v = make_uint4(0u, 0u, 0u, 0u);
                ch.runs = 0u;
                if (li >= i1) return;
                const uint2 mj = imeta[li];
                const uint32_t ng = (mj.y + kGroup - 1) / kGroup, c = (uint32_t)(lc + w), first = c * kChunkGroups;
                if (first + lane < ng) {
                    const uint32_t gc = min((uint32_t)kChunkGroups, ng - first);
                    const uint8_t *chunk = p.stream + (size_t)mj.x * 16 + (size_t)c * (kChunkGroups * 20);
                    ch.v = __ldg(reinterpret_cast<const uint4 *>(chunk + 16 * lane));
                    ch.runs = __ldg(reinterpret_cast<const uint32_t *>(chunk + 16 * gc + 4 * lane));
                }
                next(li, lc);
            };
            // The rows a chunk spans (Algorithm 1: inclusive scan over the lanes), posted for the group's other warps.
            struct Spans { uint32_t even, odd, span, sum; };
            auto scan = [&](const Chunk &ch, int i, int c) {
                Spans sp;
                const uint32_t e0 = ((uint32_t)(c + w) * kChunkGroups + lane) * kGroup;
                uint32_t total;
                decode_group(ch.runs, sp.even, sp.odd, total);
                sp.span = i < i1 && e0 < imeta[i].y ? total + kGroup : 0u;
                sp.sum = sp.span;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const uint32_t prev = __shfl_up_sync(kFull, sp.sum, d);
                    if (lane >= d) sp.sum += prev;
                }
                if (p.W > 1 && lane == 31) spans[32 * parity + w] = sp.sum;
                return sp;
            };
            Chunk c0, c1, c2;
            load(c0);
            load(c1);
            uint32_t carry = 0;                                        // rows of the column before the group's chunks
            while (pi < i1) {
                load(c2);
                const uint32_t nent = imeta[pi].y, e0 = ((uint32_t)(pc + w) * kChunkGroups + lane) * kGroup;
                const Spans now = scan(c0, pi, pc);
                uint32_t row0 = carry + now.sum - now.span;
                if (p.W > 1) {
                    asm volatile("bar.sync %0, %1;" ::"r"(1 + g), "r"(32 * p.W) : "memory");
                    const uint32_t t = lane < p.W ? spans[32 * parity + lane] : 0u;
                    row0 += __reduce_add_sync(kFull, lane < w ? t : 0u);
                    carry += __reduce_add_sync(kFull, t);
                    parity ^= 1u;
                } else {
                    carry += __shfl_sync(kFull, now.sum, 31);
                    __syncwarp();                                      // the lanes' stores of the column before this one
                }
                const uint16_t xj = (uint16_t)items[pi].y;
                const uint32_t have = nent > e0 ? min(nent - e0, (uint32_t)kGroup) : 0u;
                // A lane's rows grow, so its last one tells whether all are in range.
                const uint32_t last = row0 + entry_offset(now.even, now.odd, kGroup - 1);
                uint32_t cell[kGroup];
                const uint32_t cell0 = acc0 + 4u * row0;
                cell[0] = __dp4a(now.even, 0x00000004u, cell0);
                cell[1] = __dp4a(now.odd, 0x00000004u, cell0);
                cell[2] = __dp4a(now.even, 0x00000400u, cell0);
                cell[3] = __dp4a(now.odd, 0x00000400u, cell0);
                cell[4] = __dp4a(now.even, 0x00040000u, cell0);
                cell[5] = __dp4a(now.odd, 0x00040000u, cell0);
                cell[6] = __dp4a(now.even, 0x04000000u, cell0);
                cell[7] = __dp4a(now.odd, 0x04000000u, cell0);
                if (!__all_sync(kFull, have == kGroup && last < (uint32_t)p.M)) {   // the end of a column, or of the image
#pragma unroll
                    for (int e = 0; e < kGroup; ++e) {
                        const bool in = cell[e] < acc0 + 4u * (uint32_t)p.M && row0 < (uint32_t)p.M;
                        if ((uint32_t)e < have && !in) out_of_range = true;
                        if ((uint32_t)e >= have || !in) cell[e] = dump;
                    }
                }
                float c[kGroup], d[kGroup];
#pragma unroll
                for (int e = 0; e < kGroup; ++e) c[e] = lds_f32(cell[e]);
                const int before = pi;                                 // (while these loads are on their way: 0.3 us)
                next(pi, pc);
                if (pi != before) carry = 0;
                fma_pair(c0.v.x, xj, c[0], c[1], d[0], d[1]);
                fma_pair(c0.v.y, xj, c[2], c[3], d[2], d[3]);
                fma_pair(c0.v.z, xj, c[4], c[5], d[4], d[5]);
                fma_pair(c0.v.w, xj, c[6], c[7], d[6], d[7]);
#pragma unroll
                for (int e = 0; e < kGroup; ++e) sts_f32(cell[e], d[e]);
                c0 = c1;
                c1 = c2;
            }
        }
        __syncthreads();
    }
    if (out_of_range) atomicOr(p.status, kStatusBounds);
    if (p0 >= p1) return;                                              // (the same for the whole block)
    // ---- a5: the groups' accumulators, then one bulk reduce-add per 512 rows of y
    if (p.groups > 1) {
        float4 *acc4 = reinterpret_cast<float4 *>(acc);
        for (int i = tid; i < Mp / 4; i += kColumnThreads) {
            float4 v = acc4[i];
            for (int gg = 1; gg < p.groups; ++gg) {
                const float4 t = acc4[gg * (Mp / 4) + i];
                v.x += t.x; v.y += t.y; v.z += t.z; v.w += t.w;
            }
            acc4[i] = v;
        }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    for (int r0 = tid * 512; r0 < p.M; r0 += kColumnThreads * 512) {
        // the clearing of y (generic proxy) comes before these adds (asynchronous proxy)
        asm volatile("fence.proxy.async.global;" ::: "memory");
        const int nrows = min(512, p.M - r0);
        const uint32_t bytes = ((uint32_t)nrows * 4u) & ~15u;
        if (bytes)
            asm volatile("cp.reduce.async.bulk.global.shared::cta.bulk_group.add.f32 [%0], [%1], %2;" ::"l"(p.y + r0),
                         "r"(smem_u32(acc + r0)), "r"(bytes)
                         : "memory");
        for (int i = (int)(bytes >> 2); i < nrows; ++i) atomicAdd(p.y + r0 + i, acc[r0 + i]);
    }
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
    asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}
