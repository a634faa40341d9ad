// The single-launch kernel for layers whose blocks own few columns, and for products from a list (included by
// celty_kernels.cu inside its anonymous namespace, after celty_fused.cuh, whose streaming steps, waits and copies it uses):
// LANE_TILE layout, one slab per block, bulk reduce-add merge, no clusters.
//
// What bounds a call on such a layer is a chain of dependent steps, and in k_spmspv_fused the longest part of it is the way
// from x to the first copy: threshold all of x, rank the survivors, cut the list into equal shares, look the shares up,
// 4 100 cycles.  Here columns are dealt to blocks whatever x is (direct_column): runs of two neighbouring columns go round
// the blocks of a row part, and every round starts three blocks further on.  If each block streamed the survivors of its own
// columns, the busiest block, which sets the time, would have a quarter more than the mean (4096 x 4096 at 50 %: 35 columns, mean
// 28).  So up to 16 neighbouring blocks form a group (direct_groups), whose warps hold the group's columns, one per lane: every
// block of a group thresholds the same up to 512 activations, and takes every size-th survivor (direct_taker; busiest block 31
// columns).  The lane that holds one of the block's columns takes the next place among the block's items, notes the column, and
// starts its copy itself if it is one of a team's first; the sub-block offset was loaded while the previous kernel drained.
// Neither a block barrier nor a look-up lies between x and the first copy.  The
// accumulators, which no offset window needs before the first copies here, are cleared while the previous kernel drains as
// well (a tenth of a call's time at 4096 x 4096: cleared under the first copies they held these up).
//
// What is left of imbalance is the difference between groups.  Device time with 50 % of the weights, in us, k_spmspv_fused / blocks with columns of their
// own / this kernel, by columns per block (mean of 6 draws; the first figure of 16):
//    14 (1024 x 1024, d = 0.5)              3.80 / 3.20 / 3.22
//    56 (4096 x 4096, 0.1 / 0.5 / 0.7)      4.82 / 3.94 / 3.86, 7.79 / 6.24 / 5.80, 8.65 / 7.82 / 7.27
//    70 (5120 x 5120, 0.4)                  7.38 -> 6.58
//    75 (4096 x 11008, 0.5)                 12.26 / 11.80 / 10.91
//    84 (11008 x 4096, 0.1 / 0.5)           6.92 / 5.63 / 5.22, 11.63 / 11.43 / 10.68
//   111 (14336 x 4096, 0.5)                 12.86 / 12.97 / 12.19
//   111 (8192 x 8192, 0.5)                  14.26 / 14.80 / 13.57
// Beyond 128 columns per block a ranking lane may hold one, two or four of the group's columns, k_spmspv_fused -> this one, one vector:
//   128 (40 x 18945, 0.5)                   6.83 -> 5.73
//   139 (13824 x 5120, 0.1 / 0.5)           7.16 -> 5.73, 14.92 -> 14.03
//   187 (5120 x 13824, 0.1 / 0.5)           7.30 -> 6.01, 15.69 -> 13.75
//   139 (8192 x 10240, 0.1 / 0.3 / 0.5 / 0.7)   7.79 -> 6.34, 12.61 -> 11.79, 16.57 -> 15.71, 20.50 -> 19.60
//   198 (9700 x 9700, 0.5)                  18.52 -> 17.00
//   276 (20000 x 8000, 0.5)                 26.15 -> 26.06
//   332 (16384 x 12288, 0.1 / 0.5 / 0.7)    10.89 -> 9.99, 30.57 -> 30.50, 40.26 -> 39.78
//   387 (8192 x 28672, 0.3 / 0.5)           24.55 -> 23.59, 35.47 -> 34.38
// The gain shrinks with the
// columns, whose streaming outgrows what is saved ahead of it; the line, 512 (four members' columns at four per lane), lies beyond
// what was measured.  Where k_spmspv_fused lets the left-over blocks serve several row parts (one vector, eight or twelve parts), which
// saves it 2 % of the streaming, the line is 384:
//   144 (28672 x 2600, 0.1 / 0.3 / 0.5 / 0.7)   7.18 -> 6.19, 11.38 -> 9.79, 15.10 -> 14.44, 18.79 -> 17.80
//   228 (28672 x 4096, 0.1 / 0.3 / 0.5 / 0.7)   8.30 -> 7.39, 15.06 -> 13.89, 19.94 -> 19.63, 25.63 -> 24.71
//   361 (28672 x 6500, 0.1 / 0.3 / 0.5 / 0.7)   10.58 -> 9.80, 19.88 -> 19.02, 27.76 -> 27.58, 36.26 -> 36.32
//   455 (28672 x 8192, 0.1 / 0.5)               11.7 -> 10.9, 33.3 -> 33.6
// and for several vectors, with so many groups that one of them is far from the mean, columns times rows per lane may be 20 000 (N
// vectors at 50 %; the last three beyond the line):
//   4096 x 4096, N = 4 / 5 (14 100, 18 000)     14.3 -> 13.4, 17.3 -> 15.9
//   2048 x 6200, N = 4 (10 700)                 12.1 -> 11.0;     2000 x 9000, N = 4 (15 600)   15.6 -> 14.1
//   2558 x 6286, N = 6 (21 000)                 17.7 -> 17.8 (with 39 % of the weights 16.7 -> 18.3)
//   6000 x 3000, N = 6 (24 000)                 18.2 -> 18.9;     4928 x 3456, N = 7 (27 600)   20.1 -> 19.9 (35 %: 20.7 -> 23.3)
// Runs of two, so that survivors that lie together in x (zeroed heads of an attention output) are shared about as evenly as independent ones.
// A list is shared evenly whatever its length; the second
// product of the 5504 x 2048 MLP chain gains 1.9 of 15.4 us from this kernel.
//
// Roles of a block's warps: the first ones threshold the group's columns and stream (a2 - a4; with pairs warps t and t + 8 for team t), the
// next make the survivor list that the API reports, in a few blocks; the last clears the block's share of y, takes its ticket, waits
// for the others' and works out where the block's row segments go.
constexpr int kDirectHelpers = 3;        // at least; 20 warps leave a thread 96 registers
constexpr int kDirectThreads = 32 * (16 + kDirectHelpers + 1);

// kPairs: two warps per team that take turns at its accumulator; kBatch: one launch for several vectors
// (DirectParams::ldx); kHeld: columns of the group per ranking lane; 0: the survivors come as a list (DirectParams::list), in
// equal shares for all teams.
template <bool kPairs, bool kBatch, int kHeld>
__device__ __forceinline__ void dealt_product(const DirectParams p)
{
    constexpr bool kList = kHeld == 0;
    constexpr int kArray = kList ? 1 : kHeld;
    const uint16_t *const x = kBatch ? p.x + (size_t)blockIdx.y * p.ldx : p.x;
    float *const y = kBatch ? p.y + (size_t)blockIdx.y * p.ldy : p.y;
    uint32_t *const tickets = kBatch ? p.tickets + blockIdx.y : p.tickets;
    const bool lists = !kList && (!kBatch || blockIdx.y + 1 == gridDim.y);    // the survivor list reported is the last vector's
    extern __shared__ __align__(128) uint8_t smem[];
    const int tid = threadIdx.x, lane = tid & 31, nthreads = blockDim.x, nwarps = nthreads >> 5;
    const int warp = __shfl_sync(kFull, tid >> 5, 0);             // the same for all lanes, and the compiler knows it
    const int slab_words = (p.R + kTileSlack) * 32;
    const int G = p.G;
    constexpr int pp = kPairs ? 1 : 0, stride = 1 + pp;
    const bool streams = kPairs ? (warp & 7) < G && warp < 16 : warp < G;
    const int g = streams ? (kPairs ? (warp & 7) : warp) : 0;     // the team
    const int half = streams && kPairs ? warp >> 3 : 0;           // which of its two warps
    const int Dw = p.D / stride;                                  // ring slots per warp
    const DirectSmem &lay = p.lay;
    float *acc = reinterpret_cast<float *>(smem);
    uint8_t *ring = smem + lay.ring;
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + lay.bars);
    uint2 *items = reinterpret_cast<uint2 *>(smem + lay.items);   // [team][cap] {offset/16, units of 16 bytes << 16 | x bits}
    int *zero_group = reinterpret_cast<int *>(smem + lay.zero);
    int *taken = reinterpret_cast<int *>(smem + lay.taken);       // survivors that the block has taken
    uint32_t *kbw = reinterpret_cast<uint32_t *>(smem + lay.keep);
    volatile int *flags = reinterpret_cast<volatile int *>(smem + lay.flag);     // [G] a warp of the team gave up

    // Row part s (one slab) and place of this block in it.
    const int per_part = idiv_small(gridDim.x, p.P), kslice = idiv_small(blockIdx.x, p.P), s = blockIdx.x - kslice * p.P;
    const bool long_part = s < (int)gridDim.x - per_part * p.P;
    const int nK = per_part + (long_part ? 1 : 0);
    const float nK_inv = __fdividef(1.f, (float)nK);
    const DirectGroup group = kList ? DirectGroup{} : direct_group(kslice, long_part ? p.sizes[1] : p.sizes[0]);
    const int rankers = kList ? 0 : p.rankers;                    // warps that rank the group's columns
    const int takers = kPairs ? 16 : max(rankers, G);             // these and those that stream: they meet at barrier 15
    const int first_helper = takers, helpers = nwarps - 1 - first_helper;
    int column[kArray];                                        // that the lane holds (K or more: none)
#pragma unroll
    for (int c = 0; c < kHeld; ++c) column[c] = warp < rankers ? direct_held(kHeld * (tid - lane) + 32 * c + lane, group, nK, nK_inv) : p.K;

    // Programmatic dependent launch: see k_spmspv_fused.
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    uint32_t place0[kArray], place1[kArray];                // offset/16 of the columns' sub-blocks, and of the next ones
    auto load_place = [&]() {
#pragma unroll
        for (int c = 0; c < kHeld; ++c) {
            place0[c] = place1[c] = 0u;
            if (column[c] >= p.K) continue;
            place0[c] = p.meta[(size_t)column[c] * p.S + s];
            place1[c] = p.meta[(size_t)column[c] * p.S + s + 1];
        }
    };
    if (p.image_early) load_place();
    if (tid < 4) zero_group[tid] = 0;
    if (tid == 0) *taken = 0;
    if (tid < G) const_cast<int *>(flags)[tid] = 0;
    if (streams && lane == 0) {
#pragma unroll 1
        for (int d = 0; d < Dw; ++d) mbar_init(smem_u32(&bars[g * p.D + half * Dw + d]), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (streams) {
        float4 *slab4 = reinterpret_cast<float4 *>(acc + (size_t)g * slab_words);
#pragma unroll 1
        for (int i = half * 32 + lane; i < slab_words / 4; i += 32 * stride) slab4[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __syncthreads();
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (!p.image_early) load_place();

    const uint32_t lt_mask = (1u << lane) - 1u;
    // The lane has found item k of team `to`: it notes it, and starts its copy if it is one of the first.  (Copies that an
    // elected lane starts when all are found: 0.2 us slower at 4096 x 4096.)
    auto found = [&](int to, int k, const uint2 at, uint32_t xb) {
        (items + (size_t)to * p.cap)[k] = make_uint2(at.x, at.y << 16 | xb);
        if (k >= p.D) return;
        const int slot = to * p.D + (kPairs ? (k & 1) * Dw + (k >> 1) : k);          // a pair's warps take turns
        bulk_load(smem_u32(ring + (size_t)slot * p.slot_bytes), p.stream + (size_t)at.x * 16, at.y * 16u, smem_u32(&bars[slot]));
    };
    // The group's survivors are dealt to its blocks, a ranking warp's one after the other, beginning with a block of the warp's
    // own: what a block has differs by one per warp at most, and no warp has to know the others' counts.  In the block they go
    // to the teams in the order in which they are found.  (Exact ranks through shared memory, a barrier and two reductions:
    // 5120 x 5120 at 40 % 7.08 us instead of 6.83, 4096 x 11008 at 50 % 11.1 instead of 10.9, 4096 x 4096 level.)
    if (warp < rankers) {
        uint32_t xb[kArray];
        int n = 0;
#pragma unroll
        for (int c = 0; c < kHeld; ++c) xb[c] = column[c] < p.K ? x[column[c]] : 0u;
#pragma unroll
        for (int c = 0; c < kHeld; ++c) {
            const bool keep = column[c] < p.K && !(fabsf(__half2float(__ushort_as_half((uint16_t)xb[c]))) <= p.tau);
            const uint32_t kept = __ballot_sync(kFull, keep);
            if (keep && direct_taker(n + __popc(kept & lt_mask), warp, p.rankers_inv, group) == kslice - group.first) {
                const int i = atomicAdd(taken, 1), k = i * (int)p.G_inv >> 16;
                found(i - k * G, k, make_uint2(place0[c], place1[c] - place0[c]), xb[c]);
            }
            n += __popc(kept);
        }
    }
    if (!kList && warp < takers) asm volatile("bar.sync 15, %0;" ::"r"(32 * takers) : "memory");       // the items are there

    // The list that the API reports is made by a few blocks, eight words of x each (2048 x 5504 with 16 each: 0.3 us slower).
    const int nfull = p.K >> 5, nwords = (p.K + 31) >> 5;
    const int list_blocks = min((int)gridDim.x, (nwords + 7) >> 3);
    const bool listing = lists && (int)blockIdx.x < list_blocks;
    if (streams) {
        const uint32_t slab0 = smem_u32(acc + (size_t)g * slab_words);
        const uint32_t cell0 = slab0 + 4u * lane;
        const uint32_t ring0 = smem_u32(ring + ((size_t)g * p.D + (size_t)half * Dw) * p.slot_bytes);
        const uint32_t bar0 = smem_u32(&bars[g * p.D + half * Dw]);
        uint2 *const mine = items + (size_t)g * p.cap;
        auto team_sync = [&]() {                                  // the warp alone, or the two warps of the team
            if (kPairs) asm volatile("bar.sync %0, 64;" ::"r"(2 + g) : "memory");
            else __syncwarp();
        };
        int cnt = 0;
        if (kList) {
            const int n = __shfl_sync(kFull, max(0, min(p.K, __ldcg(p.list_count))), 0);
            if (blockIdx.x == 0 && tid == 0) *p.count = n;
            const int units = nK * G, u = kslice * G + g;
            const uint32_t units_inv = long_part ? p.list.units_inv_long : p.list.units_inv;
            uint32_t each = __umulhi((uint32_t)n, units_inv), extra = (uint32_t)n - each * (uint32_t)units;
            if (extra >= (uint32_t)units) { ++each; extra -= (uint32_t)units; }
            const int r0 = u * (int)each + min(u, (int)extra);
            cnt = (int)each + (u < (int)extra ? 1 : 0);
            for (int k = half + stride * lane; k < cnt; k += stride * 32) {
                const int j = min(max(__ldcg(p.list.idx + r0 + k), 0), p.K - 1);
                const uint32_t xb = __ldcg(p.x + r0 + k);
                const uint32_t at = p.meta[(size_t)j * p.S + s];
                found(g, k, make_uint2(at, p.meta[(size_t)j * p.S + s + 1] - at), xb);
            }
        } else {
            const int n = *taken;
            cnt = n > g ? idiv_small(n - g + G - 1, G) : 0;
        }
        uint32_t slot = 0, parity = 0, consumed = 0;              // of this warp's Dw slots
        uint32_t issued = (uint32_t)min(Dw, (cnt - half + pp) >> pp), islot = issued == (uint32_t)Dw ? 0 : issued;   // (cnt >= 0, half <= 1)
        auto issue = [&](const uint2 it) {
            bulk_load_elected(ring0 + islot * (uint32_t)p.slot_bytes, p.stream + (size_t)it.x * 16, (it.y >> 16) * 16u, bar0 + 8u * islot);
            ++issued;
            if (++islot == (uint32_t)Dw) islot = 0;
        };
        if (kList) team_sync();
        bool failed = false;
        const uint32_t zeros = smem_u32(zero_group), spare_cell = cell0 + (uint32_t)p.R * 128u;
        StepBuf b0, b1;                                           // pipeline registers, live across items
#pragma unroll 1
        for (int i = half; i < cnt; i += stride) {
            uint32_t xbits;                                       // the column's activation: asked for before the wait
            asm volatile("ld.shared.u32 %0, [%1];" : "=r"(xbits) : "r"(smem_u32(&mine[i].y)));
            if (!failed && !mbar_wait_bounded(bar0 + 8u * slot, parity, p.spin_limit)) failed = true;
            failed = __any_sync(kFull, failed);
            if (__builtin_expect(failed, 0)) {
                // The copies still in flight are awaited below.  A warp that gave up keeps meeting its partner at the
                // hand-overs, so that nobody waits for it in vain.
                if (!kPairs) break;
                if (lane == 0) flags[g] = 1;
                if (i > 0) team_sync();
                if (i + 1 < cnt) team_sync();
                continue;
            }
            const uint32_t sub = ring0 + slot * (uint32_t)p.slot_bytes;
            // what the refill at the end of this sub-block will need, read now so that it does not wait then
            const bool refill = i + stride * Dw < cnt;
            const uint2 next = refill ? mine[i + stride * Dw] : make_uint2(0u, 0u);
            const uint16_t xj = (uint16_t)xbits;
            // ---- a3 + a4.  Header: groups per lane, vectors and steps (see kSubHeader).
            uint32_t gl, hw;
            asm volatile("ld.shared.u8 %0, [%1];" : "=r"(gl) : "r"(sub + lane));
            asm volatile("ld.shared.u32 %0, [%1];" : "=r"(hw) : "r"(sub + 32));       // vectors | steps << 16
            const uint32_t steps = hw >> 16, Gs = hw & 0xFFFFu;
            const uint32_t vbase = sub + kSubHeader, rbase = vbase + 16 * Gs;
            uint32_t cum = 0, cell = cell0;
            step_fetch(b0, gl, 0, steps, cum, lt_mask, vbase, rbase, zeros);
            step_fetch(b1, gl, 1, steps, cum, lt_mask, vbase, rbase, zeros);
            // nothing above touches the accumulator: here the partner hands it over (it has finished the column
            // before this one)
            if (kPairs && i > 0) team_sync();
            step_decode<0>(b0, cell, spare_cell, 0);                                    // step 0
            step_fetch(b0, gl, 2, steps, cum, lt_mask, vbase, rbase, zeros);
            uint32_t q = 1;
#pragma unroll 2
            for (; q + 1 < steps; q += 2) {                                            // two real steps per pass
                step_decode<0>(b1, cell, spare_cell, 0);                                // step q
                step_finish(b0, xj);                                                   // step q-1
                step_fetch(b1, gl, q + 2, steps, cum, lt_mask, vbase, rbase, zeros);
                step_decode<0>(b0, cell, spare_cell, 0);                                // step q+1
                step_finish(b1, xj);                                                   // step q
                step_fetch(b0, gl, q + 3, steps, cum, lt_mask, vbase, rbase, zeros);
            }
            if (q < steps) {                                                           // one real step left
                step_decode<0>(b1, cell, spare_cell, 0);
                step_finish(b0, xj);
                step_finish(b1, xj);
            } else {                                                                   // only the last one to finish
                step_finish(b0, xj);
            }
            // The slot's contents were consumed by loads whose values have been used, and the barrier orders
            // every lane's reads before this point: the copy may overwrite it.
            __syncwarp();
            if (refill) issue(next);
            if (kPairs && i + 1 < cnt) team_sync();               // the accumulator goes to the partner
            ++consumed;
            if (++slot == (uint32_t)Dw) { slot = 0; parity ^= 1u; }
        }
        if (kPairs) team_sync();                                  // both warps are through with the accumulator
        if (__builtin_expect(failed || (kPairs && flags[g]), 0)) {
            // The copies that are still in flight have to land before the block goes on: after it their place is another
            // block's.  With the library's limit, whatever the call's is.
#pragma unroll 1
            for (; consumed < issued; ++consumed) {
                mbar_wait_bounded(bar0 + 8u * slot, parity, kSpinLimit);
                if (++slot == (uint32_t)Dw) { slot = 0; parity ^= 1u; }
            }
            // the rows of this slab are NaN then: celty_spmspv_static has no status word that its caller could read
#pragma unroll 1
            for (int w = lane; w < slab_words; w += 32) acc[(size_t)g * slab_words + w] = __int_as_float(0x7FC00000);
            if (lane == 0) atomicOr(p.status, kStatusTimeout);
        }
    } else if (warp == nwarps - 1) {
        // The adds at the end need a cleared y: this warp clears the block's share and announces it.
        const int b = (int)blockIdx.x;
        const int r0 = b * p.clear_rows + min(b, p.clear_extra), r1 = r0 + p.clear_rows + (b < p.clear_extra ? 1 : 0);
        uint32_t ticket = 0;
        if (p.tickets) {
#pragma unroll 1
            for (int i = r0 + lane; i < r1; i += 32) y[i] = 0.f;
            __syncwarp();
            if (lane == 0) {
                asm volatile("fence.acq_rel.gpu;" ::: "memory");
                // The ticket counts modulo 2 * gridDim.x, so it never has to be reset: calls alternate between
                // waiting for the lower and for the upper half.
                ticket = atomicInc(&tickets[0], 2u * gridDim.x - 1u);
            }
        }
        if (listing) {                                            // the word that the end of x cuts short
            const int j = 32 * nfull + lane;
            const bool kept = j < p.K && !(fabsf(__half2float(__ushort_as_half(x[j]))) <= p.tau);
            const uint32_t word = __ballot_sync(kFull, kept);
            if (lane == 0 && nfull < nwords) kbw[nfull] = word;
            __syncwarp();
            asm volatile("bar.arrive 1, %0;" ::"r"(32 * helpers + 32) : "memory");
        }
        if (!kBatch && blockIdx.x == 0 && lane == 0 && p.ep_count) *p.ep_count = 0;      // k_epilogue appends to it
        if (lane == 0) {
            if (__builtin_expect(p.tickets && !ticket_wait<true>(tickets, ticket, p.spin_limit), 0)) atomicOr(p.status, kStatusTimeout);
            // the others' clearing stores (generic proxy) come before this block's reduce-adds (asynchronous proxy)
            asm volatile("fence.proxy.async.global;" ::: "memory");
        }
    } else if (listing && warp >= first_helper) {
        // ---- a1 for all of x: a thread makes keep words of 32 activations each
        const int hw = warp - first_helper;
        const __half2 tau2 = __half2half2(__float2half_rd(p.tau));   // |x| > tau decided in FP16, as in k_spmspv_fused
#pragma unroll 1
        for (int w = tid - 32 * first_helper; w < nfull; w += 32 * helpers) kbw[w] = keep_word32(x + 32 * w, tau2);
        asm volatile("bar.sync 1, %0;" ::"r"(32 * helpers + 32) : "memory");   // with the last warp, for the short word
        // the list, a few words per block and warp
#pragma unroll 1
        for (int w = (int)blockIdx.x + list_blocks * hw; w < nwords; w += list_blocks * helpers) {
            uint32_t before = 0;
            for (int e = lane; e < w; e += 32) before += (uint32_t)__popc(kbw[e]);
            before = __reduce_add_sync(kFull, before);
            const uint32_t word = kbw[w];
            if (word >> lane & 1u) {
                const int pos = (int)before + __popc(word & ((1u << lane) - 1u)), j = 32 * w + lane;
                p.idx[pos] = j;
                p.val[pos] = x[j];
            }
            if (w == nwords - 1 && lane == 0) *p.count = (int)before + __popc(word);
        }
    }
    // Row segments, see k_spmspv_fused.  The last warp, one segment per lane, works out where they go under the streaming.
    const int seg = p.S == 1 ? 16 : p.C, nseg = idiv_small(p.R + seg - 1, seg);
    struct Segment { float *to; const float *from; int nrows; };
    auto segment = [&](int k) {
        const int i0 = k * seg, i1 = min(p.R, i0 + seg);
        const int64_t row0 = p.S == 1 ? (int64_t)i0 * 32 : ((int64_t)(k * p.S + s) * p.C) * 32;
        return Segment{y + row0, acc + (size_t)i0 * 32, row0 >= p.M ? 0 : min((i1 - i0) * 32, p.M - (int)row0)};
    };
    Segment early{nullptr, nullptr, 0};
    if (kPairs && warp == nwarps - 1 && lane < nseg) early = segment(lane);
    __syncthreads();

    // ---- a5: the G accumulators are added into the first one, and each row segment goes to y as one bulk reduce-add.
    if (G > 1) {
        float4 *acc4 = reinterpret_cast<float4 *>(acc);
        const int team4 = slab_words / 4;
#pragma unroll 1
        for (int q4 = tid; q4 < p.R * 8; q4 += nthreads) {
            float4 v = acc4[q4];
#pragma unroll 4
            for (int t = 1; t < G; ++t) {
                const float4 u = acc4[(size_t)t * team4 + q4];
                v.x += u.x; v.y += u.y; v.z += u.z; v.w += u.w;
            }
            acc4[q4] = v;
        }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
#pragma unroll 1
    for (int o = kPairs ? (warp == nwarps - 1 ? lane : nseg) : tid; o < nseg; o += kPairs ? 32 : nthreads) {
        const Segment sg = kPairs && o == lane ? early : segment(o);
        const uint32_t bytes = ((uint32_t)sg.nrows * 4u) & ~15u;
        if (sg.nrows <= 0) continue;
        if (bytes)
            asm volatile("cp.reduce.async.bulk.global.shared::cta.bulk_group.add.f32 [%0], [%1], %2;" ::"l"(sg.to),
                         "r"(smem_u32(sg.from)), "r"(bytes)
                         : "memory");
#pragma unroll 1
        for (int i = (int)(bytes >> 2); i < sg.nrows; ++i)
            if (sg.from[i] != 0.f) atomicAdd(sg.to + i, sg.from[i]);
    }
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
    asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");   // shared memory may go once it has been read
}

// (The same body in the kernel itself compiles to slower code: 11008 x 4096 with its FP16 copy 10.55 us instead of 10.51.)
template <bool kPairs, bool kBatch, int kHeld>
__global__ void __launch_bounds__(kDirectThreads, 1) k_spmspv_direct(const DirectParams p)
{
    dealt_product<kPairs, kBatch, kHeld>(p);
}
