// The single-launch kernel for layers whose blocks own few columns, and for products from a list (included by
// celty_kernels.cu inside its anonymous namespace, after celty_fused.cuh, whose streaming steps, waits and copies it uses):
// LANE_TILE layout, one slab per block, bulk reduce-add merge, no clusters.
//
// What bounds a call on such a layer is a chain of dependent steps, and in k_spmspv_fused the longest part of it is the way
// from x to the first copy: threshold all of x, rank the survivors, cut the list into equal shares, look the shares up,
// 4 100 cycles.  Here columns are dealt to blocks whatever x is (direct_column): runs of two neighbouring columns go round
// the blocks of a row part, and every round starts three blocks further on.  Every streaming
// warp loads the activations of all the block's columns, one column per lane and chunk of 32; ballots tell each lane the place
// of its column among the block's survivors, and survivor i goes to team i mod G.  The lane that holds one of its team's
// columns notes it, and starts the copy itself if it is one of the first; the sub-block offsets were loaded while the
// previous kernel drained.  Neither a barrier nor a look-up lies between x and the first copy, 1 400 cycles.  The
// accumulators, which no offset window needs before the first copies here, are cleared while the previous kernel drains as
// well (a tenth of a call's time at 4096 x 4096: cleared under the first copies they held these up).
//
// What it costs is balance: the survivors per block differ as they fall, sqrt((1 - d) / (d n)) of n columns at density d,
// where the ranked list is even to one column.  Device time with 50 % of the weights, in us, mean over 16 draws of
// independent survivors, ranked -> this kernel, by columns per block:
//    14 (1024 x 1024, d = 0.1 / 0.5)              3.74 -> 3.30, 3.80 -> 3.30
//    56 (4096 x 4096, 0.1 / 0.3 / 0.5 / 0.7)      4.82 -> 3.95, 6.32 -> 5.29, 7.79 -> 6.89, 8.65 -> 7.94
//    70 (5120 x 5120, 0.3 / 0.5)                  7.27 -> 6.64, 9.29 -> 8.60
//    75 (4096 x 11008, 0.1 / 0.5 / 0.7)           7.70 -> 5.92, 12.26 -> 11.64, 14.36 -> 13.64
//    84 (11008 x 4096, 0.1 / 0.5 / 0.7)           6.92 -> 5.64, 11.63 -> 11.39, 14.19 -> 13.37
//   111 (14336 x 4096, 0.1 / 0.3 / 0.5 / 0.7)     7.01 -> 5.91, 9.87 -> 9.38, 12.86 -> 12.82, 15.64 -> 15.45
//   111 (8192 x 8192, 0.1 / 0.3 / 0.5 / 0.7)      7.68 -> 6.43, 10.77 -> 10.91, 14.26 -> 14.63, 17.58 -> 17.56
// and with a build for six chunks
//   138 (8192 x 10240, 0.1 / 0.3 / 0.5 / 0.7)     8.06 -> 7.20, 12.59 -> 12.77, 16.40 -> 16.77, 20.54 -> 20.66
//   139 (13824 x 5120, 0.1 / 0.5 / 0.7)           7.09 -> 6.61, 14.60 -> 14.60, 18.18 -> 17.87
//   187 (5120 x 13824, 0.1 / 0.5 / 0.7)           7.29 -> 6.41, 15.42 -> 14.39, 18.62 -> 17.77
// so the line, four chunks, lies where the first layer is slower from 30 % on; it gives away what other shapes would gain beyond.
// Survivors that lie together in x are shared about as evenly as independent ones.  Half of the 128-column heads zeroed,
// ranked / runs of 32 columns / of 8 / of 4 / of two:   4096 x 4096 7.7 / 8.5 / 7.2 / 6.9 / 6.6;   4096 x 11008 12.2 / 15.2 / 15.7 /
// 12.2 / 11.5;   8192 x 8192 14.3 / 18.6 / 15.8 / 14.9 / 13.9.  Single columns are no more even, and loads of x that touch a
// sector per column cost 1 to 6 %.  Independent survivors take 1 to 3 % more with runs of two than with runs of 32 on layers
// of 84 columns per block and more (8192 x 8192 at 10 %: 4 %), whose blocks now reach over all of a large image, and 2 to 6 % less
// below.  One warp per chunk that shares its ballot and its activations with the others through shared memory behind a barrier,
// or the two warps of a pair half of the chunks each: 0 to 2 % slower.
// Groups of 2 to 32 blocks that share their columns' survivors evenly, ranked
// shares of the columns beyond a fixed core under the streaming: both slower (more code and loads on the way to the first
// copy, or a streaming loop that the compiler schedules worse).  A list is shared evenly whatever its length; the second
// product of the 5504 x 2048 MLP chain gains 1.9 of 15.4 us from this kernel.
//
// Roles of a block's warps: the first ones stream (a2 - a4; with pairs warps t and t + 8 for team t), the next make the
// survivor list that the API reports, in a few blocks; the last clears the block's share of y, takes its ticket, waits
// for the others' and works out where the block's row segments go.
constexpr int kDirectHelpers = 3;        // at least; 20 warps leave a thread 96 registers
constexpr int kDirectThreads = 32 * (16 + kDirectHelpers + 1);
static_assert(kDirectChunks <= kDirectHelpers + 1, "a thread of the warps that do not stream for each of a block's columns");

// kPairs: two warps per team that take turns at its accumulator; kBatch: one launch for several vectors
// (FusedParams::ldx); kChunks: chunks of 32 columns that the block's columns fit in, 2 or 4; 0: the
// survivors come as a list (FusedParams::list_count), in equal shares for all teams.
template <bool kPairs, bool kBatch, int kChunks>
__global__ void __launch_bounds__(kDirectThreads, 1) k_spmspv_direct(const FusedParams p)
{
    constexpr bool kList = kChunks == 0;
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
    const int first_helper = kPairs ? 16 : G, helpers = nwarps - 1 - first_helper;
    const int g = streams ? (kPairs ? (warp & 7) : warp) : 0;     // the team
    const int half = streams && kPairs ? warp >> 3 : 0;           // which of its two warps
    const int Dw = p.D / stride;                                  // ring slots per warp
    const DirectSmem &lay = p.direct;
    float *acc = reinterpret_cast<float *>(smem + lay.acc);
    uint8_t *ring = smem + lay.ring;
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + lay.bars);
    uint2 *items = reinterpret_cast<uint2 *>(smem + lay.items);   // [team][cap] {offset/16, units of 16 bytes << 16 | x bits}
    int *zero_group = reinterpret_cast<int *>(smem + lay.zero);
    uint2 *place = reinterpret_cast<uint2 *>(smem + lay.place);
    uint32_t *kbw = reinterpret_cast<uint32_t *>(smem + lay.keep);
    volatile int *flags = reinterpret_cast<volatile int *>(smem + lay.flag);     // [G] a warp of the team gave up

    // Row part s (one slab) and place of this block in it.
    const int per_part = idiv_small(gridDim.x, p.P), kslice = idiv_small(blockIdx.x, p.P), s = blockIdx.x - kslice * p.P;
    const bool long_part = s < (int)gridDim.x - per_part * p.P;
    const int nK = per_part + (long_part ? 1 : 0);
    const uint32_t g_inv = (uint32_t)idiv_small(65535 + G, G);    // i / G = i * g_inv >> 16 for i < 4096
    const float nK_inv = __fdividef(1.f, (float)nK);
    int column[kChunks + 1];                                  // the lane's columns of the block's (K or more: none)
#pragma unroll
    for (int c = 0; c < kChunks; ++c) column[c] = direct_column(32 * c + lane, kslice, nK, nK_inv);

    // Programmatic dependent launch: see k_spmspv_fused.
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // {offset/16, units of 16 bytes} of the block's columns' sub-blocks: once per block, by the last warps, which do not stream
    // (each streaming warp for itself, in registers: 0.05 to 0.3 us slower, their loads touch a sector per run of columns).
    // The streaming warps meet them at barrier 15, when x is on its way (at the barrier of all warps below, ahead of the wait for
    // the previous kernel: 1024 x 1024 3.34 us instead of 3.30, 4096 x 4096 6.93 instead of 6.87).
    const int own = tid - (nthreads - 32 * kDirectChunks), own_column = direct_column(max(own, 0), kslice, nK, nK_inv);
    const bool owns = own >= 0 && own < 32 * kChunks && own_column < p.K;
    uint2 own_place = make_uint2(0u, 0u);
    auto load_place = [&]() {
        if (!owns) return;
        own_place.x = p.meta[(size_t)own_column * p.S + s];
        own_place.y = p.meta[(size_t)own_column * p.S + s + 1];
    };
    auto give_place = [&]() {
        if (owns) place[own] = make_uint2(own_place.x, own_place.y - own_place.x);
        asm volatile("bar.arrive 15, %0;" ::"r"(nthreads) : "memory");
    };
    if (!kList && p.image_early) load_place();
    if (tid < 4) zero_group[tid] = 0;
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
    if (!kList && p.image_early && !streams) give_place();
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (!kList && !p.image_early && !streams) {
        load_place();
        give_place();
    }

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
        // The lane has found item k of the team: it notes it, and starts its copy if it is one of the first.  (Copies that an
        // elected lane starts when all chunks are through: 0.2 us slower at 4096 x 4096.)
        auto found = [&](int k, const uint2 at, uint32_t xb) {
            if (kPairs && (k & 1) != half) return;
            mine[k] = make_uint2(at.x, at.y << 16 | xb);
            const int slot = k >> pp;
            if (slot < Dw) bulk_load(ring0 + (uint32_t)(slot * p.slot_bytes), p.stream + (size_t)at.x * 16, at.y * 16u, bar0 + 8u * slot);
        };
        const uint32_t lt_mask = (1u << lane) - 1u;
        int cnt = 0;
        if (kList) {
            const int n = __shfl_sync(kFull, max(0, min(p.K, __ldcg(p.list_count))), 0);
            if (blockIdx.x == 0 && tid == 0) *p.count = n;
            const int units = nK * G, u = kslice * G + g;
            const uint32_t units_inv = long_part ? p.units_inv_long : p.units_inv;
            uint32_t each = __umulhi((uint32_t)n, units_inv), extra = (uint32_t)n - each * (uint32_t)units;
            if (extra >= (uint32_t)units) { ++each; extra -= (uint32_t)units; }
            const int r0 = u * (int)each + min(u, (int)extra);
            cnt = (int)each + (u < (int)extra ? 1 : 0);
            for (int k = half + stride * lane; k < cnt; k += stride * 32) {
                const int j = min(max(__ldcg(p.list_idx + r0 + k), 0), p.K - 1);
                const uint32_t xb = __ldcg(p.list_val + r0 + k);
                const uint32_t at = p.meta[(size_t)j * p.S + s];
                found(k, make_uint2(at, p.meta[(size_t)j * p.S + s + 1] - at), xb);
            }
        } else {
            uint32_t xb[kChunks + 1];
#pragma unroll
            for (int c = 0; c < kChunks; ++c) xb[c] = column[c] < p.K ? x[column[c]] : 0u;
            asm volatile("bar.sync 15, %0;" ::"r"(nthreads) : "memory");                // the places are there
            uint32_t n = 0;
#pragma unroll
            for (int c = 0; c < kChunks; ++c) {
                const bool keep = column[c] < p.K && !(fabsf(__half2float(__ushort_as_half((uint16_t)xb[c]))) <= p.tau);
                const uint32_t kept = __ballot_sync(kFull, keep), i = n + __popc(kept & lt_mask), k = i * g_inv >> 16;
                if (keep && (int)(i - k * G) == g) found((int)k, place[32 * c + lane], xb[c]);
                n += __popc(kept);
            }
            cnt = (int)n > g ? idiv_small((int)n - g + G - 1, G) : 0;
        }
        uint32_t slot = 0, parity = 0, consumed = 0;              // of this warp's Dw slots
        uint32_t issued = (uint32_t)min(Dw, (cnt - half + pp) >> pp), islot = issued == (uint32_t)Dw ? 0 : issued;   // (cnt >= 0, half <= 1)
        auto issue = [&](const uint2 it) {
            bulk_load_elected(ring0 + islot * (uint32_t)p.slot_bytes, p.stream + (size_t)it.x * 16, (it.y >> 16) * 16u, bar0 + 8u * islot);
            ++issued;
            if (++islot == (uint32_t)Dw) islot = 0;
        };
        team_sync();
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
