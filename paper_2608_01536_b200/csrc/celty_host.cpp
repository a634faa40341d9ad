// Host half of the library: offline packing into RLC-CSC (Section 3.2, Fig. 2(a)), the handle,
// host-side decoding for round-trip tests and byte accounting.  No CUDA calls in this file.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>
#include <exception>
#include <memory>
#include <new>
#include <thread>
#ifdef __SSE2__
#include <immintrin.h>
#endif

#include "celty_internal.h"
#include "celty_signal.h"

using namespace celty;

namespace {

// ---- packing.  The weights are row-major and the format is column-major, so the encoder works on blocks of 64
// columns: one row of a block is a cache line or two of W and of the mask, its kept positions one 64-bit word.  The
// words of 64 rows, transposed, are the kept rows of 64 columns, and entries, gaps and padding follow from bit scans.
// Blocks are independent but for the places their entries go to, which the counts of a first pass give; host threads
// share them.  A row of W or of the mask is another page than the one before it, so what the passes read next is prefetched.
// 2048 x 4096, half kept, 16 threads: 1.6 to 2.1 ms (2.1 to 2.4 with threads started for each pass, weights gathered entry by entry
// and pages first touched where they are filled); 27 ms on one.  Bound by the rows of W, 128 bytes of a page each (0.6 ms), the mask
// (0.3), first touches (0.2) and the start and end of the threads (0.25).
constexpr int kBlockCols = 64;

// What a thread keeps from one block to the next (fresh large vectors would be fresh pages every time).
struct SubBlock {
    uint8_t *at;
    uint32_t vectors;
    uint16_t slot[(kMaxTileRows + kGroup - 1) / kGroup + 2];      // [q]: next free one of step q
};

struct Scratch {
    std::vector<uint64_t> row_word;
    std::vector<SubBlock> subs;
    std::vector<uint16_t> values;
    std::vector<int32_t> pos;
};

int64_t host_threads(int64_t n, bool worth_threads)
{
    return worth_threads ? std::max<int64_t>(1, std::min<int64_t>({n, 16, (int64_t)std::thread::hardware_concurrency()})) : 1;      // (0: not known)
}

// Phases of work that several host threads go through together: work(phase, scratch) on each of them, then between(phase) on one
// while the others wait.  The threads are started once (starting 15 takes 0.2 ms).  false = memory ran out in one.
template <typename Work, typename Between>
bool in_phases(int64_t want, int phases, Work work, Between between)
{
    std::atomic<bool> failed(false);
    std::atomic<int64_t> arrived(0);
    std::atomic<int> open(0);                                     // the phase that may run
    Signal all_arrived, opened;
    auto phase = [&](int p, Scratch &scratch) {
        try {
            if (!failed) work(p, scratch);
        } catch (const std::exception &) {
            failed = true;
        }
    };
    std::vector<std::thread> threads;
    try {
        threads.reserve((size_t)want);
        for (int64_t t = 1; t < want; ++t)
            threads.emplace_back([&]() {
                Scratch scratch;
                for (int p = 0; p < phases; ++p) {
                    opened.wait([&] { return open >= p; });
                    phase(p, scratch);
                    ++arrived;
                    all_arrived.raise();
                }
            });
    } catch (const std::exception &) {                            // no (more) threads to be had: those there are do it
    }
    Scratch scratch;
    for (int p = 0; p < phases; ++p) {
        phase(p, scratch);
        all_arrived.wait([&] { return arrived >= (int64_t)threads.size() * (p + 1); });
        try {
            if (!failed) between(p);
        } catch (const std::exception &) {
            failed = true;
        }
        open = p + 1;
        opened.raise();
    }
    for (std::thread &t : threads) t.join();
    return !failed;
}

// f(i, scratch) for i = 0 .. n - 1, on several host threads where there is work for them; false = memory ran out in one.
template <typename F>
bool for_blocks(int64_t n, bool worth_threads, F f)
{
    std::atomic<int64_t> next(0);
    return in_phases(host_threads(n, worth_threads), 1,
                     [&](int, Scratch &scratch) { for (int64_t i; (i = next.fetch_add(1)) < n;) f(i, scratch); }, [](int) {});
}

// Kept positions of columns j0 .. j0 + n - 1 of row r, n <= 64.
inline uint64_t kept_word(const uint16_t *W, int64_t ldw, const uint8_t *mask, int64_t K, int64_t r, int64_t j0, int n)
{
    uint64_t word = 0;
    int c = 0;
    if (mask) {
        const uint8_t *m = mask + r * K + j0;
#if defined(__SSE2__) && !defined(CELTY_PLAIN_ENCODER)
        for (; c + 16 <= n; c += 16) {
            const __m128i v = _mm_loadu_si128(reinterpret_cast<const __m128i *>(m + c));
            word |= (uint64_t)(~_mm_movemask_epi8(_mm_cmpeq_epi8(v, _mm_setzero_si128())) & 0xFFFF) << c;
        }
#endif
        for (; c < n; ++c) word |= (uint64_t)(m[c] != 0) << c;
    } else {
        const uint16_t *w = W + r * ldw + j0;
#if defined(__SSE2__) && !defined(CELTY_PLAIN_ENCODER)
        const __m128i magnitude = _mm_set1_epi16(0x7FFF);
        for (; c + 16 <= n; c += 16) {
            const __m128i a = _mm_and_si128(_mm_loadu_si128(reinterpret_cast<const __m128i *>(w + c)), magnitude);
            const __m128i b = _mm_and_si128(_mm_loadu_si128(reinterpret_cast<const __m128i *>(w + c + 8)), magnitude);
            const __m128i z = _mm_packs_epi16(_mm_cmpeq_epi16(a, _mm_setzero_si128()), _mm_cmpeq_epi16(b, _mm_setzero_si128()));
            word |= (uint64_t)(~_mm_movemask_epi8(z) & 0xFFFF) << c;
        }
#endif
        for (; c < n; ++c) word |= (uint64_t)((w[c] & 0x7FFFu) != 0) << c;
    }
    return word;
}

// 64 x 64 bits: bit c of a[k] goes to bit k of a[c] (halves swapped recursively: H. S. Warren, Hacker's Delight, 7-3).
inline void transpose64(uint64_t *a)
{
    uint64_t m = 0x00000000FFFFFFFFull;
    for (int d = 32; d; d >>= 1, m ^= m << d)
        for (int k = 0; k < 64; k = (k + d + 1) & ~d) {
            const uint64_t t = ((a[k] >> d) ^ a[k + d]) & m;
            a[k] ^= t << d;
            a[k + d] ^= t;
        }
}

// The rows behind a tile's local rows, and the kept bits of a block of columns in tile order:
// bits[(t * words + i / 64) * 64 + c], bit i mod 64, is local row i of tile t in the block's column c.
struct TileRows {
    const celty_matrix *m;
    int64_t words;                                                // 64-bit words per tile
    std::vector<int32_t> row0;                                    // rows of lane 0's tile of every slab (tile_row divides)
    explicit TileRows(const celty_matrix *mat) : m(mat), words((mat->R + 63) / 64), row0((size_t)(mat->S * mat->R))
    {
        for (int64_t s = 0; s < m->S; ++s)
            for (int64_t i = 0; i < m->R; ++i)
                row0[(size_t)(s * m->R + i)] = (int32_t)(m->layout == CELTY_LAYOUT_LANE_TILE ? tile_row(m->S, m->C, s, 0, i) : i);
    }
    // tile t's local row i is row rows(t)[i] + (t mod 32); >= M: does not exist (a tile's rows grow with i)
    const int32_t *rows(int64_t t) const { return row0.data() + t / 32 * m->R; }
    void bits_of_block(const uint64_t *row_word, uint64_t *bits) const
    {
        for (int64_t t = 0; t < m->T; ++t)
            for (int64_t w = 0; w < words; ++w, bits += kBlockCols) {
                for (int k = 0; k < 64; ++k) {
                    const int64_t i = w * 64 + k, r = i < m->R ? rows(t)[i] + t % 32 : m->M;
                    bits[k] = r < m->M ? row_word[(size_t)r] : 0;
                }
                transpose64(bits);
            }
    }
};

// Kept weights and padding entries of one column of one tile (words at a stride of 64): a gap of g dropped rows
// before a kept one costs floor(g / 16) padding entries (Section 3.2).
inline void count_entries(const uint64_t *bits, int64_t words, uint32_t *kept, uint32_t *pads)
{
    uint32_t n = 0, p = 0;
    int64_t prev = -1;
    for (int64_t w = 0; w < words; ++w) {
        uint64_t b = bits[w * kBlockCols];
        if (!b) continue;
        n += (uint32_t)__builtin_popcountll(b);
        const int lo = __builtin_ctzll(b), hi = 63 - __builtin_clzll(b);
        p += (uint32_t)((w * 64 + lo - prev - 1) >> 4);
        prev = w * 64 + hi;
        // 16 dropped rows in a row between the word's first and last kept one?
        uint64_t z = ~b;
        z &= z >> 1; z &= z >> 2; z &= z >> 4; z &= z >> 8;
        if (hi > lo && (z & ((1ull << hi) - 1) & ~((1ull << lo) - 1)))
            for (int last = lo; b &= b - 1;) {
                const int i = __builtin_ctzll(b);
                p += (uint32_t)((i - last - 1) >> 4);
                last = i;
            }
    }
    *kept = n;
    *pads = p;
}

#if defined(__x86_64__) && !defined(CELTY_PLAIN_ENCODER)
// The kept weights of one column of one tile (weight of local row i in values[i], words of its kept bits at a stride of 64), one after
// the other and zeros up to the end of their last group, and their runs, eight to a word; returns how many.  For a tile without
// padding entries (a run takes four bits).  A compression of 32 weights or 64 positions is one instruction here, where a scan
// bit by bit is a dozen per entry.
__attribute__((target("avx512f,avx512bw,avx512vbmi,avx512vbmi2,popcnt")))
uint64_t compress_tile(const uint64_t *bits, int64_t words, const uint16_t *values, uint16_t *kept, uint8_t *pos /* and one before */, uint32_t *runs)
{
    const __m512i ascending = _mm512_set_epi8(
        63, 62, 61, 60, 59, 58, 57, 56, 55, 54, 53, 52, 51, 50, 49, 48, 47, 46, 45, 44, 43, 42, 41, 40, 39, 38, 37, 36, 35, 34, 33, 32, 31, 30, 29, 28,
        27, 26, 25, 24, 23, 22, 21, 20, 19, 18, 17, 16, 15, 14, 13, 12, 11, 10, 9, 8, 7, 6, 5, 4, 3, 2, 1, 0);
    uint64_t n = 0;
    for (int64_t w = 0; w < words; ++w) {
        const uint64_t b = bits[w * kBlockCols];
        const __mmask32 lo = (__mmask32)b, hi = (__mmask32)(b >> 32);
        const uint64_t half = n + (uint64_t)__builtin_popcountll((uint32_t)b);
        _mm512_storeu_si512(pos + n, _mm512_maskz_compress_epi8(b, _mm512_add_epi8(ascending, _mm512_set1_epi8((char)(64 * w)))));
        _mm512_storeu_si512(kept + n, _mm512_maskz_compress_epi16(lo, _mm512_loadu_si512(values + 64 * w)));
        _mm512_storeu_si512(kept + half, _mm512_maskz_compress_epi16(hi, _mm512_loadu_si512(values + 64 * w + 32)));
        n += (uint64_t)__builtin_popcountll(b);
    }
    _mm_storeu_si128(reinterpret_cast<__m128i *>(kept + n), _mm_setzero_si128());
    pos[-1] = 0xFF;                                               // the row before the first
    for (uint64_t k = 0; k < n; k += 64) {
        const __mmask64 there = n - k >= 64 ? ~0ull : (1ull << (n - k)) - 1;
        const __m512i gap = _mm512_sub_epi8(_mm512_loadu_si512(pos + k), _mm512_loadu_si512(pos + k - 1));
        const __m512i run = _mm512_maskz_sub_epi8(there, gap, _mm512_set1_epi8(1));
        _mm256_storeu_si256(reinterpret_cast<__m256i *>(runs + k / 8), _mm512_cvtepi16_epi8(_mm512_or_si512(run, _mm512_srli_epi16(run, 4))));
    }
    return n;
}
const bool kCompress = [] {
    __builtin_cpu_init();
    return __builtin_cpu_supports("avx512f") && __builtin_cpu_supports("avx512bw") && __builtin_cpu_supports("avx512vbmi") && __builtin_cpu_supports("avx512vbmi2");
}();
#else
constexpr bool kCompress = false;
uint64_t compress_tile(const uint64_t *, int64_t, const uint16_t *, uint16_t *, uint8_t *, uint32_t *) { return 0; }
#endif

// Writes the entries of one column of one tile, whose local row i has weight values[kStride i]: group by group into places that
// `place(q)` gives (16 bytes of values, one run word each, zeroed beforehand), entry e of a group in bits 4e .. 4e+3 of its run word.
template <int kStride, typename Place>
void emit_entries(celty_matrix *m, const TileRows &tr, const uint64_t *bits, const uint16_t *values, uint64_t logical, uint64_t entries,
                  int32_t *pos /* [R] */, Place place)
{
    uint64_t n = 0;
    if (kStride == 1 && kCompress) {
        alignas(64) uint16_t kept[kMaxTileRows + 96];
        alignas(64) uint8_t at[64 + kMaxTileRows + 144];
        alignas(64) uint32_t runs[(kMaxTileRows + 64) / 8 + 8];
        for (int64_t w = 0; w < tr.words; ++w) n += (uint64_t)__builtin_popcountll(bits[w * kBlockCols]);
        if (n == entries) {
            compress_tile(bits, tr.words, values, kept, at + 64, runs);
            for (uint64_t q = 0; q * kGroup < n; ++q) {
                uint8_t *vp, *rp;
                place((uint32_t)q, &vp, &rp);
                std::memcpy(vp, kept + q * kGroup, 16);
                std::memcpy(rp, runs + q, 4);
            }
            return;
        }
        n = 0;
    }
    for (int64_t w = 0; w < tr.words; ++w)
        for (uint64_t b = bits[w * kBlockCols]; b; b &= b - 1) pos[n++] = (int32_t)(w * 64) + __builtin_ctzll(b);
    if (n == entries) {                                           // no padding entries: whole groups without branches
        int32_t last = -1;
        for (uint64_t k = 0; k < n; k += kGroup) {
            const int have = (int)std::min<uint64_t>(kGroup, n - k);
            uint8_t *vp, *rp;
            place((uint32_t)(k / kGroup), &vp, &rp);
            uint16_t v[kGroup] = {};
            uint32_t runs = 0;
            auto one = [&](int e) {
                const int32_t i = pos[k + (uint64_t)e];
                v[e] = values[(size_t)i * kStride];
                runs |= (uint32_t)(i - last - 1) << (4 * e);
                last = i;
            };
            if (have == kGroup)
                for (int e = 0; e < kGroup; ++e) one(e);
            else
                for (int e = 0; e < have; ++e) one(e);
            std::memcpy(vp, v, sizeof v);
            std::memcpy(rp, &runs, 4);
        }
        return;
    }
    uint8_t *vp = nullptr, *rp = nullptr;
    uint32_t runs = 0, e = 0, q = 0;
    auto put = [&](uint16_t v, uint32_t run) {
        if (e == 0) {
            place(q++, &vp, &rp);
            runs = 0;
        }
        std::memcpy(vp + 2 * e, &v, 2);
        runs |= run << (4 * e);
        if (++e == kGroup) {
            std::memcpy(rp, &runs, 4);
            e = 0;
        }
    };
    int32_t prev = -1;
    for (uint64_t k = 0; k < n; ++k) {
        const int32_t i = pos[k];
        uint32_t gap = (uint32_t)(i - prev - 1);
        for (; gap > 15; gap -= 16) {
            put(0, 15);
            __atomic_fetch_or(&m->pad_bits[(size_t)(logical >> 3)], (uint8_t)(1u << (logical & 7)), __ATOMIC_RELAXED);
            ++logical;
        }
        put(values[(size_t)i * kStride], gap);
        ++logical;
        prev = i;
    }
    if (e) std::memcpy(rp, &runs, 4);
}

// Slabs S, local rows per tile R and chunk C of the LANE_TILE row map for M rows (tile_rows = 0: library's
// choice).  Up to 128 local rows per lane: a lane's run stream is then ~8 groups per column at 50% density,
// and eight or nine teams with their accumulators and rings fit one SM's shared memory.  Measured on B200 over
// the configured shapes, S = ceil(M / 4096) was the best or within 6% of the best slab count everywhere.
// On very tall layers (6 slabs or more) the streaming loop dominates, and what counts there is that eight warp
// teams fit one SM's 227 KB of shared memory (accumulator slab + two ring slots each): when the density of the
// kept weights makes the sub-blocks too large for that at 128 local rows, fewer rows per tile (in steps of 8, down
// to 96) and correspondingly more slabs are taken: 104 rows at 70% of the weights kept, 120 at 50%, 128 at 30% on
// 28672 x 8192 (measured: 44.4 us against 53.0 at 128 rows and 47.0 at 96; 37.1 against 37.7; no change).
void choose_shape(int64_t M, int64_t K, double density, int tile_rows, int64_t *S_out, int32_t *R_out, int32_t *C_out)
{
    const int64_t Q = (M + 31) / 32;                                  // groups of 32 rows
    int64_t S, R;
    if (tile_rows > 0) {
        R = tile_rows;
        S = (Q + R - 1) / R;
    } else {
        S = std::max<int64_t>(1, (M + 4095) / 4096);
        // A layer of one slab and few columns streams for so short a time that the merge dominates: two slabs
        // halve what every block adds up and adds into y (and the contributors per row), for twice as many
        // sub-blocks of half the size.  Measured at 4096 x 4096: 8.3 us against 8.8; at 4096 x 11008, where a team
        // has five sub-blocks to stream, no gain, so the rule stops short of it.
        if (S == 1 && Q >= 32 && K <= 6144) S = 2;
        // (Taller layers of few columns would gain from slabs of 2048 rows in calls for one vector, 6 to 17 % at 10 % of the
        // activations and up to 7 at 50, and lose more in batches, whose blocks have N times the columns; the image is the same for both.
        // Slabs of 4096 -> of 2048 rows, us, one vector at 10 / 50 %, N = 4, 8 at 50 %:  8192 x 2048 4.66 / 5.94, 12.7, 22.0 -> 3.92 /
        // 6.07, 13.5, 27.2;  5504 x 2048 4.24 / 5.03, 9.3, 16.5 -> 3.87 / 4.99, 10.6, 19.2;  20000 x 800 4.71 / 6.06, 12.6, 24.9 -> 3.93 /
        // 5.62, 14.7, 29.9;  8192 x 512 4.56 / 4.64, 6.1, 8.3 -> 3.89 / 3.92, 5.9, 9.0.)
        auto rows_for = [&](int64_t slabs) { return std::max<int64_t>(16, ((Q + slabs - 1) / slabs + 15) / 16 * 16); };
        auto teams_that_fit = [&](int64_t rows) {
            const double entries = 32.0 * rows * density;             // of one sub-block, mean; + 3.5 sigma for the largest
            const double largest = entries + 3.5 * std::sqrt(entries * (1.0 - density)) + 32 * 3.5;  // + group filling
            const double slot = std::ceil((kSubHeader + 2.5 * largest) / 128.0) * 128.0;
            const double misc = 2.0 * ((K + 31) / 32) * 4 + 17.0 * ((K + 255) / 256) * 4 + 1024;
            return (int64_t)((232448.0 - misc) / ((rows + kTileSlack) * 128.0 + 2.0 * slot + 1024.0));
        };
        R = rows_for(S);
        if (S >= 6)
            for (int fewer = 1; fewer <= 4 && teams_that_fit(R) < 8 && R > 32; ++fewer) {
                R -= 8;                                                // in steps of 8 rows: the chunk of the row map halves
                S = (Q + R - 1) / R;
            }
    }
    *S_out = S;
    *R_out = (int32_t)R;
    // chunks of 16 groups = 2 KB of consecutive rows of y: the merge adds them with one bulk copy each, and 2 KB
    // copies measured 3-4% faster per call than 512-byte ones on the mid-size shapes
    *C_out = R % 16 == 0 ? 16 : R % 8 == 0 ? 8 : R % 4 == 0 ? 4 : 1;
}

// Weights of a column of a tile in the encoder's copy: whole vectors of 32 and a row of 64 positions are read.
inline size_t tile_pitch(int64_t R) { return round_up((size_t)R, 64) + 8; }

// Eight rows of a block of columns (null: zeros), to[c * ld + k] = from[k][c].
inline void copy_transposed(uint16_t *to, size_t ld, const uint16_t *const from[8], int cols)
{
    int c = 0;
#if defined(__SSE2__) && !defined(CELTY_PLAIN_ENCODER)
    for (; c + 8 <= cols; c += 8) {
        __m128i r[8], a[8];
        for (int k = 0; k < 8; ++k)
            r[k] = from[k] ? _mm_loadu_si128(reinterpret_cast<const __m128i *>(from[k] + c)) : _mm_setzero_si128();
        for (int k = 0; k < 4; ++k) {                             // rows 2k and 2k + 1 interleaved, then pairs, then fours
            a[2 * k] = _mm_unpacklo_epi16(r[2 * k], r[2 * k + 1]);
            a[2 * k + 1] = _mm_unpackhi_epi16(r[2 * k], r[2 * k + 1]);
        }
        for (int h = 0; h < 2; ++h)
            for (int k = 0; k < 2; ++k) {
                r[4 * h + 2 * k] = _mm_unpacklo_epi32(a[4 * h + k], a[4 * h + 2 + k]);
                r[4 * h + 2 * k + 1] = _mm_unpackhi_epi32(a[4 * h + k], a[4 * h + 2 + k]);
            }
        for (int k = 0; k < 4; ++k) {
            _mm_storeu_si128(reinterpret_cast<__m128i *>(to + (c + 2 * k) * ld), _mm_unpacklo_epi64(r[k], r[4 + k]));
            _mm_storeu_si128(reinterpret_cast<__m128i *>(to + (c + 2 * k + 1) * ld), _mm_unpackhi_epi64(r[k], r[4 + k]));
        }
    }
#endif
    for (; c < cols; ++c)
        for (int k = 0; k < 8; ++k) to[(size_t)c * ld + k] = from[k] ? from[k][c] : 0;
}

// A row of a block of columns.
inline void copy_row(uint16_t *to, const uint16_t *from, int cols)
{
    if (cols == kBlockCols) std::memcpy(to, from, 2 * kBlockCols);
    else std::memcpy(to, from, (size_t)cols * 2);
}

// COLUMN image: meta uint2[K] {off16, entries}, then per column its chunks of up to 32 groups;
// chunk = [groups x 16 B values][groups x 4 B runs]; column block padded to 16 bytes.
void write_column(celty_matrix *m, const TileRows &tr, const uint64_t *bits, const uint16_t *values, int32_t *pos, int64_t j,
                  int c)
{
    uint32_t *meta = reinterpret_cast<uint32_t *>(m->image.data());
    const uint64_t e0 = m->block_ptr[(size_t)j], n = m->block_ptr[(size_t)j + 1] - e0, groups = (n + kGroup - 1) / kGroup;
    uint8_t *col = m->image.data() + m->meta_bytes + (size_t)meta[2 * j] * 16;
    meta[2 * j + 1] = (uint32_t)n;
    std::memset(col, 0, round_up((size_t)groups * 20, 16));
    emit_entries<kBlockCols>(m, tr, bits + c, values + c, e0, n, pos, [&](uint32_t g, uint8_t **vp, uint8_t **rp) {
        const uint64_t chunk = g / kChunkGroups, in = g % kChunkGroups, gc = std::min<uint64_t>(kChunkGroups, groups - chunk * kChunkGroups);
        uint8_t *at = col + chunk * (kChunkGroups * 20);
        *vp = at + 16 * in;
        *rp = at + 16 * gc + 4 * in;
    });
}

// LANE_TILE image: meta uint32[K*S + 1] (offset/16 of each sub-block), then per (column j, slab s) a sub-block
//   [48 B header: 32 x u8 groups of lane L's tile 32s+L, u32 vectors | steps << 16][G x 16 B values][G x 4 B runs],
// padded to 16 bytes,
// G = sum of the lanes' group counts.  Vectors are stored step-major: for step q = 0, 1, ... the
// lanes that still have a q-th group, in lane order, so that a warp reads one contiguous span per step.
// W points at the block's first column.  A tile's rows of the block are copied together, column by column: 8 to 32 KB, which stay in
// L1 or L2 while the tile is packed.  (Two or four blocks at a time, 256 or 512 bytes of a row: 20 % slower.)
void write_lane_tile(celty_matrix *m, const TileRows &tr, const uint64_t *bits, const uint16_t *W, int64_t ldw, Scratch &scratch, int64_t j0,
                     int cols)
{
    const int64_t S = m->S, T = m->T;
    const size_t ld = tile_pitch(m->R);
    const uint32_t *meta = reinterpret_cast<const uint32_t *>(m->image.data());
    scratch.values.resize((size_t)cols * ld);
    scratch.pos.resize((size_t)m->R);
    scratch.subs.resize((size_t)cols);
    uint16_t *values = scratch.values.data();
    int32_t *pos = scratch.pos.data();
    SubBlock *sub = scratch.subs.data();
    for (int64_t s = 0; s < S; ++s) {
        for (int c = 0; c < cols; ++c) {
            const size_t b = (size_t)((j0 + c) * S + s);
            SubBlock &sb = sub[c];
            sb.at = m->image.data() + m->meta_bytes + (size_t)meta[b] * 16;
            std::memset(sb.at, 0, ((size_t)meta[b + 1] - meta[b]) * 16);
            uint16_t lanes[(kMaxTileRows + kGroup - 1) / kGroup + 2] = {};                     // lanes that have a q-th group
            uint32_t steps = 0;
            sb.vectors = 0;
            for (int L = 0; L < 32; ++L) {
                const size_t k = (size_t)((j0 + c) * T + 32 * s + L);
                const uint32_t g = (m->block_ptr[k + 1] - m->block_ptr[k] + kGroup - 1) / kGroup;
                sb.at[L] = (uint8_t)g;
                sb.vectors += g;
                steps = std::max(steps, g);
                for (uint32_t q = 0; q < g; ++q) ++lanes[q];
            }
            sb.slot[0] = 0;
            for (uint32_t q = 0; q < steps; ++q) sb.slot[q + 1] = (uint16_t)(sb.slot[q] + lanes[q]);
            const uint32_t gs = sb.vectors | (steps << 16);
            std::memcpy(sb.at + 32, &gs, 4);
        }
        for (int L = 0; L < 32; ++L) {
            const int64_t t = 32 * s + L;
            const int32_t *rows = tr.rows(t);
            for (int64_t i = 0; i < m->R; i += 8) {
                const uint16_t *from[8];
                for (int k = 0; k < 8; ++k) {
                    const int64_t r = i + k < m->R ? rows[i + k] + L : m->M;
                    from[k] = r < m->M ? W + r * ldw : nullptr;
                    if (r + 1 < m->M)                                // of the next tile
                        for (int c = 0; c < cols; c += 32) __builtin_prefetch(from[k] + ldw + c);
                }
                copy_transposed(values + i, ld, from, cols);
            }
            for (int c = 0; c < cols; ++c) {
                SubBlock &sb = sub[c];
                uint8_t *vbase = sb.at + kSubHeader, *rbase = vbase + 16 * (size_t)sb.vectors;
                const uint64_t e0 = m->block_ptr[(size_t)((j0 + c) * T + t)], e1 = m->block_ptr[(size_t)((j0 + c) * T + t + 1)];
                emit_entries<1>(m, tr, bits + t * tr.words * kBlockCols + c, values + (size_t)c * ld, e0, e1 - e0, pos,
                             [&](uint32_t q, uint8_t **vp, uint8_t **rp) {
                                 const uint32_t slot = sb.slot[q]++;
                                 *vp = vbase + 16 * (size_t)slot;
                                 *rp = rbase + 4 * (size_t)slot;
                             });
            }
        }
    }
}

}  // namespace

extern "C" int celty_encode(const uint16_t *W, int64_t ldw, const uint8_t *mask, int64_t M, int64_t K,
                            const celty_encode_opts *opts, celty_matrix **out)
{
    if (!W || !out || M <= 0 || K <= 0 || ldw < K || M > kMaxM || K >= ((int64_t)1 << 31)) return CELTY_EINVAL;
    celty_encode_opts o = {4, CELTY_LAYOUT_LANE_TILE, 0, 0};
    if (opts) o = *opts;
    if (o.run_bits != 4 || o.slabs_per_block < 0 || o.slabs_per_block > 15) return CELTY_EINVAL;
    if (o.layout == CELTY_LAYOUT_COLUMN && o.slabs_per_block != 0) return CELTY_EINVAL;
    if (o.layout != CELTY_LAYOUT_COLUMN && o.layout != CELTY_LAYOUT_LANE_TILE) return CELTY_EINVAL;
    if (o.layout == CELTY_LAYOUT_COLUMN && o.tile_rows != 0) return CELTY_EINVAL;
    if (o.layout == CELTY_LAYOUT_LANE_TILE && (o.tile_rows < 0 || o.tile_rows > kMaxTileRows)) return CELTY_EINVAL;
    *out = nullptr;
    try {
        std::unique_ptr<celty_matrix> owner(new celty_matrix());   // released to the caller only on success
        celty_matrix *m = owner.get();
        m->M = M; m->K = K; m->layout = o.layout;
        const bool threads = M * K >= (1 << 18);                  // a quarter of a million weights: 1 ms of one thread
        if (o.layout == CELTY_LAYOUT_COLUMN) {
            m->R = (int32_t)M; m->T = 1; m->S = 1;
        } else {
            double density = 0.5;
            if (o.tile_rows == 0 && M > 5 * 4096) {                   // only very tall layers look at the density
                std::atomic<uint64_t> kept_weights(0);
                if (!for_blocks((M + 255) / 256, threads, [&](int64_t b, Scratch &) {
                        uint64_t n = 0;
                        for (int64_t r = b * 256; r < std::min(M, b * 256 + 256); ++r)
                            for (int64_t j = 0; j < K; j += kBlockCols)
                                n += (uint64_t)__builtin_popcountll(kept_word(W, ldw, mask, K, r, j, (int)std::min<int64_t>(kBlockCols, K - j)));
                        kept_weights += n;
                    }))
                    return CELTY_ENOMEM;
                density = (double)kept_weights.load() / ((double)M * (double)K);
            }
            choose_shape(M, K, density, o.tile_rows, &m->S, &m->R, &m->C);
            m->T = 32 * m->S;
            if (m->S > 32) return CELTY_EINVAL;                 // one warp per slab, 32 warps per block
        }
        const int64_t T = m->T, S = m->S;
        const bool lane_tile = m->layout == CELTY_LAYOUT_LANE_TILE;
        const TileRows tr(m);
        const int64_t blocks = (K + kBlockCols - 1) / kBlockCols;
        auto columns = [&](int64_t b) { return (int)std::min<int64_t>(kBlockCols, K - b * kBlockCols); };
        // Phase 0: kept bits of every block of columns, entries of every (column, tile), groups of every unit the image is
        // made of (COLUMN: a column, LANE_TILE: a sub-block).  Entries and units are summed within the block.
        m->block_ptr.allocate((size_t)(K * T + 1));
        const size_t block_bits = (size_t)(T * tr.words * kBlockCols);
        Raw<uint64_t> bits;
        bits.allocate(block_bits * (size_t)blocks);
        Raw<uint32_t> unit_at;                                    // units before unit u in its block, in 16-byte steps
        unit_at.allocate((size_t)(K * S));
        struct Sum { uint64_t kept = 0, pads = 0, units16 = 0; uint32_t largest = 0; };
        std::vector<Sum> sums((size_t)blocks);
        uint32_t *meta = nullptr;
        size_t units16 = 0;
        std::atomic<int64_t> next[3] = {{0}, {0}, {0}}, touched(0);
        const int64_t want = host_threads(blocks, threads);
        // blocks that a thread takes together in phase 0, row by row: the mask is read 256 bytes at a time
        const int64_t together = std::max<int64_t>(1, std::min<int64_t>(4, blocks / want));
        auto count_block = [&](int64_t b, const uint64_t *row_word) {
            uint64_t *bb = bits.data() + block_bits * (size_t)b;
            tr.bits_of_block(row_word, bb);
            Sum &sum = sums[(size_t)b];
            uint32_t entries = 0;
            for (int c = 0; c < columns(b); ++c) {
                const int64_t j = b * kBlockCols + c;
                for (int64_t s = 0; s < S; ++s) {
                    uint32_t groups = 0;
                    for (int64_t t = s * (T / S); t < (s + 1) * (T / S); ++t) {
                        uint32_t kept, pads;
                        count_entries(bb + t * tr.words * kBlockCols + c, tr.words, &kept, &pads);
                        entries += kept + pads;
                        m->block_ptr[(size_t)(j * T + t + 1)] = entries;
                        groups += (kept + pads + kGroup - 1) / kGroup;
                        sum.kept += kept;
                        sum.pads += pads;
                    }
                    const uint32_t units16 = (uint32_t)(((lane_tile ? kSubHeader : 0) + (size_t)groups * 20 + 15) / 16);
                    unit_at[(size_t)(j * S + s)] = (uint32_t)sum.units16;
                    sum.units16 += units16;
                    sum.largest = std::max(sum.largest, units16);
                }
            }
        };
        auto work = [&](int phase, Scratch &scratch) {
            if (phase == 0) {
                scratch.row_word.resize((size_t)(M * together));
                for (int64_t b0; (b0 = next[0].fetch_add(together)) < blocks;) {
                    const int64_t b1 = std::min(blocks, b0 + together);
                    for (int64_t r = 0; r < M; ++r) {
                        const int64_t ahead = std::min<int64_t>(M - 1, r + 16);
                        for (int64_t b = b0; b < b1; ++b) {
                            if (mask) __builtin_prefetch(mask + ahead * K + b * kBlockCols);
                            else __builtin_prefetch(W + ahead * ldw + b * kBlockCols);
                            scratch.row_word[(size_t)((b - b0) * M + r)] = kept_word(W, ldw, mask, K, r, b * kBlockCols, columns(b));
                        }
                    }
                    for (int64_t b = b0; b < b1; ++b) count_block(b, scratch.row_word.data() + (b - b0) * M);
                }
                return;
            }
            // Phase 1: places of the block's entries and units.  Phase 2: values and runs.  The large arrays are first touched here,
            // a 2 MB page per thread: in phase 2 all threads would wait for the few pages that they are in at a time.
            if (phase == 1) {
                constexpr size_t page = (size_t)2 << 20;
                const size_t pages = (m->image.size() + page - 1) / page;
                for (size_t k; (k = (size_t)touched.fetch_add(1)) * page < pages * page + m->pad_bits.size();) {
                    const size_t at = k < pages ? std::max(k * page, m->meta_bytes) : (k - pages) * page;      // (meta is written below)
                    if (k >= pages) std::memset(m->pad_bits.data() + at, 0, std::min(page, m->pad_bits.size() - at));
                    else if (at < std::min((k + 1) * page, m->image.size())) *(volatile uint8_t *)(m->image.data() + at) = 0;
                }
            }
            if (phase == 1) {
                for (int64_t b; (b = next[1].fetch_add(1)) < blocks;) {
                    const Sum &before = sums[(size_t)b];          // of all blocks before this one by now
                    const int64_t j0 = b * kBlockCols, j1 = j0 + columns(b);
                    const uint32_t entries = (uint32_t)(before.kept + before.pads);
                    for (int64_t k = j0 * T; k < j1 * T; ++k) m->block_ptr[(size_t)(k + 1)] += entries;
                    for (int64_t u = j0 * S; u < j1 * S; ++u) meta[lane_tile ? u : 2 * u] = unit_at[(size_t)u] + (uint32_t)before.units16;
                    if (b + 1 < blocks) continue;
                    const size_t used = lane_tile ? (size_t)(K * S + 1) * 4 : (size_t)K * 8;
                    if (lane_tile) meta[K * S] = (uint32_t)units16;
                    std::memset(m->image.data() + used, 0, m->meta_bytes - used);
                    std::memset(m->image.data() + m->meta_bytes + units16 * 16, 0, m->stream_bytes - units16 * 16);
                }
                return;
            }
            for (int64_t b; (b = next[2].fetch_add(1)) < blocks;) {
                const uint64_t *bb = bits.data() + block_bits * (size_t)b;
                const int n = columns(b);
                if (lane_tile) {
                    write_lane_tile(m, tr, bb, W + b * kBlockCols, ldw, scratch, b * kBlockCols, n);
                    continue;
                }
                // (read column by column where they are, a power-of-two row pitch maps them all to a few sets of the cache)
                scratch.values.resize((size_t)M * kBlockCols);
                scratch.pos.resize((size_t)M);
                for (int64_t r = 0; r < M; ++r) copy_row(&scratch.values[(size_t)r * kBlockCols], W + r * ldw + b * kBlockCols, n);
                for (int c = 0; c < n; ++c) write_column(m, tr, bb, scratch.values.data(), scratch.pos.data(), b * kBlockCols + c, c);
            }
        };
        bool too_large = false;
        auto between = [&](int phase) {
            if (phase != 0) return;
            Sum all;
            for (Sum &sum : sums) {                               // the sum of a block becomes that of those before it
                const Sum own = sum;
                sum = all;
                all.kept += own.kept;
                all.pads += own.pads;
                all.units16 += own.units16;
                all.largest = std::max(all.largest, own.largest);
            }
            const uint64_t total = all.kept + all.pads;
            m->nnz = (int64_t)all.kept;
            m->n_pad = (int64_t)all.pads;
            m->max_unit16 = all.largest;
            if (total > 0xFFFFFFFFull) {
                too_large = true;
                for (auto &n : next) n = blocks;                  // nothing of the later phases
                return;
            }
            m->block_ptr[0] = 0;
            m->pad_bits.allocate((size_t)(total + 7) / 8);
            m->meta_bytes = round_up(lane_tile ? (size_t)(K * S + 1) * 4 : (size_t)K * 8, kAlign);
            units16 = (size_t)all.units16;
            m->stream_bytes = round_up(units16 * 16, kAlign);
            m->image.allocate(m->meta_bytes + m->stream_bytes);
            meta = reinterpret_cast<uint32_t *>(m->image.data());
        };
        if (!in_phases(want, 3, work, between)) return CELTY_ENOMEM;
        if (too_large) return CELTY_EINVAL;
        const int64_t spb = o.slabs_per_block > 0 ? o.slabs_per_block : kSlabsPerBlock;
        m->P = (int32_t)((m->S + spb - 1) / spb);
        m->Sc = (int32_t)((m->S + m->P - 1) / m->P);
        m->ws = workspace_layout(K, T, m->layout == CELTY_LAYOUT_LANE_TILE ? (int64_t)m->Sc * m->R * 32 : 0);
        *out = owner.release();
        return CELTY_OK;
    } catch (const std::exception &) {
        return CELTY_ENOMEM;
    }
}

extern "C" void celty_destroy(celty_matrix *m) { delete m; }

extern "C" int celty_clone(const celty_matrix *m, celty_matrix **out)
{
    if (!m || !out) return CELTY_EINVAL;
    *out = nullptr;
    try {
        std::unique_ptr<celty_matrix> copy(new celty_matrix(*m));
        copy->d_image = nullptr;                  // the copy starts unbound, with the library's launch choices
        copy->d_ws = nullptr;
        copy->last_grid = 0;
        copy->last_merge = -1;
        for (int32_t &g : copy->last_batch_grid) g = 0;
        copy->forget_launches();
        *out = copy.release();
        return CELTY_OK;
    } catch (const std::exception &) {
        return CELTY_ENOMEM;
    }
}

extern "C" int celty_info(const celty_matrix *m, int64_t *M, int64_t *K, int64_t *nnz, int64_t *n_pad,
                          int64_t *compressed_bytes, int32_t *layout, int32_t *tile_rows)
{
    if (!m) return CELTY_EINVAL;
    if (M) *M = m->M;
    if (K) *K = m->K;
    if (nnz) *nnz = m->nnz;
    if (n_pad) *n_pad = m->n_pad;
    if (compressed_bytes) *compressed_bytes = (m->nnz + m->n_pad) * 5 / 2 + 4 * (m->K + 1);
    if (layout) *layout = m->layout;
    if (tile_rows) *tile_rows = m->layout == CELTY_LAYOUT_COLUMN ? 0 : m->R;
    return CELTY_OK;
}

extern "C" int celty_row_map(const celty_matrix *m, int32_t *slabs, int32_t *tile_rows, int32_t *chunk)
{
    if (!m) return CELTY_EINVAL;
    if (slabs) *slabs = (int32_t)m->S;
    if (tile_rows) *tile_rows = m->R;
    if (chunk) *chunk = m->C;
    return CELTY_OK;
}

// Decode column `col` from the packed image (not from the encoder's temporaries).
extern "C" int celty_decode_host(const celty_matrix *m, int64_t col, int32_t *rows, uint16_t *vals,
                                 uint8_t *runs, uint8_t *is_pad, int64_t cap, int64_t *n_out)
{
    if (!m || col < 0 || col >= m->K) return CELTY_EINVAL;
    const int64_t T = m->T;
    const int64_t n = (int64_t)m->block_ptr[(col + 1) * T] - (int64_t)m->block_ptr[col * T];
    if (n_out) *n_out = n;
    if (n > cap) return CELTY_ENOMEM;
    const uint8_t *stream = m->image.data() + m->meta_bytes;
    const uint32_t *meta = reinterpret_cast<const uint32_t *>(m->image.data());
    int64_t o = 0;
    // A pad cannot be told from a kept +0 that follows 15 dropped rows by looking at the image, so
    // the flag comes from the bit the encoder recorded for the entry's logical position.
    auto emit = [&](uint64_t logical, int64_t row, uint16_t v, uint8_t run) {
        if (rows) rows[o] = (int32_t)row;
        if (vals) vals[o] = v;
        if (runs) runs[o] = run;
        if (is_pad) is_pad[o] = (m->pad_bits[logical >> 3] >> (logical & 7)) & 1u;
        ++o;
    };
    if (m->layout == CELTY_LAYOUT_COLUMN) {
        const uint8_t *colp = stream + (size_t)meta[2 * col] * 16;
        const int64_t groups = (n + kGroup - 1) / kGroup;
        int64_t s = 0;
        for (int64_t e = 0; e < n; ++e) {
            const int64_t g = e / kGroup, c = g / kChunkGroups, gl = g % kChunkGroups;
            const int64_t gc = std::min<int64_t>(kChunkGroups, groups - c * kChunkGroups);
            const uint8_t *chunk = colp + c * (kChunkGroups * 20);
            uint16_t v; uint32_t w;
            std::memcpy(&v, chunk + 16 * gl + 2 * (e % kGroup), 2);
            std::memcpy(&w, chunk + 16 * gc + 4 * gl, 4);
            const uint8_t run = (w >> (4 * (e % kGroup))) & 15u;
            s += run;
            emit((uint64_t)m->block_ptr[col] + e, s + e, v, run);
        }
    } else {
        for (int64_t sl = 0; sl < m->S; ++sl) {
            const uint8_t *sub = stream + (size_t)meta[col * m->S + sl] * 16;
            int64_t G = 0;
            for (int L = 0; L < 32; ++L) G += sub[L];
            const uint8_t *vbase = sub + kSubHeader, *rbase = vbase + 16 * G;
            for (int L = 0; L < 32; ++L) {
                const int64_t t = 32 * sl + L;
                if (t >= T) break;
                const int64_t nt = (int64_t)m->block_ptr[col * T + t + 1] - (int64_t)m->block_ptr[col * T + t];
                int64_t s = 0;
                for (int64_t e = 0; e < nt; ++e) {
                    const int64_t q = e / kGroup;
                    // slot of (step q, lane L): all lanes' groups of earlier steps + lower lanes of this step
                    int64_t slot = 0;
                    for (int L2 = 0; L2 < 32; ++L2) slot += std::min<int64_t>(sub[L2], q) + (L2 < L && sub[L2] > q ? 1 : 0);
                    uint16_t v; uint32_t w;
                    std::memcpy(&v, vbase + 16 * slot + 2 * (e % kGroup), 2);
                    std::memcpy(&w, rbase + 4 * slot, 4);
                    const uint8_t run = (w >> (4 * (e % kGroup))) & 15u;
                    s += run;
                    emit((uint64_t)m->block_ptr[col * T + t] + e, tile_row(m->S, m->C, sl, L, s + e), v, run);
                }
            }
        }
    }
    return CELTY_OK;
}

extern "C" int celty_host_image(const celty_matrix *m, const void **image, size_t *image_bytes, size_t *stream_offset)
{
    if (!m) return CELTY_EINVAL;
    if (image) *image = m->image.data();
    if (image_bytes) *image_bytes = m->image.size();
    if (stream_offset) *stream_offset = m->meta_bytes;
    return CELTY_OK;
}

extern "C" int celty_device_bytes(const celty_matrix *m, size_t *image_bytes, size_t *workspace_bytes)
{
    if (!m) return CELTY_EINVAL;
    if (image_bytes) *image_bytes = m->image.size();
    if (workspace_bytes) *workspace_bytes = m->ws.total;
    return CELTY_OK;
}

extern "C" int celty_fetched_bytes(const celty_matrix *m, const int32_t *idx, int64_t n, int64_t *stream_bytes,
                                   int64_t *total_bytes)
{
    if (!m || (!idx && n > 0) || n < 0) return CELTY_EINVAL;
    const uint32_t *meta = reinterpret_cast<const uint32_t *>(m->image.data());
    int64_t sb = 0, mb = 0;
    for (int64_t p = 0; p < n; ++p) {
        const int64_t j = idx[p];
        if (j < 0 || j >= m->K) return CELTY_EINVAL;
        if (m->layout == CELTY_LAYOUT_COLUMN) {
            const int64_t groups = ((int64_t)meta[2 * j + 1] + kGroup - 1) / kGroup;
            sb += (int64_t)round_up((size_t)groups * 20, 16);
            mb += 8;
        } else {
            sb += ((int64_t)meta[(j + 1) * m->S] - (int64_t)meta[j * m->S]) * 16;
            mb += 4 * (m->S + 1);
        }
    }
    if (stream_bytes) *stream_bytes = sb;
    // x read once, the list written (4-byte index + 2-byte value), y written once.  Scratch traffic of
    // the split-K merge (per-block partial sums) is not counted: it is overhead, not work.
    if (total_bytes) *total_bytes = sb + mb + 2 * m->K + 6 * n + 4 * m->M;
    return CELTY_OK;
}

extern "C" int celty_stored_entries(const celty_matrix *m, const int32_t *idx, int64_t n, int64_t *entries)
{
    if (!m || (!idx && n > 0) || n < 0 || !entries) return CELTY_EINVAL;
    int64_t e = 0;
    for (int64_t p = 0; p < n; ++p) {
        const int64_t j = idx[p];
        if (j < 0 || j >= m->K) return CELTY_EINVAL;
        e += (int64_t)m->block_ptr[(j + 1) * m->T] - (int64_t)m->block_ptr[j * m->T];
    }
    *entries = e;
    return CELTY_OK;
}

extern "C" int celty_layout_stats(const celty_matrix *m, int64_t *sub_blocks, int64_t *steps, int64_t *groups)
{
    if (!m) return CELTY_EINVAL;
    if (m->layout != CELTY_LAYOUT_LANE_TILE) return CELTY_EINVAL;
    const uint32_t *meta = reinterpret_cast<const uint32_t *>(m->image.data());
    const uint8_t *stream = m->image.data() + m->meta_bytes;
    int64_t nb = 0, st = 0, gr = 0;
    for (int64_t b = 0; b < m->K * m->S; ++b) {
        uint32_t hw;
        std::memcpy(&hw, stream + (size_t)meta[b] * 16 + 32, 4);      // vectors | steps << 16 (see kSubHeader)
        ++nb;
        st += hw >> 16;
        gr += hw & 0xFFFFu;
    }
    if (sub_blocks) *sub_blocks = nb;
    if (steps) *steps = st;
    if (groups) *groups = gr;
    return CELTY_OK;
}

extern "C" int celty_shard_columns(int64_t K, int32_t world, int32_t rank, int64_t *k_begin, int64_t *k_end)
{
    if (K <= 0 || world < 1 || rank < 0 || rank >= world || !k_begin || !k_end) return CELTY_EINVAL;
    // groups of 8 columns (16 bytes of FP16 activations) dealt as evenly as they go: a shard's slice of x then
    // starts on the 16-byte boundary the kernels ask for
    const int64_t groups = (K + 7) / 8, base = groups / world, extra = groups % world;
    const int64_t g0 = rank * base + std::min<int64_t>(rank, extra), g1 = g0 + base + (rank < extra ? 1 : 0);
    *k_begin = std::min<int64_t>(K, g0 * 8);
    *k_end = std::min<int64_t>(K, g1 * 8);
    return CELTY_OK;
}

extern "C" int celty_count_entries(const uint8_t *mask, int64_t ldm, int64_t M, int64_t K, int run_bits,
                                   int64_t *nnz, int64_t *n_pad)
{
    if (!mask || M <= 0 || K <= 0 || ldm < K || run_bits < 1 || run_bits > 8) return CELTY_EINVAL;
    // rows outermost (the mask is row-major); gap[j] = dropped rows of column j since its last kept row
    std::vector<int64_t> gap;
    try {
        gap.assign((size_t)K, 0);
    } catch (const std::bad_alloc &) {
        return CELTY_ENOMEM;
    }
    int64_t kept = 0, pads = 0;
    for (int64_t i = 0; i < M; ++i) {
        const uint8_t *row = mask + i * ldm;
        for (int64_t j = 0; j < K; ++j) {
            if (!row[j]) {
                ++gap[(size_t)j];
                continue;
            }
            ++kept;
            pads += gap[(size_t)j] >> run_bits;      // a padding entry covers 2^run_bits rows: its run and itself
            gap[(size_t)j] = 0;
        }
    }
    if (nnz) *nnz = kept;
    if (n_pad) *n_pad = pads;
    return CELTY_OK;
}

extern "C" int celty_set_launch(celty_matrix *m, int32_t grid, int32_t variant, int32_t groups, int32_t depth,
                                int32_t cluster)
{
    if (!m || grid < 0 || variant < 0 || variant > 509 || groups < 0 || groups > 16 || depth < 0 || depth > 16 ||
        !(cluster == 0 || cluster == 1 || cluster == 2 || cluster == 4))
        return CELTY_EINVAL;
    m->grid = grid;
    // variant: bit 0 selects the two-launch path; 2 / 4 force the ordered two-stage / the bulk reduce-add merge
    m->merge = (variant & 2) ? 0 : (variant & 4) ? 1 : -1;
    m->no_overlap = (variant & 8) ? 1 : 0;
    m->variant = variant & 1;
    m->pairs = (variant & 16) ? 1 : (variant & 32) ? 0 : -1;
    m->mix = (variant & 64) ? 0 : (variant & 128) ? 1 : -1;
    m->lean = (variant & 256) ? 0 : -1;
    m->groups = groups;
    m->depth = depth;
    m->cluster = cluster;
    m->forget_launches();
    return CELTY_OK;
}

extern "C" int celty_set_register_rows(celty_matrix *m, int32_t rows)
{
    if (!m || !(rows == 0 || rows == 32 || rows == 64 || rows == 96 || rows == 128)) return CELTY_EINVAL;
    m->reg_rows = rows;
    m->forget_launches();
    return CELTY_OK;
}

extern "C" int celty_set_wait_limit(celty_matrix *m, uint32_t polls)
{
    if (!m) return CELTY_EINVAL;
    m->spin_limit = polls;
    m->forget_launches();
    return CELTY_OK;
}

extern "C" const char *celty_strerror(int status)
{
    switch (status) {
        case CELTY_OK: return "ok";
        case CELTY_EINVAL: return "invalid argument";
        case CELTY_ENOMEM: return "out of memory or buffer too small";
        case CELTY_ECUDA: return "CUDA runtime error";
        case CELTY_ESTATE: return "handle is not bound to device memory";
        case CELTY_ETIMEOUT: return "a bounded wait inside a kernel ran out";
        case CELTY_EBOUNDS: return "a decoded index was out of range";
        case CELTY_ELIMIT: return "size exceeds the fixed scratch of the no-allocation entry point";
        default: return "unknown status";
    }
}
