"""The host encoder with and without vector instructions packs the same image, byte for byte (the plain build's entries are
held to the oracle's rule where the library runs without them; the vector build's in test_host_encoder).  No GPU needed."""
import os
import subprocess

import pytest

from conftest import ROOT

CSRC = os.path.join(ROOT, "paper_2608_01536_b200", "csrc")
MAIN = r'''
#include <cstdio>
#include <cstdlib>
#include <random>
#include <thread>
#include <vector>
#include "celty.h"
#ifdef NO_COUNT                                  // a system that does not say how many processors it has
unsigned std::thread::hardware_concurrency() noexcept { return 0; }
#endif
int main(int, char **v) {
    const int M = atoi(v[1]), K = atoi(v[2]), tile_rows = atoi(v[3]), kept = atoi(v[4]), column = atoi(v[5]);
    std::mt19937 r(M * 31 + K);
    std::vector<uint16_t> W((size_t)M * K);
    std::vector<uint8_t> mask((size_t)M * K);
    for (size_t i = 0; i < W.size(); ++i) { W[i] = (uint16_t)r(); mask[i] = (int)(r() % 1000) < kept; }
    celty_encode_opts o = {4, column ? CELTY_LAYOUT_COLUMN : CELTY_LAYOUT_LANE_TILE, tile_rows, 0};
    for (int with_mask = 0; with_mask < 2; ++with_mask) {
        celty_matrix *m;
        if (celty_encode(W.data(), K, with_mask ? mask.data() : nullptr, M, K, &o, &m)) return 1;
        const void *image; size_t bytes, at;
        celty_host_image(m, &image, &bytes, &at);
        fwrite(image, 1, bytes, stdout);
        for (int j = 0; j < K; j += 1 + K / 7) {
            std::vector<uint8_t> runs(4 * M + 64), pads(4 * M + 64);
            int64_t n;
            if (celty_decode_host(m, j, nullptr, nullptr, runs.data(), pads.data(), 4 * M + 64, &n)) return 2;
            fwrite(runs.data(), 1, n, stdout);
            fwrite(pads.data(), 1, n, stdout);
        }
        celty_destroy(m);
    }
}
'''


@pytest.fixture(scope="module")
def encoders(tmp_path_factory):
    d = tmp_path_factory.mktemp("encoders")
    (d / "main.cpp").write_text(MAIN)
    exes = []
    for k, flags in enumerate(([], ["-DCELTY_PLAIN_ENCODER"], ["-DNO_COUNT"])):
        exes.append(str(d / ("encoder%d" % k)))
        subprocess.check_call(["g++", "-O2", "-std=c++17", "-pthread", *flags, "-I", os.path.join(ROOT, "include"), "-I", CSRC,
                               os.path.join(CSRC, "celty_host.cpp"), str(d / "main.cpp"), "-o", exes[-1]])
    return exes


# rows per tile on both sides of a 64-bit word of kept bits and the largest; ragged rows and columns; all, half, few and no padding
@pytest.mark.parametrize("M,K,tile_rows,kept,column", [
    (1, 1, 0, 500, 0), (33, 63, 0, 500, 0), (40, 65, 1, 1000, 0), (2016, 130, 63, 500, 0), (2048, 64, 64, 1000, 0), (2080, 129, 65, 300, 0),
    (7680, 70, 240, 500, 0), (7681, 70, 240, 900, 0), (4100, 200, 128, 60, 0), (2048, 300, 0, 500, 0), (1000, 200, 0, 1, 0), (777, 130, 0, 500, 1),
    (3000, 64, 96, 980, 0)])
def test_plain_and_vector_builds_agree(encoders, M, K, tile_rows, kept, column):
    outs = [subprocess.check_output([e, *map(str, (M, K, tile_rows, kept, column))]) for e in encoders[:2]]
    assert len(outs[0]) > 0 and outs[0] == outs[1]


@pytest.mark.parametrize("M,K,column", [(1024, 1024, 0), (1024, 1024, 1), (21000, 70, 0), (100, 100, 0)])
def test_a_system_without_a_processor_count(encoders, M, K, column):
    outs = [subprocess.check_output([e, *map(str, (M, K, 0, 500, column))]) for e in (encoders[0], encoders[2])]
    assert len(outs[0]) > 0 and outs[0] == outs[1]


def test_encoder_threads_that_wait_leave_the_processor(tmp_path):
    """One of eight threads takes 0.3 s of wall-clock time over each of two phases: the others look for a moment and sleep."""
    (tmp_path / "main.cpp").write_text(r'''
#include "celty_host.cpp"
#include <cstdio>
#include <ctime>
int main() {
    std::atomic<int> turn[2] = {{0}, {0}}, seen(0), between(0);
    if (!in_phases(8, 2, [&](int p, Scratch &) {
            if (between != p) exit(2);                            // nobody is ahead
            if (turn[p]++ == 3) std::this_thread::sleep_for(std::chrono::milliseconds(300));
            ++seen;
        }, [&](int) { if (seen != 8 * ++between) exit(3); }))
        return 1;
    printf("%.4f", (double)clock() / CLOCKS_PER_SEC);
}
''')
    exe = str(tmp_path / "phases")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-pthread", "-I", os.path.join(ROOT, "include"), "-I", CSRC, str(tmp_path / "main.cpp"), "-o", exe])
    assert float(subprocess.check_output([exe])) < 0.1            # seconds of processor time; seven threads that poll: up to 4
