"""Totals of a tick at and above 2^30 and 2^32, on the host, in the code that
the kernels and the C ABI share (mqr_internal.cuh): a leaf's filter work, the
look-back's status words, and which totals refuse a tick."""
import subprocess

from paper_1411_3212_gb300 import build

PROGRAM = r"""
#include <cstdio>
#include "mqr_internal.cuh"
using namespace mqr;
using u64 = unsigned long long;
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); bad = 1; } } while (0)

// The prefixes that consecutive tiles read back from each other's status words.
template <typename T>
static bool prefixes_hold(const u64 *agg, int n) {
    u64 want = 0;
    T word = status_word<T>(2, 0);
    for (int i = 0; i < n; ++i) {
        if (status_flag(word) != 2u || status_sum(word) != want) return false;
        const T own = status_word<T>(1, (T)agg[i]);
        if (status_flag(own) != 1u || status_sum(own) != agg[i]) return false;
        want += agg[i];
        word = status_word<T>(2, (T)(status_sum(word) + status_sum(own)));
    }
    return status_flag(word) == 2u && status_sum(word) == want;
}

static LeafScanSum *scan_status(void (*)(cudaStream_t, int, uint32_t, const uint32_t *, const uint32_t *, uint32_t *,
                                         uint32_t *, uint32_t *, uint32_t *, LeafScanSum *, uint32_t *, Caps, Info *)) {
    return nullptr;
}

static PairSum *pair_status(void (*)(cudaStream_t, const float4 *, uint32_t, float, float, float, float, Worlds,
                                     const uint32_t *, const uint32_t *, const uint32_t *, uint2 *, uint4 *, uint32_t *,
                                     uint32_t *, u64, PairSum *, u64 *, uint32_t *, Info *)) {
    return nullptr;
}

int main() {
    int bad = 0;
    // a leaf's words and items
    CHECK(leaf_work(1, 1).words == 1 && leaf_work(1, 1).items == 1);
    CHECK(leaf_work(128, 0).words == 0 && leaf_work(128, 0).items == 0);
    CHECK(leaf_work(257, 33).words == 9 * 33 && leaf_work(257, 33).items == 2 * 2);
    CHECK(leaf_work(4000000, 10000).words == 1250000000ull && leaf_work(4000000, 10000).items == 15625ull * 313);
    CHECK(leaf_work(4000000, 40000).words == 5000000000ull);
    CHECK(leaf_work((1u << 30) - 1, (1u << 30) - 1).words == (u64)(1u << 25) * ((1u << 30) - 1));
    CHECK(leaf_work((1u << 30) - 1, (1u << 30) - 1).items == (u64)(1u << 22) * (1u << 25));
    // what tiles hand on: the leaf scan's sums pass 2^30 and 2^32
    const u64 pile[] = {1250000000ull, 176000000ull, 3000000000ull, 0ull, 1ull << 40};
    (void)scan_status(launch_leaf_scan);                  // the kernel's status words are these
    CHECK(prefixes_hold<LeafScanSum>(pile, 5));
    // and so do nine pairs of each of up to 2^30 queries
    const u64 pairs[] = {9ull * 119304648, 9ull * 119304648, 9ull * 400000000, 0ull, 504ull};
    (void)pair_status(launch_query_blocks);
    CHECK(prefixes_hold<PairSum>(pairs, 5) && !prefixes_hold<uint32_t>(pairs, 1));
    const u64 leaves[] = {2048, 0, (1u << 30) - 2049};     // leaves: fewer than 2^30
    CHECK(prefixes_hold<uint32_t>(leaves, 3));
    CHECK(!prefixes_hold<uint32_t>(pile, 1));              // why 32-bit words do not do
    // which totals refuse a tick
    Info in{};
    CHECK(tick_limit(in, true) == kTickFits);
    for (u64 w : {1ull << 30, (1ull << 32) - 1}) {
        in.n_words = w;
        CHECK(tick_limit(in, true) == kTickFits);
    }
    for (u64 w : {1ull << 32, (1ull << 32) + (1ull << 30), 1ull << 40}) {
        in.n_words = w;
        CHECK(tick_limit(in, true) == kTickWords);
        CHECK(tick_limit(in, false) == kTickFits);         // no bitmaps
    }
    in.n_words = 0;
    in.n_items = (1ull << 32) - 256;
    CHECK(tick_limit(in, true) == kTickFits && in.n_items + 4 < (1ull << 32));
    in.n_items = 1ull << 32;
    CHECK(tick_limit(in, true) == kTickWords && tick_limit(in, false) == kTickWords);
    in.n_cand = kMaxCandTiles * 32;
    in.n_items = 0;
    CHECK(tick_limit(in, true) == kTickFits);
    in.n_cand += 1;
    CHECK(tick_limit(in, true) == kTickCandidates);
    // the result scan's tiles: none past the records starts at one of them, and
    // no thread of the last tile takes records past the last
    CHECK(res_tile_begin((1u << 21) + 5) == (1ull << 32) + 5 * (u64)kResTile);
    const uint32_t most = (uint32_t)(kMaxCandTiles * 32), last = most / kResTile * kResTile;
    CHECK(res_tile_begin(most / kResTile) == last && most - last < (uint32_t)kResTile);
    for (uint32_t nsub : {most, most - 8, most - 31, 2048u, 2049u, 7u, 8u})
        for (uint32_t t = 0; t < (uint32_t)kResThreads; ++t) {
            const uint32_t kb = (nsub - 1) / kResTile * kResTile + t * kResItems;
            CHECK(res_items_whole(kb, nsub) == ((u64)kb + kResItems <= nsub));
        }
    return bad;
}
"""


def test_totals_beyond_32_bits(tmp_path):
    build.build()
    src, exe = tmp_path / "limits.cu", tmp_path / "limits"
    src.write_text(PROGRAM)
    subprocess.run([build._nvcc(), *build.ARCH, *build.FLAGS, "-I" + build.CSRC, "-o", str(exe), str(src), "-L" + build.HERE,
                    "-lmqr", "-Xlinker", "-rpath=" + build.HERE], check=True)
    r = subprocess.run([str(exe)], stdout=subprocess.PIPE, text=True)
    assert r.returncode == 0, r.stdout
