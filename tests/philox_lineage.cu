// Host program: philox4x32_10_lineage, philox_lineage_b and philox_lineage_words
// against Philox4x32-10 of the plain counter.  Prints the number of counters that
// differ.
#include <cstdio>

#include "gm_common.cuh"

using namespace gm;

struct RoundKey {
    uint2 k;
    __host__ __device__ uint2 operator()(int r) const { return philox_round_key(k, r); }
};

int main() {
    const uint32_t edge[] = {0u, 1u, 2u, 0x7FFFFFFFu, 0x80000000u, 0xFFFFFFFEu, 0xFFFFFFFFu, 0x9E3779B9u};
    uint64_t state = 1;
    auto word = [&]() {  // an edge value for one word in four
        state = state * 6364136223846793005ull + 1442695040888963407ull;
        const uint32_t r = (uint32_t)(state >> 32);
        return (r & 3u) == 0u ? edge[r >> 29] : r * 2654435761u;
    };
    long bad = 0;
    const long n = 2000000;
    for (long i = 0; i < n; ++i) {
        const uint32_t draw = word(), lo = word(), hi = word(), hist = word();
        const uint2 k = make_uint2(word(), word());
        const RoundKey key{k};
        const uint4 want = philox4x32_10(make_uint4(draw, lo, hi, hist), k);
        PhiloxLineage l = philox_lineage(lo, hi, key(0), key(1));
        const uint4 got = philox4x32_10_lineage(draw, hist, l, key);
        // a record keeps a and c
        l.b = philox_lineage_b(l.c, key(1));
        const uint4 again = philox4x32_10_lineage(draw, hist, l, key);
        const uint2 own = philox_lineage_words(l.a, l.c, key(0), key(1));
        const bool ok = got.x == want.x && got.y == want.y && got.z == want.z && got.w == want.w &&
                        again.x == want.x && again.y == want.y && again.z == want.z && again.w == want.w &&
                        own.x == lo && own.y == hi;
        bad += !ok;
    }
    printf("%ld of %ld differ\n", bad, n);
    return bad != 0;
}
