// Prints the tiles of the grouped GEMM (make_tiles of the library) for one task of M x N outputs (herm: the lower triangle of
// M x M) over K: checks that they follow one another without a gap, in 64 bits, and that split tiles' partial sums do too.
#include <cstdio>
#include <cstdlib>

#include "internal.h"

int main(int argc, char** argv) {
    using namespace tdmrg;
    if (argc != 5) return 2;
    TaskList tl;
    Task t{};
    Seg s{};
    t.M = atoi(argv[1]); t.N = atoi(argv[2]); t.herm = (int8_t)atoi(argv[4]);
    t.seg_end = 1;
    s.K = atoi(argv[3]);
    tl.tasks.push_back(t);
    tl.segs.push_back(s);
    make_tiles(tl);
    const int64_t outs = t.herm ? (int64_t)t.M * (t.M + 1) / 2 : (int64_t)t.M * t.N;
    int64_t next = 0, partial = 0;
    for (const Tile& x : tl.tiles) {   // one cost but for the last tile's, so they stay in order
        const int64_t o = t.herm ? (int64_t)x.m0 * (x.m0 + 1) / 2 + x.o0 : (int64_t)x.m0 * t.N + x.o0;
        if (x.m0 < 0 || x.m0 >= t.M || x.o0 < 0 || x.cnt < 1 || x.cnt > 256 || (outs > kFlatOuts && x.o0 >= (t.herm ? x.m0 + 1 : t.N))) {
            printf("tile out of range: row %d column %d count %d\n", x.m0, x.o0, x.cnt);
            return 1;
        }
        const int64_t want = x.split < 0 || x.part == 0 ? next : next - x.cnt;
        if (o != want) {
            printf("tile at %lld instead of %lld\n", (long long)o, (long long)want);
            return 1;
        }
        if (x.split < 0 || x.part == 0) next += x.cnt;
        if (x.split >= 0 && x.part == 0) {
            if (32 * (int64_t)x.split_base != partial) { printf("partial sums at %lld\n", (long long)x.split_base); return 1; }
            partial += (int64_t)x.nparts * ((x.cnt + 31) & ~31);
        }
    }
    if (next != outs || partial != tl.npartial) { printf("covered %lld of %lld\n", (long long)next, (long long)outs); return 1; }
    return 0;
}
