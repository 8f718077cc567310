// The batch autotuner over made-up rounds (see test_autotune_host.py); argv[1]:
// a file to keep measurements in.
#include <cstdio>

#include "autotune.h"

using namespace snp;

// A machine on which candidate `fast` is 1.5 times as fast as the others.
static int round(Autotune& t, double work, int fast) {
    const int c = t.pick(2, 16, work);
    t.record(2, 16, c, work, work / (c == fast ? 1.5e9 : 1e9));
    return c;
}

int main(int, char** argv) {
    int bad = 0;
    {  // one large round, then a steady load of smaller ones: tried and tuned
        Autotune t;
        round(t, 1e9, 2);
        int last = -1, seen = 0;
        for (int i = 0; i < 20; ++i) seen |= 1 << (last = round(t, 1e8, 2));
        bad += last != 2 || seen != 7;
    }
    {  // what a file holds outlives a small first round and one of far more work
        Autotune a;
        for (int i = 0; i < 5; ++i) round(a, 4e9, 1);
        bad += a.pick(2, 16, 4e9) != 1;
        a.save(argv[1]);
        Autotune b;
        b.load(argv[1]);
        bad += round(b, 1e6, 1) != 1;  // a level of its own: the nearest one's choice
        for (int i = 0; i < 5; ++i) bad += round(b, 4e9, 1) != 1;
        b.save(argv[1]);
        Autotune c;
        c.load(argv[1]);
        bad += c.pick(2, 16, 4e9) != 1 || c.pick(2, 16, 5e10) != 1;
        bad += c.pick(2, 15, 4e9) != 0 || c.pick(4, 16, 4e9) != 0;  // other sizes and widths: nothing known
    }
    {  // small rounds, in which everything is slow, leave a large one's choice alone
        Autotune t;
        for (int i = 0; i < 4; ++i) round(t, 4e9, 0);
        for (int i = 0; i < 9; ++i) {
            const int c = t.pick(2, 16, 1e5);
            t.record(2, 16, c, 1e5, 1.0);
        }
        bad += t.pick(2, 16, 4e9) != 0;
    }
    {  // a load that falls through many levels once keeps to the known choice
        Autotune t;
        for (int i = 0; i < 4; ++i) round(t, 4e9, 2);
        for (double w = 1e9; w > 1e3; w /= 4) bad += round(t, w, 2) != 2;
    }
    {  // lines without a level, and of an earlier set of candidates
        FILE* f = std::fopen(argv[1], "w");
        std::fprintf(f, "2 16 6 1e9 1\n2 16 7 1e9 3\n2 16 8 1e9 0.5\n2 16 3 1e9 1e-3\n");
        std::fclose(f);
        Autotune t;
        t.load(argv[1]);
        bad += t.pick(2, 16, 1e7) != 2;
    }
    std::printf("bad=%d\n", bad);
    return bad;
}
