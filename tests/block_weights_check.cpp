// Host check of the block trees' leaf records (csrc/blocks_planner.cpp, leaf_weight): a weight is
// accepted only when both records give it back exactly, and every merged weight of the library's
// operators named on the command line is.  Built and run by tests/test_blocks_cpu.py; prints "OK
// <count>" or the first failure.
#include "blocks.hpp"

#include <cstdio>
#include <cstdlib>
#include <cstring>

using namespace mbc;

static bool exact(cplx w) {                 // what the device trees compute with
    uint32_t fb, hw;
    if (!leaf_weight(w, fb, hw)) return false;
    float f;
    double d;
    const uint64_t bits = (uint64_t)hw << 32;
    std::memcpy(&f, &fb, 4);
    std::memcpy(&d, &bits, 8);
    if (w.imag() != 0.0 || (double)f != w.real() || d != w.real()) {
        printf("FAIL accepted %.17g + %.17g i\n", w.real(), w.imag());
        exit(1);
    }
    return true;
}

int main(int argc, char** argv) {
    long done = 0;
    for (double x : {0.0, 1.0, -1.0, 48.0, -2.5, 2097151.0, -2097151.0, 4194302.0, 4194304.0 * 3, 0.375})
        if (!exact(x)) { printf("FAIL refused %.17g\n", x); return 1; } else ++done;
    for (double x : {2097152.0 + 0.5, 4194307.0, -4194307.0, 8388609.0, 16777217.0, 1.0 / 3.0, 1e300, 1e-300})
        if (exact(x)) { printf("FAIL accepted %.17g\n", x); return 1; } else ++done;
    if (exact(cplx(1.0, 1.0)) || exact(cplx(0.0, -1.0))) { printf("FAIL accepted a complex weight\n"); return 1; }
    for (int a = 1; a < argc; ++a) {
        BlockHostPlan p;
        p.op = atoi(argv[a]);
        const std::string err = plan_blocks(p);
        if (!err.empty()) { printf("FAIL %s\n", err.c_str()); return 1; }
        for (const cplx& w : p.w)
            if (!exact(w)) { printf("FAIL operator %d refused %.17g + %.17g i\n", p.op, w.real(), w.imag()); return 1; } else ++done;
    }
    printf("OK %ld\n", done);
    return 0;
}
