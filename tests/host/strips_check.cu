// Host-side check of the 2D strip kernels' work split (no GPU call): a call that
// reduces is taken only where its CTAs' partials fit the reduction scratch, and
// a call that does not reduce is taken at every size.  Prints one line per
// violation and "ok <cases>" at the end.
#include <cstdio>
#include <cstring>

#include "stencil_fx2d.cuh"

using namespace jfnk;

template <typename T>
static int check(int n, RedOut red, bool want) {
    StencilArgs<T> a;
    memset(&a, 0, sizeof(a));
    a.g = Grid::make(2, n);
    a.node_scale = T(1);
    a.red = red;
    const bool got = fx2d_use<T>(Prob::BRATU2, a, Mode::JV);
    if (got != want) printf("n=%d red=%d: taken %d, expected %d\n", n, (int)red, got, want);
    return got == want ? 0 : 1;
}

int main() {
    int bad = 0, cases = 0;
    // one CTA a strip of 30 node columns at the least: 2 kMaxRedBlocks strips
    const int last = 30 * 2 * kMaxRedBlocks + 1;
    for (int n : {2, 31, 32, 4096, last - 1, last, last + 1, 2 * last}) {
        bad += check<double>(n, RedOut::NONE, true) + check<float>(n, RedOut::NONE, true);
        bad += check<double>(n, RedOut::EPS, n <= last) + check<float>(n, RedOut::NORM, n <= last);
        cases += 4;
    }
    if (bad == 0) printf("ok %d\n", cases);
    return bad == 0 ? 0 : 1;
}
