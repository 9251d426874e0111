// The factor loads of the fixed-point operator (ax_fx_core.cuh, fx_operator) on
// one element, for every order and thread layout that is launched: prints the
// number of loads outside the element's 3 n^3 entries.
#include "device_on_host.h"

#include <stdio.h>

#include "../../paper_2005_13425_gb300/csrc/ax_fx_core.cuh"

using namespace nekgb;

template <int N, bool EO, int G>
static void run() {
    constexpr int A = fx_array(N), N3 = N * N * N;
    auto D = std::make_unique<typename FxConsts<N, EO>::type>();
    memset(D.get(), 0, sizeof *D);
    std::vector<int2> sm(4 * A);
    std::vector<int4> g(3 * N3);
    unsigned low = 0;
    host::lo = (const char *)g.data();
    host::hi = (const char *)(g.data() + g.size());
    host::outside = 0;
    host::cta(fx_threads(N, G), [&] {
        FxThread<N, G> th;
        th.init();
        int2 *X = sm.data(), *R = X + A, *S = X + 2 * A, *TT = G == 3 ? X + 3 * A : X;
        const bool on = th.active && th.el == 0;    // one element; the CTA's others are past the end
        fx_operator<N, EO>(th, on, X, R, S, TT, g.data() + th.column(), *D, &low);
    });
    printf("%d %d %d %ld\n", N, (int)EO, G, host::outside);
}

template <int N>
static void orders() {
    run<N, true, 1>();
    run<N, true, 3>();
    run<N, false, 1>();
    if constexpr (N > 2) orders<N - 1>();
}

int main() {
    orders<16>();
    return 0;
}
