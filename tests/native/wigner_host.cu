// The float-pair functions of the Wigner noise (csrc/wigner.cuh, host branch) against long double: the largest
// relative errors (log2) of the Box-Muller radius, the cosine and the sine over the words where the reductions
// change (0, 2^k and the table intervals' and directions' edges, each with its neighbours) and argv[1] random ones.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <random>

#include "wigner.cuh"

using namespace twa;
static constexpr WignerTables W = make_wigner_tables();

int main(int, char** argv) {
    double worst[3] = {0, 0, 0};
    uint32_t at[3] = {0, 0, 0};
    const long double pi = 3.14159265358979323846264338327950288L;
    long long words = 0;
    auto hold = [&](int i, uint32_t c, Pair<float> got, long double want) {
        const double e = std::fabs((double)(((long double)got.hi + got.lo - want) / want));
        if (!(e <= worst[i])) {   // NaN too
            worst[i] = e;
            at[i] = c;
        }
    };
    auto check = [&](uint32_t c) {
        ++words;
        const long double u = ((long double)c + 0.5L) / 4294967296.0L;
        const RadiusWord r = radius_word(c, W.rec);
        hold(0, c, bm_radius(r.mh, r.ml, r.T.x, r.T.y, r.T.z, r.E), sqrtl(-2.0L * (u < 0.5L ? logl(u) : log1pl(u - 1.0L))));
        // the angle 2 pi (2 c + 1) / 2^33 to the nearest quarter turn, in integers
        const uint64_t a = 2ull * c + 1, quarter = (a + (1ull << 30)) >> 31;
        const long double d = (long double)((int64_t)a - (int64_t)(quarter << 31)) * 2.0L * pi / 8589934592.0L;
        const long double co = cosl(d), si = sinl(d);
        const int q = quarter & 3;
        const DirectionWord w = direction_word(c, W.dir);
        Pair<float> pc, ps;
        bm_direction(w.rest, w.D.x, w.D.y, w.D.z, w.D.w, pc, ps);
        hold(1, c, pc, q == 0 ? co : (q == 1 ? -si : (q == 2 ? -co : si)));
        hold(2, c, ps, q == 0 ? si : (q == 1 ? co : (q == 2 ? -si : -co)));
    };
    for (uint32_t i = 0; i < 5000; ++i) {
        check(i);
        check(~i);
    }
    for (int b = 0; b < 32; ++b)
        for (int d = -600; d < 600; ++d) check((1u << b) + d);
    for (uint32_t j = 0; j < 256; ++j)
        for (int d = -300; d < 300; ++d) {
            check((j << 24) + d);
            check((j << 24) + (1u << 23) + d);
        }
    for (uint32_t j = 0; j < 128; ++j)
        for (int e = 0; e < 25; ++e)
            for (int d = -30; d < 30; ++d) check(((0x80000000u | (j << 24)) >> e) + d);
    std::mt19937 g(1);
    for (long long i = std::atoll(argv[1]); i > 0; --i) check((uint32_t)g());
    std::printf("%lld", words);
    for (int i = 0; i < 3; ++i) std::printf(" %.3f %u", std::log2(worst[i]), at[i]);
    std::printf("\n");
}
