// Host check of the following's integer filter (csrc/abg.cuh): the 32-bit form against the 64-bit
// form on random chains over the whole 16-bit input range (also far outside the pads and the drift
// length) and on extensions whose hits lie at the ends of the search window, so that states wrap
// around the word.  Both must take the same decisions at every row.  Compiled with signed overflow
// trapping.  Prints the number of predictions compared and of chains that left the 32-bit range.
#include <cstdio>
#include <cstdlib>
#include <random>

#include "abg.cuh"

using namespace tpc;

constexpr int M_MISS = 8, W_F0 = 77, W_F1 = 38, V_MAX = 320;

static std::mt19937 rng(7);
static int uni(int lo, int hi) { return std::uniform_int_distribution<int>(lo, hi)(rng); }

struct Chain {
    int n, y[40], z[40], d[40];
};

template <class T>
struct Run {
    Abg<T> y, z;
    void filter(const Chain &c) {
        abg_init(y, c.y[0], c.y[1], c.d[1]);
        abg_init(z, c.z[0] - Abg<T>::ZB, c.z[1] - Abg<T>::ZB, c.d[1]);
        for (int k = 1; k < c.n; k++) {
            for (int j = 0; j < c.d[k]; j++) {
                abg_predict(y);
                abg_predict(z);
            }
            abg_update(y, c.y[k]);
            abg_update(z, c.z[k] - Abg<T>::ZB);
        }
    }
    // one row further: whether the prediction is inside, and where
    bool step(int ymax, int zmax, int *py, int *pz) {
        abg_predict(y);
        abg_predict(z);
        *py = q16_round(y.p);
        *pz = q16_round(z.p) + Abg<T>::ZB;
        return !(abs(*py) > ymax || *pz < 0 || *pz > zmax || y.v > (T)V_MAX * 65536 || y.v < -(T)V_MAX * 65536);
    }
    void hit(int my, int mz) {
        abg_update(y, my);
        abg_update(z, mz - Abg<T>::ZB);
    }
};

int main(int argc, char **argv) {
    const int chains = argc > 1 ? atoi(argv[1]) : 200000;
    long long compared = 0, wrapped = 0;
    for (int it = 0; it < chains; it++) {
        // links reach 384 LSB a row (768 across a skipped one); steps that change slowly or at random,
        // and chains that run towards the ends of the range; every second one starts inside the detector
        Chain c;
        c.n = uni(5, 39);
        const int kind = uni(0, 3);
        c.y[0] = kind == 3 ? (uni(0, 1) ? 32767 : -32768) : uni(-32768, 32767);
        c.z[0] = kind == 2 ? uni(48000, 65535) : kind == 3 ? uni(0, 1) * 65535 : uni(0, 65535);
        if (it % 2) c.y[0] = uni(-12000, 12000), c.z[0] = uni(0, NARROW_ZMAX);
        int sy = uni(-384, 384), sz = uni(-384, 384);
        for (int k = 1; k < c.n; k++) {
            c.d[k] = uni(0, 9) == 0 ? 2 : 1;
            if (kind == 0) sy = uni(-384, 384), sz = uni(-384, 384);
            else sy = std::min(std::max(sy + uni(-58, 58), -384), 384), sz = std::min(std::max(sz + uni(-58, 58), -384), 384);
            c.y[k] = std::min(std::max(c.y[k - 1] + sy * c.d[k], -32768), 32767);
            c.z[k] = std::min(std::max(c.z[k - 1] + sz * c.d[k], 0), 65535);
        }
        Run<int32_t> a;
        Run<long long> b;
        a.filter(c);
        b.filter(c);
        const int ymax = it & 2 ? NARROW_YMAX : uni(1000, NARROW_YMAX), zmax = it & 4 ? NARROW_ZMAX : uni(1000, NARROW_ZMAX);
        if (b.y.p > INT32_MAX || b.y.p < INT32_MIN || b.z.p - (16384ll << 16) > INT32_MAX) wrapped++;
        int misses = 0;
        const int bias = uni(0, 2);      // hits always at one end of the window, or anywhere in it
        for (int row = 0; row < 512; row++) {
            int ya, za, yb, zb;
            const bool ib = b.step(ymax, zmax, &yb, &zb);
            const bool ia = c.z[c.n - 1] <= NARROW_ZHIT && a.step(ymax, zmax, &ya, &za);
            compared++;
            if (ia != ib || (ib && (ya != yb || za != zb))) {
                printf("chain %d row %d: %d (%d, %d) against %d (%d, %d)\n", it, row, ia, ya, za, ib, yb, zb);
                return 1;
            }
            if (!ib) break;
            const int w = W_F0 + W_F1 * misses;
            if (uni(0, 3) == 0 && misses < M_MISS - 1) { misses++; continue; }
            const int dy = bias == 2 ? uni(-w, w) : bias ? w : -w, dz = bias == 2 ? uni(-w, w) : uni(0, 1) ? w : -w;
            const int my = std::min(std::max(yb + dy, -32768), 32767), mz = std::min(std::max(zb + (uni(0, 1) ? dz : w), 0), 65535);
            a.hit(my, mz);
            b.hit(my, mz);
            misses = 0;
        }
    }
    printf("compared %lld wrapped %lld\n", compared, wrapped);
    return 0;
}
