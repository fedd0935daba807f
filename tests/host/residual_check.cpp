// Host-side check of the refinement residual's items (no GPU): for every number
// of slots, each slab of each block meets each chunk of each source block
// exactly once and each slot of its rows is written exactly once; and with less
// memory than the usual slots take, fewer are used instead of refusing the solve.
// Prints "ok" and exits 0 on success.
#include <cstdio>
#include <vector>

#include "krr_internal.h"

namespace {

int check(const krr::ResGrid &q) {
    const int64_t nt = q.nt, S = q.S, KC = q.KC, slots = q.slots();
    std::vector<uint8_t> met(nt * S * nt * KC), wrote(slots * nt * S);
    for (int64_t t = 0; t < q.items(); ++t) {
        krr::ResItem it;
        if (!krr::res_decode(q, (int)t, it)) continue;
        if (it.i < 0 || it.i >= nt || it.sl < 0 || it.sl >= S || it.j0 < 0 || it.j1 > nt || it.kc0 < 0 ||
            it.kc1 > KC || it.j0 >= it.j1 || it.kc0 >= it.kc1 || it.slot < 0 || it.slot >= slots)
            return 1;
        if (wrote[(it.slot * nt + it.i) * S + it.sl]++) return 2;
        for (int64_t j = it.j0; j < it.j1; ++j)
            for (int64_t k = it.kc0; k < it.kc1; ++k)
                if (met[((it.i * S + it.sl) * nt + j) * KC + k]++) return 3;
    }
    for (uint8_t w : wrote)
        if (!w) return 4;
    for (uint8_t m : met)
        if (!m) return 5;
    return 0;
}

}  // namespace

int main() {
    const int64_t edges[][2] = {{2, 4}, {4, 8}, {8, 16}, {32, 64}};  // tile edge 256, 512, 1024, 4096
    for (int64_t nt : {1, 2, 3, 5, 7, 10, 20, 47, 48, 49, 51, 97, 130})
        for (const auto &e : edges) {
            if (nt * nt * e[0] * e[1] > 4000000) continue;
            for (int64_t ctas : {152, 48})
                for (int most : {48, 24, 10, 5, 3, 2, 1}) {
                    const krr::ResGrid q = krr::res_grid(nt, e[0], e[1], ctas, most);
                    const int bad = (q.slots() > most || (q.g > 1 && q.h > 1)) ? 9 : check(q);
                    if (bad) {
                        std::printf("nt %d S %d KC %d slots %d: %d\n", (int)nt, (int)e[0], (int)e[1], most, bad);
                        return 1;
                    }
                }
        }
    // an allocator with room for `room` slots: the solve gets at least half of
    // them, a refusal only if one does not fit, and the next solve asks for no more
    for (int64_t nt : {1, 5, 40, 97, 1024})
        for (int room : {100, 48, 47, 30, 7, 2, 1, 0}) {
            int most = krr::RES_SLOTS, asked = 0;
            krr::ResGrid q;
            const auto alloc = [&](const krr::ResGrid &g) {
                ++asked;
                return g.slots() <= room ? KRR_OK : KRR_ENOMEM;
            };
            const int want = krr::res_grid(nt, 8, 16, 152, krr::RES_SLOTS).slots();
            const krr_status st = krr::res_reserve(nt, 8, 16, 152, &most, alloc, &q);
            if (st != (room > 0 ? KRR_OK : KRR_ENOMEM)) return 2;
            if (st == KRR_OK && !(q.slots() <= room && (q.slots() == want || 4 * q.slots() > room))) {
                std::printf("nt %d room %d: %d slots\n", (int)nt, room, q.slots());
                return 3;
            }
            asked = 0;
            if (krr::res_reserve(nt, 8, 16, 152, &most, alloc, &q) != st || (st == KRR_OK && asked != 1)) return 4;
        }
    // any other error is passed on
    int most = krr::RES_SLOTS;
    krr::ResGrid q;
    if (krr::res_reserve(9, 8, 16, 152, &most, [](const krr::ResGrid &) { return KRR_ECUDA; }, &q) != KRR_ECUDA) return 5;
    std::printf("ok\n");
    return 0;
}
