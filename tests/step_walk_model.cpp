// A model of the barriers between the loads, the decoding warps and the MMAs of gemm_tmw_kernel, for tests/test_step_walk.py: agents
// that take their steps in random order, loads that land in any order.  It walks the kernel's own index arithmetic (StepWalk).
//   step_walk_model SPR A_STAGES KBLOCKS TILES SEEDS ASKS
// ASKS 1: as the kernel; 0: no group asks whether a slot is empty before it asks whether it is full, no load waits for one before.
// Prints how many of the runs went wrong: a stage read that was not (or no longer) the wanted one, or no agent able to move.
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>

#include "../paper_2307_15517_b200/csrc/mx_step_walk.h"

namespace {

constexpr int GROUPS = 3, WARPS = 2, RS = 4;         // two warps stand for a group's four in either CTA

struct Barrier {
    int count = 1, arrived = 0;
    uint32_t phase = 0;
    void arrive(int n = 1)
    {
        arrived += n;
        if (arrived >= count) { arrived -= count; ++phase; }
    }
    bool test(uint32_t parity) const { return (phase & 1u) != parity; }      // as mbarrier.test_wait.parity
};

template <int SPR> bool run(int as, int kblocks, int tiles, unsigned seed, bool asks)
{
    using Walk = mx::StepWalk<SPR, GROUPS>;
    std::mt19937 rng(seed);
    const int raws = (kblocks + SPR - 1) / SPR;
    const uint32_t total_raws = (uint32_t)raws * tiles, total_steps = (uint32_t)kblocks * tiles;
    std::vector<Barrier> r_full(RS), r_empty(RS), a_full(as), a_empty(as);
    for (auto &b : r_full) b.count = 2;              // mantissas and exponents
    for (auto &b : r_empty) b.count = SPR * WARPS;
    for (auto &b : a_full) b.count = WARPS;
    std::vector<int64_t> slot(2 * RS, -1), astage(as * WARPS, -1);
    struct Load { uint32_t raw; int part; double weight; };
    std::vector<Load> loads;
    uint32_t filled = 0, multiplied = 0, committed = 0;
    std::uniform_real_distribution<double> u(0, 1);

    struct Warp {
        Walk walk;
        int index, state;                            // 0: is the slot empty of the stage before, 1: is it full, 2: read it, 3: wait for a place
        uint32_t ri;
        bool there, done;
    };
    std::vector<Warp> warps;
    for (int g = 0; g < GROUPS; ++g)
        for (int w = 0; w < WARPS; ++w) {
            Warp x{Walk{g, 0, 0, (uint32_t)g}, w, 0, 0, false, false};
            x.walk.settle(kblocks, raws, 1);
            x.ri = x.walk.raw();
            x.done = x.walk.tile >= tiles;
            warps.push_back(x);
        }
    bool wrong = false;
    auto holds = [&](uint32_t r) { return slot[2 * (r % RS)] == (int64_t)r && slot[2 * (r % RS) + 1] == (int64_t)r; };
    auto full = [&](uint32_t r) { return r_full[r % RS].test((r / RS) & 1u); };
    auto empty = [&](uint32_t r) { return r_empty[r % RS].test(((r / RS) & 1u) ^ 1u); };
    auto move = [&](Warp &w) -> bool {
        if (w.done) return false;
        if (w.state == 0) {
            if (!w.there && asks && Walk::ASKS_EMPTY && !empty(w.ri)) return false;
            w.state = 1;
            return true;
        }
        if (w.state == 1) {
            if (!w.there && !full(w.ri)) return false;
            if (!holds(w.ri)) wrong = true;
            w.state = 2;
            return true;
        }
        const uint32_t step = w.walk.step, a = step % as;
        if (w.state == 2) {
            if (!holds(w.ri)) wrong = true;          // still there at the end of the reads
            w.state = 3;
            return true;
        }
        if (!a_empty[a].test(((step / as) & 1u) ^ 1u)) return false;
        if (step >= (uint32_t)as && committed <= step - as) wrong = true;
        astage[a * WARPS + w.index] = step;
        const uint32_t was = w.ri;
        const bool last = w.walk.kb == kblocks - 1;
        w.walk.step += GROUPS;
        w.walk.kb += GROUPS;
        w.walk.settle(kblocks, raws, 1);
        w.ri = w.walk.raw();
        w.there = (!asks || !Walk::ASKS_EMPTY || empty(w.ri)) && full(w.ri);
        a_full[a].arrive();
        r_empty[was % RS].arrive(last ? 1 + raws * SPR - kblocks : 1);
        w.done = w.walk.tile >= tiles;
        w.state = 0;
        return true;
    };

    std::vector<double> pace(warps.size() + 3);
    for (auto &p : pace) p = u(rng) < 0.3 ? 0.02 : 1.0;
    long idle = 0;
    while (!wrong && idle < 20000) {
        bool moved = false;
        const size_t who = rng() % (pace.size() + 1);
        if (who < pace.size() && u(rng) > pace[who]) continue;
        if (who < warps.size()) {
            moved = move(warps[who]);
        } else if (who == warps.size()) {            // the loads' issuer
            const bool last_there = !asks || !Walk::waits_for_last(kblocks) || filled % raws != 0 || filled == 0 || full(filled - 1);
            if (filled < total_raws && last_there && r_empty[filled % RS].test(((filled / RS) & 1u) ^ 1u)) {
                for (int part = 0; part < 2; ++part) {
                    slot[2 * (filled % RS) + part] = -1;
                    loads.push_back({filled, part, u(rng) < 0.25 ? 0.005 : 0.5});
                }
                ++filled;
                moved = true;
            }
        } else if (who == warps.size() + 1) {        // the MMAs' issuer
            if (multiplied < total_steps && a_full[multiplied % as].test((multiplied / as) & 1u)) {
                for (int w = 0; w < WARPS; ++w) wrong |= astage[multiplied % as * WARPS + w] != (int64_t)multiplied;
                ++multiplied;
                moved = true;
            }
        } else if (who == warps.size() + 2) {
            if (committed < multiplied) {
                a_empty[committed % as].arrive();
                ++committed;
                moved = true;
            }
        } else if (!loads.empty()) {
            const size_t l = rng() % loads.size();
            if (u(rng) < loads[l].weight) {
                slot[2 * (loads[l].raw % RS) + loads[l].part] = loads[l].raw;
                r_full[loads[l].raw % RS].arrive();
                loads.erase(loads.begin() + l);
            }
            moved = true;
        }
        idle = moved ? 0 : idle + 1;
        if (committed == total_steps) break;
    }
    for (auto &w : warps) wrong |= !w.done;
    return !wrong && committed == total_steps;
}

}  // namespace

int main(int argc, char **argv)
{
    if (argc != 7) return 2;
    const int spr = atoi(argv[1]), as = atoi(argv[2]), kblocks = atoi(argv[3]), tiles = atoi(argv[4]), seeds = atoi(argv[5]);
    int bad = 0;
    for (int s = 0; s < seeds; ++s) bad += !(spr == 4 ? run<4>(as, kblocks, tiles, s, atoi(argv[6])) : run<2>(as, kblocks, tiles, s, atoi(argv[6])));
    printf("%d\n", bad);
    return 0;
}
