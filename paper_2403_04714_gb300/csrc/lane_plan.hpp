// lane_plan.hpp -- launch plan of the lane = instance bytecode with areas
// packed by process (lane_inst_packed in kernels.cu): the search over CTA
// sizes, apart from the CUDA queries, so that CPU tests run it too.
#pragma once
#include <algorithm>
#include <cstddef>
#include <cstdint>

#include "abi_device.h"

namespace rtl {

struct LanePlanInput {
    uint32_t n_proc = 0, groups = 0;    // a task per process and group of 32 instances
    int sms = 1;
    uint32_t share = 1;                 // the launch may hold 1 / share of the CTAs that fit on the GPU
    size_t smem_limit = 0;              // dynamic shared memory of a CTA
    uint32_t warps = 0;                 // configured warps per CTA, 0 = chosen here
    bool per_cycle = false;             // launches of one cycle: a warp for every task
};

struct LanePlan {
    int warps = 0, grid = 0, max_grid = 0;
    uint32_t banded = 0;                // see LaunchArgs
    uint64_t rounds = ~0ull;            // ~0: nothing fits
    size_t smem = 0;
};

// Persistent launches: the CTA size and grid with the fewest rounds of tasks,
// then the fewest warps.  slots(i): value slots of the i-th process, descending.  occ(threads,
// smem, &ctas): CTAs that fit on an SM, or an error code, which ends the search.
template <class Slots, class Occ>
int plan_lane(const LanePlanInput& in, Slots&& slots, Occ&& occ, LanePlan& best) {
    const uint32_t n_tasks = in.n_proc * in.groups, share = std::max(1u, in.share);
    // CTA 0 has the largest areas
    auto area_bytes = [&](int w, uint32_t band) {
        uint64_t words = 0;
        for (int i = 0; i < w && uint64_t(i) * band < n_tasks; i++) words += slots(size_t(i) * band / in.groups) * 32ull + kBlockWords;
        return size_t(words) * 8;
    };
    best = LanePlan();
    if (in.per_cycle && !in.warps) {
        // The CTAs of a launch of one cycle follow one another on an SM as they
        // finish, and a large one leaves it to its last warps.  So CTAs of four
        // warps (fewer where there are not four tasks for every SM), or of as many
        // as make fewer waves of resident warps.  Chosen as for persistent
        // launches, us a cycle: 2k-op netlist x 2,500 19 warps 32.2, 4 warps 18.1;
        // 20k-op x 2,500 32 warps 298, 4 warps 219; 200k-op x 2,500 4 warps 1,840,
        // 20 warps 1,647.
        const int base = int(std::min<uint64_t>(4, std::max<uint64_t>(1, (n_tasks + in.sms - 1) / in.sms)));
        for (int i = 0; i <= 32; i++) {
            const int w = i ? i : base;
            const uint32_t need = (n_tasks + w - 1) / w;
            const size_t smem = area_bytes(w, need);
            if (smem > in.smem_limit) continue;
            int ctas = 0;
            if (int rc = occ(w * 32, smem, &ctas)) return rc;
            const uint64_t warps = uint64_t(ctas) * w * in.sms;
            if (!warps || (n_tasks + warps - 1) / warps >= best.rounds) continue;
            best.rounds = (n_tasks + warps - 1) / warps;
            best.warps = w;
            best.smem = smem;
            best.max_grid = ctas * in.sms;
            best.grid = int(std::min(need, std::max(1u, uint32_t(best.max_grid) / share)));
        }
        if (best.warps) best.rounds = (n_tasks + uint64_t(best.grid) * best.warps - 1) / (uint64_t(best.grid) * best.warps);
        return 0;
    }
    int lo = in.warps ? int(std::min(32u, in.warps)) : 1, hi = in.warps ? lo : 32;
    // (a configured CTA size that does not fit is halved until it does)
    for (; best.rounds == ~0ull && lo >= 1; lo = lo / 2, hi = lo) {
        for (int w = lo; w <= hi; w++) {
            for (int k = in.warps ? 32 / w : 1; k >= 1; k--) {        // CTAs per SM
                const uint32_t need = (n_tasks + w - 1) / w;
                const uint32_t grid = std::max(1u, std::min(need, std::max(1u, uint32_t(k * in.sms) / share)));
                const uint64_t rounds = (n_tasks + uint64_t(grid) * w - 1) / (uint64_t(grid) * w);
                if (rounds >= best.rounds) continue;
                bool banded = false;
                size_t smem = area_bytes(w, in.per_cycle ? need : grid);
                if (smem > in.smem_limit && !in.per_cycle) banded = true, smem = area_bytes(w, uint32_t(rounds * grid));
                if (smem > in.smem_limit) continue;
                int ctas = 0;
                if (int rc = occ(w * 32, smem, &ctas)) return rc;
                // k CTAs per SM were wished for; the share is of those that fit
                if (ctas < 1 || grid > std::max(1u, uint32_t(ctas * in.sms) / share)) continue;
                best.rounds = rounds;
                best.banded = banded;
                best.warps = w;
                best.smem = smem;
                best.max_grid = ctas * in.sms;
                best.grid = int(grid);
            }
        }
    }
    return 0;
}

}  // namespace rtl
