// plan_internal.hpp -- the plan object behind the opaque bmmc_plan handle:
// the validated matrix (Sec. 3), its one or two tiled passes (Sec. 5.1, 5.2)
// and each pass's launch tables (Sec. 4.1-4.3).
#pragma once
#include <stdint.h>

#include <mutex>

#include "bmmc.h"
#include "f2.hpp"
#include "pass_desc.h"
#include "plan.hpp"

struct bmmc_plan_s {
    int n = 0;
    int e_log = 0;
    uint64_t c = 0;
    bmmc::f2::Mat a;
    bmmc::PlanOptions opt;
    int npass = 0;
    bmmc::f2::Mat t[2];
    uint64_t tc[2] = {0, 0};
    bmmc::PassDesc desc[2];
    bmmc::PassInfo info[2];
    // A two-pass plan whose permutation runs as one launch: `whole` holds the
    // tables of (A, c) over generic tiles (see create_impl in capi.cpp).  The
    // two factors' tables then serve the queries only and are derived by the
    // first one that asks (factors_derived, under derive_mu).
    bool fused = false;
    bmmc::PassDesc whole;
    bmmc::PassInfo whole_info;
    std::mutex derive_mu;
    bool factors_derived = false;
    // Workspace owned by the plan for bmmc_execute (plans of two launches only).
    std::mutex ws_mu;
    void *ws = nullptr;
    int ws_device = -1;

    uint64_t bytes() const { return (1ull << n) << e_log; }
    // Kernel launches of one execution, and the tables of launch i.
    int launches() const { return fused ? 1 : npass; }
    const bmmc::PassDesc &launch_desc(int i) const { return fused ? whole : desc[i]; }
};
