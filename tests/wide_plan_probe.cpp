// Which plans go to the wide pass, and how many records their passes hold
// (test support only): plans made by the library's own planner with the
// parameters its entry points use.
#include <algorithm>
#include <vector>

#include "../paper_1608_00263_gb300/csrc/qs_internal.h"

using namespace qs;

// One state's plan.  narrow: as the gradient's forward evolution.  out: the
// register bits the plan was made for, its wide form's (0: none), passes of
// the lowered plan, most records of one of them, most ops of a planned pass.
extern "C" int probe_state(int n, int dtype, int mode, int tile, int narrow, const qs_gate *g, size_t ng, int *out)
{
    qs_opts o{};
    o.mode = mode;
    o.tile_log2 = tile;
    PlanParams pp = default_plan_params(n, (qs_dtype)dtype, &o);
    if (narrow) pp = narrow_plan_params(pp);
    Plan plan;
    if (build_plan(pp, g, ng, &plan) != QS_OK) return -1;
    WidePlan w;
    lower_wide(plan, &w);
    out[0] = plan.r;
    out[1] = plan.wide;
    out[2] = (int)w.passes.size();
    out[3] = out[4] = 0;
    for (const WidePass &p : w.passes) out[3] = std::max(out[3], (int)p.nops);
    for (const DevPass &p : plan.passes) {
        const DevPhase *h = plan.phases.data() + p.phase_begin;
        out[4] = std::max(out[4], h[p.nphases - 1].op_end - h[0].op_begin);
    }
    return 0;
}

// Instances of one batch, planned with five register bits of the (re, im)
// form or for the wide pass, and lowered together.  Returns the number of
// lowered passes (0: the batch runs the plans as they are); *regs: their
// register bits.
extern "C" int probe_batch(int count, const int *n, const qs_gate *g, const uint64_t *offsets, int wide, int *regs)
{
    std::vector<Plan> plans(count);
    std::vector<int> idx(count);
    for (int i = 0; i < count; ++i) {
        idx[i] = i;
        const size_t ng = (size_t)(offsets[i + 1] - offsets[i]);
        if (ng && build_plan(batch_plan_params(n[i], 0, wide != 0), g + offsets[i], ng, &plans[i]) != QS_OK) return -1;
    }
    WidePlan w;
    lower_instances(plans, std::vector<FoldArgs>(count), idx, &w);
    *regs = 0;
    for (const WidePass &p : w.passes) *regs |= p.r;
    return (int)w.passes.size();
}

// A plan that says it was made for the wide pass and holds more ops than one
// (the mistake is planted here): what lowering it returns.
extern "C" int probe_oversize(int n, const qs_gate *g, size_t ng)
{
    Plan plan;
    if (build_plan(batch_plan_params(n, 0, false), g, ng, &plan) != QS_OK) return -1;
    plan.wide = kWideRegBits;
    WidePlan w;
    const qs_status st = lower_wide(plan, &w);
    if (lower_instances({plan}, {FoldArgs{}}, {0}, &w) != st) return -1;
    return (int)st;
}

// The reverse sweep's plan: most records of a pass, or -1.
extern "C" int probe_sweep(int n, const qs_gate *g, size_t ng)
{
    WidePlan w;
    std::vector<int> slots;
    if (build_adjoint(n, g, ng, &w, &slots) != QS_OK) return -1;
    int most = 0;
    for (const WidePass &p : w.passes) most = std::max(most, (int)p.nops);
    return most;
}

// Register bits of the wide form a list is planned for on a state that its
// first pass reads (0: the (re, im) form), and the plan's passes.
extern "C" int probe_held(int n, int dtype, int mode, int tile, const qs_gate *g, size_t ng, int *passes)
{
    qs_opts o{};
    o.mode = mode;
    o.tile_log2 = tile;
    Plan plan;
    if (build_plan(held_plan_params(default_plan_params(n, (qs_dtype)dtype, &o), g, ng), g, ng, &plan) != QS_OK) return -1;
    *passes = (int)plan.passes.size();
    return plan.wide;
}
