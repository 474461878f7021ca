// Dataflow schedule of the fused runs of small steps (k_small_steps): host
// side, made once per plan.
//
// A run is a tree of gate-sized contractions listed in path order; its depth
// is 15-25 levels where it has 180-730 steps (the 12- and 30-qubit brickwork
// blocks).  Steps are put on the lowest level above every earlier step of the
// run that they read, overwrite, or whose operands they overwrite (address
// ranges of the arenas), so the steps of a level are independent of each other
// and one CTA barrier per level orders the run.  Every output element of a
// level becomes one entry (step, element, operand offsets of its first term).
#include <algorithm>
#include <map>

#include "ptn_internal.h"

namespace ptn {

namespace {

struct Range {
    int32_t arena;
    int64_t off, size;
};
bool meets(const Range& a, const Range& b) {
    return a.arena == b.arena && a.off < b.off + b.size && b.off < a.off + a.size;
}
Range out_range(const StepDesc& s) { return {s.out_arena, s.out_off, s.out_size}; }
bool reads(const StepDesc& s, const Range& r) {
    for (const OperandDesc& d : s.op)
        if (d.mode == OP_BUF && meets({d.arena, d.arena_off, d.inst_size}, r)) return true;
    return false;
}

// Offsets of every combination of the given bit strides, at most 2^14 - 1.
std::vector<uint32_t> combos(const int64_t* stride, int n) {
    std::vector<uint32_t> v((size_t)1 << n, 0);
    for (size_t i = 1; i < v.size(); i++) {
        const int p = __builtin_ctzll(i);
        v[i] = v[i & (i - 1)] + (uint32_t)stride[p];
    }
    return v;
}

void add_part(const StepDesc* st, int n, SmallRuns& sr) {
    SmallPart part;
    part.step0 = (int32_t)sr.steps.size();
    part.n_steps = n;
    part.cls = st[0].out_cls;
    std::vector<int> level(n, 0);
    int n_lvl = 0;
    for (int k = 0; k < n; k++) {
        const Range out = out_range(st[k]);
        for (int j = 0; j < k; j++) {
            if (level[j] < level[k]) continue;
            const Range oj = out_range(st[j]);
            if (reads(st[k], oj) || meets(out, oj) || reads(st[j], out)) level[k] = level[j] + 1;
        }
        n_lvl = std::max(n_lvl, level[k] + 1);
    }
    for (int k = 0; k < n; k++) {
        SmallStep s{};
        bool dense = true;
        for (int o = 0; o < 2; o++) {
            const OperandDesc& d = st[k].op[o];
            SmallOp& p = s.op[o];
            p.size = (int32_t)d.inst_size;
            p.col = -1;
            if (d.mode == OP_LEAF) {
                p.src = -1;
                p.base = d.leaf_base;
                p.col = d.leaf_col;
            } else {
                p.src = d.arena;
                p.base = d.arena_off;
                p.inst = d.cls;
                p.cache = d.cls == CLS_TRAJ ? d.cache : 0;
            }
            p.slice0 = (int32_t)sr.slices.size();
            p.n_slice = d.n_slice;
            for (int q = 0; q < d.n_slice; q++) sr.slices.push_back({d.slice_qubit[q], (int32_t)d.slice_stride[q]});
            for (int q = 0; q < st[k].n_sum; q++) dense = dense && st[k].sum_stride[o][q] == (int64_t)1 << q;
        }
        s.out_off = st[k].out_off;
        s.out_size = (int32_t)st[k].out_size;
        s.out_arena = st[k].out_arena;
        const uint32_t nk = 1u << st[k].n_sum;
        s.loop = nk | (st[k].op[0].conj ? kSmallConjA : 0u) | (st[k].op[1].conj ? kSmallConjB : 0u);
        if (dense) {
            s.loop |= kSmallDense;
        } else {
            s.ktab = (int32_t)sr.ktab.size();
            const auto a = combos(st[k].sum_stride[0], st[k].n_sum), b = combos(st[k].sum_stride[1], st[k].n_sum);
            for (uint32_t i = 0; i < nk; i++) sr.ktab.push_back(a[i] | (b[i] << 16));
        }
        sr.steps.push_back(s);
    }
    // levels in order; within a level steps of equal length of the summed loop
    // stand together, so the threads of a warp mostly run the same loop
    std::vector<int> order(n);
    for (int k = 0; k < n; k++) order[k] = k;
    std::stable_sort(order.begin(), order.end(), [&](int x, int y) {
        return level[x] != level[y] ? level[x] < level[y] : st[x].n_sum > st[y].n_sum;
    });
    part.lvl0 = (int32_t)sr.lvl.size();
    part.n_lvl = n_lvl;
    int cur = -1;
    for (int k : order) {
        while (cur < level[k]) {
            sr.lvl.push_back((int32_t)sr.ent.size());
            cur++;
        }
        const auto a = combos(st[k].out_stride[0], st[k].n_out), b = combos(st[k].out_stride[1], st[k].n_out);
        for (size_t o = 0; o < a.size(); o++)
            sr.ent.push_back({a[o] | (b[o] << 16), (uint16_t)k, (uint16_t)o});
    }
    sr.lvl.push_back((int32_t)sr.ent.size());
    sr.parts.push_back(part);
}

}  // namespace

int small_run_len(const std::vector<StepDesc>& steps, size_t k, int fuse_max) {
    size_t en = k + 1;
    while (en < steps.size() && en - k < (size_t)fuse_max && steps[en].fuse_prev) en++;
    return (int)(en - k);
}

void build_small_runs(const std::vector<StepDesc>& steps, int fuse_max, SmallRuns& sr) {
    sr = SmallRuns();
    for (size_t k = 0; k < steps.size(); k++) {
        const int len = small_run_len(steps, k, fuse_max);
        if (len < 2) continue;
        sr.run_at[(int32_t)k] = {(int32_t)sr.parts.size(), 0};
        for (int done = 0; done < len; done += kSmallPartSteps)
            add_part(&steps[k + done], std::min(kSmallPartSteps, len - done), sr);
        sr.run_at[(int32_t)k].second = (int32_t)sr.parts.size();
        k += len - 1;
    }
}

}  // namespace ptn
