// Hand-out order of a plan's tasks.
//
// CTAs take items in one fixed order, and a CTA whose next item waits for its inputs waits
// with it.  A stage of one frame keeps the SMs busy for only 5-17 us while an item takes
// 6-10 us from its ticket to its published result, so an order that runs layer by layer and
// frame by frame leaves CTAs waiting at every layer.  The order is therefore chosen: a few
// candidates (tiles of a group staggered against each other, the frames of a batch overlapped
// by different amounts) are run through a small model of the kernel, and the one that ends
// first is kept.  Every candidate is a topological order of the task dependencies, so an item
// only ever waits for items handed out before it, whatever the model gets wrong.
#include <algorithm>
#include <queue>

#include "planner.h"

namespace mafat {
namespace {

// What the model knows of a stage's items (microseconds).
struct StageCost {
    double mma, epi, load, period;
};

// Times of the tensor-core kernel, fitted to its per-item trace on GB300: an MMA of 128 x N x 16
// takes max(N / 2, 32 + N / 4) cycles (tensor core, or shared memory at 128 bytes a cycle) and
// about half as much again in an item; a 64-channel chunk takes 0.36 us to arrive; the epilogue
// handles a unit of one block x 32 columns in ~0.45 us on each of two warpgroups.
StageCost tc_cost(const MafatStageDev& s, double blocks) {
    StageCost c;
    const double steps = (double)s.n_chunks * s.n_bsteps * s.kst * blocks;
    c.mma = std::max(0.36 * s.n_chunks, 1.5 * steps * std::max(s.n_blk / 2.0, 32.0 + s.n_blk / 4.0) / 2070.0);
    const double units = blocks * std::max(1, s.n_blk / 32);
    c.epi = 0.3 + 0.45 * ((units + 1.0) / 2.0);
    c.load = s.in_mode == MAFAT_IN_GATHER ? 2.0 : 0.8;
    c.period = std::max(std::max(c.mma + 0.7, c.epi), 1.6);
    return c;
}

// fp32 kernel: an item's chunks one after another, at the pace of an item by itself, and ~5 us for the
// ticket, first loads and publication.  The order matters where SMs have little to do; with the
// pace of three items an SM (3 x F32Cost::full) 16 64x64 frames took 983 us instead of 934 and six 96x96
// frames cut after layer 11 742 instead of 733 (four 224x224 frames 858 instead of 870).
StageCost f32_stage_cost(const MafatStageDev& s) {
    StageCost c{};
    c.mma = 5.0 + s.f32_chunks * f32_cost(s.k, s.f32_ct).item;
    c.period = c.mma;
    return c;
}

struct Model {
    const PlanTables& t;
    const std::vector<TaskDep>& deps;
    std::vector<StageCost> cost;
    bool tc;
    int n_ctas;

    // Makespan of the tasks in `order` (others are taken as absent); start_of and end_of, where wanted,
    // get when a task's first item could start and when its last one was published.
    double run(const std::vector<int>& order, std::vector<double>* start_of = nullptr, std::vector<double>* end_of = nullptr) const {
        struct Cta {
            double mma_free = 0, mma_prev = 0, epi_free = 0, epi_prev = 0;
        };
        const int n = tc ? n_ctas : 3 * n_ctas;
        std::vector<Cta> cta(n);
        // CTAs by the time they take their next ticket: a binary heap whose top is replaced
        struct Slot {
            double at;
            int cta;
        };
        std::vector<Slot> take(n);
        for (int i = 0; i < n; ++i) take[i] = {0.0, i};
        auto replace_top = [&](double at) {
            Slot v = take[0];
            v.at = at;
            int i = 0;
            for (int c = 1; c < n; c = 2 * i + 1) {
                if (c + 1 < n && take[c + 1].at < take[c].at) ++c;
                if (take[c].at >= at) break;
                take[i] = take[c];
                i = c;
            }
            take[i] = v;
        };
        std::vector<double> done(t.tasks.size(), 0.0), group((size_t)t.cfg.batch * t.cfg.n_groups + 1, 0.0);
        double end = 0.0;
        for (int ti : order) {
            const TaskDep& d = deps[ti];
            const StageCost& c = cost[t.tasks[ti].stage];
            const bool look = t.stages[t.tasks[ti].stage].lookahead != 0;
            double ready = 0.0, fin = 0.0;
            if (d.prev_task >= 0) ready = std::max(ready, done[d.prev_task]);
            if (d.group_ctr >= 0) ready = std::max(ready, group[d.group_ctr]);
            for (int k = 0; k < t.tasks[ti].n_items; ++k) {
                Cta& q = cta[take[0].cta];
                const double dep = std::max(take[0].at + (tc ? 1.7 : 2.5), ready + 0.5);
                if (start_of && k == 0) (*start_of)[ti] = dep;
                double out, next;
                if (tc) {
                    const double load = std::max(dep, q.mma_prev) + c.load;  // two A stages
                    const double start = std::max(std::max(load, q.mma_free + 0.7), q.epi_prev);
                    next = look ? dep : std::max(dep, q.mma_free);
                    q.mma_prev = q.mma_free;
                    q.mma_free = start + c.mma;
                    q.epi_prev = q.epi_free;
                    q.epi_free = std::max(q.mma_free, q.epi_free) + c.epi;
                    out = q.epi_free + 0.9;
                } else {
                    out = next = dep + c.mma;
                }
                fin = std::max(fin, out);
                replace_top(next);
            }
            done[ti] = fin;
            if (end_of) (*end_of)[ti] = fin;
            if (d.bump_ctr >= 0) group[d.bump_ctr] = std::max(group[d.bump_ctr], fin);
            end = std::max(end, fin);
        }
        return end;
    }
};

// The model of a plan; items: each stage's items of one frame.
Model make_model(const PlanTables& t, const std::vector<TaskDep>& deps, std::vector<double>& items) {
    Model m{t, deps, {}, t.cfg.dtype == 0, t.cfg.n_ctas > 0 ? t.cfg.n_ctas : 152};
    std::vector<double> blocks(t.stages.size(), 0.0);
    items.assign(t.stages.size(), 0.0);
    for (const MafatTaskDev& k : t.tasks) {
        if (k.frame != 0) continue;
        blocks[k.stage] += (double)k.nby * k.nbx * t.stages[k.stage].n_nblk;
        items[k.stage] += k.n_items;
    }
    for (size_t s = 0; s < t.stages.size(); ++s)
        m.cost.push_back(m.tc ? tc_cost(t.stages[s], items[s] > 0 ? blocks[s] / items[s] : 1.0) : f32_stage_cost(t.stages[s]));
    return m;
}

std::vector<int> prefix_of(const PlanTables& t, const std::vector<int>& order, int frames) {
    std::vector<int> prefix;
    for (int i : order)
        if (t.tasks[i].frame < frames) prefix.push_back(i);
    return prefix;
}

// Topological order of the tasks with smallest key first.
std::vector<int> topological(const PlanTables& t, const std::vector<TaskDep>& deps, const std::vector<double>& key,
                             int frames) {
    const int n = (int)t.tasks.size();
    std::vector<int> wait(n, 0), group_left((size_t)t.cfg.batch * t.cfg.n_groups + 1, 0);
    std::vector<std::vector<int>> next(n), group_next(group_left.size());
    for (int i = 0; i < n; ++i) {
        if (t.tasks[i].frame >= frames) continue;
        if (deps[i].prev_task >= 0) ++wait[i], next[deps[i].prev_task].push_back(i);
        if (deps[i].group_ctr >= 0) ++wait[i], group_next[deps[i].group_ctr].push_back(i);
        if (deps[i].bump_ctr >= 0) ++group_left[deps[i].bump_ctr];
    }
    typedef std::pair<double, int> Entry;
    std::priority_queue<Entry, std::vector<Entry>, std::greater<Entry>> open;
    for (int i = 0; i < n; ++i)
        if (t.tasks[i].frame < frames && wait[i] == 0) open.push({key[i], i});
    std::vector<int> order;
    while (!open.empty()) {
        const int i = open.top().second;
        open.pop();
        order.push_back(i);
        for (int j : next[i])
            if (--wait[j] == 0) open.push({key[j], j});
        const int b = deps[i].bump_ctr;
        if (b >= 0 && --group_left[b] == 0)
            for (int j : group_next[b])
                if (--wait[j] == 0) open.push({key[j], j});
    }
    return order;
}

}  // namespace

int rings_enough(const PlanTables& t, const std::vector<TaskDep>& deps, const std::vector<int>& order,
                 const std::vector<int>& first, const std::vector<int>& last) {
    const int n = (int)t.tasks.size(), frames = std::min(t.cfg.batch, 4 * t.ring_sets);
    std::vector<double> items, start(n, 0.0), end(n, 0.0);
    make_model(t, deps, items).run(prefix_of(t, order, frames), &start, &end);
    std::vector<int> at(n);
    for (int k = 0; k < n; ++k) at[order[k]] = k;
    for (int rings = 2; rings < t.ring_sets; ++rings) {
        bool same = true;
        for (size_t q = (size_t)t.ring_slots * rings; q < first.size() && same; ++q) {
            const int i = first[q], p = last[q - (size_t)t.ring_slots * rings];
            same = at[p] < at[i] && (t.tasks[i].frame >= frames || end[p] + 0.5 <= start[i]);
        }
        if (same) return rings;
    }
    return t.ring_sets;
}

std::vector<int> hand_out_order(const PlanTables& t, const std::vector<TaskDep>& deps, const std::vector<int>& given) {
    const int G = t.cfg.n_groups, n = (int)t.tasks.size(), batch = t.cfg.batch;
    std::vector<double> items;
    const Model m = make_model(t, deps, items);
    const size_t n_st = t.stages.size();
    std::vector<int> tile(n, 0), tiles(n_st, 0);  // tile index of a task among its stage's of the frame
    int64_t frame_items = 0;
    for (int i = 0; i < n; ++i) {
        if (t.tasks[i].frame != 0) continue;
        frame_items += t.tasks[i].n_items;
        ++tiles[t.tasks[i].stage];
    }
    {
        std::vector<int> seen((size_t)batch * n_st, 0);
        for (int i = 0; i < n; ++i) tile[i] = seen[(size_t)t.tasks[i].frame * n_st + t.tasks[i].stage]++;
    }
    std::vector<double> work(n_st, 0.0);  // microseconds of all SMs for a stage of one frame
    for (size_t s = 0; s < n_st; ++s) work[s] = items[s] * m.cost[s].period / (m.tc ? m.n_ctas : 3 * m.n_ctas);
    std::vector<double> gw(G, 0.0), off(n_st, 0.0);
    double total = 0.0;
    for (int g = 0; g < G; ++g) {
        for (int s = t.stage_first[g]; s <= t.stage_last[g]; ++s) {
            off[s] = gw[g];
            gw[g] += work[s];
        }
        total += gw[g];
    }
    // A model run costs ~0.05 us per item, so the candidates are first compared over a few frames; but
    // what a ring's reuse costs shows only where there are more frames than rings (16 608x608 frames
    // through four rings: all stages in lockstep promise 23 % less over three frames and take 2149 us
    // instead of 678), so those that promise enough are compared again over twice as many.
    const int few = (int)std::max<int64_t>(1, std::min<int64_t>(batch, std::max<int64_t>(2, 8000 / std::max<int64_t>(1, frame_items))));
    const int many = std::max(few, std::min(batch, 2 * t.ring_sets));
    auto keyed = [&](double rate, double stagger, double lead, double stretch) {
        // virtual time of a task: its frame's start, a lead before every later group (in frames'
        // work), the stages of later groups stretched, tiles of a group staggered
        std::vector<double> key(n);
        for (int i = 0; i < n; ++i) {
            const MafatTaskDev& k = t.tasks[i];
            int g = 0;
            while (g + 1 < G && k.stage > t.stage_last[g]) ++g;
            double v = (double)k.frame * rate * total;
            for (int h = 0; h < g; ++h) v += gw[h] * (h == 0 ? 1.0 : stretch) + lead * total;
            v += off[k.stage] * (g == 0 ? 1.0 : stretch) + stagger * gw[g] * tile[i] / std::max(1, tiles[k.stage]);
            key[i] = v + 1e-9 * (double)i;
        }
        return key;
    };
    // the model is good to a few per cent: another order has to promise more than that (eight
    // 1216x1216 frames: promised 2.7 % less, measured 0.8 % more)
    const double margin = 0.96, limit_few = margin * m.run(prefix_of(t, given, few));
    double best = few == many ? limit_few : 0.0;
    std::vector<double> best_key;
    auto offer = [&](double rate, double stagger, double lead, double stretch) {
        std::vector<double> key = keyed(rate, stagger, lead, stretch);
        double us = m.run(topological(t, deps, key, few));
        if (us >= limit_few) return;
        if (few < many) {
            if (best == 0.0) best = margin * m.run(prefix_of(t, given, many));
            us = m.run(topological(t, deps, key, many));
        }
        if (us < best) {
            best = us;
            best_key.swap(key);
        }
    };
    offer(0.0, 0.0, 0.0, 1.0);  // all frames stage by stage
    offer(0.5, 0.0, 0.0, 1.0);
    if (G > 1) {
        for (double stretch : {2.0, 3.0})
            for (double lead : {0.0, 0.15}) offer(0.5, 0.0, lead, stretch);
        offer(1.0, 0.0, 0.0, 2.0);
        offer(1.0, 0.0, 0.15, 2.0);
        offer(1.0, 0.0, 0.15, 4.0);
    }
    return best_key.empty() ? given : topological(t, deps, best_key, batch);
}

}  // namespace mafat
