// Host build of the library's plan code (no launches): the split workspaces of a replayed handle,
// the tile shapes of grouped contractions.
#include "../paper_1911_00242_gb300/csrc/ccsd_api.cu"

namespace ccsdk {
void launch_zgemm(int, int, const GemmArgs&, int, cudaStream_t) {}
void launch_zgemm_grouped(int, int, const GemmArgs*, const long long*, int, long long, int, cudaStream_t) {}
}  // namespace ccsdk

namespace {

struct Dry {
    ccsd_ctx h;
    int rc;
    Dry(const ccsd_config* c, int use, int dtype = CCSD_C128) {
        init_ctx(&h, c);
        h.use = (HandleUse)use;
        Alloc al{&h};
        al.dry = true;
        const bool on_dev[9] = {true, true, true, true, true, true, true, true, true};
        rc = setup_handle(&h, al, nullptr, on_dev, dtype, false);
    }
};

}  // namespace

extern "C" long long probe_bytes(const ccsd_config* c, int use) {
    Dry d(c, use);
    return d.rc ? -1 : (long long)d.h.owned_bytes;
}

// Bit w: replayed in arithmetic w; bit 8: the handle stages ccsd_residual's arguments.
extern "C" int probe_replays(const ccsd_config* c, int use) {
    Dry d(c, use);
    if (d.rc) return -1;
    int m = d.h.stage ? 256 : 0;
    for (int w = 0; w < ZG_ARITH; ++w) m |= d.h.graphable[w] ? 1 << w : 0;
    return m;
}

// Pairs of steps whose partials or counters share memory although no path of the graph's edges
// orders them, in every arithmetic the handle replays; *shared counts the pairs that are ordered.
extern "C" int probe_conflicts(const ccsd_config* c, int use, int* shared) {
    Dry d(c, use);
    *shared = 0;
    if (d.rc) return -1;
    ccsd_ctx* h = &d.h;
    int bad = 0;
    for (int w = 0; w < ZG_ARITH; ++w) {
        if (!h->graphable[w]) continue;
        h->fp32 = w == ZG_FP32;
        h->oz_on = w == ZG_DF;
        struct Use { int step, kind; long long off, n; };
        std::vector<Use> us;
        std::map<int, std::vector<int>> next;
        HazardMap hz;
        for (int i = 0; i < (int)h->seq.size(); ++i) {
            const Step& st = h->seq[i];
            if (!step_active(h, st)) continue;
            for (int p : hz.add(i, step_access(h, st))) next[p].push_back(i);
            if (st.kind == 0) {
                const GemmPlan& g = h->gemms[st.idx];
                const GemmVar& v = g.var[w];
                if (v.nsplit < 2) continue;
                us.push_back({i, 0, v.work_off, (long long)v.nsplit * g.args.nbatch * g.args.M * g.args.N});
                us.push_back({i, 1, v.cnt_off, v.blocks});
            } else if (st.kind == 6 && h->tcs[st.idx].oz && h->tcs[st.idx].z.nsplit > 1) {
                const TcPlan& t = h->tcs[st.idx];
                us.push_back({i, 2, t.work_off, (long long)t.z.nsplit * t.z.nbatch * t.z.M * (t.z.Nr / 2)});
            }
        }
        for (const Use& a : us) {
            std::set<int> seen{a.step};
            std::vector<int> todo{a.step};
            while (!todo.empty()) {
                const int x = todo.back();
                todo.pop_back();
                for (int y : next[x]) if (seen.insert(y).second) todo.push_back(y);
            }
            for (const Use& b : us) {
                if (b.step <= a.step || b.kind != a.kind) continue;
                if (a.off + a.n <= b.off || b.off + b.n <= a.off) continue;
                if (seen.count(b.step)) ++*shared; else ++bad;
            }
            const long long cap = a.kind == 0 ? (long long)h->work_elems : a.kind == 1 ? (long long)h->cnt_need
                                                                                        : h->oz_work_elems;
            if (a.off < 0 || a.off + a.n > cap) ++bad;
        }
    }
    return bad;
}

// Shapes of contraction step number `gemm` (of those active in mixed or FP64 iterations) in rank
// order, for a group of this one member; the shape its own plan takes in *own.  -1: no such step.
extern "C" int probe_rank(const ccsd_config* c, int dtype, int fp32, int gemm, int* order, int* own) {
    Dry d(c, 1, dtype);
    if (d.rc) return -1;
    ccsd_ctx* h = &d.h;
    h->fp32 = fp32;
    for (size_t si = 0; si < h->seq.size(); ++si) {
        const Step& st = h->seq[si];
        if (st.kind != 0 || !step_active(h, st) || gemm-- > 0) continue;
        const GemmPlan& p = h->gemms[st.idx];
        if (p.args.nbatch == 0) return 0;
        const std::vector<int> r = rank_shapes({h}, si, fp32 ? ZG_FP32 : ZG_FP64);
        for (size_t i = 0; i < r.size(); ++i) order[i] = r[i];
        *own = p.var[fp32 ? ZG_FP32 : ZG_FP64].shape;
        return (int)r.size();
    }
    return -1;
}

// Elements of split partials in one launch of contraction step `gemm` (as in probe_rank) over n
// members like this one, in tile shape cfg; *least: what the FP32 sums alone need.  -1: no such step.
extern "C" long long probe_group_partials(const ccsd_config* c, int n, int fp32, int gemm, int cfg, long long* least) {
    Dry d(c, 1);
    if (d.rc) return -1;
    ccsd_ctx* h = &d.h;
    h->fp32 = fp32;
    for (size_t si = 0; si < h->seq.size(); ++si) {
        const Step& st = h->seq[si];
        if (st.kind != 0 || !step_active(h, st) || gemm-- > 0) continue;
        const GemmArgs& a = h->gemms[st.idx].args;
        const std::vector<ccsd_ctx*> m((size_t)n, h);
        long long out[2];
        for (int q = 0; q < 2; ++q) {
            out[q] = 0;
            for (int ns : group_splits(m, si, cfg, fp32 ? ZG_FP32 : ZG_FP64, q == 1))
                if (ns > 1) out[q] += (long long)ns * a.nbatch * a.M * a.N;
        }
        *least = out[1];
        return out[0];
    }
    return -1;
}

// Grouping key of a served solve in FP64 (fp32 = 0) or mixed iterations, its lane first; returns
// its length.
extern "C" int probe_key(const ccsd_config* c, int fp32, long long* out, int cap) {
    Dry d(c, 2);
    if (d.rc) return -1;
    d.h.fp32 = fp32;
    const std::vector<long long> k = server_key(&d.h);
    out[0] = lane_of(*c);
    for (size_t i = 0; i < k.size() && (int)i + 1 < cap; ++i) out[i + 1] = k[i];
    return (int)k.size() + 1;
}

// Launches of contraction step `gemm` (as in probe_rank) over two served members: how many, and
// bit 8 set if a launch mixes shapes of different K groups with its members' own.
extern "C" int probe_classes(const ccsd_config* c0, const ccsd_config* c1, int fp32, int gemm) {
    Dry a(c0, 2), b(c1, 2);
    if (a.rc || b.rc || a.h.seq.size() != b.h.seq.size()) return -1;
    a.h.fp32 = b.h.fp32 = fp32;
    const int arith = fp32 ? ZG_FP32 : ZG_FP64;
    for (size_t si = 0; si < a.h.seq.size(); ++si) {
        const Step& st = a.h.seq[si];
        if (st.kind != 0 || !step_active(&a.h, st) || gemm-- > 0) continue;
        const std::vector<KGroupClass> cl = kgroup_classes({&a.h, &b.h}, si, arith);
        int out = (int)cl.size();
        for (const KGroupClass& c : cl)
            for (const ccsd_ctx* h : c.m)
                if (kZgShapes[h->gemms[h->seq[si].idx].var[arith].shape].ks != kZgShapes[c.shape].ks) out |= 256;
        return out;
    }
    return -1;
}
