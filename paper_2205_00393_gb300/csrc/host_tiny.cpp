// Host side of the tiny-network kernel (kernels_tiny.cu): which networks it runs,
// and the tables of their plan.
#include "host.hpp"

namespace tnc_host {

// Complex multiply-accumulates of a slice, its share of the invariants included, up
// to which a CTA takes it: a CTA alone (one slice) takes 20 us up to 2^14, 32 at
// 2^16.3, 44-74 at 2^17.3 to 2^18 where the levels' launches spread the work over
// the chip and take 60-73 us throughout. From 64 slices on these take 95-110 us and
// a CTA each still 50-73 at 2^18 (1000 slices: 56 us instead of 624 at 2^14, 245
// instead of 593 at 2^16.9), and a call of several variants repeats the launches for
// each. Shared memory ends the range at about 2^18.5.
constexpr double kTinyMaxCmacs = 3 << 16, kTinyMaxCmacsMany = 3 << 17;
constexpr int64_t kTinyMany = 64;
constexpr int64_t kTinyMaxPartials = 1 << 20;  // FP64 partial results of a call: 16 MiB

namespace {

struct Tables {
    std::vector<uint32_t> w;
    int here() const { return (int)w.size(); }
    // offsets of every value of the bits with strides str, the first bit lowest
    int offsets(const std::vector<int64_t>& str) {
        const int o = here();
        for (uint32_t x = 0; x < 1u << str.size(); ++x) {
            int64_t off = 0;
            for (size_t j = 0; j < str.size(); ++j)
                if ((x >> j) & 1) off += str[j];
            w.push_back((uint32_t)off);
        }
        return o;
    }
};

// Tables of the network's plan; false if it is not tiny in this mode.
bool build_tiny(tnc_net* net, int mode, Tables& T, tnc::TinyParams& p, double& cmacs) {
    const Plan& P = net->plan;
    const int nl = net->n_leaves, nt = net->tree->n_tensors();
    if (P.nodes.empty() || P.nodes.back().kind != K_ROOT_F64 || P.nodes.back().chunks != 1 || nt > 4096) return false;
    cmacs = 0;
    for (const NodePlan& np : P.nodes) {
        if (shape_choice(net, mode, np.mb, np.nb, np.kb, np.is_root)) return false;
        if (np.mb + np.nb > 14 || np.kb > 12 || np.mb + np.kb > 15 || np.nb + np.kb > 15) return false;
        cmacs += std::ldexp(1.0, np.mb + np.nb + np.kb);
    }
    if (cmacs > kTinyMaxCmacsMany || net->total_leaf_elems > 16384) return false;
    // places of the intermediates behind the leaves: the outputs of a level are live
    // together, its inputs die after it (invariant ones used per slice stay)
    std::vector<int64_t> at(nt, 0);
    std::map<int64_t, int64_t> used;  // element offset -> length
    used[0] = (net->total_leaf_elems + 1) / 2 * 2;
    int64_t top = used[0];
    auto alloc = [&](int64_t len) {
        len = (len + 1) / 2 * 2;
        int64_t end = 0;
        for (auto& kv : used) {
            if (kv.first - end >= len) break;
            end = kv.first + kv.second;
        }
        used[end] = len;
        top = std::max(top, end + len);
        return end;
    };
    std::vector<std::vector<const NodePlan*>> levels;
    int inv = 0;
    for (bool per : {false, true}) {
        for (const Group& g : level_groups(net, mode, per)) {
            levels.emplace_back();
            for (auto* list : {&g.fp32, &g.tc})
                for (int v : *list) {
                    const NodePlan& np = P.nodes[v - nl];
                    at[v] = alloc(1ll << (np.mb + np.nb));
                    levels.back().push_back(&np);
                }
            for (const NodePlan* np : levels.back())
                for (int c : {np->A, np->B})
                    if (c >= nl && (P.per_slice[c] != 0) == per) used.erase(at[c]);
        }
        if (!per) inv = (int)levels.size();
    }
    if (top > 0xFFFF) return false;
    for (int v = 0; v < nl; ++v) at[v] = net->leaf_off[v];
    // tables
    auto op_words = [&](const NodePlan& np, uint32_t item0) {
        std::vector<uint32_t> o(tnc::kTinyOpWords);
        o[0] = np.A;
        o[1] = np.B;
        o[2] = np.is_root ? 0 : (uint32_t)at[np.v];
        o[3] = np.mb | np.nb << 8 | np.kb << 16;
        o[4] = T.offsets(np.am);
        o[5] = T.offsets(np.bn);
        o[6] = T.offsets(np.ak);
        const int b = T.offsets(np.bk);
        for (int k = 0; k < 1 << np.kb; ++k) T.w[o[6] + k] |= T.w[b + k] << 16;
        T.w.resize(b);
        o[7] = item0;
        return o;
    };
    std::vector<uint32_t> ops, lv;
    std::vector<std::vector<uint16_t>> maps;
    for (const auto& level : levels) {
        maps.emplace_back();
        for (const NodePlan* np : level) {
            const uint32_t id = (uint32_t)(ops.size() / tnc::kTinyOpWords), items = 1u << (np->mb + np->nb);
            const auto o = op_words(*np, (uint32_t)maps.back().size() * 4);
            ops.insert(ops.end(), o.begin(), o.end());
            maps.back().insert(maps.back().end(), (items + 3) / 4, (uint16_t)id);
        }
    }
    const auto root = op_words(P.nodes.back(), 0);
    p.o_root = T.here();
    T.w.insert(T.w.end(), root.begin(), root.end());
    p.o_ops = T.here();
    T.w.insert(T.w.end(), ops.begin(), ops.end());
    for (const auto& m : maps) {
        lv.push_back((uint32_t)m.size() * 4);
        lv.push_back(T.here());
        for (size_t i = 0; i < m.size(); i += 2) T.w.push_back(m[i] | (i + 1 < m.size() ? (uint32_t)m[i + 1] << 16 : 0));
    }
    p.o_levels = T.here();
    T.w.insert(T.w.end(), lv.begin(), lv.end());
    p.inv_levels = inv;
    p.levels = (int)levels.size();
    p.o_static = T.here();
    for (int v = 0; v < nt; ++v) T.w.push_back((uint32_t)at[v]);
    p.o_base = T.here();
    for (int v = 0; v < nt; ++v) T.w.push_back((uint32_t)at[v]);
    std::vector<uint32_t> sliced, var;
    const int sbits = (int)net->S_sorted.size();
    for (int v = 0; v < nl; ++v) {
        const int o = T.here();
        int n = 0;
        for (const auto& [bit, stride] : P.sl[v])
            if (bit < sbits) {  // (the bits above name the variant)
                T.w.push_back(bit);
                T.w.push_back((uint32_t)stride);
                ++n;
            }
        if (n)
            for (uint32_t x : {(uint32_t)v, (uint32_t)o, (uint32_t)n}) sliced.push_back(x);
        if (!net->var_off.empty() && net->var_off[v] >= 0) {
            if (net->var_off[v] + (net->leaf_elems[v] << net->variant_bits) > 0x7fffffffll) return false;
            for (int64_t e = 0; e < net->leaf_elems[v]; ++e)
                for (uint32_t x : {(uint32_t)(net->var_off[v] + e), (uint32_t)(net->leaf_off[v] + e), (uint32_t)net->leaf_elems[v]})
                    var.push_back(x);
        }
    }
    p.o_sliced = T.here();
    p.n_sliced = (int)sliced.size() / 3;
    T.w.insert(T.w.end(), sliced.begin(), sliced.end());
    p.o_var = T.here();
    p.n_var = (int)var.size() / 3;
    T.w.insert(T.w.end(), var.begin(), var.end());
    T.w.resize((T.w.size() + 3) / 4 * 4);
    p.words = (int)T.w.size();
    p.data_elems = (int)((top + 1) / 2 * 2);
    p.leaf_elems = (int)net->total_leaf_elems;
    return p.n_sliced <= tnc::kTinyThreads && tnc::tiny_smem_bytes(p.data_elems, p.words) <= tnc::kTinySmem;
}

}  // namespace

tnc_status tiny_contract(tnc_net* net, int mode, int64_t first, int64_t stride, int64_t per, int64_t groups, double2* out,
                         cudaStream_t s, bool* done) {
    *done = false;
    const Plan& P = net->plan;
    const int64_t fit = kTinyMaxPartials >> std::min(P.obits, 40);
    if (net->persist_test_stall || per < 1 || groups < 1 || per > fit || groups > fit / per) return TNC_OK;
    const std::string key = plan_key(net, mode, 0);
    auto it = net->tiny_plans.find(key);
    // a graph that a call is captured into keeps the addresses of its tables and
    // buffer: neither is made during a capture (a call alike comes before it; else
    // the other executors see to the call), and neither is freed while the network lives
    const bool capture = capturing(s);
    if (it == net->tiny_plans.end()) {
        if (capture) return TNC_OK;
        auto tp = std::make_unique<TinyPlan>();
        Tables T;
        if (build_tiny(net, mode, T, tp->prm, tp->cmacs)) {
            CUDA_TRY(cudaMalloc(&tp->mem, T.w.size() * 4));
            CUDA_TRY(cudaMemcpyAsync(tp->mem, T.w.data(), T.w.size() * 4, cudaMemcpyHostToDevice, s));
            CUDA_TRY(cudaStreamSynchronize(s));  // the host words may go
            tp->prm.tables = static_cast<const uint32_t*>(tp->mem);
        }
        if (net->tiny_plans.size() >= 8) {
            for (auto& [k, plan] : net->tiny_plans)
                if (plan->captured) net->tiny_kept.push_back(std::move(plan));
            net->tiny_plans.clear();
        }
        it = net->tiny_plans.emplace(key, std::move(tp)).first;
    }
    TinyPlan& tp = *it->second;
    if (!tp.mem || tp.cmacs > (per * groups >= kTinyMany ? kTinyMaxCmacsMany : kTinyMaxCmacs)) return TNC_OK;
    const size_t given = net->ws_user ? net->ws_user_bytes : 0;
    if (tp.want != per || tp.given != given) {
        tp.want = per;
        tp.given = given;
        tp.nb = call_batch(net, per, mode, batch_budget(net, mode));
    }
    if (tp.nb < 1) return TNC_OK;
    // Partial results: in the caller's workspace, in rounds of as many as it holds (calls
    // on several streams then share no memory that their workspaces do not), or in a
    // buffer of the network's own.
    const size_t need = (size_t)(per * groups) << P.obits;
    const int64_t room = net->ws_user ? (int64_t)(given / sizeof(double2) >> P.obits) : per * groups;
    if (room < 1) return TNC_OK;
    if (!net->ws_user && need > net->d_tiny_cap) {
        if (capture) return TNC_OK;
        double2* m = nullptr;
        const size_t size = std::max(need, std::min<size_t>(2 * net->d_tiny_cap, kTinyMaxPartials));  // (so few are kept)
        if (cudaMalloc(&m, size * sizeof(double2)) != cudaSuccess) {  // the workspace's executors need none
            (void)cudaGetLastError();
            return TNC_OK;
        }
        if (net->d_tiny_captured) net->d_tiny_kept.push_back(net->d_tiny);
        else if (net->d_tiny) CUDA_TRY(cudaFree(net->d_tiny));
        net->d_tiny = m;
        net->d_tiny_cap = size;
        net->d_tiny_captured = false;
    }
    if (capture) {
        tp.captured = true;
        net->d_tiny_captured |= !net->ws_user;
    }
    tnc::TinyParams p = tp.prm;
    p.leaves = net->d_leaves;
    p.variants = net->d_var;
    p.stride = stride;
    p.sbits = (int)net->S_sorted.size();
    p.obits = P.obits;
    p.partials = net->ws_user ? static_cast<double2*>(net->ws_user) : net->d_tiny;
    p.err = net->d_err;
    tnc::PermParams pp{};
    pp.obits = P.obits;
    for (int j = 0; j < P.obits; ++j) pp.ostride[j] = P.out_stride[j];
    double cm = 0;
    if (net->timing)
        for (const NodePlan& np : P.nodes)
            cm += std::ldexp(1.0, np.mb + np.nb + np.kb) * (np.per_slice ? (double)(per * groups) : 1.0);
    CUDA_TRY(timed_begin(net, -1, K_PERSIST, (int)std::min<int64_t>(per, 0x7fffffff), s, cm));
    net->launches -= 1;
    const int64_t dg = std::max<int64_t>(1, std::min(groups, room / per)), dj = std::min(per, room);
    for (int64_t g = 0; g < groups; g += dg)
        for (int64_t j = 0; j < per; j += dj) {
            p.first = first + g * stride + j;
            p.per = std::min(dj, per - j);
            p.groups = std::min(dg, groups - g);
            p.out = out + (g << P.obits);
            p.clear = j == 0;
            CUDA_TRY(tnc::launch_tiny(p, pp, s));
            net->launches += 2;  // the slices and their sum
        }
    CUDA_TRY(timed_end(net, s));
    net->last_batch = tp.nb;
    net->last_arena_bytes[0] = net->last_arena_bytes[1] = 0;  // no layout of tensors, no task dependencies
    net->last_persist_deps = false;
    net->inv_key.clear();  // the workspace may hold partial results
    *done = true;
    return TNC_OK;
}

}  // namespace tnc_host
