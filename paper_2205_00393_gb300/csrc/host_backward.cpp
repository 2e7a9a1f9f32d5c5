// Host side of the adjoint pass (tnc_contract_backward) and the gate-parameter
// chain rule (tnc_param_grads).
#include "host.hpp"

namespace tnc_host {

// ------------------------------------------------------------ adjoint pass

// First-fit allocator over a workspace (also used as a dry run to size it).
struct FitAlloc {
    std::map<int64_t, int64_t> used;
    int64_t top = 0;
    int64_t alloc(int64_t len) {
        len = align_up(std::max<int64_t>(len, 1));
        int64_t prev_end = 0;
        for (auto& kv : used) {
            if (kv.first - prev_end >= len) break;
            prev_end = kv.first + kv.second;
        }
        used[prev_end] = len;
        top = std::max(top, prev_end + len);
        return prev_end;
    }
    void release(int64_t off) { used.erase(off); }
};

struct Backward {
    tnc_net* net;
    int mode;
    int64_t nb;
    bool exec;
    char* ws = nullptr;
    cudaStream_t s = nullptr;
    FitAlloc A;
    Arena fwd;                                     // offsets of forward intermediates and planes
    std::vector<char> needs;                       // per tensor: environment required
    std::vector<std::vector<int>> env_layout;      // per tensor
    std::vector<int64_t> env_off;                  // per tensor (current env buffer)
    std::vector<int64_t> inv_acc;                  // per invariant tensor: FP64 env accumulator
    int64_t leaf_grad = -1;                        // FP64 gradients of all leaves, packed
    // per-level checkpointing of per-slice intermediates
    int keep_every = 1;                            // keep tensors at levels divisible by this
    std::vector<char> keep, present;               // per tensor
    int64_t recomputed = 0;                        // nodes recomputed in the reverse walk
};

int64_t layout_stride(const std::vector<int>& layout, int mode) {
    const int L = (int)layout.size();
    for (int p = 0; p < L; ++p)
        if (layout[p] == mode) return 1ll << (L - 1 - p);
    return -1;
}

// The contraction that gives the environment of child c of node np (into
// env_off[c]) from the node's environment and the sibling's value.
tnc::GemmParams env_gemm(const Backward& bw, const NodePlan& np, int c, int64_t b) {
    const tnc_net* net = bw.net;
    const Plan& P = net->plan;
    const bool is_a = (c == np.A);
    tnc::GemmParams g{};
    const std::vector<int>& ev = bw.env_layout[np.v];
    tnc::Operand E{};
    E.ptr = reinterpret_cast<const float2*>(bw.ws + bw.env_off[np.v]);
    E.batch_stride = P.per_slice[np.v] || np.is_root ? ((int64_t)1 << ev.size()) : 0;
    tnc::Operand S = operand(net, bw.fwd, bw.ws, is_a ? np.B : np.A, b);
    if (is_a) {
        // E_A[m, k] = sum_n E_v[m, n] B[k, n]
        g.A = E;
        g.B = S;
        g.mb = np.mb;
        g.nb = np.kb;
        g.kb = np.nb;
        for (int j = 0; j < np.mb; ++j) g.am[j] = layout_stride(ev, np.mm[np.mb - 1 - j]);
        for (int j = 0; j < np.nb; ++j) {
            g.ak[j] = layout_stride(ev, np.nm[np.nb - 1 - j]);
            g.bk[j] = np.bn[j];
        }
        for (int j = 0; j < np.kb; ++j) g.bn[j] = np.bk[j];
    } else {
        // E_B[k, n] = sum_m A[m, k] E_v[m, n]
        g.A = S;
        g.B = E;
        g.mb = np.kb;
        g.nb = np.nb;
        g.kb = np.mb;
        for (int j = 0; j < np.kb; ++j) g.am[j] = np.ak[j];
        for (int j = 0; j < np.mb; ++j) {
            g.ak[j] = np.am[j];
            g.bk[j] = layout_stride(ev, np.mm[np.mb - 1 - j]);
        }
        for (int j = 0; j < np.nb; ++j) g.bn[j] = layout_stride(ev, np.nm[np.nb - 1 - j]);
    }
    g.C = reinterpret_cast<float2*>(bw.ws + bw.env_off[c]);
    g.c_batch_stride = 1ll << bw.env_layout[c].size();
    return g;
}

// Layout of child c's environment: its modes in np's order.
std::vector<int> env_child_layout(const NodePlan& np, int c) {
    std::vector<int> lay = c == np.A ? np.mm : np.km;
    const std::vector<int>& rest = c == np.A ? np.km : np.nm;
    lay.insert(lay.end(), rest.begin(), rest.end());
    return lay;
}

// Parameters that fold leaf c's environments into its FP64 gradient.
tnc::LeafEnvParams leaf_env_params(const Backward& bw, int c) {
    const tnc_net* net = bw.net;
    tnc::LeafEnvParams lp{};
    lp.env = reinterpret_cast<const float2*>(bw.ws + bw.env_off[c]);
    lp.env_batch_stride = 1ll << bw.env_layout[c].size();
    int q = 0;
    for (int64_t e : net->leaf_idx[c])
        for (int bit = 0; bit < net->logd[e]; ++bit, ++q) {
            const int mode = net->mode_base[e] + bit;
            lp.sl_bit[q] = net->plan.slice_bit_of_mode[mode];
            lp.env_stride[q] = lp.sl_bit[q] >= 0 ? 0 : layout_stride(bw.env_layout[c], mode);
        }
    lp.L = q;
    lp.grad = reinterpret_cast<double2*>(bw.ws + bw.leaf_grad) + net->leaf_off[c];
    return lp;
}

// Environment of child `c` of node np from the node's environment.
tnc_status env_child(Backward& bw, const NodePlan& np, int c, int64_t b, int64_t slice0) {
    tnc_net* net = bw.net;
    const bool is_a = (c == np.A);
    bw.env_layout[c] = env_child_layout(np, c);
    const int64_t elems = 1ll << bw.env_layout[c].size();
    bw.env_off[c] = bw.A.alloc(b * elems * 8);  // environments of every child, batch b
    // GEMM dims of this environment: E_A is (mb, kb) over nb; E_B is (kb, nb) over mb
    const int gmb = is_a ? np.mb : np.kb, gnb = is_a ? np.kb : np.nb, gkb = is_a ? np.nb : np.mb;
    const int env_choice = shape_choice(net, bw.mode, gmb, gnb, gkb, false);
    const bool tc = env_choice != 0;
    int64_t pa = -1, pb = -1;
    if (tc) {  // split-precision planes (allocated in the sizing pass too)
        pa = bw.A.alloc(tc_bytes_a(bw.net, bw.mode, gmb, gnb, gkb, b));
        pb = bw.A.alloc(tc_bytes_b(bw.net, bw.mode, gmb, gnb, gkb, b));
    }
    if (!bw.exec) {
        if (tc) {
            bw.A.release(pa);
            bw.A.release(pb);
        }
        return TNC_OK;
    }
    tnc::GemmParams g = env_gemm(bw, np, c, b);
    g.slice0 = slice0;
    if (tc) {
        // split precision with FP32 accumulation, as in the forward
        tnc_status st =
            launch_tc_contraction(net, g, (int)b, bw.mode, bw.ws + pa, bw.ws + pb, np.v, bw.s, env_choice, b);
        bw.A.release(pa);
        bw.A.release(pb);
        return st;
    }
    CUDA_TRY(timed_begin(net, np.v, K_GEMM_F32, (int)b, bw.s, std::ldexp(1.0, g.mb + g.nb + g.kb) * b));
    CUDA_TRY(tnc::launch_gemm_f32(g, (int)b, bw.s));
    CUDA_TRY(timed_end(net, bw.s));
    return TNC_OK;
}

// Fold the environment of child c (batch b) into its destination: leaves
// accumulate into their FP64 gradient; invariant tensors reached from a
// per-slice parent accumulate (over slices) into their FP64 environment;
// anything else keeps its environment for its own children.
tnc_status env_fold(Backward& bw, int c, int64_t b, int64_t slice0, bool from_per_slice) {
    tnc_net* net = bw.net;
    const Plan& P = net->plan;
    const int64_t elems = 1ll << bw.env_layout[c].size();
    if (c < net->n_leaves) {
        if (bw.exec) {
            tnc::LeafEnvParams lp = leaf_env_params(bw, c);
            lp.slice0 = slice0;
            CUDA_TRY(timed_begin(net, c, -2, (int)b, bw.s, 0.0));
            CUDA_TRY(tnc::launch_leaf_env_accum(lp, (int)b, bw.s));
            CUDA_TRY(timed_end(net, bw.s));
        }
        bw.A.release(bw.env_off[c]);
    } else if (from_per_slice && !P.per_slice[c]) {
        if (bw.exec) {
            CUDA_TRY(tnc::launch_accum_batch_f64(reinterpret_cast<const float2*>(bw.ws + bw.env_off[c]), elems,
                                                 (int)b, elems,
                                                 reinterpret_cast<double2*>(bw.ws + bw.inv_acc[c]), bw.s));
            net->launches += 1;
        }
        bw.A.release(bw.env_off[c]);
    }
    return TNC_OK;
}

tnc_status fwd_node(Backward& bw, const NodePlan& np, int64_t b, int64_t slice0);

// Make the value of per-slice tensor v available, recomputing it (and, as
// needed, its own per-slice inputs) from the nearest kept tensors.
tnc_status materialize(Backward& bw, int v, int64_t b, int64_t slice0) {
    tnc_net* net = bw.net;
    if (v < net->n_leaves || !net->plan.per_slice[v] || bw.present[v]) return TNC_OK;
    const NodePlan& np = net->plan.nodes[v - net->n_leaves];
    tnc_status st;
    for (int c : {np.A, np.B})
        if ((st = materialize(bw, c, b, slice0)) != TNC_OK) return st;
    if ((st = fwd_node(bw, np, b, slice0)) != TNC_OK) return st;
    bw.present[v] = 1;
    bw.recomputed += 1;
    for (int c : {np.A, np.B})
        if (c >= net->n_leaves && net->plan.per_slice[c] && !bw.keep[c]) {
            bw.A.release(bw.fwd.off[c]);
            bw.present[c] = 0;
        }
    return TNC_OK;
}

// Reverse walk over the nodes of one class (per-slice or invariant).
tnc_status reverse_walk(Backward& bw, bool per_slice, int64_t b, int64_t slice0) {
    tnc_net* net = bw.net;
    const Plan& P = net->plan;
    tnc_status st;
    for (int i = (int)P.nodes.size() - 1; i >= 0; --i) {
        const NodePlan& np = P.nodes[i];
        const bool node_per = np.per_slice;
        if (node_per != per_slice) continue;
        if (!bw.needs[np.v]) continue;
        if (per_slice) {  // siblings feed the environment contractions
            if (bw.needs[np.A] && (st = materialize(bw, np.B, b, slice0)) != TNC_OK) return st;
            if (bw.needs[np.B] && (st = materialize(bw, np.A, b, slice0)) != TNC_OK) return st;
        }
        for (int c : {np.A, np.B}) {
            if (!bw.needs[c]) continue;
            if ((st = env_child(bw, np, c, b, slice0)) != TNC_OK) return st;
            if ((st = env_fold(bw, c, b, slice0, per_slice)) != TNC_OK) return st;
        }
        bw.A.release(bw.env_off[np.v]);
        if (per_slice)  // the children's values are not needed again
            for (int c : {np.A, np.B})
                if (c >= net->n_leaves && P.per_slice[c] && bw.present[c]) {
                    bw.A.release(bw.fwd.off[c]);
                    bw.present[c] = 0;
                }
    }
    return TNC_OK;
}

// One forward node kept for the reverse walk (all per-slice intermediates live).
tnc_status fwd_node(Backward& bw, const NodePlan& np, int64_t b, int64_t slice0) {
    tnc_net* net = bw.net;
    const Plan& P = net->plan;
    const bool per = np.per_slice;
    bw.fwd.off[np.v] = bw.A.alloc((per ? b : 1) * tensor_bytes(P, np.v));
    const bool tc = shape_choice(net, bw.mode, np.mb, np.nb, np.kb, np.is_root) != 0;
    const size_t i = np.v - net->n_leaves;
    if (tc) {
        bw.fwd.planes_a[i] = bw.A.alloc(tc_bytes_a(net, bw.mode, np.mb, np.nb, np.kb, per ? b : 1));
        bw.fwd.planes_b[i] = bw.A.alloc(tc_bytes_b(net, bw.mode, np.mb, np.nb, np.kb, per ? b : 1));
    }
    if (bw.exec) {
        tnc::GemmParams g = gemm_params(net, bw.fwd, bw.ws, np, b);
        g.C = reinterpret_cast<float2*>(bw.ws + bw.fwd.off[np.v]);
        g.c_batch_stride = per ? tensor_bytes(P, np.v) / 8 : 0;
        g.slice0 = slice0;
        tnc_status st = launch_node(net, bw.fwd, bw.ws, np, g, per ? (int)b : 1, bw.mode, bw.s);
        if (st != TNC_OK) return st;
    }
    if (tc) {
        bw.A.release(bw.fwd.planes_a[i]);
        bw.A.release(bw.fwd.planes_b[i]);
    }
    return TNC_OK;
}

// The whole backward computation; with exec == false only the workspace is sized.
tnc_status backward_run(Backward& bw, int64_t lo, int64_t hi, const double* grad_out) {
    tnc_net* net = bw.net;
    const Plan& P = net->plan;
    const tnc::Tree& T = *net->tree;
    tnc_status st;
    bw.fwd.off.assign(T.n_tensors(), -1);
    bw.fwd.planes_a.assign(P.nodes.size(), -1);
    bw.fwd.planes_b.assign(P.nodes.size(), -1);
    bw.env_layout.assign(T.n_tensors(), {});
    bw.env_off.assign(T.n_tensors(), -1);
    bw.inv_acc.assign(T.n_tensors(), -1);
    // checkpoint levels: per-slice dependency depth; the root's inputs are kept
    bw.keep.assign(T.n_tensors(), 0);
    bw.present.assign(T.n_tensors(), 0);
    {
        std::vector<int> level(T.n_tensors(), 0);
        for (const NodePlan& np : P.nodes) {
            if (!np.per_slice || np.is_root) continue;
            int l = 0;
            for (int c : {np.A, np.B})
                if (c >= net->n_leaves && P.per_slice[c]) l = std::max(l, level[c]);
            level[np.v] = l + 1;
            bw.keep[np.v] = (level[np.v] % std::max(1, bw.keep_every)) == 0;
        }
        if (!P.nodes.empty())
            for (int c : {P.nodes.back().A, P.nodes.back().B}) bw.keep[c] = 1;
    }
    bw.leaf_grad = bw.A.alloc(net->total_leaf_elems * 16);
    if (bw.exec) CUDA_TRY(cudaMemsetAsync(bw.ws + bw.leaf_grad, 0, net->total_leaf_elems * 16, bw.s));
    // invariant forward, kept for the whole call
    for (const NodePlan& np : P.nodes)
        if (!np.per_slice && !np.is_root)
            if ((st = fwd_node(bw, np, 1, 0)) != TNC_OK) return st;
    // FP64 environment accumulators of invariant tensors whose parent is per-slice
    for (int v = net->n_leaves; v < T.n_tensors(); ++v) {
        if (P.per_slice[v] || v == T.root || !bw.needs[v]) continue;
        const int par = T.parent[v];
        if (par < 0 || !(P.per_slice[par] || par == T.root)) continue;
        const int64_t bytes = (int64_t)16 << P.layout[v].size();
        bw.inv_acc[v] = bw.A.alloc(bytes);
        if (bw.exec) CUDA_TRY(cudaMemsetAsync(bw.ws + bw.inv_acc[v], 0, bytes, bw.s));
    }
    const int root = T.root;
    for (int64_t s0 = lo; s0 < hi; s0 += bw.nb) {
        const int64_t b = std::min<int64_t>(bw.nb, hi - s0);
        FitAlloc saved = bw.A;
        // per-slice forward, root excluded; tensors off the checkpoint levels are
        // dropped once consumed and recomputed in the reverse walk
        std::fill(bw.present.begin(), bw.present.end(), 0);
        for (const NodePlan& np : P.nodes) {
            if (!np.per_slice || np.is_root) continue;
            if ((st = fwd_node(bw, np, b, s0)) != TNC_OK) return st;
            bw.present[np.v] = 1;
            for (int c : {np.A, np.B})
                if (c >= net->n_leaves && P.per_slice[c] && !bw.keep[c] && bw.present[c]) {
                    bw.A.release(bw.fwd.off[c]);
                    bw.present[c] = 0;
                }
        }
        // seed: the root's environment is grad_out (in the root's layout)
        bw.env_layout[root] = P.layout[root];
        const int64_t relems = 1ll << P.layout[root].size();
        bw.env_off[root] = bw.A.alloc(b * relems * 8);
        if (bw.exec) {
            tnc::SeedParams sp{};
            sp.grad = reinterpret_cast<const double2*>(grad_out);
            sp.obits = P.obits;
            for (int j = 0; j < P.obits; ++j) sp.ostride[j] = P.out_stride[j];
            sp.E = reinterpret_cast<float2*>(bw.ws + bw.env_off[root]);
            sp.batch_stride = relems;
            CUDA_TRY(tnc::launch_env_seed(sp, (int)b, bw.s));
            net->launches += 1;
        }
        if (root < net->n_leaves) {
            if ((st = env_fold(bw, root, b, s0, true)) != TNC_OK) return st;
        } else if ((st = reverse_walk(bw, true, b, s0)) != TNC_OK) {
            return st;
        }
        bw.A.used = saved.used;  // the batch's buffers are dead; keep the peak
    }
    // invariant reverse walk from the accumulated environments (batch 1)
    for (int v = net->n_leaves; v < T.n_tensors(); ++v) {
        if (bw.inv_acc[v] < 0) continue;
        // the accumulator holds the environment in the layout its per-slice
        // parent produced (env_layout[v], set by env_child; same size as v)
        const int64_t elems = (int64_t)1 << P.layout[v].size();
        if (bw.env_layout[v].empty() && !P.layout[v].empty()) bw.env_layout[v] = P.layout[v];
        bw.env_off[v] = bw.A.alloc(elems * 8);
        if (bw.exec)
            CUDA_TRY(tnc::launch_f64_to_f32(reinterpret_cast<const double2*>(bw.ws + bw.inv_acc[v]), elems,
                                            reinterpret_cast<float2*>(bw.ws + bw.env_off[v]), bw.s));
    }
    if ((st = reverse_walk(bw, false, 1, 0)) != TNC_OK) return st;
    return TNC_OK;
}


// ------------------------------------------------------ adjoint pass by levels
//
// The same computation in few launches: the contractions of a tree level, forward
// and reverse, run as one grouped launch (those of the tensor cores, of 256 tiles
// or more, or of a long K on their own), and so do the folds of the
// environments that a level produces. Node by node, a 16-qubit gradient took
// 659 launches, planned anew (and sized several times) on every call. Every
// contraction and every FP64 sum is the same as node by node.
// This way is taken when every intermediate is kept (no checkpoints) and its
// workspace fits the budget at the batch that the node-by-node pass would take.

struct LevelBuilder {
    Backward& bw;
    BackwardPlan& bp;

    // an FP32 or tensor-core contraction (node: its record in the timings)
    void add(std::vector<std::pair<tnc::GemmParams, int>>& grouped, std::vector<BackwardOp>& singles, const tnc::GemmParams& g,
             int node, bool per_slice) {
        const tnc_net* net = bw.net;
        const int choice = shape_choice(net, bw.mode, g.mb, g.nb, g.kb, false);
        if (!choice && tnc::gemm_f32_tiles(g.mb, g.nb) < 256 && !tnc::gemm_f32_long(g.kb)) {
            grouped.emplace_back(g, node);
            return;
        }
        BackwardOp op;
        op.type = BackwardOp::NODE;
        op.per_slice = per_slice;
        op.g = g;
        op.node = node;
        op.choice = choice;
        op.cmacs = std::ldexp(1.0, g.mb + g.nb + g.kb);
        singles.push_back(op);
    }
    // the level's launches, the grouped one first. Called when every output of the
    // level has its place: a contraction's planes may then take any free bytes,
    // the next one's planes the same ones.
    void emit(std::vector<BackwardOp>& ops, const std::vector<std::pair<tnc::GemmParams, int>>& grouped,
              std::vector<BackwardOp>& singles, bool per_slice, int64_t b) {
        const tnc_net* net = bw.net;
        for (BackwardOp& op : singles) {
            if (!op.choice) continue;
            op.pa = bw.A.alloc(tc_bytes_a(net, bw.mode, op.g.mb, op.g.nb, op.g.kb, b));
            op.pb = bw.A.alloc(tc_bytes_b(net, bw.mode, op.g.mb, op.g.nb, op.g.kb, b));
            bw.A.release(op.pa);
            bw.A.release(op.pb);
        }
        if (!grouped.empty()) {
            BackwardOp op;
            op.per_slice = per_slice;
            op.first = (int)bp.gemm.size();
            op.off_first = (int64_t)bp.map.size();
            op.n = (int)grouped.size();
            for (const auto& [g, node] : grouped) {
                bp.gemm.push_back(g);
                tnc::gemm_f32_group_map(bp.map, (int)bp.gemm.size() - 1 - op.first, g.mb, g.nb);
                op.cmacs += std::ldexp(1.0, g.mb + g.nb + g.kb);
            }
            op.blocks = (int64_t)bp.map.size() - op.off_first;
            ops.push_back(op);
        }
        for (BackwardOp& op : singles) ops.push_back(std::move(op));
        singles.clear();
    }
    // one launch over the entries [first, table size) of a fold table, elems elements each
    void emit_fold(std::vector<BackwardOp>& ops, BackwardOp::Type type, int first, const std::vector<int64_t>& elems) {
        if (elems.empty()) return;
        BackwardOp op;
        op.type = type;
        op.first = first;
        op.n = (int)elems.size();
        op.off_first = (int64_t)bp.off.size();
        for (int64_t n : elems) {
            bp.off.push_back(op.blocks);
            op.blocks += (n + 255) / 256;
        }
        bp.off.push_back(op.blocks);
        ops.push_back(op);
    }
    // forward contractions of one class, every output kept
    void forward(std::vector<BackwardOp>& ops, bool per_slice, int64_t b) {
        tnc_net* net = bw.net;
        const Plan& P = net->plan;
        for (const Group& lg : level_groups(net, bw.mode, per_slice)) {
            std::vector<std::pair<tnc::GemmParams, int>> grouped;
            std::vector<BackwardOp> singles;
            for (auto* list : {&lg.fp32, &lg.tc})
                for (int v : *list) {
                    const NodePlan& np = P.nodes[v - net->n_leaves];
                    bw.fwd.off[v] = bw.A.alloc((per_slice ? b : 1) * tensor_bytes(P, v));
                    tnc::GemmParams g = gemm_params(net, bw.fwd, bw.ws, np, b);
                    g.C = reinterpret_cast<float2*>(bw.ws + bw.fwd.off[v]);
                    g.c_batch_stride = per_slice ? tensor_bytes(P, v) / 8 : 0;
                    add(grouped, singles, g, v, per_slice);
                }
            emit(ops, grouped, singles, per_slice, per_slice ? b : 1);
        }
    }
    // reverse walk of one class, a level of nodes at a time (level 0: the root, or
    // the invariant tensors whose environments were summed)
    void reverse(std::vector<BackwardOp>& ops, bool per_slice, int64_t b) {
        tnc_net* net = bw.net;
        const Plan& P = net->plan;
        const int nl = net->n_leaves;
        std::vector<int> level(net->tree->n_tensors(), 0);
        std::vector<std::vector<int>> by_level;
        for (int i = (int)P.nodes.size() - 1; i >= 0; --i) {
            const NodePlan& np = P.nodes[i];
            if (np.per_slice != per_slice || !bw.needs[np.v]) continue;
            const int l = level[np.v];
            if ((int)by_level.size() <= l) by_level.resize(l + 1);
            by_level[l].push_back(i);
            for (int c : {np.A, np.B})
                if (c >= nl && (P.per_slice[c] != 0) == per_slice) level[c] = l + 1;
        }
        for (const auto& nodes : by_level) {
            std::vector<std::pair<tnc::GemmParams, int>> grouped;
            std::vector<BackwardOp> singles;
            std::vector<int64_t> leaf_elems, inv_elems;
            const int leaf0 = (int)bp.leaf.size(), inv0 = (int)bp.inv.size();
            std::vector<int> folded;
            for (int i : nodes) {
                const NodePlan& np = P.nodes[i];
                for (int c : {np.A, np.B}) {
                    if (!bw.needs[c]) continue;
                    bw.env_layout[c] = env_child_layout(np, c);
                    const int64_t elems = 1ll << bw.env_layout[c].size();
                    bw.env_off[c] = bw.A.alloc(b * elems * 8);
                    add(grouped, singles, env_gemm(bw, np, c, b), np.v, per_slice);
                    if (c < nl) {
                        bp.leaf.push_back(leaf_env_params(bw, c));
                        leaf_elems.push_back(net->leaf_elems[c]);
                        folded.push_back(c);
                    } else if (per_slice && !P.per_slice[c]) {
                        tnc::InvEnvParams ip{};
                        ip.env = reinterpret_cast<float2*>(bw.ws + bw.env_off[c]);
                        ip.acc = reinterpret_cast<double2*>(bw.ws + bw.inv_acc[c]);
                        ip.n = elems;
                        bp.inv.push_back(ip);
                        inv_elems.push_back(elems);
                        folded.push_back(c);
                    }
                }
            }
            emit(ops, grouped, singles, per_slice, b);
            emit_fold(ops, BackwardOp::LEAF, leaf0, leaf_elems);
            emit_fold(ops, BackwardOp::INV_SUM, inv0, inv_elems);
            for (int c : folded) bw.A.release(bw.env_off[c]);
            for (int i : nodes) {
                const NodePlan& np = P.nodes[i];
                bw.A.release(bw.env_off[np.v]);
                if (per_slice)  // the children's values are not needed again
                    for (int c : {np.A, np.B})
                        if (c >= nl && P.per_slice[c]) bw.A.release(bw.fwd.off[c]);
            }
        }
    }
};

// The whole pass for batches of nb slices and a last one of `tail` (0: none); bw.ws
// may be null to size the workspace.
void build_backward_plan(Backward& bw, int64_t nb, int64_t tail, BackwardPlan& bp) {
    tnc_net* net = bw.net;
    const Plan& P = net->plan;
    const tnc::Tree& T = *net->tree;
    struct NoFuse {  // no fused stem groups in the forward levels
        tnc_net* net;
        bool was;
        explicit NoFuse(tnc_net* n) : net(n), was(n->in_many) { n->in_many = true; }
        ~NoFuse() { net->in_many = was; }
    } no_fuse(net);
    LevelBuilder lb{bw, bp};
    bw.fwd.off.assign(T.n_tensors(), -1);
    bw.env_layout.assign(T.n_tensors(), {});
    bw.env_off.assign(T.n_tensors(), -1);
    bw.inv_acc.assign(T.n_tensors(), -1);
    bw.leaf_grad = bw.A.alloc(net->total_leaf_elems * 16);
    bp.zero_bytes = bw.leaf_grad + align_up(std::max<int64_t>(net->total_leaf_elems * 16, 1));
    for (int v = net->n_leaves; v < T.n_tensors(); ++v) {
        if (P.per_slice[v] || v == T.root || !bw.needs[v]) continue;
        const int par = T.parent[v];
        if (par < 0 || !(P.per_slice[par] || par == T.root)) continue;
        bw.inv_acc[v] = bw.A.alloc((int64_t)16 << P.layout[v].size());  // right behind the one before
        bp.zero_bytes = bw.inv_acc[v] + align_up((int64_t)16 << P.layout[v].size());
    }
    lb.forward(bp.inv_fwd, false, 1);
    const FitAlloc saved = bw.A;
    for (int q = 0; q < (tail ? 2 : 1); ++q) {
        const int64_t b = q ? tail : nb;
        auto& ops = bp.slices[q];
        lb.forward(ops, true, b);
        bw.env_layout[T.root] = P.layout[T.root];
        const int64_t relems = 1ll << P.layout[T.root].size();
        bw.env_off[T.root] = bw.A.alloc(b * relems * 8);
        BackwardOp seed;
        seed.type = BackwardOp::SEED;
        seed.seed.obits = P.obits;
        for (int j = 0; j < P.obits; ++j) seed.seed.ostride[j] = P.out_stride[j];
        seed.seed.E = reinterpret_cast<float2*>(bw.ws + bw.env_off[T.root]);
        seed.seed.batch_stride = relems;
        ops.push_back(seed);
        lb.reverse(ops, true, b);
        bw.A.used = saved.used;  // the batch's buffers are dead; keep the peak
    }
    const int inv0 = (int)bp.inv.size();
    std::vector<int64_t> inv_elems;
    for (int v = net->n_leaves; v < T.n_tensors(); ++v) {
        if (bw.inv_acc[v] < 0) continue;
        if (bw.env_layout[v].empty() && !P.layout[v].empty()) bw.env_layout[v] = P.layout[v];
        const int64_t elems = (int64_t)1 << P.layout[v].size();
        bw.env_off[v] = bw.A.alloc(elems * 8);
        tnc::InvEnvParams ip{};
        ip.env = reinterpret_cast<float2*>(bw.ws + bw.env_off[v]);
        ip.acc = reinterpret_cast<double2*>(bw.ws + bw.inv_acc[v]);
        ip.n = elems;
        bp.inv.push_back(ip);
        inv_elems.push_back(elems);
    }
    lb.emit_fold(bp.inv_rev, BackwardOp::INV_READ, inv0, inv_elems);
    lb.reverse(bp.inv_rev, false, 1);
    bp.top = bw.A.top;
}

tnc_status upload_backward_plan(BackwardPlan& bp, cudaStream_t s) {
    size_t off = 0;
    auto slot = [&](size_t bytes) {
        const size_t o = off;
        off += (bytes + 255) / 256 * 256;
        return o;
    };
    const size_t o_gemm = slot(bp.gemm.size() * sizeof(bp.gemm[0])), o_leaf = slot(bp.leaf.size() * sizeof(bp.leaf[0])),
                 o_inv = slot(bp.inv.size() * sizeof(bp.inv[0])), o_off = slot(bp.off.size() * sizeof(bp.off[0])),
                 o_map = slot(bp.map.size() * sizeof(bp.map[0]));
    CUDA_TRY(cudaMalloc(&bp.mem, std::max<size_t>(off, 256)));
    char* base = static_cast<char*>(bp.mem);
    auto up = [&](size_t o, const void* src, size_t bytes) -> cudaError_t {
        return bytes ? cudaMemcpyAsync(base + o, src, bytes, cudaMemcpyHostToDevice, s) : cudaSuccess;
    };
    CUDA_TRY(up(o_gemm, bp.gemm.data(), bp.gemm.size() * sizeof(bp.gemm[0])));
    CUDA_TRY(up(o_leaf, bp.leaf.data(), bp.leaf.size() * sizeof(bp.leaf[0])));
    CUDA_TRY(up(o_inv, bp.inv.data(), bp.inv.size() * sizeof(bp.inv[0])));
    CUDA_TRY(up(o_off, bp.off.data(), bp.off.size() * sizeof(bp.off[0])));
    CUDA_TRY(up(o_map, bp.map.data(), bp.map.size() * sizeof(bp.map[0])));
    CUDA_TRY(cudaStreamSynchronize(s));  // the host vectors may go
    bp.d_gemm = reinterpret_cast<const tnc::GemmParams*>(base + o_gemm);
    bp.d_leaf = reinterpret_cast<const tnc::LeafEnvParams*>(base + o_leaf);
    bp.d_inv = reinterpret_cast<const tnc::InvEnvParams*>(base + o_inv);
    bp.d_off = reinterpret_cast<const int64_t*>(base + o_off);
    bp.d_map = reinterpret_cast<const int2*>(base + o_map);
    bp.gemm.clear();
    bp.leaf.clear();
    bp.inv.clear();
    bp.map.clear();
    return TNC_OK;
}

tnc_status run_backward_ops(tnc_net* net, const BackwardPlan& bp, const std::vector<BackwardOp>& ops, int64_t batch,
                            int64_t slice0, int mode, const double* grad_out, char* ws, cudaStream_t s) {
    tnc_status st;
    for (const BackwardOp& op : ops) {
        const int b = op.per_slice ? (int)batch : 1;
        switch (op.type) {
            case BackwardOp::GROUP:
                CUDA_TRY(timed_begin(net, -1, K_GEMM_F32, b, s, op.cmacs * b));
                CUDA_TRY(tnc::launch_gemm_f32_group(bp.d_gemm + op.first, bp.d_map + op.off_first, op.blocks, slice0, b, s));
                CUDA_TRY(timed_end(net, s));
                break;
            case BackwardOp::NODE: {
                tnc::GemmParams g = op.g;
                g.slice0 = slice0;
                if (op.choice) {
                    if ((st = launch_tc_contraction(net, g, b, mode, ws + op.pa, ws + op.pb, op.node, s, op.choice, b)) != TNC_OK)
                        return st;
                } else {
                    CUDA_TRY(timed_begin(net, op.node, K_GEMM_F32, b, s, op.cmacs * b));
                    CUDA_TRY(tnc::launch_gemm_f32(g, b, s));
                    CUDA_TRY(timed_end(net, s));
                }
                break;
            }
            case BackwardOp::LEAF:
                CUDA_TRY(timed_begin(net, -1, -2, (int)batch, s, 0.0));
                CUDA_TRY(tnc::launch_leaf_env_accum_group(bp.d_leaf + op.first, bp.d_off + op.off_first, op.n, op.blocks, slice0,
                                                          (int)batch, s));
                CUDA_TRY(timed_end(net, s));
                break;
            case BackwardOp::INV_SUM:
            case BackwardOp::INV_READ:
                net->launches += 1;
                CUDA_TRY(tnc::launch_inv_env_group(bp.d_inv + op.first, bp.d_off + op.off_first, op.n, op.blocks,
                                                   op.type == BackwardOp::INV_SUM ? (int)batch : 0, s));
                break;
            case BackwardOp::SEED: {
                tnc::SeedParams sp = op.seed;
                sp.grad = reinterpret_cast<const double2*>(grad_out);
                net->launches += 1;
                CUDA_TRY(tnc::launch_env_seed(sp, (int)batch, s));
                break;
            }
        }
    }
    return TNC_OK;
}

}  // namespace tnc_host

extern "C" {

tnc_status tnc_contract_backward(tnc_net_t net, int64_t lo, int64_t hi, int mode, const double* grad_out_c128,
                                 float* grad_leaves_c64, const unsigned char* leaf_mask, size_t budget_bytes,
                                 void* stream) {
    if (!net) return fail(TNC_E_INVALID, "NULL network");
    if (!grad_out_c128 || !grad_leaves_c64) return fail(TNC_E_INVALID, "NULL gradient buffer");
    if (mode < TNC_FP32 || mode > TNC_SPLIT_FP16X2) return fail(TNC_E_INVALID, "unknown mode");
    tnc_status st = ensure_plan(net);
    if (st != TNC_OK) return st;
    if (net->variant_bits || net->n_variants)
        return fail(TNC_E_STATE, "the adjoint pass does not take leaf variants (tnc_set_leaf_variants)");
    const int64_t n_slices = 1ll << std::min<size_t>(net->S_sorted.size(), 62);
    if (lo < 0 || hi < lo || hi > n_slices) return fail(TNC_E_INVALID, "slice range outside [0, 2^|S|]");
    cudaStream_t s = (cudaStream_t)stream;
    if ((st = ensure_leaves(net, s)) != TNC_OK) return st;
    const tnc::Tree& T = *net->tree;
    Backward bw;
    bw.net = net;
    bw.mode = mode;
    bw.s = s;
    bw.needs.assign(T.n_tensors(), 0);
    for (int v = 0; v < net->n_leaves; ++v) bw.needs[v] = leaf_mask ? (leaf_mask[v] != 0) : 1;
    for (size_t i = 0; i < T.children.size(); ++i) {
        const int v = net->n_leaves + (int)i;
        bw.needs[v] = bw.needs[T.children[i].first] || bw.needs[T.children[i].second];
    }
    if (budget_bytes == 0) budget_bytes = (size_t)32 << 30;
    if (hi == lo) {
        CUDA_TRY(cudaMemsetAsync(grad_leaves_c64, 0, net->total_leaf_elems * 8, s));
        return TNC_OK;
    }
    // checkpoint spacing, then the largest slice batch, that fit the budget (dry runs;
    // kept for calls alike)
    const std::string mask(bw.needs.begin(), bw.needs.begin() + net->n_leaves);
    const std::string key = plan_key(net, mode, 0) + ":" + std::to_string(budget_bytes) + ":" + std::to_string(hi - lo) + ":" +
                            std::to_string(net->backward_keep_every) + ":" + mask;
    auto known = net->backward_sizes.find(key);
    if (known == net->backward_sizes.end()) {
        BackwardSizes sz;
        int keep_every = 1;
        auto need_for = [&](int64_t nb) {
            Backward d = bw;
            d.exec = false;
            d.nb = nb;
            d.keep_every = keep_every;
            // a whole batch and the smaller last one, which can need more: its operand
            // planes may stay below the cap at which the others are cut into panels
            backward_run(d, lo, std::min(hi, lo + nb + (hi - lo) % nb), grad_out_c128);
            return (size_t)d.A.top;
        };
        if (net->backward_keep_every > 0) keep_every = net->backward_keep_every;
        else
            while (need_for(1) > budget_bytes && keep_every < 64) keep_every *= 2;
        sz.need = need_for(1);
        sz.keep_every = keep_every;
        if (sz.need <= budget_bytes) {
            int64_t nb = 1;
            const int64_t hi_b = std::min<int64_t>(hi - lo, 1024);
            while (nb < hi_b) {
                int64_t nx = std::min<int64_t>(nb * 2, hi_b);
                const size_t need = need_for(nx);
                if (need > budget_bytes) break;
                nb = nx;
                sz.need = need;
            }
            sz.nb = nb;
            if (keep_every == 1 && T.root >= net->n_leaves) {
                Backward d = bw;
                BackwardPlan dry;
                build_backward_plan(d, nb, (hi - lo) % nb, dry);
                if ((size_t)dry.top <= budget_bytes) sz.need_levels = (size_t)dry.top;
            }
        }
        if (net->backward_sizes.size() >= 64) net->backward_sizes.clear();
        known = net->backward_sizes.emplace(key, sz).first;
    }
    const BackwardSizes sz = known->second;
    if (sz.nb == 0)
        return fail(TNC_E_OOM, "backward workspace for one slice exceeds the budget (" + std::to_string(sz.need) + " bytes)");
    net->last_keep_every = sz.keep_every;
    const int64_t nb = sz.nb;
    // by levels when its workspace is there or can be had, and, during a capture, its
    // plan: a plan is uploaded, the node-by-node pass has its parameters in its launches
    const int64_t tail = (hi - lo) % nb;
    auto place = [&](size_t bytes) -> char* {
        if (net->ws_user && net->ws_user_bytes >= bytes) return (char*)net->ws_user;
        return net->ws_own && net->ws_own_bytes >= bytes ? (char*)net->ws_own : nullptr;
    };
    auto plan_at = [&](const char* at) {
        return plan_key(net, mode, nb) + ":" + std::to_string(tail) + ":" + std::to_string((uintptr_t)at) + ":" +
               std::to_string((uintptr_t)net->d_leaves) + ":" + mask;
    };
    const bool capture = capturing(s);
    bool levels = sz.need_levels > 0;
    if (net->ws_user && net->ws_user_bytes < sz.need_levels && net->ws_user_bytes >= sz.need)
        levels = false;  // the caller's workspace fits node by node only
    if (levels && capture) {
        char* const at = place(sz.need_levels);
        levels = at && net->backward_plans.count(plan_at(at));
    }
    size_t need = levels ? sz.need_levels : sz.need;
    char* ws = place(need);
    if (!ws) {
        if (net->ws_own) CUDA_TRY(cudaFree(net->ws_own));
        net->ws_own = nullptr;
        net->ws_own_bytes = 0;
        size_t bytes = std::max(need, sz.need);  // (either way fits then)
        if (bytes > sz.need && cudaMalloc(&net->ws_own, bytes) != cudaSuccess) {
            (void)cudaGetLastError();
            net->ws_own = nullptr;
            levels = false;
            need = bytes = sz.need;
        }
        if (!net->ws_own) CUDA_TRY(cudaMalloc(&net->ws_own, bytes));
        net->ws_own_bytes = bytes;
        ws = (char*)net->ws_own;
    }
    net->last_backward_bytes = need;
    net->last_batch = nb;
    net->group_key.clear();  // the workspace may now hold other data
    net->inv_key.clear();
    CUDA_TRY(cudaMemsetAsync(net->d_err, 0, sizeof(int), s));
    bw.exec = true;
    bw.nb = nb;
    bw.ws = ws;
    bw.keep_every = sz.keep_every;
    if (levels) {
        const std::string pkey = plan_at(ws);
        auto it = net->backward_plans.find(pkey);
        if (it == net->backward_plans.end()) {
            auto bp = std::make_unique<BackwardPlan>();
            build_backward_plan(bw, nb, tail, *bp);
            if ((st = upload_backward_plan(*bp, s)) != TNC_OK) return st;
            if (net->backward_plans.size() >= 4) {
                for (auto& [k, plan] : net->backward_plans)
                    if (plan->captured) net->backward_kept.push_back(std::move(plan));
                net->backward_plans.clear();
            }
            it = net->backward_plans.emplace(pkey, std::move(bp)).first;
        }
        it->second->captured |= capture;
        const BackwardPlan& bp = *it->second;
        bw.leaf_grad = 0;
        CUDA_TRY(cudaMemsetAsync(ws, 0, bp.zero_bytes, s));
        auto run = [&](const std::vector<BackwardOp>& ops, int64_t batch, int64_t s0) {
            return run_backward_ops(net, bp, ops, batch, s0, mode, grad_out_c128, ws, s);
        };
        if ((st = run(bp.inv_fwd, 1, 0)) != TNC_OK) return st;
        for (int64_t s0 = lo; s0 < hi; s0 += nb) {
            const int64_t b = std::min<int64_t>(nb, hi - s0);
            if ((st = run(bp.slices[b < nb ? 1 : 0], b, s0)) != TNC_OK) return st;
        }
        if ((st = run(bp.inv_rev, 1, 0)) != TNC_OK) return st;
    } else if ((st = backward_run(bw, lo, hi, grad_out_c128)) != TNC_OK) {
        return st;
    }
    CUDA_TRY(tnc::launch_f64_to_f32(reinterpret_cast<const double2*>(ws + bw.leaf_grad), net->total_leaf_elems,
                                    reinterpret_cast<float2*>(grad_leaves_c64), s));
    net->launches += 1;
    return TNC_OK;
}

tnc_status tnc_param_grads(tnc_net_t net, int n_params, const int* leaf_ids, const float* dleaf_c64,
                           const float* env_packed_c64, double* out_c128, void* stream) {
    if (!net) return fail(TNC_E_INVALID, "NULL network");
    if (n_params < 0 || (n_params > 0 && (!leaf_ids || !dleaf_c64 || !env_packed_c64 || !out_c128)))
        return fail(TNC_E_INVALID, "bad argument");
    if (n_params == 0) return TNC_OK;
    std::vector<int64_t> host(3 * (size_t)n_params);
    int64_t doff = 0;
    for (int q = 0; q < n_params; ++q) {
        const int l = leaf_ids[q];
        if (l < 0 || l >= net->n_leaves) return fail(TNC_E_INVALID, "leaf id out of range");
        host[q] = net->leaf_off[l];
        host[n_params + q] = doff;
        host[2 * n_params + q] = net->leaf_elems[l];
        doff += net->leaf_elems[l];
    }
    cudaStream_t s = (cudaStream_t)stream;
    const size_t bytes = host.size() * sizeof(int64_t);
    if (net->pg_cap < bytes) {
        if (net->d_pg) CUDA_TRY(cudaFree(net->d_pg));
        net->d_pg = nullptr;
        net->pg_cap = 0;
        CUDA_TRY(cudaMalloc(&net->d_pg, bytes));
        net->pg_cap = bytes;
    }
    CUDA_TRY(cudaMemcpyAsync(net->d_pg, host.data(), bytes, cudaMemcpyHostToDevice, s));
    CUDA_TRY(tnc::launch_param_grads(n_params, net->d_pg, net->d_pg + n_params, net->d_pg + 2 * n_params,
                                     reinterpret_cast<const float2*>(env_packed_c64),
                                     reinterpret_cast<const float2*>(dleaf_c64),
                                     reinterpret_cast<double2*>(out_c128), s));
    CUDA_TRY(cudaStreamSynchronize(s));  // the staged offsets above are host memory
    return TNC_OK;
}


}  // extern "C"
