// sg_vb.cu -- Viana-Bray model, host side: validation, greedy colouring, device layouts
// (plain colour-major CSR and packed sliced-ELL), measurement bookkeeping.
//
// Update order: the vertices of a graph are coloured greedily in vertex order (each vertex gets
// the smallest colour not used by an already-coloured neighbour), then greedily once more in the
// order of decreasing colour (increasing label inside a colour); a sweep updates colour class
// 0, then 1, ...  Each class is an independent set, so its vertices can be updated in parallel;
// this generalises the bipartite half-updates of SI section 3 to the Poissonian graphs of the
// Viana-Bray ensemble (Eq. 3).  The random number of a vertex is keyed by its original label,
// so relabelling and slicing never change the trajectory.
#include <math.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <atomic>
#include <memory>
#include <string>
#include <thread>
#include <vector>

#include "../../include/sg.h"
#include "sg_internal.cuh"
#include "sg_model.h"
#include "vb_resident.h"

namespace sg {
namespace {

struct Graph {
    int32_t n = 0;
    int64_t edges = 0;  // undirected
    std::vector<int32_t> row_ptr, col;
    std::vector<uint64_t> jb;
    std::vector<int32_t> colour;
    int n_colours = 0;
    uint64_t seed = 0;
    std::vector<double> temps;
};

void load_graph(const sg_vb_graph& in, int R, int idx, Graph& g) {
    const std::string tag = "graph " + std::to_string(idx) + ": ";
    if (in.n < 2 || in.n > SG_VB_MAX_N) fail(SG_EINVAL, tag + "n out of range");
    if (!in.row_ptr || !in.col || !in.jbits || !in.temps) fail(SG_EINVAL, tag + "null array");
    const int32_t n = in.n;
    if (in.row_ptr[0] != 0) fail(SG_EINVAL, tag + "row_ptr[0] != 0");
    for (int32_t i = 0; i < n; ++i) {
        const int32_t d = in.row_ptr[i + 1] - in.row_ptr[i];
        if (d < 0) fail(SG_EINVAL, tag + "row_ptr not monotone");
        if (d > SG_VB_MAX_DEGREE) fail(SG_EINVAL, tag + "degree above " + std::to_string(SG_VB_MAX_DEGREE));
    }
    const int64_t nnz = in.row_ptr[n];
    if (nnz % 2) fail(SG_EINVAL, tag + "odd number of directed entries (not symmetric)");
    g.n = n;
    g.edges = nnz / 2;
    g.row_ptr.assign(in.row_ptr, in.row_ptr + n + 1);
    g.col.assign(in.col, in.col + nnz);
    g.jb.assign(in.jbits, in.jbits + nnz);
    // sorted copy of every row for the structural checks
    std::vector<std::pair<int32_t, uint64_t>> srt(nnz);
    for (int64_t e = 0; e < nnz; ++e) {
        if (g.col[e] < 0 || g.col[e] >= n) fail(SG_EINVAL, tag + "neighbour index out of range");
        srt[e] = {g.col[e], g.jb[e]};
    }
    for (int32_t i = 0; i < n; ++i) {
        auto b = srt.begin() + g.row_ptr[i], e = srt.begin() + g.row_ptr[i + 1];
        std::sort(b, e);
        for (auto it = b; it != e; ++it) {
            if (it->first == i) fail(SG_EINVAL, tag + "self-loop at vertex " + std::to_string(i));
            if (it + 1 != e && (it + 1)->first == it->first)
                fail(SG_EINVAL, tag + "duplicate edge at vertex " + std::to_string(i));
        }
    }
    for (int32_t i = 0; i < n; ++i)
        for (int32_t e = g.row_ptr[i]; e < g.row_ptr[i + 1]; ++e) {
            const int32_t j = srt[e].first;
            auto b = srt.begin() + g.row_ptr[j], en = srt.begin() + g.row_ptr[j + 1];
            auto it = std::lower_bound(b, en, std::make_pair(i, (uint64_t)0),
                                       [](const std::pair<int32_t, uint64_t>& a,
                                          const std::pair<int32_t, uint64_t>& c) {
                                           return a.first < c.first;
                                       });
            if (it == en || it->first != i)
                fail(SG_EINVAL, tag + "edge (" + std::to_string(i) + "," + std::to_string(j) +
                                    ") has no reverse entry");
            if (it->second != srt[e].second)
                fail(SG_EINVAL, tag + "couplings of edge (" + std::to_string(i) + "," +
                                    std::to_string(j) + ") differ between directions");
        }
    g.temps.assign(in.temps, in.temps + R);
    for (double T : g.temps)
        if (!(T >= 0.0)) fail(SG_EINVAL, tag + "temperature must be >= 0 (or +inf)");
    g.seed = in.seed;
    // greedy colouring in vertex order
    g.colour.assign(n, -1);
    std::vector<char> used(SG_VB_MAX_DEGREE + 2, 0);
    int nc = 0;
    for (int32_t i = 0; i < n; ++i) {
        for (int32_t e = g.row_ptr[i]; e < g.row_ptr[i + 1]; ++e) {
            const int c = g.colour[g.col[e]];
            if (c >= 0) used[c] = 1;
        }
        int c = 0;
        while (used[c]) ++c;
        g.colour[i] = c;
        nc = std::max(nc, c + 1);
        for (int32_t e = g.row_ptr[i]; e < g.row_ptr[i + 1]; ++e) {
            const int cj = g.colour[g.col[e]];
            if (cj >= 0) used[cj] = 0;
        }
    }
    // one recolouring pass: greedy again, visiting the classes from the last to the first
    // (vertex order inside a class).  Each old class is an independent set, so no colour is
    // added, and the thin last classes of the first pass are folded into the others.
    std::vector<int32_t> start(nc + 1, 0), order(n);
    for (int32_t i = 0; i < n; ++i) ++start[nc - g.colour[i]];
    for (int c = 0; c < nc; ++c) start[c + 1] += start[c];
    for (int32_t i = 0; i < n; ++i) order[start[nc - 1 - g.colour[i]]++] = i;
    std::vector<int32_t> fresh(n, -1);
    int nc2 = 0;
    for (int32_t i : order) {
        for (int32_t e = g.row_ptr[i]; e < g.row_ptr[i + 1]; ++e) {
            const int c = fresh[g.col[e]];
            if (c >= 0) used[c] = 1;
        }
        int c = 0;
        while (used[c]) ++c;
        fresh[i] = c;
        nc2 = std::max(nc2, c + 1);
        for (int32_t e = g.row_ptr[i]; e < g.row_ptr[i + 1]; ++e) {
            const int cj = fresh[g.col[e]];
            if (cj >= 0) used[cj] = 0;
        }
    }
    g.colour.swap(fresh);
    g.n_colours = nc2;
}

// Validate and colour every graph of a batch, one graph per task on the host's cores (the
// graphs are independent; a batch of hundreds of uneven graphs is mostly this work).  The first
// failing graph's error, in graph order, is raised after all tasks have ended.
void load_graphs(const sg_vb_graph* in, int n_graphs, int R, std::vector<Graph>& out) {
    out.resize(n_graphs);
    const unsigned hw = std::max(1u, std::thread::hardware_concurrency());
    const int nt = (int)std::min<unsigned>(hw, (unsigned)n_graphs);
    std::vector<std::unique_ptr<Error>> errs(n_graphs);
    std::atomic<int> next{0};
    auto work = [&] {
        for (;;) {
            const int b = next.fetch_add(1);
            if (b >= n_graphs) return;
            try {
                load_graph(in[b], R, b, out[b]);
            } catch (const Error& e) {
                errs[b].reset(new Error(e));
            } catch (const std::bad_alloc&) {
                errs[b].reset(new Error{SG_ENOMEM, "host allocation failed"});
            }
        }
    };
    if (nt <= 1) {
        work();
    } else {
        std::vector<std::thread> pool;
        for (int t = 0; t < nt; ++t) pool.emplace_back(work);
        for (auto& th : pool) th.join();
    }
    for (auto& e : errs)
        if (e) throw *e;
}

// Run f(lo, hi) over [0, n) cut into contiguous ranges, one per host thread (f must only write
// what its own range owns).
template <class F>
void parallel_ranges(int64_t n, F&& f) {
    const unsigned hw = std::max(1u, std::thread::hardware_concurrency());
    const int64_t nt = std::min<int64_t>((int64_t)hw, std::max<int64_t>(1, n / 4096));
    if (nt <= 1) {
        f((int64_t)0, n);
        return;
    }
    std::vector<std::thread> pool;
    for (int64_t t = 0; t < nt; ++t) pool.emplace_back([&, t] { f(n * t / nt, n * (t + 1) / nt); });
    for (auto& th : pool) th.join();
}

std::vector<uint32_t> vb_table(double T) {
    std::vector<uint32_t> t(kVbThrStride);
    const double beta = 1.0 / T;
    t[0] = 0xFFFFFFFFu;
    for (int m = 1; m < kVbThrStride; ++m) t[m] = metropolis_threshold(-2.0 * beta * m);
    return t;
}

class VbModel : public Model {
public:
    VbModel(const sg_vb_graph* graphs, int n_graphs, int n_lanes, int n_replicas, int kernel,
            const std::vector<int64_t>& tw_, const std::vector<int64_t>& tm_) {
        if (kernel != SG_VB_PLAIN && kernel != SG_VB_PACKED) fail(SG_EINVAL, "unknown VB kernel");
        if (n_lanes < 1 || n_lanes > 64) fail(SG_EINVAL, "n_lanes must be 1..64");
        if (n_replicas < 1) fail(SG_EINVAL, "n_replicas must be >= 1");
        if (kernel == SG_VB_PACKED && !(n_replicas == 1 || n_replicas == 2 || n_replicas == 4))
            fail(SG_EINVAL, "packed kernel supports 1, 2 or 4 replicas");
        if (kernel == SG_VB_PLAIN && n_graphs != 1) fail(SG_EINVAL, "plain kernel takes one graph");
        kernel_ = kernel;
        n_inst = n_graphs;
        R = n_replicas;
        L = n_lanes;
        Lc_ = kernel == SG_VB_PACKED ? 64 : L;
        tw = tw_;
        tm = tm_;
        load_graphs(graphs, n_graphs, R, graphs_);
        for (const Graph& g : graphs_)
            for (int r = 0; r < R; ++r) {
                auto t = vb_table(g.temps[r]);
                for (int m = 1; m < kVbThrStride; ++m)
                    if (t[m] > t[m - 1]) fail(SG_EINVAL, "threshold table not monotone");
                thr_.insert(thr_.end(), t.begin(), t.end());
            }
        if (kernel == SG_VB_PACKED) build_packed();
        else build_plain();
        Carver c;
        carve(c);
        ws_bytes_ = c.off;
    }

    // computed once at construction: carving with a null base would reset the device views
    size_t workspace_bytes() const override { return ws_bytes_; }

    void attach(char* ws, cudaStream_t st) override {
        Carver c;
        c.base = ws;
        carve(c);
        auto up = [&](void* dst, const void* src, size_t bytes) {
            if (bytes) check_cuda(cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, st), "H2D copy");
            h2d_bytes += (int64_t)bytes;
        };
        up((void*)d_thr_, thr_.data(), thr_.size() * 4);
        if (kernel_ == SG_VB_PACKED) {
            up((void*)pk_.vinfo, h_vinfo_.data(), h_vinfo_.size() * 4);
            up((void*)pk_.slice_base, h_slice_base_.data(), h_slice_base_.size() * 4);
            up((void*)pk_.slice_graph, h_slice_graph_.data(), h_slice_graph_.size() * 4);
            up((void*)pk_.col, h_col_.data(), h_col_.size() * 4);
            up((void*)pk_.slice_meta, h_slice_meta_.data(), h_slice_meta_.size() * sizeof(uint4));
            check_cuda(cudaMemsetAsync(pk_.err, 0, 4, st), "memset");
            check_cuda(cudaMemsetAsync(pk_.gbar, 0, 8, st), "memset");
            check_cuda(cudaMemsetAsync(pk_.claims, 0, (size_t)kVbClaimGroups * 2 * kVbMaxColours * 4, st), "memset");
            up((void*)rs_.graph_class_slice, graph_class_slice_.data(), graph_class_slice_.size() * 4);
            up((void*)pk_.class_slice, colour_slice_.data(), colour_slice_.size() * 4);
            up((void*)pk_.jb, h_jb_.data(), h_jb_.size() * 8);
            std::vector<uint64_t> seeds(n_inst);
            for (int b = 0; b < n_inst; ++b) seeds[b] = graphs_[b].seed;
            up((void*)pk_.seeds, seeds.data(), seeds.size() * 8);
            std::vector<int64_t> gw(1, 0);
            for (const Graph& g : graphs_) gw.push_back(gw.back() + (int64_t)R * g.n);
            up((void*)d_graph_words_, gw.data(), gw.size() * 8);
            up((void*)pk_.up_slice_base, h_up_base_.data(), h_up_base_.size() * 4);
            launches += vb_packed_build_upper(pk_, st);  // from col and jb, on the device
            launches += vb_packed_init(pk_, st);
            form_ = plan_resident() ? kResident : kGrid;
        } else {
            up((void*)pl_.row_ptr, h_row_ptr_.data(), h_row_ptr_.size() * 4);
            up((void*)pl_.col, h_col_i_.data(), h_col_i_.size() * 4);
            up((void*)pl_.jb, h_jb_.data(), h_jb_.size() * 8);
            up((void*)pl_.orig, h_orig_.data(), h_orig_.size() * 4);
            launches += vb_plain_init(pl_, st);
        }
        check_cuda(cudaMemsetAsync(dC_, 0, nC() * 8, st), "memset");
        check_cuda(cudaMemsetAsync(dQ_, 0, nQ() * 8, st), "memset");
        check_cuda(cudaMemsetAsync(dE_, 0, nE() * 8, st), "memset");
        if (n_bins) {
            check_cuda(cudaMemsetAsync(wC_, 0, nwC() * 8, st), "memset");
            check_cuda(cudaMemsetAsync(wQ_, 0, nwQ() * 8, st), "memset");
            check_cuda(cudaMemsetAsync(wE_, 0, nwE() * 8, st), "memset");
        }
        check_cuda(cudaGetLastError(), "init launch");
        check_cuda(cudaStreamSynchronize(st), "attach");
    }

    // The plan with 2^lc CTAs for every graph, and the entries of the largest graph; false: some graph does
    // not fit.
    bool resident_layout(uint32_t lc, bool copies, VbResident& rs, int64_t& graph_entries) const {
        const int nc = pk_.n_colours;
        const uint32_t C = 1u << lc;
        rs = rs_;
        rs.cluster = C;
        rs.log_cluster = lc;
        rs.copies = copies;
        rs.graph_slices = 0;
        rs.max_slices = 0;
        rs.max_entries = 0;
        graph_entries = 0;
        for (int b = 0; b < n_inst; ++b) {
            int64_t ns[kResMaxCluster] = {}, ne[kResMaxCluster] = {}, all = 0, entries = 0;
            for (int c = 0; c < nc; ++c) {
                const uint32_t lo = graph_class_slice_[(size_t)c * n_inst + b],
                               hi = graph_class_slice_[(size_t)c * n_inst + b + 1];
                if (hi - lo > C * 1024u) return false;  // far beyond shared memory
                all += hi - lo;
                for (uint32_t s = lo; s < hi; ++s) {
                    const uint32_t k = (s - lo) & (C - 1);
                    ++ns[k];
                    ne[k] += h_slice_base_[s + 1] - h_slice_base_[s];
                }
            }
            for (uint32_t k = 0; k < C; ++k) {
                rs.max_slices = std::max(rs.max_slices, (int)ns[k]);
                rs.max_entries = std::max(rs.max_entries, (uint32_t)ne[k]);
                entries += ne[k];
            }
            graph_entries = std::max(graph_entries, entries);
            rs.graph_slices = std::max(rs.graph_slices, (int)all);
            if (vb_resident_smem(R, copies ? rs.graph_slices : rs.max_slices, rs.max_slices,
                                 rs.max_entries) > (size_t)kResMaxSmem)
                return false;
        }
        return vb_resident_clusters(R, rs) >= n_inst;
    }

    // What a class takes in a cluster, and grid-wide (us, the average over the classes), for one, two and
    // four replicas.  Fitted to bipartite graphs of degree 3 to 6 and Poissonian ones of mean degree 2 to 16,
    // N = 1000 .. 48000, alone and in batches of up to 100; within 15 %.
    // With copies of all words a CTA sends each slice that it updates to the others; without, it gathers
    // its slices' entries, a row of 32 at a time, from them.  Examples (us a sweep, one replica where not
    // said, cluster against grid): bipartite N = 8192 3.6, 4.0; 16384 5.7, 4.1; 32768 13.5, 4.2; two replicas
    // 4096 3.0, 4.5; 16384 7.8, 4.6; four replicas 4096 4.8, 4.9; 8192 8.2, 4.9; eight Poissonian graphs of degree 4,
    // N = 5000, 13.0, 14.8; one of them, one replica, N = 16384 8.1, 10.9; 24000 14.5, 11.6; nine bipartite graphs of
    // 9000, two replicas, 6.0, 6.8.
    double cluster_us(const VbResident& rs, int64_t graph_entries, int more) const {
        static const double kCopies[3][3] = {{0.8, 0.03, 0.0065}, {0.75, 0.04, 0.0125}, {1.5, 0.132, 0.017}};
        static const double kGather[3][3] = {{0.95, 0.045, 0.15}, {0.85, 0.047, 0.25}, {0.9, 0.096, 0.6}};
        const int q = R == 4 ? 2 : R - 1;
        const double slices = (double)rs.max_slices / pk_.n_colours;
        const double rows = (double)graph_entries / rs.cluster / 32 / pk_.n_colours;
        if (rs.copies) return kCopies[q][0] + slices * (kCopies[q][1] + kCopies[q][2] * (rs.cluster - 1));
        return kGather[q][0] + rows * kGather[q][1] + more * kGather[q][2];
    }
    double grid_us(int more) const {
        static const double kGridWide[3][3] = {{2.0, 0.00055, 0.15}, {2.2, 0.0007, 0.3}, {2.4, 0.00105, 0.33}};
        const int q = R == 4 ? 2 : R - 1;
        return kGridWide[q][0] + kGridWide[q][1] * pk_.n_slices / pk_.n_colours + more * kGridWide[q][2];
    }

    // Which graphs run in shared memory, and how (R = 2, Poissonian of degree 4, us a sweep).
    // One CTA as long as its 12 updating warps take a class in two rounds at most: N = 1000 4.5,
    // against 4.8 in a cluster and 11.4 in the grid-wide form; N = 2500 7.8, 5.0 in a cluster.
    // A cluster whose CTAs each hold a copy of all words: 8 CTAs where that fits (N = 2500 5.0, 16 CTAs
    // 5.5, without copies 6.3; N = 6000 6.4, 6.9, 7.6), else 16 (N = 9000 8.1, without copies 8.6;
    // one replica, N = 18000 8.3, 11.4).  Each update goes to all CTAs, so four replicas do not gain
    // from 16 (N = 4500 13.6, without copies 10.9), nor does a graph of degree 4, whose words
    // arrive in one round (bipartite N = 4096: 16 CTAs without copies 2.9, 8 with copies 3.2).
    // A cluster only where it is estimated to take no longer than the grid-wide form.
    // A batch takes the first of these for which the GPU holds all its clusters at once.
    bool plan_resident() {
        if (pk_.n_colours < 1) return false;
        int widest = 0;  // slices of the largest class of one graph
        for (size_t i = 0; i + 1 < graph_class_slice_.size(); ++i)
            widest = std::max(widest, (int)(graph_class_slice_[i + 1] - graph_class_slice_[i]));
        const uint32_t width = pk_.max_width;
        rs_.wide = width > 15;
        const int more = width > 8 ? (int)(width - 1) / 8 : 0;
        VbResident rs;
        int64_t entries = 0;
        auto take = [&](uint32_t lc, bool copies) {
            if (!resident_layout(lc, copies, rs, entries)) return false;
            if (lc > 0 && cluster_us(rs, entries, more) > grid_us(more)) return false;
            rs_ = rs;
            return true;
        };
        if (widest <= kResMain + kResMain / 3 && take(0, false)) return true;
        if (width <= 4 && R >= 2 && take(4, false)) return true;
        return take(3, true) || (R < 4 && take(4, true)) || take(4, false) || take(2, true) ||
               take(3, false) || take(1, true) || take(2, false) || take(1, false);
    }

    // The packed sweeps of a call, without a captured graph: a launch takes as many sweeps as run in a few
    // milliseconds, so nothing is left of the launches' gaps.  A single sweep is done grid-wide, whatever the
    // form: taking the instance into shared memory and the words back costs more than the sweep saves
    // (us a call of one sweep, shared memory against grid: N = 1000 20, 12 with one replica and 27, 17 with
    // four; N = 14000, two replicas 29, 17; 140 graphs of 1000, four replicas 30, 25; of two sweeps 27, 27 and 35,
    // 31; 39, 31; 37, 46).
    bool sweep_direct(int64_t t0, int64_t n, cudaStream_t st) override {
        if (kernel_ != SG_VB_PACKED) return false;
        const int64_t most = std::max<int64_t>(1, std::min<int64_t>(1024, ((int64_t)1 << 28) / (n_slots_ * R)));
        for (int64_t done = 0; done < n;) {
            const int m = (int)std::min<int64_t>(n - done, most);
            const uint32_t t = (uint32_t)(t0 + done);
            const int k = form_ == kResident && m > 1 ? vb_resident_sweeps(pk_, rs_, t, m, st)
                                             : vb_packed_sweeps(pk_, max_class_slices_, t, m, st);
            if (k < 0) fail(SG_ECUDA, "sweep launch failed");
            launches += k;
            done += m;
        }
        return true;
    }

    void sweep(uint32_t t_off, cudaStream_t st) override {
        if (kernel_ == SG_VB_PACKED) fail(SG_EINVAL, "packed sweeps are queued by sweep_direct");
        for (size_t c = 0; c + 1 < colour_begin_.size(); ++c)
            launches += vb_plain_colour(pl_, colour_begin_[c], colour_begin_[c + 1], clock_dev, t_off, st);
    }

    void snapshot(int w, cudaStream_t st) override {
        if (kernel_ == SG_VB_PACKED) launches += vb_packed_snapshot(pk_, w, st);
        else if (vb_plain_snapshot(pl_, w, st) < 0) fail(SG_ECUDA, "snapshot copy failed");
    }

    // add the raw counts at time tau into column u of count arrays with ncol columns
    void measure_into(int64_t* Cb, int64_t* Qb, int64_t* Eb, int64_t ncol, int64_t u, int64_t tau,
                      cudaStream_t st) {
        const int64_t ntw = (int64_t)tw.size();
        int active = 0;
        while (active < (int)ntw && tw[active] <= tau) ++active;
        VbMeasure m{};
        m.n_c = active;
        m.c = Cb + u;
        m.c_w = ncol;
        m.c_k = ntw * ncol;
        m.c_r = (int64_t)Lc_ * m.c_k;
        m.c_g = R * m.c_r;
        m.q = R >= 2 ? Qb + u : nullptr;
        m.q_k = ncol;
        m.q_r = (int64_t)Lc_ * ncol;
        m.q_g = (R / 2) * m.q_r;
        m.e = Eb + u;
        m.e_k = ncol;
        m.e_r = (int64_t)Lc_ * ncol;
        m.e_g = R * m.e_r;
        if (kernel_ == SG_VB_PACKED) {
            const int n = vb_packed_measure(pk_, m, st);
            if (n < 0) fail(SG_ECUDA, "measurement launch failed");
            launches += n;
            return;
        }
        for (int w = 0; w < active; ++w)
            launches += vb_plain_count(pl_, VbCountJob{0, w, m.c + w * m.c_w, m.c_r, m.c_k}, st);
        if (m.q) launches += vb_plain_count(pl_, VbCountJob{1, 0, m.q, m.q_r, m.q_k}, st);
        launches += vb_plain_count(pl_, VbCountJob{2, 0, m.e, m.e_r, m.e_k}, st);
    }

    void measure_scheduled(int u, int64_t tau, cudaStream_t st) override {
        measure_into(dC_, dQ_, dE_, (int64_t)tm.size(), u, tau, st);
    }

    void set_windows(int64_t nb) override {
        n_bins = nb;
        Carver c;
        carve(c);
        ws_bytes_ = c.off;
    }

    void measure_window(int m, int64_t tau, cudaStream_t st) override {
        measure_into(wC_, wQ_, wE_, n_bins, m, tau, st);
    }

    void read_windows(const int64_t* cnt_c, const int64_t* cnt_q, int64_t* C, int64_t* q,
                      int64_t* E, cudaStream_t st) override {
        const Counts all = read_counts(wC_, wQ_, wE_, nwE(), st, "read windows");
        const int64_t *c = all.c, *qq = all.q, *e = all.e;
        const int64_t ntw = (int64_t)tw.size(), nb = n_bins;
        for (int b = 0; b < n_inst; ++b) {
            const int64_t N = graphs_[b].n, M = graphs_[b].edges;
            for (int r = 0; r < R; ++r)
                for (int k = 0; k < L; ++k)
                    for (int64_t m = 0; m < nb; ++m) {
                        for (int64_t w = 0; w < ntw; ++w) {
                            const int64_t src = ((((int64_t)b * R + r) * Lc_ + k) * ntw + w) * nb + m;
                            const int64_t dst = ((((int64_t)b * R + r) * L + k) * ntw + w) * nb + m;
                            C[dst] = cnt_c[w * nb + m] * N - 2 * c[src];
                        }
                        const int64_t se = (((int64_t)b * R + r) * Lc_ + k) * nb + m;
                        const int64_t de = (((int64_t)b * R + r) * L + k) * nb + m;
                        E[de] = cnt_q[m] * M - e[se];
                        if (r < R / 2) {
                            const int64_t sq = (((int64_t)b * (R / 2) + r) * Lc_ + k) * nb + m;
                            const int64_t dq = (((int64_t)b * (R / 2) + r) * L + k) * nb + m;
                            q[dq] = cnt_q[m] * N - 2 * qq[sq];
                        }
                    }
        }
    }

    void measure_now(int64_t tau, cudaStream_t st) override {
        check_cuda(cudaMemsetAsync(mC_, 0, (size_t)(mE_ - mC_ + (int64_t)nmE()) * 8, st), "memset");
        measure_into(mC_, mQ_, mE_, 1, 0, tau, st);
    }

    void read_scheduled(int64_t tau, int64_t* C, int64_t* q, int64_t* E, cudaStream_t st) override {
        const Counts all = read_counts(dC_, dQ_, dE_, nE(), st, "read results");
        const int64_t *c = all.c, *qq = all.q, *e = all.e;
        const int64_t ntw = (int64_t)tw.size(), ntm = (int64_t)tm.size();
        for (int b = 0; b < n_inst; ++b) {
            const int64_t N = graphs_[b].n, M = graphs_[b].edges;
            for (int r = 0; r < R; ++r)
                for (int k = 0; k < L; ++k)
                    for (int64_t u = 0; u < ntm; ++u) {
                        const bool done = tm[u] <= tau;
                        for (int64_t w = 0; w < ntw; ++w) {
                            const bool ok = done && tw[w] <= tm[u];
                            const int64_t src = ((((int64_t)b * R + r) * Lc_ + k) * ntw + w) * ntm + u;
                            const int64_t dst = ((((int64_t)b * R + r) * L + k) * ntw + w) * ntm + u;
                            C[dst] = ok ? N - 2 * c[src] : 0;
                        }
                        const int64_t se = (((int64_t)b * R + r) * Lc_ + k) * ntm + u;
                        const int64_t de = (((int64_t)b * R + r) * L + k) * ntm + u;
                        E[de] = done ? M - e[se] : 0;
                        if (r < R / 2) {
                            const int64_t sq = (((int64_t)b * (R / 2) + r) * Lc_ + k) * ntm + u;
                            const int64_t dq = (((int64_t)b * (R / 2) + r) * L + k) * ntm + u;
                            q[dq] = done ? N - 2 * qq[sq] : 0;
                        }
                    }
        }
    }

    void read_now(int64_t tau, int64_t* C, int64_t* q, int64_t* E, cudaStream_t st) override {
        const Counts all = read_counts(mC_, mQ_, mE_, nmE(), st, "read measurement");
        const int64_t *c = all.c, *qq = all.q, *e = all.e;
        const int64_t ntw = (int64_t)tw.size();
        for (int b = 0; b < n_inst; ++b) {
            const int64_t N = graphs_[b].n, M = graphs_[b].edges;
            for (int r = 0; r < R; ++r)
                for (int k = 0; k < L; ++k) {
                    for (int64_t w = 0; w < ntw; ++w) {
                        const int64_t src = (((int64_t)b * R + r) * Lc_ + k) * ntw + w;
                        const int64_t dst = (((int64_t)b * R + r) * L + k) * ntw + w;
                        C[dst] = tw[w] <= tau ? N - 2 * c[src] : 0;
                    }
                    E[((int64_t)b * R + r) * L + k] = M - e[((int64_t)b * R + r) * Lc_ + k];
                    if (r < R / 2)
                        q[((int64_t)b * (R / 2) + r) * L + k] =
                            N - 2 * qq[((int64_t)b * (R / 2) + r) * Lc_ + k];
                }
        }
    }

    size_t spins_bytes() const override {
        int64_t tot = 0;
        for (const Graph& g : graphs_) tot += (int64_t)R * g.n;
        return (size_t)tot * 8;
    }

    void get_spins(void* dst, cudaStream_t st) override {
        uint64_t* out = static_cast<uint64_t*>(dst);
        if (kernel_ == SG_VB_PACKED) {
            // laid out in the caller's order on the device, a part at a time, and copied straight
            // to the caller
            const int64_t total = (int64_t)(spins_bytes() / 8);
            for (int64_t lo = 0; lo < total; lo += spin_part()) {
                const int64_t hi = std::min(total, lo + spin_part());
                launches += vb_packed_spins(pk_, d_graph_words_, lo, hi, d_spins_, st);
                check_cuda(cudaGetLastError(), "spins launch");
                down(out + lo, d_spins_, (size_t)(hi - lo) * 8, st);
            }
            check_cuda(cudaStreamSynchronize(st), "read spins");
        } else {
            const int32_t N = pl_.N;
            std::vector<int8_t> s((size_t)R * L * N);
            down(s.data(), pl_.s, s.size(), st);
            check_cuda(cudaStreamSynchronize(st), "read spins");
            for (int r = 0; r < R; ++r)
                for (int32_t v = 0; v < N; ++v) {
                    const int32_t nv = new_of_[v];
                    uint64_t w = 0;
                    for (int k = 0; k < L; ++k)
                        if (s[((size_t)r * L + k) * N + nv] < 0) w |= 1ull << k;
                    out[(int64_t)r * N + v] = w;
                }
        }
    }

    std::vector<uint32_t> thresholds() const override { return thr_; }

    std::vector<int32_t> colouring(int b, int* n_colours) const override {
        if (b < 0 || b >= n_inst) fail(SG_EINVAL, "graph index out of range");
        *n_colours = graphs_[b].n_colours;
        return graphs_[b].colour;
    }

    int device_status(cudaStream_t st) override {
        int v = 0;
        if (kernel_ == SG_VB_PACKED && pk_.err) {
            check_cuda(cudaMemcpyAsync(&v, pk_.err, 4, cudaMemcpyDeviceToHost, st), "status copy");
            check_cuda(cudaStreamSynchronize(st), "status");
        }
        return v;
    }

    std::vector<std::pair<void*, size_t>> state_regions() override {
        std::vector<std::pair<void*, size_t>> v;
        if (kernel_ == SG_VB_PACKED) {
            v.push_back({pk_.S, (size_t)pk_.n_slots * R * 8});
            v.push_back({pk_.snap, (size_t)tw.size() * pk_.n_slots * R * 8});
        } else {
            const size_t n = (size_t)R * L * pl_.N;
            v.push_back({pl_.s, n});
            v.push_back({pl_.snap, tw.size() * n});
        }
        v.push_back({dC_, nC() * 8});
        v.push_back({dQ_, nQ() * 8});
        v.push_back({dE_, nE() * 8});
        if (n_bins) {
            v.push_back({wC_, nwC() * 8});
            v.push_back({wQ_, nwQ() * 8});
            v.push_back({wE_, nwE() * 8});
        }
        return v;
    }

private:
    // words of the configuration copied at a time (64 MB bounds the workspace for it)
    int64_t spin_part() const { return std::min<int64_t>((int64_t)(spins_bytes() / 8), (int64_t)8 << 20); }
    size_t nC() const { return (size_t)n_inst * R * Lc_ * tw.size() * tm.size(); }
    size_t nQ() const { return (size_t)n_inst * (R / 2) * Lc_ * tm.size(); }
    size_t nE() const { return (size_t)n_inst * R * Lc_ * tm.size(); }
    size_t nmC() const { return (size_t)n_inst * R * Lc_ * tw.size(); }
    size_t nwC() const { return (size_t)n_inst * R * Lc_ * tw.size() * n_bins; }
    size_t nwQ() const { return (size_t)n_inst * (R / 2) * Lc_ * n_bins; }
    size_t nwE() const { return (size_t)n_inst * R * Lc_ * n_bins; }
    size_t nmQ() const { return (size_t)n_inst * (R / 2) * Lc_; }
    size_t nmE() const { return (size_t)n_inst * R * Lc_; }

    // C, q and E counts, which lie one after the other in the workspace, in one copy
    struct Counts {
        std::vector<int64_t> buf;
        const int64_t *c, *q, *e;
    };
    Counts read_counts(const int64_t* c, const int64_t* q, const int64_t* e, size_t n_e,
                       cudaStream_t st, const char* what) {
        Counts r;
        r.buf.resize((size_t)(e - c) + n_e);
        down(r.buf.data(), c, r.buf.size() * 8, st);
        check_cuda(cudaStreamSynchronize(st), what);
        r.c = r.buf.data();
        r.q = r.c + (q - c);
        r.e = r.c + (e - c);
        return r;
    }

    void down(void* dst, const void* src, size_t bytes, cudaStream_t st) {
        d2h_bytes += (int64_t)bytes;
        if (bytes) check_cuda(cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDeviceToHost, st), "D2H copy");
    }

    void carve(Carver& c) {
        clock_dev = c.take<uint32_t>(1);
        d_thr_ = c.take<uint32_t>(thr_.size());
        if (kernel_ == SG_VB_PACKED) {
            pk_.vinfo = c.take<uint32_t>(h_vinfo_.size());
            pk_.slice_base = c.take<uint32_t>(h_slice_base_.size());
            pk_.slice_graph = c.take<uint32_t>(h_slice_graph_.size());
            pk_.col = c.take<uint32_t>(h_col_.size());
            pk_.slice_meta = c.take<uint4>(h_slice_meta_.size());
            pk_.err = c.take<int>(1);
            pk_.gbar = c.take<uint32_t>(2);
            pk_.claims = c.take<uint32_t>((size_t)kVbClaimGroups * 2 * kVbMaxColours);
            rs_.graph_class_slice = c.take<uint32_t>(graph_class_slice_.size());
            pk_.class_slice = c.take<uint32_t>(colour_slice_.size());
            // of the 129 MB L2 about 96 MB for graph and spins together
            pk_.far_beyond_l2 = (size_t)n_slots_ * 8 * R > ((size_t)176 << 20);
            pk_.stream_first = h_col_.size() * 12 + (size_t)n_slots_ * (4 + 8 * R) > ((size_t)96 << 20);
            pk_.jb = c.take<uint64_t>(h_jb_.size());
            pk_.seeds = c.take<uint64_t>(n_inst);
            pk_.up_slice_base = c.take<uint32_t>(h_up_base_.size());
            pk_.up_row_slice = c.take<uint32_t>(up_entries_ / 32);
            pk_.up_rows = (uint32_t)(up_entries_ / 32);
            pk_.up_col = c.take<uint32_t>(up_entries_);
            pk_.up_jb = c.take<uint64_t>(up_entries_);
            pk_.S = c.take<uint64_t>((size_t)n_slots_ * R);
            pk_.snap = c.take<uint64_t>((size_t)n_slots_ * R * tw.size());
            d_spins_ = c.take<uint64_t>((size_t)spin_part());
            d_graph_words_ = c.take<int64_t>((size_t)n_inst + 1);
            pk_.thr = d_thr_;
            pk_.n_slots = n_slots_;
            pk_.n_slices = (int32_t)(n_slots_ / 32);
            pk_.R = R;
            pk_.n_graphs = n_inst;
            pk_.max_width = max_width_;
            pk_.n_rows = (uint32_t)(h_col_.size() / 32);
            pk_.n_colours = (int32_t)colour_slice_.size() - 1;
            // SG_TEST_STAGE_WAIT_NS shortens the waits at the grid-wide barrier: a test of the timeout
            // path (the kernel gives up, flags SG_ETIMEOUT and exits cleanly)
            pk_.stage_wait_ns = 2000000000ull;
            if (const char* w = getenv("SG_TEST_STAGE_WAIT_NS")) pk_.stage_wait_ns = strtoull(w, nullptr, 10);
            if (pk_.n_colours > kVbMaxColours) fail(SG_EINVAL, "more colour classes than supported");
        } else {
            const Graph& g = graphs_[0];
            pl_.row_ptr = c.take<int32_t>(h_row_ptr_.size());
            pl_.col = c.take<int32_t>(h_col_i_.size());
            pl_.jb = c.take<uint64_t>(h_jb_.size());
            pl_.orig = c.take<uint32_t>(h_orig_.size());
            pl_.s = c.take<int8_t>((size_t)R * L * g.n);
            pl_.snap = c.take<int8_t>((size_t)R * L * g.n * tw.size());
            pl_.thr = d_thr_;
            pl_.seed = g.seed;
            pl_.N = g.n;
            pl_.R = R;
            pl_.L = L;
        }
        dC_ = c.take<int64_t>(nC());
        dQ_ = c.take<int64_t>(nQ());
        dE_ = c.take<int64_t>(nE());
        mC_ = c.take<int64_t>(nmC());
        mQ_ = c.take<int64_t>(nmQ());
        mE_ = c.take<int64_t>(nmE());
        wC_ = c.take<int64_t>(nwC());
        wQ_ = c.take<int64_t>(nwQ());
        wE_ = c.take<int64_t>(nwE());
    }

    // colour-major CSR of the single graph (plain kernel)
    void build_plain() {
        const Graph& g = graphs_[0];
        const int32_t n = g.n;
        colour_begin_.assign(g.n_colours + 1, 0);
        for (int32_t i = 0; i < n; ++i) colour_begin_[g.colour[i] + 1]++;
        for (int c = 0; c < g.n_colours; ++c) colour_begin_[c + 1] += colour_begin_[c];
        std::vector<int32_t> cursor(colour_begin_.begin(), colour_begin_.end() - 1);
        new_of_.assign(n, 0);
        h_orig_.assign(n, 0);
        for (int32_t i = 0; i < n; ++i) {
            const int32_t nv = cursor[g.colour[i]]++;
            new_of_[i] = nv;
            h_orig_[nv] = (uint32_t)i;
        }
        h_row_ptr_.assign(n + 1, 0);
        for (int32_t nv = 0; nv < n; ++nv) {
            const int32_t i = (int32_t)h_orig_[nv];
            h_row_ptr_[nv + 1] = h_row_ptr_[nv] + (g.row_ptr[i + 1] - g.row_ptr[i]);
        }
        h_col_i_.resize(g.col.size());
        h_jb_.resize(g.col.size());
        for (int32_t nv = 0; nv < n; ++nv) {
            const int32_t i = (int32_t)h_orig_[nv];
            int32_t o = h_row_ptr_[nv];
            for (int32_t e = g.row_ptr[i]; e < g.row_ptr[i + 1]; ++e, ++o) {
                h_col_i_[o] = new_of_[g.col[e]];
                h_jb_[o] = g.jb[e];
            }
        }
    }

    // sliced-ELL over slots ordered by (colour, graph, degree descending, original label)
    void build_packed() {
        int cmax = 0;
        for (const Graph& g : graphs_) cmax = std::max(cmax, g.n_colours);
        slot_of_.resize(n_inst);
        for (int b = 0; b < n_inst; ++b) slot_of_[b].assign(graphs_[b].n, -1);
        // bucket vertices by (colour, degree) per graph, in original-label order
        std::vector<std::vector<std::vector<int32_t>>> bucket(n_inst);
        for (int b = 0; b < n_inst; ++b) {
            const Graph& g = graphs_[b];
            bucket[b].assign((size_t)g.n_colours * (SG_VB_MAX_DEGREE + 1), {});
            for (int32_t i = 0; i < g.n; ++i) {
                const int d = g.row_ptr[i + 1] - g.row_ptr[i];
                bucket[b][(size_t)g.colour[i] * (SG_VB_MAX_DEGREE + 1) + d].push_back(i);
            }
        }
        int64_t cursor = 0;
        colour_slice_.assign(cmax + 1, 0);
        std::vector<int32_t> slot_graph_vertex;  // original label per slot, -1 for padding
        std::vector<int32_t> slot_graph;
        for (int c = 0; c < cmax; ++c) {
            colour_slice_[c] = (uint32_t)(cursor / 32);
            for (int b = 0; b < n_inst; ++b) {
                const Graph& g = graphs_[b];
                graph_class_slice_.push_back((uint32_t)(cursor / 32));
                if (c >= g.n_colours) continue;
                const int64_t start = cursor;
                // highest degree first: the longest slices start early instead of forming the tail
                for (int d = SG_VB_MAX_DEGREE; d >= 0; --d)
                    for (int32_t i : bucket[b][(size_t)c * (SG_VB_MAX_DEGREE + 1) + d]) {
                        slot_of_[b][i] = cursor++;
                        slot_graph_vertex.push_back(i);
                        slot_graph.push_back(b);
                    }
                if (cursor == start) continue;
                while (cursor % 32) {
                    ++cursor;
                    slot_graph_vertex.push_back(-1);
                    slot_graph.push_back(b);
                }
            }
        }
        colour_slice_[cmax] = (uint32_t)(cursor / 32);
        graph_class_slice_.push_back((uint32_t)(cursor / 32));
        for (int c = 0; c < cmax; ++c)
            max_class_slices_ = std::max(max_class_slices_, (int)(colour_slice_[c + 1] - colour_slice_[c]));
        n_slots_ = cursor;
        const int64_t n_slices = n_slots_ / 32;
        h_vinfo_.assign(n_slots_, kInactive);
        h_slice_graph_.assign(n_slices, 0);
        h_slice_base_.assign(n_slices + 1, 0);
        std::vector<int32_t> width_of(n_slices, 0);
        parallel_ranges(n_slices, [&](int64_t s0, int64_t s1) {
            for (int64_t s = s0; s < s1; ++s) {
                const int b = slot_graph[s * 32];
                h_slice_graph_[s] = (uint32_t)b;
                const Graph& g = graphs_[b];
                int width = 0;
                for (int l = 0; l < 32; ++l) {
                    const int32_t i = slot_graph_vertex[s * 32 + l];
                    if (i < 0) continue;
                    const int d = g.row_ptr[i + 1] - g.row_ptr[i];
                    width = std::max(width, d);
                    h_vinfo_[s * 32 + l] = (uint32_t)i | ((uint32_t)d << kDegShift);
                }
                width_of[s] = width;
            }
        });
        int64_t entries = 0;
        for (int64_t s = 0; s < n_slices; ++s) {
            max_width_ = std::max(max_width_, (uint32_t)width_of[s]);
            h_slice_base_[s] = (uint32_t)entries;
            entries += 32 * (int64_t)width_of[s];
            if (entries >= (int64_t(1) << 32)) fail(SG_EINVAL, "too many graph entries for one batch");
        }
        h_slice_base_[n_slices] = (uint32_t)entries;
        h_col_.assign(entries, 0);
        h_jb_.assign(entries, 0);
        // every slice writes only its own entries
        parallel_ranges(n_slices, [&](int64_t s0, int64_t s1) {
            for (int64_t s = s0; s < s1; ++s) {
                const int b = (int)h_slice_graph_[s];
                const Graph& g = graphs_[b];
                const int64_t base = h_slice_base_[s];
                const int width = (int)((h_slice_base_[s + 1] - base) / 32);
                for (int l = 0; l < 32; ++l) {
                    const int64_t slot = s * 32 + l;
                    const int32_t i = slot_graph_vertex[slot];
                    int e = 0;
                    if (i >= 0)
                        for (int32_t k = g.row_ptr[i]; k < g.row_ptr[i + 1]; ++k, ++e) {
                            h_col_[base + (int64_t)e * 32 + l] = (uint32_t)slot_of_[b][g.col[k]];
                            h_jb_[base + (int64_t)e * 32 + l] = g.jb[k];
                        }
                    for (; e < width; ++e) {
                        h_col_[base + (int64_t)e * 32 + l] = (uint32_t)slot;
                        h_jb_[base + (int64_t)e * 32 + l] = 0;
                    }
                }
            }
        });
        // upper entries (energy measurement): neighbours in later colour classes only
        h_up_base_.assign(n_slices + 1, 0);
        std::vector<int32_t> up_width(n_slices, 0);
        parallel_ranges(n_slices, [&](int64_t s0, int64_t s1) {
            for (int64_t s = s0; s < s1; ++s) {
                const int b = (int)h_slice_graph_[s];
                const Graph& g = graphs_[b];
                int w = 0;
                for (int l = 0; l < 32; ++l) {
                    const int64_t slot = s * 32 + l;
                    const int32_t i = slot_graph_vertex[slot];
                    if (i < 0) continue;
                    int n_up = 0;
                    for (int32_t k = g.row_ptr[i]; k < g.row_ptr[i + 1]; ++k)
                        n_up += slot_of_[b][g.col[k]] > slot;
                    w = std::max(w, n_up);
                }
                up_width[s] = w;
            }
        });
        int64_t up_entries = 0;
        for (int64_t s = 0; s < n_slices; ++s) {
            h_up_base_[s] = (uint32_t)up_entries;
            up_entries += 32 * (int64_t)up_width[s];
        }
        h_up_base_[n_slices] = (uint32_t)up_entries;
        up_entries_ = up_entries;  // filled on the device at attach (vb_packed_build_upper)
        h_slice_meta_.resize(n_slices);
        for (int64_t s = 0; s < n_slices; ++s) {
            uint4 m;
            m.x = h_slice_base_[s];
            m.y = (h_slice_base_[s + 1] - h_slice_base_[s]) / 32;
            m.z = h_slice_graph_[s];
            m.w = 0;
            h_slice_meta_[s] = m;
        }
    }

    int kernel_ = SG_VB_PACKED;
    enum Form { kGrid, kResident };
    Form form_ = kGrid;         // vb_sweep.cu or vb_resident.cu, chosen at attach
    int max_class_slices_ = 0;  // slices of the largest class
    uint32_t max_width_ = 0;    // entries of the widest slice
    VbResident rs_{};
    std::vector<uint32_t> graph_class_slice_;  // first slice of every (class, graph)
    int Lc_ = 64;
    size_t ws_bytes_ = 0;
    std::vector<Graph> graphs_;
    std::vector<uint32_t> thr_;
    // packed host layout
    std::vector<uint32_t> colour_slice_;
    std::vector<uint4> h_slice_meta_;
    std::vector<std::vector<int64_t>> slot_of_;
    int64_t n_slots_ = 0;
    std::vector<uint32_t> h_slice_base_, h_slice_graph_;
    pinned_vector<uint32_t> h_vinfo_, h_col_;  // the large images copied at attach: page-locked
    pinned_vector<uint64_t> h_jb_;
    std::vector<uint32_t> h_up_base_;  // upper entries (energy measurement): slice bases
    int64_t up_entries_ = 0;
    // plain host layout
    std::vector<int32_t> colour_begin_, new_of_, h_row_ptr_, h_col_i_;
    std::vector<uint32_t> h_orig_;
    // device views
    VbPackedDev pk_{};
    VbPlainDev pl_{};
    uint32_t* d_thr_ = nullptr;
    uint64_t* d_spins_ = nullptr;       // a part of the configuration in the caller's order
    int64_t* d_graph_words_ = nullptr;  // [n_graphs + 1] first word of each graph in it
    int64_t *dC_ = nullptr, *dQ_ = nullptr, *dE_ = nullptr;
    int64_t *mC_ = nullptr, *mQ_ = nullptr, *mE_ = nullptr;
    int64_t *wC_ = nullptr, *wQ_ = nullptr, *wE_ = nullptr;  // window sums of raw counts
};

}  // namespace

Model* make_vb_model(const void* graphs, int n_graphs, int n_lanes, int n_replicas, int kernel,
                     const std::vector<int64_t>& tw, const std::vector<int64_t>& tm) {
    return new VbModel(static_cast<const sg_vb_graph*>(graphs), n_graphs, n_lanes, n_replicas,
                       kernel, tw, tm);
}

}  // namespace sg
