// Batched evaluation: many problems per sweep launch, optionally replayed as a CUDA graph.
//
// Problems of one shape (levels, subsystems), solver, kernel family and tile size (threads)
// form a group; a group's sweep launch takes the concatenation of its problems' tile lists (each
// tile names its problem), so problems of different durations and window counts share every
// wave of the GPU instead of each filling a fraction of it, and no tile runs with more threads
// than its own problem's.  The groups' launches of one sweep run concurrently, each on a stream
// of its own forked from the caller's stream and joined back.  The per-problem steps (controls,
// terminal conditions, final reductions) stay per problem.  With MSQOC_BATCH_GRAPH the whole sequence is captured once
// into a CUDA graph and replayed; every buffer it touches belongs to the problems and stays
// where it is, so replays only need the problems' inputs staged with msqoc_set_inputs.
#include <algorithm>
#include <new>
#include <vector>

#include "msqoc_host.h"

using namespace msqoc;

struct msqoc_batch {
    struct Group {
        int L = 0, q = 0, solver = 0, pair = 0, lean = 0;   // shape, solver and kernel family of the group
        int nthreads = 0;                          // threads of its tiles
        int pthreads = 0, plean = 0;               // propagator tiles (0: no member is sliced)
        std::vector<int> members;     // indices into probs
        SweepArgs pargs{};            // the members' propagator sweep
        int nptiles = 0, E_max = 1, M_max = 1;
        Tile* ptiles = nullptr;
        int* plmap = nullptr;
        std::vector<Tile> host_ptiles;
        std::vector<int> pfirst, pcount;      // per member: its tiles in host_ptiles
        Tile* slot_ptiles[MSQOC_BATCH_SLOTS] = {};
        Tile* slot_phost[MSQOC_BATCH_SLOTS] = {};
        SweepArgs args{};             // pds / tiles / lanemap / geometry of the group's launches
        int ntiles = 0;
        int nseg_max = 1, nsub_max = 1;
        long slots = 1;               // tiles the GPU holds at a time
        int qmode = 0;                // the members' form of the gradient products (QuadArgs::mode)
        int quad_blocks = 0;          // blocks of a row of the quadrature launch: the most of the members
        ProbDev* pds = nullptr;
        Tile* tiles = nullptr;
        int* lanemap = nullptr;
        std::vector<Tile> host_tiles;         // the group's tiles, longest windows first
        std::vector<int> first, count;        // per member: its tiles in host_tiles (by member k)
        Tile* slot_tiles[MSQOC_BATCH_SLOTS] = {};   // per slot: the tiles of a subset evaluation
        Tile* slot_host[MSQOC_BATCH_SLOTS] = {};    // pinned staging of those tiles
        int* slot_list[MSQOC_BATCH_SLOTS] = {};     // per slot: the subset's members (rows of the
        int* slot_lhost[MSQOC_BATCH_SLOTS] = {};    // quadrature launch), and their pinned staging
    };
    std::vector<msqoc_problem*> probs;
    std::vector<int> group_of, member_of;   // per problem: its group and index within it
    std::vector<Group> groups;
    int flags = 0;
    int device = 0;
    cudaStream_t cap = nullptr;                   // capture stream (graph mode)
    cudaGraphExec_t exec[2] = {nullptr, nullptr};  // [objective, gradient]
    cudaEvent_t slot_done[MSQOC_BATCH_SLOTS] = {};  // the slot's staging copies have been read
    // per stream set (one per subset slot, the last for whole-batch evaluations): the groups'
    // streams, the fork event on the caller's stream and each group's join event
    std::vector<cudaStream_t> gstream[MSQOC_BATCH_SLOTS + 1];
    std::vector<cudaEvent_t> gjoin[MSQOC_BATCH_SLOTS + 1];
    cudaEvent_t gfork[MSQOC_BATCH_SLOTS + 1] = {};
};

namespace {

int ipow(int b, int e) {
    int r = 1;
    while (e-- > 0) r *= b;
    return r;
}

void free_batch(msqoc_batch* b) {
    for (auto& g : b->groups) {
        if (g.pds) cudaFree(g.pds);
        if (g.tiles) cudaFree(g.tiles);
        if (g.lanemap) cudaFree(g.lanemap);
        if (g.ptiles) cudaFree(g.ptiles);
        if (g.plmap) cudaFree(g.plmap);
        for (int k = 0; k < MSQOC_BATCH_SLOTS; ++k) {
            if (g.slot_tiles[k]) cudaFree(g.slot_tiles[k]);
            if (g.slot_host[k]) cudaFreeHost(g.slot_host[k]);
            if (g.slot_ptiles[k]) cudaFree(g.slot_ptiles[k]);
            if (g.slot_phost[k]) cudaFreeHost(g.slot_phost[k]);
            if (g.slot_list[k]) cudaFree(g.slot_list[k]);
            if (g.slot_lhost[k]) cudaFreeHost(g.slot_lhost[k]);
        }
    }
    for (auto& e : b->slot_done)
        if (e) cudaEventDestroy(e);
    for (int k = 0; k <= MSQOC_BATCH_SLOTS; ++k) {
        for (cudaStream_t gs : b->gstream[k])
            if (gs) cudaStreamDestroy(gs);
        for (cudaEvent_t e : b->gjoin[k])
            if (e) cudaEventDestroy(e);
        if (b->gfork[k]) cudaEventDestroy(b->gfork[k]);
    }
    for (auto& e : b->exec)
        if (e) cudaGraphExecDestroy(e);
    if (b->cap) cudaStreamDestroy(b->cap);
}

// One sweep of every group with tiles, each group's launches issued by launch(gi, stream): on
// the caller's stream s when at most one group has tiles, else concurrently on the groups'
// streams of stream set `set`, forked from s and joined back into it (both also under graph
// capture, where the fork and join become the graph's branches).
template <typename F>
msqoc_status for_groups(msqoc_batch* b, const int* ntiles, int set, cudaStream_t s, F&& launch) {
    const int ng = static_cast<int>(b->groups.size());
    int active = 0;
    for (int gi = 0; gi < ng; ++gi) active += ntiles[gi] > 0;
    if (active <= 1 || b->gstream[set].empty()) {
        for (int gi = 0; gi < ng; ++gi)
            if (ntiles[gi] > 0) CUDA_TRY(launch(gi, s));
        return MSQOC_OK;
    }
    CUDA_TRY(cudaEventRecord(b->gfork[set], s));
    for (int gi = 0; gi < ng; ++gi) {
        if (ntiles[gi] <= 0) continue;
        cudaStream_t gs = b->gstream[set][gi];
        CUDA_TRY(cudaStreamWaitEvent(gs, b->gfork[set], 0));
        CUDA_TRY(launch(gi, gs));
        CUDA_TRY(cudaEventRecord(b->gjoin[set][gi], gs));
        CUDA_TRY(cudaStreamWaitEvent(s, b->gjoin[set][gi], 0));
    }
    return MSQOC_OK;
}

// What one batched evaluation launches of a group: its tiles, its propagator tiles and its members
// (list: device array, nullptr for every member in order).
struct GroupWork {
    Tile* tiles = nullptr;
    Tile* ptiles = nullptr;
    int* list = nullptr;
    int ntiles = 0, nptiles = 0, nlist = 0;
};
// The history (or a segment's recomputation) and the adjoint sweep of n tiles each in one launch:
// always for slices; for segments where that takes fewer waves (4 transmons, 16 windows, checkpoints
// every 64 steps: one problem 11.7 -> 7.9 ms, but four, whose tiles fill the GPU, 15.0 -> 15.2).
bool both_sweeps(const msqoc_batch::Group& g, long n) {
    if (g.nsub_max != 1 || g.pair != 0 || g.solver != SOLVER_MIXED) return false;
    auto waves = [&](long t) { return (t + g.slots - 1) / g.slots; };
    return g.pthreads || (g.nseg_max > 1 && waves(2 * n) < 2 * waves(n));
}
// fn(pds, list, n) for the n members of a launch whose rows are problems, in parts of what a grid's y and z
// dimensions hold
template <class Fn>
cudaError_t in_rows(const ProbDev* pds, const int* list, int n, Fn fn) {
    constexpr int most = 65535;
    for (int i = 0; i < n; i += most) {
        const cudaError_t e = fn(list ? pds : pds + i, list ? list + i : nullptr, std::min(n - i, most));
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}
// The launch sequence of one batched evaluation of the problems `sel`; work[g]: the part of group g;
// set: the stream set of the groups.
msqoc_status enqueue(msqoc_batch* b, const std::vector<msqoc_problem*>& sel, const std::vector<GroupWork>& work,
                     bool grad, int set, cudaStream_t s) {
    std::vector<int> ntiles;
    for (const GroupWork& w : work) ntiles.push_back(w.ntiles);
    auto compose = [&](int gi, bool bwd, cudaStream_t gs) {
        const auto& g = b->groups[gi];
        return in_rows(g.pds, work[gi].list, work[gi].nlist, [&](const ProbDev* pds, const int* list, int n) {
            return launch_compose(pds, list, g.E_max, g.M_max, n, ipow(g.L, g.q), bwd, gs);
        });
    };
    msqoc_status st;
    for (msqoc_problem* p : sel)
        if ((st = launch_controls(p, p->pd.pair, s))) return st;
    st = for_groups(b, ntiles.data(), set, s, [&](int gi, cudaStream_t gs) {
        const auto& g = b->groups[gi];
        if (g.pthreads) {
            SweepArgs pa = g.pargs;
            pa.tiles = work[gi].ptiles;
            cudaError_t e = launch_sweep(pa, work[gi].nptiles, gs);
            if (e == cudaSuccess)
                e = compose(gi, false, gs);
            if (e != cudaSuccess) return e;
        }
        if (g.pthreads && (!grad || g.nsub_max == 1)) return cudaSuccess;   // (history: with the adjoint)
        SweepArgs a = g.args;
        a.tiles = work[gi].tiles;
        a.mode = grad ? SWEEP_HISTORY : SWEEP_OBJECTIVE;
        a.seg = 0;
        return launch_sweep(a, work[gi].ntiles, gs);
    });
    if (st) return st;
    for (msqoc_problem* p : sel)
        if ((st = launch_terminal(p, grad, s))) return st;
    if (!grad) {
        for (msqoc_problem* p : sel) {
            double* o = p->out_dev;
            if ((st = launch_objective_outputs(p, o, o + 1, o + 2, s))) return st;
        }
        return MSQOC_OK;
    }
    st = for_groups(b, ntiles.data(), set, s, [&](int gi, cudaStream_t gs) {
        const auto& g = b->groups[gi];
        if (g.pthreads) {
            const cudaError_t e = compose(gi, true, gs);
            if (e != cudaSuccess) return e;
        }
        const bool both = both_sweeps(g, work[gi].ntiles);
        for (int seg = g.nseg_max - 1; seg >= 0; --seg) {
            SweepArgs a = g.args;
            a.tiles = work[gi].tiles;
            a.seg = seg;
            if (g.nseg_max > 1 && !both) {
                a.mode = SWEEP_RECOMPUTE;
                const cudaError_t e = launch_sweep(a, work[gi].ntiles, gs);
                if (e != cudaSuccess) return e;
            }
            for (int sub = g.nsub_max - 1; sub >= 0; --sub) {
                a.mode = both ? SWEEP_BOTH : SWEEP_ADJOINT;
                a.sub = sub;
                cudaError_t e = launch_sweep(a, work[gi].ntiles, gs);
                if (e != cudaSuccess) return e;
                QuadArgs qa = quad_args(b->probs[g.members[0]]->pd, g.pds, seg, sub);
                e = in_rows(g.pds, work[gi].list, work[gi].nlist, [&](const ProbDev* pds, const int* list, int n) {
                    qa.pds = pds;
                    qa.list = list;
                    return launch_quad(qa, g.quad_blocks, n, gs);
                });
                if (e != cudaSuccess) return e;
            }
        }
        return cudaSuccess;
    });
    if (st) return st;
    for (msqoc_problem* p : sel) {
        const OutLayout ol = out_layout(p->npen, p->pd.d, p->nW);
        double* o = p->out_dev;
        if ((st = launch_gradient_outputs(p, o, o + ol.ga, p->pd.M > 1 ? o + ol.gw : nullptr, s))) return st;
    }
    return MSQOC_OK;
}

msqoc_status enqueue_all(msqoc_batch* b, bool grad, cudaStream_t s) {
    std::vector<GroupWork> work;
    for (auto& g : b->groups)
        work.push_back(GroupWork{g.tiles, g.ptiles, nullptr, g.ntiles, g.nptiles, static_cast<int>(g.members.size())});
    return enqueue(b, b->probs, work, grad, MSQOC_BATCH_SLOTS, s);
}

msqoc_status eval(msqoc_batch* b, bool grad, cudaStream_t s) {
    if (grad && !(b->flags & MSQOC_BATCH_GRADIENT))
        return fail(MSQOC_ERR_INVALID_ARG, "batch was created without MSQOC_BATCH_GRADIENT");
    if (!(b->flags & MSQOC_BATCH_GRAPH)) return enqueue_all(b, grad, s);
    cudaGraphExec_t& ex = b->exec[grad ? 1 : 0];
    if (!ex) {
        // capture on a private stream; the first replay below runs it
        CUDA_TRY(cudaStreamBeginCapture(b->cap, cudaStreamCaptureModeRelaxed));
        const msqoc_status st = enqueue_all(b, grad, b->cap);
        cudaGraph_t graph = nullptr;
        const cudaError_t e = cudaStreamEndCapture(b->cap, &graph);
        if (st) {
            if (graph) cudaGraphDestroy(graph);
            return st;
        }
        CUDA_TRY(e);
        const cudaError_t ei = cudaGraphInstantiate(&ex, graph, 0);
        cudaGraphDestroy(graph);
        CUDA_TRY(ei);
    }
    CUDA_TRY(cudaGraphLaunch(ex, s));
    return MSQOC_OK;
}

// frees a batch under construction unless released
struct BatchOwner {
    msqoc_batch* b = nullptr;
    ~BatchOwner() {
        if (b) {
            free_batch(b);
            delete b;
        }
    }
};

msqoc_status batch_create(msqoc_problem* const* problems, int32_t n, int32_t flags, msqoc_batch** out) {
    if (!out) return fail(MSQOC_ERR_INVALID_ARG, "out is NULL");
    *out = nullptr;
    if (!problems || n < 1) return fail(MSQOC_ERR_INVALID_ARG, "no problems");
    if (flags & ~(MSQOC_BATCH_GRADIENT | MSQOC_BATCH_GRAPH)) return fail(MSQOC_ERR_INVALID_ARG, "unknown flags %d", flags);
    int dev = 0;
    CUDA_TRY(cudaGetDevice(&dev));
    for (int i = 0; i < n; ++i) {
        if (!problems[i]) return fail(MSQOC_ERR_INVALID_ARG, "problem %d is NULL", i);
        if (problems[i]->device != dev) return fail(MSQOC_ERR_INVALID_ARG, "problem %d lives on another device", i);
        if (is_shard(problems[i]->pd))
            return fail(MSQOC_ERR_UNSUPPORTED, "problem %d is a window range; batches take whole problems", i);
        for (int j = 0; j < i; ++j)
            if (problems[j] == problems[i]) return fail(MSQOC_ERR_INVALID_ARG, "problem %d appears twice", i);
    }
    BatchOwner owner{new (std::nothrow) msqoc_batch()};
    msqoc_batch* b = owner.b;
    if (!b) return fail(MSQOC_ERR_OUT_OF_MEMORY, "host allocation failed");
    b->flags = flags;
    b->device = dev;
    b->probs.assign(problems, problems + n);
    msqoc_status st = MSQOC_OK;
    // the history buffers first: the problems' device records then hold their final pointers
    if (flags & MSQOC_BATCH_GRADIENT)
        for (msqoc_problem* p : b->probs)
            if (!st) st = ensure_gradient_buffers(p, nullptr);
    if (!st && cudaDeviceSynchronize() != cudaSuccess) st = fail(MSQOC_ERR_CUDA, "synchronize failed");
    // groups by (levels, subsystems, solver, kernel family, tile threads, propagator tiles, form of the
    // gradient products: a member's results do not depend on the others)
    for (int i = 0; i < n && !st; ++i) {
        const ProbDev& pd = b->probs[i]->pd;
        const int qmode = flags & MSQOC_BATCH_GRADIENT ? quad_args(pd, nullptr, 0, 0).mode : 0;
        auto it = std::find_if(b->groups.begin(), b->groups.end(), [&](const msqoc_batch::Group& g) {
            return g.L == pd.L && g.q == pd.q && g.solver == pd.solver && g.pair == pd.pair && g.lean == pd.lean &&
                   g.nthreads == pd.nthreads && g.pthreads == b->probs[i]->prop.nthreads &&
                   g.plean == b->probs[i]->prop.lean && g.qmode == qmode;
        });
        if (it == b->groups.end()) {
            b->groups.emplace_back();
            it = b->groups.end() - 1;
            it->L = pd.L;
            it->q = pd.q;
            it->solver = pd.solver;
            it->pair = pd.pair;
            it->lean = pd.lean;
            it->nthreads = pd.nthreads;
            it->pthreads = b->probs[i]->prop.nthreads;
            it->plean = b->probs[i]->prop.lean;
            it->qmode = qmode;
        }
        it->members.push_back(i);
    }
    b->group_of.assign(n, 0);
    b->member_of.assign(n, 0);
    for (size_t gi = 0; gi < b->groups.size(); ++gi)
        for (size_t k = 0; k < b->groups[gi].members.size(); ++k) {
            b->group_of[b->groups[gi].members[k]] = static_cast<int>(gi);
            b->member_of[b->groups[gi].members[k]] = static_cast<int>(k);
        }
    for (auto& g : b->groups) {
        if (st) break;
        int nthreads = 32, cpt = 1, gmax = 1;
        for (int i : g.members) {
            const ProbDev& pd = b->probs[i]->pd;
            nthreads = std::max(nthreads, pd.nthreads);
            cpt = std::max(cpt, pd.cb);
            gmax = std::max(gmax, pd.glocal);
            g.nseg_max = std::max(g.nseg_max, pd.nseg);
            g.nsub_max = std::max(g.nsub_max, pd.nsub);
            g.quad_blocks = std::max(g.quad_blocks, quad_blocks(pd));
        }
        std::vector<ProbDev> pds;
        std::vector<Tile> tiles, ptiles;
        std::vector<int> maps, pmaps;
        SweepPlan plan{0, g.pthreads, g.plean, 0};
        // a member's tiles and lane maps (V windows of E columns) behind those of the others
        auto append = [](std::vector<Tile>& ts, std::vector<int>& ms, const ProbDev& pd, int k, int V, int E, int cb,
                         int nt, int pair) {
            const int map_base = static_cast<int>(ms.size() / nt);
            const int n = static_cast<int>(tile_count(V, E, cb));
            for (int t = 0; t < n; ++t) {
                Tile x = tile_at(t, V, E, cb, k);
                x.map += map_base;
                ts.push_back(x);
            }
            const Tile last = tile_at(n - 1, V, E, cb, 0);
            ms.resize(ms.size() + size_t(cb + 1) * nt);
            int* mp = ms.data() + size_t(map_base) * nt;
            for (int j = 0; j <= cb; ++j)
                build_lanemap(pd.L, pd.q, j < cb ? cb : last.ncol, j < cb ? j + 1 : last.ncol0, nt, pair,
                              mp + size_t(j) * nt);
            return n;
        };
        for (size_t k = 0; k < g.members.size(); ++k) {
            const ProbDev& pd = b->probs[g.members[k]]->pd;
            const msqoc_problem* pr = b->probs[g.members[k]];
            g.first.push_back(static_cast<int>(tiles.size()));
            g.count.push_back(append(tiles, maps, pd, static_cast<int>(k), pd.M * pd.C, pd.E, pd.cb, nthreads, pd.pair));
            g.E_max = std::max(g.E_max, pd.E);
            g.M_max = std::max(g.M_max, pd.M);
            if (g.pthreads) {
                g.pfirst.push_back(static_cast<int>(ptiles.size()));
                g.pcount.push_back(append(ptiles, pmaps, pd, static_cast<int>(k), pd.M * pd.C, pd.N, pr->prop.cpt,
                                          g.pthreads, 0));
                plan.cpt = std::max(plan.cpt, pr->prop.cpt);
            }
            pds.push_back(pd);
        }
        // longest windows first: the CTAs that take longest start in the first wave
        auto tile_len = [&](const Tile& x) {
            const ProbDev& pd = b->probs[g.members[x.prob]]->pd;
            return (pd.nsteps + pd.M * pd.C - 1) / (pd.M * pd.C);
        };
        g.host_ptiles = ptiles;
        std::stable_sort(ptiles.begin(), ptiles.end(), [&](const Tile& x, const Tile& y) { return tile_len(x) > tile_len(y); });
        g.nptiles = static_cast<int>(ptiles.size());
        g.host_tiles = tiles;
        std::stable_sort(tiles.begin(), tiles.end(), [&](const Tile& x, const Tile& y) { return tile_len(x) > tile_len(y); });
        g.ntiles = static_cast<int>(tiles.size());
        cudaError_t e = cudaMalloc(reinterpret_cast<void**>(&g.pds), pds.size() * sizeof(ProbDev));
        if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void**>(&g.tiles), tiles.size() * sizeof(Tile));
        if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void**>(&g.lanemap), maps.size() * sizeof(int));
        if (e == cudaSuccess) e = cudaMemcpy(g.pds, pds.data(), pds.size() * sizeof(ProbDev), cudaMemcpyHostToDevice);
        if (e == cudaSuccess) e = cudaMemcpy(g.tiles, tiles.data(), tiles.size() * sizeof(Tile), cudaMemcpyHostToDevice);
        if (e == cudaSuccess) e = cudaMemcpy(g.lanemap, maps.data(), maps.size() * sizeof(int), cudaMemcpyHostToDevice);
        if (g.pthreads) {
            if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void**>(&g.ptiles), ptiles.size() * sizeof(Tile));
            if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void**>(&g.plmap), pmaps.size() * sizeof(int));
            if (e == cudaSuccess) e = cudaMemcpy(g.ptiles, ptiles.data(), ptiles.size() * sizeof(Tile), cudaMemcpyHostToDevice);
            if (e == cudaSuccess) e = cudaMemcpy(g.plmap, pmaps.data(), pmaps.size() * sizeof(int), cudaMemcpyHostToDevice);
        }
        for (int k = 0; k < MSQOC_BATCH_SLOTS && e == cudaSuccess; ++k) {
            if (g.pthreads) {
                e = cudaMalloc(reinterpret_cast<void**>(&g.slot_ptiles[k]), ptiles.size() * sizeof(Tile));
                if (e == cudaSuccess) e = cudaMallocHost(reinterpret_cast<void**>(&g.slot_phost[k]), ptiles.size() * sizeof(Tile));
                if (e != cudaSuccess) break;
            }
            e = cudaMalloc(reinterpret_cast<void**>(&g.slot_tiles[k]), tiles.size() * sizeof(Tile));
            if (e == cudaSuccess) e = cudaMallocHost(reinterpret_cast<void**>(&g.slot_host[k]), tiles.size() * sizeof(Tile));
            if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void**>(&g.slot_list[k]), g.members.size() * sizeof(int));
            if (e == cudaSuccess) e = cudaMallocHost(reinterpret_cast<void**>(&g.slot_lhost[k]), g.members.size() * sizeof(int));
        }
        if (e != cudaSuccess) {
            st = fail(e == cudaErrorMemoryAllocation ? MSQOC_ERR_OUT_OF_MEMORY : MSQOC_ERR_CUDA, "batch tables: %s",
                      cudaGetErrorString(e));
            break;
        }
        const ProbDev& p0 = b->probs[g.members[0]]->pd;
        g.args = sweep_args(p0, g.pds, g.tiles, g.lanemap, SWEEP_OBJECTIVE, 0);
        // one history depth for the launch: the smallest of the members' (it always fits)
        for (int mi : g.members) g.args.hdepth = std::min(g.args.hdepth, b->probs[mi]->pd.hdepth);
        g.args.cpt = cpt;
        g.args.gmax = gmax;
        g.args.nthreads = nthreads;
        if (g.pthreads) g.pargs = prop_args(plan, p0, g.pds, g.ptiles, g.plmap);
        SweepArgs adj = g.args;
        adj.mode = SWEEP_ADJOINT;
        int sms = 0;
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        g.slots = std::max<long>(1, long(sms) * sweep_ctas_per_sm(adj));
        SweepArgs both = g.args;
        both.mode = SWEEP_BOTH;
        if (admission_bytes(g.q, g.L, p0.N, cpt, nthreads, gmax, g.solver, g.pair, g.args.hdepth) > 227 * 1024) {
            st = fail(MSQOC_ERR_UNSUPPORTED, "batched tiles need too much shared memory");
            break;
        }
        // set the kernels' shared-memory limits now (a launch of no tiles only does that), so
        // that a graph capture later makes no attribute calls
        if (launch_sweep(g.args, 0, nullptr) != cudaSuccess || launch_sweep(adj, 0, nullptr) != cudaSuccess ||
            launch_quad(quad_args(p0, g.pds, 0, 0), 0, 0, nullptr) != cudaSuccess ||
            (g.pthreads && launch_sweep(g.pargs, 0, nullptr) != cudaSuccess) ||
            (both_sweeps(g, 1) && launch_sweep(both, 0, nullptr) != cudaSuccess))
            st = fail(MSQOC_ERR_CUDA, "sweep kernel attributes could not be set");
    }
    if (!st && (flags & MSQOC_BATCH_GRAPH) && cudaStreamCreateWithFlags(&b->cap, cudaStreamNonBlocking) != cudaSuccess)
        st = fail(MSQOC_ERR_CUDA, "capture stream creation failed");
    for (int k = 0; k < MSQOC_BATCH_SLOTS && !st; ++k)
        if (cudaEventCreateWithFlags(&b->slot_done[k], cudaEventDisableTiming) != cudaSuccess)
            st = fail(MSQOC_ERR_CUDA, "event creation failed");
    // the groups' streams and events (several groups only)
    const size_t ng = b->groups.size();
    for (int k = 0; k <= MSQOC_BATCH_SLOTS && !st && ng > 1; ++k) {
        b->gstream[k].assign(ng, nullptr);
        b->gjoin[k].assign(ng, nullptr);
        cudaError_t e = cudaEventCreateWithFlags(&b->gfork[k], cudaEventDisableTiming);
        for (size_t gi = 0; gi < ng && e == cudaSuccess; ++gi) {
            e = cudaStreamCreateWithFlags(&b->gstream[k][gi], cudaStreamNonBlocking);
            if (e == cudaSuccess) e = cudaEventCreateWithFlags(&b->gjoin[k][gi], cudaEventDisableTiming);
        }
        if (e != cudaSuccess) st = fail(MSQOC_ERR_CUDA, "group streams: %s", cudaGetErrorString(e));
    }
    if (st) return st;
    *out = b;
    owner.b = nullptr;
    return MSQOC_OK;
}

msqoc_status batch_eval_subset(msqoc_batch* b, const int32_t* members, int32_t n, int32_t gradient, int32_t slot,
                               void* stream) {
    if (!b || !members || n < 1) return fail(MSQOC_ERR_INVALID_ARG, "batch or members is NULL / empty");
    if (slot < 0 || slot >= MSQOC_BATCH_SLOTS) return fail(MSQOC_ERR_INVALID_ARG, "slot %d out of range", slot);
    if (gradient && !(b->flags & MSQOC_BATCH_GRADIENT))
        return fail(MSQOC_ERR_INVALID_ARG, "batch was created without MSQOC_BATCH_GRADIENT");
    const int np = static_cast<int>(b->probs.size());
    std::vector<char> seen(np, 0);
    for (int i = 0; i < n; ++i) {
        if (members[i] < 0 || members[i] >= np) return fail(MSQOC_ERR_INVALID_ARG, "member %d out of range", members[i]);
        if (seen[members[i]]++) return fail(MSQOC_ERR_INVALID_ARG, "member %d listed twice", members[i]);
    }
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    // the slot's staging buffers are rewritten only after its previous copies were read
    CUDA_TRY(cudaEventSynchronize(b->slot_done[slot]));
    std::vector<msqoc_problem*> sel;
    std::vector<GroupWork> work(b->groups.size());
    for (int i = 0; i < n; ++i) sel.push_back(b->probs[members[i]]);
    for (size_t gi = 0; gi < b->groups.size(); ++gi) {
        auto& g = b->groups[gi];
        GroupWork& w = work[gi];
        Tile* h = g.slot_host[slot];
        Tile* ph = g.slot_phost[slot];
        for (int i = 0; i < n; ++i) {
            if (b->group_of[members[i]] != static_cast<int>(gi)) continue;
            const int k = b->member_of[members[i]];
            std::copy(g.host_tiles.begin() + g.first[k], g.host_tiles.begin() + g.first[k] + g.count[k], h + w.ntiles);
            w.ntiles += g.count[k];
            if (g.pthreads) {
                std::copy(g.host_ptiles.begin() + g.pfirst[k], g.host_ptiles.begin() + g.pfirst[k] + g.pcount[k],
                          ph + w.nptiles);
                w.nptiles += g.pcount[k];
            }
            g.slot_lhost[slot][w.nlist++] = k;
        }
        if (!w.ntiles) continue;
        auto longer = [&](const Tile& x, const Tile& y) {
            auto len = [&](const Tile& t) {
                const ProbDev& pd = b->probs[g.members[t.prob]]->pd;
                return (pd.nsteps + pd.M * pd.C - 1) / (pd.M * pd.C);
            };
            return len(x) > len(y);
        };
        std::stable_sort(h, h + w.ntiles, longer);
        CUDA_TRY(cudaMemcpyAsync(g.slot_tiles[slot], h, w.ntiles * sizeof(Tile), cudaMemcpyHostToDevice, s));
        if (w.nptiles) {
            std::stable_sort(ph, ph + w.nptiles, longer);
            CUDA_TRY(cudaMemcpyAsync(g.slot_ptiles[slot], ph, w.nptiles * sizeof(Tile), cudaMemcpyHostToDevice, s));
        }
        CUDA_TRY(cudaMemcpyAsync(g.slot_list[slot], g.slot_lhost[slot], w.nlist * sizeof(int), cudaMemcpyHostToDevice, s));
        w.tiles = g.slot_tiles[slot];
        w.ptiles = g.slot_ptiles[slot];
        w.list = g.slot_list[slot];
    }
    CUDA_TRY(cudaEventRecord(b->slot_done[slot], s));
    return enqueue(b, sel, work, gradient != 0, slot, s);
}

}  // namespace

extern "C" {

msqoc_status msqoc_batch_create(msqoc_problem* const* problems, int32_t n, int32_t flags, msqoc_batch** out) {
    if (out) *out = nullptr;
    return guarded([&] { return batch_create(problems, n, flags, out); });
}

msqoc_status msqoc_batch_eval_objective(msqoc_batch* b, void* stream) {
    if (!b) return fail(MSQOC_ERR_INVALID_ARG, "batch is NULL");
    return guarded([&] { return eval(b, false, static_cast<cudaStream_t>(stream)); });
}

msqoc_status msqoc_batch_eval_gradient(msqoc_batch* b, void* stream) {
    if (!b) return fail(MSQOC_ERR_INVALID_ARG, "batch is NULL");
    return guarded([&] { return eval(b, true, static_cast<cudaStream_t>(stream)); });
}

msqoc_status msqoc_batch_eval_subset(msqoc_batch* b, const int32_t* members, int32_t n, int32_t gradient,
                                     int32_t slot, void* stream) {
    return guarded([&] { return batch_eval_subset(b, members, n, gradient, slot, stream); });
}

msqoc_status msqoc_batch_destroy(msqoc_batch* b) {
    if (!b) return MSQOC_OK;
    cudaDeviceSynchronize();
    free_batch(b);
    delete b;
    return MSQOC_OK;
}

msqoc_status msqoc_set_inputs(msqoc_problem* p, const double* alpha, const double* W, void* stream) {
    if (!p) return fail(MSQOC_ERR_INVALID_ARG, "problem is NULL");
    return stage_inputs(p, alpha, W, static_cast<cudaStream_t>(stream));
}

msqoc_status msqoc_get_objective(msqoc_problem* p, double* P_out, double* J_out, double* pen_out, void* stream) {
    if (!p || !P_out) return fail(MSQOC_ERR_INVALID_ARG, "problem or P_out is NULL");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const double* o = p->out_dev;
    CUDA_TRY(cudaMemcpyAsync(P_out, o, sizeof(double), cudaMemcpyDefault, s));
    if (J_out) CUDA_TRY(cudaMemcpyAsync(J_out, o + 1, sizeof(double), cudaMemcpyDefault, s));
    if (pen_out && p->pd.M > 1)
        CUDA_TRY(cudaMemcpyAsync(pen_out, o + 2, (p->pd.M - 1) * sizeof(double), cudaMemcpyDefault, s));
    const bool host = !is_device_ptr(P_out) || (J_out && !is_device_ptr(J_out)) || (pen_out && !is_device_ptr(pen_out));
    return host ? check_status_sync(p, s) : MSQOC_OK;
}

msqoc_status msqoc_get_gradient(msqoc_problem* p, double* P_out, double* grad_alpha, double* grad_W, void* stream) {
    if (!p || !grad_alpha) return fail(MSQOC_ERR_INVALID_ARG, "problem or grad_alpha is NULL");
    if (p->pd.M > 1 && !grad_W) return fail(MSQOC_ERR_INVALID_ARG, "grad_W is NULL but M > 1");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const double* o = p->out_dev;
    const OutLayout ol = out_layout(p->npen, p->pd.d, p->nW);
    if (P_out) CUDA_TRY(cudaMemcpyAsync(P_out, o, sizeof(double), cudaMemcpyDefault, s));
    CUDA_TRY(cudaMemcpyAsync(grad_alpha, o + ol.ga, p->pd.d * sizeof(double), cudaMemcpyDefault, s));
    if (p->pd.M > 1) CUDA_TRY(cudaMemcpyAsync(grad_W, o + ol.gw, p->nW * sizeof(double), cudaMemcpyDefault, s));
    const bool host = (P_out && !is_device_ptr(P_out)) || !is_device_ptr(grad_alpha) ||
                      (p->pd.M > 1 && !is_device_ptr(grad_W));
    return host ? check_status_sync(p, s) : MSQOC_OK;
}

}  // extern "C"
