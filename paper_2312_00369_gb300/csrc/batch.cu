// batch.cu -- many independent lattices advanced by one persistent launch
// per time step (the extern "C" pflbm_batch_* entry points of pflbm.h).
//
// A batch holds, in device memory, one step descriptor per lattice for each
// parity of the ping-pong state (set 0: in = current copy, out = the other;
// set 1: swapped). A step is, by schedule kernel: 1, one launch of
// k_step_batch over a work list of (lattice, first tile) items; 2, one launch
// of the staged kernel over its work list; 3 (the default for FP32 and 16-bit
// storage), one launch of the two-node kernel per group of lattices of one
// size and viscosity mode, its descriptors passed in the launch's parameters
// (grid = tiles x lattices), the groups' launches forked onto side streams and
// joined back. With use_graph the launches of PFLBM_BATCH_GRAPH_STEPS steps
// are captured once in a CUDA graph and replayed; in it each group takes its
// steps back to back on its stream, and the streams join once per replay.
//
// Runs of 16 steps and more with schedule kernel 3 or 0 step the members that
// fit the chip's shared memory there, many steps per launch (resident.cu), in
// waves of as many members as it holds, and the rest of the batch as above, where
// that is estimated to be faster.
#include <algorithm>
#include <climits>
#include <cstring>
#include <set>
#include <string>
#include <utility>
#include <vector>

#include "pflbm_internal.cuh"

namespace pfk {
int set_error(int code, const char* msg);
int materialize_handle(pflbm_t* h);
int post_status(pflbm_t* h);
}  // namespace pfk

using namespace pfk;

struct pflbm_batch {
    int precision = PFLBM_FP32;
    int device = 0;
    cudaStream_t stream = nullptr;
    pflbm_schedule_t sched{};
    std::vector<pflbm_t*> hs;
    std::vector<int> cur0;        // each lattice's state copy when descriptors were written
    int phase = 0;                // steps taken since then, mod 2
    size_t args_bytes = 0;
    int cap_lattices = 0, cap_work = 0;
    void* d_args[2] = {nullptr, nullptr};
    bool staged = false;          // staged (TMA ring) kernel, int4 items; else int2 items
    bool by_class = false;        // two-node kernel, one launch per group of same-size lattices
    struct ClassLaunch {
        int vv, nx, ny, count;
        std::vector<unsigned char> descs[2];   // count step descriptors of each set (host)
    };
    std::vector<ClassLaunch> classes;
    // runs of many steps: members that fit the chip's shared memory are stepped
    // there (resident.cu), as many of them side by side as it holds (a wave),
    // wave by wave; the others as above (their own groups and graph)
    struct Wave {
        int first, count;                  // its items
        std::vector<int> members;
    };
    std::vector<Wave> waves;
    bool no_resident = false;              // a cooperative launch was refused: launches from then on
    int route = 0;                         // test aid: 0 by the estimate, 1 waves, 2 launches
    double launch_us = 0, wave_us = 0;     // estimates of a step: launches; waves and the rest
    double setup_us = 0;                   // and of the waves' set-up
    int refuse_after = -1;                 // test aid: resident launches until one is taken as refused
    std::vector<ClassLaunch> rest;
    uint4* d_items = nullptr;
    ResidentCut* d_cuts = nullptr;
    // exchange words and the lists' overflow, in buffers of their own: whatever
    // members come and go, the words' memory holds zeros or words of earlier tags
    // only (list entries there could be taken for a word that has arrived)
    void *d_words = nullptr, *d_spill = nullptr;
    size_t cap_items = 0, cap_cuts = 0, cap_words = 0, cap_spill = 0;   // bytes
    unsigned long long half_words = 0;     // exchange words of one buffer
    unsigned res_tag = 0;
    // per-class launches run side by side: forked from the batch's stream to
    // these streams and joined back (in the captured graph as well)
    static constexpr int kForks = 4;
    cudaStream_t fork_stream[kForks] = {};
    cudaEvent_t fork_ev = nullptr, join_ev[kForks] = {};
    void* d_work = nullptr;
    int n_work = 0;
    int grid = 0;
    long long nodes = 0;
    // PFLBM_BATCH_GRAPH_STEPS steps of all members, and of those not resident
    struct Captured {
        cudaGraph_t graph = nullptr;
        cudaGraphExec_t exec = nullptr;
    } graph, rest_graph;
    void* (*alloc_fn)(size_t, void*) = nullptr;
    void (*free_fn)(void*, size_t, void*) = nullptr;
    void* alloc_ctx = nullptr;
};

namespace {

int balloc(pflbm_batch_t* b, void** p, size_t bytes)
{
    *p = nullptr;
    if (b->alloc_fn) {
        *p = b->alloc_fn(bytes, b->alloc_ctx);
        return *p ? PFLBM_OK : set_error(PFLBM_ENOMEM, "batch: allocator callback returned NULL");
    }
    cudaError_t e = cudaMalloc(p, bytes);
    if (e != cudaSuccess) {
        cudaGetLastError();
        *p = nullptr;
        return set_error(PFLBM_ENOMEM, "batch: cudaMalloc failed");
    }
    return PFLBM_OK;
}

void bfree(pflbm_batch_t* b, void* p, size_t bytes)
{
    if (!p) return;
    if (b->free_fn)
        b->free_fn(p, bytes, b->alloc_ctx);
    else
        cudaFree(p);
}

void drop_graph(pflbm_batch_t* b)
{
    for (pflbm_batch::Captured* g : {&b->graph, &b->rest_graph}) {
        if (g->exec) cudaGraphExecDestroy(g->exec);
        if (g->graph) cudaGraphDestroy(g->graph);
        g->exec = nullptr;
        g->graph = nullptr;
    }
}

// Interleave per-lattice item lists: lattice by lattice (order 0), or the
// largest lattices first with items interleaved across lattices (order 1).
template <typename I>
std::vector<I> order_items(std::vector<std::vector<I>>& per, int order)
{
    std::vector<I> w;
    if (order == 1) {
        std::vector<size_t> idx(per.size());
        for (size_t i = 0; i < idx.size(); ++i) idx[i] = i;
        std::stable_sort(idx.begin(), idx.end(), [&](size_t a, size_t b) { return per[a].size() > per[b].size(); });
        size_t longest = idx.empty() ? 0 : per[idx[0]].size();
        for (size_t j = 0; j < longest; ++j)
            for (size_t i : idx)
                if (j < per[i].size()) w.push_back(per[i][j]);
    } else {
        for (auto& v : per) w.insert(w.end(), v.begin(), v.end());
    }
    return w;
}

// Global-load kernel: (lattice, first tile) items of tiles_per_item tiles.
std::vector<int2> build_work(const std::vector<pflbm_t*>& hs, const pflbm_schedule_t& s)
{
    const int G = std::max(1, s.tiles_per_item);
    std::vector<std::vector<int2>> per(hs.size());
    for (size_t i = 0; i < hs.size(); ++i) {
        int ntx = tiles_x(hs[i]->nx), nty = tiles_y(hs[i]->ny);
        for (int by = 0; by < nty; by += G)
            for (int bx = 0; bx < ntx; ++bx) per[i].push_back(make_int2((int)i, by * ntx + bx));
    }
    return order_items(per, s.order);
}

// Staged kernel: (lattice, strip, first block, blocks | shape << 16) items,
// shape and blocks per item by size class.
std::vector<int4> build_work_staged(const std::vector<pflbm_t*>& hs, const pflbm_schedule_t& s)
{
    std::vector<std::vector<int4>> per(hs.size());
    for (size_t i = 0; i < hs.size(); ++i) {
        const long long nodes = (long long)hs[i]->nx * hs[i]->ny;
        int shape = 0, L = std::max(1, s.tiles_per_item);
        for (int k = 0; k < std::min(8, s.n_classes); ++k)
            if (nodes <= s.class_max_nodes[k]) {
                shape = s.class_shape[k] == 1 ? 1 : 0;
                L = std::max(1, s.class_tiles[k]);
                break;
            }
        const int TXs = shape ? 64 : 32, TYs = shape ? 4 : 8;
        const int nsx = (hs[i]->nx + TXs - 1) / TXs, nby = (hs[i]->ny + TYs - 1) / TYs;
        L = std::min(L, std::min(nby, 0xffff));
        for (int b0 = 0; b0 < nby; b0 += L)
            for (int sx = 0; sx < nsx; ++sx)
                per[i].push_back(make_int4((int)i, sx, b0, std::min(L, nby - b0) | (shape << 16)));
    }
    return order_items(per, s.order);
}

// Groups of the members `idx` with the same size and viscosity mode, largest
// first, each cut into launches of at most step2_class_capacity().
std::vector<pflbm_batch::ClassLaunch> build_classes(const pflbm_batch_t* b, std::vector<int> idx,
                                                    const std::vector<unsigned char>& a0,
                                                    const std::vector<unsigned char>& a1)
{
    std::vector<pflbm_batch::ClassLaunch> out;
    const int K = step2_class_capacity(b->precision), n = (int)idx.size();
    auto vv = [&](int i) { return (b->hs[i]->prm.nu_l > 0 && b->hs[i]->prm.nu_g > 0) ? 1 : 0; };
    std::stable_sort(idx.begin(), idx.end(), [&](int p, int q) {
        const long long np = (long long)b->hs[p]->nx * b->hs[p]->ny, nq = (long long)b->hs[q]->nx * b->hs[q]->ny;
        if (np != nq) return np > nq;
        if (b->hs[p]->nx != b->hs[q]->nx) return b->hs[p]->nx > b->hs[q]->nx;
        return vv(p) < vv(q);
    });
    for (int j = 0; j < n;) {
        const pflbm_t* h0 = b->hs[idx[j]];
        int e = j;
        while (e < n && e - j < K && b->hs[idx[e]]->nx == h0->nx && b->hs[idx[e]]->ny == h0->ny && vv(idx[e]) == vv(idx[j]))
            ++e;
        pflbm_batch::ClassLaunch cl;
        cl.vv = vv(idx[j]);
        cl.nx = h0->nx;
        cl.ny = h0->ny;
        cl.count = e - j;
        for (int set = 0; set < 2; ++set) {
            const std::vector<unsigned char>& src = set ? a1 : a0;
            cl.descs[set].resize(b->args_bytes * cl.count);
            for (int m = 0; m < cl.count; ++m)
                std::memcpy(cl.descs[set].data() + b->args_bytes * m, src.data() + b->args_bytes * idx[j + m], b->args_bytes);
        }
        out.push_back(std::move(cl));
        j = e;
    }
    return out;
}

// A device buffer of at least `bytes` (its contents are not kept when it grows).
int grow(pflbm_batch_t* b, void** p, size_t* cap, size_t bytes)
{
    if (bytes <= *cap) return PFLBM_OK;
    bfree(b, *p, *cap);
    *p = nullptr;
    *cap = 0;
    if (int rc = balloc(b, p, bytes)) return rc;
    *cap = bytes;
    return PFLBM_OK;
}

// Time of a step (us) by launches per size group and by waves, from what each has to do.
// Launches: 64 x 8 tiles without a solid node near, with some, and without fluid;
// groups past the four forked streams queue. A wave: what a step of its largest
// patch takes, the exchange, and the set-up of its launch spread over the run (43 us for
// small patches, 65 to 109 for full ones; counted low, since short runs of many
// mixes are close and the launches' estimate errs to the low side). Fitted to 184 mixes
// in FP16 and FP32 (2 to 300 lattices of 128 x 64 to 784 x 392, flat and with obstacles,
// requests of many sizes), runs of 200 steps: either estimate is within 12 % in nearly
// all. With the lines below a mix runs 0.3 to 0.5 % above the faster of the two on
// average, at most 1 % (FP16) or 6 % (FP32) above the launches. (In FP32 the lines nearly touch from 0.3 to 2 M nodes; at
// more than 2^21 the launches run at 0.9 of the HBM bandwidth and are left alone.)
// Measured (us a step, launches and waves): FP16 16 requests 47.5 and 33.6, 64 requests
// 160 and 154, 256 uneven with obstacles 213 and 196, without 186 and 208, 18 of 528 x 264
// 54.6 and 78.3; FP32 8 requests 18.8 and 13.8, 6 of 256 x 256 with a shallow slope 13.8 and
// 12.7, 16 uneven 14.3 and 19.9, 9 of 512 x 256 33.9 and 45.4.
struct RouteCost {
    double fixed, plain, mixed, solid, group;   // launches
    double wave, cycle, setup, setup_cycle;     // waves
    double line;                                // waves below this times the launches
    long long most;                             // nodes
};
constexpr RouteCost kRoute16{5.77, 8.29e-3, 19.4e-3, 4.83e-3, 0.45, 1.79, 7.49e-4, 25.0, 8e-3, 0.97, LLONG_MAX};
constexpr RouteCost kRoute32{4.33, 10.33e-3, 18.57e-3, 8.1e-3, 0.57, 2.55, 8.52e-4, 25.0, 8e-3, 1.0, 1LL << 21};
const RouteCost& route_cost(int precision) { return precision == PFLBM_FP32 ? kRoute32 : kRoute16; }

// Estimate of a step of the members `idx` by launches.
double launch_estimate(const pflbm_batch_t* b, const std::vector<int>& idx)
{
    if (idx.empty()) return 0.0;
    const RouteCost& c = route_cost(b->precision);
    std::set<std::pair<int, int>> sizes;
    double us = c.fixed;
    for (int i : idx) {
        const pflbm_t* h = b->hs[i];
        sizes.insert({h->nx, h->ny});
        if (h->map.sum.empty())   // a large lattice
            us += c.plain * ((h->nx + 63) / 64) * ((h->ny + 7) / 8);
        else
            us += c.plain * h->map.tiles[kTilePlain] + c.mixed * h->map.tiles[kTileMixed] + c.solid * h->map.tiles[kTileSolid];
    }
    return us + c.group * std::max(0, (int)sizes.size() - pflbm_batch::kForks);
}

// Whether a run of n steps takes the waves; n = 0: whether any run may.
bool waves_pay(const pflbm_batch_t* b, int64_t n)
{
    if (b->route) return b->route == 1;
    const RouteCost& c = route_cost(b->precision);
    return b->nodes <= c.most && b->wave_us + (n ? b->setup_us / (double)n : 0.0) < c.line * b->launch_us;
}

// Waves of members stepped resident, largest members first, each into the first
// wave with room for its patches; removes them from *idx. Where the patches
// of the last wave leave SMs idle, the members are cut into more rows of
// patches, as long as that takes no more waves.
int plan_waves(pflbm_batch_t* b, std::vector<int>* idx)
{
    const int cls = resident_batch_class(b->precision);
    int coop = 0, sms = 0;
    cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, b->device);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, b->device);
    if (!coop || cls < 0 || b->no_resident || b->route == 2) return PFLBM_OK;
    if (!b->route && b->nodes > route_cost(b->precision).most) return PFLBM_OK;
    const int n = (int)b->hs.size();
    struct Member { int i, active; ResidentCut cut; unsigned long long words; };
    auto pack = [&](double split, std::vector<Member>& ms, std::vector<int>& wave, std::vector<int>& others) {
        ms.clear();
        others.clear();
        for (int i : *idx) {
            Member m;
            m.i = i;
            const pflbm_t* h = b->hs[i];
            if (cut_resident(h->nx, h->ny, b->precision, h->map, cls, split, &m.cut, &m.active, &m.words) && m.active > 0 &&
                m.active <= sms)
                ms.push_back(m);
            else
                others.push_back(i);
        }
        std::stable_sort(ms.begin(), ms.end(), [](const Member& p, const Member& q) { return p.active > q.active; });
        std::vector<int> room;
        wave.assign(ms.size(), 0);
        for (size_t k = 0; k < ms.size(); ++k) {
            size_t w = 0;
            while (w < room.size() && room[w] < ms[k].active) ++w;
            if (w == room.size()) room.push_back(sms);
            room[w] -= ms[k].active;
            wave[k] = (int)w;
        }
        return (int)room.size();
    };
    std::vector<Member> ms, ms2;
    std::vector<int> wave, wave2, others, others2;
    int nw = pack(1.0, ms, wave, others);
    if (nw == 0) return PFLBM_OK;
    long long total = 0;
    for (const Member& m : ms) total += m.active;
    const double spare = (double)nw * sms / (double)total;
    for (double split = spare; split > 1.05; split -= 0.1 * (spare - 1.0) + 0.02)
        if (pack(split, ms2, wave2, others2) <= nw && others2.size() <= others.size()) {
            ms.swap(ms2);
            wave.swap(wave2);
            others.swap(others2);
            nw = 1 + *std::max_element(wave.begin(), wave.end());
            break;
        }
    const RouteCost& rate = route_cost(b->precision);
    b->launch_us = launch_estimate(b, *idx);
    b->wave_us = launch_estimate(b, others) + nw * rate.wave;
    b->setup_us = nw * rate.setup;
    for (int w = 0; w < nw; ++w) {
        double most = 0;
        for (size_t k = 0; k < ms.size(); ++k)
            if (wave[k] == w) most = std::max(most, step_cycles(b->precision, ms[k].cut.w, ms[k].cut.h));
        b->wave_us += rate.cycle * most;
        b->setup_us += rate.setup_cycle * most;
    }
    if (!waves_pay(b, 0)) return PFLBM_OK;
    std::vector<uint4> items;
    std::vector<ResidentCut> cuts(n);
    int most = 0;
    b->half_words = 0;
    for (int w = 0; w < nw; ++w) {
        pflbm_batch::Wave wv{(int)items.size(), 0, {}};
        unsigned long long at = 0;
        for (size_t k = 0; k < ms.size(); ++k) {
            if (wave[k] != w) continue;
            const Member& m = ms[k];
            cuts[m.i] = m.cut;
            wv.members.push_back(m.i);
            unsigned rank = 0;
            for (int p = 0; p < m.cut.px * m.cut.py; ++p)
                if (m.cut.active[p >> 5] >> (p & 31) & 1u)
                    items.push_back(make_uint4((unsigned)m.i, rank++ << 16 | (unsigned)p, (unsigned)at, (unsigned)(at >> 32)));
            at += m.words;
        }
        wv.count = (int)items.size() - wv.first;
        most = std::max(most, wv.count);
        b->half_words = std::max(b->half_words, at);
        b->waves.push_back(std::move(wv));
    }
    const size_t bytes = 2 * b->half_words * resident_word_bytes();
    const bool fresh = bytes > b->cap_words;
    void *pi = b->d_items, *pc = b->d_cuts;
    int rc = grow(b, &pi, &b->cap_items, items.size() * sizeof(uint4));
    b->d_items = (uint4*)pi;
    if (!rc) rc = grow(b, &pc, &b->cap_cuts, cuts.size() * sizeof(ResidentCut));
    b->d_cuts = (ResidentCut*)pc;
    if (!rc) rc = grow(b, &b->d_spill, &b->cap_spill, (size_t)most * resident_spill(b->precision, cls).words() * 4);
    if (!rc) rc = grow(b, &b->d_words, &b->cap_words, bytes);
    if (rc) {   // no memory for it: all members take single steps
        b->waves.clear();
        return PFLBM_OK;
    }
    cudaError_t e = cudaMemcpyAsync(b->d_items, items.data(), items.size() * sizeof(uint4), cudaMemcpyHostToDevice, b->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(b->d_cuts, cuts.data(), cuts.size() * sizeof(ResidentCut), cudaMemcpyHostToDevice, b->stream);
    if (e == cudaSuccess && fresh) {
        e = cudaMemsetAsync(b->d_words, 0, bytes, b->stream);
        b->res_tag = 0;
    }
    // the host vectors go out of scope on return: finish the copies first
    if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
    if (e != cudaSuccess) return set_error(PFLBM_ECUDA, cudaGetErrorString(e));
    idx->swap(others);
    return PFLBM_OK;
}

int upload(pflbm_batch_t* b)
{
    const int n = (int)b->hs.size();
    std::vector<unsigned char> a0(b->args_bytes * n), a1(b->args_bytes * n);
    b->cur0.resize(n);
    b->nodes = 0;
    for (int i = 0; i < n; ++i) {
        pflbm_t* h = b->hs[i];
        write_step_args(h, 0, a0.data() + b->args_bytes * i);
        write_step_args(h, 1, a1.data() + b->args_bytes * i);
        b->cur0[i] = h->cur;
        b->nodes += (long long)h->nx * h->ny;
    }
    b->staged = b->precision != PFLBM_FP64 && b->sched.kernel == 2;
    for (pflbm_t* h : b->hs)
        if (!h->tma) b->staged = false;
    // the default kernel is the two-node one, one launch per group of
    // same-size lattices (measured fastest on mixes of small lattices in
    // FP32 and 16-bit storage)
    b->by_class = b->precision != PFLBM_FP64 && (b->sched.kernel == 3 || b->sched.kernel == 0);
    b->classes.clear();
    b->rest.clear();
    b->waves.clear();
    if (b->by_class) {
        std::vector<int> idx(n);
        for (int i = 0; i < n; ++i) idx[i] = i;
        b->classes = build_classes(b, idx, a0, a1);
        if (int rc = plan_waves(b, &idx)) return rc;
        if (!b->waves.empty()) b->rest = build_classes(b, idx, a0, a1);
    }
    std::vector<unsigned char> wbytes;
    size_t item = b->staged ? sizeof(int4) : sizeof(int2);
    if (b->by_class) {
        // no work list: each launch's grid is (tiles, lattices)
    } else if (b->staged) {
        std::vector<int4> w4 = build_work_staged(b->hs, b->sched);
        wbytes.resize(w4.size() * item);
        if (!w4.empty()) std::memcpy(wbytes.data(), w4.data(), wbytes.size());
    } else {
        std::vector<int2> w2 = build_work(b->hs, b->sched);
        wbytes.resize(w2.size() * item);
        if (!w2.empty()) std::memcpy(wbytes.data(), w2.data(), wbytes.size());
    }
    const int n_items = (int)(wbytes.size() / item);
    if (n > b->cap_lattices) {
        int cap = std::max(n, 2 * b->cap_lattices);
        for (int k = 0; k < 2; ++k) {
            bfree(b, b->d_args[k], b->args_bytes * b->cap_lattices);
            b->d_args[k] = nullptr;
        }
        for (int k = 0; k < 2; ++k)
            if (int rc = balloc(b, &b->d_args[k], b->args_bytes * cap)) return rc;
        b->cap_lattices = cap;
        drop_graph(b);
    }
    if (n_items > b->cap_work) {
        int cap = std::max(n_items, 2 * b->cap_work);
        bfree(b, b->d_work, sizeof(int4) * b->cap_work);
        b->d_work = nullptr;
        void* p;
        if (int rc = balloc(b, &p, sizeof(int4) * cap)) return rc;
        b->d_work = p;
        b->cap_work = cap;
        drop_graph(b);
    }
    cudaError_t e = cudaMemcpyAsync(b->d_args[0], a0.data(), a0.size(), cudaMemcpyHostToDevice, b->stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(b->d_args[1], a1.data(), a1.size(), cudaMemcpyHostToDevice, b->stream);
    if (e == cudaSuccess && !wbytes.empty())
        e = cudaMemcpyAsync(b->d_work, wbytes.data(), wbytes.size(), cudaMemcpyHostToDevice, b->stream);
    // the host vectors go out of scope on return: finish the copies first
    if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
    if (e != cudaSuccess) return set_error(PFLBM_ECUDA, cudaGetErrorString(e));
    drop_graph(b);   // kernel, work list or grid may differ from the captured ones
    b->n_work = n_items;
    b->phase = 0;
    int per_sm = b->staged ? staged_batch_ctas_per_sm(b->precision) : batch_max_ctas_per_sm(b->precision);
    if (b->sched.ctas_per_sm > 0) per_sm = std::min(per_sm, b->sched.ctas_per_sm);
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, b->device);
    b->grid = std::max(1, std::min(b->n_work, std::max(1, per_sm) * std::max(1, sms)));
    if (b->by_class) {
        // info: the CTAs (one 64 x 8 tile each) of all launches, and the launches
        long long ctas = 0;
        for (const auto& cl : b->classes) ctas += (long long)cl.count * ((cl.nx + 63) / 64) * ((cl.ny + 7) / 8);
        b->n_work = (int)std::min(ctas, (long long)INT_MAX);
        b->grid = (int)b->classes.size();
    }
    if (b->by_class && b->classes.size() > 1) {
        // the forked streams and events of the per-class launches (made here,
        // outside any stream capture)
        const int nf = std::min((int)b->classes.size(), (int)pflbm_batch::kForks);
        for (int k = 0; k < nf; ++k) {
            cudaError_t e2 = cudaSuccess;
            if (!b->fork_stream[k]) e2 = cudaStreamCreateWithFlags(&b->fork_stream[k], cudaStreamNonBlocking);
            if (e2 == cudaSuccess && !b->join_ev[k])
                e2 = cudaEventCreateWithFlags(&b->join_ev[k], cudaEventDisableTiming);
            if (e2 != cudaSuccess) return set_error(PFLBM_ECUDA, cudaGetErrorString(e2));
        }
        if (!b->fork_ev) {
            cudaError_t e2 = cudaEventCreateWithFlags(&b->fork_ev, cudaEventDisableTiming);
            if (e2 != cudaSuccess) return set_error(PFLBM_ECUDA, cudaGetErrorString(e2));
        }
    }
    return PFLBM_OK;
}

int check_members(pflbm_t* const* hs, int count, int precision, int device, cudaStream_t stream)
{
    for (int i = 0; i < count; ++i) {
        if (!hs[i]) return set_error(PFLBM_EINVAL, "batch: NULL handle");
        if (hs[i]->precision != precision || hs[i]->device != device || hs[i]->stream != stream)
            return set_error(PFLBM_EINVAL, "batch: all handles need the same precision, device and stream");
        for (int j = 0; j < i; ++j)
            if (hs[j] == hs[i]) return set_error(PFLBM_EINVAL, "batch: a handle appears twice");
    }
    return PFLBM_OK;
}

// Steps per captured graph (even). One graph replay runs each size group's
// steps back to back: measured on 256 small lattices (BF16, MLUPS) 46.8k with
// a join after every step, 47.6k at 2 steps per graph, 48.3k at 8, 47.9k at 32
// (300 steps), and over 400 steps 48.55k at 8 against 48.7k at 16. 8 divides
// the 200-step ticks of the server.
#ifndef PFLBM_BATCH_GRAPH_STEPS
#define PFLBM_BATCH_GRAPH_STEPS 8
#endif

cudaError_t launch_set(pflbm_batch_t* b, const std::vector<pflbm_batch::ClassLaunch>& classes, int set);

// nsteps steps from descriptor set `set0` on. With one launch per size group,
// each group takes its steps back to back on its own forked stream, and the
// streams join once at the end: a group's lattices need only their own
// previous step, so small groups run ahead instead of waiting each step for
// the largest.
cudaError_t launch_steps(pflbm_batch_t* b, const std::vector<pflbm_batch::ClassLaunch>& classes, int set0, int nsteps)
{
    const int nc = (int)classes.size();
    if (!b->by_class || nc <= 1) {
        cudaError_t e = cudaSuccess;
        for (int s = 0; s < nsteps && e == cudaSuccess; ++s) e = launch_set(b, classes, (set0 + s) & 1);
        return e;
    }
    const int nf = std::min(nc, (int)pflbm_batch::kForks);
    cudaError_t e = cudaEventRecord(b->fork_ev, b->stream);
    for (int k = 0; k < nf && e == cudaSuccess; ++k) e = cudaStreamWaitEvent(b->fork_stream[k], b->fork_ev, 0);
    for (int c = 0; c < nc && e == cudaSuccess; ++c) {
        const auto& cl = classes[c];
        for (int s = 0; s < nsteps && e == cudaSuccess; ++s)
            e = launch_step2_class(b->precision, cl.vv, cl.descs[(set0 + s) & 1].data(), cl.count, cl.nx, cl.ny,
                                   b->fork_stream[c % nf]);
    }
    for (int k = 0; k < nf && e == cudaSuccess; ++k) e = cudaEventRecord(b->join_ev[k], b->fork_stream[k]);
    for (int k = 0; k < nf && e == cudaSuccess; ++k) e = cudaStreamWaitEvent(b->stream, b->join_ev[k], 0);
    return e;
}

cudaError_t launch_set(pflbm_batch_t* b, const std::vector<pflbm_batch::ClassLaunch>& classes, int set)
{
    if (b->staged)
        return launch_step_staged_batch(b->precision, b->d_args[set], (const int4*)b->d_work, b->n_work, b->grid,
                                        b->stream);
    if (b->by_class) {
        const int nc = (int)classes.size();
        if (nc == 1)
            return launch_step2_class(b->precision, classes[0].vv, classes[0].descs[set].data(), classes[0].count,
                                      classes[0].nx, classes[0].ny, b->stream);
        const int nf = std::min(nc, (int)pflbm_batch::kForks);   // streams made by upload()
        cudaError_t e = cudaEventRecord(b->fork_ev, b->stream);
        for (int k = 0; k < nf && e == cudaSuccess; ++k) e = cudaStreamWaitEvent(b->fork_stream[k], b->fork_ev, 0);
        // largest groups first, dealt round-robin over the forked streams
        for (int c = 0; c < nc && e == cudaSuccess; ++c) {
            const auto& cl = classes[c];
            e = launch_step2_class(b->precision, cl.vv, cl.descs[set].data(), cl.count, cl.nx, cl.ny,
                                   b->fork_stream[c % nf]);
        }
        for (int k = 0; k < nf && e == cudaSuccess; ++k) e = cudaEventRecord(b->join_ev[k], b->fork_stream[k]);
        for (int k = 0; k < nf && e == cudaSuccess; ++k) e = cudaStreamWaitEvent(b->stream, b->join_ev[k], 0);
        return e;
    }
    return launch_step_batch(b->precision, b->d_args[set], (const int2*)b->d_work, b->n_work,
                             std::max(1, b->sched.tiles_per_item), b->grid, b->stream);
}

int ensure_graph(pflbm_batch_t* b, const std::vector<pflbm_batch::ClassLaunch>& classes, pflbm_batch::Captured* g)
{
    if (g->exec) return PFLBM_OK;
    cudaError_t e = cudaStreamBeginCapture(b->stream, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) return set_error(PFLBM_ECUDA, cudaGetErrorString(e));
    cudaError_t e1 = launch_steps(b, classes, 0, PFLBM_BATCH_GRAPH_STEPS);
    e = cudaStreamEndCapture(b->stream, &g->graph);
    if (e1 != cudaSuccess || e != cudaSuccess) {
        drop_graph(b);
        return set_error(PFLBM_ECUDA, "batch: graph capture failed");
    }
    e = cudaGraphInstantiate(&g->exec, g->graph, 0);
    if (e != cudaSuccess) {
        drop_graph(b);
        return set_error(PFLBM_ECUDA, cudaGetErrorString(e));
    }
    return PFLBM_OK;
}

// n steps of the members in `classes` (all members where the kernel has no
// size groups) from parity `phase` on, by graph replays where asked.
int step_launches(pflbm_batch_t* b, const std::vector<pflbm_batch::ClassLaunch>& classes, pflbm_batch::Captured* g, int phase,
                  int64_t n)
{
    static_assert(PFLBM_BATCH_GRAPH_STEPS >= 2 && PFLBM_BATCH_GRAPH_STEPS % 2 == 0, "an even step count per graph");
    auto single = [&]() -> int {
        cudaError_t e = launch_set(b, classes, phase);
        if (e != cudaSuccess) return set_error(PFLBM_ECUDA, cudaGetErrorString(e));
        phase ^= 1;
        --n;
        return PFLBM_OK;
    };
    if (phase == 1 && n > 0)
        if (int rc = single()) return rc;
    if (b->sched.use_graph && n >= PFLBM_BATCH_GRAPH_STEPS) {
        if (int rc = ensure_graph(b, classes, g)) return rc;
        for (; n >= PFLBM_BATCH_GRAPH_STEPS; n -= PFLBM_BATCH_GRAPH_STEPS) {
            cudaError_t e = cudaGraphLaunch(g->exec, b->stream);
            if (e != cudaSuccess) return set_error(PFLBM_ECUDA, cudaGetErrorString(e));
        }
    }
    while (n > 0)
        if (int rc = single()) return rc;
    return PFLBM_OK;
}

// A resident launch; cudaErrorCooperativeLaunchTooLarge and the like when fewer
// SMs are to be had than the device reports.
cudaError_t launch_wave(pflbm_batch_t* b, const ResidentWave& a, int cls)
{
    if (b->refuse_after >= 0 && b->refuse_after-- == 0) return cudaErrorCooperativeLaunchTooLarge;
    return launch_resident_wave(b->precision, a, cls, b->stream);
}

// n steps of the members `idx` from parity `phase` on, one launch per size group
// and step. Each member's copy named by its handle is that of the batch's phase.
int step_members(pflbm_batch_t* b, const std::vector<int>& idx, int phase, int64_t n)
{
    std::vector<unsigned char> a0(b->args_bytes * b->hs.size()), a1(b->args_bytes * b->hs.size());
    for (int i : idx) {
        write_step_args(b->hs[i], b->phase, a0.data() + b->args_bytes * i);
        write_step_args(b->hs[i], b->phase ^ 1, a1.data() + b->args_bytes * i);
    }
    const std::vector<pflbm_batch::ClassLaunch> classes = build_classes(b, idx, a0, a1);
    for (int64_t left = n; left > 0;) {
        const int c = (int)std::min<int64_t>(left, kResidentMaxSteps);
        cudaError_t e = launch_steps(b, classes, phase, c);
        if (e != cudaSuccess) return set_error(PFLBM_ECUDA, cudaGetErrorString(e));
        phase ^= c & 1;
        left -= c;
    }
    return PFLBM_OK;
}

// n steps of the waves' members. When a launch is refused, what is left of its
// wave and the waves after it are taken by the size groups' launches, each from
// the copy that it has come to, and so is everything from then on.
int step_waves(pflbm_batch_t* b, int64_t n)
{
    const int cls = resident_batch_class(b->precision);
    for (const pflbm_batch::Wave& w : b->waves) {
        int phase = b->phase;
        int64_t left = n;
        while (left > 0 && !b->no_resident) {
            const int c = (int)std::min<int64_t>(left, kResidentMaxSteps);
            if (b->res_tag > UINT_MAX - 2u * kResidentMaxSteps) {   // tags start again
                cudaError_t e = cudaMemsetAsync(b->d_words, 0, b->cap_words, b->stream);
                if (e != cudaSuccess) return set_error(PFLBM_ECUDA, cudaGetErrorString(e));
                b->res_tag = 0;
            }
            ResidentWave a{};
            a.args = b->d_args[phase];
            a.cuts = b->d_cuts;
            a.items = b->d_items + w.first;
            a.words = b->d_words;
            a.half = b->half_words;
            a.spill = (uint32_t*)b->d_spill;
            a.tag = b->res_tag;
            a.steps = c;
            a.n_items = w.count;
            if (launch_wave(b, a, cls) != cudaSuccess) {
                cudaGetLastError();
                b->no_resident = true;
                break;
            }
            b->res_tag += (unsigned)c;
            phase ^= c & 1;
            left -= c;
        }
        if (left > 0)
            if (int rc = step_members(b, w.members, phase, left)) return rc;
    }
    return PFLBM_OK;
}

// Whether a run of n steps takes the waves.
bool runs_resident(const pflbm_batch_t* b, int64_t n)
{
    return !b->waves.empty() && !b->no_resident && n >= kResidentMinSteps && waves_pay(b, n);
}

}  // namespace

extern "C" {

void pflbm_schedule_default(pflbm_schedule_t* s)
{
    if (!s) return;
    std::memset(s, 0, sizeof(*s));
    s->ctas_per_sm = 0;
    s->tiles_per_item = 1;
    s->order = 0;
    s->use_graph = 1;
    s->kernel = 0;
    s->n_classes = 0;
}

int pflbm_batch_create(pflbm_batch_t** out, pflbm_t* const* hs, int count, const pflbm_schedule_t* sched)
{
    if (!out) return set_error(PFLBM_EINVAL, "batch: NULL out");
    *out = nullptr;
    if (!hs || count < 1) return set_error(PFLBM_EINVAL, "batch: need at least one handle");
    if (!hs[0]) return set_error(PFLBM_EINVAL, "batch: NULL handle");
    if (int rc = check_members(hs, count, hs[0]->precision, hs[0]->device, hs[0]->stream)) return rc;
    pflbm_batch_t* b = new pflbm_batch();
    b->precision = hs[0]->precision;
    b->device = hs[0]->device;
    b->stream = hs[0]->stream;
    // the batch's own small buffers come from cudaMalloc: a member's
    // allocator may belong to a handle that is destroyed while the batch lives
    pflbm_schedule_default(&b->sched);
    if (sched) b->sched = *sched;
    if (b->sched.tiles_per_item < 1) b->sched.tiles_per_item = 1;
    b->args_bytes = step_args_bytes(b->precision);
    b->hs.assign(hs, hs + count);
    DeviceGuard g(b->device);
    if (int rc = upload(b)) {
        pflbm_batch_destroy(b);
        return rc;
    }
    *out = b;
    return PFLBM_OK;
}

int pflbm_batch_set(pflbm_batch_t* b, pflbm_t* const* hs, int count)
{
    if (!b || !hs || count < 1) return set_error(PFLBM_EINVAL, "batch: invalid arguments");
    if (int rc = check_members(hs, count, b->precision, b->device, b->stream)) return rc;
    DeviceGuard g(b->device);
    b->hs.assign(hs, hs + count);
    return upload(b);
}

int pflbm_batch_step(pflbm_batch_t* b, int64_t n)
{
    if (!b) return set_error(PFLBM_EINVAL, "batch: NULL batch");
    if (n < 0) return set_error(PFLBM_EINVAL, "batch: negative step count");
    if (n == 0) return PFLBM_OK;
    DeviceGuard g(b->device);
    NvtxRange range("pflbm_batch_step");
    bool stale = false;
    for (size_t i = 0; i < b->hs.size(); ++i) {
        pflbm_t* h = b->hs[i];
        if (h->hstatus && (h->hstatus[0] & 4))
            return set_error(PFLBM_ETIMEOUT, "batch: a wait in the step kernel gave up");
        if (h->hstatus && h->hstatus[0] != 0)
            return set_error(PFLBM_ENUMERIC, "batch: NaN or |u| >= 0.3 detected on the device");
        if (h->init_pending) {
            if (int rc = materialize_handle(h)) return rc;
        }
        if (h->cur != (b->cur0[i] ^ b->phase)) stale = true;
    }
    if (stale) {  // a member was stepped on its own: rewrite the descriptors
        if (int rc = upload(b)) return rc;
    }
    if (runs_resident(b, n) && !capturing(b->stream)) {
        if (int rc = step_waves(b, n)) return rc;
        if (!b->rest.empty())
            if (int rc = step_launches(b, b->rest, &b->rest_graph, b->phase, n)) return rc;
    } else if (int rc = step_launches(b, b->classes, &b->graph, b->phase, n)) {
        return rc;
    }
    b->phase ^= (int)(n & 1);
    for (pflbm_t* h : b->hs) {
        if (n & 1) h->cur ^= 1;
        h->steps += n;
        h->replace_phi = true;
        if (int rc = post_status(h)) return rc;
    }
    // invariant: every member's current copy is cur0[i] ^ phase
    return PFLBM_OK;
}

int pflbm_batch_kernel(const pflbm_batch_t* b)
{
    if (!b) return set_error(PFLBM_EINVAL, "batch: NULL batch");
    return b->staged ? 2 : (b->by_class ? 3 : 1);
}

int pflbm_batch_info(const pflbm_batch_t* b, int* n_work, int* grid, int64_t* nodes)
{
    if (!b) return set_error(PFLBM_EINVAL, "batch: NULL batch");
    if (n_work) *n_work = b->n_work;
    if (grid) *grid = b->grid;
    if (nodes) *nodes = b->nodes;
    return PFLBM_OK;
}

int pflbm_debug_batch(pflbm_batch_t* b, int64_t n, int route, int refuse_after, int* waves)
{
    if (!b || route < 0 || route > 2) return set_error(PFLBM_EINVAL, "batch: invalid arguments");
    b->refuse_after = refuse_after;
    if (route != b->route) {
        DeviceGuard g(b->device);
        b->route = route;
        if (int rc = upload(b)) return rc;
    }
    if (waves) *waves = runs_resident(b, n) ? (int)b->waves.size() : 0;
    return PFLBM_OK;
}

void pflbm_batch_destroy(pflbm_batch_t* b)
{
    if (!b) return;
    DeviceGuard g(b->device);
    if (b->stream) cudaStreamSynchronize(b->stream);
    drop_graph(b);
    for (int k = 0; k < pflbm_batch::kForks; ++k) {
        if (b->fork_stream[k]) {
            cudaStreamSynchronize(b->fork_stream[k]);
            cudaStreamDestroy(b->fork_stream[k]);
        }
        if (b->join_ev[k]) cudaEventDestroy(b->join_ev[k]);
    }
    if (b->fork_ev) cudaEventDestroy(b->fork_ev);
    for (int k = 0; k < 2; ++k) bfree(b, b->d_args[k], b->args_bytes * b->cap_lattices);
    bfree(b, b->d_work, sizeof(int4) * b->cap_work);
    bfree(b, b->d_items, b->cap_items);
    bfree(b, b->d_cuts, b->cap_cuts);
    bfree(b, b->d_words, b->cap_words);
    bfree(b, b->d_spill, b->cap_spill);
    delete b;
}

}  // extern "C"
