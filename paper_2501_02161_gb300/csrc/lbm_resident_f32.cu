// lbm_resident_f32.cu -- resident kernels of the 32-bit arithmetic (FP32 and
// 16-bit flow storage; the adjoint and temperature populations are FP32 in
// all three) and the planner of resident launches.
#include <algorithm>
#include <vector>

#include "lbm_dispatch.cuh"
#include "lbm_resident.cuh"

namespace lbm {

namespace {
constexpr int kSMs = 152;
constexpr int kSmemSM = 233472;   // shared memory of an SM; a block of m on it may use kSmemSM / m - 1 KB

int ceil_div(int a, int b) { return (a + b - 1) / b; }
}  // namespace

namespace {
// words of an inbox (res_first of the last group, in closed form)
int inbox_words(bool heat, bool d2, int real, int bx, int by, int bz) {
    const int np = real == 8 ? 1 : 3;
    const int x = ceil_div(by * bz, np), y = ceil_div(bx * bz, np), z = ceil_div(bx * by, np);
    if (heat) return 2 * (x + y + z);
    if (d2) return 6 * (x + y) + 4 * ceil_div(bz, np);
    return 10 * (x + y + z) + 4 * (ceil_div(bx, np) + ceil_div(by, np) + ceil_div(bz, np));
}
}  // namespace

namespace {
// The cut into at most 152 m boxes, m to an SM, that is estimated to be fastest.
// A step of a box costs the SM its instructions over four schedulers (about 320
// of a border task, 250 of an interior one, 40 for 32 words to send and
// receive; less than half for the smaller lattices), and the block itself the
// rounds of its warps and the way of the words.
ResPlan plan_boxes(int stencil, int storage, ResPhase ph, int nx, int ny, int nz, int m, int& tasks) {
    ResPlan best = {};
    const bool d2 = stencil == 0;
    const bool heat = ph == RP_THERM || ph == RP_TADJ;
    const int Q = heat ? 7 : (d2 ? 9 : 19);
    const int naux = heat ? (ph == RP_THERM ? 6 : 5) : (ph == RP_ADJ_T ? 7 : 4);  // constants and boundary values
    const int rb = (int)aux_bytes(storage);
    const int tb = heat ? (int)heat_bytes(storage) : (ph == RP_FLOW ? (int)pop_bytes(storage) : (int)adj_bytes(storage));
    const int limit = kSMs * m, smem_max = kSmemSM / m - 1024, most = kResThreads(rb) / m / 32;
    if ((long long)nx * ny * nz * Q * tb > (long long)kSMs * kSmemSM) return best;
    double best_cost = 1e30;
    for (int pz = 1; pz <= std::min(nz, limit); ++pz) {
        const int bz = ceil_div(nz, pz);
        if (bz > 255 || ceil_div(nz, bz) != pz) continue;
        for (int py = 1; py <= std::min(ny, limit / pz); ++py) {
            const int by = ceil_div(ny, py);
            if (by > 255 || ceil_div(ny, by) != py) continue;
            for (int px = 1; px <= std::min(nx, limit / (pz * py)); ++px) {
                const int bx = ceil_div(nx, px);
                if (bx > 255 || ceil_div(nx, bx) != px) continue;
                ResGeom g = {};
                g.nx = nx; g.ny = ny; g.nz = nz;
                g.px = px; g.py = py; g.pz = pz;
                g.bx = bx; g.by = by; g.bz = bz;
                g.pitch = bx | 1;
                const long long nodes = (long long)bx * by * bz, cap = (long long)g.pitch * by * bz;
                if (cap > 8192) continue;  // 13-bit places
                const long long aux_at = (kResHead + (Q * cap + 1) * tb + 15) / 16 * 16;
                const long long word_at = (aux_at + (nodes + 96) * ((long long)naux * rb + 4) + 15) / 16 * 16;
                if (word_at > smem_max) continue;
                g.inbox = ceil_div(inbox_words(heat, d2, rb, bx, by, bz), 32) * 32;
                const long long smem = word_at + std::max(16LL * g.inbox, cap);
                if (smem > smem_max) continue;
                const long long inner = (long long)std::max(bx - 2, 0) * std::max(by - 2, 0) *
                                        (d2 ? bz : std::max(bz - 2, 0));
                const int nb = (int)(nodes - inner + 31) / 32, ni = (int)(inner + 31) / 32;
                // warps, and how many of them exchange: half of a full set, those
                // with the fewest tasks among them, or for a small box up to
                // eight of their own
                const int need = g.inbox / 32;
                int warps = most, exchange = std::min(most / 2, need);
                if (nb + ni + std::min(need, 8) <= most) {
                    exchange = std::min(need, 8);
                    warps = nb + ni + exchange;
                }
                const int words = ceil_div(need, exchange);
                const double scale = heat || d2 ? 0.45 : 1.0;
                const double issue = (scale * (320.0 * nb + 250.0 * ni) + 40.0 * need) / 4 / 0.75;
                const double travel = 900.0 * scale * ceil_div(nb, warps) + 1600.0 + 250.0 * words;
                const double cost = std::max(issue, travel + 0.5 * issue) + 0.01 * px * py * pz;
                if (cost >= best_cost) continue;
                best_cost = cost;
                tasks = nb + ni;
                g.cap = (int)cap;
                g.list = (int)nodes + 96;
                g.aux_at = (int)aux_at;
                g.word_at = (int)word_at;
                g.parity = (long long)g.inbox * px * py * pz;
                g.silent = 32 * (warps - exchange);
                g.words = words;
                best.g = g;
                best.threads = 32 * warps;
                best.per_sm = m;
                best.smem = (size_t)smem;
                best.inbox_bytes = (size_t)(2 * g.parity) * sizeof(ResWord);
                best.ok = true;
            }
        }
    }
    return best;
}
}  // namespace

// One block per SM; two for a temperature lattice whose boxes would have more
// than one task per warp (192 x 48 x 24: 1.84 / 1.67 us a step against 2.06 /
// 1.92 with one; the flow's boxes lose more to their larger surface: 64^3 5.28 /
// 5.11 against 4.42 / 4.34).
ResPlan resident_plan(int stencil, int storage, ResPhase ph, int nx, int ny, int nz) {
    int tasks = 0;
    ResPlan p = plan_boxes(stencil, storage, ph, nx, ny, nz, 1, tasks);
    if ((ph == RP_THERM || ph == RP_TADJ) && storage != 0 && (!p.ok || tasks > kResThreads(4) / 32)) {
        const ResPlan two = plan_boxes(stencil, storage, ph, nx, ny, nz, 2, tasks);
        if (two.ok) p = two;
    }
    return p;
}

namespace {
// Every population of every border node, for one cut and set of symmetry
// planes: the item of a word it is sent in has to be the one that its receiver
// (the node and population it reaches by plain wrapping and reflecting) takes
// it from, inside the inboxes and used once; and every word that is waited for
// has to be sent.
template <class P>
long long exchange_mismatches(const ResGeom& g, int mirror, std::vector<long long>& leaves) {
    using L = typename P::L;
    constexpr int NP = res_per_word<P>();
    const int dim[3] = {g.nx, g.ny, g.nz};
    const int blocks = g.px * g.py * g.pz;
    std::vector<long long> reader((size_t)g.parity * 3, -1);  // per item place: node * Q + population
    std::vector<int> waits((size_t)g.parity, 0);
    long long bad = 0, sent = 0, read = 0;
    bad += res_first<P>(g, 3 * L::Q) > g.inbox;
    for (int pass = 0; pass < 2; ++pass)
        for (int blk = 0; blk < blocks; ++blk) {
            const ResBox b = res_box(g, blk);
            long long items = 0;
            for (int e = 0; e < 3 * L::Q; ++e) {
                const ResLink l = res_link<P>(g, mirror, b, e);
                const int first = res_first<P>(g, e), next = res_first<P>(g, e + 1);
                for (int w = first; w < next; ++w) {
                    int got = 0;
                    for (int u = 0; u < NP; ++u) {
                        int at[3];
                        if (!res_item<P>(g, b, e, l.own_key, w - first + u * (next - first), at)) continue;
                        ++items;
                        const int q[3] = {b.x0 + at[0], b.y0 + at[1], b.z0 + at[2]};
                        const long long n = q[0] + (long long)g.nx * (q[1] + (long long)g.ny * q[2]);
                        if (pass == 0) {
                            const long long p = 3 * ((long long)blk * g.inbox + w) + got++;
                            if (p < 0 || p >= 3 * g.parity) { ++bad; continue; }
                            reader[p] = n * L::Q + L::opp(e / 3);
                            waits[p / 3] = 1;
                            ++read;
                            continue;
                        }
                        const long long place = (long long)l.block * g.inbox + res_first<P>(g, l.back) + w - first;
                        const long long p = 3 * place + got++;
                        if (p < 0 || p >= 3 * g.parity) { ++bad; continue; }
                        ++sent;
                        waits[place] = 0;
                        int to[3], arr[3];
                        for (int c = 0; c < 3; ++c) {
                            arr[c] = res_move<P>(e / 3, c);
                            to[c] = q[c] + arr[c];
                            if (to[c] < 0 || to[c] >= dim[c]) {
                                if (mirror >> c & 1) {
                                    to[c] = to[c] < 0 ? -1 - to[c] : 2 * dim[c] - 1 - to[c];
                                    arr[c] = -arr[c];
                                } else {
                                    to[c] = (to[c] + dim[c]) % dim[c];
                                }
                            }
                        }
                        int j = 0;
                        for (int c = 1; c < L::Q; ++c)
                            if (res_move<P>(c, 0) == arr[0] && res_move<P>(c, 1) == arr[1] && res_move<P>(c, 2) == arr[2]) j = c;
                        const long long r = to[0] + (long long)g.nx * (to[1] + (long long)g.ny * to[2]);
                        bad += reader[p] != r * L::Q + j;
                        reader[p] = -2;  // a second sender would find it taken
                    }
                }
            }
            // the items are all (node, population) pairs that leave (whatever the
            // symmetry planes); the others stay in the box
            if (mirror || pass) {
                bad += items != leaves[blk];
                continue;
            }
            long long leaving = 0;
            for (int lz = 0; lz < b.ez; ++lz)
                for (int ly = 0; ly < b.ey; ++ly)
                    for (int lx = 0; lx < b.ex; ++lx)
                        for (int i = 1; i < L::Q; ++i) {
                            const int out = res_out_bit<P>(i, 0) | res_out_bit<P>(i, 1) | res_out_bit<P>(i, 2);
                            if (res_mask(b, lx, ly, lz) & out) {
                                ++leaving;
                                continue;
                            }
                            const int far = lx + b.sy * ly + b.sz * lz + res_move<P>(i, 0) + res_move<P>(i, 1) * b.sy +
                                            res_move<P>(i, 2) * b.sz;
                            bad += far < 0 || far >= g.cap;
                        }
            leaves[blk] = leaving;
            bad += items != leaving;
        }
    for (int w : waits) bad += w;
    return bad + (sent != read);
}

// the exchange is the same for phases of equal cuts whose populations move the
// same way, as one or three to a word
struct Checked {
    ResGeom g;
    int way, per_word;
};

template <class P>
long long exchange_check(int stencil, int storage, ResPhase ph, int nx, int ny, int nz, std::vector<Checked>& done) {
    const ResPlan p = resident_plan(stencil, storage, ph, nx, ny, nz);
    if (!p.ok) return 0;
    for (const Checked& d : done)
        if (d.way == P::S && d.per_word == res_per_word<P>() && d.g.bx == p.g.bx && d.g.by == p.g.by &&
            d.g.bz == p.g.bz && d.g.cap == p.g.cap && d.g.inbox == p.g.inbox)
            return 0;
    done.push_back({p.g, P::S, res_per_word<P>()});
    long long bad = 0;
    std::vector<long long> leaves((size_t)p.g.px * p.g.py * p.g.pz);
    for (int mirror = 0; mirror < (stencil == 0 ? 4 : 8); ++mirror) bad += exchange_mismatches<P>(p.g, mirror, leaves);
    return bad;
}

// every phase that a context of one storage can have
template <typename R>
long long exchange_checks(int stencil, int storage, int nx, int ny, int nz, std::vector<Checked>& done) {
    auto check = [&](auto phase, ResPhase ph) {
        return exchange_check<decltype(phase)>(stencil == 0 ? 0 : 1, storage, ph, nx, ny, nz, done);
    };
    if (stencil == 0) return check(ResFlow<D2Q9, R, R, R>(), RP_FLOW) + check(ResAdjoint<D2Q9, R, R, false>(), RP_ADJ);
    if (stencil == 1)
        return check(ResFlow<D3Q19, R, R, R>(), RP_FLOW) + check(ResAdjoint<D3Q19, R, R, false>(), RP_ADJ) +
               check(ResAdjoint<D3Q19, R, R, true>(), RP_ADJ_T);
    return check(ResHeat<R, R, R>(), RP_THERM) + check(ResHeatAdjoint<R, R>(), RP_TADJ);
}
}  // namespace

long long resident_mismatches(int stencil, int nx, int ny, int nz) {
    std::vector<Checked> done;
    long long bad = exchange_checks<double>(stencil, 0, nx, ny, nz, done);
    for (int storage = 1; storage < (stencil == 0 ? 2 : 4); ++storage)
        bad += exchange_checks<float>(stencil, storage, nx, ny, nz, done);
    return bad;
}

cudaError_t resident_flow_f64(int stencil, ResPhase ph, const FlowLaunch& a, const ResPlan& p, const ResWords& w,
                              int steps, cudaStream_t s);
cudaError_t resident_thermal_f64(ResPhase ph, const ThermLaunch& a, const ResPlan& p, const ResWords& w,
                                 int steps, cudaStream_t s);

cudaError_t resident_flow(int stencil, int storage, ResPhase ph, const FlowLaunch& a, const ResPlan& p, const ResWords& w,
                          int steps, cudaStream_t s) {
    using dispatch::flow_args;
    if (storage == 0) return resident_flow_f64(stencil, ph, a, p, w, steps, s);
    if (ph == RP_FLOW) {
        if (stencil == 0) return launch_resident<ResFlow<D2Q9, float, float, float>>(flow_args<1>(a), p, w, steps, s);
        if (storage == 1) return launch_resident<ResFlow<D3Q19, float, float, float>>(flow_args<1>(a), p, w, steps, s);
        if (storage == 2) return launch_resident<ResFlow<D3Q19, __half, float, float>>(flow_args<2>(a), p, w, steps, s);
        return launch_resident<ResFlow<D3Q19, __nv_bfloat16, float, float>>(flow_args<3>(a), p, w, steps, s);
    }
    // the adjoint populations are FP32 in every 32-bit mode
    const auto x = flow_args<1>(a);
    if (stencil == 0) return launch_resident<ResAdjoint<D2Q9, float, float, false>>(x, p, w, steps, s);
    if (ph == RP_ADJ) return launch_resident<ResAdjoint<D3Q19, float, float, false>>(x, p, w, steps, s);
    return launch_resident<ResAdjoint<D3Q19, float, float, true>>(x, p, w, steps, s);
}

cudaError_t resident_thermal(int storage, ResPhase ph, const ThermLaunch& a, const ResPlan& p, const ResWords& w,
                             int steps, cudaStream_t s) {
    if (storage == 0) return resident_thermal_f64(ph, a, p, w, steps, s);
    const auto x = dispatch::therm_args<1>(a);
    if (ph == RP_THERM) return launch_resident<ResHeat<float, float, float>>(x, p, w, steps, s);
    return launch_resident<ResHeatAdjoint<float, float>>(x, p, w, steps, s);
}

}  // namespace lbm
