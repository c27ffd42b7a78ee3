// lbm_resident.cuh -- many steps of one lattice in one launch, the populations
// held in shared memory.
//
// A step of a small or middle-sized lattice through its own launch costs the
// fixed 2.1-2.3 us of a dependent launch, and moves every population through
// L2 twice.  Here one co-resident block per SM owns a box of the lattice and
// keeps its populations in shared memory for all the steps of a launch; only
// the populations that cross into a neighbour's box travel through L2.
//
// In place (two-step pattern): at the start of an even step slot i of a node
// holds the population that arrives there in direction i; the step writes the
// post-collision value of i to the node's own slot opp(i).  An odd step reads
// value i from slot opp(i) of the node it comes from and writes the result
// to slot i of the node it goes to.  Either way a node reads value i and writes
// value opp(i) at the same slot, so one copy of the populations suffices and
// the nodes of a step may run in any order; a barrier separates the steps of a
// block.  Where the node that value i comes from lies outside the box, that
// slot is the node's own slot i in both kinds of step.
//
// Exchange: the populations that leave the box are stored, three with the
// number of the step in one 128-bit word (64-bit values: one), into the inbox
// of the box they enter.  A reader polls the word itself until it carries the
// expected number, so there is no flag, no fence and no barrier between
// blocks: measured 0.43 us a step for such an exchange over 152 blocks against
// 1.8-2.4 us with data, fence and flag.  A word's place in an inbox is that of
// the word which answers it, so one list per box says for each word which slots
// it is sent from and received into, and the same thread does both.  Two
// inboxes alternate.  A word is overwritten two steps later, when the sender
// has received all words of the step between, which its neighbours sent after
// a barrier that followed their reading.
//
// The nodes are listed border first, 32 to a task, a node's lane its place
// modulo 32: with an odd number of populations per place the lanes of a task
// then meet 32 different banks wherever the rows of the box end (1.9 instead of
// 1 accesses per request without, and the shared memory was what 64^3 waited
// for).  Every warp computes border tasks first.  The last warps, which have
// the fewest tasks left, then send, take their interior tasks while the words
// travel, and receive; the others only announce that their border is done.  A
// wall node reflects every population: value opp(i) becomes value i, which is
// the slot's content already, so walls take no part in the steps.
//
// Every wait is bounded: after kWaitLimit polls the block sets an error flag,
// waits no more and the launch ends; the input populations are untouched.
//
// The node arithmetic is that of the one-step kernels, operation by operation.
//
// Measured, us a step (forward / adjoint) in launches of 500 steps against one
// launch per step: 16^3 1.73 / 1.63 against 2.27 / 2.56, 32^3 2.23 / 2.21 against
// 3.1 / 2.8, 64^3 FP32 4.40 / 4.36 against 5.65 / 5.73, temperature at
// 192 x 48 x 24 1.78 / 1.70 against 4.13 / 4.38; 32^3 FP64 16.7 / 14.8 against
// 29.5 / 31.5.  The set-up of a launch takes 20 us at 16^3 and 90 at 64^3 (the
// nodes of a box are listed by one warp each), so short blocks do not go resident.
// At 64^3 a block issues 20000 warp instructions a step (5000 cycles of each
// scheduler) and takes about 8500 cycles: what bounds it is the chain border -
// barrier - words - barrier, of which the travel of the words is about 1500.
#pragma once

#include "lbm_device.cuh"
#include "lbm_internal.h"

namespace lbm {

// ---------------------------------------------------------------------------
// one exchanged word: values and step number, written and read whole
// ---------------------------------------------------------------------------
struct alignas(16) ResWord {
    unsigned long long lo, hi;
};
// (volatile without a memory clobber: the shared-memory accesses around them
// are ordered by the barriers, and those of the next words may overlap)
__device__ __forceinline__ void word_st(ResWord* p, ResWord w) {
    asm volatile("{\n.reg .b128 w;\nmov.b128 w, {%1, %2};\nst.relaxed.gpu.global.b128 [%0], w;\n}" ::"l"(p),
                 "l"(w.lo), "l"(w.hi));
}
__device__ __forceinline__ ResWord word_ld(const ResWord* p) {
    ResWord w;
    asm volatile("{\n.reg .b128 w;\nld.relaxed.gpu.global.b128 w, [%2];\nmov.b128 {%0, %1}, w;\n}"
                 : "=l"(w.lo), "=l"(w.hi)
                 : "l"(p));
    return w;
}
__device__ __forceinline__ uint32_t word_tag(const ResWord& w) { return (uint32_t)(w.hi >> 32); }

// stored population <-> compute value <-> the bits of an exchanged word
template <typename T> struct Slot;
template <> struct Slot<float> {
    __device__ __forceinline__ static float dec(float v) { return v; }
    __device__ __forceinline__ static float enc(float v) { return v; }
    __device__ __forceinline__ static uint32_t bits(float v) { return __float_as_uint(v); }
    __device__ __forceinline__ static float unbits(uint32_t b) { return __uint_as_float(b); }
};
template <> struct Slot<double> {
    __device__ __forceinline__ static double dec(double v) { return v; }
    __device__ __forceinline__ static double enc(double v) { return v; }
};
template <> struct Slot<__half> {
    __device__ __forceinline__ static float dec(__half v) { return __half2float(v); }
    __device__ __forceinline__ static __half enc(float v) { return __float2half_rn(v); }
    __device__ __forceinline__ static uint32_t bits(__half v) { return __half_as_ushort(v); }
    __device__ __forceinline__ static __half unbits(uint32_t b) { return __ushort_as_half((unsigned short)b); }
};
template <> struct Slot<__nv_bfloat16> {
    __device__ __forceinline__ static float dec(__nv_bfloat16 v) { return __bfloat162float(v); }
    __device__ __forceinline__ static __nv_bfloat16 enc(float v) { return __float2bfloat16_rn(v); }
    __device__ __forceinline__ static uint32_t bits(__nv_bfloat16 v) { return __bfloat16_as_ushort(v); }
    __device__ __forceinline__ static __nv_bfloat16 unbits(uint32_t b) { return __ushort_as_bfloat16((unsigned short)b); }
};

// a word's slots, as byte offsets: 64-bit values one, the others three (a word
// with fewer nodes fills up with a spare slot that nothing reads)
template <typename T>
__device__ __forceinline__ T& slot_at(unsigned char* sm, uint32_t offset) {
    return *reinterpret_cast<T*>(sm + offset);
}
template <typename T>
__device__ __forceinline__ ResWord word_pack(unsigned char* sm, const uint4& e, uint32_t tag) {
    ResWord w;
    if constexpr (sizeof(T) == 8) {
        w.lo = (unsigned long long)__double_as_longlong(slot_at<T>(sm, e.x));
        w.hi = (unsigned long long)tag << 32;
    } else {
        const uint32_t a = Slot<T>::bits(slot_at<T>(sm, e.x)), b = Slot<T>::bits(slot_at<T>(sm, e.y)),
                       c = Slot<T>::bits(slot_at<T>(sm, e.z));
        asm("mov.b64 %0, {%1, %2};" : "=l"(w.lo) : "r"(a), "r"(b));
        asm("mov.b64 %0, {%1, %2};" : "=l"(w.hi) : "r"(c), "r"(tag));
    }
    return w;
}
template <typename T>
__device__ __forceinline__ void word_unpack(unsigned char* sm, const uint4& e, const ResWord& w) {
    if constexpr (sizeof(T) == 8) {
        slot_at<T>(sm, e.x) = __longlong_as_double((long long)w.lo);
    } else {
        slot_at<T>(sm, e.x) = Slot<T>::unbits((uint32_t)w.lo);
        slot_at<T>(sm, e.y) = Slot<T>::unbits((uint32_t)(w.lo >> 32));
        slot_at<T>(sm, e.z) = Slot<T>::unbits((uint32_t)w.hi);
    }
}

// ---------------------------------------------------------------------------
// the four phases: what a node keeps beside its populations, and its update
// ---------------------------------------------------------------------------
template <class L_, typename T_, typename TA, typename R_>
struct ResFlow {
    using L = L_;
    using T = T_;
    using R = R_;
    using Args = FlowArgs<T, TA, R>;
    static constexpr int S = 1;      // a population moves along S e_i
    static __device__ __forceinline__ bool reflects(int fl) { return (fl & 7) == WALL; }  // and does nothing else
    static constexpr int NAUX = 1;   // gamma
    static constexpr int NBC = 3;    // boundary values, read at open nodes only
    static __device__ __forceinline__ int bc_at(int c) { return c; }
    static __device__ __forceinline__ const T* in(const Args& a) { return a.fin; }
    static __device__ __forceinline__ T* out(const Args& a) { return a.fout; }
    static __device__ __forceinline__ void aux(const Args& a, long long n, int fl, R (&x)[NAUX]) {
        x[0] = (fl & 7) != WALL ? a.gamma[n] : R(0);
    }
    static __device__ __forceinline__ bool special(int fl) { return (fl & 7) != FLUID; }
    // SPECIAL: the node may be other than fluid
    template <bool SPECIAL, class Bc>
    static __device__ __forceinline__ void update(const Args& a, int fl, const R (&x)[NAUX], R (&f)[L::Q], Bc bc) {
        const int type = fl & 7;
        if (SPECIAL && type >= VEL) {
            const R v[3] = {bc(0), bc(1), bc(2)};
            zou_he<L, true>(f, type, (fl >> 3) & 7, v, a.rho0);
        }
        double acc[2];
        flow_collide<L, T, TA, R, false>(a, 0, SPECIAL ? fl : FLUID, x[0], f, acc);
    }
};

template <class L_, typename TA, typename R_, bool THERMAL>
struct ResAdjoint {
    using L = L_;
    using T = TA;
    using R = R_;
    using Args = FlowArgs<TA, TA, R>;
    static constexpr int S = -1;
    static __device__ __forceinline__ bool reflects(int fl) { return (fl & 7) == WALL; }
    static constexpr int NAUX = THERMAL ? 7 : 4;  // gamma, u, coupling
    static constexpr int NBC = 0;
    static __device__ __forceinline__ int bc_at(int c) { return c; }
    static __device__ __forceinline__ const T* in(const Args& a) { return a.ain; }
    static __device__ __forceinline__ T* out(const Args& a) { return a.aout; }
    static __device__ __forceinline__ void aux(const Args& a, long long n, int, R (&x)[NAUX]) {
        x[0] = a.gamma[n];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            x[1 + k] = a.u[k * a.np + n];
            if constexpr (THERMAL) x[4 + k] = a.cpl[k * a.np + n];
        }
    }
    static __device__ __forceinline__ bool special(int fl) { return (fl & 7) != FLUID; }
    template <bool SPECIAL, class Bc>
    static __device__ __forceinline__ void update(const Args& a, int fl, const R (&x)[NAUX], R (&s)[L::Q], Bc) {
        const int type = fl & 7;
        R v0 = 0, v1 = 0, v2 = 0;
        if constexpr (THERMAL) { v0 = x[4]; v1 = x[5]; v2 = x[6]; }
        adjoint_collide_values<L, R>(a.omega, a.model, a.src_in, SPECIAL && type == VEL, x[0], x[1], x[2], x[3], v0, v1,
                                         v2, s);
        if (SPECIAL && type >= VEL) zou_he_adjoint<L, true>(s, type, (fl >> 3) & 7);
    }
};

template <typename TG, typename TA, typename R_>
struct ResHeat {
    using L = D3Q7;
    using T = TG;
    using R = R_;
    using Args = ThermArgs<TG, TA, R>;
    static constexpr int S = 1;
    static __device__ __forceinline__ bool reflects(int fl) { return (fl & (7 | HEAT_BIT)) == WALL; }
    static constexpr int NAUX = 5;  // 1/tau_g, gamma, u
    static constexpr int NBC = 1;   // T_in
    static __device__ __forceinline__ int bc_at(int) { return 3; }
    static __device__ __forceinline__ const T* in(const Args& a) { return a.gin; }
    static __device__ __forceinline__ T* out(const Args& a) { return a.gout; }
    static __device__ __forceinline__ void aux(const Args& a, long long n, int, R (&x)[NAUX]) {
        x[1] = a.gamma[n];
        x[0] = R(1) / tau_g<R>(x[1], a.kappa_f, a.k_ratio);
#pragma unroll
        for (int k = 0; k < 3; ++k) x[2 + k] = a.u[k * a.np + n];
    }
    static __device__ __forceinline__ bool special(int fl) { return (fl & 7) != FLUID; }
    template <bool SPECIAL, class Bc>
    static __device__ __forceinline__ void update(const Args& a, int fl, const R (&x)[NAUX], R (&g)[7], Bc bc) {
        const int type = fl & 7;
        if (SPECIAL && type != FLUID) {
            const R v[4] = {R(0), R(0), R(0), bc(0)};
            thermal_bc<R>(g, fl, v, x[1], x[2], x[3], x[4], a.q);
        }
        if (!SPECIAL || type != WALL) {
            R tem = 0;
#pragma unroll
            for (int k = 0; k < 7; ++k) tem = Ex<R>::add(tem, g[k]);
            thermal_collide_values<R>(a.beta, g, tem, x[0], x[1], x[2], x[3], x[4]);
        }
    }
};

template <typename TA, typename R_>
struct ResHeatAdjoint {
    using L = D3Q7;
    using T = TA;
    using R = R_;
    using Args = ThermArgs<TA, TA, R>;
    static constexpr int S = -1;
    static __device__ __forceinline__ bool reflects(int fl) { return (fl & 7) == WALL; }
    static constexpr int NAUX = 5;
    static constexpr int NBC = 0;
    static __device__ __forceinline__ int bc_at(int c) { return c; }
    static __device__ __forceinline__ const T* in(const Args& a) { return a.ain; }
    static __device__ __forceinline__ T* out(const Args& a) { return a.aout; }
    static __device__ __forceinline__ void aux(const Args& a, long long n, int fl, R (&x)[NAUX]) {
        ResHeat<TA, TA, R>::aux(a, n, fl, x);
    }
    static __device__ __forceinline__ bool special(int fl) { return (fl & 7) != FLUID; }
    template <bool SPECIAL, class Bc>
    static __device__ __forceinline__ void update(const Args& a, int fl, const R (&x)[NAUX], R (&s)[7], Bc) {
        R ckn;
        thermal_adjoint_update<R>(a.src_q, a.src_T, a.beta, SPECIAL ? fl : FLUID, x[0], x[1], x[2], x[3], x[4], s, ckn);
    }
};

// ---------------------------------------------------------------------------
// lattice geometry of the exchange
// ---------------------------------------------------------------------------
// component a of the displacement of population i in a step
template <class P>
__host__ __device__ constexpr int res_move(int i, int a) {
    return P::S * ecomp_of<typename P::L>(i, a);
}
// face bit that population i enters a box through along axis a (bit 2a low, 2a + 1 high), and leaves it
template <class P>
__host__ __device__ constexpr int res_in_bit(int i, int a) {
    const int m = a < 0 ? 0 : res_move<P>(i, a);
    return m > 0 ? 1 << (2 * a) : (m < 0 ? 2 << (2 * a) : 0);
}
template <class P>
__host__ __device__ constexpr int res_out_bit(int i, int a) {
    const int m = a < 0 ? 0 : res_move<P>(i, a);
    return m > 0 ? 2 << (2 * a) : (m < 0 ? 1 << (2 * a) : 0);
}
struct ResShared {
    int first[3 * 19 + 1];  // inbox place of each group's first word
    int move[3 * 19];       // from there to its place in the receiving inbox
    int own_key[3 * 19];    // numbering of its items (res_link)
    int tasks[3];           // of the border, the interior, the walls
    int lane[3][32];        // nodes of a list and lane
    int over[3];            // nodes placed beyond their lane's share
    int bail;
    int limit;              // polls of a wait
};
static_assert(sizeof(ResShared) <= kResHead, "head of the shared memory");

// the block's own constants
struct ResBox {
    int q[3];             // place among the boxes
    int x0, y0, z0;       // first node
    int ex, ey, ez;       // nodes per axis
    int sy, sz;           // shared-memory slots between rows, between planes
};

__host__ __device__ __forceinline__ ResBox res_box(const ResGeom& g, int block) {
    ResBox b;
    b.q[0] = block % g.px;
    b.q[1] = (block / g.px) % g.py;
    b.q[2] = block / (g.px * g.py);
    b.x0 = b.q[0] * g.bx;
    b.y0 = b.q[1] * g.by;
    b.z0 = b.q[2] * g.bz;
    b.ex = g.nx - b.x0 < g.bx ? g.nx - b.x0 : g.bx;
    b.ey = g.ny - b.y0 < g.by ? g.ny - b.y0 : g.by;
    b.ez = g.nz - b.z0 < g.bz ? g.nz - b.z0 : g.bz;
    b.sy = g.pitch;
    b.sz = g.pitch * g.by;
    return b;
}

// faces of the box that a node lies on
__host__ __device__ __forceinline__ int res_mask(const ResBox& b, int lx, int ly, int lz) {
    return (lx == 0) | (lx == b.ex - 1) << 1 | (ly == 0) << 2 | (ly == b.ey - 1) << 3 | (lz == 0) << 4 |
           (lz == b.ez - 1) << 5;
}

// A group is one population and one set of axes across which it leaves a box
// (e = 3 i + 0: its first axis, 1: its second, 2: both).  Its words have places
// [first, next group's first) in every inbox, sized for a whole box.
template <class P>
__host__ __device__ __forceinline__ int res_crosses(int e, int a) {  // the crossing's direction along axis a, 0: none
    int m[3], k = 0, at = -1;
    for (int c = 0; c < 3; ++c) {
        m[c] = P::S * ecomp_of<typename P::L>(e / 3, c);
        if (m[c]) {
            if (c == a) at = k;
            ++k;
        }
    }
    const int cse = e % 3;
    if (at < 0 || (cse > 0 && k < 2)) return 0;
    return cse == 2 || cse == at ? m[a] : 0;
}
template <class P>
__host__ __device__ __forceinline__ int res_items(const ResGeom& g, int e) {  // nodes of a whole box in the group
    const int b[3] = {g.bx, g.by, g.bz};
    int n = 1;
    bool any = false;
    for (int a = 0; a < 3; ++a) {
        if (res_crosses<P>(e, a)) any = true;
        else n *= b[a];
    }
    return any ? n : 0;
}
template <class P>
__host__ __device__ constexpr int res_per_word() {
    return sizeof(typename P::R) == 8 ? 1 : 3;
}
template <class P>
__host__ __device__ __forceinline__ int res_first(const ResGeom& g, int e) {
    int n = 0;
    for (int c = 0; c < e; ++c) n += (res_items<P>(g, c) + res_per_word<P>() - 1) / res_per_word<P>();
    return n;
}

// where a group's populations arrive
struct ResLink {
    int block;     // the box they enter
    int back;      // group of that box which travels the same way back
    bool own_key;  // items are numbered by this box's nodes (else by the receivers')
};
template <class P>
__host__ __device__ ResLink res_link(const ResGeom& g, int mirror, const ResBox& b, int e) {
    using L = typename P::L;
    const int i = e / 3;
    const int parts[3] = {g.px, g.py, g.pz};
    int blk[3] = {b.q[0], b.q[1], b.q[2]}, back[3];  // back: displacement of the way back
    for (int a = 0; a < 3; ++a) {
        back[a] = -P::S * ecomp_of<L>(i, a);
        const int m = res_crosses<P>(e, a);
        if (!m) continue;
        const int to = blk[a] + m;
        if (to >= 0 && to < parts[a]) blk[a] = to;
        else if (mirror >> a & 1) back[a] = m;       // symmetry plane: stays, and leaves by the same face
        else blk[a] = to < 0 ? parts[a] - 1 : 0;
    }
    int k = 0;
    for (int c = 1; c < L::Q; ++c)
        if (P::S * L::cx(c) == back[0] && P::S * L::cy(c) == back[1] && P::S * L::cz(c) == back[2]) k = c;
    ResLink l;
    l.block = blk[0] + g.px * (blk[1] + g.py * blk[2]);
    l.back = 3 * k + e % 3;
    l.own_key = i <= k;
    return l;
}

// node of item p of a group: false when this (cut) box has none.  Both boxes of
// a link number the items alike: by the coordinates of the side with the lower
// population, along the axes that are not crossed.  Word w of a group of n has
// the items w, w + n and w + 2 n: neighbouring lanes, neighbouring nodes.
template <class P>
__host__ __device__ bool res_item(const ResGeom& g, const ResBox& b, int e, bool own_key, int p, int (&at)[3]) {
    const int nom[3] = {g.bx, g.by, g.bz}, ext[3] = {b.ex, b.ey, b.ez};
    for (int a = 0; a < 3; ++a) {
        const int m = P::S * ecomp_of<typename P::L>(e / 3, a);
        if (const int c = res_crosses<P>(e, a)) {
            at[a] = c > 0 ? ext[a] - 1 : 0;
            continue;
        }
        at[a] = p % nom[a] - (own_key ? 0 : m);
        p /= nom[a];
        const int to = at[a] + m;
        if (at[a] < 0 || at[a] >= ext[a] || to < 0 || to >= ext[a]) return false;
    }
    return p == 0;
}

// ---------------------------------------------------------------------------
// the block's words
// ---------------------------------------------------------------------------
constexpr uint32_t kNoNode = 0xffffffffu;

template <class P>
struct ResBlock {
    using R = typename P::R;
    using T = typename P::T;
    ResBox b;
    ResShared* sh;
    T* sm;                 // populations
    const R* aux;          // per-node constants
    const uint32_t* info;  // per listed node: place (13 bits), faces (6), flag (7); kNoNode: none
    const uint4* word;     // per inbox place: three slots, in w the place in the receiving inbox (from this box's)
    ResWord* boxes;        // all inboxes
    int* err;
    int border, inner, walls;  // places of the three lists (multiples of 32)
    int syq, szq;          // slots between rows, between planes
    uint32_t my, mz;       // 2^32 / row length, / plane size, rounded up
};

// Exchanging thread t has the places t, t + nt, ... of the inbox, n at most.
// A place without a node is sent to itself: no lane differs from its
// neighbours, and every load of a batch of U is under way before the first is
// looked at.
template <class P, int U>
__device__ __forceinline__ void res_send(const ResBlock<P>& B, const ResGeom& g, ResWord* __restrict__ own, uint32_t tag,
                                         int t, int nt) {
    using T = typename P::T;
    unsigned char* const sm = reinterpret_cast<unsigned char*>(B.sm);
#pragma unroll 1
    for (; t < g.inbox; t += U * nt) {
        uint4 e[U];
        ResWord v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) e[u] = B.word[t + u * nt < g.inbox ? t + u * nt : t];
#pragma unroll
        for (int u = 0; u < U; ++u) v[u] = word_pack<T>(sm, e[u], tag);
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (t + u * nt < g.inbox) word_st(own + (int)e[u].w, v[u]);
    }
}

// wait for the words and put them into their slots
template <class P, int U>
__device__ __forceinline__ void res_receive(const ResBlock<P>& B, const ResGeom& g, const ResWord* __restrict__ own,
                                            uint32_t tag, int t, int nt) {
    unsigned char* const sm = reinterpret_cast<unsigned char*>(B.sm);
#pragma unroll 1
    for (; t < g.inbox; t += U * nt) {
        ResWord v[U];
        for (int spins = 0;; ++spins) {
            // one vote: a lane that left by itself would be missing in the others'
            // next one (the flag is read while the words travel: 64^3 loses 0.3 % of a
            // step to it, 0.7 % with a vote of its own)
            const int gone = *(volatile int*)&B.sh->bail;
            uint32_t bad = 0;
#pragma unroll
            for (int u = 0; u < U; ++u) v[u] = word_ld(own + (t + u * nt < g.inbox ? t + u * nt : t));
#pragma unroll
            for (int u = 0; u < U; ++u) bad |= word_tag(v[u]) ^ tag;
            if (!__any_sync(0xffffffffu, gone ? 0u : bad)) break;
            if (spins >= B.sh->limit) {
                *(volatile int*)&B.sh->bail = 1;
                atomicExch(B.err, 1);
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (t + u * nt < g.inbox) word_unpack<typename P::T>(sm, B.word[t + u * nt], v[u]);
    }
}

// ---------------------------------------------------------------------------
// steps
// ---------------------------------------------------------------------------
enum ResStep { RES_FIRST = 0, RES_EVEN, RES_ODD };

// one node of a step.  RES_FIRST pulls from global memory as the one-step
// kernels do and writes as an even step; last: store to global memory.
template <class P, int STEP, bool BORDER, bool REFLECTS = false>
__device__ __forceinline__ void res_node(const typename P::Args& a, const ResGeom& g, const ResBlock<P>& B, int j,
                                         bool last) {
    using L = typename P::L;
    using R = typename P::R;
    using T = typename P::T;
    constexpr int Q = L::Q;
    const uint32_t w = B.info[j];
    if (w == kNoNode) return;
    const int k = w & 0x1fff, mask = (w >> 13) & 63, fl = w >> 19;
    int x0, y0, z0;  // the node, computed where it is needed
    auto place = [&]() {
        const int lz = B.b.sz == 1 ? k : (int)__umulhi((uint32_t)k, B.mz), r = k - lz * B.b.sz;
        const int ly = B.b.sy == 1 ? r : (int)__umulhi((uint32_t)r, B.my);
        x0 = B.b.x0 + r - ly * B.b.sy;
        y0 = B.b.y0 + ly;
        z0 = B.b.z0 + lz;
        return x0 + g.nx * (y0 + g.ny * z0);
    };
    R x[P::NAUX], f[Q];
#pragma unroll
    for (int c = 0; c < P::NAUX; ++c) x[c] = B.aux[c * g.list + j];
    // slot of value i (read) and of value opp(i) (written): a row of nodes, and a
    // constant within it
    const int own = k * Q;
    int row[9];
#pragma unroll
    for (int dz = -1; dz <= 1; ++dz)
#pragma unroll
        for (int dy = -1; dy <= 1; ++dy)
            row[4 + dy + 3 * dz] = own - (dy == 0 ? 0 : (dy > 0 ? B.syq : -B.syq)) -
                                   (dz == 0 ? 0 : (dz > 0 ? B.szq : -B.szq));
    int at[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        at[i] = own + i;
        if (STEP == RES_ODD) {
            const int from = row[4 + res_move<P>(i, 1) + 3 * res_move<P>(i, 2)] + (L::opp(i) - res_move<P>(i, 0) * Q);
            const int enters = res_in_bit<P>(i, 0) | res_in_bit<P>(i, 1) | res_in_bit<P>(i, 2);
            if (!BORDER || !(mask & enters)) at[i] = from;
        }
    }
    // opaque, or the multiples of the plane stride are kept in registers for all
    // nodes of all steps
    long long np = a.np;
    asm volatile("" : "+l"(np));
    if (STEP == RES_FIRST) {
        Cell c;
        c.n = place();
        c.x = x0;
        c.y = y0;
        c.z = z0;
        if (a.mirror && on_mirror_face(c, g.nx, g.ny, g.nz, a.mirror)) {
#pragma unroll
            for (int i = 0; i < L::Q; ++i)
                f[i] = Slot<T>::dec(__ldg(P::in(a) + mirror_src<L>(c, g.nx, g.ny, g.nz, np, a.mirror, i, -P::S)));
        } else {
            const Nbr o = neighbours(c, g.nx, g.ny, g.nz);
            const T* __restrict__ p = P::in(a) + c.n;
#pragma unroll
            for (int i = 0; i < L::Q; ++i, p += np) f[i] = Slot<T>::dec(__ldg(p + nbr_offset<L>(o, i, -P::S)));
        }
    } else {
#pragma unroll
        for (int i = 0; i < Q; ++i) f[i] = Slot<T>::dec(B.sm[at[i]]);
    }
    if (REFLECTS)
        bounce<L>(f);
    else
        P::template update<BORDER>(a, fl, x, f, [&](int c) { return B.aux[(P::NAUX + c) * g.list + j]; });
    if (last) {
        T* __restrict__ q = P::out(a) + place();
#pragma unroll
        for (int i = 0; i < Q; ++i, q += np) *q = Slot<T>::enc(f[i]);
    } else {
#pragma unroll
        for (int i = 0; i < Q; ++i) B.sm[at[i]] = Slot<T>::enc(f[L::opp(i)]);
    }
}

// a warp's share of a step; the words sent after it carry the number tag
template <class P, int STEP>
__device__ __forceinline__ void res_step(const typename P::Args& a, const ResGeom& g, const ResBlock<P>& B, uint32_t tag,
                                         bool last) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, warps = blockDim.x >> 5;
    const int nb = B.border >> 5, ni = B.inner >> 5;
    // walls: into their slots in the first step, reflected to global memory in the last
    if (STEP == RES_FIRST || last)
#pragma unroll 1
        for (int j = threadIdx.x; j < B.walls; j += blockDim.x)
            res_node<P, STEP, true, true>(a, g, B, B.border + B.inner + j, last);
#pragma unroll 1
    for (int q = warp; q < nb; q += warps) res_node<P, STEP, true>(a, g, B, 32 * q + lane, last);
    __syncwarp();
    const int t = (int)threadIdx.x - g.silent, nt = blockDim.x - g.silent;
    const int n = g.words;
    ResWord* const own = B.boxes + (tag & 1) * g.parity + (long long)blockIdx.x * g.inbox;
    if (t < 0) {
        asm volatile("bar.arrive 1, %0;" ::"r"((int)blockDim.x) : "memory");
    } else {
        asm volatile("bar.sync 1, %0;" ::"r"((int)blockDim.x) : "memory");
        if (!last) {
            if (n == 1) res_send<P, 1>(B, g, own, tag, t, nt);
            else if (n == 2) res_send<P, 2>(B, g, own, tag, t, nt);
            else res_send<P, 4>(B, g, own, tag, t, nt);
        }
    }
    // the warps that the last border round left idle come first
    int q = warp - nb % warps;
    if (q < 0) q += warps;
#pragma unroll 1
    for (; q < ni; q += warps) res_node<P, STEP, false>(a, g, B, B.border + 32 * q + lane, last);
    if (t >= 0 && !last) {
        __syncwarp();
        if (n == 1) res_receive<P, 1>(B, g, own, tag, t, nt);
        else if (n == 2) res_receive<P, 2>(B, g, own, tag, t, nt);
        else res_receive<P, 4>(B, g, own, tag, t, nt);
    }
    asm volatile("bar.sync 0, %0;" ::"r"((int)blockDim.x) : "memory");
}

// 64 registers a thread in 32-bit arithmetic, 168 in 64-bit: no phase spills
template <class P>
__global__ void __launch_bounds__(kResThreads(sizeof(typename P::R)), 1)
    k_resident(typename P::Args a, ResGeom g, void* inboxes, const unsigned* __restrict__ base, int* err, int limit,
               int steps) {
    using L = typename P::L;
    using R = typename P::R;
    using T = typename P::T;
    extern __shared__ __align__(16) unsigned char raw[];
    ResShared& sh = *reinterpret_cast<ResShared*>(raw);
    R* const aux = reinterpret_cast<R*>(raw + g.aux_at);
    uint32_t* const info = reinterpret_cast<uint32_t*>(aux + (size_t)(P::NAUX + P::NBC) * g.list);
    uint4* const word = reinterpret_cast<uint4*>(raw + g.word_at);
    ResBlock<P> B;
    B.b = res_box(g, blockIdx.x);
    B.sh = &sh;
    B.sm = reinterpret_cast<T*>(raw + kResHead);
    B.aux = aux;
    B.info = info;
    B.word = word;
    B.boxes = static_cast<ResWord*>(inboxes);
    B.err = err;
    const ResBox& b = B.b;
    if (threadIdx.x == 0) {
        sh.bail = 0;
        sh.limit = limit;
        for (int c = 0; c < 3; ++c) sh.over[c] = 0;
    }
    B.syq = b.sy * L::Q;
    B.szq = b.sz * L::Q;
    B.my = b.sy == 1 ? 0 : (uint32_t)((0x100000000ull + b.sy - 1) / b.sy);
    B.mz = b.sz == 1 ? 0 : (uint32_t)((0x100000000ull + b.sz - 1) / b.sz);
    constexpr int NP = res_per_word<P>();
    for (int e = threadIdx.x; e < 3 * L::Q; e += blockDim.x) sh.first[e + 1] = (res_items<P>(g, e) + NP - 1) / NP;
    __syncthreads();
    if (threadIdx.x == 0) {
        sh.first[0] = 0;
        for (int e = 0; e < 3 * L::Q; ++e) sh.first[e + 1] += sh.first[e];
    }
    __syncthreads();
    for (int e = threadIdx.x; e < 3 * L::Q; e += blockDim.x) {
        const ResLink l = res_link<P>(g, a.mirror, b, e);
        sh.move[e] = (l.block - (int)blockIdx.x) * g.inbox + sh.first[l.back] - sh.first[e];
        sh.own_key[e] = l.own_key;
    }
    __syncthreads();
    // the three lists.  First every place's list and order in it: 0..2 border (the
    // open nodes first, so that they fill warps of their own; those inside the
    // box too, so that interior tasks are free of their code), 3 interior, 4
    // wall, 5 not a node.
    unsigned char* const cls = raw + g.word_at;  // the words' list comes here later
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    auto coordinates = [&](int k, int& lx, int& ly, int& lz) {
        lz = k / b.sz;
        ly = (k - lz * b.sz) / b.sy;
        lx = k - lz * b.sz - ly * b.sy;
        return lx < b.ex && ly < b.ey && lz < b.ez;
    };
    auto faces = [&](int lx, int ly, int lz) { return res_mask(b, lx, ly, lz) & (L::Q == 9 ? 15 : 63); };
    for (int k = threadIdx.x; k < g.cap; k += blockDim.x) {
        int lx, ly, lz, c = 5;
        if (coordinates(k, lx, ly, lz)) {
            const int fl = a.flags[(b.x0 + lx) + (long long)g.nx * ((b.y0 + ly) + (long long)g.ny * (b.z0 + lz))];
            const int mask = faces(lx, ly, lz);
            if (P::reflects(fl)) c = 4;
            else if (P::special(fl)) c = 0;
            else c = !mask ? 3 : (mask & 60 ? 1 : 2);
        }
        cls[k] = (unsigned char)c;
    }
    __syncthreads();
    // a warp per list: lane r counts the nodes whose place is r modulo 32
    for (int c = wid; c < 3; c += nwarp) {
        int n = 0;
        for (int k = lane; k < g.cap; k += 32) n += (cls[k] < 3 ? 0 : cls[k] - 2) == c;
        sh.lane[c][lane] = n;
        for (int o = 16; o > 0; o >>= 1) n += __shfl_xor_sync(0xffffffffu, n, o);
        if (lane == 0) sh.tasks[c] = (n + 31) >> 5;
    }
    __syncthreads();
    B.border = 32 * sh.tasks[0];
    B.inner = 32 * sh.tasks[1];
    B.walls = 32 * sh.tasks[2];
    for (int j = threadIdx.x; j < g.list; j += blockDim.x) info[j] = kNoNode;
    __syncthreads();
    // place them: a lane's share in its column, what is beyond into the holes of
    // the others
    for (int c = wid; c < 3; c += nwarp) {
        const int start = c == 0 ? 0 : (c == 1 ? B.border : B.border + B.inner), share = sh.tasks[c];
        int n = 0;
        for (int sub = c == 0 ? 0 : c + 2; sub <= (c == 0 ? 2 : c + 2); ++sub)
            for (int k = lane; k < g.cap; k += 32) {
                if (cls[k] != sub) continue;
                int at = start + 32 * n + lane;
                if (n >= share) {
                    int hole = atomicAdd(&sh.over[c], 1), r = 0;
                    for (;; ++r) {
                        const int free = max(share - sh.lane[c][r], 0);
                        if (hole < free) break;
                        hole -= free;
                    }
                    at = start + 32 * (sh.lane[c][r] + hole) + r;
                }
                ++n;
                int lx, ly, lz;
                coordinates(k, lx, ly, lz);
                const int node = (b.x0 + lx) + g.nx * ((b.y0 + ly) + g.ny * (b.z0 + lz));
                info[at] = (uint32_t)k | (uint32_t)faces(lx, ly, lz) << 13 | (uint32_t)a.flags[node] << 19;
            }
    }
    __syncthreads();
    for (int j = threadIdx.x; j < g.list; j += blockDim.x) {
        const uint32_t w = info[j];
        if (w == kNoNode) continue;
        int lx, ly, lz;
        coordinates(w & 0x1fff, lx, ly, lz);
        R x[P::NAUX];
        const long long n = (b.x0 + lx) + (long long)g.nx * ((b.y0 + ly) + (long long)g.ny * (b.z0 + lz));
        P::aux(a, n, w >> 19, x);
#pragma unroll
        for (int c = 0; c < P::NAUX; ++c) aux[c * g.list + j] = x[c];
#pragma unroll
        for (int c = 0; c < P::NBC; ++c) aux[(P::NAUX + c) * g.list + j] = a.bc[4 * n + P::bc_at(c)];
    }
    __syncthreads();
    for (int w = threadIdx.x; w < g.inbox; w += blockDim.x) {
        const uint32_t spare = g.cap * L::Q;
        uint32_t slot[3] = {spare, spare, spare};
        int got = 0, to = w;
        if (w < sh.first[3 * L::Q]) {
            int e = 0;
            while (sh.first[e + 1] <= w) ++e;
            for (int u = 0; u < NP; ++u) {
                int at[3];
                if (!res_item<P>(g, b, e, sh.own_key[e], w - sh.first[e] + u * (sh.first[e + 1] - sh.first[e]), at))
                    continue;
                const uint32_t v = (at[0] + b.sy * at[1] + b.sz * at[2]) * L::Q + L::opp(e / 3);
                if (got == 0) slot[0] = v;
                else if (got == 1) slot[1] = v;
                else slot[2] = v;
                ++got;
            }
            if (got) to = w + sh.move[e];
        }
        word[w] = make_uint4(slot[0] * sizeof(T), slot[1] * sizeof(T), slot[2] * sizeof(T), (uint32_t)to);
    }
    __syncthreads();
    const uint32_t tag0 = *base;
    res_step<P, RES_FIRST>(a, g, B, tag0 + 1, steps == 1);
#pragma unroll 1
    for (int t = 1; t < steps; t += 2) {
        res_step<P, RES_ODD>(a, g, B, tag0 + t + 1, t == steps - 1);
        if (t + 1 < steps) res_step<P, RES_EVEN>(a, g, B, tag0 + t + 2, t + 1 == steps - 1);
    }
}

// launch with the arguments of a phase (returns the launch's error)
template <class P>
cudaError_t launch_resident(const typename P::Args& a, const ResPlan& p, const ResWords& w, int steps, cudaStream_t s) {
    cudaError_t e = cudaFuncSetAttribute(k_resident<P>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)p.smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(p.g.px * p.g.py * p.g.pz);
    cfg.blockDim = dim3(p.threads);
    cfg.dynamicSmemBytes = p.smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;  // all blocks are resident together
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_resident<P>, a, p.g, w.inboxes, w.base, w.err, w.limit, steps);
}

}  // namespace lbm
