// The walker update with several commits per round (mucal_launch_config
// .multi_commit): device code, one instantiation per lane count in
// walker_scan_<lanes>.cu.  The chain is the one-thread chain of
// walker_chain.cuh, bit for bit.
#pragma once

#include "walker_chain.cuh"

namespace mucal {
namespace {

// ---------------------------------------------------------------------------
// Several commits per round (multi-commit rounds) on a sliding window of W
// attempts, one per lane of the walker's group: slot (lane) t mod W holds
// attempt t, for the W attempts from the first undecided one (t0) on.  The
// place of a slot is its distance from t0's slot.
//
// A round evaluates the energy changes of the whole window against the state
// at its start.  Such a value stays right until an earlier attempt of the
// window commits a move next to one of the attempt's two sites or in one of
// its two list slots; which attempts touch which is a matter of the sites
// alone.  Taking all energy changes as they are, the decisions are a short
// serial recurrence in the energy, which every lane of the group runs
// redundantly in registers: T(E, dE_i) >= r_i ? E += dE_i.  The round then
// ends at the first attempt that an earlier accepted one touches: the
// attempts before it are decided as the serial chain decides them, commit
// together and give way to the next ones, and the window slides on.  The first
// attempt is never stopped, so every round decides at least one, mostly the
// whole window; no group of a warp waits for another's conflicts.
//
// Where the last round had few accepted moves in each walker of the warp, a
// round takes all decisions at its first energy, one threshold a lane, and
// ends with the first accepted attempt: no recurrence, no tests for touching,
// one commit to look for in the lists.  (Rounds of the recurrence without the
// tests for touching took, at 2D L = 40, N = 60, 64 walkers, 60 sweeps and
// acceptance 0.03, 0.254 ms, these 0.149; 2D L = 16, N = 32 at 0.04 0.319 and
// 0.209, rounds that always end at the first accepted attempt 0.223.  Few is a
// quarter of the window: an eighth 0.155 and 0.227, more than a quarter of the
// warp's attempts together instead 2D L = 64 1.12 -> 1.43 at 0.45.)
//
// The rounds are bound by the latency of dependent integer instructions and by
// issue slots (a walker is one serial chain, and an SM holds only tens of
// walkers): on 2D L = 64 at 8 lanes and 28 walkers per SM a round was about 540
// warp instructions, one issued every 4.0 cycles per warp, for 7.3 attempts
// per walker (18.3 warp instructions per attempt against 24 with one commit
// per round).  So independent work stands beside the recurrence, in the same
// straight line of code: the random numbers (2.77e10 -> 2.86e10 attempts/s)
// and the comparisons of the moves' sites (-> 2.95e10; one commit per round
// 1.7e10); with the rounds of few moves a path of their own the others have
// fewer instructions to choose between (20 sweeps 1.22 -> 1.15 ms).  Two attempts
// per lane, which halve what is done once per lane, issued as much and ran at
// half the warps: 2.07e10.
//
// A step of the recurrence is one threshold load from shared memory and a few
// dependent integer instructions: from the whole table (kThrShared), or from
// the walker's window of rows (kThrWindow, see ThrWindow), where an attempt
// reached with an energy whose row has not arrived is stopped like one with a
// conflict.  Where neither fits, the thresholds are read from global memory
// (kThrGlobal) ahead of the recurrence: every lane turns the kScanWords
// thresholds of an attempt's dE around the round's energy, contiguous in the
// table's dE-major copy, into a bit mask of decisions by energy, and the
// attempt is stopped when reached with another energy.
// ---------------------------------------------------------------------------
constexpr int kScanWords = 24;    // energies of a decision mask (bits 0-23; the lane's dE above)
constexpr int kScanReach = 10;    // of which at least this many on either side of the round's energy
template <int W>
constexpr int kScanFew = W / 4;   // accepted moves of a walker's round that are still few
// A window's centre follows an energy further from it than this (ms of 3D
// L = 32, N = 3277, 8192 walkers, 10 sweeps at 5 / 7 / 9 rows: 12.81 / 12.40 / 12.23).
constexpr int kScanDrift = 9;
static_assert(kThrTPad >= kScanReach + 3 && kThrTPad >= kScanWords - kScanReach, "window in the padding");

// Occupation as the rounds read it: de() is the energy change but for the
// adjacency of the two sites, commit() applies this lane's move (several
// lanes of a group may commit at once, so through atomics).
template <int D, bool SB>
struct ScanBits {
    uint32_t *bits;
    __device__ __forceinline__ uint32_t bit(uint32_t s) const
    {
        uint32_t v;
        if constexpr (SB) {
            const uint32_t base = (uint32_t)__cvta_generic_to_shared(bits);
            asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(base + ((s >> 5) << 2)) : "memory");
        } else {
            v = __ldcg(bits + (s >> 5));
        }
        return (v >> (s & 31u)) & 1u;
    }
    __device__ __forceinline__ int de(uint32_t, uint32_t, const uint32_t (&na)[2 * D],
                                      const uint32_t (&nb)[2 * D]) const
    {
        int n = 0;
#pragma unroll
        for (int i = 0; i < 2 * D; ++i) n += (int)bit(na[i]) - (int)bit(nb[i]);
        return n;
    }
    __device__ __forceinline__ void commit(uint32_t a, uint32_t b, const uint32_t (&)[2 * D],
                                           const uint32_t (&)[2 * D]) const
    {
        atomicXor(bits + (a >> 5), 1u << (a & 31u));
        atomicXor(bits + (b >> 5), 1u << (b & 31u));
    }
};

template <int D>
struct ScanField {
    uint32_t fbase;      // shared byte address of the walker's field (see FieldView)
    __device__ __forceinline__ int de(uint32_t a, uint32_t b, const uint32_t (&)[2 * D],
                                      const uint32_t (&)[2 * D]) const
    {
        uint32_t va, vb;
        asm volatile("ld.shared.u8 %0, [%1];" : "=r"(va) : "r"(fbase + a) : "memory");
        asm volatile("ld.shared.u8 %0, [%1];" : "=r"(vb) : "r"(fbase + b) : "memory");
        return ((int)va - (int)vb) >> 2;
    }
    __device__ __forceinline__ void commit(uint32_t, uint32_t, const uint32_t (&na)[2 * D],
                                           const uint32_t (&nb)[2 * D]) const
    {
#pragma unroll
        for (int i = 0; i < 2 * D; ++i) {
            // -4 and +4 in the sites' bytes (shifts modulo 32)
            asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(fbase + (na[i] & ~3u)),
                         "r"(__funnelshift_l(0u, 0xFFFFFFFCu, na[i] << 3)) : "memory");
            asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(fbase + (nb[i] & ~3u)),
                         "r"(__funnelshift_l(0u, 4u, nb[i] << 3)) : "memory");
        }
    }
};

// The sizes a round needs, in registers: the parameter table is in global
// memory, and the rounds' stores would have it read again every time.
struct Sizes {
    int32_t L, V, L2;
    uint32_t magL;
};

// The round's comparisons as chains of predicates, one instruction each (the
// compiled form of the same C++ expressions materialised every comparison as a
// number: 505 against 270 comparing and selecting instructions a round in 2D).

// set |= bit if one of the sites s is x or y, or pa == a or pb == b.
template <int D>
__device__ __forceinline__ void or_if_touch(uint32_t &set, uint32_t bit, const uint32_t (&na)[2 * D],
                                            const uint32_t (&nb)[2 * D], uint32_t a, uint32_t b,
                                            uint32_t pa, uint32_t pb)
{
    if constexpr (D == 2)
        asm("{\n\t.reg .pred p, q;\n\t"
            "setp.eq.u32 p, %10, %12;\n\tsetp.eq.u32 q, %11, %13;\n\t"
            "setp.eq.or.u32 p, %2, %12, p;\n\tsetp.eq.or.u32 q, %2, %13, q;\n\t"
            "setp.eq.or.u32 p, %3, %12, p;\n\tsetp.eq.or.u32 q, %3, %13, q;\n\t"
            "setp.eq.or.u32 p, %4, %12, p;\n\tsetp.eq.or.u32 q, %4, %13, q;\n\t"
            "setp.eq.or.u32 p, %5, %12, p;\n\tsetp.eq.or.u32 q, %5, %13, q;\n\t"
            "setp.eq.or.u32 p, %6, %12, p;\n\tsetp.eq.or.u32 q, %6, %13, q;\n\t"
            "setp.eq.or.u32 p, %7, %12, p;\n\tsetp.eq.or.u32 q, %7, %13, q;\n\t"
            "setp.eq.or.u32 p, %8, %12, p;\n\tsetp.eq.or.u32 q, %8, %13, q;\n\t"
            "setp.eq.or.u32 p, %9, %12, p;\n\tsetp.eq.or.u32 q, %9, %13, q;\n\t"
            "@p or.b32 %0, %0, %1;\n\t@q or.b32 %0, %0, %1;\n\t}"
            : "+r"(set)
            : "r"(bit), "r"(na[0]), "r"(na[1]), "r"(na[2]), "r"(na[3]), "r"(nb[0]), "r"(nb[1]),
              "r"(nb[2]), "r"(nb[3]), "r"(a), "r"(b), "r"(pa), "r"(pb));
    else
        asm("{\n\t.reg .pred p, q;\n\t"
            "setp.eq.u32 p, %14, %16;\n\tsetp.eq.u32 q, %15, %17;\n\t"
            "setp.eq.or.u32 p, %2, %16, p;\n\tsetp.eq.or.u32 q, %2, %17, q;\n\t"
            "setp.eq.or.u32 p, %3, %16, p;\n\tsetp.eq.or.u32 q, %3, %17, q;\n\t"
            "setp.eq.or.u32 p, %4, %16, p;\n\tsetp.eq.or.u32 q, %4, %17, q;\n\t"
            "setp.eq.or.u32 p, %5, %16, p;\n\tsetp.eq.or.u32 q, %5, %17, q;\n\t"
            "setp.eq.or.u32 p, %6, %16, p;\n\tsetp.eq.or.u32 q, %6, %17, q;\n\t"
            "setp.eq.or.u32 p, %7, %16, p;\n\tsetp.eq.or.u32 q, %7, %17, q;\n\t"
            "setp.eq.or.u32 p, %8, %16, p;\n\tsetp.eq.or.u32 q, %8, %17, q;\n\t"
            "setp.eq.or.u32 p, %9, %16, p;\n\tsetp.eq.or.u32 q, %9, %17, q;\n\t"
            "setp.eq.or.u32 p, %10, %16, p;\n\tsetp.eq.or.u32 q, %10, %17, q;\n\t"
            "setp.eq.or.u32 p, %11, %16, p;\n\tsetp.eq.or.u32 q, %11, %17, q;\n\t"
            "setp.eq.or.u32 p, %12, %16, p;\n\tsetp.eq.or.u32 q, %12, %17, q;\n\t"
            "setp.eq.or.u32 p, %13, %16, p;\n\tsetp.eq.or.u32 q, %13, %17, q;\n\t"
            "@p or.b32 %0, %0, %1;\n\t@q or.b32 %0, %0, %1;\n\t}"
            : "+r"(set)
            : "r"(bit), "r"(na[0]), "r"(na[1]), "r"(na[2]), "r"(na[3]), "r"(na[4]), "r"(na[5]),
              "r"(nb[0]), "r"(nb[1]), "r"(nb[2]), "r"(nb[3]), "r"(nb[4]), "r"(nb[5]), "r"(a), "r"(b),
              "r"(pa), "r"(pb));
}

// x += v if y == z.
__device__ __forceinline__ void add_if_eq(uint32_t &x, uint32_t v, uint32_t y, uint32_t z)
{
    asm("{\n\t.reg .pred p;\n\tsetp.eq.u32 p, %2, %3;\n\t@p add.u32 %0, %0, %1;\n\t}"
        : "+r"(x) : "r"(v), "r"(y), "r"(z));
}

// A step of the recurrence: if T >= r, x += v and set |= bit.
__device__ __forceinline__ void step_if_ge(int &x, int v, unsigned &set, unsigned bit, uint32_t T, uint32_t r)
{
    asm("{\n\t.reg .pred p;\n\tsetp.ge.u32 p, %4, %5;\n\t@p add.s32 %0, %0, %2;\n\t"
        "@p or.b32 %1, %1, %3;\n\t}"
        : "+r"(x), "+r"(set) : "r"(v), "r"(bit), "r"(T), "r"(r));
}

// Bits of x turned left by n places in W bits (n <= W).
template <int W>
__device__ __forceinline__ unsigned turn_left(unsigned x, uint32_t n)
{
    if constexpr (W == 32) return __funnelshift_l(x, x, n);
    else return ((x << n) | ((x << n) >> W)) & ((1u << W) - 1u);
}

template <int D, typename IdxT, int W, int TM, typename View>
__device__ __forceinline__ void chain_scan(const SysParams &p, int w, bool active, const View v,
                                           const uint32_t *thr, unsigned long long *hist,
                                           uint64_t A, uint32_t iter, uint32_t ring_s, uint32_t mbar_s,
                                           uint32_t *stage_all)
{
    constexpr unsigned FULL = 0xffffffffu;
    constexpr unsigned WM = (uint32_t)(W - 1);
    constexpr int NS = 2 * D;
    constexpr int TS = (4 * D + 1 + 3) & ~3;   // words of a table row (SysParams::tstride)
    constexpr bool PAIR = sizeof(IdxT) == 2;   // two list values fit one word
    // dE + 2D of an attempt; one past the last, where T = 0 (a row's padding, or
    // the row behind the dE-major copy), stands for an attempt past the end
    constexpr uint32_t DEAD = 4 * D + 1;
    constexpr unsigned GMASK = W == 32 ? 0xffffffffu : ((1u << W) - 1u);
    const int lane = threadIdx.x & 31;
    const int j = lane & (W - 1);
    const int gbase = lane - j;
    const unsigned gm = GMASK << gbase;
    // the group's words of shared memory, one per slot: used in turns, with a
    // warp barrier before each write and after it
    uint32_t *stage = stage_all + (threadIdx.x / W) * W;
    IdxT *S = walker_S<IdxT>(p, w);
    const uint32_t N = (uint32_t)p.N;
    const uint32_t holes = (uint32_t)(p.V - p.N);
    const uint64_t seed = p.seed_base + (uint64_t)w;
    const uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
    const Sizes sz{p.L, p.V, p.L2, p.magL};
    const uint32_t pitch = (uint32_t)p.thrT_pitch;
    const bool ahead = p.prefetch != 0;
    int bin = active ? p.E[w] - p.e_lo : 0;
    const uint32_t rbase = TM == kThrShared ? (uint32_t)__cvta_generic_to_shared(thr) : ring_s;
    uint32_t carry = 0;      // attempts of the run at the current energy not recorded yet
    uint32_t acc = 0;
    // tunnelling bookkeeping (Sec. 4): every energy the walker takes is
    // compared with the two ends
    const bool tun = p.tunnel != 0;
    const int tlo = p.tun_lo, thi = p.tun_hi;
    uint32_t tst = tun && active ? p.tun_state[w] : 0u;
    uint32_t tcnt = 0;
    if (tun && bin <= tlo) {
        tcnt += tst == 2u ? 1u : 0u;
        tst = 1u;
    } else if (tun && bin >= thi) {
        tcnt += tst == 1u ? 1u : 0u;
        tst = 2u;
    }
    ThrWindow tw;
    int vlo = 0, vhi = 0;    // rows of the window that have arrived
    constexpr int WLO = kThrWindowRows / 2 - 1, WHI = kThrWindowRows / 2;
    if constexpr (TM == kThrWindow) {
        tw.ring = ring_s;
        tw.mbar = mbar_s;
        tw.table = thr;
        tw.n_rows = p.n_bins;
        tw.tstride = TS;
        tw.c = bin;
        if (active) {
            if (j == 0) mbar_init(mbar_s, 1u);
            __syncwarp(gm);
            tw.fetch(bin - WLO, bin + WHI, j == 0);
            tw.wait_group(p, gm);
        }
        vlo = bin - WLO;
        vhi = bin + WHI;
    }
    // the slot's attempt t: the current one (k, m, a, b, r2p), its next
    // (n: attempt t + W; its list entries are read in every round) and the one
    // after it (q: its random numbers are drawn in every round, and its list
    // entries prefetched into L2 where the lists are larger than L2)
    auto draw = [&](uint64_t t, uint32_t &kk, uint32_t &mm, uint32_t &rr) {
        const uint4 r = philox10(make_uint4((uint32_t)t, (uint32_t)(t >> 32), iter, 0u), k0, k1);
        kk = __umulhi(r.x, N);
        mm = __umulhi(r.y, holes);
        // acceptance T == 2^32 - 1 || r2 < T, as the single compare T >= rr
        rr = (r.z == 0xFFFFFFFFu) ? r.z : r.z + 1u;
    };
    uint64_t t0 = 0;             // (the same in the whole group)
    uint32_t k, m, r2p, kn, mn, r2n, a, b;
    const uint64_t t = (uint64_t)j;
    draw(t, k, m, r2p);
    draw(t + W, kn, mn, r2n);
    a = 0;                       // any two sites, where there is no attempt
    b = 1;
    if (active && t < A) {
        a = __ldcg(S + k);
        b = __ldcg(S + N + m);
    }
    // A round's values: attempts left, as far as the window and the next two
    // windows reach; the place of t0's slot and of this one; the slot's next
    // list entries and the random numbers of the attempt after; the sites
    // around its move and dE + 2D.
    uint32_t near, h, place, an, bn, kq, mq, r2q, code;
    uint32_t na[NS], nb[NS];
    unsigned am;              // accepted attempts, by place
    int x0 = 0;
    int xs[W];                // the energy bin after each attempt
    auto begin = [&]() {
        const uint64_t left = active && t0 < A ? A - t0 : 0u;
        near = left < 3u * W ? (uint32_t)left : 3u * W;
        h = (uint32_t)t0 & WM;
        place = ((uint32_t)j - h) & WM;
        an = a;
        bn = b;
        if (place + W < near) {
            an = __ldcg(S + kn);
            bn = __ldcg(S + N + mn);
        }
        neighbours<D>(sz, a, na);
        neighbours<D>(sz, b, nb);
        uint32_t de = (uint32_t)(v.de(a, b, na, nb) + 2 * D);
#pragma unroll
        for (int i = 0; i < NS; ++i) add_if_eq(de, 1u, na[i], b);    // (at most one of them)
        // (a state whose list and occupation disagree, as one may be restored, can
        // give any dE: never a threshold outside the table)
        code = place < near ? min(de, DEAD) : DEAD;
    };
    // The recurrence, and beside it, since its steps wait for one another,
    // the slots' random numbers two windows ahead.
    auto recurrence = [&]() {
        am = 0;
        draw(t0 + place + 2 * W, kq, mq, r2q);
        if constexpr (TM != kThrGlobal) {
            uint32_t rs[W], cs[W / 4];
            __syncwarp(FULL);
            stage[place] = r2p;
            __syncwarp(FULL);
#pragma unroll
            for (int i = 0; i < W; i += 4) *reinterpret_cast<uint4 *>(rs + i) = *reinterpret_cast<const uint4 *>(stage + i);
            __syncwarp(FULL);
            reinterpret_cast<uint8_t *>(stage)[place] = (uint8_t)code;
            __syncwarp(FULL);
#pragma unroll
            for (int i = 0; i < W / 4; ++i) cs[i] = stage[i];
            int x = bin;
#pragma unroll
            for (int i = 0; i < W; ++i) {
                const uint32_t ci = (cs[i / 4] >> (8 * (i & 3))) & 0xFFu;
                const uint32_t row = TM == kThrWindow ? (uint32_t)x & (kThrWindowRows - 1u) : (uint32_t)x;
                uint32_t T;
                asm volatile("ld.shared.u32 %0, [%1];" : "=r"(T) : "r"(row * (4u * TS) + (rbase + 4u * ci)));
                step_if_ge(x, (int)ci - 2 * D, am, 1u << i, T, rs[i]);
                xs[i] = x;
            }
        } else {
            const int e0 = (bin + kThrTPad - kScanReach) & ~3;
            x0 = bin + kThrTPad - e0;
            uint32_t word;
            const bool valid = place < near;
            const uint4 *q = reinterpret_cast<const uint4 *>(
                thr + ((valid ? code : 0u) * pitch + (uint32_t)e0));
            uint32_t ok = 0;
#pragma unroll
            for (int g = 0; g < kScanWords / 4; ++g) {
                const uint4 y = __ldg(q + g);
                ok |= (y.x >= r2p ? 1u << (4 * g) : 0u) | (y.y >= r2p ? 2u << (4 * g) : 0u) |
                      (y.z >= r2p ? 4u << (4 * g) : 0u) | (y.w >= r2p ? 8u << (4 * g) : 0u);
            }
            word = (code << 24) | (valid ? ok : 0u);
            uint32_t ws[W];
            __syncwarp(FULL);
            stage[place] = word;
            __syncwarp(FULL);
#pragma unroll
            for (int i = 0; i < W; i += 4) *reinterpret_cast<uint4 *>(ws + i) = *reinterpret_cast<const uint4 *>(stage + i);
            int x = x0;
#pragma unroll
            for (int i = 0; i < W; ++i) {
                step_if_ge(x, (int)(ws[i] >> 24) - 2 * D, am, 1u << i,
                           __funnelshift_r(ws[i], ws[i], (uint32_t)x) & 1u, 1u);
                xs[i] = bin + x - x0;
            }
        }
    };
    // the window's places that hold an attempt
    auto places = [&]() {
        return W == 32 && near >= 32u ? 0xffffffffu : (1u << (near < W ? near : W)) - 1u;
    };
    auto prefetch = [&]() {
        if (ahead && place + 2 * W < near) {
            asm volatile("prefetch.L2 [%0];" ::"l"(S + kq));
            asm volatile("prefetch.L2 [%0];" ::"l"(S + N + mq));
        }
    };
    // what the slot goes on with: its next attempt, or the same one again
    auto advance = [&](bool decided) {
        k = decided ? kn : k;
        m = decided ? mn : m;
        a = decided ? an : a;
        b = decided ? bn : b;
        r2p = decided ? r2n : r2p;
        kn = decided ? kq : kn;
        mn = decided ? mq : mn;
        r2n = decided ? r2q : r2n;
    };
    bool many = true;            // (the same in the whole warp) the last round had many accepted moves
    while (__any_sync(FULL, active && t0 < A)) {
        if constexpr (TM == kThrWindow) {
            // rows asked for a round ago; then the window follows the energy
            if (active && t0 < A) {
                if (tw.pend) {
                    tw.wait_group(p, gm);
                    vlo = tw.c - WLO;
                    vhi = tw.c + WHI;
                }
                const int off = bin - tw.c;
                if (!tw.broken && (off > kScanDrift || off < -kScanDrift)) {
                    if (off > 0) tw.fetch(max(tw.c + WHI + 1, bin - WLO), bin + WHI, j == 0);
                    else tw.fetch(bin - WLO, min(tw.c - WLO - 1, bin + WHI), j == 0);
                    vlo = max(vlo, bin - WLO);
                    vhi = min(vhi, bin + WHI);
                    tw.c = bin;
                    if (tw.pend && (bin < vlo || bin > vhi)) tw.wait_group(p, gm);
                    if (!tw.pend) {
                        vlo = bin - WLO;
                        vhi = bin + WHI;
                    }
                }
                // the walker stops, in all lanes of its group; the host reports the iteration invalid
                if (tw.broken) t0 = A;
            }
        }
        begin();
        const unsigned bit = 1u << place;
        const uint32_t nv = near < W ? near : (uint32_t)W;
        if (!many) {
            // Few accepted moves: the decisions at the round's energy alone,
            // one threshold a lane, up to the first accepted attempt.
            uint32_t T;
            if constexpr (TM == kThrGlobal) {
                T = __ldg(thr + ((place < near ? code : 0u) * pitch + (uint32_t)(bin + kThrTPad)));
            } else {
                const uint32_t row = TM == kThrWindow ? (uint32_t)bin & (kThrWindowRows - 1u) : (uint32_t)bin;
                asm volatile("ld.shared.u32 %0, [%1];" : "=r"(T) : "r"(row * (4u * TS) + (rbase + 4u * code)));
            }
            draw(t0 + place + 2 * W, kq, mq, r2q);
            prefetch();
            const unsigned votes = __ballot_sync(FULL, place < nv && T >= r2p);
            if (votes == 0u) {
                advance(place < nv);
                carry += nv;
                t0 += nv;
            } else {
                const unsigned mine = (votes >> gbase) & GMASK;
                am = turn_left<W>(mine, (uint32_t)W - h);
                many = __any_sync(FULL, __popc(am) > kScanFew<W>);
                const uint32_t first = am ? (uint32_t)__ffs(am) - 1u : 0u;
                const uint32_t nd = am ? first + 1u : nv;
                const int src = gbase + (int)((first + h) & WM);
                const uint32_t cc = __shfl_sync(FULL, code, src);
                uint32_t ck, cm, ca, cb;
                shfl_pair<IdxT>(k, m, src, ck, cm);
                shfl_pair<IdxT>(a, b, src, ca, cb);
                const int de = am ? (int)cc - 2 * D : 0;
                if (am && place == first) {
                    v.commit(a, b, na, nb);
                    S[k] = (IdxT)b;
                    S[N + m] = (IdxT)a;
                    ++acc;
                    const uint32_t cnt = carry + first;
                    if (de != 0 && cnt != 0u) atomicAdd(hist + bin, (unsigned long long)cnt);
                }
                carry = de != 0 ? 1u : carry + nd;
                bin += de;
                if (tun && am) {
                    if (bin <= tlo) {
                        tcnt += tst == 2u ? 1u : 0u;
                        tst = 1u;
                    } else if (bin >= thi) {
                        tcnt += tst == 1u ? 1u : 0u;
                        tst = 2u;
                    }
                }
                advance(place < nd);
                a = am && ck == k ? cb : a;
                b = am && cm == m ? ca : b;
                t0 += nd;
            }
            if (carry >= 0x40000000u) {
                if (active && j == 0) atomicAdd(hist + bin, (unsigned long long)carry);
                carry = 0;
            }
            __syncwarp(FULL);
            continue;
        }
        // Many: every pair of slots is tried for touching ahead of the
        // recurrence, slot s against the W / 2 behind it in the ring.
        unsigned behind = 0;       // places of the touched ones
        {
            uint32_t pa[W / 2], pb[W / 2];
            __syncwarp(FULL);
            stage[j] = PAIR ? (a | (b << 16)) : a;
            __syncwarp(FULL);
#pragma unroll
            for (int d = 1; d <= W / 2; ++d) {
                const uint32_t x = stage[(j + d) & WM];
                pa[d - 1] = PAIR ? (x & 0xFFFFu) : x;
                pb[d - 1] = PAIR ? (x >> 16) : 0u;
            }
            if constexpr (!PAIR) {
                __syncwarp(FULL);
                stage[j] = b;
                __syncwarp(FULL);
#pragma unroll
                for (int d = 1; d <= W / 2; ++d) pb[d - 1] = stage[(j + d) & WM];
            }
            recurrence();      // (the comparisons below fill its waits too)
            unsigned c = 0;
#pragma unroll
            for (int d = 1; d <= W / 2; ++d)
                or_if_touch<D>(c, 1u << (d - 1), na, nb, a, b, pa[d - 1], pb[d - 1]);
            behind = turn_left<W>(c, place + 1);
        }
        prefetch();
        // the energy bin after the own attempt
        __syncwarp(FULL);
        if (j == 0) {
#pragma unroll
            for (int i = 0; i < W; i += 4)
                *reinterpret_cast<int4 *>(stage + i) = make_int4(xs[i], xs[i + 1], xs[i + 2], xs[i + 3]);
        }
        __syncwarp(FULL);
        const int x1 = (int)stage[place];
        // attempts that have to wait (bad) and those whose move changes the
        // energy (up), by place, over the group
        const int de = (int)code - 2 * D;
        const bool yes = (am & bit) != 0u && place < near;
        const int x = x1 - (yes ? de : 0);
        unsigned bad = 0, up = yes && de != 0 ? bit : 0u;
        if constexpr (TM == kThrGlobal) bad |= (uint32_t)(x - bin + x0) >= (uint32_t)kScanWords ? bit : 0u;
        if constexpr (TM == kThrWindow) bad |= x < vlo || x > vhi ? bit : 0u;
        am &= places();
        bad |= (behind & am & (bit - 1u)) ? bit : 0u;
        bad |= yes ? behind & ~(bit | (bit - 1u)) : 0u;
        if constexpr (W <= 16) {
            unsigned y = bad | (up << 16);
#pragma unroll
            for (int o = 1; o < W; o <<= 1) y |= __shfl_xor_sync(FULL, y, o);
            bad = y & 0xFFFFu;
            up = y >> 16;
        } else {
#pragma unroll
            for (int o = 1; o < W; o <<= 1) {
                bad |= __shfl_xor_sync(FULL, bad, o);
                up |= __shfl_xor_sync(FULL, up, o);
            }
        }
        // attempts decided (a bad one past the end is none)
        const uint32_t nd = bad ? min((uint32_t)__ffs(bad) - 1u, nv) : nv;
        const unsigned done = W == 32 && nd >= 32u ? 0xffffffffu : (1u << nd) - 1u;
        const unsigned chg = up & done;
        many = __any_sync(FULL, __popc(am) > kScanFew<W>);
        const bool commit = yes && place < nd;
        // the list slots a commit rewrites
        const uint32_t moved = commit && PAIR ? (k | (m << 16)) : 0xFFFFFFFFu;   // (indices below 65535)
        if (commit) {
            v.commit(a, b, na, nb);
            S[k] = (IdxT)b;
            S[N + m] = (IdxT)a;
            ++acc;
            // a move ends the run at the energy before it
            const unsigned prev = chg & (bit - 1u);
            const uint32_t cnt = prev ? place - 31u + (uint32_t)__clz(prev) : carry + place;
            if (de != 0 && cnt != 0u) atomicAdd(hist + (x1 - de), (unsigned long long)cnt);
        }
        carry = chg ? nd - 31u + (uint32_t)__clz(chg) : carry + nd;
        if (tun) {      // (the same in the whole block)
            unsigned tl = commit && x1 <= tlo ? bit : 0u;
            unsigned th = commit && x1 >= thi ? bit : 0u;
#pragma unroll
            for (int o = 1; o < W; o <<= 1) {
                tl |= __shfl_xor_sync(FULL, tl, o);
                th |= __shfl_xor_sync(FULL, th, o);
            }
            while (tl | th) {      // events in attempt order, runs of one end at once
                if (th == 0u || (tl != 0u && __ffs(tl) < __ffs(th))) {
                    tcnt += tst == 2u ? 1u : 0u;
                    tst = 1u;
                    tl = th ? tl & ~((th & (0u - th)) - 1u) : 0u;
                } else {
                    tcnt += tst == 1u ? 1u : 0u;
                    tst = 2u;
                    th = tl ? th & ~((tl & (0u - tl)) - 1u) : 0u;
                }
            }
            __syncwarp(FULL);
        }
        // the energy the window goes on from: after its last decided attempt
        bin = nd ? (int)stage[nd - 1u] : bin;
        const uint32_t a_i = a, b_i = b, k_i = k, m_i = m;
        advance(place < nd);
        // its list entries, read before this round's commits, where a commit
        // moved one of its slots (at most one commit of a round per slot)
        if constexpr (PAIR) {
            __syncwarp(FULL);
            stage[j] = moved;
            __syncwarp(FULL);
            uint32_t ms[W];
#pragma unroll
            for (int i = 0; i < W; i += 4) *reinterpret_cast<uint4 *>(ms + i) = *reinterpret_cast<const uint4 *>(stage + i);
            const uint32_t own = k | (m << 16);
            uint32_t low = 0xFFFFFFFFu;     // the least of each half
#pragma unroll
            for (int i = 0; i < W; i += 2) low = __vimin3_u16x2(low, ms[i] ^ own, ms[i + 1] ^ own);
            if (__any_sync(FULL, (low & 0xFFFFu) == 0u || low < 0x10000u)) {
                int of_k = -1, of_m = -1;
#pragma unroll
                for (int i = 0; i < W; ++i) {
                    const uint32_t x = ms[i] ^ (k | (m << 16));
                    of_k = (x & 0xFFFFu) == 0u ? i : of_k;
                    of_m = x < 0x10000u ? i : of_m;
                }
                const uint32_t to_k = __shfl_sync(FULL, b_i, of_k & (W - 1), W);
                const uint32_t to_m = __shfl_sync(FULL, a_i, of_m & (W - 1), W);
                a = of_k >= 0 ? to_k : a;
                b = of_m >= 0 ? to_m : b;
            }
        } else {
            if (__any_sync(FULL, commit)) {
#pragma unroll
                for (int i = 0; i < W; ++i) {
                    const bool ci = __shfl_sync(FULL, (int)commit, i, W) != 0;
                    const uint32_t ki = __shfl_sync(FULL, k_i, i, W);
                    const uint32_t mi = __shfl_sync(FULL, m_i, i, W);
                    const uint32_t ai = __shfl_sync(FULL, a_i, i, W);
                    const uint32_t bi = __shfl_sync(FULL, b_i, i, W);
                    a = ci && ki == k ? bi : a;
                    b = ci && mi == m ? ai : b;
                }
            }
        }
        t0 += nd;
        if (carry >= 0x40000000u) {
            if (active && j == 0) atomicAdd(hist + bin, (unsigned long long)carry);
            carry = 0;
        }
        __syncwarp(FULL);       // the commits, before the next round's reads
    }
    if constexpr (TM == kThrWindow) {
        if (active) {
            // no copy may still write into the ring when the block moves on
            if (!tw.broken) {
                tw.wait_group(p, gm);
            } else if (tw.pend) {
                uint32_t ok = 0;
                for (uint32_t i = 0; i < kWaitLimit && !ok; ++i) ok = mbar_try_wait(mbar_s, tw.phase);
            }
            __syncwarp(gm);
            if (j == 0) mbar_inval(mbar_s);
        }
    }
#pragma unroll
    for (int o = W / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(FULL, acc, o);
    if (active && j == 0) {
        if (carry) atomicAdd(hist + bin, (unsigned long long)carry);
        p.E[w] = bin + p.e_lo;
        p.accepts[w] = acc;
        if (tun) {
            p.tun_state[w] = (uint8_t)tst;
            p.tun_count[w] += tcnt;
        }
    }
}

// How the rounds read a walker's occupation.
enum ScanView { kViewBitsShared, kViewBitsGlobal, kViewField };

template <int D, typename IdxT, int W, int TM, int VIEW>
__device__ __forceinline__ void scan_item(const SysParams &p, const BlockWork &wk, uint32_t *smem,
                                          uint32_t *stage, uint64_t sweeps, uint32_t iter)
{
    const int lw = threadIdx.x / W;
    const bool active = lw < wk.count;
    const int w = wk.walker0 + (active ? lw : 0);
    const uint32_t *thr = TM == kThrShared ? smem : (TM == kThrWindow ? p.thr : p.thrT);
    unsigned long long *hist = hist_row(p, w, wk.hist_row);
    const uint64_t A = sweeps * (uint64_t)p.N;
    uint32_t *state = smem + (TM == kThrShared ? thr_words_aligned(p) : 0);
    uint32_t ring_s = 0u, mbar_s = 0u;
    if constexpr (TM == kThrWindow) {
        const int wpb = (int)blockDim.x / W;
        const uint32_t used = VIEW == kViewField ? (uint32_t)wpb * (uint32_t)field_bytes(p)
                              : VIEW == kViewBitsShared ? (uint32_t)wpb * (uint32_t)p.words * 4u : 0u;
        window_addrs(p, (uint32_t)__cvta_generic_to_shared(state) + used, wpb, active ? lw : 0,
                     ring_s, mbar_s);
    }
    if constexpr (VIEW == kViewField) {
        if constexpr (TM == kThrShared) block_copy_words(smem, p.thr, (size_t)p.n_bins * (size_t)p.tstride);
        field_build<D, IdxT>(p, wk, state);   // ends with a block barrier, which also covers the table
        const ScanField<D> v{(uint32_t)__cvta_generic_to_shared(state) +
                             (uint32_t)((size_t)(active ? lw : 0) * field_bytes(p))};
        chain_scan<D, IdxT, W, TM>(p, w, active, v, thr, hist, A, iter, ring_s, mbar_s, stage);
        field_finish<IdxT>(p, wk, state);
    } else {
        constexpr bool SB = VIEW == kViewBitsShared;
        const BlockSetup bs = block_setup(p, wk, smem, SB ? 1 : 0, TM == kThrShared ? 1 : 0);
        uint32_t *bits0 = SB ? state : p.bits + (size_t)wk.walker0 * (size_t)p.words;
        const ScanBits<D, SB> v{bits0 + (size_t)(active ? lw : 0) * p.words};
        chain_scan<D, IdxT, W, TM>(p, w, active, v, thr, hist, A, iter, ring_s, mbar_s, stage);
        block_finish(bs, SB ? 1 : 0);
    }
}

// Block b takes work item b; with a counter (persistent launches), then the
// items that it pulls from it.
template <int W, int TM, int VIEW>
__global__ void __launch_bounds__(kGroupMaxThreads, 1)
walker_update_scan(const SysParams *__restrict__ sys, const BlockWork *__restrict__ work,
                   uint64_t sweeps, uint32_t iter, int n_items, int *next_item)
{
    extern __shared__ __align__(16) uint32_t smem[];
    __shared__ __align__(16) uint32_t stage[kGroupMaxThreads];
    __shared__ int s_item;
    int item = blockIdx.x;
    for (;;) {
        const BlockWork wk = work[item];
        const SysParams &p = sys[wk.sys];
        if (p.d == 2) {
            if (p.idx16) scan_item<2, uint16_t, W, TM, VIEW>(p, wk, smem, stage, sweeps, iter);
            else scan_item<2, uint32_t, W, TM, VIEW>(p, wk, smem, stage, sweeps, iter);
        } else {
            if (p.idx16) scan_item<3, uint16_t, W, TM, VIEW>(p, wk, smem, stage, sweeps, iter);
            else scan_item<3, uint32_t, W, TM, VIEW>(p, wk, smem, stage, sweeps, iter);
        }
        if (!next_item) break;
        item = next_work_item(next_item, &s_item);
        if (item >= n_items) break;
    }
}

template <int G>
void walker_scan_fns_t(const void *(&fns)[kWalkerScanFns])
{
    int i = 0;
#define MUCAL_SCAN_FNS(VIEW)                                            \
    fns[i++] = (const void *)walker_update_scan<G, kThrGlobal, VIEW>;  \
    fns[i++] = (const void *)walker_update_scan<G, kThrShared, VIEW>;  \
    fns[i++] = (const void *)walker_update_scan<G, kThrWindow, VIEW>;
    MUCAL_SCAN_FNS(kViewBitsShared)
    MUCAL_SCAN_FNS(kViewBitsGlobal)
    MUCAL_SCAN_FNS(kViewField)
#undef MUCAL_SCAN_FNS
}

}  // namespace
}  // namespace mucal
