// The walker update with several commits per round (mucal_launch_config
// .multi_commit): device code, one instantiation per lane count in
// walker_scan_<lanes>.cu.  The chain is the one-thread chain of
// walker_chain.cuh, bit for bit.
#pragma once

#include "walker_chain.cuh"

namespace mucal {
namespace {

// ---------------------------------------------------------------------------
// Several commits per round (multi-commit rounds) on a sliding window of G
// attempts: lane t mod G of the group holds attempt t, for the G attempts from
// the first undecided one (t0) on.
//
// A round evaluates the energy changes of the whole window against the state
// at its start.  Such a value stays right until an earlier attempt of the
// window commits a move next to one of the lane's two sites or in one of its
// two list slots; which earlier lanes could do so (cm, a bit mask) is a matter
// of the sites alone.  Taking all energy changes as they are, the decisions
// are a short serial recurrence in the energy, which every lane of the group
// runs redundantly in registers: T(E, dE_i) >= r_i ? E += dE_i.  The round
// then ends at the first lane whose cm meets an accepted lane: the lanes
// before it are decided as the serial chain decides them, commit together and
// take the next attempts, and the window slides on.  The first lane is never
// stopped, so every round decides at least one attempt, mostly the whole
// window; no group of a warp waits for another's conflicts.
//
// A step of the recurrence is one threshold load from shared memory and a few
// dependent integer instructions: from the whole table (kThrShared), or from
// the walker's window of rows (kThrWindow, see ThrWindow), where a lane
// reached with an energy whose row has not arrived is stopped like one with a
// conflict.  Where neither fits, the thresholds are read from global memory
// (kThrGlobal) ahead of the recurrence: every lane turns the kScanWords
// thresholds of its dE around the round's energy, contiguous in the table's
// dE-major copy, into a bit mask of decisions by energy, and is stopped when
// reached with another energy.
// ---------------------------------------------------------------------------
constexpr int kScanWords = 24;    // energies of a decision mask (bits 0-23; the lane's dE above)
constexpr int kScanDrift = 5;     // a window's centre follows an energy further from it than this
constexpr int kScanReach = 10;    // of which at least this many on either side of the round's energy
static_assert(kThrTPad >= kScanReach + 3 && kThrTPad >= kScanWords - kScanReach, "window in the padding");

// Occupation as the rounds read it: d4() is 4 times the energy change but for
// the adjacency of the two sites, commit() applies this lane's move (several
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
    __device__ __forceinline__ int d4(uint32_t, uint32_t, const uint32_t (&na)[2 * D],
                                      const uint32_t (&nb)[2 * D]) const
    {
        int n = 0;
#pragma unroll
        for (int i = 0; i < 2 * D; ++i) n += (int)bit(na[i]) - (int)bit(nb[i]);
        return 4 * n;
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
    __device__ __forceinline__ int d4(uint32_t a, uint32_t b, const uint32_t (&)[2 * D],
                                      const uint32_t (&)[2 * D]) const
    {
        uint32_t va, vb;
        asm volatile("ld.shared.u8 %0, [%1];" : "=r"(va) : "r"(fbase + a) : "memory");
        asm volatile("ld.shared.u8 %0, [%1];" : "=r"(vb) : "r"(fbase + b) : "memory");
        return (int)va - (int)vb;
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

template <int D, typename IdxT, int G, int TM, typename View>
__device__ __forceinline__ void chain_scan(const SysParams &p, int w, bool active, const View v,
                                           const uint32_t *thr, unsigned long long *hist,
                                           uint64_t A, uint32_t iter, uint32_t ring_s, uint32_t mbar_s)
{
    constexpr unsigned FULL = 0xffffffffu;
    constexpr unsigned GMASK = (G == 32) ? 0xffffffffu : ((1u << G) - 1u);
    constexpr int NS = 2 * D;
    constexpr int TS = (4 * D + 1 + 3) & ~3;   // words of a table row (SysParams::tstride)
    // an entry of a row's padding, where T = 0: what lanes without a decision to take read
    constexpr uint32_t DEAD = 4u * (2 * D + 1);
    const int lane = threadIdx.x & 31;
    const int j = lane & (G - 1);
    const int gbase = lane - j;
    const unsigned gm = GMASK << gbase;
    IdxT *S = walker_S<IdxT>(p, w);
    const uint32_t N = (uint32_t)p.N;
    const uint32_t holes = (uint32_t)(p.V - p.N);
    const uint64_t seed = p.seed_base + (uint64_t)w;
    const uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
    const Sizes sz{p.L, p.V, p.L2, p.magL};
    const uint32_t pitch = (uint32_t)p.thrT_pitch;
    int bin = active ? p.E[w] - p.e_lo : 0;
    const uint32_t rbase = TM == kThrShared ? (uint32_t)__cvta_generic_to_shared(thr) + 8u * D : 0u;
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
            tw.wait(p);
        }
        vlo = bin - WLO;
        vhi = bin + WHI;
    }
    // lane masks of a group turned so that bit o is the window's o-th attempt
    auto turned = [](unsigned x, uint32_t h) -> unsigned {
        if constexpr (G == 32) return __funnelshift_r(x, x, h);
        else return ((x | (x << G)) >> h) & GMASK;
    };
    // attempt t0 + pos of this lane: the current one (k, m, a, b, r2p), the
    // lane's next (n: attempt + G; its list entries are read in every round)
    // and the one after it (q: its random numbers are drawn in every round,
    // and its list entries prefetched into L2)
    auto draw = [&](uint64_t t, uint32_t &kk, uint32_t &mm, uint32_t &rr) {
        const uint4 r = philox10(make_uint4((uint32_t)t, (uint32_t)(t >> 32), iter, 0u), k0, k1);
        kk = __umulhi(r.x, N);
        mm = __umulhi(r.y, holes);
        // acceptance T == 2^32 - 1 || r2 < T, as the single compare T >= rr
        rr = (r.z == 0xFFFFFFFFu) ? r.z : r.z + 1u;
    };
    uint64_t t0 = 0;             // (the same in the whole group)
    uint32_t k, m, r2p, kn, mn, r2n;
    draw((uint64_t)j, k, m, r2p);
    draw((uint64_t)j + G, kn, mn, r2n);
    uint32_t a = 0, b = 1;       // any two sites, where there is no attempt
    if (active && (uint64_t)j < A) {
        a = __ldcg(S + k);
        b = __ldcg(S + N + m);
    }
    while (__any_sync(FULL, active && t0 < A)) {
        if constexpr (TM == kThrWindow) {
            // rows asked for a round ago; then the window follows the energy
            if (active && t0 < A) {
                if (tw.pend) {
                    tw.wait(p);
                    vlo = tw.c - WLO;
                    vhi = tw.c + WHI;
                }
                const int off = bin - tw.c;
                if (off > kScanDrift || off < -kScanDrift) {
                    if (off > 0) tw.fetch(max(tw.c + WHI + 1, bin - WLO), bin + WHI, j == 0);
                    else tw.fetch(bin - WLO, min(tw.c - WLO - 1, bin + WHI), j == 0);
                    vlo = max(vlo, bin - WLO);
                    vhi = min(vhi, bin + WHI);
                    tw.c = bin;
                    if (tw.pend && (bin < vlo || bin > vhi)) tw.wait(p);
                    if (!tw.pend) {
                        vlo = bin - WLO;
                        vhi = bin + WHI;
                    }
                }
                if (tw.broken) t0 = A;     // the walker stops; the host reports the iteration invalid
            }
        }
        const uint32_t h = (uint32_t)t0 & (uint32_t)(G - 1);
        const uint32_t pos = ((uint32_t)j - h) & (uint32_t)(G - 1);
        const unsigned before = (1u << pos) - 1u;
        const uint64_t t = t0 + pos;
        const bool valid = active && t < A;
        const uint32_t nv = !active || t0 >= A ? 0u : (A - t0 < (uint64_t)G ? (uint32_t)(A - t0) : (uint32_t)G);
        uint32_t an = a, bn = b;
        if (active && t + G < A) {
            an = __ldcg(S + kn);
            bn = __ldcg(S + N + mn);
        }
        uint32_t kq, mq, r2q;
        draw(t + 2 * G, kq, mq, r2q);
        if (active && t + 2 * G < A) {
            asm volatile("prefetch.L2 [%0];" ::"l"(S + kq));
            asm volatile("prefetch.L2 [%0];" ::"l"(S + N + mq));
        }
        uint32_t na[NS], nb[NS];
        neighbours<D>(sz, a, na);
        neighbours<D>(sz, b, nb);
        uint32_t adj4 = 0;
#pragma unroll
        for (int i = 0; i < NS; ++i) adj4 |= (na[i] == b) ? 4u : 0u;
        const int d4 = v.d4(a, b, na, nb) + (int)adj4;
        const int de4 = valid ? d4 : 0;
        // every pair of lanes once, lane l with lane l + d: bit l of ballot d
        // tells whether their moves touch
        unsigned cm = 0;
#pragma unroll
        for (int d = 1; d <= G / 2; ++d) {
            uint32_t pa, pb;
            shfl_pair<IdxT>(a, b, gbase + ((j + d) & (G - 1)), pa, pb);
            bool c = (pa == a) | (pb == b);
#pragma unroll
            for (int i = 0; i < NS; ++i)
                c |= (na[i] == pa) | (na[i] == pb) | (nb[i] == pa) | (nb[i] == pb);
            const unsigned B = (__ballot_sync(FULL, c) & gm) >> gbase;
            cm |= B & (1u << ((j - d) & (G - 1)));
            cm |= ((B >> j) & 1u) << ((j + d) & (G - 1));
        }
        cm = turned(cm, h) & before;
        // the recurrence
        unsigned am = 0;          // accepted attempts, by place in the window
        int x0 = 0;
        if constexpr (TM == kThrShared) {
            const uint32_t d_own = valid ? (uint32_t)de4 : DEAD;
            uint32_t row = rbase + (uint32_t)bin * (4u * TS);
#pragma unroll
            for (int i = 0; i < G; ++i) {
                const uint32_t di = __shfl_sync(FULL, d_own, (int)h + i, G);
                const uint32_t ri = __shfl_sync(FULL, r2p, (int)h + i, G);
                uint32_t T;
                asm("ld.shared.u32 %0, [%1];" : "=r"(T) : "r"(row + di));
                const bool ok = T >= ri;
                row += ok ? di * (uint32_t)TS : 0u;
                am |= ok ? 1u << i : 0u;
            }
        } else if constexpr (TM == kThrWindow) {
            const uint32_t d_own = valid ? (uint32_t)de4 : DEAD;
            int x = bin;
#pragma unroll
            for (int i = 0; i < G; ++i) {
                const uint32_t di = __shfl_sync(FULL, d_own, (int)h + i, G);
                const uint32_t ri = __shfl_sync(FULL, r2p, (int)h + i, G);
                uint32_t T;
                asm volatile("ld.shared.u32 %0, [%1];" : "=r"(T)
                             : "r"(((uint32_t)x & (kThrWindowRows - 1u)) * (4u * TS) + (ring_s + 8u * D + di)));
                const bool ok = T >= ri;
                x += ok ? (int)di >> 2 : 0;
                am |= ok ? 1u << i : 0u;
            }
        } else {
            const int e0 = (bin + kThrTPad - kScanReach) & ~3;
            x0 = bin + kThrTPad - e0;
            const uint4 *q = reinterpret_cast<const uint4 *>(
                thr + ((uint32_t)((de4 >> 2) + 2 * D) * pitch + (uint32_t)e0));
            uint32_t ok[kScanWords / 8];
#pragma unroll
            for (int g = 0; g < kScanWords / 8; ++g) {
                const uint4 u = __ldg(q + 2 * g), u2 = __ldg(q + 2 * g + 1);
                const uint32_t tv[8] = {u.x, u.y, u.z, u.w, u2.x, u2.y, u2.z, u2.w};
                ok[g] = 0;
#pragma unroll
                for (int o = 0; o < 8; ++o) ok[g] |= tv[o] >= r2p ? 1u << (8 * g + o) : 0u;
            }
            const uint32_t word = ((uint32_t)(de4 >> 2) << 24) | (valid ? ok[0] | ok[1] | ok[2] : 0u);
            int x = x0;
#pragma unroll
            for (int i = 0; i < G; ++i) {
                const uint32_t wi = __shfl_sync(FULL, word, (int)h + i, G);
                const bool yes = (__funnelshift_r(wi, wi, (uint32_t)x) & 1u) != 0u;
                x += yes ? (int)wi >> 24 : 0;
                am |= yes ? 1u << i : 0u;
            }
        }
        // the energy after this lane's attempt is bin + incl
        const int de = de4 >> 2;
        const bool yes = valid && ((am >> pos) & 1u);
        int incl = yes ? de : 0;
#pragma unroll
        for (int o = 1; o < G; o <<= 1) {
            const int y = __shfl_sync(FULL, incl, (j - o) & (G - 1), G);
            incl += pos >= (uint32_t)o ? y : 0;
        }
        bool bad = (cm & am) != 0u;
        if constexpr (TM == kThrGlobal)
            bad = bad || (uint32_t)(x0 + incl - (yes ? de : 0)) >= (uint32_t)kScanWords;
        if constexpr (TM == kThrWindow) {
            const int e = bin + incl - (yes ? de : 0);
            bad = bad || e < vlo || e > vhi;
        }
        const unsigned bb = turned((__ballot_sync(FULL, valid && bad) & gm) >> gbase, h);
        const uint32_t nd = bb ? (uint32_t)__ffs(bb) - 1u : nv;    // attempts decided
        const bool decided = pos < nd;
        const bool commit = yes && decided;
        const unsigned chg = turned((__ballot_sync(FULL, commit && de != 0) & gm) >> gbase, h);
        if (commit) {
            v.commit(a, b, na, nb);
            S[k] = (IdxT)b;
            S[N + m] = (IdxT)a;
            ++acc;
            // a move ends the run at the energy before it
            const unsigned prev = chg & before;
            const uint32_t cnt = prev ? pos - 31u + (uint32_t)__clz(prev) : carry + pos;
            if (de != 0 && cnt != 0u) atomicAdd(hist + (bin + incl - de), (unsigned long long)cnt);
        }
        carry = chg ? nd - 31u + (uint32_t)__clz(chg) : carry + nd;
        if (tun) {      // (the same in the whole block)
            unsigned tl = turned((__ballot_sync(FULL, commit && bin + incl <= tlo) & gm) >> gbase, h);
            unsigned th = turned((__ballot_sync(FULL, commit && bin + incl >= thi) & gm) >> gbase, h);
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
        // (with nd = 0 no attempt is left and every lane's incl is 0)
        bin += __shfl_sync(FULL, incl, (int)(h + nd) - 1, G);
        // what this lane goes on with: its next attempt, or the same one again
        const uint32_t a_i = a, b_i = b, k_i = k, m_i = m;
        k = decided ? kn : k;
        m = decided ? mn : m;
        a = decided ? an : a;
        b = decided ? bn : b;
        r2p = decided ? r2n : r2p;
        kn = decided ? kq : kn;
        mn = decided ? mq : mn;
        r2n = decided ? r2q : r2n;
        // its list entries, read before this round's commits, where a commit
        // moved one of its slots (at most one commit of a round per slot)
        bool hit = false;
        const uint32_t s_i = commit ? k_i : 0xFFFFFFFFu, t_i = commit ? m_i : 0xFFFFFFFFu;
        if constexpr (sizeof(IdxT) == 2) {
            const uint32_t slots = (s_i & 0xFFFFu) | (t_i << 16);   // slot indices are below 65535
            const uint32_t own = k | (m << 16);
            uint32_t low = 0xFFFFFFFFu;      // the least of each half over the lanes
#pragma unroll
            for (int i = 0; i < G; ++i) low = __vminu2(low, __shfl_sync(FULL, slots, i, G) ^ own);
            hit = (low & 0xFFFFu) == 0u || low < 0x10000u;
        } else {
#pragma unroll
            for (int i = 0; i < G; ++i) {
                const uint32_t ki = __shfl_sync(FULL, s_i, i, G), mi = __shfl_sync(FULL, t_i, i, G);
                hit = hit || ki == k || mi == m;
            }
        }
        if (__any_sync(FULL, hit)) {
#pragma unroll
            for (int i = 0; i < G; ++i) {
                const uint32_t ki = __shfl_sync(FULL, s_i, i, G), mi = __shfl_sync(FULL, t_i, i, G);
                const uint32_t ai = __shfl_sync(FULL, a_i, i, G), bi = __shfl_sync(FULL, b_i, i, G);
                a = ki == k ? bi : a;
                b = mi == m ? ai : b;
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
            if (tw.broken) {
                uint32_t ok = 0;
                for (uint32_t i = 0; i < kWaitLimit && !ok; ++i) ok = mbar_try_wait(mbar_s, tw.phase);
            } else {
                tw.wait(p);
            }
            __syncwarp(gm);
            if (j == 0) mbar_inval(mbar_s);
        }
    }
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(FULL, acc, o);
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

template <int D, typename IdxT, int G, int TM, int VIEW>
__device__ __forceinline__ void scan_item(const SysParams &p, const BlockWork &wk, uint32_t *smem,
                                          uint64_t sweeps, uint32_t iter)
{
    const int lw = threadIdx.x / G;
    const bool active = lw < wk.count;
    const int w = wk.walker0 + (active ? lw : 0);
    const uint32_t *thr = TM == kThrShared ? smem : (TM == kThrWindow ? p.thr : p.thrT);
    unsigned long long *hist = hist_row(p, w, wk.hist_row);
    const uint64_t A = sweeps * (uint64_t)p.N;
    uint32_t *state = smem + (TM == kThrShared ? thr_words_aligned(p) : 0);
    uint32_t ring_s = 0u, mbar_s = 0u;
    if constexpr (TM == kThrWindow) {
        const uint32_t wpb = blockDim.x / G;
        const uint32_t used = VIEW == kViewField ? wpb * (uint32_t)field_bytes(p)
                              : VIEW == kViewBitsShared ? wpb * (uint32_t)p.words * 4u : 0u;
        window_addrs(p, (uint32_t)__cvta_generic_to_shared(state) + used, (int)wpb, active ? lw : 0,
                     ring_s, mbar_s);
    }
    if constexpr (VIEW == kViewField) {
        if constexpr (TM == kThrShared) block_copy_words(smem, p.thr, (size_t)p.n_bins * (size_t)p.tstride);
        field_build<D, IdxT>(p, wk, state);   // ends with a block barrier, which also covers the table
        const ScanField<D> v{(uint32_t)__cvta_generic_to_shared(state) +
                             (uint32_t)((size_t)(active ? lw : 0) * field_bytes(p))};
        chain_scan<D, IdxT, G, TM>(p, w, active, v, thr, hist, A, iter, ring_s, mbar_s);
        field_finish<IdxT>(p, wk, state);
    } else {
        constexpr bool SB = VIEW == kViewBitsShared;
        const BlockSetup bs = block_setup(p, wk, smem, SB ? 1 : 0, TM == kThrShared ? 1 : 0);
        uint32_t *bits0 = SB ? state : p.bits + (size_t)wk.walker0 * (size_t)p.words;
        const ScanBits<D, SB> v{bits0 + (size_t)(active ? lw : 0) * p.words};
        chain_scan<D, IdxT, G, TM>(p, w, active, v, thr, hist, A, iter, ring_s, mbar_s);
        block_finish(bs, SB ? 1 : 0);
    }
}

// Block b takes work item b; with a counter (persistent launches), then the
// items that it pulls from it.
template <int G, int TM, int VIEW>
__global__ void __launch_bounds__(kGroupMaxThreads, 1)
walker_update_scan(const SysParams *__restrict__ sys, const BlockWork *__restrict__ work,
                   uint64_t sweeps, uint32_t iter, int n_items, int *next_item)
{
    extern __shared__ __align__(16) uint32_t smem[];
    __shared__ int s_item;
    int item = blockIdx.x;
    for (;;) {
        const BlockWork wk = work[item];
        const SysParams &p = sys[wk.sys];
        if (p.d == 2) {
            if (p.idx16) scan_item<2, uint16_t, G, TM, VIEW>(p, wk, smem, sweeps, iter);
            else scan_item<2, uint32_t, G, TM, VIEW>(p, wk, smem, sweeps, iter);
        } else {
            if (p.idx16) scan_item<3, uint16_t, G, TM, VIEW>(p, wk, smem, sweeps, iter);
            else scan_item<3, uint32_t, G, TM, VIEW>(p, wk, smem, sweeps, iter);
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
