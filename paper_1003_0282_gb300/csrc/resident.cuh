// resident.cuh -- many lattice steps of a small domain (or of a small batch) in one launch.
//
// A domain whose populations fit the L2 cache spends most of a step outside
// the collision: the launches of a step (an even bulk kernel, an odd bulk
// kernel, the ring kernels) each cost microseconds and fill few of the 152
// SMs.  The kernels here advance a whole run of plain steps instead.  Each
// thread keeps the nodes it owns for the whole launch; a step is "load the
// node's slots, collide, store the same slots, meet the neighbours".  In the
// AA pattern a node reads and writes one set of slots per step (its own in
// even steps, in odd steps the slots it pulls from, which are the ones it
// pushes to), and no other node touches them in that step, so one meeting per
// step is enough.  The boundary rules are the addresses of those slots and
// are worked out once per launch, from classify() as the ring kernels use it.
//
// Three forms, chosen by res_build():
//   k_resident_cluster  one thread-block cluster (up to 8 CTAs), one node
//     pair per thread (FP64: one node), the state in shared memory for the
//     whole launch; neighbours' slots are reached through distributed shared
//     memory and a step ends with the cluster barrier.
//   k_resident_one, k_resident_slab  a cooperative grid, one CTA per SM, each
//     with the state of a tile of one domain in shared memory (one pair, or
//     several, per thread); populations that cross tiles travel through L2 as
//     words of value and step that the reader polls with a bound.
//   k_resident_grid     (FP32, FP64) a cooperative grid, the state in global
//     memory (L2); a CTA owns a contiguous range of node pairs of one domain
//     and after every step waits only for the CTAs whose nodes its own
//     exchange populations with (a step counter per CTA, polled with a bound).
//
// Arithmetic and storage are those of the step kernels (PairArith, NodeArith,
// Codec), rounding included: a run here equals the same steps launched one by
// one.  With 16-bit storage (S) shared memory holds the FP32 value (R) of what
// would be stored, rounded through S on every store, and the nodes that the
// ring kernels update take their arithmetic in odd steps.
#pragma once

#include <cooperative_groups.h>

#include <vector>

#include "ops_impl.cuh"

namespace axl {

constexpr int kResThreads = 256;  // threads of a CTA, at most
constexpr int kResAz = 256;       // steps whose force a(t) is kept ready (even)
constexpr int kResPad = 32;       // 32-bit words between two CTAs' step counters (one 128-byte line each)
constexpr long long kResWait = kWaitCycles;
__host__ __device__ constexpr int res_up32(int v) { return (v + 31) / 32 * 32; }

// One domain as the resident kernels see it, and the CTAs it has.
template <class S, class R>
struct ResDom {
    S* pop;
    Geom G;
    Coef<R> C;
    double az0, omega_t;
    double* az;      // a(t) by AA parity: where the step kernels read it (two values)
    double* az16;    // a batch domain's copy for the bulk kernel, or null
    void* mail;      // words between CTAs: [CTA][plane][lane][place on the tile's outline]
    int th;
    int npairs;      // node pairs (FP64: nodes), pair p = (row pair p / nr, column p % nr)
    int cta0, ncta;  // CTAs [cta0, cta0 + ncta)
    int chunk;       // cluster, grid in L2: consecutive pairs of a CTA; else the most pairs of a CTA
    int tx, w, h;    // state in shared memory: tiles of w columns x h row pairs, tx in a row
    int max_tab, max_ghost;  // rows of a CTA's slot table, slots of other CTAs, at most
};

// The rectangle of pairs that CTA `rank` of domain D keeps in shared memory.
struct ResTile {
    int j0, k0, w, h;
    template <class D>
    __host__ __device__ ResTile(const D& d, int nkp, int rank)
        : j0((rank % d.tx) * d.w), k0((rank / d.tx) * d.h), w(d.G.nr - j0 < d.w ? d.G.nr - j0 : d.w),
          h(nkp - k0 < d.h ? nkp - k0 : d.h) {}
    // place of a pair of the tile's outline along it: first row, last row, first column, last column
    __host__ __device__ int outline(int j, int kp) const {
        const int jl = j - j0, kl = kp - k0;
        return kl == 0 ? jl : (kl == h - 1 ? w + jl : (jl == 0 ? 2 * w + kl : 2 * w + h + kl));
    }
    // index of pair (j, kp) in the tile, or -1
    __host__ __device__ int index(int j, int kp) const {
        return j >= j0 && j < j0 + w && kp >= k0 && kp < k0 + h ? (kp - k0) * w + (j - j0) : -1;
    }
};

// The slot that population (er, ez) of node (j, k) is pulled from in an odd
// step -- and pushed to in the opposite direction: its D2Q9 or D2Q4 plane,
// its node, and how a value changes on the way: 0 not at all, 1 through the
// axis (g changes sign), 2 + face off a solid face.
struct ResSlot {
    int plane, j, k, how;
};
__host__ __device__ __forceinline__ ResSlot res_slot9(const Geom& G, int a, int j, int k) {
    const Site s = classify(G, j, k, -cr9(a), -cz9(a));
    if (s.solid) return {a, j, k, 2 + s.face};
    return {opp9(idx9(s.fr ? -cr9(a) : cr9(a), s.fz ? -cz9(a) : cz9(a))), s.j, s.k, s.fr ? 1 : 0};
}
__host__ __device__ __forceinline__ ResSlot res_slot4(const Geom& G, int q, int j, int k) {
    const Site s = classify(G, j, k, -cr4(q), -cz4(q));
    if (s.solid) return {q, j, k, 2 + s.face};
    return {opp4(idx4(s.fr ? -cr4(q) : cr4(q), s.fz ? -cz4(q) : cz4(q))), s.j, s.k, s.fr ? 1 : 0};
}

// g and h on their way through a slot, as the step kernels' boundary rules
// round them, without a branch: g' = sg g + cg with sg = 1, -1 (axis, or off a
// wall: cg = rho0 u_w / 2), h' = (sh h + ch) + ct with sh = -1, ch = -T_ref/2,
// ct = T_w/2 off a wall of given temperature, else h.  What adds nothing is
// -0, which leaves either zero as it is.
template <class R>
__device__ __forceinline__ void res_through_g(const Geom& G, const Coef<R>& C, int how, int j, R& sg, R& cg) {
    sg = how == 0 ? R(1) : R(-1);
    cg = how >= 2 ? mul_rn(R(0.5) * C.rho0, wall_uth(G, C, how - 2, j)) : R(-0.0);
}
template <class R>
__device__ __forceinline__ void res_through_h(const Coef<R>& C, int how, R& sh, R& ch, R& ct) {
    const bool dirichlet = how >= 2 && pick4(C.t_dir, how - 2);
    sh = dirichlet ? R(-1) : R(1);
    ch = dirichlet ? R(-0.5) * C.t_ref : R(-0.0);
    ct = dirichlet ? R(0.5) * pick4(C.t_w, how - 2) : R(-0.0);
}

// The slot of plane-ordered population q of node (j, k): plane-ordered slot
// and lane (ql), pair, and how a value changes on the way.
template <int NL>
__host__ __device__ __forceinline__ void res_where(const Geom& G, int q, int j, int k, int& ql, int& p, int& how) {
    const ResSlot s = q < 9 ? res_slot9(G, q, j, k) : res_slot4(G, (q - 9) & 3, j, k);
    ql = (q < 9 ? s.plane : 9 + ((q - 9) & ~3) + s.plane) * NL + s.k % NL;
    p = (s.k / NL) * G.nr + s.j;
    how = s.how;
}

// a(t) in R, as the step kernels round it.
template <class R>
__device__ __forceinline__ R res_az(double az0, double omega_t, long long t) {
    return R(force_at(az0, omega_t, t));
}

// The time level a launch starts from.  The device clock alone knows it (a
// replay of steps that the caller captured moves it on without the host).
// A thread loads it when the kernel starts, so that its set-up hides the load.
__device__ __forceinline__ long long res_start(const Clock* clock) {
    return *reinterpret_cast<const volatile long long*>(&clock->t);
}

// A CTA of a grid has its time level t0 (one thread, behind the barrier that
// shared it).  The last CTA to say so moves the clock on: nobody is left to
// read it.  `taken` wraps to zero.
__device__ __forceinline__ void res_taken(Clock* clock, unsigned* taken, long long t0, int nsteps) {
    if (atomicInc(taken, gridDim.x - 1) == gridDim.x - 1) clock->t = t0 + nsteps;
}

// The force after the last step of a launch, at level t1 (an even level; the
// odd entry holds the last step's force, as after single steps).
template <class S, class R>
__device__ __forceinline__ void res_finish(const ResDom<S, R>& D, long long t1) {
    const double a0 = force_at(D.az0, D.omega_t, t1), a1 = force_at(D.az0, D.omega_t, t1 - 1);
    D.az[0] = a0;
    D.az[1] = a1;
    if (D.az16) {
        D.az16[0] = a0;
        *reinterpret_cast<float*>(D.az16 + 1) = (float)a0;
        D.az16[2] = a1;
        *reinterpret_cast<float*>(D.az16 + 3) = (float)a1;
    }
}

template <class RC>
__device__ __forceinline__ RC res_make(typename ScalarOf<RC>::type a, typename ScalarOf<RC>::type b);
template <>
__device__ __forceinline__ F2 res_make<F2>(float a, float b) { return F2(a, b); }
template <>
__device__ __forceinline__ D1 res_make<D1>(double a, double) { return D1(a); }

// What one thread holds of its pair for a whole launch: how g and h change on
// their way through its slots (the slots' addresses are the kernels' own).
template <class RC, bool SW, bool TH>
struct ResLinks {
    RC sg[SW ? 4 : 1], cg[SW ? 4 : 1], sh[TH ? 4 : 1], ch[TH ? 4 : 1], ct[TH ? 4 : 1];
    __device__ __forceinline__ void set_g(int q, const RC& s, const RC& c) {
        if (SW) sg[SW ? q : 0] = s, cg[SW ? q : 0] = c;
    }
    __device__ __forceinline__ RC g(int q, RC v) const { return SW ? fmaR(v, sg[SW ? q : 0], cg[SW ? q : 0]) : v; }
    __device__ __forceinline__ RC h(int q, RC v) const {
        return TH ? fmaR(v, sh[TH ? q : 0], ch[TH ? q : 0]) + ct[TH ? q : 0] : v;
    }
};

// v as storage S keeps it.
template <class S, class R>
__device__ __forceinline__ R res_keep(R v) {
    if constexpr (std::is_same<S, R>::value) return v;
    S t;
    Codec<S>::store(&t, v);
    return Codec<S>::load(&t);
}

// Lanes (bit l: row k0 + l) of a pair of column j that the ring kernels update
// in odd steps with an arithmetic of their own, which is so with 16-bit
// storage only: the outer ring, without the side columns where the bulk
// kernels take them (Geom::side).
template <class S, class R>
__device__ __forceinline__ unsigned res_ring(const Geom& G, int j, int k0) {
    if constexpr (std::is_same<S, R>::value) return 0;
    const bool column = (j == 0 || j == G.nr - 1) && !(G.inner == AXLBM_INNER_AXIS && G.nr >= 3 && G.nz >= 3);
    return (column || k0 == 0 || k0 == G.nz - 1 ? 1u : 0u) | (column || k0 + 1 == G.nz - 1 ? 2u : 0u);
}

// A node of the ring kernels.  Plain float expressions are fused by the
// compiler within a basic block, and what it hoists out of a loop over steps is
// no longer there to fuse: a call keeps the expressions as a ring kernel has
// them, and with them the rounding.
template <class R, bool SW, bool TH>
__device__ __noinline__ void res_ring_collide(Cell<R, SW, TH>& s, R inv_r, const Coef<R>& C, R az) {
    s.collide(inv_r, C, az);
}

// Collides a pair: the lanes of `ring` as the ring kernels do, at 1/r = inv_ring().
template <class S, class RC, class R, bool SW, bool TH, class Inv>
__device__ __forceinline__ void res_collide(Cell<RC, SW, TH>& c, R inv_r, const Coef<R>& C, R az, unsigned ring,
                                            const Coef<R>& Cg, const Inv& inv_ring) {
    if constexpr (!std::is_same<S, R>::value) {
        if (ring) {
            const Cell<RC, SW, TH> in = c;
            if (ring != 3u) c.collide(inv_r, C, az);
            const R inv = inv_ring();
#pragma unroll 1
            for (int l = 0; l < 2; ++l) {
                if (!((ring >> l) & 1u)) continue;
                Cell<R, SW, TH> s;
                auto put = [&](RC& to, R v) { to = l ? RC(Lanes<RC>::get(to, 0), v) : RC(v, Lanes<RC>::get(to, 1)); };
#pragma unroll
                for (int a = 0; a < 9; ++a) s.d[a] = Lanes<RC>::get(in.d[a], l);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (SW) s.g[q] = Lanes<RC>::get(in.g[q], l);
                    if (TH) s.h[q] = Lanes<RC>::get(in.h[q], l);
                }
                res_ring_collide(s, inv, Cg, az);
#pragma unroll
                for (int a = 0; a < 9; ++a) put(c.d[a], s.d[a]);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (SW) put(c.g[q], s.g[q]);
                    if (TH) put(c.h[q], s.h[q]);
                }
            }
            return;
        }
    }
    c.collide(inv_r, C, az);
}

// Load / store the populations of a pair: at(q, l) is the value of plane-
// ordered slot q of lane l; in odd steps links change g and h on the way, and
// slot q takes the opposite population.
template <class RC, bool SW, bool TH, int PAR, class At, class Links>
__device__ __forceinline__ void res_load(Cell<RC, SW, TH>& c, const At& at, const Links& L) {
    constexpr int NL = Lanes<RC>::n, HP = SW ? 13 : 9;
#pragma unroll
    for (int a = 0; a < 9; ++a) c.d[a] = res_make<RC>(at(a, 0), at(a, NL - 1));
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        if (SW) c.g[q] = res_make<RC>(at(9 + q, 0), at(9 + q, NL - 1));
        if (TH) c.h[q] = res_make<RC>(at(HP + q, 0), at(HP + q, NL - 1));
        if (SW && PAR) c.g[q] = L.g(q, c.g[q]);
        if (TH && PAR) c.h[q] = L.h(q, c.h[q]);
    }
}
template <class S, class RC, bool SW, bool TH, int PAR, class To, class Links>
__device__ __forceinline__ void res_store(const Cell<RC, SW, TH>& c, const To& to, const Links& L) {
    constexpr int NL = Lanes<RC>::n, HP = SW ? 13 : 9;
#pragma unroll
    for (int q = 0; q < 9 + (SW ? 4 : 0) + (TH ? 4 : 0); ++q) {
        const int o = opp4((q - 9) & 3), m = (q - 9) & 3;
        RC x = q < 9 ? c.d[opp9(q)] : (SW && q < 13 ? c.g[o] : c.h[o]);
        if (PAR && SW && q >= 9 && q < 13) x = L.g(m, x);
        if (PAR && TH && q >= HP) x = L.h(m, x);
#pragma unroll
        for (int l = 0; l < NL; ++l) to(q, l, res_keep<S>(Lanes<RC>::get(x, l)));
    }
}

// Links of the pair in rows k0 and k0 + 1 of column j, and its slots as
// put(q, l, ql, p) takes them; a lane without a node keeps to itself (p = -1).
template <class RC, class R, bool SW, bool TH, class Put>
__device__ __forceinline__ void res_links(const Geom& G, const Coef<R>& C, int j, int k0, ResLinks<RC, SW, TH>& L,
                                          const Put& put) {
    constexpr int NL = Lanes<RC>::n, P = 9 + (SW ? 4 : 0) + (TH ? 4 : 0), HP = SW ? 13 : 9;
#pragma unroll
    for (int q = 0; q < P; ++q) {
        R sg[NL], cg[NL], sh[NL], ch[NL], ct[NL];
#pragma unroll
        for (int l = 0; l < NL; ++l) {
            int ql = q * NL + l, p = -1, how = 0;
            if (k0 + l < G.nz) res_where<NL>(G, q, j, k0 + l, ql, p, how);
            put(q, l, ql, p);
            if (SW && q >= 9 && q < 13) res_through_g<R>(G, C, how, j, sg[l], cg[l]);
            if (TH && q >= HP) res_through_h<R>(C, how, sh[l], ch[l], ct[l]);
        }
        const int m = (q - 9) & 3;
        if (SW && q >= 9 && q < 13) {
            L.sg[SW ? m : 0] = res_make<RC>(sg[0], sg[NL - 1]);
            L.cg[SW ? m : 0] = res_make<RC>(cg[0], cg[NL - 1]);
        }
        if (TH && q >= HP) {
            L.sh[TH ? m : 0] = res_make<RC>(sh[0], sh[NL - 1]);
            L.ch[TH ? m : 0] = res_make<RC>(ch[0], ch[NL - 1]);
            L.ct[TH ? m : 0] = res_make<RC>(ct[0], ct[NL - 1]);
        }
    }
}

// ---------------------------------------------------------------------------- cluster

__device__ __forceinline__ uint32_t res_mapa(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void res_dst(uint32_t a, float v) {
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void res_dst(uint32_t a, double v) {
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
__device__ __forceinline__ void res_dld(uint32_t a, float& v) {
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
}
__device__ __forceinline__ void res_dld(uint32_t a, double& v) {
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory");
}

// One cluster of D.ncta CTAs, thread i of a CTA owning pair rank * chunk + i.
// Shared memory: the force table, then the state [plane][lane][chunk].
//
// What bounds it: the latency of one step of one thread (slots, the chain of
// the collision, barrier); the throughput of one scheduler for more pairs.
// FP64: the FP64 pipe, whatever a warp's active lanes (64 cycles per warp
// instruction of a warp alone on its SM, 76 with one on each scheduler).
template <class S, class R, bool SW, bool TH>
__global__ void __launch_bounds__(kResThreads, 1)
k_resident_cluster(const ResDom<S, R>* __restrict__ doms, Clock* clock, int nsteps) {
    using RC = typename PairArith<R>::type;
    constexpr int NL = Lanes<RC>::n, P = nplanes<SW, TH>();
    extern __shared__ __align__(16) unsigned char res_smem[];
    const ResDom<S, R>& D = doms[0];
    const Geom& G = D.G;
    uint32_t nclust;
    asm("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(nclust));
    if ((int)nclust != D.ncta) {  // not launched as one cluster: nothing is touched
        if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(&clock->err, 1u);
        return;
    }
    const long long t0 = res_start(clock);
    R* az_tab = reinterpret_cast<R*>(res_smem);
    R* st = az_tab + kResAz;
    const int tid = threadIdx.x, chunk = D.chunk, ncta = D.ncta, rank = blockIdx.x;
    const int p = rank * chunk + tid;
    const bool on = tid < chunk && p < D.npairs;
    const int nr = G.nr, kp = on ? p / nr : 0, j = on ? p - kp * nr : 0, k0 = NL * kp;
    const Coef<R> C = D.C;
    R* const mine = st + tid;
    uint32_t at[P][NL];
    ResLinks<RC, SW, TH> L;
    if (on) {  // natural-layout state into shared memory; the slots of odd steps
#pragma unroll
        for (int q = 0; q < P; ++q)
#pragma unroll
            for (int l = 0; l < NL; ++l) mine[(q * NL + l) * chunk] = k0 + l < G.nz ? Codec<S>::load(slot(D.pop, G, q, j, k0 + l)) : R(0);
        res_links<RC, R, SW, TH>(G, C, j, k0, L, [&](int q, int l, int ql, int sp) {
            if (sp < 0) sp = p;
            const int sr = sp / chunk, si = sp - sr * chunk;
            at[q][l] = res_mapa(smem_u32(st) + (uint32_t)((ql * chunk + si) * sizeof(R)), sr);
        });
    }
    const R inv_r = step_inv_radius<R>(G, j);
    const unsigned ring = res_ring<S, R>(G, j, k0);
    auto meet = [&]() {
        if (ncta == 1) {
            __syncthreads();
        } else {
            asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
        }
    };
    for (int s = 0; s < nsteps; ++s) {
        if (s % kResAz == 0) {  // (the meeting that ended the last step has everybody past the old entries)
            for (int i = tid; i < kResAz && s + i < nsteps; i += blockDim.x)
                az_tab[i] = res_az<R>(D.az0, D.omega_t, t0 + s + i);
            if (s == 0) meet();  // and the state of every CTA is in place
            else __syncthreads();
        }
        if (on) {
            const R az = az_tab[s % kResAz];
            Cell<RC, SW, TH> c;
            if ((s & 1) == 0) {  // even step: own slots, back into the opposite ones
                res_load<RC, SW, TH, 0>(c, [&](int q, int l) { return mine[(q * NL + l) * chunk]; }, L);
                c.collide(inv_r, C, az);
                res_store<S, RC, SW, TH, 0>(c, [&](int q, int l, R v) { mine[(q * NL + l) * chunk] = v; }, L);
            } else {
                R v[P][NL];
#pragma unroll
                for (int q = 0; q < P; ++q)
#pragma unroll
                    for (int l = 0; l < NL; ++l) res_dld(at[q][l], v[q][l]);
                res_load<RC, SW, TH, 1>(c, [&](int q, int l) { return v[q][l]; }, L);
                res_collide<S>(c, inv_r, C, az, ring, D.C, [&]() { return inv_radius<R>(G, j); });
                res_store<S, RC, SW, TH, 1>(c, [&](int q, int l, R x) { res_dst(at[q][l], x); }, L);
            }
        }
        meet();
    }
    if (on) {
#pragma unroll
        for (int l = 0; l < NL; ++l) {
            if (k0 + l >= G.nz) continue;
#pragma unroll
            for (int q = 0; q < P; ++q) Codec<S>::store(slot(D.pop, G, q, j, k0 + l), mine[(q * NL + l) * chunk]);
        }
    }
    if (rank == 0 && tid == 0) {  // (every CTA took its time level before the first meeting)
        res_finish(D, t0 + nsteps);
        clock->t = t0 + nsteps;
    }
}

// ---------------------------------------------------------------------------- grid, state in shared memory

// A population on its way between two CTAs: the value and the step it is for
// in one 8-byte word (FP64: two halves, each with the step), written and read
// with relaxed 8-byte accesses.  The reader polls the word itself, so a hop
// costs one store and one load of L2 (590 to 1170 cycles one way on GB300,
// median 1070) where a flag behind a release costs 1730 to 2500.
// One word serves a slot in both directions: its owner and the node that uses
// it in odd steps take turns.
template <class R>
struct ResWord;
template <>
struct ResWord<float> {
    using type = unsigned long long;
    __device__ static __forceinline__ void store(type* p, float v, unsigned step) {
        const type w = ((type)step << 32) | __float_as_uint(v);
        asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(w) : "memory");
    }
    __device__ static __forceinline__ type load(const type* p) {
        type w;
        asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(w) : "l"(p) : "memory");
        return w;
    }
    __device__ static __forceinline__ bool is(type w, unsigned step) { return (unsigned)(w >> 32) == step; }
    __device__ static __forceinline__ float value(type w) { return __uint_as_float((unsigned)w); }
};
template <>
struct ResWord<double> {
    using type = ulonglong2;
    __device__ static __forceinline__ void store(type* p, double v, unsigned step) {
        const unsigned long long b = (unsigned long long)__double_as_longlong(v), t = (unsigned long long)step << 32;
        asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(t | (b & 0xffffffffull)),
                     "l"(t | (b >> 32))
                     : "memory");
    }
    __device__ static __forceinline__ type load(const type* p) {
        type w;
        asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(w.x), "=l"(w.y) : "l"(p) : "memory");
        return w;
    }
    __device__ static __forceinline__ bool is(const type& w, unsigned step) {
        return (unsigned)(w.x >> 32) == step && (unsigned)(w.y >> 32) == step;
    }
    __device__ static __forceinline__ double value(const type& w) {
        return __longlong_as_double((long long)((w.y << 32) | (w.x & 0xffffffffull)));
    }
};

// Shared memory of a CTA whose state sits there: the force table; the values
// (its own slots [plane][lane][chunk], then copies of other CTAs' slots that
// its nodes use in odd steps, the "ghosts"); per ghost this CTA's own slot
// that the same neighbour uses, and the words of the two.
template <class R>
struct ResSlab {
    R *az, *st;
    int *own, *even, *odd;  // [max_ghost]
    unsigned char* rest;
    __device__ ResSlab(unsigned char* smem, int values, int max_ghost) {
        az = reinterpret_cast<R*>(smem);
        st = az + kResAz;
        own = reinterpret_cast<int*>(st + values + max_ghost);
        even = own + max_ghost;
        odd = even + max_ghost;
        rest = reinterpret_cast<unsigned char*>(odd + max_ghost);
    }
};
template <class R, bool SW, bool TH>
__host__ __device__ constexpr size_t res_slab_smem(int chunk, int max_ghost) {
    return (kResAz + (size_t)nplanes<SW, TH>() * Lanes<typename PairArith<R>::type>::n * chunk + max_ghost) * sizeof(R) +
           (size_t)max_ghost * 3 * sizeof(int);
}

// Words of a step into shared memory (PAR 0: the CTA's own slots, 1: the
// ghosts), a thread's polls all in flight together; a poll gives up after
// kResWait cycles, or when another CTA has.
template <class R, int PAR>
__device__ __forceinline__ void res_gather(const ResSlab<R>& S, const typename ResWord<R>::type* mail, int gbase, int ng,
                                           unsigned want, Clock* clock, int* bad) {
    using W = ResWord<R>;
    constexpr int U = 2;  // a tile's outline rarely has more than two words per thread
    const int T = blockDim.x;
    for (int g0 = threadIdx.x; g0 < ng; g0 += U * T) {
        typename W::type w[U];
        int from[U];
        unsigned miss = 0;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            from[u] = 0;
            if (g0 + u * T < ng) {
                from[u] = (PAR ? S.odd : S.even)[g0 + u * T];
                miss |= 1u << u;
            }
        }
        const long long w0 = clock64();
        for (int tries = 0; miss; ++tries) {
#pragma unroll
            for (int u = 0; u < U; ++u)
                if ((miss >> u) & 1u) w[u] = W::load(mail + from[u]);
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (((miss >> u) & 1u) && W::is(w[u], want)) {
                    S.st[PAR ? gbase + g0 + u * T : S.own[g0 + u * T]] = W::value(w[u]);
                    miss &= ~(1u << u);
                }
            if ((tries & 255) == 255) {
                const bool late = clock64() - w0 > kResWait;
                if (late || *reinterpret_cast<volatile int*>(bad) || *reinterpret_cast<volatile unsigned*>(&clock->err)) {
                    if (late) atomicOr(&clock->err, 1u);
                    *bad = 1;
                    break;
                }
            }
        }
    }
}
// The step's results that belong to other CTAs (odd) or that they use next (even).
template <class R, int PAR>
__device__ __forceinline__ void res_scatter(const ResSlab<R>& S, typename ResWord<R>::type* mail, int gbase, int ng,
                                            unsigned step) {
    for (int g = threadIdx.x; g < ng; g += blockDim.x)
        ResWord<R>::store(mail + (PAR ? S.odd : S.even)[g], S.st[PAR ? gbase + g : S.own[g]], step);
}

// The word of slot ql of pair (j, kp), which lies on the outline of its tile:
// words of one side of a tile lie side by side, apart from other tiles'.
template <int PL, class D>
__host__ __device__ __forceinline__ int res_word(const D& d, int nkp, int ql, int j, int kp) {
    const int rank = (kp / d.h) * d.tx + j / d.w;
    return (rank * PL + ql) * (2 * (d.w + d.h)) + ResTile(d, nkp, rank).outline(j, kp);
}

// A lane's slot in another CTA becomes a ghost: its number (consecutive within
// the warp, so that copies and words lie side by side), or -1.
__device__ __forceinline__ int res_new_ghost(bool remote, int* count) {
    const unsigned act = __activemask(), m = __ballot_sync(act, remote);
    const int lane = threadIdx.x & 31, first = __ffs(m) - 1;
    int g = 0;
    if (remote && lane == first) g = atomicAdd(count, __popc(m));
    if (m) g = __shfl_sync(act, g, first);
    return remote ? g + __popc(m & ((1u << lane) - 1u)) : -1;
}

// The common part of the kernels that keep the state in shared memory: loads
// it, runs nsteps steps of update(par, force), each between the words of its
// neighbours coming in and going out, and writes it back.
template <class S_, class R, bool SW, bool TH, class Update>
__device__ __forceinline__ void res_slab_run(const ResDom<S_, R>& D, const ResSlab<R>& S, Clock* clock, int nsteps,
                                             unsigned epoch, unsigned* taken, long long t_start, int ng, int* bad,
                                             const Update& update) {
    constexpr int NL = Lanes<typename PairArith<R>::type>::n, PL = nplanes<SW, TH>() * NL;
    const Geom& G = D.G;
    const int tid = threadIdx.x, T = blockDim.x, chunk = D.chunk;
    const int rank = blockIdx.x - D.cta0, gbase = PL * chunk;
    const ResTile tile(D, (G.nz + NL - 1) / NL, rank);
    auto* mail = static_cast<typename ResWord<R>::type*>(D.mail);
    auto step = [&](auto par_tag, int s) {
        constexpr int PAR = decltype(par_tag)::value;
        if (s > 0 && ng > 0) {
            res_gather<R, PAR>(S, mail, gbase, ng, epoch + (unsigned)s, clock, bad);
            __syncthreads();
        }
        update(par_tag, S.az[s % kResAz]);
        __syncthreads();
        if (ng > 0) res_scatter<R, PAR>(S, mail, gbase, ng, epoch + (unsigned)s + 1u);
    };
    __shared__ long long t0;
    if (tid == 0) t0 = t_start;
    int stop = __syncthreads_or(*bad);
    if (tid == 0) res_taken(clock, taken, t_start, nsteps);
    for (int s = 0; s < nsteps && !stop; s += 2) {
        if (s % kResAz == 0) {
            for (int i = tid; i < kResAz && s + i < nsteps; i += T) S.az[i] = res_az<R>(D.az0, D.omega_t, t0 + s + i);
            __syncthreads();
        }
        step(std::integral_constant<int, 0>{}, s);
        step(std::integral_constant<int, 1>{}, s + 1);
        // (a wait that gives up ends the loop for the whole CTA: looked at rarely, and after the last step)
        if ((s & 62) == 62) stop = __syncthreads_or(*bad);
    }
    if (!stop && ng > 0) res_gather<R, 0>(S, mail, gbase, ng, epoch + (unsigned)nsteps, clock, bad);
    if (__syncthreads_or(*bad)) {
        if (tid == 0) atomicOr(&clock->err, 1u);
        return;
    }
    const int n = tile.w * tile.h;
    for (int m = tid; m < PL * n; m += T) {
        const int ql = m / n, i = m - ql * n, kl = i / tile.w, j = tile.j0 + i - kl * tile.w, k = NL * (tile.k0 + kl) + ql % NL;
        if (k < G.nz) Codec<S_>::store(slot(D.pop, G, ql / NL, j, k), S.st[ql * chunk + i]);
    }
    if (rank == 0 && tid == 0) res_finish(D, t0 + nsteps);
}

// One pair per thread: addresses and links stay in registers.
template <class S_, class R, bool SW, bool TH>
__device__ __forceinline__ void res_one_cta(const ResDom<S_, R>& D, Clock* clock, int nsteps, unsigned epoch, unsigned* taken,
                                            unsigned char* smem) {
    using RC = typename PairArith<R>::type;
    constexpr int NL = Lanes<RC>::n, P = nplanes<SW, TH>();
    __shared__ int ghosts, bad;
    const long long t_start = res_start(clock);
    const Geom& G = D.G;
    const Coef<R> C = D.C;
    const int tid = threadIdx.x, chunk = D.chunk, nr = G.nr, nkp = (G.nz + NL - 1) / NL;
    const int gbase = P * NL * chunk, max_ghost = D.max_ghost;
    const ResTile tile(D, nkp, blockIdx.x - D.cta0);
    const int n = tile.w * tile.h;
    const ResSlab<R> S(smem, gbase, max_ghost);
    if (tid == 0) ghosts = bad = 0;
    __syncthreads();
    const bool on = tid < n;
    const int kl = (on ? tid : 0) / tile.w, j = tile.j0 + (on ? tid : 0) - kl * tile.w, kp = tile.k0 + kl, k0 = NL * kp;
    R* const mine = S.st + tid;
    int at[P][NL];
    ResLinks<RC, SW, TH> L;
    if (tid < res_up32(n)) {  // whole warps
        res_links<RC, R, SW, TH>(G, C, j, k0, L, [&](int q, int l, int ql, int sp) {
            const int here = sp < 0 ? tid : tile.index(sp % nr, sp / nr);
            const int g = res_new_ghost(on && here < 0, &ghosts);
            at[q][l] = g < 0 ? ql * chunk + max(here, 0) : gbase + g;
            if (g >= max_ghost) {
                bad = 2;
                at[q][l] = gbase;
            } else if (g >= 0) {
                S.own[g] = (q * NL + l) * chunk + tid;
                S.even[g] = res_word<P * NL>(D, nkp, q * NL + l, j, kp);
                S.odd[g] = res_word<P * NL>(D, nkp, ql, sp % nr, sp / nr);
            }
            if (on) mine[(q * NL + l) * chunk] = k0 + l < G.nz ? Codec<S_>::load(slot(D.pop, G, q, j, k0 + l)) : R(0);
        });
    }
    __syncthreads();
    const R inv_r = step_inv_radius<R>(G, j);
    const unsigned ring = res_ring<S_, R>(G, j, k0);
    res_slab_run<S_, R, SW, TH>(D, S, clock, nsteps, epoch, taken, t_start, min(ghosts, max_ghost), &bad, [&](auto par_tag, R az) {
        constexpr int PAR = decltype(par_tag)::value;
        if (!on) return;
        Cell<RC, SW, TH> c;
        if (PAR == 0) {
            res_load<RC, SW, TH, 0>(c, [&](int q, int l) { return mine[(q * NL + l) * chunk]; }, L);
            c.collide(inv_r, C, az);
            res_store<S_, RC, SW, TH, 0>(c, [&](int q, int l, R v) { mine[(q * NL + l) * chunk] = v; }, L);
        } else {
            res_load<RC, SW, TH, 1>(c, [&](int q, int l) { return S.st[at[q][l]]; }, L);
            res_collide<S_>(c, inv_r, C, az, ring, D.C, [&]() { return inv_radius<R>(G, j); });
            res_store<S_, RC, SW, TH, 1>(c, [&](int q, int l, R v) { S.st[at[q][l]] = v; }, L);
        }
    });
}

// Cooperative grid, one CTA per SM, one pair per thread; CTA b works for
// domain cta_dom[b].
//
// What bounds it: the latency of a step -- the neighbours' words (a store and
// a polled load of L2), one node's chain, two barriers.
template <class S, class R, bool SW, bool TH>
__global__ void __launch_bounds__(kResThreads, 1)
k_resident_one(const ResDom<S, R>* __restrict__ doms, const int* __restrict__ cta_dom, Clock* clock, int nsteps,
               unsigned epoch, unsigned* taken) {
    extern __shared__ __align__(16) unsigned char res_smem[];
    const ResDom<S, R>& D = doms[cta_dom[blockIdx.x]];
    if (TH && D.th) res_one_cta<S, R, SW, TH>(D, clock, nsteps, epoch, taken, res_smem);
    else res_one_cta<S, R, SW, false>(D, clock, nsteps, epoch, taken, res_smem);
}

constexpr int kResSlabThreads = 384;

constexpr int kResRingShift = 28;  // a pair's index in the tile below, the lanes of res_ring above
constexpr int kResPairMask = (1 << kResRingShift) - 1;

// A pair of the kernel below: its index in the tile; tab: its row of the slot
// table, or -1 away from the tile's outline, where every slot is the CTA's own.
template <class R>
struct ResPair {
    float inv_r;
    int i, tab;
};
template <>
struct ResPair<double> {
    int col, i, tab;  // col: column of the tile
};
// Bytes of the pairs, so that what follows lies on an 8-byte boundary.
template <class R>
__host__ __device__ constexpr size_t res_pairs_bytes(int chunk, int max_ghost) {
    const size_t b = (size_t)chunk * sizeof(ResPair<R>);
    return b + (sizeof(R) == 8 ? (8 - (b + (size_t)max_ghost * 3 * sizeof(int)) % 8) % 8 : 0);
}
// A row of the slot table: where population (q, l) is pulled from in an odd
// step (index into the values), then the links.
template <class R, bool SW, bool TH>
__host__ __device__ constexpr size_t res_row_bytes() {
    return Lanes<typename PairArith<R>::type>::n *
           (nplanes<SW, TH>() * sizeof(int) + ((SW ? 8 : 0) + (TH ? 12 : 0)) * sizeof(R));
}

// FP64: what the collision takes of each column of the tile, in shared memory
// (recomputed per node it would be a tenth of the FP64 instructions).
template <class R, bool SW, bool TH>
__host__ __device__ constexpr size_t res_column_bytes(int w) {
    return sizeof(R) == 8 ? (size_t)w * sizeof(ColCoef<SW, TH>) : 0;
}

// Several pairs per thread.
template <class S_, class R, bool SW, bool TH>
__device__ __forceinline__ void res_slab_cta(const ResDom<S_, R>& D, Clock* clock, int nsteps, unsigned epoch, unsigned* taken,
                                             unsigned char* smem) {
    using RC = typename PairArith<R>::type;
    constexpr int NL = Lanes<RC>::n, P = nplanes<SW, TH>(), PL = P * NL, NF = (SW ? 8 : 0) + (TH ? 12 : 0);
    __shared__ int ghosts, bad, rows;
    const long long t_start = res_start(clock);
    const Geom& G = D.G;
    const Coef<R> C = D.C;
    const int tid = threadIdx.x, T = blockDim.x, chunk = D.chunk, nr = G.nr, nkp = (G.nz + NL - 1) / NL;
    const int gbase = PL * chunk, max_ghost = D.max_ghost, max_tab = D.max_tab;
    const ResTile tile(D, nkp, blockIdx.x - D.cta0);
    const int tw = tile.w, n = tw * tile.h;
    const ResSlab<R> S(smem, gbase, max_ghost);
    ResPair<R>* pairs = reinterpret_cast<ResPair<R>*>(S.rest);
    R* tf = reinterpret_cast<R*>(S.rest + res_pairs_bytes<R>(chunk, max_ghost));  // [NF][NL][max_tab]: sg, cg, then sh, ch, ct, four each
    ColCoef<SW, TH>* columns = reinterpret_cast<ColCoef<SW, TH>*>(tf + NF * NL * max_tab);  // [w], FP64 only
    int* tab = reinterpret_cast<int*>(reinterpret_cast<unsigned char*>(columns) + res_column_bytes<R, SW, TH>(D.w));  // [P][NL][max_tab]
    if (tid == 0) ghosts = bad = 0;
    __syncthreads();
    // pairs in order, those with a row of the table last (a warp's slots and words then lie side by side)
    if (tid < 32) {
        int plain = 0;
        for (int pass = 0; pass < 2; ++pass) {
            int at0 = 0, at1 = plain;
            for (int i0 = 0; i0 < n; i0 += 32) {
                const int i = i0 + tid, kl = i / tw, jl = i - kl * tw;
                const bool row = jl == 0 || jl == tw - 1 || kl == 0 || kl == tile.h - 1;  // the tile's outline
                const unsigned m0 = __ballot_sync(0xffffffffu, i < n && !row), m1 = __ballot_sync(0xffffffffu, i < n && row);
                if (pass && i < n) {
                    ResPair<R> r;
                    if constexpr (sizeof(R) == 8) r.col = jl;
                    else r.inv_r = step_inv_radius<R>(G, tile.j0 + jl);
                    r.i = i | (int)(res_ring<S_, R>(G, tile.j0 + jl, NL * (tile.k0 + kl)) << kResRingShift);
                    const int to = row ? at1 + __popc(m1 & ((1u << tid) - 1u)) : at0 + __popc(m0 & ((1u << tid) - 1u));
                    r.tab = row ? to - plain : -1;
                    pairs[to] = r;
                }
                at0 += __popc(m0);
                at1 += __popc(m1);
            }
            if (!pass) plain = at0;
        }
        if (tid == 0) {
            rows = n - plain;
            if (rows > max_tab) bad = 2;
        }
    }
    __syncthreads();
    const int nt = rows, n0 = n - nt;
    if (!bad) {
        const int blocks = (nt + 31) / 32, lane = tid & 31;
        for (int w = tid >> 5; w < blocks * PL; w += T >> 5) {  // 32 pairs of one population and lane
            const int x = w / blocks, t = (w - x * blocks) * 32 + lane, q = x / NL, l = x - q * NL;
            const bool on = t < nt;
            const int i = pairs[n0 + (on ? t : 0)].i & kResPairMask, kl = i / tw, j = tile.j0 + i - kl * tw, kp = tile.k0 + kl, k = NL * kp + l;
            int ql = x, sp = kp * nr + j, how = 0;  // (a lane without a node keeps to itself)
            if (k < G.nz) res_where<NL>(G, q, j, k, ql, sp, how);
            const int here = tile.index(sp % nr, sp / nr);
            const int g = res_new_ghost(on && here < 0, &ghosts);
            int e = here >= 0 ? ql * chunk + here : gbase + g;
            if (g >= max_ghost) {
                bad = 2;
                e = gbase;
            } else if (g >= 0) {
                S.own[g] = x * chunk + i;
                S.even[g] = res_word<PL>(D, nkp, x, j, kp);
                S.odd[g] = res_word<PL>(D, nkp, ql, sp % nr, sp / nr);
            }
            if (on) {
                tab[x * max_tab + t] = e;
                const int m = (q - 9) & 3;
                R* f = tf + l * max_tab + t;
                
                if (SW && q >= 9 && q < 13) {
                    R sg, cg;
                    res_through_g<R>(G, C, how, j, sg, cg);
                    f[m * NL * max_tab] = sg;
                    f[(4 + m) * NL * max_tab] = cg;
                }
                if (TH && q >= (SW ? 13 : 9)) {
                    R sh, ch, ct;
                    res_through_h<R>(C, how, sh, ch, ct);
                    constexpr int B = SW ? 8 : 0;
                    f[(B + m) * NL * max_tab] = sh;
                    f[(B + 4 + m) * NL * max_tab] = ch;
                    f[(B + 8 + m) * NL * max_tab] = ct;
                }
            }
        }
    }
    if constexpr (sizeof(R) == 8)
        for (int jl = tid; jl < tw; jl += T) columns[jl].set(step_inv_radius<R>(G, tile.j0 + jl), C);
    for (int m = tid; m < PL * n; m += T) {  // the state, natural layout
        const int ql = m / n, i = m - ql * n, kl = i / tw, j = tile.j0 + i - kl * tw, k = NL * (tile.k0 + kl) + ql % NL;
        S.st[ql * chunk + i] = k < G.nz ? Codec<S_>::load(slot(D.pop, G, ql / NL, j, k)) : R(0);
    }
    __syncthreads();
    // links read from the table where they are used
    struct TabLinks {
        const R* f;
        int stride;
        __device__ __forceinline__ RC of(int x) const {
            return res_make<RC>(f[x * NL * stride], f[(x * NL + NL - 1) * stride]);
        }
        __device__ __forceinline__ RC g(int q, RC v) const { return fmaR(v, of(q), of(4 + q)); }
        __device__ __forceinline__ RC h(int q, RC v) const {
            constexpr int B = SW ? 8 : 0;
            return fmaR(v, of(B + q), of(B + 4 + q)) + of(B + 8 + q);
        }
    };
    res_slab_run<S_, R, SW, TH>(D, S, clock, nsteps, epoch, taken, t_start, min(ghosts, max_ghost), &bad, [&](auto par_tag, R az) {
        constexpr int PAR = decltype(par_tag)::value;
        for (int m = tid; m < n; m += T) {
            const ResPair<R> r = pairs[m];
            const int i = std::is_same<S_, R>::value ? r.i : r.i & kResPairMask;
            R* const mine = S.st + i;
            // index (from `mine`) of the slot of population q, lane l, in an odd step without a table row
            auto inside = [&](int q, int l) {
                const int er = q < 9 ? cr9(q) : cr4((q - 9) & 3), ez = q < 9 ? cz9(q) : cz4((q - 9) & 3);
                const int pl = q < 9 ? opp9(q) : 9 + ((q - 9) & ~3) + opp4((q - 9) & 3);
                if (NL == 1) return pl * chunk - ez * tw - er;
                const int row = l - ez;  // -1, 0, 1, 2: of the pair below, this pair, this pair, the pair above
                return (pl * NL + (row & 1)) * chunk + (row < 0 ? -tw : (row > 1 ? tw : 0)) - er;
            };
            const TabLinks tl{tf + r.tab, max_tab};
            struct NoLinks {
                __device__ __forceinline__ RC g(int, RC v) const { return v; }
                __device__ __forceinline__ RC h(int, RC v) const { return v; }
            } none;
            const int* e = tab + r.tab;
            Cell<RC, SW, TH> c;
            if (PAR == 0) res_load<RC, SW, TH, 0>(c, [&](int q, int l) { return mine[(q * NL + l) * chunk]; }, none);
            else if (r.tab < 0) res_load<RC, SW, TH, 1>(c, [&](int q, int l) { return mine[inside(q, l)]; }, none);
            else res_load<RC, SW, TH, 1>(c, [&](int q, int l) { return S.st[e[(q * NL + l) * max_tab]]; }, tl);
            if constexpr (sizeof(R) == 8) c.collide_d1(columns[r.col], C, az);
            else if (PAR == 0) c.collide(r.inv_r, C, az);
            else
                res_collide<S_>(c, r.inv_r, C, az, (unsigned)r.i >> kResRingShift, D.C,
                                [&]() { return inv_radius<R>(G, tile.j0 + i % tw); });
            if (PAR == 0) res_store<S_, RC, SW, TH, 0>(c, [&](int q, int l, R v) { mine[(q * NL + l) * chunk] = v; }, none);
            else if (r.tab < 0) res_store<S_, RC, SW, TH, 1>(c, [&](int q, int l, R v) { mine[inside(q, l)] = v; }, none);
            else res_store<S_, RC, SW, TH, 1>(c, [&](int q, int l, R v) { S.st[e[(q * NL + l) * max_tab]] = v; }, tl);
        }
    });
}

// Cooperative grid, one CTA per SM, several pairs per thread.
//
// What bounds it: FP32 latency at three warps a scheduler (words in, barrier,
// update, barrier, words out in series; a third of the issue slots used); the
// FP64 pipe.
template <class S, class R, bool SW, bool TH>
__global__ void __launch_bounds__(kResSlabThreads, 1)
k_resident_slab(const ResDom<S, R>* __restrict__ doms, const int* __restrict__ cta_dom, Clock* clock, int nsteps,
                unsigned epoch, unsigned* taken) {
    extern __shared__ __align__(16) unsigned char res_smem[];
    const ResDom<S, R>& D = doms[cta_dom[blockIdx.x]];
    if (TH && D.th) res_slab_cta<S, R, SW, TH>(D, clock, nsteps, epoch, taken, res_smem);
    else res_slab_cta<S, R, SW, false>(D, clock, nsteps, epoch, taken, res_smem);
}

// ---------------------------------------------------------------------------- grid, state in L2

// Shared memory of a grid CTA: the force table, a record per pair, and for
// the pairs with a node on the domain's outline the slots of odd steps.
template <class R>
struct ResRec {
    R inv_r;
    int x;     // offset of the pair's first node in a plane; bit 30: the second lane is empty
    int ring;  // entry of the outline table, or -1
};
constexpr int kResHowShift = 28;   // an outline entry: offset below, ResSlot::how above
constexpr int kResOff = (1 << kResHowShift) - 1;

template <class R, bool SW, bool TH>
__host__ __device__ constexpr size_t res_ring_bytes() {
    return Lanes<typename PairArith<R>::type>::n * (nplanes<SW, TH>() * sizeof(int) + (SW ? 4 * sizeof(R) : 0));
}
template <class R, bool SW, bool TH>
__host__ __device__ constexpr size_t res_grid_smem(int chunk, int max_ring) {
    return kResAz * sizeof(R) + (size_t)chunk * sizeof(ResRec<R>) + (size_t)max_ring * res_ring_bytes<R, SW, TH>();
}

__device__ __forceinline__ unsigned res_ld_acquire(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void res_st_release(unsigned* p, unsigned v) {
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

template <class R>
__device__ __forceinline__ R res_ring_g(R v, int how, R cg) {
    return how == 0 ? v : (how == 1 ? -v : cg - v);
}
template <class R>
__device__ __forceinline__ R res_ring_h(R v, int how, const Coef<R>& C) {
    return how < 2 ? v : bounce_h(C, how - 2, v);
}

// One step of the CTA's pairs.  PAR 1: an odd step (neighbours' slots).
template <class S, class R, bool SW, bool TH, int PAR>
__device__ __forceinline__ void res_grid_step(const ResDom<S, R>& D, const Coef<R>& C, const ResRec<R>* rec, int n,
                                              const int* ring_at, const R* ring_cg, R az) {
    using RC = typename PairArith<R>::type;
    constexpr int NL = Lanes<RC>::n, P = nplanes<SW, TH>(), HP = SW ? 13 : 9;
    const int plane = (int)D.G.plane, pitch = (int)D.G.pitch;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const ResRec<R> r = rec[i];
        const bool two = NL == 2 && !(r.x & (1 << 30));
        S* const base = D.pop + (r.x & ~(1 << 30));
        const int row1 = two ? pitch : 0;  // an empty lane repeats the first one's node (never stored)
        const bool ring = PAR == 1 && r.ring >= 0;
        const int* at = ring_at + r.ring * (P * NL);
        const R* cg = ring_cg + r.ring * (4 * NL);
        // offset from `base` of the slot of plane-ordered population q in an odd step, away from the outline
        auto inside = [&](int q) {
            const int er = q < 9 ? cr9(q) : cr4((q - 9) & 3), ez = q < 9 ? cz9(q) : cz4((q - 9) & 3);
            const int pl = q < 9 ? opp9(q) : 9 + ((q - 9) & ~3) + opp4((q - 9) & 3);
            return pl * plane - ez * pitch - er;
        };
        R v[P][NL];
        if (PAR == 0) {
#pragma unroll
            for (int q = 0; q < P; ++q)
#pragma unroll
                for (int l = 0; l < NL; ++l) v[q][l] = __ldcg(base + (q * plane + l * row1));
        } else if (!ring) {
#pragma unroll
            for (int q = 0; q < P; ++q)
#pragma unroll
                for (int l = 0; l < NL; ++l) v[q][l] = __ldcg(base + (inside(q) + l * row1));
        } else {
#pragma unroll
            for (int q = 0; q < P; ++q)
#pragma unroll
                for (int l = 0; l < NL; ++l) v[q][l] = __ldcg(D.pop + (at[q * NL + l] & kResOff));
#pragma unroll
            for (int q = 9; q < P; ++q)
#pragma unroll
                for (int l = 0; l < NL; ++l) {
                    const int how = (unsigned)at[q * NL + l] >> kResHowShift;
                    v[q][l] = SW && q < 13 ? res_ring_g<R>(v[q][l], how, cg[(q - 9) * NL + l])
                                           : res_ring_h<R>(v[q][l], how, C);
                }
        }
        Cell<RC, SW, TH> c;
#pragma unroll
        for (int a = 0; a < 9; ++a) c.d[a] = res_make<RC>(v[a][0], v[a][NL - 1]);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (SW) c.g[q] = res_make<RC>(v[9 + q][0], v[9 + q][NL - 1]);
            if (TH) c.h[q] = res_make<RC>(v[HP + q][0], v[HP + q][NL - 1]);
        }
        c.collide(r.inv_r, C, az);
        // slot q takes the opposite population (even steps: of the node itself)
#pragma unroll
        for (int l = 0; l < NL; ++l) {
            if (l && !two) continue;
            if (!ring) {
#pragma unroll
                for (int q = 0; q < P; ++q) {
                    const RC x = q < 9 ? c.d[opp9(q)] : (SW && q < 13 ? c.g[opp4((q - 9) & 3)] : c.h[opp4((q - 9) & 3)]);
                    S* to = base + ((PAR ? inside(q) : q * plane) + l * row1);
                    *to = (S)Lanes<RC>::get(x, l);
                }
            } else {
#pragma unroll
                for (int q = 0; q < P; ++q) {
                    const int e = at[q * NL + l], how = (unsigned)e >> kResHowShift;
                    const RC x = q < 9 ? c.d[opp9(q)] : (SW && q < 13 ? c.g[opp4((q - 9) & 3)] : c.h[opp4((q - 9) & 3)]);
                    R y = Lanes<RC>::get(x, l);
                    if (SW && q >= 9 && q < 13) y = res_ring_g<R>(y, how, cg[(q - 9) * NL + l]);
                    if (TH && q >= HP) y = res_ring_h<R>(y, how, C);
                    D.pop[e & kResOff] = (S)y;
                }
            }
        }
    }
}

// The work of one CTA: a contiguous range of pairs of domain D.
template <class S, class R, bool SW, bool TH>
__device__ __forceinline__ void res_grid_cta(const ResDom<S, R>& D, unsigned* flags, Clock* clock, int nsteps,
                                             unsigned epoch, unsigned* taken, unsigned char* smem) {
    using RC = typename PairArith<R>::type;
    constexpr int NL = Lanes<RC>::n, P = nplanes<SW, TH>();
    __shared__ int n_ring, abort_flag;
    __shared__ long long t0;
    const long long t_start = res_start(clock);
    const Geom& G = D.G;
    const Coef<R> C = D.C;
    const int tid = threadIdx.x, chunk = D.chunk, nr = G.nr;
    const int rank = blockIdx.x - D.cta0;
    const int p0 = rank * chunk, n = min(chunk, D.npairs - p0);
    R* az_tab = reinterpret_cast<R*>(smem);
    ResRec<R>* rec = reinterpret_cast<ResRec<R>*>(az_tab + kResAz);
    if (tid == 0) n_ring = abort_flag = 0;
    __syncthreads();
    for (int i = tid; i < n; i += blockDim.x) {
        const int p = p0 + i, kp = p / nr, j = p - kp * nr, k = NL * kp;
        const bool two = NL == 2 && k + 1 < G.nz;
        ResRec<R> r;
        r.inv_r = step_inv_radius<R>(G, j);
        r.x = (int)((long long)(G.row0 + k) * G.pitch + G.col0 + j) | (NL == 2 && !two ? 1 << 30 : 0);
        r.ring = j == 0 || j == nr - 1 || k == 0 || k + (two ? 1 : 0) == G.nz - 1 ? atomicAdd(&n_ring, 1) : -1;
        rec[i] = r;
    }
    if (tid == 0) t0 = t_start;
    __syncthreads();
    if (tid == 0) res_taken(clock, taken, t_start, nsteps);
    // outline table: the slots, and rho0 u_w / 2 where a g population meets a wall
    R* ring_cg = reinterpret_cast<R*>(rec + chunk);
    int* ring_at = reinterpret_cast<int*>(ring_cg + (SW ? n_ring * 4 * NL : 0));
    for (int i = tid; i < n; i += blockDim.x) {
        const int e = rec[i].ring;
        if (e < 0) continue;
        const int p = p0 + i, kp = p / nr, j = p - kp * nr;
        for (int l = 0; l < NL; ++l) {
            const int k = NL * kp + l < G.nz ? NL * kp + l : NL * kp;
            for (int q = 0; q < P; ++q) {
                const ResSlot s = q < 9 ? res_slot9(G, q, j, k) : res_slot4(G, (q - 9) & 3, j, k);
                const int plane = q < 9 ? s.plane : 9 + ((q - 9) & ~3) + s.plane;
                ring_at[(e * P + q) * NL + l] = (int)(slot(D.pop, G, plane, s.j, s.k) - D.pop) | (s.how << kResHowShift);
                if (SW && q >= 9 && q < 13)
                    ring_cg[(e * 4 + (q - 9)) * NL + l] =
                        s.how >= 2 ? mul_rn(R(0.5) * C.rho0, wall_uth(G, C, s.how - 2, j)) : R(0);
            }
        }
    }
    // the CTAs this one meets: owners of pairs within one node of its range,
    // and across periodic ends
    const int last = D.npairs - 1;
    const int a0 = max(p0 - nr - 1, 0) / chunk, a1 = min(p0 + n + nr, last) / chunk;
    int b0 = 0, b1 = -1, c0 = 0, c1 = -1;
    if (G.z_lo == AXLBM_Z_PERIODIC) {
        if (p0 <= nr) b0 = max(last - 2 * nr, 0) / chunk, b1 = last / chunk;
        if (p0 + n - 1 >= last - nr) c0 = 0, c1 = min(2 * nr, last) / chunk;
    }
    const int na = a1 - a0 + 1, nb = b1 - b0 + 1, nc = c1 - c0 + 1, nmeet = na + nb + nc;
    const unsigned* dom_flags = flags + (long long)D.cta0 * kResPad;
    unsigned* my_flag = flags + (long long)blockIdx.x * kResPad;
    for (int s = 0; s < nsteps; ++s) {
        if (s % kResAz == 0) {
            __syncthreads();
            for (int i = tid; i < kResAz && s + i < nsteps; i += blockDim.x)
                az_tab[i] = res_az<R>(D.az0, D.omega_t, t0 + s + i);
        }
        if (s > 0 && tid < 32) {
            const unsigned want = epoch + (unsigned)s;
            for (int m = tid; m < nmeet; m += 32) {
                const int c = m < na ? a0 + m : (m < na + nb ? b0 + (m - na) : c0 + (m - na - nb));
                if (c == rank) continue;
                const unsigned* f = dom_flags + (long long)c * kResPad;
                if ((int)(res_ld_acquire(f) - want) >= 0) continue;
                const long long w0 = clock64();
                int tries = 0;
                while ((int)(res_ld_acquire(f) - want) < 0) {
                    if (clock64() - w0 > kResWait ||
                        ((++tries & 1023) == 0 && *reinterpret_cast<volatile unsigned*>(&clock->err) != 0u)) {
                        abort_flag = 1;
                        break;
                    }
                }
            }
        }
        __syncthreads();
        if (abort_flag) break;
        const R az = az_tab[s % kResAz];
        if ((s & 1) == 0) res_grid_step<S, R, SW, TH, 0>(D, C, rec, n, ring_at, ring_cg, az);
        else res_grid_step<S, R, SW, TH, 1>(D, C, rec, n, ring_at, ring_cg, az);
        __syncthreads();
        if (tid == 0) {
            res_st_release(my_flag, epoch + (unsigned)s + 1u);
        }
    }
    if (abort_flag) {
        if (tid == 0) atomicOr(&clock->err, 1u);
        return;
    }
    if (rank == 0 && tid == 0) res_finish(D, t0 + nsteps);
}

// Cooperative grid; CTA b works for domain cta_dom[b].
//
// What bounds it: for few pairs per CTA the latency of a step -- the slots
// from L2, the collision's chain, a fence, a release store and the
// neighbours' polls -- also for many in FP32, at three warps a scheduler (38 %
// of the issue slots, 37 % of L2's rate at 512 x 1280); in FP64 the FP64 pipe.
template <class S, class R, bool SW, bool TH>
__global__ void __launch_bounds__(kResThreads, 2)
k_resident_grid(const ResDom<S, R>* __restrict__ doms, const int* __restrict__ cta_dom, unsigned* flags, Clock* clock,
                int nsteps, unsigned epoch, unsigned* taken) {
    extern __shared__ __align__(16) unsigned char res_smem[];
    const ResDom<S, R>& D = doms[cta_dom[blockIdx.x]];
    if (TH && D.th) res_grid_cta<S, R, SW, true>(D, flags, clock, nsteps, epoch, taken, res_smem);
    else res_grid_cta<S, R, SW, false>(D, flags, clock, nsteps, epoch, taken, res_smem);
}

}  // namespace axl
