// resident_ops.cuh -- which domains run on the multi-step kernels, and their launches.
#pragma once

#include <algorithm>

#include "resident.cuh"

namespace axl {

// Populations that a grid keeps in L2 between steps: beyond this the step
// kernels, which stream them through shared memory by TMA, are faster.
constexpr size_t kResMaxBytes = 64u << 20;
constexpr int kResSmemMax = 224 << 10;  // dynamic shared memory of a CTA (half of it with two CTAs per SM)
constexpr int kResClusterMax = 8;  // CTAs of a portable cluster

// Pairs of CTA [p0, p1) with a node on the outline of an nr x nz domain (nl nodes per pair).
inline int res_ring_pairs(int p0, int p1, int nr, int nz, int nl) {
    const int last = (nz - 1) / nl;
    int count = 0;
    for (int kp = p0 / nr; kp * (long long)nr < p1; ++kp) {
        const int ja = std::max(p0 - kp * nr, 0), jb = std::min(p1 - kp * nr, nr) - 1;
        if (kp == 0 || kp == last) count += jb - ja + 1;
        else count += (ja == 0) + (jb == nr - 1 && nr > 1);
    }
    return count;
}

// Tables of CTA `rank` of domain y: pairs on its tile's outline, and how many
// of their slots other CTAs own.
template <int NL, class Dom>
void res_tile_tables(const Dom& y, int rank, bool sw, bool th, int* pairs, int* ghosts) {
    const int nr = y.G.nr, nz = y.G.nz, planes = 9 + (sw ? 4 : 0) + (th ? 4 : 0);
    const ResTile t(y, (nz + NL - 1) / NL, rank);
    *pairs = *ghosts = 0;
    for (int kl = 0; kl < t.h; ++kl)
        for (int jl = 0; jl < t.w; jl += (kl == 0 || kl == t.h - 1 || t.w < 3) ? 1 : t.w - 1) {
            const int j = t.j0 + jl, kp = t.k0 + kl;
            const bool two = NL == 2 && NL * kp + 1 < nz;
            const bool ring = j == 0 || j == nr - 1 || kp == 0 || NL * kp + (two ? 1 : 0) == nz - 1;
            *pairs += 1;
            for (int q = 1; q < planes; ++q) {
                const int er = q < 9 ? cr9(q) : cr4((q - 9) & 3), ez = q < 9 ? cz9(q) : cz4((q - 9) & 3);
                for (int l = 0; l < (two ? 2 : 1); ++l) {
                    if (ring) {  // the link may be wrapped, mirrored or bounced back
                        int ql, p, how;
                        res_where<NL>(y.G, q, j, NL * kp + l, ql, p, how);
                        *ghosts += t.index(p % nr, p / nr) < 0;
                        continue;
                    }
                    const int row = NL == 1 ? -2 * ez : l - ez;  // below 0 or above 1: another row of pairs
                    const int kq = kl + (row < 0 ? -1 : (row > 1 ? 1 : 0));
                    *ghosts += kq < 0 || kq >= t.h || jl - er < 0 || jl - er >= t.w;
                }
            }
        }
}

// Splits a domain of nr x nkp pairs (nl nodes each) into the fewest tiles of
// at most `most` pairs that are no longer than three times their width where
// the domain lets them; the words a tile exchanges grow with its outline.
inline int res_tiling(int nr, int nkp, int nl, int most, int* w, int* h) {
    int best = 0x7fffffff, edge = 0;
    for (int square = 1; square >= 0 && best == 0x7fffffff; --square)
        for (int tx = 1; tx <= nr; ++tx) {
            const int tw = (nr + tx - 1) / tx;
            if (tx > 1 && tw == (nr + tx - 2) / (tx - 1)) continue;  // the same width in fewer tiles
            if (tw > most) continue;
            const int ty = (nkp + most / tw - 1) / (most / tw), th = (nkp + ty - 1) / ty;
            if (square && ((tw > 3 * nl * th && th < nkp) || (nl * th > 3 * tw && tw < nr))) continue;
            const int tiles = ((nr + tw - 1) / tw) * ((nkp + th - 1) / th);
            if (tiles < best || (tiles == best && tw + nl * th < edge)) {
                best = tiles;
                edge = tw + nl * th;
                *w = tw;
                *h = th;
            }
        }
    return best;
}

template <class R>
int res_lanes() { return std::is_same<R, float>::value ? 2 : 1; }

template <class S, bool SW, bool TH>
cudaError_t res_build(Resident* r, const ResidentDomain* d, int n, int num_sms, cudaStream_t stream) {
    using R = typename std::conditional<std::is_same<S, double>::value, double, float>::type;
    const int nl = res_lanes<R>();
    size_t state = 0;
    long long pairs = 0;
    std::vector<ResDom<S, R>> doms(n);
    for (int i = 0; i < n; ++i) {
        const ResidentDomain& x = d[i];
        const Geom& G = x.G;
        // grids whose steps end with passes of their own (wet walls, Zou-He walls, the mirror column) and
        // cut domains keep the step kernels
        if (G.inner == AXLBM_INNER_AXIS_NODE || G.outer != AXLBM_OUTER_BB || G.z_lo == AXLBM_Z_NEE ||
            G.z_hi == AXLBM_Z_NEE || G.z_lo == AXLBM_Z_HALO || G.z_hi == AXLBM_Z_HALO)
            return cudaSuccess;
        const int planes = 9 + (SW ? 4 : 0) + (TH ? 4 : 0);
        if (planes * G.plane >= (1ll << kResHowShift)) return cudaSuccess;  // offsets of the outline table
        state += (size_t)G.nr * G.nz * (9 + (SW ? 4 : 0) + (x.th ? 4 : 0)) * sizeof(S);
        const long long np = (long long)((G.nz + nl - 1) / nl) * G.nr;
        if (state > kResMaxBytes) return cudaSuccess;
        pairs += np;
        ResDom<S, R>& y = doms[i];
        y.pop = static_cast<S*>(x.pop);
        y.G = G;
        y.C = make_coef<R>(x.tau, x.forcing, x.boundary);
        y.C.mrt = x.mrt;
        y.az0 = x.forcing.az0;
        y.omega_t = x.forcing.omega_t;
        y.az = x.az;
        y.az16 = x.az16;
        y.mail = nullptr;
        y.th = x.th;
        y.npairs = (int)np;
    }
    r->sw = SW;
    r->th = TH;
    cudaError_t e;
    std::vector<int> cta_dom;
    // One domain of up to 8 x 256 pairs: a cluster.  A warp of FP32 pairs per
    // scheduler of an SM keeps a step at the latency of one thread, so an SM
    // takes 128 pairs before the next CTA is added; FP64 nodes are spread at a
    // warp per SM, whose FP64 pipe one warp already fills.
    if (n == 1 && pairs <= kResClusterMax * kResThreads) {
        const int full = nl == 2 ? 128 : 32;
        int c = 1;
        while (c < kResClusterMax && pairs > (long long)c * full) c *= 2;
        const int chunk = (int)((pairs + c - 1) / c);
        doms[0].cta0 = 0;
        doms[0].ncta = c;
        doms[0].chunk = chunk;
        r->cluster = true;
        r->grid = c;
        r->threads = res_up32(chunk);
        r->smem = kResAz * sizeof(R) + (size_t)nplanes<SW, TH>() * nl * chunk * sizeof(R);
        auto kern = k_resident_cluster<S, R, SW, TH>;
        // the attribute belongs to the kernel, not to this handle: always the largest a handle can ask for
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kResSmemMax);
        if (e != cudaSuccess) return e;
        r->kernel = reinterpret_cast<const void*>(kern);
        cta_dom.assign(c, 0);
    } else {
        bool fits = false;
        auto place = [&](int chunk) {  // every domain has CTAs of its own
            int cta = 0;
            cta_dom.clear();
            for (int i = 0; i < n; ++i) {
                ResDom<S, R>& y = doms[i];
                y.cta0 = cta;
                y.chunk = chunk;
                y.ncta = (y.npairs + chunk - 1) / chunk;
                cta += y.ncta;
                cta_dom.insert(cta_dom.end(), y.ncta, i);
            }
            r->grid = cta;
        };
        auto chunk_for = [&](int most) {
            int chunk = std::max(32, res_up32((int)((pairs + most - 1) / most)));
            for (;; chunk += 32) {
                long long ctas = 0;
                for (int i = 0; i < n; ++i) ctas += (doms[i].npairs + chunk - 1) / chunk;
                if (ctas <= most) return chunk;
            }
        };
        r->cluster = false;
        // the state in shared memory, one CTA per SM: the smallest tiles that give no more CTAs than SMs
        const int room = (int)(kResSmemMax / (nplanes<SW, TH>() * nl * sizeof(R)));
        int most = std::max<int>(32, (int)((pairs + num_sms - 1) / num_sms));
        for (; n <= num_sms && most < room; most += std::max(1, most / 64)) {
            long long ctas = 0;
            for (int i = 0; i < n; ++i) {
                ResDom<S, R>& y = doms[i];
                ctas += y.ncta = res_tiling(y.G.nr, (y.G.nz + nl - 1) / nl, nl, most, &y.w, &y.h);
            }
            if (ctas > num_sms) continue;
            r->grid = (int)ctas;
            int cta = 0, chunk = 0;
            cta_dom.clear();
            for (int i = 0; i < n; ++i) {
                ResDom<S, R>& y = doms[i];
                y.tx = (y.G.nr + y.w - 1) / y.w;
                y.cta0 = cta;
                y.chunk = y.w * y.h;
                cta += y.ncta;
                cta_dom.insert(cta_dom.end(), y.ncta, i);
                chunk = std::max(chunk, y.chunk);
            }
            const bool one = chunk <= kResThreads;
            size_t smem = 0;
            for (ResDom<S, R>& y : doms) {
                const bool h = TH && y.th;
                y.max_tab = y.max_ghost = 1;
                bool inner_seen = false;
                for (int c = 0; c < y.ncta; ++c) {
                    // whole tiles away from the domain's outline are alike: the first one stands for all
                    const int nkp = (y.G.nz + nl - 1) / nl;
                    const ResTile T(y, nkp, c);
                    const bool inner = T.j0 > 0 && T.k0 > 0 && T.j0 + T.w < y.G.nr && T.k0 + T.h < nkp && T.w == y.w && T.h == y.h;
                    if (inner && inner_seen) continue;
                    inner_seen |= inner;
                    int t, g;
                    res_tile_tables<Lanes<typename PairArith<R>::type>::n>(y, c, SW, h, &t, &g);
                    y.max_tab = std::max(y.max_tab, t);
                    y.max_ghost = std::max(y.max_ghost, g);
                }
                // (a domain without h in a batch with it has fewer planes)
                size_t need = h ? res_slab_smem<R, SW, TH>(y.chunk, y.max_ghost) : res_slab_smem<R, SW, false>(y.chunk, y.max_ghost);
                if (!one)
                    need += res_pairs_bytes<R>(y.chunk, y.max_ghost) + res_column_bytes<R, SW, TH>(y.w) +
                            y.max_tab * (h ? res_row_bytes<R, SW, TH>() : res_row_bytes<R, SW, false>());
                smem = std::max(smem, need);
            }
            if (smem > (size_t)kResSmemMax) break;
            r->smem = smem;
            const int iters = (chunk + kResSlabThreads - 1) / kResSlabThreads;
            r->threads = one ? kResThreads : std::max(kResThreads, res_up32((chunk + iters - 1) / iters));
            const auto k1 = k_resident_one<S, R, SW, TH>;
            const auto k2 = k_resident_slab<S, R, SW, TH>;
            r->kernel = one ? reinterpret_cast<const void*>(k1) : reinterpret_cast<const void*>(k2);
            e = cudaFuncSetAttribute(r->kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kResSmemMax);
            if (e != cudaSuccess) return e;
            int got = 0;
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&got, r->kernel, r->threads, r->smem);
            if (e != cudaSuccess) return e;
            fits = (long long)got * num_sms >= r->grid;
            r->slab = true;
            r->one = one;
            break;
        }
        // The state in L2.  Not with 16-bit storage: shared memory takes domains up
        // to where a step kernel already has 300 k pairs to work on (in shared
        // memory and with the step kernels: 512 x 768, 100 steps: 0.72 and 1.39 ms;
        // 96 x 144, 300 steps: 0.55 and 2.58 ms).
        if constexpr (std::is_same<S, R>::value) {
            auto kern = k_resident_grid<S, R, SW, TH>;
            for (int per_sm = 2; per_sm >= 1 && !fits; --per_sm) {
                const int most = per_sm * num_sms;
                if (n > most) return cudaSuccess;
                const int chunk = chunk_for(most);
                place(chunk);
                int ring = 0;
                for (const ResDom<S, R>& y : doms)
                    for (int c = 0; c < y.ncta; ++c)
                        ring = std::max(ring, res_ring_pairs(c * chunk, std::min((c + 1) * chunk, y.npairs), y.G.nr, y.G.nz, nl));
                const int iters = (chunk + kResThreads - 1) / kResThreads;
                r->slab = false;
                r->kernel = reinterpret_cast<const void*>(kern);
                r->threads = res_up32((chunk + iters - 1) / iters);
                r->smem = res_grid_smem<R, SW, TH>(chunk, ring);
                if (r->smem > (size_t)(per_sm == 2 ? kResSmemMax / 2 : kResSmemMax)) continue;
                e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kResSmemMax);
                if (e != cudaSuccess) return e;
                int got = 0;
                e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&got, kern, r->threads, r->smem);
                if (e != cudaSuccess) return e;
                fits = (long long)got * num_sms >= r->grid;
            }
        }
        if (!fits) return cudaSuccess;
    }
    // descriptors, CTA map, step counters or words, count of CTAs with their time level: one allocation of the library's own
    const size_t b_doms = (n * sizeof(ResDom<S, R>) + 255) / 256 * 256;
    const size_t b_map = (cta_dom.size() * sizeof(int) + 255) / 256 * 256;
    auto words = [&](const ResDom<S, R>& y) {  // (whole 128-byte lines per domain)
        const size_t b = (size_t)y.ncta * nplanes<SW, TH>() * nl * 2 * (y.w + y.h) * sizeof(typename ResWord<R>::type);
        return (b + 127) / 128 * 128;
    };
    size_t b_flags = (size_t)r->grid * kResPad * sizeof(unsigned);
    if (r->slab) {
        b_flags = 0;
        for (const ResDom<S, R>& y : doms) b_flags += words(y);
    }
    b_flags = (b_flags + 127) / 128 * 128;
    const size_t b_taken = 128;
    if (cudaMalloc(&r->scratch, b_doms + b_map + b_flags + b_taken) != cudaSuccess) {
        cudaGetLastError();
        r->scratch = nullptr;
        return cudaSuccess;  // no room for it: the step kernels run
    }
    r->off_map = b_doms;
    r->off_flags = b_doms + b_map;
    r->off_taken = r->off_flags + b_flags;
    char* m = static_cast<char*>(r->scratch);
    if (r->slab) {
        size_t off = r->off_flags;
        for (ResDom<S, R>& y : doms) {
            y.mail = m + off;
            off += words(y);
        }
    }
    e = cudaMemcpyAsync(m, doms.data(), n * sizeof(ResDom<S, R>), cudaMemcpyHostToDevice, stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(m + r->off_map, cta_dom.data(), cta_dom.size() * sizeof(int), cudaMemcpyHostToDevice, stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(m + r->off_flags, 0, b_flags + b_taken, stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(stream);  // the lists live on this stack
    r->epoch = 0;
    r->on = e == cudaSuccess;
    return e;
}

template <class S>
cudaError_t res_build_any(Resident* r, const ResidentDomain* d, int n, bool sw, bool th, int num_sms, cudaStream_t st) {
    if (sw && th) return res_build<S, true, true>(r, d, n, num_sms, st);
    if (sw) return res_build<S, true, false>(r, d, n, num_sms, st);
    if (th) return res_build<S, false, true>(r, d, n, num_sms, st);
    return res_build<S, false, false>(r, d, n, num_sms, st);
}

template <class S>
ResidentOps make_resident_ops() {
    ResidentOps o;
    o.build = &res_build_any<S>;
    return o;
}

}  // namespace axl
