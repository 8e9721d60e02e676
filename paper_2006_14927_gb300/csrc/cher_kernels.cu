// cher_kernels.cu -- every bunch of a tile of track steps, in FP64 and in
// FP32-bulk precision: the yields, the trace and, in a curved atmosphere, the
// crossings (steps a1-a5; in flat layers cher_hits.cu forms those without
// propagating every bunch).
//
// A CTA owns a tile of `BLOCK` consecutive steps:
//   phase A  one thread per step: Cherenkov yield (CERENK, paper section
//            3.2; the FP32 path screens it in FP32 and takes the FP64 chain
//            wherever the count or the photons per bunch would not be
//            certain), bunch count nb = ceil(N / B), per-step constants
//            staged in shared memory; a CTA-wide exclusive scan of nb gives
//            every bunch of the tile a slot;
//   phase B  the CTA's threads stride over the tile's bunches (the paper's
//            sub-step loop, Appendix A, unrolled across threads): Philox
//            randoms, emission point / azimuth / wavelength, the rare
//            conditions first (Algorithm 2's hoisting becomes a per-lane
//            predicate), Snell + one fine-table index for n(h) and one
//            (height, sin^2) cell for both refraction corrections (the
//            single-search refactor of section 3.3.1 and the repeated-call
//            hoisting of Algorithm 3), the ground point and arrival time
//            (RAYBND, Appendix B listing), candidate spheres from the ground
//            grid, and warp-aggregated compaction of the crossings (TELOUT;
//            the curved hits kernels queue their crossings per warp and
//            record them 32 at a time, see flush_ring).
// In the persistent variant CTAs pull tiles from an atomic queue, so showers
// of very uneven size share one launch (the paper's independent-shower
// parallelism, section 2, inside one GPU).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <type_traits>

#include "cher_internal.h"
#include "cher_path.cuh"

namespace cher {
namespace {

// The curved hits kernels record their crossings from a per-warp queue instead
// of in the window where they are found.  About 1-2 % of bunches cross a
// sphere, so a window usually holds none or one, and recording it there
// keeps 31 of 32 lanes idle through the record's ~70 instructions.  The
// window queues each (bunch, candidate) pair as 8 bytes (step in tile and
// bunch index; grid and candidate entry) in a ring of 64 in shared memory;
// once 32 are queued, and at the end of the tile while its step constants
// are still in shared memory, each lane takes one pair, computes its bunch
// again (the same function on the same inputs, so the same values) and
// writes the record with the per-(warp, telescope) atomics of record_hits.
// (The bound on a step's azimuths that cher_hits.cu uses was tried for the
// curved atmosphere too: at 70 deg, 10 bunches a step, it costs more than it
// saves, 79 -> 133 us per 3e5 steps.)
constexpr int kRing = 64;

template <class R, int BLOCK, bool TR, int FB, bool DS, bool CV>
__device__ __forceinline__ void flush_ring(const KParams &p, const Consts<R> &c, R np1o,
                                           const Seg<R> *seg, const SegD<R> *segd,
                                           const uint2 *ring, int head, int n, int64_t base,
                                           int lane, unsigned &st_over) {
    int tel = -1;
    R tx = R(0), ty = R(0), tz = R(0);
    BunchOut<R> o;
    o.status = -1;
    o.zg = R(0);
    int s = 0, j = 0;
    if (lane < n) {
        const uint2 e = ring[(head + lane) & (kRing - 1)];
        s = dbg_index(p, static_cast<int>(e.x >> 22), BLOCK, DBG_SMEM);
        j = static_cast<int>(e.x & 0x3fffffu);
        bunch<R, TR, FB, DS, CV>(p, c, seg[s], DS ? segd + s : nullptr, j, o);
        const int g = static_cast<int>(e.y >> 31);
        const int m = static_cast<int>(e.y & 0x7fffffffu);
        tel = cand_info<R>(p, g, dbg_index(p, m, g ? p.grid[1].n_cand : p.grid[0].n_cand,
                                           DBG_GRID), tx, ty, tz);
    }
    // from here on as record_hits, one crossing per lane
    const unsigned grp = __match_any_sync(kFull, tel);
    if (tel >= 0) {
        const int leader = __ffs(grp) - 1;
        const unsigned rank = __popc(grp & ((1u << lane) - 1u));
        unsigned long long slot0 = 0;
        if (lane == leader)
            slot0 = atomicAdd(p.count + tel, static_cast<unsigned long long>(__popc(grp)));
        slot0 = __shfl_sync(grp, slot0, leader);
        const unsigned long long slot = slot0 + rank;
        if (slot < static_cast<unsigned long long>(p.cap)) {
            const Seg<R> &S = seg[s];
            const int64_t gstep = p.track_base + base + s;
            const uint64_t key = (static_cast<uint64_t>(gstep) << 32) | static_cast<uint32_t>(j);
            const R lam = o.lam, tg = o.t;
            const R np1 = DS ? R(1) + o.kap * c.eta_o : np1o;
            const R sl = (tz - o.zg) / o.cz;   // to the plane through the centre
            const int64_t r = dbg_index(p, static_cast<int64_t>(tel) * p.cap +
                                               static_cast<int64_t>(slot),
                                        int64_t(p.n_tel) * p.cap, DBG_OUT);
            store4<R>(p.pos, r, o.X + sl * o.cx - tx, o.Y + sl * o.cy - ty, o.cx, o.cy);
            store4<R>(p.tim, r, tg + sl * np1 * R(1.0 / kC), o.he, S.w, lam);
            p.key[r] = key;
        } else {
            ++st_over;
        }
    }
}

// ------------------------------------------------------------------------
// The fused kernel.
// ------------------------------------------------------------------------
// TR: the atmospheric transmission draw is compiled in (a separate
// instantiation: present but switched off it cost 2 % of the launch).
// FB: bunches past the tables' zenith range are queued for the fallback
// pass (1, hits) or integrated in place (2, trace).
// DS: the index depends on the wavelength (per-step spectra in shared memory).
template <class R, int BLOCK>
__host__ __device__ constexpr size_t segd_offset() {
    return (sizeof(Seg<R>) * BLOCK + sizeof(int) * (BLOCK + 1 + 32) + 15) & ~size_t(15);
}

// the crossing queue of the curved hits kernels, after the spectra (DS)
template <class R, int BLOCK, bool DS>
__host__ __device__ constexpr size_t ring_offset() {
    return segd_offset<R, BLOCK>() + (DS ? sizeof(SegD<R>) * BLOCK : 0);
}

// CV: a curved atmosphere (radial heights, spherical shells).
template <class R, int BLOCK, int MODE, bool TR, int FB, bool DS, bool CV>
__device__ __forceinline__ void gen_prop(const KParams &p) {
    extern __shared__ __align__(16) unsigned char smem[];
    Seg<R> *seg = reinterpret_cast<Seg<R> *>(smem);
    int *off = reinterpret_cast<int *>(seg + BLOCK);          // BLOCK + 1
    int *wsum = off + BLOCK + 1;                                // BLOCK / 32
    SegD<R> *segd = reinterpret_cast<SegD<R> *>(smem + segd_offset<R, BLOCK>());   // DS only
    // the hits kernels queue their crossings (flush_ring) in a ring after
    // the spectra (the entry packs the step in the tile in 10 bits above the
    // bunch index in 22: a step has at most 2^22 bunches)
    constexpr bool kQueue = MODE == MODE_HITS;
    static_assert(BLOCK <= 1024, "the queue entry holds the step in the tile in 10 bits");
    __shared__ unsigned s_tile;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint2 *ring = reinterpret_cast<uint2 *>(smem + ring_offset<R, BLOCK, DS>()) + warp * kRing;
    int q_tail = 0, q_cnt = 0;       // (warp-uniform)
    // the candidate grids (a few KB) are read through L1; their sizes and
    // pointers come straight from the kernel parameters (selects, nothing
    // held in registers across the bunch loop)

    Consts<R> c;
    R np1o;
    make_consts<R>(p, c, np1o);

    unsigned st_steps = 0, st_emit = 0, st_inval = 0, st_bunch = 0, st_up = 0, st_below = 0,
             st_above = 0, st_angle = 0, st_absorb = 0, st_hits = 0, st_over = 0;

    // Persistent CTAs claim their next tile one tile ahead, during the scan
    // (its barriers publish the claim), and prefetch that tile's step
    // arrays into L2 while they work through the current tile's bunches; one
    // barrier per tile separates its bunch loop from the next phase A.
    int64_t tile = blockIdx.x;
    if (p.tile_counter) {
        __syncthreads();
        if (tid == 0) s_tile = atomicAdd(p.tile_counter, 1u);
        __syncthreads();
        tile = static_cast<int64_t>(s_tile);
    }
    for (;;) {
        if (tile >= p.n_tiles) break;
        const int64_t base = tile * p.tile;

        // ---- phase A: one step per thread ----------------------------------
        const int64_t i = base + tid;
        int nb = 0;
        if (tid < p.tile && i < p.n) {
            // the FP32 path screens the yield in FP32 (same bunch counts as FP64)
            using YT = typename std::conditional<std::is_same<R, float>::value, YieldF,
                                                 Yield>::type;
            YT y;
            // in a curved atmosphere the yield needs the midpoint's horizontal place
            double xyd[4];
            float xyf[4];
            if constexpr (CV) {
                xyd[0] = __ldg(p.x0 + i);
                xyd[1] = __ldg(p.y0 + i);
                xyd[2] = static_cast<double>(load_dir<R>(p.ux, i));
                xyd[3] = static_cast<double>(load_dir<R>(p.uy, i));
                xyf[0] = d2f_rn(xyd[0]);
                xyf[1] = d2f_rn(xyd[1]);
                xyf[2] = static_cast<float>(load_dir<R>(p.ux, i));
                xyf[3] = static_cast<float>(load_dir<R>(p.uy, i));
            }
            const double *pxyd = CV ? xyd : nullptr;
            const float *pxyf = CV ? xyf : nullptr;
            if constexpr (DS) {
                if constexpr (std::is_same<YT, YieldF>::value)
                    step_yield_screened_disp(p, step_valid<R>(p, i), __ldg(p.z0 + i),
                                             __ldg(p.len + i), __ldg(p.ekin + i),
                                             load_dir<float>(p.uz, i), y, segd[tid], pxyf, pxyd);
                else
                    step_yield_disp<R>(p, step_valid<R>(p, i), __ldg(p.z0 + i), __ldg(p.len + i),
                                       __ldg(p.ekin + i), static_cast<double>(load_dir<R>(p.uz, i)),
                                       y, segd[tid], pxyd);
            } else if constexpr (std::is_same<YT, YieldF>::value) {
                step_yield_screened(p, step_valid<R>(p, i), __ldg(p.z0 + i), __ldg(p.len + i),
                                    __ldg(p.ekin + i), load_dir<float>(p.uz, i), y, pxyf, pxyd);
            } else {
                step_yield(p, step_valid<R>(p, i), __ldg(p.z0 + i), __ldg(p.len + i),
                           __ldg(p.ekin + i), static_cast<double>(load_dir<R>(p.uz, i)), y, pxyd);
            }
            nb = y.nb;
            ++st_steps;
            st_emit += (nb > 0);
            st_inval += !y.valid;
            if constexpr (MODE == MODE_YIELD) {
                p.y_nb[i] = nb;
                p.y_w[i] = nb > 0 ? static_cast<double>(y.N) / static_cast<double>(nb) : 0.0;
            } else {
                prep_step<R>(p, i, y, seg[tid]);
            }
        }
        if constexpr (MODE == MODE_YIELD) {
            if (!p.tile_counter) break;
            __syncthreads();
            if (tid == 0) s_tile = atomicAdd(p.tile_counter, 1u);
            __syncthreads();
            tile = static_cast<int64_t>(s_tile);
            continue;
        }
        st_bunch += nb;

        // ---- CTA exclusive scan of nb ---------------------------------------
        int v = nb;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(kFull, v, o);
            if (lane >= o) v += t;
        }
        if (lane == 31) wsum[warp] = v;
        if (tid == 0 && p.tile_counter) s_tile = atomicAdd(p.tile_counter, 1u);
        __syncthreads();
        const int64_t next = p.tile_counter ? static_cast<int64_t>(s_tile) : p.n_tiles;
        if (warp == 0) {
            int w = lane < BLOCK / 32 ? wsum[lane] : 0;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(kFull, w, o);
                if (lane >= o) w += t;
            }
            if (lane < BLOCK / 32) wsum[lane] = w;   // inclusive warp totals
        }
        __syncthreads();
        const int excl = v - nb + (warp > 0 ? wsum[warp - 1] : 0);
        // (past the tile's steps no more starts: place `tile` is the total)
        off[tid] = tid <= p.tile ? excl : 0x7fffffff;
        if (tid == BLOCK - 1) off[BLOCK] = p.tile == BLOCK ? excl + nb : 0x7fffffff;
        __syncthreads();
        const int total = off[p.tile];
        if (next < p.n_tiles) {
            const int64_t ni = next * p.tile + tid;
            if (tid < p.tile && ni < p.n) {
                prefetch_l2(p.x0 + ni);
                prefetch_l2(p.y0 + ni);
                prefetch_l2(p.z0 + ni);
                prefetch_l2(p.t0 + ni);
                prefetch_l2(p.len + ni);
                prefetch_l2(p.ekin + ni);
                prefetch_l2(static_cast<const R *>(p.ux) + ni);
                prefetch_l2(static_cast<const R *>(p.uy) + ni);
                prefetch_l2(static_cast<const R *>(p.uz) + ni);
                if (p.shower) prefetch_l2(p.shower + ni);
            }
        }

        // ---- phase B: the tile's bunches -------------------------------------
        // Each warp takes an even share of contiguous 32-bunch windows (shares
        // differ by at most one window).  The step of a window's first bunch
        // comes from the previous window (one search per warp and tile);
        // inside a window a lane's step is the last step whose first bunch is
        // <= its own, counted from the at most 32 step starts that follow with
        // one ballot and a few shuffles.
        const int nwin = (total + 31) >> 5;
        const int w_lo = (warp * nwin) / (BLOCK / 32);
        const int w_hi = ((warp + 1) * nwin) / (BLOCK / 32);
        int s_cur = 0;
        if (w_lo < w_hi) {
            int lo = 0, hi = BLOCK;
            const int b_first = w_lo * 32;
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (off[mid] <= b_first) lo = mid; else hi = mid;
            }
            s_cur = lo;
        }
        for (int win = w_lo; win < w_hi; ++win) {
            const int bidx = win * 32 + lane;
            const bool live = bidx < total;
            int s = s_cur;
            for (int batch = s_cur;; batch += 32) {
                const int idx = batch + 1 + lane;
                const int v = (idx <= BLOCK ? off[idx] : 0x7fffffff) - win * 32;
                const int k = __popc(__ballot_sync(kFull, v <= 31));
                for (int q = 0; q < k; ++q) s += (__shfl_sync(kFull, v, q) <= lane);
                if (k < 32) break;
            }
            s_cur = __shfl_sync(kFull, s, 31);
            BunchOut<R> o;
            o.status = -1;
            o.zg = R(0);
            int j = 0;
            if (live) {
                s = dbg_index(p, s, BLOCK, DBG_SMEM);
                j = bidx - off[s];
                bunch<R, TR, FB, DS, CV>(p, c, seg[s], DS ? segd + s : nullptr, j, o);
                if (o.status != ST_GROUND) {       // rare: the drops
                    st_up += o.status == ST_UPWARD;
                    st_below += o.status == ST_BELOW;
                    st_above += o.status == ST_ABOVE;
                    st_angle += o.status == ST_ANGLE;
                    st_absorb += o.status == ST_ABSORBED;
                }
            }
            int s0 = 0, gsel = 0;
            unsigned hm = live ? sphere_hits<R, CV>(p, c, o, s0, gsel) : 0u;
            if constexpr (MODE == MODE_TRACE) {
                st_hits += __popc(hm);
                if (live) {
                    const int64_t gb =
                        dbg_index(p, __ldg(p.bunch_off + base + s) + j, p.t_nbunch, DBG_TRACE);
                    const R w = seg[s].w;
                    if (o.status == ST_GROUND) {
                        store4<R>(p.pos, gb, o.X, o.Y, o.cx, o.cy);
                        store4<R>(p.tim, gb, o.t, o.he, w, o.lam);
                    } else {
                        store4<R>(p.pos, gb, R(0), R(0), R(0), R(0));
                        store4<R>(p.tim, gb, R(0), o.he, w, o.lam);
                    }
                    p.t_status[gb] = o.status;
                    p.t_nhit[gb] = __popc(hm);
                    int first = -1;
                    for (unsigned mm = hm; mm; mm &= mm - 1u) {      // lowest telescope index
                        R tx, ty, tz;
                        const int k = cand_info<R>(p, gsel, s0 + __ffs(mm) - 1, tx, ty, tz);
                        first = (first < 0 || k < first) ? k : first;
                    }
                    p.t_first[gb] = first;
                }
            } else if constexpr (kQueue) {
                // one pair per lane and round (a lane with several crossings
                // takes several rounds), so at most 32 join a ring of < 32
                for (;;) {
                    const unsigned has = __ballot_sync(kFull, hm != 0u);
                    if (!has) break;
                    if (hm) {
                        const int bit = __ffs(hm) - 1;
                        hm &= hm - 1u;
                        const int slot =
                            (q_tail + __popc(has & ((1u << lane) - 1u))) & (kRing - 1);
                        ring[slot] = make_uint2(
                            (static_cast<uint32_t>(s) << 22) | static_cast<uint32_t>(j),
                            (static_cast<uint32_t>(gsel) << 31) | static_cast<uint32_t>(s0 + bit));
                        ++st_hits;
                    }
                    q_tail = (q_tail + __popc(has)) & (kRing - 1);
                    q_cnt += __popc(has);
                    if (q_cnt >= 32) {
                        __syncwarp();
                        flush_ring<R, BLOCK, TR, FB, DS, CV>(p, c, np1o, seg, segd, ring,
                                                             (q_tail - q_cnt) & (kRing - 1), 32,
                                                             base, lane, st_over);
                        q_cnt -= 32;
                        __syncwarp();
                    }
                }
            }
        }
        if constexpr (kQueue) {
            // the rest of the queue, while the tile's step constants are there
            __syncwarp();
            if (q_cnt > 0) {
                flush_ring<R, BLOCK, TR, FB, DS, CV>(p, c, np1o, seg, segd, ring,
                                                     (q_tail - q_cnt) & (kRing - 1), q_cnt, base,
                                                     lane, st_over);
                q_cnt = 0;
            }
            __syncwarp();
        }
        if (!p.tile_counter) break;
        // every warp is done with this tile's step constants and offsets
        // before the next tile's phase A and scan overwrite them
        __syncthreads();
        tile = next;
    }

    unsigned long long *S = p.stats;
    if (S) {
        flush_stat(S, CHER_STAT_STEPS, st_steps);
        flush_stat(S, CHER_STAT_EMITTING, st_emit);
        flush_stat(S, CHER_STAT_INVALID, st_inval);
        if (MODE != MODE_YIELD) {
            flush_stat(S, CHER_STAT_BUNCHES, st_bunch);
            flush_stat(S, CHER_STAT_UPWARD, st_up);
            flush_stat(S, CHER_STAT_BELOW_OBS, st_below);
            flush_stat(S, CHER_STAT_ABOVE_MAX, st_above);
            flush_stat(S, CHER_STAT_ANGLE, st_angle);
            flush_stat(S, CHER_STAT_ABSORBED, st_absorb);
            // reached the ground = generated - dropped (a per-thread partial
            // may be negative; the sum modulo 2^64 is exact)
            flush_stat_signed(S, CHER_STAT_GROUND,
                              static_cast<int>(st_bunch) -
                                  static_cast<int>(st_up + st_below + st_above + st_angle + st_absorb));
            flush_stat(S, CHER_STAT_HITS, st_hits);
            flush_stat(S, CHER_STAT_OVERFLOW, st_over);
        }
    }
}

// The kernels: every instantiation at the register budget of 1024 / BLOCK
// threads per SM (FP32) or of one CTA (FP64).
template <class R, int BLOCK, int MODE, bool TR, int FB, bool DS, bool CV>
__global__ void __launch_bounds__(BLOCK, std::is_same<R, float>::value ? 1024 / BLOCK : 1)
    k_gen_prop(const KParams p) {
    gen_prop<R, BLOCK, MODE, TR, FB, DS, CV>(p);
}

// ------------------------------------------------------------------------
// The fallback pass: one thread per queued bunch (warps walk the queue 32
// entries at a time so that the compaction stays warp-synchronous).
// ------------------------------------------------------------------------
template <class R, bool TR, bool DS>
__global__ void __launch_bounds__(128) k_fallback(const KParams p) {
    Consts<R> c;
    R np1o;
    make_consts<R>(p, c, np1o);
    const int lane = threadIdx.x & 31;
    const unsigned long long queued = *p.fb_count;
    const unsigned long long cap = static_cast<unsigned long long>(p.fb_cap);
    const int64_t n = static_cast<int64_t>(queued < cap ? queued : cap);
    unsigned st_fb = 0, st_absorb = 0, st_hits = 0, st_over = 0;
    const int64_t warps = static_cast<int64_t>(gridDim.x) * (blockDim.x >> 5);
    const int64_t wid = static_cast<int64_t>(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5);
    for (int64_t first = wid * 32; first < n; first += warps * 32) {
        const int64_t e = first + lane;
        const bool live = e < n;
        BunchOut<R> o;
        o.status = -1;
        o.zg = R(0);
        R w = R(0);
        uint64_t key = 0;
        if (live) {
            const FbEntry<R> E =
                static_cast<const FbEntry<R> *>(p.fb_list)[dbg_index(p, e, p.fb_cap, DBG_FB)];
            R D, L;
            if constexpr (std::is_same<R, float>::value)
                ray_integrals_f(p, E.dh, E.s_obs, E.c2, DS ? E.kap : 1.0f, D, L);
            else
                ray_integrals(p, p.h_obs + E.dh, E.s_obs, DS ? E.kap : 1.0, D, L);
            const R co = sqrt(E.c2);
            o.X = E.xe + D * E.hx;
            o.Y = E.ye + D * E.hy;
            o.t = E.te + L * R(1.0 / kC);
            o.cx = E.s_obs * E.hx;
            o.cy = E.s_obs * E.hy;
            o.cz = -co;
            o.he = E.he;
            o.lam = E.lam;
            o.kap = DS ? E.kap : R(1);
            o.status = ST_GROUND;
            w = E.w;
            key = E.key;
            const uint32_t step_hi = E.step_hi;
            ++st_fb;
            if constexpr (TR) {
                // the bunch's fourth Philox word decides, as in the main pass
                const uint4 x = philox4x32_10(
                    make_uint4(static_cast<uint32_t>(key >> 32), step_hi, static_cast<uint32_t>(key),
                               0u),
                    p.key0, p.key1);
                const R tau = trans_tau<R>(p, o.lam, o.he);
                R P, u3;
                if constexpr (std::is_same<R, float>::value) {
                    P = __expf(-(tau / co));
                    u3 = u01f(x.w);
                } else {
                    P = exp(-(tau / co));
                    u3 = u01d(x.w);
                }
                if (!(u3 < P)) {
                    o.status = ST_ABSORBED;
                    ++st_absorb;
                }
            }
        }
        int s0 = 0, gsel = 0;
        unsigned hm = live ? sphere_hits<R>(p, c, o, s0, gsel) : 0u;
        const R np1 = DS ? R(1) + o.kap * c.eta_o : np1o;
        const R lam_o = o.lam, t_o = o.t;
        record_hits<R>(p, o, hm, s0, gsel,
                       [w, key, lam_o, t_o](R &w_, uint64_t &k_, R &l_, R &t_) {
                           w_ = w;
                           k_ = key;
                           l_ = lam_o;
                           t_ = t_o;
                       },
                       np1, lane, st_hits, st_over);
    }
    unsigned long long *S = p.stats;
    if (S) {
        // the main pass counted the queued bunches as reaching the ground
        flush_stat(S, CHER_STAT_FALLBACK, st_fb);
        flush_stat(S, CHER_STAT_ABSORBED, st_absorb);
        flush_stat_signed(S, CHER_STAT_GROUND, -static_cast<int>(st_absorb));
        flush_stat(S, CHER_STAT_HITS, st_hits);
        flush_stat(S, CHER_STAT_OVERFLOW, st_over);
        if (blockIdx.x == 0 && threadIdx.x == 0 && queued > cap) {
            atomicAdd(S + CHER_STAT_FB_LOST, queued - cap);
            atomicAdd(S + CHER_STAT_GROUND, ~(queued - cap) + 1ull);     // minus the lost
        }
    }
}

// The trace arrays as a bunch that nothing traces leaves them: zeros, status
// -1.  One pass of stores over 44 bytes (FP32) a bunch instead of a launch for
// each of the five arrays, which the host could not issue as fast as they ran
// (yields and trace of 3e4 steps: 223 -> 199 us from call to result).  Array by
// array in 16-byte stores by as many CTAs as there are 1024 bunches: bound by the
// stores (3.2e7 bunches, FP32, 1.43 GB: 187 us; five fills 190, 1216 CTAs walking
// over all of it 213).
__device__ __forceinline__ void fill_words(void *base, int64_t bytes, int v, int64_t at,
                                           int64_t stride) {
    // (4-byte stores where the array or its end is not 16-byte aligned)
    const int64_t n16 = reinterpret_cast<uintptr_t>(base) % 16 ? 0 : bytes / 16;
    for (int64_t k = at; k < n16; k += stride) static_cast<int4 *>(base)[k] = make_int4(v, v, v, v);
    for (int64_t k = 4 * n16 + at; k < bytes / 4; k += stride) static_cast<int *>(base)[k] = v;
}

template <class R>
__global__ void __launch_bounds__(256) k_clear_trace(const cher_trace t) {
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    const int64_t at = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    fill_words(t.pos, t.n_bunches * 4 * static_cast<int64_t>(sizeof(R)), 0, at, stride);
    fill_words(t.tim, t.n_bunches * 4 * static_cast<int64_t>(sizeof(R)), 0, at, stride);
    fill_words(t.status, t.n_bunches * 4, -1, at, stride);
    fill_words(t.nhit, t.n_bunches * 4, 0, at, stride);
    fill_words(t.first_hit, t.n_bunches * 4, 0, at, stride);
}

template <class R, int BLOCK>
size_t smem_bytes(const KParams &p) {
    size_t b = segd_offset<R, BLOCK>();
    if (p.disp_k > 0) b += sizeof(SegD<R>) * BLOCK;
    // every launch reserves the crossing queue (the hits kernels use it;
    // 2 KB per 128 threads)
    b += sizeof(uint2) * kRing * (BLOCK / 32);
    return b;
}

template <class R, int BLOCK, int MODE, bool DS, bool CV>
const void *kernel_ptr_ds(bool tr, bool fb) {
    if constexpr (MODE == MODE_YIELD) {
        return reinterpret_cast<const void *>(&k_gen_prop<R, BLOCK, MODE, false, 0, DS, CV>);
    } else if constexpr (CV) {
        // the curved atmosphere has no beyond-table fallback
        if (fb) return nullptr;
        return tr ? reinterpret_cast<const void *>(&k_gen_prop<R, BLOCK, MODE, true, 0, DS, CV>)
                  : reinterpret_cast<const void *>(&k_gen_prop<R, BLOCK, MODE, false, 0, DS, CV>);
    } else {
        if (fb)
            return tr ? reinterpret_cast<const void *>(&k_gen_prop<R, BLOCK, MODE, true, 2, DS, CV>)
                      : reinterpret_cast<const void *>(&k_gen_prop<R, BLOCK, MODE, false, 2, DS, CV>);
        return tr ? reinterpret_cast<const void *>(&k_gen_prop<R, BLOCK, MODE, true, 0, DS, CV>)
                  : reinterpret_cast<const void *>(&k_gen_prop<R, BLOCK, MODE, false, 0, DS, CV>);
    }
}

// the wavelength-dependent index and the curved atmosphere come in 128-step
// tiles; the hits kernel of flat layers is cher_hits.cu's
template <class R, int BLOCK, int MODE>
const void *kernel_ptr(bool tr, bool fb, bool ds, bool cv) {
    if constexpr (BLOCK == kDispBlock) {
        if (cv)
            return ds ? kernel_ptr_ds<R, BLOCK, MODE, true, true>(tr, fb)
                      : kernel_ptr_ds<R, BLOCK, MODE, false, true>(tr, fb);
        if constexpr (MODE != MODE_HITS)
            if (ds) return kernel_ptr_ds<R, BLOCK, MODE, true, false>(tr, fb);
    }
    if constexpr (MODE != MODE_HITS)
        if (!ds && !cv) return kernel_ptr_ds<R, BLOCK, MODE, false, false>(tr, fb);
    return nullptr;
}

template <class R, int MODE>
const void *pick(int block, bool tr, bool fb, bool ds, bool cv) {
    switch (block) {
    case 128: return kernel_ptr<R, 128, MODE>(tr, fb, ds, cv);
    case 256: return kernel_ptr<R, 256, MODE>(tr, fb, ds, cv);
    case 512: return kernel_ptr<R, 512, MODE>(tr, fb, ds, cv);
    }
    return nullptr;
}

// mode: a Mode, plus kTransBit / kFbBit / kDispBit / kCurvBit for the
// instantiations with the transmission draw / the beyond-table fallback /
// the wavelength-dependent index / the curved atmosphere
const void *pick_kernel(bool fp32, int block, int mode) {
    if (hits_kernel_serves(mode)) return hits_kernel(fp32, mode);
    const bool tr = (mode & kTransBit) != 0;
    const bool fb = (mode & kFbBit) != 0;
    const bool ds = (mode & kDispBit) != 0;
    const bool cv = (mode & kCurvBit) != 0;
    mode &= ~(kTransBit | kFbBit | kDispBit | kCurvBit);
    if (fp32) {
        switch (mode) {
        case MODE_HITS: return pick<float, MODE_HITS>(block, tr, fb, ds, cv);
        case MODE_TRACE: return pick<float, MODE_TRACE>(block, tr, fb, ds, cv);
        case MODE_YIELD: return pick<float, MODE_YIELD>(block, tr, fb, ds, cv);
        }
    } else {
        switch (mode) {
        case MODE_HITS: return pick<double, MODE_HITS>(block, tr, fb, ds, cv);
        case MODE_TRACE: return pick<double, MODE_TRACE>(block, tr, fb, ds, cv);
        case MODE_YIELD: return pick<double, MODE_YIELD>(block, tr, fb, ds, cv);
        }
    }
    return nullptr;
}

}  // namespace

void fill_float_constants(KParams &p) {
    p.f.h_obs = static_cast<float>(p.h_obs);
    p.f.dH_max = static_cast<float>(p.h_max - p.h_obs);
    p.f.eta_o = static_cast<float>(p.eta_obs);
    p.f.inv_np1o = static_cast<float>(1.0 / (1.0 + p.eta_obs));
    p.f.np1o = static_cast<float>(1.0 + p.eta_obs);
    p.f.q_max = static_cast<float>(p.q_max);
    p.f.inv_dht = static_cast<float>(p.inv_dht);
    p.f.inv_dq = static_cast<float>(p.inv_dq);
    p.f.inv_dh = static_cast<float>(p.inv_dh);
    p.f.lam_inv1 = static_cast<float>(p.lam_inv1);
    p.f.lam_dinv = static_cast<float>(p.lam_dinv);
    for (int g = 0; g < 2; ++g) {
        p.f.gx0[g] = static_cast<float>(p.grid[g].x0);
        p.f.gy0[g] = static_cast<float>(p.grid[g].y0);
        p.f.inv_gcs[g] = static_cast<float>(p.grid[g].inv_cs);
    }
    p.f.q_band = static_cast<float>(p.q_band);
    p.f.inv_me = static_cast<float>(p.inv_me);
    p.f.K = static_cast<float>(p.K);
    p.f.inv_B = static_cast<float>(p.inv_B);
    p.f.h_max = static_cast<float>(p.h_max);
    p.f.dh = static_cast<float>(1.0 / p.inv_dh);
    p.f.eta_slope = static_cast<float>(p.eta_slope * 1.01);
    p.f.eta_jump = static_cast<float>(p.eta_jump);
    p.f.rcut2 = static_cast<float>(p.rcut2);
    p.cull.r_cut = static_cast<float>(std::sqrt(p.rcut2) * (1.0 + 1e-6));
    p.f.fb_q = static_cast<float>(p.fb_q);
    p.f.trans_l0 = static_cast<float>(p.trans_l0);
    p.f.trans_lscale = static_cast<float>(p.trans_lscale);
    p.f.trans_h0 = static_cast<float>(p.trans_h0);
    p.f.trans_hscale = static_cast<float>(p.trans_hscale);
    p.f.prof_dx = static_cast<float>(p.prof_dx);
    p.f.prof_inv_dx = static_cast<float>(p.prof_inv_dx);
    for (int m = 0; m < kDispMax; ++m) p.f.kap[m] = static_cast<float>(p.kap[m]);
    p.f.disp_Kd = static_cast<float>(p.disp_Kd);
    p.f.disp_u1 = static_cast<float>(p.disp_u1);
    p.f.disp_du = static_cast<float>(p.disp_du);
    p.f.kap_lo = static_cast<float>(p.kap_lo);
    p.f.kap_winv = static_cast<float>(p.kap_winv);
    for (int l = 0; l < 5; ++l) p.f.eta_coef[l] = static_cast<float>(p.atm.eta_coef[l]);
    p.f.earth_radius = static_cast<float>(p.earth_radius);
    p.f.r_o = static_cast<float>(p.r_o);
    p.f.inv_ro = static_cast<float>(p.inv_ro);
    p.f.inv_dsec = static_cast<float>(p.inv_dsec);
    for (int q = 0; q < 12; ++q) {
        p.f.gl_x[q] = static_cast<float>(p.gl_x[q]);
        p.f.gl_w[q] = static_cast<float>(p.gl_w[q]);
    }
    for (int l = 0; l < 6; ++l) p.f.hb[l] = static_cast<float>(p.atm.hb[l]);
    for (int l = 0; l < 5; ++l) {
        p.f.a[l] = static_cast<float>(p.atm.a[l]);
        p.f.b[l] = static_cast<float>(p.atm.b[l]);
        p.f.c[l] = static_cast<float>(p.atm.c[l]);
        p.f.inv_c[l] = static_cast<float>(p.atm.inv_c[l]);
        p.f.t_top[l] = static_cast<float>(p.atm.t_top[l]);
    }
}

namespace {
__global__ void k_round_to_float(const double *in, float *out, float *lo, int64_t n) {
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n;
         i += int64_t(gridDim.x) * blockDim.x) {
        if (lo)
            d2f_split(in[i], out[i], lo[i]);
        else
            out[i] = d2f_rn(in[i]);
    }
}
}  // namespace

size_t fallback_record_bytes(bool fp32) {
    static_assert(sizeof(FbEntry<float>) == 64 && sizeof(FbEntry<double>) == 112,
                  "fallback queue records");
    return fp32 ? sizeof(FbEntry<float>) : sizeof(FbEntry<double>);
}

template <class R>
void fallback_r(bool tr, bool disp, const KParams &p, int grid, cudaStream_t st) {
    if (disp) {
        if (tr) k_fallback<R, true, true><<<grid, 128, 0, st>>>(p);
        else k_fallback<R, false, true><<<grid, 128, 0, st>>>(p);
    } else {
        if (tr) k_fallback<R, true, false><<<grid, 128, 0, st>>>(p);
        else k_fallback<R, false, false><<<grid, 128, 0, st>>>(p);
    }
}

cudaError_t launch_fallback(bool fp32, bool tr, bool disp, const KParams &p, int num_sms,
                            void *stream) {
    const int grid = num_sms * 8;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (fp32) fallback_r<float>(tr, disp, p, grid, st);
    else fallback_r<double>(tr, disp, p, grid, st);
    return cudaGetLastError();
}

cudaError_t round_to_float(const double *in, float *out, float *lo, int64_t n, int num_sms,
                           void *stream) {
    if (n <= 0) return cudaSuccess;
    const int64_t blocks = std::min<int64_t>((n + 255) / 256, int64_t(num_sms) * 8);
    k_round_to_float<<<static_cast<int>(blocks), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        in, out, lo, n);
    return cudaGetLastError();
}

size_t kernel_smem_bytes(bool fp32, int block, int mode, const KParams &p) {
    if (hits_kernel_serves(mode)) return hits_smem_bytes(fp32, mode, block);
    if (fp32) {
        switch (block) {
        case 128: return smem_bytes<float, 128>(p);
        case 256: return smem_bytes<float, 256>(p);
        case 512: return smem_bytes<float, 512>(p);
        }
    } else {
        switch (block) {
        case 128: return smem_bytes<double, 128>(p);
        case 256: return smem_bytes<double, 256>(p);
        case 512: return smem_bytes<double, 512>(p);
        }
    }
    return 0;
}

cudaError_t kernel_prepare(bool fp32, int block, int mode, size_t smem) {
    const void *k = pick_kernel(fp32, block, mode);
    if (!k) return cudaErrorInvalidValue;
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                static_cast<int>(smem));
}

int kernel_max_ctas_per_sm(bool fp32, int block, int mode, size_t smem) {
    const void *k = pick_kernel(fp32, block, mode);
    int n = 0;
    if (!k || cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, block, smem) != cudaSuccess)
        return 0;
    return n;
}

cudaError_t clear_trace(bool fp32, const cher_trace &t, int num_sms, void *stream) {
    const int grid = static_cast<int>(
        std::min<int64_t>((t.n_bunches + 1023) / 1024, int64_t(num_sms) * 256));
    const cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (fp32) k_clear_trace<float><<<grid, 256, 0, s>>>(t);
    else k_clear_trace<double><<<grid, 256, 0, s>>>(t);
    return cudaGetLastError();
}

cudaError_t kernel_launch(bool fp32, int block, int mode, int grid, size_t smem,
                          const KParams &p, void *stream) {
    const void *k = pick_kernel(fp32, block, mode);
    if (!k) return cudaErrorInvalidValue;
    void *args[] = {const_cast<KParams *>(&p)};
    return cudaLaunchKernel(k, dim3(grid), dim3(block), args, smem,
                            static_cast<cudaStream_t>(stream));
}

}  // namespace cher
