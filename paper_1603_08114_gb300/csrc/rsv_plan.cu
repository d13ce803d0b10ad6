// rsv_plan.cu -- host-side work plan of the trajectory kernels.
//
// A plan fixes the block shape (threads nt, sites per thread j; the window of
// a block is W = nt * j sites) and cuts the series into segments placed in
// bins:
//  - a series that fits a window (and, for a single series, that the cost
//    model keeps whole) is one segment on ceil(T / (32 j)) whole warps; such
//    segments are packed side by side into bins first-fit-decreasing;
//  - a longer series is cut into tiles of `tile` owned sites, each with a
//    halo of K = (force evaluations per trajectory) + 1 sites per side, one
//    tile per bin.
// Segment ids run series by series so that the tiles of one series are
// consecutive (their partial dH are summed in that order).
#include <algorithm>
#include <cstring>
#include <numeric>
#include <vector>

#include "rsv_traj.cuh"

namespace rsv {

namespace {

const int kJ_fp64[] = {1, 2, 4, 8, 16, 28};
const int kJ_mixed[] = {4, 8, 12, 16, 20};
const int kNJ_fp64 = 6, kNJ_mixed = 5;

// mixed: (a, k) float2 + x0 (hi, lo) + p0 per site (+ dtau/m with a mass,
// + the leverage v with leverage), the start state in j rows of
// mixed_row(nt, j) slots each; FP64:
// a' (or y e^{-mu/2}), kc (+ 1/m) per site
size_t smem_for(bool mixed, bool mass, bool lev, int nt, int j)
{
    if (mixed)
        return ((2 + (mass ? 1 : 0) + (lev ? 1 : 0)) * (size_t)mixed_ntp(nt) +
                3 * (size_t)mixed_row(nt, j)) *
               (size_t)j * sizeof(float);
    return (2 + (mass ? 1 : 0)) * (size_t)nt * (size_t)j * sizeof(double);
}

bool valid_j(bool mixed, int j)
{
    const int* js = mixed ? kJ_mixed : kJ_fp64;
    const int n = mixed ? kNJ_mixed : kNJ_fp64;
    for (int i = 0; i < n; ++i)
        if (js[i] == j) return true;
    return false;
}

// Time in us of one round of a trajectory -- the blocks an SM holds at once,
// with `warps` warps of j sites per thread between them, through n_force force
// evaluations -- as fitted to sweeps of every block shape.
//
// FP64 (T = 500 .. 2^18, 10 .. 80 steps): a step is the longer of one warp's own
// latency (0.30 + 0.36 j) and the SM's FP64 pipe, which all its warps share (0.50
// + 0.0625 j per warp); the draws, energies and decision take about 16 + 3 j.
// Off by 10 % at most near the optimum: T = 2000, 50 steps 46 us (87 blocks of
// 128 x 1) against 121 us (4 blocks of 192 x 4, the fewest sites in flight), T =
// 30000, 50 steps 72 us (160 x 2) against 106 us (128 x 4).
//
// Mixed (persistent chains of T = 500 .. 2^20, 10 .. 100 steps, theta sampled): a
// step has a latency that grows with j up to four warps and then with every
// further warp; so has the fixed part.  T = 2000, 50 steps 20.8 us a trajectory
// (5 blocks of 128 x 4) against 33.0 (one block of 544 x 4), T = 30000 21.4
// (74 of 128 x 4) against 33.0, T = 700000, 90 steps 66 (142 of 640 x 8)
// against 72 (256 x 20); at 2^20 sites only the windows of 384 x 20 fit in one
// round of 12 warps (87 us with 78 steps and a mass; 448 x 16: 90, 608 x 12:
// 94).  Below four warps the draws, the sweep and the decision wait for one
// another: T = 2000, 6 force evaluations 13.5 us (5 blocks of 128 x 4) against 19.4
// (19 of 32 x 4) and 17.1 (one of 512 x 4).  T = 500 .. 2^20, 2 .. 60 evaluations:
// the shape taken is 0.8 % off the fastest on average (17 % without that term).
//
// Mixed with leverage (a launch per trajectory; T = 700 .. 2^22, 8 .. 100 steps,
// with and without a mass): a step takes about 1.4 times as long (1.3 with runs
// of 12), and the energies at both ends, per site here, 0.75 j more.  2^20
// sites: 8 steps 608 x 12 52.6 us against 57.7 (352 x 20), 100 steps 139.3 against
// 136.0 (384 x 20); over 72 sizes the shape taken is 1.0 % off the fastest on
// average (1.9 % without the 0.75 j, which took 352 x 20 at 8 steps).
double round_cost(bool mixed, bool lev, int j, double warps, double n_force)
{
    if (!mixed)
        return 16.0 + 3.0 * j + n_force * std::max(0.30 + 0.36 * j, 0.50 + 0.0625 * j * warps);
    const double more = std::max(0.0, warps - 4.0);
    // few warps take the serial phases one after another
    const double alone = lev ? (warps < 2.0 ? 1.5 : 0.0)
                         : warps < 2.0 ? 4.0 : warps < 3.0 ? 1.5 : warps < 4.0 ? 0.6 : 0.0;
    double step, fixed;
    switch (j) {
        case 4: step = 0.147 + 0.0119 * more, fixed = 13.3 + 0.22 * warps + alone; break;
        case 8: step = 0.21 + 0.0195 * more, fixed = 16.0 + 0.22 * warps; break;
        case 12: step = 0.32 + 0.031 * more, fixed = 20.0 + 0.55 * warps; break;
        case 16: step = 0.305 + 0.045 * more, fixed = 19.9 + 0.7 * warps; break;
        default: step = 0.36 + 0.038 * more, fixed = 19.1 + 0.9 * warps; break;
    }
    if (lev) return fixed + 0.75 * j + n_force * step * (j == 12 ? 1.3 : 1.4);
    return fixed + n_force * step;
}

// Time in us of a trajectory of a mixed batch: `bins` bins on blocks of W warps of
// 20 sites per thread, `bps` blocks to an SM, in rounds of all the blocks that fit
// and a last one of what is left, as fitted to sweeps of every block size (20 ..
// 6000 series of 10 .. 7600 sites, 4 .. 50 steps).  k blocks on an SM put k ceil(W /
// 4) warps on its fullest scheduler, which paces a step; blocks beside one another
// hide each other's serial phases.  4000 series of 300 .. 640, 50 steps: 128 x 20
// 142 us, 384 x 20 196, 32 x 20 217 (many one-warp blocks, each in a phase of its
// own, are slow: blocks below four warps only where every SM has one).  The shape
// taken is 0.8 % off the fastest on average and 1.4 % with leverage, whose blocks
// hide less, and at most 1.4 % slower than 384 x 20 (by the model of one block's
// warps 9 % and 13 % off, and up to 53 % slower than 384 x 20).
double batch_cost(bool lev, int W, int64_t bins, int64_t bps, int num_sms, double n_force)
{
    auto round = [&](int64_t k) {
        const double s = (double)(k * ((W + 3) / 4)), more = (double)(k - 1);
        return lev ? 26.7 + 2.4 * s - 0.5 * more + n_force * (0.273 + 0.232 * s + 0.05 * more)
                   : 19.6 + 2.7 * s - 2.3 * more + n_force * (0.202 + 0.174 * s - 0.109 * more);
    };
    const int64_t full = bins / (bps * num_sms), rest = bins % (bps * num_sms);
    return full * round(bps) + (rest ? round((rest + num_sms - 1) / num_sms) : 0.0);
}

// Bins that whole series of cnt[w] x w warps need at NW warps a bin, larger
// ones first, each into the fullest bin with room (an estimate of the packing
// below, which takes the first such bin).
int64_t packed_bins(const std::vector<int64_t>& cnt, int NW)
{
    std::vector<int64_t> room(NW + 1, 0);  // bins by the warps they have left
    int64_t bins = 0;
    for (int w = NW; w >= 1; --w) {
        int64_t left = cnt[w];
        for (int r = w; r <= NW && left > 0; ++r) {
            while (room[r] > 0 && left > 0) {
                const int64_t per = r / w, use = std::min(room[r], (left + per - 1) / per);
                const int64_t put = std::min(left, use * per);
                const int64_t full = put / per, rest = put % per;
                room[r] -= full + (rest ? 1 : 0);
                room[r - per * w] += full;
                if (rest) room[r - rest * w] += 1;
                left -= put;
            }
        }
        const int64_t per = NW / w, full = left / per, rest = left % per;
        bins += full + (rest ? 1 : 0);
        room[NW - per * w] += full;
        if (rest) room[NW - rest * w] += 1;
    }
    return bins;
}

int ntmax(bool mixed, bool mass, int j) { return mixed ? mixed_max_threads(j, mass) : 256; }

}  // namespace

void free_plan(Plan& p)
{
    if (p.d_segs) cudaFree(p.d_segs);
    if (p.d_bin_first) cudaFree(p.d_bin_first);
    if (p.d_bin_seg) cudaFree(p.d_bin_seg);
    if (p.d_ser) cudaFree(p.d_ser);
    p = Plan();
}

bool make_plan(const int64_t* off, int n, int n_md, int integrator, double lambda, bool mixed,
               bool mass, bool lev, int num_sms, int sched_nt, int sched_j, int64_t sched_tile,
               Plan& P, const char** why, bool chain)
{
    // one site of staleness per force evaluation
    const int64_t K = (int64_t)n_md * make_scheme(integrator, lambda).nk + 1;
    const size_t smem_cap = 227 * 1024;
    if (n < 1) {
        *why = "no series";
        return false;
    }
    int64_t Tmax = 0;
    for (int s = 0; s < n; ++s) {
        const int64_t T = off[s + 1] - off[s];
        if (T < 1) {
            *why = "every series needs T >= 1";
            return false;
        }
        Tmax = std::max(Tmax, T);
    }

    // ---- block shape and tile ----------------------------------------------
    int nt = 0, j = 0;
    int64_t tile = 0;
    if (sched_nt > 0) {
        // a single series no longer than the tile is kept whole: it needs the
        // window only, no halo
        const bool whole1 = n == 1 && sched_tile >= Tmax && Tmax <= (int64_t)sched_nt * sched_j;
        if (!valid_j(mixed, sched_j) || sched_nt % 32 || sched_nt > ntmax(mixed, mass, sched_j) ||
            sched_tile < 1 || (!whole1 && sched_tile + 2 * K + 3 > (int64_t)sched_nt * sched_j) ||
            smem_for(mixed, mass, lev, sched_nt, sched_j) > smem_cap) {
            *why = "the fixed schedule does not fit this call";
            return false;
        }
        nt = sched_nt;
        j = sched_j;
        tile = sched_tile;
    } else if (n == 1) {
        // one series: fewest waves of the smallest windows (latency per
        // trajectory ~ sites per thread), whole if one window holds it
        const int64_t T = Tmax;
        double best = 1e300;
        const int* js = mixed ? kJ_mixed : kJ_fp64;
        const int nj = mixed ? kNJ_mixed : kNJ_fp64;
        for (int ji = 0; ji < nj; ++ji) {
            const int tmax = ntmax(mixed, mass, js[ji]);
            for (int t = 32; t <= tmax; t += 32) {
                const int64_t cap = (int64_t)t * js[ji];
                if (smem_for(mixed, mass, lev, t, js[ji]) > smem_cap) continue;
                const int64_t tl = cap - 2 * K - 3;
                int64_t bins;
                int64_t use_tile;
                if (T <= cap) {
                    bins = 1;
                    use_tile = T;
                } else {
                    if (tl < 1) continue;
                    bins = (T + tl - 1) / tl;
                    use_tile = tl;
                }
                // also consider splitting a series that would fit
                for (int pass = 0; pass < 2; ++pass) {
                    int64_t b = bins, ut = use_tile;
                    if (pass == 1) {
                        if (T <= cap && tl >= 1 && tl < T) {
                            b = (T + tl - 1) / tl;
                            ut = tl;
                        } else {
                            continue;
                        }
                    }
                    // blocks resident per SM share it: an SM's work per wave
                    // is bps windows
                    int bps = blocks_per_sm(mixed, mass, lev, js[ji], t,
                                            smem_for(mixed, mass, lev, t, js[ji]));
                    if (bps < 1) continue;
                    const int64_t waves = (b + (int64_t)num_sms * bps - 1) / ((int64_t)num_sms * bps);
                    double cost = (double)waves * (double)cap * bps;
                    if (!mixed) {
                        const int64_t per = std::min<int64_t>(bps, (b + num_sms - 1) / num_sms);
                        cost = (double)((b + per * num_sms - 1) / (per * num_sms)) *
                               round_cost(false, lev, js[ji], (double)per * (t / 32), (double)(K - 1)) *
                               (1.0 + 1e-6 * b);
                    } else if (chain) {
                        // one block per SM; a round more of a chain without
                        // leverage is a launch more
                        const int64_t w = (b + num_sms - 1) / num_sms;
                        cost = (double)w * (round_cost(true, lev, js[ji], t / 32, (double)(K - 1)) +
                                            (w > 1 ? 6.0 : 0.0)) + 0.005 * b;
                    }
                    // single trajectories (mixed): measured at T = 2^20, J = 12
                    // with ~600 threads is the fastest, J = 20 close, J = 16 and
                    // 8 slower; a series cut into tiles runs at the throughput
                    // of its blocks, which falls with fewer warps, a whole one
                    // keeps the smallest window (a tie-break toward more threads)
                    if (mixed && !chain) {
                        cost *= js[ji] == 12 ? 1.0 : js[ji] == 20 ? 1.03 : 1.08;
                        cost *= 1.0 + (b > 1 ? 1.0 : 1e-3) * (double)(tmax - t) / tmax;
                    }
                    if (cost < best) {
                        best = cost;
                        nt = t;
                        j = js[ji];
                        tile = ut;
                    }
                }
            }
        }
        if (nt == 0) {
            *why = "n_md too large for an on-chip window";
            return false;
        }
    } else {
        // many series: the shape with the least estimated time, in rounds of the
        // bins an SM holds at once.  Mixed plans keep runs of 20 sites, and the
        // largest block where a series is longer than its window, so that a
        // series' double-float sums are taken in the same order whatever it
        // is packed with; smaller blocks spread few short series over the SMs
        // (10 series of 300 .. 1000 sites, 40 steps: 64 x 20 in 7 blocks 54 us a
        // trajectory, 384 x 20 in 2 78).  FP64, whose sums have no order, takes
        // any run (64 series of 300 .. 2000: 192 x 2 120 us a trajectory, 256 x 28
        // 702).
        double best = 1e300;
        const int big_j = mixed ? 20 : 28, big_t = ntmax(mixed, mass, big_j);
        if ((int64_t)big_t * big_j - 2 * K - 3 < 1) {
            *why = "n_md too large for an on-chip window";
            return false;
        }
        const int only[] = {20};
        const int* js = mixed ? only : kJ_fp64;
        const int nj = mixed ? 1 : kNJ_fp64;
        for (int ji = 0; ji < nj; ++ji) {
            const int tmax = ntmax(mixed, mass, js[ji]);
            for (int t = 32; t <= tmax; t += 32) {
                const int64_t cap = (int64_t)t * js[ji], tl = cap - 2 * K - 3, pw = 32LL * js[ji];
                const size_t sm = smem_for(mixed, mass, lev, t, js[ji]);
                if (sm > smem_cap || (tl < 1 && Tmax > cap)) continue;
                if (mixed && Tmax > cap && t < tmax) continue;
                std::vector<int64_t> cnt(t / 32 + 1, 0);
                int64_t b = 0, segs = 0;
                for (int s = 0; s < n; ++s) {
                    const int64_t T = off[s + 1] - off[s];
                    if (T <= cap) {
                        ++cnt[(T + pw - 1) / pw];
                        ++segs;
                    } else {
                        b += (T + tl - 1) / tl;
                    }
                }
                segs += b;
                // prefer shapes within the segments rsv_reserve grows the
                // partials for (a whole series is one, whatever its length)
                if (segs > reserved_segs(off[n], n)) continue;
                b += packed_bins(cnt, t / 32);
                const int bps = blocks_per_sm(mixed, mass, lev, js[ji], t, sm);
                if (bps < 1) continue;
                const int64_t per = std::min<int64_t>(bps, (b + num_sms - 1) / num_sms);
                if (mixed && t < 128 && b > num_sms) continue;
                const double cost =
                    mixed ? batch_cost(lev, t / 32, b, bps, num_sms, (double)(K - 1))
                          : (double)((b + per * num_sms - 1) / (per * num_sms)) *
                                (round_cost(false, lev, js[ji], (double)per * (t / 32),
                                            (double)(K - 1)) + 6.0);
                if (cost < best) {
                    best = cost;
                    nt = t;
                    j = js[ji];
                    tile = std::max<int64_t>(tl, 1);
                }
            }
        }
        if (nt == 0) {  // tiles of a few sites in every shape: the largest window
            nt = big_t;
            j = big_j;
            tile = (int64_t)big_t * big_j - 2 * K - 3;
        }
    }
    const int64_t cap = (int64_t)nt * j;
    const int NW = nt / 32;
    const int64_t per_warp = 32LL * j;

    // ---- segments --------------------------------------------------------------
    std::vector<Seg> segs;
    std::vector<SerInfo> ser(n);
    for (int s = 0; s < n; ++s) {
        const int64_t T = off[s + 1] - off[s];
        ser[s].off = off[s];
        ser[s].T = T;
        ser[s].seg0 = (int)segs.size();
        const bool whole = (n == 1) ? (tile >= T && T <= cap) : (T <= cap);
        if (whole) {
            Seg g;
            g.lo = 0;
            g.hi = T;
            g.wlo = 0;
            g.whi = T;
            g.series = s;
            g.warp0 = 0;
            g.nwarp = (int)((T + per_warp - 1) / per_warp);
            g.split = 0;
            segs.push_back(g);
            ser[s].nseg = 1;
        } else {
            int cnt = 0;
            for (int64_t lo = 0; lo < T; lo += tile) {
                Seg g;
                g.lo = lo;
                g.hi = std::min(T, lo + tile);
                g.wlo = std::max(lo - K, (int64_t)0) & ~(int64_t)3;
                g.whi = std::min(T, g.hi + K);
                g.series = s;
                g.warp0 = 0;
                g.nwarp = NW;
                g.split = 1;
                if (g.whi - g.wlo > cap) {
                    *why = "internal: tile window exceeds the block";
                    return false;
                }
                segs.push_back(g);
                ++cnt;
            }
            ser[s].nseg = cnt;
        }
    }

    // ---- bins ------------------------------------------------------------------
    std::vector<int> bin_first{0};
    std::vector<int> bin_seg;
    int nsplit = 0;
    for (int s = 0; s < n; ++s) {
        if (ser[s].nseg > 1 || segs[ser[s].seg0].split) {
            ++nsplit;
            for (int k = 0; k < ser[s].nseg; ++k) {
                bin_seg.push_back(ser[s].seg0 + k);
                bin_first.push_back((int)bin_seg.size());
            }
        }
    }
    std::vector<int> whole;
    for (int i = 0; i < (int)segs.size(); ++i)
        if (!segs[i].split) whole.push_back(i);
    std::stable_sort(whole.begin(), whole.end(),
                     [&](int a, int b) { return segs[a].nwarp > segs[b].nwarp; });
    // each into the first bin with room: the bins before k have none for the
    // present size, and never will (rooms only shrink), so the search goes on from k
    std::vector<std::vector<int>> bins;
    std::vector<int> room;
    int k = 0, size = 0;
    for (int id : whole) {
        const int need = segs[id].nwarp;
        if (need != size) {
            size = need;
            k = 0;
        }
        while (k < (int)bins.size() && room[k] < need) ++k;
        if (k == (int)bins.size()) {
            bins.emplace_back();
            room.push_back(NW);
        }
        segs[id].warp0 = NW - room[k];
        room[k] -= need;
        bins[k].push_back(id);
    }
    for (auto& b : bins) {
        for (int id : b) bin_seg.push_back(id);
        bin_first.push_back((int)bin_seg.size());
    }
    const int nbins = (int)bin_first.size() - 1;

    // ---- launch shape ----------------------------------------------------------
    Plan p;
    p.nt = nt;
    p.j = j;
    p.nbins = nbins;
    p.smem = smem_for(mixed, mass, lev, nt, j);
    p.nsegs = (int64_t)segs.size();
    p.nseries = n;
    p.nsplit = nsplit;
    p.total = off[n];
    p.n_md = n_md;
    p.integrator = integrator;
    p.lambda = lambda;
    p.mixed = mixed;
    p.mass = mass;
    p.lev = lev;
    const int bps = blocks_per_sm(mixed, mass, lev, j, nt, p.smem);
    if (bps < 1) {  // a fixed schedule whose block does not fit on an SM
        *why = "the block shape does not fit on one SM (shared memory or registers)";
        return false;
    }
    p.grid = std::min(nbins, num_sms * bps);

    // ---- device copy -----------------------------------------------------------
    cudaError_t e = cudaMalloc(&p.d_segs, sizeof(Seg) * segs.size());
    if (e == cudaSuccess) e = cudaMalloc(&p.d_bin_first, sizeof(int) * bin_first.size());
    if (e == cudaSuccess) e = cudaMalloc(&p.d_bin_seg, sizeof(int) * std::max<size_t>(1, bin_seg.size()));
    if (e == cudaSuccess) e = cudaMalloc(&p.d_ser, sizeof(SerInfo) * ser.size());
    if (e == cudaSuccess)
        e = cudaMemcpy(p.d_segs, segs.data(), sizeof(Seg) * segs.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
        e = cudaMemcpy(p.d_bin_first, bin_first.data(), sizeof(int) * bin_first.size(),
                       cudaMemcpyHostToDevice);
    if (e == cudaSuccess && !bin_seg.empty())
        e = cudaMemcpy(p.d_bin_seg, bin_seg.data(), sizeof(int) * bin_seg.size(),
                       cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
        e = cudaMemcpy(p.d_ser, ser.data(), sizeof(SerInfo) * ser.size(), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        free_plan(p);
        *why = "plan upload failed (out of device memory?)";
        return false;
    }
    P = p;
    return true;
}

}  // namespace rsv
