// Three- and four-step row strips: several time steps per pass over the lattice, with every
// intermediate row in registers.  Included by lbm_kernels.cuh (inside its namespaces).
//
// A warp owns a window of 64 columns (lane: one column pair) and walks down the rows of its range.  In
// one iteration phase 0 collides row y of step t, phase 1 row y - 1 of step t + 1, ..., phase NS - 1 row
// y - NS + 1 of step t + NS - 1, whose streamed populations go to the other lattice.  Between two phases
// a population is needed one row later per unit of c_y, so a ring keeps two rows of the c_y = +1 group
// and one row of the c_y = 0 group (nine pairs, 18 registers per ring; the c_y = -1 group passes straight
// on); the row loop is unrolled by two so that every ring slot is a fixed register.  The shift by c_x is
// a warp shuffle.  No phase touches shared memory and no barrier separates them: warps run on their own.
// A launch moves every population through HBM once per NS steps: NS = 4 with FP32 storage (18 B per
// update), 3 with 16-bit storage (12 B; its stores round, so the steps per launch are part of the result).
//
// Window and halo: a value is right if the columns within one per step are, so after NS collisions and
// the last stream the outer NS columns on each side are not.  The useful columns of a window are those
// of lanes [2, 30); two lanes on each side are halo, computed again by the neighbouring windows.  A row
// of an even number of columns that fits a warp needs no halo: its lanes shuffle in a circle (closed).
// Rows rarely fill whole windows, so the windows of T rows of T samples (at the same height) are laid
// end to end over G warps (StripPacker): 256 columns take 14 warps for three samples where one sample
// alone takes five, 0.857 useful lanes against 0.8.
//
// Work: the rows of the running samples, T samples side by side, are split into equal ranges, one per
// group of G warps.  A piece (range x sample) of L rows runs L + 2 (NS - 1) iterations, so a batch with
// fewer groups of samples than ranges splits each group into equal parts instead: no range then holds
// parts of two (strip_part; 20 x 100^2 FP32: 2.8 us per step, equal ranges 4.1, both before idle lanes
// loaded pairs of their own; 2.6 now).
//
// What bounds it (625 x 256^2 FP32): the register file's read ports and HBM.  A packed FMA of three
// distinct registers takes three cycles (two with a reused or immediate operand, measured), about 600 of
// the 800 cycles a warp's iteration takes; a launch of 0.498 ms moves its 2.95 GB at 0.87 of the copy
// bandwidth.  Kernel GLUPS against the strips with their rings in shared memory, three steps per launch, two
// barriers per row: 329 / 243 (125 against 168 us per step); 128^2 322 / 242, 512^2 329 / 202, 1024^2 325 / 206,
// 255^2 277 / 210, 200^2 303 / 166; BF16 at 256^2 294 / 235, FP16 280 / 231, FX16 232 / 217 (bound by its
// conversions).
#pragma once

// Number of phases (time steps) per launch.
template <typename S>
constexpr int kStripSteps = sizeof(S) == 4 ? kStripStepsF32 : 3;
constexpr int kStripThreads = 128;
constexpr int kStripWarps = kStripThreads / 32;

// Rows in flight ahead of the one in use when rows are staged in shared memory, and the slots they
// rotate through: a row is copied into the slot that was read one iteration before.
constexpr int kStripDepth = 3, kStripSlots = kStripDepth + 1;

// Default staging of the phase-0 rows (the kernel's D) and the blocks of 128 threads per SM that the
// register budget is sized for.  Measured at 625 x 256^2 (kernel GLUPS): FP32 staged in shared memory 1 / 2
// / 3 rows ahead 271 / 305 / 311 at 3 blocks, 258 at 4 (spills), in registers 271, not staged 224; BF16 292
// at 3 blocks, 287 at 4, 272 in registers; FX16 225 in registers at 4 blocks, 216 staged at 3.
template <typename S, bool ODD>
constexpr int kStripDefaultD = std::is_same<S, int16_t>::value && !ODD ? 2 : 1;
template <typename S, int D, bool ODD>
constexpr int kStripMinBlocks = sizeof(S) == 2 && D == 2 ? 4 : 3;

// Widest rows (columns) of the scheme.
template <typename S>
constexpr int kStripMaxNx = sizeof(S) == 4 ? 1280 : 1600;

__device__ __forceinline__ f2 shift_from_left(f2 v, int left) {
    float a, b;
    upk(v, a, b);
    return pk(__shfl_sync(0xffffffffu, b, left), a);
}
__device__ __forceinline__ f2 shift_from_right(f2 v, int right) {
    float a, b;
    upk(v, a, b);
    return pk(b, __shfl_sync(0xffffffffu, a, right));
}

// One piece (the rows ya .. yb - 1 of one sample per lane) as this lane sees it.
template <typename S>
struct StripPiece {
    const S* src;   // the lane's first column in the lattice that holds the state
    S* dst;         // the same column in the other lattice
    int pitch, plane, ny, ya, yb;
    int xa, xb;     // the lane's columns
    int left, right;  // lanes of the neighbouring pairs
    bool use_b;     // column xb belongs to the pair (not past an odd width)
    uint32_t sid;
    PackedBGK om;
    typename Storage<S>::Q qz;
};

// Runs the piece for n steps; lanes with `put` write their columns.  REC: red[k] takes this lane's sum
// of u.u at step t + k where k is a recorded step.
template <typename S, int D, bool ODD, bool REC>
__device__ __forceinline__ void strip_piece(const KParams& p, const StripPiece<S>& c, PairRaw<S>* const stage, const int t,
                                            const int n, const bool put, double (&red)[kStripSteps<S>]) {
    constexpr int NS = kStripSteps<S>;
    constexpr unsigned kAll = 0xffffffffu;
    using Raw = PairRaw<S>;
    const bool sr = sizeof(S) == 2 && p.stochastic != 0;
    const int pitch = c.pitch, plane = c.plane, ny = c.ny, ya = c.ya, yb = c.yb, xa = c.xa, xb = c.xb;
    const int left = c.left, right = c.right;
    const bool use_b = c.use_b;
    const uint32_t sid = c.sid;
    const PackedBGK om = c.om;
    const typename Storage<S>::Q qz = c.qz;
    const S* const src = c.src;
    S* const dst = c.dst;
    bool want[NS];
#pragma unroll
    for (int k = 0; k < NS; ++k) want[k] = REC && k < n && ((t + k) % p.qoi_every) == 0;
    const int L = yb - ya, total = L + 2 * (n - 1);
    int yl = (ya - (n - 1)) % ny;
    yl += yl < 0 ? ny : 0;
    // a row of odd width closes on itself between an even and an odd column, so a pair beyond its ends
    // is not aligned (or not adjacent): two copies
    const bool whole = !ODD || ((xa & 1) == 0 && xb == xa + 1);
    const bool all_whole = !ODD || __all_sync(kAll, whole);
    constexpr int kSecond = kStripWarps * kStripSlots * 9 * 32;
    const uint32_t halves = whole ? 0x3210u : ((xa & 1 ? 0x32u : 0x10u) | (xb & 1 ? 0x7600u : 0x5400u));
    Raw pre[9];
    int ahead = total;  // rows still to be fetched
    int put_at = 0, get_at = 0;  // D == 1: slot of the next row to fetch and to use
    auto next_slot = [](int s) { return s == kStripDepth * (9 * 32) ? 0 : s + 9 * 32; };
    auto fetch = [&]() {
        const S* s0 = src + yl * pitch;
        if constexpr (D == 1) {
            if (ahead > 0) {
                if (all_whole) {
#pragma unroll
                    for (int i = 0; i < 9; ++i) cp_async<2 * sizeof(S)>(stage + put_at + i * 32, s0 + i * plane);
                } else if constexpr (sizeof(S) == 4) {
#pragma unroll
                    for (int i = 0; i < 9; ++i) {
                        S* at = reinterpret_cast<S*>(stage + put_at + i * 32);
                        cp_async<4>(at, s0 + i * plane);
                        cp_async<4>(at + 1, s0 + i * plane + (xb - xa));
                    }
                } else {
                    // the two words that hold the columns, in two sets of slots
#pragma unroll
                    for (int i = 0; i < 9; ++i) {
                        cp_async<4>(stage + put_at + i * 32, s0 + i * plane - (xa & 1));
                        cp_async<4>(stage + kSecond + put_at + i * 32, s0 + i * plane + ((xb & ~1) - xa));
                    }
                }
            }
            cp_async_commit();
            put_at = next_slot(put_at);
            --ahead;
        } else {
#pragma unroll
            for (int i = 0; i < 9; ++i) pre[i] = __ldg(reinterpret_cast<const Raw*>(s0 + i * plane));
        }
        yl = yl + 1 == ny ? 0 : yl + 1;
    };
    // destination rows of the row being finished: y - 1, y, y + 1
    int yp = ya + 1 == ny ? 0 : ya + 1;
    int om_ = (ya == 0 ? ny - 1 : ya - 1) * pitch, oz = ya * pitch, op = yp * pitch;
    auto push = [&](const f2(&g)[9], int y) {
        if constexpr (sizeof(S) == 4) {
            f2 v[9];
#pragma unroll
            for (int i = 0; i < 9; ++i)
                v[i] = cx(i) == 0 ? g[i] : (cx(i) > 0 ? shift_from_left(g[i], left) : shift_from_right(g[i], right));
            if (put) {
#pragma unroll
                for (int i = 0; i < 9; ++i) {
                    S* d = dst + ((cy(i) > 0 ? op : (cy(i) < 0 ? om_ : oz)) + i * plane);
                    *reinterpret_cast<f2*>(d) = v[i];  // past an odd width: the row's padding
                }
            }
        } else {
            // one hash per pair (even column and the next) and step gives the random bits; in a row of
            // odd width the pairs beyond its ends straddle two pairs of the row
            const uint32_t salt = (uint32_t)(t + n - 1) * 0x85EBCA77u + sid * 0xC2B2AE3Du;
            uint32_t h = 0u, hb = 0u;
            if (sr) {
                h = mix32((uint32_t)(y * pitch + (xa & ~1)) * 0x9E3779B1u + salt);
                if (ODD && !all_whole) hb = mix32((uint32_t)(y * pitch + (xb & ~1)) * 0x9E3779B1u + salt);
            }
            uint32_t v[9];
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                uint32_t w;
                if (sr) {
                    uint32_t bits = sr_bits(h, i);
                    if (ODD && !all_whole) bits = __byte_perm(bits, sr_bits(hb, i), halves);
                    w = pair_word_sr<S>(g[i], bits, qz, i);
                } else {
                    w = pair_word<S>(g[i], qz, i);
                }
                if (cx(i) > 0)
                    w = __byte_perm(__shfl_sync(kAll, w, left), w, 0x5432);
                else if (cx(i) < 0)
                    w = __byte_perm(w, __shfl_sync(kAll, w, right), 0x5432);
                v[i] = w;
            }
            if (put) {
#pragma unroll
                for (int i = 0; i < 9; ++i) {
                    S* d = dst + ((cy(i) > 0 ? op : (cy(i) < 0 ? om_ : oz)) + i * plane);
                    *reinterpret_cast<uint32_t*>(d) = v[i];
                }
            }
        }
        om_ = oz;
        oz = op;
        yp = yp + 1 == ny ? 0 : yp + 1;
        op = yp * pitch;
    };
    // rings between the phases: P two rows of populations 2, 5, 6 (slot: parity of the
    // iteration), Z one row of populations 0, 1, 3
    f2 P[NS - 1][2][3], Z[NS - 1][3];
#pragma unroll
    for (int k = 0; k < NS - 1; ++k)
#pragma unroll
        for (int q = 0; q < 3; ++q) P[k][0][q] = P[k][1][q] = Z[k][q] = 0ull;
    // SLOW: the first iterations, whose later phases have no input yet, the last launches
    // with fewer steps, and launches that record K
    auto iterate = [&](auto par_c, auto slow_c, const int it) {
        constexpr int PAR = decltype(par_c)::value;
        constexpr bool SLOW = decltype(slow_c)::value;
        f2 g[9];
        if constexpr (D == 0) fetch();
        if constexpr (D == 1) {
            cp_async_wait<kStripDepth - 1>();
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                Raw w = stage[get_at + i * 32];
                if constexpr (ODD && sizeof(S) == 2)
                    if (!all_whole) w = __byte_perm(w, stage[kSecond + get_at + i * 32], halves);
                g[i] = pair_from_raw<S>(w, qz, i);
            }
            get_at = next_slot(get_at);
            fetch();
        } else {
#pragma unroll
            for (int i = 0; i < 9; ++i) g[i] = pair_from_raw<S>(pre[i], qz, i);
        }
        if constexpr (D == 2) {
            if (it + 1 < total) fetch();
        }
        auto collide = [&](f2(&h)[9], int k) {
            if constexpr (REC) {
                const int row = it - k - (n - 1);
                // one branch for the warp: on `put` as well, halo and useful lanes would collide one after
                // the other.  Odd widths form u.u in every phase, whose one copy of the collision leaves
                // the other rows' code better off (128 x 127^2 with a series every 100 steps 11.81 against
                // 11.92 us per step; 625 x 256^2 130.3 against 127.8)
                f2 q;
                const bool sum = want[k] && row >= 0 && row < L;
                if (ODD || sum)
                    collide_packed(h, om, &q);
                else
                    collide_packed(h, om, nullptr);
                if (sum && put) {
                    float a, b;
                    upk(q, a, b);
                    red[k] += (double)a + (use_b ? (double)b : 0.0);
                }
            } else {
                // FP32: the last two phases in scalar instructions (the same bits), which balances the
                // register ports against the issue slots: 516 us per launch at 625 x 256^2, all packed
                // 527, all scalar 529 (an earlier build; 498 now); 16-bit storage all packed 421, all
                // scalar 449
                if (sizeof(S) == 4 && k >= 2)
                    collide_halves(h, om);
                else
                    collide_packed(h, om, nullptr);
            }
        };
        collide(g, 0);
#pragma unroll
        for (int k = 1; k < NS; ++k) {
            if (SLOW && k == n) break;
            f2 h[9];
            h[0] = Z[k - 1][0];
            h[1] = shift_from_left(Z[k - 1][1], left);
            h[3] = shift_from_right(Z[k - 1][2], right);
            h[2] = P[k - 1][PAR][0];
            h[5] = shift_from_left(P[k - 1][PAR][1], left);
            h[6] = shift_from_right(P[k - 1][PAR][2], right);
            h[4] = g[4];
            h[7] = shift_from_right(g[7], right);
            h[8] = shift_from_left(g[8], left);
            Z[k - 1][0] = g[0];
            Z[k - 1][1] = g[1];
            Z[k - 1][2] = g[3];
            P[k - 1][PAR][0] = g[2];
            P[k - 1][PAR][1] = g[5];
            P[k - 1][PAR][2] = g[6];
            if (SLOW && it < 2 * k) return;
            collide(h, k);
#pragma unroll
            for (int i = 0; i < 9; ++i) g[i] = h[i];
        }
        push(g, ya + it - 2 * (n - 1));
    };
    const std::integral_constant<int, 0> even{};
    const std::integral_constant<int, 1> odd{};
    const std::true_type slow{};
    const std::false_type fast{};
    if constexpr (D == 1)
        for (int k = 0; k < kStripDepth; ++k) fetch();
    if constexpr (D == 2) fetch();
    const int lead = n < NS || REC ? total : 2 * (NS - 1);
    int it = 0;
    for (; it < lead; it += 2) {
        iterate(even, slow, it);
        if (it + 1 < total) iterate(odd, slow, it + 1);
    }
    if constexpr (!REC) {
        for (; it < total; it += 2) {
            iterate(even, fast, it);
            if (it + 1 < total) iterate(odd, fast, it + 1);
        }
    }
}

// Sums of NS <= 4 values over the warp, value k in the lanes 8 k of the result: at the first two levels a lane
// keeps half of the values and sends the others (6 FP64 adds instead of 5 NS, whose units all warps share),
// in the order of one butterfly per value.
template <int NS>
__device__ __forceinline__ double strip_warp_sums(const double (&v)[NS], int lane) {
    static_assert(NS == 3 || NS == 4, "two levels of halves");
    const bool hi = (lane & 16) != 0, odd = (lane & 8) != 0;
    const double v3 = NS == 4 ? v[NS - 1] : 0.0;
    const double a = (hi ? v[2] : v[0]) + __shfl_xor_sync(0xffffffffu, hi ? v[0] : v[2], 16);
    const double b = (hi ? v3 : v[1]) + __shfl_xor_sync(0xffffffffu, hi ? v[1] : v3, 16);
    double r = (odd ? b : a) + __shfl_xor_sync(0xffffffffu, odd ? a : b, 8);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
    return r;
}

// Sum over the warp of n slots of one sample: `nw` consecutive warps of every piece, G T NS apart.  Eight
// slots of a lane are in flight at once.  Not inlined: its registers are its own, not the row loop's.
template <int NS>
__device__ __noinline__ double strip_slots_sum(const double* slots, int n, int nw, int G, int T) {
    constexpr int kAhead = 8;
    const int lane = threadIdx.x & 31;
    double acc[NS];
#pragma unroll
    for (int k = 0; k < NS; ++k) acc[k] = 0.0;
    for (int q0 = lane; q0 < n; q0 += 32 * kAhead) {
        double v[kAhead][NS];
#pragma unroll
        for (int i = 0; i < kAhead; ++i) {
            const int q = q0 + 32 * i, at = q / nw;
            const double* from = slots + ((int64_t)at * G + (q - at * nw)) * T * NS;
#pragma unroll
            for (int k = 0; k < NS; ++k) v[i][k] = q < n ? __ldcg(from + k) : 0.0;
        }
#pragma unroll
        for (int i = 0; i < kAhead; ++i)
#pragma unroll
            for (int k = 0; k < NS; ++k) acc[k] += v[i][k];
    }
    return strip_warp_sums<NS>(acc, lane);
}

// What the sums of a piece need besides the kernel's parameters.
struct StripSums {
    const SampleDev* samples;
    double *kpart, *series;
    int32_t* counters;
    int64_t qoi_every, series_ld;
    int spl, t, nact, T, G, slot, task, m, ny, rb, ya, yb, per, parts, group;
};

// K: the warp's sum of each of its tasks into the slot of (range, warp, sample); the last warp of a sample to
// finish sums its slots in a fixed order.  The warp's tasks share one fence, which waits for the rows' stores
// too, and count in parallel, a lane each.  Three 256 x 256 samples with the energy of every step, us per
// step: FP32 6.9, FX16 8.3 (2.7 and 3.4 without); with a fence, a count and a butterfly per value for each
// task, one slot after the other and halo lanes that collided apart from the others 13.4 and 20.0.
template <int NS>
__device__ __forceinline__ void strip_record(const StripSums& a, const StripMap& map, const double (&red)[NS]) {
    constexpr unsigned kAll = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    // Lane c looks after task c.  A sample is summed if one of its own steps of this launch is a recorded one:
    // every warp that holds it has to come to the same answer (its counter waits for all of them),
    // whatever other samples the warp holds.
    const int64_t wait = (a.qoi_every - a.t % a.qoi_every) % a.qoi_every;  // steps from t to the next recorded one
    const int mine = a.m * a.T + lane;
    int w0 = 0, nw = 0;  // the group's warps that hold columns of the task
    if (lane < a.T && mine < a.nact && wait < min(a.spl, a.samples[mine].steps - a.t)) {
        nw = map.closed ? 1 : map.warps_of[lane];
        w0 = map.closed ? 0 : map.first_warp[lane];
    }
    const unsigned held = __ballot_sync(kAll, a.slot >= w0 && a.slot < w0 + nw);
    // pieces are numbered along the ranges: a piece is one range's part of one group of samples
    const int piece = a.parts > 0 ? a.group : a.m + a.group;
    for (unsigned left = held; left != 0; left &= left - 1) {
        const int c = __ffs(left) - 1;
        double part[NS];
#pragma unroll
        for (int k = 0; k < NS; ++k) part[k] = a.task == c ? red[k] : 0.0;
        const double sum = strip_warp_sums<NS>(part, lane);
        if ((lane & 7) == 0 && lane / 8 < NS)
            a.kpart[(((int64_t)piece * a.G + a.slot) * a.T + c) * NS + lane / 8] = sum;
    }
    __threadfence();
    __syncwarp();
    bool last = false;
    if ((held >> lane) & 1) last = atomicAdd(a.counters + mine, a.yb - a.ya) + (a.yb - a.ya) == a.ny * nw;
    const unsigned done = __ballot_sync(kAll, last);
    if (done == 0) return;
    __threadfence();
    const int first = a.parts > 0 ? a.m * a.parts : a.m + a.rb / a.per;
    const int pieces = a.parts > 0 ? a.parts : (a.rb + a.ny - 1) / a.per - a.rb / a.per + 1;
    for (unsigned left = done; left != 0; left &= left - 1) {
        const int c = __ffs(left) - 1, jc = a.m * a.T + c;
        const int cw0 = __shfl_sync(kAll, w0, c), cnw = __shfl_sync(kAll, nw, c);
        const double* slots = a.kpart + (((int64_t)first * a.G + cw0) * a.T + c) * NS;
        const double total = strip_slots_sum<NS>(slots, pieces * cnw, cnw, a.G, a.T);
        const SampleDev* sc = a.samples + jc;
        const int k = lane / 8;
        if ((lane & 7) == 0 && k < min(a.spl, sc->steps - a.t) && (a.t + k) % a.qoi_every == 0)
            a.series[(int64_t)sc->sample_id * a.series_ld + (a.t + k) / a.qoi_every] = total * sc->u_ref_inv2;
        if (lane == 0) a.counters[jc] = 0;
    }
}

// W: compile-time width (0: map.nx; 256 columns 564 instead of 527 us per launch).  D: the phase-0 row is
// loaded when it is used (0), kStripDepth rows ahead into shared memory by cp.async (1) or one row ahead
// into registers (2).  ODD: odd widths.  SERIES: launches of runs that record K at some step; the others' kernel
// holds no second copy of the rows' code with its sums (625 x 256^2 124.9 against 125.7 us per step, 1 x 128^2 1.52
// / 1.69, FX16 128 x 256^2 38.2 / 39.5).
template <typename S, int W, int D, bool ODD, bool SERIES>
__global__ void __launch_bounds__(kStripThreads, kStripMinBlocks<S, D, ODD>) strip_regs_kernel(KParams p, const __grid_constant__ StripMap map) {
    static_assert(!ODD || D == 1, "unaligned pairs are put together in shared memory");
    constexpr int NS = kStripSteps<S>;
    constexpr unsigned kAll = 0xffffffffu;
    using Raw = PairRaw<S>;
    // 16-bit rows of odd width: a second set of slots for the pairs that are not one word
    __shared__ Raw s_stage[D == 1 ? (ODD && sizeof(S) == 2 ? 2 : 1) * kStripWarps * kStripSlots * 9 * 32 : 1];
    const int lane = threadIdx.x & 31;
    Raw* const stage = D == 1 ? s_stage + (threadIdx.x >> 5) * (kStripSlots * 9 * 32) + lane : nullptr;
    const int wid = (int)((blockIdx.x * (unsigned)kStripThreads + threadIdx.x) >> 5);
    const int G = map.warps, T = map.samples;
    const int ngroups = (int)(gridDim.x * (unsigned)kStripWarps) / G;
    const int group = wid / G, slot = wid - group * G;
    if (group >= ngroups) return;
    const int nx = W > 0 ? W : map.nx;
    const int U = (nx + 1) >> 1;

    // this lane's sample within the group of T (task), column pair and neighbours.  Idle lanes load pairs of
    // their own too: all on one pair, its copies into their slots came one after the other (1 x 57 x 33: 2.48
    // against 1.93 us per step, 1 x 512^2 3.15 / 2.78, 16 x 97^2 2.97 / 2.76)
    int task = -1, px = lane % U, left = (lane + 31) & 31, right = (lane + 1) & 31;
    bool useful = false;
    if (map.closed) {
        if (lane / U < T) {
            task = lane / U;
            px = lane - task * U;
            left = task * U + (px == 0 ? U - 1 : px - 1);
            right = task * U + (px == U - 1 ? 0 : px + 1);
            useful = true;
        }
    } else {
        for (int q = map.start[slot]; q < map.start[slot + 1]; ++q) {
            const StripStretch s = map.stretch[q];
            const int at = lane - s.lane0;
            if (at >= 0 && at < s.count + 2 * kStripHalo) {
                task = s.task;
                px = s.first + at - kStripHalo;
                useful = at >= kStripHalo && at < s.count + kStripHalo;
            }
        }
    }
    int xa = (2 * px) % nx;
    xa += xa < 0 ? nx : 0;
    const int xb = xa + 1 == nx ? 0 : xa + 1;
    const bool use_b = !ODD || 2 * px + 1 < nx;

    const int t = (int)p.step_counter[0] + p.dt;
    const int t0 = (int)p.step_counter[1];
    // the table is ordered by descending steps, so mostly either all samples still run or none
    const int nact = p.steps_sorted[p.nsamples - 1] > t ? p.nsamples : active_samples(p, t);
    const int nsup = (nact + T - 1) / T;
    const int rows = map.ny > 0 ? nsup * map.ny : p.row_base[nact];
    // ranges: equal shares of all rows, or (small batches) `part` rows of one group of samples, so that no
    // range holds parts of two
    const int parts = map.part > 0 ? (map.ny + map.part - 1) / map.part : 0;
    const int per = parts > 0 ? map.part : (rows + ngroups - 1) / ngroups;
    const int r0 = parts > 0 ? group / parts * map.ny + group % parts * per : group * per;
    const int r1 = parts > 0 ? min(min(rows, r0 + per), (group / parts + 1) * map.ny) : min(rows, r0 + per);

    for (int r = r0; r < r1;) {
        int m, rb, ny;
        if (map.ny > 0) {
            ny = map.ny;
            m = r / ny;
            rb = m * ny;
        } else {
            int lo = 0, hi = nact - 1;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (p.row_base[mid] <= r)
                    lo = mid;
                else
                    hi = mid - 1;
            }
            m = lo;
            rb = p.row_base[m];
            ny = p.row_base[m + 1] - rb;
        }
        const int ya = r - rb, yb = min(ny, r1 - rb);
        r = rb + yb;
        const bool have = task >= 0 && m * T + task < nact;
        const int j = have ? m * T + task : m * T;
        const SampleDev* sp = p.samples + j;
        const int steps = __ldg(&sp->steps);
        const int sslot = __ldg(&sp->slot);
        const float omega = (float)__ldg(&sp->omega);
        const int64_t f_off = __ldg(&sp->f_off);
        const bool second = ((p.sel[sslot] ^ ((t - t0) / p.spl)) & 1) != 0;
        StripPiece<S> pc;
        pc.src = static_cast<const S*>(second ? p.arena2 : p.arena) + f_off + xa;
        pc.dst = static_cast<S*>(second ? p.arena : p.arena2) + f_off + xa;
        pc.pitch = W > 0 ? 9 * W : __ldg(&sp->pitch);
        pc.plane = W > 0 ? W : (int)__ldg(&sp->plane);
        pc.ny = ny;
        pc.ya = ya;
        pc.yb = yb;
        pc.xa = xa;
        pc.xb = xb;
        pc.left = left;
        pc.right = right;
        pc.use_b = use_b;
        pc.sid = (uint32_t)__ldg(&sp->sample_id);
        pc.om = packed_bgk(omega);
        pc.qz = quanta_of<S>(p, j);
        const int n_mine = have ? min(p.spl, steps - t) : 0;

        const int n_max = __reduce_max_sync(kAll, n_mine);
        bool rec = false;
        if (SERIES && p.qoi_every > 0 && p.series != nullptr)
            for (int k = 0; k < n_max; ++k) rec = rec || (t + k) % p.qoi_every == 0;
        double red[NS];
#pragma unroll
        for (int k = 0; k < NS; ++k) red[k] = 0.0;
        // samples of one group may end at different steps of this launch: one pass per step count
        for (int n = n_max; n >= 1; --n) {
            if (!__any_sync(kAll, n_mine == n)) continue;
            const bool put = useful && n_mine == n;
            if (SERIES && rec)
                strip_piece<S, D, ODD, true>(p, pc, stage, t, n, put, red);
            else
                strip_piece<S, D, ODD, false>(p, pc, stage, t, n, put, red);
        }
        if (!SERIES || !rec) continue;
        double sums[NS];
#pragma unroll
        for (int k = 0; k < NS; ++k) sums[k] = red[k];
        const StripSums a{p.samples, p.kpart, p.series, p.counters, p.qoi_every, p.series_ld, p.spl, t, nact, T, G,
                          slot, task, m, ny, rb, ya, yb, per, parts, group};
        strip_record<NS>(a, map, sums);
    }
}
