// sidm_pairs.cu -- (a2, a3) pair interaction probabilities and scatter draws.
//
// For every unordered pair of a halo with d_ij < h_i + h_j (Sect. 3.5: the
// geometric factor Lambda of the interaction probability is the overlap of
// the two spline kernels):
//   P_ij = (sigma(v_ij)/m) m_j v_ij Lambda_ij dt,  v_ij = |v_i - v_j|,
//   sigma/m = s0 or s0 / (1 + (v/w)^2)^2 (Sect. 3.8, Eq. vel_dep),
// and a counter-based Philox4x32-10 draw keyed by (seed; step, min id,
// max id, halo), so the draw is independent of thread order.  Event iff
// u = x0 2^-32 < P (no clamp: P >= 1 always fires).
//
// Each unordered pair is tested once, in the frame of the lower leaf: a query
// leaf A meets the leaves B >= A.  k_pairs draws; k_pairs_all forms every P
// (per-particle sums of P) and the FP64 form's moments.
#include "sidm_internal.cuh"
#include "sidm_tile.cuh"

namespace sidm {
namespace {

struct PairParams {
    int H, L;
    const int32_t* leaf_halo;
    const int32_t* leaf_off;
    const int64_t* halo_off;
    const int32_t* lvl_off;
    const int32_t* top;
    const HaloFrame* frame;
    const float4* cell;
    const float4* nlo;
    const float4* nhi;
    const void* P4;
    const void* S4;     // FP32 offsets (mixed form: P4, with the kernel size)
    const float* reach; // FP64 form: reach in place of the kernel size (k_leaf_hmax)
    const void* V4;
    const uint32_t* ID;
    const void* vel;    // the caller's velocities [3][N] (unchanged until the resolve)
    int64_t N;
    const void* lam;
    const float4* lam4; // the mixed form's table as groups of four along x (forward-dominated halos, k_pairs)
    const sidm_xs* xs;
    const double* dt;
    const double* mass;
    uint32_t seed_lo, seed_hi, step_lo;
    uint32_t rk[20];    // Philox round keys of the seed
    const int32_t* bins;  // individual power-of-two steps (NULL: one step dt[h] for all)
    int n_bins, substep;
    double dt_max;
    sidm_event* ev;
    unsigned long long ev_cap;
    float* sump;
    int use_sump;
    int parts;          // warps that share a query leaf's candidate leaves (a power of two)
    int parts_log;
    // what a warp leaves after kPTiles candidate leaves, (leaf, part | run << 8, first
    // candidate leaf, accepted leaves before it), and the second launch that takes it
    int4* rest;
    int rest_cap;       // 0: a warp leaves nothing
    double* dacc;       // local diagnostics: [5][nacc] kernel-weighted moments
    int64_t nacc;
    DevCounters* cnt;
    sidm_step_stats* st;
    double* evg;        // forward-dominated halos: G = m_j Lambda dt of each record (NULL: none allowed)
    double glx[8], glw[8];  // 8-point Gauss-Legendre rule on [-1, 1] (Lambda by quadrature)
};

// what one traversal of the in-range pairs computes
constexpr int kModeDrawExact = 1;   // draws, every P formed (per-particle sums of P)
constexpr int kModeDiag = 2;        // no draws: kernel-weighted moments for the local diagnostics (FP64 form)

// spline kernel of Sect. 2, support h, normalised to one
template <class R>
__device__ __forceinline__ R spline_w(R d, R h)
{
    const R q = d / h;
    if (!(q < R(1))) return R(0);
    const R norm = R(8.0 / 3.14159265358979323846) / (h * h * h);
    if (q < R(0.5)) return norm * (R(1) - R(6) * q * q * (R(1) - q));
    const R t = R(1) - q;
    return norm * R(2) * t * t * t;
}

// groups of 32 pairs drawn together (a launch knob)
constexpr int kPerRoundMax = 4, kPerRoundDefault = 2;
// moments: pairs a lane queues per round, and the queue entries per warp, a power
// of two: a round adds up to 32 kQueuePerRound pairs to fewer than 32 waiting
constexpr int kQueuePerRound = 4;
constexpr int kQueue = 256;
static_assert(kQueue >= 32 * (kQueuePerRound + 1), "one round must fit behind the entries still waiting");

template <class R>
__device__ __forceinline__ uint32_t id_of(R w)
{
    if constexpr (sizeof(R) == 4) return __float_as_uint((float)w);
    else return (uint32_t)(double)w;
}

// individual power-of-two steps: a particle of bin b (step dt_max / 2^b) opens a
// step at sub-step s of the 2^(n_bins-1) sub-steps of the smallest bin iff s is
// a multiple of 2^(n_bins-1-b)
__device__ __forceinline__ bool step_opens(int b, int n_bins, int s)
{
    return (s & ((1 << (n_bins - 1 - b)) - 1)) == 0;
}

// a length in the halo's FP32 unit, rounded up
template <class R>
__device__ __forceinline__ float to_float_ru_p(R v, double down)
{
    if constexpr (sizeof(R) == 8) return __double2float_ru((double)v * down);
    else return (float)v;
}

// per warp: staging buffers (the bulk-copy path lands a candidate leaf in the
// first; the plain path keeps the query leaf's own points there), the shifted
// candidate leaf, queue of in-range pairs (slot i, slot j), traversal stack,
// boxes of the nodes under test (32 lo + 32 hi)
template <class R>
constexpr size_t pair_warp_bytes()
{
    return (TileStageT<R, false>::bytes() + kQueue * 8 + kStack * 4 + 64 * 16 + 8 * 8 + 15) / 16 * 16;
}

// Every P formed (kModeDrawExact: per-particle sums of P), or the FP64 form's
// moments for the local diagnostics (kModeDiag: no draws; each pair adds
// m W(d, h_i) and its velocity moments of j to particle i when d < h_i, and the
// same for j; the mixed form gathers them per particle, k_knn_warm).  In-range
// pairs are compacted into a per-warp queue of (slot i, slot j) that persists
// across candidate leaves, filled in rounds of ballots.  The sums take one FP32
// addition per pair and particle, in this kernel's order of pairs within a warp
// and in the order of arrival between warps, so their last bits differ from run
// to run.  What would change them for good is left out: the query's terms added
// up per run of its pairs in k_pairs (31.5 ms where this takes 38 of a satellite's
// big step of 2^22 particles; 5e-7 off), and FP64 sums rounded once (89.2 against
// 86.7 ms a big step; 1e-7 to 1e-6 off, the FP32 order's own rounding).  The table
// is read by scalar loads: rows of four (lambda_f_rows) give the same bits and
// 87.4 ms.
template <class R, int MODE, bool DRAG>
__global__ void __launch_bounds__(256, sizeof(R) == 4 ? 4 : 2) k_pairs_all(PairParams p)
{
    constexpr int PR = kQueuePerRound;
    using V = typename Vec4<R>::T;
    using Stage = TileStageT<R, false>;
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned char* base = smem + wid * pair_warp_bytes<R>();
    Stage st_pos(base);
    uint32_t* q_si = (uint32_t*)(base + Stage::bytes());
    uint32_t* q_sj = q_si + kQueue;
    int* stack = (int*)(q_sj + kQueue);
    float4* blo = (float4*)(stack + kStack);
    float4* bhi = blo + 32;
    // the warp's statistics (64-bit, added to once per query leaf, so the
    // per-lane counters of a leaf stay 32-bit registers): pairs, P > 1,
    // |P - u| < 1e-6, tests, Lambda lookups, tiles, most tiles of one leaf
    unsigned long long* wst = (unsigned long long*)(bhi + 32);
    if (lane < 8) wst[lane] = 0ull;
    st_pos.init(lane);
    const R* __restrict__ T = (const R*)p.lam;
    const V* __restrict__ P4 = (const V*)p.P4;
    const V* __restrict__ V4 = (const V*)p.V4;
    const uint32_t lt = (1u << lane) - 1u;


    while (true) {
        int leaf = 0;
        if (lane == 0) leaf = (int)atomicAdd(&p.cnt->work[1], 1u);
        leaf = __shfl_sync(0xffffffffu, leaf, 0);
        if (leaf >= p.L) break;
        const int h = p.leaf_halo[leaf];
        const int leaf0 = p.leaf_off[h];
        const int64_t hb = p.halo_off[h];
        const int64_t nh = p.halo_off[h + 1] - hb;
        const int64_t slot2u = hb - (int64_t)leaf0 * kLeaf;   // padded slot -> particle index
        const int A = leaf - leaf0;
        const int countA = (int)min((int64_t)kLeaf, nh - (int64_t)A * kLeaf);
        // with individual steps only particles whose step opens at this sub-step
        // take part; a leaf without such a particle has no pair to test
        const bool active = lane < countA &&
                            (!p.bins || step_opens(p.bins[hb + (int64_t)A * kLeaf + lane], p.n_bins, p.substep));
        if (p.bins && !__any_sync(0xffffffffu, active)) continue;
        const HaloFrame fr = p.frame[h];
        const float4 cA = p.cell[leaf];
        const sidm_xs xs = p.xs[h];
        const int kind = xs.kind;
        // forward-dominated halo: every in-range pair becomes a record (no draw);
        // only the instantiation for contexts with SIDM_FLAG_DRAG has room for them
        const bool drag = DRAG && MODE != kModeDiag && xs.angular != 0;
        if (!DRAG && MODE != kModeDiag && xs.angular != 0) {
            if (lane == 0) raise_status(p.cnt, SIDM_DEV_BAD_INPUT);
            continue;
        }
        const R pref = p.bins ? R(0) : (R)xs.s0 * (R)p.mass[h] * (R)p.dt[h];
        const R inv_w = kind == 1 ? R(1) / (R)xs.w : R(0);
        const float4 qlo = p.nlo[leaf], qhi = p.nhi[leaf];
        const float hmaxA = qlo.w;
        const uint32_t slotA = (uint32_t)leaf * kLeaf + lane;
        const V q = P4[slotA];
        // the queries in their own frame, for tiles tested candidate by lane (the
        // plain path stages tiles in registers, so the first staging buffer is free)
        V* qsh = st_pos.raw();
        __syncwarp();
        qsh[lane] = q;
        __syncwarp();
        int qhead = 0, qn = 0;
        uint32_t n_pairs = 0u, n_gt1 = 0u, n_near = 0u, n_tested = 0u, n_lam = 0u, n_tiles = 0u;

        // d^2 of a queued pair, recomputed exactly as in the in-range test
        // (candidate shifted into the frame of the query's leaf)
        auto pair_d2 = [&](uint32_t si, uint32_t sj, const V& pi, const V& pj) -> R {
            R cx = pj.x, cy = pj.y, cz = pj.z;
            if constexpr (sizeof(R) == 4) {
                const float4 ci = p.cell[si / kLeaf], cj = p.cell[sj / kLeaf];
                cx = __fadd_rn(cx, __fsub_rn(cj.x, ci.x));
                cy = __fadd_rn(cy, __fsub_rn(cj.y, ci.y));
                cz = __fadd_rn(cz, __fsub_rn(cj.z, ci.z));
            }
            const R dx = sub_rn(cx, pi.x), dy = sub_rn(cy, pi.y), dz = sub_rn(cz, pi.z);
            return fma_rn(dz, dz, fma_rn(dy, dy, mul_rn(dx, dx)));
        };

        // P, draw and event (or the diagnostic moments) for queue entries
        // qhead .. qhead+nb-1, one per lane
        auto run_batch = [&](int nb) {
            __syncwarp();
            if constexpr (MODE == kModeDiag) {
                if (lane < nb) {
                    const int e = (qhead + lane) & (kQueue - 1);
                    const uint32_t si = q_si[e], sj = q_sj[e];
                    const V vi = V4[si], vj = V4[sj];
                    const V pi = P4[si], pj = P4[sj];
                    const R d2 = pair_d2(si, sj, pi, pj);
                    const R d = sqrt_rn(d2);
                    const R mh = (R)p.mass[h];
                    const int64_t ui = slot2u + si, uj = slot2u + sj;
                    if (d2 < mul_rn(pi.w, pi.w)) {
                        const double wt = (double)(mh * spline_w<R>(d, pi.w));
                        atomicAdd(p.dacc + ui, wt);
                        atomicAdd(p.dacc + p.nacc + ui, wt * (double)vj.x);
                        atomicAdd(p.dacc + 2 * p.nacc + ui, wt * (double)vj.y);
                        atomicAdd(p.dacc + 3 * p.nacc + ui, wt * (double)vj.z);
                        atomicAdd(p.dacc + 4 * p.nacc + ui,
                                  wt * ((double)vj.x * vj.x + (double)vj.y * vj.y + (double)vj.z * vj.z));
                    }
                    if (d2 < mul_rn(pj.w, pj.w)) {
                        const double wt = (double)(mh * spline_w<R>(d, pj.w));
                        atomicAdd(p.dacc + uj, wt);
                        atomicAdd(p.dacc + p.nacc + uj, wt * (double)vi.x);
                        atomicAdd(p.dacc + 2 * p.nacc + uj, wt * (double)vi.y);
                        atomicAdd(p.dacc + 3 * p.nacc + uj, wt * (double)vi.z);
                        atomicAdd(p.dacc + 4 * p.nacc + uj,
                                  wt * ((double)vi.x * vi.x + (double)vi.y * vi.y + (double)vi.z * vi.z));
                    }
                }
            } else if (lane < nb) {
                const int e = (qhead + lane) & (kQueue - 1);
                const uint32_t si = q_si[e], sj = q_sj[e];
                const V vi = V4[si], vj = V4[sj];
                const R hi = ((const R*)(P4 + si))[3], hj = ((const R*)(P4 + sj))[3];
                const R ux = vj.x - vi.x, uy = vj.y - vi.y, uz = vj.z - vi.z;
                const R v2 = ux * ux + uy * uy + uz * uz;
                const uint32_t ida = id_of<R>(vi.w), idb = id_of<R>(vj.w);
                const uint32_t a = min(ida, idb), b = max(ida, idb);
                const Philox4 x = philox4x32_10_rk(p.step_lo, a, b, (uint32_t)h, p.rk);
                // individual steps: the pair's longer step dt_max / 2^min(b_i, b_j)
                R prefp = pref;
                int bmin = 0;
                if (p.bins) {
                    bmin = min(p.bins[slot2u + si], p.bins[slot2u + sj]);
                    prefp = (R)xs.s0 * (R)p.mass[h] * (R)ldexp(p.dt_max, -bmin);
                }
                R P, pre, inv, u;
                if constexpr (sizeof(R) == 4) {
                    // P needs ~1e-6 relative accuracy only (the event decision below is
                    // exact for the P computed here): reciprocal square roots and
                    // approximate divisions are enough.
                    const float v = v2 > 0.f ? v2 * rsqrtf(v2) : 0.f;
                    float sig = 1.f;
                    if (kind == 1) { const float qq = v * inv_w; const float tt = 1.f + qq * qq; sig = __fdividef(1.f, tt * tt); }
                    pre = prefp * sig * v;
                    inv = __fdividef(1.f, fmaxf(hi, hj));
                    u = (R)((float)x.x[0] * 0x1p-32f);
                } else {
                    const R v = sqrt(v2);
                    R sig = R(1);
                    if (kind == 1) { const R qq = v * inv_w; const R tt = R(1) + qq * qq; sig = R(1) / (tt * tt); }
                    pre = prefp * sig * v;
                    inv = R(1) / (hi > hj ? hi : hj);
                    u = (R)ldexp((double)x.x[0], -32);
                }
                P = R(0);
                R gfac = R(0);
                bool fire = false;
                {
                    ++n_lam;
                    const R d2 = pair_d2(si, sj, P4[si], P4[sj]);
                    R f;
                    if constexpr (sizeof(R) == 4) {
                        const float d = d2 > 0.f ? d2 * rsqrtf(d2) : 0.f;
                        f = lambda_f_fast(T, d, hi, hj, inv);
                    } else {
                        f = lambda_f<R>(T, sqrt_rn(d2), hi, hj);
                    }
                    P = pre * (f * inv * inv * inv);
                    if (drag) {
                        // the record keeps G = m_j Lambda dt; D = P / 3 at the step start.
                        // The turn's sine is the square root of a multiple of Lambda, so
                        // Lambda must be accurate relative to itself where it falls to
                        // zero, which neither the table nor an FP32 quadrature (its
                        // integrand cancels there) is: FP64 quadrature beyond half the
                        // support (everywhere in the FP64 form), the table inside, where
                        // Lambda > Lambda(0)/4 bounds its relative error
                        R lam = f * inv * inv * inv;
                        const R d2q = pair_d2(si, sj, P4[si], P4[sj]);
                        const R dq = sqrt_rn(d2q);
                        if (sizeof(R) == 8 || dq >= R(0.5) * (hi + hj))
                            lam = (R)lambda_quad<double>((double)dq, (double)hi, (double)hj, p.glx, p.glw);
                        fire = true;
                        P = pre * lam;
                        gfac = (R)p.mass[h] * lam * (p.bins ? (R)ldexp(p.dt_max, -bmin) : (R)p.dt[h]);
                        if (P > R(3)) ++n_gt1;
                    } else {
                        if constexpr (sizeof(R) == 4) fire = P >= R(1) || x.x[0] < (uint32_t)ceilf((float)P * 0x1p32f);
                        else fire = u < P;
                        if (P > R(1)) ++n_gt1;
                        if (fabs(P - u) < R(1e-6)) ++n_near;
                    }
                }
                const int64_t ui = slot2u + si, uj = slot2u + sj;
                if constexpr (MODE == kModeDrawExact) {
                    if (p.use_sump) {
                        // on individual steps a rate, scaled to dt_max (exact power of two)
                        const float ps = (float)(p.bins ? P * (R)ldexp(1.0, bmin) : P);
                        atomicAdd(p.sump + ui, ps);
                        atomicAdd(p.sump + uj, ps);
                    }
                }
                if (fire) {
                    const unsigned long long slot = atomicAdd(&p.cnt->ev_count, 1ull);
                    if (slot < p.ev_cap) {
                        sidm_event E;
                        E.key = ((unsigned long long)h << 54) | ((unsigned long long)a << 27) | (unsigned long long)b;
                        E.i = (uint32_t)(ida < idb ? ui : uj);
                        E.j = (uint32_t)(ida < idb ? uj : ui);
                        E.x1 = x.x[1];
                        E.x2 = x.x[2];
                        E.P = (float)P;
                        E.x0 = x.x[0];
                        p.ev[slot] = E;
                        if (drag) p.evg[slot] = (double)gfac;
                    }
                }
            }
            qhead = (qhead + nb) & (kQueue - 1);
            qn -= nb;
            __syncwarp();
        };

        // this lane's entry of candidate leaf Bl (the plain path loads it straight
        // into a register, so the walk can fetch the next leaf early)
        auto fetch = [&](int Bl) -> V {
            return P4[(int64_t)(leaf0 + Bl) * kLeaf + lane];
        };
        // craw: fetch(Bl) (unused on the bulk-copy path, which stages the leaf here)
        auto process = [&](int Bl, bool mine, const V& craw) {
            const int Bg = leaf0 + Bl;
            ++n_tiles;
            const int countB = (int)min((int64_t)kLeaf, nh - (int64_t)Bl * kLeaf);
            V c = craw;
            if constexpr (sizeof(R) == 4) {
                const float4 cB = p.cell[Bg];
                c.x = __fadd_rn(c.x, __fsub_rn(cB.x, cA.x));
                c.y = __fadd_rn(c.y, __fsub_rn(cB.y, cA.y));
                c.z = __fadd_rn(c.z, __fsub_rn(cB.z, cA.z));
            }
            __syncwarp();
            V* tp = st_pos.shifted();
            tp[lane] = c;
            __syncwarp();
            const uint32_t slotB = (uint32_t)Bg * kLeaf;
            // candidates that cannot reach any query of A (box gap > h_t + hmax_A) are skipped
            float3 pc;
            if constexpr (sizeof(R) == 4) {
                pc = make_float3(__fadd_rn(cA.x, c.x), __fadd_rn(cA.y, c.y), __fadd_rn(cA.z, c.z));
            } else {
                pc = make_float3(__double2float_rn(((double)c.x - fr.O[0]) * fr.down),
                                 __double2float_rn(((double)c.y - fr.O[1]) * fr.down),
                                 __double2float_rn(((double)c.z - fr.O[2]) * fr.down));
            }
            const float rc = __fadd_ru(__fmul_ru(__fadd_ru(to_float_ru_p<R>(c.w, fr.down), hmaxA), 1.0f + 0x1p-20f), fr.margin);
            const uint32_t cmask = __ballot_sync(
                0xffffffffu, lane < countB && point_gap2_rd(pc, qlo, qhi) <= __fmul_ru(rc, rc) &&
                                 (!p.bins || step_opens(p.bins[hb + (int64_t)Bl * kLeaf + lane], p.n_bins, p.substep)));
            // (i) the pairs to test: queries that reach B (qmask) x candidates that
            //     can reach some query (cmask), inside A only candidate > query.  The
            //     warp loops over the smaller mask: lane = query, candidates from the
            //     staged tile (bits of okm = candidates), or lane = candidate, queries
            //     from their staged copy (bits = queries).  Same tests, same operands.
            const uint32_t qmask = __ballot_sync(0xffffffffu, mine);
            const bool by_cand = __popc(qmask) < __popc(cmask);
            uint32_t okm = 0u, allow;
            if (!by_cand) {
                for (uint32_t mm = cmask; mm; mm &= mm - 1u) {
                    const int t = __ffs(mm) - 1;
                    const V pj = tp[t];
                    const R dx = sub_rn(pj.x, q.x), dy = sub_rn(pj.y, q.y), dz = sub_rn(pj.z, q.z);
                    const R d2 = fma_rn(dz, dz, fma_rn(dy, dy, mul_rn(dx, dx)));
                    const R hs = add_rn(q.w, pj.w);
                    okm |= (d2 < mul_rn(hs, hs) ? 1u : 0u) << t;
                }
                allow = mine ? cmask : 0u;
                if (Bl == A) allow &= 0xFFFFFFFEu << lane;
            } else {
                for (uint32_t mm = qmask; mm; mm &= mm - 1u) {
                    const int i = __ffs(mm) - 1;
                    const V qi = qsh[i];
                    const R dx = sub_rn(c.x, qi.x), dy = sub_rn(c.y, qi.y), dz = sub_rn(c.z, qi.z);
                    const R d2 = fma_rn(dz, dz, fma_rn(dy, dy, mul_rn(dx, dx)));
                    const R hs = add_rn(qi.w, c.w);
                    okm |= (d2 < mul_rn(hs, hs) ? 1u : 0u) << i;
                }
                allow = ((cmask >> lane) & 1u) ? qmask : 0u;
                if (Bl == A) allow &= (1u << lane) - 1u;
            }
            n_tested += (uint32_t)__popc(allow);
            okm &= allow;
            // queue entry of bit t: (query slot, candidate slot)
            const uint32_t own = by_cand ? slotB + lane : slotA;
            const uint32_t base = by_cand ? (uint32_t)leaf * kLeaf : slotB;
            // (ii) queue the pairs in rounds: every lane with pairs left adds up to
            //      PR, after the entries of the lanes below it
            for (uint32_t m = __ballot_sync(0xffffffffu, okm != 0u); m; m = __ballot_sync(0xffffffffu, okm != 0u)) {
                const int cnt = __popc(okm);
                int e = qhead + qn + __popc(m & lt);
                int c2 = __popc(m);
#pragma unroll
                for (int k = 2; k <= PR; ++k) {
                    const uint32_t mk = __ballot_sync(0xffffffffu, cnt >= k);
                    e += __popc(mk & lt);
                    c2 += __popc(mk);
                }
                const int take = min(cnt, PR);
                for (int k = 0; k < take; ++k, ++e) {
                    const int t = __ffs(okm) - 1;
                    okm &= okm - 1u;
                    q_si[e & (kQueue - 1)] = by_cand ? base + t : own;
                    q_sj[e & (kQueue - 1)] = by_cand ? own : base + t;
                }
                qn += c2;
                n_pairs += (uint32_t)c2;
                while (qn >= 32) run_batch(32);
            }
            __syncwarp();
        };

        // tree walk over leaves B >= A.  A node is visited iff some lane's point
        // lies within (h_i + hmax_node)(1 + 2^-20) + margin of the node's box.
        float3 pq;                                     // query point in the halo frame
        if constexpr (sizeof(R) == 4) {
            pq = make_float3(__fadd_rn(cA.x, (float)q.x), __fadd_rn(cA.y, (float)q.y), __fadd_rn(cA.z, (float)q.z));
        } else {
            pq = make_float3(__double2float_rn(((double)q.x - fr.O[0]) * fr.down),
                             __double2float_rn(((double)q.y - fr.O[1]) * fr.down),
                             __double2float_rn(((double)q.z - fr.O[2]) * fr.down));
        }
        const float hq = active ? to_float_ru_p<R>(q.w, fr.down) : -INFINITY;
        // this lane's query reaches box c: within (h_i + hmax_node)(1 + 2^-20) + margin
        auto near_box = [&](int c) -> bool {
            const float4 lo = blo[c], hi = bhi[c];
            const float r = __fadd_ru(__fmul_ru(__fadd_ru(hq, lo.w), 1.0f + 0x1p-20f), fr.margin);
            return active && point_gap2_rd(pq, lo, hi) <= __fmul_ru(r, r);
        };
        // boxes of nodes g0 .. g0+n-1 (n <= kArity = 32), one per lane
        auto load_boxes = [&](int g0, int n) {
            __syncwarp();
            if (lane < n) { blo[lane] = p.nlo[g0 + lane]; bhi[lane] = p.nhi[g0 + lane]; }
            __syncwarp();
        };
        // bit c: some lane's query reaches box c (each lane keeps its own bits
        // for the leaves of this node).  Every query point lies in the leaf's
        // box, so a child farther from that box than the reach of the largest
        // h_i is out of reach of every lane: one box test per child (a lane
        // each) leaves the per-lane point tests to the children that pass it.
        float hqmax = hq;
        for (int o = 16; o > 0; o >>= 1) hqmax = fmaxf(hqmax, __shfl_xor_sync(0xffffffffu, hqmax, o));
        uint32_t lane_bits = 0u;
        auto accept = [&](int n, uint32_t eligible) -> uint32_t {
            bool reach = false;
            if (lane < n && ((eligible >> lane) & 1u)) {
                const float4 lo = blo[lane], hi = bhi[lane];
                const float r = __fadd_ru(__fmul_ru(__fadd_ru(hqmax, lo.w), 1.0f + 0x1p-20f), fr.margin);
                reach = box_gap2_rd(qlo, qhi, lo, hi) <= __fmul_ru(r, r);
            }
            const uint32_t near = __ballot_sync(0xffffffffu, reach);
            uint32_t bits = 0u;
            if (active)
                for (uint32_t m = near; m; m &= m - 1u) {
                    const int c = __ffs(m) - 1;
                    bits |= (near_box(c) ? 1u : 0u) << c;
                }
            lane_bits = bits;
            return __reduce_or_sync(0xffffffffu, bits);
        };
        // nodes whose subtree holds a leaf >= A (level lev, local indices first ..)
        auto eligible_mask = [&](int lev, int first, int n) -> uint32_t {
            return __ballot_sync(0xffffffffu, lane < n && ((int64_t)(first + lane + 1) << (kArityLog * lev)) > A);
        };
        // accepted leaves in index order; the next one is fetched before this one
        // is processed, so its load overlaps this leaf's tests
        auto visit_leaves = [&](uint32_t acc, int first) {
            if (acc == 0u) return;
            int c = __ffs(acc) - 1;
            acc &= acc - 1u;
            V cur = fetch(first + c);
            while (true) {
                const int cn = __ffs(acc) - 1;         // -1: none left
                acc &= acc - 1u;
                V nxt{};
                if (cn >= 0) nxt = fetch(first + cn);
                process(first + c, (lane_bits >> c) & 1u, cur);
                if (cn < 0) break;
                c = cn;
                cur = nxt;
            }
        };
        auto push = [&](uint32_t acc, int lev, int first, int& sp) -> bool {
            const int cnt = __popc(acc);
            if (sp + cnt > kStack) return false;
            // descending local index on the stack, so the lowest is visited first
            if ((acc >> lane) & 1u) stack[sp + cnt - 1 - __popc(acc & lt)] = (lev << 24) | (first + lane);
            sp += cnt;
            __syncwarp();
            return true;
        };
        const int top = p.top[h];
        const int Hp = p.H + 1;
        int sp = 0;
        bool failed = false;
        {
            const int nb = p.lvl_off[top * Hp + h];
            const int ntop = p.lvl_off[top * Hp + h + 1] - nb;
            load_boxes(nb, ntop);
            const uint32_t acc = accept(ntop, eligible_mask(top, 0, ntop));
            if (top == 0) visit_leaves(acc, 0);
            else if (!push(acc, top, 0, sp)) failed = true;
        }
        while (sp > 0 && !failed) {
            const int e = stack[--sp];
            __syncwarp();
            const int lev = e >> 24, idx = e & 0xFFFFFF;
            const int cl = lev - 1;
            const int cb = p.lvl_off[cl * Hp + h];
            const int cc = p.lvl_off[cl * Hp + h + 1] - cb;
            const int first = idx * kArity;
            const int nch = min(kArity, cc - first);
            load_boxes(cb + first, nch);
            const uint32_t acc = accept(nch, eligible_mask(cl, first, nch));
            if (cl == 0) visit_leaves(acc, first);
            else if (!push(acc, cl, first, sp)) failed = true;
        }
        // the queue outlives the staged tiles (entries are slots), so one partial
        // batch per query leaf remains
        if (qn > 0) run_batch(qn);
        if (failed && lane == 0) raise_status(p.cnt, SIDM_DEV_STACK);
        // this leaf's counts into the warp's 64-bit statistics (the per-lane
        // ones summed over the warp; pairs and tiles are the same in every lane)
        {
            const uint32_t g1 = __reduce_add_sync(0xffffffffu, n_gt1);
            const uint32_t nr = __reduce_add_sync(0xffffffffu, n_near);
            const uint32_t te = __reduce_add_sync(0xffffffffu, n_tested);
            const uint32_t la = __reduce_add_sync(0xffffffffu, n_lam);
            if (lane == 0) {
                wst[0] += n_pairs; wst[1] += g1; wst[2] += nr; wst[3] += te; wst[4] += la; wst[5] += n_tiles;
                wst[6] = max(wst[6], (unsigned long long)n_tiles);
            }
            __syncwarp();
        }
    }
    // warp totals -> step statistics
    if (lane == 0) {
        if (wst[0]) atomicAdd(&p.st->n_pairs, wst[0]);
        if (wst[1]) atomicAdd(&p.st->n_p_gt1, wst[1]);
        if (wst[2]) atomicAdd(&p.st->n_near, wst[2]);
        if (wst[3]) atomicAdd(&p.st->n_tested, wst[3]);
        atomicAdd(&p.cnt->diag[4], wst[5]);
        atomicMax(&p.cnt->diag[5], wst[6]);
        if (wst[4]) atomicAdd(&p.cnt->diag[6], wst[4]);
    }
    st_pos.finish(lane, p.cnt);
}

// ---------------------------------------------------------------- draws
// Most in-range pairs never come near an event (P ~ 1e-6 .. 1e-4), and whether
// a draw can fire at all is decided by integers: P_ij <= T 2^-32 for every pair
// of a query leaf, with T from the largest sigma(v) v and Lambda <= 4 / h_i^3
// (kLamFUp), so a pair needs the two ids and Philox word 0 only; the few pairs
// with x0 <= T take the full evaluation (velocities, P, event).  One warp per
// query leaf, one query per lane:
//  * the tree is walked with the box of the queries and their largest h (one box
//    test per child, a lane each); accepted leaves are listed and loaded two at
//    a time;
//  * a listed leaf's candidates are kept if they come within h_j + the largest
//    h of the queries' box (tested in the query leaf's own frame, with room for
//    the rounding of the gap) and go to a ring;
//  * batches of kPBatch ring entries are tested against all 32 queries, two
//    candidates per packed FP32 operation, into one bit mask per lane;
//  * one warp scan of the masks' bit counts per batch gives every lane its place
//    in the warp's queue of (query lane, candidate) pairs, which is emptied 32
//    pairs at a time, all lanes busy.
// The FP64 form runs the same search on FP32 offsets (S4, in units of
// 2^HaloFrame::E) with a reach w = h and the rounding errors' bound (k_leaf_hmax),
// where a pair is out of range, in range for certain, or (about 1 in 10^3) settled
// by its FP64 distance before its draw;
// only pairs whose draw can fire take FP64 arithmetic.  2^20 NFW halo: 2.8 ms
// per launch against 39 ms with every test and P on the FP64 pipe, 16384
// particles 0.13 against 1.30 ms.
// Issue-bound (2.9 of 4 instructions per cycle): mixed form 1.95 ms for the 2^20
// NFW halo at N_ngb = 64 (3.28 ms before), 2.65e8 in-range pairs, 1.16e9 tests.
// Filling the queue in rounds of ballots and forming sigma(v) and
// a bound of P for every pair, with masked tests, took 331 lane instructions
// per in-range pair (52 % of them queueing and masks); a queue per lane, without
// the scan, left 54 % of the lanes idle in the draws (a leaf's partners lie
// after it in Morton order, and their number varies over its lanes).  Walk boxes
// of 2, 4 and 8 lane groups (1.97, 2.00, 2.07 ms), batches of 8 (2.19), runs of
// width 2, 2.5 and 4 (2.11, 1.95, 1.97), 1 and 3 groups of 32 pairs drawn together
// (2.10, 1.99 against 1.94 for 2) and 64 registers (2.17) were slower.
constexpr int kPBatch = 16;     // candidates per batch (batches start at multiples of it: never wrap)
constexpr int kPRing = 128;     // candidate ring entries (x, y, z and h apart)
constexpr int kPCand = 256;     // candidates whose ids and slots are kept for queued pairs
constexpr int kPQueue = 32 * (kPBatch + kPerRoundMax);   // queued pairs: a batch behind less than one draw's
constexpr int kPList = 64;      // accepted leaves listed before they are streamed
constexpr float kPSpread = 3.0f;   // widest box of a run of queries / its largest h
// Candidate leaves after which a warp leaves the rest of its item to a second launch,
// whose warps share it: the kernel of an outlier reaches the centre, and one warp would
// test the whole halo while the SMs idle.  Hernquist halos, N_ngb = 128: 200,000
// particles 1.39 ms (2.08 without; 1.87 with 1024), 400,000 1.92 (5.66; 2.05).  256
// leaves rests to ordinary warps of the 64-halo batch (72 against 50 ms).
constexpr uint32_t kPTiles = 512;
// Warps that share such a rest, at least and at most (powers of two): beside many short
// rests there can be a long one, so every rest is cut.  At least 1, 4, 8, 16: a core of
// 400,000 particles within six cells, with outliers, N_ngb = 16, 11.7, 6.9, 4.6, 3.5 ms,
// a dense halo beside a wide one 18.8, 8.1, 6.3, 6.4; ordinary halos alike.
constexpr int kPRestMin = 16, kPRest = 32;
static_assert((kPRing & (kPRing - 1)) == 0 && kPRing >= kPBatch - 1 + 2 * kLeaf, "the ring holds a batch's leftover plus two leaves");
static_assert(kPCand == 256, "a queued pair is (query lane << 8 | candidate mod 256)");

constexpr size_t draw_warp_bytes()
{
    return (size_t)kPRing * 16 + (size_t)kPCand * 8 + 32 * 4 + (size_t)(kPList + kStack) * 4 +
           (size_t)4 * 16 + (size_t)kPQueue * 2 + 8 * 8;
}
static_assert(draw_warp_bytes() % 16 == 0 && (kPList + kStack) % 4 == 0 && kPQueue % 8 == 0, "16-byte aligned parts");

constexpr uint32_t kUnsure = 0x80000000u;   // on a candidate's id (below 2^27): its pairs are settled in FP64

// max over v of sigma(v) v / s0 for kind 1: v / (1 + (v/w)^2)^2 peaks at v = w / sqrt(3)
constexpr float kSvMax = 0.32475953f;    // 3 sqrt(3) / 16, rounded up

// speed from its square, to a few FP32 units in the last place, with room for what
// squares below the form's normal numbers lose
__device__ __forceinline__ double speed_of(float v2) { return (double)(sqrtf(v2) + 4e-19f); }
__device__ __forceinline__ double speed_of(double v2)
{
    return (v2 > 1e-30 && v2 < 1e30 ? (double)sqrtf((float)v2) : sqrt(v2)) + 4e-154;
}

// REST: the launch that takes up the rests that the warps of the first one left
template <class R, int PR, bool DRAG, bool REST>
__global__ void __launch_bounds__(256, 3) k_pairs(PairParams p)
{
    static_assert(PR >= 1 && PR <= kPerRoundMax, "32-pair groups drawn together");
    using V = typename Vec4<R>::T;
    constexpr unsigned FULL = 0xffffffffu;
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned char* base = smem + wid * draw_warp_bytes();
    float* ring = (float*)base;                        // [4][kPRing] x, y, z, h
    float4* wbox = (float4*)(base + kPRing * 16);      // the queries' box: lo, hi (halo frame), centre, half widths (leaf frame)
    uint32_t* cid = (uint32_t*)(wbox + 4);             // [kPCand] candidate ids
    uint32_t* cslot = cid + kPCand;                    // [kPCand] and slots
    uint32_t* qid = cslot + kPCand;                    // [32] query ids
    int* list = (int*)(qid + 32);
    int* stack = list + kPList;
    unsigned long long* wst = (unsigned long long*)(stack + kStack);
    uint16_t* queue = (uint16_t*)(wst + 8);
    if (lane < 8) wst[lane] = 0ull;
    const R* __restrict__ T = (const R*)p.lam;
    constexpr bool kF32 = sizeof(R) == 4;
    const V* __restrict__ P4 = (const V*)p.P4;
    const float4* __restrict__ S4 = (const float4*)p.S4;
    const V* __restrict__ V4 = (const V*)p.V4;
    const uint32_t lt = (1u << lane) - 1u;
    const int Hp = p.H + 1;
    int64_t items = (int64_t)p.L * p.parts;
    int share = kPRestMin;                                 // warps that share a rest: more while some would have none
    if constexpr (REST) {
        items = min(p.cnt->pair_rest[0], (unsigned)p.rest_cap);
        while (share < kPRest && items * share < (int64_t)gridDim.x * blockDim.x / 32) share *= 2;
        items *= share;
    }

    while (true) {
        unsigned int item = 0u;
        if (lane == 0) item = atomicAdd(REST ? &p.cnt->pair_rest[1] : &p.cnt->work[1], 1u);
        item = __shfl_sync(FULL, item, 0);
        if ((int64_t)item >= items) break;
        // (leaf, part | runs before << 8, first candidate leaf, accepted leaves before it)
        int4 it = make_int4(0, 0, 0, 0);
        if constexpr (REST) it = p.rest[item / (unsigned)share];
        const int leaf = REST ? it.x : (int)(item / (unsigned)p.parts);
        const int part = REST ? it.y & 255 : (int)(item & (unsigned)(p.parts - 1));
        int run = REST ? -(it.y >> 8) : 0;                 // below 0: a run before the rest's
        const int h = p.leaf_halo[leaf];
        const int leaf0 = p.leaf_off[h];
        const int A = leaf - leaf0;
        const uint32_t nh = (uint32_t)(p.halo_off[h + 1] - p.halo_off[h]);   // n_max < 2^31
        auto index_of = [&](uint32_t slot) {                  // padded slot -> particle index
            return p.halo_off[h] + (int64_t)slot - (int64_t)leaf0 * kLeaf;
        };
        // with individual steps only particles whose step opens at this sub-step
        // take part; a leaf without such a particle has no pair to test
        const uint32_t slotA = (uint32_t)leaf * kLeaf + lane;
        const bool active = (uint32_t)A * kLeaf + lane < nh &&
                            (!p.bins || step_opens(p.bins[index_of(slotA)], p.n_bins, p.substep));
        if (p.bins && !__any_sync(FULL, active)) continue;
        const float4 cA = p.cell[leaf];
        const float margin = p.frame[h].margin;
        // forward-dominated halo: every in-range pair becomes a record (no draw);
        // only the instantiation for contexts with SIDM_FLAG_DRAG has room for them
        const bool drag = DRAG && p.xs[h].angular != 0;
        if (!DRAG && p.xs[h].angular != 0) {
            if (lane == 0) raise_status(p.cnt, SIDM_DEV_BAD_INPUT);
            continue;
        }
        float4 q = S4[slotA];
        if constexpr (!kF32) q.w = p.reach[slotA];
        // FP64 form: a pair below this share of (w_i + w_j)^2 is in range for certain
        const float sure = kF32 ? 1.f : q.w < 0.f ? 0.f : 1.0f - 0x1p-11f;
        if constexpr (!kF32) q.w = fabsf(q.w);
        // the draws' integer bound: no pair's P exceeds thr 2^-32 - 2e-6 (the factor
        // 1.001 and the 3e-6 cover every rounding and the |P - u| < 1e-6 count); a
        // bound that is not a number below one keeps every pair
        uint32_t thr = FULL;
        {
            const sidm_xs xs = p.xs[h];
            // Lengths, speeds and cross-sections may lie anywhere in the form's range, so
            // the factors meet in FP64 (a few operations per leaf); what the mixed form's
            // FP32 products of P can gain by rounding below the normal numbers is added
            double sv;
            if (xs.kind == 1) {
                sv = (double)kSvMax * fabs((double)(R)xs.w);
            } else {
                R vi2 = R(0);
                if (active) {
                    const R* vel = (const R*)p.vel;
                    const int64_t uA = index_of(slotA);
                    const R vx = vel[uA], vy = vel[p.N + uA], vz = vel[2 * p.N + uA];
                    vi2 = vx * vx + vy * vy + vz * vz;
                }
                sv = speed_of(vi2) + speed_of((R)__longlong_as_double((long long)p.cnt->vmax2[h]));
            }
            R X = (R)xs.s0 * (R)p.mass[h] * (p.bins ? (R)p.dt_max : (R)p.dt[h]);
            if (p.bins) {                                     // the longest step that opens now
                const int tz = p.substep ? __ffs(p.substep) - 1 : 31;
                X *= (R)__int_as_float((127 - max(0, p.n_bins - 1 - tz)) << 23);
            }
            double b;
            if constexpr (kF32) {
                const float inv = 1.f / q.w;
                b = (double)X * sv * (1.001 * kLamFUp * ((double)inv * inv * inv) + 0x1p-146);
                if (X > 0.f && X < 0x1p-100f) b = 1.0;
            } else {
                const double down = p.frame[h].down;
                const float inv = 1.f / ((1.0f - 0x1p-20f) * (float)((double)P4[slotA].w * down));
                b = (double)X * down * down * down * sv * (1.001 * kLamFUp * ((double)inv * inv * inv));
            }
            const float bf = __double2float_ru(b + 3e-6);
            uint32_t t = FULL;
            if (bf < 1.f) t = (uint32_t)(fmaxf(bf, 3e-6f) * 4294967296.f) + 1u;
            thr = __reduce_max_sync(FULL, active ? t : 0u);
            if (drag) thr = FULL;
        }
        qid[lane] = active ? p.ID[slotA] : 0u;
        uint32_t n_pairs = 0u, n_tested = 0u, n_tiles = 0u;       // the same in every lane

        // the halo's factors of P in the form's precision (FP64 conversions are
        // slow); plain draws form them for their few pairs only
        struct Factors { R pref, inv_w, dt; bool vdep; };
        auto factors = [&]() {
            const sidm_xs xs = p.xs[h];
            const R m = (R)p.mass[h], t = p.bins ? (R)p.dt_max : (R)p.dt[h];
            return Factors{(R)xs.s0 * m * t, xs.kind == 1 ? R(1) / (R)xs.w : R(0), t, xs.kind == 1};
        };
        constexpr bool kEvery = DRAG;
        const Factors fac = kEvery ? factors() : Factors{};
        // canonical d^2 of query pi and candidate pj (mixed form: the candidate
        // shifted into the query leaf's frame)
        auto pair_d2 = [&](const V& pi, const V& pj, uint32_t sj) -> R {
            R cx = pj.x, cy = pj.y, cz = pj.z;
            if constexpr (kF32) {
                const float4 cj = p.cell[sj / kLeaf];
                cx = __fadd_rn(cx, __fsub_rn(cj.x, cA.x));
                cy = __fadd_rn(cy, __fsub_rn(cj.y, cA.y));
                cz = __fadd_rn(cz, __fsub_rn(cj.z, cA.z));
            }
            const R dx = sub_rn(cx, pi.x), dy = sub_rn(cy, pi.y), dz = sub_rn(cz, pi.z);
            return fma_rn(dz, dz, fma_rn(dy, dy, mul_rn(dx, dx)));
        };
        // the full evaluation of the in-range pair (query lane li, slot sj): P,
        // decision, record
        auto evaluate = [&](int li, uint32_t sj, uint32_t idi, uint32_t idj) {
            const Philox4 x = philox4x32_10_rk(p.step_lo, min(idi, idj), max(idi, idj), (uint32_t)h, p.rk);
            const Factors fc = kEvery ? fac : factors();
            const uint32_t si = (uint32_t)leaf * kLeaf + li;
            const int64_t ui = index_of(si), uj = index_of(sj);
            R ux, uy, uz;
            if constexpr (!DRAG) {
                const R* vel = (const R*)p.vel;
                ux = vel[uj] - vel[ui];
                uy = vel[p.N + uj] - vel[p.N + ui];
                uz = vel[2 * p.N + uj] - vel[2 * p.N + ui];
            } else {
                const V vi = V4[si], vj = V4[sj];
                ux = vj.x - vi.x; uy = vj.y - vi.y; uz = vj.z - vi.z;
            }
            const V pi = P4[si], pj = P4[sj];
            const R hi = pi.w, hj = pj.w;
            const R v2 = ux * ux + uy * uy + uz * uz;
            const uint32_t a = min(idi, idj), b = max(idi, idj);
            // individual steps: the pair's longer step dt_max / 2^min(b_i, b_j)
            const float down = p.bins ? __int_as_float((127 - min(p.bins[ui], p.bins[uj])) << 23) : 1.f;   // 2^-min(b_i, b_j)
            const R prefp = fc.pref * down;
            // mixed form: P needs ~1e-6 relative accuracy only (the event decision
            // below is exact for the P computed here): reciprocal square roots and
            // approximate divisions are enough.
            R v, sig = R(1), inv, u;
            if constexpr (kF32) {
                v = v2 > 0.f ? v2 * rsqrtf(v2) : 0.f;
                if (fc.vdep) {
                    const float qq = v * fc.inv_w, tt = 1.f + qq * qq;
                    sig = __fdividef(1.f, tt * tt);
                }
                inv = __fdividef(1.f, fmaxf(hi, hj));
                u = (R)((float)x.x[0] * 0x1p-32f);
            } else {
                v = sqrt(v2);
                if (fc.vdep) { const R qq = v * fc.inv_w, tt = R(1) + qq * qq; sig = R(1) / (tt * tt); }
                inv = R(1) / (hi > hj ? hi : hj);
                u = (R)ldexp((double)x.x[0], -32);
            }
            const R pre = prefp * sig * v;
            const R P_up = pre * (R(kLamFUp) * inv * inv * inv);
            const bool need = drag || !(u >= P_up + R(2e-6));
            R P = R(0), gfac = R(0);
            bool fire = false;
            if (need) {
                atomicAdd(&wst[4], 1ull);
                const R d2 = pair_d2(pi, pj, sj);
                R f;
                if constexpr (kF32) {
                    const float d = d2 > 0.f ? d2 * rsqrtf(d2) : 0.f;
                    f = kEvery ? lambda_f_rows(p.lam4, d, hi, hj, inv) : lambda_f_fast(T, d, hi, hj, inv);
                } else {
                    f = lambda_f<R>(T, sqrt_rn(d2), hi, hj);
                }
                P = pre * (f * inv * inv * inv);
                if (drag) {
                    // the record keeps G = m_j Lambda dt; D = P / 3 at the step start.
                    // The turn's sine is the square root of a multiple of Lambda, so
                    // Lambda must be accurate relative to itself where it falls to
                    // zero, which neither the table nor an FP32 quadrature (its
                    // integrand cancels there) is: FP64 quadrature beyond half the
                    // support (everywhere in the FP64 form), the table inside, where
                    // Lambda > Lambda(0)/4 bounds its relative error
                    R lam = f * inv * inv * inv;
                    const R dq = sqrt_rn(d2);
                    if (!kF32 || dq >= R(0.5) * (hi + hj))
                        lam = (R)lambda_quad<double>((double)dq, (double)hi, (double)hj, p.glx, p.glw);
                    fire = true;
                    P = pre * lam;
                    gfac = (R)p.mass[h] * lam * (fc.dt * down);
                    if (P > R(3)) atomicAdd(&wst[1], 1ull);
                } else {
                    if constexpr (kF32) fire = P >= R(1) || x.x[0] < (uint32_t)ceilf((float)P * 0x1p32f);
                    else fire = u < P;
                    if (P > R(1)) atomicAdd(&wst[1], 1ull);
                    if (fabs(P - u) < R(1e-6)) atomicAdd(&wst[2], 1ull);
                }
            }
            if (fire) {
                // one counter update for the lanes that fire together
                const unsigned am = __activemask();
                const int lead = __ffs(am) - 1;
                unsigned long long slot = 0ull;
                if (lane == lead) slot = atomicAdd(&p.cnt->ev_count, (unsigned long long)__popc(am));
                slot = __shfl_sync(am, slot, lead) + (unsigned long long)__popc(am & lt);
                if (slot < p.ev_cap) {
                    sidm_event E;
                    E.key = ((unsigned long long)h << 54) | ((unsigned long long)a << 27) | (unsigned long long)b;
                    E.i = (uint32_t)(idi < idj ? ui : uj);
                    E.j = (uint32_t)(idi < idj ? uj : ui);
                    E.x1 = x.x[1];
                    E.x2 = x.x[2];
                    E.P = (float)P;
                    E.x0 = x.x[0];
                    p.ev[slot] = E;
                    if (drag) p.evg[slot] = (double)gfac;
                }
            }
        };

        // Consecutive particles of the Morton curve can lie far apart (on the sparse
        // outer shell on opposite sides of the halo), and boxes around them would
        // reach most of it: the queries are taken in runs of lanes whose box is at
        // most kPSpread times their largest h wide (nearly always one run).  Lanes no
        // wider apart than two of the cells that order them are not split: in a core
        // denser than the cells, leaves lie on one another, and each run would load them
        // all.  The runs follow from the lanes left alone, so that both launches cut
        // them alike
        uint32_t todo = __ballot_sync(FULL, active);
        while (todo) {
        bool act = (todo >> lane) & 1u;
        {
            const float px = __fadd_rn(cA.x, q.x), py = __fadd_rn(cA.y, q.y), pz = __fadd_rn(cA.z, q.z);
            float v[7] = {act ? px : INFINITY,  act ? py : INFINITY,  act ? pz : INFINITY,
                          act ? -px : INFINITY, act ? -py : INFINITY, act ? -pz : INFINITY, act ? -q.w : INFINITY};
            float w[7];
            auto box = [&]() {                               // of the act lanes: lo, -hi, -largest h
#pragma unroll
                for (int i = 0; i < 7; ++i) w[i] = act ? v[i] : INFINITY;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
                    for (int i = 0; i < 7; ++i) w[i] = fminf(w[i], __shfl_xor_sync(FULL, w[i], o));
                }
            };
            auto wide = [&]() {
                return fmaxf(fmaxf(-w[3] - w[0], -w[4] - w[1]), -w[5] - w[2]) > kPSpread * -w[6];
            };
            box();
            const bool whole = fmaxf(fmaxf(-w[3] - w[0], -w[4] - w[1]), -w[5] - w[2]) <= 2.f * p.frame[h].fine;
            if (!whole && wide()) {                          // the same in every lane
                // boxes of the lanes up to this one: the run ends before the first that is too wide
#pragma unroll
                for (int i = 0; i < 7; ++i) w[i] = v[i];
                for (int o = 1; o < 32; o <<= 1) {
#pragma unroll
                    for (int i = 0; i < 7; ++i) {
                        const float y = __shfl_up_sync(FULL, w[i], o);
                        if (lane >= o) w[i] = fminf(w[i], y);
                    }
                }
                const uint32_t over = __ballot_sync(FULL, act && wide());
                if (over) act = act && lane < __ffs(over) - 1;
                box();
            }
            todo &= ~__ballot_sync(FULL, act);
            if (REST && run < 0) { ++run; continue; }
            float f[6] = {act ? q.x : INFINITY,  act ? q.y : INFINITY,  act ? q.z : INFINITY,
                          act ? -q.x : INFINITY, act ? -q.y : INFINITY, act ? -q.z : INFINITY};
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
                for (int i = 0; i < 6; ++i) f[i] = fminf(f[i], __shfl_xor_sync(FULL, f[i], o));
            }
            __syncwarp();
            if (lane == 0) {
                wbox[0] = make_float4(w[0], w[1], w[2], 0.f);
                wbox[1] = make_float4(-w[3], -w[4], -w[5], -w[6]);
                // centre and half widths; with c = RN(x - centre) the computed gap
                // |c| - half of a point x exceeds the true one by less than 2^-22 (gap +
                // half), which the factors here and on the reach cover
                const float cx = 0.5f * (f[0] - f[3]), cy = 0.5f * (f[1] - f[4]), cz = 0.5f * (f[2] - f[5]);
                const float s = 1.0f + 0x1p-18f;
                wbox[2] = make_float4(-cx, -cy, -cz, 0.f);
                wbox[3] = make_float4(s * fmaxf(-f[3] - cx, cx - f[0]), s * fmaxf(-f[4] - cy, cy - f[1]),
                                      s * fmaxf(-f[5] - cz, cz - f[2]), -w[6]);
            }
            __syncwarp();
        }
        // the query, negated, in both halves (NaN: in range of nothing)
        const float nx = act ? -q.x : __int_as_float(0x7fffffff);
        const unsigned long long qx2 = pack2(nx, nx), qy2 = pack2(-q.y, -q.y), qz2 = pack2(-q.z, -q.z), qw2 = pack2(q.w, q.w);

        // the accepted children of a node: local leaf indices into the list (this
        // part's share: every parts-th one), or nodes onto the stack.  A child is
        // visited iff the queries' box comes within (h + hmax_child)(1 + 2^-20) +
        // margin of the child's box, h the queries' largest, and its subtree holds a
        // leaf >= A
        int nl = 0, seen = REST ? it.w : 0, sp = 0;
        const int from = REST ? max(A, it.z) : A;          // the first leaf of this walk
        it.z = it.w = 0;                                   // later runs start anew
        bool failed = false;
        auto visit = [&](int lev, int first, int base, int n) {
            float4 lo = make_float4(0.f, 0.f, 0.f, 0.f), hi = lo;
            const bool in = lane < n && ((int64_t)(first + lane + 1) << (kArityLog * lev)) > (int64_t)from;
            if (in) { lo = p.nlo[base + first + lane]; hi = p.nhi[base + first + lane]; }
            const float4 qhi = wbox[1];
            const float r = __fadd_ru(__fmul_ru(__fadd_ru(qhi.w, lo.w), 1.0f + 0x1p-20f), margin);
            const bool ok = box_gap2_rd(wbox[0], qhi, lo, hi) <= __fmul_ru(r, r);
            uint32_t acc = __ballot_sync(FULL, in && ok);
            if (lev == 0) {
                const int no = seen + __popc(acc & lt);
                const bool mine = ((acc >> lane) & 1u) && (no & (p.parts - 1)) == part &&
                                  (!REST || ((unsigned)(no >> p.parts_log) & (share - 1)) == (item & (share - 1)));
                seen += __popc(acc);
                acc = __ballot_sync(FULL, mine);
                if (mine) list[nl + __popc(acc & lt)] = first + lane;
                nl += __popc(acc);
            } else if (sp + __popc(acc) > kStack) {
                failed = true;
            } else {
                // descending local index on the stack, so the lowest is visited first
                sp += __popc(acc);
                if ((acc >> lane) & 1u) stack[sp - 1 - __popc(acc & lt)] = (lev << 24) | (first + lane);
            }
            __syncwarp();
        };
        const int top = p.top[h];
        {
            const int nb = p.lvl_off[top * Hp + h];
            visit(top, 0, nb, p.lvl_off[top * Hp + h + 1] - nb);
        }
        // ring entries: candidate numbers cnum .. cnum + navail - 1; queued pairs qn,
        // the oldest candidate number they may name, entries of the query leaf
        // itself still in the ring and this lane's rank among them
        int navail = 0, qn = 0, nself = 0, rank = 0, li = 0;
        uint32_t cnum = 0u, oldest = 0u;
        const int n_act = __popc(__ballot_sync(FULL, act));
        while (true) {
            bool fin = false;
            if (li < nl) {
                // two listed leaves: shift, filter, append to the ring
                const int Bl[2] = {list[li], list[min(li + 1, nl - 1)]};
                float4 c[2], cB[2];
                uint32_t id[2];
                bool open[2];
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const uint32_t s = (uint32_t)(leaf0 + Bl[u]) * kLeaf + lane;
                    c[u] = S4[s];
                    if constexpr (!kF32) c[u].w = p.reach[s];
                    cB[u] = p.cell[leaf0 + Bl[u]];
                    id[u] = p.ID[s];
                    if constexpr (!kF32) {
                        if (c[u].w < 0.f) id[u] |= kUnsure;
                        c[u].w = fabsf(c[u].w);
                    }
                    open[u] = (uint32_t)Bl[u] * kLeaf + lane < nh && li + u < nl;
                    if (p.bins) open[u] = open[u] && step_opens(p.bins[index_of(s)], p.n_bins, p.substep);
                }
                const float4 fc = wbox[2], fw = wbox[3];
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    c[u].x = __fadd_rn(c[u].x, __fsub_rn(cB[u].x, cA.x));     // exact shift into the query leaf's frame
                    c[u].y = __fadd_rn(c[u].y, __fsub_rn(cB[u].y, cA.y));
                    c[u].z = __fadd_rn(c[u].z, __fsub_rn(cB[u].z, cA.z));
                    const float gx = fmaxf(fabsf(c[u].x + fc.x) - fw.x, 0.f), gy = fmaxf(fabsf(c[u].y + fc.y) - fw.y, 0.f),
                                gz = fmaxf(fabsf(c[u].z + fc.z) - fw.z, 0.f);
                    const float r = (c[u].w + fw.w) * (1.0f + 0x1p-18f);
                    const bool keep = open[u] && gx * gx + gy * gy + gz * gz <= r * r;
                    const uint32_t m = __ballot_sync(FULL, keep);
                    if (u == 0 && Bl[0] == A) {                           // A is the first of its walk
                        nself = __popc(m);
                        rank = __popc(m & lt);
                        n_tested -= __reduce_add_sync(FULL, act ? (unsigned)rank + 1u : 0u);   // each of its pairs once
                    }
                    if (keep) {
                        const uint32_t e = cnum + navail + __popc(m & lt);
                        float* at = ring + (e & (kPRing - 1));
                        at[0] = c[u].x; at[kPRing] = c[u].y; at[2 * kPRing] = c[u].z; at[3 * kPRing] = c[u].w;
                        uint32_t* ca = cid + (e & (kPCand - 1));
                        ca[0] = id[u];
                        ca[kPCand] = (uint32_t)(leaf0 + Bl[u]) * kLeaf + lane;
                    }
                    navail += __popc(m);
                    n_tested += (uint32_t)(n_act * __popc(m));
                }
                n_tiles += min(2, nl - li);
                li += 2;
                __syncwarp();
            } else if (!REST && sp > 0 && n_tiles > kPTiles && p.rest_cap > 0 && !failed) {
                // the rest of this walk (the unvisited leaves are those from the stack's
                // top node on) and the later runs go to the second launch
                const int e = stack[sp - 1];
                unsigned int slot = 0u;
                if (lane == 0) slot = atomicAdd(&p.cnt->pair_rest[0], 1u);
                slot = __shfl_sync(FULL, slot, 0);
                if (slot >= (unsigned)p.rest_cap) { raise_status(p.cnt, SIDM_DEV_STACK); break; }   // cannot happen: one per item
                if (lane == 0) p.rest[slot] = make_int4(leaf, part | (run << 8), (e & 0xFFFFFF) << (kArityLog * (e >> 24)), seen);
                sp = 0;
                todo = 0u;
            } else if (sp > 0 && !failed) {
                // walk until the list may not hold another node's leaves, or the tree is done
                nl = li = 0;
                do {
                    const int e = stack[--sp];
                    __syncwarp();
                    const int cl = (e >> 24) - 1, first = (e & 0xFFFFFF) * kArity;
                    const int cb = p.lvl_off[cl * Hp + h];
                    visit(cl, first, cb, min(kArity, p.lvl_off[cl * Hp + h + 1] - cb - first));
                } while (sp > 0 && nl <= kPList - kArity && !failed);
            } else {
                // at the very end fill the partial batch with infinitely far entries
                fin = true;
                const int fill = (kPBatch - navail % kPBatch) % kPBatch;
                if (lane < fill) {
                    float* at = ring + ((cnum + navail + lane) & (kPRing - 1));
                    at[0] = INFINITY; at[kPRing] = INFINITY; at[2 * kPRing] = INFINITY; at[3 * kPRing] = 0.f;
                }
                navail += fill;
                __syncwarp();
            }
            while (navail >= kPBatch || (fin && qn > 0)) {
                int full = qn;                           // pairs to draw now: all of them at the very end
                if (navail >= kPBatch) {
                    // the ring's first kPBatch candidates against all queries
                    uint32_t okm = 0u, surem = 0u;          // in range; FP64 form: for certain
                    const unsigned long long sure2 = pack2(sure, sure);
#pragma unroll
                    for (int t = 0; t < kPBatch; t += 4) {
                        const float* at = ring + (cnum & (kPRing - 1)) + t;
                        const ulonglong2 x = *(const ulonglong2*)at, y = *(const ulonglong2*)(at + kPRing),
                                         z = *(const ulonglong2*)(at + 2 * kPRing), w = *(const ulonglong2*)(at + 3 * kPRing);
#pragma unroll
                        for (int u = 0; u < 2; ++u) {
                            const unsigned long long dx = add2(u ? x.y : x.x, qx2), dy = add2(u ? y.y : y.x, qy2),
                                                     dz = add2(u ? z.y : z.x, qz2);
                            const unsigned long long d2 = fma2(dz, dz, fma2(dy, dy, mul2(dx, dx)));
                            const unsigned long long hs = add2(qw2, u ? w.y : w.x), hs2 = mul2(hs, hs);
                            float da, db, ha, hb;
                            unpack2(d2, da, db);
                            unpack2(hs2, ha, hb);
                            if (da < ha) okm |= 1u << (t + 2 * u);
                            if (db < hb) okm |= 2u << (t + 2 * u);
                            if constexpr (!kF32) {
                                unpack2(mul2(hs2, sure2), ha, hb);
                                if (da < ha) surem |= 1u << (t + 2 * u);
                                if (db < hb) surem |= 2u << (t + 2 * u);
                            }
                        }
                    }
                    if (nself > 0) {                     // inside the leaf each pair once: candidates after the query
                        const int after = rank + 1;      // candidate number of the leaf, counted from the first
                        okm &= after - (int)cnum >= 32 ? 0u : after > (int)cnum ? FULL << (after - (int)cnum) : FULL;
                        nself -= kPBatch;
                    }
                    // this lane's place in the queue, then its pairs
                    const int n = __popc(okm);
                    int inc = n;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const int y = __shfl_up_sync(FULL, inc, o);
                        if (lane >= o) inc += y;
                    }
                    const int total = __shfl_sync(FULL, inc, 31);
                    uint16_t* qp = queue + qn + inc - n;
                    const uint32_t tag = (uint32_t)lane << 8;
#pragma unroll
                    for (int t = 0; t < kPBatch; ++t)
                        if ((okm >> t) & 1u)
                            *qp++ = (uint16_t)(tag | ((cnum + t) & (kPCand - 1)) | (kF32 || ((surem >> t) & 1u) ? 0u : 0x8000u));
                    if (qn == 0) oldest = cnum;
                    qn += total;
                    n_pairs += (uint32_t)total;
                    const int rest = qn % (32 * PR);
                    full = qn - rest;
                    // the waiting pairs keep their candidates: draw them too before those are overwritten
                    if (total < rest) { if (cnum + 2 * kPBatch + 2 * kLeaf - oldest > kPCand) full = qn; }
                    else oldest = cnum;
                    cnum += kPBatch;
                    navail -= kPBatch;
                    __syncwarp();
                }
                for (int f0 = 0; f0 < full; f0 += 32 * PR) {
                    uint32_t ent[PR], idi[PR], idj[PR];
                    uint32_t maybe = 0u;
#pragma unroll
                    for (int k = 0; k < PR; ++k) {
                        const int at = f0 + 32 * k + lane;
                        ent[k] = queue[at < full ? at : f0];
                        idi[k] = qid[(ent[k] >> 8) & 31u];
                        idj[k] = cid[ent[k] & (kPCand - 1)];
                        bool valid = at < full;
                        if constexpr (!kF32) {               // settled in FP64 where FP32 is not sure
                            const bool ask = valid && ((ent[k] & 0x8000u) || (idj[k] & kUnsure));
                            idj[k] &= ~kUnsure;
                            if (__any_sync(FULL, ask)) {
                                if (ask) {
                                    const uint32_t sj = cslot[ent[k] & (kPCand - 1)];
                                    const V pi = P4[(uint32_t)leaf * kLeaf + ((ent[k] >> 8) & 31u)], pj = P4[sj];
                                    const R hs = add_rn(pi.w, pj.w);
                                    valid = pair_d2(pi, pj, sj) < mul_rn(hs, hs);
                                }
                                n_pairs -= (uint32_t)__popc(__ballot_sync(FULL, ask && !valid));
                            }
                            ent[k] &= 0x7fffu;
                        }
                        const Philox4 x = philox4x32_10_rk(p.step_lo, min(idi[k], idj[k]), max(idi[k], idj[k]), (uint32_t)h, p.rk);
                        maybe |= (valid && x.x[0] <= thr ? 1u : 0u) << k;
                    }
                    if (maybe) {
#pragma unroll 1
                        for (int k = 0; k < PR; ++k) {
                            if (!((maybe >> k) & 1u)) continue;
                            uint32_t en = ent[0], di = idi[0], dj = idj[0];
#pragma unroll
                            for (int r = 1; r < PR; ++r)
                                if (r == k) { en = ent[r]; di = idi[r]; dj = idj[r]; }
                            evaluate((int)(en >> 8), cslot[en & (kPCand - 1)], di, dj);
                        }
                    }
                }
                // the rest moves to the queue's front
                if (full > 0) {
                    const int rest = qn - full;          // < 32 PR <= full: no overlap
                    __syncwarp();
#pragma unroll
                    for (int k = 0; k < PR; ++k)
                        if (32 * k + lane < rest) queue[32 * k + lane] = queue[full + 32 * k + lane];
                    qn = rest;
                    __syncwarp();
                }
            }
            if (fin) break;
        }
        if (failed && lane == 0) raise_status(p.cnt, SIDM_DEV_STACK);
        ++run;
        }   // runs of queries
        // this leaf's counts into the warp's 64-bit statistics
        {
            __syncwarp();
            if (lane == 0) {
                wst[0] += n_pairs; wst[3] += n_tested; wst[5] += n_tiles;
                wst[6] = max(wst[6], (unsigned long long)n_tiles);
            }
            __syncwarp();
        }
    }
    // warp totals -> step statistics
    if (lane == 0) {
        if (wst[0]) atomicAdd(&p.st->n_pairs, wst[0]);
        if (wst[1]) atomicAdd(&p.st->n_p_gt1, wst[1]);
        if (wst[2]) atomicAdd(&p.st->n_near, wst[2]);
        if (wst[3]) atomicAdd(&p.st->n_tested, wst[3]);
        atomicAdd(&p.cnt->diag[4], wst[5]);
        atomicMax(&p.cnt->diag[5], wst[6]);
        if (wst[4]) atomicAdd(&p.cnt->diag[6], wst[4]);
    }
}

// Largest squared speed of every halo whose cross-section does not depend on the
// speed (kind 0), for the bound of P: kSplit CTAs per reduction chunk, one atomic
// each.  A NaN drops out of the maximum: its pairs have P = NaN and never fire.
constexpr int kVmaxSplit = 4, kVmaxChunk = 16384;
template <class R>
__global__ void __launch_bounds__(256) k_vmax(const R* __restrict__ vel, int64_t N, const int32_t* __restrict__ chunk_halo,
                                              const int64_t* __restrict__ chunk_begin, const int64_t* __restrict__ halo_off,
                                              const sidm_xs* __restrict__ xs, DevCounters* __restrict__ cnt)
{
    const int c = blockIdx.x / kVmaxSplit, part = blockIdx.x % kVmaxSplit;
    const int h = chunk_halo[c];
    if (xs[h].kind == 1) return;
    const int64_t b = chunk_begin[c] + (int64_t)part * (kVmaxChunk / kVmaxSplit);
    const int64_t e = min(min(chunk_begin[c] + kVmaxChunk, halo_off[h + 1]), b + kVmaxChunk / kVmaxSplit);
    R m = R(0);
#pragma unroll 4
    for (int64_t s = b + threadIdx.x; s < e; s += blockDim.x) {
        const R x = vel[s], y = vel[N + s], z = vel[2 * N + s];
        const R v2 = x * x + y * y + z * z;
        m = v2 > m ? v2 : m;
    }
    for (int o = 16; o > 0; o >>= 1) { const R y = __shfl_xor_sync(0xffffffffu, m, o); m = y > m ? y : m; }
    if ((threadIdx.x & 31) == 0 && m > R(0)) atomicMax(&cnt->vmax2[h], (unsigned long long)__double_as_longlong((double)m));
}

void fill_params(sidm_ctx* c, PairParams& p, uint64_t seed, uint64_t step, const sidm_xs* xs, const double* dt,
                 const double* mass, const void* vel, sidm_step_stats* st)
{
    const LayoutHost& L = c->lay;
    p = PairParams{};
    p.H = L.H; p.L = L.L;
    p.leaf_halo = c->d_leaf_halo; p.leaf_off = c->d_leaf_off; p.halo_off = c->d_halo_off;
    p.lvl_off = c->d_lvl_off; p.top = c->d_top; p.frame = c->d_frame; p.cell = c->d_cell;
    p.nlo = c->d_nlo; p.nhi = c->d_nhi; p.P4 = c->d_P4; p.S4 = c->cfg.precision == SIDM_FP64 ? (const void*)c->d_S4 : c->d_P4; p.reach = c->d_reach; p.V4 = c->d_V4; p.ID = c->d_ID; p.lam = c->d_lam; p.lam4 = c->d_lam4;
    p.vel = vel; p.N = L.N; p.parts = 1;
    p.xs = xs; p.dt = dt; p.mass = mass;
    p.seed_lo = (uint32_t)seed; p.seed_hi = (uint32_t)(seed >> 32); p.step_lo = (uint32_t)step;
    for (int r = 0; r < 10; ++r) {
        p.rk[2 * r] = p.seed_lo + (uint32_t)r * 0x9E3779B9u;
        p.rk[2 * r + 1] = p.seed_hi + (uint32_t)r * 0xBB67AE85u;
    }
    p.ev = c->d_ev; p.ev_cap = (unsigned long long)c->cfg.event_cap;
    p.sump = c->d_sump; p.use_sump = (c->cfg.flags & SIDM_FLAG_SUM_P) ? 1 : 0;
    p.dacc = c->d_dacc; p.nacc = L.N;
    p.bins = c->step_bins; p.n_bins = c->step_nbins; p.substep = c->step_sub; p.dt_max = c->step_dtmax;
    p.cnt = c->d_cnt; p.st = st;
    p.evg = c->d_evg;
    for (int g = 0; g < 8; ++g) { p.glx[g] = c->gl8x[g]; p.glw[g] = c->gl8w[g]; }
}

template <class R, int MODE, bool DRAG>
int launch_all(sidm_ctx* c, uint64_t seed, uint64_t step, const sidm_xs* xs, const double* dt, const double* mass,
               const void* vel, sidm_step_stats* st, cudaStream_t s)
{
    PairParams p;
    fill_params(c, p, seed, step, xs, dt, mass, vel, st);
    const LayoutHost& L = c->lay;
    const int warps = c->pair_warps;
    const size_t smem = (size_t)warps * pair_warp_bytes<R>();
    auto kern = k_pairs_all<R, MODE, DRAG>;
    int occ = 0;
    if (int rc = occupancy(c, (const void*)kern, warps * 32, smem, &occ)) return rc;
    if (occ < 1) return set_err(c, SIDM_ECAPACITY, "pair kernel does not fit on an SM");
    int grid = c->cfg.grid_ctas > 0 ? c->cfg.grid_ctas : c->sm_count * occ;
    grid = std::max(1, std::min(grid, (L.L + warps - 1) / warps));
    c->pair_grid = grid;
    cudaError_t e = cudaMemsetAsync(&c->d_cnt->work[1], 0, sizeof(unsigned int), s);
    if (e != cudaSuccess) return cuda_check(c, e, "pair work reset");
    const int tidx = MODE == kModeDiag ? -1 : timer_begin(c, 2, s);
    kern<<<grid, warps * 32, smem, s>>>(p);
    timer_end(c, tidx, s);
    c->launches++;
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_check(c, e, "pair launch");
    return SIDM_OK;
}

// With few query leaves each is shared by several warps (a
// power of two, at most kPartsMax), so that every resident warp has about
// N_ngb / 16 items, 2 to 4: the last wave stays short, at the price of the walk that
// the parts repeat, which weighs more the fewer neighbours there are (N_ngb = 16,
// 100,000 uniform particles: 147 us with 4 parts, 181 with 8; Hernquist 179, 230).
constexpr int kPartsMax = 16;
template <class R, int PR, bool DRAG>
int launch_draws(sidm_ctx* c, uint64_t seed, uint64_t step, const sidm_xs* xs, const double* dt, const double* mass,
                 const void* vel, sidm_step_stats* st, cudaStream_t s)
{
    PairParams p;
    fill_params(c, p, seed, step, xs, dt, mass, vel, st);
    const LayoutHost& L = c->lay;
    const int warps = c->pair_warps;
    const size_t smem = (size_t)warps * draw_warp_bytes();
    auto kern = k_pairs<R, PR, DRAG, false>;
    auto kern_rest = k_pairs<R, DRAG ? 1 : kPerRoundDefault, DRAG, true>;   // the groups drawn together change no result
    int occ = 0;
    if (int rc = occupancy(c, (const void*)kern, warps * 32, smem, &occ)) return rc;
    if (occ < 1) return set_err(c, SIDM_ECAPACITY, "pair kernel does not fit on an SM");
    int grid = c->cfg.grid_ctas > 0 ? c->cfg.grid_ctas : c->sm_count * occ;
    // (four, too, where a warp's kPTiles leaves are much of the halo)
    const int64_t want = (int64_t)(L.L < 2 * (int)kPTiles ? 4 : std::max(2, std::min(4, c->kmax_cur / 16))) * grid * warps;
    while (p.parts < kPartsMax && (int64_t)L.L * p.parts < want) { p.parts *= 2; ++p.parts_log; }
    int rest_occ = 0;
    if (int rc = occupancy(c, (const void*)kern_rest, warps * 32, smem, &rest_occ)) return rc;
    if (rest_occ < 1) return set_err(c, SIDM_ECAPACITY, "pair kernel does not fit on an SM");
    const int rest_grid = std::max(1, c->cfg.grid_ctas > 0 ? c->cfg.grid_ctas : c->sm_count * rest_occ);
    p.rest = c->d_pair_rest;
    // a halo of few leaves has no warp that wants so many; every item may leave one rest
    p.rest_cap = L.L > (int)kPTiles && (int64_t)L.L * p.parts <= c->pair_rest_cap ? c->pair_rest_cap : 0;
    grid = (int)std::max<int64_t>(1, std::min<int64_t>(grid, ((int64_t)L.L * p.parts + warps - 1) / warps));
    c->pair_grid = grid;
    cudaError_t e = cudaMemsetAsync(&c->d_cnt->work[1], 0, sizeof(unsigned int), s);
    if (e != cudaSuccess) return cuda_check(c, e, "pair work reset");
    {
        k_vmax<R><<<L.nchunk * kVmaxSplit, 256, 0, s>>>((const R*)vel, L.N, c->d_chunk_halo, c->d_chunk_begin, c->d_halo_off,
                                                        xs, c->d_cnt);
        c->launches++;
    }
    const int tidx = timer_begin(c, 2, s);
    kern<<<grid, warps * 32, smem, s>>>(p);
    c->launches++;
    if (p.rest_cap > 0) {
        kern_rest<<<rest_grid, warps * 32, smem, s>>>(p);
        c->launches++;
    }
    timer_end(c, tidx, s);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_check(c, e, "pair launch");
    return SIDM_OK;
}

}  // namespace

template <class R>
static int launch_form(sidm_ctx* c, uint64_t seed, uint64_t step, const sidm_xs* xs, const double* dt, const double* mass,
                       const void* vel, sidm_step_stats* st, cudaStream_t s)
{
    const bool exact = (c->cfg.flags & SIDM_FLAG_SUM_P) != 0;
    if (c->cfg.flags & SIDM_FLAG_DRAG)                  // forward-dominated halos allowed
        return exact ? launch_all<R, kModeDrawExact, true>(c, seed, step, xs, dt, mass, vel, st, s)
                     : launch_draws<R, 1, true>(c, seed, step, xs, dt, mass, vel, st, s);
    if (exact) return launch_all<R, kModeDrawExact, false>(c, seed, step, xs, dt, mass, vel, st, s);
    // the hot path: groups of 32 pairs drawn together as configured (a launch knob)
    switch (c->cfg.pair_per_round > 0 ? c->cfg.pair_per_round : kPerRoundDefault) {
    case 1: return launch_draws<R, 1, false>(c, seed, step, xs, dt, mass, vel, st, s);
    case 2: return launch_draws<R, 2, false>(c, seed, step, xs, dt, mass, vel, st, s);
    case 3: return launch_draws<R, 3, false>(c, seed, step, xs, dt, mass, vel, st, s);
    default: return launch_draws<R, 4, false>(c, seed, step, xs, dt, mass, vel, st, s);
    }
}

int launch_pairs(sidm_ctx* c, uint64_t seed, uint64_t step, const sidm_xs* xs, const double* dt, const double* mass,
                 const void* vel, sidm_step_stats* st, cudaStream_t s)
{
    if (c->lay.L == 0) return SIDM_OK;
    return c->cfg.precision == SIDM_FP64 ? launch_form<double>(c, seed, step, xs, dt, mass, vel, st, s)
                                         : launch_form<float>(c, seed, step, xs, dt, mass, vel, st, s);
}

int launch_pairs_diag(sidm_ctx* c, const sidm_xs* xs, const double* mass, cudaStream_t s)
{
    if (c->lay.L == 0) return SIDM_OK;
    return launch_all<double, kModeDiag, false>(c, 0, 0, xs, nullptr, mass, nullptr, c->d_stats_own, s);
}

}  // namespace sidm
