// sidm_knn.cu -- (a1) kernel sizes: h_i = distance to the N_ngb-th nearest
// other particle of the halo (Sect. 2: each particle's kernel size adapts to
// its N_ngb nearest neighbours; Eq. hDl: h is the radius of the sphere holding
// N_ngb particles).
//
// One warp per leaf of 32 consecutive Morton-ordered particles, one query per
// lane.  Candidate leaves are staged through shared memory (plain coalesced
// 128-bit loads, or bulk asynchronous copies with an mbarrier), shifted into
// the query leaf's frame, and every lane keeps a 4-ary max-heap of its N_ngb
// smallest keys in shared memory (one 128-bit load per heap level).  The heap
// is first filled from the leaves next to the query leaf in Morton order
// (stored unsorted, then heapified once), whose k-th distance bounds the
// search radius; the bounding-volume tree is then walked with that
// (shrinking) radius, nearest children first, skipping those leaves.  Inside
// a tile a lane only appends keys below its current bound to a short pending
// list; the lists are merged into the heaps in batches, so the divergent heap
// sift runs with every lane busy instead of once per candidate.  The result
// is the exact k-th smallest of the canonical distance, so it does not depend
// on tile order, flush points or launch shape.
#include <type_traits>

#include "sidm_internal.cuh"
#include "sidm_tile.cuh"

namespace sidm {
namespace {

template <class R, bool NBR>
struct KeyOf {
    using T = typename std::conditional<(sizeof(R) == 8) || NBR, unsigned long long, uint32_t>::type;
};

struct KnnParams {
    int H, L;
    const int32_t* leaf_halo;
    const int32_t* leaf_off;
    const int64_t* halo_off;
    const int32_t* lvl_off;
    const int32_t* top;
    const int32_t* ngb;
    const HaloFrame* frame;
    const float4* cell;
    const float4* nlo;
    const float4* nhi;
    void* P4;
    const void* S4;     // FP32 offsets the warm-started search reads (mixed form: P4)
    const uint32_t* ID;
    void* h_out;
    uint32_t* nbr;
    int k_stride;
    int kcap;
    DevCounters* cnt;
    unsigned int* work;          // persistent work counter (zeroed before the launch)
    const int32_t* leaf_list;    // NULL: every leaf; else the leaves listed here ...
    const unsigned int* list_len;  // ... of which there are *list_len
    int32_t* long_list;          // k_knn_warm without teams: where leaves of more than tiles_max candidate leaves go
    unsigned tiles_max;
    unsigned int* long_len;
    void* hprev;        // out: h per particle (next call's guess), NULL for neighbour lists
    int use_guess;      // P4.w holds each particle's previous kernel size
    float slack;        // guess bound = previous h * slack
    const void* V4;     // moments: velocities, particle mass, sums [5][nacc]
    const double* mass;
    double* dacc;
    int64_t nacc;
    int flush_node;     // pending keys per lane that trigger a merge before a node's tests
};

template <class R, bool NBR>
__device__ __forceinline__ typename KeyOf<R, NBR>::T make_key(R d2, uint32_t id)
{
    if constexpr (sizeof(R) == 8) {
        return (unsigned long long)__double_as_longlong((double)d2);
    } else if constexpr (NBR) {
        return ((unsigned long long)__float_as_uint((float)d2) << 32) | id;
    } else {
        return __float_as_uint((float)d2);
    }
}

template <class R, bool NBR>
__device__ __forceinline__ R key_d2(typename KeyOf<R, NBR>::T k)
{
    if constexpr (sizeof(R) == 8) return (R)__longlong_as_double((long long)k);
    else if constexpr (NBR) return (R)__uint_as_float((uint32_t)(k >> 32));
    else return (R)__uint_as_float((uint32_t)k);
}

// Per-lane 4-ary max-heaps of keys (all keys are >= 0 as unsigned integers).
// Node t (0-based) sits at position t + 3, so the children 4t+1 .. 4t+4 of
// node t fill the aligned group t + 1.  Group g of lane l is stored at
// [g][l][0..3]: a lane reads all four children with one vector load and the
// 32 lanes of a warp hit distinct banks.  Positions past the last node read
// as 0, which never exceeds a key, so a missing child is never promoted.
template <class K>
struct Heap4 {
    K* g;        // [groups][32][4]
    int lane;
    __device__ K& at(int t) const { const int pos = t + 3; return g[((pos >> 2) * 32 + lane) * 4 + (pos & 3)]; }
    __device__ void children(int t, K c[4]) const
    {
        const K* src = g + ((t + 1) * 32 + lane) * 4;
        if constexpr (sizeof(K) == 4) {
            const uint4 v = *(const uint4*)src;
            c[0] = v.x; c[1] = v.y; c[2] = v.z; c[3] = v.w;
        } else {
            const ulonglong2 a = *(const ulonglong2*)src, b = *(const ulonglong2*)(src + 2);
            c[0] = a.x; c[1] = a.y; c[2] = b.x; c[3] = b.y;
        }
    }
    // zero the positions after node n-1 up to the end of its group
    __device__ void clear_tail(int n) const
    {
        for (int pos = n + 3; pos <= ((n + 2) | 3); ++pos) g[((pos >> 2) * 32 + lane) * 4 + (pos & 3)] = K(0);
    }
    // sift key down from node t of a heap of n nodes
    __device__ void sift(int t, int n, K key) const
    {
        while (4 * t + 1 < n) {
            K c[4];
            children(t, c);
            K m = c[0];
            int j = 0;
            if (c[1] > m) { m = c[1]; j = 1; }
            if (c[2] > m) { m = c[2]; j = 2; }
            if (c[3] > m) { m = c[3]; j = 3; }
            if (!(m > key)) break;
            at(t) = m;
            t = 4 * t + 1 + j;
        }
        at(t) = key;
    }
    // as sift, for a heap whose storage past node n-1 holds stale keys
    __device__ void sift_masked(int t, int n, K key) const
    {
        while (4 * t + 1 < n) {
            K c[4];
            children(t, c);
            if (4 * t + 2 >= n) c[1] = K(0);
            if (4 * t + 3 >= n) c[2] = K(0);
            if (4 * t + 4 >= n) c[3] = K(0);
            K m = c[0];
            int j = 0;
            if (c[1] > m) { m = c[1]; j = 1; }
            if (c[2] > m) { m = c[2]; j = 2; }
            if (c[3] > m) { m = c[3]; j = 3; }
            if (!(m > key)) break;
            at(t) = m;
            t = 4 * t + 1 + j;
        }
        at(t) = key;
    }
    __device__ void heapify(int n) const
    {
        for (int t = (n - 2) / 4; t >= 0; --t) sift(t, n, at(t));
    }
};

template <class K>
__host__ __device__ constexpr int heap4_groups(int kcap) { return (kcap + 2) / 4 + 1; }

// pending heap insertions per lane (a tile adds at most its masked candidates,
// so the lists are merged before a tile that could overflow one)
constexpr int kPend = 32;
static_assert(kPend >= kLeaf, "a tile can admit all of its candidates: one empty pending list must hold them");
// Defaults of the launch knobs (sidm_config; none changes a result): query
// groups of 32 / G consecutive lanes whose boxes filter the candidates,
// independent distance chains in the candidate loop, the pending count at
// which the lists are merged before a tree node's tests, and the warm-start
// bound factor (previous kernel size times it); values the autotuner picks on
// the GB300 for the 2^20 NFW halo at N_ngb = 64 (with the fixed-bound warm
// kernel: 1.47 ms per search at a bound of 1.07, 1.52 ms at 1.05)
constexpr int kGroupsDefault = 2;
// compacted candidate batches (knob knn_batch): candidates that pass the group
// filter are appended to a per-warp buffer and the distance loop runs over
// batches of kBatch of them; the buffer holds a batch's leftover (< kBatch)
// plus one whole leaf
constexpr int kBatch = 16;
constexpr int kBufCap = kBatch + kLeaf;
static_assert(kPend >= kBatch, "a batch can admit all of its candidates: one empty pending list must hold them");
constexpr int kChainsDefault = 4;
constexpr int kBatchDefault = 3;                   // 1: loop per staged leaf, 2: compacted batches, 3: 2 + fixed-bound warm kernel
constexpr int kFlushNodeDefault = 32;
constexpr float kGuessSlackDefault = 1.07f;

template <class R>
__device__ __forceinline__ float to_float_ru(R v)
{
    if constexpr (sizeof(R) == 8) return __double2float_ru((double)v);
    else return (float)v;
}

// shared memory of one warp: staged tile (shifted in place) | ids | traversal
// stack | heap groups | pending keys (the child boxes of a node live in
// registers, one per lane); 14.1 KB at N_ngb = 64 in the mixed form, so 16
// warps fit on an SM
template <class R, class K, int G, bool BATCH = false>
__host__ __device__ constexpr size_t knn_warp_bytes_t(int kcap)
{
    // the batch buffer takes the place of the staged tile and its ids
    return ((BATCH ? (size_t)kBufCap * sizeof(typename Vec4<R>::T) : TileStageT<R, false, 1>::bytes() + 32 * 4) +
            kStack * 4 + 2 * G * 16 +
            (size_t)heap4_groups<K>(kcap) * 32 * 4 * sizeof(K) + (size_t)kPend * 32 * sizeof(K) + 15) / 16 * 16;
}

static_assert((TileStageT<float, false, 1>::bytes() + 32 * 4 + kStack * 4) % 16 == 0 &&
                  (TileStageT<double, false, 1>::bytes() + 32 * 4 + kStack * 4) % 16 == 0 &&
                  (kBufCap * 16 + kStack * 4) % 16 == 0,
              "the heap groups are read as 16-byte vectors");
template <class R, bool NBR, bool TMA, int G, int CH, bool BATCH>
__global__ void k_knn(KnnParams p)
{
    static_assert(G == 2 || G == 4 || G == 8, "lane groups are 16, 8 or 4 lanes");
    static_assert(CH == 4 || CH == 8, "four or eight independent distance chains");
    static_assert(!(BATCH && TMA), "compacted batches read candidates straight into registers");
    using V = typename Vec4<R>::T;
    using K = typename KeyOf<R, NBR>::T;
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned char* base = smem + wid * knn_warp_bytes_t<R, K, G, BATCH>(p.kcap);
    TileStageT<R, TMA, 1> stage(base);
    V* bufv = (V*)base;                            // BATCH: [kBufCap] candidates (w: slot, or id with NBR)
    uint32_t* tids = (uint32_t*)(base + TileStageT<R, TMA, 1>::bytes());
    int* stack = BATCH ? (int*)(base + (size_t)kBufCap * sizeof(V)) : (int*)(tids + 32);
    float4* gbox = (float4*)(stack + kStack);      // [G][2]: box lo, hi of each lane group
    K* heapg = (K*)(gbox + 2 * G);                 // 16-byte aligned: 528 + 128 + 4 kStack bytes in, + boxes
    K* pend = heapg + (size_t)heap4_groups<K>(p.kcap) * 32 * 4;   // [kPend][32]
    const Heap4<K> hp{heapg, lane};
    stage.init(lane);
    unsigned long long n_cand = 0ull, n_ins = 0ull, n_tiles_all = 0ull, n_tiles_max = 0ull, n_redo = 0ull;

    while (true) {
        int leaf = 0;
        if (lane == 0) leaf = (int)atomicAdd(p.work, 1u);
        leaf = __shfl_sync(0xffffffffu, leaf, 0);
        if (p.leaf_list) {
            if ((unsigned)leaf >= *p.list_len) break;
            leaf = p.leaf_list[leaf];
        } else if (leaf >= p.L) {
            break;
        }
        const int h = p.leaf_halo[leaf];
        const int k = p.ngb[h];
        const int leaf0 = p.leaf_off[h];
        const int nleaf = p.leaf_off[h + 1] - leaf0;
        const int64_t hb = p.halo_off[h];
        const int64_t nh = p.halo_off[h + 1] - hb;
        const int A = leaf - leaf0;
        const int countA = (int)min((int64_t)kLeaf, nh - (int64_t)A * kLeaf);
        const bool active = lane < countA;
        const HaloFrame fr = p.frame[h];
        const V q = ((const V*)p.P4)[(int64_t)leaf * kLeaf + lane];
        // a buffered candidate's w holds its slot (its id with NBR), so the query
        // recognises itself
        const uint32_t own = NBR ? (BATCH && active ? p.ID[(int64_t)leaf * kLeaf + lane] : 0u)
                                 : (uint32_t)leaf * kLeaf + lane;
        const float4 cA = p.cell[leaf];
        const float4 qlo = p.nlo[leaf], qhi = p.nhi[leaf];
        unsigned long long n_tiles = 0ull;
        bool failed = false;
        // Warm start: q.w holds the particle's kernel size of the previous call.
        // Pass 0 starts with the bound key of (h_prev * slack)^2, so only
        // candidates inside that bound enter; a lane that collects fewer than k
        // of them is redone by the cold pass 1 (Morton-window fill, unbounded
        // start).  In both passes the first k admitted keys are stored unsorted
        // and heapified once.
        const bool guess = p.use_guess && active && q.w > R(0);
        K bound_key = ~K(0);
        if (guess) {
            R r;
            if constexpr (sizeof(R) == 4) r = __fmul_ru((float)q.w, p.slack);
            else r = __dmul_ru((double)q.w, (double)p.slack);
            bound_key = make_key<R, NBR>(mul_ru(r, r), 0xFFFFFFFFu);
        }
        K result = K(0);
        bool todo = active;
        for (int pass = __any_sync(0xffffffffu, guess) ? 0 : 1; pass < 2; ++pass) {
        const bool act = pass == 0 ? guess : todo;
        if (!__any_sync(0xffffffffu, act)) break;
        hp.clear_tail(k);
        K root = (pass == 0 && act) ? bound_key : ~K(0);
        int nfill = 0, np = 0;                         // heap fill level, pending keys
        bool heaped = false;

        int nbuf = 0;                                  // BATCH: candidates in the buffer
        // merge the pending keys of every lane into its heap (each lane works
        // on its own heap column; no lane reads another's)
        auto flush = [&]() {
            if (!heaped && nfill == k) {               // the heap array is full: order it once
                hp.heapify(k);
                root = hp.at(0);
                heaped = true;
            }
            for (int i = 0; i < np; ++i) {
                const K key = pend[i * 32 + lane];
                if (key < root) {
                    ++n_ins;
                    hp.sift(0, k, key);
                    root = hp.at(0);
                }
            }
            np = 0;
        };

        float3 pq;                                     // query point in the halo frame
        if constexpr (sizeof(R) == 4) {
            pq = make_float3(__fadd_rn(cA.x, (float)q.x), __fadd_rn(cA.y, (float)q.y), __fadd_rn(cA.z, (float)q.z));
        } else {
            pq = make_float3(__double2float_rn(((double)q.x - fr.O[0]) * fr.down),
                             __double2float_rn(((double)q.y - fr.O[1]) * fr.down),
                             __double2float_rn(((double)q.z - fr.O[2]) * fr.down));
        }
        // boxes of the query points of each group of 32 / G consecutive
        // lanes (shared memory): a candidate is kept if it lies within the
        // largest bound of some group's lanes from that group's box (the union is
        // tighter than the whole leaf's box; the mask stays warp-uniform)
        constexpr int kGL = 32 / G;
        {
            float lx = active ? pq.x : INFINITY, ly = active ? pq.y : INFINITY, lz = active ? pq.z : INFINITY;
            float ux = active ? pq.x : -INFINITY, uy = active ? pq.y : -INFINITY, uz = active ? pq.z : -INFINITY;
            for (int o = kGL / 2; o > 0; o >>= 1) {
                lx = fminf(lx, __shfl_xor_sync(0xffffffffu, lx, o));
                ly = fminf(ly, __shfl_xor_sync(0xffffffffu, ly, o));
                lz = fminf(lz, __shfl_xor_sync(0xffffffffu, lz, o));
                ux = fmaxf(ux, __shfl_xor_sync(0xffffffffu, ux, o));
                uy = fmaxf(uy, __shfl_xor_sync(0xffffffffu, uy, o));
                uz = fmaxf(uz, __shfl_xor_sync(0xffffffffu, uz, o));
            }
            __syncwarp();
            if (lane % kGL == 0) {
                gbox[2 * (lane / kGL)] = make_float4(lx, ly, lz, 0.f);
                gbox[2 * (lane / kGL) + 1] = make_float4(ux, uy, uz, 0.f);
            }
            __syncwarp();
        }
        auto my_r2 = [&]() -> float {
            if (!act) return -1.0f;
            R rr = sqrt_ru(key_d2<R, NBR>(root));
            if constexpr (sizeof(R) == 8) rr *= fr.down;   // to the halo's FP32 unit
            float r = to_float_ru<R>(rr);
            r = __fadd_ru(__fmul_ru(r, 1.0f + 0x1p-20f), fr.margin);
            return __fmul_ru(r, r);
        };
        // this lane's entry of candidate leaf Bl and the leaf's frame origin (the
        // plain path loads both straight into registers, so a caller can fetch
        // the next leaf early; the shift needs the origin as soon as the entry)
        struct Fetched { V c; float4 cell; };
        auto fetch = [&](int Bl) -> Fetched {
            Fetched f{};
            if constexpr (!TMA) f.c = ((const V*)p.P4)[(int64_t)(leaf0 + Bl) * kLeaf + lane];
            if constexpr (sizeof(R) == 4) f.cell = p.cell[leaf0 + Bl];
            return f;
        };
        // the largest bound of each lane group (r2g) and of all lanes (r2all),
        // from each lane's bound r2 (my_r2); an unbounded lane (its heap not yet
        // full in the cold pass) counts as infinite
        struct GroupBounds { float g[G]; float all; };
        auto group_bounds = [&](float r2, bool mine) -> GroupBounds {
            float lr2 = -1.f;
            if (act && mine) lr2 = isnan(r2) ? INFINITY : r2;
            for (int o = kGL / 2; o > 0; o >>= 1) lr2 = fmaxf(lr2, __shfl_xor_sync(0xffffffffu, lr2, o));
            GroupBounds b;
            b.all = -1.f;
#pragma unroll
            for (int g = 0; g < G; ++g) {
                b.g[g] = __shfl_sync(0xffffffffu, lr2, g * kGL);
                b.all = fmaxf(b.all, b.g[g]);
            }
            return b;
        };
        // BATCH: the distances from every active query to the first nb buffered
        // candidates (CH independent chains), admitted like the per-leaf loop
        // below; the entries after them move to the front
        auto run_batch = [&](int nb) {
            if (__any_sync(0xffffffffu, np + nb > kPend)) flush();
            __syncwarp();
            if (act) {
                n_cand += (unsigned long long)nb;
                for (int t = 0; t < nb; t += CH) {
                    K key[CH];
                    bool ok[CH];
#pragma unroll
                    for (int u = 0; u < CH; ++u) {
                        const int idx = t + u < nb ? t + u : t;
                        const V cj = bufv[idx];
                        const uint32_t who = sizeof(R) == 4 ? __float_as_uint((float)cj.w) : (uint32_t)(double)cj.w;
                        const R dx = sub_rn(cj.x, q.x), dy = sub_rn(cj.y, q.y), dz = sub_rn(cj.z, q.z);
                        const R d2 = fma_rn(dz, dz, fma_rn(dy, dy, mul_rn(dx, dx)));
                        key[u] = make_key<R, NBR>(d2, who);
                        ok[u] = t + u < nb && who != own;
                    }
#pragma unroll
                    for (int u = 0; u < CH; ++u) {
                        if (ok[u] && key[u] < root) {
                            if (nfill < k) hp.at(nfill++) = key[u];
                            else pend[(np++) * 32 + lane] = key[u];
                        }
                    }
                }
            }
            __syncwarp();
            const int rem = nbuf - nb;                 // < 32
            V tmp{};
            if (lane < rem) tmp = bufv[nb + lane];
            __syncwarp();
            if (lane < rem) bufv[lane] = tmp;
            nbuf = rem;
            __syncwarp();
        };
        auto drain = [&]() {
            if constexpr (BATCH) { if (nbuf > 0) run_batch(nbuf); }
        };
        // mine: this lane's query reaches leaf Bl; gb: group_bounds of the lanes'
        // bounds; craw: fetch(Bl) (unused on the bulk-copy path, which stages the
        // leaf here)
        auto process = [&](int Bl, bool mine, const GroupBounds& gb, const Fetched& craw) {
            const int Bg = leaf0 + Bl;
            const int countB = (int)min((int64_t)kLeaf, nh - (int64_t)Bl * kLeaf);
            V c;
            if constexpr (TMA) c = stage.load_lane((const V*)p.P4 + (int64_t)Bg * kLeaf, lane, p.cnt);
            else c = craw.c;
            // shift the candidates into the query leaf's frame (exact shift)
            if constexpr (sizeof(R) == 4) {
                const float4 cB = craw.cell;
                c.x = __fadd_rn(c.x, __fsub_rn(cB.x, cA.x));
                c.y = __fadd_rn(c.y, __fsub_rn(cB.y, cA.y));
                c.z = __fadd_rn(c.z, __fsub_rn(cB.z, cA.z));
            }
            // candidates farther from a lane group's box than the largest bound of
            // its lanes cannot enter one of their heaps: the loops skip the
            // candidates no group can reach (an unbounded lane, before its heap is
            // full in the cold pass, keeps them all)
            const float r2all = gb.all;
            uint32_t cmask;
            if (!(r2all < INFINITY)) {
                cmask = countB == kLeaf ? 0xffffffffu : ((1u << countB) - 1u);
            } else {
                float3 pc;                             // candidate in the halo frame
                if constexpr (sizeof(R) == 4) {
                    pc = make_float3(__fadd_rn(cA.x, c.x), __fadd_rn(cA.y, c.y), __fadd_rn(cA.z, c.z));
                } else {
                    pc = make_float3(__double2float_rn(((double)c.x - fr.O[0]) * fr.down),
                                     __double2float_rn(((double)c.y - fr.O[1]) * fr.down),
                                     __double2float_rn(((double)c.z - fr.O[2]) * fr.down));
                }
                bool reach = false;
#pragma unroll
                for (int g = 0; g < G; ++g)
                    reach = reach || (gb.g[g] >= 0.f && point_gap2_rd(pc, gbox[2 * g], gbox[2 * g + 1]) <= gb.g[g]);
                cmask = __ballot_sync(0xffffffffu, lane < countB && reach);
            }
            ++n_tiles;
            if (cmask == 0u) return;                   // no candidate of this leaf can enter
            if constexpr (BATCH) {
                // append the candidates that pass to the buffer, in lane order
                if ((cmask >> lane) & 1u) {
                    V e = c;
                    const uint32_t who = NBR ? p.ID[(int64_t)Bg * kLeaf + lane] : (uint32_t)Bg * kLeaf + lane;
                    if constexpr (sizeof(R) == 4) e.w = __uint_as_float(who); else e.w = (R)who;
                    bufv[nbuf + __popc(cmask & ((1u << lane) - 1u))] = e;
                }
                nbuf += __popc(cmask);
                __syncwarp();
                while (nbuf >= kBatch) run_batch(kBatch);
                return;
            }
            // room for this tile's candidates in every pending list
            if (__any_sync(0xffffffffu, np + __popc(cmask) > kPend)) flush();
            __syncwarp();
            V* sh = stage.shifted();
            sh[lane] = c;
            if (NBR) tids[lane] = p.ID[(int64_t)Bg * kLeaf + lane];
            __syncwarp();
            if (act && mine) {
                n_cand += (unsigned long long)__popc(cmask);
                // the masked candidates CH at a time (independent distance
                // chains); an admitted key fills the heap array (unsorted, heapified
                // at the next merge) until it holds k keys, then waits in the
                // pending list, for which room was made before the tile
                for (uint32_t mm = cmask; mm;) {
                    int t[CH];
#pragma unroll
                    for (int u = 0; u < CH; ++u) { t[u] = __ffs(mm) - 1; mm &= mm - 1u; }   // -1: none left
                    K key[CH];
#pragma unroll
                    for (int u = 0; u < CH; ++u) {
                        const V cj = sh[t[u] >= 0 ? t[u] : t[0]];
                        const R dx = sub_rn(cj.x, q.x), dy = sub_rn(cj.y, q.y), dz = sub_rn(cj.z, q.z);
                        const R d2 = fma_rn(dz, dz, fma_rn(dy, dy, mul_rn(dx, dx)));
                        key[u] = make_key<R, NBR>(d2, NBR ? tids[t[u] >= 0 ? t[u] : t[0]] : 0u);
                    }
#pragma unroll
                    for (int u = 0; u < CH; ++u) {
                        if (t[u] >= 0 && key[u] < root && !(Bl == A && t[u] == lane)) {
                            if (nfill < k) hp.at(nfill++) = key[u];
                            else pend[(np++) * 32 + lane] = key[u];
                        }
                    }
                }
            }
            __syncwarp();
        };

        // 1) cold pass: Morton-window leaves around A holding at least k+1 particles
        int wlo = 0, whi = -1;
        if (pass == 1) {
            wlo = A; whi = A;
            int64_t wcount = countA;
            while (wcount < k + 1 && (wlo > 0 || whi < nleaf - 1)) {
                if (whi < nleaf - 1) { ++whi; wcount += min((int64_t)kLeaf, nh - (int64_t)whi * kLeaf); }
                if (wcount < k + 1 && wlo > 0) { --wlo; wcount += kLeaf; }
            }
            // the window holds at least k other particles, so every lane's heap is
            // full after it: order it and merge the window's keys beyond the first k
            for (int Bl = wlo; Bl <= whi; ++Bl) process(Bl, true, group_bounds(my_r2(), true), fetch(Bl));
            drain();
            flush();
        }

        // 2) tree walk.  A node is visited iff the query point of some lane lies
        //    within that lane's current k-th distance (+ margin) of the node's box;
        //    accepted leaves are processed at once so the bound keeps shrinking.
        // the boxes of the children being tested, one per lane, in registers
        float4 clo = make_float4(0.f, 0.f, 0.f, 0.f), chi = clo;
        auto load_boxes = [&](int g0, int n) {
            if (lane < n) { clo = p.nlo[g0 + lane]; chi = p.nhi[g0 + lane]; }
        };
        // this lane's query within r2 of child c's box (every lane takes part)
        auto near_child = [&](int c, float r2) -> bool {
            const float4 lo = make_float4(__shfl_sync(0xffffffffu, clo.x, c), __shfl_sync(0xffffffffu, clo.y, c),
                                          __shfl_sync(0xffffffffu, clo.z, c), 0.f);
            const float4 hi = make_float4(__shfl_sync(0xffffffffu, chi.x, c), __shfl_sync(0xffffffffu, chi.y, c),
                                          __shfl_sync(0xffffffffu, chi.z, c), 0.f);
            return r2 >= 0.f && point_gap2_rd(pq, lo, hi) <= r2;
        };
        // bit c: the query of some lane lies within its bound of box c; the
        // lane's own bits and bound are kept for the leaves of this node.
        // Every query point lies in the query leaf's box, so a child farther
        // from that box than the largest lane bound is out of reach of every
        // lane: one box test per child (a lane each) leaves the per-lane
        // point tests to the children that pass it.
        uint32_t lane_bits = 0u;
        float node_r2 = -1.0f;
        auto accept = [&](int n, float r2, uint32_t skip) -> uint32_t {
            float r2max = r2;
            for (int o = 16; o > 0; o >>= 1) r2max = fmaxf(r2max, __shfl_xor_sync(0xffffffffu, r2max, o));
            const uint32_t near =
                __ballot_sync(0xffffffffu, lane < n && box_gap2_rd(qlo, qhi, clo, chi) <= r2max) & ~skip;
            uint32_t bits = 0u;
            for (uint32_t m = near; m; m &= m - 1u) {
                const int c = __ffs(m) - 1;
                if (near_child(c, r2)) bits |= 1u << c;
            }
            lane_bits = bits;
            node_r2 = r2;
            return __reduce_or_sync(0xffffffffu, bits);
        };
        // leaves of the Morton window among local leaves first .. first+n-1
        auto window_mask = [&](int first, int n) -> uint32_t {
            const int lo = max(wlo - first, 0), hi = min(whi - first, n - 1);
            if (lo > hi) return 0u;
            return ((2u << hi) - 1u) & ~((1u << lo) - 1u);
        };
        // the warm pass's bound barely moves, so a leaf reuses the lane's node test
        // (a larger, older bound only admits more); the cold pass re-tests with the
        // bound its nearer leaves have shrunk
        auto visit_leaf = [&](int Bl, int c) {
            const float r2 = my_r2();
            const bool mine = near_child(c, r2);
            if (__any_sync(0xffffffffu, mine)) process(Bl, mine, group_bounds(r2, mine), fetch(Bl));
        };
        // Accepted children are visited nearest first (box gap to the query leaf),
        // so the k-th bound shrinks early.  rank = position among the accepted.
        auto order_rank = [&](uint32_t acc, int n) -> int {
            const bool mine_acc = lane < n && ((acc >> lane) & 1u);
            const float pr = mine_acc ? box_gap2_rd(qlo, qhi, clo, chi) : INFINITY;
            int rank = 0;
            for (int j = 0; j < n; ++j) {
                const float pj = __shfl_sync(0xffffffffu, pr, j);
                if ((acc >> j) & 1u) rank += (pj < pr || (pj == pr && j < lane)) ? 1 : 0;
            }
            return rank;
        };
        // the warm pass starts from a tight bound, so it takes the accepted
        // children in index order; the cold pass visits the nearest first
        auto visit_leaves_in_order = [&](uint32_t acc, int n, int first_local) {
            if (acc == 0u) return;
            if (pass == 0) {
                // index order; the next accepted leaf is fetched before this one is
                // processed, so its load overlaps this leaf's candidate loop.  Every
                // leaf of the node reuses the lanes' node-test bounds, so the group
                // bounds of a lane set are formed once per node (a lane whose query
                // misses a leaf only widens the mask, never narrows it)
                uint32_t m = acc;
                int c = __ffs(m) - 1;
                m &= m - 1u;
                Fetched cur = fetch(first_local + c);
                const GroupBounds gb = group_bounds(node_r2, lane_bits != 0u);
                while (true) {
                    const int cn = __ffs(m) - 1;       // -1: none left
                    m &= m - 1u;
                    Fetched nxt{};
                    if (cn >= 0) nxt = fetch(first_local + cn);
                    const bool mine = (lane_bits >> c) & 1u;
                    if (__any_sync(0xffffffffu, mine)) process(first_local + c, mine, gb, cur);
                    if (cn < 0) break;
                    c = cn;
                    cur = nxt;
                }
                return;
            }
            const int rank = order_rank(acc, n);
            const int cnt = __popc(acc);
            for (int r = 0; r < cnt; ++r) {
                const uint32_t m = __ballot_sync(0xffffffffu, lane < n && ((acc >> lane) & 1u) && rank == r);
                const int c = __ffs(m) - 1;
                visit_leaf(first_local + c, c);
            }
        };
        auto push_in_order = [&](uint32_t acc, int n, int lev, int first_local, int& sp) -> bool {
            const int rank = pass == 0 ? __popc(acc & ((1u << lane) - 1u)) : order_rank(acc, n);
            const int cnt = __popc(acc);
            if (sp + cnt > kStack) return false;
            if (lane < n && ((acc >> lane) & 1u)) stack[sp + cnt - 1 - rank] = (lev << 24) | (first_local + lane);
            sp += cnt;
            __syncwarp();
            return true;
        };
        const int top = p.top[h];
        const int32_t* loff = p.lvl_off;
        const int Hp = p.H + 1;
        int sp = 0;
        {
            const int nb = loff[top * Hp + h];
            const int ntop = loff[top * Hp + h + 1] - nb;   // at most kArity
            load_boxes(nb, ntop);
            const uint32_t acc = accept(ntop, my_r2(), top == 0 ? window_mask(0, ntop) : 0u);
            if (top == 0) visit_leaves_in_order(acc, ntop, 0);
            else if (!push_in_order(acc, ntop, top, 0, sp)) failed = true;
        }
        while (sp > 0 && !failed) {
            const int e = stack[--sp];
            __syncwarp();
            const int lev = e >> 24, idx = e & 0xFFFFFF;
            const int cl = lev - 1;
            const int cb = loff[cl * Hp + h];
            const int cc = loff[cl * Hp + h + 1] - cb;
            const int first = idx * kArity;
            const int nch = min(kArity, cc - first);
            // tighten the bounds before the node tests once enough keys wait
            if (__any_sync(0xffffffffu, np >= p.flush_node)) flush();
            load_boxes(cb + first, nch);
            const uint32_t acc = accept(nch, my_r2(), cl == 0 ? window_mask(first, nch) : 0u);
            if (cl == 0) visit_leaves_in_order(acc, nch, first);
            else if (!push_in_order(acc, nch, cl, first, sp)) failed = true;
        }
        drain();
        flush();
        if (act && heaped) { result = root; todo = false; }
        if (pass == 0 && act && todo) ++n_redo;
        }   // passes
        if (failed && lane == 0) raise_status(p.cnt, SIDM_DEV_STACK);
        n_tiles_all += n_tiles;
        n_tiles_max = n_tiles > n_tiles_max ? n_tiles : n_tiles_max;

        // 3) outputs
        if (active) {
            const int64_t u = hb + (int64_t)A * kLeaf + lane;
            const R hval = sqrt_rn(key_d2<R, NBR>(result));
            if (p.h_out) {
                ((R*)p.h_out)[u] = hval;
                ((R*)((V*)p.P4 + (int64_t)leaf * kLeaf + lane))[3] = hval;
                if (p.hprev) ((R*)p.hprev)[u] = hval;
            }
            if constexpr (NBR) {
                // heap sort: repeatedly move the maximum behind the shrinking heap
                for (int end = k - 1; end > 0; --end) {
                    const K top_key = hp.at(0);
                    const K last = hp.at(end);
                    hp.at(end) = top_key;
                    hp.sift_masked(0, end, last);
                }
                for (int t = 0; t < k; ++t) p.nbr[u * p.k_stride + t] = (uint32_t)(hp.at(t) & 0xFFFFFFFFull);
            }
        }
        __syncwarp();
    }
    // diagnostics: tiles, lane-level candidates, heap insertions, worst leaf
    for (int o = 16; o > 0; o >>= 1) {
        n_cand += __shfl_xor_sync(0xffffffffu, n_cand, o);
        n_ins += __shfl_xor_sync(0xffffffffu, n_ins, o);
        n_redo += __shfl_xor_sync(0xffffffffu, n_redo, o);
    }
    if (lane == 0) {
        atomicAdd(&p.cnt->diag[0], n_tiles_all);
        atomicAdd(&p.cnt->diag[1], n_cand);
        atomicAdd(&p.cnt->diag[2], n_ins);
        atomicMax(&p.cnt->diag[3], n_tiles_max);
        if (n_redo) atomicAdd(&p.cnt->diag[7], n_redo);
    }
    stage.finish(lane, p.cnt);
}

// ---------------------------------------------------------------------------
// Fixed-bound search.  From the second call on every particle carries its
// previous kernel size, and only candidates inside slack x h_prev are admitted
// (reading C14); a first call takes a density guess instead (k_knn_guess).  The
// same walk collects neighbour lists and the moments of the local diagnostics
// inside the kernel size itself.  One warp per query leaf (or, with few leaves, the warps of a
// CTA share a leaf's candidate leaves and the first merges their keys); the
// bound is fixed for the whole leaf, so:
//  * the queries are taken in runs of lanes whose box is at most kWSpread(Team)
//    times their largest bound wide (nearly always one run; consecutive particles of
//    the Morton curve can lie on opposite sides of the halo);
//  * the tree is walked with the run's box grown by its largest bound; accepted
//    leaves are listed and loaded two at a time;
//  * a candidate is kept if it lies within the largest bound of the box, a test
//    made in the query leaf's own frame, and goes to a per-warp ring;
//  * batches of kWBatch ring entries are tested against all 32 queries, two per
//    packed FP32 operation, with branch-free admission: a lane stores every key
//    at its next free slot and advances the slot only for a key below its bound.
// The keys of a lane sit in shared memory as [slot][lane], the first kk of them
// a 4-ary max-heap once it is ordered, up to kWPend further ones waiting behind.
//
// The mixed form's keys are the canonical distances and kk = N_ngb.  The FP64
// form searches with FP32 offsets too (S4: offset to the leaf's cell corner, in
// units of 2^HaloFrame::E, w = a bound of the offset's error) and keeps kk = N_ngb + kWExtra keys with their
// slots; distances in FP64 are formed only for the candidates whose FP32 distance
// lies so near the N_ngb-th that rounding could change their order (one or two).
//
// A lane that admits fewer than N_ngb keys (its guess was too small) tries again
// with a wider bound.  A leaf goes to a list that the per-lane search (k_knn,
// warm-started after a warm start, failing lanes cold) then redoes when its
// particles have no previous kernel size, when they would take more than kWRuns
// runs, when kWAttempts bounds did not do, when the tree walk's stack overflows, or
// when the FP32 order of the FP64 form does not settle it (more than kWBand
// candidates within the error, or one that was not kept); so the result is the same
// exact k-th distance as a cold search.  A leaf that has streamed tiles_max candidate
// leaves (an outlier whose kernel reaches the centre: thousands, on one warp, while
// the SMs idle) is started anew by a team, in a launch of its own.
//
// Issue-bound and, with 10 to 15 warps per SM (their keys fill the shared memory),
// latency-bound.  Per search, this launch and the redo's together: 2^20 NFW halo,
// N_ngb = 64: 1.11 ms (1.60 ms with group boxes, one leaf and one candidate at a
// time, and spread leaves and failed guesses left to the redo, which alone took
// 0.37 ms); FP64 form 2.2 ms (11.6 ms with every distance in FP64).  Eight halos of
// 1500 to 30000 particles, N_ngb up to 128: 0.50 ms (0.98); 2048 particles 40 us
// (84), teams; FP64 16384 particles 0.22 ms (4.4).  kWSpread 2, 2.5, 3, 4: 1.15,
// 1.11, 1.12, 1.20 ms at 2^20 and 0.47, 0.58, 0.60, 0.64 ms for the eight halos.
// A first search, 300,007 NFW particles, N_ngb = 48: 0.62 ms with the guess
// (0.78 before long leaves went to teams) against 2.5 ms in the per-lane kernel
// (whose heaps fill from the Morton window, 20 of 32 lanes active); 100,003
// Hernquist particles with their lists 1.36 ms (1.55).  Neighbour lists there
// 0.45 ms (1.87 in the per-lane kernel);
// moments of the 300,007 particles 0.57 ms (1.74 ms over in-range pairs, with ten
// FP64 atomics each).
// Boxes of four lane groups in wide runs: 1.36 ms; runs of a leaf dealt out to the
// team's warps instead of shared by them: 0.42 against 0.22 ms (FP64, 16384).
constexpr int kWRing = 128;     // candidate ring entries
constexpr int kWBatch = 8;      // candidates per batch (batches start at multiples of it: never wrap)
constexpr int kWList = 64;      // accepted leaves listed before they are streamed
constexpr int kWPend = 32;      // keys a lane may hold beyond kk before a merge (room enough that
                                // merges are rare and most lanes order their heaps together)
constexpr int kWExtra = 4;      // FP64 form: keys kept beyond N_ngb
constexpr int kWBand = 4;       // FP64 form: candidates compared in FP64
static_assert((kWRing & (kWRing - 1)) == 0 && kWRing >= kWBatch - 1 + 2 * kLeaf, "the ring holds a batch's leftover plus two leaves");
static_assert(kWPend >= kWBatch, "one batch fits after a merge");
constexpr int kWarmMaxWarps = 8;   // the kernel's launch bound: 256 threads, two CTAs per SM
constexpr int kWAttempts = 8;      // bounds tried, each 1.1 to 3 times the one before, before the redo
// Runs of a leaf at most; a leaf of more goes to the redo.  Leaves of NFW and Hernquist
// halos take three at most with sizes near theirs; with guesses ten times too small
// each lane is a run: 100,000 Hernquist particles 2.76 ms with runs and attempts
// without limit, 0.95 through the redo.  4 instead of 8: 45.3 against 44.1 ms for the
// 64-halo batch, whose halos of few, far particles have leaves of five.
constexpr int kWRuns = 8;
// Candidate leaves one warp streams for a leaf; one that wants more goes to a team.
// 200,003 Hernquist particles, N_ngb = 128: 3.64 ms with one warp throughout, 1.43
// with 512, but the eight halos above 0.58 ms with 512 against 0.54 with 1024.  A first
// search has more of them: neighbours of the 100,003 particles 1.28, 1.36, 1.62,
// 1.97 ms with 192, 384, 768, 1024, first sizes of the 300,007 0.74, 0.62, 0.62, 0.62.
constexpr unsigned kWTiles = 1024, kWTilesGuess = 384;   // (from a density guess)
// widest box of a run of queries / its largest bound: a run costs a walk, a wide
// box reaches dense regions that none of its queries does; a team shares both
constexpr float kWSpread = 2.25f, kWSpreadTeam = 3.0f;

// what a fixed-bound search collects: the kernel size, the neighbour list within
// it, or the kernel-weighted moments of the neighbours within it (mixed form)
constexpr int kSizes = 0, kLists = 1, kMoments = 2;

template <class R, int MODE>
__host__ __device__ constexpr size_t warm_warp_bytes(int kcap)
{
    using K = typename KeyOf<R, MODE == kLists>::T;
    return (size_t)kWRing * (sizeof(K) == 8 || MODE == kMoments ? 16 : 12) + 4 * 16 + (size_t)(kWList + kStack + 32) * 4 +
           (size_t)(kcap + (sizeof(R) == 8 ? kWExtra : 0) + kWPend) * 32 * sizeof(K);
}

template <class R, bool TEAM, int MODE>
__global__ void __launch_bounds__(kWarmMaxWarps * 32, 2) k_knn_warm(KnnParams p, int32_t* redo_list, unsigned int* redo_len)
{
    constexpr bool NBR = MODE == kLists;
    using K = typename KeyOf<R, NBR>::T;
    using V = typename Vec4<R>::T;
    constexpr bool kF32 = sizeof(R) == 4;
    static_assert(MODE == kSizes || kF32, "lists and moments: mixed form");
    constexpr bool kTag = sizeof(K) == 8;              // keys carry the slot (FP64 form) or the id (neighbour lists)
    constexpr bool kRingTag = kTag || MODE == kMoments;   // moments keep slots alone
    constexpr unsigned FULL = 0xffffffffu;
    constexpr unsigned kRow = 32 * sizeof(K);          // bytes of one slot of all lanes
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int team_leaf;
    __shared__ unsigned int team_bad, team_stop, team_fail, team_err;
    __shared__ float team_rad[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int nw = TEAM ? (int)(blockDim.x >> 5) : 1, part = TEAM ? wid : 0;   // nw: a power of two
    const size_t warp_bytes = warm_warp_bytes<R, MODE>(p.kcap);
    unsigned char* base = smem + wid * warp_bytes;
    float* ring = (float*)base;                        // [3 or 4][kWRing] x, y, z (and the tag)
    // the run's box: lo (w: squared reach of the walk), hi (halo frame), centre,
    // half widths (leaf frame)
    float4* wbox = (float4*)(ring + (kRingTag ? 4 : 3) * kWRing);
    int* list = (int*)(wbox + 4);
    int* stack = list + kWList;
    int* held = stack + kStack;                        // [32] keys of this warp's lanes (TEAM)
    unsigned char* keys = (unsigned char*)(held + 32); // [kk + kWPend][32]
    const float4* __restrict__ S4 = (const float4*)p.S4;
    const V* P4 = (const V*)p.P4;
    const uint32_t lt = (1u << lane) - 1u;
    const int Hp = p.H + 1;
    unsigned long long n_cand = 0ull, n_ins = 0ull, n_tiles = 0ull, n_tiles_max = 0ull, n_again = 0ull;

    while (true) {
        int leaf = 0;
        if constexpr (TEAM) {
            __syncthreads();
            if (threadIdx.x == 0) {
                int next = (int)atomicAdd(p.work, 1u);
                if (p.leaf_list) next = (unsigned)next < *p.list_len ? p.leaf_list[next] : p.L;
                team_leaf = next;
                team_bad = team_fail = team_err = 0u;
            }
            __syncthreads();
            leaf = team_leaf;
        } else {
            if (lane == 0) leaf = (int)atomicAdd(p.work, 1u);
            leaf = __shfl_sync(FULL, leaf, 0);
        }
        if (leaf >= p.L) break;
        const int h = p.leaf_halo[leaf];
        const int k = p.ngb[h];
        const int kk = kF32 ? k : k + kWExtra;
        const int leaf0 = p.leaf_off[h];
        const uint32_t nh = (uint32_t)(p.halo_off[h + 1] - p.halo_off[h]);   // n_max < 2^31
        const int A = leaf - leaf0;
        const bool active = (uint32_t)A * kLeaf + lane < nh;
        const uint32_t slotA = (uint32_t)leaf * kLeaf + lane;
        const float4 q = S4[slotA];
        const R hp = P4[slotA].w;
        const unsigned long long tiles0 = n_tiles;
        // a particle without a previous kernel size sends its leaf to the redo
        // (moments: a particle without an extent has no neighbours inside it)
        bool bad = MODE != kMoments && __any_sync(FULL, active && !(hp > R(0))), too_long = false;
        const float margin = p.frame[h].margin;
        const float4 cA = p.cell[leaf];
        // the lane's bound: slack h_prev rounded up
        float rad = 0.f;
        if (active) {
            if constexpr (MODE == kMoments) rad = (float)hp;
            else if constexpr (kF32) rad = __fmul_ru((float)hp, p.slack);
            else rad = __double2float_ru(__dmul_ru((double)hp * p.frame[h].down, (double)p.slack));
        }
        uint32_t todo = bad ? 0u : __ballot_sync(FULL, active);
        const float px = __fadd_rn(cA.x, q.x), py = __fadd_rn(cA.y, q.y), pz = __fadd_rn(cA.z, q.z);
        bool act = false;
        float w[7];
        auto box = [&]() {                                   // of the act lanes: lo, -hi, -largest bound
            w[0] = act ? px : INFINITY;  w[1] = act ? py : INFINITY;  w[2] = act ? pz : INFINITY;
            w[3] = act ? -px : INFINITY; w[4] = act ? -py : INFINITY; w[5] = act ? -pz : INFINITY;
            w[6] = act ? -rad : INFINITY;
        };
        auto widest = [&]() {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
                for (int i = 0; i < 7; ++i) w[i] = fminf(w[i], __shfl_xor_sync(FULL, w[i], o));
            }
        };
        auto wide = [&]() {
            return fmaxf(fmaxf(-w[3] - w[0], -w[4] - w[1]), -w[5] - w[2]) > (TEAM ? kWSpreadTeam : kWSpread) * -w[6];
        };
        // act: the next run of the lanes left
        auto next_run = [&](uint32_t left) {
            act = (left >> lane) & 1u;
            box();
            widest();
            if (!wide()) return;                             // the same in every lane
            // boxes of the lanes up to this one: the run ends before the first that is too wide
            box();
            for (int o = 1; o < 32; o <<= 1) {
#pragma unroll
                for (int i = 0; i < 7; ++i) {
                    const float y = __shfl_up_sync(FULL, w[i], o);
                    if (lane >= o) w[i] = fminf(w[i], y);
                }
            }
            const uint32_t over = __ballot_sync(FULL, act && wide());
            if (over) act = act && lane < __ffs(over) - 1;
        };
        // a leaf no wider than two of the cells that order it is taken whole (in a core
        // denser than the cells, leaves lie on one another, and each run would load them
        // all), another of more than kWRuns runs goes to the redo, which takes all its
        // lanes through one walk
        act = (todo >> lane) & 1u;
        box();
        widest();
        bool whole = !wide() || fmaxf(fmaxf(-w[3] - w[0], -w[4] - w[1]), -w[5] - w[2]) <= 2.f * p.frame[h].fine;
        if (!whole && MODE != kMoments) {
            uint32_t left = todo;
            for (int r = 0; r < kWRuns && left; ++r) {
                next_run(left);
                left &= ~__ballot_sync(FULL, act);
            }
            if (left) { bad = true; todo = 0u; }
        }
        while (todo) {
        if (whole) act = (todo >> lane) & 1u;
        else next_run(todo);
        todo &= ~__ballot_sync(FULL, act);
        // a lane that admits fewer than N_ngb keys tries again with a wider bound
        int found = 0;                                 // keys of the last attempt
        for (int attempt = 0;; ++attempt) {
        uint32_t root = act ? __float_as_uint(MODE == kMoments ? __fmul_rn(rad, rad) : __fmul_ru(rad, rad)) : 0u;   // bits of the lane's d^2 bound
        float err = 0.f;                               // FP64 form: largest offset error of a candidate
        // the filter's bound follows the lanes': squared, or for the FP64 form, which
        // adds a candidate's error, plain
        float rf = 0.f;
        auto reach = [&]() {
            const float r = sqrtf(__uint_as_float(__reduce_max_sync(FULL, root))) * (1.0f + 0x1p-17f);
            rf = kF32 ? r * r : r;
            const float rw = __fadd_ru(r, margin);
            __syncwarp();
            if (lane == 0) wbox[0].w = __fmul_ru(rw, rw);    // and the walk's
            __syncwarp();
        };
        {
            box();
            widest();
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
                wbox[1] = make_float4(-w[3], -w[4], -w[5], 0.f);
                // centre and half widths; with c = RN(x - centre) the computed gap
                // |c| - half of a point x exceeds the true one by less than 2^-22 (gap +
                // half), which the factors here and on the bound cover
                const float cx = 0.5f * (f[0] - f[3]), cy = 0.5f * (f[1] - f[4]), cz = 0.5f * (f[2] - f[5]);
                const float s = 1.0f + 0x1p-18f;
                wbox[2] = make_float4(-cx, -cy, -cz, 0.f);
                wbox[3] = make_float4(s * fmaxf(-f[3] - cx, cx - f[0]), s * fmaxf(-f[4] - cy, cy - f[1]),
                                      s * fmaxf(-f[5] - cz, cz - f[2]), 0.f);
            }
            __syncwarp();
            reach();
        }
        // the query, negated, in both halves; lanes outside the run admit nothing
        const unsigned long long qx2 = pack2(-q.x, -q.x), qy2 = pack2(-q.y, -q.y), qz2 = pack2(-q.z, -q.z);
        const unsigned off0 = (unsigned)sizeof(K) * lane;
        unsigned off = off0;                           // end of the lane's keys (bytes)
        const unsigned room = off0 + kRow * (unsigned)(kk + kWPend - kWBatch);
        bool heaped = false, dropped = false;
        double mom[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
        auto at = [&](int t) -> K& { return *(K*)(keys + off0 + kRow * (unsigned)t); };
        auto sift = [&](int t, K key) {
            while (true) {
                const int c0 = 4 * t + 1;
                if (c0 >= kk) break;
                K m = at(c0);
                int j = c0;
#pragma unroll
                for (int u = 1; u < 4; ++u) {
                    const K c = c0 + u < kk ? at(c0 + u) : K(0);
                    if (c > m) { m = c; j = c0 + u; }
                }
                if (!(m > key)) break;
                at(t) = m;
                t = j;
            }
            at(t) = key;
        };
        auto bits = [](K key) -> uint32_t { if constexpr (kTag) return (uint32_t)(key >> 32); else return key; };
        // moments: the waiting neighbours of every lane, added up in FP64
        auto gather = [&]() {
            const V* V4 = (const V*)p.V4;
            const R m = (R)p.mass[h], hq = (R)rad;
            const R norm = R(8.0 / 3.14159265358979323846) / (hq * hq * hq);
            for (unsigned o = off0; o < off; o += kRow) {
                const uint32_t sj = *(const uint32_t*)(keys + o);
                const V pj = P4[sj], vj = V4[sj];
                const float4 cj = p.cell[sj / kLeaf];
                const R dx = sub_rn(__fadd_rn(pj.x, __fsub_rn(cj.x, cA.x)), q.x), dy = sub_rn(__fadd_rn(pj.y, __fsub_rn(cj.y, cA.y)), q.y),
                        dz = sub_rn(__fadd_rn(pj.z, __fsub_rn(cj.z, cA.z)), q.z);
                const R d = sqrt_rn(fma_rn(dz, dz, fma_rn(dy, dy, mul_rn(dx, dx))));
                const R t = d / hq, u = R(1) - t;
                const R w = t < R(0.5) ? norm * (R(1) - R(6) * t * t * u) : norm * R(2) * u * u * u;
                const double wt = (double)(m * w), vx = (double)vj.x, vy = (double)vj.y, vz = (double)vj.z;
                mom[0] = __dadd_rn(mom[0], wt);
                mom[1] = __fma_rn(wt, vx, mom[1]);
                mom[2] = __fma_rn(wt, vy, mom[2]);
                mom[3] = __fma_rn(wt, vz, mom[3]);
                mom[4] = __fma_rn(wt, __fma_rn(vx, vx, __fma_rn(vy, vy, __dmul_rn(vz, vz))), mom[4]);
            }
            off = off0;
        };
        // merge the waiting keys into the heap (each lane its own column)
        auto flush = [&]() {
            if constexpr (MODE == kMoments) { gather(); __syncwarp(); return; }
            const int cnt = (int)((off - off0) / kRow);
            if (cnt >= kk) {
                if (!heaped) {
                    for (int t = (kk - 2) / 4; t >= 0; --t) sift(t, at(t));
                    heaped = true;
                }
                for (int i = kk; i < cnt; ++i) {
                    const K key = at(i);
                    if (key < at(0)) {
                        ++n_ins;
                        sift(0, key);
                    }
                }
                dropped = dropped || cnt > kk;
                root = min(root, bits(at(0)) + (kTag ? 1u : 0u));   // tagged keys: equal FP32 distances still enter
                off = off0 + kRow * (unsigned)kk;
            }
            reach();
        };

        // the accepted children of a node: local leaf indices into the list (this
        // part's share), or nodes onto the stack
        int nl = 0, sp = 0;
        if (part == 0) { if (lane == 0) list[0] = A; nl = 1; }   // the query leaf first
        __syncwarp();
        auto visit = [&](int lev, int first, int nb, int n) {
            float4 lo = make_float4(INFINITY, INFINITY, INFINITY, 0.f), hi = lo;
            const bool in = lane < n && !(lev == 0 && first + lane == A);
            if (in) { lo = p.nlo[nb + first + lane]; hi = p.nhi[nb + first + lane]; }
            const float4 qlo = wbox[0];
            uint32_t acc = __ballot_sync(FULL, in && box_gap2_rd(qlo, wbox[1], lo, hi) <= qlo.w);
            if (lev == 0) {
                // a team's leaves are dealt by number: its warps' bounds, and so the
                // leaves they accept, differ once keys have been merged
                const bool mine = ((acc >> lane) & 1u) && ((first + lane) & (nw - 1)) == part;
                acc = __ballot_sync(FULL, mine);
                if (mine) list[nl + __popc(acc & lt)] = first + lane;
                nl += __popc(acc);
            } else if (sp + __popc(acc) > kStack) {
                bad = true;
            } else {
                sp += __popc(acc);
                if ((acc >> lane) & 1u) stack[sp - 1 - __popc(acc & lt)] = (lev << 24) | (first + lane);
            }
            __syncwarp();
        };
        const int top = p.top[h];
        bool started = false;
        // ring entries: candidate numbers cnum .. cnum + navail - 1; entries of the
        // query leaf still in the ring, and this lane's own number
        int navail = 0, nself = 0, li = 0;
        uint32_t cnum = 0u;
        while (true) {
            bool fin = false;
            if (li < nl) {
                // two listed leaves: shift, filter, append to the ring
                const int Bl[2] = {list[li], list[min(li + 1, nl - 1)]};
                float4 c[2], cB[2];
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    c[u] = S4[(uint32_t)(leaf0 + Bl[u]) * kLeaf + lane];
                    cB[u] = p.cell[leaf0 + Bl[u]];
                }
                const float4 fc = wbox[2], fw = wbox[3];
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    c[u].x = __fadd_rn(c[u].x, __fsub_rn(cB[u].x, cA.x));     // exact shift into the query leaf's frame
                    c[u].y = __fadd_rn(c[u].y, __fsub_rn(cB[u].y, cA.y));
                    c[u].z = __fadd_rn(c[u].z, __fsub_rn(cB[u].z, cA.z));
                    const float gx = fmaxf(fabsf(c[u].x + fc.x) - fw.x, 0.f), gy = fmaxf(fabsf(c[u].y + fc.y) - fw.y, 0.f),
                                gz = fmaxf(fabsf(c[u].z + fc.z) - fw.z, 0.f);
                    const float re = rf + c[u].w, r2 = kF32 ? rf : re * re;
                    // the query leaf's entries all stay: their numbers are their lanes
                    const bool self = u == 0 && Bl[0] == A;
                    const bool keep = (uint32_t)Bl[u] * kLeaf + lane < nh && li + u < nl &&
                                      (gx * gx + gy * gy + gz * gz <= r2 || self);
                    const uint32_t m = __ballot_sync(FULL, keep);
                    if (self) nself = __popc(m);
                    if constexpr (!kF32) err = fmaxf(err, keep ? c[u].w : 0.f);
                    if (keep) {
                        float* e = ring + ((cnum + navail + __popc(m & lt)) & (kWRing - 1));
                        e[0] = c[u].x; e[kWRing] = c[u].y; e[2 * kWRing] = c[u].z;
                        const uint32_t slot = (uint32_t)(leaf0 + Bl[u]) * kLeaf + lane;
                        if constexpr (kRingTag) e[3 * kWRing] = __uint_as_float(NBR ? p.ID[slot] : slot);
                    }
                    navail += __popc(m);
                }
                n_tiles += (unsigned long long)min(2, nl - li);
                li += 2;
                __syncwarp();
            } else if (!started || sp > 0) {
                // walk until the list may not hold another node's leaves, or the tree is done
                if (!TEAM && (unsigned)(n_tiles - tiles0) > p.tiles_max) { bad = too_long = true; break; }
                nl = li = 0;
                if (!started) {
                    const int nb = p.lvl_off[top * Hp + h];
                    visit(top, 0, nb, p.lvl_off[top * Hp + h + 1] - nb);
                    started = true;
                }
                while (sp > 0 && nl <= kWList - kArity && !bad) {
                    const int e = stack[--sp];
                    __syncwarp();
                    const int cl = (e >> 24) - 1, first = (e & 0xFFFFFF) * kArity;
                    const int cb = p.lvl_off[cl * Hp + h];
                    visit(cl, first, cb, min(kArity, p.lvl_off[cl * Hp + h + 1] - cb - first));
                }
            } else {
                // at the very end fill the partial batch with infinitely far entries
                fin = true;
                const int fill = (kWBatch - navail % kWBatch) % kWBatch;
                if (lane < fill) {
                    float* e = ring + ((cnum + navail + lane) & (kWRing - 1));
                    e[0] = INFINITY; e[kWRing] = INFINITY; e[2 * kWRing] = INFINITY;
                }
                navail += fill;
                __syncwarp();
            }
            if (bad) break;
            while (navail >= kWBatch) {
                if (__any_sync(FULL, off > room)) flush();
                const bool own = nself > 0;
                const int me = own ? lane - (int)cnum : -1;   // this lane's own entry in the batch
#pragma unroll
                for (int t = 0; t < kWBatch; t += 4) {
                    const float* e = ring + (cnum & (kWRing - 1)) + t;
                    const ulonglong2 x = *(const ulonglong2*)e, y = *(const ulonglong2*)(e + kWRing),
                                     z = *(const ulonglong2*)(e + 2 * kWRing);
                    uint4 sl = make_uint4(0u, 0u, 0u, 0u);
                    if constexpr (kRingTag) sl = *(const uint4*)(e + 3 * kWRing);
                    const uint32_t s4[4] = {sl.x, sl.y, sl.z, sl.w};
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        const unsigned long long dx = add2(u ? x.y : x.x, qx2), dy = add2(u ? y.y : y.x, qy2),
                                                 dz = add2(u ? z.y : z.x, qz2);
                        const unsigned long long d2 = fma2(dz, dz, fma2(dy, dy, mul2(dx, dx)));
                        const uint32_t db[2] = {(uint32_t)d2, (uint32_t)(d2 >> 32)};
#pragma unroll
                        for (int r = 0; r < 2; ++r) {
                            const int i = t + 2 * u + r;
                            if constexpr (!kTag) *(uint32_t*)(keys + off) = MODE == kMoments ? s4[2 * u + r] : db[r];
                            else *(unsigned long long*)(keys + off) = ((unsigned long long)db[r] << 32) | s4[2 * u + r];
                            off += db[r] < root && i != me ? kRow : 0u;
                        }
                    }
                }
                if (act) n_cand += kWBatch;
                cnum += kWBatch;
                navail -= kWBatch;
                nself -= kWBatch;
                __syncwarp();
            }
            if (fin) break;
        }
        if (too_long) break;
        if constexpr (MODE == kMoments) {
            // the warps' moments, added in order by the first
            gather();
            __syncwarp();                                      // the sums go where other lanes' queued slots were
            double* part_mom = (double*)(keys) + lane;         // [5][32], the queue is empty
            for (int i = 0; TEAM && i < 5; ++i) part_mom[32 * i] = mom[i];
            if constexpr (TEAM) {
                if (bad && lane == 0) atomicOr(&team_bad, 1u);
                __syncthreads();
                bad = team_bad != 0u;
            }
            if (bad && part == 0 && lane == 0) raise_status(p.cnt, SIDM_DEV_STACK);
            if (part == 0 && act) {
                for (int w = 1; w < nw; ++w)
                    for (int i = 0; i < 5; ++i)
                        mom[i] = __dadd_rn(mom[i], *(const double*)((const unsigned char*)(part_mom + 32 * i) + w * warp_bytes));
                const int64_t u = p.halo_off[h] + (int64_t)slotA - (int64_t)leaf0 * kLeaf;
                for (int i = 0; i < 5; ++i) p.dacc[i * p.nacc + u] = mom[i];
            }
            if constexpr (TEAM) __syncthreads();
            break;
        }
        // the first warp takes over the other warps' keys
        if constexpr (TEAM && MODE != kMoments) {
            flush();
            held[lane] = (int)((off - off0) / kRow);
            if (dropped) held[lane] |= 0x10000;
            if (!kF32) atomicMax(&team_err, __float_as_uint(err));
            if (bad && lane == 0) atomicOr(&team_bad, 1u);
            __syncthreads();
            bad = team_bad != 0u;
            if (!kF32) err = __uint_as_float(team_err);
            if (wid == 0 && !bad) {
                for (int w = 1; w < nw; ++w) {
                    const int hw = *(const int*)((const unsigned char*)(held + lane) + w * warp_bytes);
                    dropped = dropped || (hw & 0x10000);
                    const unsigned char* src = keys + w * warp_bytes + off0;
                    const int most = __reduce_max_sync(FULL, hw & 0xffff);
                    for (int i = 0; i < most; ++i) {
                        if (__any_sync(FULL, off > room)) flush();
                        if (i < (hw & 0xffff)) {
                            const K key = *(const K*)(src + kRow * (unsigned)i);
                            *(K*)(keys + off) = key;
                            off += bits(key) < root ? kRow : 0u;
                            dropped = dropped || bits(key) >= root;
                        }
                    }
                }
            }
        }
        uint32_t fail = 0u;                            // lanes that try again
        if (!bad && part == 0) {
            flush();
            const int n = (int)((off - off0) / kRow);
            bool ok = !act || n >= k, again = !ok;
            R hval = R(0);
            if constexpr (!kF32) {
                // every FP32 distance is within `err` of the exact one
                err = q.w + __uint_as_float(__reduce_max_sync(FULL, __float_as_uint(err))) + 0x1p-19f * rad;
            }
            if constexpr (kF32) {
                if (!NBR && act && ok) hval = sqrt_rn(__uint_as_float(bits(at(0))));
            } else if (act && ok) {
                // the k-th smallest FP32 distance: the (n - k + 1)-th largest of the n kept
                float v[kWExtra + 1];
#pragma unroll
                for (int j = 0; j <= kWExtra; ++j) v[j] = -1.f;
                for (int i = 0; i < n; ++i) {
                    float x = __uint_as_float(bits(at(i)));
#pragma unroll
                    for (int j = 0; j <= kWExtra; ++j) { const float y = fmaxf(v[j], x); x = fminf(v[j], x); v[j] = y; }
                }
                float dk = v[0];
#pragma unroll
                for (int j = 1; j <= kWExtra; ++j) if (n - k == j) dk = v[j];
                // candidates that may come before, or after, the k-th exact distance
                dk = sqrtf(dk);
                const float lo = dk - 2.f * err, hi = dk + 2.f * err;
                const float lo2 = lo > 0.f ? lo * lo * (1.0f - 0x1p-20f) : -1.f, hi2 = hi * hi * (1.0f + 0x1p-20f);
                ok = dropped ? v[0] > hi2 : hi2 < rad * rad * (1.0f - 0x1p-20f);
                again = !ok && !dropped;
                if (ok) {
                    const V qd = P4[slotA];
                    int below = 0, nb = 0;
                    double d2[kWBand];
                    for (int j = 0; j < kWBand; ++j) d2[j] = INFINITY;
                    for (int i = 0; i < n; ++i) {
                        const K key = at(i);
                        const float x = __uint_as_float(bits(key));
                        if (x < lo2) { ++below; continue; }
                        if (x > hi2) continue;
                        const V pj = P4[(uint32_t)key];
                        const double dx = sub_rn((double)pj.x, (double)qd.x), dy = sub_rn((double)pj.y, (double)qd.y),
                                     dz = sub_rn((double)pj.z, (double)qd.z);
                        double e = fma_rn(dz, dz, fma_rn(dy, dy, mul_rn(dx, dx)));
#pragma unroll
                        for (int j = 0; j < kWBand; ++j) { const double y = fmin(d2[j], e); e = fmax(d2[j], e); d2[j] = y; }
                        ++nb;
                    }
                    ok = nb <= kWBand && k - below >= 1 && k - below <= nb;
                    double e = d2[0];
#pragma unroll
                    for (int j = 1; j < kWBand; ++j) if (k - below - 1 == j) e = d2[j];
                    hval = (R)sqrt_rn(e);
                }
            }
            fail = __ballot_sync(FULL, again);
            // the next bound: what holds N_ngb and two standard deviations of its Poisson
            // count at the density that the keys found suggest
            // (three times as far where the last step found nothing more)
            if (again) rad *= attempt > 0 && n == found ? 3.f : fminf(fmaxf(cbrtf(((float)k + 2.f * sqrtf((float)k) + 1.f) / ((float)n + 1.f)), 1.1f), 3.f);
            found = n;
            if (__any_sync(FULL, !ok && !again) || (fail && attempt == kWAttempts - 1)) bad = true;
            if (act && ok) {
                const int64_t u = p.halo_off[h] + (int64_t)slotA - (int64_t)leaf0 * kLeaf;
                if constexpr (NBR) {
                    // heap sort: repeatedly move the maximum behind the shrinking heap
                    for (int end = k - 1; end > 0; --end) {
                        const K top_key = at(0), key = at(end);
                        int t = 0;
                        while (4 * t + 1 < end) {
                            int j = 4 * t + 1;
                            K mk = at(j);
                            for (int c = 4 * t + 2; c < min(4 * t + 5, end); ++c) if (at(c) > mk) { mk = at(c); j = c; }
                            if (!(mk > key)) break;
                            at(t) = mk;
                            t = j;
                        }
                        at(t) = key;
                        at(end) = top_key;
                    }
                    for (int t = 0; t < k; ++t) p.nbr[u * p.k_stride + t] = (uint32_t)at(t);
                } else {
                    ((R*)p.h_out)[u] = hval;
                    if (p.hprev) ((R*)p.hprev)[u] = hval;
                    ((R*)((V*)p.P4 + slotA))[3] = hval;
                }
            }
            if (attempt == 0) n_again += (unsigned long long)__popc(fail);
        }
        if constexpr (TEAM) {
            // written between this attempt's two barriers only (team_bad may be set
            // again by a warp that has begun the next attempt)
            if (wid == 0) {
                team_rad[lane] = rad;
                if (lane == 0) { team_fail = fail; team_stop = bad ? 1u : 0u; }
            }
            __syncthreads();
            fail = team_fail;
            bad = team_stop != 0u;
            rad = team_rad[lane];
        }
        if (bad || fail == 0u) break;
        act = (fail >> lane) & 1u;
        }   // attempts
        if (bad) break;
        }   // runs of queries
        if ((MODE != kMoments || too_long) && bad && part == 0 && lane == 0) {
            const unsigned r = atomicAdd(too_long ? p.long_len : redo_len, 1u);
            (too_long ? p.long_list : redo_list)[r] = leaf;
        }
        n_tiles_max = n_tiles - tiles0 > n_tiles_max ? n_tiles - tiles0 : n_tiles_max;
        __syncwarp();
    }
    for (int o = 16; o > 0; o >>= 1) {
        n_cand += __shfl_xor_sync(FULL, n_cand, o);
        n_ins += __shfl_xor_sync(FULL, n_ins, o);
    }
    if (lane == 0) {
        atomicAdd(&p.cnt->diag[0], n_tiles);
        atomicAdd(&p.cnt->diag[1], n_cand);
        atomicAdd(&p.cnt->diag[2], n_ins);
        atomicMax(&p.cnt->diag[3], n_tiles_max);
        if (n_again) atomicAdd(&p.cnt->diag[7], n_again);
    }
}

void fill_params(sidm_ctx* c, KnnParams& p, void* h_out, uint32_t* nbr, int k_stride, bool use_guess)
{
    const LayoutHost& L = c->lay;
    p.H = L.H; p.L = L.L;
    p.leaf_halo = c->d_leaf_halo; p.leaf_off = c->d_leaf_off; p.halo_off = c->d_halo_off;
    p.lvl_off = c->d_lvl_off; p.top = c->d_top; p.ngb = c->d_ngb; p.frame = c->d_frame;
    p.cell = c->d_cell; p.nlo = c->d_nlo; p.nhi = c->d_nhi; p.P4 = c->d_P4; p.ID = c->d_ID;
    p.S4 = c->cfg.precision == SIDM_FP64 ? (const void*)c->d_S4 : c->d_P4;
    p.h_out = h_out; p.nbr = nbr; p.k_stride = k_stride; p.kcap = c->kmax_cur; p.cnt = c->d_cnt;
    p.work = &c->d_cnt->work[0];
    p.leaf_list = nullptr; p.list_len = nullptr; p.long_list = nullptr; p.long_len = nullptr; p.tiles_max = ~0u;
    p.hprev = nbr ? nullptr : c->d_hprev;
    p.use_guess = use_guess ? 1 : 0;
    p.slack = c->cfg.knn_slack > 0.f ? c->cfg.knn_slack : kGuessSlackDefault;
    p.flush_node = c->cfg.knn_flush > 0 ? c->cfg.knn_flush : kFlushNodeDefault;
}

// warps per CTA: at most the configured number, and of those the one with the
// most resident warps per SM (with large N_ngb the per-warp heaps make two
// small CTAs hold more warps than one large one); a CTA may use at most 227 KB
// of shared memory.  Also the persistent grid.
int pick_shape(sidm_ctx* c, const void* kern, size_t per_warp, int* warps_out, int* grid_out, int max_warps = 16)
{
    int warps = 0, occ = 0;
    for (int w = std::min(c->knn_warps, max_warps); w >= 1; --w) {
        if ((size_t)w * per_warp > (size_t)227 * 1024) continue;
        int o = 0;
        const int rc = occupancy(c, kern, w * 32, (size_t)w * per_warp, &o);
        if (rc) return rc;
        if (o * w > occ * warps) { warps = w; occ = o; }
    }
    if (warps < 1 || occ < 1) return set_err(c, SIDM_ECAPACITY, "knn kernel does not fit on an SM (ngb_max too large)");
    int grid = c->cfg.grid_ctas > 0 ? c->cfg.grid_ctas : c->sm_count * occ;
    grid = std::max(1, std::min(grid, (c->lay.L + warps - 1) / warps));
    *warps_out = warps;
    *grid_out = grid;
    return SIDM_OK;
}

// redo: the leaves the fixed-bound warm kernel listed (their count and the
// work counter were zeroed before it ran)
template <class R, bool NBR, bool TMA, int G, int CH, bool BATCH = false>
int launch_t(sidm_ctx* c, void* h_out, uint32_t* nbr, int k_stride, bool use_guess, cudaStream_t s, bool redo = false)
{
    using K = typename KeyOf<R, NBR>::T;
    KnnParams p;
    fill_params(c, p, h_out, nbr, k_stride, use_guess);
    if (redo) {
        p.leaf_list = c->d_knn_redo;
        p.list_len = &c->d_cnt->knn_redo[0];
        p.work = &c->d_cnt->knn_redo[1];
    }
    auto kern = k_knn<R, NBR, TMA, G, CH, BATCH>;
    const size_t per_warp = knn_warp_bytes_t<R, K, G, BATCH>(p.kcap);
    int warps = 0, grid = 0;
    if (int rc = pick_shape(c, (const void*)kern, per_warp, &warps, &grid)) return rc;
    if (!redo) c->knn_grid = grid;
    cudaError_t e;
    if (!redo) {
        e = cudaMemsetAsync(&c->d_cnt->work[0], 0, sizeof(unsigned int), s);
        if (e != cudaSuccess) return cuda_check(c, e, "knn work reset");
    }
    const int tidx = timer_begin(c, 1, s);
    kern<<<grid, warps * 32, (size_t)warps * per_warp, s>>>(p);
    timer_end(c, tidx, s);
    c->launches++;
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_check(c, e, "knn launch");
    return SIDM_OK;
}

// the plain-load kernel-size search with the configured lane groups, chains
// and candidate loop (per staged leaf, or compacted batches)
template <class R>
int launch_tuned(sidm_ctx* c, void* h_out, bool use_guess, cudaStream_t s, bool redo = false)
{
    const int g = c->cfg.knn_groups > 0 ? c->cfg.knn_groups : kGroupsDefault;
    const int ch = c->cfg.knn_chains > 0 ? c->cfg.knn_chains : kChainsDefault;
    const bool batch = (c->cfg.knn_batch > 0 ? c->cfg.knn_batch : kBatchDefault) >= 2;
#define SIDM_KNN_CASE(GG, CC, BB) \
    if (g == GG && ch == CC && batch == BB) return launch_t<R, false, false, GG, CC, BB>(c, h_out, nullptr, 0, use_guess, s, redo);
    SIDM_KNN_CASE(2, 4, false) SIDM_KNN_CASE(4, 4, false) SIDM_KNN_CASE(8, 4, false) SIDM_KNN_CASE(4, 8, false)
    SIDM_KNN_CASE(2, 4, true) SIDM_KNN_CASE(4, 4, true) SIDM_KNN_CASE(8, 4, true) SIDM_KNN_CASE(4, 8, true)
#undef SIDM_KNN_CASE
    return set_err(c, SIDM_EINVAL, "knn_chains 8 takes knn_groups 4");
}

// warm-started search with the fixed-bound kernel, then the per-lane search
// (itself warm-started: a lane whose guess fails there is redone cold) of the
// leaves it could not finish.  With fewer than kTeamItems leaves per resident
// warp the warps of a CTA share a leaf.
constexpr int64_t kTeamItems = 1;
template <class R, int MODE = kSizes>
int launch_warm(sidm_ctx* c, void* h_out, cudaStream_t s, uint32_t* nbr = nullptr, int k_stride = 0, const double* mass = nullptr,
                bool guessed = false)
{
    constexpr bool NBR = MODE == kLists;
    KnnParams p;
    fill_params(c, p, h_out, nbr, k_stride, true);
    p.V4 = c->d_V4; p.mass = mass; p.dacc = c->d_dacc; p.nacc = c->lay.N;
    if (guessed) p.slack = 1.0f;                   // a density guess (k_knn_guess)
    if (NBR) p.slack = 1.0f + 0x1p-20f;            // the kernel size itself is the bound
    const size_t per_warp = warm_warp_bytes<R, MODE>(p.kcap);
    int warps = 0, grid = 0;
    if (int rc = pick_shape(c, (const void*)k_knn_warm<R, false, MODE>, per_warp, &warps, &grid, kWarmMaxWarps)) return rc;
    int tw = kWarmMaxWarps, occ = 0;                // a team's warps
    while (tw > 1 && (tw > c->knn_warps || (size_t)tw * per_warp > (size_t)226 * 1024)) tw /= 2;
    if (int rc = occupancy(c, (const void*)k_knn_warm<R, true, MODE>, tw * 32, (size_t)tw * per_warp, &occ)) return rc;
    const bool can_team = occ >= 1 && tw > 1;
    const int team_grid = std::max(1, std::min(c->cfg.grid_ctas > 0 ? c->cfg.grid_ctas : c->sm_count * occ, c->lay.L));
    const bool team = can_team && c->lay.L < kTeamItems * grid * warps;
    const unsigned tiles_max = guessed ? kWTilesGuess : kWTiles;
    // a halo of few leaves has none that streams so many of them
    const bool longs = can_team && !team && c->lay.L > (int)tiles_max;
    if (team) { warps = tw; grid = team_grid; }
    c->knn_grid = grid;
    cudaError_t e = cudaMemsetAsync(&c->d_cnt->work[0], 0, sizeof(unsigned int), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(&c->d_cnt->knn_redo[0], 0, 4 * sizeof(unsigned int), s);
    if (e != cudaSuccess) return cuda_check(c, e, "knn work reset");
    const int tidx = MODE == kMoments ? -1 : timer_begin(c, 1, s);
    p.tiles_max = longs ? tiles_max : ~0u;
    if (longs) { p.long_list = c->d_knn_long; p.long_len = &c->d_cnt->knn_redo[2]; }
    if (team) k_knn_warm<R, true, MODE><<<grid, warps * 32, (size_t)warps * per_warp, s>>>(p, c->d_knn_redo, &c->d_cnt->knn_redo[0]);
    else k_knn_warm<R, false, MODE><<<grid, warps * 32, (size_t)warps * per_warp, s>>>(p, c->d_knn_redo, &c->d_cnt->knn_redo[0]);
    c->launches++;
    if (longs) {
        p.leaf_list = c->d_knn_long;
        p.list_len = &c->d_cnt->knn_redo[2];
        p.work = &c->d_cnt->knn_redo[3];
        k_knn_warm<R, true, MODE><<<team_grid, tw * 32, (size_t)tw * per_warp, s>>>(p, c->d_knn_redo, &c->d_cnt->knn_redo[0]);
        c->launches++;
    }
    timer_end(c, tidx, s);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_check(c, e, "knn launch");
    if constexpr (MODE == kMoments) return SIDM_OK;
    else if constexpr (NBR) return launch_t<float, true, false, kGroupsDefault, kChainsDefault>(c, nullptr, nbr, k_stride, false, s, true);
    else return launch_tuned<R>(c, h_out, !guessed, s, true);
}

// A guess for every particle of a search that has no earlier kernel sizes, into
// P4.w: the radius of the kGuessRank-th nearest of the leaf's other particles (of
// the kGuessNear-th where that radius jumps: the leaf holds clumps), scaled to
// N_ngb with two standard deviations of a Poisson count, so that few guesses fail,
// and at most kGuessWide times the leaf's lower quartile for particles near it
// (those at the leaf's rim see a part of their neighbourhood only).  One warp per
// leaf; a wrong guess costs time, never accuracy.
// A guess that holds more than N_ngb particles of the kGuessSpan leaves on either
// side in Morton order is lowered to the radius that holds N_ngb of them: on the
// sparse shell even the quartile can reach across the halo.  In a leaf wider than
// kGuessMixed times the quartile's guess (dense and sparse particles side by side,
// where the quartile is far too small for some) every particle takes that radius, which
// cannot fail: first sizes of 2003 Hernquist particles, N_ngb = 128, 0.56 ms (0.93).
constexpr int kGuessRank = 10, kGuessNear = 4, kGuessSpan = 4;
constexpr float kGuessWide = 1.0f;
constexpr float kGuessMixed = 9.0f;   // about four runs of kWSpread
template <class R>
__global__ void __launch_bounds__(256) k_knn_guess(int L, const int32_t* __restrict__ leaf_halo, const int32_t* __restrict__ leaf_off,
                                                   const int64_t* __restrict__ halo_off, const int32_t* __restrict__ ngb,
                                                   const HaloFrame* __restrict__ frame, const float4* __restrict__ S4,
                                                   const float4* __restrict__ cell, typename Vec4<R>::T* __restrict__ P4)
{
    constexpr unsigned FULL = 0xffffffffu;
    __shared__ float4 window[8][(2 * kGuessSpan + 1) * kLeaf];
    const int lane = threadIdx.x & 31;
    float4* win = window[threadIdx.x >> 5];
    const int leaf = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (leaf >= L) return;                                     // whole warps
    const int h = leaf_halo[leaf];
    const int n = (int)min((int64_t)kLeaf, halo_off[h + 1] - halo_off[h] - (int64_t)(leaf - leaf_off[h]) * kLeaf);
    const float4 q = S4[(int64_t)leaf * kLeaf + lane];
    float d2[kLeaf];
    float hi = 0.f;
#pragma unroll
    for (int t = 0; t < kLeaf; ++t) {
        const float dx = __shfl_sync(FULL, q.x, t) - q.x, dy = __shfl_sync(FULL, q.y, t) - q.y, dz = __shfl_sync(FULL, q.z, t) - q.z;
        d2[t] = t < n ? dx * dx + dy * dy + dz * dz : INFINITY;
        if (t < n) hi = fmaxf(hi, d2[t]);
    }
    // squared radius holding m others (and the particle itself) by bisection on the bits
    auto radius2 = [&](int m) -> float {
        uint32_t lo = 0u, up = __float_as_uint(hi);
        for (int it = 0; it < 20 && up - lo > 1u; ++it) {
            const uint32_t mid = lo + (up - lo) / 2u;
            const float x = __uint_as_float(mid);
            int c = 0;
#pragma unroll
            for (int t = 0; t < kLeaf; ++t) c += d2[t] <= x ? 1 : 0;
            if (c >= m + 1) up = mid; else lo = mid;
        }
        return __uint_as_float(up);
    };
    const int far = min(kGuessRank, max(1, n / 3)), near = min(kGuessNear, far);
    // r^3 per particle, from the far rank or, where that is several times the near one's, from the near
    const float rf = radius2(far), rn = radius2(near);
    const float vf = rf * sqrtf(rf) / (float)far, vn = rn * sqrtf(rn) / (float)near;
    const float v = lane < n ? (vf > 6.f * vn ? 1.5f * vn : vf) : INFINITY;
    float ext = 0.f;                                           // the leaf's width
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float x = a == 0 ? q.x : a == 1 ? q.y : q.z;
        float lo = lane < n ? x : INFINITY, up = lane < n ? x : -INFINITY;
        for (int o = 16; o > 0; o >>= 1) { lo = fminf(lo, __shfl_xor_sync(FULL, lo, o)); up = fmaxf(up, __shfl_xor_sync(FULL, up, o)); }
        ext = fmaxf(ext, up - lo);
    }
    int rank = 0;
    for (int t = 0; t < kLeaf; ++t) {
        const float y = __shfl_sync(FULL, v, t);
        rank += y < v || (y == v && t < lane) ? 1 : 0;
    }
    const uint32_t at = __ballot_sync(FULL, rank == n / 4);
    const float quart = __shfl_sync(FULL, v, __ffs(at) - 1);
    constexpr float wide = kGuessWide * kGuessWide * kGuessWide;
    const float vg = fminf(v, wide * quart);
    const float k = (float)ngb[h];
    float g = cbrtf(vg * (k + 2.f * sqrtf(k) + 1.f)), g2 = g * g;
    // the window, in this leaf's frame
    const int first = max(leaf_off[h], leaf - kGuessSpan), last = min(leaf_off[h + 1] - 1, leaf + kGuessSpan);
    const int64_t end = (int64_t)leaf_off[h] * kLeaf + (halo_off[h + 1] - halo_off[h]);
    const float4 cA = cell[leaf];
    for (int b = first; b <= last; ++b) {
        float4 c = S4[(int64_t)b * kLeaf + lane];
        const float4 cB = cell[b];
        c.x += cB.x - cA.x; c.y += cB.y - cA.y; c.z += cB.z - cA.z;
        if ((int64_t)b * kLeaf + lane >= end) c.x = INFINITY;
        win[(b - first) * kLeaf + lane] = c;
    }
    __syncwarp();
    const int nw = (last - first + 1) * kLeaf;
    auto within = [&](float r2) -> int {
        int c = 0;
#pragma unroll 8
        for (int t = 0; t < nw; ++t) {
            const float4 w = win[t];
            const float dx = w.x - q.x, dy = w.y - q.y, dz = w.z - q.z;
            c += dx * dx + dy * dy + dz * dz <= r2 ? 1 : 0;
        }
        return c;
    };
    const int want = ngb[h] + 1;                               // the particle itself among them
    float low = 0.f, high = g2;
    const bool more = lane < n && within(g2) > want;
    const float gq = cbrtf(wide * quart * (k + 2.f * sqrtf(k) + 1.f));
    if (ext > kGuessMixed * gq) {                              // the same in every lane
        // dense and sparse particles in one leaf: the radius that holds N_ngb of the window
        uint32_t a = 0u, b = __float_as_uint(3.f * ext * ext);
        while (within(__uint_as_float(b)) < want && b < 0x7f000000u) b += 0x1000000u;      // four times the square
        for (int it = 0; it < 12; ++it) {
            const uint32_t mid = a + (b - a) / 2u;
            if (within(__uint_as_float(mid)) >= want) b = mid; else a = mid;
        }
        g = sqrtf(__uint_as_float(b)) * 1.001f;
    } else if (__any_sync(FULL, more)) {
        for (int it = 0; it < 8; ++it) {
            const float mid = 0.5f * (low + high);
            if (within(mid) >= want) high = mid; else low = mid;
        }
        if (more) g = sqrtf(high) * 1.001f;
    }
    if (lane < n) P4[(int64_t)leaf * kLeaf + lane].w = sizeof(R) == 8 ? (R)((double)g * frame[h].up) : (R)g;
}

template <class R>
int launch_guess(sidm_ctx* c, cudaStream_t s)
{
    using V = typename Vec4<R>::T;
    const float4* S4 = c->cfg.precision == SIDM_FP64 ? c->d_S4 : (const float4*)c->d_P4;
    k_knn_guess<R><<<(unsigned)(((int64_t)c->lay.L * 32 + 255) / 256), 256, 0, s>>>(c->lay.L, c->d_leaf_halo, c->d_leaf_off, c->d_halo_off,
                                                                                  c->d_ngb, c->d_frame, S4, c->d_cell, (V*)c->d_P4);
    c->launches++;
    return cuda_check(c, cudaGetLastError(), "knn guess launch");
}

}  // namespace

int launch_knn(sidm_ctx* c, void* h_out, uint32_t* nbr, int k_stride, bool use_guess, cudaStream_t s)
{
    if (c->lay.L == 0) return SIDM_OK;
    const bool tma = c->cfg.use_tma != 0;
    constexpr int G = kGroupsDefault, CH = kChainsDefault;   // neighbour lists and bulk copies: defaults
    // the fixed-bound kernel, from the previous kernel sizes or a density guess,
    // unless the knobs ask for bulk copies or the per-lane kernel (knn_batch 1 or 2)
    const bool fixed = !tma && (c->cfg.knn_batch > 0 ? c->cfg.knn_batch : kBatchDefault) == 3;
    if (c->cfg.precision == SIDM_FP64) {
        if (nbr) return set_err(c, SIDM_EINVAL, "neighbour lists: mixed form only");
        if (fixed) {
            if (!use_guess) { if (int rc = launch_guess<double>(c, s)) return rc; }
            return launch_warm<double>(c, h_out, s, nullptr, 0, nullptr, !use_guess);
        }
        return tma ? launch_t<double, false, true, G, CH>(c, h_out, nullptr, 0, use_guess, s)
                   : launch_tuned<double>(c, h_out, use_guess, s);
    }
    if (nbr && fixed) return launch_warm<float, kLists>(c, nullptr, s, nbr, k_stride);
    if (nbr) return tma ? launch_t<float, true, true, G, CH>(c, nullptr, nbr, k_stride, false, s)
                        : launch_t<float, true, false, G, CH>(c, nullptr, nbr, k_stride, false, s);
    if (fixed) {
        if (!use_guess) { if (int rc = launch_guess<float>(c, s)) return rc; }
        return launch_warm<float>(c, h_out, s, nullptr, 0, nullptr, !use_guess);
    }
    return tma ? launch_t<float, false, true, G, CH>(c, h_out, nullptr, 0, use_guess, s)
               : launch_tuned<float>(c, h_out, use_guess, s);
}

// kernel-weighted moments of every particle's neighbours (local diagnostics, mixed form)
int launch_moments(sidm_ctx* c, const double* mass, cudaStream_t s)
{
    if (c->lay.L == 0) return SIDM_OK;
    return launch_warm<float, kMoments>(c, nullptr, s, nullptr, 0, mass);
}

}  // namespace sidm
