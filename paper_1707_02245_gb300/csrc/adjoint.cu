// Exact transpose K^T of the circular-mean projector (Sec. 3.3.1, Sec. 4.2 eq. (K_def)) by
// pixel tiles with fixed-point accumulation, and the K^T entry points.
#include <algorithm>
#include <initializer_list>

#include "pat_internal.cuh"

namespace pat {

// ---------------------------------------------------------------------------------
// K^T by pixel tiles with exact fixed-point accumulation.
//
// A CTA owns a share of one WTILE x WTILE pixel tile's candidate points.  Its shared
// accumulators (with a one-pixel ring, so every point whose taps touch the tile can add
// all four weights) hold int32 fixed-point values: every pixel satisfies
//   |(K^T y)(p)| <= max|y| * (K^T 1)(p)        (all entries of K are >= 0),
// so with the scale S = 2^30 / (max|y| * max over the ATILE tile of K^T 1) no partial sum
// of a tile pixel exceeds 2^30 and integer addition (native shared atomics, associative,
// hence deterministic) replaces floating-point atomics.  The resolution 2^-30 of that
// bound is finer than FP32 accumulation of the same terms.  Ring cells are dropped.
//
// Work: geometry creation cuts every ray (detector, angle) of a tile's polar box to the
// segment of radii whose points can have taps in the tile, concatenates the segments
// into the tile's candidate list, and cuts the lists into nearly equal work items of whole
// segments that fill one wave of resident CTAs.  Every candidate uses the forward projector's
// FP32 position and tap arithmetic, so the CTA adds exactly the entries of K^T that belong to
// its pixels.  Items of one scale tile share its scale, so their fixed-point tiles add exactly
// (in any order) into one image with integer atomics.
//
// Bound: issue slots and the shared-memory atomics together.  At 256^2 with 256 detectors
// (8.4 M points): 18.2 us per launch, against 26.5 us for a kernel whose threads walked
// contiguous runs of the candidate list one point at a time: there nearly every step of a
// warp held some lane's segment change, and its lanes' pixels lay on random banks (3.6
// wavefronts per atomic, 19 M warp instructions).  64^2 with 64 detectors: 6.0 -> 5.2 us;
// an uneven batch of 8: 77 -> 57 us.  Tiles of 64 pixels with 16 lanes to a segment: 19.2 us.
// ---------------------------------------------------------------------------------
// Threads of a K^T CTA and resident CTAs per SM.  Fewer, larger CTAs zero and flush fewer tile
// copies; the 64 registers of 2 x 512 threads hold the loop without spills (us per launch at
// 256^2 / 64^2: 2 x 512 18.2 / 4.8, 1 x 1024 19.3 / 4.6, 4 x 256 18.7 / 5.3, 3 x 384 18.7 / 5.3).
constexpr int ATHREADS = 512;
constexpr int ADJ_MIN_BLOCKS = 2;
constexpr int ACELL = WTILE + 3;     // cells per axis: the tile, its ring and one more for points outside
constexpr int ACOPY = 48;            // columns from an accumulator to its second copy (16 banks on)
constexpr int AKIND = 96;            // columns to the accumulators of the other kind of segment (0 banks on)
constexpr int ASTRIDE = 192;         // row stride: a multiple of 32 words, so a cell's column alone is its bank
static_assert(ACELL <= ACOPY && ACOPY + ACELL <= AKIND && AKIND + ACOPY + ACELL <= ASTRIDE, "accumulators side by side");
static_assert(ASTRIDE % 32 == 0 && ACOPY % 32 == 16 && AKIND % 32 == 0, "banks of the accumulators");

// One work item of K^T: the ray segments of its records.  ALANES lanes share a segment, each
// with two neighbouring points at a time (their data are one aligned 8-byte load), so a warp
// walks AROWS segments of nearly equal length at once with no segment change inside its loop.
// Each candidate is evaluated with the forward's FP32 point arithmetic, two points per paired
// instruction; a point whose taps fall outside the tile window adds to the cells past the
// ring, which are dropped with it, so the loop has no branch.
//
// Banks: segments that advance fastest along x add to accumulators with x along a row, the
// others to accumulators with y along a row, so the lanes of a segment stand in different
// columns, and with a row stride of a multiple of 32 words the column alone is the bank.
// Every second segment of a warp adds to a copy 16 banks on.  All four accumulators are added
// before the tile leaves the CTA.  Wavefronts per atomic and lanes in use at 256^2: 3.1 and
// 26.6 of 32 without the copies, 2.1 with them (16 lanes to a segment: 1.6 and 23.8).
//
// The order of the products of a tap is that of the axes, not of the kind of segment, so
// tiles and work items of any shape give the same bits.
struct AdjConst {
    float2 dr, rh, scale;
    const float* wk;
    int T;
};

// The points of one segment that this lane takes.  FAST_Y: the row of the accumulator runs
// along y.
template <bool PREMUL, bool FAST_Y>
__device__ __forceinline__ void adjoint_segment(const AdjConst& a, const float4 geo, const float4 seg, const float* __restrict__ y,
                                                int sub2, int bm, int bs, int* cells) {
    const float2 magic = make_float2(FLOOR_MAGIC, FLOOR_MAGIC), nmagic = make_float2(-FLOOR_MAGIC, -FLOOR_MAGIC);
    const float2 one = make_float2(1.f, 1.f), mone = make_float2(-1.f, -1.f);
    const int n = __float_as_int(seg.w);
    const float2 dm = make_float2(geo.x, geo.x), ds = make_float2(geo.y, geo.y);
    const float2 cm = make_float2(geo.z, geo.z), cs = make_float2(geo.w, geo.w);
    const float* __restrict__ yp = y + (size_t)__float_as_uint(PREMUL ? seg.x : seg.y);
    const float k0 = seg.z + (float)sub2;
    float2 kf = make_float2(k0, k0 + 1.f);
    for (int p = sub2; p < n; p += 2 * ALANES) {
        float2 yv;
        if (PREMUL) {
            yv = __ldg(reinterpret_cast<const float2*>(yp + p));
        } else {   // (the caller's array may lie on any 4-byte boundary and its rows have no padding)
            const int k = min((int)seg.z + p, a.T - 1);   // (seg.z may be rounded beyond 2^28)
            yv = make_float2(__ldg(yp + p) * __ldg(a.wk + k), k + 1 < a.T ? __ldg(yp + p + 1) * __ldg(a.wk + k + 1) : 0.f);
        }
        const float2 c = __fmul2_rn(yv, a.scale);
        const float2 r = __ffma2_rn(kf, a.dr, a.rh);   // = rk[k], bit for bit (see radius())
        kf = __fadd2_rn(kf, make_float2(2.f * ALANES, 2.f * ALANES));
        const float2 fm = __ffma2_rn(r, cm, dm), fs = __ffma2_rn(r, cs, ds);
        const float2 tm = __fadd2_rd(fm, magic), ts = __fadd2_rd(fs, magic);   // floor + 1.5 * 2^23, exactly
        const float2 frm = __ffma2_rn(__fadd2_rn(tm, nmagic), mone, fm), frs = __ffma2_rn(__fadd2_rn(ts, nmagic), mone, fs);
        const float2 omm = __ffma2_rn(frm, mone, one), oms = __ffma2_rn(frs, mone, one);
        // taps (c (1 - ay)) (1 - ax), ...
        const float2 c0 = __fmul2_rn(c, FAST_Y ? omm : oms), c1 = __fmul2_rn(c, FAST_Y ? frm : frs);
        const float2 wl = FAST_Y ? oms : omm, wh = FAST_Y ? frs : frm;
        const float2 v00 = __fmul2_rn(c0, wl), v11 = __fmul2_rn(c1, wh);
        const float2 vx = __fmul2_rn(c0, wh), vy = __fmul2_rn(c1, wl);   // the tap further along x, along y
        const float2 v10 = FAST_Y ? vy : vx, v01 = FAST_Y ? vx : vy;     // along the row, across rows
        // tile-local cells straight from the floors' bits
        {
            const unsigned lm = min((unsigned)(__float_as_int(tm.x) - bm), (unsigned)(WTILE + 1));
            const unsigned ls = min((unsigned)(__float_as_int(ts.x) - bs), (unsigned)(WTILE + 1));
            int* t = cells + ls * ASTRIDE + lm;
            atomicAdd(t, __float2int_rn(v00.x));
            atomicAdd(t + 1, __float2int_rn(v10.x));
            atomicAdd(t + ASTRIDE, __float2int_rn(v01.x));
            atomicAdd(t + ASTRIDE + 1, __float2int_rn(v11.x));
        }
        {
            const unsigned lm = min((unsigned)(__float_as_int(tm.y) - bm), (unsigned)(WTILE + 1));
            const unsigned ls = min((unsigned)(__float_as_int(ts.y) - bs), (unsigned)(WTILE + 1));
            int* t = cells + ls * ASTRIDE + lm;
            atomicAdd(t, __float2int_rn(v00.y));
            atomicAdd(t + 1, __float2int_rn(v10.y));
            atomicAdd(t + ASTRIDE, __float2int_rn(v01.y));
            atomicAdd(t + ASTRIDE + 1, __float2int_rn(v11.y));
        }
    }
}

// Maximum of n <= ATHREADS words, in every thread of the CTA.
__device__ __forceinline__ unsigned max_of_slots(const unsigned* slots, int n) {
    __shared__ unsigned s_max[ATHREADS / 32];
    const int tid = threadIdx.x;
    const unsigned v = __reduce_max_sync(0xffffffffu, tid < n ? slots[tid] : 0u);
    if ((tid & 31) == 0) s_max[tid >> 5] = v;
    __syncthreads();
    unsigned m = 0u;
#pragma unroll
    for (int w = 0; w < ATHREADS / 32; ++w) m = max(m, s_max[w]);
    return m;
}

// n_items work items of one tile: item (with SEVERAL: items[0], items[1], ...).  max |y| comes from
// a.ymax_bits, or (n_slots > 0) is the maximum of that many block maxima.
template <bool PREMUL, bool SEVERAL>
__device__ __forceinline__ void adjoint_items(const AdjArgs& a, int item_index, const int* __restrict__ items, int n_items,
                                              const unsigned* slots = nullptr, int n_slots = 0) {
    const int N = a.g.n;
    int4 item = __ldg(reinterpret_cast<const int4*>(a.items + (SEVERAL ? __ldg(items) : item_index)));
    const int tile = item.x;
    int nrec = item.z, split = item.w;
    const int x0 = (tile % a.wtiles_x) * WTILE, y0 = (tile / a.wtiles_x) * WTILE;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    __shared__ __align__(16) int acc[ACELL * ASTRIDE];
    for (int c = tid; c < ACELL * ASTRIDE / 4; c += ATHREADS) reinterpret_cast<int4*>(acc)[c] = make_int4(0, 0, 0, 0);
    constexpr int STEP = ATHREADS / ALANES;      // segments the CTA walks at once
    const int sub2 = 2 * (lane % ALANES);
    int first = warp * AROWS, j = first + lane / ALANES;
    const float4* __restrict__ recs = reinterpret_cast<const float4*>(a.recs + item.y);
    float4 q = make_float4(0.f, 0.f, 0.f, 0.f), s = q;
    if (j < nrec) {
        q = __ldg(recs + 2 * j);
        s = __ldg(recs + 2 * j + 1);
    }
    await_predecessor();
    if (a.stop && *(volatile const int*)a.stop) return;
    // the scale of the ATILE tile that holds this work tile
    const float bound = __uint_as_float(n_slots > 0 ? max_of_slots(after_wait(slots), n_slots) : *after_wait(a.ymax_bits)) * __ldg(&a.tile_kmax[(y0 / ATILE) * a.tiles_x + x0 / ATILE]);
    const float scale = 1073741824.0f / bound;  // 2^30 / bound
    const float* __restrict__ y = after_wait(a.y);
    const AdjConst ac{make_float2(a.g.dr_f, a.g.dr_f), make_float2(a.g.rh_f, a.g.rh_f), make_float2(scale, scale), a.g.wk, a.g.n_t};
    const bool run = bound > 0.f && isfinite(bound);
    __syncthreads();
    if (run) {
        int* cells = acc + (lane / ALANES % 2) * ACOPY;
        const int bx = FLOOR_MAGIC_BITS + x0 - 1, by = FLOOR_MAGIC_BITS + y0 - 1;
        // the next segment is loaded while this one is walked
        auto advance = [&](float4& geo, float4& seg) {
            geo = q;
            seg = s;
            j += STEP;
            first += STEP;
            s.w = 0.f;
            if (j < nrec) {
                q = __ldg(recs + 2 * j);
                s = __ldg(recs + 2 * j + 1);
            }
        };
        float4 geo, seg;
        while (true) {
            while (first < split) {
                advance(geo, seg);
                adjoint_segment<PREMUL, false>(ac, geo, seg, y, sub2, bx, by, cells);
            }
            while (first < nrec) {
                advance(geo, seg);
                adjoint_segment<PREMUL, true>(ac, geo, seg, y, sub2, by, bx, cells + AKIND);
            }
            if (!SEVERAL || --n_items == 0) break;
            item = __ldg(reinterpret_cast<const int4*>(a.items + __ldg(++items)));
            recs = reinterpret_cast<const float4*>(a.recs + item.y);
            nrec = item.z;
            split = item.w;
            first = warp * AROWS;
            j = first + lane / ALANES;
            if (j < nrec) {
                q = __ldg(recs + 2 * j);
                s = __ldg(recs + 2 * j + 1);
            }
        }
    }
    __syncthreads();
    dependents_may_start();
    // the accumulators with x along a row += those with y along a row, along diagonals: a
    // warp's cells lie in 32 different columns of each
    for (int c = tid; c < WTILE * WTILE; c += ATHREADS) {
        const int lx = c % WTILE, ly = (lx + c / WTILE) % WTILE;
        const int* ty = acc + (lx + 1) * ASTRIDE + AKIND + ly + 1;
        acc[(ly + 1) * ASTRIDE + lx + 1] += ty[0] + ty[ACOPY];
    }
    __syncthreads();
    // work items of one tile share its scale, so their fixed-point partial sums add
    // exactly (and in any order) with integer atomics
    for (int c = tid; c < WTILE * WTILE; c += ATHREADS) {
        const int lx = c % WTILE, ly = c / WTILE;
        const int gx = x0 + lx, gy = y0 + ly;
        if (gx >= N || gy >= N) continue;
        const int* t = acc + (ly + 1) * ASTRIDE + lx + 1;
        const int v = t[0] + t[ACOPY];
        if (v) atomicAdd(&a.acc_out[(size_t)gy * N + gx], v);
    }
}

// K^T of one data set: slots hold the block maxima of |y| that k_adjoint_prep leaves; the
// maximum goes to ymax_out for the conversion that follows.
template <bool PREMUL>
__global__ void __launch_bounds__(ATHREADS, ADJ_MIN_BLOCKS) k_adjoint_tiles(const __grid_constant__ AdjArgs a,
                                                                            const unsigned* __restrict__ slots, int n_slots,
                                                                            unsigned* __restrict__ ymax_out) {
    adjoint_items<PREMUL, false>(a, blockIdx.x, nullptr, 1, slots, n_slots);
    if (blockIdx.x == 0) {
        const unsigned m = max_of_slots(slots, n_slots);
        if (threadIdx.x == 0) *ymax_out = m;
    }
    dependents_may_start();
}

// Before K^T of one data set: clears the fixed-point image, leaves each block's max |y| (as
// float bits) in its slot and, when qw is not NULL, writes the data times the arc weights in
// rows of row_stride(T).  One launch instead of a clear and a maximum, and the aligned copy
// serves K^T's paired loads (pat_adjoint, 256^2 with 256 detectors: 36.9 -> 24.6 us per call).
__global__ void __launch_bounds__(512) k_adjoint_prep(const float* __restrict__ y, const float* __restrict__ wk, int D, int T,
                                                      float* __restrict__ qw, int* __restrict__ acc, long long nn,
                                                      unsigned* __restrict__ slots) {
    const long long first = blockIdx.x * (long long)blockDim.x + threadIdx.x, step = (long long)gridDim.x * blockDim.x;
    for (long long i = first; i < nn; i += step) acc[i] = 0;
    unsigned m = 0u;
    const unsigned Tp = row_stride(T);
    // rows padded to an even length: entry k == T of an odd row is zero
    for (long long i = first; i < (long long)D * Tp; i += step) {
        const unsigned d = (unsigned)i / Tp, k = (unsigned)i - d * Tp;   // D * Tp <= 2^32
        float v = 0.f;
        if (k < (unsigned)T) {
            v = __ldg(y + (size_t)d * T + k);
            m = max(m, __float_as_uint(fabsf(v)));
            v *= __ldg(wk + k);
        }
        if (qw) qw[i] = v;
    }
    __shared__ unsigned s_max[16];
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0) s_max[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x < 32) {
        m = __reduce_max_sync(0xffffffffu, threadIdx.x < blockDim.x / 32 ? s_max[threadIdx.x] : 0u);
        if (threadIdx.x == 0) slots[blockIdx.x] = m;
    }
    dependents_may_start();
}

template <bool PREMUL, bool SEVERAL>
__global__ void __launch_bounds__(ATHREADS, ADJ_MIN_BLOCKS) k_adjoint_tiles_b(const AdjArgs* __restrict__ args,
                                                                              const int2* __restrict__ map,
                                                                              const int* __restrict__ list) {
    const int2 pm = map[blockIdx.x];
    const AdjArgs& a = args[adj_map_problem(pm)];   // (a shared copy would be reloaded after every shared atomic)
    adjoint_items<PREMUL, SEVERAL>(a, pm.y, list + pm.y, adj_map_count(pm));
}

// out = the fixed-point K^T image in floating point
__global__ void k_kt_to_float(KtView kt, int N, float* __restrict__ out) {
    const int gx = blockIdx.x * blockDim.x + threadIdx.x, gy = blockIdx.y * blockDim.y + threadIdx.y;
    await_predecessor();
    if (gx >= N || gy >= N) return;
    kt.acc = after_wait(kt.acc);
    kt.ymax_bits = after_wait(kt.ymax_bits);
    out[(size_t)gy * N + gx] = kt.at(gx, gy, N);
}

// max of K^T 1 over each K^T tile, with headroom for the FP32 rounding of the terms
KtView kt_view(const pat_geometry* g, const int* acc, const unsigned* ymax_bits) {
    KtView v;
    v.acc = acc;
    v.ymax_bits = ymax_bits;
    v.tile_kmax = g->pc.tile_kmax;
    v.tiles_x = g->adj_tiles_x;
    return v;
}

AdjArgs make_adj_args(const pat_geometry* g, const float* y, const float* premul, const unsigned* ymax_bits, int* acc,
                      const int* stop) {
    AdjArgs a;
    const GeomView& v = g->view;
    a.g = AdjGeom{v.n, v.n_t, v.wk, v.dr_f, v.rh_f};
    a.y = premul ? premul : y;
    a.premul = premul ? 1 : 0;
    a.ymax_bits = ymax_bits;
    a.tile_kmax = g->pc.tile_kmax;
    a.recs = g->adj_rec;
    a.items = g->adj_item;
    a.acc_out = acc;
    a.tiles_x = g->adj_tiles_x;
    a.wtiles_x = g->adj_wtiles_x;
    a.stop = stop;
    return a;
}

int adjoint_blocks_per_sm() {
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_adjoint_tiles_b<true, true>, ATHREADS, 0) != cudaSuccess || n < 1) {
        cudaGetLastError();
        n = 4;
    }
    return n;
}

// Waves of CTAs a batch's K^T keeps.  A geometry's items fill one wave, so a batch of B has B waves
// of them, and with few candidates an item is mostly its CTA's fixed cost: the chain of loads before
// the first point, and clearing, merging and flushing the accumulators.  Beyond this many waves a
// CTA takes several items of a tile.  us per launch with one item a CTA and with this rule: 64
// problems of 64^2 with 64 detectors 204, 91; 8 of them 26.8, 19.2; 64 of 32^2 with 16 44, 25; 8 of
// 96^2 with 330 171, 74; 16 of 256^2 with 128 139, 121; 8 uneven ones 61.6, 57.0.  2 waves cost 4
// problems of 256^2 with 256 detectors 65.3 against 62.4; 8 waves left the 8 of 64^2 at 26.7.
constexpr int ADJ_BATCH_WAVES = 3;

AdjMap adjoint_map(const pat_geometry* const* g, int B) {
    long long total = 0;
    for (int b = 0; b < B; ++b) total += g[b]->adj_items;
    const int most = (int)std::min<long long>(ADJ_MAP_ITEMS, std::max<long long>(1, total / (ADJ_BATCH_WAVES * g[0]->adj_slots)));
    AdjMap map;
    map.several = most > 1;
    if (B == 1 && !map.several) {   // (a geometry's items are heaviest first)
        map.entries.resize(g[0]->adj_items);
        for (int i = 0; i < g[0]->adj_items; ++i) map.entries[i] = adj_map_entry(0, i, 1);
        return map;
    }
    std::vector<std::pair<float, int2>> v;
    v.reserve((size_t)total);
    for (int b = 0; b < B; ++b) {
        const std::vector<float>& cost = g[b]->adj_item_cost;
        const std::vector<int>&tile = g[b]->adj_item_tile, &by_tile = g[b]->adj_by_tile;
        const int items = g[b]->adj_items;
        for (int i = 0; !map.several && i < items; ++i) v.push_back({cost[i], adj_map_entry(b, i, 1)});
        for (int i = 0, n; map.several && i < items; i += n) {
            for (n = 1; i + n < items && tile[by_tile[i + n]] == tile[by_tile[i]]; ++n) {}
            const int parts = ceil_div(n, most);
            for (int p = 0; p < parts; ++p) {
                const int i0 = i + n * p / parts, i1 = i + n * (p + 1) / parts;
                float sum = 0.f;
                for (int k = i0; k < i1; ++k) sum += cost[by_tile[k]];
                v.push_back({sum, adj_map_entry(b, (int)map.list.size(), i1 - i0)});
                map.list.insert(map.list.end(), by_tile.begin() + i0, by_tile.begin() + i1);
            }
        }
    }
    std::stable_sort(v.begin(), v.end(), [](const std::pair<float, int2>& x, const std::pair<float, int2>& y) { return x.first > y.first; });
    map.entries.reserve(v.size());
    for (const auto& e : v) map.entries.push_back(e.second);
    return map;
}

int launch_adjoint_b(const AdjArgs* args, const int2* map, const int* list, int nblocks, bool several, bool premul,
                     cudaStream_t st) {
    if (nblocks <= 0) return PAT_OK;
    prof_mark(PAT_PHASE_ADJOINT, st, true);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)nblocks);
    cfg.blockDim = dim3(ATHREADS);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    set_dependent_launch(attr[0]);
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    auto kernel = premul ? (several ? k_adjoint_tiles_b<true, true> : k_adjoint_tiles_b<true, false>)
                         : (several ? k_adjoint_tiles_b<false, true> : k_adjoint_tiles_b<false, false>);
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, args, map, list);
    if (e != cudaSuccess) return cuda_fail(e, "k_adjoint_tiles_b");
    PAT_LAUNCH_CHECK("k_adjoint_tiles_b");
    prof_mark(PAT_PHASE_ADJOINT, st, false);
    return PAT_OK;
}

// K^T y through caller-provided scratch: head (a word for the maximum and n_slots for block
// maxima), the fixed-point image acc (N*N int32) and, when not NULL, qw
// (D * row_stride(T) floats, 8-byte aligned).  No allocation and no profiling events.
int launch_adjoint_into(const pat_geometry* g, const float* y, unsigned* head, int n_slots, int* acc, float* qw,
                        float* out, cudaStream_t st) {
    const int N = g->desc.n, D = g->desc.n_det, T = g->desc.n_t;
    const long long work = std::max((long long)N * N, (long long)D * T);
    unsigned *ymax = head, *slots = head + 1;
    n_slots = std::max(1, std::min({n_slots, ATHREADS, 2 * sm_count(), ceil_div(work, 512)}));
    k_adjoint_prep<<<n_slots, 512, 0, st>>>(y, g->view.wk, D, T, qw, acc, (long long)N * N, slots);
    PAT_LAUNCH_CHECK("k_adjoint_prep");
    const AdjArgs a = make_adj_args(g, y, qw, ymax, acc, nullptr);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)g->adj_items);
    cfg.blockDim = dim3(ATHREADS);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    set_dependent_launch(attr[0]);
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const unsigned* cslots = slots;
    cudaError_t e = qw ? cudaLaunchKernelEx(&cfg, k_adjoint_tiles<true>, a, cslots, n_slots, ymax)
                       : cudaLaunchKernelEx(&cfg, k_adjoint_tiles<false>, a, cslots, n_slots, ymax);
    count_launch();
    if (e != cudaSuccess) return cuda_fail(e, "k_adjoint_tiles");
    cfg.gridDim = dim3((unsigned)ceil_div(N, 32), (unsigned)ceil_div(N, 8));
    cfg.blockDim = dim3(32, 8);
    e = cudaLaunchKernelEx(&cfg, k_kt_to_float, kt_view(g, acc, ymax), N, out);
    count_launch();
    return e == cudaSuccess ? PAT_OK : cuda_fail(e, "k_kt_to_float");
}

int launch_adjoint(const pat_geometry* g, const float* y, float* out, cudaStream_t st) {
    int rc = ensure_precond(g, st);
    if (rc) return rc;
    char* scratch = nullptr;
    const size_t head = 4096, acc = ((size_t)g->desc.n * g->desc.n * sizeof(int) + 255) & ~(size_t)255;
    const size_t weighted = (size_t)g->desc.n_det * row_stride(g->desc.n_t) * sizeof(float);
    bool qw = cudaMallocAsync((void**)&scratch, head + acc + weighted, st) == cudaSuccess;
    if (!qw) {   // no room for the weighted data: the kernel weights them itself
        cudaGetLastError();
        PAT_CUDA(cudaMallocAsync((void**)&scratch, head + acc, st));
    }
    rc = launch_adjoint_into(g, y, (unsigned*)scratch, (int)(head / 4) - 1, (int*)(scratch + head),
                             qw ? (float*)(scratch + head + acc) : nullptr, out, st);
    cudaFreeAsync(scratch, st);
    return rc;
}

}  // namespace pat

using namespace pat;

extern "C" int pat_adjoint(const pat_geometry* g, const float* y_dev, float* u_dev, void* stream) {
    if (!g || !u_dev || !y_dev) return fail(PAT_ERR_INVALID_ARG, "pat_adjoint: NULL argument");
    return launch_adjoint(g, y_dev, u_dev, (cudaStream_t)stream);
}
