// Exact transpose K^T of the circular-mean projector (Sec. 3.3.1, Sec. 4.2 eq. (K_def)) by
// pixel tiles with fixed-point accumulation, and the K^T entry points.
#include <algorithm>

#include "pat_internal.cuh"

namespace pat {

// ---------------------------------------------------------------------------------
// K^T by pixel tiles with exact fixed-point accumulation.
//
// A CTA owns a share of one WTILE x WTILE pixel tile's candidate points (WTILE: see
// work_tile_side).  Its shared accumulator (with a one-pixel ring, so every point whose taps
// touch the tile can add all four weights) holds int32 fixed-point values: every pixel satisfies
//   |(K^T y)(p)| <= max|y| * (K^T 1)(p)        (all entries of K are >= 0),
// so with the scale S = 2^30 / (max|y| * max over the work tile of K^T 1) no partial sum
// of a tile pixel exceeds 2^30 and integer addition (native shared atomics, associative,
// hence deterministic) replaces floating-point atomics.  The resolution 2^-30 of that
// bound is finer than FP32 accumulation of the same terms.  Ring cells are dropped.
//
// Work: geometry creation cuts every ray (detector, angle) of a tile's polar box to the
// segment of radii whose points can have taps in the tile, concatenates the segments
// into the tile's candidate list, and cuts the lists into nearly equal work items of whole
// segments that fill one wave of resident CTAs.  Every candidate uses the forward projector's
// FP32 position and tap arithmetic, so the CTA adds exactly the entries of K^T that belong to
// its pixels.  Items of one tile share its scale, so their fixed-point tiles add exactly (in
// any order) into one image with integer atomics.
//
// Bound: issue slots and the shared-memory atomics together.  At 256^2 with 256 detectors
// (8.4 M points): 19.2 us per launch, 2.0 wavefronts per atomic and 14 M warp instructions,
// against 26.5 us, 3.6 and 19 M for a kernel whose threads walked contiguous runs of the
// candidate list one point at a time: there nearly every step of a warp held some lane's
// segment change, and its lanes' pixels lay on random banks.
// ---------------------------------------------------------------------------------
// Threads of a K^T CTA and resident CTAs per SM.  Fewer, larger CTAs zero and flush fewer tile
// copies; the 64 registers of 2 x 512 threads hold the loop without spills (measured at 256^2:
// 2 x 512 19.2 us, 1 x 1024 19.9, 4 x 256 20.5, 3 x 512 with spills 30).
constexpr int ATHREADS = 512;
constexpr int ADJ_MIN_BLOCKS = 2;
constexpr int acell(int side) { return side + 3; }   // cells per axis: the tile, its ring and one more for points outside
constexpr int astride(int side) { return (2 * acell(side) + 31) / 32 * 32; }   // row stride of the accumulators: a cell's bank is its column mod 32

// One work item of K^T: the ray segments of its records.  ALANES lanes share a segment, each
// with two neighbouring points at a time (their data are one aligned 8-byte load), so a warp
// walks AROWS segments of nearly equal length at once with no segment change inside its loop.
// Each candidate is evaluated with the forward's FP32 point arithmetic, two points per paired
// instruction; a point whose taps fall outside the tile window adds to the cells past the
// ring, which are dropped with it, so the loop has no branch.
//
// Two accumulators hold the tile: the first with x along a row, the second with y along a
// row.  A segment adds to the one whose rows run along its fast axis: its lanes then stand in
// different columns, and with a row stride of a multiple of 32 words the column alone is the
// bank.  Both are added before the tile leaves the CTA.
template <bool PREMUL, int WTILE>
__device__ __forceinline__ void adjoint_tile(const AdjArgs& a, int item_index, int* acc) {
    constexpr int ACELL = acell(WTILE), ASTRIDE = astride(WTILE);
    const AdjGeom& g = a.g;
    const int N = g.n;
    const int4 item = __ldg(reinterpret_cast<const int4*>(a.items + item_index));
    const int tile = item.x, nrec = item.z, split = item.w;
    const int x0 = (tile % a.wtiles_x) * WTILE, y0 = (tile / a.wtiles_x) * WTILE;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int c = tid; c < ACELL * ASTRIDE / 4; c += ATHREADS) reinterpret_cast<int4*>(acc)[c] = make_int4(0, 0, 0, 0);
    // the scale of the ATILE tile that holds this work tile
    const float bound = __uint_as_float(*a.ymax_bits) * __ldg(&a.tile_kmax[(y0 / ATILE) * a.tiles_x + x0 / ATILE]);
    const float scale = 1073741824.0f / bound;  // 2^30 / bound
    const float* __restrict__ wk = g.wk;
    const float* __restrict__ y = a.y;
    const int T = g.n_t;
    const float4* __restrict__ recs = reinterpret_cast<const float4*>(a.recs + item.y);
    constexpr int STEP = ATHREADS / ALANES;      // segments the CTA walks at once
    const int sub2 = 2 * (lane % ALANES);
    const float sub2f = (float)sub2;
    int j = warp * AROWS + lane / ALANES;
    const bool run = bound > 0.f && isfinite(bound);
    float4 q = make_float4(0.f, 0.f, 0.f, 0.f), s = q;
    if (run && j < nrec) {
        q = __ldg(recs + 2 * j);
        s = __ldg(recs + 2 * j + 1);
    }
    const float2 dr2 = make_float2(g.dr_f, g.dr_f), rh2 = make_float2(g.rh_f, g.rh_f);
    const float2 magic = make_float2(FLOOR_MAGIC, FLOOR_MAGIC), nmagic = make_float2(-FLOOR_MAGIC, -FLOOR_MAGIC);
    const float2 one = make_float2(1.f, 1.f), mone = make_float2(-1.f, -1.f), scale2 = make_float2(scale, scale);
    __syncthreads();
    if (run) {
        for (int first = warp * AROWS; first < nrec; first += STEP) {
            const float4 geo = q, seg = s;
            j += STEP;
            s.w = 0.f;
            if (j < nrec) {   // the next segment, while this one is walked
                q = __ldg(recs + 2 * j);
                s = __ldg(recs + 2 * j + 1);
            }
            const int n = __float_as_int(seg.w);
            const float2 dm = make_float2(geo.x, geo.x), ds = make_float2(geo.y, geo.y);
            const float2 cm = make_float2(geo.z, geo.z), cs = make_float2(geo.w, geo.w);
            // tile-local cells straight from the floors' bits
            const bool fast_y = first >= split;
            const int bm = FLOOR_MAGIC_BITS + (fast_y ? y0 : x0) - 1, bs = FLOOR_MAGIC_BITS + (fast_y ? x0 : y0) - 1;
            int* cells = acc + (fast_y ? ACELL : 0);
            const float* __restrict__ yp = y + (size_t)__float_as_uint(PREMUL ? seg.x : seg.y);
            float2 kf = make_float2(seg.z + sub2f, seg.z + sub2f + 1.f);
            for (int p = sub2; p < n; p += 2 * ALANES) {
                float2 yv;
                if (PREMUL) {
                    yv = __ldg(reinterpret_cast<const float2*>(yp + p));
                } else {   // (the caller's array may lie on any 4-byte boundary and its rows have no padding)
                    const int k = (int)seg.z + p;
                    yv = make_float2(__ldg(yp + p) * __ldg(wk + k), k + 1 < T ? __ldg(yp + p + 1) * __ldg(wk + k + 1) : 0.f);
                }
                const float2 c = __fmul2_rn(yv, scale2);
                const float2 r = __ffma2_rn(kf, dr2, rh2);   // = rk[k], bit for bit (see radius())
                kf = __fadd2_rn(kf, make_float2(2.f * ALANES, 2.f * ALANES));
                const float2 fm = __ffma2_rn(r, cm, dm), fs = __ffma2_rn(r, cs, ds);
                const float2 tm = __fadd2_rd(fm, magic), ts = __fadd2_rd(fs, magic);   // floor + 1.5 * 2^23, exactly
                const float2 frm = __ffma2_rn(__fadd2_rn(tm, nmagic), mone, fm), frs = __ffma2_rn(__fadd2_rn(ts, nmagic), mone, fs);
                const float2 omm = __ffma2_rn(frm, mone, one), oms = __ffma2_rn(frs, mone, one);
                const float2 c0 = __fmul2_rn(c, oms), c1 = __fmul2_rn(c, frs);
                const float2 v00 = __fmul2_rn(c0, omm), v10 = __fmul2_rn(c0, frm);
                const float2 v01 = __fmul2_rn(c1, omm), v11 = __fmul2_rn(c1, frm);
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
    }
    __syncthreads();
    // the first accumulator += the second transposed, along diagonals: a warp's cells lie in
    // 32 different columns of both
    for (int c = tid; c < WTILE * WTILE; c += ATHREADS) {
        const int lx = c & (WTILE - 1), ly = (lx + c / WTILE) & (WTILE - 1);
        acc[(ly + 1) * ASTRIDE + lx + 1] += acc[(lx + 1) * ASTRIDE + ACELL + ly + 1];
    }
    __syncthreads();
    // work items of one tile share its scale, so their fixed-point partial sums add
    // exactly (and in any order) with integer atomics
    for (int c = tid; c < WTILE * WTILE; c += ATHREADS) {
        const int lx = c % WTILE, ly = c / WTILE;
        const int gx = x0 + lx, gy = y0 + ly;
        if (gx >= N || gy >= N) continue;
        const int v = acc[(ly + 1) * ASTRIDE + lx + 1];
        if (v) atomicAdd(&a.acc_out[(size_t)gy * N + gx], v);
    }
}

template <bool PREMUL>
__device__ __forceinline__ void adjoint_item(const AdjArgs& a, int item_index) {
    __shared__ __align__(16) int acc[acell(WTILE_LARGE) * astride(WTILE_LARGE)];
    if (a.side == WTILE_SMALL)
        adjoint_tile<PREMUL, WTILE_SMALL>(a, item_index, acc);
    else
        adjoint_tile<PREMUL, WTILE_LARGE>(a, item_index, acc);
}

__global__ void __launch_bounds__(ATHREADS, ADJ_MIN_BLOCKS) k_adjoint_tiles(AdjArgs a) {
    adjoint_item<false>(a, blockIdx.x);
}

template <bool PREMUL>
__global__ void __launch_bounds__(ATHREADS, ADJ_MIN_BLOCKS) k_adjoint_tiles_b(const AdjArgs* __restrict__ args,
                                                            const int2* __restrict__ map) {
    const int2 pm = map[blockIdx.x];
    const AdjArgs& a = args[pm.x];   // (a shared copy would be reloaded after every shared atomic)
    if (a.stop && *(volatile const int*)a.stop) return;
    adjoint_item<PREMUL>(a, pm.y);
}

// out = the fixed-point K^T image in floating point
__global__ void k_kt_to_float(KtView kt, int N, float* __restrict__ out) {
    const int gx = blockIdx.x * blockDim.x + threadIdx.x, gy = blockIdx.y * blockDim.y + threadIdx.y;
    if (gx >= N || gy >= N) return;
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
    a.side = g->adj_side;
    a.wtiles_x = g->adj_wtiles_x;
    a.stop = stop;
    return a;
}

int adjoint_blocks_per_sm() {
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_adjoint_tiles_b<true>, ATHREADS, 0) != cudaSuccess || n < 1) {
        cudaGetLastError();
        n = 4;
    }
    return n;
}

int launch_adjoint_b(const AdjArgs* args, const int2* map, int nblocks, bool premul, cudaStream_t st) {
    if (nblocks <= 0) return PAT_OK;
    prof_mark(PAT_PHASE_ADJOINT, st, true);
    if (premul)
        k_adjoint_tiles_b<true><<<nblocks, ATHREADS, 0, st>>>(args, map);
    else
        k_adjoint_tiles_b<false><<<nblocks, ATHREADS, 0, st>>>(args, map);
    PAT_LAUNCH_CHECK("k_adjoint_tiles_b");
    prof_mark(PAT_PHASE_ADJOINT, st, false);
    return PAT_OK;
}

// K^T y through caller-provided scratch: the max word at ymax_bits and the fixed-point
// image at acc (N*N int32), both already zero; no allocation and no profiling events.
int launch_adjoint_into(const pat_geometry* g, const float* y, unsigned* ymax_bits, int* acc, float* out,
                        cudaStream_t st) {
    const int N = g->desc.n;
    const long long S = (long long)g->desc.n_det * g->desc.n_t;
    const int arc = launch_absmax(y, S, ymax_bits, st);
    if (arc) return arc;
    const AdjArgs a = make_adj_args(g, y, nullptr, ymax_bits, acc, nullptr);
    k_adjoint_tiles<<<g->adj_items, ATHREADS, 0, st>>>(a);
    PAT_LAUNCH_CHECK("k_adjoint_tiles");
    dim3 blk(32, 8), grd(ceil_div(N, 32), ceil_div(N, 8));
    k_kt_to_float<<<grd, blk, 0, st>>>(kt_view(g, acc, ymax_bits), N, out);
    PAT_LAUNCH_CHECK("k_kt_to_float");
    return PAT_OK;
}

int launch_adjoint(const pat_geometry* g, const float* y, float* out, cudaStream_t st) {
    int rc = ensure_precond(g, st);
    if (rc) return rc;
    char* scratch = nullptr;
    const size_t bytes = 256 + (size_t)g->desc.n * g->desc.n * sizeof(int);
    PAT_CUDA(cudaMallocAsync((void**)&scratch, bytes, st));
    const cudaError_t e = cudaMemsetAsync(scratch, 0, bytes, st);
    rc = e == cudaSuccess ? launch_adjoint_into(g, y, (unsigned*)scratch, (int*)(scratch + 256), out, st)
                          : cuda_fail(e, "launch_adjoint: scratch");
    cudaFreeAsync(scratch, st);
    return rc;
}

}  // namespace pat

using namespace pat;

extern "C" int pat_adjoint(const pat_geometry* g, const float* y_dev, float* u_dev, void* stream) {
    if (!g || !u_dev || !y_dev) return fail(PAT_ERR_INVALID_ARG, "pat_adjoint: NULL argument");
    return launch_adjoint(g, y_dev, u_dev, (cudaStream_t)stream);
}
