// Batched projector, transpose and CG over many independent problems of
// uneven sizes (cube side, image count and image size differ per problem).
//
// Ray kernels are persistent: one grid of (SM count x resident CTAs) CTAs
// strides over the work list until it is exhausted.  A work unit is one warp
// tile (32 pixels) of one pixel tile of one image of one problem; the
// schedule deals groups of kSchedGroup tiles round-robin over the problems,
// so every warp's share mixes all problems evenly, and the transposes of all
// problems run side by side with their float atomics spread over every cube
// instead of piling onto one small cube at a time.  Each problem carries its own tile shape (256
// threads per CTA for all of them), chosen by the autotuner.  The walk is the same
// Siddon walk as the single-problem kernels (walk.cuh).
//
// Vector kernels run over (problem, chunk of kChunk elements) items: a CTA
// handles one chunk, writes its FP64 partial sums, and the CTA that finishes
// a problem's last chunk adds that problem's partials in a fixed order and
// applies the CG scalar step (reduce.cuh).  Every problem has its own FP64
// slots and "done" flag, so problems that converge early stop working while
// the others continue.
#include <cuda_bf16.h>

#include "batch.cuh"
#include "plane.cuh"
#include "reduce.cuh"
#include "walk.cuh"

namespace tomo {

namespace {

constexpr int kThreads = 256;

// Problem owning `item`: the largest p with prefix[p] <= item.
__device__ __forceinline__ int owner(const int64_t *__restrict__ prefix,
                                     int n_probs, int64_t item)
{
    int lo = 0, hi = n_probs - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(prefix + mid) <= item)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

template <bool kAdjoint>
__global__ void __launch_bounds__(kThreads, 6)
k_walk_batched(const WalkDesc *__restrict__ descs,
               const int64_t *__restrict__ prefix,
               const int2 *__restrict__ sched, int64_t n_chunks,
               unsigned long long *next_item)
{
    // CTAs take tiles from a work queue (one atomic counter); warp w of the
    // CTA walks warp tile w of the tile, and a barrier per tile keeps the
    // CTA's warps together: their rays are neighbours that sweep the same
    // voxels at the same depth, which is what the L1 reuses (measured:
    // without the barrier, or with static striding, the walks run slower).
    // The fetch of the next tile is issued when the current one starts and
    // read after its walk: in the transpose the counter shares the L2 atomic
    // units with every segment's reduction, and a fetch waited for at the
    // barrier would park the whole CTA in that queue.
    __shared__ long long s_item;
    const int lane = threadIdx.x & 31;
    const int wt = threadIdx.x >> 5;  // warp tile in the tile
    const int64_t n_items = n_chunks * kSchedGroup;
    if (threadIdx.x == 0) s_item = (long long)atomicAdd(next_item, 1ull);
    __syncthreads();
    int64_t item = s_item;
    while (item < n_items) {
        unsigned long long ahead = 0;
        if (threadIdx.x == 0) ahead = atomicAdd(next_item, 1ull);
        do {
            const int2 ch = sched[item / kSchedGroup];
            const int p = ch.x;
            const int t = ch.y + (int)(item % kSchedGroup);
            if (t >= (int)(prefix[p + 1] - prefix[p])) continue;
            const WalkDesc d = descs[p];
            if (d.done != nullptr && *d.done != 0.0) continue;
            const int tu = t % d.tiles_u;
            const int rest = t / d.tiles_u;
            const int tv = rest % d.tiles_v;
            const int img = rest / d.tiles_v;
            // the pixel of this lane: warp tile wt of tile (tu, tv), laid out as
            // in the single-problem kernels
            const int rows = 32 / d.tl.warp_u;
            const int warps_u = d.tl.tile_u / d.tl.warp_u;
            const int iu = tu * d.tl.tile_u + (wt % warps_u) * d.tl.warp_u +
                           (lane % d.tl.warp_u);
            const int iv = tv * d.tl.tile_v + (wt / warps_u) * rows +
                           (lane / d.tl.warp_u);
            if (iu >= d.nu || iv >= d.nv) continue;
            const int64_t id = ((int64_t)img * d.nv + iv) * d.nu + iu;
            const bool masked = d.mask != nullptr && d.mask[id] != 0;
            const float gain = d.prm[img].gain;
            if (!kAdjoint) {
                float y = 0.0f;
                if (!masked) {
                    const RayRec r = load_ray(d.rays + id);
                    if (r.chord > 0.0f) {
                        GatherOp<float> op;
                        op.c = d.src;
                        op.acc = 0.0f;
                        siddon_gather(r, d.nx, d.nxny, op);
                        y = gain * op.acc;
                    }
                }
                d.dst[id] = y;
            } else if (!masked) {
                const float yv = gain * d.src[id];
                if (yv != 0.0f) {
                    const RayRec r = load_ray(d.rays + id);
                    if (r.chord > 0.0f) {
                        ScatterOp op;
                        op.c = d.dst;
                        op.y = yv;
                        siddon_walk(r, d.nx, d.nxny, op);
                    }
                }
            }
        } while (false);
        __syncthreads();  // every thread has read s_item
        if (threadIdx.x == 0) s_item = (long long)ahead;
        __syncthreads();
        item = s_item;
    }
}

// Plane-synchronous transpose over the plane tiles of every problem, with
// the work queue of k_walk_batched.  All lanes of a warp take part in the
// plane walk's votes, so lanes outside the image only vote.
__global__ void __launch_bounds__(kThreads, 5)
k_adjoint_plane_batched(const WalkDesc *__restrict__ descs,
                        const int64_t *__restrict__ prefix,
                        const int2 *__restrict__ sched, int64_t n_chunks,
                        unsigned long long *next_item)
{
    __shared__ long long s_item;
    const int lane = threadIdx.x & 31;
    const int wt = threadIdx.x >> 5;  // image row of the tile
    const int64_t n_items = n_chunks * kSchedGroup;
    if (threadIdx.x == 0) s_item = (long long)atomicAdd(next_item, 1ull);
    __syncthreads();
    int64_t item = s_item;
    while (item < n_items) {
        unsigned long long ahead = 0;
        if (threadIdx.x == 0) ahead = atomicAdd(next_item, 1ull);
        const int2 ch = sched[item / kSchedGroup];
        const int p = ch.x;
        const int t = ch.y + (int)(item % kSchedGroup);
        // t, p and the done flag are the same for every thread of the CTA
        if (t < (int)(prefix[p + 1] - prefix[p])) {
            const WalkDesc d = descs[p];
            if (d.done == nullptr || *d.done == 0.0) {
                const int tiles_u = (d.nu + kPlaneTileU - 1) / kPlaneTileU;
                const int tiles_v = (d.nv + kPlaneTileV - 1) / kPlaneTileV;
                const int tu = t % tiles_u;
                const int rest = t / tiles_u;
                const int tv = rest % tiles_v;
                const int img = rest / tiles_v;
                const int iu = tu * kPlaneTileU + lane;
                const int iv = tv * kPlaneTileV + wt;
                const bool in_img = iu < d.nu && iv < d.nv;
                const int64_t id = ((int64_t)img * d.nv + iv) * d.nu + iu;
                const ImgParam q = d.prm[img];
                RayRec r;
                r.chord = -1.0f;
                float yv = 0.0f;
                if (in_img && (d.mask == nullptr || d.mask[id] == 0)) {
                    yv = q.gain * d.src[id];
                    if (yv != 0.0f) r = load_ray(d.rays + id);
                }
                const bool live = r.chord > 0.0f;
                PlaneRay pr;
                const bool regular =
                    live && plane_ray(r, q.pad, d.nx, d.ny, d.nz, pr,
                                         sizeof(float));
                const int L = (q.pad >> 2) & 3;
                PlaneScatterOp op;
                op.c = L == 1 ? d.lay1 : (L == 2 ? d.lay2 : d.dst);
                op.y = yv;
                plane_walk_for(q.pad, pr, regular, op);
                if (live && !regular) {
                    ScatterOp op2;
                    op2.c = d.dst;
                    op2.y = yv;
                    siddon_walk(r, d.nx, d.nxny, op2);
                }
            }
        }
        __syncthreads();  // every thread has read s_item
        if (threadIdx.x == 0) s_item = (long long)ahead;
        __syncthreads();
        item = s_item;
    }
}

// Layout accumulators back into the native cubes: one CTA per 32 x 32 tile
// of (x, b) at one c, reading the accumulator along b and adding into the
// cube along x (both coalesced, the additions atomic); the accumulator is
// zeroed as it is read.
__global__ void __launch_bounds__(kThreads)
k_add_from_layout_batched(const LayoutJob *__restrict__ jobs,
                          const int64_t *__restrict__ prefix, int n_jobs)
{
    __shared__ float tile[32][33];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int64_t n_items = prefix[n_jobs];
    for (int64_t item = blockIdx.x; item < n_items; item += gridDim.x) {
        const int j = owner(prefix, n_jobs, item);
        const LayoutJob J = jobs[j];
        // the same for every thread of the CTA
        if (!(*J.used & J.bit) || (J.done != nullptr && *J.done != 0.0))
            continue;
        const int64_t k = item - prefix[j];
        const int x0 = (int)(k % J.tiles_x) * 32;
        const int64_t r = k / J.tiles_x;
        const int b0 = (int)(r % J.tiles_b) * 32;
        const int c = (int)(r / J.tiles_b);
        for (int i = ty; i < 32; i += 8) {
            const int x = x0 + i, b = b0 + tx;
            if (b < J.nb && x < J.nx) {
                const int64_t a = b + (int64_t)J.nb * (x + (int64_t)J.nx * c);
                tile[tx][i] = J.acc[a];
                J.acc[a] = 0.0f;
            }
        }
        __syncthreads();
        // the jobs of layouts 1 and 2 of one problem run in this same launch
        // and add into the same cube: the additions must be atomic
        for (int i = ty; i < 32; i += 8) {
            const int b = b0 + i, x = x0 + tx;
            if (b < J.nb && x < J.nx) red_add(J.cube + x + J.sb * b + J.sc * c, tile[i][tx]);
        }
        __syncthreads();
    }
}

// The problems' cubes into their layout copies (the inverse tile move of
// k_add_from_layout_batched: read along x, write along b).
__global__ void __launch_bounds__(kThreads)
k_to_layout_batched(const LayoutJob *__restrict__ jobs,
                    const int64_t *__restrict__ prefix, int n_jobs)
{
    __shared__ float tile[32][33];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int64_t n_items = prefix[n_jobs];
    for (int64_t item = blockIdx.x; item < n_items; item += gridDim.x) {
        const int j = owner(prefix, n_jobs, item);
        const LayoutJob J = jobs[j];
        // the same for every thread of the CTA
        if (!(*J.used & J.bit) || (J.done != nullptr && *J.done != 0.0))
            continue;
        const int64_t k = item - prefix[j];
        const int x0 = (int)(k % J.tiles_x) * 32;
        const int64_t r = k / J.tiles_x;
        const int b0 = (int)(r % J.tiles_b) * 32;
        const int c = (int)(r / J.tiles_b);
        for (int i = ty; i < 32; i += 8) {
            const int b = b0 + i, x = x0 + tx;
            if (b < J.nb && x < J.nx) tile[i][tx] = J.cube[x + J.sb * b + J.sc * c];
        }
        __syncthreads();
        for (int i = ty; i < 32; i += 8) {
            const int x = x0 + i, b = b0 + tx;
            if (b < J.nb && x < J.nx)
                J.acc[b + (int64_t)J.nb * (x + (int64_t)J.nx * c)] = tile[tx][i];
        }
        __syncthreads();
    }
}

// Forward projection over the plane tiles of every problem: one CTA per
// tile, tiles taken problem by problem (a CTA finds its problem by a binary
// search of the tile prefix), so the CTAs resident at one time gather from
// one problem's cube and layout copies.  A CTA covers 32 x 8 pixels of one
// image; when the image's hint selects the plane forward the warps walk
// plane by plane on the layout copies, with the gather bodies free of slot
// predicates (irregular lanes per ray on the native cube), otherwise every
// lane walks its own ray.  Voxels go by 32-bit offset, with six slabs of
// loads in flight in 64 registers (a walk by address needs every problem's
// cube and copies between two multiples of 2^32).  When it came, 10.34
// ms per projection of the 32-problem workload against 11.0 for a persistent
// work-queue kernel, whose loop state left no registers for the predicate-free
// bodies.
__global__ void __launch_bounds__(kThreads, 4)
k_forward_plane_batched(const WalkDesc *__restrict__ descs,
                        const int64_t *__restrict__ prefix, int n_probs)
{
    const int lane = threadIdx.x & 31;
    const int wt = threadIdx.x >> 5;  // image row of the tile
    const int64_t tile = (int64_t)blockIdx.y * gridDim.x + blockIdx.x;
    if (tile >= prefix[n_probs]) return;
    int lo = 0, hi = n_probs;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (prefix[mid] <= tile) lo = mid;
        else hi = mid;
    }
    const int p = lo;
    const int t = (int)(tile - prefix[p]);
    const WalkDesc &d = descs[p];
    if (d.done != nullptr && *d.done != 0.0) return;
    const int tiles_u = (d.nu + kPlaneTileU - 1) / kPlaneTileU;
    const int tiles_v = (d.nv + kPlaneTileV - 1) / kPlaneTileV;
    const int tu = t % tiles_u;
    const int rest = t / tiles_u;
    const int tv = rest % tiles_v;
    const int img = rest / tiles_v;
    const int iu = tu * kPlaneTileU + lane;
    const int iv = tv * kPlaneTileV + wt;
    const bool in_img = iu < d.nu && iv < d.nv;
    const int64_t id = ((int64_t)img * d.nv + iv) * d.nu + iu;
    const ImgParam q = d.prm[img];
    RayRec r;
    r.chord = -1.0f;
    if (in_img && (d.mask == nullptr || d.mask[id] == 0))
        r = load_ray(d.rays + id);
    const bool live = r.chord > 0.0f;
    float acc = 0.0f;
    if (q.pad & kPlaneFwdBit) {
        PlaneRay pr;
        const bool regular =
            live && plane_ray(r, q.pad, d.nx, d.ny, d.nz, pr, sizeof(float));
        const int L = (q.pad >> 2) & 3;
        PlaneGatherOp<float> op;
        op.c = L == 1 ? d.lay1 : (L == 2 ? d.lay2 : d.src);
        op.acc = 0.0f;
        plane_walk_for<6>(q.pad, pr, regular, op);
        acc = op.acc;
        if (live && !regular) {
            GatherOp<float> op2;
            op2.c = d.src;
            op2.acc = 0.0f;
            siddon_gather(r, d.nx, d.nxny, op2);
            acc = op2.acc;
        }
    } else if (live) {
        GatherOp<float> op2;
        op2.c = d.src;
        op2.acc = 0.0f;
        siddon_gather(r, d.nx, d.nxny, op2);
        acc = op2.acc;
    }
    if (in_img) d.dst[id] = q.gain * acc;
}

// Operation codes (batch.cuh): what one vector pass does.
constexpr int V_SUMSQ = BV_SUMSQ, V_ZERO = BV_ZERO, V_INIT = BV_INIT,
              V_PRIOR = BV_PRIOR, V_PQ = BV_PQ, V_UPDATE = BV_UPDATE,
              V_DIR = BV_DIR, V_PRIOR_X = BV_PRIOR_X;

// Elements a thread takes of a chunk at once: their loads are issued together
// (the passes are bound by the latency of their loads: the problems of a
// batch are small and their vectors stay in L2).
constexpr int kVecUnroll = 4;
static_assert(kChunk % (kThreads * kVecUnroll) == 0, "whole groups per chunk");

// Calls f(i, k) for the elements i = c0 + threadIdx.x + (g + k) blockDim.x of
// a chunk that lie below c1, k = 0 .. kVecUnroll - 1 inside one group g.
template <class F>
__device__ __forceinline__ void vec_group(int64_t c0, int64_t c1, int g, const F &f)
{
#pragma unroll
    for (int k = 0; k < kVecUnroll; ++k) {
        const int64_t i = c0 + (int64_t)(g + k) * kThreads + threadIdx.x;
        if (i < c1) f(i, k);
    }
}

// One pass over every problem.  A work item is a chunk of kChunk elements of
// one problem; with sums, the CTA that finishes a problem's last item (one
// counter per problem, no waiting) adds the problem's partial sums in item
// order and applies the CG scalar step, so the sums do not depend on which
// CTA that is.  Bound by load latency and, in the passes with sums, by the
// FP64 additions of block_sums: 8 problems (31^3 to 96^3), 10 iterations, took
// 4.08 ms with chunks of 16384 elements, one kernel for all passes (64-bit
// divisions and a run-time choice of pass per element) and separate kernels
// for the scalar steps, and take 2.81 ms.  At six CTAs per SM (40 registers) a
// prior pass spills 28 bytes and the first residual 8; the update, 72 there, 40
// at five (19.3 -> 17.8 us a pass).
template <int kOp>
__global__ void __launch_bounds__(kThreads, kOp == V_UPDATE ? 5 : 6)
k_vec_batched(const VecDesc *__restrict__ descs,
              const int64_t *__restrict__ prefix, int n_probs, bool warm,
              double tol2, double *partials, unsigned int *counters)
{
    constexpr bool kSums = kOp == V_SUMSQ || kOp == V_INIT || kOp == V_PQ ||
                           kOp == V_UPDATE;
    constexpr int kGroups = (int)(kChunk / kThreads);
    constexpr int kValues = kOp == V_INIT || kOp == V_UPDATE ? 2 : 1;
    __shared__ double sm[kValues][kSumThreads];
    __shared__ bool last;
    const int64_t n_items = prefix[n_probs];
    for (int64_t item = blockIdx.x; item < n_items; item += gridDim.x) {
        const int p = owner(prefix, n_probs, item);
        const VecDesc d = descs[p];  // a copy: stores below cannot alias it
        // (not V_SUMSQ, V_ZERO, V_INIT: the slots hold the last solve's state)
        if (kOp != V_SUMSQ && kOp != V_ZERO && kOp != V_INIT && d.S[S_DONE] != 0.0)
            continue;
        const int64_t len = (kOp == V_SUMSQ) ? d.m : d.n;
        // this item's chunk of its problem: elements [c0, c1)
        const int64_t c0 = (item - prefix[p]) * kChunk;
        const int64_t c1 = c0 + kChunk < len ? c0 + kChunk : len;
        // per-thread sums in compensated float pairs (SumF2), then FP64
        SumF2 a0, a1;
        for (int g = 0; g < kGroups; g += kVecUnroll) {
            if constexpr (kOp == V_SUMSQ) {
                float y[kVecUnroll] = {};
                vec_group(c0, c1, g, [&](int64_t i, int k) {
                    if (d.mask == nullptr || d.mask[i] == 0) y[k] = d.y[i];
                });
#pragma unroll
                for (int k = 0; k < kVecUnroll; ++k) a0.add_prod(y[k], y[k]);
            } else if constexpr (kOp == V_ZERO) {
                vec_group(c0, c1, g, [&](int64_t i, int) {
                    d.b[i] = 0.0f;
                    if (!warm || (d.mm != nullptr && d.mm[i] != 0)) d.x[i] = 0.0f;
                });
            } else if constexpr (kOp == V_INIT) {
                // map mask: b, r, p are 0 on the excluded voxels, so every
                // iterate stays in the restricted space
                float b[kVecUnroll] = {}, q[kVecUnroll] = {}, x[kVecUnroll] = {};
                bool out[kVecUnroll] = {};
                vec_group(c0, c1, g, [&](int64_t i, int k) {
                    out[k] = d.mm != nullptr && d.mm[i] != 0;
                    b[k] = out[k] ? 0.0f : d.b[i];
                    if (warm) {
                        q[k] = d.q[i];
                        x[k] = d.x[i];
                    }
                });
                vec_group(c0, c1, g, [&](int64_t i, int k) {
                    if (out[k]) d.b[i] = 0.0f;
                    const float r = out[k] ? 0.0f : (warm ? b[k] - q[k] : b[k]);
                    d.r[i] = r;
                    d.p[i] = r;
                    a0.add_prod(r, r);
                    if (warm) a1.add_prod_sum(x[k], r, b[k]);
                });
            } else if constexpr (kOp == V_PRIOR || kOp == V_PRIOR_X) {
                const float *__restrict__ src = (kOp == V_PRIOR_X) ? d.x : d.p;
                const unsigned nx = d.nx, ny = d.ny;
                float val[kVecUnroll] = {};
                vec_group(c0, c1, g, [&](int64_t v, int k) {
                    const unsigned r = (unsigned)v / nx;  // v < 2^31
                    const int i = (int)((unsigned)v - r * nx);
                    const int j = (int)(r % ny), z = (int)(r / ny);
                    val[k] = prior_at(src, d.w, v, i, j, z, d.nx, d.ny, d.nz, d.lam);
                });
                vec_group(c0, c1, g, [&](int64_t v, int k) { d.q[v] = val[k]; });
            } else if constexpr (kOp == V_PQ) {
                float u[kVecUnroll] = {}, v[kVecUnroll] = {};
                vec_group(c0, c1, g, [&](int64_t i, int k) {
                    u[k] = d.p[i];
                    v[k] = d.q[i];
                });
#pragma unroll
                for (int k = 0; k < kVecUnroll; ++k) a0.add_prod(u[k], v[k]);
            } else if constexpr (kOp == V_UPDATE) {
                const StepF2 alpha = step_of(d.S[S_ALPHA]);
                float x[kVecUnroll] = {}, r[kVecUnroll] = {}, b[kVecUnroll] = {};
                vec_group(c0, c1, g, [&](int64_t i, int k) {
                    x[k] = axpy(alpha, d.p[i], d.x[i]);
                    r[k] = (d.mm != nullptr && d.mm[i] != 0)
                               ? 0.0f
                               : axpy(alpha, -d.q[i], d.r[i]);
                    b[k] = d.b[i];
                });
                vec_group(c0, c1, g, [&](int64_t i, int k) {
                    d.x[i] = x[k];
                    d.r[i] = r[k];
                    a0.add_prod(r[k], r[k]);
                    a1.add_prod_sum(x[k], r[k], b[k]);
                });
            } else if constexpr (kOp == V_DIR) {
                const StepF2 beta = step_of(d.S[S_BETA]);
                float v[kVecUnroll] = {};
                vec_group(c0, c1, g, [&](int64_t i, int k) {
                    v[k] = axpy(beta, d.p[i], d.r[i]);
                });
                vec_group(c0, c1, g, [&](int64_t i, int k) { d.p[i] = v[k]; });
            }
        }
        if constexpr (kSums) {
            static_assert(kThreads == kSumThreads, "one value per thread");
            double v[kValues], t[kValues];
            v[0] = a0.value();
            if (kValues > 1) v[kValues - 1] = a1.value();
            block_sums<kValues>(v, t, sm);
            const int64_t first = prefix[p], end = prefix[p + 1];
            if (threadIdx.x == 0) {
                for (int k = 0; k < kValues; ++k) partials[2 * item + k] = t[k];
                __threadfence();
                last = atomicAdd(counters + p, 1u) == (unsigned)(end - first) - 1u;
            }
            __syncthreads();
            if (last) {
                __threadfence();
                for (int k = 0; k < kValues; ++k) v[k] = 0.0;
                for (int64_t i = first + threadIdx.x; i < end; i += blockDim.x)
                    for (int k = 0; k < kValues; ++k) v[k] += __ldcg(partials + 2 * i + k);
                block_sums<kValues>(v, t, sm);
                const double s0 = t[0], s1 = t[kValues - 1];
                if (threadIdx.x == 0) {
                    counters[p] = 0u;
                    if (kOp == V_SUMSQ) d.S[S_YMY] = s0;
                    else if (kOp == V_INIT) cg_finalize_init(d.S, d.report, s0, s1, tol2);
                    else if (kOp == V_PQ) cg_finalize_pq(d.S, s0);
                    else cg_finalize_update(d.S, d.report, s0, s1);
                }
            }
            __syncthreads();  // `last` is read before the next item writes it
        }
    }
}

}  // namespace

int walk_batched_blocks_per_sm()
{
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &n, k_walk_batched<false>, kThreads, 0) != cudaSuccess)
        return 1;
    int m = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &m, k_walk_batched<true>, kThreads, 0) != cudaSuccess)
        return 1;
    return n < m ? (n > 0 ? n : 1) : (m > 0 ? m : 1);
}

int plane_batched_blocks_per_sm()
{
    int q = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &q, k_adjoint_plane_batched, kThreads, 0) != cudaSuccess)
        return 1;
    return q > 0 ? q : 1;
}

cudaError_t launch_walk_batched(bool adjoint, const WalkDesc *descs,
                                const int64_t *prefix, const int2 *sched,
                                int64_t n_chunks, unsigned long long *next_item,
                                int grid, cudaStream_t s)
{
    if (adjoint)
        k_walk_batched<true><<<grid, kThreads, 0, s>>>(descs, prefix, sched,
                                                        n_chunks, next_item);
    else
        k_walk_batched<false><<<grid, kThreads, 0, s>>>(descs, prefix, sched,
                                                         n_chunks, next_item);
    return cudaGetLastError();
}

cudaError_t launch_adjoint_plane_batched(const WalkDesc *descs,
                                         const int64_t *prefix,
                                         const int2 *sched, int64_t n_chunks,
                                         unsigned long long *next_item,
                                         int grid, cudaStream_t s)
{
    k_adjoint_plane_batched<<<grid, kThreads, 0, s>>>(descs, prefix, sched,
                                                      n_chunks, next_item);
    return cudaGetLastError();
}

cudaError_t launch_add_from_layout_batched(const LayoutJob *jobs,
                                           const int64_t *prefix, int n_jobs,
                                           int grid, cudaStream_t s)
{
    if (n_jobs <= 0) return cudaSuccess;
    k_add_from_layout_batched<<<grid, kThreads, 0, s>>>(jobs, prefix, n_jobs);
    return cudaGetLastError();
}

cudaError_t launch_to_layout_batched(const LayoutJob *jobs,
                                     const int64_t *prefix, int n_jobs,
                                     int grid, cudaStream_t s)
{
    if (n_jobs <= 0) return cudaSuccess;
    k_to_layout_batched<<<grid, kThreads, 0, s>>>(jobs, prefix, n_jobs);
    return cudaGetLastError();
}

cudaError_t launch_forward_plane_batched(const WalkDesc *descs,
                                         const int64_t *prefix, int n_probs,
                                         int64_t n_tiles, cudaStream_t s)
{
    if (n_tiles <= 0) return cudaSuccess;
    const int64_t gx = n_tiles < 65536 ? n_tiles : 65536;
    const dim3 grid((unsigned)gx, (unsigned)((n_tiles + gx - 1) / gx));
    k_forward_plane_batched<<<grid, kThreads, 0, s>>>(descs, prefix, n_probs);
    return cudaGetLastError();
}

cudaError_t launch_vec_batched(int op, const VecDesc *descs,
                               const int64_t *prefix, int n_probs, bool warm,
                               double tol2, double *partials,
                               unsigned int *counters, int grid, cudaStream_t s)
{
    auto launch = [&](auto kernel) {
        kernel<<<grid, kThreads, 0, s>>>(descs, prefix, n_probs, warm, tol2,
                                         partials, counters);
    };
    switch (op) {
    case BV_SUMSQ: launch(k_vec_batched<BV_SUMSQ>); break;
    case BV_ZERO: launch(k_vec_batched<BV_ZERO>); break;
    case BV_INIT: launch(k_vec_batched<BV_INIT>); break;
    case BV_PRIOR: launch(k_vec_batched<BV_PRIOR>); break;
    case BV_PQ: launch(k_vec_batched<BV_PQ>); break;
    case BV_UPDATE: launch(k_vec_batched<BV_UPDATE>); break;
    case BV_DIR: launch(k_vec_batched<BV_DIR>); break;
    case BV_PRIOR_X: launch(k_vec_batched<BV_PRIOR_X>); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace tomo
