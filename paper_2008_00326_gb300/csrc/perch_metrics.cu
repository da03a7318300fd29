// ADD / ADD-S pose errors (the accuracy measure of Sec. VI): the mean over a
// mesh's vertices x of || A x - B x || (ADD) or of the distance from A x to
// the closest B y (ADD-S, for symmetric objects).  ADD, and ADD-S of a mesh
// without sorted vertices: one block per pose pair, B's transformed vertices
// staged through shared memory in tiles.  ADD-S over sorted vertices: a few
// blocks per pair that visit only the groups of vertices that can be closest.
#include "perch_internal.cuh"

#include <algorithm>
#include <cmath>
#include <cooperative_groups.h>
#include <vector>

namespace perch {

namespace {

constexpr int kAddThreads = 256;
constexpr int kAddTile = 1024;      // B-transformed vertices per shared-memory tile
constexpr int kAddPer = 4;          // A-transformed vertices per thread per pass

__device__ __forceinline__ float3 xform(const float* P, float4 v)
{
    return make_float3(P[0] * v.x + P[1] * v.y + P[2] * v.z + P[3],
                       P[4] * v.x + P[5] * v.y + P[6] * v.z + P[7],
                       P[8] * v.x + P[9] * v.y + P[10] * v.z + P[11]);
}

__global__ void __launch_bounds__(kAddThreads) k_add_s(const float4* verts, int nv, const float* A_all,
                                                      const float* B_all, long long n, int symmetric,
                                                      double* out)
{
    __shared__ float3 tile[kAddTile];
    __shared__ float sA[12], sB[12];
    __shared__ double red[kAddThreads / 32];
    for (long long q = blockIdx.x; q < n; q += gridDim.x) {
        if (threadIdx.x < 12) {
            sA[threadIdx.x] = A_all[q * 12 + threadIdx.x];
            sB[threadIdx.x] = B_all[q * 12 + threadIdx.x];
        }
        __syncthreads();
        double acc = 0.0;
        for (int base = 0; base < nv; base += kAddThreads * kAddPer) {
            float3 pa[kAddPer];
            float best[kAddPer];
#pragma unroll
            for (int k = 0; k < kAddPer; ++k) {
                const int i = base + k * kAddThreads + threadIdx.x;
                pa[k] = i < nv ? xform(sA, verts[i]) : make_float3(0.f, 0.f, 0.f);
                best[k] = 3.0e38f;
                if (!symmetric && i < nv) {
                    const float3 pb = xform(sB, verts[i]);
                    const float dx = pa[k].x - pb.x, dy = pa[k].y - pb.y, dz = pa[k].z - pb.z;
                    best[k] = dx * dx + dy * dy + dz * dz;
                }
            }
            if (symmetric) {
                for (int t0 = 0; t0 < nv; t0 += kAddTile) {
                    const int tn = min(kAddTile, nv - t0);
                    __syncthreads();
                    for (int j = threadIdx.x; j < tn; j += kAddThreads) tile[j] = xform(sB, verts[t0 + j]);
                    __syncthreads();
                    for (int j = 0; j < tn; ++j) {
                        const float3 pb = tile[j];
#pragma unroll
                        for (int k = 0; k < kAddPer; ++k) {
                            const float dx = pa[k].x - pb.x, dy = pa[k].y - pb.y, dz = pa[k].z - pb.z;
                            best[k] = fminf(best[k], dx * dx + dy * dy + dz * dz);
                        }
                    }
                }
            }
#pragma unroll
            for (int k = 0; k < kAddPer; ++k)
                if (base + k * kAddThreads + (int)threadIdx.x < nv) acc += sqrt((double)best[k]);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
        __syncthreads();
        if (threadIdx.x == 0) {
            double s = 0.0;
            for (int w = 0; w < kAddThreads / 32; ++w) s += red[w];
            out[q] = s / (double)nv;
        }
        __syncthreads();
    }
}

// ---- ADD-S over sorted vertices -------------------------------------------
//
// A warp takes a group of 32 neighbouring vertices under A, and a group under B
// is visited only if its bounding sphere comes closer to the warp's than the
// worst nearest distance its lanes have so far: the nearest group first, then
// whatever is left in reach, some 17 of the 313 groups of a 10,000-vertex
// ellipsoid for estimates ten degrees and a centimetre off.  A skipped vertex is
// farther than every lane's nearest one, so the minima are those of all V^2
// distances, bit for bit.  The bounds allow for rounding (kAddSlack of the
// coordinates' size, some twenty times the error of a transformed distance) and
// for poses that are not rotations (a group's radius grows with the largest
// singular value, bounded from R^T R); a bound that is not a number skips
// nothing.
//
// Bound by instruction issue: a visit is 32 broadcast loads and 9 operations
// each.  200 pairs of 10,001 vertices take 0.52 ms, against 5.39 ms for all
// pairs of vertices (and 1.69 ms with groups along a space-filling curve).
constexpr int kNnThreads = 128;
constexpr int kNnWarps = kNnThreads / 32;
constexpr int kNnCluster = 8;        // blocks per pose pair when there are few pairs
constexpr int kNnSums = kNnCluster * kNnWarps;   // partial sums of a pair, however many blocks it has
constexpr int kNnGroups = 1024;      // groups under B held in shared memory
constexpr float kAddSlack = 1e-5f;

// An upper bound of the factor by which P stretches a length.
__device__ __forceinline__ float stretch(const float* P)
{
    float most = 0.0f;
    for (int i = 0; i < 3; ++i) {
        float row = 0.0f;
        for (int j = 0; j < 3; ++j) row += fabsf(P[i] * P[j] + P[4 + i] * P[4 + j] + P[8 + i] * P[8 + j]);
        most = row > most || row != row ? row : most;
    }
    return sqrtf(most) * 1.00001f;
}

__global__ void __launch_bounds__(kNnThreads) k_add_nn(const float4* verts, const float4* spheres, int nv, int ng,
                                                       float size, const float* A_all, const float* B_all,
                                                       long long n, double* out)
{
    namespace cg = cooperative_groups;
    __shared__ float4 near_group[kNnGroups];
    __shared__ float4 staged[kNnWarps][32];
    __shared__ float sA[12], sB[12];
    __shared__ double sum[kNnSums];
    const cg::cluster_group cluster = cg::this_cluster();
    const int parts = (int)cluster.num_blocks(), part = (int)cluster.block_rank();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (long long q = blockIdx.x / parts; q < n; q += gridDim.x / parts) {
        if (threadIdx.x < 12) {
            sA[threadIdx.x] = A_all[q * 12 + threadIdx.x];
            sB[threadIdx.x] = B_all[q * 12 + threadIdx.x];
        }
        __syncthreads();
        const float fa = stretch(sA), fb = stretch(sB);
        const float slack = kAddSlack * (fa * size + fb * size + fabsf(sA[3]) + fabsf(sA[7]) + fabsf(sA[11]) +
                                         fabsf(sB[3]) + fabsf(sB[7]) + fabsf(sB[11]));
        const auto sphere_b = [&](int g) {
            const float4 c = __ldg(&spheres[g]);
            const float3 p = xform(sB, c);
            return make_float4(p.x, p.y, p.z, c.w * fb);
        };
        if (ng <= kNnGroups)
            for (int g = threadIdx.x; g < ng; g += kNnThreads) near_group[g] = sphere_b(g);
        __syncthreads();
        // group i goes to partial sum i % kNnSums and a warp adds up whole partial
        // sums, so that a pair's mean has one summation order and does not depend on
        // the number of pairs that share the call
        const int n_sums = min(kNnSums, ng);
        for (int slot = part * kNnWarps + warp; slot < n_sums; slot += parts * kNnWarps) {
            double acc = 0.0;
            for (int i = slot; i < ng; i += kNnSums) {
                const int vi = 32 * i + lane;
                const float3 x = xform(sA, __ldg(&verts[vi]));
                const float4 ci = __ldg(&spheres[i]);
                const float3 c = xform(sA, ci);
                const float reach = ci.w * fa + slack;
                // distance from the warp's centre to group g's sphere
                const auto gap = [&](int g) {
                    const float4 s = ng <= kNnGroups ? near_group[g] : sphere_b(g);
                    const float dx = c.x - s.x, dy = c.y - s.y, dz = c.z - s.z;
                    return sqrtf(dx * dx + dy * dy + dz * dz) - s.w;
                };
                float best = 3.0e38f;
                const auto visit = [&](int g) {
                    const float3 y = xform(sB, __ldg(&verts[32 * g + lane]));
                    staged[warp][lane] = 32 * g + lane < nv ? make_float4(y.x, y.y, y.z, 0.0f)
                                                            : make_float4(1.0e30f, 1.0e30f, 1.0e30f, 0.0f);
                    __syncwarp();
#pragma unroll 8
                    for (int k = 0; k < 32; ++k) {
                        const float4 p = staged[warp][k];
                        const float dx = x.x - p.x, dy = x.y - p.y, dz = x.z - p.z;
                        best = fminf(best, dx * dx + dy * dy + dz * dz);
                    }
                    __syncwarp();
                };
                // the group whose sphere is nearest first (any group if none compares)
                float low = 3.0e38f;
                int first = 0;
                for (int g = lane; g < ng; g += 32) {
                    const float d = gap(g);
                    if (d < low) { low = d; first = g; }
                }
                for (int o = 16; o > 0; o >>= 1) {
                    const float d = __shfl_xor_sync(0xffffffffu, low, o);
                    const int g = __shfl_xor_sync(0xffffffffu, first, o);
                    if (d < low || (d == low && g < first)) { low = d; first = g; }
                }
                visit(first);
                for (int g0 = 0; g0 < ng; g0 += 32) {
                    // of these 32 groups the nearest first, as long as it is within what the lanes'
                    // worst nearest distance reaches (distances are non-negative: their bits order
                    // like the values; a gap below zero counts as zero, one that does not compare too)
                    const int g = g0 + lane;
                    unsigned ahead = 0xFFFFFFFFu;
                    if (g < ng && g != first) {
                        const float d = gap(g);
                        ahead = d > 0.0f ? __float_as_uint(d) : 0u;
                    }
                    for (;;) {
                        const unsigned next = __reduce_min_sync(0xffffffffu, ahead);
                        const float worst =
                            __uint_as_float(__reduce_max_sync(0xffffffffu, vi < nv ? __float_as_uint(best) : 0u));
                        const float limit = sqrtf(worst) * 1.00001f + reach;
                        if (next == 0xFFFFFFFFu || __uint_as_float(next) > limit) break;
                        const unsigned at = __ballot_sync(0xffffffffu, ahead == next);
                        const int k = __ffs(at) - 1;
                        if (lane == k) ahead = 0xFFFFFFFFu;
                        visit(g0 + k);
                    }
                }
                if (vi < nv) acc += sqrt((double)best);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            if (lane == 0) sum[slot] = acc;
        }
        cluster.sync();
        if (part == 0 && threadIdx.x == 0) {
            double total = 0.0;
            for (int k = 0; k < n_sums; ++k) total += cluster.map_shared_rank(sum, k / kNnWarps % parts)[k];
            out[q] = total / (double)nv;
        }
        cluster.sync();              // the sums have been read, and with them the pose arrays
    }
}

}  // namespace

// Vertices split into compact groups of 32 (the widest side of a box halved, at a
// multiple of 32, until 32 are left) with bounding spheres: out holds
// 32 ceil(n / 32) vertices (the last group filled up with its last vertex), then
// a sphere (centre, radius) for each group.  On a 10,000-vertex ellipsoid the
// spheres are 6.3 mm wide and a group has 17 others in reach; groups along a
// space-filling curve are 11 mm and 48.
size_t add_groups_count(int n_verts) { return 33 * (((size_t)n_verts + 31) / 32); }

static void split_groups(const float* v4, int* first, int* last)
{
    while (last - first > 32) {
        float lo[3], hi[3];
        for (int a = 0; a < 3; ++a) lo[a] = hi[a] = v4[4 * (size_t)*first + a];
        for (const int* i = first; i != last; ++i)
            for (int a = 0; a < 3; ++a) {
                lo[a] = std::min(lo[a], v4[4 * (size_t)*i + a]);
                hi[a] = std::max(hi[a], v4[4 * (size_t)*i + a]);
            }
        int axis = 0;
        for (int a = 1; a < 3; ++a)
            if (hi[a] - lo[a] > hi[axis] - lo[axis]) axis = a;
        int* const mid = first + ((last - first + 31) / 32 + 1) / 2 * 32;
        std::nth_element(first, mid, last, [&](int i, int j) {
            const float x = v4[4 * (size_t)i + axis], y = v4[4 * (size_t)j + axis];
            return x < y || (x == y && i < j);
        });
        split_groups(v4, mid, last);
        last = mid;
    }
}

void add_groups(const float* v4, int n_verts, float* out)
{
    const size_t ng = ((size_t)n_verts + 31) / 32;
    std::vector<int> order(n_verts);
    for (int i = 0; i < n_verts; ++i) order[i] = i;
    split_groups(v4, order.data(), order.data() + n_verts);
    for (int i = 0; i < n_verts; ++i) std::copy(v4 + 4 * (size_t)order[i], v4 + 4 * (size_t)order[i] + 4, out + 4 * (size_t)i);
    for (size_t i = n_verts; i < 32 * ng; ++i) std::copy(out + 4 * (size_t)(n_verts - 1), out + 4 * (size_t)n_verts, out + 4 * i);
    for (size_t g = 0; g < ng; ++g) {
        const float* p = out + 128 * g;
        float* s = out + 128 * ng + 4 * g;
        for (int a = 0; a < 3; ++a) {
            float mn = p[a], mx = p[a];
            for (int i = 1; i < 32; ++i) { mn = std::min(mn, p[4 * i + a]); mx = std::max(mx, p[4 * i + a]); }
            s[a] = 0.5f * mn + 0.5f * mx;
        }
        double r = 0.0;
        for (int i = 0; i < 32; ++i) {
            const double dx = (double)p[4 * i] - s[0], dy = (double)p[4 * i + 1] - s[1], dz = (double)p[4 * i + 2] - s[2];
            r = std::max(r, std::sqrt(dx * dx + dy * dy + dz * dz));
        }
        s[3] = (float)(r * 1.000001);
    }
}

cudaError_t launch_add_nn(const float4* groups, int n_verts, float size, const float* poses, const float* poses_true,
                          long long n, double* out, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    if (n_verts < 1) return cudaErrorInvalidValue;
    const int ng = (n_verts + 31) / 32;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // enough blocks to fill the device several times over, at most one warp per group
    int parts = 1;
    while (parts < kNnCluster && n * parts < 16ll * sms && 2 * parts * kNnWarps <= ng) parts *= 2;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(parts * std::min<long long>(n, 65535)));
    cfg.blockDim = dim3(kNnThreads);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)parts;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_add_nn, groups, groups + 32 * (size_t)ng, n_verts, ng, size, poses, poses_true, n,
                              out);
}

cudaError_t launch_add_s(const float4* verts, int n_verts, const float* poses, const float* poses_true,
                         long long n, int symmetric, double* out, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    if (n_verts < 1) return cudaErrorInvalidValue;
    const unsigned grid = (unsigned)(n < 65535 ? n : 65535);
    k_add_s<<<grid, kAddThreads, 0, s>>>(verts, n_verts, poses, poses_true, n, symmetric, out);
    return cudaGetLastError();
}

}  // namespace perch
