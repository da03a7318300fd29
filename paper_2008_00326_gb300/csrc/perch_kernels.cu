// libperch kernels for sm_103a: observation build (back-projection, CIELAB,
// cell index over I), the fused per-hypothesis scorer (fixed-point raster with
// an atomicMin z-buffer in shared memory, resolve with occluder removal and
// image-space down-sampling, warp-cooperative 27-cell radius search,
// CIEDE2000 check, J_r / J_o counts) and the warp-shuffle argmin.
//
// Bit-exactness: every step whose result decides an integer (snapping,
// coverage, depth, back-projection, squared distances, the cylinder test) is
// written with explicit round-to-nearest single-precision intrinsics
// (__fadd_rn, __fmul_rn, __fdiv_rn) and the file is compiled with -fmad=false,
// so no multiply-add is contracted.  Edge functions are exact int32.
#include "perch_internal.cuh"

#include <algorithm>
#include <climits>
#include <cstdint>
#include <cuda_runtime.h>
#include <map>
#include <mutex>
#include <set>
#include <tuple>
#include <utility>

namespace perch {

// ---------------------------------------------------------------------------
// colour: sRGB -> CIELAB (D65) and CIEDE2000 (Sec. IV-B, Eq. 4), binary32
// ---------------------------------------------------------------------------

__device__ float g_srgb_lin[256];   // sRGB decoding of each 8-bit code, filled at start-up

__global__ void k_init_tables()
{
    int i = threadIdx.x;
    if (i < 256) {
        float c = __fdiv_rn((float)i, 255.0f);
        g_srgb_lin[i] = (c <= 0.04045f) ? __fdiv_rn(c, 12.92f)
                                        : powf(__fdiv_rn(__fadd_rn(c, 0.055f), 1.055f), 2.4f);
    }
}

cudaError_t init_device_tables(cudaStream_t s)
{
    k_init_tables<<<1, 256, 0, s>>>();
    return cudaGetLastError();
}

// The colour test only decides whether a difference exceeds tau_c, and the
// parity contract leaves the decisions within 1e-3 of tau_c to rounding (the
// band): the constants' divisions are multiplications by reciprocals, the
// other divisions approximate (__fdividef), the angles in half-turns
// (sinpif / cospif reduce their argument exactly) -- a few 1e-6 relative at
// most, far inside the band.
__device__ __forceinline__ float cie_f(float t)
{
    // cube root above (6/29)^3, the linear toe below it
    return (t > 0.0088564517f) ? cbrtf(t) : (t * 903.29630f + 16.0f) * (1.0f / 116.0f);
}

__device__ __forceinline__ float3 srgb8_to_lab(uint32_t r8, uint32_t g8, uint32_t b8)
{
    float r = g_srgb_lin[r8], g = g_srgb_lin[g8], b = g_srgb_lin[b8];
    float x = 0.4124564f * r + 0.3575761f * g + 0.1804375f * b;
    float y = 0.2126729f * r + 0.7151522f * g + 0.0721750f * b;
    float z = 0.0193339f * r + 0.1191920f * g + 0.9503041f * b;
    float fx = cie_f(x * (1.0f / 0.95047f)), fy = cie_f(y), fz = cie_f(z * (1.0f / 1.08883f));
    return make_float3(116.0f * fy - 16.0f, 500.0f * (fx - fy), 200.0f * (fy - fz));
}

// Hue angle in [0, 360) degrees, 0 on the neutral axis.
__device__ __forceinline__ float hue_degrees(float b, float a)
{
    const float kDeg = 57.295779513082321f;      // degrees per radian
    float h = (a == 0.0f && b == 0.0f) ? 0.0f : atan2f(b, a) * kDeg;
    if (h < 0.0f) h += 360.0f;
    return h;
}

// CIEDE2000 with kL = kC = kH = 1, angles in degrees.
__device__ __forceinline__ float ciede2000(float3 p, float3 q)
{
    const float k25p7 = 6103515625.0f;
    float c1 = sqrtf(p.y * p.y + p.z * p.z);
    float c2 = sqrtf(q.y * q.y + q.z * q.z);
    float cm = 0.5f * (c1 + c2);
    float cm2 = cm * cm, cm7 = cm2 * cm2 * cm2 * cm;
    float g = 0.5f * (1.0f - sqrtf(__fdividef(cm7, cm7 + k25p7)));
    float ap1 = p.y * (1.0f + g), ap2 = q.y * (1.0f + g);
    float cp1 = sqrtf(ap1 * ap1 + p.z * p.z), cp2 = sqrtf(ap2 * ap2 + q.z * q.z);
    const float hp1 = hue_degrees(p.z, ap1), hp2 = hue_degrees(q.z, ap2);
    float prod = cp1 * cp2;
    float dh = 0.0f, hm;
    if (prod == 0.0f) {
        hm = hp1 + hp2;
    } else {
        dh = hp2 - hp1;
        if (dh > 180.0f) dh -= 360.0f;
        else if (dh < -180.0f) dh += 360.0f;
        float s = hp1 + hp2;
        if (fabsf(hp1 - hp2) <= 180.0f) hm = 0.5f * s;
        else hm = (s < 360.0f) ? 0.5f * (s + 360.0f) : 0.5f * (s - 360.0f);
    }
    float dL = q.x - p.x;
    float dC = cp2 - cp1;
    float dH = 2.0f * sqrtf(prod) * sinpif(dh * (1.0f / 360.0f));     // sin(dh / 2 degrees)
    float lm = 0.5f * (p.x + q.x) - 50.0f;
    float lm2 = lm * lm;
    float cpm = 0.5f * (cp1 + cp2);
    float t = 1.0f - 0.17f * cospif((hm - 30.0f) * (1.0f / 180.0f)) + 0.24f * cospif(hm * (1.0f / 90.0f))
              + 0.32f * cospif((3.0f * hm + 6.0f) * (1.0f / 180.0f))
              - 0.20f * cospif((4.0f * hm - 63.0f) * (1.0f / 180.0f));
    float e = (hm - 275.0f) * (1.0f / 25.0f);
    float dtheta = 30.0f * __expf(-e * e);
    float cpm2 = cpm * cpm, cpm7 = cpm2 * cpm2 * cpm2 * cpm;
    float rc = 2.0f * sqrtf(__fdividef(cpm7, cpm7 + k25p7));
    float sl = 1.0f + __fdividef(0.015f * lm2, sqrtf(20.0f + lm2));
    float sc = 1.0f + 0.045f * cpm;
    float sh = 1.0f + 0.015f * cpm * t;
    float rt = -sinpif(dtheta * (1.0f / 90.0f)) * rc;                  // sin(2 dtheta degrees)
    float a = __fdividef(dL, sl), b = __fdividef(dC, sc), c = __fdividef(dH, sh);
    return sqrtf(a * a + b * b + c * c + rt * b * c);
}

// ---------------------------------------------------------------------------
// geometry helpers (exact op order)
// ---------------------------------------------------------------------------

// fl(a / b) from rb = fl(1 / b): an estimate corrected twice by its exact
// remainder.  Markstein, "Computation of elementary functions on the IBM RISC
// System/6000 processor" (1990): with rb correctly rounded and q within one unit
// in the last place, fl(q + fl(a - b q) rb) is the correctly rounded quotient;
// the first correction brings q there.  Holds while nothing underflows or
// overflows: kDivLo < |a| < kDivHi (or a = 0) and kDivLo < b < kDivHi.  Five
// operations against some nineteen issue slots of __fdiv_rn.
constexpr float kDivLo = 8.6736174e-19f, kDivHi = 1.1529215e18f;       // 2^-60, 2^60

__device__ __forceinline__ float div_by(float a, float b, float rb)
{
    float q = __fmul_rn(a, rb);
    q = __fmaf_rn(__fmaf_rn(-b, q, a), rb, q);
    return __fmaf_rn(__fmaf_rn(-b, q, a), rb, q);
}

// Quotients outside that range (rare, kept out of line).
__device__ __noinline__ float div_any(float a, float b) { return __fdiv_rn(a, b); }

__device__ __forceinline__ bool div_fits(float a) { return (fabsf(a) > kDivLo && fabsf(a) < kDivHi) || a == 0.0f; }

// Back-projection of pixel (u,v) at integer depth d (0.1 mm units), Sec. IV-A.
// sc.rfx, sc.rfy: fl(1 / fx), fl(1 / fy), or 0 when fx or fy is out of div_by's range.
__device__ __forceinline__ float3 back_project(const DevScene& sc, int u, int v, unsigned d)
{
    const float z = div_by(__uint2float_rn(d), 10000.0f, 1.0f / 10000.0f);
    const float ax = __fmul_rn(__fsub_rn(__int2float_rn(u), sc.cx), z);
    const float ay = __fmul_rn(__fsub_rn(__int2float_rn(v), sc.cy), z);
    if (sc.rfx != 0.0f && div_fits(ax) && div_fits(ay))
        return make_float3(div_by(ax, sc.fx, sc.rfx), div_by(ay, sc.fy, sc.rfy), z);
    return make_float3(div_any(ax, sc.fx), div_any(ay, sc.fy), z);
}

// Hash-cell coordinate floor(x / cell), taken as floor(fl(x * fl(1 / cell))):
// for two points within delta of each other on an axis the two products
// differ by at most delta (1 + 2^-22) / cell + 2 * 1e5 * 2^-24 < 0.997 (cell =
// delta (1 + 1/64), coordinates below 1e5 cells), so their cells are at most
// one apart -- the radius search's 27 cells hold every point within delta.
__device__ __forceinline__ int cell_coord(float x, float inv_cell)
{
    return __float2int_rd(__fmul_rn(x, inv_cell));
}

__device__ __forceinline__ unsigned long long cell_key(int cx, int cy, int cz)
{
    return ((unsigned long long)((unsigned)(cx + kCellBias) & 0x1FFFFFu) << 42) |
           ((unsigned long long)((unsigned)(cy + kCellBias) & 0x1FFFFFu) << 21) |
           (unsigned long long)((unsigned)(cz + kCellBias) & 0x1FFFFFu);
}

__device__ __forceinline__ uint32_t hash_slot(unsigned long long k, uint32_t mask)
{
    k ^= k >> 31;
    k *= 0x7fb5d329728ea185ull;
    k ^= k >> 27;
    k *= 0x81dadef4bc2dd44dull;
    k ^= k >> 33;
    return (uint32_t)k & mask;
}

// ---------------------------------------------------------------------------
// observation build: per-pixel CIELAB, cloud I, voxel hash (cell = delta*(1+1/64))
// ---------------------------------------------------------------------------

__global__ void k_obs_insert(DevScene sc, const uint8_t* __restrict__ rgb, float4* lab, float4* pxyz,
                             int32_t* slot_of_pixel, unsigned long long* keys, uint32_t* count,
                             uint32_t mask, int* n_valid, int* err)
{
    int npx = sc.W * sc.H;
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= npx) return;
    int u = i % sc.W, v = i / sc.W;
    float3 L = srgb8_to_lab(rgb[3 * i], rgb[3 * i + 1], rgb[3 * i + 2]);
    lab[i] = make_float4(L.x, L.y, L.z, 0.0f);
    unsigned d = sc.depth[i];
    int slot = -1;
    pxyz[i] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (d != 0 && u % sc.stride == 0 && v % sc.stride == 0) {
        float3 p = back_project(sc, u, v, d);
        pxyz[i] = make_float4(p.x, p.y, p.z, 1.0f);
        unsigned long long k = cell_key(cell_coord(p.x, sc.inv_cell), cell_coord(p.y, sc.inv_cell),
                                        cell_coord(p.z, sc.inv_cell));
        uint32_t h = hash_slot(k, mask);
        for (uint32_t probe = 0; probe <= mask; ++probe) {
            unsigned long long prev = atomicCAS(&keys[h], kEmptyKey, k);
            if (prev == kEmptyKey || prev == k) {
                slot = (int)h;
                break;
            }
            h = (h + 1) & mask;
        }
        if (slot < 0) atomicOr(err, kErrHashFull);
        else atomicAdd(&count[slot], 1u);
        atomicAdd(n_valid, 1);
    }
    slot_of_pixel[i] = slot;
}

// Exclusive scan of count[0..n) into start[], in tiles of 1024 (one block per
// tile), then a second pass over the tile sums, then the offsets.
__device__ __forceinline__ uint32_t block_incl_scan_1024(uint32_t x, uint32_t* warp_sums)
{
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t t = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += t;
    }
    if (lane == 31) warp_sums[w] = x;
    __syncthreads();
    if (w == 0) {
        uint32_t s = warp_sums[lane];
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t t = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += t;
        }
        warp_sums[lane] = s;
    }
    __syncthreads();
    if (w > 0) x += warp_sums[w - 1];
    return x;
}

__global__ void __launch_bounds__(1024) k_scan_tiles(const uint32_t* count, uint32_t* start,
                                                    uint32_t* tile_sums, uint32_t n)
{
    __shared__ uint32_t ws[32];
    uint32_t i = blockIdx.x * 1024u + threadIdx.x;
    uint32_t x = i < n ? count[i] : 0u;
    uint32_t incl = block_incl_scan_1024(x, ws);
    if (i < n) start[i] = incl - x;
    if (threadIdx.x == 1023) tile_sums[blockIdx.x] = incl;
}

__global__ void __launch_bounds__(1024) k_scan_sums(uint32_t* tile_sums, uint32_t n_tiles)
{
    // n_tiles <= 1024 * k; sequential over chunks of 1024
    __shared__ uint32_t ws[32];
    __shared__ uint32_t carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (uint32_t base = 0; base < n_tiles; base += 1024) {
        uint32_t i = base + threadIdx.x;
        uint32_t x = i < n_tiles ? tile_sums[i] : 0u;
        uint32_t incl = block_incl_scan_1024(x, ws);
        uint32_t c = carry;
        if (i < n_tiles) tile_sums[i] = c + incl - x;
        __syncthreads();
        if (threadIdx.x == 1023) carry = c + incl;
        __syncthreads();
    }
}

__global__ void k_finish_table(const unsigned long long* keys, const uint32_t* count,
                               uint32_t* start, const uint32_t* tile_offsets, uint4* table,
                               uint32_t n)
{
    uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    uint32_t s = start[i] + tile_offsets[i >> 10];
    start[i] = s;
    unsigned long long k = keys[i];
    table[i] = make_uint4((uint32_t)k, (uint32_t)(k >> 32), s, k == kEmptyKey ? 0u : count[i]);
}

// Re-insert the occupied slots of the build table into a table sized for
// them (twice the occupied count, rounded up to a power of two), so that the
// lookups of the radius search touch a compact, cache-friendly array.
__global__ void k_compact_table(const uint4* big, uint32_t cap_big, uint4* small, uint32_t mask,
                                int* err)
{
    uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= cap_big) return;
    uint4 e = big[i];
    unsigned long long k = (unsigned long long)e.x | ((unsigned long long)e.y << 32);
    if (k == kEmptyKey) return;
    uint32_t h = hash_slot(k, mask);
    for (uint32_t probe = 0; probe <= mask; ++probe) {
        unsigned long long prev = atomicCAS(reinterpret_cast<unsigned long long*>(&small[h]), kEmptyKey, k);
        if (prev == kEmptyKey) {
            small[h].z = e.z;
            small[h].w = e.w;
            return;
        }
        h = (h + 1) & mask;
    }
    atomicOr(err, kErrHashFull);
}

// ---- near-cell bitmap: lets a query whose 27 neighbour cells are all empty
// skip the hash lookups (exact: such a query has no candidate at all)

__device__ __forceinline__ long long near_index(const DevScene& sc, int x, int y, int z)
{
    const int ix = x - sc.near_lo[0], iy = y - sc.near_lo[1], iz = z - sc.near_lo[2];
    if (ix < 0 || iy < 0 || iz < 0 || ix >= sc.near_n[0] || iy >= sc.near_n[1] || iz >= sc.near_n[2]) return -1;
    return ((long long)iz * sc.near_n[1] + iy) * sc.near_n[0] + ix;
}

__global__ void k_cell_occupancy(DevScene sc, uint32_t* occ)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < sc.n_pts; i += gridDim.x * blockDim.x) {
        const float4 p = sc.pts[i];
        const long long b = near_index(sc, cell_coord(p.x, sc.inv_cell), cell_coord(p.y, sc.inv_cell),
                                       cell_coord(p.z, sc.inv_cell));
        if (b >= 0) atomicOr(&occ[b >> 5], 1u << (b & 31));
    }
}

__global__ void k_cell_dilate(DevScene sc, const uint32_t* occ, uint32_t* near_bits)
{
    const long long n = (long long)sc.near_n[0] * sc.near_n[1] * sc.near_n[2];
    for (long long b = blockIdx.x * (long long)blockDim.x + threadIdx.x; b < n;
         b += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(b % sc.near_n[0]) + sc.near_lo[0];
        const int y = (int)((b / sc.near_n[0]) % sc.near_n[1]) + sc.near_lo[1];
        const int z = (int)(b / ((long long)sc.near_n[0] * sc.near_n[1])) + sc.near_lo[2];
        bool any = false;
        for (int k = 0; k < 27 && !any; ++k) {
            const long long q = near_index(sc, x + k % 3 - 1, y + (k / 3) % 3 - 1, z + k / 9 - 1);
            any = q >= 0 && ((occ[q >> 5] >> (q & 31)) & 1u);
        }
        if (any) atomicOr(&near_bits[b >> 5], 1u << (b & 31));
    }
}

cudaError_t launch_near_cells(const DevScene& sc, uint32_t* occ, uint32_t* near_bits, cudaStream_t s)
{
    if (sc.n_pts <= 0) return cudaSuccess;
    k_cell_occupancy<<<min(1024, (sc.n_pts + 255) / 256), 256, 0, s>>>(sc, occ);
    const long long n = (long long)sc.near_n[0] * sc.near_n[1] * sc.near_n[2];
    k_cell_dilate<<<(unsigned)std::min<long long>(4096, (n + 255) / 256), 256, 0, s>>>(sc, occ, near_bits);
    return cudaGetLastError();
}

// ---- observation build over the dense cell index: points and their cell box,
// count per cell, exclusive scan, scatter by cell.  Five small launches read and
// write each pixel two or three times (the cell arrays, four bytes a cell, are
// the larger part at a million cells); the hash build they replace for clouds
// whose cell box is small enough took thirteen.

// n / d for 0 <= n < 2^24 and 1 <= d < 2^24 without an integer division: a
// binary32 estimate (both operands exact, error below one) corrected once.
__device__ __forceinline__ int div_small(int n, int d)
{
    int q = __float2int_rz(__fmul_rn(__int2float_rn(n), __frcp_rn(__int2float_rn(d))));
    const int r = n - q * d;
    q += (r >= d) - (r < 0);
    return q;
}

__device__ __forceinline__ bool on_lattice(const DevScene& sc, int u, int v)
{
    return div_small(u, sc.stride) * sc.stride == u && div_small(v, sc.stride) * sc.stride == v;
}

// Per pixel CIELAB and observed point; stats = (smallest, largest cell
// coordinates of the points, their count), initialised to (INT_MAX x 3,
// INT_MIN x 3, 0).
__global__ void __launch_bounds__(256) k_obs_points(DevScene sc, const uint8_t* __restrict__ rgb, float4* lab,
                                                   float4* pxyz, int* stats)
{
    __shared__ int red[7];
    if (threadIdx.x < 7) red[threadIdx.x] = threadIdx.x < 3 ? INT_MAX : threadIdx.x < 6 ? INT_MIN : 0;
    __syncthreads();
    const int i = blockIdx.x * 256 + threadIdx.x;
    int c[3] = {INT_MAX, INT_MAX, INT_MAX};
    bool in = false;
    if (i < sc.W * sc.H) {
        const int v = div_small(i, sc.W), u = i - v * sc.W;
        const float3 L = srgb8_to_lab(rgb[3 * i], rgb[3 * i + 1], rgb[3 * i + 2]);
        lab[i] = make_float4(L.x, L.y, L.z, 0.0f);
        const unsigned d = sc.depth[i];
        in = d != 0 && on_lattice(sc, u, v);
        float4 p = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (in) {
            const float3 q = back_project(sc, u, v, d);
            p = make_float4(q.x, q.y, q.z, 1.0f);
            c[0] = cell_coord(q.x, sc.inv_cell);
            c[1] = cell_coord(q.y, sc.inv_cell);
            c[2] = cell_coord(q.z, sc.inv_cell);
        }
        pxyz[i] = p;
    }
    const unsigned any = __ballot_sync(0xffffffffu, in);
    if (any != 0u) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const int lo = __reduce_min_sync(0xffffffffu, c[a]), hi = __reduce_max_sync(0xffffffffu, in ? c[a] : INT_MIN);
            if ((threadIdx.x & 31) == 0) {
                atomicMin(&red[a], lo);
                atomicMax(&red[3 + a], hi);
            }
        }
        if ((threadIdx.x & 31) == 0) atomicAdd(&red[6], __popc(any));
    }
    __syncthreads();
    if (red[6] == 0) return;
    if (threadIdx.x < 3) atomicMin(&stats[threadIdx.x], red[threadIdx.x]);
    else if (threadIdx.x < 6) atomicMax(&stats[threadIdx.x], red[threadIdx.x]);
    else if (threadIdx.x == 6) atomicAdd(&stats[6], red[6]);
}

// Linear cell of an observed point (its cell lies inside the box's border).
__device__ __forceinline__ int point_cell(const DevScene& sc, float4 p)
{
    const int x = cell_coord(p.x, sc.inv_cell) - sc.near_lo[0], y = cell_coord(p.y, sc.inv_cell) - sc.near_lo[1];
    const int z = cell_coord(p.z, sc.inv_cell) - sc.near_lo[2];
    return (z * sc.near_n[1] + y) * sc.near_n[0] + x;
}

// Points per cell; the first point of a cell marks the cell's 27 neighbours, nine
// rows of three consecutive bits, in the near-cell bitmap (both arrays zeroed).
__global__ void __launch_bounds__(256) k_cell_count(DevScene sc, uint32_t* count, uint32_t* near_bits)
{
    const int i = blockIdx.x * 256 + threadIdx.x;
    if (i >= sc.W * sc.H) return;
    const float4 p = sc.pxyz[i];
    if (p.w == 0.0f) return;
    const int c = point_cell(sc, p);
    if (atomicAdd(&count[c], 1u) != 0u) return;
    const int nx = sc.near_n[0], nxy = nx * sc.near_n[1];
    for (int dz = -1; dz <= 1; ++dz)
        for (int dy = -1; dy <= 1; ++dy) {
            const int b = c + dz * nxy + dy * nx - 1;
            atomicOr(&near_bits[b >> 5], 7u << (b & 31));
            if ((b & 31) > 29) atomicOr(&near_bits[(b >> 5) + 1], 7u >> (32 - (b & 31)));
        }
}

// start[i] += its tile's offset; start[n] = total.
__global__ void k_add_tile_offsets(uint32_t* start, const uint32_t* tile_offsets, uint32_t n, uint32_t total)
{
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) start[i] += tile_offsets[i >> 10];
    else if (i == n) start[n] = total;
}

// The points by cell (any order within a cell: a nearest neighbour's ties go by
// pixel); count runs down to zero.
__global__ void __launch_bounds__(256) k_cell_scatter(DevScene sc, const uint32_t* start, uint32_t* count, float4* out)
{
    const int i = blockIdx.x * 256 + threadIdx.x;
    if (i >= sc.W * sc.H) return;
    float4 p = sc.pxyz[i];
    if (p.w == 0.0f) return;
    const int c = point_cell(sc, p), v = div_small(i, sc.W);
    // the pixel as (v << 16 | u): ordered like the index v W + u, and its
    // coordinates come back without a division
    p.w = __uint_as_float(((uint32_t)v << 16) | (uint32_t)(i - v * sc.W));
    out[start[c] + atomicSub(&count[c], 1u) - 1u] = p;
}

cudaError_t launch_obs_points(const DevScene& sc, const uint8_t* rgb, float4* lab, float4* pxyz, int* stats,
                              cudaStream_t s)
{
    k_obs_points<<<(sc.W * sc.H + 255) / 256, 256, 0, s>>>(sc, rgb, lab, pxyz, stats);
    return cudaGetLastError();
}

cudaError_t launch_dense_cells(const DevScene& sc, uint32_t* count, uint32_t* tile_sums, uint32_t* near_bits,
                               uint32_t* cell_start, float4* out, cudaStream_t s)
{
    const long long n = (long long)sc.near_n[0] * sc.near_n[1] * sc.near_n[2];
    if (sc.n_pts <= 0 || n <= 0 || n > 0x7FFFFFFFll) return cudaErrorInvalidValue;
    const unsigned blocks = (unsigned)((sc.W * sc.H + 255) / 256);
    cudaError_t e = cudaMemsetAsync(count, 0, (size_t)n * 4, s);
    if (!e) e = cudaMemsetAsync(near_bits, 0, (size_t)((n + 31) / 32) * 4, s);
    if (e) return e;
    k_cell_count<<<blocks, 256, 0, s>>>(sc, count, near_bits);
    const uint32_t n_tiles = (uint32_t)((n + 1023) / 1024);
    k_scan_tiles<<<n_tiles, 1024, 0, s>>>(count, cell_start, tile_sums, (uint32_t)n);
    k_scan_sums<<<1, 1024, 0, s>>>(tile_sums, n_tiles);
    k_add_tile_offsets<<<(unsigned)(n / 256 + 1), 256, 0, s>>>(cell_start, tile_sums, (uint32_t)n, (uint32_t)sc.n_pts);
    k_cell_scatter<<<blocks, 256, 0, s>>>(sc, cell_start, count, out);
    return cudaGetLastError();
}

cudaError_t launch_compact_table(const uint4* big, uint32_t cap_big, uint4* small, uint32_t cap_small,
                                 int* err, cudaStream_t s)
{
    cudaError_t e = cudaMemsetAsync(small, 0xFF, sizeof(uint4) * cap_small, s);
    if (e != cudaSuccess) return e;
    k_compact_table<<<(cap_big + 255) / 256, 256, 0, s>>>(big, cap_big, small, cap_small - 1, err);
    return cudaGetLastError();
}

__global__ void k_count_cells(const uint4* table, uint32_t n, int* n_cells)
{
    uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    bool occ = false;
    if (i < n) {
        uint4 e = table[i];
        occ = !(e.x == 0xFFFFFFFFu && e.y == 0xFFFFFFFFu);
    }
    unsigned b = __ballot_sync(0xffffffffu, occ);
    if ((threadIdx.x & 31) == 0 && b) atomicAdd(n_cells, __popc(b));
}

__global__ void k_obs_scatter(DevScene sc, const int32_t* slot_of_pixel, const uint32_t* start,
                              uint32_t* cursor, float4* pts)
{
    int npx = sc.W * sc.H;
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= npx) return;
    int slot = slot_of_pixel[i];
    if (slot < 0) return;
    int u = i % sc.W, v = i / sc.W;
    float3 p = back_project(sc, u, v, sc.depth[i]);
    uint32_t pos = start[slot] + atomicAdd(&cursor[slot], 1u);
    // the pixel as (v << 16 | u): ordered like the index v W + u, and its
    // coordinates come back without a division
    pts[pos] = make_float4(p.x, p.y, p.z, __uint_as_float(((uint32_t)v << 16) | (uint32_t)u));
}

cudaError_t launch_build(const DevScene& sc, const BuildBuffers& b, uint32_t cap,
                         const uint8_t* rgb_dev, int* err, cudaStream_t s)
{
    int npx = sc.W * sc.H;
    cudaError_t e;
    if ((e = cudaMemsetAsync(b.keys, 0xFF, sizeof(unsigned long long) * cap, s))) return e;
    if ((e = cudaMemsetAsync(b.count, 0, sizeof(uint32_t) * cap, s))) return e;
    if ((e = cudaMemsetAsync(b.cursor, 0, sizeof(uint32_t) * cap, s))) return e;
    if ((e = cudaMemsetAsync(b.n_valid, 0, 2 * sizeof(int), s))) return e;
    int blocks = (npx + 255) / 256;
    k_obs_insert<<<blocks, 256, 0, s>>>(sc, rgb_dev, b.lab, b.pxyz, b.slot_of_pixel, b.keys, b.count,
                                        cap - 1, b.n_valid, err);
    uint32_t n_tiles = (cap + 1023) / 1024;
    // the tile sums of the scan live just past the cursors
    uint32_t* tile_sums = b.cursor + cap;   // BuildBuffers::cursor has cap + n_tiles words
    k_scan_tiles<<<n_tiles, 1024, 0, s>>>(b.count, b.start, tile_sums, cap);
    k_scan_sums<<<1, 1024, 0, s>>>(tile_sums, n_tiles);
    k_finish_table<<<(cap + 255) / 256, 256, 0, s>>>(b.keys, b.count, b.start, tile_sums, b.table,
                                                     cap);
    k_obs_scatter<<<blocks, 256, 0, s>>>(sc, b.slot_of_pixel, b.start, b.cursor, b.pts);
    k_count_cells<<<(cap + 255) / 256, 256, 0, s>>>(b.table, cap, b.n_valid + 1);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// scoring kernel
// ---------------------------------------------------------------------------


struct TriSetup {
    int x[3], y[3];               // snapped positions, 1/16 px
    float iz[3];                  // 1/Z
    int vid[3];                   // mesh vertex ids after the orientation swap
    int A;                        // doubled area > 0
};

// A set-up triangle staged for its warp (48 bytes, 3 x 16-byte moves): the values
// of edges 0 and 1 at its pixel box's first sample, less their tie bias, and
// their increments per column (a) and row (b); edge 2 holds the rest of K.  Its
// items, numbered from `first`, are the samples of the box or, when thin, its
// rows.
struct __align__(16) TriStage {
    int a0, a1, b0, b1;
    int t0, t1, K, tri;
    unsigned idx;                 // z-buffer index of the first sample | its flags (DepthItem) | thin << 18
    int bw;                       // box width
    float rbw;                    // fl(1 / bw)
    int first;
};

__device__ __forceinline__ int edge_fn(int ax, int ay, int bx, int by, int px, int py)
{
    return (bx - ax) * (py - ay) - (by - ay) * (px - ax);
}

__device__ __forceinline__ bool owns(int dx, int dy)
{
    return dy > 0 || (dy == 0 && dx < 0);
}

__device__ __forceinline__ int floor16(int x) { return x >> 4; }         // arithmetic shift
__device__ __forceinline__ int ceil16(int x) { return -((-x) >> 4); }

// Doubled area and orientation of a loaded triangle: a negative area swaps
// vertices 1 and 2 (two-sided rendering).  False if degenerate (A == 0).
__device__ __forceinline__ bool orient_triangle(TriSetup& o)
{
    int A = edge_fn(o.x[0], o.y[0], o.x[1], o.y[1], o.x[2], o.y[2]);
    if (A == 0) return false;
    if (A < 0) {
        int tx = o.x[1], ty = o.y[1], tvid = o.vid[1];
        float ti = o.iz[1];
        o.x[1] = o.x[2]; o.y[1] = o.y[2]; o.iz[1] = o.iz[2]; o.vid[1] = o.vid[2];
        o.x[2] = tx; o.y[2] = ty; o.iz[2] = ti; o.vid[2] = tvid;
        A = -A;
    }
    o.A = A;
    return true;
}

// Triangle loaded at a pose: transform, near/guard-band cull, projection,
// 4-bit snap (orient_triangle completes the set-up).  False if culled.
// (C: a DevScene, or what the rasteriser keeps of one.)
template <class C>
__device__ __forceinline__ bool load_triangle(const C& sc, const float4* verts, const float* P, int4 tv, TriSetup& o)
{
    int vids[3] = {tv.x, tv.y, tv.z};
    const float gx0 = (float)(-16 * sc.W), gx1 = (float)(32 * sc.W);
    const float gy0 = (float)(-16 * sc.H), gy1 = (float)(32 * sc.H);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        float4 v = __ldg(&verts[vids[k]]);
        float X = __fadd_rn(__fadd_rn(__fadd_rn(__fmul_rn(P[0], v.x), __fmul_rn(P[1], v.y)),
                                      __fmul_rn(P[2], v.z)), P[3]);
        float Y = __fadd_rn(__fadd_rn(__fadd_rn(__fmul_rn(P[4], v.x), __fmul_rn(P[5], v.y)),
                                      __fmul_rn(P[6], v.z)), P[7]);
        float Z = __fadd_rn(__fadd_rn(__fadd_rn(__fmul_rn(P[8], v.x), __fmul_rn(P[9], v.y)),
                                      __fmul_rn(P[10], v.z)), P[11]);
        if (!(Z >= sc.z_near)) return false;
        const float iz = __frcp_rn(Z);     // = fl(1 / Z), as the division would give
        const bool fits = fminf(fabsf(X), fminf(fabsf(Y), Z)) > kDivLo && fmaxf(fabsf(X), fmaxf(fabsf(Y), Z)) < kDivHi;
        float px = __fadd_rn(__fmul_rn(sc.fx, fits ? div_by(X, Z, iz) : div_any(X, Z)), sc.cx);
        float py = __fadd_rn(__fmul_rn(sc.fy, fits ? div_by(Y, Z, iz) : div_any(Y, Z)), sc.cy);
        float sx = __fmul_rn(px, 16.0f), sy = __fmul_rn(py, 16.0f);
        if (!(sx >= gx0) || !(sx < gx1) || !(sy >= gy0) || !(sy < gy1)) return false;
        o.x[k] = __float2int_rn(sx);
        o.y[k] = __float2int_rn(sy);
        o.iz[k] = iz;
        o.vid[k] = vids[k];
    }
    return true;
}

template <bool K32>
__device__ __forceinline__ void zmin(uint32_t* zbuf, int idx, unsigned d, int tri, int* err)
{
    if (K32) {
        if (d > 0xFFFFu) {
            atomicOr(err, kErrKeyRange);
            return;
        }
        atomicMin(&zbuf[idx], (d << 16) | (unsigned)tri);
    } else {
        unsigned long long* z64 = reinterpret_cast<unsigned long long*>(zbuf);
        atomicMin(&z64[idx], ((unsigned long long)d << 32) | (unsigned)tri);
    }
}

// ---- resolve queue and per-warp cell groups -------------------------------

constexpr int kWarpQueue = 64;    // kept rendered points queued per warp (a ring)

// A group of G queries shares a 27-cell candidate list; k = floor(32 / G)
// lanes test each query's candidates.  Lane l serves query floor(l / k),
// taken as (l * ceil(1024 / k)) >> 10 (exact for l < 32 and k <= 32), so the
// split needs no integer division.
__constant__ unsigned char c_lanes_per_query[33] = {
    32, 32, 16, 10, 8, 6, 5, 4, 4, 3, 3, 2, 2, 2, 2, 2, 2,
    1, 1, 1, 1, 1, 1, 1, 1, 1, 1, 1, 1, 1, 1, 1, 1};
__constant__ unsigned short c_lane_div[33] = {
    1024, 1024, 512, 342, 256, 205, 171, 147, 128, 114, 103, 94, 86, 79, 74, 69, 64,
    61, 57, 54, 52, 49, 47, 45, 43, 41, 40, 38, 37, 36, 35, 34, 32};

struct __align__(16) KeptPoint {  // a rendered point of R \ C waiting for its radius search
    float x, y, z;
    uint32_t pix;                 // its pixel u | v << 16 (the colour is interpolated only if needed)
};

// Per-warp scratch of the radius search (shared memory).
struct __align__(16) WarpProbe {
    int2 runs[27];                // hash: non-empty cells as (start - first candidate, end candidate);
                                  // dense index: runs[r].x of the non-empty rows
    int total;                    // hash: candidates of the group's 27 cells
    unsigned char qlist[32];      // hash: the lanes of the group's queries, in lane order
    float4 q[32];                 // the group's queries as -x, -x, -y, -y (hash: the query of each lane)
    unsigned long long best[32];  // hash: nearest-neighbour key of each lane's query
    float4 stage[64];             // hash: a chunk of the group's candidates, shared by its queries;
                                  // dense index: .xyz = -z, -z, pixel of the group's queries
};

// Per-warp scratch: the radius search and the rasteriser's triangle stage
// use the same bytes (the two phases are separated by block barriers).
constexpr size_t kRasterScratch = 64 * sizeof(uint4) + 21 * sizeof(TriStage);   // its triangle ring and staged triangles
constexpr size_t kWarpScratch = sizeof(WarpProbe) > kRasterScratch ? sizeof(WarpProbe) : kRasterScratch;
static_assert(kWarpQueue * sizeof(float4) >= 64 * 16, "the depth ring fits the kept-point queue it aliases");
static_assert(sizeof(KeptPoint) == 16, "kept-point queue entries are 16 bytes");
static_assert(sizeof(TriStage) == 48, "staged triangles are 48 bytes");
static_assert(kWarpScratch % 16 == 0, "per-warp scratch keeps 16-byte alignment");
static_assert(sizeof(WarpProbe) % 16 == 0, "per-warp scratch keeps 16-byte alignment");

// Warp-cooperative lookup of the 27 cells around cell (gx, gy, gz) in the voxel
// hash (an observation whose cell box is too large for the dense index): lane
// j < 27 probes the table for neighbour j (the table lives in L2, so the loads
// overlap).  The non-empty runs are stored in order with a running candidate
// count, so that candidate i is point runs[r].x + i for the first run r with
// i < runs[r].y.  Returns the number of runs.
__device__ __forceinline__ int lookup_hash(const DevScene& sc, int gx, int gy, int gz, WarpProbe& W, int lane)
{
    uint32_t start = 0, cnt = 0;
    if (lane < 27) {
        const unsigned long long key = cell_key(gx + lane % 3 - 1, gy + (lane / 3) % 3 - 1, gz + lane / 9 - 1);
        uint32_t slot = hash_slot(key, sc.table_mask);
        for (uint32_t probe = 0; probe <= sc.table_mask; ++probe) {
            const uint4 x = __ldg(&sc.table[slot]);
            unsigned long long k = (unsigned long long)x.x | ((unsigned long long)x.y << 32);
            if (k == key) {
                start = x.z;
                cnt = x.w;
                break;
            }
            if (k == kEmptyKey) break;
            slot = (slot + 1) & sc.table_mask;
        }
    }
    uint32_t incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    const unsigned nonempty = __ballot_sync(0xffffffffu, cnt != 0);
    if (cnt != 0)
        W.runs[__popc(nonempty & ((1u << lane) - 1u))] = make_int2((int)start - (int)(incl - cnt), (int)incl);
    if (lane == 31) W.total = (int)incl;
    return __popc(nonempty);
}

// Admissible band of the observed-side keys (jo_mode 1: for every observed
// point of the band, the key (d2 bits << 32 | rendered pixel) of its nearest
// rendered point within delta, kEmptyKey if none).
struct MarkBand {
    uint32_t* marks;
    int u0, u1, v0, v1, vw;
    int* err;                     // debug builds: where index violations are reported
};

// Candidates j, j + k, ... of a staged chunk of n against query q, folded
// into local: the minimum (d2 bits << 32 | pixel) within delta, or kEmptyKey.
// MARK (jo_mode 1) also folds the pair into the key of every observed point
// within delta that lies in the admissible band: its nearest rendered point
// is the smallest (d2, rendered pixel), the rendered pixel carried in q.w.
template <bool MARK>
__device__ __forceinline__ unsigned long long scan_staged(float delta2, const float4 q, const float4* stage,
                                                          int n, int j, int k, const MarkBand& mb,
                                                          unsigned long long local)
{
    for (int i = j; i < n; i += k) {
        const float4 c = stage[i];
        float ex = __fsub_rn(q.x, c.x), ey = __fsub_rn(q.y, c.y), ez = __fsub_rn(q.z, c.z);
        float d2 = __fadd_rn(__fadd_rn(__fmul_rn(ex, ex), __fmul_rn(ey, ey)), __fmul_rn(ez, ez));
        if (d2 <= delta2) {
            unsigned long long key = ((unsigned long long)__float_as_uint(d2) << 32) | __float_as_uint(c.w);
            local = key < local ? key : local;
            if (MARK) {
                const uint32_t pw = __float_as_uint(c.w);
                const int pu = (int)(pw & 0xFFFFu), pv = (int)(pw >> 16);
                if (pu >= mb.u0 && pu < mb.u1 && pv >= mb.v0 && pv < mb.v1) {
                    const int i = (pv - mb.v0) * mb.vw + (pu - mb.u0);
                    atomicMin(reinterpret_cast<unsigned long long*>(mb.marks) + i,
                              ((unsigned long long)__float_as_uint(d2) << 32) | __float_as_uint(q.w));
                }
            }
        }
    }
    return local;
}

// Candidates c0 .. c0 + 63 of a group's runs staged in the warp's shared
// memory (two coalesced loads per lane).  Lane j < (the group's run count)
// holds run j as run = (start - first candidate index, end candidate index)
// (the other lanes: end = INT_MAX); the run of candidate c is the first whose
// end exceeds c, found by a five-step binary search over the lanes.
__device__ __forceinline__ int candidate_point(int2 run, int c)
{
    int r = 0;
#pragma unroll
    for (int step = 16; step >= 1; step >>= 1) {
        const int e = __shfl_sync(0xffffffffu, run.y, r + step - 1);
        if (e <= c) r += step;
    }
    return __shfl_sync(0xffffffffu, run.x, r) + c;
}

__device__ __forceinline__ void stage_chunk(const DevScene& sc, WarpProbe& W, int2 run, int c0, int T, int lane,
                                            int* err)
{
    const int ci = c0 + lane, cj = ci + 32;
    const int pi = candidate_point(run, ci), pj = candidate_point(run, cj);
    if (ci < T && PERCH_CHECKED((unsigned)pi < (unsigned)sc.n_pts, err)) W.stage[lane] = __ldg(&sc.pts[pi]);
    if (cj < T && PERCH_CHECKED((unsigned)pj < (unsigned)sc.n_pts, err)) W.stage[lane + 32] = __ldg(&sc.pts[pj]);
}

// Radius search of up to 32 points through the voxel hash.  Lanes whose points
// fall in the same cell form a group; its 27-cell neighbourhood is looked up
// once, its candidates are staged in shared memory 64 at a time and tested by
// all 32 lanes: floor(32 / G) lanes per query (G = the group's queries) split
// each chunk, each keeps its minimum (d2 bits, pixel) in a register and folds
// it into the query's result with one shared-memory atomicMin.
template <bool MARK>
__device__ __noinline__ unsigned long long probe_hash(const DevScene& sc, bool valid, float4 query, WarpProbe& W,
                                                      int lane, const MarkBand& band)
{
    // copies: the caller's lie in memory that the marks' atomics might change, and were
    // read again for every candidate (Eq. 3 over 700 poses at 1023x455, 2 mm: 11.2
    // against 9.4 ms)
    const MarkBand mb = band;
    const float delta2 = sc.delta2;
    int cx = 0, cy = 0, cz = 0;
    unsigned long long key = kEmptyKey;
    if (valid) {
        cx = cell_coord(query.x, sc.inv_cell);
        cy = cell_coord(query.y, sc.inv_cell);
        cz = cell_coord(query.z, sc.inv_cell);
        if (sc.near_bits) {
            // no observed point in the 27 cells: nothing to look up
            const long long b = near_index(sc, cx, cy, cz);
            valid = b >= 0 && ((__ldg(&sc.near_bits[b >> 5]) >> (b & 31)) & 1u);
        }
        if (valid) key = cell_key(cx, cy, cz);
    }
    W.q[lane] = query;
    W.best[lane] = kEmptyKey;
    const unsigned grp = __match_any_sync(0xffffffffu, key);
    const int leader = __ffs(grp) - 1;
    const int my_pos = __popc(grp & ((1u << lane) - 1u));
    for (unsigned rest = __ballot_sync(0xffffffffu, valid && lane == leader); rest != 0; rest &= rest - 1) {
        const int L = __ffs(rest) - 1;
        if (valid && leader == L) W.qlist[my_pos] = (unsigned char)lane;
        const int nruns = lookup_hash(sc, __shfl_sync(0xffffffffu, cx, L), __shfl_sync(0xffffffffu, cy, L),
                                      __shfl_sync(0xffffffffu, cz, L), W, lane);
        const int G = __popc(__shfl_sync(0xffffffffu, grp, L));
        __syncwarp();
        const int T = W.total;
        // k = floor(32 / G) lanes per query; lane j of a query takes
        // candidates j, j + k, ... of each staged chunk and keeps its
        // minimum in a register
        const int k = c_lanes_per_query[G];
        const int qj = (lane * (int)c_lane_div[k]) >> 10;
        const bool active = lane < G * k;
        const int ql = active ? W.qlist[qj] : 0;
        const float4 q = W.q[ql];
        unsigned long long local = kEmptyKey;
        const int2 run = lane < nruns ? W.runs[lane] : make_int2(0, INT_MAX);
        for (int c0 = 0; c0 < T; c0 += 64) {
            stage_chunk(sc, W, run, c0, T, lane, mb.err);
            __syncwarp();
            const int n = min(64, T - c0);
            if (active) local = scan_staged<MARK>(delta2, q, W.stage, n, lane - qj * k, k, mb, local);
            __syncwarp();
        }
        if (active && local != kEmptyKey) atomicMin(&W.best[ql], local);
        __syncwarp();
    }
    return W.best[lane];
}

// Packed binary32 pairs, each half rounded to nearest like the scalar operation.
// A square is a fused multiply-add of the pair (-0, -0), which changes no bit of
// the product.  The pair is read from constant memory: a packed multiplication,
// or an addend the assembler can see through, is contracted with the addition
// that follows it (.rn and -fmad=false notwithstanding: measured, 22 % of the
// sums then differ in their last bit).
__constant__ unsigned long long c_negzero2 = 0x8000000080000000ull;

__device__ __forceinline__ unsigned long long pack2(float a, float b)
{
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}

__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b)
{
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

__device__ __forceinline__ unsigned long long square2(unsigned long long a)
{
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %1, %2;" : "=l"(r) : "l"(a), "l"(c_negzero2));
    return r;
}

// Bits of the squared distances of a query (negated, each coordinate twice: the
// differences only change sign) to two candidates, by packed binary32 operations
// that round each half as the scalar ones do.  The values are non-negative, so
// the bits order like them; a NaN compares above every radius.
__device__ __forceinline__ uint2 dist2_pair(ulonglong2 qxy, unsigned long long qz, unsigned long long x,
                                            unsigned long long y, unsigned long long z)
{
    const unsigned long long ex = add2(x, qxy.x), ey = add2(y, qxy.y), ez = add2(z, qz);
    const unsigned long long d = add2(add2(square2(ex), square2(ey)), square2(ez));
    return make_uint2((unsigned)d, (unsigned)(d >> 32));
}

// jo_mode 1: fold the pair (query of rendered pixel qpix, observed point of pixel
// pw, squared distance d2) into the observed point's key if the two lie within
// delta of each other and the point in the admissible band.
__device__ __forceinline__ void mark_pair(const MarkBand& mb, unsigned d2, unsigned d2max, uint32_t qpix, uint32_t pw)
{
    if (d2 > d2max) return;
    const int pu = (int)(pw & 0xFFFFu), pv = (int)(pw >> 16);
    if (pu >= mb.u0 && pu < mb.u1 && pv >= mb.v0 && pv < mb.v1)
        atomicMin(reinterpret_cast<unsigned long long*>(mb.marks) + (pv - mb.v0) * mb.vw + (pu - mb.u0),
                  ((unsigned long long)d2 << 32) | qpix);
}

// 32 candidates c .. c + 31 of a group of T (c uniform; lane l takes c + l), one
// per lane.  Lane j < 9 holds row j of the group: cnt points, the first of them
// the group's candidate off.  base[r] is the point index of the r-th non-empty
// row's candidate 0; begun counts the rows begun before c (advanced).
__device__ __forceinline__ float4 group_candidate(const DevScene& sc, const int2* base, int off, int cnt, int c, int T,
                                                  int lane, int& begun, int* err)
{
    const float far = 1.0e30f;                            // beyond every radius: d2 = inf
    float4 p = make_float4(far, far, far, 0.0f);
    const unsigned rel = (unsigned)(off - c);
    const unsigned starts = __reduce_or_sync(0xffffffffu, cnt != 0 && rel < 32u ? 1u << rel : 0u);
    begun += __popc(starts & (0xffffffffu >> (31 - lane)));
    if (c + lane < T) {
        // the candidate lies in the last row begun at or before it
        const int i = base[begun - 1].x + c + lane;
        if (PERCH_CHECKED((unsigned)i < (unsigned)sc.n_pts, err)) p = __ldg(&sc.pts[i]);
    }
    begun = __shfl_sync(0xffffffffu, begun, 31);
    return p;
}

// Radius search of up to 32 points through the dense cell index.  Lanes whose
// points fall in the same cell form a group; the groups are taken in order of
// their cells.  A group's candidates -- nine
// rows of three cells, each row one run of the cell-sorted points -- are held
// two or four per lane in registers, loaded once by coalesced reads; every
// query of the group is then broadcast to them, and the warp's minimum of the
// squared distances and of the pixels that attain it is the query's nearest
// point (two warp-wide integer minima).  The cell box has a border of empty
// cells, so rows that run over its faces only wrap into empty cells or into
// further observed points, which cannot change a nearest neighbour within
// delta; only the ends of the whole index are clamped.  NEAR: the caller has
// tested the near-cell bits.
//
// Bound by instruction issue: about 90 instructions a group and 30 a query per 64
// candidates (45 per 128), against the 16 to 230 candidates of a mean query on
// the tabletop and 6-DoF scenes.  Staging the candidates in shared memory and
// splitting the lanes over the group's queries costs about half as much again
// (155k against 105k warp instructions per pose of an ellipsoid, 771k against
// 487k per 6-DoF pose), and four lanes per query walking its nine rows alone
// 142k and 628k: the longest row of eight queries counts for all of them.
template <bool MARK, bool NEAR>
__device__ __forceinline__ unsigned long long probe_dense(const DevScene& sc, bool valid, float4 query, WarpProbe& W,
                                                          int lane, const MarkBand& mb)
{
    const int nx = sc.near_n[0], nxy = nx * sc.near_n[1], ncell = nxy * sc.near_n[2];
    int cell = -1;
    if (valid) {
        const int ix = cell_coord(query.x, sc.inv_cell) - sc.near_lo[0];
        const int iy = cell_coord(query.y, sc.inv_cell) - sc.near_lo[1];
        const int iz = cell_coord(query.z, sc.inv_cell) - sc.near_lo[2];
        if ((unsigned)ix < (unsigned)nx && (unsigned)iy < (unsigned)sc.near_n[1] && (unsigned)iz < (unsigned)sc.near_n[2]) {
            const int c = iz * nxy + iy * nx + ix;
            if (NEAR || ((__ldg(&sc.near_bits[c >> 5]) >> (c & 31)) & 1u)) cell = c;
        }
    }
    const unsigned lt = (1u << lane) - 1u;
    const unsigned d2max = __float_as_uint(sc.delta2);
    // lane j < 9: from a cell to the first of the three cells of its row j
    const int row_off = (lane % 3 - 1) * nx + (lane / 3 - 1) * nxy - 1;
    unsigned bd = 0xFFFFFFFFu, bp = 0xFFFFFFFFu;          // the lane's own nearest point
    for (;;) {
        // the lowest cell not yet searched (-1, none, is the largest unsigned)
        const int c = (int)__reduce_min_sync(0xffffffffu, (unsigned)cell);
        if (c < 0) break;
        const bool mine = cell == c;
        const unsigned members = __ballot_sync(0xffffffffu, mine);
        const int G = __popc(members), pos = mine ? __popc(members & lt) : -1;
        if (mine) {
            cell = -1;
            W.q[pos] = make_float4(-query.x, -query.x, -query.y, -query.y);
            W.stage[pos] = make_float4(-query.z, -query.z, query.w, 0.0f);
        }
        int s0 = 0, cnt = 0;
        if (lane < 9) {
            s0 = (int)__ldg(&sc.cell_start[min(max(c + row_off, 0), ncell)]);
            cnt = (int)__ldg(&sc.cell_start[min(max(c + row_off + 3, 0), ncell)]) - s0;
        }
        int off = cnt;                                    // the row's first candidate
#pragma unroll
        for (int o = 1; o < 16; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, off, o);
            if (lane >= o) off += t;
        }
        const int T = __shfl_sync(0xffffffffu, off, 8);
        off -= cnt;
        const unsigned nonempty = __ballot_sync(0xffffffffu, cnt != 0);
        if (cnt != 0) W.runs[__popc(nonempty & lt)].x = s0 - off;
        __syncwarp();
        int begun = 0;
#pragma unroll 1
        for (int c0 = 0; c0 < T; c0 += 128) {
            const float4 ca = group_candidate(sc, W.runs, off, cnt, c0, T, lane, begun, mb.err);
            const float4 cb = group_candidate(sc, W.runs, off, cnt, c0 + 32, T, lane, begun, mb.err);
            const unsigned long long x0 = pack2(ca.x, cb.x), y0 = pack2(ca.y, cb.y), z0 = pack2(ca.z, cb.z);
            const unsigned pa = __float_as_uint(ca.w), pb = __float_as_uint(cb.w);
            if (T - c0 <= 64) {
#pragma unroll 1
                for (int i = 0; i < G; ++i) {
                    const ulonglong2 qa = *reinterpret_cast<const ulonglong2*>(&W.q[i]);
                    const unsigned long long qz = *reinterpret_cast<const unsigned long long*>(&W.stage[i]);
                    const uint2 d = dist2_pair(qa, qz, x0, y0, z0);
                    if (MARK) {
                        const uint32_t qp = __float_as_uint(W.stage[i].z);
                        mark_pair(mb, d.x, d2max, qp, pa);
                        mark_pair(mb, d.y, d2max, qp, pb);
                    }
                    const unsigned dm = __reduce_min_sync(0xffffffffu, min(d.x, d.y));
                    if (dm > d2max) continue;
                    const unsigned pm = __reduce_min_sync(
                        0xffffffffu, min(d.x == dm ? pa : 0xFFFFFFFFu, d.y == dm ? pb : 0xFFFFFFFFu));
                    if (pos == i && (dm < bd || (dm == bd && pm < bp))) {
                        bd = dm;
                        bp = pm;
                    }
                }
            } else {
                const float4 cc = group_candidate(sc, W.runs, off, cnt, c0 + 64, T, lane, begun, mb.err);
                const float4 cd = group_candidate(sc, W.runs, off, cnt, c0 + 96, T, lane, begun, mb.err);
                const unsigned long long x1 = pack2(cc.x, cd.x), y1 = pack2(cc.y, cd.y), z1 = pack2(cc.z, cd.z);
                const unsigned pc = __float_as_uint(cc.w), pd = __float_as_uint(cd.w);
#pragma unroll 1
                for (int i = 0; i < G; ++i) {
                    const ulonglong2 qa = *reinterpret_cast<const ulonglong2*>(&W.q[i]);
                    const unsigned long long qz = *reinterpret_cast<const unsigned long long*>(&W.stage[i]);
                    const uint2 d = dist2_pair(qa, qz, x0, y0, z0), e = dist2_pair(qa, qz, x1, y1, z1);
                    if (MARK) {
                        const uint32_t qp = __float_as_uint(W.stage[i].z);
                        mark_pair(mb, d.x, d2max, qp, pa);
                        mark_pair(mb, d.y, d2max, qp, pb);
                        mark_pair(mb, e.x, d2max, qp, pc);
                        mark_pair(mb, e.y, d2max, qp, pd);
                    }
                    const unsigned dm = __reduce_min_sync(0xffffffffu, min(min(d.x, d.y), min(e.x, e.y)));
                    if (dm > d2max) continue;
                    const unsigned pm = __reduce_min_sync(
                        0xffffffffu, min(min(d.x == dm ? pa : 0xFFFFFFFFu, d.y == dm ? pb : 0xFFFFFFFFu),
                                         min(e.x == dm ? pc : 0xFFFFFFFFu, e.y == dm ? pd : 0xFFFFFFFFu)));
                    if (pos == i && (dm < bd || (dm == bd && pm < bp))) {
                        bd = dm;
                        bp = pm;
                    }
                }
            }
        }
        __syncwarp();
    }
    return ((unsigned long long)bd << 32) | bp;
}

// Radius search for up to 32 queued points (one per lane; `valid` marks the
// lanes holding one).  Returns the lane's own result: the nearest observed
// point within delta (smallest FP32 squared distance, ties to the lowest pixel)
// as (d2 bits << 32 | pixel), or kEmptyKey.  All 32 lanes must call it.
template <bool MARK, bool NEAR>
__device__ __forceinline__ unsigned long long probe_batch(const DevScene& sc, bool valid, float qx, float qy, float qz,
                                                          uint32_t qpix, WarpProbe& W, int lane, const MarkBand& mb)
{
    const float4 q = make_float4(qx, qy, qz, __uint_as_float(qpix));
    return sc.cell_start ? probe_dense<MARK, NEAR>(sc, valid, q, W, lane, mb) : probe_hash<MARK>(sc, valid, q, W, lane, mb);
}

// Conservative pixel box of an object-frame box [lo,hi] at pose P (2 px
// margin), clipped to [cu0,cu1) x [cv0,cv1).  Falls back to the clip box
// when a corner is not in front of the camera.  Also returns the largest Z.
// A whole warp calls it, corner c in lanes c, c + 8, ...: one corner's latency
// instead of eight, and a fraction of the code (the kernel's loops compete for
// the instruction cache, so it is also called, not inlined).
struct PixelBox {
    int4 box;
    float zmax;
};

__device__ __noinline__ PixelBox project_box(float4 camera, const float* P, float3 lo, float3 hi, int4 clip)
{
    const int lane = threadIdx.x & 31;
    const float x = (lane & 1) ? hi.x : lo.x;
    const float y = (lane & 2) ? hi.y : lo.y;
    const float z = (lane & 4) ? hi.z : lo.z;
    const float X = P[0] * x + P[1] * y + P[2] * z + P[3];
    const float Y = P[4] * x + P[5] * y + P[6] * z + P[7];
    const float Z = P[8] * x + P[9] * y + P[10] * z + P[11];
    float zm = fmaxf(-3.0e38f, Z), umin = 3.0e38f, umax = -3.0e38f, vmin = 3.0e38f, vmax = -3.0e38f;
    const bool front = Z > 1e-4f;
    if (front) {
        const float u = camera.x * div_any(X, Z) + camera.z, v = camera.y * div_any(Y, Z) + camera.w;
        umin = fminf(umin, u); umax = fmaxf(umax, u);
        vmin = fminf(vmin, v); vmax = fmaxf(vmax, v);
    }
#pragma unroll 1
    for (int o = 4; o > 0; o >>= 1) {
        zm = fmaxf(zm, __shfl_xor_sync(0xffffffffu, zm, o));
        umin = fminf(umin, __shfl_xor_sync(0xffffffffu, umin, o));
        umax = fmaxf(umax, __shfl_xor_sync(0xffffffffu, umax, o));
        vmin = fminf(vmin, __shfl_xor_sync(0xffffffffu, vmin, o));
        vmax = fmaxf(vmax, __shfl_xor_sync(0xffffffffu, vmax, o));
    }
    const bool ok = __ballot_sync(0xffffffffu, !front) == 0u;
    PixelBox r = {clip, zm};
    if (ok && umax - umin < 1.0e7f && vmax - vmin < 1.0e7f) {
        const int u0 = (int)floorf(fmaxf(umin, -1.0e7f)) - 2, u1 = (int)ceilf(fminf(umax, 1.0e7f)) + 3;
        const int v0 = (int)floorf(fmaxf(vmin, -1.0e7f)) - 2, v1 = (int)ceilf(fminf(vmax, 1.0e7f)) + 3;
        r.box.x = max(u0, clip.x);
        r.box.y = max(v0, clip.y);
        r.box.z = max(min(u1, clip.z), r.box.x);
        r.box.w = max(min(v1, clip.w), r.box.y);
    }
    return r;
}

// Shared-memory carve-up of one scoring block.
struct ScoreSmem {
    uint32_t* zbuf;               // z-buffer tile (32- or 64-bit keys), at offset 0
    uint32_t* marks;              // admissible-band bitset
    int* next_batch;
    int* refused;                 // tree edges: the object would occlude a placed one
    int* bin_cnt;                 // kBinTiles: triangles binned per z-buffer tile
    int* jo_next;                 // plain scoring: next chunk of J_o's |I cap V|
    int* vbounds;                 // snapped vertex bounds of the hypothesis (vertex_pass)
};

// rint(x) for |x| < 2^22: adding 1.5 x 2^23 rounds to an integer, ties to even,
// and leaves it in the low bits (a conversion holds its unit for eight issue
// slots; the vertex pass is a sixteenth of a search).
__device__ __forceinline__ int rint_small(float x)
{
    return __float_as_int(__fadd_rn(x, 12582912.0f)) - 0x4B400000;
}

// ---- per-hypothesis vertex cache (one slot of global scratch per block) ----
//
// Each vertex is transformed, projected and snapped once per hypothesis and
// kept as (x16, y16 : unsigned 16 bits, biased by kSnapBias, 1/Z : float), so
// that a triangle's box comes from packed unsigned minima and maxima; a vertex
// that fails the near-plane or guard-band test is stored as x16 = y16 = 0xFFFF,
// which culls every triangle that uses it.  Used when W and H are at most 1023
// (snapped coordinates in [-16 x 1023, 32 x 1023)).
constexpr int kSnapBias = 1 << 14;            // 1024 pixels in 1/16 px
constexpr uint32_t kCulledXY = 0xFFFFFFFFu;

// bounds (optional, shared memory, initialised to INT_MAX, INT_MAX, INT_MIN,
// INT_MIN): the smallest and largest snapped x and y of the vertices kept.
__device__ __forceinline__ void vertex_pass(const DevScene& sc, const DevMesh& m, const float* P,
                                            unsigned long long* vc, int nt, int* bounds = nullptr)
{
    const float gx0 = (float)(-16 * sc.W), gx1 = (float)(32 * sc.W);
    const float gy0 = (float)(-16 * sc.H), gy1 = (float)(32 * sc.H);
    int xmin = INT_MAX, ymin = INT_MAX, xmax = INT_MIN, ymax = INT_MIN;
#pragma unroll 1
    for (int i = threadIdx.x; i < m.n_verts; i += nt) {
        float4 v = __ldg(&m.verts[i]);
        float X = __fadd_rn(__fadd_rn(__fadd_rn(__fmul_rn(P[0], v.x), __fmul_rn(P[1], v.y)),
                                      __fmul_rn(P[2], v.z)), P[3]);
        float Y = __fadd_rn(__fadd_rn(__fadd_rn(__fmul_rn(P[4], v.x), __fmul_rn(P[5], v.y)),
                                      __fmul_rn(P[6], v.z)), P[7]);
        float Z = __fadd_rn(__fadd_rn(__fadd_rn(__fmul_rn(P[8], v.x), __fmul_rn(P[9], v.y)),
                                      __fmul_rn(P[10], v.z)), P[11]);
        unsigned long long rec = kCulledXY;
        if (Z >= sc.z_near) {
            const float iz = __frcp_rn(Z);
            float xz, yz;
            const float small = fminf(fabsf(X), fminf(fabsf(Y), Z)), large = fmaxf(fabsf(X), fmaxf(fabsf(Y), Z));
            if (small > kDivLo && large < kDivHi) {
                xz = div_by(X, Z, iz);
                yz = div_by(Y, Z, iz);
            } else {
                xz = div_any(X, Z);
                yz = div_any(Y, Z);
            }
            const float sx = __fmul_rn(__fadd_rn(__fmul_rn(sc.fx, xz), sc.cx), 16.0f);
            const float sy = __fmul_rn(__fadd_rn(__fmul_rn(sc.fy, yz), sc.cy), 16.0f);
            if (sx >= gx0 && sx < gx1 && sy >= gy0 && sy < gy1) {
                const int xi = rint_small(sx), yi = rint_small(sy);
                xmin = min(xmin, xi); xmax = max(xmax, xi);
                ymin = min(ymin, yi); ymax = max(ymax, yi);
                rec = (unsigned long long)((uint32_t)(xi + kSnapBias) | ((uint32_t)(yi + kSnapBias) << 16)) |
                      ((unsigned long long)__float_as_uint(iz) << 32);
            }
        }
        vc[i] = rec;
    }
    if (bounds) {
        xmin = __reduce_min_sync(0xffffffffu, xmin);
        ymin = __reduce_min_sync(0xffffffffu, ymin);
        xmax = __reduce_max_sync(0xffffffffu, xmax);
        ymax = __reduce_max_sync(0xffffffffu, ymax);
        if ((threadIdx.x & 31) == 0) {
            atomicMin(&bounds[0], xmin);
            atomicMin(&bounds[1], ymin);
            atomicMax(&bounds[2], xmax);
            atomicMax(&bounds[3], ymax);
        }
    }
}

__device__ __forceinline__ bool load_cached(const unsigned long long* vc, int4 tv, TriSetup& o)
{
    // the three records are loaded before any is tested, so that all three
    // loads are in flight together
    const unsigned long long rec[3] = {vc[tv.x], vc[tv.y], vc[tv.z]};
    const int vids[3] = {tv.x, tv.y, tv.z};
    bool ok = true;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const unsigned long long r = rec[k];
        ok = ok && (uint32_t)r != kCulledXY;
        o.x[k] = (int)(r & 0xFFFFu) - kSnapBias;
        o.y[k] = (int)((r >> 16) & 0xFFFFu) - kSnapBias;
        o.iz[k] = __uint_as_float((uint32_t)(r >> 32));
        o.vid[k] = vids[k];
    }
    return ok;
}

// Triangle t (its vertex ids tv) loaded at pose P: from the vertex cache, or
// transformed and snapped here.  False if culled.
template <bool VC>
__device__ __forceinline__ bool load_tri(const DevScene& sc, const DevMesh& m, const float* P,
                                         const unsigned long long* vc, int4 tv, TriSetup& o)
{
    if (VC) return load_cached(vc, tv, o);
    return load_triangle(sc, m.verts, P, tv, o);
}

// Full set-up of triangle t at pose P: load, then orientation.  False if
// culled or degenerate.
template <bool VC>
__device__ __forceinline__ bool get_triangle(const DevScene& sc, const DevMesh& m, const float* P,
                                             const unsigned long long* vc, int t, TriSetup& o)
{
    return load_tri<VC>(sc, m, P, vc, __ldg(&m.tris[t]), o) && orient_triangle(o);
}

// ---- rasteriser: rings of triangles and covered samples --------------------
//
// A fine mesh leaves few lanes of a warp anything to do at a time: a third to a
// half of its triangles hold no sample, and about one sample in four that is
// tested is covered.  So the triangles whose boxes hold samples are queued in
// shared memory and set up by 32 full lanes, and the covered samples are queued
// again until 32 of them can have their depth (a division) and z-buffer update.
constexpr int kRing = 64;         // entries of a warp's ring of triangles or samples
constexpr int kStaged = 21;       // larger triangles expanded at a time (the scratch's size)
constexpr int kTinyBox = 8;       // boxes of up to this many samples are walked in one lane

// A covered sample: edges 0 and 1 less their tie bias, the triangle, and the
// z-buffer index with the biases in bits 16 and 17.
struct __align__(16) DepthItem {
    int t0, t1, tri;
    unsigned idx;
};

extern __shared__ __align__(16) unsigned char g_smem[];

// The rasteriser's arguments, by value: it is called, not inlined, so that its
// loops have the registers to themselves (inlined, they ran from spilled
// values).  Shared-memory places are byte offsets from the block's base, so that
// every access is a shared-memory one.
struct RasterArgs {
    const int4* tris;
    const unsigned long long* vc; // vertex cache (raster_whole: nullptr)
    const int* list;              // the tile's bin, or nullptr: triangles 0 .. n - 1
    int n;
    int tu0, tv0, tu1, tv1, tw;   // tile [tu0,tu1) x [tv0,tv1), row pitch tw
    unsigned scratch, ring;       // the warp's triangle ring and staged triangles; its depth ring
    int* err;
};

// Depth and z-buffer update of the n <= 32 oldest samples of the ring at `at`:
// the triangle is read again (its weights and 1/Z in the orientation's order),
// z = A / ((w0/Z0 + w1/Z1) + w2/Z2) with one division, d = rint(10000 z).
template <bool K32>
__device__ __forceinline__ void depth_flush(const RasterArgs& a, int at, int n, int lane)
{
    __syncwarp();
    if (lane < n) {
        const DepthItem e = reinterpret_cast<const DepthItem*>(g_smem + a.ring)[(at + lane) & (kRing - 1)];
        const int4 tv = __ldg(&a.tris[e.tri]);
        TriSetup o;
        load_cached(a.vc, tv, o);
        const int A = edge_fn(o.x[0], o.y[0], o.x[1], o.y[1], o.x[2], o.y[2]);
        const int idx = (int)(e.idx & 0xFFFFu);
        const int w0 = e.t0 + (int)((e.idx >> 16) & 1u), wa = e.t1 + (int)((e.idx >> 17) & 1u);
        const int wb = (int)((unsigned)abs(A) - (unsigned)w0 - (unsigned)wa);
        // a triangle of negative area has its vertices 1 and 2 exchanged
        const float f1 = __fmul_rn(__int2float_rn(wa), o.iz[1]), f2 = __fmul_rn(__int2float_rn(wb), o.iz[2]);
        const float f0 = __fmul_rn(__int2float_rn(w0), o.iz[0]);
        const float num = __fadd_rn(__fadd_rn(f0, A < 0 ? f2 : f1), A < 0 ? f1 : f2);
        const float dz = __fmul_rn(__fdiv_rn(__int2float_rn(abs(A)), num), 10000.0f);
        // dz >= 0 (every weight and 1/Z is), so dz in [0, 2^32) rounds to
        // nearest in 32 bits (the largest binary32 below 2^32 is an integer)
        if (dz < 4294967296.0f && PERCH_CHECKED((unsigned)idx < (unsigned)(a.tw * (a.tv1 - a.tv0)), a.err)) {
            const unsigned d = __float2uint_rn(dz);
            if (d >= 1u) zmin<K32>(reinterpret_cast<uint32_t*>(g_smem), idx, d, e.tri, a.err);
        }
    }
    __syncwarp();
}

// Rasterise triangles at a pose into the z-buffer tile at the start of the
// block's shared memory.  A warp reads 32 triangles at a time and queues those
// whose pixel box holds a sample of the tile; 32 queued ones are set up, one per
// lane.  Boxes of up to kTinyBox samples are walked in their lanes by edge
// increments.  Larger triangles are staged in shared memory (kStaged at a time,
// the rest go back to the queue) and their items -- samples, or rows when the
// triangle covers less than a quarter of its box, like the wedges of a can's end
// caps -- spread over the lanes; a row is narrowed to the samples between the
// edges (with a margin; coverage is still tested) and walked by its lane.
// Covered samples go through the depth ring.  No barrier inside.
//
// Bound by instruction issue: the two rings keep the lanes full, and the walk,
// the depth and the set-up each stand in the code once, because the kernel's
// loops together are at the size of the instruction cache (a version with the
// walk and the depth inlined three times issued fewer instructions and took 1.5
// times as long, 5 to 9 warps in 16 waiting for instructions).  A render of a
// 20,000-triangle ellipsoid or a 9,984-triangle can costs 127k and 122k warp
// instructions, against 202k and 159k without the triangle ring.  With it, three
// 640x480 objects x 29,584 poses 42.0 -> 36.2 ms, five 6-DoF objects of 30,000
// triangles x 4,096 poses 1.41 times the former rate.
template <int NT, bool K32>
__device__ __noinline__ void raster_tile(const RasterArgs a)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    uint4* const TR = reinterpret_cast<uint4*>(g_smem + a.scratch);
    TriStage* const TS = reinterpret_cast<TriStage*>(g_smem + a.scratch + kRing * sizeof(uint4));
    DepthItem* const DQ = reinterpret_cast<DepthItem*>(g_smem + a.ring);
    int head = 0, count = 0, dhead = 0, dcount = 0;     // the rings of triangles and samples
    constexpr int kPix = kSnapBias / 16;                // pixels are biased like the cached coordinates
    const uint32_t tlo = (uint32_t)(a.tu0 + kPix) | ((uint32_t)(a.tv0 + kPix) << 16);
    const uint32_t thi = (uint32_t)(a.tu1 - 1 + kPix) | ((uint32_t)(a.tv1 - 1 + kPix) << 16);
    // vertex ids are loaded two iterations ahead, the vertices' snapped positions
    // (the low halves of their records) one
    int base = warp * 32, t_next = base + lane;
    uint4 e_next = make_uint4(0u, 0u, 0u, 0u);          // positions and id of the next triangle
    int4 tv_next = make_int4(0, 0, 0, 0);               // vertex ids of the one after it
    if (base + lane < a.n) {
        if (a.list) t_next = a.list[t_next];
        e_next.w = (unsigned)t_next;
        tv_next = __ldg(&a.tris[t_next]);
        e_next.x = (uint32_t)a.vc[tv_next.x]; e_next.y = (uint32_t)a.vc[tv_next.y]; e_next.z = (uint32_t)a.vc[tv_next.z];
    }
    if (base + lane + NT < a.n) {
        t_next = a.list ? a.list[base + lane + NT] : base + lane + NT;
        tv_next = __ldg(&a.tris[t_next]);
    }
    for (;;) {
        if (count < 32 && base < a.n) {
            const int i = base + lane;
            const int4 tv = tv_next;
            uint4 e = e_next;
            if (i + NT < a.n) {
                e_next = make_uint4((uint32_t)a.vc[tv.x], (uint32_t)a.vc[tv.y], (uint32_t)a.vc[tv.z], (unsigned)t_next);
                if (i + 2 * NT < a.n) {
                    t_next = a.list ? a.list[i + 2 * NT] : i + 2 * NT;
                    tv_next = __ldg(&a.tris[t_next]);
                }
            }
            base += NT;
            bool some = false;
            if (i < a.n) {
                const uint32_t lo = __vimin3_u16x2(e.x, e.y, e.z), hi = __vimax3_u16x2(e.x, e.y, e.z);
                const uint32_t pl = __vmaxu2(((lo + 0x000F000Fu) >> 4) & 0x0FFF0FFFu, tlo);
                const uint32_t ph = __vminu2((hi >> 4) & 0x0FFF0FFFu, thi);
                some = __vmaxu2(pl, ph) == ph && (hi & 0xFFFFu) != 0xFFFFu;
            }
            const unsigned bal = __ballot_sync(0xffffffffu, some);
            if (some) TR[(head + count + __popc(bal & lt)) & (kRing - 1)] = e;
            count += __popc(bal);
            continue;
        }
        const bool last = count == 0;                   // only covered samples left
        if (last && dcount == 0) break;
        __syncwarp();
        // ---- set-up of the 32 oldest, one per lane: sample state (x0, x1, K, tri,
        // idx), per column (a0, a1) and, at the end of a row of bw, (r0, r1)
        int x0, x1, K, tri, a0, a1, r0, r1, bw, left, items = 0, first, total;
        unsigned idx;
        {
            const bool have = lane < count;
            const uint4 e = TR[(head + lane) & (kRing - 1)];
            tri = (int)e.w;
            head = (head + 32) & (kRing - 1);
            count = max(0, count - 32);
            const uint32_t lo = __vimin3_u16x2(e.x, e.y, e.z), hi = __vimax3_u16x2(e.x, e.y, e.z);
            const uint32_t pl = __vmaxu2(((lo + 0x000F000Fu) >> 4) & 0x0FFF0FFFu, tlo);
            const uint32_t ph = __vminu2((hi >> 4) & 0x0FFF0FFFu, thi);
            const int u0 = (int)(pl & 0xFFFFu), v0 = (int)(pl >> 16), bh = (int)(ph >> 16) - v0 + 1;
            bw = (int)(ph & 0xFFFFu) - u0 + 1;
            const int x[3] = {(int)(e.x & 0xFFFFu), (int)(e.y & 0xFFFFu), (int)(e.z & 0xFFFFu)};
            const int y[3] = {(int)(e.x >> 16), (int)(e.y >> 16), (int)(e.z >> 16)};
            // edge i runs from vertex i + 1 to vertex i + 2 (mod 3), all reversed when
            // the area is negative (two-sided rendering)
            int A = edge_fn(x[0], y[0], x[1], y[1], x[2], y[2]);
            const int sg = A < 0 ? -1 : 1;
            A = abs(A);
            const int area = have && A != 0 ? bw * bh : 0;  // 0: nothing to do
            const int dx0 = sg * (x[2] - x[1]), dy0 = sg * (y[2] - y[1]), dx1 = sg * (x[0] - x[2]), dy1 = sg * (y[0] - y[2]);
            const int n0 = owns(dx0, dy0) ? 0 : 1, n1 = owns(dx1, dy1) ? 0 : 1;
            K = A - n0 - n1 - (owns(sg * (x[1] - x[0]), sg * (y[1] - y[0])) ? 0 : 1);
            a0 = -16 * dy0; a1 = -16 * dy1;
            // edge values at the box's first sample, less the tie bias
            x0 = (int)((unsigned)dx0 * (unsigned)(16 * v0 - y[1]) - (unsigned)dy0 * (unsigned)(16 * u0 - x[1]) - (unsigned)n0);
            x1 = (int)((unsigned)dx1 * (unsigned)(16 * v0 - y[2]) - (unsigned)dy1 * (unsigned)(16 * u0 - x[2]) - (unsigned)n1);
            idx = (unsigned)((v0 - kPix - a.tv0) * a.tw + (u0 - kPix - a.tu0)) | (unsigned)((n0 << 16) | (n1 << 17));
            left = area <= kTinyBox ? area : 0;
            r0 = 16 * dx0 - (bw - 1) * a0;
            r1 = 16 * dx1 - (bw - 1) * a1;
            // ---- the larger boxes: staged, or back to the queue
            const unsigned big = __ballot_sync(0xffffffffu, area > kTinyBox);
            first = total = 0;
            if (big != 0u) {
                const int rank = __popc(big & lt), n_big = __popc(big);
                if (area > kTinyBox && rank >= kStaged) TR[(head + count + rank - kStaged) & (kRing - 1)] = e;
                count += max(0, n_big - kStaged);
                // thin: the triangle's area (A / 512 samples) is under a quarter of the box's
                const bool thin = bw > 2 && (long long)A < 128ll * area;
                items = area > kTinyBox && rank < kStaged ? (thin ? bh : area) : 0;
                first = items;
#pragma unroll
                for (int off = 1; off < 32; off <<= 1) {
                    const int v = __shfl_up_sync(0xffffffffu, first, off);
                    if (lane >= off) first += v;
                }
                total = __shfl_sync(0xffffffffu, first, 31);
                first -= items;
                if (items > 0)
                    TS[rank] = TriStage{a0, a1, 16 * dx0, 16 * dx1, x0, x1, K, tri, idx | (thin ? 1u << 18 : 0u), bw,
                                        __frcp_rn(__int2float_rn(bw)), first};
                __syncwarp();
            }
        }
        int du = bw, begun = 0;                         // begun: staged triangles whose items began before f0
        for (int f0 = 0;; f0 += 32) {
            // ---- walk the lanes' samples
            while (__ballot_sync(0xffffffffu, left > 0) != 0u || (last && dcount > 0)) {
                // covered: every edge value, less its tie bias, is non-negative
                const bool cov = left > 0 && (x0 | x1 | (int)((unsigned)K - (unsigned)x0 - (unsigned)x1)) >= 0;
                const unsigned bal = __ballot_sync(0xffffffffu, cov);
                if (cov) DQ[(dhead + dcount + __popc(bal & lt)) & (kRing - 1)] = DepthItem{x0, x1, tri, idx};
                dcount += __popc(bal);
                --left;
                const bool wrap = --du == 0;            // on to the next row
                x0 = (int)((unsigned)x0 + (unsigned)(wrap ? r0 : a0));
                x1 = (int)((unsigned)x1 + (unsigned)(wrap ? r1 : a1));
                idx += wrap ? (unsigned)(a.tw - (bw - 1)) : 1u;
                if (wrap) du = bw;
                if (dcount >= 32 || last) {
                    const int n = min(dcount, 32);
                    depth_flush<K32>(a, dhead, n, lane);
                    dhead = (dhead + n) & (kRing - 1);
                    dcount -= n;
                }
            }
            if (f0 >= total) break;
            // ---- the next 32 items: item f belongs to the last triangle begun at or before it
            const unsigned rel = (unsigned)(first - f0);
            const unsigned starts = __reduce_or_sync(0xffffffffu, items > 0 && rel < 32u ? 1u << rel : 0u);
            begun += __popc(starts & (lt | (1u << lane)));
            const TriStage s = TS[begun - 1];
            begun = __shfl_sync(0xffffffffu, begun, 31);
            const int f = f0 + lane, local = f - s.first;
            int u, v = local;                           // the item's samples: `left` of row v from column u
            x0 = s.t0; x1 = s.t1; K = s.K; tri = s.tri; a0 = s.a0; a1 = s.a1;
            if (s.idx & (1u << 18)) {
                x0 = (int)((unsigned)x0 + (unsigned)s.b0 * (unsigned)v);
                x1 = (int)((unsigned)x1 + (unsigned)s.b1 * (unsigned)v);
                // where the row crosses the edges: u < 2^16 and the quotient's relative
                // error is below 2^-21, so the margin of 1/16 keeps every covered sample
                float lo = 0.0f, hi = (float)(s.bw - 1);
                const int xs[3] = {x0, x1, (int)((unsigned)K - (unsigned)x0 - (unsigned)x1)};
                const int as[3] = {a0, a1, -a0 - a1};
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const float r = __fdividef(-__int2float_rn(xs[k]), __int2float_rn(as[k]));
                    if (as[k] > 0) lo = fmaxf(lo, r - 0.0625f);
                    else if (as[k] < 0) hi = fminf(hi, r + 0.0625f);
                    else if (xs[k] < 0) hi = -1.0f;
                }
                u = __float2int_ru(fminf(lo, 65536.0f));
                left = __float2int_rd(fmaxf(hi, -1.0f)) - u + 1;
            } else {
                v = __float2int_rz(__fmul_rn(__int2float_rn(local), s.rbw));
                const int r = local - v * s.bw;
                v += (r >= s.bw) - (r < 0);
                u = local - v * s.bw;
                left = 1;
                x0 = (int)((unsigned)x0 + (unsigned)s.b0 * (unsigned)v);
                x1 = (int)((unsigned)x1 + (unsigned)s.b1 * (unsigned)v);
            }
            if (f >= total) left = 0;
            x0 = (int)((unsigned)x0 + (unsigned)a0 * (unsigned)u);
            x1 = (int)((unsigned)x1 + (unsigned)a1 * (unsigned)u);
            idx = (s.idx & 0x3FFFFu) + (unsigned)(v * a.tw + u);
            du = INT_MAX;
        }
    }
}

// ---- rasteriser of staged triangles: large ones, or no vertex cache (images over 1023
// pixels, or a block that found no cache slot)

struct RasterCamera {             // without the vertex cache
    const float4* verts;
    const float* P;
    int W, H;
    float fx, fy, cx, cy, z_near;
};
struct CachedVertices {};         // with it

// A triangle staged with all that its samples need, since its vertices would have to
// be transformed again (64 bytes, 4 x 16-byte moves): TriStage's fields, and the
// doubled area and the 1/Z of its vertices in the orientation's order.
struct __align__(16) TriWhole {
    int a0, a1, b0, b1;
    int t0, t1, K, A;
    float iz0, iz1, iz2;
    int tri;
    unsigned idx;                 // z-buffer index of the first sample | tie biases of edges 0 and 1 in bits 16 and 17
    int bw;
    float rbw;
    int first;
};
static_assert(32 * sizeof(TriWhole) <= kWarpScratch, "a warp's triangles fit its scratch");

// A triangle's snapped positions and 1/Z, from the vertex cache or transformed here.
__device__ __forceinline__ bool load_whole(const RasterArgs& a, CachedVertices, int4 tv, TriSetup& o)
{
    return load_cached(a.vc, tv, o);
}
__device__ __forceinline__ bool load_whole(const RasterArgs&, const RasterCamera& c, int4 tv, TriSetup& o)
{
    return load_triangle(c, c.verts, c.P, tv, o);
}

// Coverage, depth and z-buffer update of one sample of a staged triangle: x0 and x1 are
// edges 0 and 1 there less their tie bias, idx its place in the tile of cap words.
template <bool K32>
__device__ __forceinline__ void whole_sample(const TriWhole& s, int x0, int x1, int idx, int cap, int* err)
{
    if ((x0 | x1 | (int)((unsigned)s.K - (unsigned)x0 - (unsigned)x1)) < 0) return;
    if (!PERCH_CHECKED((unsigned)idx < (unsigned)cap, err)) return;
    uint32_t* const zbuf = reinterpret_cast<uint32_t*>(g_smem);
    // Early out for a sample that cannot beat the depth already stored here: its depth
    // is at least 1e4 / max(1/Z) less a few 2^-24 relative, so if max(1/Z) (d_here + 2)
    // < 9999 its depth is at least d_here + 2 and its key is larger.  The stored key
    // only decreases, so reading it while other samples update it can only make this
    // test skip less.
    unsigned dh;
    if (K32) {
        const uint32_t w = zbuf[idx];
        dh = w == 0xFFFFFFFFu ? 0xFFFFFFFFu : (w >> 16);
    } else {
        const unsigned long long w = reinterpret_cast<const unsigned long long*>(zbuf)[idx];
        dh = w == kEmptyKey ? 0xFFFFFFFFu : (unsigned)(w >> 32);
    }
    const float izmax = fmaxf(s.iz0, fmaxf(s.iz1, s.iz2));
    if (dh < 0xFFFFFFF0u && __fmul_rn(izmax, __uint2float_rn(dh + 2u)) < 9999.0f) return;
    const int w0 = x0 + (int)((s.idx >> 16) & 1u), w1 = x1 + (int)((s.idx >> 17) & 1u);
    const int w2 = (int)((unsigned)s.A - (unsigned)w0 - (unsigned)w1);
    const float num = __fadd_rn(__fadd_rn(__fmul_rn(__int2float_rn(w0), s.iz0), __fmul_rn(__int2float_rn(w1), s.iz1)),
                                __fmul_rn(__int2float_rn(w2), s.iz2));
    const float dz = __fmul_rn(__fdiv_rn(__int2float_rn(s.A), num), 10000.0f);
    if (dz < 4294967296.0f) {                           // (as in depth_flush)
        const unsigned d = __float2uint_rn(dz);
        if (d >= 1u) zmin<K32>(zbuf, idx, d, s.tri, err);
    }
}

// The tile's triangles, 32 at a time, one per lane: loaded and set up once.
// Boxes of one sample are tested in their lanes; the others are staged and their
// samples spread evenly over the lanes.  Without the cache every z-buffer tile
// transforms the mesh again; reading a triangle's vertices for its set-up and for each
// covered sample too, as raster_tile does, took 1.1 to 1.8 times as long (700 poses at
// 1,200x380, 20,000 triangles, stride 2: 2.47 against 1.35 ms).
template <int NT, bool K32, class Camera>
__device__ __noinline__ void raster_whole(const RasterArgs a, const Camera cam)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    TriWhole* const TS = reinterpret_cast<TriWhole*>(g_smem + a.scratch);
    const int cap = a.tw * (a.tv1 - a.tv0);
    int t_next = 0;                                     // the lane's next triangle, loaded one iteration ahead
    int4 tv_next = make_int4(0, 0, 0, 0);
    if (warp * 32 + lane < a.n) {
        t_next = a.list ? a.list[warp * 32 + lane] : warp * 32 + lane;
        tv_next = __ldg(&a.tris[t_next]);
    }
    for (int base = warp * 32; base < a.n; base += NT) {
        const int i = base + lane, t = t_next;
        const int4 tv = tv_next;
        if (i + NT < a.n) {
            t_next = a.list ? a.list[i + NT] : i + NT;
            tv_next = __ldg(&a.tris[t_next]);
        }
        int area = 0;
        TriWhole s = {};
        TriSetup o;
        // the box first: many triangles hold no sample of the tile
        if (i < a.n && load_whole(a, cam, tv, o)) {
            const int u0 = max(ceil16(min(o.x[0], min(o.x[1], o.x[2]))), a.tu0);
            const int u1 = min(floor16(max(o.x[0], max(o.x[1], o.x[2]))), a.tu1 - 1);
            const int v0 = max(ceil16(min(o.y[0], min(o.y[1], o.y[2]))), a.tv0);
            const int v1 = min(floor16(max(o.y[0], max(o.y[1], o.y[2]))), a.tv1 - 1);
            if (u0 <= u1 && v0 <= v1 && orient_triangle(o)) {
                const int dx0 = o.x[2] - o.x[1], dy0 = o.y[2] - o.y[1], dx1 = o.x[0] - o.x[2], dy1 = o.y[0] - o.y[2];
                const int n0 = owns(dx0, dy0) ? 0 : 1, n1 = owns(dx1, dy1) ? 0 : 1;
                s.a0 = -16 * dy0; s.a1 = -16 * dy1;
                s.b0 = 16 * dx0; s.b1 = 16 * dx1;
                s.t0 = (int)((unsigned)dx0 * (unsigned)(16 * v0 - o.y[1]) - (unsigned)dy0 * (unsigned)(16 * u0 - o.x[1]) -
                             (unsigned)n0);
                s.t1 = (int)((unsigned)dx1 * (unsigned)(16 * v0 - o.y[2]) - (unsigned)dy1 * (unsigned)(16 * u0 - o.x[2]) -
                             (unsigned)n1);
                s.K = o.A - n0 - n1 - (owns(o.x[1] - o.x[0], o.y[1] - o.y[0]) ? 0 : 1);
                s.A = o.A;
                s.iz0 = o.iz[0]; s.iz1 = o.iz[1]; s.iz2 = o.iz[2];
                s.tri = t;
                s.idx = (unsigned)((v0 - a.tv0) * a.tw + (u0 - a.tu0)) | (unsigned)((n0 << 16) | (n1 << 17));
                s.bw = u1 - u0 + 1;
                s.rbw = __frcp_rn(__int2float_rn(s.bw));
                area = s.bw * (v1 - v0 + 1);
            }
        }
        if (area == 1) whole_sample<K32>(s, s.t0, s.t1, (int)(s.idx & 0xFFFFu), cap, a.err);
        const int items = area > 1 ? area : 0;
        const unsigned some = __ballot_sync(0xffffffffu, items > 0);
        if (some == 0u) continue;
        int first = items;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int x = __shfl_up_sync(0xffffffffu, first, off);
            if (lane >= off) first += x;
        }
        const int total = __shfl_sync(0xffffffffu, first, 31);
        first -= items;
        s.first = first;
        if (items > 0) TS[__popc(some & lt)] = s;
        __syncwarp();
        int begun = 0;                                  // staged triangles whose samples began before f0
        for (int f0 = 0; f0 < total; f0 += 32) {
            // sample f belongs to the last triangle begun at or before it
            const unsigned rel = (unsigned)(first - f0);
            const unsigned starts = __reduce_or_sync(0xffffffffu, items > 0 && rel < 32u ? 1u << rel : 0u);
            begun += __popc(starts & (lt | (1u << lane)));
            if (f0 + lane < total) {
                const TriWhole e = TS[begun - 1];
                const int local = f0 + lane - e.first;
                int v = __float2int_rz(__fmul_rn(__int2float_rn(local), e.rbw));
                const int r = local - v * e.bw;
                v += (r >= e.bw) - (r < 0);
                const int u = local - v * e.bw;
                whole_sample<K32>(e, (int)((unsigned)e.t0 + (unsigned)e.b0 * (unsigned)v + (unsigned)e.a0 * (unsigned)u),
                                  (int)((unsigned)e.t1 + (unsigned)e.b1 * (unsigned)v + (unsigned)e.a1 * (unsigned)u),
                                  (int)(e.idx & 0xFFFFu) + v * a.tw + u, cap, a.err);
            }
            begun = __shfl_sync(0xffffffffu, begun, 31);
        }
        __syncwarp();
    }
}

// Which rasteriser the render of a mesh with stout triangles takes (DevMesh::stout).
// raster_tile keeps its lanes full where most triangles hold few samples or their boxes
// few covered ones; where a triangle holds several, setting it up with its depths at
// hand beats reading it again for each.  us for 1,452 poses, raster_tile /
// raster_whole, at 160x120, 320x240 and 640x480 (stride 3, mostly render): boxes of 588
// triangles 128 / 109, 300 / 243, 1,344 / 1,147 and of 10,800 209 / 238, 386 / 433, 1,390
// / 1,198; ellipsoids of 1,104 103 / 95, 233 / 189, 730 / 641 and of 18,240 232 / 305,
// 393 / 472, 1,089 / 1,115.  They meet at about one sample a triangle.  A cylinder of
// 8,200 with end caps of thin wedges, which fill little of their boxes, is the rings'
// throughout: 193 / 265, 353 / 599, 2,187 / 4,620.
__device__ __forceinline__ bool few_large_triangles(const DevMesh& m, int px) { return px >= m.n_tris; }

// The tile's render of mesh m (or of its triangles list[0 .. n_list)) at pose P.
// probe_off and ring_off: byte offsets of the block's per-warp scratch and of its
// warps' depth rings in shared memory.  EITHER: the rasteriser is chosen by the px
// samples of the hypothesis's whole render, else raster_tile with the vertex cache.
template <int NT, bool K32, bool VC, bool EITHER = false>
__device__ __forceinline__ void raster(const DevScene& sc, const DevMesh& m, const float* P,
                                       const unsigned long long* vc, unsigned probe_off, unsigned ring_off, int tu0,
                                       int tv0, int tu1, int tv1, int tw, int* err, const int* list = nullptr,
                                       int n_list = 0, int px = 0)
{
    const unsigned warp = threadIdx.x >> 5;
    const RasterArgs a = {m.tris, vc, list, list ? n_list : m.n_tris, tu0, tv0, tu1, tv1, tw,
                          probe_off + warp * (unsigned)kWarpScratch,
                          ring_off + warp * (unsigned)(kRing * sizeof(DepthItem)), err};
    if (!VC)
        raster_whole<NT, K32>(a, RasterCamera{m.verts, P, sc.W, sc.H, sc.fx, sc.fy, sc.cx, sc.cy, sc.z_near});
    else if (EITHER && few_large_triangles(m, px))
        raster_whole<NT, K32>(a, CachedVertices{});
    else
        raster_tile<NT, K32>(a);
}

// Tile bins of one hypothesis: the pixel box rbox is rasterised in tiles of tw
// x th pixels (n_tx per row of tiles); every triangle whose sample box meets a
// tile is listed in that tile's bin (bins + tile * cap, count in cnt[tile];
// a count above cap marks a bin that overflowed).  A triangle covers samples
// only inside its sample box, so a tile rasterised from its bin gets the same
// z-buffer as from the whole mesh.  Bin order depends on timing; the
// z-buffer does not (atomicMin).
template <int NT, bool VC>
__device__ void bin_triangles(const DevScene& sc, const DevMesh& mesh, const float* P, const unsigned long long* vc,
                              const int* rbox, int tw, int th, int n_tx, int* bins, int cap, int* cnt)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int4 tv_next = warp * 32 + lane < mesh.n_tris ? __ldg(&mesh.tris[warp * 32 + lane]) : make_int4(0, 0, 0, 0);
    for (int base = warp * 32; base < mesh.n_tris; base += NT) {
        const int t = base + lane;
        const int4 tv = tv_next;
        if (t + NT < mesh.n_tris) tv_next = __ldg(&mesh.tris[t + NT]);
        TriSetup o;
        if (t >= mesh.n_tris || !load_tri<VC>(sc, mesh, P, vc, tv, o)) continue;
        const int u0 = max(ceil16(min(o.x[0], min(o.x[1], o.x[2]))), rbox[0]);
        const int u1 = min(floor16(max(o.x[0], max(o.x[1], o.x[2]))), rbox[2] - 1);
        const int v0 = max(ceil16(min(o.y[0], min(o.y[1], o.y[2]))), rbox[1]);
        const int v1 = min(floor16(max(o.y[0], max(o.y[1], o.y[2]))), rbox[3] - 1);
        if (u0 > u1 || v0 > v1) continue;
        const int tx0 = div_small(u0 - rbox[0], tw), tx1 = div_small(u1 - rbox[0], tw);
        const int ty0 = div_small(v0 - rbox[1], th), ty1 = div_small(v1 - rbox[1], th);
        for (int ty = ty0; ty <= ty1; ++ty)
            for (int tx = tx0; tx <= tx1; ++tx) {
                const int tile = ty * n_tx + tx;
                const int k = atomicAdd(&cnt[tile], 1);
                if (k < cap) bins[tile * cap + k] = t;
            }
    }
}

// Affine integer colour at pixel (u, v) of the set-up triangle o: per channel
// (w0 c0 + w1 c1 + w2 c2 + floor(A / 2)) / A with the edge values w of the
// pixel's sample (screen-space interpolation of the per-vertex colour, rounded
// half up), packed r | g << 8 | b << 16.
__device__ __forceinline__ uint32_t interp_colour(const DevMesh& m, const TriSetup& o, int u, int v)
{
    const int sx = 16 * u, sy = 16 * v;
    const long long w0 = edge_fn(o.x[1], o.y[1], o.x[2], o.y[2], sx, sy);
    const long long w1 = edge_fn(o.x[2], o.y[2], o.x[0], o.y[0], sx, sy);
    const long long w2 = edge_fn(o.x[0], o.y[0], o.x[1], o.y[1], sx, sy);
    const uint32_t c0 = __float_as_uint(__ldg(&m.verts[o.vid[0]].w));
    const uint32_t c1 = __float_as_uint(__ldg(&m.verts[o.vid[1]].w));
    const uint32_t c2 = __float_as_uint(__ldg(&m.verts[o.vid[2]].w));
    const long long half = o.A / 2;
    // floor(num / A) without a 64-bit division: a binary32 estimate from the
    // reciprocal of A (relative error a few 2^-24, and the quotient is below
    // 256, so the estimate is off by at most one) corrected exactly with
    // integer arithmetic
    const float rA = __frcp_rn(__int2float_rn(o.A));
    uint32_t crgb = 0;
#pragma unroll 1
    for (int ch = 0; ch < 24; ch += 8) {
        const long long num = w0 * ((c0 >> ch) & 255) + w1 * ((c1 >> ch) & 255) + w2 * ((c2 >> ch) & 255) + half;
        // num < 2^41: its binary32 value from two 32-bit halves (the
        // estimate needs only relative accuracy, the correction makes it exact)
        const float numf = __fadd_rn(__fmul_rn(__int2float_rn((int)(num >> 16)), 65536.0f),
                                     __int2float_rn((int)(num & 0xFFFF)));
        long long q = __float2int_rz(__fmul_rn(numf, rA));
        const long long r = num - q * o.A;
        q += (r >= o.A) - (r < 0);
        crgb |= (uint32_t)q << ch;
    }
    return crgb;
}

// jo_mode 1 with the colour check (Eq. 3 with Eq. 4 applied from the observed
// side): every observed point p of rows [mv0, mv1) of the admissible box
// holds the key of its nearest rendered point q; p stays an inlier iff the
// CIEDE2000 difference between q's rendered colour and p's colour is at most
// tau_c, else its key is cleared.  This handles the p whose q lies in the
// z-buffer tile [tu0, tu1) x [tv0, tv1) now in shared memory (q's winning
// triangle gives its colour).
template <int NT, bool K32, bool VC>
__device__ __forceinline__ void jo_colour_pass(const Job& J, const float* P, const unsigned long long* vc, const ScoreSmem& S,
                               int tu0, int tv0, int tu1, int tv1, int tw, const int* vbox, int mv0, int mv1)
{
    const DevScene& sc = J.sc;
    const int vw = vbox[2] - vbox[0];
    const int n = vw * (mv1 - mv0);
    unsigned long long* keys = reinterpret_cast<unsigned long long*>(S.marks);
    for (int i = threadIdx.x; i < n; i += NT) {
        const unsigned long long k = keys[i];
        if (k == kEmptyKey) continue;
        const uint32_t qp = (uint32_t)k;
        const int qu = (int)(qp & 0xFFFFu), qv = (int)(qp >> 16);
        if (qu < tu0 || qu >= tu1 || qv < tv0 || qv >= tv1) continue;
        const int zi = (qv - tv0) * tw + (qu - tu0);
        // q is a kept rendered point: its z-buffer word holds its triangle
        const int tri = K32 ? (int)(S.zbuf[zi] & 0xFFFFu)
                            : (int)(uint32_t)reinterpret_cast<const unsigned long long*>(S.zbuf)[zi];
        TriSetup o;
        get_triangle<VC>(sc, J.m, P, vc, tri, o);
        const uint32_t crgb = interp_colour(J.m, o, qu, qv);
        const int pu = vbox[0] + i % vw, pv = mv0 + i / vw;
        const float4 lp = __ldg(&sc.lab[pv * sc.W + pu]);
        const float3 lq = srgb8_to_lab(crgb & 255, (crgb >> 8) & 255, (crgb >> 16) & 255);
        if (ciede2000(lq, make_float3(lp.x, lp.y, lp.z)) > sc.tau_c) keys[i] = kEmptyKey;
    }
}

// Specialisations of the scoring kernel: plain scoring (jo_mode 0), edges of
// the Monotone Scene Generation tree, and jo_mode 1 (Eq. 3 as written, with
// per-pixel nearest-rendered-point keys).  Each is compiled separately so the
// plain path carries none of the other two's code.
enum : int { kModePlain = 0, kModeTree = 1, kModeEq3 = 2 };

// Forms of plain scoring, compiled separately too: the rings' rasteriser alone, with
// tile bins, or the choice between the two rasterisers.  The choice in every kernel cost
// the renders that never take it 1 to 3 % (three 640x480 objects x 29,584 poses 36.5
// against 35.9 ms, the tree search 53.4 against 51.6), so it is compiled for meshes that
// can gain by it: stout triangles, no more of them than the region of interest holds
// pixels nor than kEitherTris (a render of more samples than that takes three tiles).
// The other modes search and count more than they render, and take the rings.
enum : int { kFormRings = 0, kFormBins = 1, kFormEither = 2 };
constexpr int kEitherTris = 16384;

// Is the observed point p of pixel pix in the admissible set V(O) at pose P
// (Sec. IV-A J_o; labels Sec. V-C)?  The inscribed cylinder about the
// object's z-axis (radius^2 rr, height vol_h) in the object frame, R^T (p - t),
// or the pixel's label.
__device__ __forceinline__ bool in_admissible(const DevScene& sc, const Job& J, const float* P, float rr, int pix,
                                              float4 p)
{
    if (J.label >= 0) return __ldg(&sc.labels[pix]) == J.label;
    float e0 = __fsub_rn(p.x, P[3]), e1 = __fsub_rn(p.y, P[7]), e2 = __fsub_rn(p.z, P[11]);
    float q0 = __fadd_rn(__fadd_rn(__fmul_rn(P[0], e0), __fmul_rn(P[4], e1)), __fmul_rn(P[8], e2));
    float q1 = __fadd_rn(__fadd_rn(__fmul_rn(P[1], e0), __fmul_rn(P[5], e1)), __fmul_rn(P[9], e2));
    float q2 = __fadd_rn(__fadd_rn(__fmul_rn(P[2], e0), __fmul_rn(P[6], e1)), __fmul_rn(P[10], e2));
    return __fadd_rn(__fmul_rn(q0, q0), __fmul_rn(q1, q1)) <= rr && q2 >= 0.0f && q2 <= J.m.vol_h;
}

// |I cap V| of plain scoring, counted in chunks of kJoChunk lattice pixels of
// the whole admissible box taken from a shared counter (zero at the start of
// the hypothesis).  It needs nothing rendered: a warp counts chunks once the
// search leaves it idle, so the warps that finish early count most of them.
constexpr int kJoChunk = 256;

__device__ __forceinline__ void jo_count_in(const DevScene& sc, const Job& J, const float* P, const int* vbox,
                                            int* counter, int& n_in)
{
    const int s = sc.stride, lane = threadIdx.x & 31;
    const int us0 = div_small(vbox[0] + s - 1, s) * s, vs0 = div_small(vbox[1] + s - 1, s) * s;
    const int nu = us0 < vbox[2] ? div_small(vbox[2] - 1 - us0, s) + 1 : 0;
    const int nv = vs0 < vbox[3] ? div_small(vbox[3] - 1 - vs0, s) + 1 : 0;
    const int npx = nu * nv;
    const float rr = __fmul_rn(J.m.vol_r, J.m.vol_r);
    for (;;) {
        int c = 0;
        if (lane == 0) c = atomicAdd(counter, 1);
        const int k0 = __shfl_sync(0xffffffffu, c, 0) * kJoChunk;
        if (k0 >= npx) break;
        const int k1 = min(k0 + kJoChunk, npx);
#pragma unroll 1
        for (int k = k0 + lane; k < k1; k += 32) {
            const int kv = div_small(k, nu);
            const int pix = (vs0 + kv * s) * sc.W + us0 + (k - kv * nu) * s;
            const float4 p = __ldg(&sc.pxyz[pix]);
            if (p.w != 0.0f && in_admissible(sc, J, P, rr, pix, p)) ++n_in;
        }
    }
}

// Rasterise, resolve and radius-search the pixel box rbox in z-buffer tiles.
// J_r is accumulated when count_jr; marks are set for nearest neighbours that
// fall in rows [mv0, mv1) of the admissible box vbox.
template <int NT, bool K32, bool VC, int MODE, int FORM>
__device__ __forceinline__ void score_tiles(const ScoreArgs& a, const Job& J, const float* P, const unsigned long long* vc,
                            const int* rbox, const ScoreSmem& S, const int* vbox, int mv0, int mv1,
                            bool count_jr, int& jr_local, int& n_in, int& n_marked)
{
    constexpr bool TREE = MODE == kModeTree, EQ3 = MODE == kModeEq3, BINS = FORM == kFormBins;
    const DevScene& sc = J.sc;
    const float rr = __fmul_rn(J.m.vol_r, J.m.vol_r);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    WarpProbe& WP = *reinterpret_cast<WarpProbe*>(g_smem + a.probe_off + warp * (unsigned)kWarpScratch);
    const int s = sc.stride;
    const int rw = rbox[2] - rbox[0], rh = rbox[3] - rbox[1];
    // (plain scoring goes through one empty tile, to count J_o's |I cap V|)
    if (MODE != kModePlain && (rw <= 0 || rh <= 0)) return;
    const int cap_px = K32 ? a.zcap_words : a.zcap_words / 2;
    const int tw = max(1, min(rw, cap_px));
    const int th = max(1, div_small(cap_px, tw));
    const uint32_t empty32 = 0xFFFFFFFFu;
    const int vw = vbox[2] - vbox[0];
    uint32_t* const zbuf = reinterpret_cast<uint32_t*>(g_smem);
    uint32_t* const marks = reinterpret_cast<uint32_t*>(g_smem + a.marks_off);
    // a pixel box of several tiles: each tile's triangles binned first
    const int n_tx = BINS ? (rw + tw - 1) / tw : 1, n_tiles = BINS ? n_tx * ((rh + th - 1) / th) : 1;
    const bool binned = BINS && VC && a.bin_cap > 0 && n_tiles > 1 && n_tiles <= kBinTiles;
    int* bins = binned ? reinterpret_cast<int*>(const_cast<unsigned long long*>(vc) + a.bin_off) : nullptr;
    if (binned) {
        for (int i = threadIdx.x; i < n_tiles; i += NT) S.bin_cnt[i] = 0;
        __syncthreads();
        if (BINS) bin_triangles<NT, VC>(sc, J.m, P, vc, rbox, tw, th, n_tx, bins, a.bin_cap, S.bin_cnt);
        __syncthreads();
    }
    int tile = 0;
    int tv0 = rbox[1];
    do {
        int tu0 = rbox[0];
        do {
            const int tu1 = min(tu0 + tw, rbox[2]), tv1 = min(tv0 + th, rbox[3]);
            const int tpx = tw * (tv1 - tv0);
            const int words = K32 ? tpx : 2 * tpx;
#pragma unroll 1
            for (int i = threadIdx.x; i < words; i += NT) zbuf[i] = empty32;
            if (threadIdx.x == 0) *S.next_batch = 0;
            __syncthreads();
            // (the depth rings take the place of the kept-point queues, idle meanwhile)
            const bool in_bin = BINS && binned && S.bin_cnt[tile] <= a.bin_cap;
            if (MODE != kModePlain || (rw > 0 && rh > 0))
                raster<NT, K32, VC, FORM == kFormEither>(sc, J.m, P, vc, a.probe_off, a.kept_off, tu0, tv0, tu1, tv1, tw,
                                                         a.err, in_bin ? bins + tile * a.bin_cap : nullptr,
                                                         in_bin ? S.bin_cnt[tile] : 0, rw * rh);
            __syncthreads();
            if (a.dump) {
                for (int i = threadIdx.x; i < tpx; i += NT) {
                    int u = tu0 + i % tw, v = tv0 + i / tw;
                    if (u >= tu1) continue;
                    unsigned long long k;
                    if (K32) {
                        uint32_t w = zbuf[i];
                        k = (w == empty32) ? kEmptyKey
                                           : (((unsigned long long)(w >> 16) << 32) | (w & 0xFFFFu));
                    } else {
                        k = reinterpret_cast<unsigned long long*>(zbuf)[i];
                    }
                    a.dump[(size_t)v * sc.W + u] = k;
                }
            }
            // ---- resolve + radius search.  The stride lattice of the tile is
            // cut into 8 x 4 pixel blocks that warps take from a counter; a
            // warp resolves a block (occluder test, colour, back-projection)
            // and appends its kept points to its own queue, which it searches
            // 32 at a time -- no block-wide barrier until the tile is done.
            const int us0 = div_small(tu0 + s - 1, s) * s, vs0 = div_small(tv0 + s - 1, s) * s;
            const int nu = us0 < tu1 ? div_small(tu1 - 1 - us0, s) + 1 : 0;
            const int nv = vs0 < tv1 ? div_small(tv1 - 1 - vs0, s) + 1 : 0;
            const int nbx = (nu + 7) / 8, nby = (nv + 3) / 4;
            const int nblocks = nbx * nby;
            KeptPoint* const wq = reinterpret_cast<KeptPoint*>(g_smem + a.kept_off) + warp * kWarpQueue;
            const MarkBand mband = {marks, vbox[0], vbox[2], mv0, mv1, vw, a.err};
            __syncwarp();
            int wq_head = 0, wq_count = 0;
            for (;;) {
                int blk = 0;
                if (lane == 0) blk = atomicAdd(S.next_batch, 1);
                blk = __shfl_sync(0xffffffffu, blk, 0);
                const bool more = blk < nblocks;
                if (more) {
                    bool kept = false;
                    KeptPoint kp;
                    const int by = div_small(blk, nbx);
                    const int lu = (blk - by * nbx) * 8 + (lane & 7), lv = by * 4 + (lane >> 3);
                    if (lu < nu && lv < nv) {
                        int u = us0 + lu * s, v = vs0 + lv * s;
                        int zi = (v - tv0) * tw + (u - tu0);
                        unsigned d = 0;
                        int tri = -1;
                        if (!PERCH_CHECKED((unsigned)zi < (unsigned)(tw * (tv1 - tv0)), a.err)) {
                        } else if (K32) {
                            uint32_t w = zbuf[zi];
                            if (w != empty32) { d = w >> 16; tri = (int)(w & 0xFFFFu); }
                        } else {
                            unsigned long long w = reinterpret_cast<unsigned long long*>(zbuf)[zi];
                            if (w != kEmptyKey) { d = (unsigned)(w >> 32); tri = (int)(uint32_t)w; }
                        }
                        int pix = v * sc.W + u;
                        if (TREE && tri >= 0) {
                            // a placed object in front hides the pixel; one behind
                            // by more than the margin refuses the edge
                            const unsigned sd = __ldg(&J.tree.depth[pix]);
                            if (sd != 0) {
                                if ((unsigned long long)d + (unsigned)J.tree.margin < sd) *S.refused = 1;
                                if (!(d < sd)) tri = -1;
                            }
                            if (tri >= 0 && J.tree.out_depth) J.tree.out_depth[pix] = d;
                        }
                        if (tri >= 0) {
                            unsigned dobs = __ldg(&sc.depth[pix]);
                            bool occluded = sc.occ_margin >= 0 && dobs > 0 &&
                                            (unsigned long long)dobs + (unsigned)sc.occ_margin < d &&
                                            (J.label < 0 || __ldg(&sc.labels[pix]) != J.label);
                            if (!occluded) {
                                float3 q = back_project(sc, u, v, d);
                                kp.x = q.x; kp.y = q.y; kp.z = q.z; kp.pix = (uint32_t)u | ((uint32_t)v << 16);
                                kept = true;
                                if (sc.near_bits) {
                                    // no observed point in the 27 cells: unexplained
                                    // without a search (the radius search's own filter)
                                    const long long b = near_index(sc, cell_coord(q.x, sc.inv_cell),
                                                                   cell_coord(q.y, sc.inv_cell),
                                                                   cell_coord(q.z, sc.inv_cell));
                                    if (b < 0 || !((__ldg(&sc.near_bits[b >> 5]) >> (b & 31)) & 1u)) {
                                        kept = false;
                                        if (count_jr) ++jr_local;
                                    }
                                }
                            }
                        }
                    }
                    const unsigned bal = __ballot_sync(0xffffffffu, kept);
                    if (kept) wq[(wq_head + wq_count + __popc(bal & ((1u << lane) - 1u))) & (kWarpQueue - 1)] = kp;
                    wq_count += __popc(bal);
                }
                // search a full batch, or what is left once the blocks run out
                while (wq_count >= 32 || (!more && wq_count > 0)) {
                    __syncwarp();
                    const int nb = min(wq_count, 32);
                    const bool valid = lane < nb;
                    KeptPoint kq = {0.f, 0.f, 0.f, 0u};
                    if (valid) kq = wq[(wq_head + lane) & (kWarpQueue - 1)];
                    wq_head = (wq_head + nb) & (kWarpQueue - 1);
                    wq_count -= nb;
                    const uint32_t qpix = (EQ3 && valid) ? kq.pix : 0u;
                    const unsigned long long nn = probe_batch<EQ3, true>(sc, valid, kq.x, kq.y, kq.z, qpix, WP, lane, mband);
                    if (valid) {
                        bool explained = nn != kEmptyKey;
                        const int pnn = (int)(uint32_t)nn;
                        const int pu = pnn & 0xFFFF, pv = pnn >> 16;
                        if (explained && sc.color_check) {
                            // the rendered colour of q, from the triangle its z-buffer word holds
                            const int qu = (int)(kq.pix & 0xFFFFu), qv = (int)(kq.pix >> 16);
                            const int qi = (qv - tv0) * tw + (qu - tu0);
                            const int qtri = K32 ? (int)(zbuf[qi] & 0xFFFFu)
                                                 : (int)(uint32_t)reinterpret_cast<const unsigned long long*>(zbuf)[qi];
                            TriSetup o;
                            get_triangle<VC>(sc, J.m, P, vc, qtri, o);
                            const uint32_t rgb = interp_colour(J.m, o, qu, qv);
                            float4 lp = __ldg(&sc.lab[pv * sc.W + pu]);
                            float3 lq = srgb8_to_lab(rgb & 255, (rgb >> 8) & 255, (rgb >> 16) & 255);
                            if (ciede2000(lq, make_float3(lp.x, lp.y, lp.z)) > sc.tau_c) explained = false;
                        }
                        if (TREE && explained && J.tree.out_mark) {
                            const int npix = pv * sc.W + pu;
                            atomicOr(&J.tree.out_mark[npix >> 5], 1u << (npix & 31));
                        }
                        if (!explained) {
                            if (count_jr) ++jr_local;
                        } else if (!EQ3) {
                            if (pu >= vbox[0] && pu < vbox[2] && pv >= mv0 && pv < mv1) {
                                int bit = (pv - mv0) * vw + (pu - vbox[0]);
                                if (PERCH_CHECKED((unsigned)bit < 32u * (unsigned)a.mark_words, a.err)) {
                                    const unsigned m = 1u << (bit & 31);
                                    const unsigned was = atomicOr(&marks[bit >> 5], m);
                                    if (MODE == kModePlain && !(was & m)) {
                                        // J_o's marked part: the first mark of a pixel of V
                                        const int npix = pv * sc.W + pu;
                                        const float4 pn = __ldg(&sc.pxyz[npix]);
                                        if (pn.w != 0.0f && in_admissible(sc, J, P, rr, npix, pn)) ++n_marked;
                                    }
                                }
                            }
                        }
                    }
                }
                if (!more) break;
            }
            // J_o's |I cap V|, by the warps that finish the search first (all of it
            // with the first tile)
            if (MODE == kModePlain && count_jr) jo_count_in(sc, J, P, vbox, S.jo_next, n_in);
            __syncthreads();
            if (threadIdx.x == 0) *S.next_batch = 0;
            __syncthreads();
            ++tile;
            tu0 += tw;
        } while (tu0 < rbox[2]);
        tv0 += th;
    } while (tv0 < rbox[3]);
}

// score_tiles without the vertex cache (images over 1023 pixels) or with 64-bit
// keys (65,536 triangles or more, poses beyond 6.5 m): called, so that the
// common case has the kernel's registers and instruction cache to itself.
// Returns (J_r, |I cap V|, marked) of this thread.
template <int NT, int MODE, int FORM>
__device__ __noinline__ int3 score_tiles_rare(const ScoreArgs& a, const float* P, const unsigned long long* vc,
                                              const int* rbox, ScoreSmem S, const int* vbox, int mv0, int mv1,
                                              bool count_jr, int k32)
{
    int3 r = make_int3(0, 0, 0);
    if (vc)
        score_tiles<NT, false, true, MODE, FORM>(a, a.job, P, vc, rbox, S, vbox, mv0, mv1, count_jr, r.x, r.y, r.z);
    else if (k32)
        score_tiles<NT, true, false, MODE, FORM>(a, a.job, P, vc, rbox, S, vbox, mv0, mv1, count_jr, r.x, r.y, r.z);
    else
        score_tiles<NT, false, false, MODE, FORM>(a, a.job, P, vc, rbox, S, vbox, mv0, mv1, count_jr, r.x, r.y, r.z);
    return r;
}

// jo_mode 1 with the colour check, after score_tiles has made every key of
// the band final: the colour pass over the same z-buffer tiles.  With one
// tile its z-buffer is still in shared memory; otherwise each tile is
// rendered again.
template <int NT, bool K32, bool VC>
__device__ __noinline__ void jo_colour_band(const ScoreArgs& a, const Job& J, const float* P,
                                            const unsigned long long* vc, const int* rbox, const ScoreSmem& S,
                                            const int* vbox, int mv0, int mv1)
{
    const int rw = rbox[2] - rbox[0], rh = rbox[3] - rbox[1];
    if (rw <= 0 || rh <= 0) return;
    const int cap_px = K32 ? a.zcap_words : a.zcap_words / 2;
    const int tw = min(rw, cap_px);
    const int th = max(1, cap_px / tw);
    if (th >= rh) {
        jo_colour_pass<NT, K32, VC>(J, P, vc, S, rbox[0], rbox[1], rbox[2], rbox[3], tw, vbox, mv0, mv1);
        __syncthreads();
        return;
    }
    for (int tv0 = rbox[1]; tv0 < rbox[3]; tv0 += th) {
        for (int tu0 = rbox[0]; tu0 < rbox[2]; tu0 += tw) {
            const int tu1 = min(tu0 + tw, rbox[2]), tv1 = min(tv0 + th, rbox[3]);
            const int words = K32 ? tw * (tv1 - tv0) : 2 * tw * (tv1 - tv0);
            for (int i = threadIdx.x; i < words; i += NT) S.zbuf[i] = 0xFFFFFFFFu;
            __syncthreads();
            raster<NT, K32, VC>(J.sc, J.m, P, vc, a.probe_off, a.kept_off, tu0, tv0, tu1, tv1, tw, a.err);
            __syncthreads();
            jo_colour_pass<NT, K32, VC>(J, P, vc, S, tu0, tv0, tu1, tv1, tw, vbox, mv0, mv1);
            __syncthreads();
        }
    }
}

// Score hypothesis h (one block).  Writes costs[2h] = J_o, costs[2h+1] = J_r.
template <int NT, int MODE, int FORM>
__device__ void score_one(const ScoreArgs& a, const Job& J, long long h, const ScoreSmem& S, float* s_pose,
                          int* s_rbox, int* s_vbox, int* s_k32, int (*s_red)[NT / 32],
                          unsigned long long* vc)
{
    constexpr bool TREE = MODE == kModeTree;
    const DevScene& sc = J.sc;
    if (threadIdx.x < 12) s_pose[threadIdx.x] = J.poses[h * 12 + threadIdx.x];
    if (TREE && threadIdx.x == 0) *S.refused = 0;
    if (threadIdx.x == 0) *S.jo_next = 0;
    if (threadIdx.x < 4) S.vbounds[threadIdx.x] = threadIdx.x < 2 ? INT_MAX : INT_MIN;
    __syncthreads();
    // the two boxes by two warps, while the others begin the vertex pass
    if (threadIdx.x < 64) {
        const DevMesh& m = J.m;
        const bool vol = threadIdx.x >= 32;
        const PixelBox b = project_box(
            make_float4(sc.fx, sc.fy, sc.cx, sc.cy), s_pose,
            vol ? make_float3(-m.vol_r, -m.vol_r, 0.0f) : make_float3(m.lo[0], m.lo[1], m.lo[2]),
            vol ? make_float3(m.vol_r, m.vol_r, m.vol_h) : make_float3(m.hi[0], m.hi[1], m.hi[2]),
            vol ? make_int4(0, 0, sc.W, sc.H) : make_int4(J.roi[0], J.roi[1], J.roi[2], J.roi[3]));
        if ((threadIdx.x & 31) == 0) {
            int* const out = vol ? s_vbox : s_rbox;
            out[0] = b.box.x; out[1] = b.box.y; out[2] = b.box.z; out[3] = b.box.w;
            if (!vol) *s_k32 = (m.n_tris <= 65535 && b.zmax < 6.5f) ? 1 : 0;
            else if (J.label >= 0) for (int i = 0; i < 4; ++i) out[i] = J.roi[i];
        }
    }
    const bool use_vc = vc != nullptr;
    if (use_vc) vertex_pass(sc, J.m, s_pose, vc, NT, S.vbounds);
    __syncthreads();
    // The pixel box of the render: the projected object-frame box, tightened
    // (with the vertex cache) to the samples between the kept vertices'
    // smallest and largest snapped coordinates -- every covered sample lies
    // in its triangle's vertex box, so nothing outside can be covered.
    if (threadIdx.x == 0 && use_vc) {
        const int* vb = S.vbounds;
        if (vb[0] > vb[2]) {
            s_rbox[2] = s_rbox[0];
            s_rbox[3] = s_rbox[1];
        } else {
            s_rbox[0] = max(s_rbox[0], ceil16(vb[0]));
            s_rbox[1] = max(s_rbox[1], ceil16(vb[1]));
            s_rbox[2] = max(s_rbox[0], min(s_rbox[2], floor16(vb[2]) + 1));
            s_rbox[3] = max(s_rbox[1], min(s_rbox[3], floor16(vb[3]) + 1));
        }
    }

    // The admissible box is handled in bands of rows that fit the marks
    // bitset (jo_mode 1: one 64-bit key per pixel); each band repeats the
    // render + search (J_r counted once).
    constexpr bool jo1 = MODE == kModeEq3;
    const int vw = s_vbox[2] - s_vbox[0], vh = s_vbox[3] - s_vbox[1];
    const int band_rows = vw > 0 ? max(1, div_small(jo1 ? a.mark_words / 2 : 32 * a.mark_words, vw)) : 1;
    const int n_bands = vh > 0 ? div_small(vh + band_rows - 1, band_rows) : 1;
    int jr = 0, n_in = 0, n_marked = 0;
    const int s = sc.stride;
    const float* P = s_pose;
    const float rr = __fmul_rn(J.m.vol_r, J.m.vol_r);
#pragma unroll 1
    for (int band = 0; band < n_bands; ++band) {
        const int mv0 = s_vbox[1] + band * band_rows;
        const int mv1 = min(mv0 + band_rows, s_vbox[3]);
        const int mwords = jo1 ? 2 * vw * max(0, mv1 - mv0) : (vw * max(0, mv1 - mv0) + 31) / 32;
        const uint32_t mfill = jo1 ? 0xFFFFFFFFu : 0u;     // empty keys / clear bits
#pragma unroll 1
        for (int i = threadIdx.x; i < mwords; i += NT) S.marks[i] = mfill;
        __syncthreads();
        if (*s_k32 && use_vc) {
            score_tiles<NT, true, true, MODE, FORM>(a, J, P, vc, s_rbox, S, s_vbox, mv0, mv1, band == 0, jr, n_in, n_marked);
        } else {
            const int3 r = score_tiles_rare<NT, MODE, FORM>(a, P, vc, s_rbox, S, s_vbox, mv0, mv1, band == 0, *s_k32);
            jr += r.x;
            n_in += r.y;
            n_marked += r.z;
        }
        __syncthreads();
        if (jo1 && sc.color_check) {
            // Eq. 4 from the observed side, once the band's keys are final
            if (*s_k32) {
                if (use_vc) jo_colour_band<NT, true, true>(a, J, P, vc, s_rbox, S, s_vbox, mv0, mv1);
                else jo_colour_band<NT, true, false>(a, J, P, vc, s_rbox, S, s_vbox, mv0, mv1);
            } else {
                if (use_vc) jo_colour_band<NT, false, true>(a, J, P, vc, s_rbox, S, s_vbox, mv0, mv1);
                else jo_colour_band<NT, false, false>(a, J, P, vc, s_rbox, S, s_vbox, mv0, mv1);
            }
        }
        // plain scoring: J_o's marked part was counted as the marks were set
        // (each pixel of V once, by the lane whose atomicOr set its bit) and
        // |I cap V| is counted by jo_count_in
        if (MODE == kModePlain) continue;
        // ---- J_o over the admissible set V(h), rows [mv0, mv1)
        const int us0 = div_small(s_vbox[0] + s - 1, s) * s, vs0 = div_small(mv0 + s - 1, s) * s;
        const int nu = us0 < s_vbox[2] ? div_small(s_vbox[2] - 1 - us0, s) + 1 : 0;
        const int nv = vs0 < mv1 ? div_small(mv1 - 1 - vs0, s) + 1 : 0;
        // pixel k = (row k / nu, column k % nu), the row and column carried
        // from one k to the next (k advances by NT) instead of divided out
        int kr = nu > 0 ? div_small(threadIdx.x, nu) : 0, kc = threadIdx.x - kr * nu;
        const int rstep = nu > 0 ? div_small(NT, nu) : 0, cstep = NT - rstep * nu;
        for (int k = threadIdx.x; k < nu * nv; k += NT) {
            const int u = us0 + kc * s, v = vs0 + kr * s;
            kc += cstep;
            kr += rstep;
            if (kc >= nu) { kc -= nu; ++kr; }
            int pix = v * sc.W + u;
            // the observed point of the pixel, back-projected once per scene
            const float4 p = __ldg(&sc.pxyz[pix]);
            if (p.w == 0.0f) continue;
            bool in;
            if (J.label >= 0) {
                in = __ldg(&sc.labels[pix]) == J.label;
            } else {
                float e0 = __fsub_rn(p.x, P[3]), e1 = __fsub_rn(p.y, P[7]), e2 = __fsub_rn(p.z, P[11]);
                float q0 = __fadd_rn(__fadd_rn(__fmul_rn(P[0], e0), __fmul_rn(P[4], e1)), __fmul_rn(P[8], e2));
                float q1 = __fadd_rn(__fadd_rn(__fmul_rn(P[1], e0), __fmul_rn(P[5], e1)), __fmul_rn(P[9], e2));
                float q2 = __fadd_rn(__fadd_rn(__fmul_rn(P[2], e0), __fmul_rn(P[6], e1)), __fmul_rn(P[10], e2));
                in = __fadd_rn(__fmul_rn(q0, q0), __fmul_rn(q1, q1)) <= rr && q2 >= 0.0f && q2 <= J.m.vol_h;
            }
            if (in) {
                if (TREE) {
                    if (J.tree.out_vol) atomicOr(&J.tree.out_vol[pix >> 5], 1u << (pix & 31));
                    if ((__ldg(&J.tree.vol[pix >> 5]) >> (pix & 31)) & 1u) continue;   // counted before
                }
                ++n_in;
                int bit = (v - mv0) * vw + (u - s_vbox[0]);
                if (!PERCH_CHECKED((unsigned)bit < (jo1 ? (unsigned)a.mark_words / 2u : 32u * (unsigned)a.mark_words), a.err))
                    continue;
                unsigned mk = jo1 ? (reinterpret_cast<const unsigned long long*>(S.marks)[bit] != kEmptyKey)
                                  : (S.marks[bit >> 5] >> (bit & 31)) & 1u;
                if (TREE && !mk) mk = (__ldg(&J.tree.mark[pix >> 5]) >> (pix & 31)) & 1u;
                n_marked += mk;
            }
        }
        __syncthreads();
    }
    // ---- warp-shuffle reduction of (J_r, |I cap V|, marked)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        jr += __shfl_xor_sync(0xffffffffu, jr, o);
        n_in += __shfl_xor_sync(0xffffffffu, n_in, o);
        n_marked += __shfl_xor_sync(0xffffffffu, n_marked, o);
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) { s_red[0][warp] = jr; s_red[1][warp] = n_in; s_red[2][warp] = n_marked; }
    __syncthreads();
    if (threadIdx.x < 32) {
        int x = lane < NT / 32 ? s_red[0][lane] : 0;
        int y = lane < NT / 32 ? s_red[1][lane] : 0;
        int z = lane < NT / 32 ? s_red[2][lane] : 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            x += __shfl_xor_sync(0xffffffffu, x, o);
            y += __shfl_xor_sync(0xffffffffu, y, o);
            z += __shfl_xor_sync(0xffffffffu, z, o);
        }
        if (lane == 0) {
            const bool refused = TREE && *S.refused;
            J.costs[2 * h] = refused ? -1 : y - z;
            J.costs[2 * h + 1] = refused ? -1 : x;
        }
    }
    __syncthreads();
}

// Byte offsets of the dynamic shared-memory regions of a scoring block; every
// region starts on a 16-byte boundary (the queues and the per-warp scratch
// hold float4 and 64-bit fields).
struct SmemLayout {
    size_t marks, kept, probe, total;
};

__host__ __device__ inline size_t align16(size_t x) { return (x + 15) & ~(size_t)15; }

__host__ __device__ inline SmemLayout smem_layout(int zcap_words, int mark_words, int threads)
{
    SmemLayout L;
    L.marks = align16(sizeof(uint32_t) * (size_t)zcap_words);
    L.kept = align16(L.marks + sizeof(uint32_t) * (size_t)mark_words);
    L.probe = align16(L.kept + sizeof(KeptPoint) * kWarpQueue * (size_t)(threads / 32));
    L.total = align16(L.probe + kWarpScratch * (size_t)(threads / 32));
    return L;
}

// Claim one vertex-cache slot from a pool of nslots (bit set = in use).
// Blocks of every scoring kernel that runs at the same time with the same
// launch shape draw from one pool sized for the device's resident blocks, so
// a free slot exists; should none be found the block runs without the cache
// (same results).  Bounded: every failed attempt adds a bit to `seen`.
__device__ int claim_vslot(unsigned* mask, int nslots)
{
    const int words = (nslots + 31) >> 5;
    for (int k = 0; k < words; ++k) {
        const int w = (int)((blockIdx.x + k) % words);
        const int rem = nslots - 32 * w;
        const unsigned valid = rem >= 32 ? 0xFFFFFFFFu : ((1u << rem) - 1u);
        unsigned seen = *(volatile unsigned*)&mask[w];
        while (~seen & valid) {
            const int b = __ffs(~seen & valid) - 1;
            const unsigned prev = atomicOr(&mask[w], 1u << b);
            if (!(prev & (1u << b))) {
                __threadfence();    // the previous holder's writes precede ours
                return 32 * w + b;
            }
            seen |= prev | (1u << b);
        }
    }
    return -1;
}

// Persistent scoring kernel over one job: each block repeatedly takes the
// next hypothesis index from a device counter (zero at launch) and scores
// it.  The job is read from the kernel parameters, so its fields are
// constant-bank operands.  MODE kModeTree: the job's hypotheses are edges of the
// Monotone Scene Generation tree from the state in job.tree.  At most 64
// registers per thread (128 and 256 threads): four 256-thread blocks, 32 warps,
// fit an SM when the block's shared memory allows (the default launch shape),
// which hides latency better than three blocks of 80 registers (36.6 against
// 39.9 ms for three 640x480 objects x 29,584 poses).  The Eq. 3 scorer, which
// holds more, would run from spilled values: 80 registers (2.44 against 2.84 ms
// for two objects x 2,527 poses at 517x389).
template <int NT, int MODE, int FORM>
__global__ void __launch_bounds__(NT, NT == 512 ? 1 : (MODE == kModeEq3 ? 768 : 1024) / NT) k_score(const __grid_constant__ ScoreArgs a)
{
    unsigned char* const smem = g_smem;
    __shared__ float s_pose[12];
    __shared__ int s_rbox[4], s_vbox[4], s_k32, s_next, s_slot, s_refused, s_bin_cnt[kBinTiles], s_jo_next,
        s_vbounds[4];
    __shared__ long long s_h;
    __shared__ int s_red[3][NT / 32];

    ScoreSmem S;
    S.zbuf = reinterpret_cast<uint32_t*>(smem);
    S.marks = reinterpret_cast<uint32_t*>(smem + a.marks_off);
    S.next_batch = &s_next;
    S.refused = &s_refused;
    S.bin_cnt = s_bin_cnt;
    S.jo_next = &s_jo_next;
    S.vbounds = s_vbounds;
    if (threadIdx.x == 0) s_slot = a.vcache ? claim_vslot(a.vmask, a.vslots) : -1;
    __syncthreads();
    unsigned long long* vc = s_slot >= 0 ? a.vcache + (size_t)s_slot * a.vstride : nullptr;
    for (;;) {
        if (threadIdx.x == 0) s_h = (long long)atomicAdd(a.next, 1u);
        __syncthreads();
        const long long h = s_h;
        if (h >= a.n) break;
        score_one<NT, MODE, FORM>(a, a.job, h, S, s_pose, s_rbox, s_vbox, &s_k32, s_red, vc);
    }
    // every thread has passed the barrier after its last use of the slot
    if (threadIdx.x == 0 && s_slot >= 0) {
        __threadfence();
        atomicAnd(&a.vmask[s_slot >> 5], ~(1u << (s_slot & 31)));
    }
}

size_t score_smem_bytes(const ScoreConfig& cfg, int mark_words)
{
    return smem_layout(cfg.zcap_words, mark_words, cfg.threads).total;
}

// Let fn use all the shared memory a block may have, once per device: the limit
// is a property of the function, so calls that set it to what each needs would
// undercut one another between threads (and cost a driver call per launch).
static cudaError_t allow_smem(const void* fn)
{
    static std::mutex mu;
    static std::set<std::pair<int, const void*>> done;
    int dev = 0, most = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lk(mu);
    if (done.count({dev, fn})) return cudaSuccess;
    cudaFuncAttributes fa{};
    e = cudaFuncGetAttributes(&fa, fn);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, most - (int)fa.sharedSizeBytes);
    if (e == cudaSuccess) done.insert({dev, fn});
    return e;
}

template <int NT, int MODE, int FORM>
static int score_grid_nt(size_t smem)
{
    int dev = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (allow_smem((const void*)k_score<NT, MODE, FORM>) != cudaSuccess) return -1;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_score<NT, MODE, FORM>, NT, smem) != cudaSuccess)
        return -1;
    return max(1, per) * max(1, sms);
}

template <int NT>
static int score_grid_all(size_t smem)
{
    // the specialisations share one grid and one vertex-cache pool: sized for the
    // one with most resident blocks (of another, the blocks past its own share
    // start as others end and find the counter spent)
    const int g[5] = {score_grid_nt<NT, kModePlain, kFormRings>(smem), score_grid_nt<NT, kModePlain, kFormBins>(smem),
                      score_grid_nt<NT, kModePlain, kFormEither>(smem), score_grid_nt<NT, kModeTree, kFormRings>(smem),
                      score_grid_nt<NT, kModeEq3, kFormRings>(smem)};
    int most = g[0];
    for (int k = 1; k < 5; ++k) most = g[k] < 0 || most < 0 ? -1 : max(most, g[k]);
    return most;
}

int score_grid(const ScoreConfig& cfg, int mark_words)
{
    // a function of the device and the shape alone, asked for on every call
    static std::mutex mu;
    static std::map<std::tuple<int, int, size_t>, int> known;
    const size_t smem = score_smem_bytes(cfg, mark_words);
    int dev = 0;
    cudaGetDevice(&dev);
    const std::tuple<int, int, size_t> key(dev, cfg.threads, smem);
    std::lock_guard<std::mutex> lk(mu);
    const auto it = known.find(key);
    if (it != known.end()) return it->second;
    const int g = cfg.threads == 128 ? score_grid_all<128>(smem)
                                     : cfg.threads == 512 ? score_grid_all<512>(smem) : score_grid_all<256>(smem);
    if (g > 0 && known.size() < 4096) known[key] = g;
    return g;
}

// a with the places of the block's shared-memory regions, which the kernel reads
// from the parameter bank instead of holding them in registers.
static ScoreArgs with_layout(ScoreArgs a, int threads)
{
    const SmemLayout L = smem_layout(a.zcap_words, a.mark_words, threads);
    a.marks_off = (unsigned)L.marks;
    a.kept_off = (unsigned)L.kept;
    a.probe_off = (unsigned)L.probe;
    return a;
}

// The kernel specialisation a launch runs on (tile bins: plain scoring only;
// the other modes rasterise every tile from the whole mesh).
template <int NT>
static const void* score_kernel(const ScoreArgs& a)
{
    const Job& J = a.job;
    if (J.tree.depth) return (const void*)k_score<NT, kModeTree, kFormRings>;
    if (J.sc.jo_mode == 1) return (const void*)k_score<NT, kModeEq3, kFormRings>;
    if (a.bin_cap > 0) return (const void*)k_score<NT, kModePlain, kFormBins>;
    const long long px = (long long)(J.roi[2] - J.roi[0]) * (J.roi[3] - J.roi[1]);
    if (J.m.stout && J.m.n_tris <= kEitherTris && J.m.n_tris <= px) return (const void*)k_score<NT, kModePlain, kFormEither>;
    return (const void*)k_score<NT, kModePlain, kFormRings>;
}

template <int NT>
static cudaError_t launch_score_nt(const ScoreArgs& a, const ScoreConfig& cfg, int grid, cudaStream_t s)
{
    const size_t smem = score_smem_bytes(cfg, a.mark_words);
    const unsigned g = (unsigned)(a.n < grid ? a.n : grid);
    const void* fn = score_kernel<NT>(a);
    cudaError_t e = allow_smem(fn);
    if (e != cudaSuccess) return e;
    ScoreArgs copy = with_layout(a, NT);
    void* args[] = {&copy};
    return cudaLaunchKernel(fn, dim3(g), dim3(NT), args, smem, s);
}

template <int NT>
static cudaError_t add_score_node_nt(cudaGraph_t g, const cudaGraphNode_t* deps, size_t ndeps,
                                     const ScoreArgs& a, const ScoreConfig& cfg, int grid,
                                     cudaGraphNode_t* out)
{
    const size_t smem = score_smem_bytes(cfg, a.mark_words);
    const void* fn = score_kernel<NT>(a);
    cudaError_t e = allow_smem(fn);
    if (e != cudaSuccess) return e;
    ScoreArgs copy = with_layout(a, NT);
    void* args[] = {&copy};
    cudaKernelNodeParams kp{};
    kp.func = const_cast<void*>(fn);
    kp.gridDim = dim3((unsigned)(a.n < grid ? a.n : grid));
    kp.blockDim = dim3(NT);
    kp.sharedMemBytes = (unsigned)smem;
    kp.kernelParams = args;
    return cudaGraphAddKernelNode(out, g, deps, ndeps, &kp);
}

cudaError_t add_score_node(cudaGraph_t g, const cudaGraphNode_t* deps, size_t ndeps,
                           const ScoreArgs& a, const ScoreConfig& cfg, int grid, cudaGraphNode_t* out)
{
    if (a.n <= 0 || a.n > 0xFFFFFFF0ll || grid <= 0 || a.job.tree.depth) return cudaErrorInvalidValue;
    switch (cfg.threads) {
    case 128: return add_score_node_nt<128>(g, deps, ndeps, a, cfg, grid, out);
    case 512: return add_score_node_nt<512>(g, deps, ndeps, a, cfg, grid, out);
    default: return add_score_node_nt<256>(g, deps, ndeps, a, cfg, grid, out);
    }
}

cudaError_t launch_score(const ScoreArgs& a, const ScoreConfig& cfg, int grid, cudaStream_t s)
{
    if (a.n <= 0) return cudaSuccess;
    if (grid <= 0) return cudaErrorInvalidValue;
    if (a.n > 0xFFFFFFF0ll) return cudaErrorInvalidValue;   // the counter is 32-bit
    switch (cfg.threads) {
    case 128: return launch_score_nt<128>(a, cfg, grid, s);
    case 512: return launch_score_nt<512>(a, cfg, grid, s);
    default: return launch_score_nt<256>(a, cfg, grid, s);
    }
}

// ---------------------------------------------------------------------------
// M2M GICP refinement (Sec. IV-A "Parallel M2M GICP")
// ---------------------------------------------------------------------------
//
// Per hypothesis (one block): render the mesh at the input pose, keep the
// visible, unoccluded pixels on the stride lattice as the source cloud (each
// with the camera-frame normal of its triangle), then iterate Gauss-Newton
// steps of the GICP objective against the observed cloud: every source point
// moved by the current increment is matched to its nearest observed point
// within delta (the radius search of the scorer), contributes 28 binary32
// terms (the 6x6 normal matrix's upper triangle, the gradient and r^T M r)
// that are rounded to multiples of 2^-24 and summed exactly in int64, and
// warp 0 solves the system in binary64 and updates the increment.  The
// fixed-point sums make the result independent of the summation order.

constexpr int kGicpTerms = 28;
// Three blocks of 256 threads (80 registers) per SM: 24 warps.  With the warp-wide
// solve: 26.8 ms for 20,480 refinements, against 32.0 ms for four blocks of 128
// threads (128 registers, 16 warps) and 29.8 ms for five (96 registers).
constexpr int kGicpThreads = 256;
constexpr float kGicpScale = 16777216.0f;    // 2^24
constexpr float kGicpLimit = 1048576.0f;     // a correspondence with a larger |term| is skipped

__device__ __forceinline__ float3 cross_rn(float3 a, float3 b)
{
    return make_float3(__fsub_rn(__fmul_rn(a.y, b.z), __fmul_rn(a.z, b.y)),
                       __fsub_rn(__fmul_rn(a.z, b.x), __fmul_rn(a.x, b.z)),
                       __fsub_rn(__fmul_rn(a.x, b.y), __fmul_rn(a.y, b.x)));
}

__device__ __forceinline__ float3 unit_or_zero(float3 c)
{
    const float len2 = __fadd_rn(__fadd_rn(__fmul_rn(c.x, c.x), __fmul_rn(c.y, c.y)), __fmul_rn(c.z, c.z));
    if (!(len2 > 0.0f)) return make_float3(0.0f, 0.0f, 0.0f);
    const float inv = __fdiv_rn(1.0f, __fsqrt_rn(len2));
    return make_float3(__fmul_rn(c.x, inv), __fmul_rn(c.y, inv), __fmul_rn(c.z, inv));
}

__device__ __forceinline__ float3 sub_rn(float4 a, float4 b)
{
    return make_float3(__fsub_rn(a.x, b.x), __fsub_rn(a.y, b.y), __fsub_rn(a.z, b.z));
}

// Object-frame unit normal of triangle t, vertex order as stored.
__device__ __forceinline__ float3 triangle_normal(const DevMesh& m, int t)
{
    const int4 tv = __ldg(&m.tris[t]);
    const float4 a = __ldg(&m.verts[tv.x]), b = __ldg(&m.verts[tv.y]), c = __ldg(&m.verts[tv.z]);
    return unit_or_zero(cross_rn(sub_rn(b, a), sub_rn(c, a)));
}

// R v for the 3x3 rotation stored row-major with row pitch `pitch`.
__device__ __forceinline__ float3 rotate_rn(const float* R, int pitch, float x, float y, float z)
{
    return make_float3(
        __fadd_rn(__fadd_rn(__fmul_rn(R[0], x), __fmul_rn(R[1], y)), __fmul_rn(R[2], z)),
        __fadd_rn(__fadd_rn(__fmul_rn(R[pitch], x), __fmul_rn(R[pitch + 1], y)), __fmul_rn(R[pitch + 2], z)),
        __fadd_rn(__fadd_rn(__fmul_rn(R[2 * pitch], x), __fmul_rn(R[2 * pitch + 1], y)),
                  __fmul_rn(R[2 * pitch + 2], z)));
}

__global__ void k_obs_normals(DevScene sc, int jump, float4* nrm)
{
    const int n = sc.W * sc.H;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int u = i % sc.W, v = i / sc.W;
        float3 nv = make_float3(0.0f, 0.0f, 0.0f);
        const int dc = sc.depth[i];
        if (dc != 0 && u >= 1 && v >= 1 && u + 1 < sc.W && v + 1 < sc.H) {
            const int nu[4] = {u - 1, u + 1, u, u}, nvv[4] = {v, v, v - 1, v + 1};
            float3 P[4];
            bool ok = true;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int d = sc.depth[nvv[k] * sc.W + nu[k]];
                if (d == 0 || abs(d - dc) > jump) ok = false;
                else P[k] = back_project(sc, nu[k], nvv[k], (unsigned)d);
            }
            if (ok) {
                const float3 a = make_float3(__fsub_rn(P[1].x, P[0].x), __fsub_rn(P[1].y, P[0].y),
                                             __fsub_rn(P[1].z, P[0].z));
                const float3 b = make_float3(__fsub_rn(P[3].x, P[2].x), __fsub_rn(P[3].y, P[2].y),
                                             __fsub_rn(P[3].z, P[2].z));
                nv = unit_or_zero(cross_rn(a, b));
            }
        }
        nrm[i] = make_float4(nv.x, nv.y, nv.z, 0.0f);
    }
}

cudaError_t launch_obs_normals(const DevScene& sc, int normal_jump, float4* nrm, cudaStream_t s)
{
    const int n = sc.W * sc.H;
    if (n <= 0) return cudaSuccess;
    k_obs_normals<<<(n + 255) / 256, 256, 0, s>>>(sc, normal_jump, nrm);
    return cudaGetLastError();
}

// The 28 terms of one correspondence: p = Rf a + tf (already moved), m = Rf na,
// observed b with normal nb.  False (no terms) when the combined covariance is
// not positive or a term is out of bounds.
__device__ __forceinline__ bool gicp_terms(const float* Rf, float3 p, float4 na, float3 b, float4 nb,
                                           float eps, float* out)
{
    const float3 m = rotate_rn(Rf, 3, na.x, na.y, na.z);
    const float e = __fsub_rn(1.0f, eps);
    // C = 2 I - e (nb nb^T + m m^T)
    const float c00 = __fsub_rn(2.0f, __fmul_rn(e, __fadd_rn(__fmul_rn(nb.x, nb.x), __fmul_rn(m.x, m.x))));
    const float c11 = __fsub_rn(2.0f, __fmul_rn(e, __fadd_rn(__fmul_rn(nb.y, nb.y), __fmul_rn(m.y, m.y))));
    const float c22 = __fsub_rn(2.0f, __fmul_rn(e, __fadd_rn(__fmul_rn(nb.z, nb.z), __fmul_rn(m.z, m.z))));
    const float c01 = -__fmul_rn(e, __fadd_rn(__fmul_rn(nb.x, nb.y), __fmul_rn(m.x, m.y)));
    const float c02 = -__fmul_rn(e, __fadd_rn(__fmul_rn(nb.x, nb.z), __fmul_rn(m.x, m.z)));
    const float c12 = -__fmul_rn(e, __fadd_rn(__fmul_rn(nb.y, nb.z), __fmul_rn(m.y, m.z)));
    // M = C^-1 (adjugate over determinant)
    const float a00 = __fsub_rn(__fmul_rn(c11, c22), __fmul_rn(c12, c12));
    const float a01 = __fsub_rn(__fmul_rn(c02, c12), __fmul_rn(c01, c22));
    const float a02 = __fsub_rn(__fmul_rn(c01, c12), __fmul_rn(c02, c11));
    const float a11 = __fsub_rn(__fmul_rn(c00, c22), __fmul_rn(c02, c02));
    const float a12 = __fsub_rn(__fmul_rn(c01, c02), __fmul_rn(c00, c12));
    const float a22 = __fsub_rn(__fmul_rn(c00, c11), __fmul_rn(c01, c01));
    const float det = __fadd_rn(__fadd_rn(__fmul_rn(c00, a00), __fmul_rn(c01, a01)), __fmul_rn(c02, a02));
    if (!(det > 0.0f)) return false;
    const float id = __fdiv_rn(1.0f, det);
    float M[3][3];
    M[0][0] = __fmul_rn(a00, id); M[0][1] = __fmul_rn(a01, id); M[0][2] = __fmul_rn(a02, id);
    M[1][1] = __fmul_rn(a11, id); M[1][2] = __fmul_rn(a12, id); M[2][2] = __fmul_rn(a22, id);
    M[1][0] = M[0][1]; M[2][0] = M[0][2]; M[2][1] = M[1][2];
    const float r[3] = {__fsub_rn(b.x, p.x), __fsub_rn(b.y, p.y), __fsub_rn(b.z, p.z)};
    // Jacobian of r with respect to (w, v) is [ [p]x , -I ]; MA = M [p]x
    float MA[3][3], AMA[3][3], Mr[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        MA[i][0] = __fsub_rn(__fmul_rn(M[i][1], p.z), __fmul_rn(M[i][2], p.y));
        MA[i][1] = __fsub_rn(__fmul_rn(M[i][2], p.x), __fmul_rn(M[i][0], p.z));
        MA[i][2] = __fsub_rn(__fmul_rn(M[i][0], p.y), __fmul_rn(M[i][1], p.x));
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        AMA[0][j] = __fsub_rn(__fmul_rn(p.z, MA[1][j]), __fmul_rn(p.y, MA[2][j]));
        AMA[1][j] = __fsub_rn(__fmul_rn(p.x, MA[2][j]), __fmul_rn(p.z, MA[0][j]));
        AMA[2][j] = __fsub_rn(__fmul_rn(p.y, MA[0][j]), __fmul_rn(p.x, MA[1][j]));
    }
#pragma unroll
    for (int i = 0; i < 3; ++i)
        Mr[i] = __fadd_rn(__fadd_rn(__fmul_rn(M[i][0], r[0]), __fmul_rn(M[i][1], r[1])), __fmul_rn(M[i][2], r[2]));
    int k = 0;
#pragma unroll
    for (int i = 0; i < 6; ++i) {
#pragma unroll
        for (int j = i; j < 6; ++j) {
            float h;
            if (i < 3 && j < 3) h = AMA[i][j];
            else if (i < 3) h = -MA[j - 3][i];
            else h = M[i - 3][j - 3];
            out[k++] = h;
        }
    }
    out[k++] = __fsub_rn(__fmul_rn(p.z, Mr[1]), __fmul_rn(p.y, Mr[2]));
    out[k++] = __fsub_rn(__fmul_rn(p.x, Mr[2]), __fmul_rn(p.z, Mr[0]));
    out[k++] = __fsub_rn(__fmul_rn(p.y, Mr[0]), __fmul_rn(p.x, Mr[1]));
    out[k++] = -Mr[0];
    out[k++] = -Mr[1];
    out[k++] = -Mr[2];
    out[k++] = __fadd_rn(__fadd_rn(__fmul_rn(r[0], Mr[0]), __fmul_rn(r[1], Mr[1])), __fmul_rn(r[2], Mr[2]));
    bool ok = true;
#pragma unroll
    for (int i = 0; i < kGicpTerms; ++i) ok = ok && fabsf(out[i]) < kGicpLimit;
    return ok;
}

// rint(2^24 term) of each lane, summed over the warp: hi 2^22 + lo, |term| < 2^20.
// Adding 1.5 x 2^23 rounds a binary32 value below 2^22 to an integer, ties to
// even, and leaves it in the low bits: first 4 term (the multiples of 2^22, any
// rounding will do), then the exact remainder, whose ties fall as the whole's
// because 2^22 is even.  The biased bits of 32 lanes wrap, and the wrapped sum
// less 32 biases is each sum exactly (|sum| < 2^27).  Two warp-wide integer
// additions in place of five 64-bit shuffles, and no conversion instructions.
__device__ __forceinline__ void warp_fixed_sum(float term, int& hi, int& lo)
{
    const float magic = 12582912.0f;             // 0x4B400000
    const float t = __fmaf_rn(term, 4.0f, magic);
    const float rest = __fmaf_rn(-__fsub_rn(t, magic), 4194304.0f, __fmul_rn(term, kGicpScale));
    const unsigned h = __reduce_add_sync(0xffffffffu, __float_as_uint(t));
    const unsigned l = __reduce_add_sync(0xffffffffu, __float_as_uint(__fadd_rn(rest, magic)));
    hi = (int)(h - 32u * 0x4B400000u);
    lo = (int)(l - 32u * 0x4B400000u);
}

// H xi = -g from the fixed-point sums, by Cholesky in binary64, by one warp.
// Lane k < 21 holds element (column c, row r >= c) of the lower triangle in the
// sums' order, lane 21 + c the right-hand side as a row 6; column q is finished
// (pivot, quotients) and subtracted from the columns after it, so every element
// sees its subtractions in the order of q, as a row-by-row evaluation does, and
// the result is that evaluation's to the bit.  The back substitution subtracts
// in rising order too, which leaves it serial; all lanes do it.  One thread
// alone took a sixth of a step: binary64 quotients and roots are long chains,
// and here 12 of them follow one another instead of 33.
__constant__ unsigned char c_gicp_col[27] = {0, 0, 0, 0, 0, 0, 1, 1, 1, 1, 1, 2, 2, 2, 2, 3, 3, 3, 4, 4, 5, 0, 1, 2, 3, 4, 5};
__constant__ unsigned char c_gicp_row[27] = {0, 1, 2, 3, 4, 5, 1, 2, 3, 4, 5, 2, 3, 4, 5, 3, 4, 5, 4, 5, 5, 6, 6, 6, 6, 6, 6};

__host__ __device__ constexpr int gicp_lane(int c, int r)
{
    return r == 6 ? 21 + c : 6 * c - c * (c - 1) / 2 + r - c;
}

__device__ __forceinline__ bool gicp_solve(const unsigned long long* S, int lane, double* xi)
{
    const int k = min(lane, 26), c = c_gicp_col[k], r = c_gicp_row[k];
    double t = __dmul_rn(__ll2double_rn((long long)S[k]), 1.0 / 16777216.0);     // exact scaling
    if (r == 6) t = -t;
#pragma unroll 1
    for (int q = 0; q < 6; ++q) {
        const double p = __shfl_sync(0xffffffffu, t, gicp_lane(q, q));
        if (!(p > 0.0)) return false;
        const double d = __dsqrt_rn(p);
        if (c == q) t = r == q ? d : __ddiv_rn(t, d);
        const double lr = __shfl_sync(0xffffffffu, t, gicp_lane(q, max(r, q)));
        const double lc = __shfl_sync(0xffffffffu, t, gicp_lane(q, max(c, q)));
        if (c > q) t = __dsub_rn(t, __dmul_rn(lr, lc));
    }
#pragma unroll
    for (int i = 5; i >= 0; --i) {
        double x = __shfl_sync(0xffffffffu, t, gicp_lane(i, 6));
#pragma unroll
        for (int q = i + 1; q < 6; ++q) x = __dsub_rn(x, __dmul_rn(__shfl_sync(0xffffffffu, t, gicp_lane(i, q)), xi[q]));
        xi[i] = __ddiv_rn(x, __shfl_sync(0xffffffffu, t, gicp_lane(i, i)));
    }
    return true;
}

// Apply the step xi to the increment (R, t): R <- dR R, t <- dR t + v, with
// dR the rotation of the quaternion (1, w/2) normalised; by one warp, lane 3 i +
// j on R[i][j] and lane 9 + i on t[i].  True when the step is below the
// stopping thresholds.
__device__ __forceinline__ bool gicp_update(double* R, double* t, const double* xi, float stop_rot, float stop_trans,
                                            int lane)
{
    const double hx = __dmul_rn(xi[0], 0.5), hy = __dmul_rn(xi[1], 0.5), hz = __dmul_rn(xi[2], 0.5);
    const double nrm = __dsqrt_rn(__dadd_rn(__dadd_rn(__dadd_rn(1.0, __dmul_rn(hx, hx)), __dmul_rn(hy, hy)),
                                            __dmul_rn(hz, hz)));
    const double qk = __ddiv_rn(lane == 0 ? 1.0 : lane == 1 ? hx : lane == 2 ? hy : hz, nrm);
    const double qw = __shfl_sync(0xffffffffu, qk, 0), qx = __shfl_sync(0xffffffffu, qk, 1);
    const double qy = __shfl_sync(0xffffffffu, qk, 2), qz = __shfl_sync(0xffffffffu, qk, 3);
    double d[9];
    d[0] = __dsub_rn(1.0, __dmul_rn(2.0, __dadd_rn(__dmul_rn(qy, qy), __dmul_rn(qz, qz))));
    d[1] = __dmul_rn(2.0, __dsub_rn(__dmul_rn(qx, qy), __dmul_rn(qw, qz)));
    d[2] = __dmul_rn(2.0, __dadd_rn(__dmul_rn(qx, qz), __dmul_rn(qw, qy)));
    d[3] = __dmul_rn(2.0, __dadd_rn(__dmul_rn(qx, qy), __dmul_rn(qw, qz)));
    d[4] = __dsub_rn(1.0, __dmul_rn(2.0, __dadd_rn(__dmul_rn(qx, qx), __dmul_rn(qz, qz))));
    d[5] = __dmul_rn(2.0, __dsub_rn(__dmul_rn(qy, qz), __dmul_rn(qw, qx)));
    d[6] = __dmul_rn(2.0, __dsub_rn(__dmul_rn(qx, qz), __dmul_rn(qw, qy)));
    d[7] = __dmul_rn(2.0, __dadd_rn(__dmul_rn(qy, qz), __dmul_rn(qw, qx)));
    d[8] = __dsub_rn(1.0, __dmul_rn(2.0, __dadd_rn(__dmul_rn(qx, qx), __dmul_rn(qy, qy))));
    const int i = lane < 9 ? lane / 3 : min(lane - 9, 2), j = lane % 3;
    const double d0 = i == 0 ? d[0] : i == 1 ? d[3] : d[6], d1 = i == 0 ? d[1] : i == 1 ? d[4] : d[7];
    const double d2 = i == 0 ? d[2] : i == 1 ? d[5] : d[8];
    const double* const col = lane < 9 ? R + j : t;
    const int pitch = lane < 9 ? 3 : 1;
    double x = __dadd_rn(__dadd_rn(__dmul_rn(d0, col[0]), __dmul_rn(d1, col[pitch])), __dmul_rn(d2, col[2 * pitch]));
    if (lane >= 9) x = __dadd_rn(x, i == 0 ? xi[3] : i == 1 ? xi[4] : xi[5]);
    __syncwarp();
    if (lane < 9) R[lane] = x;
    else if (lane < 12) t[i] = x;
    __syncwarp();
    const double sr = (double)stop_rot, st = (double)stop_trans;
    const double w2 = __dadd_rn(__dadd_rn(__dmul_rn(xi[0], xi[0]), __dmul_rn(xi[1], xi[1])), __dmul_rn(xi[2], xi[2]));
    const double v2 = __dadd_rn(__dadd_rn(__dmul_rn(xi[3], xi[3]), __dmul_rn(xi[4], xi[4])), __dmul_rn(xi[5], xi[5]));
    return w2 < __dmul_rn(sr, sr) && v2 < __dmul_rn(st, st);
}

// Render the hypothesis in z-buffer tiles and append its source cloud
// (visible, unoccluded pixels on the stride lattice) to src; *count ends as
// the number of source points (entries past cap are not written).
template <int NT, bool K32, bool VC>
__device__ void gicp_source(const GicpArgs& a, const Job& J, const float* P, const unsigned long long* vc,
                            const int* rbox, uint32_t* zbuf, unsigned probe_off, float4* src, int* count)
{
    const DevScene& sc = J.sc;
    const int s = sc.stride;
    const int rw = rbox[2] - rbox[0], rh = rbox[3] - rbox[1];
    if (rw <= 0 || rh <= 0) return;
    const int cap_px = K32 ? a.zcap_words : a.zcap_words / 2;
    const int tw = min(rw, cap_px);
    const int th = max(1, cap_px / tw);
    for (int tv0 = rbox[1]; tv0 < rbox[3]; tv0 += th) {
        for (int tu0 = rbox[0]; tu0 < rbox[2]; tu0 += tw) {
            const int tu1 = min(tu0 + tw, rbox[2]), tv1 = min(tv0 + th, rbox[3]);
            const int words = K32 ? tw * (tv1 - tv0) : 2 * tw * (tv1 - tv0);
            for (int i = threadIdx.x; i < words; i += NT) zbuf[i] = 0xFFFFFFFFu;
            __syncthreads();
            raster<NT, K32, VC>(sc, J.m, P, vc, probe_off, probe_off + (unsigned)kWarpScratch * (NT / 32), tu0, tv0,
                                tu1, tv1, tw, a.err);
            __syncthreads();
            const int us0 = ((tu0 + s - 1) / s) * s, vs0 = ((tv0 + s - 1) / s) * s;
            const int nu = us0 < tu1 ? (tu1 - 1 - us0) / s + 1 : 0;
            const int nv = vs0 < tv1 ? (tv1 - 1 - vs0) / s + 1 : 0;
            for (int k = threadIdx.x; k < nu * nv; k += NT) {
                const int kv = div_small(k, nu);
                const int u = us0 + (k - kv * nu) * s, v = vs0 + kv * s;
                const int zi = (v - tv0) * tw + (u - tu0);
                unsigned d = 0;
                int tri = -1;
                if (K32) {
                    const uint32_t w = zbuf[zi];
                    if (w != 0xFFFFFFFFu) { d = w >> 16; tri = (int)(w & 0xFFFFu); }
                } else {
                    const unsigned long long w = reinterpret_cast<unsigned long long*>(zbuf)[zi];
                    if (w != kEmptyKey) { d = (unsigned)(w >> 32); tri = (int)(uint32_t)w; }
                }
                if (tri < 0) continue;
                const int pix = v * sc.W + u;
                const unsigned dobs = __ldg(&sc.depth[pix]);
                const bool occluded = sc.occ_margin >= 0 && dobs > 0 &&
                                      (unsigned long long)dobs + (unsigned)sc.occ_margin < d &&
                                      (J.label < 0 || __ldg(&sc.labels[pix]) != J.label);
                if (occluded) continue;
                const float3 q = back_project(sc, u, v, d);
                const float3 no = triangle_normal(J.m, tri);
                const float3 nc = rotate_rn(P, 4, no.x, no.y, no.z);
                const int idx = atomicAdd(count, 1);
                if (idx < a.src_cap) {
                    src[2 * (size_t)idx] = make_float4(q.x, q.y, q.z, 0.0f);
                    src[2 * (size_t)idx + 1] = make_float4(nc.x, nc.y, nc.z, 0.0f);
                }
            }
            __syncthreads();
        }
    }
}

__host__ __device__ inline size_t gicp_probe_offset(int zcap_words)
{
    return align16(sizeof(uint32_t) * (size_t)zcap_words);
}

template <int NT>
__global__ void __launch_bounds__(NT, 768 / NT) k_gicp(const __grid_constant__ GicpArgs a)
{
    unsigned char* const smem = g_smem;
    __shared__ float s_pose[12], s_Rf[9], s_tf[3];
    __shared__ double s_R[9], s_t[3];
    __shared__ unsigned long long s_sum[kGicpTerms];
    __shared__ int s_rbox[4], s_k32, s_slot, s_nsrc, s_corr, s_done, s_updates, s_last;
    __shared__ long long s_h;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const Job& J = a.job;
    const DevScene& sc = J.sc;
    uint32_t* zbuf = reinterpret_cast<uint32_t*>(smem);
    const unsigned probe_off = (unsigned)gicp_probe_offset(a.zcap_words);
    char* probe = reinterpret_cast<char*>(smem) + probe_off;
    WarpProbe& WP = *reinterpret_cast<WarpProbe*>(probe + warp * kWarpScratch);
    if (threadIdx.x == 0) {
        s_slot = claim_vslot(a.smask, a.slots);
        if (s_slot < 0) atomicOr(a.err, kErrNoSlot);
    }
    __syncthreads();
    if (s_slot < 0) return;
    const unsigned long long* vc = a.vcache ? a.vcache + (size_t)s_slot * a.vstride : nullptr;
    float4* src = a.src + (size_t)s_slot * 2 * (size_t)a.src_cap;
    const MarkBand nomark = {nullptr, 0, 0, 0, 0, 0, a.err};
    for (;;) {
        if (threadIdx.x == 0) s_h = (long long)atomicAdd(a.next, 1u);
        __syncthreads();
        const long long h = s_h;
        if (h >= a.n) break;
        if (threadIdx.x < 12) s_pose[threadIdx.x] = J.poses[h * 12 + threadIdx.x];
        if (threadIdx.x == 0) s_nsrc = 0;
        __syncthreads();
        if (threadIdx.x < 32) {
            const PixelBox b = project_box(make_float4(sc.fx, sc.fy, sc.cx, sc.cy), s_pose,
                                           make_float3(J.m.lo[0], J.m.lo[1], J.m.lo[2]),
                                           make_float3(J.m.hi[0], J.m.hi[1], J.m.hi[2]),
                                           make_int4(J.roi[0], J.roi[1], J.roi[2], J.roi[3]));
            if (lane == 0) {
                s_rbox[0] = b.box.x; s_rbox[1] = b.box.y; s_rbox[2] = b.box.z; s_rbox[3] = b.box.w;
                s_k32 = (J.m.n_tris <= 65535 && b.zmax < 6.5f) ? 1 : 0;
            }
        }
        if (vc) vertex_pass(sc, J.m, s_pose, const_cast<unsigned long long*>(vc), NT);
        __syncthreads();
        if (s_k32) {
            if (vc) gicp_source<NT, true, true>(a, J, s_pose, vc, s_rbox, zbuf, probe_off, src, &s_nsrc);
            else gicp_source<NT, true, false>(a, J, s_pose, vc, s_rbox, zbuf, probe_off, src, &s_nsrc);
        } else {
            if (vc) gicp_source<NT, false, true>(a, J, s_pose, vc, s_rbox, zbuf, probe_off, src, &s_nsrc);
            else gicp_source<NT, false, false>(a, J, s_pose, vc, s_rbox, zbuf, probe_off, src, &s_nsrc);
        }
        const int nsrc = s_nsrc;
        if (nsrc > a.src_cap) {
            // the source cloud does not fit its slot: the pose is returned unchanged
            if (threadIdx.x < 12) a.poses_out[h * 12 + threadIdx.x] = s_pose[threadIdx.x];
            if (threadIdx.x == 0) {
                atomicOr(a.err, kErrSourceCap);
                if (a.info) { a.info[2 * h] = -1; a.info[2 * h + 1] = nsrc; }
            }
            __syncthreads();
            continue;
        }
        if (threadIdx.x == 0) {
            for (int i = 0; i < 9; ++i) { s_R[i] = (i % 4 == 0) ? 1.0 : 0.0; s_Rf[i] = (float)s_R[i]; }
            for (int i = 0; i < 3; ++i) { s_t[i] = 0.0; s_tf[i] = 0.0f; }
            s_done = 0;
            s_updates = 0;
            s_last = 0;
        }
        __syncthreads();
        for (int it = 0; it < a.max_iters; ++it) {
            if (threadIdx.x < kGicpTerms) s_sum[threadIdx.x] = 0ull;
            if (threadIdx.x == 0) s_corr = 0;
            __syncthreads();
            long long acc = 0;
            int corr = 0;
            for (int base = warp * 32; base < nsrc; base += NT) {
                const int i = base + lane;
                const bool valid = i < nsrc;
                float4 A = make_float4(0.f, 0.f, 0.f, 0.f), NA = A;
                if (valid) { A = src[2 * (size_t)i]; NA = src[2 * (size_t)i + 1]; }
                const float3 r0 = rotate_rn(s_Rf, 3, A.x, A.y, A.z);
                const float3 p = make_float3(__fadd_rn(r0.x, s_tf[0]), __fadd_rn(r0.y, s_tf[1]),
                                             __fadd_rn(r0.z, s_tf[2]));
                const unsigned long long nn = probe_batch<false, false>(sc, valid, p.x, p.y, p.z, 0u, WP, lane, nomark);
                bool ok = valid && nn != kEmptyKey;
                float terms[kGicpTerms];
#pragma unroll
                for (int j = 0; j < kGicpTerms; ++j) terms[j] = 0.0f;
                if (ok) {
                    const uint32_t pw = (uint32_t)nn;
                    const int pu = (int)(pw & 0xFFFFu), pv = (int)(pw >> 16);
                    const int pix = pv * sc.W + pu;
                    const float3 b = back_project(sc, pu, pv, __ldg(&sc.depth[pix]));
                    ok = gicp_terms(s_Rf, p, NA, b, __ldg(&a.nrm[pix]), a.epsilon, terms);
                }
                const unsigned bal = __ballot_sync(0xffffffffu, ok);
                corr += __popc(bal);
                if (bal) {
#pragma unroll
                    for (int j = 0; j < kGicpTerms; ++j) {
                        int hi, lo;
                        warp_fixed_sum(ok ? terms[j] : 0.0f, hi, lo);
                        if (lane == j) acc += (long long)hi * 4194304ll + lo;
                    }
                }
            }
            if (lane < kGicpTerms) atomicAdd(&s_sum[lane], (unsigned long long)acc);
            if (lane == 0) atomicAdd(&s_corr, corr);
            __syncthreads();
            if (warp == 0) {
                const int n_corr = s_corr;
                double xi[6];
                bool done = true, stepped = false;
                if (n_corr >= a.min_corr && gicp_solve(s_sum, lane, xi)) {
                    done = gicp_update(s_R, s_t, xi, a.stop_rot, a.stop_trans, lane);
                    stepped = true;
                    if (lane < 9) s_Rf[lane] = __double2float_rn(s_R[lane]);
                    else if (lane < 12) s_tf[lane - 9] = __double2float_rn(s_t[lane - 9]);
                }
                if (lane == 0) {
                    s_last = n_corr;
                    s_done = done;
                    s_updates += stepped;
                }
            }
            __syncthreads();
            if (s_done) break;
        }
        // refined pose = increment o input pose
        if (threadIdx.x < 12) {
            const int i = threadIdx.x / 4, j = threadIdx.x % 4;
            const float* P = s_pose;
            double x;
            if (j < 3) {
                x = __dadd_rn(__dadd_rn(__dmul_rn(s_R[3 * i], (double)P[j]), __dmul_rn(s_R[3 * i + 1], (double)P[4 + j])),
                              __dmul_rn(s_R[3 * i + 2], (double)P[8 + j]));
            } else {
                x = __dadd_rn(__dadd_rn(__dadd_rn(__dmul_rn(s_R[3 * i], (double)P[3]),
                                                  __dmul_rn(s_R[3 * i + 1], (double)P[7])),
                                        __dmul_rn(s_R[3 * i + 2], (double)P[11])), s_t[i]);
            }
            a.poses_out[h * 12 + threadIdx.x] = __double2float_rn(x);
        }
        if (threadIdx.x == 0 && a.info) {
            a.info[2 * h] = s_updates;
            a.info[2 * h + 1] = s_last;
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAnd(&a.smask[s_slot >> 5], ~(1u << (s_slot & 31)));
    }
}

size_t gicp_smem_bytes(int zcap_words)
{
    return gicp_probe_offset(zcap_words) + (kWarpScratch + sizeof(DepthItem) * kRing) * (kGicpThreads / 32);
}

int gicp_grid(int zcap_words)
{
    int dev = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const size_t smem = gicp_smem_bytes(zcap_words);
    if (allow_smem((const void*)k_gicp<kGicpThreads>) != cudaSuccess) return -1;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_gicp<kGicpThreads>, kGicpThreads, smem) != cudaSuccess)
        return -1;
    return max(1, per) * max(1, sms);
}

cudaError_t launch_gicp(const GicpArgs& a, int grid, cudaStream_t s)
{
    if (a.n <= 0) return cudaSuccess;
    if (a.n > 0xFFFFFFF0ll || grid <= 0 || grid > a.slots) return cudaErrorInvalidValue;
    const size_t smem = gicp_smem_bytes(a.zcap_words);
    cudaError_t e = allow_smem((const void*)k_gicp<kGicpThreads>);
    if (e != cudaSuccess) return e;
    k_gicp<kGicpThreads><<<(unsigned)(a.n < grid ? a.n : grid), kGicpThreads, smem, s>>>(a);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// 6-DoF pose proposals (Sec. V-B, Eq. 5 and Eq. 6)
// ---------------------------------------------------------------------------

__global__ void k_mask_depth_range(ProposalArgs a)
{
    const int bw = a.box[2] - a.box[0], bh = a.box[3] - a.box[1];
    unsigned lo = 0xFFFFFFFFu, hi = 0u;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < bw * bh; i += gridDim.x * blockDim.x) {
        const int u = a.box[0] + i % bw, v = a.box[1] + i / bw;
        const int pix = v * a.sc.W + u;
        const unsigned d = a.sc.depth[pix];
        if (d != 0 && a.sc.labels[pix] == a.label) {
            lo = min(lo, d);
            hi = max(hi, d);
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    if ((threadIdx.x & 31) == 0 && hi != 0u) {
        atomicMin(&a.zr[0], lo);
        atomicMax(&a.zr[1], hi);
    }
}

__global__ void k_proposals(ProposalArgs a)
{
    const long long total = (long long)a.M * a.N * a.K;
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx == 0 && a.z_out) {
        const bool any = a.zr[1] != 0u;
        a.z_out[0] = any ? (int32_t)a.zr[0] : 0;
        a.z_out[1] = any ? (int32_t)a.zr[1] : 0;
    }
    if (idx >= total) return;
    const int j = (int)(idx % a.K);
    const int k = (int)((idx / a.K) % a.N);
    const int i = (int)(idx / ((long long)a.K * a.N));
    // viewpoint i of the Fibonacci lattice (object frame, towards the camera)
    const float golden = 2.39996322972865332f;          // pi (3 - sqrt 5)
    const float y = 1.0f - (2.0f * i + 1.0f) / (float)a.M;
    const float rad = sqrtf(fmaxf(0.0f, 1.0f - y * y));
    const float phi = golden * (float)i;
    const float vx = rad * cosf(phi), vy = y, vz = rad * sinf(phi);
    // camera axes in the object frame: forward = -v, right, down
    const float fx = -vx, fy = -vy, fz = -vz;
    float rx = fy * 1.0f - fz * 0.0f, ry = fz * 0.0f - fx * 1.0f, rz = 0.0f;   // forward x (0,0,1)
    float rn = sqrtf(rx * rx + ry * ry + rz * rz);
    if (rn < 1e-6f) {                                   // forward parallel to z: use (0,1,0)
        rx = fy * 0.0f - fz * 1.0f;
        ry = fz * 0.0f - fx * 0.0f;
        rz = fx * 1.0f - fy * 0.0f;
        rn = sqrtf(rx * rx + ry * ry + rz * rz);
    }
    rx /= rn; ry /= rn; rz /= rn;
    const float dx = fy * rz - fz * ry, dy = fz * rx - fx * rz, dz = fx * ry - fy * rx;
    // in-plane rotation about the optical axis
    const float th = 6.28318530717958648f * (float)k / (float)a.N;
    const float c = cosf(th), s = sinf(th);
    const float R[9] = {c * rx - s * dx, c * ry - s * dy, c * rz - s * dz,
                        s * rx + c * dx, s * ry + c * dy, s * rz + c * dz,
                        fx, fy, fz};
    // translation: the box centre back-projected at depth z_j
    const bool any = a.zr[1] != 0u;
    const float zmin = any ? (float)a.zr[0] / 10000.0f : 0.0f;
    const float zmax = any ? (float)a.zr[1] / 10000.0f : 0.0f;
    const float z = a.K > 1 ? zmin + (zmax - zmin) * (float)j / (float)(a.K - 1) : 0.5f * (zmin + zmax);
    const float uc = 0.5f * (float)(a.box[0] + a.box[2] - 1), vc = 0.5f * (float)(a.box[1] + a.box[3] - 1);
    const float cxp = (uc - a.sc.cx) * z / a.sc.fx, cyp = (vc - a.sc.cy) * z / a.sc.fy;
    float* out = a.poses + 12 * idx;
    const float m0 = a.centre[0], m1 = a.centre[1], m2 = a.centre[2];
    out[0] = R[0]; out[1] = R[1]; out[2] = R[2];
    out[3] = cxp - (R[0] * m0 + R[1] * m1 + R[2] * m2);
    out[4] = R[3]; out[5] = R[4]; out[6] = R[5];
    out[7] = cyp - (R[3] * m0 + R[4] * m1 + R[5] * m2);
    out[8] = R[6]; out[9] = R[7]; out[10] = R[8];
    out[11] = z - (R[6] * m0 + R[7] * m1 + R[8] * m2);
}

cudaError_t launch_proposals(const ProposalArgs& a, cudaStream_t s)
{
    cudaError_t e = cudaMemsetAsync(a.zr, 0xFF, sizeof(unsigned), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(a.zr + 1, 0, sizeof(unsigned), s);
    if (e != cudaSuccess) return e;
    const int area = (a.box[2] - a.box[0]) * (a.box[3] - a.box[1]);
    if (area > 0) k_mask_depth_range<<<min(1024, (area + 255) / 256), 256, 0, s>>>(a);
    const long long total = (long long)a.M * a.N * a.K;
    k_proposals<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(a);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// argmin of J = J_o + J_r (the last block reduces the blocks' results)
// ---------------------------------------------------------------------------
//
// Bound by latency, not by bytes: a launch is one or a few rounds of loads, the
// block's reduction, the ticket and the last block's reduction in a row.  So the
// costs are read first, kBestUnroll pairs in flight per thread, and only a thread
// that holds the block's smallest J reads an id (all of its equal ones, in a second
// pass over its pairs, when it holds several); reductions are warp-wide integer
// minima of 32 bits, one per part of the key.  A call in a queue of calls, with
// ids: 500 pairs 4.1 us (6.2 with one pair in flight per thread, every id read and
// 64-bit shuffles), 300,001 pairs 6.2 (9.2), 2,000,000 pairs 8.2 (12.3) and, all
// equal, 10.3 (13.3).
constexpr int kBestThreads = 256;
constexpr int kBestUnroll = 4;
constexpr int kBestGrid = 608;           // blocks at most, on any device: four per SM of 152
static_assert(kBestGrid <= kBestMaxBlocks, "a block's result has its place in the scratch");

struct BestKey {
    unsigned J;              // compared as unsigned, like the upper half of the packed key
    unsigned long long id;   // caller id or index
    unsigned idx;            // below 2^31; the key of nothing has all bits set
};

__device__ __forceinline__ BestKey best_none() { return {0xFFFFFFFFu, ~0ull, 0xFFFFFFFFu}; }

// The smallest key of the warp's lanes by (J, id, index), in every lane.
__device__ __forceinline__ BestKey warp_best(const BestKey& k)
{
    const unsigned full = 0xffffffffu, hi = (unsigned)(k.id >> 32), lo = (unsigned)k.id;
    const unsigned J = __reduce_min_sync(full, k.J);
    const unsigned h = __reduce_min_sync(full, k.J == J ? hi : full);
    const unsigned l = __reduce_min_sync(full, k.J == J && hi == h ? lo : full);
    const unsigned x = __reduce_min_sync(full, k.J == J && hi == h && lo == l ? k.idx : full);
    return {J, ((unsigned long long)h << 32) | l, x};
}

// The smallest key of the block's threads (in every lane of every warp).
__device__ __forceinline__ BestKey block_best(BestKey k, BestKey* sh)
{
    const int lane = threadIdx.x & 31;
    k = warp_best(k);
    if (lane == 0) sh[threadIdx.x >> 5] = k;
    __syncthreads();
    return warp_best(lane < kBestThreads / 32 ? sh[lane] : best_none());
}

// J of pair i (its low 32 bits); costs may be aligned to 4 bytes only.
__device__ __forceinline__ unsigned pair_cost(const BestArgs& a, bool wide, long long i)
{
    if (wide) {
        const int2 c = reinterpret_cast<const int2*>(a.costs)[i];
        return (unsigned)c.x + (unsigned)c.y;
    }
    return (unsigned)a.costs[2 * i] + (unsigned)a.costs[2 * i + 1];
}

__global__ void __launch_bounds__(kBestThreads) k_best(BestArgs a)
{
    __shared__ BestKey sh[2][kBestThreads / 32];
    __shared__ unsigned low[kBestThreads / 32];
    __shared__ bool last;
    const bool wide = (reinterpret_cast<uintptr_t>(a.costs) & 7) == 0;
    const long long first = blockIdx.x * (long long)(kBestThreads * kBestUnroll) + threadIdx.x;
    const long long step = gridDim.x * (long long)(kBestThreads * kBestUnroll);
    unsigned best = 0xFFFFFFFFu, at = 0xFFFFFFFFu;    // smallest J and the first index that has it
    bool ties = false;
    for (long long b = first; b < a.n; b += step) {
        unsigned J[kBestUnroll];
#pragma unroll
        for (int u = 0; u < kBestUnroll; ++u)
            J[u] = b + u * kBestThreads < a.n ? pair_cost(a, wide, b + u * kBestThreads) : 0xFFFFFFFFu;
#pragma unroll
        for (int u = 0; u < kBestUnroll; ++u) {
            const long long i = b + u * kBestThreads;
            if (i >= a.n) continue;
            if (J[u] < best || at == 0xFFFFFFFFu) {
                best = J[u];
                at = (unsigned)i;
                ties = false;
            } else if (J[u] == best) {
                ties = true;
            }
        }
    }
    const unsigned w = __reduce_min_sync(0xffffffffu, best);
    if ((threadIdx.x & 31) == 0) low[threadIdx.x >> 5] = w;
    __syncthreads();
    unsigned m = low[0];
#pragma unroll
    for (int i = 1; i < kBestThreads / 32; ++i) m = min(m, low[i]);
    BestKey k = best_none();
    if (best == m && at != 0xFFFFFFFFu) {
        k = {m, a.ids ? a.ids[at] : (unsigned long long)at, at};
        if (a.ids && ties) {
            for (long long b = first; b < a.n; b += step) {
                unsigned long long id[kBestUnroll];
                bool eq[kBestUnroll];
#pragma unroll
                for (int u = 0; u < kBestUnroll; ++u) {
                    const long long i = b + u * kBestThreads;
                    eq[u] = i < a.n && pair_cost(a, wide, i) == m;
                    id[u] = eq[u] ? a.ids[i] : ~0ull;
                }
#pragma unroll
                for (int u = 0; u < kBestUnroll; ++u)      // indices ascend: the first of equal ids stays
                    if (eq[u] && id[u] < k.id) {
                        k.id = id[u];
                        k.idx = (unsigned)(b + u * kBestThreads);
                    }
            }
        }
    }
    k = block_best(k, sh[0]);
    if (gridDim.x > 1) {
        if (threadIdx.x == 0) {
            a.partial[3 * blockIdx.x + 0] = k.J;
            a.partial[3 * blockIdx.x + 1] = k.id;
            a.partial[3 * blockIdx.x + 2] = k.idx;
            __threadfence();
            last = atomicAdd(a.ticket, 1u) == gridDim.x - 1;
        }
        __syncthreads();
        if (!last) return;
        __threadfence();
        k = best_none();
        for (unsigned b = threadIdx.x; b < gridDim.x; b += kBestThreads) {
            const volatile unsigned long long* const p = a.partial + 3 * b;
            const BestKey c = {(unsigned)p[0], p[1], (unsigned)p[2]};
            if (c.J < k.J || (c.J == k.J && (c.id < k.id || (c.id == k.id && c.idx < k.idx)))) k = c;
        }
        k = block_best(k, sh[1]);
        if (threadIdx.x == 0) *a.ticket = 0u;
    }
    if (threadIdx.x == 0) {
        if (a.best_index) *a.best_index = k.idx;
        if (a.best_cost) *a.best_cost = (int32_t)k.J;
        // (J << 32) | id: the smallest such key over several shards is their winner
        if (a.key) *a.key = ((unsigned long long)k.J << 32) | (k.id & 0xFFFFFFFFull);
    }
}

int best_blocks(long long n)
{
    const long long b = (n + kBestThreads * kBestUnroll - 1) / (kBestThreads * kBestUnroll);
    return (int)(b < 1 ? 1 : (b > kBestGrid ? kBestGrid : b));
}

cudaError_t launch_best(const BestArgs& a, cudaStream_t s)
{
    k_best<<<best_blocks(a.n), kBestThreads, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace perch
