// majorant.cu -- field ingest and the majorant pyramid (sm_103a).
//
// K2+K1 fused (relayout_l1): the row-major extinction field is rewritten into
// 8x8x8 bricks (Sec. 3.1.2: voxels kept in fixed-size spatially coherent
// blocks) and, in the same pass, the max of every brick -- the level-1 cell of
// the pyramid -- is reduced.  One pass over HBM: 4 B read + 4 B (or 2 B) written
// per voxel plus 4 B per 512 voxels.
// K1 (reduce_level): level L >= 2 cells take the exact max and min of their (up to)
// 8x8x8 children (Sec. 3.1.1: merged voxels store the max).  Max is exact and
// order-free, so the result is bit-identical to any other evaluation order.
// Octree (oct_bricks, oct_reduce2): the paper's own grid, Sec. 3.1.1 --
// groups of 2^3 cells merged recursively, each cell keeping the max and the
// min of the voxels it covers.  Levels 1 to 3 come from one pass over the
// stored voxels (bricks); level L >= 4 reduces 2^3 cells of level L - 1.
// Leaf map (either grid): for each level-1 cell, the coarsest ancestor whose
// majorant times its height is <= tau~ (Sec. 4.2's merge criterion), with
// its majorant, its minorant (the min levels, built alongside the max) and
// its size as a voxel shift.
#include <cuda_bf16.h>

#include "mcrt_internal.h"

namespace mcrt {

namespace {

// One block of 256 threads = 4 consecutive bricks along x.  Thread t holds
// row r = t >> 2 (y & 7 = r & 7, z & 7 = r >> 3) of brick q = t & 3.
template <bool BF16>
__global__ void __launch_bounds__(256) relayout_l1_kernel(const float* __restrict__ src, int nx, int ny, int nz,
                                                          int nbx, int nby, void* __restrict__ dst,
                                                          float* __restrict__ l1, float* __restrict__ l1min)
{
    const int t = threadIdx.x;
    const int q = t & 3;
    const int r = t >> 2;
    const int bx = blockIdx.x * 4 + q;
    const int by = blockIdx.y;
    const int bz = blockIdx.z;
    const int y = by * 8 + (r & 7);
    const int z = bz * 8 + (r >> 3);
    const int x0 = bx * 8;
    float v[8];
    const bool row_ok = (bx < nbx) && (y < ny) && (z < nz);
    const size_t row = ((size_t)z * ny + y) * (size_t)nx;
    if (row_ok && x0 + 8 <= nx && (nx & 3) == 0 &&
        ((reinterpret_cast<uintptr_t>(src) & 15u) == 0)) {
        const float4 a = __ldcs(reinterpret_cast<const float4*>(src + row + x0));
        const float4 b = __ldcs(reinterpret_cast<const float4*>(src + row + x0 + 4));
        v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
        v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = (row_ok && x0 + i < nx) ? src[row + x0 + i] : 0.0f;
    }
    float m = 0.0f;
    float mn = __int_as_float(0x7f800000);   // min over the existing voxels (as stored)
    if (BF16) {
        // stored voxels: nearest bf16; majorant: smallest bf16 >= the FP32 max,
        // which bounds every nearest-rounded voxel of the brick
        uint32_t packed[4];
#pragma unroll
        for (int i = 0; i < 8; i += 2) {
            const uint32_t lo = __bfloat16_as_ushort(__float2bfloat16_rn(v[i]));
            const uint32_t hi = __bfloat16_as_ushort(__float2bfloat16_rn(v[i + 1]));
            packed[i / 2] = lo | (hi << 16);
            m = fmaxf(m, fmaxf(v[i], v[i + 1]));
            if (row_ok && x0 + i < nx) mn = fminf(mn, __uint_as_float(lo << 16));
            if (row_ok && x0 + i + 1 < nx) mn = fminf(mn, __uint_as_float(hi << 16));
        }
        m = __bfloat162float(__float2bfloat16_ru(m));
        if (bx < nbx) {
            const size_t brick = ((size_t)bz * nby + by) * (size_t)nbx + bx;
            uint4* o = reinterpret_cast<uint4*>(static_cast<uint16_t*>(dst) + brick * 512 + r * 8);
            __stcs(o, make_uint4(packed[0], packed[1], packed[2], packed[3]));
        }
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            m = fmaxf(m, v[i]);
            if (row_ok && x0 + i < nx) mn = fminf(mn, v[i]);
        }
        if (bx < nbx) {
            const size_t brick = ((size_t)bz * nby + by) * (size_t)nbx + bx;
            float4* o = reinterpret_cast<float4*>(static_cast<float*>(dst) + brick * 512 + r * 8);
            __stcs(o, make_float4(v[0], v[1], v[2], v[3]));
            __stcs(o + 1, make_float4(v[4], v[5], v[6], v[7]));
        }
    }
    // max over the 64 rows of each brick: lanes sharing q differ in bits 2..4
    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 4));
    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 8));
    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 16));
    mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, 4));
    mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, 8));
    mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, 16));
    __shared__ float part[8][4], partmin[8][4];
    if ((t & 31) < 4) { part[t >> 5][q] = m; partmin[t >> 5][q] = mn; }
    __syncthreads();
    if (t < 4) {
        float mm = part[0][t], mmn = partmin[0][t];
#pragma unroll
        for (int w = 1; w < 8; ++w) { mm = fmaxf(mm, part[w][t]); mmn = fminf(mmn, partmin[w][t]); }
        const int bxx = blockIdx.x * 4 + t;
        if (bxx < nbx) {
            l1[((size_t)bz * nby + by) * (size_t)nbx + bxx] = mm;
            l1min[((size_t)bz * nby + by) * (size_t)nbx + bxx] = mmn;
        }
    }
}

// One warp per coarse cell, its max and its min; lane l takes children l,
// l + 32, ... of 512.
__global__ void __launch_bounds__(256) reduce_level_kernel(const float* __restrict__ pmax, const float* __restrict__ pmin,
                                                           int px, int py, int pz, float* __restrict__ omax,
                                                           float* __restrict__ omin, int cx, int cy, int cz)
{
    const long long cell = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (cell >= (long long)cx * cy * cz) return;
    const int ix = (int)(cell % cx);
    const int iy = (int)((cell / cx) % cy);
    const int iz = (int)(cell / ((long long)cx * cy));
    float m = 0.0f, mn = __int_as_float(0x7f800000);
#pragma unroll 4
    for (int c = lane; c < 512; c += 32) {
        const int x = ix * 8 + (c & 7), y = iy * 8 + ((c >> 3) & 7), z = iz * 8 + (c >> 6);
        if (x < px && y < py && z < pz) {
            const size_t j = ((size_t)z * py + y) * (size_t)px + x;
            m = fmaxf(m, pmax[j]);
            mn = fminf(mn, pmin[j]);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
    }
    if (lane == 0) {
        omax[cell] = m;
        omin[cell] = mn;
    }
}

// Octree levels 1 to 3 as oct_bricks_kernel writes them.
struct LevelOut {
    float* mx[4];
    float* mn[4];
    int dims[4][3];
};

struct LevelTable {
    const float* p[kMaxGridLevels + 1];
    const float* pmin[kMaxGridLevels + 1];
    int dims[kMaxGridLevels + 1][3];
    float hz[kMaxGridLevels + 1];
};

// Leaf of each level-1 cell of the pyramid: search from the top level down to
// finest + 1.  A level-L cell spans 2^(3 L) voxels per axis, which is the
// shift the entry records.
__global__ void __launch_bounds__(256) leafmap_kernel(LevelTable T, int levels, int finest, float tau,
                                                      int n1x, int n1y, int n1z, uint2* __restrict__ leaf)
{
    constexpr int lb = 3;
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (long long)n1x * n1y * n1z) return;
    const int cx = (int)(i % n1x), cy = (int)((i / n1x) % n1y), cz = (int)(i / ((long long)n1x * n1y));
    for (int L = levels; L > finest; --L) {
        const int s = lb * (L - 1);
        const int ax = cx >> s, ay = cy >> s, az = cz >> s;
        const size_t c = ((size_t)az * T.dims[L][1] + ay) * T.dims[L][0] + ax;
        const float M = T.p[L][c];
        if (__fmul_rn(M, T.hz[L]) <= tau) {
            // .y: the minorant rounded down to bfloat16 (high half) | the shift
            leaf[i] = make_uint2(__float_as_uint(M),
                                 (__float_as_uint(T.pmin[L][c]) & 0xFFFF0000u) | (unsigned)(lb * L));
            return;
        }
    }
    if (finest == 0) {
        // voxel leaves: the majorant is the voxel itself, so the entry names the cell's brick
        leaf[i] = make_uint2((uint32_t)i, 0u);
    } else {
        const int s = lb * (finest - 1);
        const size_t c = ((size_t)(cz >> s) * T.dims[finest][1] + (cy >> s)) * T.dims[finest][0] + (cx >> s);
        const float M = T.p[finest][c];
        leaf[i] = make_uint2(__float_as_uint(M),
                             (__float_as_uint(T.pmin[finest][c]) & 0xFFFF0000u) | (unsigned)(lb * finest));
    }
}

// Octree levels 1 to 3 of one brick: max and min of each group of 2^3, 4^3
// and 8^3 voxels (the stored values: FP32, or the nearest-bfloat16 voxels of
// a BF16 field, whose max bounds exactly what the tracer reads).  One warp
// per brick: lane (z2, y2, xh) reads the 16 voxels of two level-1 cells next
// to each other in x, four rows of four, and the coarser levels are shuffles.
// Bound by HBM: the field read once, 1/7 of it written twice, 863 MB in 157 us
// (5.5 TB/s) for the 1024 x 1024 x 160 field.
template <bool BF16>
__global__ void __launch_bounds__(256) oct_bricks_kernel(const void* __restrict__ vox, int nx, int ny, int nz, int nbx,
                                                         int nby, unsigned nbricks, int levels, LevelOut O)
{
    const unsigned b = blockIdx.x * 8u + (threadIdx.x >> 5);
    if (b >= nbricks) return;
    const int lane = threadIdx.x & 31, xh = lane & 1, y2 = (lane >> 1) & 3, z2 = lane >> 3;
    const int bx = (int)(b % (unsigned)nbx), by = (int)((b / (unsigned)nbx) % (unsigned)nby),
              bz = (int)(b / ((unsigned)nbx * (unsigned)nby));
    const int x0 = bx * 8 + 4 * xh, y0 = by * 8 + 2 * y2, z0 = bz * 8 + 2 * z2;
    const float kInf = __int_as_float(0x7f800000);
    float m[2] = {0.0f, 0.0f}, mn[2] = {kInf, kInf};
    float v[4][4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const size_t off = (size_t)b * 512u + (unsigned)(((2 * z2 + (r >> 1)) * 8 + 2 * y2 + (r & 1)) * 8 + 4 * xh);
        if (BF16) {
            const uint2 w = __ldg(reinterpret_cast<const uint2*>(static_cast<const uint16_t*>(vox) + off));
            v[r][0] = __uint_as_float(w.x << 16); v[r][1] = __uint_as_float(w.x & 0xFFFF0000u);
            v[r][2] = __uint_as_float(w.y << 16); v[r][3] = __uint_as_float(w.y & 0xFFFF0000u);
        } else {
            const float4 w = __ldg(reinterpret_cast<const float4*>(static_cast<const float*>(vox) + off));
            v[r][0] = w.x; v[r][1] = w.y; v[r][2] = w.z; v[r][3] = w.w;
        }
    }
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (x0 + i < nx && y0 + (r & 1) < ny && z0 + (r >> 1) < nz) {
                m[i >> 1] = fmaxf(m[i >> 1], v[r][i]);
                mn[i >> 1] = fminf(mn[i >> 1], v[r][i]);
            }
    {
        const int cx = bx * 4 + 2 * xh, cy = by * 4 + y2, cz = bz * 4 + z2;
        const int* d = O.dims[1];
        if (cx < d[0] && cy < d[1] && cz < d[2]) {
            const size_t c = ((size_t)cz * d[1] + cy) * d[0] + cx;
            if ((d[0] & 1) == 0) {
                *reinterpret_cast<float2*>(O.mx[1] + c) = make_float2(m[0], m[1]);
                *reinterpret_cast<float2*>(O.mn[1] + c) = make_float2(mn[0], mn[1]);
            } else {
                O.mx[1][c] = m[0];
                O.mn[1][c] = mn[0];
                if (cx + 1 < d[0]) {
                    O.mx[1][c + 1] = m[1];
                    O.mn[1][c + 1] = mn[1];
                }
            }
        }
    }
    if (levels < 2) return;
    float M = fmaxf(m[0], m[1]), N = fminf(mn[0], mn[1]);
    for (int o : {2, 8}) {
        M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
        N = fminf(N, __shfl_xor_sync(0xffffffffu, N, o));
    }
    {
        const int cx = bx * 2 + xh, cy = by * 2 + (y2 >> 1), cz = bz * 2 + (z2 >> 1);
        const int* d = O.dims[2];
        if (!(y2 & 1) && !(z2 & 1) && cx < d[0] && cy < d[1] && cz < d[2]) {
            const size_t c = ((size_t)cz * d[1] + cy) * d[0] + cx;
            O.mx[2][c] = M;
            O.mn[2][c] = N;
        }
    }
    if (levels < 3) return;
    for (int o : {1, 4, 16}) {
        M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
        N = fminf(N, __shfl_xor_sync(0xffffffffu, N, o));
    }
    if (lane == 0) {
        O.mx[3][b] = M;
        O.mn[3][b] = N;
    }
}

// Leaf map of the octree, 32 bricks per block.  The levels from 8^3 voxels up
// are the same for a whole brick: each warp looks at its levels for the 32
// bricks (lane = brick, reads next to each other), then expands four of them,
// and only where no coarse level qualifies do the lanes (as in
// oct_bricks_kernel) look at their own 4^3 and 2^3 cells.  Bound by the 8
// bytes written per 2^3 voxels, 16 per lane.  For the 1024 x 1024 x 160 field:
// one thread per cell walking down from the top level 162 us, one warp per
// brick with a lane per level 104 us, this 52 us.  finest: 0 (voxel leaves)
// or 1.
__global__ void __launch_bounds__(256) oct_leafmap_kernel(LevelTable T, int levels, int finest, float tau, int nbx,
                                                          int nby, unsigned nbricks, uint2* __restrict__ leaf)
{
    __shared__ int coarse[32];
    __shared__ uint2 coarse_e[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned b0 = blockIdx.x * 32u;
    auto brick = [&](unsigned b, int& bx, int& by, int& bz) {
        bx = (int)(b % (unsigned)nbx);
        by = (int)((b / (unsigned)nbx) % (unsigned)nby);
        bz = (int)(b / ((unsigned)nbx * (unsigned)nby));
    };
    // .y: the minorant rounded down to bfloat16 (high half) | the shift
    auto entry = [](float M, float mn, int L) {
        return make_uint2(__float_as_uint(M), (__float_as_uint(mn) & 0xFFFF0000u) | (unsigned)L);
    };
    if (warp == 0) coarse[lane] = 0;
    __syncthreads();
    {
        int bx, by, bz;
        const bool have = b0 + lane < nbricks;
        brick(have ? b0 + lane : 0u, bx, by, bz);
        int best = 0;
        uint2 e = make_uint2(0u, 0u);
        for (int L = 3 + warp; L <= levels; L += 8) {
            const int s = L - 3;
            const size_t c = ((size_t)(bz >> s) * T.dims[L][1] + (by >> s)) * T.dims[L][0] + (bx >> s);
            const float M = T.p[L][c], mn = T.pmin[L][c];
            if (have && __fmul_rn(M, T.hz[L]) <= tau) {
                best = L;
                e = entry(M, mn, L);
            }
        }
        if (best) atomicMax(&coarse[lane], best);
        __syncthreads();
        if (best && coarse[lane] == best) coarse_e[lane] = e;
        __syncthreads();
    }
    const int xh = lane & 1, y2 = (lane >> 1) & 3, z2 = lane >> 3;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const unsigned b = b0 + 4u * warp + q;
        if (b >= nbricks) return;
        int bx, by, bz;
        brick(b, bx, by, bz);
        const int cx = bx * 4 + 2 * xh, cy = by * 4 + y2, cz = bz * 4 + z2;
        if (cx >= T.dims[1][0] || cy >= T.dims[1][1] || cz >= T.dims[1][2]) continue;
        const size_t c1 = ((size_t)cz * T.dims[1][1] + cy) * T.dims[1][0] + cx;
        uint2 e[2];
        bool done = coarse[4 * warp + q] != 0;
        if (done) {
            e[0] = e[1] = coarse_e[4 * warp + q];
        } else if (levels >= 2) {
            const size_t c = ((size_t)(cz >> 1) * T.dims[2][1] + (cy >> 1)) * T.dims[2][0] + (cx >> 1);
            const float M = T.p[2][c];
            if (__fmul_rn(M, T.hz[2]) <= tau) {
                e[0] = e[1] = entry(M, T.pmin[2][c], 2);
                done = true;
            }
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            if (done || cx + i >= T.dims[1][0]) continue;
            const float M = T.p[1][c1 + i];
            if (finest == 1 || __fmul_rn(M, T.hz[1]) <= tau) e[i] = entry(M, T.pmin[1][c1 + i], 1);
            else e[i] = make_uint2(b, 0u);     // voxel leaves: the entry names the brick
        }
        if ((T.dims[1][0] & 1) == 0) {
            *reinterpret_cast<uint4*>(leaf + c1) = make_uint4(e[0].x, e[0].y, e[1].x, e[1].y);
        } else {
            leaf[c1] = e[0];
            if (cx + 1 < T.dims[1][0]) leaf[c1 + 1] = e[1];
        }
    }
}

// Octree level L >= 4: max and min over the (up to) 2^3 children.
__global__ void __launch_bounds__(256) oct_reduce2_kernel(const float* __restrict__ pmax, const float* __restrict__ pmin,
                                                          int px, int py, int pz, float* __restrict__ omax,
                                                          float* __restrict__ omin, int dx, int dy, int dz)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (long long)dx * dy * dz) return;
    const int cx = (int)(i % dx), cy = (int)((i / dx) % dy), cz = (int)(i / ((long long)dx * dy));
    float m = 0.0f, mn = __int_as_float(0x7f800000);
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const int x = 2 * cx + (c & 1), y = 2 * cy + ((c >> 1) & 1), z = 2 * cz + (c >> 2);
        if (x < px && y < py && z < pz) {
            const size_t j = ((size_t)z * py + y) * (size_t)px + x;
            m = fmaxf(m, pmax[j]);
            mn = fminf(mn, pmin[j]);
        }
    }
    omax[i] = m;
    omin[i] = mn;
}

}  // namespace

cudaError_t launch_relayout(const float* src, const mcrt_scene* sc, cudaStream_t st)
{
    dim3 grid((sc->nb[0] + 3) / 4, sc->nb[1], sc->nb[2]);
    float* l1 = sc->d_pyr + sc->lev_off[1];
    float* l1min = sc->d_pyr + sc->pyr_capacity + sc->lev_off[1];
    if (sc->storage == MCRT_STORAGE_BF16)
        relayout_l1_kernel<true><<<grid, 256, 0, st>>>(src, sc->n[0], sc->n[1], sc->n[2], sc->nb[0], sc->nb[1],
                                                       sc->d_vox, l1, l1min);
    else
        relayout_l1_kernel<false><<<grid, 256, 0, st>>>(src, sc->n[0], sc->n[1], sc->n[2], sc->nb[0], sc->nb[1],
                                                        sc->d_vox, l1, l1min);
    return cudaGetLastError();
}

cudaError_t launch_reduce_level(const float* pmax, const float* pmin, const int* pd, float* omax, float* omin,
                                const int* d, cudaStream_t st)
{
    const long long cells = (long long)d[0] * d[1] * d[2];
    const int warps = 8;
    const long long blocks = (cells + warps - 1) / warps;
    reduce_level_kernel<<<(unsigned)blocks, 32 * warps, 0, st>>>(pmax, pmin, pd[0], pd[1], pd[2], omax, omin, d[0], d[1],
                                                                d[2]);
    return cudaGetLastError();
}

cudaError_t launch_leafmap(const mcrt_scene* sc, float tau, int finest, int grid, cudaStream_t st)
{
    LevelTable T{};
    const bool oct = grid == MCRT_GRID_OCTREE;
    const int levels = oct ? sc->oct_levels : sc->levels;
    const int lb = oct ? 1 : 3;
    if (levels < 1 || levels > kMaxGridLevels) return cudaErrorInvalidValue;
    for (int L = 1; L <= levels; ++L) {
        if (oct) {
            T.p[L] = sc->d_oct + sc->oct_off[L];
            T.pmin[L] = sc->d_oct + sc->oct_capacity + sc->oct_off[L];
            for (int a = 0; a < 3; ++a) T.dims[L][a] = sc->oct_dims[3 * L + a];
        } else {
            T.p[L] = sc->d_pyr + sc->lev_off[L];
            T.pmin[L] = sc->d_pyr + sc->pyr_capacity + sc->lev_off[L];
            for (int a = 0; a < 3; ++a) T.dims[L][a] = sc->lev_dims[3 * L + a];
        }
        T.hz[L] = sc->h[2] * (float)(1 << (lb * L));
    }
    const long long cells = (long long)sc->nb[0] * sc->nb[1] * sc->nb[2];
    if (oct) {
        oct_leafmap_kernel<<<(unsigned)((cells + 31) / 32), 256, 0, st>>>(T, levels, finest, tau, sc->nb[0], sc->nb[1],
                                                                        (unsigned)cells, sc->d_oleaf);
    } else {
        leafmap_kernel<<<(unsigned)((cells + 255) / 256), 256, 0, st>>>(T, levels, finest, tau, sc->nb[0], sc->nb[1],
                                                                        sc->nb[2], sc->d_leaf);
    }
    return cudaGetLastError();
}

cudaError_t launch_octree(const mcrt_scene* sc, cudaStream_t st)
{
    float* mx = sc->d_oct;
    float* mn = sc->d_oct + sc->oct_capacity;
    LevelOut O{};
    for (int L = 1; L <= 3 && L <= sc->oct_levels; ++L) {
        O.mx[L] = mx + sc->oct_off[L];
        O.mn[L] = mn + sc->oct_off[L];
        for (int a = 0; a < 3; ++a) O.dims[L][a] = sc->oct_dims[3 * L + a];
    }
    const unsigned nbricks = (unsigned)((size_t)sc->nb[0] * sc->nb[1] * sc->nb[2]);
    if (sc->storage == MCRT_STORAGE_BF16)
        oct_bricks_kernel<true><<<(nbricks + 7) / 8, 256, 0, st>>>(sc->d_vox, sc->n[0], sc->n[1], sc->n[2], sc->nb[0],
                                                                   sc->nb[1], nbricks, sc->oct_levels, O);
    else
        oct_bricks_kernel<false><<<(nbricks + 7) / 8, 256, 0, st>>>(sc->d_vox, sc->n[0], sc->n[1], sc->n[2], sc->nb[0],
                                                                    sc->nb[1], nbricks, sc->oct_levels, O);
    for (int L = 4; L <= sc->oct_levels; ++L) {
        const int* pd = &sc->oct_dims[3 * (L - 1)];
        const int* d = &sc->oct_dims[3 * L];
        const long long n = (long long)d[0] * d[1] * d[2];
        oct_reduce2_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(
            mx + sc->oct_off[L - 1], mn + sc->oct_off[L - 1], pd[0], pd[1], pd[2], mx + sc->oct_off[L],
            mn + sc->oct_off[L], d[0], d[1], d[2]);
    }
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Heightfield ground: max pyramid.  Level 0 holds each cell's maximum over
// its 4 corner heights (periodic), which are kept as one record per cell
// where the grid is not too large for that, level L the maximum over 4 x 4 cells of level L - 1.  Also a scan for
// invalid heights (not finite, < 0 or above the top of the field).
// ---------------------------------------------------------------------------
namespace {

// A block of 32 x 8 cells: each thread writes its cell's record (cells null:
// none, the plain heights are kept), and either
// the cell's maximum (level 0 is the only level) or, with a 4 x 4 group, the
// maximum of level 1.  (Level 0 of a taller pyramid is never read: the walk
// takes a cell's maximum from its corners.)
__global__ void __launch_bounds__(256) hf_cells_kernel(const float* __restrict__ h, int nx, int ny,
                                                       float4* __restrict__ cells, float* __restrict__ lev0,
                                                       float* __restrict__ lev1)
{
    __shared__ float rows[8][8];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const long long nbx = (nx + 31) / 32;
    const int i = (int)(blockIdx.x % nbx) * 32 + tx, j = (int)(blockIdx.x / nbx) * 8 + ty;
    const bool in = i < nx && j < ny;
    float m = 0.0f;
    if (in) {
        const int i1 = i + 1 == nx ? 0 : i + 1, j1 = j + 1 == ny ? 0 : j + 1;
        const float4 c = make_float4(h[(size_t)j * nx + i], h[(size_t)j * nx + i1], h[(size_t)j1 * nx + i],
                                     h[(size_t)j1 * nx + i1]);
        if (cells) cells[(size_t)j * nx + i] = c;
        m = fmaxf(fmaxf(c.x, c.y), fmaxf(c.z, c.w));
        if (lev0) lev0[(size_t)j * nx + i] = m;
    }
    if (!lev1) return;
    // (nx and ny are multiples of 4: a group is inside or outside as a whole)
    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 1));
    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 2));
    if ((tx & 3) == 0) rows[ty][tx >> 2] = m;
    __syncthreads();
    if (in && (tx & 3) == 0 && (ty & 3) == 0)
        lev1[(size_t)(j >> 2) * (nx >> 2) + (i >> 2)] = fmaxf(fmaxf(rows[ty][tx >> 2], rows[ty + 1][tx >> 2]),
                                                              fmaxf(rows[ty + 2][tx >> 2], rows[ty + 3][tx >> 2]));
}

__global__ void hf_reduce4_kernel(const float* __restrict__ in, int nx, int ny, float* __restrict__ out)
{
    // out is (nx / 4) x (ny / 4)
    const int ox = nx >> 2, oy = ny >> 2;
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (long long)ox * oy) return;
    const int i = (int)(idx % ox), j = (int)(idx / ox);
    float m = in[(size_t)(4 * j) * nx + 4 * i];
    for (int b = 0; b < 4; ++b)
        for (int a = 0; a < 4; ++a) m = fmaxf(m, in[(size_t)(4 * j + b) * nx + 4 * i + a]);
    out[idx] = m;
}

__global__ void hf_check_kernel(const float* __restrict__ h, long long n, float top, int* __restrict__ bad)
{
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= n) return;
    const float v = h[idx];
    if (!(v >= 0.0f && v <= top)) atomicOr(bad, 1);
}

}  // namespace

cudaError_t launch_hf_pyramid(const float* h, int nx, int ny, float4* cells, float* pyr, const int* off, int levels,
                              cudaStream_t st)
{
    const long long blocks = (long long)((nx + 31) / 32) * ((ny + 7) / 8);
    hf_cells_kernel<<<(unsigned)blocks, 256, 0, st>>>(h, nx, ny, cells, levels == 1 ? pyr + off[0] : nullptr,
                                                      levels > 1 ? pyr + off[1] : nullptr);
    for (int L = 2; L < levels; ++L) {
        const int px = nx >> (2 * (L - 1)), py = ny >> (2 * (L - 1));
        const long long n = (long long)(px >> 2) * (py >> 2);
        hf_reduce4_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(pyr + off[L - 1], px, py, pyr + off[L]);
    }
    return cudaGetLastError();
}

cudaError_t launch_hf_check(const float* h, long long n, float top, int* bad, cudaStream_t st)
{
    hf_check_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(h, n, top, bad);
    return cudaGetLastError();
}

}  // namespace mcrt
