// Linear BVH over the particles' smoothing spheres.
//
// The paper does not describe its search structure; this is a Morton-code
// LBVH: 30-bit Morton codes of the sphere centres, stable radix sort, the
// binary radix tree of Karras (2012, "Maximizing parallelism in the
// construction of BVHs, octrees and k-d trees").  The radix tree only orders
// the particles (k_leaf_order); the traversal reads an implicit 32-ary tree of
// boxes over the ordered particles, 32 to a block (one lane tests one sphere
// or one child).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <new>

#include "common.cuh"

namespace urchin {

namespace {

__device__ __forceinline__ unsigned f2ord(float f)
{
    unsigned u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__host__ __device__ __forceinline__ float ord2f(unsigned u)
{
#ifdef __CUDA_ARCH__
    return __uint_as_float((u & 0x80000000u) ? (u & 0x7fffffffu) : ~u);
#else
    unsigned v = (u & 0x80000000u) ? (u & 0x7fffffffu) : ~u;
    float f;
    memcpy(&f, &v, 4);
    return f;
#endif
}

// bounds[0..2] min centre, [3..5] max centre, [6] max h (ordered encoding);
// bounds[7] error bits: 1 = non-finite, 2 = h <= 0 or mass < 0
// logh_sum accumulates sum ln h (the geometric mean of h sets the shape of
// the traversal's ray packets)
__global__ void k_bounds(const float* __restrict__ x, const float* __restrict__ y,
                         const float* __restrict__ z, const float* __restrict__ h,
                         const double* __restrict__ m, int64_t n, unsigned* bounds, double* logh_sum)
{
    unsigned mn[3] = {0xffffffffu, 0xffffffffu, 0xffffffffu};
    unsigned mx[4] = {0u, 0u, 0u, 0u};
    unsigned err = 0;
    double lsum = 0.0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        float c[3] = {x[i], y[i], z[i]};
        float hi = h[i];
        double mi = m[i];
        bool fin = isfinite(c[0]) && isfinite(c[1]) && isfinite(c[2]) && isfinite(hi) && isfinite(mi);
        if (!fin) { err |= 1u; continue; }
        if (!(hi > 0.f) || mi < 0.0) err |= 2u;
        else lsum += (double)logf(hi);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            unsigned o = f2ord(c[a]);
            mn[a] = min(mn[a], o);
            mx[a] = max(mx[a], o);
        }
        mx[3] = max(mx[3], f2ord(hi));
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            mn[a] = min(mn[a], __shfl_xor_sync(0xffffffffu, mn[a], off));
            mx[a] = max(mx[a], __shfl_xor_sync(0xffffffffu, mx[a], off));
        }
        mx[3] = max(mx[3], __shfl_xor_sync(0xffffffffu, mx[3], off));
        err |= __shfl_xor_sync(0xffffffffu, err, off);
        lsum += __shfl_xor_sync(0xffffffffu, lsum, off);
    }
    if ((threadIdx.x & 31) == 0) {
        for (int a = 0; a < 3; ++a) {
            atomicMin(&bounds[a], mn[a]);
            atomicMax(&bounds[3 + a], mx[a]);
        }
        atomicMax(&bounds[6], mx[3]);
        if (err) atomicOr(&bounds[7], err);
        atomicAdd(logh_sum, lsum);
    }
}

__device__ __forceinline__ unsigned spread10(unsigned v)
{
    v = (v * 0x00010001u) & 0xFF0000FFu;
    v = (v * 0x00000101u) & 0x0F00F00Fu;
    v = (v * 0x00000011u) & 0xC30C30C3u;
    v = (v * 0x00000005u) & 0x49249249u;
    return v;
}

__global__ void k_morton(const float* __restrict__ x, const float* __restrict__ y,
                         const float* __restrict__ z, int64_t n, const unsigned* bounds,
                         uint32_t* codes, int32_t* idx)
{
    float lo[3], inv[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        lo[a] = ord2f(bounds[a]);
        float ext = ord2f(bounds[3 + a]) - lo[a];
        inv[a] = ext > 0.f ? 1.0f / ext : 0.f;
    }
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        float c[3] = {x[i], y[i], z[i]};
        unsigned q[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            float u = (c[a] - lo[a]) * inv[a];
            u = fminf(fmaxf(u * 1024.f, 0.f), 1023.f);
            q[a] = (unsigned)u;
        }
        codes[i] = (spread10(q[0]) << 2) | (spread10(q[1]) << 1) | spread10(q[2]);
        idx[i] = (int32_t)i;
    }
}

__global__ void k_gather(const float* __restrict__ x, const float* __restrict__ y,
                         const float* __restrict__ z, const float* __restrict__ h,
                         const double* __restrict__ m, const int32_t* __restrict__ order, int64_t n,
                         double mass_to_A, double unit_cm, float4* xyzh, float* A32, double* A64,
                         int32_t* perm, int32_t* inv, unsigned* err)
{
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < n;
         s += (int64_t)gridDim.x * blockDim.x) {
        int32_t i = order[s];
        if (i < 0 || i >= n) {     // a permutation from the sort; never true
            atomicOr(err, 8u);
            continue;
        }
        float hi = h[i];
        xyzh[s] = make_float4(x[i], y[i], z[i], hi);
        double hcm = (double)hi * unit_cm;
        // A_j = sigma_th (m_j/m_p) (8/pi) / h_j^2: threshold optical depth per
        // unit dimensionless chord integral of a fully neutral particle
        double A = mass_to_A * m[i] / (hcm * hcm);
        A64[s] = A;
        A32[s] = (float)A;
        perm[s] = i;
        inv[i] = (int32_t)s;
    }
}

__device__ __forceinline__ int delta(const uint32_t* __restrict__ codes, int n, int i, int j)
{
    if (j < 0 || j >= n) return -1;
    uint32_t a = codes[i], b = codes[j];
    if (a != b) return __clz(a ^ b);
    return 32 + __clz((unsigned)i ^ (unsigned)j);
}

// Karras (2012) binary radix tree: internal node i covers a Morton range and
// splits it at the highest differing bit.  Children are encoded >= 0 for an
// internal node, ~leaf for a leaf (particle).
__global__ void k_karras(const uint32_t* __restrict__ codes, int n, int32_t* child_l, int32_t* child_r,
                         int32_t* first, int32_t* last, int32_t* parent_int)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n - 1) return;
    int d = (delta(codes, n, i, i + 1) - delta(codes, n, i, i - 1)) >= 0 ? 1 : -1;
    int dmin = delta(codes, n, i, i - d);
    int lmax = 2;
    while (delta(codes, n, i, i + lmax * d) > dmin) lmax <<= 1;
    int l = 0;
    for (int t = lmax >> 1; t >= 1; t >>= 1)
        if (delta(codes, n, i, i + (l + t) * d) > dmin) l += t;
    int j = i + l * d;
    int dnode = delta(codes, n, i, j);
    int s = 0;
    for (int div = 2;; div <<= 1) {
        int t = (l + div - 1) / div;
        if (delta(codes, n, i, i + (s + t) * d) > dnode) s += t;
        if (t <= 1) break;
    }
    int g = i + s * d + min(d, 0);
    int lo = min(i, j), hi = max(i, j);
    first[i] = lo;
    last[i] = hi;
    if (lo == g) child_l[i] = ~g;
    else { child_l[i] = g; parent_int[g] = i; }
    if (hi == g + 1) child_r[i] = ~(g + 1);
    else { child_r[i] = g + 1; parent_int[g + 1] = i; }
    if (i == 0) parent_int[0] = -1;
}

// Conservative sphere bounds: rounded outward and padded by 1e-6 of the
// coordinate scale so float slab tests never cull a sphere a ray crosses.
__device__ __forceinline__ void sphere_box(float4 p, float lo[3], float hi[3])
{
    float pad = 1e-6f * (fmaxf(fmaxf(fabsf(p.x), fabsf(p.y)), fabsf(p.z)) + p.w);
    lo[0] = __fsub_rd(__fsub_rd(p.x, p.w), pad);
    lo[1] = __fsub_rd(__fsub_rd(p.y, p.w), pad);
    lo[2] = __fsub_rd(__fsub_rd(p.z, p.w), pad);
    hi[0] = __fadd_ru(__fadd_ru(p.x, p.w), pad);
    hi[1] = __fadd_ru(__fadd_ru(p.y, p.w), pad);
    hi[2] = __fadd_ru(__fadd_ru(p.z, p.w), pad);
}

// Particles of child c of an inner node (c < 0: the single particle ~c).
__device__ __forceinline__ int child_size(int32_t c, const int32_t* __restrict__ first,
                                          const int32_t* __restrict__ last)
{
    return c < 0 ? 1 : last[c] - first[c] + 1;
}

// order[s] = the particle of slot s (and mslot, the slots in Morton order): the subtrees of at most kLeafMax
// particles ("leaves": the children of at most kLeafMax particles of the root
// and of every larger inner node) in the order of a depth-first walk that
// takes a node's leaf children before its inner ones, left before right, a
// leaf's particles in Morton order.  A leaf's first slot is the sum, over its
// ancestors, of the particles that precede it below each.
__global__ void k_leaf_order(int n, const int32_t* __restrict__ child_l, const int32_t* __restrict__ child_r,
                             const int32_t* __restrict__ first, const int32_t* __restrict__ last,
                             const int32_t* __restrict__ parent_int, const int32_t* __restrict__ idx, int32_t* order,
                             int32_t* mslot, unsigned* err)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n - 1 || (i > 0 && last[i] - first[i] + 1 <= kLeafMax)) return;
    const int32_t cl = child_l[i], cr = child_r[i];
    const int nl = child_size(cl, first, last), nr = child_size(cr, first, last);
    if (nl > kLeafMax && nr > kLeafMax) return;
    int at = 0, c = i;
    int p = i > 0 ? parent_int[i] : -1;
    // the tree is at most 62 levels deep; the cap only guards against a
    // malformed parent chain
    for (int level = 0; p >= 0; ++level) {
        if (level > 128) {
            atomicOr(err, 4u);
            return;
        }
        const int32_t pl = child_l[p], pr = child_r[p];
        if (c == pr) {
            at += child_size(pl, first, last);
        } else {
            const int m = child_size(pr, first, last);
            if (m <= kLeafMax) at += m;
        }
        c = p;
        p = p > 0 ? parent_int[p] : -1;
    }
    const int f = first[i];
    if (at < 0 || at + (nl <= kLeafMax ? nl : 0) + (nr <= kLeafMax ? nr : 0) > n) {   // never true for a well-formed tree
        atomicOr(err, 4u);
        return;
    }
    if (nl <= kLeafMax)
        for (int q = 0; q < nl; ++q, ++at) {
            order[at] = idx[f + q];
            mslot[f + q] = at;
        }
    if (nr <= kLeafMax)
        for (int q = nl; q < nl + nr; ++q, ++at) {
            order[at] = idx[f + q];
            mslot[f + q] = at;
        }
}

// Level 0 of the 32-ary tree: a warp bounds the spheres of 32 slots.
__global__ void k_blocks(const float4* __restrict__ xyzh, int n, float4* out, int n_out)
{
    const int g = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5);
    const int lane = threadIdx.x & 31;
    if (g >= n_out) return;
    float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
    if (32 * g + lane < n) sphere_box(xyzh[32 * g + lane], lo, hi);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            lo[a] = fminf(lo[a], __shfl_xor_sync(0xffffffffu, lo[a], o));
            hi[a] = fmaxf(hi[a], __shfl_xor_sync(0xffffffffu, hi[a], o));
        }
    if (lane == 0) {
        out[2 * (int64_t)g] = make_float4(lo[0], lo[1], lo[2], 0.f);
        out[2 * (int64_t)g + 1] = make_float4(hi[0], hi[1], hi[2], 0.f);
    }
}

// One level of the 32-ary tree: a warp bounds 32 entries of the level below.
__global__ void k_level(const float4* __restrict__ in, int n_in, float4* out, int n_out)
{
    const int g = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5);
    const int lane = threadIdx.x & 31;
    if (g >= n_out) return;
    const int e = 32 * g + lane;
    float4 lo = make_float4(INFINITY, INFINITY, INFINITY, 0.f), hi = make_float4(-INFINITY, -INFINITY, -INFINITY, 0.f);
    if (e < n_in) {
        lo = in[2 * (int64_t)e];
        hi = in[2 * (int64_t)e + 1];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        lo.x = fminf(lo.x, __shfl_xor_sync(0xffffffffu, lo.x, o));
        lo.y = fminf(lo.y, __shfl_xor_sync(0xffffffffu, lo.y, o));
        lo.z = fminf(lo.z, __shfl_xor_sync(0xffffffffu, lo.z, o));
        hi.x = fmaxf(hi.x, __shfl_xor_sync(0xffffffffu, hi.x, o));
        hi.y = fmaxf(hi.y, __shfl_xor_sync(0xffffffffu, hi.y, o));
        hi.z = fmaxf(hi.z, __shfl_xor_sync(0xffffffffu, hi.z, o));
    }
    if (lane == 0) {
        lo.w = hi.w = 0.f;
        out[2 * (int64_t)g] = lo;
        out[2 * (int64_t)g + 1] = hi;
    }
}

void free_bvh_arrays(urchin_bvh* b)
{
    if (!b) return;
    cudaFree(b->boxes);
    cudaFree(b->xyzh);
    cudaFree(b->A32);
    cudaFree(b->A64);
    cudaFree(b->perm);
    cudaFree(b->inv);
    cudaFree(b->mslot);
    cudaFree(b->ktab);
    b->ktab = nullptr;
    b->boxes = nullptr;
    b->xyzh = nullptr;
    b->A32 = nullptr;
    b->A64 = nullptr;
    b->perm = nullptr;
    b->inv = nullptr;
    b->mslot = nullptr;
}

int build(const urchin_particles* p, const urchin_box* box, urchin_bvh* b, cudaStream_t s)
{
    const int64_t n = p->n;
    b->n = n;
    b->periodic = box->periodic ? 1 : 0;
    b->L = box->L;
    b->unit_cm = box->unit_cm;
    URCHIN_TRY_CUDA(cudaGetDevice(&b->device));
    URCHIN_TRY_CUDA(cudaMalloc(&b->xyzh, sizeof(float4) * (size_t)n));
    URCHIN_TRY_CUDA(cudaMalloc(&b->A32, sizeof(float) * (size_t)n));
    URCHIN_TRY_CUDA(cudaMalloc(&b->A64, sizeof(double) * (size_t)n));
    URCHIN_TRY_CUDA(cudaMalloc(&b->perm, sizeof(int32_t) * (size_t)n));
    URCHIN_TRY_CUDA(cudaMalloc(&b->inv, sizeof(int32_t) * (size_t)n));
    URCHIN_TRY_CUDA(cudaMalloc(&b->mslot, sizeof(int32_t) * (size_t)n));
    URCHIN_TRY_CUDA(cudaMalloc(&b->ktab, sizeof(float2) * (kKTab + 1)));
    {
        static float2 table[kKTab + 1];
        static bool ready = false;
        static std::mutex mu;
        std::lock_guard<std::mutex> lock(mu);
        if (!ready) {
            m4_full_table(table);
            ready = true;
        }
        URCHIN_TRY_CUDA(cudaMemcpyAsync(b->ktab, table, sizeof(table), cudaMemcpyHostToDevice, s));
        URCHIN_TRY_CUDA(cudaStreamSynchronize(s));
    }

    const int64_t ni = std::max<int64_t>(1, n - 1);
    Layout lay;
    size_t o_bounds = lay.take(8 * sizeof(unsigned));
    size_t o_logh = lay.take(sizeof(double));
    size_t o_codes = lay.take((size_t)n * 4);
    size_t o_idx = lay.take((size_t)n * 4);
    size_t o_radix = lay.take(radix_tmp_bytes(n));
    size_t o_cl = lay.take((size_t)ni * 4);
    size_t o_cr = lay.take((size_t)ni * 4);
    size_t o_first = lay.take((size_t)ni * 4);
    size_t o_last = lay.take((size_t)ni * 4);
    size_t o_pint = lay.take((size_t)ni * 4);
    size_t o_order = lay.take((size_t)n * 4);
    Scratch scr;
    URCHIN_TRY(scr.alloc(lay.bytes, s));
    unsigned* bounds = scr.at<unsigned>(o_bounds);
    uint32_t* codes = scr.at<uint32_t>(o_codes);
    int32_t* idx = scr.at<int32_t>(o_idx);

    unsigned init[8] = {0xffffffffu, 0xffffffffu, 0xffffffffu, 0u, 0u, 0u, 0u, 0u};
    URCHIN_TRY_CUDA(cudaMemcpyAsync(bounds, init, sizeof(init), cudaMemcpyHostToDevice, s));
    double* logh = scr.at<double>(o_logh);
    URCHIN_TRY_CUDA(cudaMemsetAsync(logh, 0, sizeof(double), s));
    unsigned grid = (unsigned)std::min<int64_t>((n + 255) / 256, 2048);
    k_bounds<<<grid, 256, 0, s>>>(p->pos_x, p->pos_y, p->pos_z, p->h, p->mass_H, n, bounds, logh);
    URCHIN_TRY(launched());
    unsigned hb[8];
    double lh = 0.0;
    URCHIN_TRY_CUDA(cudaMemcpyAsync(hb, bounds, sizeof(hb), cudaMemcpyDeviceToHost, s));
    URCHIN_TRY_CUDA(cudaMemcpyAsync(&lh, logh, sizeof(double), cudaMemcpyDeviceToHost, s));
    URCHIN_TRY_CUDA(cudaStreamSynchronize(s));
    b->hgeo = (float)std::exp(lh / (double)n);
    if (hb[7] & 1u) return set_error(URCHIN_ERR_NONFINITE, "urchin_build_bvh: NaN/Inf in positions, h or mass_H");
    if (hb[7] & 2u) return set_error(URCHIN_ERR_ARG, "urchin_build_bvh: h must be > 0 and mass_H >= 0");
    b->hmax = ord2f(hb[6]);

    k_morton<<<grid, 256, 0, s>>>(p->pos_x, p->pos_y, p->pos_z, n, bounds, codes, idx);
    URCHIN_TRY(launched());
    URCHIN_TRY(radix_sort_pairs(codes, idx, n, 30, scr.at<void>(o_radix), s));
    int32_t* order = idx;
    if (n == 1) URCHIN_TRY_CUDA(cudaMemsetAsync(b->mslot, 0, sizeof(int32_t), s));
    if (n > 1) {
        int32_t* cl = scr.at<int32_t>(o_cl);
        int32_t* cr = scr.at<int32_t>(o_cr);
        int32_t* first = scr.at<int32_t>(o_first);
        int32_t* last = scr.at<int32_t>(o_last);
        int32_t* pint = scr.at<int32_t>(o_pint);
        const unsigned gi = (unsigned)((ni + 255) / 256);
        order = scr.at<int32_t>(o_order);
        k_karras<<<gi, 256, 0, s>>>(codes, (int)n, cl, cr, first, last, pint);
        URCHIN_TRY(launched());
        k_leaf_order<<<gi, 256, 0, s>>>((int)n, cl, cr, first, last, pint, idx, order, b->mslot, bounds + 7);
        URCHIN_TRY(launched());
    }
    const double mass_to_A = sigma_th_cm2() * 8.0 / kPi;
    k_gather<<<grid, 256, 0, s>>>(p->pos_x, p->pos_y, p->pos_z, p->h, p->mass_H, order, n, mass_to_A,
                                  b->unit_cm, b->xyzh, b->A32, b->A64, b->perm, b->inv,
                                  bounds + 7);
    URCHIN_TRY(launched());
    // levels up to the first of one entry above the blocks
    int64_t entries = 0;
    b->n_lev = 0;
    for (int l = 0, c = (int)((n + 31) / 32);; ++l, c = (c + 31) / 32) {
        if (l >= kMaxLevels) return set_error(URCHIN_ERR_CUDA, "urchin_build_bvh: too many tree levels");
        b->lev_off[l] = (int)entries;
        b->lev_cnt[l] = c;
        b->n_lev = l;
        entries += c;
        if (l > 0 && c == 1) break;
    }
    URCHIN_TRY_CUDA(cudaMalloc(&b->boxes, sizeof(float4) * 2 * (size_t)entries));
    k_blocks<<<(unsigned)((b->lev_cnt[0] + 7) / 8), 256, 0, s>>>(b->xyzh, (int)n, b->boxes, b->lev_cnt[0]);
    URCHIN_TRY(launched());
    for (int l = 1; l <= b->n_lev; ++l) {
        const int c = b->lev_cnt[l];
        k_level<<<(unsigned)((c + 7) / 8), 256, 0, s>>>(b->boxes + 2 * (int64_t)b->lev_off[l - 1], b->lev_cnt[l - 1],
                                                        b->boxes + 2 * (int64_t)b->lev_off[l], c);
        URCHIN_TRY(launched());
    }
    float4 root[2];
    URCHIN_TRY_CUDA(cudaMemcpyAsync(root, b->boxes + 2 * (int64_t)b->lev_off[b->n_lev], sizeof(root),
                                    cudaMemcpyDeviceToHost, s));
    URCHIN_TRY_CUDA(cudaMemcpyAsync(hb, bounds, sizeof(hb), cudaMemcpyDeviceToHost, s));
    URCHIN_TRY_CUDA(cudaStreamSynchronize(s));
    if (hb[7] & 12u) return set_error(URCHIN_ERR_CUDA, "urchin_build_bvh: internal consistency check failed (%u)",
                                      hb[7]);
    b->root_lo[0] = root[0].x;
    b->root_lo[1] = root[0].y;
    b->root_lo[2] = root[0].z;
    b->root_hi[0] = root[1].x;
    b->root_hi[1] = root[1].y;
    b->root_hi[2] = root[1].z;
    scr.release();
    URCHIN_TRY_CUDA(cudaStreamSynchronize(s));
    return URCHIN_OK;
}

}  // namespace

}  // namespace urchin

extern "C" int urchin_build_bvh(const urchin_particles* p, const urchin_box* box, urchin_bvh** out,
                                urchin_stream_t stream)
{
    using namespace urchin;
    clear_error();
    if (!out) return set_error(URCHIN_ERR_ARG, "urchin_build_bvh: out is NULL");
    *out = nullptr;
    if (!p || !box) return set_error(URCHIN_ERR_ARG, "urchin_build_bvh: particles or box is NULL");
    if (p->n < 1 || p->n > (int64_t)0x3fffffff)
        return set_error(URCHIN_ERR_ARG, "urchin_build_bvh: n = %lld out of range [1, 2^30)", (long long)p->n);
    if (!p->pos_x || !p->pos_y || !p->pos_z || !p->h || !p->mass_H)
        return set_error(URCHIN_ERR_ARG, "urchin_build_bvh: a particle array is NULL");
    if (!(box->unit_cm > 0.0) || !std::isfinite(box->unit_cm))
        return set_error(URCHIN_ERR_ARG, "urchin_build_bvh: unit_cm must be finite and > 0");
    if (box->periodic && (!(box->L > 0.0) || !std::isfinite(box->L)))
        return set_error(URCHIN_ERR_ARG, "urchin_build_bvh: periodic box needs finite L > 0");
    urchin_bvh* b = new (std::nothrow) urchin_bvh();
    if (!b) return set_error(URCHIN_ERR_NOMEM, "urchin_build_bvh: host allocation failed");
    int st = build(p, box, b, (cudaStream_t)stream);
    if (st != URCHIN_OK) {
        free_bvh_arrays(b);
        delete b;
        return st;
    }
    *out = b;
    return URCHIN_OK;
}

extern "C" void urchin_free_bvh(urchin_bvh* bvh)
{
    if (!bvh) return;
    cudaDeviceSynchronize();
    urchin::free_bvh_arrays(bvh);
    delete bvh;
}

extern "C" int64_t urchin_bvh_size(const urchin_bvh* bvh) { return bvh ? bvh->n : -1; }
