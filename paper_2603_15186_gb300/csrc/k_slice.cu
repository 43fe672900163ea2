// GS-slice occupancy (NavGSim Sec. III-C): every leaf Gaussian is cut by a set
// of horizontal planes z_k = z0 + k dz; on each plane the cut is the 2D
// Gaussian
//   G2D(x, z) = exp(-1/2 lambda (z - mu_z)^2) exp(-1/2 [x - mu(z)]^T C [x - mu(z)])
// with C the xy block of Sigma^-1, mu(z) = mu_xy - (z - mu_z) (alpha, beta) and
// lambda the Schur complement. Per plane and grid cell the kernel keeps the
// largest slice value a = min(0.99, o G2D(cell centre, z_k)) over the leaves
// whose a reaches 1/255; a cell is occupied where that value reaches the
// threshold.
//
// In float32 the slice parameters are taken in their well-conditioned forms
// (equal to the paper's by the block-inverse identities): lambda = 1 /
// Sigma_zz, (alpha, beta) = -(Sigma_xz, Sigma_yz) / Sigma_zz, C = (R S^-2 R^T)
// restricted to xy, so no difference of large terms appears.
//
// One thread per node takes the planes within the slice's vertical support and the
// box of cells of each slice's support (the ellipse where a >= 1/255, widened by a
// relative 1e-4 and 1e-6 m). Boxes differ (a few cells to hundreds: log-normal
// scales, interior nodes none), so a warp puts its leaves' boxes, every leaf on its
// first plane, then every leaf on its second, end to end and its lanes take the cells
// one each; a value is folded into its cell with atomicMax on its bits (non-negative
// floats order like their bit patterns, so the result does not depend on the order). 4M
// leaves, 13 planes, 528 x 276 cells of 5 cm (60 M cells in boxes): 1740 us with a loop per
// thread over its own boxes (6.6 of 32 lanes active) and a count per thread on one
// address, 350 us so; its atomics do not bound it (a look at the cell before each, to
// leave out those that change nothing: 538 us). Plane by plane for the whole warp, a plane
// that one leaf reaches costs as much as one that all reach: 300 planes 1 cm apart,
// 20 cm cells, 1M leaves of a floor 682 us (620 with the loop per thread), 525 us so;
// 60k leaves of a box, where the leaves of most planes end the call, 165 (120), 126 us.
#include "ngs_internal.cuh"

namespace ngs {

template <typename A>
__device__ __forceinline__ void load_sop(const void *p, int64_t i, float v[4]);
template <>
__device__ __forceinline__ void load_sop<float>(const void *p, int64_t i, float v[4]) {
    const float4 t = reinterpret_cast<const float4 *>(p)[i];
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
template <>
__device__ __forceinline__ void load_sop<__half>(const void *p, int64_t i, float v[4]) {
    const uint2 t = reinterpret_cast<const uint2 *>(p)[i];
    const float2 a = __half22float2(*reinterpret_cast<const __half2 *>(&t.x));
    const float2 b = __half22float2(*reinterpret_cast<const __half2 *>(&t.y));
    v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}
template <>
__device__ __forceinline__ void load_sop<__nv_bfloat16>(const void *p, int64_t i, float v[4]) {
    const uint2 t = reinterpret_cast<const uint2 *>(p)[i];
    v[0] = __uint_as_float(t.x << 16); v[1] = __uint_as_float(t.x & 0xffff0000u);
    v[2] = __uint_as_float(t.y << 16); v[3] = __uint_as_float(t.y & 0xffff0000u);
}

// One leaf's slice by one plane: what its cells' values need, and its support box.
struct __align__(16) SliceItem {
    float ez, cxx, cxy, cyy;
    float o, mx, my, inv_w;
    int32_t i0, j0, w;
    uint32_t plane;       // the plane's first cell in the grid
};

constexpr int kSliceThreads = 256;
// a slice of more cells is spread over the warp by itself
constexpr uint32_t kSliceBig = 1u << 16;

template <typename A>
__global__ void __launch_bounds__(kSliceThreads)
k_slice(SceneDev sc, SliceGrid g, uint32_t *__restrict__ value_bits,
        unsigned long long *work) {
    __shared__ SliceItem s_item[kSliceThreads / 32][32];
    __shared__ uint32_t s_start[kSliceThreads / 32][32];   // an item's first cell in the warp's list
    __shared__ unsigned long long s_evals[kSliceThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t node = (int64_t)blockIdx.x * kSliceThreads + threadIdx.x;
    int k0 = 0, k1 = -1;   // the planes that cut this thread's leaf
    float4 p = make_float4(0.f, 0.f, 0.f, 0.f);
    float o = 0.f, K = 0.f, lambda = 0.f, alpha = 0.f, beta = 0.f;
    float cxx = 0.f, cxy = 0.f, cyy = 0.f, ixx = 0.f, iyy = 0.f;
    // leaves only, and only those that reach 255 o >= 1
    if (node < sc.n && __float_as_int(sc.box_hi[node].w) == 0) p = sc.pos4[node];
    else p.w = __uint_as_float(kNodeCullOpacity);
    if (!(__float_as_uint(p.w) & kNodeCullOpacity)) {
        float so[4];
        load_sop<A>(sc.sop, node, so);
        o = so[3];
        K = 2.0f * logf(255.0f * o);                               // a >= 1/255 <=> q <= K
        const float4 q4 = sc.quat[node];
        const float qn = rsqrtf(q4.x * q4.x + q4.y * q4.y + q4.z * q4.z + q4.w * q4.w);
        const float w = q4.x * qn, x = q4.y * qn, y = q4.z * qn, z = q4.w * qn;
        const float R[9] = {1.f - 2.f * (y * y + z * z), 2.f * (x * y - w * z), 2.f * (x * z + w * y),
                            2.f * (x * y + w * z), 1.f - 2.f * (x * x + z * z), 2.f * (y * z - w * x),
                            2.f * (x * z - w * y), 2.f * (y * z + w * x), 1.f - 2.f * (x * x + y * y)};
        float s2[3], is2[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            s2[k] = expf(2.0f * so[k]);
            is2[k] = expf(-2.0f * so[k]);
        }
        // Sigma's z row and Sigma^-1's xy block
        float sxz = 0.f, syz = 0.f, szz = 0.f;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            sxz += R[k] * s2[k] * R[6 + k];
            syz += R[3 + k] * s2[k] * R[6 + k];
            szz += R[6 + k] * s2[k] * R[6 + k];
            cxx += R[k] * is2[k] * R[k];
            cxy += R[k] * is2[k] * R[3 + k];
            cyy += R[3 + k] * is2[k] * R[3 + k];
        }
        lambda = 1.0f / szz;
        alpha = -sxz / szz;
        beta = -syz / szz;
        const float det = cxx * cyy - cxy * cxy;
        if (det > 0.0f && K >= 0.0f) {
            // planes within the vertical support lambda z'^2 <= K
            const float rz = sqrtf(K / lambda) * 1.0001f + 1e-6f;
            k0 = max((int)ceilf((p.z - rz - g.z0) / g.dz), 0);
            k1 = min((int)floorf((p.z + rz - g.z0) / g.dz), g.nz - 1);
            ixx = cyy / det;                                       // C^-1 diagonal
            iyy = cxx / det;
        }
    }
    const uint32_t plane = (uint32_t)g.nx * (uint32_t)g.ny;   // the grid has < 2^31 cells
    unsigned long long evals = 0;
    const int span = k0 <= k1 ? k1 - k0 : -1;
    // the value of cell (i, j) of item t, folded into the plane's cell
    auto fold = [&](const SliceItem &t, int i, int j) {
        const float dy = g.y0 + ((float)j + 0.5f) * g.cell - t.my;
        const float dx = g.x0 + ((float)i + 0.5f) * g.cell - t.mx;
        // the terms in this order, the last one rounded before it is added
        const float q = __fadd_rn(__fmaf_rn(2.0f * t.cxy * dx, dy, __fmaf_rn(t.cxx * dx, dx, t.ez)),
                                  __fmul_rn(t.cyy * dy, dy));
        const float a = t.o * expf(-0.5f * q);
        if (a >= (1.0f / 255.0f))
            atomicMax(value_bits + t.plane + (uint32_t)j * (uint32_t)g.nx + (uint32_t)i,
                      __float_as_uint(fminf(0.99f, a)));
    };
    SliceItem *items = s_item[warp];
    uint32_t *starts = s_start[warp];
    // every lane's first plane, then every lane's second
    const int most = __reduce_max_sync(0xffffffffu, span);
    for (int at_plane = 0; at_plane <= most; ++at_plane) {
        SliceItem t;
        uint32_t n = 0, h = 0;   // cells and rows of this thread's slice
        if (at_plane <= span) {
            const int k = k0 + at_plane;
            const float zp = (g.z0 + (float)k * g.dz) - p.z;
            const float ez = lambda * zp * zp;
            const float rem = K - ez;
            if (rem >= 0.0f) {
                const float hx = sqrtf(rem * ixx) * 1.0001f + 1e-6f, hy = sqrtf(rem * iyy) * 1.0001f + 1e-6f;
                const float mx = p.x - zp * alpha, my = p.y - zp * beta;
                const int i0 = max(0, (int)ceilf((mx - hx - g.x0) / g.cell - 0.5f));
                const int i1 = min(g.nx - 1, (int)floorf((mx + hx - g.x0) / g.cell - 0.5f));
                const int j0 = max(0, (int)ceilf((my - hy - g.y0) / g.cell - 0.5f));
                const int j1 = min(g.ny - 1, (int)floorf((my + hy - g.y0) / g.cell - 0.5f));
                if (i0 <= i1 && j0 <= j1) {
                    t.ez = ez; t.cxx = cxx; t.cxy = cxy; t.cyy = cyy;
                    t.o = o; t.mx = mx; t.my = my;
                    t.i0 = i0; t.j0 = j0; t.w = i1 - i0 + 1;
                    t.plane = (uint32_t)k * plane;
                    t.inv_w = 1.0f / (float)t.w;
                    h = (uint32_t)(j1 - j0 + 1);
                    n = (uint32_t)t.w * h;      // < 2^31, the grid's cells
                    evals += n;
                }
            }
        }
        for (uint32_t big = __ballot_sync(0xffffffffu, n > kSliceBig); big; big &= big - 1) {
            const int src = __ffs(big) - 1;
            if (lane == src) items[0] = t;
            const uint32_t rows = __shfl_sync(0xffffffffu, h, src);
            __syncwarp();
            const SliceItem u = items[0];
            __syncwarp();
            for (uint32_t j = 0; j < rows; ++j)
                for (int i = lane; i < u.w; i += 32) fold(u, u.i0 + i, u.j0 + (int)j);
        }
        if (n > kSliceBig) n = 0;
        // the items that have cells, in lane order, and their cells end to end
        const uint32_t has = __ballot_sync(0xffffffffu, n > 0);
        if (has == 0) continue;
        if ((has & (has - 1)) == 0) {   // one item: a leaf of more planes than its neighbours
            const int src = __ffs(has) - 1;
            const uint32_t total = __shfl_sync(0xffffffffu, n, src);
            if (lane == src) items[0] = t;
            __syncwarp();
            const SliceItem u = items[0];
            __syncwarp();
            for (uint32_t r = lane; r < total; r += 32) {
                const uint32_t jj = (uint32_t)(((float)r + 0.5f) * u.inv_w);
                fold(u, u.i0 + (int)(r - jj * (uint32_t)u.w), u.j0 + (int)jj);
            }
            continue;
        }
        uint32_t incl = n;
#pragma unroll
        for (int s = 1; s < 32; s <<= 1) {
            const uint32_t v = __shfl_up_sync(0xffffffffu, incl, s);
            if (lane >= s) incl += v;
        }
        const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
        if (n > 0) {
            const int q = __popc(has & lanemask_lt());
            items[q] = t;
            starts[q] = incl - n;
        }
        __syncwarp();
        // lane l also holds the start of item l
        const uint32_t start = lane < __popc(has) ? starts[lane] : 0xffffffffu;
        for (uint32_t c0 = 0; c0 < total; c0 += 32) {
            // the item of cell c0 + lane: the last that starts at or before c0, plus
            // the items that start between
            const uint32_t at = __popc(__ballot_sync(0xffffffffu, start <= c0)) - 1;
            const uint32_t off = start - c0;
            const uint32_t marks =
                __reduce_or_sync(0xffffffffu, start > c0 && off < 32u ? 1u << off : 0u);
            const uint32_t c = c0 + lane;
            if (c < total) {
                const int q = at + __popc(marks & (lanemask_lt() | 1u << lane));
                const SliceItem u = items[q];
                // row and column in the box: exact, (r + 1/2) / w is at least
                // 1 / (2 w) from an integer and r < 2^17
                const uint32_t r = c - starts[q];
                const uint32_t jj = (uint32_t)(((float)r + 0.5f) * u.inv_w);
                fold(u, u.i0 + (int)(r - jj * (uint32_t)u.w), u.j0 + (int)jj);
            }
        }
        __syncwarp();
    }
    // one count per CTA: a count per thread, all on one address, took most of the
    // kernel's time
    if (work) {
#pragma unroll
        for (int s = 16; s > 0; s >>= 1) evals += __shfl_down_sync(0xffffffffu, evals, s);
        if (lane == 0) s_evals[warp] = evals;
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int w = 1; w < kSliceThreads / 32; ++w) evals += s_evals[w];
            if (evals) atomicAdd(work, evals);
        }
    }
}

__global__ void k_slice_mask(const uint32_t *__restrict__ value_bits, int64_t n, float threshold,
                             uint8_t *__restrict__ occ) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        occ[i] = __uint_as_float(value_bits[i]) >= threshold ? 1 : 0;
}

void launch_slice(const SceneDev &sc, const SliceGrid &g, float *value, uint8_t *occ,
                  unsigned long long *work, int num_sms, cudaStream_t st) {
    const int64_t cells = (int64_t)g.nx * g.ny * g.nz;
    cudaMemsetAsync(value, 0, (size_t)cells * sizeof(float), st);
    const int64_t blocks = (sc.n + kSliceThreads - 1) / kSliceThreads;
    uint32_t *bits = reinterpret_cast<uint32_t *>(value);
    if (blocks > 0) {
        switch (sc.attr_dtype) {
        case NGS_F16: k_slice<__half><<<(unsigned)blocks, kSliceThreads, 0, st>>>(sc, g, bits, work); break;
        case NGS_BF16:
            k_slice<__nv_bfloat16><<<(unsigned)blocks, kSliceThreads, 0, st>>>(sc, g, bits, work);
            break;
        default: k_slice<float><<<(unsigned)blocks, kSliceThreads, 0, st>>>(sc, g, bits, work); break;
        }
    }
    if (occ)
        k_slice_mask<<<std::max(1, (int)std::min<int64_t>((cells + 255) / 256, 16 * num_sms)), 256, 0,
                       st>>>(bits, cells, g.threshold, occ);
}

}  // namespace ngs
