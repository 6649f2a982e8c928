// kernels.cu -- the GB300 hot path of the 3DPV shadow-sample method.
//
// Per wave (a chunk of sun steps of one or more jobs), in stream order:
//   k_window      light window: bounding box of every module corner projected
//                 on the sun's light plane (Section 2, step 3: orthographic view
//                 from the sun, field of view limited to the generator)
//   k_light       light frame, texel size and origin per (job, step)
//   k_modsetup    each module at each step in texel space; marks the raster
//                 tiles that hold samples, their far plane (max sample depth +
//                 bias) and counts the receiver modules per tile
//   k_bin         (triangle, tile) pairs: one warp per 32 meshlets and step,
//                 meshlet boxes tested against the light window one per lane,
//                 then against the far planes of occupied tiles; the
//                 survivors' triangles transformed and binned one per lane;
//                 pairs counted per tile and appended to the wave's pair list
//   k_bin_big     same for triangles that span many tiles, one warp each
//   k_scan_*      bin offsets, the list of non-empty tiles, receiver offsets
//   k_scatter, k_recv_fill   write the bins and receiver lists
//   k_tile_warp   one warp per non-empty tile: one bit per texel and receiver
//                 plane, covered by something in front of that plane (Fig. 3:
//                 the depth buffer keeps the surface nearest the sun -- the
//                 samples of a plane need to know only whether that surface is
//                 in front of them), and the few texels where a triangle
//                 crosses the plane and depths must be compared
//   k_raster_test one CTA per tile that a warp cannot take (many triangles)
//   k_pv          per (step, module), one per lane: the maximum power point of
//                 modules over lit tiles, the list of the others
//   k_cells       per listed module, one warp: shaded samples per cell from
//                 the tiles' bits, irradiance per cell, substring currents,
//                 bypass-diode maximum power point (Section 2, step 4)
//   k_string, k_array   series strings and strings in parallel (when asked)
//   k_gen_step, k_heat  sky map of the effective shading (when asked)
//   k_epilogue    Kahan-compensated FP32 sums over the wave's steps in step
//                 order, per module, string and array (energy) and per cell
//                 (beam loss, when asked)
// A job may cover one window group of a generator (its own light window);
// the generator's other modules then enter its map as occluder meshlets.
// The map path replaces the tile kernels, k_pv and k_cells by k_raster_map (tiles stored
// to an HBM shadow map with 16-byte stores) + k_sample (texel gathers, ballot
// tallies, PV model).  Outside the waves: the clear-sky sun table and ideal
// tracker poses (k_sun_table, k_gather_sun, k_ideal_poses) and the diffuse
// sky view (k_sky_patches, then the waves over the patches, k_sky_fraction).
#include <cfloat>
#include <climits>
#include <cstdint>

#include "pv3d_dev.cuh"

namespace pv3d {

// ---------------------------------------------------------------------------
// helpers
// ---------------------------------------------------------------------------

// Order-preserving map float -> uint32 (a < b  <=>  key(a) < key(b)).
__device__ __forceinline__ uint32_t okey(float d)
{
    uint32_t b = __float_as_uint(d);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float okey_inv(uint32_t k)
{
    uint32_t b = (k & 0x80000000u) ? (k & 0x7FFFFFFFu) : ~k;
    return __uint_as_float(b);
}

constexpr uint32_t kEmpty = 0xFFFFFFFFu;

// Per-(step, cell) shaded samples, one byte per entry e (a count is at most
// n^2 <= 225).
__device__ __forceinline__ uint32_t tally_get(const uint32_t* words, int64_t e)
{
    return reinterpret_cast<const uint8_t*>(words)[e];
}
__device__ __forceinline__ void tally_set(uint32_t* words, int64_t e, uint32_t v)
{
    reinterpret_cast<uint8_t*>(words)[e] = (uint8_t)v;
}

// Largest job index j with base(j) <= item (bases ascend with j).
template <typename F>
__device__ __forceinline__ int job_of(int n_jobs, int64_t item, F base)
{
    int lo = 0, hi = n_jobs - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (base(mid) <= item) lo = mid; else hi = mid - 1;
    }
    return lo;
}

struct Basis {
    float ux, uy, uz, vx, vy, vz, sx, sy, sz;
};

// Light frame from the sun vector: w = s, u = normalize(s x z) (x at the
// zenith), v = s x u.  Below 2 degrees of elevation the frame is built in FP64.
__device__ __forceinline__ Basis light_basis(const double* sp)
{
    Basis b;
    double sx = sp[0], sy = sp[1], sz = sp[2];
    if (sz < 0.03489949670250097) {  // sin(2 deg)
        double h2 = sx * sx + sy * sy;
        double ux = 1.0, uy = 0.0;
        if (h2 >= 1e-12) {
            double r = 1.0 / sqrt(h2);
            ux = sy * r;
            uy = -sx * r;
        }
        b.ux = (float)ux; b.uy = (float)uy; b.uz = 0.f;
        b.vx = (float)(-sz * uy);
        b.vy = (float)(sz * ux);
        b.vz = (float)(sx * uy - sy * ux);
    } else {
        float fx = (float)sx, fy = (float)sy, fz = (float)sz;
        float h2 = fx * fx + fy * fy;
        float ux = 1.f, uy = 0.f;
        if (h2 >= 1e-12f) {
            float r = rsqrtf(h2);
            ux = fy * r;
            uy = -fx * r;
        }
        b.ux = ux; b.uy = uy; b.uz = 0.f;
        b.vx = -fz * uy;
        b.vy = fz * ux;
        b.vz = fx * uy - fy * ux;
    }
    b.sx = (float)sx; b.sy = (float)sy; b.sz = (float)sz;
    return b;
}

// Posed module frame relative to the job's reference point.  Tracker rotation
// R = Rz(pi - az) * Rx(tilt) about the pivot (pv3d_set_poses).
__device__ __forceinline__ void posed_module(const JobDev& J, const ModuleDev& M, int step,
                                             float3& o, float3& u, float3& v)
{
    o = make_float3(M.o[0], M.o[1], M.o[2]);
    u = make_float3(M.u[0], M.u[1], M.u[2]);
    v = make_float3(M.v[0], M.v[1], M.v[2]);
    if (M.tracker >= 0) {
        const float* pz = J.poses + 2 * ((size_t)step * (size_t)J.n_trk + (size_t)M.tracker);
        float sb, cb, sa, ca;
        sincosf(pz[1], &sb, &cb);
        sincosf(pz[0], &sa, &ca);
        float cg = -ca, sg = sa;
        float r00 = cg, r01 = -sg * cb, r02 = sg * sb;
        float r10 = sg, r11 = cg * cb, r12 = -cg * sb;
        float r20 = 0.f, r21 = sb, r22 = cb;
        const float* pv = J.pivots + 3 * M.tracker;
        float3 oo = o, uu = u, vv = v;
        o = make_float3(pv[0] + r00 * oo.x + r01 * oo.y + r02 * oo.z,
                        pv[1] + r10 * oo.x + r11 * oo.y + r12 * oo.z,
                        pv[2] + r20 * oo.x + r21 * oo.y + r22 * oo.z);
        u = make_float3(r00 * uu.x + r01 * uu.y + r02 * uu.z, r10 * uu.x + r11 * uu.y + r12 * uu.z,
                        r20 * uu.x + r21 * uu.y + r22 * uu.z);
        v = make_float3(r00 * vv.x + r01 * vv.y + r02 * vv.z, r10 * vv.x + r11 * vv.y + r12 * vv.z,
                        r20 * vv.x + r21 * vv.y + r22 * vv.z);
    }
}

__device__ __forceinline__ float dot3(float3 a, float ax, float ay, float az)
{
    return a.x * ax + a.y * ay + a.z * az;
}

// Sample (I, J) of a module, I = cu * n + i and J = cv * n + j, sits at
// a = (I + 1/2) p/n, b = (J + 1/2) p/n along the module axes (Section 2,
// step 3: n x n areas per cell, centred).  Its texel-space position is the
// row's base (the b terms) plus a times the module's first axis, so the
// samples of a row share the base.  The rasteriser's needed-texel mask, the
// fused test and the map gather all evaluate this one rounding sequence, so
// they agree bit for bit on the texel every sample reads.
struct SampleRow {
    float x, y, d;
};
__device__ __forceinline__ SampleRow sample_row(const ModStep& s, int Jr, float p_over_n)
{
    const float b = __fmul_rn(__fadd_rn((float)Jr, 0.5f), p_over_n);
    return SampleRow{__fmaf_rn(b, s.tbx, s.tx0), __fmaf_rn(b, s.tby, s.ty0), __fmaf_rn(b, s.db, s.d0)};
}

// floor(x) clamped to [0, r_max] (r_max = R - 1 < 2^22) without a conversion
// instruction: x is clamped as a float (NaN goes to 0), then 1.5 * 2^23 is
// added rounding toward minus infinity, which leaves floor(x) in the low
// mantissa bits.
__device__ __forceinline__ int texel_floor(float x, float r_max)
{
    const float c = fminf(fmaxf(x, 0.f), r_max);
    return __float_as_int(__fadd_rd(c, 12582912.f)) - 0x4B400000;
}

// Texel (ix, iy) and depth d of sample I of a row; ih = I + 1/2 (exact).
__device__ __forceinline__ void sample_texel(const ModStep& s, const SampleRow& row, float ih, float p_over_n,
                                             float r_max, int& ix, int& iy, float& d)
{
    const float a = __fmul_rn(ih, p_over_n);
    ix = texel_floor(__fmaf_rn(a, s.tax, row.x), r_max);
    iy = texel_floor(__fmaf_rn(a, s.tay, row.y), r_max);
    d = __fmaf_rn(a, s.da, row.d);
}

// (float)k + 1/2 for 0 <= k < 2^22, by the same exponent trick.
__device__ __forceinline__ float texel_centre(int k)
{
    return __fadd_rn(__fadd_rn(__int_as_float(0x4B400000 | k), -12582912.f), 0.5f);
}

// Inclusive prefix sum over the lanes of a warp.
__device__ __forceinline__ int warp_incl_scan(int v)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, v, off);
        if (lane >= off) v += y;
    }
    return v;
}

// Edge function A px + B py + C of a set-up triangle at a texel centre, and
// its interpolated depth.  The rasteriser, the sample-driven test and the
// culling masks all evaluate them with this one rounding sequence, so the
// paths agree bit for bit on which triangles cover a texel and at what depth.
__device__ __forceinline__ float edge_at(float A, float Bc, float C, float px, float py)
{
    return __fmaf_rn(A, px, __fmaf_rn(Bc, py, C));
}
__device__ __forceinline__ float depth_at(float w0, float w1, float w2, float e0, float e1, float e2)
{
    return __fmaf_rn(w2, e2, __fmaf_rn(w1, e1, __fmul_rn(w0, e0)));
}

// Is a sample at depth d with bias b behind the stored depth key `key`
// (Section 2, step 3: shaded iff farther from the sun than the nearest
// surface; equality is lit)?
__device__ __forceinline__ bool behind_key(float d, float bias, uint32_t key, float dnear, float qscale,
                                           int u24)
{
    if (u24) return __fmul_rn(__fsub_rn(d, dnear), qscale) > __fmaf_rn(bias, qscale, (float)key);
    return d > __fadd_rn(okey_inv(key), bias);
}

// The largest far plane of each block of kFarBlock x kFarBlock tiles lies at
// the start of the step's stretch of t_off, which has no other use until the
// scan fills it.
constexpr unsigned int kSmallWave = 4096;      // fused path: up to so many tiles those over share_bins are counted
constexpr int kShareSteps = 3;
__host__ __device__ constexpr unsigned int share_bins(int q) { return 8u << q; }
constexpr int kFarSh = 3, kFarBlock = 1 << kFarSh;
__device__ __forceinline__ int64_t far_block(int64_t te0, int tiles_x, int tx, int ty)
{
    return te0 + (int64_t)(ty >> kFarSh) * ((tiles_x + kFarBlock - 1) >> kFarSh) + (tx >> kFarSh);
}

// ---------------------------------------------------------------------------
// k_clear: reset the wave's accumulators (sizes read from the wave descriptor,
// so the whole wave can be replayed from one captured graph)
// ---------------------------------------------------------------------------

// Zero n bytes from p by threads i0, i0 + 1, ... of `stride`: 16 bytes at a time between the first
// and the last 16-byte boundary.
__device__ __forceinline__ void clear_bytes(void* p, int64_t n, int64_t i0, int64_t stride)
{
    uint8_t* b = static_cast<uint8_t*>(p);
    const int64_t head = min(n, (int64_t)((16u - (uint32_t)((uintptr_t)b & 15u)) & 15u)), quads = (n - head) / 16;
    const int64_t tail = head + 16 * quads;
    uint4* q = reinterpret_cast<uint4*>(b + head);
    for (int64_t i = i0; i < quads; i += stride) q[i] = make_uint4(0u, 0u, 0u, 0u);
    for (int64_t i = i0; i < head + n - tail; i += stride) b[i < head ? i : tail + i - head] = 0;
}

// Zero the rows of a per-cell output of job J (E bytes a cell; out_cstride
// cells a row, of which the job's n_cells).
template <int E>
__device__ __forceinline__ void clear_rows(uint8_t* p, const JobDev& J, int64_t i0, int64_t stride)
{
    p += (int64_t)J.out_row0 * J.out_cstride * E;
    if (J.out_cstride == J.n_cells) {
        clear_bytes(p, (int64_t)J.k * J.n_cells * E, i0, stride);
    } else {
        for (int64_t i = i0; i < (int64_t)J.k * J.n_cells; i += stride) {
            const int64_t r = i / J.n_cells;
            uint8_t* q = p + (r * J.out_cstride + i - r * J.n_cells) * E;
            if (E == 8) *reinterpret_cast<unsigned long long*>(q) = 0ull;
            else *q = 0;
        }
    }
}

__global__ void k_clear(const WaveDev* __restrict__ W, const JobDev* __restrict__ jobs, Buffers B)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i0 == 0) {
        B.ctr->n_big = 0u;
        B.ctr->n_nonempty = 0u;
        B.ctr->raster_next = 0u;
        B.ctr->n_heavy = 0u;
        B.ctr->n_pairs = 0ull;
        B.ctr->cov_next = 0ull;
        B.ctr->n_touch = 0u;
        B.ctr->n_first = 0u;
        B.ctr->n_rest = 0u;
        for (int q = 0; q < kShareSteps; ++q) B.ctr->n_over[q] = 0u;
        B.ctr->heavy_next = 0u;
    }
    const int64_t nw = 4 * W->tot_js, nt = W->tot_te;
    for (int64_t i = i0; i < nw; i += stride) B.win[i] = 0xFFFFFFFFu;
    for (int64_t i = i0; i < nt; i += stride) {
        B.t_far[i] = 0u;
        B.t_cnt[i] = 0u;
        B.t_rcnt[i] = 0u;
        B.t_plane[i] = kPlaneNone;
    }
    // the jobs' own, a share of the blocks each: the far planes of blocks of
    // tiles, and on the fused path the outputs per cell (k_cells writes the
    // cells that may be shaded).  (Cleared by the whole grid one after the
    // other, 500 jobs' took 379 us; the set-up stage went from 437 to 134.)
    const int nj = W->n_jobs, per = max((int)gridDim.x / nj, 1);
    const int64_t j0 = (blockIdx.x % per) * (int64_t)blockDim.x + threadIdx.x, js = (int64_t)per * blockDim.x;
    for (int q = blockIdx.x / per; q < nj; q += gridDim.x / per) {
        const JobDev& J = jobs[q];
        const int tw = J.tiles_x, cn = (tw + kFarBlock - 1) >> kFarSh, nc = cn * cn;
        for (int64_t i = j0; i < (int64_t)J.k * nc; i += js)
            B.t_off[J.te_base + i / nc * ((int64_t)tw * tw) + i % nc] = 0u;
        if (!W->fused) continue;
        if (J.kahan_cell)
            clear_bytes(reinterpret_cast<uint8_t*>(B.cs_cnt) + J.cs_base, (int64_t)J.k * J.n_cells, j0, js);
        if (J.out_counts) clear_rows<1>(J.out_counts, J, j0, js);
        if (J.out_bits) clear_rows<8>(reinterpret_cast<uint8_t*>(J.out_bits), J, j0, js);
    }
}

// ---------------------------------------------------------------------------
// k_window: projected bounding box of the generator per (job, step)
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kWinPerItem) k_window(const WaveDev* __restrict__ W,
                                                         const JobDev* __restrict__ jobs, Buffers B)
{
    __shared__ float red[4][kWinPerItem / 32];
    const int64_t tot = W->tot_win;
    const int nj = W->n_jobs;
    for (int64_t item = blockIdx.x; item < tot; item += gridDim.x) {
        int j = job_of(nj, item, [&](int q) { return jobs[q].it_win; });
        const JobDev& J = jobs[j];
        int64_t li = item - J.it_win;
        int groups = (J.n_mods + kWinPerItem - 1) / kWinPerItem;
        int ls = (int)(li / groups), g = (int)(li % groups);
        const double* sp = J.sun + 3 * (size_t)(J.step0 + ls);
        if (!(sp[2] > 0.0)) continue;  // uniform over the block
        Basis bs = light_basis(sp);
        float umin = FLT_MAX, umax = -FLT_MAX, vmin = FLT_MAX, vmax = -FLT_MAX;
        int m = g * kWinPerItem + threadIdx.x;
        if (m < J.n_mods) {
            const ModuleDev& M = J.mods[m];
            float3 o, u, v;
            posed_module(J, M, J.step0 + ls, o, u, v);
            float lu = M.cu * M.pitch, lv = M.cv * M.pitch;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                float a = (c == 1 || c == 2) ? lu : 0.f;
                float b = (c >= 2) ? lv : 0.f;
                float3 p = make_float3(o.x + a * u.x + b * v.x, o.y + a * u.y + b * v.y,
                                       o.z + a * u.z + b * v.z);
                float pu = dot3(p, bs.ux, bs.uy, bs.uz), pv = dot3(p, bs.vx, bs.vy, bs.vz);
                umin = fminf(umin, pu); umax = fmaxf(umax, pu);
                vmin = fminf(vmin, pv); vmax = fmaxf(vmax, pv);
            }
        }
#pragma unroll
        for (int off = 16; off; off >>= 1) {
            umin = fminf(umin, __shfl_xor_sync(0xffffffffu, umin, off));
            umax = fmaxf(umax, __shfl_xor_sync(0xffffffffu, umax, off));
            vmin = fminf(vmin, __shfl_xor_sync(0xffffffffu, vmin, off));
            vmax = fmaxf(vmax, __shfl_xor_sync(0xffffffffu, vmax, off));
        }
        int w = threadIdx.x >> 5;
        if ((threadIdx.x & 31) == 0) {
            red[0][w] = umin; red[1][w] = -umax; red[2][w] = vmin; red[3][w] = -vmax;
        }
        __syncthreads();
        if (threadIdx.x < 4) {
            float r = red[threadIdx.x][0];
            for (int q = 1; q < kWinPerItem / 32; ++q) r = fminf(r, red[threadIdx.x][q]);
            if (r < FLT_MAX) atomicMin(&B.win[4 * (size_t)(J.js_base + ls) + threadIdx.x], okey(r));
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// k_light: light frame, texel size delta = extent / (R - 2), window origin
// ---------------------------------------------------------------------------
__global__ void k_light(const WaveDev* __restrict__ W, const JobDev* __restrict__ jobs, Buffers B)
{
    const int64_t tot = W->tot_js;
    const int nj = W->n_jobs;
    for (int64_t js = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; js < tot;
         js += (int64_t)gridDim.x * blockDim.x) {
        int j = job_of(nj, js, [&](int q) { return (int64_t)jobs[q].js_base; });
        const JobDev& J = jobs[j];
        int ls = (int)(js - J.js_base);
        int step = J.step0 + ls;
        const double* sp = J.sun + 3 * (size_t)step;
        LightParams lp;
        Basis bs = light_basis(sp);
        lp.ux = bs.ux; lp.uy = bs.uy; lp.uz = bs.uz;
        lp.vx = bs.vx; lp.vy = bs.vy; lp.vz = bs.vz;
        lp.sx = bs.sx; lp.sy = bs.sy; lp.sz = bs.sz;
        lp.valid = sp[2] > 0.0;
        lp.dni = J.dni[step];
        lp.dhi = J.dhi[step];
        lp.dt = J.dt[step];
        lp.pad = 0;
        if (lp.valid) {
            float umin = okey_inv(B.win[4 * js + 0]), umax = -okey_inv(B.win[4 * js + 1]);
            float vmin = okey_inv(B.win[4 * js + 2]), vmax = -okey_inv(B.win[4 * js + 3]);
            float ext = fmaxf(fmaxf(umax - umin, vmax - vmin), 1e-6f);
            float delta = ext / (float)(J.R - 2);
            lp.delta = delta;
            lp.inv_delta = 1.f / delta;
            lp.u0 = 0.5f * (umin + umax) - 0.5f * J.R * delta;
            lp.v0 = 0.5f * (vmin + vmax) - 0.5f * J.R * delta;
            // depth range of everything (scene and generator bounds) for 24-bit depth
            float dmin = FLT_MAX, dmax = -FLT_MAX;
            for (int c = 0; c < 8; ++c) {
                float x = (c & 1) ? J.scene_hi[0] : J.scene_lo[0];
                float y = (c & 2) ? J.scene_hi[1] : J.scene_lo[1];
                float z = (c & 4) ? J.scene_hi[2] : J.scene_lo[2];
                float d = -(x * lp.sx + y * lp.sy + z * lp.sz);
                dmin = fminf(dmin, d); dmax = fmaxf(dmax, d);
            }
            float pad = 0.01f * (dmax - dmin) + 1.f;
            lp.dnear = dmin - pad;
            lp.qscale = 16777214.f / ((dmax + pad) - lp.dnear);
        } else {
            lp.delta = 0.f; lp.inv_delta = 0.f; lp.u0 = 0.f; lp.v0 = 0.f;
            lp.dnear = 0.f; lp.qscale = 0.f;
        }
        B.lp[js] = lp;
    }
}

// Depth key stored in the map for depth d (FP32 order bits, or 24-bit fixed point).
__device__ __forceinline__ uint32_t depth_store_key(float d, const LightParams& lp, int u24)
{
    if (!u24) return okey(d);
    float q = (d - lp.dnear) * lp.qscale;
    q = fminf(fmaxf(q, 0.f), 16777214.f);
    return (uint32_t)q;  // truncation: a surface is never stored farther than it is
}

// ---------------------------------------------------------------------------
// k_modsetup: module frames in texel space, bias, tile occupancy, far planes,
// receiver counts; k_recv_fill lists the receivers of the non-empty tiles
// ---------------------------------------------------------------------------
struct TileRange {
    int tx0, tx1, ty0, ty1;
    float dmax;
};

// Tiles touched by the bounding box of a module's corners in texel space.
__device__ __forceinline__ TileRange module_tiles(const ModStep& s, const ModuleDev& M, int R, int sh)
{
    const float lu = M.cu * M.pitch, lv = M.cv * M.pitch;
    float xmin = FLT_MAX, xmax = -FLT_MAX, ymin = FLT_MAX, ymax = -FLT_MAX, dmax = -FLT_MAX;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float a = (k == 1 || k == 2) ? lu : 0.f;
        const float b = (k >= 2) ? lv : 0.f;
        const float x = s.tx0 + a * s.tax + b * s.tbx;
        const float y = s.ty0 + a * s.tay + b * s.tby;
        const float d = s.d0 + a * s.da + b * s.db;
        xmin = fminf(xmin, x); xmax = fmaxf(xmax, x);
        ymin = fminf(ymin, y); ymax = fmaxf(ymax, y);
        dmax = fmaxf(dmax, d);
    }
    TileRange t;
    t.tx0 = max(0, min(R - 1, (int)floorf(xmin))) >> sh;
    t.tx1 = max(0, min(R - 1, (int)floorf(xmax))) >> sh;
    t.ty0 = max(0, min(R - 1, (int)floorf(ymin))) >> sh;
    t.ty1 = max(0, min(R - 1, (int)floorf(ymax))) >> sh;
    if ((R >> sh) == 0) t.ty1 = t.ty0 - 1;  // a map smaller than a tile has none
    t.dmax = dmax;
    return t;
}

// Threads that share a (step, module) item's tiles: a warp when the wave has
// too few items to fill the grid otherwise (a module may touch a hundred tiles:
// for two modules over a day of suns, R = 1024, a thread each made the set-up
// kernels 105 us, a warp each 32 us).
__device__ __forceinline__ int mod_group(int64_t tot)
{
    return tot * 32 <= (int64_t)gridDim.x * blockDim.x ? 32 : 1;
}

__global__ void k_modsetup(const WaveDev* __restrict__ W, const JobDev* __restrict__ jobs, Buffers B)
{
    const int64_t tot = W->tot_mod;
    const int nj = W->n_jobs;
    const int sh = W->tile_sh;
    const int u24 = W->depth_u24;
    const int grp = mod_group(tot), sub = threadIdx.x & (grp - 1);
    for (int64_t item = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / grp; item < tot;
         item += (int64_t)gridDim.x * blockDim.x / grp) {
        int j = job_of(nj, item, [&](int q) { return jobs[q].it_mod; });
        const JobDev& J = jobs[j];
        int64_t li = item - J.it_mod;
        int ls = (int)(li / J.n_mods), m = (int)(li % J.n_mods);
        int64_t js = J.js_base + ls;
        const LightParams& lp = B.lp[js];
        if (!lp.valid) continue;
        const ModuleDev& M = J.mods[m];
        float3 o, u, v;
        posed_module(J, M, J.step0 + ls, o, u, v);
        ModStep s;
        float lo_u = dot3(o, lp.ux, lp.uy, lp.uz), lo_v = dot3(o, lp.vx, lp.vy, lp.vz);
        s.tx0 = (lo_u - lp.u0) * lp.inv_delta;
        s.ty0 = (lo_v - lp.v0) * lp.inv_delta;
        s.d0 = -dot3(o, lp.sx, lp.sy, lp.sz);
        s.tax = dot3(u, lp.ux, lp.uy, lp.uz) * lp.inv_delta;
        s.tay = dot3(u, lp.vx, lp.vy, lp.vz) * lp.inv_delta;
        s.da = -dot3(u, lp.sx, lp.sy, lp.sz);
        s.tbx = dot3(v, lp.ux, lp.uy, lp.uz) * lp.inv_delta;
        s.tby = dot3(v, lp.vx, lp.vy, lp.vz) * lp.inv_delta;
        s.db = -dot3(v, lp.sx, lp.sy, lp.sz);
        float3 n = make_float3(u.y * v.z - u.z * v.y, u.z * v.x - u.x * v.z, u.x * v.y - u.y * v.x);
        float nl = rsqrtf(n.x * n.x + n.y * n.y + n.z * n.z);
        n.x *= nl; n.y *= nl; n.z *= nl;
        float c = dot3(n, lp.sx, lp.sy, lp.sz);
        s.cosi = c;
        s.nz = n.z;
        // slope-scaled bias: half a texel diagonal times the receiver slope
        // (tan of incidence, clamped at 89 deg) plus 1/32 texel
        float cc = fmaxf(c, 0.017452406f);
        float tan_i = sqrtf(fmaxf(0.f, 1.f - cc * cc)) / cc;
        s.bias = lp.delta * (0.70710678f * tan_i + 0.03125f);
        if (u24) s.bias += 2.f / lp.qscale;
        // the depth plane of the samples over the light plane, and how far a
        // sample's depth may lie from the plane's at the centre of its texel:
        // the slope over half a texel, the rounding of positions and depths
        // (of this module and of others on the plane, whose bias may differ by
        // the rounding of cos i under the square root), of the plane's own
        // coefficients, and a few steps of 24-bit depth.  No plane within a
        // degree of the sun.
        const float lu = M.cu * M.pitch, lv = M.cv * M.pitch;
        const float det = s.tax * s.tby - s.tay * s.tbx;
        const float dsum = fabsf(s.tax * s.tby) + fabsf(s.tay * s.tbx);
        if (fabsf(det) > 1e-6f * dsum && fabsf(c) > 0.017452406f) {
            const float inv_det = 1.f / det;
            s.pa = (s.da * s.tby - s.db * s.tay) * inv_det;
            s.pb = (s.db * s.tax - s.da * s.tbx) * inv_det;
            const float ex = fabsf(lu * s.tax) + fabsf(lv * s.tbx) + 256.f;
            const float ey = fabsf(lu * s.tay) + fabsf(lv * s.tby) + 256.f;
            s.hs = 0.52f * (fabsf(s.pa) + fabsf(s.pb)) +
                   4e-6f * fabsf(dsum * inv_det) * (fabsf(s.pa) * ex + fabsf(s.pb) * ey) +
                   2e-6f * (fabsf(o.x) + fabsf(o.y) + fabsf(o.z) + lu + lv) + 2e-5f + 1e-3f * lp.delta +
                   (u24 ? 8.f / lp.qscale : 0.f);
        } else {
            s.pa = s.pb = 0.f;
            s.hs = INFINITY;
        }
        s.pad = 0.f;
        if (sub == 0) B.ms[J.ms_base + li] = s;
        // A triangle shades a sample only where its depth is below the
        // sample's depth minus the bias, so a tile may drop every triangle whose
        // nearest point is not nearer than (max sample depth - bias).
        const TileRange tr = module_tiles(s, M, J.R, sh);
        const uint32_t far_key = u24 ? depth_store_key(tr.dmax - s.bias, lp, 1) + 2u : okey(tr.dmax - s.bias);
        const int64_t te0 = J.te_base + (int64_t)ls * J.tiles_x * J.tiles_x;
        for (int ty = tr.ty0; ty <= tr.ty1; ++ty)
            for (int tx = tr.tx0 + sub; tx <= tr.tx1; tx += grp) {
                const int64_t te = te0 + (int64_t)ty * J.tiles_x + tx;
                atomicMax(&B.t_far[te], far_key);
                // (once per module and block of tiles, and most are no farther
                // than one before)
                if ((tx == tr.tx0 || (tx & (kFarBlock - 1)) == 0) && (ty == tr.ty0 || (ty & (kFarBlock - 1)) == 0)) {
                    uint32_t* fb = &B.t_off[far_block(te0, J.tiles_x, tx, ty)];
                    if (__ldcg(fb) < far_key) atomicMax(fb, far_key);
                }
                atomicAdd(&B.t_rcnt[te], 1u);
                // the plane group shared by every receiver of the tile
                const uint32_t pl = (uint32_t)M.plane;
                const uint32_t old = atomicCAS(&B.t_plane[te], kPlaneNone, pl);
                // fused path: a module of the tile, for the plane of a tile of one group
                if (old == kPlaneNone) B.t_roff[te] = (uint32_t)m;
                if (old != kPlaneNone && old != pl && old != kPlaneMixed) atomicExch(&B.t_plane[te], kPlaneMixed);
            }
    }
}

// After the scan: list each module as a receiver of the non-empty tiles it
// touches (fused path: only of tiles of several plane groups, the others need
// no list).
__global__ void k_recv_fill(const WaveDev* __restrict__ W, const JobDev* __restrict__ jobs, Buffers B)
{
    const int64_t tot = W->tot_mod;
    const int nj = W->n_jobs;
    const int sh = W->tile_sh;
    const int64_t cap = W->recv_cap;
    const int fused = W->fused;
    const int grp = mod_group(tot), sub = threadIdx.x & (grp - 1);
    for (int64_t item = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / grp; item < tot;
         item += (int64_t)gridDim.x * blockDim.x / grp) {
        int j = job_of(nj, item, [&](int q) { return jobs[q].it_mod; });
        const JobDev& J = jobs[j];
        int64_t li = item - J.it_mod;
        int ls = (int)(li / J.n_mods), m = (int)(li % J.n_mods);
        if (!B.lp[J.js_base + ls].valid) continue;
        const ModStep s = B.ms[J.ms_base + li];
        const TileRange tr = module_tiles(s, J.mods[m], J.R, sh);
        const int64_t te0 = J.te_base + (int64_t)ls * J.tiles_x * J.tiles_x;
        for (int ty = tr.ty0; ty <= tr.ty1; ++ty)
            for (int tx = tr.tx0 + sub; tx <= tr.tx1; tx += grp) {
                const int64_t te = te0 + (int64_t)ty * J.tiles_x + tx;
                if (B.t_cnt[te] == 0u || (fused && B.t_plane[te] != kPlaneMixed)) continue;
                const uint32_t pos = atomicAdd(&B.t_rcur[te], 1u);
                if (pos < (uint64_t)cap) B.recv[pos] = (uint32_t)m;
            }
    }
}

// ---------------------------------------------------------------------------
// triangles in texel space
// ---------------------------------------------------------------------------
struct TriT {
    float x[3], y[3], d[3];
};

// Light-space texel coordinates and depth of a point (world, relative to the
// job's reference), with every rounding written out: the tile kernels and
// the map path inline this in different contexts, and must get the same
// bits for the same vertex whatever the compiler would otherwise fuse.
__device__ __forceinline__ void project_point(const LightParams& lp, float x, float y, float z, float& tx, float& ty,
                                              float& d)
{
    tx = __fmul_rn(__fsub_rn(__fmaf_rn(z, lp.uz, __fmaf_rn(y, lp.uy, __fmul_rn(x, lp.ux))), lp.u0), lp.inv_delta);
    ty = __fmul_rn(__fsub_rn(__fmaf_rn(z, lp.vz, __fmaf_rn(y, lp.vy, __fmul_rn(x, lp.vx))), lp.v0), lp.inv_delta);
    d = -__fmaf_rn(z, lp.sz, __fmaf_rn(y, lp.sy, __fmul_rn(x, lp.sx)));
}

// Triangle q of a window group's occluder modules (every module of the
// generator, posed for the step and projected like the scene).  Not inlined:
// the pose's sines and cosines would sit in every kernel that reads triangles.
__device__ __noinline__ void occ_tri_texel(const JobDev& J, const LightParams& lp, int ls, int q, TriT& T)
{
    float3 o, u, v;
    const ModuleDev& M = J.occ_mods[q >> 1];
    posed_module(J, M, J.step0 + ls, o, u, v);
    const float lu = M.cu * M.pitch, lv = M.cv * M.pitch;
    // corners c0 = O, c1 = O + lu U, c2 = O + lu U + lv V, c3 = O + lv V;
    // triangles (c0, c1, c2) and (c0, c2, c3)
    const float a1 = lu, b1 = (q & 1) ? lv : 0.f;
    const float a2 = (q & 1) ? 0.f : lu, b2 = lv;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float a = k == 0 ? 0.f : (k == 1 ? a1 : a2), b = k == 0 ? 0.f : (k == 1 ? b1 : b2);
        const float x = __fmaf_rn(b, v.x, __fmaf_rn(a, u.x, o.x));
        const float y = __fmaf_rn(b, v.y, __fmaf_rn(a, u.y, o.y));
        const float z = __fmaf_rn(b, v.z, __fmaf_rn(a, u.z, o.z));
        project_point(lp, x, y, z, T.x[k], T.y[k], T.d[k]);
    }
}

// Triangle `t` of job J (scene triangle, or module triangle after the scene's)
// at local step ls in texel coordinates.  Module triangles come from the
// job's own module frames (ModStep), or, for a window group, from every
// module of the generator posed for the step and projected like the scene.
__device__ __forceinline__ void tri_texel(const JobDev& J, const Buffers& B, const LightParams& lp,
                                          int ls, int t, TriT& T)
{
    if (t >= J.n_tris && J.occ_mods) {
        TriT O;
        occ_tri_texel(J, lp, ls, t - J.n_tris, O);
        T = O;
        return;
    }
    if (t < J.n_tris) {
        const float4* p = J.tri + 3 * (size_t)t;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const float4 q = __ldg(p + k);
            project_point(lp, __fsub_rn(q.x, J.ref[0]), __fsub_rn(q.y, J.ref[1]), __fsub_rn(q.z, J.ref[2]), T.x[k],
                          T.y[k], T.d[k]);
        }
    } else {
        int q = t - J.n_tris;
        int m = q >> 1;
        const ModuleDev& M = J.mods[m];
        const ModStep s = B.ms[J.ms_base + (int64_t)ls * J.n_mods + m];
        float lu = M.cu * M.pitch, lv = M.cv * M.pitch;
        // quad corners c0 = O, c1 = O + lu U, c2 = O + lu U + lv V, c3 = O + lv V;
        // triangles (c0, c1, c2) and (c0, c2, c3)
        float a1 = lu, b1 = (q & 1) ? lv : 0.f;
        float a2 = (q & 1) ? 0.f : lu, b2 = lv;
        T.x[0] = s.tx0; T.y[0] = s.ty0; T.d[0] = s.d0;
        T.x[1] = __fmaf_rn(b1, s.tbx, __fmaf_rn(a1, s.tax, s.tx0));
        T.y[1] = __fmaf_rn(b1, s.tby, __fmaf_rn(a1, s.tay, s.ty0));
        T.d[1] = __fmaf_rn(b1, s.db, __fmaf_rn(a1, s.da, s.d0));
        T.x[2] = __fmaf_rn(b2, s.tbx, __fmaf_rn(a2, s.tax, s.tx0));
        T.y[2] = __fmaf_rn(b2, s.tby, __fmaf_rn(a2, s.tay, s.ty0));
        T.d[2] = __fmaf_rn(b2, s.db, __fmaf_rn(a2, s.da, s.d0));
    }
}

// Plane group of triangle t if it is a module triangle (the job's own
// modules, or the generator's occluder modules of a window group), else
// kPlaneNone.  Modules of one plane group cannot shade one another, so a
// module triangle is not binned into a tile whose receivers all share its
// plane group (t_plane).
__device__ __forceinline__ uint32_t module_tri_plane(const JobDev& J, int t)
{
    if (t < J.n_tris) return kPlaneNone;
    const int m = (t - J.n_tris) >> 1;
    return (uint32_t)(J.occ_mods ? J.occ_mods[m].plane : J.mods[m].plane);
}

// Edge functions of a counter-clockwise triangle: E_k(p) = A_k px + B_k py + C_k,
// inside iff every E_k >= 0.  Returns false for a degenerate (edge-on) triangle.
struct Edges {
    float A[3], Bc[3], C[3];
    float area2;
};

__device__ __forceinline__ bool make_edges(TriT& T, Edges& e)
{
    float area2 = __fsub_rn(__fmul_rn(__fsub_rn(T.x[1], T.x[0]), __fsub_rn(T.y[2], T.y[0])),
                            __fmul_rn(__fsub_rn(T.y[1], T.y[0]), __fsub_rn(T.x[2], T.x[0])));
    if (!(fabsf(area2) > 0.f)) return false;
    if (area2 < 0.f) {
        float tx = T.x[1], ty = T.y[1], td = T.d[1];
        T.x[1] = T.x[2]; T.y[1] = T.y[2]; T.d[1] = T.d[2];
        T.x[2] = tx; T.y[2] = ty; T.d[2] = td;
        area2 = -area2;
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        // edge k is opposite vertex k: from vertex k+1 to vertex k+2
        int a = (k + 1) % 3, b = (k + 2) % 3;
        e.A[k] = -__fsub_rn(T.y[b], T.y[a]);
        e.Bc[k] = __fsub_rn(T.x[b], T.x[a]);
        e.C[k] = -__fadd_rn(__fmul_rn(e.A[k], T.x[a]), __fmul_rn(e.Bc[k], T.y[a]));
    }
    e.area2 = area2;
    return true;
}

// Could the triangle cover a texel centre of the rectangle [x0,x1] x [y0,y1]?
__device__ __forceinline__ bool rect_overlap(const Edges& e, float x0, float x1, float y0, float y1)
{
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        float x = e.A[k] > 0.f ? x1 : x0;
        float y = e.Bc[k] > 0.f ? y1 : y0;
        if (e.A[k] * x + e.Bc[k] * y + e.C[k] < 0.f) return false;
    }
    return true;
}

// ---------------------------------------------------------------------------
// k_bin: (triangle, tile) pairs in one pass -- vertex transform batched over
// steps; each pair is counted into its tile and appended to the wave's pair
// list, which k_scatter distributes into the bins after the scan
// ---------------------------------------------------------------------------

// Append this lane's pairs (te[q], tri) for the set bits q of `valid` to the
// pair list: one atomic per warp.  Called by all 32 lanes together.
__device__ __forceinline__ void append_pairs(const Buffers& B, const WaveDev* W, const uint32_t* te, uint32_t valid,
                                             uint32_t tri)
{
    const int lane = threadIdx.x & 31;
    const int c = __popc(valid);
    const int inc = warp_incl_scan(c);
    const int tot = __shfl_sync(0xffffffffu, inc, 31);
    if (tot == 0) return;
    unsigned long long base = 0;
    if (lane == 31) base = atomicAdd(&B.ctr->n_pairs, (unsigned long long)tot);
    base = __shfl_sync(0xffffffffu, base, 31);
    unsigned long long pos = base + (unsigned long long)(inc - c);
    const uint64_t cap = (uint64_t)W->bin_cap;
#pragma unroll
    for (int q = 0; q < kBigTiles; ++q)
        if (valid & (1u << q)) {
            if (pos < cap) B.pairs[pos] = make_uint2(te[q], tri);
            ++pos;
        }
}

constexpr int kLaneTiles = 16;   // a meshlet over at most this many tiles is tested by its own lane,
constexpr int kFineTiles = 512;  // over at most this many tile by tile, over more by blocks of tiles only

// Texel extents of a world box under a light.
struct TexBox {
    float x0, x1, y0, y1, d0;
};
__device__ __forceinline__ TexBox project_box(const float4* box, const JobDev& J, const LightParams& lp)
{
    const float4 lo = box[0], hi = box[1];
    TexBox b = {FLT_MAX, -FLT_MAX, FLT_MAX, -FLT_MAX, FLT_MAX};
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const float x = ((c & 1) ? hi.x : lo.x) - J.ref[0];
        const float y = ((c & 2) ? hi.y : lo.y) - J.ref[1];
        const float z = ((c & 4) ? hi.z : lo.z) - J.ref[2];
        const float tx = (x * lp.ux + y * lp.uy + z * lp.uz - lp.u0) * lp.inv_delta;
        const float ty = (x * lp.vx + y * lp.vy + z * lp.vz - lp.v0) * lp.inv_delta;
        b.x0 = fminf(b.x0, tx); b.x1 = fmaxf(b.x1, tx);
        b.y0 = fminf(b.y0, ty); b.y1 = fmaxf(b.y1, ty);
        b.d0 = fminf(b.d0, -(x * lp.sx + y * lp.sy + z * lp.sz));
    }
    return b;
}

__global__ void __launch_bounds__(256, 4) k_bin(const WaveDev* __restrict__ W, const JobDev* __restrict__ jobs,
                                             Buffers B)
{
    // One warp per (32 groups of 32 meshlets, step), the step fastest so that
    // consecutive warps reuse the groups' triangles from cache.  Each lane
    // projects one group's bounding box; in the groups that overlap the light
    // window, one after the other, each lane then projects one scene meshlet's
    // box and keeps it if it overlaps the window; each kept box is tested
    // against the far planes of the tiles it covers: if no tile can receive a
    // shadow from the meshlet, its 32 triangles are skipped together.
    // Otherwise each lane bins one of its triangles.  Generator module
    // triangles follow the scene's, in meshlets of 32, without the box test.
    // A triangle over more than kBigTiles tiles is listed for k_bin_big.
    //
    // Bound by instruction issue (65 % of the slots while an SM has work).
    // 500 light windows over 560 000 triangles, 29 suns: almost every meshlet
    // is outside a window, and with a box each tested by every window the
    // kernel took 4.49 ms, with groups first 0.6.  One window over all of them,
    // 47 suns: at a low sun a meshlet's box covers thousands of tiles, and the
    // warps that had to read them all took 652 us while the others had long
    // finished; by blocks of tiles 223.
    const int64_t tot = W->tot_tri;
    const int nj = W->n_jobs;
    const int sh = W->tile_sh;
    const int TS = 1 << sh;
    const int u24 = W->depth_u24;
    const int lane = threadIdx.x & 31;
    const int64_t n_warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    // few items: several warps share one's groups, each testing all boxes
    int parts = 1;
    while (parts < 32 && tot * parts < n_warps) parts *= 2;
    for (int64_t item = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; item < tot * parts; item += n_warps) {
        const int j = job_of(nj, item, [&](int q) { return jobs[q].it_tri * parts; });
        const JobDev& J = jobs[j];
        const uint32_t li = (uint32_t)(item - J.it_tri * parts);
        const int sp = (int)(li / (uint32_t)J.k), ls = (int)(li - (uint32_t)sp * (uint32_t)J.k);
        const int R = J.R;
        const int64_t js = J.js_base + ls;
        const LightParams& lp = B.lp[js];
        if (!lp.valid || J.tiles_x == 0) continue;  // (a map smaller than a tile has none)
        const int64_t te0 = J.te_base + (int64_t)ls * J.tiles_x * J.tiles_x;
        // scene meshlets, then (window groups) occluder-module meshlets, both
        // with boxes, then the job's own module meshlets
        const int n_boxed = J.n_ml + J.n_oml;
        const int n_all = n_boxed + ((J.n_mtris + 31) >> 5);
        // this lane's group of 32 meshlets: those of the scene have a box
        const int gl = (sp / parts) * 32 + lane;
        bool in_window = gl * 32 < n_all && (lane & (parts - 1)) == (sp & (parts - 1));
        if (in_window && gl * 32 + 31 < J.n_ml) {
            const TexBox bx = project_box(J.ml_box + 2 * (J.n_ml + gl), J, lp);
            in_window = bx.x1 >= 0.f && bx.y1 >= 0.f && bx.x0 <= (float)R && bx.y0 <= (float)R;
        }
#pragma unroll 1
        for (unsigned int gm = __ballot_sync(0xffffffffu, in_window); gm; gm &= gm - 1u) {
            const int g = (sp / parts) * 32 + __ffs((int)gm) - 1;
            // this lane's boxed meshlet: window test, covered tiles, nearest depth key
            const int ml = g * 32 + lane;
            int btx0 = 0, btx1 = -1, bty0 = 0, bty1 = -1;
            uint32_t bkey = 0u;
            bool pass = false;
            if (ml < n_boxed) {
                const TexBox bx = project_box(ml < J.n_ml ? J.ml_box + 2 * ml : J.oml_box + 2 * (ml - J.n_ml), J, lp);
                const float xmin = bx.x0, xmax = bx.x1, ymin = bx.y0, ymax = bx.y1, dmin = bx.d0;
                pass = xmax >= 0.5f && ymax >= 0.5f && xmin <= R - 0.5f && ymin <= R - 0.5f;
                if (pass) {
                    btx0 = max(0, (int)floorf(xmin - 0.5f)) >> sh;
                    btx1 = min(R - 1, (int)ceilf(xmax)) >> sh;
                    bty0 = max(0, (int)floorf(ymin - 0.5f)) >> sh;
                    bty1 = min(R - 1, (int)ceilf(ymax)) >> sh;
                    // the box's nearest point, less a margin for the rounding of
                    // the projection
                    bkey = depth_store_key(dmin - 1e-3f * (1.f + fabsf(dmin)), lp, u24);
                }
            } else {
                pass = ml < n_all;
            }
            // the meshlet's nearest point against the far plane of each tile it
            // covers: each lane tests its own meshlet's tiles (independent loads
            // across the warp), the warp together those of a meshlet over many
            // tiles
            bool keep_lane = false, coop = false;
            if (pass && ml < n_boxed) {
                const int ntl = (btx1 - btx0 + 1) * (bty1 - bty0 + 1);
                if (ntl <= kLaneTiles) {
                    // no early exit: the loads of a row of tiles are issued together
                    for (int ty = bty0; ty <= bty1; ++ty) {
                        const uint32_t* far_row = B.t_far + te0 + (int64_t)ty * J.tiles_x;
    #pragma unroll 4
                        for (int tx = btx0; tx <= btx1; ++tx) keep_lane |= bkey < far_row[tx];
                    }
                } else {
                    coop = true;
                }
            } else if (pass) {
                keep_lane = true;  // module meshlets: no box
            }
            unsigned int kept = __ballot_sync(0xffffffffu, keep_lane);
            for (unsigned int cm = __ballot_sync(0xffffffffu, coop); cm; cm &= cm - 1u) {
                const int q = __ffs(cm) - 1;
                const int mx0 = __shfl_sync(0xffffffffu, btx0, q), mx1 = __shfl_sync(0xffffffffu, btx1, q);
                const int my0 = __shfl_sync(0xffffffffu, bty0, q), my1 = __shfl_sync(0xffffffffu, bty1, q);
                const uint32_t mkey = __shfl_sync(0xffffffffu, bkey, q);
                const int wx = mx1 - mx0 + 1, ntl = wx * (my1 - my0 + 1);
                // blocks of tiles first
                const int cx0 = mx0 >> kFarSh, cy0 = my0 >> kFarSh, cw = (mx1 >> kFarSh) - cx0 + 1;
                const int nc = cw * ((my1 >> kFarSh) - cy0 + 1);
                bool keep = false;
                for (int q0 = 0; q0 < nc && !keep; q0 += 32) {
                    const int k = q0 + lane;
                    keep = __any_sync(0xffffffffu,
                                      k < nc && mkey < B.t_off[far_block(te0, J.tiles_x, (cx0 + k % cw) << kFarSh,
                                                                         (cy0 + k / cw) << kFarSh)]);
                }
                if (keep && ntl > kFineTiles) {
                    kept |= 1u << q;
                    continue;
                }
                if (!keep) continue;
                keep = false;
                for (int q0 = 0; q0 < ntl && !keep; q0 += 32) {
                    const int k = q0 + lane;
                    bool kk = false;
                    if (k < ntl) {
                        const int ty = my0 + k / wx, tx = mx0 + k % wx;
                        kk = mkey < B.t_far[te0 + (int64_t)ty * J.tiles_x + tx];
                    }
                    keep = __any_sync(0xffffffffu, kk);
                }
                if (keep) kept |= 1u << q;
            }
            for (unsigned int cand = kept; cand; cand &= cand - 1u) {
                const int q = __ffs(cand) - 1;
                const int mi = g * 32 + q;
                int t;
                bool act;
                if (mi < n_boxed) {
                    if (mi < J.n_ml) {
                        t = mi * 32 + lane;
                        act = t < J.n_tris;
                    } else {
                        t = J.n_tris + (mi - J.n_ml) * 32 + lane;
                        act = t < J.n_tris + 2 * J.n_occ;
                    }
                } else {
                    t = J.n_tris + (mi - n_boxed) * 32 + lane;
                    act = t < J.n_tris + J.n_mtris;
                }
                // per lane: the tiles its triangle may shade (at most kBigTiles), in
                // registers until the warp appends them together
                uint32_t te[kBigTiles];
                uint32_t valid = 0u;
                if (act) {
                    TriT T;
                    tri_texel(J, B, lp, ls, t, T);
                    const uint32_t tplane = module_tri_plane(J, t);
                    Edges e;
                    const float xmin = fminf(T.x[0], fminf(T.x[1], T.x[2])), xmax = fmaxf(T.x[0], fmaxf(T.x[1], T.x[2]));
                    const float ymin = fminf(T.y[0], fminf(T.y[1], T.y[2])), ymax = fmaxf(T.y[0], fmaxf(T.y[1], T.y[2]));
                    // covered texel centres (ix + 0.5) lie in [xmin, xmax]
                    const int ix0 = max(0, (int)ceilf(xmin - 0.5f)), ix1 = min(R - 1, (int)floorf(xmax - 0.5f));
                    const int iy0 = max(0, (int)ceilf(ymin - 0.5f)), iy1 = min(R - 1, (int)floorf(ymax - 0.5f));
                    if (make_edges(T, e) && xmax >= 0.5f && ymax >= 0.5f && xmin <= R - 0.5f && ymin <= R - 0.5f &&
                        ix0 <= ix1 && iy0 <= iy1) {
                        const uint32_t dkey = depth_store_key(fminf(T.d[0], fminf(T.d[1], T.d[2])), lp, u24);
                        const int tx0 = ix0 >> sh, tx1 = ix1 >> sh, ty0 = iy0 >> sh, ty1 = iy1 >> sh;
                        const int wx = tx1 - tx0 + 1, ntiles = wx * (ty1 - ty0 + 1);
                        if (ntiles > kBigTiles) {
                            const unsigned int pos = atomicAdd(&B.ctr->n_big, 1u);
                            if (pos < (uint64_t)W->big_cap) B.big[pos] = make_uint2((uint32_t)t, (uint32_t)js);
                        } else {
                            int nx = tx0, ny = ty0;
    #pragma unroll
                            for (int q = 0; q < kBigTiles; ++q) {
                                te[q] = 0u;
                                if (q >= ntiles) continue;
                                const int tx = nx, ty = ny;
                                if (++nx > tx1) {
                                    nx = tx0;
                                    ++ny;
                                }
                                if (ntiles > 1 && !rect_overlap(e, tx * TS + 0.5f, tx * TS + TS - 0.5f, ty * TS + 0.5f,
                                                                ty * TS + TS - 0.5f))
                                    continue;
                                const uint32_t x = (uint32_t)(te0 + (int64_t)ty * J.tiles_x + tx);
                                // unoccupied tile (far 0) or triangle wholly behind its far plane
                                if (!(dkey < B.t_far[x])) continue;
                                // a module triangle in the plane of every receiver of the tile
                                if (tplane != kPlaneNone && B.t_plane[x] == tplane) continue;
                                atomicAdd(&B.t_cnt[x], 1u);
                                te[q] = x;
                                valid |= 1u << q;
                            }
                        }
                    }
                }
                append_pairs(B, W, te, valid, (uint32_t)t);
            }
        }
    }
}

// Triangles spanning more than kBigTiles tiles: one warp per triangle, lanes
// over its tiles.
__global__ void __launch_bounds__(256) k_bin_big(const WaveDev* __restrict__ W,
                                                 const JobDev* __restrict__ jobs, Buffers B)
{
    const unsigned int n_big = min((unsigned long long)B.ctr->n_big, (unsigned long long)W->big_cap);
    const int nj = W->n_jobs;
    const int sh = W->tile_sh;
    const int TS = 1 << sh;
    const int u24 = W->depth_u24;
    const int lane = threadIdx.x & 31;
    const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t n_warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t e = warp; e < n_big; e += n_warps) {
        uint2 en = B.big[e];
        int t = (int)en.x;
        int64_t js = en.y;
        int j = job_of(nj, js, [&](int q) { return (int64_t)jobs[q].js_base; });
        const JobDev& J = jobs[j];
        int ls = (int)(js - J.js_base);
        const LightParams lp = B.lp[js];
        TriT T;
        tri_texel(J, B, lp, ls, t, T);
        Edges ed;
        if (!make_edges(T, ed)) continue;
        const int R = J.R;
        float xmin = fminf(T.x[0], fminf(T.x[1], T.x[2])), xmax = fmaxf(T.x[0], fmaxf(T.x[1], T.x[2]));
        float ymin = fminf(T.y[0], fminf(T.y[1], T.y[2])), ymax = fmaxf(T.y[0], fmaxf(T.y[1], T.y[2]));
        int ix0 = max(0, (int)ceilf(xmin - 0.5f)), ix1 = min(R - 1, (int)floorf(xmax - 0.5f));
        int iy0 = max(0, (int)ceilf(ymin - 0.5f)), iy1 = min(R - 1, (int)floorf(ymax - 0.5f));
        if (ix0 > ix1 || iy0 > iy1) continue;
        float dmin = fminf(T.d[0], fminf(T.d[1], T.d[2]));
        uint32_t dkey = depth_store_key(dmin, lp, u24);
        const uint32_t tplane = module_tri_plane(J, t);
        int tx0 = ix0 >> sh, tx1 = ix1 >> sh, ty0 = iy0 >> sh, ty1 = iy1 >> sh;
        int wx = tx1 - tx0 + 1;
        int ntiles = wx * (ty1 - ty0 + 1);
        int64_t te0 = J.te_base + (int64_t)ls * J.tiles_x * J.tiles_x;
        for (int q0 = 0; q0 < ntiles; q0 += 32) {
            const int q = q0 + lane;
            uint32_t te[kBigTiles];
            uint32_t valid = 0u;
            te[0] = 0u;
            if (q < ntiles) {
                const int tx = tx0 + q % wx, ty = ty0 + q / wx;
                const uint32_t x = (uint32_t)(te0 + (int64_t)ty * J.tiles_x + tx);
                if (rect_overlap(ed, tx * TS + 0.5f, tx * TS + TS - 0.5f, ty * TS + 0.5f, ty * TS + TS - 0.5f) &&
                    dkey < B.t_far[x] && !(tplane != kPlaneNone && B.t_plane[x] == tplane)) {
                    atomicAdd(&B.t_cnt[x], 1u);
                    te[0] = x;
                    valid = 1u;
                }
            }
            append_pairs(B, W, te, valid, (uint32_t)t);
        }
    }
}

// After the scan: each (tile, triangle) pair to its place in the tile's bin.
__global__ void __launch_bounds__(256) k_scatter(const WaveDev* __restrict__ W, Buffers B)
{
    const unsigned long long np = min(B.ctr->n_pairs, (unsigned long long)W->bin_cap);
    const uint64_t cap = (uint64_t)W->bin_cap;
    for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < np;
         i += (unsigned long long)gridDim.x * blockDim.x) {
        const uint2 p = B.pairs[i];
        const uint32_t pos = atomicAdd(&B.t_cur[p.x], 1u);
        if (pos < cap) B.bins[pos] = p.y;
    }
}

// ---------------------------------------------------------------------------
// scan over the wave's tile entries: triangle-bin offsets, the list of
// non-empty tiles (= map slots) and receiver-list offsets of non-empty tiles
// ---------------------------------------------------------------------------
constexpr int kScanThreads = 1024;
constexpr int kScanPer = 4;
constexpr unsigned long long kFirstBins = 48;  // fused path: tiles of more triangles are taken first
constexpr int kScanTile = kScanThreads * kScanPer;

// Block-wide exclusive scan of three counters; returns the block totals.
__device__ __forceinline__ void block_scan3(unsigned long long v[3], unsigned long long tot[3])
{
    __shared__ unsigned long long ws[3][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    unsigned long long inc[3] = {v[0], v[1], v[2]};
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            unsigned long long y = __shfl_up_sync(0xffffffffu, inc[q], off);
            if (lane >= off) inc[q] += y;
        }
    }
    if (lane == 31)
        for (int q = 0; q < 3; ++q) ws[q][w] = inc[q];
    __syncthreads();
    if (w == 0) {
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            unsigned long long x = lane < nw ? ws[q][lane] : 0ull;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                unsigned long long y = __shfl_up_sync(0xffffffffu, x, off);
                if (lane >= off) x += y;
            }
            if (lane < nw) ws[q][lane] = x;
        }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        tot[q] = ws[q][nw - 1];
        v[q] = (w ? ws[q][w - 1] : 0ull) + inc[q] - v[q];
    }
    __syncthreads();
}

__device__ __forceinline__ void scan_values(const Buffers& B, int64_t i, int fused, unsigned long long v[3])
{
    const uint32_t c = B.t_cnt[i];
    v[0] = c;
    v[1] = c ? 1u : 0u;
    v[2] = c && (!fused || B.t_plane[i] == kPlaneMixed) ? B.t_rcnt[i] : 0u;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_a(const WaveDev* __restrict__ W, Buffers B)
{
    const int64_t tot = W->tot_te;
    const int64_t n_tiles = (tot + kScanTile - 1) / kScanTile;
    for (int64_t st = blockIdx.x; st < n_tiles; st += gridDim.x) {
        unsigned long long v[3] = {0, 0, 0};
        int64_t base = st * kScanTile + (int64_t)threadIdx.x * kScanPer;
#pragma unroll
        for (int q = 0; q < kScanPer; ++q) {
            if (base + q < tot) {
                unsigned long long x[3];
                scan_values(B, base + q, W->fused, x);
                v[0] += x[0]; v[1] += x[1]; v[2] += x[2];
            }
        }
        unsigned long long t[3];
        block_scan3(v, t);
        if (threadIdx.x == 0)
            for (int q = 0; q < 3; ++q) B.block_sums[3 * st + q] = t[q];
    }
}

__global__ void __launch_bounds__(kScanThreads) k_scan_b(const WaveDev* __restrict__ W, Buffers B)
{
    const int64_t tot = W->tot_te;
    const int64_t n_tiles = (tot + kScanTile - 1) / kScanTile;
    unsigned long long carry[3] = {0, 0, 0};
    for (int64_t base = 0; base < n_tiles; base += blockDim.x) {
        int64_t i = base + threadIdx.x;
        unsigned long long v[3], t[3];
        for (int q = 0; q < 3; ++q) v[q] = i < n_tiles ? B.block_sums[3 * i + q] : 0ull;
        block_scan3(v, t);
        if (i < n_tiles)
            for (int q = 0; q < 3; ++q) B.block_sums[3 * i + q] = v[q] + carry[q];
        for (int q = 0; q < 3; ++q) carry[q] += t[q];
    }
    if (threadIdx.x == 0) {
        Counters* c = B.ctr;
        c->tot_bins = carry[0];
        c->n_nonempty = (unsigned int)min(carry[1], 0xFFFFFFFFull);
        c->tot_recv = carry[2];
        c->stat_bins += carry[0];
        c->stat_nonempty += carry[1];
        if (carry[0] > c->need_bins) c->need_bins = carry[0];
        if (carry[1] > c->need_tiles) c->need_tiles = carry[1];
        if (carry[2] > c->need_recv) c->need_recv = carry[2];
        unsigned long long nb = c->n_big;
        if (nb > c->need_big) c->need_big = nb;
        if (carry[0] > (unsigned long long)W->bin_cap) c->overflow |= 1u;
        if (!W->fused && carry[1] > (unsigned long long)W->map_cap_tiles) c->overflow |= 2u;
        if (nb > (unsigned long long)W->big_cap) c->overflow |= 4u;
        if (carry[2] > (unsigned long long)W->recv_cap) c->overflow |= 8u;
    }
}

__global__ void __launch_bounds__(kScanThreads) k_scan_c(const WaveDev* __restrict__ W, Buffers B)
{
    const int64_t tot = W->tot_te;
    const int64_t n_tiles = (tot + kScanTile - 1) / kScanTile;
    const bool small = W->fused && B.ctr->n_nonempty <= kSmallWave;
    for (int64_t st = blockIdx.x; st < n_tiles; st += gridDim.x) {
        unsigned long long x[kScanPer][3];
        unsigned long long v[3] = {0, 0, 0};
        int64_t base = st * kScanTile + (int64_t)threadIdx.x * kScanPer;
#pragma unroll
        for (int q = 0; q < kScanPer; ++q) {
            if (base + q < tot) scan_values(B, base + q, W->fused, x[q]);
            else x[q][0] = x[q][1] = x[q][2] = 0ull;
            v[0] += x[q][0]; v[1] += x[q][1]; v[2] += x[q][2];
        }
        unsigned long long t[3];
        block_scan3(v, t);
        for (int q = 0; q < 3; ++q) v[q] += B.block_sums[3 * st + q];
#pragma unroll
        for (int q = 0; q < kScanPer; ++q) {
            int64_t i = base + q;
            // offsets of non-empty tiles only: every reader of t_off, t_cur,
            // t_slot, t_roff and t_rcur takes a tile from the non-empty list
            // or checks t_cnt first
            if (i < tot && x[q][1]) {
                B.t_off[i] = (uint32_t)min(v[0], 0xFFFFFFFFull);
                B.t_cur[i] = (uint32_t)min(v[0], 0xFFFFFFFFull);
                B.t_slot[i] = (uint32_t)min(v[1], 0xFFFFFFFFull);
                if (x[q][2]) {  // (fused path: t_roff of a tile of one plane group keeps its module)
                    B.t_roff[i] = (uint32_t)min(v[2], 0xFFFFFFFFull);
                    B.t_rcur[i] = (uint32_t)min(v[2], 0xFFFFFFFFull);
                }
                if (!W->fused) B.nonempty[v[1]] = (uint32_t)i;
            }
            v[0] += x[q][0]; v[1] += x[q][1]; v[2] += x[q][2];
            // fused path: tiles of many triangles from the front of the list,
            // the others from its end, so that k_tile_warp starts with the
            // long ones and the short ones fill its tail
            if (W->fused) {
                const bool ne = i < tot && x[q][1], first = ne && x[q][0] > kFirstBins;
                const unsigned int bf = __ballot_sync(0xffffffffu, first), br = __ballot_sync(0xffffffffu, ne && !first);
                const int lane = threadIdx.x & 31;
                unsigned int pos = 0;
                if (lane == 0 && bf) pos = atomicAdd(&B.ctr->n_first, (unsigned int)__popc(bf));
                if (lane == 1 && br) pos = atomicAdd(&B.ctr->n_rest, (unsigned int)__popc(br));
                const unsigned int pf = __shfl_sync(0xffffffffu, pos, 0), pr = __shfl_sync(0xffffffffu, pos, 1);
                const unsigned int below = (1u << lane) - 1u;
                if (first) B.nonempty[pf + __popc(bf & below)] = (uint32_t)i;
                else if (ne) B.nonempty[tot - 1 - (int64_t)(pr + __popc(br & below))] = (uint32_t)i;
                if (small && (bf | br)) {
#pragma unroll
                    for (int p = 0; p < kShareSteps; ++p) {
                        const unsigned int bo = __ballot_sync(0xffffffffu, ne && x[q][0] > share_bins(p));
                        if (lane == 0 && bo) atomicAdd(&B.ctr->n_over[p], (unsigned int)__popc(bo));
                    }
                }
            }
        }
    }
}

// ---------------------------------------------------------------------------
// per-tile work: receivers and the tile rasteriser (map path)
// ---------------------------------------------------------------------------
constexpr int kRecvChunk = 64;  // receivers staged in shared memory at a time (two per lane of one warp)
constexpr int kTriBatchMax = 128;  // triangles set up in shared memory at a time by the rasteriser (one per thread)
// Sub-blocks per tile side (4, 8 and 16 texels on 32-, 64- and 128-texel tiles).
template <int TS>
struct SubGrid {
    static constexpr int side = 8;
    static constexpr int blocks = side * side;
};
static_assert(kRecvChunk == 64, "receiver prefix sums take two entries per lane of one warp");

// Exclusive prefix sum of up to 64 entries, two per lane; called by one full
// warp.  Returns the total in every lane.
__device__ __forceinline__ int warp_excl_scan64(int& a0, int& a1)
{
    const int s = a0 + a1;
    const int inc = warp_incl_scan(s);
    const int ex = inc - s;
    a1 = ex + a0;
    a0 = ex;
    return __shfl_sync(0xffffffffu, inc, 31);
}

// Exclusive prefix sum of n <= 32 K entries a[0, n), K consecutive entries
// per lane of one warp, in place; a[n] receives the total.  Called by one
// full warp.
template <int K>
__device__ __forceinline__ void warp_excl_scan_k(int* a, int n)
{
    const int lane = threadIdx.x & 31;
    int v[K], sum = 0;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int i = lane * K + k;
        v[k] = i < n ? a[i] : 0;
        sum += v[k];
    }
    const int inc = warp_incl_scan(sum);
    int ex = inc - sum;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int i = lane * K + k;
        if (i < n) a[i] = ex;
        ex += v[k];
    }
    if (lane == 31) a[n] = inc;
}

// A triangle set up for one tile: edge functions, scaled depths, its texel
// box and the sub-blocks in which it may shade a sample (tri_sub_mask).  The
// rasteriser visits rows y0 .. y0 + rows - 1 of the box, one row per lane.
// 17 words: lanes reading different triangles' fields hit different banks.
struct TriSetup {
    float A[3], Bc[3], C[3];
    float e0, e1, e2;
    short x0, bw;
    int y0, rows;        // rows = 0: not kept
    uint32_t sm_lo, sm_hi;  // sub-block bits 0-31, 32-63
};
static_assert(sizeof(TriSetup) == 17 * 4, "odd word stride");

// q / d for 0 <= q < 2^24 (one float estimate, one correction).
__device__ __forceinline__ int fdiv(int q, int d, float inv_d)
{
    int r = (int)((float)q * inv_d);
    const int rem = q - r * d;
    if (rem < 0) --r;
    else if (rem >= d) ++r;
    return r;
}

// A receiver module of the tile, staged in shared memory.  Its samples that
// may read the tile form the index box [I0, I1] x [J0, J1] (I = cu * n + i,
// J = cv * n + j), walked as (sample row, cell column) items; each item's
// samples are further clipped to the row's stretch that crosses the tile.
struct RecvSm {
    ModStep s;
    float p_over_n, inv_p;     // sample spacing along the module axes (m) and its inverse
    float pa, pb, pc;          // receiver depth plane d = pa x + pb y + pc in tile-local texel coordinates
    float cull_tol;            // plane tolerance (half the bias slack), or -1 if the plane may not cull
    float cx0, cy0;            // module origin, tile-local texel coordinates
    float inv_tax, inv_tay;    // inverse texels per metre along the module's U axis (0: no row clip by it)
    float xlo, xhi, ylo, yhi;  // the tile's texel range, tile-local (open towards the map border)
    float bx0, bx1, by0, by1;  // the module's texel-space bounding box, tile-local, one texel wider
    float inv_ncol;
    int cu;                    // cells across the module
    int cell_base;             // first cell of the module in the generator
    int I0, I1, J0;            // sample-index box (J1 = J0 + rows - 1)
    int cI0, ncol;             // cell columns of the box
    int item_pref;             // (row, cell column) items of the receivers staged before this one
};

static_assert(SubGrid<32>::blocks == 64 && SubGrid<64>::blocks == 64 && SubGrid<128>::blocks == 64,
              "a triangle's sub-block set is one 64-bit mask");

// Summary of a tile's sub-block depth limits (sub_summary).
struct SubInfo {
    uint2 occ;   // sub-blocks some receiver meets
    float dlo;   // smallest limit among them
};

template <int TS>
struct TileSm {
    uint32_t tile[TS * TS];          // depth keys of the tile
    float dlim[SubGrid<TS>::blocks]; // per sub-block depth limit (sub_limits)
    SubInfo si;                      // their summary (sub_summary)
    uint32_t mask[TS * TS / 32];     // texels read by some sample (sparse tiles)
    int n_need;                      // how many (sparse tiles)
    RecvSm recv[kRecvChunk];
    int n_recv;                      // receivers staged
    int total_items;                 // (sample row, cell column) items over the staged receivers
    TriSetup tri[kTriBatchMax];      // a batch of set-up triangles, one per thread
    int row_pref[kTriBatchMax + 1];  // prefix of their rows
};

// Stage receiver module m of tile (tx, ty): sample-index box (the tile
// corners mapped back onto the module plane, widened by one sample), row
// clipping, bounding box and depth plane.  item_pref receives the receiver's
// own item count.
template <int TS>
__device__ __forceinline__ void stage_one(RecvSm& R, const JobDev& J, const Buffers& B, int ls, int tx, int ty,
                                          int m)
{
    const ModuleDev& M = J.mods[m];
    const ModStep s = B.ms[J.ms_base + (int64_t)ls * J.n_mods + m];
    const int n = J.n;
    const float X0 = (float)(tx * TS), Y0 = (float)(ty * TS);
    R.s = s;
    R.p_over_n = __fdiv_rn(M.pitch, (float)n);
    R.inv_p = 1.f / R.p_over_n;
    R.cu = M.cu;
    R.cell_base = M.cell_base;
    R.cx0 = s.tx0 - X0;
    R.cy0 = s.ty0 - Y0;
    R.inv_tax = fabsf(s.tax) > 1e-6f ? 1.f / s.tax : 0.f;
    R.inv_tay = fabsf(s.tay) > 1e-6f ? 1.f / s.tay : 0.f;
    R.xlo = tx == 0 ? -FLT_MAX : 0.f;
    R.xhi = tx == J.tiles_x - 1 ? FLT_MAX : (float)TS;
    R.ylo = ty == 0 ? -FLT_MAX : 0.f;
    R.yhi = ty == J.tiles_x - 1 ? FLT_MAX : (float)TS;
    {
        const float lu = M.cu * M.pitch, lv = M.cv * M.pitch;
        float x0 = FLT_MAX, x1 = -FLT_MAX, y0 = FLT_MAX, y1 = -FLT_MAX;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const float a = (c & 1) ? lu : 0.f, b = (c & 2) ? lv : 0.f;
            const float x = R.cx0 + a * s.tax + b * s.tbx, y = R.cy0 + a * s.tay + b * s.tby;
            x0 = fminf(x0, x); x1 = fmaxf(x1, x);
            y0 = fminf(y0, y); y1 = fmaxf(y1, y);
        }
        R.bx0 = x0 - 1.f; R.bx1 = x1 + 1.f;
        R.by0 = y0 - 1.f; R.by1 = y1 + 1.f;
    }
    int I0 = 0, I1 = M.cu * n - 1, J0 = 0, J1 = M.cv * n - 1;
    const float det = s.tax * s.tby - s.tay * s.tbx;
    const bool planar = fabsf(det) > 1e-6f * (fabsf(s.tax * s.tby) + fabsf(s.tay * s.tbx));
    R.cull_tol = -1.f;
    R.pa = R.pb = R.pc = 0.f;
    if (planar) {
        const float inv_det = 1.f / det;
        float amin = FLT_MAX, amax = -FLT_MAX, bmin = FLT_MAX, bmax = -FLT_MAX;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const float dx = ((c & 1) ? (float)TS : 0.f) - R.cx0;
            const float dy = ((c & 2) ? (float)TS : 0.f) - R.cy0;
            const float a = (dx * s.tby - dy * s.tbx) * inv_det;
            const float b = (dy * s.tax - dx * s.tay) * inv_det;
            amin = fminf(amin, a); amax = fmaxf(amax, a);
            bmin = fminf(bmin, b); bmax = fmaxf(bmax, b);
        }
        // samples at a = (I + 1/2) p/n: I in [a_min n/p - 1/2, a_max n/p - 1/2], one more each side
        I0 = max(I0, (int)fmaxf(floorf(amin * R.inv_p - 0.5f) - 1.f, -1.f));
        I1 = min(I1, (int)fminf(ceilf(amax * R.inv_p - 0.5f) + 1.f, 1e6f));
        J0 = max(J0, (int)fmaxf(floorf(bmin * R.inv_p - 0.5f) - 1.f, -1.f));
        J1 = min(J1, (int)fminf(ceilf(bmax * R.inv_p - 0.5f) + 1.f, 1e6f));
        // depth of the receiver plane over the tile: a triangle lying on or
        // behind the plane (by less than half the bias slack) shades none
        // of its samples, so it may be skipped for this receiver
        R.pa = (s.da * s.tby - s.db * s.tay) * inv_det;
        R.pb = (s.db * s.tax - s.da * s.tbx) * inv_det;
        R.pc = s.d0 - R.pa * R.cx0 - R.pb * R.cy0;
        if (s.cosi > 0.017452406f) R.cull_tol = B.lp[J.js_base + ls].delta * (1.f / 64.f);
    }
    R.I0 = I0;
    R.I1 = I1;
    R.J0 = J0;
    R.cI0 = I0 / n;
    R.ncol = (I0 <= I1) ? I1 / n - I0 / n + 1 : 0;
    R.inv_ncol = 1.f / (float)max(R.ncol, 1);
    R.item_pref = (I0 <= I1 && J0 <= J1) ? R.ncol * (J1 - J0 + 1) : 0;  // prefixed by the caller
}

// Stage receivers [r0, r0 + cnt) of tile (tx, ty) for the whole block (cnt <=
// kRecvChunk), with their item prefixes.
template <int TS>
__device__ void stage_receivers(TileSm<TS>& sm, const JobDev& J, const Buffers& B, int ls, int tx, int ty,
                                uint64_t r0, int cnt)
{
    const int tid = threadIdx.x;
    if (tid < cnt) stage_one<TS>(sm.recv[tid], J, B, ls, tx, ty, (int)B.recv[r0 + tid]);
    __syncthreads();
    if (tid < 32) {
        const int q0 = 2 * tid, q1 = q0 + 1;
        int i0 = q0 < cnt ? sm.recv[q0].item_pref : 0, i1 = q1 < cnt ? sm.recv[q1].item_pref : 0;
        const int ti = warp_excl_scan64(i0, i1);
        if (q0 < cnt) sm.recv[q0].item_pref = i0;
        if (q1 < cnt) sm.recv[q1].item_pref = i1;
        if (tid == 0) {
            sm.n_recv = cnt;
            sm.total_items = ti;
        }
    }
    __syncthreads();
}

// Receiver of staged item `it` (items prefixed in item_pref).
__device__ __forceinline__ int recv_of_item(const RecvSm* recv, int n_recv, int it)
{
    int lo = 0, hi = n_recv - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (recv[mid].item_pref <= it) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// Clip [Ib, Ie] to the samples of row Jr whose texel may lie in the tile:
// the stretch of the row's line a -> (cx0 + a tax + b tbx, cy0 + a tay + b tby)
// inside the tile's texel range, widened by one sample each side (the exact
// test is the caller's, per sample).
__device__ __forceinline__ void row_range(const RecvSm& R, int Jr, int& Ib, int& Ie)
{
    const float b = __fmul_rn(__fadd_rn((float)Jr, 0.5f), R.p_over_n);
    float amin = -FLT_MAX, amax = FLT_MAX;
    if (R.inv_tax != 0.f) {
        const float c = fmaf(b, R.s.tbx, R.cx0);
        const float a0 = (R.xlo - c) * R.inv_tax, a1 = (R.xhi - c) * R.inv_tax;
        amin = fminf(a0, a1);
        amax = fmaxf(a0, a1);
    }
    if (R.inv_tay != 0.f) {
        const float c = fmaf(b, R.s.tby, R.cy0);
        const float a0 = (R.ylo - c) * R.inv_tay, a1 = (R.yhi - c) * R.inv_tay;
        amin = fmaxf(amin, fminf(a0, a1));
        amax = fminf(amax, fmaxf(a0, a1));
    }
    const float lo = floorf(amin * R.inv_p - 0.5f) - 1.f, hi = ceilf(amax * R.inv_p - 0.5f) + 1.f;
    Ib = max(Ib, (int)fminf(fmaxf(lo, -1.f), 1e7f));
    Ie = min(Ie, (int)fmaxf(fminf(hi, 1e7f), -2.f));
}

// Decode staged item `it`: receiver, sample row Jr, cell (cu, cv), row jj
// within the cell and the item's sample range [Ib, Ie].
__device__ __forceinline__ const RecvSm& decode_item(const RecvSm* recv, int n_recv, int it, int n, float inv_n,
                                                     int& Jr, int& cu, int& cv, int& jj, int& Ib, int& Ie)
{
    const RecvSm& R = recv[recv_of_item(recv, n_recv, it)];
    const int q = it - R.item_pref;
    const int row = fdiv(q, R.ncol, R.inv_ncol);
    cu = R.cI0 + q - row * R.ncol;
    Jr = R.J0 + row;
    cv = fdiv(Jr, n, inv_n);
    jj = Jr - cv * n;
    Ib = max(R.I0, cu * n);
    Ie = min(R.I1, cu * n + n - 1);
    row_range(R, Jr, Ib, Ie);
    return R;
}

// Visit the samples of the staged receivers that read tile (tx, ty): one
// thread per (sample row, cell column) item walks the row's samples inside
// the cell, the box and the row's stretch over the tile.  f(R, k, ix, iy, d)
// is called per sample inside the tile (k = j * n + i within the cell);
// g(R, cu, cv) after each item.
template <int TS, bool PROF, typename F, typename G>
__device__ __forceinline__ void for_tile_samples(const RecvSm* recv, int n_recv, int total_items, const JobDev& J,
                                                 int tx, int ty, int it_begin, int it_stride, unsigned int& cand,
                                                 F f, G g)
{
    constexpr int SH = TS == 128 ? 7 : (TS == 64 ? 6 : 5);
    const int n = J.n;
    const float r_max = (float)(J.R - 1);
    const float inv_n = 1.f / (float)n;
    for (int it = it_begin; it < total_items; it += it_stride) {
        int Jr, cu, cv, jj, Ib, Ie;
        const RecvSm& R = decode_item(recv, n_recv, it, n, inv_n, Jr, cu, cv, jj, Ib, Ie);
        if (PROF) cand += (unsigned int)max(0, Ie - Ib + 1);
        const SampleRow row = sample_row(R.s, Jr, R.p_over_n);
        float ih = (float)Ib + 0.5f;
        for (int I = Ib; I <= Ie; ++I, ih += 1.f) {
            float d;
            int ix, iy;
            sample_texel(R.s, row, ih, R.p_over_n, r_max, ix, iy, d);
            if ((ix >> SH) == tx && (iy >> SH) == ty) f(R, jj * n + (I - cu * n), ix, iy, d);
        }
        g(R, cu, cv);
    }
}

// Can triangle T (tile-local texel coordinates) shade a sample of a staged
// receiver?  False only if it lies on or behind every receiver's plane.
__device__ __forceinline__ bool may_shade(const RecvSm* recv, int n_recv, const TriT& T, bool cull_ok)
{
    if (!cull_ok) return true;
    for (int r = 0; r < n_recv; ++r) {
        const RecvSm& R = recv[r];
        if (R.cull_tol < 0.f) return true;
        float gap = FLT_MAX;
#pragma unroll
        for (int k = 0; k < 3; ++k) gap = fminf(gap, T.d[k] - (R.pa * T.x[k] + R.pb * T.y[k] + R.pc));
        if (!(gap >= -R.cull_tol)) return true;
    }
    return false;
}

// Tile-local texel-centre range [x0, x1] x [y0, y1] of a triangle's bounding box.
template <int TS>
__device__ __forceinline__ bool tri_box(const TriT& T, int& x0, int& x1, int& y0, int& y1)
{
    const float xmin = fminf(T.x[0], fminf(T.x[1], T.x[2])), xmax = fmaxf(T.x[0], fmaxf(T.x[1], T.x[2]));
    const float ymin = fminf(T.y[0], fminf(T.y[1], T.y[2])), ymax = fmaxf(T.y[0], fmaxf(T.y[1], T.y[2]));
    x0 = max(0, (int)ceilf(xmin - 0.5f));
    x1 = min(TS - 1, (int)floorf(xmax - 0.5f));
    y0 = max(0, (int)ceilf(ymin - 0.5f));
    y1 = min(TS - 1, (int)floorf(ymax - 0.5f));
    return x0 <= x1 && y0 <= y1;
}

// Summary of a tile's sub-block depth limits, for tri_sub_mask's fast path:
// the sub-blocks that any receiver meets (limit above -inf) and the smallest
// limit among them.  Called by one full warp once the limits are written.
__device__ __forceinline__ SubInfo sub_summary(const float* dlim)
{
    const int lane = threadIdx.x & 31;
    const float a = dlim[lane], b = dlim[lane + 32];
    SubInfo si;
    si.occ.x = __ballot_sync(0xffffffffu, a > -FLT_MAX);
    si.occ.y = __ballot_sync(0xffffffffu, b > -FLT_MAX);
    float lo = fminf(a > -FLT_MAX ? a : FLT_MAX, b > -FLT_MAX ? b : FLT_MAX);
#pragma unroll
    for (int off = 16; off; off >>= 1) lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, off));
    si.dlo = lo;
    return si;
}

// The sub-blocks of the tile in which a set-up triangle may shade a sample
// (bit sb = sy * side + sx): its nearest vertex is nearer than the
// sub-block's depth limit, and each edge function is non-negative at the
// texel centre of (its texel box within the sub-block) farthest inside the
// edge -- exact, since edge_at is monotone in px and py, so a texel centre
// of the sub-block that the triangle covers implies a non-negative value
// there.  Row by row of sub-blocks: when every edge is non-negative at the
// row's corner farthest outside it, the triangle covers every texel centre
// of its box in that row, and when its nearest vertex is also nearer than the
// tile's smallest limit, the row's bits are the occupied sub-blocks of the
// box's columns.  A triangle with no such sub-block cannot shade any sample
// of the tile and is not kept.
template <int TS>
__device__ __forceinline__ uint64_t tri_sub_mask(const Edges& ed, int x0, int x1, int y0, int y1, float dmin,
                                                 const float* dlim, const SubInfo& si)
{
    constexpr int kSubSide = SubGrid<TS>::side;
    constexpr int SW = TS / kSubSide;  // sub-block side, texels
    static_assert(kSubSide == 8, "a row of sub-blocks is one byte of the mask");
    const uint64_t occ = (uint64_t)si.occ.x | ((uint64_t)si.occ.y << 32);
    const int sx0 = x0 / SW, sx1 = x1 / SW;
    const uint64_t cols = (uint64_t)((2u << sx1) - (1u << sx0));  // bits sx0..sx1 of a row
    const bool near_all = dmin < si.dlo;
    const float fxl = texel_centre(x0), fxh = texel_centre(x1);
    uint64_t m = 0ull;
    for (int sy = y0 / SW; sy <= y1 / SW; ++sy) {
        const float fy0 = texel_centre(max(y0, sy * SW)), fy1 = texel_centre(min(y1, sy * SW + SW - 1));
        float t[3];
        bool full = true;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            t[k] = __fmaf_rn(ed.Bc[k], ed.Bc[k] > 0.f ? fy1 : fy0, ed.C[k]);
            full = full && edge_at(ed.A[k], ed.Bc[k], ed.C[k], ed.A[k] > 0.f ? fxl : fxh,
                                   ed.Bc[k] > 0.f ? fy0 : fy1) >= 0.f;
        }
        const uint64_t row = (cols << (8 * sy)) & occ;
        if (full && near_all) {
            m |= row;
            continue;
        }
        for (uint64_t r = row; r; r &= r - 1ull) {
            const int sb = __ffsll((long long)r) - 1;
            if (!(dmin < dlim[sb])) continue;
            if (!full) {
                const int sx = sb & 7;
                const float fx0 = texel_centre(max(x0, sx * SW)), fx1 = texel_centre(min(x1, sx * SW + SW - 1));
                bool in = true;
#pragma unroll
                for (int k = 0; k < 3; ++k) in = in && __fmaf_rn(ed.A[k], ed.A[k] > 0.f ? fx1 : fx0, t[k]) >= 0.f;
                if (!in) continue;
            }
            m |= 1ull << sb;
        }
    }
    return m;
}

// Per sub-block, the depth below which a triangle must reach to shade one of
// its samples: the largest over the receivers whose box meets the sub-block
// of (receiver plane over the sub-block - bias), plus twice the plane
// tolerance and, for 24-bit depth, the one-step truncation of the stored
// key.  A sample at depth d is shaded only by a surface nearer than d - bias
// (less the truncation), and interpolated depths inside a triangle are no
// nearer than its nearest vertex (up to rounding, which the tolerance
// covers).  A sub-block with a receiver whose plane may not cull gets no
// limit; one that no receiver meets gets -inf.  Entries sb = q_begin,
// q_begin + q_stride, ... are written.
template <int TS>
__device__ __forceinline__ void sub_limits(const RecvSm* recv, int n_recv, float* dlim, float q1, int q_begin,
                                           int q_stride)
{
    constexpr int kSubSide = SubGrid<TS>::side, kSubBlocks = SubGrid<TS>::blocks;
    constexpr int SW = TS / kSubSide;
    for (int sb = q_begin; sb < kSubBlocks; sb += q_stride) {
        const float x0 = (float)((sb % kSubSide) * SW), x1 = x0 + (float)SW;
        const float y0 = (float)((sb / kSubSide) * SW), y1 = y0 + (float)SW;
        float lim = -FLT_MAX;
        for (int r = 0; r < n_recv; ++r) {
            const RecvSm& R = recv[r];
            if (R.bx1 < x0 || R.bx0 > x1 || R.by1 < y0 || R.by0 > y1) continue;
            if (R.cull_tol < 0.f) { lim = FLT_MAX; break; }
            const float pm = R.pc + fmaxf(R.pa * x0, R.pa * x1) + fmaxf(R.pb * y0, R.pb * y1);
            lim = fmaxf(lim, pm - R.s.bias + 2.f * R.cull_tol + q1);
        }
        dlim[sb] = lim;
    }
}

// ---- tile rasteriser ------------------------------------------------------

// Narrow the texel range [lo, hi] of a row to the texels whose centre px
// has fma(A, px, t) >= 0 -- edge_at on that row, which is monotone in px,
// so the texels form an interval: an estimate of its end from the edge's
// root, corrected by evaluating the edge exactly as the per-texel test does
// (at most the range's width of steps, one or two in practice).
__device__ __forceinline__ void edge_span(float A, float t, int& lo, int& hi)
{
    if (lo > hi) return;
    if (A > 0.f) {
        const float f = ceilf(__fdividef(-t, A) - 0.5f);
        int i = (int)fminf(fmaxf(f, (float)lo), (float)(hi + 1));
        while (i > lo && __fmaf_rn(A, (float)(i - 1) + 0.5f, t) >= 0.f) --i;
        while (i <= hi && __fmaf_rn(A, (float)i + 0.5f, t) < 0.f) ++i;
        lo = i;
    } else if (A < 0.f) {
        const float f = floorf(__fdividef(-t, A) - 0.5f);
        int i = (int)fminf(fmaxf(f, (float)(lo - 1)), (float)hi);
        while (i < hi && __fmaf_rn(A, (float)(i + 1) + 0.5f, t) >= 0.f) ++i;
        while (i >= lo && __fmaf_rn(A, (float)i + 0.5f, t) < 0.f) --i;
        hi = i;
    } else if (!(t >= 0.f)) {
        hi = lo - 1;  // fma(0, px, t) = t for every texel of the row
    }
}

// Bits of the texels lo .. hi (tile-local) that fall in word w of a row.
__device__ __forceinline__ uint32_t span_word(int lo, int hi, int w)
{
    const int a = max(lo - 32 * w, 0), b = min(hi - 32 * w, 31);
    return b < a ? 0u : (0xFFFFFFFFu >> (31 - b)) & (0xFFFFFFFFu << a);
}

// Texel bits of word w of a row from the row's byte of sub-block bits (bit
// sx covers texels sx * TS / 8 .. sx * TS / 8 + TS / 8 - 1).
template <int TS>
__device__ __forceinline__ uint32_t sub_word(uint32_t sbyte, int w)
{
    if constexpr (TS == 32) {
        uint32_t x = sbyte;  // bit i -> bit 4 i, then a nibble each
        x = (x | (x << 12)) & 0x000F000Fu;
        x = (x | (x << 6)) & 0x03030303u;
        x = (x | (x << 3)) & 0x11111111u;
        return x * 0xFu;
    } else if constexpr (TS == 64) {
        uint32_t x = (sbyte >> (4 * w)) & 0xFu;  // bit i -> bit 8 i, then a byte each
        x = (x | (x << 14)) & 0x00030003u;
        x = (x | (x << 7)) & 0x01010101u;
        return x * 0xFFu;
    } else {
        uint32_t x = (sbyte >> (2 * w)) & 0x3u;  // bit i -> bit 16 i, then a half-word each
        x = (x | (x << 15)) & 0x00010001u;
        return x * 0xFFFFu;
    }
}

// Set up binned triangle t of tile (ox, oy) for the rasteriser in S and
// return its rows: 0 (not kept) if it lies behind every staged receiver's
// plane, covers no texel centre of the tile, or may shade no sample of any
// sub-block (tri_sub_mask with the sub-block depth limits dlim).
template <int TS, bool PROF>
__device__ __forceinline__ int setup_raster_tri(const JobDev& J, const Buffers& B, const LightParams& lp, int ls,
                                                int t, float ox, float oy, const RecvSm* recv, int n_recv,
                                                bool cull_ok, const float* dlim, const SubInfo& si, TriSetup& S,
                                                unsigned int& culled)
{
    constexpr int SWS = (TS == 128 ? 7 : (TS == 64 ? 6 : 5)) - 3;  // log2 of the sub-block side
    TriT T;
    tri_texel(J, B, lp, ls, t, T);
#pragma unroll
    for (int k = 0; k < 3; ++k) { T.x[k] -= ox; T.y[k] -= oy; }
    if (!may_shade(recv, n_recv, T, cull_ok)) {
        if (PROF) ++culled;
        return 0;
    }
    Edges ed;
    int x0, x1, y0, y1;
    if (!make_edges(T, ed) || !tri_box<TS>(T, x0, x1, y0, y1)) return 0;
    const uint64_t sb = tri_sub_mask<TS>(ed, x0, x1, y0, y1, fminf(T.d[0], fminf(T.d[1], T.d[2])), dlim, si);
    if (sb == 0ull) return 0;
    const float inv_a = 1.f / ed.area2;
#pragma unroll
    for (int k = 0; k < 3; ++k) { S.A[k] = ed.A[k]; S.Bc[k] = ed.Bc[k]; S.C[k] = ed.C[k]; }
    S.e0 = T.d[0] * inv_a; S.e1 = T.d[1] * inv_a; S.e2 = T.d[2] * inv_a;
    S.sm_lo = (uint32_t)sb;
    S.sm_hi = (uint32_t)(sb >> 32);
    S.x0 = (short)x0; S.bw = (short)(x1 - x0 + 1);
    // the box's rows within the sub-block rows it may shade
    const int sy0 = (__ffsll((long long)sb) - 1) >> 3, sy1 = (63 - __clzll((long long)sb)) >> 3;
    const int ry0 = max(y0, sy0 << SWS), ry1 = min(y1, (sy1 << SWS) + (1 << SWS) - 1);
    S.y0 = ry0;
    S.rows = ry1 - ry0 + 1;
    return S.rows;
}

// Draw rows [u_beg, u_end) of set-up triangles tri[0, nb) (rows prefixed in
// row_pref) into the depth tile, 32 at a time, one (triangle, row) per lane
// of the calling warp: the row's texels inside all three edges, exactly
// (edge_at on a row is fma(A, px, t_k), monotone in px: edge_span), within
// the triangle's sub-blocks and, unless mask is null, marked in mask.
template <int TS, bool PROF>
__device__ __forceinline__ void draw_rows(const TriSetup* tri, const int* row_pref, int nb, int u_beg, int u_end,
                                          const uint32_t* mask, uint32_t* tile, const LightParams& lp, int u24,
                                          unsigned int& visits, unsigned int& writes)
{
    constexpr int WPR = TS / 32;
    constexpr int SWS = (TS == 128 ? 7 : (TS == 64 ? 6 : 5)) - 3;
    const int lane = threadIdx.x & 31;
    // a lane finds its triangle by walking forward from the last
    int t = 0;
    {
        int lo = 0, hi = nb - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (row_pref[mid] <= u_beg) lo = mid; else hi = mid - 1;
        }
        t = lo;
    }
    for (int ub = u_beg; ub < u_end; ub += 32) {
        const int u = ub + lane;
        if (u >= u_end) break;
        while (row_pref[t + 1] <= u) ++t;
        const TriSetup& S = tri[t];
        const int iy = S.y0 + (u - row_pref[t]);
        const int sy = iy >> SWS;
        const uint32_t sbyte = ((sy < 4 ? S.sm_lo : S.sm_hi) >> ((sy & 3) << 3)) & 0xFFu;
        if (sbyte == 0u) continue;
        if (mask) {
            uint32_t any = 0u;
#pragma unroll
            for (int w = 0; w < WPR; ++w) any |= mask[iy * WPR + w];
            if (any == 0u) continue;
        }
        const float py = (float)iy + 0.5f;
        const float A0 = S.A[0], A1 = S.A[1], A2 = S.A[2];
        const float t0 = __fmaf_rn(S.Bc[0], py, S.C[0]);
        const float t1 = __fmaf_rn(S.Bc[1], py, S.C[1]);
        const float t2 = __fmaf_rn(S.Bc[2], py, S.C[2]);
        int lo = S.x0, hi = S.x0 + S.bw - 1;
        edge_span(A0, t0, lo, hi);
        edge_span(A1, t1, lo, hi);
        edge_span(A2, t2, lo, hi);
        if (lo > hi) continue;
        const float e0 = S.e0, e1 = S.e1, e2 = S.e2;
        for (int w = lo >> 5; w <= (hi >> 5); ++w) {
            uint32_t bits = span_word(lo, hi, w) & sub_word<TS>(sbyte, w);
            if (mask) bits &= mask[iy * WPR + w];
            while (bits) {
                const int ix = (w << 5) + __ffs(bits) - 1;
                bits &= bits - 1u;
                const float px = (float)ix + 0.5f;
                const float w0 = __fmaf_rn(A0, px, t0);
                const float w1 = __fmaf_rn(A1, px, t1);
                const float w2 = __fmaf_rn(A2, px, t2);
                atomicMin(&tile[iy * TS + ix], depth_store_key(depth_at(w0, w1, w2, e0, e1, e2), lp, u24));
                if (PROF) { ++visits; ++writes; }
            }
        }
    }
}

// The tile's sub-block depth limits (sub_limits, or no limit when the
// receivers are staged in chunks) and their summary, for the whole block.
template <int TS>
__device__ __forceinline__ void tile_limits(TileSm<TS>& sm, const LightParams& lp, int u24, bool cull_ok)
{
    const int tid = threadIdx.x, bd = blockDim.x;
    if (cull_ok) sub_limits<TS>(sm.recv, sm.n_recv, sm.dlim, u24 ? 1.f / lp.qscale : 0.f, tid, bd);
    else
        for (int q = tid; q < SubGrid<TS>::blocks; q += bd) sm.dlim[q] = FLT_MAX;
    __syncthreads();
    if (tid < 32) {
        const SubInfo si = sub_summary(sm.dlim);
        if (tid == 0) sm.si = si;
    }
    __syncthreads();
}

// Rasterise the tile's triangles into sm.tile.  Sparse tiles (fewer samples
// than two per texel) are rasterised only at the texels their samples read.
// A triangle is drawn only in the sub-blocks where it may shade a sample
// (tri_sub_mask with the sub-block depth limits): the stored nearest depth
// may then differ at a texel, but never the decision of a sample there (the
// dropped triangles are behind every sample they cover, and "shaded" is
// "some covering triangle is nearer than the sample less its bias").  Each
// (triangle, row) goes to one lane, which visits only the texels of the row
// inside all three edges (edge_span), of the triangle's sub-blocks and, in
// sparse tiles, marked.  Receivers [r0, r0 + nrecv) must be staged (the
// first kRecvChunk of them) on entry.
template <int TS, bool PROF>
__device__ void tile_raster(TileSm<TS>& sm, const JobDev& J, const Buffers& B, const WaveDev* W, int ls, int tx,
                           int ty, int64_t te, uint64_t r0, int nrecv, unsigned int& visits,
                           unsigned int& writes, unsigned int& culled, unsigned int& cand, unsigned int& dense_n)
{
    constexpr int WPR = TS / 32;
    static_assert(SubGrid<TS>::side == 8, "sub-block index by shifts");
    const int tid = threadIdx.x, bd = blockDim.x;
    const int warp = tid >> 5, n_warps = bd >> 5;
    const int u24 = W->depth_u24;
    const LightParams& lp = B.lp[J.js_base + ls];
    const bool cull_ok = nrecv <= kRecvChunk;
    // samples reading the tile, at most (estimated from the staged receivers)
    const int64_t est = (int64_t)sm.total_items * J.n * ((nrecv + kRecvChunk - 1) / kRecvChunk);
    // dense only when the samples clearly outnumber the texels: marking costs
    // about as much per sample as a texel visit, and sparse tiles visit only
    // the texels that samples read
    const bool dense = est >= 2 * TS * TS;
    if (PROF && threadIdx.x == 0 && dense) ++dense_n;
    tile_limits<TS>(sm, lp, u24, cull_ok);
    int n_need = TS * TS;
    if (!dense) {
        for (int q = tid; q < TS * WPR; q += bd) sm.mask[q] = 0u;
        __syncthreads();
        for (int c0 = 0; c0 < nrecv; c0 += kRecvChunk) {
            if (c0 > 0) stage_receivers<TS>(sm, J, B, ls, tx, ty, r0 + c0, min(kRecvChunk, nrecv - c0));
            for_tile_samples<TS, PROF>(
                sm.recv, sm.n_recv, sm.total_items, J, tx, ty, threadIdx.x, blockDim.x, cand,
                [&](const RecvSm&, int, int ix, int iy, float) {
                    atomicOr(&sm.mask[(iy & (TS - 1)) * WPR + ((ix & (TS - 1)) >> 5)], 1u << (ix & 31));
                },
                [&](const RecvSm&, int, int) {});
            __syncthreads();
        }
        if (nrecv > kRecvChunk) stage_receivers<TS>(sm, J, B, ls, tx, ty, r0, kRecvChunk);
        if (tid < 32) {
            unsigned int c = 0;
            for (int q = tid; q < TS * WPR; q += 32) c += __popc(sm.mask[q]);
            c = __reduce_add_sync(0xffffffffu, c);
            if (tid == 0) sm.n_need = (int)c;
        }
        __syncthreads();
        n_need = sm.n_need;
    }
    uint4* t4 = reinterpret_cast<uint4*>(sm.tile);
    for (int q = tid; q < TS * TS / 4; q += bd) t4[q] = make_uint4(kEmpty, kEmpty, kEmpty, kEmpty);
    __syncthreads();
    if (n_need == 0) return;
    const float ox = (float)(tx * TS), oy = (float)(ty * TS);
    const uint64_t off = B.t_off[te];
    uint64_t cnt = B.t_cnt[te];
    const uint64_t cap = (uint64_t)W->bin_cap;
    if (off + cnt > cap) cnt = off < cap ? cap - off : 0;
    // triangles in batches of one per thread (at most kTriBatchMax): set-up,
    // then all warps share the batch's rows, one (triangle, row) per lane
    const int batch = min(bd, kTriBatchMax);
    for (uint64_t b0 = 0; b0 < cnt; b0 += batch) {
        const int nb = (int)min((uint64_t)batch, cnt - b0);
        if (tid < nb)
            sm.row_pref[tid] = setup_raster_tri<TS, PROF>(J, B, lp, ls, (int)B.bins[off + b0 + tid], ox, oy, sm.recv,
                                                          sm.n_recv, cull_ok, sm.dlim, sm.si, sm.tri[tid], culled);
        __syncthreads();
        if (tid < 32) warp_excl_scan_k<kTriBatchMax / 32>(sm.row_pref, nb);
        __syncthreads();
        // each warp takes a contiguous range of the batch's rows
        const int n_rows = sm.row_pref[nb];
        draw_rows<TS, PROF>(sm.tri, sm.row_pref, nb, (int)(((int64_t)n_rows * warp) / n_warps),
                            (int)(((int64_t)n_rows * (warp + 1)) / n_warps), dense ? nullptr : sm.mask, sm.tile,
                            lp, u24, visits, writes);
        __syncthreads();
    }
}
// Add per-thread work counters to the global profile counters (warp-reduced).
__device__ __forceinline__ void flush_profile(const Buffers& B, unsigned int samples, unsigned int visits,
                                              unsigned int writes, unsigned int culled)
{
#pragma unroll
    for (int off = 16; off; off >>= 1) {
        samples += __shfl_xor_sync(0xffffffffu, samples, off);
        visits += __shfl_xor_sync(0xffffffffu, visits, off);
        writes += __shfl_xor_sync(0xffffffffu, writes, off);
        culled += __shfl_xor_sync(0xffffffffu, culled, off);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&B.ctr->prof_samples, (unsigned long long)samples);
        atomicAdd(&B.ctr->prof_visits, (unsigned long long)visits);
        atomicAdd(&B.ctr->prof_writes, (unsigned long long)writes);
        atomicAdd(&B.ctr->prof_culled, (unsigned long long)culled);
    }
}

__device__ __forceinline__ void flush_profile2(const Buffers& B, unsigned int cand, unsigned int tiles,
                                               unsigned int dense, unsigned int stiles, unsigned int pairs)
{
#pragma unroll
    for (int off = 16; off; off >>= 1) {
        cand += __shfl_xor_sync(0xffffffffu, cand, off);
        tiles += __shfl_xor_sync(0xffffffffu, tiles, off);
        dense += __shfl_xor_sync(0xffffffffu, dense, off);
        stiles += __shfl_xor_sync(0xffffffffu, stiles, off);
        pairs += __shfl_xor_sync(0xffffffffu, pairs, off);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&B.ctr->prof_cand, (unsigned long long)cand);
        atomicAdd(&B.ctr->prof_tiles, (unsigned long long)tiles);
        atomicAdd(&B.ctr->prof_dense, (unsigned long long)dense);
        atomicAdd(&B.ctr->prof_stiles, (unsigned long long)stiles);
        atomicAdd(&B.ctr->prof_pairs, (unsigned long long)pairs);
    }
}

// The heavy-tile kernel's share of the work counters (also in the totals).
__device__ __forceinline__ void flush_heavy(const Buffers& B, unsigned int samples, unsigned int writes,
                                            unsigned int tiles)
{
#pragma unroll
    for (int off = 16; off; off >>= 1) {
        samples += __shfl_xor_sync(0xffffffffu, samples, off);
        writes += __shfl_xor_sync(0xffffffffu, writes, off);
        tiles += __shfl_xor_sync(0xffffffffu, tiles, off);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&B.ctr->prof_h_samples, (unsigned long long)samples);
        atomicAdd(&B.ctr->prof_h_writes, (unsigned long long)writes);
        atomicAdd(&B.ctr->prof_h_tiles, (unsigned long long)tiles);
    }
}

// Decode a non-empty tile entry.
__device__ __forceinline__ void decode_tile(const JobDev* jobs, int nj, uint32_t te, int& j, int& ls, int& tx,
                                            int& ty)
{
    j = job_of(nj, te, [&](int q) { return jobs[q].te_base; });
    const JobDev& J = jobs[j];
    const uint32_t lte = (uint32_t)(te - J.te_base);  // tile entries of a wave are numbered in 32 bits
    const uint32_t tps = (uint32_t)(J.tiles_x * J.tiles_x);
    ls = (int)(lte / tps);
    const uint32_t tl = lte - (uint32_t)ls * tps;
    ty = (int)(tl / (uint32_t)J.tiles_x);
    tx = (int)(tl - (uint32_t)ty * (uint32_t)J.tiles_x);
}

// Receivers of a tile entry, clamped to the receiver pool.
__device__ __forceinline__ void tile_receivers(const Buffers& B, const WaveDev* W, int64_t te, uint64_t& r0, int& n)
{
    r0 = B.t_roff[te];
    uint64_t r1 = r0 + B.t_rcnt[te];
    if (r1 > (uint64_t)W->recv_cap) r1 = (uint64_t)W->recv_cap;
    n = r1 > r0 ? (int)(r1 - r0) : 0;
}

// ---------------------------------------------------------------------------
// k_raster_map: map path -- rasterise the tile and store it in HBM for the
// gather kernel (coalesced 16-byte stores)
// ---------------------------------------------------------------------------
template <int TS, bool PROF>
__global__ void __launch_bounds__(256) k_raster_map(const WaveDev* __restrict__ W,
                                                    const JobDev* __restrict__ jobs, Buffers B)
{
    extern __shared__ __align__(16) unsigned char tile_smem[];  // sizeof(TileSm<TS>), set at launch
    TileSm<TS>& sm = *reinterpret_cast<TileSm<TS>*>(tile_smem);
    unsigned int p_visits = 0, p_writes = 0, p_culled = 0, p_cand = 0, p_dense = 0;
    __shared__ unsigned int s_item;
    // incomplete bins (pool overflow, the wave is rerun): nothing to read
    const unsigned int n_ne = (B.ctr->overflow & 1u) ? 0u : B.ctr->n_nonempty;
    const int64_t map_cap = W->map_cap_tiles;
    const int nj = W->n_jobs;
    const int tid = threadIdx.x, bd = blockDim.x;
    for (;;) {
        if (tid == 0) s_item = atomicAdd(&B.ctr->raster_next, 1u);
        __syncthreads();
        const unsigned int item = s_item;
        __syncthreads();
        if (item >= n_ne || item >= map_cap) break;
        const uint32_t te = B.nonempty[item];
        int j, ls, tx, ty;
        decode_tile(jobs, nj, te, j, ls, tx, ty);
        const JobDev& J = jobs[j];
        uint64_t r0;
        int nrecv;
        tile_receivers(B, W, te, r0, nrecv);
        stage_receivers<TS>(sm, J, B, ls, tx, ty, r0, min(nrecv, kRecvChunk));
        // the tile is stored even when nothing was drawn: its samples read it
        tile_raster<TS, PROF>(sm, J, B, W, ls, tx, ty, te, r0, nrecv, p_visits, p_writes, p_culled, p_cand,
                              p_dense);
        const uint4* t4 = reinterpret_cast<const uint4*>(sm.tile);
        uint4* dst = reinterpret_cast<uint4*>(B.map + ((size_t)item * (TS * TS)));
        for (int q = tid; q < TS * TS / 4; q += bd) dst[q] = t4[q];
        __syncthreads();
    }
    if (PROF) {
        flush_profile(B, 0u, p_visits, p_writes, p_culled);
        flush_profile2(B, p_cand, 0u, p_dense, 0u, 0u);
    }
}

// ---------------------------------------------------------------------------
// fused path: coverage of a tile's texels, and the samples that look it up
//
// A sample is shaded iff some triangle covers its texel's centre at a depth
// that the sample, less its bias, is behind.  The samples of the modules of
// one plane (a tracker's table, a facade) lie on that plane, so at a texel a
// triangle is in front of all of them, behind all of them, or in a thin band
// about the plane (the plane's slope over the texel and rounding) where each
// sample must compare depths.  A tile therefore keeps one bit per texel and
// plane: covered by something in front of the plane.  Triangles wholly in
// front of a plane set whole row spans, those wholly behind are dropped, and
// only those that cross the plane's band in the tile compare depths, texel by
// texel; texels in the band are "open", and the few samples that read them
// test the triangles there one by one (or the tile's nearest depth).  The
// decisions are those of a depth map, sample by sample.
//
// The kernels of this path are bound by instruction issue and fetch (a tile
// runs a few thousand instructions of straight-line code, and the warps of an
// SM are all at different places in it), so the code is kept small: one copy
// of each loop, none unrolled that is not short and hot.
// ---------------------------------------------------------------------------

// Planes that a warp of k_tile_warp keeps bits of; tiles of more go to
// k_raster_test.  The less shared memory a warp takes, the more of them an SM
// holds.
template <int TS>
struct WarpLevels {
    static constexpr int n = TS == 32 ? 12 : (TS == 64 ? 8 : 1);
};

// Planes that k_raster_test keeps bits of at a time (its blocks an SM stay
// what they are without), and in all: a tile of more of them has them drawn in
// turns.  In a tile of more than kMaxLevels the last of a single turn stands
// for every plane without bits of its own.
template <int TS>
struct PassLevels {
    static constexpr int n = TS == 32 ? 32 : (TS == 64 ? 28 : 10);
};
constexpr int kMaxLevels = 64;
static_assert(kMaxLevels >= kRecvChunk, "a tile that culls by all planes (Level::cull) has all of them in its list");

template <int TS>
struct TileSh {  // log2 of the tile side
    static constexpr int v = TS == 128 ? 7 : (TS == 64 ? 6 : 5);
};

// A plane of the tile's receivers: depth d = pa x + pb y + pc at tile-local
// texel coordinates.  A triangle's depth at a texel centre less the plane's is
// below -front: it shades every sample of the plane that reads the texel; not
// below back: none.  front = inf, back = inf where no such bound is known (the
// sun within a degree of the plane, planes that share a level): every texel
// that a triangle covers is open.
struct Level {
    float pa, pb, pc;
    float front, back;
    float cull;  // a triangle nowhere nearer than the plane by more shades no sample of it; -1: no such bound
    int plane;  // plane group, or -1: any group without a level of its own
};

// What tile entry t_cnt holds once the tile kernels are done: kTileLit, a
// tile that shades every sample of every receiver, or 1 + the 16-byte offset
// of the tile's record in the pool B.cov:
//   word 0      levels | kRecOpen | kRecDepth | kRecHeavy | open triangles << 16
//   word 4 ...  plane group of each level, as many words as a multiple of four
//               holds (kNoPlane in the others)
//   then        box of each level's covered and open texels, x0 | x1 << 8 | y0
//               << 16 | y1 << 24 (kBoxNone: none), as many words
//   then        TS * TS / 32 words of coverage bits per level (bit x & 31 of
//               word y * TS / 32 + x / 32)
// and, with kRecOpen, as many words of open texels, then the open triangles
// (TriS, 12 words each) or, with kRecDepth, TS * TS depth keys.
constexpr uint32_t kTileLit = 0u;
constexpr uint32_t kTileFull = 0xFFFFFFFFu, kTileFullHeavy = 0xFFFFFFFEu;  // (heavy: k_raster_test's, for the counters)
constexpr uint32_t kRecLevels = 0xFFu, kRecOpen = 1u << 8, kRecDepth = 1u << 9, kRecHeavy = 1u << 10;
constexpr int kRecPlane = 4;
constexpr uint32_t kNoPlane = 0xFFFFFFFEu;
constexpr uint32_t kBoxNone = 0x000000FFu;
__device__ __forceinline__ int rec_planes(int nl) { return (nl + 3) & ~3; }
__device__ __forceinline__ int rec_box(int nl) { return kRecPlane + rec_planes(nl); }
__device__ __forceinline__ int rec_head(int nl) { return kRecPlane + 2 * rec_planes(nl); }
static_assert(kMaxLevels <= (int)kRecLevels, "record header");

// A triangle set up for the sample-driven test (48 bytes, three 16-byte loads):
// edge functions k = 0..2 in tile-local texel coordinates and depths scaled by
// the inverse doubled area.
struct TriS {
    float4 p;  // A0, B0, C0, A1
    float4 q;  // B1, C1, A2, B2
    float4 r;  // C2, e0, e1, e2
};

// Does triangle T cover texel centre (px, py) at a depth that the sample
// (depth d, bias) is behind?
__device__ __forceinline__ bool tri_shades(const TriS& T, float px, float py, float d, float bias,
                                           const LightParams& lp, int u24)
{
    const float4 p = T.p, q = T.q, r = T.r;
    const float w0 = edge_at(p.x, p.y, p.z, px, py);
    const float w1 = edge_at(p.w, q.x, q.y, px, py);
    const float w2 = edge_at(q.z, q.w, r.x, px, py);
    if (!(w0 >= 0.f && w1 >= 0.f && w2 >= 0.f)) return false;
    const float depth = depth_at(w0, w1, w2, r.y, r.z, r.w);
    if (u24) return behind_key(d, bias, depth_store_key(depth, lp, 1), lp.dnear, lp.qscale, 1);
    return d > __fadd_rn(depth, bias);  // = behind_key(d, bias, okey(depth), ...): okey is invertible
}

// A triangle set up for drawing: edge functions, depths scaled by the inverse
// doubled area, its texel box, the levels it is in front of and those it is
// to be compared with texel by texel (bit l of front, deep).  21 words: lanes
// reading different triangles' fields hit different banks.
struct TriDraw {
    float A[3], Bc[3], C[3];
    float inv[3];        // -1 / A, about (infinite for A = 0)
    float e[3];
    short x0, x1;
    int y0;
    float err;           // bound on the rounding of its depths
    uint32_t front, deep;
    int rows;
};
static_assert(sizeof(TriDraw) == 21 * 4, "odd word stride");

// Triangles being drawn by a warp, one per lane, and the inclusive prefix of
// their rows.
struct DrawSm {
    TriDraw tri[32];
    int pref[32];
    uint32_t open;  // triangles that left a texel open
};

// Level of module m (ModStep s) in tile (tx, ty).
template <int TS>
__device__ __forceinline__ void fill_level(Level& L, const ModStep& s, int plane, int tx, int ty, float cull)
{
    L.pa = s.pa;
    L.pb = s.pb;
    L.pc = s.d0 - s.pa * (s.tx0 - (float)(tx * TS)) - s.pb * (s.ty0 - (float)(ty * TS));
    L.front = s.hs + s.bias;
    L.back = s.hs - s.bias;
    // (less than half of the bias that is no slope: what lies in the plane or
    // behind it, which at a low sun rounding alone may bring past the bias)
    L.cull = s.cosi > 0.017452406f && s.hs < FLT_MAX ? cull : -1.f;
    L.plane = plane;
}

// Put nl levels in order, front to back; true if each is in front of the next
// all over the tile (planes that do not cross in it, such as parallel tables):
// what is in front of one level is then in front of all after it.
template <int TS>
__device__ __forceinline__ bool order_levels(Level* lv, int nl)
{
    const int lane = threadIdx.x & 31;
    const Level L = lv[min(lane, nl - 1)];
    // levels without a plane last, in their order: the shared level stays the last
    const float key = L.front < FLT_MAX ? L.pc + (L.pa + L.pb) * (0.5f * TS) - L.front : INFINITY;
    int rank = 0;
#pragma unroll 1
    for (int q = 0; q < nl; ++q) {
        const float o = __shfl_sync(0xffffffffu, key, q);
        rank += o < key || (o == key && q < lane) ? 1 : 0;
    }
    __syncwarp();
    if (lane < nl) lv[rank] = L;
    __syncwarp();
    bool ok = true;
    if (lane < nl) {
        const Level& a = lv[max(lane - 1, 0)];
        const Level& b = lv[lane];
        const float d = (b.pc - b.front) - (a.pc - a.front), x = (b.pa - a.pa) * TS, y = (b.pb - a.pb) * TS;
        ok = b.front < FLT_MAX && d + fminf(x, 0.f) + fminf(y, 0.f) >= 0.f;
    }
    return __all_sync(0xffffffffu, ok);
}

// The levels of tile te, at most `cap`, for one full warp; returns their
// number, or cap + 1 if there are more.  A tile of one plane group takes the
// plane from any of its modules (t_roff), others go through the receiver list.
template <int TS>
__device__ __forceinline__ int build_levels(Level* lv, int cap, const JobDev& J, const Buffers& B, const WaveDev* W,
                                            uint32_t te, int ls, int tx, int ty, uint32_t plane)
{
    const int lane = threadIdx.x & 31;
    const ModStep* ms = B.ms + J.ms_base + (int64_t)ls * J.n_mods;
    const uint32_t r0 = B.t_roff[te];
    const float cull = B.t_rcnt[te] <= (uint32_t)kRecvChunk ? B.lp[J.js_base + ls].delta * (1.f / 64.f) : -1.f;
    if (plane != kPlaneMixed) {
        if (lane == 0) fill_level<TS>(lv[0], ms[r0], (int)plane, tx, ty, cull);
        __syncwarp();
        return 1;
    }
    uint32_t r1 = r0 + B.t_rcnt[te];
    if (r1 > (uint64_t)W->recv_cap) r1 = (uint32_t)W->recv_cap;
    int nl = 0;
#pragma unroll 1
    for (uint32_t r = r0; r < r1; r += 32) {
        const bool have = r + lane < r1;
        const int m = have ? (int)B.recv[r + lane] : 0;
        const int pl = have ? J.mods[m].plane : -1;
        bool known = !have;
        for (int q = 0; q < nl; ++q) known = known || lv[q].plane == pl;
        unsigned int todo = __ballot_sync(0xffffffffu, !known);
#pragma unroll 1
        while (todo) {
            if (nl == cap) return cap + 1;
            const int lead = __ffs((int)todo) - 1;
            const int p = __shfl_sync(0xffffffffu, pl, lead);
            todo &= ~__ballot_sync(0xffffffffu, have && pl == p);
            if (lane == lead) fill_level<TS>(lv[nl], ms[m], pl, tx, ty, cull);
            ++nl;
            __syncwarp();
        }
    }
    return nl;
}

// A binned triangle over the tile: its texel-space vertices (tile-local,
// counter-clockwise), edges and texel box, and what it is to the tile's
// levels.
struct TriWork {
    TriT T;
    Edges ed;
    int x0, x1, y0, y1;
    float err;             // bound on the rounding of its depths
    uint32_t front, deep;  // bit l: in front of level l; to be compared with it texel by texel
    bool whole;            // covers every texel centre of the tile
};

// Set up binned triangle t of tile (ox, oy) for levels [s0, s0 + np) of nl (bit
// l of front and deep: level s0 + l); front = deep = 0 if it covers no texel
// centre of the tile or is behind every level, or lies in or behind the planes
// of all nl.
//
// The triangle's depth less a plane's is linear, so over the tile it lies
// between its values at the vertices, up to what rounding makes of the depth
// at a texel (depth_at): the mean of the vertex depths d_k weighted by the
// edge functions w_k >= 0 as computed, over the doubled area as computed, is
// off by at most |d| (|sum w_k / area - 1| + 6 u), u = 2^-24.  Each w_k is off
// its exact value by at most 5 u (|A_k| (|px| + |x_a|) + |B_k| (|py| + |y_a|))
// (the rounding of A, B, C and of the two multiply-adds; x_a, y_a the vertex C
// was taken at, |px|, |py| <= TS) and the area by 3 u of the same sum S over
// the three edges: |sum w_k / area - 1| <= 8 u S / area = 4.8e-7 S / area.
// Twice that is allowed for, and 1e-5 of the plane's terms at the vertices.
template <int TS, bool PROF>
__device__ __forceinline__ void classify_tri(const JobDev& J, const Buffers& B, const LightParams& lp, int ls, int t,
                                             float ox, float oy, const Level* lv, int nl, int s0, int np,
                                             TriWork& w, unsigned int& culled)
{
    tri_texel(J, B, lp, ls, t, w.T);
    TriT& T = w.T;
#pragma unroll
    for (int k = 0; k < 3; ++k) { T.x[k] -= ox; T.y[k] -= oy; }
    if (!make_edges(T, w.ed) || !tri_box<TS>(T, w.x0, w.x1, w.y0, w.y1)) return;
    const Edges& e = w.ed;
    const float xm = fmaxf(fabsf(T.x[0]), fmaxf(fabsf(T.x[1]), fabsf(T.x[2]))) + (float)TS;
    const float ym = fmaxf(fabsf(T.y[0]), fmaxf(fabsf(T.y[1]), fabsf(T.y[2]))) + (float)TS;
    const float S = (fabsf(e.A[0]) + fabsf(e.A[1]) + fabsf(e.A[2])) * xm +
                    (fabsf(e.Bc[0]) + fabsf(e.Bc[1]) + fabsf(e.Bc[2])) * ym;
    const float dabs = fmaxf(fabsf(T.d[0]), fmaxf(fabsf(T.d[1]), fabsf(T.d[2])));
    const float err = dabs * (1e-6f * __fdividef(S, e.area2) + 1e-6f);
    w.err = err;
    bool keep = false;
#pragma unroll 1
    for (int l = 0; l < nl; ++l) {
        const float pa = lv[l].pa, pb = lv[l].pb, pc = lv[l].pc;
        float lo = FLT_MAX, hi = -FLT_MAX;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const float g = T.d[k] - (pa * T.x[k] + pb * T.y[k] + pc);
            lo = fminf(lo, g);
            hi = fmaxf(hi, g);
        }
        const float tol = err + 1e-5f * (fabsf(pa) * xm + fabsf(pb) * ym);
        keep = keep || lv[l].cull < 0.f || !(lo >= -lv[l].cull);
        const uint32_t bit = l >= s0 && l < s0 + np ? 1u << (l - s0) : 0u;
        if (hi + tol < -lv[l].front) w.front |= bit;
        else if (!(lo - tol >= lv[l].back)) w.deep |= bit;
    }
    if (!keep) w.deep = 0u;  // (front none)
    if (PROF && s0 == 0 && !(w.front | w.deep)) ++culled;
    // each edge at the texel centre farthest outside it (edge_at is monotone
    // in px and py)
    if (w.x0 == 0 && w.y0 == 0 && w.x1 == TS - 1 && w.y1 == TS - 1) {
        w.whole = true;
#pragma unroll
        for (int k = 0; k < 3; ++k)
            w.whole = w.whole && edge_at(e.A[k], e.Bc[k], e.C[k], e.A[k] > 0.f ? 0.5f : TS - 0.5f,
                                         e.Bc[k] > 0.f ? 0.5f : TS - 0.5f) >= 0.f;
    }
}

// Narrow the texel range [lo, hi] (whole numbers, or empty: lo = hi + 1) of a
// row to the texels whose centre px has fma(A, px, t) >= 0 -- edge_at on that
// row, which is monotone in px, so the texels form an interval that ends at
// one end of the range (the high one for A >= 0).  Its other end is found from
// the edge's root t inv, inv = -1/A about.  The sign of fma is that of A px + t exactly, and
// within the range (at most 128 texels) the root's estimate is off by far less
// than one texel, so one step either way corrects it.  A = 0 (or so small that
// the root overflows): the estimate is infinite, beyond the range on the side
// where the sign of t puts the interval's end; t = 0 then makes it NaN, which
// the clamp takes to the low end (A >= 0: every texel; A < 0: none).
__device__ __forceinline__ void row_edge(float A, float inv, float t, float& lo, float& hi)
{
    const float s = A >= 0.f ? 1.f : -1.f;
    const float begin = A >= 0.f ? lo : hi, end = (A >= 0.f ? hi : lo) + s;
    const float r = __fmaf_rn(t, inv, -0.5f);
    float i = fminf(fmaxf(A >= 0.f ? ceilf(r) : floorf(r), fminf(begin, end)), fmaxf(begin, end));
    if (i != begin && __fmaf_rn(A, i - s + 0.5f, t) >= 0.f) i -= s;
    if (i != end && __fmaf_rn(A, i + 0.5f, t) < 0.f) i += s;
    if (A >= 0.f) lo = i;
    else hi = i;
}

// Narrow the texels [lo, hi] to those where a value that is linear along them,
// from ga at lo to gb at hi, is below T: with margin < 0 to fewer (each of them
// is), with margin > 0 to more (no other is), by that part of a texel, which is
// far above what the root's estimate is off by.  False if none is.  A NaN (an
// infinite bound) leaves none and all.
__device__ __forceinline__ bool below(float ga, float gb, float T, float margin, float& lo, float& hi)
{
    const bool in_a = margin > 0.f ? !(ga >= T) : ga < T, in_b = margin > 0.f ? !(gb >= T) : gb < T;
    if (in_a != in_b) {
        const float x = __fmaf_rn(__fdividef(T - ga, gb - ga), hi - lo, lo);
        if (margin > 0.f) {
            if (in_a) hi = fminf(hi, ceilf(x + margin));
            else lo = fmaxf(lo, floorf(x - margin));
        } else {
            if (in_a) hi = fmaxf(lo - 1.f, floorf(x + margin));
            else lo = fminf(hi + 1.f, ceilf(x - margin));
        }
    }
    return (in_a || in_b) && lo <= hi;
}

// A triangle's rows are one lane each.  On 64- and 128-texel tiles a triangle
// has rows enough for the warp, so its rows are drawn together: its set-up is
// read by all lanes at once, and a warp that has the tile to itself
// (k_tile_warp) updates a row's words with one vector load and store in place
// of atomics.  On 32-texel tiles most have five to ten rows and several
// triangles share the warp.  (128 texels, the facade year: 4.7 -> 3.9 ms for
// k_tile_warp; 64 texels, 45 suns over 13 modules: 68 -> 53 us.)
//
// k_raster_test: threads of a block, blocks an SM.
template <int TS>
struct HeavyCfg {
    static constexpr int threads = TS == 32 ? 128 : 256;
    static constexpr int stride = TS + 1;  // of a row of depths: the lanes' rows lie in different banks
    static constexpr int min_blocks = TS == 32 ? 8 : (TS == 64 ? 4 : 2);
};

// A row's texels between those in front of a plane and those behind it are
// compared one by one up to so many, above that as a span.  (A steep plane's
// band may be as wide as the tile: with this, and the depths of a row's open
// texels drawn once in place of once a level, k_raster_test took 117 us in
// place of 158 for 25 modules of all orientations, 47 suns, R = 512.)
constexpr float kBandTexels = 6.f;

// Draw the warp's triangles (w, one per lane; `full`: the levels covered
// everywhere, neither drawn nor compared any more): row spans into the coverage bits of the levels they are in
// front of (cov, TS * TS / 32 words each; nested levels: of the first of them
// only, finish_words adds the bits to the levels after it), and for the levels
// they cross, the texels in front of the plane as coverage bits and those in
// the band as open.  `open` (level-free): the open texels' bits; with TILE,
// their nearest depth in `tile` too.  D.open receives the triangles that left
// a texel open.
template <int TS, bool TILE, bool PROF>
__device__ __forceinline__ void draw_tris(DrawSm& D, const TriWork& w, uint32_t full, bool nested, const Level* lv,
                                          uint32_t* cov,
                                          uint32_t* open, uint32_t* tile, const LightParams& lp, int u24,
                                          unsigned int& visits, unsigned int& writes)
{
    constexpr int WPR = TS / 32, NW = TS * WPR;
    constexpr bool kRowsOfOne = TS >= 64, kOwnRow = kRowsOfOne && !TILE;
    const int lane = threadIdx.x & 31;
    uint32_t front = w.front & ~full, deep = w.deep & ~full;
    if (nested) {
        const uint32_t low = w.front & (0u - w.front);
        front &= low;
        deep &= low - 1u;  // low = 0: all
    }
    int rows = 0;
    if (front | deep) {
        TriDraw& S = D.tri[lane];
        const float inv_a = 1.f / w.ed.area2;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            S.A[k] = w.ed.A[k]; S.Bc[k] = w.ed.Bc[k]; S.C[k] = w.ed.C[k];
            S.inv[k] = __fdividef(-1.f, __fadd_rn(w.ed.A[k], 0.f));  // A = -0 is 0
            S.e[k] = w.T.d[k] * inv_a;
        }
        S.x0 = (short)w.x0;
        S.x1 = (short)w.x1;
        S.y0 = w.y0;
        S.err = w.err;
        S.rows = rows = w.y1 - w.y0 + 1;
        S.front = front;
        S.deep = deep;
    }
    if (lane == 0) D.open = 0u;
    auto draw_row = [&](const TriDraw& S, int t, int iy) {
        const float py = (float)iy + 0.5f;
        float a = (float)S.x0, b = (float)S.x1;
        float tk[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            tk[k] = __fmaf_rn(S.Bc[k], py, S.C[k]);
            row_edge(S.A[k], S.inv[k], tk[k], a, b);
        }
        const int lo = (int)a, hi = (int)b;
        if (lo > hi) return;
        if (PROF) visits += (unsigned int)(hi - lo + 1);
#pragma unroll 1
        for (uint32_t m = S.front; m; m &= m - 1u) {
            uint32_t* row = cov + (__ffs((int)m) - 1) * NW + iy * WPR;
            if constexpr (kOwnRow && TS == 128) {
                uint4 v = *reinterpret_cast<uint4*>(row);
                v.x |= span_word(lo, hi, 0); v.y |= span_word(lo, hi, 1);
                v.z |= span_word(lo, hi, 2); v.w |= span_word(lo, hi, 3);
                *reinterpret_cast<uint4*>(row) = v;
            } else if constexpr (kOwnRow && TS == 64) {
                uint2 v = *reinterpret_cast<uint2*>(row);
                v.x |= span_word(lo, hi, 0); v.y |= span_word(lo, hi, 1);
                *reinterpret_cast<uint2*>(row) = v;
            } else {
#pragma unroll 1
                for (int q = lo >> 5; q <= (hi >> 5); ++q) atomicOr(&row[q], span_word(lo, hi, q));
            }
        }
        uint32_t m = S.deep;
        if (m == 0u) return;
        const float A0 = S.A[0], A1 = S.A[1], A2 = S.A[2], e0 = S.e[0], e1 = S.e[1], e2 = S.e[2];
        auto depth_px = [&](float px) {
            return depth_at(__fmaf_rn(A0, px, tk[0]), __fmaf_rn(A1, px, tk[1]), __fmaf_rn(A2, px, tk[2]), e0, e1, e2);
        };
        const float pl = a + 0.5f, ph = b + 0.5f, dl = depth_px(pl), dh = depth_px(ph), err2 = 2.f * S.err;
        uint32_t left[TILE ? WPR : 1] = {};  // the row's open texels
#pragma unroll 1
        for (; m; m &= m - 1u) {
            const int l = __ffs((int)m) - 1;
            const float pa = lv[l].pa, base = __fmaf_rn(lv[l].pb, py, lv[l].pc);
            const float fr = -lv[l].front, bk = lv[l].back;
            // the gap is linear along the row, up to the depths' rounding: its
            // ends tell which texels are in front and which are behind, and
            // where there are many others which of them are in the band, but
            // for those about the roots
            const float ga = dl - __fmaf_rn(pa, pl, base), gb = dh - __fmaf_rn(pa, ph, base);
            float fa = a, fb = b, ca = a, cb = b;          // in front; not behind
            float ia = a, ib = a - 1.f, ja = a, jb = a - 1.f;  // in the band: [ia, ib] less [ja, jb]
            if (!below(ga, gb, fr - err2, -0.02f, fa, fb)) fb = fa - 1.f;
            if (!below(ga, gb, bk + err2, 0.02f, ca, cb)) continue;
            if (!(bk < FLT_MAX)) {  // no plane to compare with
                ib = b;
            } else if ((cb - ca) - (fb - fa) > kBandTexels) {
                ib = jb = b;
                if (!below(ga, gb, bk - err2, -0.02f, ia, ib)) ib = ia - 1.f;
                if (!below(ga, gb, fr + err2, 0.02f, ja, jb)) jb = ja - 1.f;
            }
            const int f0 = (int)fa, f1 = (int)fb, c0 = (int)ca, c1 = (int)cb;
            const int i0 = (int)ia, i1 = (int)ib, j0 = (int)ja, j1 = (int)jb;
#pragma unroll 1
            for (int q = c0 >> 5; q <= (c1 >> 5); ++q) {
                const int word = iy * WPR + q;
                uint32_t c = span_word(f0, f1, q);
                uint32_t r = span_word(c0, c1, q) & ~c & ~cov[l * NW + word];
                uint32_t o = r & span_word(i0, i1, q) & ~span_word(j0, j1, q);
#pragma unroll 1
                for (r &= ~o; r; r &= r - 1u) {
                    const int x = __ffs((int)r) - 1;
                    const float px = (float)(32 * q + x) + 0.5f;
                    const float gap = depth_px(px) - __fmaf_rn(pa, px, base);
                    if (PROF) ++writes;
                    if (gap < fr) c |= 1u << x;
                    else if (!(gap >= bk)) o |= 1u << x;
                }
                if (c) atomicOr(&cov[l * NW + word], c);
                if (o) {
                    atomicOr(&open[word], o);
                    atomicOr(&D.open, 1u << t);
                    if (TILE) {
#pragma unroll
                        for (int k = 0; k < WPR; ++k) left[k] |= k == q ? o : 0u;
                    }
                }
            }
        }
        // the depths of the row's open texels, of all levels together (each a
        // chain of 25 dependent instructions: four at a time, 25 modules of all
        // orientations on 128-texel tiles, 47 suns, went from 805 to 600 us)
        if constexpr (TILE) {
#pragma unroll 1
            for (int q = lo >> 5; q <= (hi >> 5); ++q) {
                uint32_t r = 0u;
#pragma unroll
                for (int k = 0; k < WPR; ++k) r |= k == q ? left[k] : 0u;
                if (r == 0u) continue;
                const int x0 = __ffs((int)r) - 1, x1 = 31 - __clz((int)r);
                uint32_t* dst = &tile[iy * HeavyCfg<TS>::stride + 32 * q];
#pragma unroll 4
                for (int x = x0; x <= x1; ++x) {
                    const uint32_t key = depth_store_key(depth_px((float)(32 * q + x) + 0.5f), lp, u24);
                    if ((r >> x) & 1u) atomicMin(&dst[x], key);
                }
            }
        }
    };
    if constexpr (kRowsOfOne) {
        unsigned int todo = __ballot_sync(0xffffffffu, rows > 0);
        __syncwarp();
#pragma unroll 1
        for (; todo; todo &= todo - 1u) {
            const int t = __ffs((int)todo) - 1;
            const TriDraw& S = D.tri[t];
            const int end = S.y0 + S.rows;
#pragma unroll 1
            for (int iy = S.y0 + lane; iy < end; iy += 32) draw_row(S, t, iy);
            __syncwarp();  // the next triangle's rows are other lanes'
        }
    } else {
        const int inc = warp_incl_scan(rows);
        D.pref[lane] = inc;
        __syncwarp();
        const int total = __shfl_sync(0xffffffffu, inc, 31);
#pragma unroll 1
        for (int u = lane; u < total; u += 32) {
            int t = 0;  // the row's triangle: the first with pref > u
#pragma unroll
            for (int step = 16; step; step >>= 1)
                if (D.pref[t + step - 1] <= u) t += step;
            const TriDraw& S = D.tri[t];
            draw_row(S, t, S.y0 + u - (t ? D.pref[t - 1] : 0));
        }
        __syncwarp();
    }
}

// Levels that are covered everywhere given that those of f are.
__device__ __forceinline__ uint32_t full_after(uint32_t f, bool nested, uint32_t all)
{
    return nested && f ? all & ~((f & (0u - f)) - 1u) : f;
}

// Coverage word q of every level in turn, with the levels' nesting and the
// full levels applied: f(l, word).
template <int TS, typename F>
__device__ __forceinline__ void for_levels(const uint32_t* cov, int nl, bool nested, uint32_t full, int q, F f)
{
    uint32_t c = 0u;
#pragma unroll 1
    for (int l = 0; l < nl; ++l) {
        const uint32_t v = cov[l * (TS * TS / 32) + q];
        c = (full >> l) & 1u ? 0xFFFFFFFFu : (nested ? c | v : v);
        f(l, c);
    }
}

// The levels whose coverage bits are all set, for one full warp.
template <int TS>
__device__ __forceinline__ uint32_t full_levels(const uint32_t* cov, int nl, bool nested, uint32_t full)
{
    uint32_t ok = (2u << (nl - 1)) - 1u;
#pragma unroll 1
    for (int q = threadIdx.x & 31; q < TS * TS / 32; q += 32)
        for_levels<TS>(cov, nl, nested, full, q, [&](int l, uint32_t c) {
            if (c != 0xFFFFFFFFu) ok &= ~(1u << l);
        });
    return __reduce_and_sync(0xffffffffu, ok);
}

// Write the levels' nesting and the full levels into the coverage words q =
// q_begin, q_begin + q_stride, ...: some = a bit is set, hole = a bit is not.
template <int TS>
__device__ __forceinline__ void finish_words(uint32_t* cov, int nl, bool nested, uint32_t full, int q_begin, int q_stride,
                                             uint32_t& some, uint32_t& hole)
{
#pragma unroll 1
    for (int q = q_begin; q < TS * TS / 32; q += q_stride)
        for_levels<TS>(cov, nl, nested, full, q, [&](int l, uint32_t c) {
            cov[l * (TS * TS / 32) + q] = c;
            some |= c;
            hole |= ~c;
        });
}

// Bins of a tile, clamped to the bin pool.
__device__ __forceinline__ void tile_bins(const Buffers& B, const WaveDev* W, uint32_t te, uint64_t& off, uint32_t& cnt)
{
    off = B.t_off[te];
    cnt = B.t_cnt[te];
    const uint64_t cap = (uint64_t)W->bin_cap;
    if (off + cnt > cap) cnt = off < cap ? (uint32_t)(cap - off) : 0u;
}

// Words of a tile's record, and its place in the pool: the 16-byte offset
// plus one, or 0 when the pool is full (the host grows it and reruns the
// wave).  Called by one thread.
__device__ __forceinline__ uint32_t alloc_record(const Buffers& B, const WaveDev* W, uint32_t words)
{
    const unsigned long long quads = (words + 3u) / 4u;
    const unsigned long long pos = atomicAdd(&B.ctr->cov_next, quads);
    return pos + quads <= (unsigned long long)W->cov_cap ? (uint32_t)pos + 1u : 0u;
}

// Box of the texels set in cov or open (TS * TS / 32 words each), packed as in
// the record's header; by one full warp.
template <int TS>
__device__ __forceinline__ uint32_t texel_box(const uint32_t* cov, const uint32_t* open)
{
    constexpr int WPR = TS / 32, NW = TS * WPR;
    int x0 = 255, x1 = -1, y0 = 255, y1 = -1;
#pragma unroll 1
    for (int q = threadIdx.x & 31; q < NW; q += 32) {
        const uint32_t c = cov[q] | open[q];
        if (c) {
            const int y = q / WPR, xb = (q % WPR) * 32;
            y0 = min(y0, y); y1 = max(y1, y);
            x0 = min(x0, xb + __ffs((int)c) - 1); x1 = max(x1, xb + 31 - __clz((int)c));
        }
    }
    x0 = __reduce_min_sync(0xffffffffu, x0); x1 = __reduce_max_sync(0xffffffffu, x1);
    y0 = __reduce_min_sync(0xffffffffu, y0); y1 = __reduce_max_sync(0xffffffffu, y1);
    return x1 < 0 ? kBoxNone : (uint32_t)x0 | ((uint32_t)x1 << 8) | ((uint32_t)y0 << 16) | ((uint32_t)y1 << 24);
}

// ---------------------------------------------------------------------------
// k_tile_warp: fused path -- one warp per non-empty tile: the tile's coverage
// bits.  A tile of more planes than WarpLevels, with more than warp_bins()
// binned triangles (fewer in waves of few tiles, see below) or more than
// kWarpOpen that leave texels open, and a 64-texel tile with more than
// kWarpRecv receivers or more than kWarpKept triangles in front of or across a
// level, is listed for k_raster_test.  A tile is a small
// work item: one warp each keeps many tiles in flight per SM, which hides the
// chain of dependent loads that starts a tile.
//
// What bounds it: instruction issue (53-70 % of the slots over full waves, the
// rest waits for the triangles' vertices).  A depth per texel and a test per
// sample cost one step per covered texel and one per sample; a bit per texel
// costs one step per row of a triangle, and a plane's samples read it as
// words.  The code is kept small (loops not unrolled, one copy of each): at
// twice the size the warps waited for instructions up to nine cycles each.
// With k_cells, against depth tiles and a test per sample: 12,000 modules on
// trackers over terrain, 47 suns: 3.2 -> 1.8 ms all told; a facade of 200
// modules, 50 000 triangles, n = 8, a year of hours: 17.5 -> 13.4 ms.
// ---------------------------------------------------------------------------
constexpr int kWarpOpen = 32;
constexpr int kWarpKept = 80;
constexpr int kWarpRecv = 16;
constexpr int kTileWarps = 4;  // warps per block

// Blocks an SM: as many as its shared memory holds.  (A bound of 8 for every
// tile side kept 64 registers a thread and spilled 60 of them for blocks that
// could not be resident; with 6 for 64 and 128 texels, 80 registers and no
// spills, this kernel's share of the facade's year went from 2.82 to 2.70 ms,
// of its report from 3.00 to 2.71, of the diffuse month from 419 to 362 us.)
template <int TS>
struct TileBlocks {
    static constexpr int n = TS == 32 ? 8 : 6;
};
constexpr size_t kSmShared = 228 * 1024, kBlockShared = 1024;  // of an SM; taken by the system for each block

template <int TS>
__device__ constexpr uint32_t warp_bins() { return TS == 32 ? 256u : (TS == 64 ? 512u : 96u); }

template <int TS>
struct __align__(16) WarpSm {
    TriS tri[kWarpOpen];
    DrawSm d;
    Level lv[WarpLevels<TS>::n];
    __align__(16) uint32_t cov[WarpLevels<TS>::n * TS * TS / 32];  // draw_tris takes a row at once
    uint32_t open[TS * TS / 32];
};
static_assert(offsetof(WarpSm<64>, cov) % 16 == 0 && sizeof(WarpSm<64>) % 16 == 0 &&
              offsetof(WarpSm<128>, cov) % 16 == 0 && sizeof(WarpSm<128>) % 16 == 0, "rows are read as vectors");

template <int TS, bool PROF>
__global__ void __launch_bounds__(kTileWarps * 32, TileBlocks<TS>::n) k_tile_warp(const WaveDev* __restrict__ W,
                                                                  const JobDev* __restrict__ jobs, Buffers B)
{
    extern __shared__ __align__(16) unsigned char tile_smem[];  // kTileWarps WarpSm, set at launch
    static_assert(TileBlocks<TS>::n * (kTileWarps * sizeof(WarpSm<TS>) + kBlockShared) <= kSmShared, "blocks an SM");
    constexpr int NW = TS * TS / 32;
    unsigned int p_visits = 0, p_writes = 0, p_culled = 0, p_tiles = 0, p_stiles = 0, p_hr = 0, p_hb = 0, p_ht = 0;
    const int lane = threadIdx.x & 31;
    WarpSm<TS>& sm = reinterpret_cast<WarpSm<TS>*>(tile_smem)[threadIdx.x >> 5];
    // the bins are incomplete when the pool overflowed: the wave is rerun
    // with a larger pool, so nothing here may read them
    const unsigned int n_ne = (B.ctr->overflow & 1u) ? 0u : B.ctr->n_nonempty;
    // tiles of many triangles come first, from the front of the list, the
    // others from its end (k_scan_c)
    const unsigned int n_first = B.ctr->n_first, last = (unsigned int)(W->tot_te - 1);
    const int nj = W->n_jobs;
    const int u24 = W->depth_u24;
    // with few tiles the largest is the kernel's time.  128 texels, a tile or
    // less for each resident warp: 32 triangles of up to 128 rows are enough
    // for a warp (77 facade modules, 72 suns: both tile kernels 353 us with 96,
    // 240 with 32).  Smaller tiles: where some are large, as many of the
    // largest as k_raster_test's blocks take in two rounds go to a block's eight
    // warps (25 modules on planes of their own, R = 512, 47 suns, 652 tiles of
    // up to 163 triangles: both 452 us, now 140; the call 641, now 345.  With
    // one round for the limit 50 modules, 100 suns, took 1 to 15 % longer; tiles
    // of at most 48 triangles are a warp's in any case: their blocks cost as
    // much as they save)
    uint32_t most = warp_bins<TS>();
    if (TS == 128) {
        if (n_ne <= gridDim.x * (unsigned int)kTileWarps) most = 32u;
    } else if (n_ne <= kSmallWave && n_first > 0u) {
        const unsigned int blocks = gridDim.x / TileBlocks<TS>::n * HeavyCfg<TS>::min_blocks;
        for (int q = kShareSteps; q-- > 0;)
            if (B.ctr->n_over[q] <= 2u * blocks) most = share_bins(q);
    }
    unsigned int next = 0;
    if (lane == 0) next = atomicAdd(&B.ctr->raster_next, 1u);
    next = __shfl_sync(0xffffffffu, next, 0);
    while (next < n_ne) {
        const unsigned int item = next;
        if (lane == 0) next = atomicAdd(&B.ctr->raster_next, 1u);  // claim the following tile now
        const uint32_t te = B.nonempty[item < n_first ? item : last - (item - n_first)];
        uint64_t off;
        uint32_t cnt;
        tile_bins(B, W, te, off, cnt);
        const uint32_t nrecv = B.t_rcnt[te], plane = B.t_plane[te];
        int j, ls, tx, ty;
        decode_tile(jobs, nj, te, j, ls, tx, ty);
        const JobDev& J = jobs[j];
        const bool crowd = TS == 64 && nrecv > (uint32_t)kWarpRecv;
        bool heavy = crowd || cnt > most;
        if (PROF && lane == 0) {
            if (crowd) ++p_hr;
            else if (heavy && cnt > warp_bins<TS>()) ++p_hb;
            else if (heavy) ++p_ht;
        }
        if (!heavy) {
            const LightParams& lp = B.lp[J.js_base + ls];
            const int nl = build_levels<TS>(sm.lv, WarpLevels<TS>::n, J, B, W, te, ls, tx, ty, plane);
            heavy = nl > WarpLevels<TS>::n;
            const bool nested = !heavy && nl > 1 && order_levels<TS>(sm.lv, nl);
#pragma unroll 4
            for (int q = lane; q < (heavy ? 0 : nl * NW); q += 32) sm.cov[q] = 0u;
#pragma unroll 4
            for (int q = lane; q < NW; q += 32) sm.open[q] = 0u;
            __syncwarp();
            const uint32_t all = (1u << nl) - 1u;
            const float ox = (float)(tx * TS), oy = (float)(ty * TS);
            uint32_t full = 0u;    // levels covered everywhere
            int n = 0, kept = 0;   // triangles that left a texel open; in front of or across a level
#pragma unroll 1
            for (uint32_t b0 = 0; b0 < cnt && !heavy && full != all; b0 += 32) {
                TriWork w;
                w.front = w.deep = 0u;
                w.whole = false;
                if (b0 + lane < cnt)
                    classify_tri<TS, PROF>(J, B, lp, ls, (int)B.bins[off + b0 + lane], ox, oy, sm.lv, nl, 0, nl, w,
                                           p_culled);
                full = full_after(full | __reduce_or_sync(0xffffffffu, w.whole ? w.front : 0u), nested, all);
                const unsigned int use = __ballot_sync(0xffffffffu, (w.front | w.deep) != 0u);
                kept += __popc(use);
                if (use == 0u || full == all) continue;
                draw_tris<TS, false, PROF>(sm.d, w, full, nested, sm.lv, sm.cov, sm.open, nullptr, lp, u24, p_visits,
                                           p_writes);
                const uint32_t op = sm.d.open;
                const int slot = n + __popc(op & ((1u << lane) - 1u));
                if (((op >> lane) & 1u) && slot < kWarpOpen) {
                    const TriDraw& S = sm.d.tri[lane];
                    sm.tri[slot].p = make_float4(S.A[0], S.Bc[0], S.C[0], S.A[1]);
                    sm.tri[slot].q = make_float4(S.Bc[1], S.C[1], S.A[2], S.Bc[2]);
                    sm.tri[slot].r = make_float4(S.C[2], S.e[0], S.e[1], S.e[2]);
                }
                n += __popc(op);
                heavy = n > kWarpOpen || (TS == 64 && kept > kWarpKept);
                __syncwarp();  // the set-up may be replaced
                if (b0 + 32 < cnt) full = full_levels<TS>(sm.cov, nl, nested, full);
            }
            if (full == all) heavy = false;
            if (PROF && lane == 0) {
                if (heavy) ++p_ht;
                else {
                    ++p_tiles;
                    if (kept == 0) ++p_stiles;
                }
            }
            if (!heavy) {
                uint32_t state = kTileFull;
                if (full != all) {
                    // does any texel matter, is any not covered?
                    uint32_t some = 0u, hole = 0u;
                    finish_words<TS>(sm.cov, nl, nested, full, lane, 32, some, hole);
                    __syncwarp();
                    if (!__any_sync(0xffffffffu, hole != 0u)) {
                        state = kTileFull;
                    } else if (n == 0 && !__any_sync(0xffffffffu, some != 0u)) {
                        state = kTileLit;
                    } else {
                        const uint32_t words = (uint32_t)(rec_head(nl) + nl * NW + (n ? NW + 12 * n : 0));
                        if (lane == 0) state = alloc_record(B, W, words);
                        state = __shfl_sync(0xffffffffu, state, 0);
                        if (state) {
                            uint32_t* rec = B.cov + 4 * (size_t)(state - 1u);
                            if (lane == 0) rec[0] = (uint32_t)nl | (n ? kRecOpen | ((uint32_t)n << 16) : 0u);
                            if (lane < rec_planes(nl))
                                rec[kRecPlane + lane] = lane < nl ? (uint32_t)sm.lv[lane].plane : kNoPlane;
#pragma unroll 1
                            for (int l = 0; l < nl; ++l) {
                                const uint32_t box = texel_box<TS>(sm.cov + l * NW, sm.open);
                                if (lane == 0) rec[rec_box(nl) + l] = box;
                            }
                            uint32_t* dst = rec + rec_head(nl);
                            for (int q = lane; q < nl * NW; q += 32) dst[q] = sm.cov[q];
                            if (n) {
                                dst += nl * NW;
                                for (int q = lane; q < NW; q += 32) dst[q] = sm.open[q];
                                dst += NW;
                                const uint32_t* src = reinterpret_cast<const uint32_t*>(sm.tri);
                                for (int q = lane; q < 12 * n; q += 32) dst[q] = src[q];
                            }
                        }
                    }
                }
                if (lane == 0) B.t_cnt[te] = state;
            }
        }
        if (heavy && lane == 0) {
            const unsigned int pos = atomicAdd(&B.ctr->n_heavy, 1u);
            if (pos < (uint64_t)W->tot_te) B.heavy[pos] = te;
        }
        __syncwarp();  // the warp's shared memory may be reused
        next = __shfl_sync(0xffffffffu, next, 0);
    }
    if (PROF) {
        flush_profile(B, 0u, p_visits, p_visits + p_writes, p_culled);
        flush_profile2(B, 0u, p_tiles, 0u, p_stiles, 0u);
#pragma unroll
        for (int off = 16; off; off >>= 1) {
            p_hr += __shfl_xor_sync(0xffffffffu, p_hr, off);
            p_hb += __shfl_xor_sync(0xffffffffu, p_hb, off);
            p_ht += __shfl_xor_sync(0xffffffffu, p_ht, off);
        }
        if (lane == 0) {
            atomicAdd(&B.ctr->prof_heavy_why[0], (unsigned long long)p_hr);
            atomicAdd(&B.ctr->prof_heavy_why[1], (unsigned long long)p_hb);
            atomicAdd(&B.ctr->prof_heavy_why[2], (unsigned long long)p_ht);
        }
    }
}

// ---------------------------------------------------------------------------
// k_raster_test: fused path, the tiles k_tile_warp listed -- one block per
// tile, its warps taking up to 32 triangles at a time by themselves (as many
// each: with 32 for some and none for others the facade year's share of this
// kernel was 0.96 ms, now 0.63); texels left open keep their nearest depth in
// a shared tile that goes to the record.  Tiles of more planes than have bits
// at a time are drawn in turns: 50 modules on planes of their own, 128-texel
// tiles, 100 suns: the call 1,045 us with all but three planes left open
// throughout, 660 with ten at a time.  Bound by the longest tile: there are
// fewer than blocks in most waves.
// ---------------------------------------------------------------------------
template <int TS>
struct __align__(16) HeavySm {
    uint32_t tile[TS * HeavyCfg<TS>::stride];  // nearest depth keys of open texels
    uint32_t cov[PassLevels<TS>::n * TS * TS / 32];
    uint32_t open[TS * TS / 32];
    DrawSm d[HeavyCfg<TS>::threads / 32];
    Level lv[kMaxLevels];
    int nl;
    int nested;
    uint32_t full, state;
    unsigned int item[2];
};

template <int TS, bool PROF>
__global__ void __launch_bounds__(HeavyCfg<TS>::threads, HeavyCfg<TS>::min_blocks)
    k_raster_test(const WaveDev* __restrict__ W, const JobDev* __restrict__ jobs, Buffers B)
{
    constexpr int NW = TS * TS / 32, kWarps = HeavyCfg<TS>::threads / 32;
    extern __shared__ __align__(16) unsigned char tile_smem[];  // HeavySm, set at launch
    static_assert(HeavyCfg<TS>::min_blocks * (sizeof(HeavySm<TS>) + kBlockShared) <= kSmShared, "blocks an SM");
    HeavySm<TS>& sm = *reinterpret_cast<HeavySm<TS>*>(tile_smem);
    unsigned int p_visits = 0, p_writes = 0, p_culled = 0, p_tiles = 0;
    // incomplete bins (pool overflow, the wave is rerun): nothing to read
    const unsigned int n_ne = (B.ctr->overflow & 1u) ? 0u : min(B.ctr->n_heavy, (unsigned int)W->tot_te);
    const int nj = W->n_jobs;
    const int u24 = W->depth_u24;
    const int tid = threadIdx.x, bd = blockDim.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) sm.item[0] = atomicAdd(&B.ctr->heavy_next, 1u);
    __syncthreads();
    for (int par = 0;; par ^= 1) {
        // the next tile is claimed while this one runs; the barriers inside
        // the tile publish it
        const unsigned int item = sm.item[par];
        if (item >= n_ne) break;
        if (tid == 0) sm.item[par ^ 1] = atomicAdd(&B.ctr->heavy_next, 1u);
        const uint32_t te = B.heavy[item];
        uint64_t off;
        uint32_t cnt;
        tile_bins(B, W, te, off, cnt);
        int j, ls, tx, ty;
        decode_tile(jobs, nj, te, j, ls, tx, ty);
        const JobDev& J = jobs[j];
        const LightParams& lp = B.lp[J.js_base + ls];
        if (warp == 0) {
            int nl = build_levels<TS>(sm.lv, kMaxLevels, J, B, W, te, ls, tx, ty, B.t_plane[te]);
            if (nl > kMaxLevels) {
                nl = PassLevels<TS>::n;
                if (lane == 0) {
                    Level& L = sm.lv[nl - 1];
                    L.pa = L.pb = L.pc = 0.f;
                    L.front = L.back = INFINITY;
                    L.cull = -1.f;
                    L.plane = -1;
                }
            }
            if (lane == 0) sm.nl = nl;
        }
        uint4* t4 = reinterpret_cast<uint4*>(sm.tile);
        for (int q = tid; q < TS * HeavyCfg<TS>::stride / 4; q += bd) t4[q] = make_uint4(kEmpty, kEmpty, kEmpty, kEmpty);
        for (int q = tid; q < NW; q += bd) sm.open[q] = 0u;
        if (PROF && tid == 0) ++p_tiles;
        __syncthreads();
        const int nl = sm.nl;
        const float ox = (float)(tx * TS), oy = (float)(ty * TS);
        // turns of as many levels each; up to 32 triangles a warp and round, the
        // same number for each
        const int n_turns = (nl + PassLevels<TS>::n - 1) / PassLevels<TS>::n, per = (nl + n_turns - 1) / max(n_turns, 1);
        const uint32_t rounds = (cnt + 32u * kWarps - 1u) / (32u * kWarps);
        const uint32_t share = (cnt + kWarps * rounds - 1u) / (kWarps * rounds);
        bool any_hole = false, any_open = false, any_some = false;
        uint32_t state = kTileLit;
        uint32_t* rec = nullptr;
#pragma unroll 1
        for (int s0 = 0; s0 < nl; s0 += per) {
            const int np = min(per, nl - s0);
            if (warp == 0) {
                const bool nested = np > 1 && order_levels<TS>(sm.lv + s0, np);
                if (lane == 0) {
                    sm.nested = nested;
                    sm.full = 0u;
                }
            }
            for (int q = tid; q < np * NW; q += bd) sm.cov[q] = 0u;
            __syncthreads();
            const Level* lv = sm.lv + s0;
            const bool nested = sm.nested != 0;
            const uint32_t all = (2u << (np - 1)) - 1u;
            uint32_t full = 0u;
#pragma unroll 1
            for (uint32_t b0 = share * warp; b0 < cnt; b0 += share * kWarps) {
                full |= *(volatile uint32_t*)&sm.full;
                full = __reduce_or_sync(0xffffffffu, full);
                if (full == all) break;  // every sample of these levels is shaded
                TriWork w;
                w.front = w.deep = 0u;
                w.whole = false;
                if ((uint32_t)lane < share && b0 + lane < cnt)
                    classify_tri<TS, PROF>(J, B, lp, ls, (int)B.bins[off + b0 + lane], ox, oy, sm.lv, nl, s0, np, w,
                                           p_culled);
                const uint32_t f = full_after(__reduce_or_sync(0xffffffffu, w.whole ? w.front : 0u), nested, all);
                if (f & ~full) {
                    full |= f;
                    if (lane == 0) atomicOr(&sm.full, f);
                }
                if (full == all || !__any_sync(0xffffffffu, (w.front | w.deep) != 0u)) continue;
                draw_tris<TS, true, PROF>(sm.d[warp], w, full, nested, lv, sm.cov, sm.open, sm.tile, lp, u24, p_visits,
                                          p_writes);
                if (b0 + share * kWarps < cnt) full = full_levels<TS>(sm.cov, np, nested, full);
            }
            __syncthreads();
            full = sm.full;
            uint32_t some = 0u, hole = 0u, op = 0u;
            finish_words<TS>(sm.cov, np, nested, full, tid, bd, some, hole);
            if (s0 + per >= nl)
                for (int q = tid; q < NW; q += bd) op |= sm.open[q];
            any_hole |= __syncthreads_or(hole != 0u) != 0;
            any_open |= __syncthreads_or(op != 0u) != 0;
            any_some |= __syncthreads_or(some != 0u) != 0;
            // the record: once it is known to be needed, or before the bits of
            // the first of several turns are replaced
            if (s0 == 0 && (n_turns > 1 || (any_hole && (any_some || any_open)))) {
                const uint32_t words = (uint32_t)(rec_head(nl) + nl * NW + (any_open || n_turns > 1 ? NW + TS * TS : 0));
                if (tid == 0) sm.state = alloc_record(B, W, words);
                __syncthreads();
                state = sm.state;
                if (state) rec = B.cov + 4 * (size_t)(state - 1u);
            }
            if (rec) {
#pragma unroll 1
                for (int l = warp; l < np; l += kWarps) {
                    const uint32_t box = texel_box<TS>(sm.cov + l * NW, sm.open);
                    if (lane == 0) rec[rec_box(nl) + s0 + l] = box;
                }
                if (tid < np) rec[kRecPlane + s0 + tid] = (uint32_t)lv[tid].plane;
                uint32_t* dst = rec + rec_head(nl) + s0 * NW;
                for (int q = tid; q < np * NW; q += bd) dst[q] = sm.cov[q];
            }
            __syncthreads();  // the bits may be replaced
        }
        if (rec) {
            if (tid == 0) rec[0] = (uint32_t)nl | kRecHeavy | (any_open ? kRecOpen | kRecDepth : 0u);
            if (nl + tid < rec_planes(nl)) rec[kRecPlane + nl + tid] = kNoPlane;
            if (any_open) {
                uint32_t* dst = rec + rec_head(nl) + nl * NW;
                for (int q = tid; q < NW; q += bd) dst[q] = sm.open[q];
                dst += NW;
                for (int q = tid; q < TS * TS; q += bd) dst[q] = sm.tile[q + q / TS * (HeavyCfg<TS>::stride - TS)];
            }
        }
        if (!any_hole) state = kTileFullHeavy;
        else if (!any_some && !any_open) state = kTileLit;
        if (tid == 0) B.t_cnt[te] = state;
        __syncthreads();  // the tile's shared memory may be reused
    }
    if (PROF) {
        flush_profile(B, 0u, p_visits, p_visits + p_writes, p_culled);
        flush_profile2(B, 0u, p_tiles, 0u, 0u, 0u);
        flush_heavy(B, 0u, p_visits + p_writes, p_tiles);
    }
}

// ---------------------------------------------------------------------------
// PV model per (step, module) from the cell tallies (Section 2, step 4)
// ---------------------------------------------------------------------------
constexpr int kPvThreads = 128;

// The diffuse shading fractions of local step ls: the row of its pose bin
// (tracked generators) or the generator's one row; nullptr when the diffuse
// term is not shaded.
__device__ __forceinline__ const float* diffuse_row(const JobDev& J, int ls)
{
    if (!J.fdiff) return nullptr;
    return J.fbin ? J.fdiff + (int64_t)J.fbin[J.step0 + ls] * J.fstride : J.fdiff;
}

// Irradiance per cell, substring currents, MPP over the bypass states.  All
// threads of the block call it with the cell counts in shared memory.
__device__ void module_pv(const JobDev& J, const ModuleDev& M, const ModStep& s, const LightParams& lp,
                          const uint32_t* s_cnt, uint32_t* s_imin, const Buffers& B, int64_t msi)
{
    const int ncell = M.cu * M.cv;
    const float beam = lp.dni * fmaxf(0.f, s.cosi);
    const float diff = lp.dhi * (1.f + s.nz) * 0.5f;
    const float inv_nn = 1.f / J.nn;
    const int* csub = J.lay_sub + J.lay_off[M.layout];
    const float* fd = diffuse_row(J, (int)((msi - J.ms_base) / J.n_mods));
    for (int c = threadIdx.x; c < ncell; c += blockDim.x) {
        const float f = s_cnt[c] * inv_nn;
        const float gd = fd ? diff * (1.f - fd[M.cell_base + c]) : diff;
        const float G = beam * (1.f - f) + gd;
        const float I = J.i_ref * G * 1e-3f;
        atomicMin(&s_imin[csub[c]], __float_as_uint(I));  // I >= 0: uint order = float order
    }
    __syncthreads();
    if (J.n_str) {  // substring currents for the series-string model (k_string)
        const int ls = (int)((msi - J.ms_base) / J.n_mods);
        const int m = (int)(&M - J.mods);
        float* ss = B.ss_i + J.ss_base + (int64_t)ls * J.n_sub_tot + J.sub_base[m];
        for (int k = threadIdx.x; k < M.n_sub; k += blockDim.x) ss[k] = __uint_as_float(s_imin[k]);
        if (threadIdx.x == 0) B.ms_iu[msi] = J.i_ref * (beam + diff) * 1e-3f;
    }
    if (threadIdx.x == 0) {
        const int* nk = J.lay_nk + J.lay_nk_off[M.layout];
        const int ns = M.n_sub;
        float best = 0.f, vsum = 0.f;
        for (int k = 0; k < ns; ++k) {
            const float ik = __uint_as_float(s_imin[k]);
            float volt = 0.f;
            for (int q = 0; q < ns; ++q)
                volt += __uint_as_float(s_imin[q]) >= ik ? nk[q] * J.v_cell : -J.v_diode;
            best = fmaxf(best, ik * volt);
            vsum += nk[k] * J.v_cell;
        }
        B.ms_p[msi] = best;
        B.ms_pu[msi] = J.i_ref * (beam + diff) * 1e-3f * vsum;
        B.ms_beam[msi] = beam;
    }
}

__device__ __forceinline__ void zero_step_module(const JobDev& J, const ModuleDev& M, int ls, int64_t msi,
                                                 const Buffers& B)
{
    const int ncell = M.cu * M.cv, C = J.n_cells;
    const int64_t row = (int64_t)(J.out_row0 + ls);
    if (threadIdx.x == 0) { B.ms_p[msi] = 0.f; B.ms_pu[msi] = 0.f; B.ms_beam[msi] = 0.f; }
    for (int c = threadIdx.x; c < ncell; c += blockDim.x) {
        tally_set(B.cs_cnt, J.cs_base + (int64_t)ls * C + M.cell_base + c, 0u);
        if (J.out_counts) J.out_counts[row * J.out_cstride + M.cell_base + c] = 0;
        if (J.out_bits) J.out_bits[row * J.out_cstride + M.cell_base + c] = 0ull;
    }
}

// ---------------------------------------------------------------------------
// k_pv, k_cells: fused path -- the PV model per (step, module) (Section 2, step
// 4), with the shaded samples per cell from the tiles' coverage
//
// k_pv, one (step, module) per lane: a module over lit tiles only (most of
// them) carries one current in every cell, so its maximum power point needs no
// cell; the others, and all when the diffuse term or an output is per cell,
// are listed.  k_cells takes the list one module a warp (the modules of a
// shaded table are neighbours: left to the warp that found them, 32 in a row
// kept one warp busy while others had none), or one a block when there are
// fewer modules than half the warps, a lane per cell: the texels of
// the cell's extreme samples box those of all (a sample's texel is monotone in
// its indices), and where nothing in that box is covered, or all of it, the
// cell is lit or shaded whole; the samples of the remaining cells are shared
// out over the lanes.  Nothing is accumulated across tiles, so there are no
// tallies to clear and no atomics in device memory.  Bound by instruction
// issue (71 % of the slots on a wave of 12,000 tracker modules, 256 suns: 1.13
// ms), most of it the samples of mixed cells.
// ---------------------------------------------------------------------------
constexpr int kPvTiles = 8;    // k_pv: a module over more tiles is looked at by the whole warp
constexpr int kPvFastSub = 8;  // up to so many substrings a module's voltages are summed in order
constexpr int kCellWarps = 8, kCellBlocks = 4;  // warps a block, blocks an SM
// k_cells: texels a sample from which a cell's few samples are looked up one by
// one without a look at the rows of their box first (23 tracked modules, 2 x 2
// samples a cell, 2048 x 2048 texels, 253 suns: the PV stage 154 -> 103 us, the
// same from 4 texels on; there the facade's year, 8 x 8 samples on cells of 11
// x 11 texels, would go from 4.55 to 4.90 ms)
constexpr int kSparseCell = 16;

// Level of plane `plane` in a tile's record (header word h), and its coverage
// bits.
__device__ __forceinline__ int level_of(const uint32_t* rec, uint32_t h, int plane)
{
    const int nl = (int)(h & kRecLevels);
    const uint4* p = reinterpret_cast<const uint4*>(rec + kRecPlane);
#pragma unroll 1
    for (int l = 0; l < nl - 1; l += 4) {
        const uint4 v = p[l >> 2];
        if (v.x == (uint32_t)plane) return l;
        if (v.y == (uint32_t)plane) return l + 1;
        if (v.z == (uint32_t)plane) return l + 2;
        if (v.w == (uint32_t)plane) return l + 3;
    }
    return nl - 1;  // the last level takes every other plane
}
__device__ __forceinline__ const uint32_t* level_words(const uint32_t* rec, uint32_t h, int plane, int words)
{
    return rec + rec_head((int)(h & kRecLevels)) + level_of(rec, h, plane) * words;
}

// The words of a row of TS / 32 coverage words, together.
template <int TS>
struct RowWords {
    uint32_t v[TS / 32];
};
template <int TS>
__device__ __forceinline__ RowWords<TS> load_row(const uint32_t* p)
{
    RowWords<TS> r;
    if constexpr (TS == 128) {
        const uint4 v = *reinterpret_cast<const uint4*>(p);
        r.v[0] = v.x; r.v[1] = v.y; r.v[2] = v.z; r.v[3] = v.w;
    } else if constexpr (TS == 64) {
        const uint2 v = *reinterpret_cast<const uint2*>(p);
        r.v[0] = v.x; r.v[1] = v.y;
    } else {
        r.v[0] = *p;
    }
    return r;
}

// Is the sample at texel (ix, iy), depth d, bias, of a receiver of plane
// `plane` shaded?  tc: the states of the step's tiles.
template <int TS, bool PROF>
__device__ __forceinline__ bool sample_shaded(const Buffers& B, const uint32_t* tc, int tiles_x, int ix, int iy, float d,
                                              float bias, int plane, const LightParams& lp, int u24,
                                              unsigned int& samples, unsigned int& h_samples, unsigned int& pairs)
{
    constexpr int SH = TileSh<TS>::v, WPR = TS / 32, NW = TS * WPR;
    const uint32_t state = tc[(iy >> SH) * tiles_x + (ix >> SH)];
    if (state == kTileLit) return false;
    if (PROF) ++samples;
    if (state >= kTileFullHeavy) {
        if (PROF && state == kTileFullHeavy) ++h_samples;
        return true;
    }
    const uint32_t* rec = B.cov + 4 * (size_t)(state - 1u);
    const uint32_t h = rec[0];
    if (PROF && (h & kRecHeavy)) ++h_samples;
    const int lx = ix & (TS - 1), ly = iy & (TS - 1), word = ly * WPR + (lx >> 5);
    if ((level_words(rec, h, plane, NW)[word] >> (lx & 31)) & 1u) return true;
    if (!(h & kRecOpen)) return false;
    const uint32_t* open = rec + rec_head((int)(h & kRecLevels)) + (int)(h & kRecLevels) * NW;
    if (!((open[word] >> (lx & 31)) & 1u)) return false;
    if (h & kRecDepth) {
        const uint32_t key = open[NW + ly * TS + lx];
        return behind_key(d, bias, key, lp.dnear, lp.qscale, u24);
    }
    const TriS* tri = reinterpret_cast<const TriS*>(open + NW);
    const float px = texel_centre(lx), py = texel_centre(ly);
#pragma unroll 1
    for (int t = 0; t < (int)(h >> 16); ++t) {
        if (PROF) ++pairs;
        if (tri_shades(tri[t], px, py, d, bias, lp, u24)) return true;
    }
    return false;
}

// The map path and all before the coverage bits look for a tile's samples by
// mapping the tile back onto the module (stage_one's box, row_range), one sample
// more each side.  Where that map magnifies the rounding of positions to more
// than that -- 2: the sun all but in the module's plane, anywhere; 1: an axis of
// texels all but constant along the module's rows, at the tile's border -- some
// samples are not found, and count as lit.  The counts stay what they were:
// sample_found asks for such samples one by one.
__device__ __forceinline__ int find_risk(const ModStep& s, float lu, float lv, float inv_p, int R)
{
    const float ext = fabsf(lu * s.tax) + fabsf(lv * s.tbx) + fabsf(lu * s.tay) + fabsf(lv * s.tby) + 256.f;
    const float e = 5e-7f * ((float)R + ext) * inv_p;
    const float p0 = fabsf(s.tax * s.tby), p1 = fabsf(s.tay * s.tbx), det = fabsf(s.tax * s.tby - s.tay * s.tbx);
    if (det > 1e-6f * (p0 + p1) &&
        e * fmaxf(fabsf(s.tbx) + fabsf(s.tby), fabsf(s.tax) + fabsf(s.tay)) > 0.5f * det)
        return 2;
    return (fabsf(s.tax) > 1e-6f && e > 0.5f * fabsf(s.tax)) || (fabsf(s.tay) > 1e-6f && e > 0.5f * fabsf(s.tay));
}

// Is sample (I, Jr) of the module of touch-list entry e among those that tile
// (tx, ty) finds?
template <int TS>
__device__ __noinline__ bool sample_found(const JobDev* jobs, const Buffers& B, unsigned int e, int tx, int ty, int I,
                                          int Jr)
{
    const uint4 entry = B.touch[e];
    RecvSm R;
    stage_one<TS>(R, jobs[entry.x & 0x7FFFFFFFu], B, (int)entry.y, tx, ty, (int)entry.z);
    if (R.item_pref == 0 || I < R.I0 || I > R.I1 || Jr < R.J0 || (Jr - R.J0) * R.ncol >= R.item_pref) return false;
    int Ib = R.I0, Ie = R.I1;
    row_range(R, Jr, Ib, Ie);
    return I >= Ib && I <= Ie;
}

// Cells of a module some of whose samples are shaded, and some not: coverage
// and open bits of their texel box (bit 8 r + c: row r, column c of the box),
// first sample indices and first texel.  A box larger than 8 x 8 (big) has no
// bits: in cov its tile's coverage words (address), in open.x the distance of
// the open words to them (0: none); or none of these (0), when it meets
// several tiles and its samples look their tiles up one by one.
struct CellQueue {
    uint2 cov[32], open[32];
    uint32_t ij[32], xy[32];
    uint32_t big;  // bit k: entry k is big
    int risk;            // the module's find_risk
    unsigned int entry;  // and its place in the list
};

// floor of one coordinate of the sample at (a, b) along the module axes, as
// sample_texel has it.
__device__ __forceinline__ int axis_texel(float a, float b, float ta, float tb, float t0, float r_max)
{
    return texel_floor(__fmaf_rn(a, ta, __fmaf_rn(b, tb, t0)), r_max);
}

// Shaded samples of cell c of a module (have: c is one), a lane per cell, for
// one full warp and one module; `bits` receives the flags of samples k = j * n
// + i < 64.  tc: the states of the step's tiles.
template <int TS, bool PROF>
__device__ __forceinline__ int cell_shaded(const Buffers& B, const JobDev& J, const ModStep& s, int cu, int plane,
                                           float p_over_n, const LightParams& lp, int u24, const uint32_t* tc, int c,
                                           bool have, const JobDev* jobs, CellQueue& Q, unsigned long long& bits, unsigned int& cand,
                                           unsigned int& samples, unsigned int& h_samples, unsigned int& pairs)
{
    constexpr int SH = TileSh<TS>::v, WPR = TS / 32, NW = TS * WPR;
    const int lane = threadIdx.x & 31;
    const int n = J.n, nn = J.nn, tiles_x = J.tiles_x;
    const float r_max = (float)(J.R - 1);
    bool full = false, mixed = false, big = false;
    int I0 = 0, J0 = 0, x0 = 0, y0 = 0, xe = -1, ye = -1;
    if (have) {
        const int cv = fdiv(c, cu, __frcp_rn((float)cu));
        I0 = (c - cv * cu) * n;
        J0 = cv * n;
        // along each module axis the end samples reach the least and the
        // largest texel of either coordinate
        const float a0 = __fmul_rn((float)I0 + 0.5f, p_over_n), a1 = __fmul_rn((float)(I0 + n - 1) + 0.5f, p_over_n);
        const float b0 = __fmul_rn((float)J0 + 0.5f, p_over_n), b1 = __fmul_rn((float)(J0 + n - 1) + 0.5f, p_over_n);
        x0 = axis_texel(s.tax > 0.f ? a0 : a1, s.tbx > 0.f ? b0 : b1, s.tax, s.tbx, s.tx0, r_max);
        y0 = axis_texel(s.tay > 0.f ? a0 : a1, s.tby > 0.f ? b0 : b1, s.tay, s.tby, s.ty0, r_max);
        const int x1 = axis_texel(s.tax > 0.f ? a1 : a0, s.tbx > 0.f ? b1 : b0, s.tax, s.tbx, s.tx0, r_max);
        const int y1 = axis_texel(s.tay > 0.f ? a1 : a0, s.tby > 0.f ? b1 : b0, s.tay, s.tby, s.ty0, r_max);
        xe = x1;
        ye = y1;
        big = x1 - x0 > 7 || y1 - y0 > 7;
    }
    uint32_t clo = 0u, chi = 0u, olo = 0u, ohi = 0u;  // rows 0-3 and 4-7 of the box's bits
    bool some = false, hole = false;
    const uint32_t* word = nullptr;  // big, one tile: its coverage words
    int odist = 0;
    if (have) {
        const int txa = x0 >> SH, txb = xe >> SH, tya = y0 >> SH, tyb = ye >> SH;
#pragma unroll 1
        for (int ty = tya; ty <= tyb; ++ty)
#pragma unroll 1
            for (int tx = txa; tx <= txb; ++tx) {
                const uint32_t state = tc[ty * tiles_x + tx];
                if (state == kTileLit) {
                    hole = true;
                    continue;
                }
                const int lx0 = max(x0 - (tx << SH), 0), lx1 = min(xe - (tx << SH), TS - 1);
                const int ly0 = max(y0 - (ty << SH), 0), ly1 = min(ye - (ty << SH), TS - 1);
                const bool all = state >= kTileFullHeavy;
                const uint32_t* w = nullptr;  // the level's coverage
                int o = 0;                    // its distance to the open bits, 0: none
                if (!all) {
                    const uint32_t* rec = B.cov + 4 * (size_t)(state - 1u);
                    const uint32_t h = rec[0];
                    w = level_words(rec, h, plane, NW);
                    const int nl = (int)(h & kRecLevels);
                    if (h & kRecOpen) o = (int)(rec + rec_head(nl) + nl * NW - w);
                }
                if (!big) {
                    const int q = lx0 >> 5, col = (tx << SH) + lx0 - x0, row = (ty << SH) + ly0 - y0;
                    const uint32_t m = (2u << (lx1 - lx0)) - 1u;
#pragma unroll 1
                    for (int r = 0; r <= ly1 - ly0; ++r) {
                        const int sh = 8 * ((row + r) & 3) + col;
                        uint32_t v = 0xFFFFFFFFu;
                        if (!all) {
                            const uint32_t* wr = w + (ly0 + r) * WPR + q;
                            const bool two = WPR > 1 && q + 1 < WPR;
                            v = WPR > 1 ? __funnelshift_r(wr[0], two ? wr[1] : 0u, lx0 & 31) : wr[0] >> lx0;
                            if (o) {
                                const uint32_t p =
                                    WPR > 1 ? __funnelshift_r(wr[o], two ? wr[o + 1] : 0u, lx0 & 31) : wr[o] >> lx0;
                                if (row + r < 4) olo |= (p & m) << sh;
                                else ohi |= (p & m) << sh;
                            }
                        }
                        if (row + r < 4) clo |= (v & m) << sh;
                        else chi |= (v & m) << sh;
                        hole = hole || (~v & m) != 0u;
                    }
                } else if (all) {
                    some = true;
                } else if ((xe - x0 + 1) * (ye - y0 + 1) >= kSparseCell * nn) {
                    some = hole = true;
                    if (txa == txb && tya == tyb) {
                        word = w;
                        odist = o;
                    }
                } else {
                    RowWords<TS> m;
                    uint32_t sm = 0u, hl = 0u;
#pragma unroll
                    for (int k = 0; k < WPR; ++k) m.v[k] = span_word(lx0, lx1, k);
#pragma unroll 4
                    for (int ly = ly0; ly <= ly1; ++ly) {
                        const RowWords<TS> v = load_row<TS>(w + ly * WPR);
#pragma unroll
                        for (int k = 0; k < WPR; ++k) {
                            sm |= v.v[k] & m.v[k];
                            hl |= ~v.v[k] & m.v[k];
                        }
                    }
                    if (o && sm == 0u) {
#pragma unroll 1
                        for (int ly = ly0; ly <= ly1; ++ly) {
                            const RowWords<TS> v = load_row<TS>(w + o + ly * WPR);
#pragma unroll
                            for (int k = 0; k < WPR; ++k) sm |= v.v[k] & m.v[k];
                        }
                    }
                    some = some || sm != 0u;
                    hole = hole || hl != 0u;
                    if (txa == txb && tya == tyb) {
                        word = w;
                        odist = o;
                    }
                }
            }
        some = some || (clo | chi | olo | ohi) != 0u;
        // (a box at a tile's border: texel coordinates 0 or TS - 1)
        const int risk = Q.risk;
        if (risk && !hole && (risk == 2 || x0 >> SH != (x0 - 1) >> SH || xe >> SH != (xe + 1) >> SH ||
                              y0 >> SH != (y0 - 1) >> SH || ye >> SH != (ye + 1) >> SH || txa != txb || tya != tyb)) {
            hole = some = big = true;
            word = nullptr;
        }
        full = !hole;
        mixed = some && hole;
        if (PROF) {
            cand += (unsigned int)nn;
            if (full) samples += (unsigned int)nn;
        }
    }
    int cnt = full ? nn : 0;
    bits = full ? (nn >= 64 ? ~0ull : (1ull << nn) - 1ull) : 0ull;
    const unsigned int mx = __ballot_sync(0xffffffffu, mixed);
    if (mx == 0u) return cnt;
    // the samples of the mixed cells, nn each, over the lanes
    const int rank = __popc(mx & ((1u << lane) - 1u));
    if (lane == 0) Q.big = 0u;
    __syncwarp();
    if (mixed) {
        if (big) {
            const unsigned long long p = (unsigned long long)(uintptr_t)word;
            clo = (uint32_t)p;
            chi = (uint32_t)(p >> 32);
            olo = (uint32_t)odist;
        }
        Q.cov[rank] = make_uint2(clo, chi);
        Q.open[rank] = make_uint2(olo, ohi);
        Q.ij[rank] = (uint32_t)I0 | ((uint32_t)J0 << 16);
        Q.xy[rank] = (uint32_t)x0 | ((uint32_t)y0 << 16);
        if (big) atomicOr(&Q.big, 1u << rank);
    }
    __syncwarp();
    const int total = __popc(mx) * nn;
    const uint32_t bigs = Q.big;
    const float inv_n = __frcp_rn((float)n);
    // sample base + lane: entry r, sample kk of its cell
    const int step_r = 32 / nn, step_k = 32 - step_r * nn;
    int r = lane / nn, kk = lane - r * nn;
#pragma unroll 1
    for (int base = 0; base < total; base += 32) {
        bool hit = false;
        if (base + lane < total) {
            const int jj = fdiv(kk, n, inv_n), ii = kk - jj * n;
            const uint32_t e = Q.ij[r], xy = Q.xy[r];
            float d;
            int ix, iy;
            sample_texel(s, sample_row(s, (int)(e >> 16) + jj, p_over_n), (float)((int)(e & 0xFFFFu) + ii) + 0.5f,
                         p_over_n, r_max, ix, iy, d);
            const uint2 cv = Q.cov[r], op = Q.open[r];
            bool look;
            if (!((bigs >> r) & 1u)) {
                const int bit = 8 * (iy - (int)(xy >> 16)) + ix - (int)(xy & 0xFFFFu);
                hit = (((bit < 32 ? cv.x : cv.y) >> (bit & 31)) & 1u) != 0u;
                look = !hit && (((bit < 32 ? op.x : op.y) >> (bit & 31)) & 1u) != 0u;
            } else {
                const uint32_t* w = reinterpret_cast<const uint32_t*>((uintptr_t)(((unsigned long long)cv.y << 32) | cv.x));
                look = w == nullptr;
                if (w) {
                    const int k2 = (iy & (TS - 1)) * WPR + ((ix & (TS - 1)) >> 5);
                    hit = ((w[k2] >> (ix & 31)) & 1u) != 0u;
                    look = !hit && op.x && ((w[(int)op.x + k2] >> (ix & 31)) & 1u) != 0u;
                }
            }
            if (PROF && !look) ++samples;
            if (look)
                hit = sample_shaded<TS, PROF>(B, tc, tiles_x, ix, iy, d, s.bias, plane, lp, u24, samples, h_samples,
                                              pairs);
            const int risk = Q.risk;
            if (risk && hit && (risk == 2 || ((ix + 1) & (TS - 1)) < 2 || ((iy + 1) & (TS - 1)) < 2))
                hit = sample_found<TS>(jobs, B, Q.entry, ix >> SH, iy >> SH, (int)(e & 0xFFFFu) + ii, (int)(e >> 16) + jj);
        }
        r += step_r;
        kk += step_k;
        if (kk >= nn) {
            kk -= nn;
            ++r;
        }
        const uint32_t ball = __ballot_sync(0xffffffffu, hit);
        if (mixed) {
            // this cell's samples among the 32: lanes [a, b)
            const int a = max(rank * nn - base, 0), b = min((rank + 1) * nn - base, 32);
            if (a < b) {
                const uint32_t part = (ball >> a) & (b - a >= 32 ? 0xFFFFFFFFu : (1u << (b - a)) - 1u);
                cnt += __popc(part);
                const int sh = base + a - rank * nn;  // the first of them, within the cell
                if (sh < 64) bits |= (unsigned long long)part << sh;
            }
        }
    }
    __syncwarp();  // the queue may be replaced
    return cnt;
}

// The cells of a module some sample of which may read a texel of the box
// [x0, x1] x [y0, y1]: first column | columns << 8 | first row << 16 | rows <<
// 24 (the box's corners, two texels wider, mapped back onto the module; every
// cell if the module is seen edge-on).  False if there are none.
__device__ __forceinline__ bool cell_box(const ModStep& s, const ModuleDev& M, int x0, int x1, int y0, int y1,
                                         uint32_t& cells)
{
    int ca = 0, cols = M.cu, ra = 0, rows = M.cv;
    if (s.hs < FLT_MAX) {  // the module has a plane
        const float inv = 1.f / ((s.tax * s.tby - s.tay * s.tbx) * M.pitch);
        const float px0 = (float)(x0 - 2) - s.tx0, px1 = (float)(x1 + 3) - s.tx0;
        const float py0 = (float)(y0 - 2) - s.ty0, py1 = (float)(y1 + 3) - s.ty0;
        const float axl = s.tby * inv, axr = -s.tbx * inv, bxl = -s.tay * inv, bxr = s.tax * inv;
        const float amin = fminf(axl * px0, axl * px1) + fminf(axr * py0, axr * py1);
        const float amax = fmaxf(axl * px0, axl * px1) + fmaxf(axr * py0, axr * py1);
        const float bmin = fminf(bxl * px0, bxl * px1) + fminf(bxr * py0, bxr * py1);
        const float bmax = fmaxf(bxl * px0, bxl * px1) + fmaxf(bxr * py0, bxr * py1);
        ca = (int)fminf(fmaxf(floorf(amin), 0.f), (float)M.cu);
        ra = (int)fminf(fmaxf(floorf(bmin), 0.f), (float)M.cv);
        cols = (int)fminf(fmaxf(ceilf(amax), 0.f), (float)M.cu) - ca;
        rows = (int)fminf(fmaxf(ceilf(bmax), 0.f), (float)M.cv) - ra;
    }
    cells = (uint32_t)ca | ((uint32_t)cols << 8) | ((uint32_t)ra << 16) | ((uint32_t)rows << 24);
    return cols > 0 && rows > 0;
}

// Add the covered and open texels of tile t of module m's range to a box.
__device__ __forceinline__ void add_tile_box(const Buffers& B, const JobDev& J, int ls, int m, const TileRange& tr, int t,
                                             int sh, int& x0, int& x1, int& y0, int& y1)
{
    const int wx = tr.tx1 - tr.tx0 + 1;
    const int ty = tr.ty0 + t / wx, tx = tr.tx0 + t % wx;
    const uint32_t state = B.t_cnt[J.te_base + (int64_t)ls * J.tiles_x * J.tiles_x + (int64_t)ty * J.tiles_x + tx];
    if (state == kTileLit) return;
    const int side = (1 << sh) - 1;
    uint32_t box = (uint32_t)side << 8 | (uint32_t)side << 24;
    if (state < kTileFullHeavy) {
        const uint32_t* rec = B.cov + 4 * (size_t)(state - 1u);
        const uint32_t h = rec[0];
        box = rec[rec_box((int)(h & kRecLevels)) + level_of(rec, h, J.mods[m].plane)];
    }
    if (box == kBoxNone) return;
    x0 = min(x0, (tx << sh) + (int)(box & 255u));
    x1 = max(x1, (tx << sh) + (int)((box >> 8) & 255u));
    y0 = min(y0, (ty << sh) + (int)((box >> 16) & 255u));
    y1 = max(y1, (ty << sh) + (int)(box >> 24));
}

__global__ void __launch_bounds__(kPvThreads) k_pv(const WaveDev* __restrict__ W, const JobDev* __restrict__ jobs,
                                                   Buffers B)
{
    const int64_t tot = W->tot_mod;
    const int nj = W->n_jobs, sh = W->tile_sh;
    // incomplete bins (pool overflow, the wave is rerun): the tiles have no state
    const bool tiles_ok = !(B.ctr->overflow & 1u);
    const int lane = threadIdx.x & 31;
    // a warp takes bw items: 32, or fewer so that a small wave spreads over
    // all warps
    const int64_t n_warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    int bw = 32;
    while (bw > 1 && n_warps * (bw >> 1) >= tot) bw >>= 1;
    for (int64_t base = ((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5) * bw; base < tot; base += n_warps * bw) {
        const int64_t item = lane < bw ? base + lane : tot;
        bool list = false, touched = false;
        int j = 0, ls = 0, m = 0;
        uint32_t cells = 0u;  // the cells that a covered or open texel may reach (cell_box)
        bool lit = false;
        float beam = 0.f, diff = 0.f;
        TileRange tr{};
        int nt = 0;
        if (item < tot) {
            j = job_of(nj, item, [&](int q) { return jobs[q].it_mod; });
            const JobDev& J = jobs[j];
            const int64_t li = item - J.it_mod;
            ls = (int)(li / J.n_mods);
            m = (int)(li - (int64_t)ls * J.n_mods);
            const int64_t msi = J.ms_base + li;
            const LightParams& lp = B.lp[J.js_base + ls];
            const ModuleDev& M = J.mods[m];
            lit = lp.valid != 0;
            list = lit && (J.fdiff || M.n_sub > kPvFastSub);
            if (lit) {
                const ModStep s = B.ms[msi];
                beam = lp.dni * fmaxf(0.f, s.cosi);
                diff = lp.dhi * (1.f + s.nz) * 0.5f;
                tr = module_tiles(s, M, J.R, sh);
                nt = tiles_ok ? (tr.tx1 - tr.tx0 + 1) * (tr.ty1 - tr.ty0 + 1) : 0;
            }
        }
        // box of the texels covered or open in the module's tiles: by its lane,
        // or by the warp for a module over many tiles
        int x0 = INT_MAX, x1 = -1, y0 = INT_MAX, y1 = -1;
        for (int t = 0; t < (nt <= kPvTiles ? nt : 0); ++t)
            add_tile_box(B, jobs[j], ls, m, tr, t, sh, x0, x1, y0, y1);
#pragma unroll 1
        for (unsigned int many = __ballot_sync(0xffffffffu, nt > kPvTiles); many; many &= many - 1u) {
            const int q = __ffs((int)many) - 1;
            const int jq = __shfl_sync(0xffffffffu, j, q), lq = __shfl_sync(0xffffffffu, ls, q);
            const int mq = __shfl_sync(0xffffffffu, m, q), nq = __shfl_sync(0xffffffffu, nt, q);
            TileRange tq;
            tq.tx0 = __shfl_sync(0xffffffffu, tr.tx0, q); tq.tx1 = __shfl_sync(0xffffffffu, tr.tx1, q);
            tq.ty0 = __shfl_sync(0xffffffffu, tr.ty0, q);
            int a0 = INT_MAX, a1 = -1, b0 = INT_MAX, b1 = -1;
            for (int t = lane; t < nq; t += 32) add_tile_box(B, jobs[jq], lq, mq, tq, t, sh, a0, a1, b0, b1);
            a0 = __reduce_min_sync(0xffffffffu, a0); a1 = __reduce_max_sync(0xffffffffu, a1);
            b0 = __reduce_min_sync(0xffffffffu, b0); b1 = __reduce_max_sync(0xffffffffu, b1);
            if (lane == q) { x0 = a0; x1 = a1; y0 = b0; y1 = b1; }
        }
        if (item < tot) {
            const JobDev& J = jobs[j];
            const ModuleDev& M = J.mods[m];
            const int64_t msi = J.ms_base + (int64_t)ls * J.n_mods + m;
            if (x1 >= 0) touched = cell_box(B.ms[msi], M, x0, x1, y0, y1, cells);
            const int ns = M.n_sub;
            list = list || touched;
            if (!list) {
                // every substring carries the module's one current, and the
                // voltage at it is the sum over all of them (k_cells' terms,
                // rounded as there)
                float best = 0.f, vsum = 0.f;
                if (lit) {
                    const float I = J.i_ref * (beam * 1.f + diff) * 1e-3f;
                    const int* nk = J.lay_nk + J.lay_nk_off[M.layout];
                    float volt = 0.f;
#pragma unroll 1
                    for (int k = 0; k < ns; ++k) {
                        volt = __fadd_rn(volt, __fmul_rn((float)nk[k], J.v_cell));
                        vsum += nk[k] * J.v_cell;
                    }
                    best = fmaxf(0.f, I * volt);
                    if (J.n_str) {  // substring currents for the series-string model (k_string)
                        float* ss = B.ss_i + J.ss_base + (int64_t)ls * J.n_sub_tot + J.sub_base[m];
                        for (int k = 0; k < ns; ++k) ss[k] = I;
                        B.ms_iu[msi] = J.i_ref * (beam + diff) * 1e-3f;
                    }
                    vsum = J.i_ref * (beam + diff) * 1e-3f * vsum;
                }
                B.ms_p[msi] = best;
                B.ms_pu[msi] = vsum;
                B.ms_beam[msi] = beam;
            }
        }
        const unsigned int bal = __ballot_sync(0xffffffffu, list);
        unsigned int pos = 0;
        if (lane == 0 && bal) pos = atomicAdd(&B.ctr->n_touch, (unsigned int)__popc(bal));
        pos = __shfl_sync(0xffffffffu, pos, 0) + __popc(bal & ((1u << lane) - 1u));
        if (list) B.touch[pos] = make_uint4((uint32_t)j | (touched ? 1u << 31 : 0u), (uint32_t)ls, (uint32_t)m, cells);
    }
}

template <int TS, bool PROF>
__global__ void __launch_bounds__(kCellWarps * 32, kCellBlocks) k_cells(const WaveDev* __restrict__ W,
                                                              const JobDev* __restrict__ jobs, Buffers B)
{
    __shared__ CellQueue s_queue[kCellWarps];
    __shared__ uint32_t s_imin[kCellWarps][kMaxSub];
    unsigned int p_cand = 0, p_samples = 0, p_hsamples = 0, p_pairs = 0;
    const unsigned int n_touch = B.ctr->n_touch;
    const int u24 = W->depth_u24;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    // few modules: the block's warps share one module's cells
    const bool shared = n_touch <= gridDim.x * (kCellWarps / 2);
    uint32_t* imin = s_imin[shared ? 0 : wib];
    CellQueue& Q = s_queue[wib];
    const unsigned int e0 = shared ? blockIdx.x : blockIdx.x * kCellWarps + wib;
    const unsigned int e_stride = shared ? gridDim.x : gridDim.x * kCellWarps;
#pragma unroll 1
    for (unsigned int e = e0; e < n_touch; e += e_stride) {
        const uint4 entry = B.touch[e];
        const bool touched = (entry.x >> 31) != 0u;
        const JobDev& J = jobs[entry.x & 0x7FFFFFFFu];
        const int ls = (int)entry.y, m = (int)entry.z;
        const int64_t msi = J.ms_base + (int64_t)ls * J.n_mods + m;
        const LightParams& lp = B.lp[J.js_base + ls];
        const ModuleDev& M = J.mods[m];
        const ModStep& s = B.ms[msi];
        const bool lit = lp.valid != 0;
        const int c0 = M.cell_base, ns = M.n_sub, cu = M.cu, plane = M.plane;
        const float p_over_n = __fdiv_rn(M.pitch, (float)J.n);
        if (lane == 0) {
            Q.risk = find_risk(s, cu * M.pitch, M.cv * M.pitch, 1.f / p_over_n, J.R);
            Q.entry = e;
        }
        __syncwarp();
        const float beam = lit ? lp.dni * fmaxf(0.f, s.cosi) : 0.f;
        const float diff = lit ? lp.dhi * (1.f + s.nz) * 0.5f : 0.f;
        const uint32_t* tc = B.t_cnt + J.te_base + (int64_t)ls * J.tiles_x * J.tiles_x;
        const int64_t cbase = J.cs_base + (int64_t)ls * J.n_cells + c0;
        const int64_t row = (int64_t)(J.out_row0 + ls) * J.out_cstride + c0;
        const float* fd = diffuse_row(J, ls);
        const int* csub = J.lay_sub + J.lay_off[M.layout];
        const float inv_nn = 1.f / J.nn;
        const bool few = ns <= kPvFastSub;
        // without a diffuse term per cell only the cells that a covered or open
        // texel reaches are looked at: the others carry the unshaded current,
        // which no cell exceeds, so every substring's minimum starts from it
        const bool every = fd != nullptr;
        uint32_t mine = 0x7F800000u;  // +inf; few substrings: lane k keeps substring k's minimum
        if (!every && lit) mine = __float_as_uint(J.i_ref * (beam * 1.f + diff) * 1e-3f);
        const int* nk = J.lay_nk + J.lay_nk_off[M.layout];
        const int nk_l = few && lane < ns ? nk[lane] : 0;
        if (shared) {
            if (wib == 0)
                for (int k = lane; k < ns; k += 32) imin[k] = mine;
            __syncthreads();
        } else if (!few) {
            for (int k = lane; k < ns; k += 32) imin[k] = mine;
            __syncwarp();
        }
        int ca = 0, cols = cu, ra = 0, rows = M.cv;
        if (!every) {
            ca = (int)(entry.w & 255u);
            cols = (int)((entry.w >> 8) & 255u);
            ra = (int)((entry.w >> 16) & 255u);
            rows = touched ? (int)(entry.w >> 24) : 0;
        }
        const int count = cols * rows;
        const float inv_cols = __frcp_rn((float)max(cols, 1));
        // cells at a time, one per lane
        const int per = shared ? min((count + kCellWarps - 1) / kCellWarps, 32) : 32;
#pragma unroll 1
        for (int cr = shared ? wib * per : 0; cr < count; cr += shared ? kCellWarps * per : 32) {
            const bool have = lane < per && cr + lane < count;
            const int rr = fdiv(cr + lane, max(cols, 1), inv_cols);
            const int c = (ra + rr) * cu + ca + cr + lane - rr * cols;
            unsigned long long bits = 0ull;
            int cnt = 0;
            if (touched)
                cnt = cell_shaded<TS, PROF>(B, J, s, cu, plane, p_over_n, lp, u24, tc, c, have, jobs, Q, bits, p_cand,
                                            p_samples, p_hsamples, p_pairs);
            uint32_t cur = 0x7F800000u;
            int sub = -1;
            if (have) {
                if (J.kahan_cell) tally_set(B.cs_cnt, cbase + c, (uint32_t)cnt);
                if (J.out_counts) J.out_counts[row + c] = (uint8_t)cnt;
                if (J.out_bits) J.out_bits[row + c] = bits;
                const float gd = fd ? diff * (1.f - fd[c0 + c]) : diff;
                const float G = beam * (1.f - (uint32_t)cnt * inv_nn) + gd;
                cur = __float_as_uint(J.i_ref * G * 1e-3f);  // I >= 0: uint order = float order
                sub = csub[c];
            }
            if (!lit) continue;
            if (few) {
#pragma unroll 1
                for (int k = 0; k < ns; ++k) {
                    const uint32_t v = __reduce_min_sync(0xffffffffu, sub == k ? cur : 0x7F800000u);
                    if (lane == k) mine = min(mine, v);
                }
            } else if (have) {
                atomicMin(&imin[sub], cur);
            }
        }
        if (shared) {
            if (few && lane < ns) atomicMin(&imin[lane], mine);
            __syncthreads();
            if (few && lane < ns) mine = imin[lane];
        } else {
            __syncwarp();
        }
        float best = 0.f, vsum = 0.f;
        if (lit && (!shared || wib == 0)) {
            float* ss = J.n_str ? B.ss_i + J.ss_base + (int64_t)ls * J.n_sub_tot + J.sub_base[m] : nullptr;
            if (few) {
                // lane k < ns takes candidate current k
                const float ik = __uint_as_float(mine);
                float volt = 0.f;
#pragma unroll 1
                for (int q = 0; q < ns; ++q) {
                    const float vq = __fmul_rn((float)__shfl_sync(0xffffffffu, nk_l, q), J.v_cell);
                    volt += __uint_as_float(__shfl_sync(0xffffffffu, mine, q)) >= ik ? vq : -J.v_diode;
                    vsum += nk[q] * J.v_cell;
                }
                if (lane < ns) best = fmaxf(0.f, ik * volt);
                if (ss && lane < ns) ss[lane] = ik;
            } else {
                for (int k = lane; k < ns; k += 32) {
                    const float ik = __uint_as_float(imin[k]);
                    float volt = 0.f;
#pragma unroll 1
                    for (int q = 0; q < ns; ++q)
                        volt += __uint_as_float(imin[q]) >= ik ? nk[q] * J.v_cell : -J.v_diode;
                    best = fmaxf(best, ik * volt);
                    vsum += nk[k] * J.v_cell;
                    if (ss) ss[k] = ik;
                }
#pragma unroll
                for (int off = 16; off; off >>= 1) vsum += __shfl_xor_sync(0xffffffffu, vsum, off);
            }
            best = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(best)));  // best >= 0
            if (ss && lane == 0) B.ms_iu[msi] = J.i_ref * (beam + diff) * 1e-3f;
            vsum = J.i_ref * (beam + diff) * 1e-3f * vsum;
        }
        if (lane == 0 && (!shared || wib == 0)) {
            B.ms_p[msi] = best;
            B.ms_pu[msi] = vsum;
            B.ms_beam[msi] = beam;
        }
        if (shared) __syncthreads();  // the minima may be reset
        else __syncwarp();
    }
    if (PROF) {
        flush_profile(B, p_samples, 0u, 0u, 0u);
        flush_profile2(B, p_cand, 0u, 0u, 0u, p_pairs);
        flush_heavy(B, p_hsamples, 0u, 0u);
    }
}

// ---------------------------------------------------------------------------
// k_sample: map path -- per (step, module) texel gathers from the HBM map,
// depth tests, warp-ballot cell tallies, then the PV model
// ---------------------------------------------------------------------------
template <bool PROF>
__global__ void __launch_bounds__(kPvThreads) k_sample(const WaveDev* __restrict__ W,
                                                       const JobDev* __restrict__ jobs, Buffers B)
{
    __shared__ uint32_t s_cnt[kMaxCellsPerModule];
    __shared__ unsigned long long s_bits[kMaxCellsPerModule];
    __shared__ uint32_t s_imin[kMaxSub];
    const int64_t tot = W->tot_mod;
    const int nj = W->n_jobs;
    const int sh = W->tile_sh;
    const int tmask = (1 << sh) - 1;
    const int64_t map_cap = W->map_cap_tiles;
    const int u24 = W->depth_u24;
    const int lane = threadIdx.x & 31;
    unsigned int p_samples = 0;
    for (int64_t item = blockIdx.x; item < tot; item += gridDim.x) {
        int j = job_of(nj, item, [&](int q) { return jobs[q].it_mod; });
        const JobDev& J = jobs[j];
        const int64_t li = item - J.it_mod;
        const int ls = (int)(li / J.n_mods), m = (int)(li % J.n_mods);
        const int64_t msi = J.ms_base + li;
        const LightParams& lp = B.lp[J.js_base + ls];
        const ModuleDev& M = J.mods[m];
        if (!lp.valid) {
            zero_step_module(J, M, ls, msi, B);
            continue;
        }
        const int cu = M.cu, ncell = M.cu * M.cv;
        const int n = J.n, nn = J.nn;
        const int C = J.n_cells;
        const int64_t row = (int64_t)(J.out_row0 + ls);
        const ModStep s = B.ms[msi];
        for (int c = threadIdx.x; c < ncell; c += blockDim.x) { s_cnt[c] = 0; s_bits[c] = 0ull; }
        if (threadIdx.x < kMaxSub) s_imin[threadIdx.x] = 0x7F800000u;
        __syncthreads();
        const int S = ncell * nn;
        const float p_over_n = __fdiv_rn(M.pitch, (float)n);
        const int R = J.R;
        const int64_t te0 = J.te_base + (int64_t)ls * J.tiles_x * J.tiles_x;
        for (int g0 = 0; g0 < S; g0 += blockDim.x) {
            const int g = g0 + threadIdx.x;
            bool shaded = false;
            if (g < S) {
                int c = g / nn, k = g - c * nn;
                int jj = k / n, ii = k - jj * n;
                int cv_ = c / cu, cu_ = c - cv_ * cu;
                float d;
                int ix, iy;
                const int I = cu_ * n + ii;
                sample_texel(s, sample_row(s, cv_ * n + jj, p_over_n), (float)I + 0.5f, p_over_n,
                             (float)(R - 1), ix, iy, d);
                const int64_t te = te0 + (int64_t)(iy >> sh) * J.tiles_x + (ix >> sh);
                if (J.tiles_x > 0 && B.t_cnt[te] != 0u) {
                    const uint32_t slot = B.t_slot[te];
                    if (slot < map_cap) {
                        if (PROF) ++p_samples;
                        const uint32_t key = B.map[((size_t)slot << (2 * sh)) + ((iy & tmask) << sh) + (ix & tmask)];
                        if (key != kEmpty) shaded = behind_key(d, s.bias, key, lp.dnear, lp.qscale, u24);
                    }
                }
            }
            const unsigned int ball = __ballot_sync(0xffffffffu, shaded);
            if (lane == 0 && ball) {
                const int gw = g;  // first sample of this warp
                const int glast = min(gw + 31, S - 1);
                for (int c = gw / nn; c <= glast / nn; ++c) {
                    const int lo = max(c * nn, gw), hi = min((c + 1) * nn, glast + 1);
                    const unsigned int msk = (hi - lo >= 32) ? 0xffffffffu : ((1u << (hi - lo)) - 1u);
                    const unsigned int part = (ball >> (lo - gw)) & msk;
                    if (part) {
                        atomicAdd(&s_cnt[c], (uint32_t)__popc(part));
                        if (nn <= 64) atomicOr(&s_bits[c], (unsigned long long)part << (lo - c * nn));
                    }
                }
            }
        }
        __syncthreads();
        for (int c = threadIdx.x; c < ncell; c += blockDim.x) {
            const uint32_t cnt = s_cnt[c];
            tally_set(B.cs_cnt, J.cs_base + (int64_t)ls * C + M.cell_base + c, cnt);
            if (J.out_counts) J.out_counts[row * J.out_cstride + M.cell_base + c] = (uint8_t)cnt;
            if (J.out_bits) J.out_bits[row * J.out_cstride + M.cell_base + c] = s_bits[c];
        }
        module_pv(J, M, s, lp, s_cnt, s_imin, B, msi);
        __syncthreads();
    }
    if (PROF) flush_profile(B, p_samples, 0u, 0u, 0u);
}

// ---------------------------------------------------------------------------
// k_string: series strings (Section 2: the generator's modules wired in
// series strings, Fig. 2) -- one current through every bypass substring of
// every module of the string; P(I) = I (sum_{k: I_k >= I} V_k - v_diode
// #{k: I_k < I}) is linear between consecutive substring currents, so the
// string's maximum power point is the best of them.  One warp per (step,
// string): lanes over candidate currents, an inner loop over the string's
// substrings.  Without shading every substring of a module carries the
// module's unshaded current.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_string(const WaveDev* __restrict__ W, const JobDev* __restrict__ jobs,
                                                Buffers B)
{
    const int64_t tot = W->tot_sq;
    const int nj = W->n_jobs;
    const int lane = threadIdx.x & 31;
    const int64_t n_warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t item = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; item < tot; item += n_warps) {
        const int j = job_of(nj, item, [&](int q) { return jobs[q].it_str; });
        const JobDev& J = jobs[j];
        const int64_t li = item - J.it_str;
        const int ls = (int)(li / J.n_str), q = (int)(li - (int64_t)ls * J.n_str);
        const int64_t sq = J.sq_base + li;
        const LightParams& lp = B.lp[J.js_base + ls];
        float best = 0.f, best_u = 0.f;
        if (lp.valid) {
            const int k0 = J.str_sub[q], k1 = J.str_sub[q + 1];
            const float* ik = B.ss_i + J.ss_base + (int64_t)ls * J.n_sub_tot;
            const float* iu = B.ms_iu + J.ms_base + (int64_t)ls * J.n_mods;
            for (int c = k0 + lane; c < k1; c += 32) {
                const float cur = ik[c], cur_u = iu[J.sub_mod[c]];
                float volt = 0.f, volt_u = 0.f;
                for (int k = k0; k < k1; ++k) {
                    const float vk = J.sub_nk[k] * J.v_cell;
                    volt += ik[k] >= cur ? vk : -J.v_diode;
                    volt_u += iu[J.sub_mod[k]] >= cur_u ? vk : -J.v_diode;
                }
                best = fmaxf(best, cur * volt);
                best_u = fmaxf(best_u, cur_u * volt_u);
            }
#pragma unroll
            for (int off = 16; off; off >>= 1) {
                best = fmaxf(best, __shfl_xor_sync(0xffffffffu, best, off));
                best_u = fmaxf(best_u, __shfl_xor_sync(0xffffffffu, best_u, off));
            }
        }
        if (lane == 0) {
            B.sq_p[sq] = best;
            B.sq_pu[sq] = best_u;
            const int64_t row = (int64_t)(J.out_row0 + ls);
            if (J.out_str_power) J.out_str_power[row * J.n_str + q] = best;
            if (J.out_str_power_u) J.out_str_power_u[row * J.n_str + q] = best_u;
        }
    }
}

// ---------------------------------------------------------------------------
// k_array: strings in parallel at one inverter input -- one voltage V across
// every string of the array; string s delivers the largest of its substring
// currents I_k whose string voltage V_s(I_k) = sum_{j: I_j >= I_k} V_j -
// v_diode #{j: I_j < I_k} still reaches V, and P(V) = V sum_s I_s(V) is
// linear between those voltages, so the array's maximum power point is the
// best of them.  One warp per (step, array): the array's substrings (current,
// string voltage at that current) staged in shared memory, then lanes over
// the candidate voltages.
// ---------------------------------------------------------------------------
constexpr int kArrayWarps = 4;

__global__ void __launch_bounds__(kArrayWarps * 32) k_array(const WaveDev* __restrict__ W,
                                                           const JobDev* __restrict__ jobs, Buffers B)
{
    __shared__ float s_i[kArrayWarps][kMaxArraySub], s_w[kArrayWarps][kMaxArraySub];
    __shared__ float s_iu[kArrayWarps][kMaxArraySub], s_wu[kArrayWarps][kMaxArraySub];
    __shared__ int s_str[kArrayWarps][kMaxArraySub];  // string of each staged substring (position in the array)
    const int64_t tot = W->tot_sa;
    const int nj = W->n_jobs;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int64_t n_warps = (int64_t)gridDim.x * kArrayWarps;
    for (int64_t item = (int64_t)blockIdx.x * kArrayWarps + wib; item < tot; item += n_warps) {
        const int j = job_of(nj, item, [&](int q) { return jobs[q].sa_base; });
        const JobDev& J = jobs[j];
        const int64_t li = item - J.sa_base;
        const int ls = (int)(li / J.n_arr), a = (int)(li - (int64_t)ls * J.n_arr);
        const LightParams& lp = B.lp[J.js_base + ls];
        float best = 0.f, best_u = 0.f;
        if (lp.valid) {
            const float* ik = B.ss_i + J.ss_base + (int64_t)ls * J.n_sub_tot;
            const float* iu = B.ms_iu + J.ms_base + (int64_t)ls * J.n_mods;
            // stage the array's substrings string by string, with each one's string voltage
            int n = 0;
            for (int t = J.arr_off[a]; t < J.arr_off[a + 1]; ++t) {
                const int q = J.arr_strs[t];
                const int k0 = J.str_sub[q], k1 = J.str_sub[q + 1];
                for (int c = k0 + lane; c < k1; c += 32) {
                    const float cur = ik[c], cur_u = iu[J.sub_mod[c]];
                    float volt = 0.f, volt_u = 0.f;
                    for (int k = k0; k < k1; ++k) {
                        const float vk = J.sub_nk[k] * J.v_cell;
                        volt += ik[k] >= cur ? vk : -J.v_diode;
                        volt_u += iu[J.sub_mod[k]] >= cur_u ? vk : -J.v_diode;
                    }
                    const int pos = n + (c - k0);
                    if (pos < kMaxArraySub) {
                        s_i[wib][pos] = cur; s_w[wib][pos] = volt;
                        s_iu[wib][pos] = cur_u; s_wu[wib][pos] = volt_u;
                        s_str[wib][pos] = t;
                    }
                }
                n += k1 - k0;
            }
            n = min(n, kMaxArraySub);
            __syncwarp();
            for (int c = lane; c < n; c += 32) {
                const float V = s_w[wib][c], Vu = s_wu[wib][c];
                float cur = 0.f, cur_u = 0.f, is = 0.f, isu = 0.f;
                int prev = s_str[wib][0];
                for (int k = 0; k < n; ++k) {
                    if (s_str[wib][k] != prev) {  // next string: add the last one's current
                        cur += is; cur_u += isu;
                        is = 0.f; isu = 0.f;
                        prev = s_str[wib][k];
                    }
                    if (s_w[wib][k] >= V && s_i[wib][k] > is) is = s_i[wib][k];
                    if (s_wu[wib][k] >= Vu && s_iu[wib][k] > isu) isu = s_iu[wib][k];
                }
                cur += is; cur_u += isu;
                if (V > 0.f) best = fmaxf(best, V * cur);
                if (Vu > 0.f) best_u = fmaxf(best_u, Vu * cur_u);
            }
#pragma unroll
            for (int off = 16; off; off >>= 1) {
                best = fmaxf(best, __shfl_xor_sync(0xffffffffu, best, off));
                best_u = fmaxf(best_u, __shfl_xor_sync(0xffffffffu, best_u, off));
            }
            __syncwarp();
        }
        if (lane == 0) {
            B.sa_p[item] = best;
            B.sa_pu[item] = best_u;
            const int64_t row = (int64_t)(J.out_row0 + ls);
            if (J.out_arr_power) J.out_arr_power[row * J.n_arr + a] = best;
            if (J.out_arr_power_u) J.out_arr_power_u[row * J.n_arr + a] = best_u;
        }
    }
}

// ---------------------------------------------------------------------------
// sky map of the effective shading (Fig. 6: the shading factor over the sun's
// azimuth and zenith): k_gen_step sums the generator's power per step and
// bins the step's sun; k_heat adds each bin's steps in step order (FP64)
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_gen_step(const WaveDev* __restrict__ W, const JobDev* __restrict__ jobs,
                                                  Buffers B)
{
    const int64_t tot = W->tot_js;
    const int nj = W->n_jobs;
    const int lane = threadIdx.x & 31;
    const int64_t n_warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t js = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; js < tot; js += n_warps) {
        const int j = job_of(nj, js, [&](int q) { return (int64_t)jobs[q].js_base; });
        const JobDev& J = jobs[j];
        if (J.heat_az == 0) continue;
        const int ls = (int)(js - J.js_base);
        float p = 0.f, pu = 0.f;
        for (int m = lane; m < J.n_mods; m += 32) {
            const int64_t msi = J.ms_base + (int64_t)ls * J.n_mods + m;
            p += B.ms_p[msi];
            pu += B.ms_pu[msi];
        }
#pragma unroll
        for (int off = 16; off; off >>= 1) {
            p += __shfl_xor_sync(0xffffffffu, p, off);
            pu += __shfl_xor_sync(0xffffffffu, pu, off);
        }
        if (lane == 0) {
            B.js_p[js] = p;
            B.js_pu[js] = pu;
            const double* sp = J.sun + 3 * (size_t)(J.step0 + ls);
            int bin = -1;
            if (sp[2] > 0.0) {
                const double deg = 57.29577951308232;  // degrees per radian
                double az = atan2(sp[0], sp[1]) * deg;
                if (az < 0.0) az += 360.0;
                const double zen = acos(fmin(1.0, sp[2])) * deg;
                const int ia = min((int)(az / 360.0 * J.heat_az), J.heat_az - 1);
                const int iz = min((int)(zen / 90.0 * J.heat_zen), J.heat_zen - 1);
                bin = iz * J.heat_az + ia;
            }
            B.js_bin[js] = bin;
        }
    }
}

__global__ void __launch_bounds__(256) k_heat(const WaveDev* __restrict__ W, const JobDev* __restrict__ jobs,
                                              Buffers B)
{
    const int64_t tot = W->tot_heat;
    const int nj = W->n_jobs;
    for (int64_t item = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; item < tot;
         item += (int64_t)gridDim.x * blockDim.x) {
        const int j = job_of(nj, item, [&](int q) { return jobs[q].it_heat; });
        const JobDev& J = jobs[j];
        const int bin = (int)(item - J.it_heat);
        double e = J.heat_e[bin], eu = J.heat_eu[bin];
        int cnt = J.heat_n[bin];
        for (int ls = 0; ls < J.k; ++ls) {
            const int64_t js = J.js_base + ls;
            if (B.js_bin[js] != bin) continue;
            const double dt = (double)B.lp[js].dt;
            e += (double)B.js_p[js] * dt;
            eu += (double)B.js_pu[js] * dt;
            ++cnt;
        }
        J.heat_e[bin] = e;
        J.heat_eu[bin] = eu;
        J.heat_n[bin] = cnt;
    }
}

// ---------------------------------------------------------------------------
// k_epilogue: Kahan sums over the wave's steps in step order
// ---------------------------------------------------------------------------
__device__ __forceinline__ void kahan_add(float2& acc, float x)
{
    float y = x - acc.y;
    float t = acc.x + y;
    acc.y = (t - acc.x) - y;
    acc.x = t;
}

// One warp per item (cell, module or string): the lanes load 32 steps at a
// time, then every lane applies the same Kahan additions in step order from
// the shuffled values, so the sums equal a sequential loop over the steps
// while the loads of 32 steps overlap.
__global__ void __launch_bounds__(256) k_epilogue(const WaveDev* __restrict__ W, const JobDev* __restrict__ jobs,
                                                  Buffers B)
{
    const int64_t tot = W->tot_epi;
    const int nj = W->n_jobs;
    const int lane = threadIdx.x & 31;
    if (W->fused && blockIdx.x == 0 && threadIdx.x == 0) {  // the tiles' records are all allocated by now
        Counters* c = B.ctr;
        if (c->cov_next > c->need_cov) c->need_cov = c->cov_next;
        if (c->cov_next > (unsigned long long)W->cov_cap) c->overflow |= 16u;
    }
    const int64_t n_warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t item = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; item < tot; item += n_warps) {
        const int j = job_of(nj, item, [&](int q) { return jobs[q].it_epi; });
        const JobDev& J = jobs[j];
        const int64_t li = item - J.it_epi;
        // cell items only when the per-cell beam loss is wanted
        const int C = J.kahan_cell ? J.n_cells : 0, Mn = J.n_mods;
        const float inv_nn = 1.f / J.nn;
        // kind 0: cell c; 1: module m; 2: string q; 3: array
        const int kind = li < C ? 0 : (li < C + Mn ? 1 : (li < C + Mn + J.n_str ? 2 : 3));
        const int idx = kind == 0 ? (int)li
                                  : (kind == 1 ? (int)(li - C) : (kind == 2 ? (int)(li - C - Mn) : (int)(li - C - Mn - J.n_str)));
        const int m_cell = kind == 0 ? J.cell_mod[idx] : 0;
        float2 a, au = make_float2(0.f, 0.f);
        if (kind == 0) a = J.kahan_cell[idx];
        else if (kind == 1) { a = J.kahan_mod[2 * idx]; au = J.kahan_mod[2 * idx + 1]; }
        else if (kind == 2) { a = J.kahan_str[2 * idx]; au = J.kahan_str[2 * idx + 1]; }
        else { a = J.kahan_arr[2 * idx]; au = J.kahan_arr[2 * idx + 1]; }
        for (int l0 = 0; l0 < J.k; l0 += 32) {
            const int ls = l0 + lane;
            float x = 0.f, xu = 0.f;
            bool v = false;
            if (ls < J.k) {
                const LightParams& lp = B.lp[J.js_base + ls];
                v = lp.valid != 0;
                if (kind == 0) {
                    if (v) {
                        const float beam = B.ms_beam[J.ms_base + (int64_t)ls * Mn + m_cell];
                        const uint32_t cnt = tally_get(B.cs_cnt, J.cs_base + (int64_t)ls * C + idx);
                        x = beam * (cnt * inv_nn) * lp.dt;
                    }
                } else if (kind == 1) {
                    const int64_t msi = J.ms_base + (int64_t)ls * Mn + idx;
                    const float p = B.ms_p[msi], pu = B.ms_pu[msi];
                    if (J.out_power) J.out_power[(int64_t)(J.out_row0 + ls) * J.out_mstride + idx] = p;
                    if (J.out_power_u) J.out_power_u[(int64_t)(J.out_row0 + ls) * J.out_mstride + idx] = pu;
                    x = p * lp.dt;
                    xu = pu * lp.dt;
                } else if (v && kind == 2) {
                    const int64_t sq = J.sq_base + (int64_t)ls * J.n_str + idx;
                    x = B.sq_p[sq] * lp.dt;
                    xu = B.sq_pu[sq] * lp.dt;
                } else if (v) {
                    const int64_t sa = J.sa_base + (int64_t)ls * J.n_arr + idx;
                    x = B.sa_p[sa] * lp.dt;
                    xu = B.sa_pu[sa] * lp.dt;
                }
            }
            const unsigned int vm = __ballot_sync(0xffffffffu, v);
            const int n_here = min(32, J.k - l0);
            for (int q = 0; q < n_here; ++q) {
                const float xq = __shfl_sync(0xffffffffu, x, q);
                const float xuq = __shfl_sync(0xffffffffu, xu, q);
                if (!((vm >> q) & 1u)) continue;
                kahan_add(a, xq);
                if (kind != 0) kahan_add(au, xuq);
            }
        }
        if (lane == 0) {
            if (kind == 0) J.kahan_cell[idx] = a;
            else if (kind == 1) { J.kahan_mod[2 * idx] = a; J.kahan_mod[2 * idx + 1] = au; }
            else if (kind == 2) { J.kahan_str[2 * idx] = a; J.kahan_str[2 * idx + 1] = au; }
            else { J.kahan_arr[2 * idx] = a; J.kahan_arr[2 * idx + 1] = au; }
        }
    }
}

// Convert Kahan pairs (sum, compensation) to double results.
__global__ void k_finalize(const float2* __restrict__ kmod, int n_mods, const float2* __restrict__ kcell,
                           int n_cells, double* energy, double* energy_u, double* cell_loss)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_mods + n_cells; i += gridDim.x * blockDim.x) {
        if (i < n_mods) {
            const float2 e = kmod[2 * i], eu = kmod[2 * i + 1];
            if (energy) energy[i] = (double)e.x - (double)e.y;
            if (energy_u) energy_u[i] = (double)eu.x - (double)eu.y;
        } else {
            const int c = i - n_mods;
            const float2 h = kcell[c];
            if (cell_loss) cell_loss[c] = (double)h.x - (double)h.y;
        }
    }
}

// ---------------------------------------------------------------------------
// clear-sky sun table and ideal tracker poses, made on the device (the inputs
// of steps 3-4; the paper takes TMY data, measured series or an unnamed
// clear-sky model).  Solar time without longitude correction or equation of
// time; Cooper's (1969) declination; hour angle 15 deg per hour from noon;
// Meinel & Meinel's (1976) beam irradiance with Kasten & Young's (1989) air
// mass; all in FP64.
// ---------------------------------------------------------------------------
__global__ void k_sun_table(double lat_deg, int day_first, int64_t per_day, double step_h, double dhi_fraction,
                            int64_t n, double* __restrict__ xyz, float* __restrict__ dni, float* __restrict__ dhi,
                            float* __restrict__ dt, uint8_t* __restrict__ lit)
{
    const double deg = 0.017453292519943295;  // radians per degree
    const double phi = lat_deg * deg;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t d = i / per_day, k = i - d * per_day;
        const double day = (double)(day_first + d);
        const double delta = 23.45 * deg * sin(360.0 * deg * (284.0 + day) / 365.0);
        const double omega = 15.0 * deg * ((double)k * step_h - 12.0);
        double e = -cos(delta) * sin(omega);
        double no = sin(delta) * cos(phi) - cos(delta) * cos(omega) * sin(phi);
        double up = sin(delta) * sin(phi) + cos(delta) * cos(omega) * cos(phi);
        const double len = sqrt(e * e + no * no + up * up);
        e /= len; no /= len; up /= len;
        double b = 0.0;
        if (up > 0.0) {
            const double z = acos(up) / deg;
            const double am = 1.0 / (up + 0.50572 * pow(96.07995 - z, -1.6364));
            b = 1353.0 * pow(0.7, pow(am, 0.678));
        }
        xyz[3 * i] = e; xyz[3 * i + 1] = no; xyz[3 * i + 2] = up;
        dni[i] = (float)b;
        dhi[i] = (float)(dhi_fraction * b);
        dt[i] = (float)step_h;
        lit[i] = up > 0.0;
    }
}

__global__ void k_gather_sun(const int64_t* __restrict__ idx, int64_t n, const double* __restrict__ xyz,
                             const float* __restrict__ dni, const float* __restrict__ dhi, double* __restrict__ oxyz,
                             float* __restrict__ odni, float* __restrict__ odhi)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t k = idx[i];
        oxyz[3 * i] = xyz[3 * k]; oxyz[3 * i + 1] = xyz[3 * k + 1]; oxyz[3 * i + 2] = xyz[3 * k + 2];
        odni[i] = dni[k];
        odhi[i] = dhi[k];
    }
}

// Diffuse shading: sky patches of equal zenith bands and azimuth sectors at
// their centre directions, solid angle (cos z0 - cos z1) 2 pi / sectors.
__global__ void k_sky_patches(int rings, int sectors, double* __restrict__ xyz, float* __restrict__ dni,
                              float* __restrict__ dhi, float* __restrict__ dt, double* __restrict__ dom)
{
    const double half_pi = 1.5707963267948966, two_pi = 6.283185307179586;
    const int n = rings * sectors;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int r = i / sectors, k = i - r * sectors;
        const double z0 = half_pi * r / rings, z1 = half_pi * (r + 1) / rings;
        const double zc = 0.5 * (z0 + z1);
        const double a = two_pi * (k + 0.5) / sectors;
        xyz[3 * i] = sin(zc) * sin(a);
        xyz[3 * i + 1] = sin(zc) * cos(a);
        xyz[3 * i + 2] = cos(zc);
        dni[i] = 1.f;
        dhi[i] = 0.f;
        dt[i] = 1.f;
        dom[i] = (cos(z0) - cos(z1)) * two_pi / sectors;
    }
}

// Per cell: f = sum_p W_p s_p / sum_p W_p, W_p = solid angle x max(0, n . w_p)
// with the module's front normal n (a tracked module's at the pose (az,
// tilt) of the sky view: R = Rz(pi - az) Rx(tilt)), s_p = shaded samples
// toward patch p / n^2 (counts[p][c]); summed in patch order in FP64.
__global__ void k_sky_fraction(const ModuleDev* __restrict__ mods, const int32_t* __restrict__ cell_mod, int n_cells,
                               const double* __restrict__ xyz, const double* __restrict__ dom, int n_patch,
                               const uint8_t* __restrict__ counts, int nn, float* __restrict__ fdiff, double az,
                               double tilt)
{
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < n_cells; c += gridDim.x * blockDim.x) {
        const ModuleDev& M = mods[cell_mod[c]];
        double nx = (double)M.u[1] * M.v[2] - (double)M.u[2] * M.v[1];
        double ny = (double)M.u[2] * M.v[0] - (double)M.u[0] * M.v[2];
        double nz = (double)M.u[0] * M.v[1] - (double)M.u[1] * M.v[0];
        const double l = sqrt(nx * nx + ny * ny + nz * nz);
        nx /= l; ny /= l; nz /= l;
        if (M.tracker >= 0) {
            const double cb = cos(tilt), sb = sin(tilt), cg = -cos(az), sg = sin(az);
            const double yy = cb * ny - sb * nz, zz = sb * ny + cb * nz;
            const double xx = nx;
            nx = cg * xx - sg * yy;
            ny = sg * xx + cg * yy;
            nz = zz;
        }
        double num = 0.0, den = 0.0;
        for (int p = 0; p < n_patch; ++p) {
            const double w = dom[p] * fmax(0.0, nx * xyz[3 * p] + ny * xyz[3 * p + 1] + nz * xyz[3 * p + 2]);
            den += w;
            num += w * ((double)counts[(size_t)p * n_cells + c] / (double)nn);
        }
        fdiff[c] = den > 0.0 ? (float)(num / den) : 0.f;
    }
}

__global__ void k_ideal_poses(const double* __restrict__ sun, int64_t n_steps, int n_trk, float tilt_max,
                              float* __restrict__ poses)
{
    const int64_t n = n_steps * n_trk;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t s = i / n_trk;
        const double* sp = sun + 3 * s;
        poses[2 * i] = (float)atan2(sp[0], sp[1]);
        poses[2 * i + 1] = fminf((float)acos(fmin(1.0, fmax(-1.0, sp[2]))), tilt_max);
    }
}

// ---------------------------------------------------------------------------
// host launchers
// ---------------------------------------------------------------------------
static inline unsigned int grid_for(int64_t items, int per_block, int cap)
{
    int64_t g = (items + per_block - 1) / per_block;
    if (g < 1) g = 1;
    if (g > cap) g = cap;
    return (unsigned int)g;
}

// Blocks of the block-per-tile kernels per SM (their shared tile is dynamic:
// TileSm<128> holds a 64 KB depth tile).
template <int TS>
constexpr int tile_blocks() { return TS == 128 ? 2 : 4; }

template <int TS, bool PROF>
static cudaError_t allow_tile_smem()
{
    cudaError_t e = cudaFuncSetAttribute(k_raster_test<TS, PROF>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(HeavySm<TS>));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_raster_map<TS, PROF>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)sizeof(TileSm<TS>));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_tile_warp<TS, PROF>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)(kTileWarps * sizeof(WarpSm<TS>)));
    return e;
}

cudaError_t prepare_tile_kernels()
{
    cudaError_t e = cudaSuccess;
    if (e == cudaSuccess) e = allow_tile_smem<32, false>();
    if (e == cudaSuccess) e = allow_tile_smem<32, true>();
    if (e == cudaSuccess) e = allow_tile_smem<64, false>();
    if (e == cudaSuccess) e = allow_tile_smem<64, true>();
    if (e == cudaSuccess) e = allow_tile_smem<128, false>();
    if (e == cudaSuccess) e = allow_tile_smem<128, true>();
    return e;
}

template <int TS, bool PROF>
static void launch_tile_kernels(const WaveDev* W, const JobDev* d_jobs, const Buffers& b, const LaunchCfg& cfg)
{
    const int sm = cfg.sm_count;
    if (cfg.fused) {
        k_tile_warp<TS, PROF><<<sm * TileBlocks<TS>::n, kTileWarps * 32, kTileWarps * sizeof(WarpSm<TS>), cfg.stream>>>(
            W, d_jobs, b);
        if (cfg.ev) cudaEventRecord(cfg.ev[3], cfg.stream);
        k_raster_test<TS, PROF><<<sm * HeavyCfg<TS>::min_blocks, HeavyCfg<TS>::threads, sizeof(HeavySm<TS>),
                                  cfg.stream>>>(W, d_jobs, b);
        if (cfg.ev) cudaEventRecord(cfg.ev[4], cfg.stream);
        k_pv<<<sm * 16, kPvThreads, 0, cfg.stream>>>(W, d_jobs, b);
        k_cells<TS, PROF><<<sm * kCellBlocks, kCellWarps * 32, 0, cfg.stream>>>(W, d_jobs, b);
    } else {
        k_raster_map<TS, PROF><<<sm * tile_blocks<TS>(), 256, sizeof(TileSm<TS>), cfg.stream>>>(W, d_jobs, b);
        if (cfg.ev) {
            cudaEventRecord(cfg.ev[3], cfg.stream);
            cudaEventRecord(cfg.ev[4], cfg.stream);
        }
        k_sample<PROF><<<sm * 16, kPvThreads, 0, cfg.stream>>>(W, d_jobs, b);
    }
}

cudaError_t launch_wave(const WaveDev* d_wave, const JobDev* d_jobs, const Buffers& b, const LaunchCfg& cfg)
{
    const WaveDev* W = d_wave;
    cudaStream_t st = cfg.stream;
    const int sm = cfg.sm_count;
    if (cfg.ev) cudaEventRecord(cfg.ev[0], st);
    k_clear<<<sm * 8, 256, 0, st>>>(W, d_jobs, b);
    k_window<<<sm * 8, kWinPerItem, 0, st>>>(W, d_jobs, b);
    k_light<<<sm, 128, 0, st>>>(W, d_jobs, b);
    k_modsetup<<<sm * 8, 256, 0, st>>>(W, d_jobs, b);
    if (cfg.ev) cudaEventRecord(cfg.ev[1], st);
    k_bin<<<sm * 16, 256, 0, st>>>(W, d_jobs, b);
    k_bin_big<<<sm * 8, 256, 0, st>>>(W, d_jobs, b);
    k_scan_a<<<sm * 2, kScanThreads, 0, st>>>(W, b);
    k_scan_b<<<1, kScanThreads, 0, st>>>(W, b);
    k_scan_c<<<sm * 2, kScanThreads, 0, st>>>(W, b);
    k_scatter<<<sm * 8, 256, 0, st>>>(W, b);
    k_recv_fill<<<sm * 8, 256, 0, st>>>(W, d_jobs, b);
    if (cfg.ev) cudaEventRecord(cfg.ev[2], st);
    if (cfg.tile == 32) {
        if (cfg.profile) launch_tile_kernels<32, true>(W, d_jobs, b, cfg);
        else launch_tile_kernels<32, false>(W, d_jobs, b, cfg);
    } else if (cfg.tile == 64) {
        if (cfg.profile) launch_tile_kernels<64, true>(W, d_jobs, b, cfg);
        else launch_tile_kernels<64, false>(W, d_jobs, b, cfg);
    } else {
        if (cfg.profile) launch_tile_kernels<128, true>(W, d_jobs, b, cfg);
        else launch_tile_kernels<128, false>(W, d_jobs, b, cfg);
    }
    if (cfg.extras & 1) k_string<<<sm * 4, 256, 0, st>>>(W, d_jobs, b);
    if (cfg.extras & 4) k_array<<<sm * 4, kArrayWarps * 32, 0, st>>>(W, d_jobs, b);
    if (cfg.extras & 2) {
        k_gen_step<<<sm * 4, 256, 0, st>>>(W, d_jobs, b);
        k_heat<<<sm * 2, 256, 0, st>>>(W, d_jobs, b);
    }
    if (cfg.ev) cudaEventRecord(cfg.ev[5], st);
    k_epilogue<<<sm * 8, 256, 0, st>>>(W, d_jobs, b);
    if (cfg.ev) cudaEventRecord(cfg.ev[6], st);
    return cudaGetLastError();
}

cudaError_t launch_sun_table(double lat_deg, int day_first, int64_t per_day, double step_h, double dhi_fraction,
                             int64_t n, double* xyz, float* dni, float* dhi, float* dt, uint8_t* lit, cudaStream_t st)
{
    k_sun_table<<<grid_for(n, 256, 4096), 256, 0, st>>>(lat_deg, day_first, per_day, step_h, dhi_fraction, n, xyz, dni,
                                                          dhi, dt, lit);
    return cudaGetLastError();
}

cudaError_t launch_gather_sun(const int64_t* idx, int64_t n, const double* xyz, const float* dni, const float* dhi,
                              double* oxyz, float* odni, float* odhi, cudaStream_t st)
{
    k_gather_sun<<<grid_for(n, 256, 4096), 256, 0, st>>>(idx, n, xyz, dni, dhi, oxyz, odni, odhi);
    return cudaGetLastError();
}

cudaError_t launch_sky_patches(int rings, int sectors, double* xyz, float* dni, float* dhi, float* dt, double* dom,
                               cudaStream_t st)
{
    k_sky_patches<<<grid_for((int64_t)rings * sectors, 256, 1024), 256, 0, st>>>(rings, sectors, xyz, dni, dhi, dt,
                                                                                 dom);
    return cudaGetLastError();
}

cudaError_t launch_sky_fraction(const ModuleDev* mods, const int32_t* cell_mod, int n_cells, const double* xyz,
                                const double* dom, int n_patch, const uint8_t* counts, int nn, float* fdiff,
                                double az, double tilt, cudaStream_t st)
{
    k_sky_fraction<<<grid_for(n_cells, 128, 4096), 128, 0, st>>>(mods, cell_mod, n_cells, xyz, dom, n_patch, counts,
                                                                  nn, fdiff, az, tilt);
    return cudaGetLastError();
}

cudaError_t launch_ideal_poses(const double* sun, int64_t n_steps, int n_trk, float tilt_max, float* poses,
                               cudaStream_t st)
{
    k_ideal_poses<<<grid_for(n_steps * n_trk, 256, 4096), 256, 0, st>>>(sun, n_steps, n_trk, tilt_max, poses);
    return cudaGetLastError();
}

cudaError_t launch_finalize_pairs(const float2* kmod, int n_mods, const float2* kcell, int n_cells,
                                  double* energy, double* energy_u, double* cell_loss, cudaStream_t st)
{
    int n = n_mods + n_cells;
    k_finalize<<<grid_for(n, 256, 1024), 256, 0, st>>>(kmod, n_mods, kcell, n_cells, energy, energy_u, cell_loss);
    return cudaGetLastError();
}

}  // namespace pv3d
