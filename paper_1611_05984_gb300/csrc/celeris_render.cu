// Headless rendering of the state into an RGBA8 image: the visualisation
// options of Sec. 3 (colormaps of eta, u, v and the velocity magnitude, water
// shaded by the Fresnel equations, a colormap on the terrain, a grid over the
// surfaces), without any graphics API.
//
// The shading is single precision with every operation rounded on its own
// (the _rn intrinsics: no contraction into fused multiply-adds, IEEE
// division and square root whatever the build's fast-math flags), and no
// transcendental functions, so the bytes are reproducible by any correct
// implementation of the same sequence of operations.  The colours, the
// lighting and the camera are this renderer's choices (the paper names only
// what is shown).
#include "celeris_internal.cuh"

namespace cel {
namespace {

__device__ __forceinline__ float ad(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float sb(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float ml(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float dv(float a, float b) { return __fdiv_rn(a, b); }
__device__ __forceinline__ float sq(float a) { return __fsqrt_rn(a); }
__device__ __forceinline__ float clamp01(float x) { return x < 0.0f ? 0.0f : (x > 1.0f ? 1.0f : x); }

constexpr float kWaterIndex = 1.333f;   // refractive index of water (air: 1)

// Colormaps through 5 control points at t = 0, 1/4, ..., 1: diverging
// blue-white-red (signed values), dark-to-bright (speed), sand-green-brown
// (terrain).
__constant__ float c_maps[3][5][3] = {
    {{0.020f, 0.188f, 0.380f}, {0.263f, 0.576f, 0.765f}, {0.969f, 0.969f, 0.969f},
     {0.957f, 0.647f, 0.510f}, {0.404f, 0.000f, 0.122f}},
    {{0.050f, 0.030f, 0.200f}, {0.150f, 0.250f, 0.550f}, {0.100f, 0.600f, 0.650f},
     {0.550f, 0.850f, 0.350f}, {0.990f, 0.950f, 0.300f}},
    {{0.780f, 0.700f, 0.500f}, {0.600f, 0.650f, 0.380f}, {0.350f, 0.550f, 0.250f},
     {0.450f, 0.480f, 0.300f}, {0.550f, 0.450f, 0.350f}}};
__constant__ float c_sky_horizon[3] = {0.780f, 0.850f, 0.920f};
__constant__ float c_sky_zenith[3] = {0.250f, 0.450f, 0.800f};
__constant__ float c_water[3] = {0.020f, 0.150f, 0.200f};

// The control points as the pixels read them, in shared memory: for each map
// and piece the colour at its start and the change to its end, (r, g, b, dr),
// (dg, db, -, -).  Lanes on different pieces read different banks (from
// constant memory each piece would be a load of its own).
struct ColorTable {
    float4 v[3][4][2];
};

__device__ __forceinline__ void fill_table(ColorTable &T, int tid)
{
    if (tid >= 96) return;
    const int map = tid >> 5, k = (tid >> 3) & 3, e = tid & 7;
    float v = 0.0f;
    if (e < 3) v = c_maps[map][k][e];
    else if (e < 6) v = sb(c_maps[map][k + 1][e - 3], c_maps[map][k][e - 3]);
    reinterpret_cast<float *>(&T.v[map][k][0])[e] = v;
}

constexpr float kTwo23 = 8388608.0f;   // 2^23: x + 2^23, rounded down, holds floor(x) in its low bits (0 <= x < 2^23)

__device__ __forceinline__ void colormap(const ColorTable &T, int map, float t, float rgb[3])
{
    const float s = ml(clamp01(t), 4.0f);
    const float k = fminf(sb(__fadd_rz(s, kTwo23), kTwo23), 3.0f);   // the piece (3 where t is no number)
    const float f = sb(s, k);
    const float4 *e = T.v[map][__float_as_int(ad(k, kTwo23)) & 3];
    const float4 a = e[0];
    const float2 b = *reinterpret_cast<const float2 *>(e + 1);
    rgb[0] = ad(a.x, ml(a.w, f));
    rgb[1] = ad(a.y, ml(b.x, f));
    rgb[2] = ad(a.z, ml(b.y, f));
}

// Fresnel equations, unpolarised light from air into water.
__device__ __forceinline__ float fresnel(float cos_i)
{
    cos_i = clamp01(cos_i);
    const float sin2_i = sb(1.0f, ml(cos_i, cos_i));
    const float sin2_t = dv(sin2_i, ml(kWaterIndex, kWaterIndex));
    const float cos_t = sq(sb(1.0f, sin2_t));
    const float rs = dv(sb(cos_i, ml(kWaterIndex, cos_t)), ad(cos_i, ml(kWaterIndex, cos_t)));
    const float rp = dv(sb(ml(kWaterIndex, cos_i), cos_t), ad(ml(kWaterIndex, cos_i), cos_t));
    return ml(ad(ml(rs, rs), ml(rp, rp)), 0.5f);
}

__device__ __forceinline__ void normalize3(float v[3])
{
    const float n = sq(ad(ad(ml(v[0], v[0]), ml(v[1], v[1])), ml(v[2], v[2])));
    v[0] = dv(v[0], n);
    v[1] = dv(v[1], n);
    v[2] = dv(v[2], n);
}

__device__ __forceinline__ float dot3(const float a[3], const float b[3])
{
    return ad(ad(ml(a[0], b[0]), ml(a[1], b[1])), ml(a[2], b[2]));
}

// The colour's byte, in the low bits (no number: 0).
__device__ __forceinline__ uint32_t to_byte(float c)
{
    return __float_as_uint(__fadd_rz(ad(ml(__saturatef(c), 255.0f), 0.5f), kTwo23));
}

template <typename real>
__device__ __forceinline__ float tofloat(real v) { return (float)v; }

constexpr int kRT = 32;        // pixels per tile edge
constexpr int kRS = kRT + 2;   // with a one-cell ring

// What the shaded water alone keeps per tile, with the ring (clamped at the
// grid's edges): w, and eta (no number where dry).
template <bool kOn>
struct WaterTile {
    float w[kRS][kRS + 1], eta[kRS][kRS + 1];
};
template <>
struct WaterTile<false> {};
// Q of the tile, transposed from its column-major array.
template <bool kOn>
struct QTile {
    float v[kRT][kRT + 1];
};
template <>
struct QTile<false> {};

// One 32 x 32 tile of pixels per block, four per thread.  Bound by instruction
// issue (most of them the IEEE divisions and square roots of the shading), so
// what is the same for all pixels is worked out once per block: the unit
// vectors of the view and the sun, the colour pieces, the columns and rows that
// carry a grid line.  A kernel per mode reads only what its mode shows: Q for v
// and the speed, neighbours' eta for shaded water.
// 2048 x 2048, FP32 (FP64): eta 37.6 -> 26.7 us (73.9 -> 62.3), speed with a
// grid 50.8 -> 38.8 (82.1 -> 78.8), shaded water 78.9 -> 57.1 (92.8 -> 70.3)
// against one kernel for all modes that did all of it per pixel.
template <typename real, int kMode>
__global__ void __launch_bounds__(256) k_render(const __grid_constant__ RenderArgs<real> A)
{
    constexpr bool kWater = kMode == CEL_RENDER_FRESNEL, kP = kMode == CEL_RENDER_U || kMode == CEL_RENDER_SPEED,
                   kQ = kMode == CEL_RENDER_V || kMode == CEL_RENDER_SPEED;
    __shared__ ColorTable T;
    __shared__ float s_dir[2][3];                // unit vectors of the view and the sun
    __shared__ unsigned char s_line[2][kRT];     // a grid line crosses the column, the row
    __shared__ float sB[kRS][kRS + 1];           // the cell bed with a ring (clamped)
    __shared__ WaterTile<kWater> S;
    __shared__ QTile<kQ> SQ;
    const Geo &G = A.geo;
    const cel_render_params &p = A.p;
    const int nx = G.nx, ny = G.ny;
    const int x0 = blockIdx.x * kRT, y0 = blockIdx.y * kRT;
    const int lane = threadIdx.x, wy = threadIdx.y, tid = wy * 32 + lane;
    const float dx = A.dx, dy = A.dy, ws = A.ws;
    auto stage = [&](int ty, int tx) {
        const int i = min(max(x0 - 1 + tx, 0), nx - 1), j = min(max(y0 - 1 + ty, 0), ny - 1);
        const float B = tofloat(bbar_at(A.Bc, G, i, j));
        sB[ty][tx] = B;
        if constexpr (kWater) {
            const float w = tofloat(A.w[(size_t)j * G.px + i]);
            S.w[ty][tx] = w;
            S.eta[ty][tx] = sb(w, B) > p.dry_h ? sb(w, ws) : __int_as_float(0x7fffffff);
        }
    };
#pragma unroll
    for (int u = 0; u < kRT / 8; u++) stage(wy + 8 * u, lane);
    if (wy < kRS - kRT) stage(kRT + wy, lane);
    if (tid >= 64 && tid < 64 + 2 * kRS) stage((tid - 64) >> 1, kRT + (tid & 1));
    if constexpr (kQ) {
#pragma unroll
        for (int u = 0; u < kRT / 8; u++) {   // a warp reads 32 consecutive j of one column
            const int c = wy + 8 * u, i = x0 + c, j = y0 + lane;
            SQ.v[lane][c] = (i < nx && j < ny) ? tofloat(A.Qc[(size_t)i * G.py + j]) : 0.0f;
        }
    }
    fill_table(T, tid);
    if (lane == 0 && wy >= 4 && wy < 6) {
        const float *d = wy == 4 ? p.view : p.sun;
        float v[3] = {d[0], d[1], d[2]};
        normalize3(v);
#pragma unroll
        for (int c = 0; c < 3; c++) s_dir[wy - 4][c] = v[c];
    }
    if (p.grid > 0.0f && wy >= 6) {   // a grid line crosses the cell where floor(x / spacing) changes across it
        const int k = (wy == 6 ? x0 : y0) + lane;
        const float d = wy == 6 ? dx : dy;
        s_line[wy - 6][lane] = floorf(dv(ml(__int2float_rn(k + 1), d), p.grid)) != floorf(dv(ml(__int2float_rn(k), d), p.grid));
    }
    __syncthreads();
    const int i = x0 + lane;
    if (i >= nx) return;
    const int iw = i > 0 ? i - 1 : i, ie = i < nx - 1 ? i + 1 : i;
    const float spanx = ml(__int2float_rn(ie - iw), dx);
    const float zspan = sb(p.zmax, p.zmin);
#pragma unroll 2
    for (int rr = 0; rr < kRT / 8; rr++) {
        const int cy = wy + rr * 8, j = y0 + cy;
        if (j >= ny) break;
        const int sx = lane + 1, sy = cy + 1;
        float wc;
        if constexpr (kWater) wc = S.w[sy][sx];
        else wc = tofloat(A.w[(size_t)j * G.px + i]);
        const float Bc = sB[sy][sx];
        const float h = sb(wc, Bc);
        const int js = j > 0 ? j - 1 : j, jn = j < ny - 1 ? j + 1 : j;
        float rgb[3];
        if (!(h > p.dry_h)) {
            const float spany = ml(__int2float_rn(jn - js), dy);
            const float gx = spanx > 0.0f ? dv(sb(sB[sy][sx + 1], sB[sy][sx - 1]), spanx) : 0.0f;
            const float gy = spany > 0.0f ? dv(sb(sB[sy + 1][sx], sB[sy - 1][sx]), spany) : 0.0f;
            float nb[3] = {-ml(p.exaggeration, gx), -ml(p.exaggeration, gy), 1.0f};
            normalize3(nb);
            const float d = dot3(nb, s_dir[1]);
            const float shade = ad(0.35f, ml(0.65f, d > 0.0f ? d : 0.0f));
            colormap(T, 2, dv(sb(Bc, p.zmin), zspan), rgb);
#pragma unroll
            for (int c = 0; c < 3; c++) rgb[c] = ml(rgb[c], shade);
        } else if constexpr (kWater) {
            const float ec = S.eta[sy][sx];
            auto eta_or = [&](int ty, int tx) {
                const float e = S.eta[ty][tx];
                return e == e ? e : ec;
            };
            const float eW = eta_or(sy, sx - 1), eE = eta_or(sy, sx + 1);
            const float eS = eta_or(sy - 1, sx), eN = eta_or(sy + 1, sx);
            const float spany = ml(__int2float_rn(jn - js), dy);
            const float gx = spanx > 0.0f ? dv(sb(eE, eW), spanx) : 0.0f;
            const float gy = spany > 0.0f ? dv(sb(eN, eS), spany) : 0.0f;
            float n[3] = {-ml(p.exaggeration, gx), -ml(p.exaggeration, gy), 1.0f};
            normalize3(n);
            const float *I = s_dir[0];
            const float idn = dot3(I, n);
            const float R = fresnel(-idn);
            const float tz = clamp01(sb(I[2], ml(ml(2.0f, idn), n[2])));
            float bed[3];
            colormap(T, 2, dv(sb(Bc, p.zmin), zspan), bed);
            const float a = dv(1.0f, ad(1.0f, ml(p.absorb, h)));
#pragma unroll
            for (int c = 0; c < 3; c++) {
                const float sky = ad(c_sky_horizon[c], ml(sb(c_sky_zenith[c], c_sky_horizon[c]), tz));
                const float refr = ad(c_water[c], ml(sb(bed[c], c_water[c]), a));
                rgb[c] = ad(ml(R, sky), ml(sb(1.0f, R), refr));
            }
        } else {
            float v, u = 0.0f, vv = 0.0f;
            if constexpr (kMode == CEL_RENDER_ETA) v = sb(wc, ws);
            const float hd = h > p.h_min ? h : p.h_min;
            if constexpr (kP) v = u = dv(tofloat(A.P[(size_t)j * G.px + i]), hd);
            if constexpr (kQ) v = vv = dv(SQ.v[cy][lane], hd);
            if constexpr (kMode == CEL_RENDER_SPEED) v = sq(ad(ml(u, u), ml(vv, vv)));
            colormap(T, kMode == CEL_RENDER_SPEED ? 1 : 0, dv(sb(v, p.vmin), sb(p.vmax, p.vmin)), rgb);
        }
        if (p.grid > 0.0f && (s_line[0][lane] | s_line[1][cy])) {
#pragma unroll
            for (int c = 0; c < 3; c++) rgb[c] = ml(rgb[c], 0.6f);
        }
        const uint32_t rg = __byte_perm(to_byte(rgb[0]), to_byte(rgb[1]), 0x0040);
        const uint32_t px = __byte_perm(rg, __byte_perm(to_byte(rgb[2]), 0xffu, 0x0040), 0x5410);
        reinterpret_cast<uint32_t *>(A.rgba)[(size_t)j * nx + i] = px;
    }
}

}  // namespace

template <typename real>
cudaError_t launch_render(const RenderArgs<real> &a, cudaStream_t st)
{
    dim3 grid((a.geo.nx + kRT - 1) / kRT, (a.geo.ny + kRT - 1) / kRT), block(32, 8);
    switch (a.p.mode) {
    case CEL_RENDER_ETA: k_render<real, CEL_RENDER_ETA><<<grid, block, 0, st>>>(a); break;
    case CEL_RENDER_U: k_render<real, CEL_RENDER_U><<<grid, block, 0, st>>>(a); break;
    case CEL_RENDER_V: k_render<real, CEL_RENDER_V><<<grid, block, 0, st>>>(a); break;
    case CEL_RENDER_SPEED: k_render<real, CEL_RENDER_SPEED><<<grid, block, 0, st>>>(a); break;
    default: k_render<real, CEL_RENDER_FRESNEL><<<grid, block, 0, st>>>(a); break;
    }
    return cudaGetLastError();
}

template cudaError_t launch_render<float>(const RenderArgs<float> &, cudaStream_t);
template cudaError_t launch_render<double>(const RenderArgs<double> &, cudaStream_t);

}  // namespace cel
