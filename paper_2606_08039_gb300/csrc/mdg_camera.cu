// Camera frames by ray casting (the RGB observation of Section 3.4.4: 48 x 64 frames from
// each drone's onboard camera, 60 degree field of view, at [0.02, 0, 0] in the body frame).
// The paper renders them with MuJoCo's OpenGL renderer and the Crazyflie meshes; here every
// frame is ray cast in a kernel from primitive shapes:
//   - pinhole camera along body +x, image right = body -y, image up = body +z, 60 degrees
//     the vertical field of view, each pixel through the centre of its cell, row 0 on top;
//   - the environment's other drones as oblate ellipsoids in their body frames, semi-axes
//     (L + r_p, L + r_p, 0.3 (L + r_p)); the ground z = 0 as a 0.5 m checkerboard seen from
//     above; the camera's own drone is not drawn;
//   - Lambert shading, ambient 0.35 + diffuse 0.65 max(0, n . l), l along (0.3, 0.2, 1);
//     ground greys 0.55 / 0.35, drone k coloured by the palette entry k mod 8, sky
//     (0.55, 0.70, 0.90) unshaded; channels round(255 c), alpha 255;
//   - depth along the optical axis to the nearest hit beyond 1e-4 m (+inf: sky);
//     segmentation -1 sky, 0 ground, 1 + the global index of the drone hit.
// A team of threads takes one camera: one warp in batches whose environments have at most 32
// drones, a 128-thread block otherwise. It first builds, in shared memory, each drone's ray
// transform (world direction -> the drone's scaled body frame), the camera origin in that frame,
// the normal transform and the drone's screen rectangle, then for each 16 x 8 pixel tile (one
// warp's pixels, four adjacent columns a lane) the mask of drones whose rectangles it meets; a
// pixel pays a ~25-flop ray-ellipsoid test only for the drones of its tile's mask (above 64
// drones per environment, the rectangles are tested per drone).
//
// What bounds it: the frames' bytes, nearly. 16,396 cameras of four drones, colour and
// segmentation (403 MB): 170 us with one pixel a thread and step (about 124 instructions a pixel)
// -> 66 us, 6.1 TB/s. Four columns a lane share the row's terms and the drones' records and store
// 16 bytes at a time; the ground's checker needs no float-to-integer conversion, and its two
// colours and the sky's are packed once; a warp per camera needs no block barrier, so that one
// camera's setup overlaps the others' pixels. Registers: 93 a thread (five blocks an SM); held to
// 80, 72 and 64 it took 72, 74 and 85 us.
#include "mdg_internal.cuh"

namespace mdg {
namespace {

constexpr int kCamH = 48, kCamW = 64, kCamPixels = kCamH * kCamW;
constexpr int kCamThreads = 128;
constexpr float kTMin = 1e-4f;
// unit light direction (0.3, 0.2, 1) / |(0.3, 0.2, 1)|
constexpr float kLx = 0.28221626f, kLy = 0.18814417f, kLz = 0.94072087f;

__constant__ float c_palette[8][3] = {{0.90f, 0.25f, 0.20f}, {0.20f, 0.70f, 0.30f}, {0.20f, 0.35f, 0.90f},
                                      {0.95f, 0.75f, 0.15f}, {0.70f, 0.30f, 0.80f}, {0.15f, 0.75f, 0.80f},
                                      {0.95f, 0.50f, 0.20f}, {0.60f, 0.60f, 0.65f}};

// Per drone of the environment, in shared memory, seven float4 (a ray test reads the first
// four): O = the camera origin in the drone's scaled body frame, M = diag(1/s) R^T (world
// ray -> scaled body ray, row r in float4 1 + r), C = |O|^2 - 1, Nm = R diag(1/s) (scaled
// body point -> world normal direction), its segment id, and the pixel rectangle
// [r0, r1] x [c0, c1] outside which no ray can meet it (the projection of its oriented
// bounding box, half-extents (a, a, c) along its body axes, padded by a pixel; empty when
// its bounding cube of half-width a lies behind the camera or beyond a side plane of the
// view frustum, or for the camera's own drone; the whole image when the cube straddles the
// image plane inside the frustum):
//   0: O0 O1 O2 C      1: M00 M01 M02 Nm0   2: M10 M11 M12 Nm1   3: M20 M21 M22 Nm2
//   4: Nm3 Nm4 Nm5 Nm6   5: Nm7 Nm8 id r0   6: r1 c0 c1 -
constexpr int kSceneF4 = 7;

// Square root and reciprocal of the special function unit (relative error near 2^-23): the
// hit distance of a ray-ellipsoid test, well inside the depth tolerance.
__device__ __forceinline__ float sqrt_approx(float x)
{
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float rcp_approx(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// 1 / x, correctly rounded, where x and the result are normal: the approximation and a Newton step (equal to
// the division for all 2^23 mantissas).
__device__ __forceinline__ float rcp_newton(float x)
{
    const float r = rcp_approx(x);
    return fmaf(r, fmaf(-x, r, 1.f), r);
}

struct Rot {
    float m[9];  // row-major, body -> world
};

__device__ __forceinline__ Rot rot_of(float w, float x, float y, float z)
{
    Rot R;
    R.m[0] = 1.f - 2.f * (y * y + z * z);
    R.m[1] = 2.f * (x * y - w * z);
    R.m[2] = 2.f * (x * z + w * y);
    R.m[3] = 2.f * (x * y + w * z);
    R.m[4] = 1.f - 2.f * (x * x + z * z);
    R.m[5] = 2.f * (y * z - w * x);
    R.m[6] = 2.f * (x * z - w * y);
    R.m[7] = 2.f * (y * z + w * x);
    R.m[8] = 1.f - 2.f * (x * x + y * y);
    return R;
}

// Four bytes of a pixel: channels round(255 c), alpha 255.
__device__ __forceinline__ uint32_t pack_rgba(float r, float g, float b)
{
    const uint32_t R8 = (uint32_t)__float2int_rn(255.f * __saturatef(r));
    const uint32_t G8 = (uint32_t)__float2int_rn(255.f * __saturatef(g));
    const uint32_t B8 = (uint32_t)__float2int_rn(255.f * __saturatef(b));
    return R8 | (G8 << 8) | (B8 << 16) | 0xff000000u;
}

// floor(2 x) in the low bits, for |2 x| < 2^22: adding 1.5 * 2^23 rounding down leaves it in the
// mantissa (no conversion, which runs at an eighth of the rate).
__device__ __forceinline__ uint32_t floor2(float x) { return __float_as_uint(__fmaf_rd(x, 2.f, 12582912.f)); }

constexpr int kTileW = 16, kTileH = 8, kTilesX = kCamW / kTileW, kTilesY = kCamH / kTileH;
constexpr int kTiles = kTilesX * kTilesY;
constexpr int kPx = 4;  // adjacent columns of a lane

// Four consecutive 4-byte pixels of an output: one 16-byte store when the outputs are 16-byte
// aligned (a frame is a multiple of 16 bytes), four otherwise.
__device__ __forceinline__ void store4(void* base, long long px, bool vec, uint32_t a, uint32_t b, uint32_t c, uint32_t d)
{
    uint32_t* p = static_cast<uint32_t*>(base) + px;
    if (vec) {
        *reinterpret_cast<uint4*>(p) = make_uint4(a, b, c, d);
    } else {
        p[0] = a, p[1] = b, p[2] = c, p[3] = d;
    }
}

template <int kTeam>
__global__ void __launch_bounds__(kCamThreads) render_kernel(const CamArgs a)
{
    constexpr bool kWarp = kTeam == 32;
    extern __shared__ float4 s_all[];  // per team: [max_env][kSceneF4]
    __shared__ unsigned long long s_mask[kWarp ? 1 : kTiles];
    const int team = threadIdx.x / kTeam, t = threadIdx.x % kTeam, lane = threadIdx.x & 31;
    const long long cam = (long long)blockIdx.x * (kCamThreads / kTeam) + team;
    if (cam >= a.n) return;  // a whole team
    float4* scene = s_all + team * a.max_env * kSceneF4;
    const float inv_a = 1.f / a.semi_a, inv_c = 1.f / a.semi_c;
    const float th = 0.57735026918962576f;  // tan(30 degrees)
    const float kInf = __int_as_float(0x7f800000);

    int first, N;
    if (a.uniform_N > 0) {
        N = a.uniform_N;
        first = (int)(cam / N * N);
    } else {
        int lo = 0, hi = a.n_envs - 1;  // largest env with env_off[env] <= cam
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (a.env_off[mid] <= cam) lo = mid;
            else hi = mid - 1;
        }
        first = a.env_off[lo];
        N = a.env_off[lo + 1] - first;
    }
    if (!MDG_CHECK(N >= 1 && N <= a.max_env && cam >= first && cam < first + N, a.status)) return;
    const float4 c0 = a.state[cam], c1 = a.state[a.n + cam];
    const Rot C = rot_of(c0.w, c1.x, c1.y, c1.z);  // the camera drone's rotation (body -> world)
    const float ox = c0.x + 0.02f * C.m[0], oy = c0.y + 0.02f * C.m[3], oz = c0.z + 0.02f * C.m[6];
    const int own_k = (int)(cam - first);
    for (int k = t; k < N; k += kTeam) {
        const long long g = first + k;
        const float4 p0 = a.state[g], p1 = a.state[a.n + g];
        const Rot R = rot_of(p0.w, p1.x, p1.y, p1.z);
        const float inv_s[3] = {inv_a, inv_a, inv_c};
        const float dx = ox - p0.x, dy = oy - p0.y, dz = oz - p0.z;
        float4* sc = scene + k * kSceneF4;
        float O[3], M[9], Nm[9];
        float Cq = -1.f;
        for (int r = 0; r < 3; ++r) {
            // row r of R^T is column r of R
            O[r] = (R.m[r] * dx + R.m[3 + r] * dy + R.m[6 + r] * dz) * inv_s[r];
            Cq += O[r] * O[r];
            M[3 * r + 0] = R.m[r] * inv_s[r];
            M[3 * r + 1] = R.m[3 + r] * inv_s[r];
            M[3 * r + 2] = R.m[6 + r] * inv_s[r];
        }
        for (int r = 0; r < 3; ++r)
            for (int q = 0; q < 3; ++q) Nm[3 * r + q] = R.m[3 * r + q] * inv_s[q];
        sc[0] = make_float4(O[0], O[1], O[2], Cq);
        sc[1] = make_float4(M[0], M[1], M[2], Nm[0]);
        sc[2] = make_float4(M[3], M[4], M[5], Nm[1]);
        sc[3] = make_float4(M[6], M[7], M[8], Nm[2]);
        sc[4] = make_float4(Nm[3], Nm[4], Nm[5], Nm[6]);
        const float seg_id = __int_as_float((int)(g + 1));
        // screen rectangle: the drone's centre in the camera drone's body frame
        const float ex = p0.x - ox, ey = p0.y - oy, ez = p0.z - oz;
        const float X = C.m[0] * ex + C.m[3] * ey + C.m[6] * ez;
        const float Y = C.m[1] * ex + C.m[4] * ey + C.m[7] * ez;
        const float Z = C.m[2] * ex + C.m[5] * ey + C.m[8] * ez;
        const float rho = a.semi_a;
        int r0 = 0, r1 = kCamH - 1, k0 = 0, k1 = kCamW - 1;
        // outside the view frustum: behind the camera, or beyond one of its four side
        // planes |nx| <= hx, |ny| <= hy (padded by two pixels); for a linear test the cube's
        // worst corner is the centre's value minus rho times the sum of |coefficients|
        const float hx = th * kCamW / kCamH * (1.f + 4.f / kCamW), hy = th * (1.f + 4.f / kCamH);
        const bool unseen = X + rho < 0.f || (-Y - hx * X) - rho * (1.f + hx) > 0.f ||
                            (Y - hx * X) - rho * (1.f + hx) > 0.f || (Z - hy * X) - rho * (1.f + hy) > 0.f ||
                            (-Z - hy * X) - rho * (1.f + hy) > 0.f;
        if (unseen) {
            r0 = 1, r1 = 0;  // empty
        } else if (X - rho > 1e-3f) {
            // the corners of the drone's own bounding box, half-extents (a, a, c) along its
            // body axes, in the camera drone's body frame: G = R_cam^T R_k (column q = the
            // drone's axis q) scaled by the half-extent
            float G[9];
            for (int r = 0; r < 3; ++r)
                for (int q = 0; q < 3; ++q)
                    G[3 * r + q] = (C.m[r] * R.m[q] + C.m[3 + r] * R.m[3 + q] + C.m[6 + r] * R.m[6 + q]) *
                                   (q == 2 ? a.semi_c : a.semi_a);
            float nx_lo = 1e30f, nx_hi = -1e30f, ny_lo = 1e30f, ny_hi = -1e30f;
            for (int corner = 0; corner < 8; ++corner) {
                const float sx = (corner & 1) ? 1.f : -1.f, sy = (corner & 2) ? 1.f : -1.f;
                const float sz = (corner & 4) ? 1.f : -1.f;
                const float cx = X + sx * G[0] + sy * G[1] + sz * G[2];
                const float cy = Y + sx * G[3] + sy * G[4] + sz * G[5];
                const float cz = Z + sx * G[6] + sy * G[7] + sz * G[8];
                const float ic = __fdividef(1.f, cx);  // the rectangle's padding covers its error
                const float nxc = -cy * ic, nyc = cz * ic;
                nx_lo = fminf(nx_lo, nxc);
                nx_hi = fmaxf(nx_hi, nxc);
                ny_lo = fminf(ny_lo, nyc);
                ny_hi = fmaxf(ny_hi, nyc);
            }
            // col = ((nx / (th W/H)) + 1) W/2 - 0.5, row = (1 - ny / th) H/2 - 0.5
            const float kx = 0.5f * kCamW / (th * kCamW / kCamH), ky = 0.5f * kCamH / th;
            k0 = max(0, (int)floorf((nx_lo * kx + 0.5f * kCamW - 0.5f)) - 1);
            k1 = min(kCamW - 1, (int)ceilf((nx_hi * kx + 0.5f * kCamW - 0.5f)) + 1);
            r0 = max(0, (int)floorf((0.5f * kCamH - ny_hi * ky - 0.5f)) - 1);
            r1 = min(kCamH - 1, (int)ceilf((0.5f * kCamH - ny_lo * ky - 0.5f)) + 1);
        }
        if (k == own_k) r0 = 1, r1 = 0;  // the camera's own drone: empty
        sc[5] = make_float4(Nm[7], Nm[8], seg_id, __int_as_float(r0));
        sc[6] = make_float4(__int_as_float(r1), __int_as_float(k0), __int_as_float(k1), 0.f);
    }
    if (kWarp) __syncwarp();
    else __syncthreads();
    // whether drone k's rectangle meets tile (tx, ty)
    auto meets = [&](int k, int tx, int ty) {
        const float4 q5 = scene[k * kSceneF4 + 5], q6 = scene[k * kSceneF4 + 6];
        return (ty + 1) * kTileH > __float_as_int(q5.w) && ty * kTileH <= __float_as_int(q6.x) &&
               (tx + 1) * kTileW > __float_as_int(q6.y) && tx * kTileW <= __float_as_int(q6.z) &&
               __float_as_int(q5.w) <= __float_as_int(q6.x);
    };
    // the drones of every tile, tile = tx * kTilesY + ty: lane `tile` of a warp team holds its mask
    uint32_t my_mask = 0;
    if (kWarp || N <= 64) {
        if (t < kTiles) {
            unsigned long long m = 0;
            for (int k = 0; k < N; ++k) m |= (unsigned long long)meets(k, t / kTilesY, t % kTilesY) << k;
            my_mask = (uint32_t)m;
            if (!kWarp) s_mask[t] = m;
        }
        if (kWarp) __syncwarp();
        else __syncthreads();
    }

    // the ground's two greys (normal +z) and the sky, packed
    const float shade_up = 0.35f + 0.65f * kLz;
    const float light = 0.55f * shade_up, dark = 0.35f * shade_up;
    const uint32_t c_light = pack_rgba(light, light, light), c_dark = pack_rgba(dark, dark, dark);
    const uint32_t c_sky = pack_rgba(0.55f, 0.70f, 0.90f);
    const bool vec = a.vec != 0, above = oz > 0.f;
    // the largest ray parameter for which both ground coordinates stay within 2^20 m (floor2), from
    // bounds of the origin and of the ray's horizontal components
    const float span = fmaxf(fabsf(C.m[0]) + fabsf(C.m[1]) + fabsf(C.m[2]), fabsf(C.m[3]) + fabsf(C.m[4]) + fabsf(C.m[5]));
    // (none, 0, where the slopes' reciprocals may leave the range of rcp_newton)
    const float rise = fabsf(C.m[6]) + fabsf(C.m[7]) + fabsf(C.m[8]);
    const uint32_t reach = __float_as_uint(
        fabsf(ox) < 262144.f && fabsf(oy) < 262144.f && rise < 0x1p120f ? 262144.f / fmaxf(span, 1.f) : 0.f);
    for (int tx = kWarp ? 0 : t >> 5; tx < (kWarp ? kTilesX : (t >> 5) + 1); ++tx) {
        const int col = tx * kTileW + (lane & 3) * kPx;
        // world direction of the body ray (1, -nx, ny), not normalised: its component along
        // the optical axis is 1, so the ray parameter t of a hit is its depth along the axis
        // (the minimum distance 1e-4 m is then taken along that axis)
        float e0[kPx], e1[kPx], e2[kPx];
#pragma unroll
        for (int i = 0; i < kPx; ++i) {
            const float nx = ((col + i + 0.5f) * (2.f / kCamW) - 1.f) * (th * kCamW / kCamH);
            e0[i] = fmaf(-nx, C.m[1], C.m[0]);
            e1[i] = fmaf(-nx, C.m[4], C.m[3]);
            e2[i] = fmaf(-nx, C.m[7], C.m[6]);
        }
#pragma unroll 1
        for (int ty = 0; ty < kTilesY; ++ty) {
            const int row = ty * kTileH + (lane >> 2);
            const float ny = (1.f - (row + 0.5f) * (2.f / kCamH)) * th;
            float d0[kPx], d1[kPx], d2[kPx], t_best[kPx];
            uint32_t color[kPx];
            int seg[kPx];
#pragma unroll
            for (int i = 0; i < kPx; ++i) {
                d0[i] = fmaf(ny, C.m[2], e0[i]);
                d1[i] = fmaf(ny, C.m[5], e1[i]);
                d2[i] = fmaf(ny, C.m[8], e2[i]);
                t_best[i] = kInf;
                color[i] = c_sky;
                seg[i] = -1;
            }
            // the ground: d2 is linear along the row, so the ends tell whether any pixel looks down
            if (above && fminf(d2[0], d2[kPx - 1]) < 0.f) {
                uint32_t far = 0;  // bits of the farthest hit (a NaN counts as farther than any)
                bool down[kPx];
#pragma unroll
                for (int i = 0; i < kPx; ++i) {
                    const float tg = -oz * rcp_newton(d2[i]);
                    down[i] = d2[i] < 0.f && !(tg <= kTMin);
                    t_best[i] = down[i] ? tg : kInf;
                    far = max(far, down[i] ? __float_as_uint(tg) : 0u);
                    seg[i] = down[i] ? 0 : -1;
                }
                if (far < reach) {
#pragma unroll
                    for (int i = 0; i < kPx; ++i) {
                        const float tg = t_best[i];  // an infinity gives no colour
                        const uint32_t odd = floor2(fmaf(tg, d0[i], ox)) ^ floor2(fmaf(tg, d1[i], oy));
                        color[i] = down[i] ? ((odd & 1u) ? c_dark : c_light) : c_sky;
                    }
                } else {  // close to the horizon: by the division itself, which takes any slope
#pragma unroll
                    for (int i = 0; i < kPx; ++i) {
                        const float tg = d2[i] < 0.f ? -oz * (1.f / d2[i]) : 0.f;
                        const bool hits = tg > kTMin;
                        t_best[i] = hits ? tg : kInf;
                        seg[i] = hits ? 0 : -1;
                        if (!hits) continue;
                        const float px = fmaf(tg, d0[i], ox), py = fmaf(tg, d1[i], oy);
                        const int odd = (int)floorf(px * 2.f) + (int)floorf(py * 2.f);
                        color[i] = (odd & 1) ? c_dark : c_light;
                    }
                }
            }
            // the tile's drones (the same for all lanes); above 64, the rectangles per drone
            unsigned long long cand = ~0ull;
            if (kWarp) cand = __shfl_sync(0xffffffffu, my_mask, tx * kTilesY + ty);
            else if (N <= 64) cand = s_mask[tx * kTilesY + ty];
            if (cand) {
                int hit[kPx] = {-1, -1, -1, -1};
                for (int k = 0;; ++k) {
                    if (kWarp || N <= 64) {
                        if (!cand) break;
                        k = __ffsll((long long)cand) - 1;
                        cand &= cand - 1;
                    } else {
                        if (k >= N) break;
                        if (!meets(k, tx, ty)) continue;
                    }
                    const float4* sc = scene + k * kSceneF4;
                    const float4 o = sc[0], m0 = sc[1], m1 = sc[2], m2 = sc[3];
#pragma unroll
                    for (int i = 0; i < kPx; ++i) {
                        const float D0 = m0.x * d0[i] + m0.y * d1[i] + m0.z * d2[i];
                        const float D1 = m1.x * d0[i] + m1.y * d1[i] + m1.z * d2[i];
                        const float D2 = m2.x * d0[i] + m2.y * d1[i] + m2.z * d2[i];
                        const float A = D0 * D0 + D1 * D1 + D2 * D2;
                        const float B = 2.f * (D0 * o.x + D1 * o.y + D2 * o.z);
                        const float disc = B * B - 4.f * A * o.w;
                        if (disc < 0.f) continue;
                        const float sq = sqrt_approx(disc), i2a = 0.5f * rcp_approx(A);
                        const float t1 = (-B - sq) * i2a, t2 = (-B + sq) * i2a;
                        const float tk = t1 > kTMin ? t1 : (t2 > kTMin ? t2 : kInf);
                        if (tk < t_best[i]) {
                            t_best[i] = tk;
                            hit[i] = k;
                        }
                    }
                }
#pragma unroll
                for (int i = 0; i < kPx; ++i) {
                    if (hit[i] < 0) continue;
                    const float4* sc = scene + hit[i] * kSceneF4;
                    const float4 o = sc[0], m0 = sc[1], m1 = sc[2], m2 = sc[3], q4 = sc[4], q5 = sc[5];
                    const float D0 = m0.x * d0[i] + m0.y * d1[i] + m0.z * d2[i];
                    const float D1 = m1.x * d0[i] + m1.y * d1[i] + m1.z * d2[i];
                    const float D2 = m2.x * d0[i] + m2.y * d1[i] + m2.z * d2[i];
                    const float P0 = o.x + t_best[i] * D0, P1 = o.y + t_best[i] * D1, P2 = o.z + t_best[i] * D2;
                    const float n0 = m0.w * P0 + m1.w * P1 + m2.w * P2;
                    const float n1 = q4.x * P0 + q4.y * P1 + q4.z * P2;
                    const float n2 = q4.w * P0 + q5.x * P1 + q5.y * P2;
                    const float in = rsqrtf(fmaxf(n0 * n0 + n1 * n1 + n2 * n2, 1e-30f));
                    const float nl = (n0 * kLx + n1 * kLy + n2 * kLz) * in;
                    const float shade = 0.35f + 0.65f * fmaxf(0.f, nl);
                    seg[i] = __float_as_int(q5.z);
                    const int pc = (seg[i] - 1) & 7;
                    color[i] = pack_rgba(c_palette[pc][0] * shade, c_palette[pc][1] * shade, c_palette[pc][2] * shade);
                }
            }
            const long long o = cam * kCamPixels + row * kCamW + col;
            if (a.rgba) store4(a.rgba, o, vec, color[0], color[1], color[2], color[3]);
            if (a.depth)  // +inf for sky
                store4(a.depth, o, vec, __float_as_uint(t_best[0]), __float_as_uint(t_best[1]), __float_as_uint(t_best[2]),
                       __float_as_uint(t_best[3]));
            if (a.seg) store4(a.seg, o, vec, (uint32_t)seg[0], (uint32_t)seg[1], (uint32_t)seg[2], (uint32_t)seg[3]);
        }
    }
}

}  // namespace

cudaError_t launch_render(const CamArgs& a, cudaStream_t s)
{
    if (a.n == 0) return cudaSuccess;
    // one warp a camera while a record per lane holds the environment (the masks are 32 bits then)
    const bool warp = a.max_env <= 32;
    const int teams = warp ? kCamThreads / 32 : 1;
    const int smem = teams * a.max_env * kSceneF4 * (int)sizeof(float4);
    if (smem > 48 * 1024) {  // the block form above 438 drones
        static bool done[64] = {};
        cudaError_t e = opt_in_shared((const void*)render_kernel<kCamThreads>, MDG_MAX_ENV_DRONES * kSceneF4 * sizeof(float4),
                                      done);
        if (e != cudaSuccess) return e;
    }
    const long long grid = (a.n + teams - 1) / teams;
    if (warp) render_kernel<32><<<(unsigned)grid, kCamThreads, smem, s>>>(a);
    else render_kernel<kCamThreads><<<(unsigned)grid, kCamThreads, smem, s>>>(a);
    return cudaGetLastError();
}

}  // namespace mdg
