// Ray casting of the fused TSDF (views of the reconstruction and tests).
//
// One thread per pixel marches camera depths z_i = depth_min + i * tau/2 up
// to depth_max through the trilinear field of observed cells (+-1 nodes
// included, unlike the fitness, which needs nodes inside the band); the
// first step from a positive to a non-positive value is refined by linear
// interpolation.  The normal is the normalised central difference of the
// field at +-voxel/2 along each world axis.
//
// Bound: the latency of a chain of dependent steps, hundreds per ray, eight
// node gathers each.  Nearly all of them cross free or unobserved space, where
// no sample can end the march: a cell whose observed corners are all positive
// interpolates to a positive value (each rounded step stays between its end
// points: fma(f, rn(b - a), a) >= min(a, b) for 0 <= f < 1).  The volume's
// surface map says which bricks of 8^3 cells have any other corner, 64 bricks
// to a word, so a ray jumps to the exit of a clear brick or of a whole clear
// word (32^3 cells), and evaluates only the samples in set bricks and the one
// before each run of them (the crossing needs its value).  Every sample that
// is evaluated is the one the plain march evaluates, at the same rounded
// depth, so the results are the same bits.
// Measured, 640x480 of an uploaded 512^3 room with normals, the same view again
// and again: 308 -> 52 us; each time a view not cast before, of a 512^3 map while
// 100 distinct views are fused into it: 372 -> 128 us for the last 50 (768^3
// half precision 599 -> 155).  A map whose set bricks consist mostly of cells
// with an unobserved corner is the one kind that loses: the plain march's first
// load told it so, here come a lookup and eight loads (64^3, solid, half of the
// nodes unobserved at random: 48 -> 62 us).  Loading that corner first took 2 to
// 8% more for every other map, and 53 to 60 us there.
#include "pf_internal.cuh"

namespace {

struct RayArgs {
    const void* tsdf;
    int nx, ny, nz;
    float inv_vs;
    float org[3];
    float half_vs;
    CamK cam;
    float R[9], t[3];
    float step;
    int nsteps;
    SurfaceMap surf;
    float* depth;
    float* normal;
};

// Trilinear value of an observed cell at world point q; false when the cell
// is outside the grid or has an unobserved node.
template <typename TS>
__device__ inline bool sample_observed(const RayArgs& a, float qx, float qy, float qz, float& out)
{
    const float gx = (qx - a.org[0]) * a.inv_vs;
    const float gy = (qy - a.org[1]) * a.inv_vs;
    const float gz = (qz - a.org[2]) * a.inv_vs;
    if (!(gx >= 0.0f && gx < (float)(a.nx - 1) && gy >= 0.0f && gy < (float)(a.ny - 1) && gz >= 0.0f &&
          gz < (float)(a.nz - 1)))
        return false;
    const float fx0 = floorf(gx), fy0 = floorf(gy), fz0 = floorf(gz);
    const int nxy = a.nx * a.ny;
    const int base = (int)fx0 + a.nx * (int)fy0 + nxy * (int)fz0;
    const int off[8] = {0, 1, a.nx, a.nx + 1, nxy, nxy + 1, nxy + a.nx, nxy + a.nx + 1};
    // all eight loads before the first test, so that they wait together
    float v[8];
    bool ok = true;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const float e = pf_to_float(static_cast<const TS*>(a.tsdf)[base + off[q]]);
        ok = ok && e == e;  // NaN: unobserved
        v[q] = pf_decode(e);
    }
    if (!ok) return false;
    const float fx = gx - fx0, fy = gy - fy0, fz = gz - fz0;
    const float x00 = fmaf(fx, v[1] - v[0], v[0]);
    const float x10 = fmaf(fx, v[3] - v[2], v[2]);
    const float x01 = fmaf(fx, v[5] - v[4], v[4]);
    const float x11 = fmaf(fx, v[7] - v[6], v[6]);
    const float y0 = fmaf(fy, x10 - x00, x00);
    const float y1 = fmaf(fy, x11 - x01, x01);
    out = fmaf(fz, y1 - y0, y0);
    return true;
}

template <typename TS>
__global__ void raycast_kernel(RayArgs a)
{
    const int u = blockIdx.x * blockDim.x + threadIdx.x;
    const int v = blockIdx.y * blockDim.y + threadIdx.y;
    if (u >= a.cam.width || v >= a.cam.height) return;
    const float dcx = __fdiv_rn((float)u - a.cam.cx, a.cam.fx);
    const float dcy = __fdiv_rn((float)v - a.cam.cy, a.cam.fy);
    const float dx = a.R[0] * dcx + a.R[1] * dcy + a.R[2];
    const float dy = a.R[3] * dcx + a.R[4] * dcy + a.R[5];
    const float dz = a.R[6] * dcx + a.R[7] * dcy + a.R[8];
    // Grid coordinate of sample i on axis r: about g0 + z_i gd.  slack covers
    // the rounding of the exact expression the samples use, several times
    // over, so that a sample whose neighbours on the ray lie in a box shrunk
    // by it lies in the box.
    const float tt[3] = {a.t[0], a.t[1], a.t[2]}, dd[3] = {dx, dy, dz};
    const int n[3] = {a.nx, a.ny, a.nz};
    const float zmax = fmaf((float)a.nsteps, a.step, a.cam.dmin);
    float slack[3], per_step[3];
    float first = 0.0f, last = (float)a.nsteps;
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        slack[r] = 0.01f + 2e-6f * (fabsf(tt[r]) + fabsf(a.org[r]) + zmax * fabsf(dd[r])) * a.inv_vs;
        per_step[r] = 1.0f / (dd[r] * a.inv_vs * a.step);  // steps per voxel (infinite when the ray keeps the axis)
        const float g0 = (fmaf(a.cam.dmin, dd[r], tt[r]) - a.org[r]) * a.inv_vs;
        const float s0 = (-1.0f - slack[r] - g0) * per_step[r], s1 = ((float)n[r] + slack[r] - g0) * per_step[r];
        first = fmaxf(first, fminf(s0, s1) - 1.0f);
        last = fminf(last, fmaxf(s0, s1) + 1.0f);
    }
    float hit = 0.0f;
    bool have_prev = false;
    float prev = 0.0f;
    int known = -1;  // the sample that have_prev and prev describe
    // (outside [first, last] every sample lies outside the grid)
    const int end = last >= 0.0f ? min((int)last, a.nsteps) : -1;
    for (int i = first <= last ? (int)first : end + 1; i <= end;) {
        const float z = fmaf((float)i, a.step, a.cam.dmin);
        const float q[3] = {fmaf(z, dx, a.t[0]), fmaf(z, dy, a.t[1]), fmaf(z, dz, a.t[2])};
        float g[3];
        int b[3];
        bool inside = true;
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            g[r] = (q[r] - a.org[r]) * a.inv_vs;
            inside = inside && g[r] >= 0.0f && g[r] < (float)(n[r] - 1);
            b[r] = (int)g[r] >> 3;
        }
        if (!inside) {
            ++i;
            continue;
        }
        const unsigned long long w =
            __ldg(a.surf.words + (b[0] >> 2) + a.surf.wx * ((b[1] >> 2) + a.surf.wy * (b[2] >> 2)));
        if ((w >> ((b[0] & 3) | ((b[1] & 3) << 2) | ((b[2] & 3) << 4)) & 1ull) == 0ull) {
            // no surface in this brick (or in its whole word): on to the last
            // sample that is certainly inside it, and one further
            const int sh = w == 0ull ? 2 : 0;
            const float side = w == 0ull ? 32.0f : 8.0f;
            float run = 1e9f;
#pragma unroll
            for (int r = 0; r < 3; ++r) {
                const float lo = (float)((b[r] >> sh) << (3 + sh)) + slack[r], hi = lo + side - 2.0f * slack[r];
                run = g[r] >= lo && g[r] <= hi ? fminf(run, fmaxf((lo - g[r]) * per_step[r], (hi - g[r]) * per_step[r]))
                                               : 0.0f;
                if (run <= 0.0f) break;
            }
            i += 1 + (int)fminf(fmaxf(run, 0.0f), 65536.0f);
            continue;
        }
        if (known != i - 1) {
            const float zp = fmaf((float)(i - 1), a.step, a.cam.dmin);
            have_prev = i > 0 && sample_observed<TS>(a, fmaf(zp, dx, a.t[0]), fmaf(zp, dy, a.t[1]), fmaf(zp, dz, a.t[2]), prev);
        }
        float t = 0.0f;
        const bool ok = sample_observed<TS>(a, q[0], q[1], q[2], t);
        if (ok && have_prev && prev > 0.0f && t <= 0.0f) {
            hit = (z - a.step) + a.step * __fdiv_rn(prev, prev - t);
            break;
        }
        have_prev = ok;
        prev = t;
        known = i++;
    }
    const size_t pix = (size_t)v * a.cam.width + u;
    a.depth[pix] = hit;
    if (a.normal) {
        float n[3] = {NAN, NAN, NAN};
        if (hit > 0.0f) {
            const float q[3] = {fmaf(hit, dx, a.t[0]), fmaf(hit, dy, a.t[1]), fmaf(hit, dz, a.t[2])};
            float g[3];
            bool ok = true;
            for (int ax = 0; ax < 3 && ok; ++ax) {
                float qp[3] = {q[0], q[1], q[2]}, qm[3] = {q[0], q[1], q[2]};
                qp[ax] += a.half_vs;
                qm[ax] -= a.half_vs;
                float tp, tm;
                ok = sample_observed<TS>(a, qp[0], qp[1], qp[2], tp) && sample_observed<TS>(a, qm[0], qm[1], qm[2], tm);
                g[ax] = tp - tm;
            }
            if (ok) {
                const float len = sqrtf(g[0] * g[0] + g[1] * g[1] + g[2] * g[2]);
                if (len > 0.0f)
                    for (int ax = 0; ax < 3; ++ax) n[ax] = g[ax] / len;
            }
        }
        for (int ax = 0; ax < 3; ++ax) a.normal[3 * pix + ax] = n[ax];
    }
}

}  // namespace

static pf_status pf_raycast_impl(const pf_volume* v, const pf_intrinsics* intr, const double P[16], float* depth_out,
                                 float* normal_out, void* stream)
{
    if (!v || !P || !depth_out) return PF_ERR_INVALID_ARG;
    pf_status st = pf::check_intrinsics(intr);
    if (st != PF_OK) return st;
    for (int q = 0; q < 12; ++q)
        if (!std::isfinite(P[q])) return PF_ERR_INVALID_ARG;
    RayArgs a;
    a.tsdf = v->tsdf;
    a.nx = v->desc.nx;
    a.ny = v->desc.ny;
    a.nz = v->desc.nz;
    a.inv_vs = 1.0f / v->desc.voxel_size;
    a.half_vs = 0.5f * v->desc.voxel_size;
    for (int q = 0; q < 3; ++q) a.org[q] = v->desc.origin[q];
    a.cam = make_cam(intr);
    for (int r = 0; r < 3; ++r) {
        for (int c = 0; c < 3; ++c) a.R[3 * r + c] = (float)P[4 * r + c];
        a.t[r] = (float)P[4 * r + 3];
    }
    a.step = 0.5f * v->desc.trunc;
    a.nsteps = (int)floor(((double)intr->depth_max - (double)intr->depth_min) / (double)a.step);
    a.surf = v->surf;
    a.depth = depth_out;
    a.normal = normal_out;
    // a warp covers 8 x 4 pixels: its rays pass the same bricks
    dim3 block(8, 16);
    dim3 grid((intr->width + 7) / 8, (intr->height + 15) / 16);
    cudaStream_t s = (cudaStream_t)stream;
    pf::timing_begin(pf::KC_RAYCAST, s);
    if (v->desc.tsdf_dtype == PF_F16)
        raycast_kernel<__half><<<grid, block, 0, s>>>(a);
    else if (v->desc.tsdf_dtype == PF_BF16)
        raycast_kernel<__nv_bfloat16><<<grid, block, 0, s>>>(a);
    else if (v->desc.tsdf_dtype == PF_FP8E4M3)
        raycast_kernel<__nv_fp8_e4m3><<<grid, block, 0, s>>>(a);
    else
        raycast_kernel<float><<<grid, block, 0, s>>>(a);
    pf::count_launch();
    pf::timing_end(pf::KC_RAYCAST, s);
    PF_LAUNCHED();
    return PF_OK;
}

// Every entry point that takes a volume keeps its last failing status
// there (pf_volume_last_error).
extern "C" {

pf_status pf_raycast(const pf_volume* v, const pf_intrinsics* intr, const double P[16], float* depth_out,
                     float* normal_out, void* stream)
{
    return pf::keep_status(v, pf_raycast_impl(v, intr, P, depth_out, normal_out, stream));
}

}  // extern "C"
