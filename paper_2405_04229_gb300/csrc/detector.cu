// Detector handle: per-shower ground histogram geometry and telescope
// spheres with a uniform grid hash, so each photon tests only the spheres
// whose reach covers its ground point (the telescope layouts of the thesis's
// App. B.3 have tens to thousands of spheres).
#include <math.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "common.cuh"

namespace {

// the largest arrival zeniths [deg] of the hash levels' lists; the last one is the level's own
constexpr double kHashTheta[cs::kHashLevels][cs::kHashSubs] = {{24.0, 34.0, 45.0}, {60.0, 67.0, 75.0}, {77.0, 79.0, 82.0}};
constexpr double kDeg = 3.14159265358979323846 / 180.0;

void split(double v, float* hi, float* lo) {
    *hi = (float)v;
    *lo = (float)(v - (double)*hi);
}

size_t align_up(size_t v) { return (v + 255) & ~(size_t)255; }

}  // namespace

extern "C" cs_status cs_detector_create(const cs_detector_desc* d, cs_detector** out) {
    if (!d || !out) return CS_ERR_INVALID_ARG;
    *out = nullptr;
    if (d->n_showers < 1) return CS_ERR_INVALID_ARG;
    if (d->hist_nx < 0 || d->hist_ny < 0 || (d->hist_nx > 0) != (d->hist_ny > 0)) return CS_ERR_INVALID_ARG;
    if (d->hist_nx > 0 && (!(d->hist_dx > 0.0) || !(d->hist_dy > 0.0))) return CS_ERR_INVALID_ARG;
    if ((double)d->hist_nx * d->hist_ny * d->n_showers > 4e9) return CS_ERR_INVALID_ARG;
    if (d->n_tel < 0 || (d->n_tel > 0 && !d->tel_xyzr)) return CS_ERR_INVALID_ARG;
    if (d->geometry != CS_GEOM_PLANAR && d->geometry != CS_GEOM_SPHERICAL && d->geometry != CS_GEOM_CYLINDRICAL)
        return CS_ERR_INVALID_ARG;
    if (d->geometry != CS_GEOM_PLANAR && (d->earth_radius < 0.0 || !isfinite(d->earth_radius)))
        return CS_ERR_INVALID_ARG;
    for (int i = 0; i < d->n_tel; ++i) {
        const double* t = d->tel_xyzr + 4 * i;
        if (!isfinite(t[0]) || !isfinite(t[1]) || !isfinite(t[2]) || !(t[3] > 0.0)) return CS_ERR_INVALID_ARG;
    }
    if (d->cam_n < 0 || d->cam_n > 4096) return CS_ERR_INVALID_ARG;
    if (d->cam_n > 0) {   // the optics: positive sizes, and every sphere must hold its instrument
        if (!(d->mirror_d > 0.0) || !(d->focal_f > 0.0) || !(d->camera_r > 0.0) || !isfinite(d->mirror_d) ||
            !isfinite(d->focal_f) || !isfinite(d->camera_r) || !isfinite(d->point_zenith) ||
            !isfinite(d->point_azimuth))
            return CS_ERR_INVALID_ARG;
        const double hold = sqrt(0.25 * d->mirror_d * d->mirror_d + 0.25 * d->focal_f * d->focal_f);
        for (int i = 0; i < d->n_tel; ++i)
            if (d->tel_xyzr[4 * i + 3] < hold) return CS_ERR_INVALID_ARG;
        if ((double)d->n_showers * d->n_tel * d->cam_n * d->cam_n > 4e9) return CS_ERR_INVALID_ARG;
        if (d->eff_n < 0 || d->eff_n > 16) return CS_ERR_INVALID_ARG;
        if (d->eff_n > 0 && (!d->eff_lambda_nm || !d->eff_mirror || !d->eff_camera)) return CS_ERR_INVALID_ARG;
        for (int i = 0; i < d->eff_n; ++i) {
            if (!isfinite(d->eff_lambda_nm[i]) || !(d->eff_mirror[i] >= 0.0 && d->eff_mirror[i] <= 1.0) ||
                !(d->eff_camera[i] >= 0.0 && d->eff_camera[i] <= 1.0))
                return CS_ERR_INVALID_ARG;
            if (i > 0 && !(d->eff_lambda_nm[i] > d->eff_lambda_nm[i - 1])) return CS_ERR_INVALID_ARG;
        }
    }
    cs_status st = cs::check_device();
    if (st != CS_OK) return st;

    cs_detector* h = new cs_detector;
    memset(h, 0, sizeof *h);
    cudaGetDevice(&h->device);
    cs::DetParams& p = h->p;
    p.n_showers = d->n_showers;
    p.spherical = d->geometry == CS_GEOM_SPHERICAL ? 1 : 0;
    p.cylindrical = d->geometry == CS_GEOM_CYLINDRICAL ? 1 : 0;
    p.R = d->earth_radius > 0.0 ? d->earth_radius : 6370000.0;
    p.h_obs = d->h_obs;
    p.h_obs_f = (float)d->h_obs;
    p.nx = d->hist_nx;
    p.ny = d->hist_ny;
    if (p.nx > 0) {
        split(d->hist_x0, &p.hx0_hi, &p.hx0_lo);
        split(d->hist_y0, &p.hy0_hi, &p.hy0_lo);
        p.inv_dx = (float)(1.0 / d->hist_dx);
        p.inv_dy = (float)(1.0 / d->hist_dy);
    }
    p.n_tel = d->n_tel;
    p.cam_n = d->n_tel > 0 ? d->cam_n : 0;
    if (p.cam_n > 0) {
        // telescope frame: axis a towards the pointing, e1 = a x z-hat (x-hat at zenith), e2 = a x e1
        const double th = d->point_zenith, ph = d->point_azimuth;
        const double a[3] = {sin(th) * cos(ph), sin(th) * sin(ph), cos(th)};
        double e1[3] = {a[1], -a[0], 0.0};
        const double n1 = sqrt(e1[0] * e1[0] + e1[1] * e1[1]);
        if (n1 < 1e-12) { e1[0] = 1.0; e1[1] = 0.0; } else { e1[0] /= n1; e1[1] /= n1; }
        const double e2[3] = {a[1] * e1[2] - a[2] * e1[1], a[2] * e1[0] - a[0] * e1[2], a[0] * e1[1] - a[1] * e1[0]};
        p.ax = (float)a[0]; p.ay = (float)a[1]; p.az = (float)a[2];
        p.e1x = (float)e1[0]; p.e1y = (float)e1[1]; p.e1z = (float)e1[2];
        p.e2x = (float)e2[0]; p.e2y = (float)e2[1]; p.e2z = (float)e2[2];
        p.cam_f = (float)d->focal_f;
        p.cam_rd2 = (float)(0.25 * d->mirror_d * d->mirror_d);
        p.cam_r = (float)d->camera_r;
        p.cam_scale = (float)(d->cam_n / (2.0 * d->camera_r));
        p.eff_n = d->eff_n;
        for (int i = 0; i < d->eff_n; ++i) {
            p.eff_l[i] = (float)d->eff_lambda_nm[i];
            p.eff_R[i] = (float)d->eff_mirror[i];
            p.eff_E[i] = (float)d->eff_camera[i];
        }
    }

    // host-side layout: tel float4, tel_lo float2, tel3 float4, then per hash level
    // its cell ranges, entry telescope indices and entry data
    std::vector<float4> tel(d->n_tel), tel3(p.spherical ? d->n_tel : 0);
    std::vector<float2> tel_lo(d->n_tel);
    for (int i = 0; i < d->n_tel; ++i) {
        const double* t = d->tel_xyzr + 4 * i;
        float lo;
        split(t[0], &tel[i].x, &lo); tel_lo[i].x = lo;
        split(t[1], &tel[i].y, &lo); tel_lo[i].y = lo;
        tel[i].z = (float)(t[2] - d->h_obs);
        tel[i].w = (float)t[3];
        if (p.spherical) {   // centre h = t[2] above the azimuthal-equidistant point (x, y)
            const double rg = p.R + d->h_obs, sx = sqrt(t[0] * t[0] + t[1] * t[1]), a = sx / rg;
            const double r = p.R + t[2], cx = sx > 0.0 ? t[0] / sx : 1.0, cy = sx > 0.0 ? t[1] / sx : 0.0;
            tel3[i] = make_float4((float)(r * sin(a) * cx), (float)(r * sin(a) * cy), (float)(r * cos(a) - p.R),
                                  (float)t[3]);
        }
    }
    std::vector<int2> range[cs::kHashLevels];
    std::vector<int> cell_tel[cs::kHashLevels];
    std::vector<float4> cell_data[cs::kHashLevels];
    for (int level = 0; level < cs::kHashLevels && d->n_tel > 0; ++level) {
        cs::TelHash& H = p.hash[level];
        // ground points whose arrival line (zenith <= theta) passes within r of
        // the centre lie within r / cos + |dz| tan of the centre's footprint
        auto reach = [&](int i, double theta) {
            const double* t = d->tel_xyzr + 4 * i;
            return t[3] / cos(theta) + fabs(t[2] - d->h_obs) * tan(theta) + 0.01;
        };
        const double theta_h = kHashTheta[level][cs::kHashSubs - 1] * kDeg;
        double reach_max = 0.0, reach_min = 0.0, x0 = 1e300, x1 = -1e300, y0 = 1e300, y1 = -1e300;
        for (int i = 0; i < d->n_tel; ++i) {
            const double* t = d->tel_xyzr + 4 * i;
            const double r = reach(i, theta_h);
            reach_max = fmax(reach_max, r);
            reach_min = fmax(reach_min, reach(i, kHashTheta[level][0] * kDeg));
            x0 = fmin(x0, t[0] - r); x1 = fmax(x1, t[0] + r);
            y0 = fmin(y0, t[1] - r); y1 = fmax(y1, t[1] + r);
        }
        // whole-metre origin and cell size: cell corners are exact in FP32.  Cells of half the
        // largest reach: a disc then covers ~25 cells, and a ground point's cell lists only the
        // spheres that can be near it (measured against 1, 1.5, 2 and 3 reaches: 2 % faster on
        // the 100-telescope grid and 4 % on the 2,000 inclined-shower telescopes than 2 reaches).
        // On the sphere, whose entries do not depend on the cells, of half the first list's reach
        // as long as the discs' cells stay few enough.
        // A level takes kHashSubs lists of 8 bytes a cell and 20 an entry.  Few spheres far apart
        // would take most of it for empty cells: their cells are larger, from 4e6 / kHashSubs cells
        // on (2,000 spheres over 20 km: 36 MB and 10 ms to create instead of 141 MB and 42 ms, the
        // same time a call); from 33,000 spheres on, whose lists lengthen with the cells, up to 4e6
        // (100,000 over 14 km, 4 % a call).
        x0 = floor(x0);
        y0 = floor(y0);
        double cell = fmax(ceil(0.5 * reach_max), 1.0);
        const double first = fmax(ceil(0.5 * reach_min), 1.0);
        if (p.spherical && (double)d->n_tel * (2.0 * reach_max / first + 1.0) * (2.0 * reach_max / first + 1.0) < 4e6 / cs::kHashSubs)
            cell = first;
        if (fabs(x0) > 8e6 || fabs(y0) > 8e6 || fabs(x1) > 8e6 || fabs(y1) > 8e6) {
            delete h;
            return CS_ERR_INVALID_ARG;
        }
        int gnx = (int)ceil((x1 - x0) / cell), gny = (int)ceil((y1 - y0) / cell);
        const double max_cells = fmin(fmax(4e6 / cs::kHashSubs, 40.0 * d->n_tel), 4e6);
        while ((double)gnx * gny > max_cells) { cell *= 2.0; gnx = (int)ceil((x1 - x0) / cell); gny = (int)ceil((y1 - y0) / cell); }
        gnx = gnx < 1 ? 1 : gnx;
        gny = gny < 1 ? 1 : gny;
        const size_t n_cells = (size_t)gnx * gny;
        // the kernel's cell index comes from FP32 coordinates: a few ulps at the grid's far corner
        const double slack = 4e-7 * fmax(fmax(fabs(x0), fabs(x1)), fmax(fabs(y0), fabs(y1)));
        // calls f(row, first column, last column) for the cells that the disc of radius r about
        // telescope i touches
        auto for_rows = [&](int i, double r, auto&& f) {
            const double* t = d->tel_xyzr + 4 * i;
            const int r0 = std::max((int)floor((t[1] - r - y0) / cell), 0), r1 = std::min((int)floor((t[1] + r - y0) / cell), gny - 1);
            for (int row = r0; row <= r1; ++row) {
                const double dy = fmax(fmax(y0 + row * cell - t[1], t[1] - (y0 + (row + 1) * cell)), 0.0);
                const double half = sqrt(fmax(r * r - dy * dy, 0.0));
                const int c0 = std::max((int)floor((t[0] - half - x0) / cell), 0);
                const int c1 = std::min((int)floor((t[0] + half - x0) / cell), gnx - 1);
                if (c0 <= c1) f(row, c0, c1);
            }
        };
        range[level].resize(n_cells * cs::kHashSubs);
        std::vector<int> fill(n_cells);
        for (int sub = 0; sub < cs::kHashSubs; ++sub) {
            int2* er = range[level].data() + sub * n_cells;
            std::fill(fill.begin(), fill.end(), 0);
            for (int i = 0; i < d->n_tel; ++i) {
                for_rows(i, reach(i, kHashTheta[level][sub] * kDeg) + slack, [&](int row, int c0, int c1) {
                    for (int c = c0; c <= c1; ++c) ++fill[(size_t)row * gnx + c];
                });
            }
            int at = (int)cell_tel[level].size();
            for (size_t c = 0; c < n_cells; ++c) {
                er[c] = make_int2(at, at + fill[c]);
                at += fill[c];
                fill[c] = er[c].x;
            }
            cell_tel[level].resize(at);
            cell_data[level].resize(at);
            for (int i = 0; i < d->n_tel; ++i) {   // ascending index within every cell
                const double* t = d->tel_xyzr + 4 * i;
                for_rows(i, reach(i, kHashTheta[level][sub] * kDeg) + slack, [&](int row, int c0, int c1) {
                    for (int c = c0; c <= c1; ++c) {
                        const int e = fill[(size_t)row * gnx + c]++;
                        cell_tel[level][e] = i;
                        cell_data[level][e] = p.spherical ? tel3[i]
                                                          : make_float4((float)(t[0] - (x0 + (double)c * cell)),
                                                                        (float)(t[1] - (y0 + (double)row * cell)),
                                                                        (float)(t[2] - d->h_obs), (float)t[3]);
                    }
                });
            }
        }
        H.gx0 = (float)x0;
        H.gy0 = (float)y0;
        H.cell = (float)cell;
        H.inv_cell = (float)(1.0 / cell);
        H.gnx = gnx;
        H.gny = gny;
        H.n_cells = (int)n_cells;
        // on the sphere the local vertical at a ground point in the box leans from
        // the frame's z axis by up to the box's extent / r_g: photons steeper than
        // a list's zenith in the local frame must be steeper in the frame's too
        double lean = 0.0;
        if (p.spherical) {
            const double ex = fmax(fabs(x0), fabs(x0 + gnx * cell)), ey = fmax(fabs(y0), fabs(y0 + gny * cell));
            lean = 1.01 * sqrt(ex * ex + ey * ey) / (p.R + d->h_obs) + 1e-6;
        }
        for (int sub = 0; sub < cs::kHashSubs; ++sub) {
            const double theta = fmax(kHashTheta[level][sub] * kDeg - lean, 0.0);
            (sub + 1 < cs::kHashSubs ? H.sub_sin2[sub] : H.sin2_max) = (float)(sin(theta) * sin(theta));
        }
    }
    const size_t o_tel = 0;
    const size_t o_lo = align_up(o_tel + tel.size() * sizeof(float4));
    const size_t o_t3 = align_up(o_lo + tel_lo.size() * sizeof(float2));
    size_t o_rg[cs::kHashLevels], o_ct[cs::kHashLevels], o_cd[cs::kHashLevels], end = align_up(o_t3 + tel3.size() * sizeof(float4));
    for (int level = 0; level < cs::kHashLevels; ++level) {
        o_rg[level] = end;
        o_ct[level] = align_up(o_rg[level] + (range[level].size() + 1) * sizeof(int2));
        o_cd[level] = align_up(o_ct[level] + (cell_tel[level].size() + 1) * sizeof(int));
        end = align_up(o_cd[level] + (cell_data[level].size() + 1) * sizeof(float4));
    }
    const size_t total = end;
    cudaError_t e = cudaMalloc(&h->d_mem, total);
    if (e != cudaSuccess) { cs::set_last_error("detector alloc", e); delete h; return CS_ERR_CUDA; }
    char* base = (char*)h->d_mem;
    std::vector<char> host(total, 0);
    if (!tel.empty()) memcpy(host.data() + o_tel, tel.data(), tel.size() * sizeof(float4));
    if (!tel_lo.empty()) memcpy(host.data() + o_lo, tel_lo.data(), tel_lo.size() * sizeof(float2));
    if (!tel3.empty()) memcpy(host.data() + o_t3, tel3.data(), tel3.size() * sizeof(float4));
    for (int level = 0; level < cs::kHashLevels; ++level) {
        if (!range[level].empty()) memcpy(host.data() + o_rg[level], range[level].data(), range[level].size() * sizeof(int2));
        if (!cell_tel[level].empty())
            memcpy(host.data() + o_ct[level], cell_tel[level].data(), cell_tel[level].size() * sizeof(int));
        if (!cell_data[level].empty())
            memcpy(host.data() + o_cd[level], cell_data[level].data(), cell_data[level].size() * sizeof(float4));
    }
    e = cudaMemcpy(h->d_mem, host.data(), total, cudaMemcpyHostToDevice);
    if (e != cudaSuccess) { cs::set_last_error("detector copy", e); cudaFree(h->d_mem); delete h; return CS_ERR_CUDA; }
    p.tel = (const float4*)(base + o_tel);
    p.tel_lo = (const float2*)(base + o_lo);
    p.tel3 = p.spherical ? (const float4*)(base + o_t3) : nullptr;
    for (int level = 0; level < cs::kHashLevels; ++level) {
        p.hash[level].cell_range = (const int2*)(base + o_rg[level]);
        p.hash[level].cell_tel = (const int*)(base + o_ct[level]);
        p.hash[level].cell_data = (const float4*)(base + o_cd[level]);
    }
    *out = h;
    return CS_OK;
}

extern "C" void cs_detector_destroy(cs_detector* det) {
    if (!det) return;
    cudaFree(det->d_mem);
    delete det;
}
