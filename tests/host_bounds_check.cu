// Host-side check of the closest-point search's bounds (no kernel is launched;
// runs on any machine): the cap that the scene builder puts around a patch of
// primitives lies at or below the distance of every primitive in it, less what
// FP32 rounds off that distance, for needles and slabs of any aspect at any
// rotation, seen from inside the scene and from far outside it.  Prints "ok" and exits 0 when every check holds.
#include <cstdio>
#include <random>

#include "../paper_2410_18944_gb300/csrc/scene.cu"

namespace wost {
void set_error(const std::string &) {}
wost_status cuda_status(cudaError_t, const char *) { return WOST_ERR_CUDA; }
void DevBuf::release() {}
}  // namespace wost

using namespace wost;

namespace {

using Vec = std::vector<double>;

double dot(const double *a, const double *b, int d) {
    double s = 0;
    for (int k = 0; k < d; ++k) s += a[k] * b[k];
    return s;
}

// distance from p to the segment ab, and (3D) to the triangle abc
double seg_dist(const double *a, const double *b, const double *p, int d) {
    double e[3], r[3], s = 0;
    for (int k = 0; k < d; ++k) { e[k] = b[k] - a[k]; r[k] = p[k] - a[k]; }
    const double ee = dot(e, e, d), t = ee > 0 ? std::min(std::max(dot(r, e, d) / ee, 0.0), 1.0) : 0.0;
    for (int k = 0; k < d; ++k) s += (r[k] - t * e[k]) * (r[k] - t * e[k]);
    return std::sqrt(s);
}
double tri_dist(const double *a, const double *b, const double *c, const double *p) {
    double m = std::min(seg_dist(a, b, p, 3), std::min(seg_dist(b, c, p, 3), seg_dist(c, a, p, 3)));
    double u[3], v[3], r[3];
    for (int k = 0; k < 3; ++k) { u[k] = b[k] - a[k]; v[k] = c[k] - a[k]; r[k] = p[k] - a[k]; }
    const double n[3] = {u[1] * v[2] - u[2] * v[1], u[2] * v[0] - u[0] * v[2], u[0] * v[1] - u[1] * v[0]};
    const double nn = dot(n, n, 3), uu = dot(u, u, 3), uv = dot(u, v, 3), vv = dot(v, v, 3), den = uu * vv - uv * uv;
    if (!(nn > 0) || !(den > 0)) return m;
    const double s = (vv * dot(r, u, 3) - uv * dot(r, v, 3)) / den, t = (uu * dot(r, v, 3) - uv * dot(r, u, 3)) / den;
    if (s >= 0 && t >= 0 && s + t <= 1) m = std::min(m, std::fabs(dot(r, n, 3)) / std::sqrt(nn));
    return m;
}

// patches of up to 8 primitives with vertices in a rotated box whose sides are
// `len` along the first axes and len / aspect along the rest
int check_caps(int d, int patches, double reach, std::mt19937_64 &rng) {
    std::normal_distribution<double> normal;
    std::uniform_real_distribution<double> unit(0, 1);
    const double far = 2 * std::sqrt((double)d);   // of a scene in [-1, 1]^d
    int bad = 0;
    for (int t = 0; t < patches; ++t) {
        const double aspect = std::pow(10, 1 + 5 * unit(rng)), len = std::pow(10, -2 * unit(rng));
        double R[3][3], mid[3];
        for (int i = 0; i < d; ++i) {   // a random rotation: Gram-Schmidt
            for (int k = 0; k < d; ++k) R[i][k] = normal(rng);
            for (int j = 0; j < i; ++j) {
                const double q = dot(R[i], R[j], d);
                for (int k = 0; k < d; ++k) R[i][k] -= q * R[j][k];
            }
            const double n = std::sqrt(dot(R[i], R[i], d));
            for (int k = 0; k < d; ++k) R[i][k] /= n;
        }
        for (int k = 0; k < d; ++k) mid[k] = 0.5 * (2 * unit(rng) - 1);
        const int n = 1 + (int)(8 * unit(rng)), longs = 1 + (int)((d - 1) * unit(rng));
        // the mean normal: along a short side, along the first long one, or random
        const int axis = (int)(3 * unit(rng));
        std::vector<float> P, N;
        for (int i = 0; i < n; ++i) {
            for (int j = 0; j < d; ++j) {
                double v[3] = {mid[0], mid[1], mid[2]};
                for (int a = 0; a < d; ++a) {
                    const double z = (a < longs ? len : len / aspect) * (2 * unit(rng) - 1);
                    for (int k = 0; k < d; ++k) v[k] += z * R[a][k];
                }
                for (int k = 0; k < d; ++k) P.push_back((float)v[k]);
            }
            for (int k = 0; k < d; ++k)
                N.push_back((float)(axis == 0 ? R[d - 1][k] : axis == 1 ? R[0][k] : 0.6 * R[0][k] + 0.8 * R[d - 1][k]));
        }
        const Cap c = cap_of(P, N, 0, n, d, 1e-6 * far);
        for (int q = 0; q < 16; ++q) {
            const double radius = q < 6 ? reach : (q < 11 ? len : 4 * len / aspect);
            float x[3] = {0, 0, 0};
            double xd[3] = {0, 0, 0};
            const int at = (int)(unit(rng) * n * d) * d;
            for (int k = 0; k < d; ++k) {   // (two along the cap's axis)
                const double step = q < 2 ? (double)c.a[k] * (q ? 1 : -1) : 2 * unit(rng) - 1;
                xd[k] = x[k] = (float)(P[at + k] + radius * step);
            }
            const double key = d == 2 ? cap_d2_2(make_float4(c.c[0], c.c[1], c.a[0], c.a[1]), c.h, c.r, x)
                                      : cap_d2_3(make_float4(c.c[0], c.c[1], c.c[2], c.h),
                                                 make_float4(c.a[0], c.a[1], c.a[2], c.r), x);
            for (int i = 0; i < n; ++i) {
                Vec v(P.begin() + (size_t)i * d * d, P.begin() + (size_t)(i + 1) * d * d);
                const double dist = d == 2 ? seg_dist(&v[0], &v[2], xd, 2) : tri_dist(&v[0], &v[3], &v[6], xd);
                // (the FP32 distance of a primitive: a difference of
                // coordinates, its products and their sum, each rounded)
                const double least = dist - 4 * std::ldexp(1.0, -24) * (far + dist);
                if (std::sqrt(key) > std::max(least, 0.0)) {
                    if (bad++ < 5)
                        std::printf("%dD, aspect %g: cap at %.9g, primitive at %.9g\n", d, aspect, std::sqrt(key), dist);
                }
            }
        }
    }
    return bad;
}

}  // namespace

int main() {
    std::mt19937_64 rng(11);
    int bad = 0;
    for (double reach : {1.0, 30.0, 1000.0})   // from points of the scene, and from outside
        for (int d = 2; d <= 3; ++d) bad += check_caps(d, 20000, reach, rng);
    if (bad) {
        std::printf("%d bounds above their primitives\n", bad);
        return 1;
    }
    std::printf("ok\n");
    return 0;
}
