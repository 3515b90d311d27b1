// bs_vel_exact.cu -- instances of the velocity kernel whose near pairs take the exact integral of Eq. 1
// over the tet (near_rule = BS_NEAR_EXACT), both precisions.
#include "bs_velocity_kernel.cuh"

namespace bs {
namespace {

#define BS_V(T, Q, P, TILE, S, MINB, INL) \
    { {P, TILE, S, MINB, INL, 1, false, 1}, &launch_t<T, Q, P, 128, TILE, S, MINB, INL, true, 1, false, 1> }

const VariantEntry kF32Q1[] = {BS_V(float, 1, 2, 32, 4, 4, true)};
const VariantEntry kF32Q4[] = {BS_V(float, 4, 3, 32, 2, 4, true), BS_V(float, 4, 1, 32, 4, 5, false)};
const VariantEntry kF32Q8[] = {BS_V(float, 8, 2, 16, 4, 4, true)};
const VariantEntry kF32Q27[] = {BS_V(float, 27, 1, 16, 4, 4, false)};
const VariantEntry kF32Q64[] = {BS_V(float, 64, 1, 8, 4, 4, false)};
const VariantEntry kF64Q1[] = {BS_V(double, 1, 2, 32, 4, 4, true)};
const VariantEntry kF64Q4[] = {BS_V(double, 4, 1, 32, 2, 4, true), BS_V(double, 4, 2, 32, 2, 3, true)};
const VariantEntry kF64Q8[] = {BS_V(double, 8, 2, 16, 4, 4, true)};
const VariantEntry kF64Q27[] = {BS_V(double, 27, 1, 16, 4, 4, false)};
const VariantEntry kF64Q64[] = {BS_V(double, 64, 1, 8, 4, 4, false)};
#undef BS_V

template <size_t N>
VariantList list(const VariantEntry (&v)[N])
{
    return {v, (int)N};
}

// One thread per tet: the table's values in float64, in units of the tet (its longest edge and largest vorticity brought
// to at most 1 by powers of two).  Bound by the float64 pipe, on which a division takes as long as ten products: the
// two-float table, whose words round at 2^-48, takes a reciprocal root per face and edge instead; the double one is
// rounded division by division (with the reciprocals its errors against 113 bits grow by a tenth).  1.5M tets: 3.24 ms
// (two-float), 2.36 ms (double); 2000 points of a 64^3 mesh that moves, two-float, 14.1 -> 13.4 ms a call.
template <typename R>
__global__ void exact_table_kernel(const double *__restrict__ near64, int64_t n_tets, R *__restrict__ table)
{
    constexpr bool TWO = std::is_same<R, dfl>::value;
    const int64_t tet = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (tet >= n_tets) return;
    const double *r = near64 + tet * kNearF64;
    R *t = table + tet * kExactTable;
    double wmax = 0.0;
    for (int i = 0; i < 12; ++i) wmax = fmax(wmax, fabs(r[nf64::W + i]));
    const int k = min(max(ilogb(r[nf64::H]) + 1, -1000), 1000);
    const int kw = wmax > 0.0 && wmax < (double)INFINITY ? min(max(ilogb(wmax) + 1, -1000), 1000) : 0;
    const double len = pow2_f64(-k), vort = pow2_f64(-kw);
    auto put = [&](int i, double v) { t[i] = ex_make<R>(v); };
    V3<double> v[4], w[4], n[4];
    for (int i = 0; i < 4; ++i) {
        v[i] = mk(r[nf64::V + 3 * i] * len, r[nf64::V + 3 * i + 1] * len, r[nf64::V + 3 * i + 2] * len);
        w[i] = mk(r[nf64::W + 3 * i] * vort, r[nf64::W + 3 * i + 1] * vort, r[nf64::W + 3 * i + 2] * vort);
    }
    auto sub = [](V3<double> a, V3<double> b) { return mk(a.x - b.x, a.y - b.y, a.z - b.z); };
    auto cross = [](V3<double> a, V3<double> b) {
        return mk(a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x);
    };
    auto put3 = [&](int i, V3<double> a) {
        put(i, a.x);
        put(i + 1, a.y);
        put(i + 2, a.z);
    };
    V3<double> g[4];  // barycentric gradients, in units of 1 / length
    const double unlen = pow2_f64(k);
    for (int i = 1; i < 4; ++i)
        g[i] = mk(r[nf64::G + 3 * i - 3] * unlen, r[nf64::G + 3 * i - 2] * unlen, r[nf64::G + 3 * i - 1] * unlen);
    g[0] = mk(-(g[1].x + g[2].x + g[3].x), -(g[1].y + g[2].y + g[3].y), -(g[1].z + g[2].z + g[3].z));
    // G[a][b] = d omega_a / d y_b = sum_i (omega_i - omega_0)_a g_i,b
    const V3<double> w1 = sub(w[1], w[0]), w2 = sub(w[2], w[0]), w3 = sub(w[3], w[0]);
    const V3<double> Gr[3] = {mk(w1.x * g[1].x + w2.x * g[2].x + w3.x * g[3].x, w1.x * g[1].y + w2.x * g[2].y + w3.x * g[3].y,
                                 w1.x * g[1].z + w2.x * g[2].z + w3.x * g[3].z),
                              mk(w1.y * g[1].x + w2.y * g[2].x + w3.y * g[3].x, w1.y * g[1].y + w2.y * g[2].y + w3.y * g[3].y,
                                 w1.y * g[1].z + w2.y * g[2].z + w3.y * g[3].z),
                              mk(w1.z * g[1].x + w2.z * g[2].x + w3.z * g[3].x, w1.z * g[1].y + w2.z * g[2].y + w3.z * g[3].y,
                                 w1.z * g[1].z + w2.z * g[2].z + w3.z * g[3].z)};
    for (int a = 0; a < 3; ++a) put3(ex::G + 3 * a, Gr[a]);
    put3(ex::W0, w[0]);
    const V3<double> curl = mk(Gr[2].y - Gr[1].z, Gr[0].z - Gr[2].x, Gr[1].x - Gr[0].y);
    auto Gmul = [&](V3<double> a) { return mk(dot3(Gr[0], a), dot3(Gr[1], a), dot3(Gr[2], a)); };
    for (int f = 0; f < 4; ++f) {
        const double g2 = dot3(g[f], g[f]), gn = TWO ? rsqrt(g2) : 1.0 / sqrt(g2);
        n[f] = mk(-g[f].x * gn, -g[f].y * gn, -g[f].z * gn);  // outward: lambda_f grows inwards
        put3(ex::N + 3 * f, n[f]);
        const V3<double> Nk = cross(n[f], Gmul(n[f]));
        put3(ex::V + 3 * f, mk(Nk.x - 0.5 * curl.x, Nk.y - 0.5 * curl.y, Nk.z - 0.5 * curl.z));
    }
    for (int e = 0; e < 6; ++e) {
        const int ev = ex::edge_vertices(e), a = ev & 3, b = ev >> 2 & 3;
        const V3<double> d = sub(v[b], v[a]);
        const double L2 = dot3(d, d);
        double L;
        V3<double> tan;
        if constexpr (TWO) {
            const double iL = rsqrt(L2);
            L = L2 * iL;
            tan = mk(d.x * iL, d.y * iL, d.z * iL);
        } else {
            L = sqrt(L2);
            tan = mk(d.x / L, d.y / L, d.z / L);
        }
        put3(ex::EDGE * e + ex::T, tan);
        put(ex::EDGE * e + ex::L, L);
        V3<double> U = mk(0.0, 0.0, 0.0);
        for (int o = 0; o < 2; ++o) {
            const int f = ev >> (4 + 2 * o) & 3, third = ev >> (6 - 2 * o) & 3;
            V3<double> m = cross(tan, n[f]);  // pointing away from the face's third vertex
            if (dot3(m, sub(v[third], v[a])) > 0.0) m = mk(-m.x, -m.y, -m.z);
            put3(ex::EDGE * e + ex::M + 3 * o, m);
            const V3<double> c = cross(n[f], Gmul(m));
            U = mk(U.x + 0.5 * c.x, U.y + 0.5 * c.y, U.z + 0.5 * c.z);
        }
        put3(ex::EDGE * e + ex::U, U);
        put(ex::EDGE * e + ex::EDGE - 1, 0.0);
    }
    *reinterpret_cast<int2 *>(t + ex::EXP) = make_int2(k, kw);
    put(ex::EXP + 1, 0.0);
}

}  // namespace

cudaError_t build_exact_table(const double *near64, int64_t n_tets, int precision, void *table, cudaStream_t st)
{
    const unsigned nb = (unsigned)((n_tets + 127) / 128);
    if (precision == BS_FP32) exact_table_kernel<dfl><<<nb, 128, 0, st>>>(near64, n_tets, reinterpret_cast<dfl *>(table));
    else exact_table_kernel<double><<<nb, 128, 0, st>>>(near64, n_tets, reinterpret_cast<double *>(table));
    return cudaGetLastError();
}

VariantList variants_exact(int precision, int Q)
{
    const bool f32 = precision == BS_FP32;
    switch (Q) {
    case 1: return f32 ? list(kF32Q1) : list(kF64Q1);
    case 4: return f32 ? list(kF32Q4) : list(kF64Q4);
    case 8: return f32 ? list(kF32Q8) : list(kF64Q8);
    case 27: return f32 ? list(kF32Q27) : list(kF64Q27);
    case 64: return f32 ? list(kF32Q64) : list(kF64Q64);
    default: return {};
    }
}

}  // namespace bs
